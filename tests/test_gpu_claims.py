"""The claims of a long slide's chunks: a claimer answers only for bytes that
it has compared, or that lie past the end or past a mismatch already reported.
claim_probe.cu drives the two claim loops on a job slot filled by hand."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_2306_17461_gb300 import build

    exe = str(tmp_path_factory.mktemp("claims") / "claim_probe")
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, os.path.join(HERE, "claim_probe.cu"), "-o", exe],
                   check=True, capture_output=True)

    def run(*args):
        out = subprocess.run([exe, *map(str, args)], check=True, capture_output=True, text=True, timeout=60).stdout
        lines = out.split("\n")
        return int(lines[0].split()[1]), {tuple(map(int, l.split())) for l in lines[1:] if l}

    return run


@pytest.mark.parametrize("small", [0, 1], ids=["staged", "small"])
@pytest.mark.parametrize("loop", [1, 2])
def test_chunks_not_compared_are_not_answered(probe, loop, small):
    # the descriptor is the claim's: chunk 0 is answered with its mismatch
    made, ans = probe(loop, 2, 2, small)
    assert made >= 1 and (0, 2, 100) in ans
    # it is still on its way (its words are an older job's): no answer at all,
    # so that the owner compares the chunk itself
    assert probe(loop, 2, 1, small) == (0, set())
    # the claim's job is over (the words are a later job's): nothing to answer
    assert probe(loop, 2, 3, small) == (0, set())
