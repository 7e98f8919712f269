// One CTA claims from a job slot that the host has filled, through each of the
// claim loops of lv_tiles.cu, and the slot's answer words are printed:
//
//     claim_probe LOOP ID TAG SMALL
//
// LOOP 1 or 2 (claim_loop, claim_loop2), the claim word's job id, the id that
// the descriptor words carry, and whether the job goes in small chunks.  The
// strings differ at offset 100.  Prints the number of claims made, and for each
// answer word that is not zero "chunk id offset".
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "../paper_2306_17461_gb300/csrc/lv_tiles.cu"

using namespace edg;

__device__ LaunchCtl g_ctl;

__global__ void __launch_bounds__(CTA_THREADS) probe_kernel(JobSlot *slot, const PairDesc *pairs, int loop, int *made)
{
    const Smem S{GRID_SMAX, 2};
    LvArgs P{};
    P.spin_ns = 2000000000ull;
    P.pairs = pairs;
    P.ctl = &g_ctl;
    P.stage = 2;
    if (threadIdx.x == 0) {
        S.jd()->jid = 0;
        S.jd()->slot = -1;
        S.jd()->pq = -1;
        for (int i = 0; i < 2; i++) {
            const Stage T = stage_of(S.stg() + i * STAGE_STRIDE);
            mbar_init(T.bar, 1);
            *T.phase = 0;
        }
        fence_mbar_init();
    }
    __syncthreads();
    const int n = loop == 2 ? claim_loop2(P, S, slot, 0, 8, nullptr) : claim_loop(P, S, slot, 0, 0ull, 8);
    if (threadIdx.x == 0)
        *made = n;
}

static void ck(cudaError_t e)
{
    if (e != cudaSuccess) {
        std::fprintf(stderr, "%s\n", cudaGetErrorString(e));
        std::exit(1);
    }
}

int main(int argc, char **argv)
{
    if (argc != 5)
        return 2;
    const int loop = std::atoi(argv[1]), small = std::atoi(argv[4]);
    const unsigned long long id = std::strtoull(argv[2], nullptr, 10) << 32, tag = std::strtoull(argv[3], nullptr, 10) << 32;
    const int64_t n = 40000, lim = 39000;
    std::vector<uint8_t> a(n, 1), b(n, 1);
    b[3 + 100] = 2; // (the slide starts at rows 2 of A and 3 of B)
    uint8_t *A, *B;
    JobSlot *slot;
    PairDesc *pairs;
    int *made;
    ck(cudaMalloc(&A, n));
    ck(cudaMalloc(&B, n));
    ck(cudaMalloc(&slot, sizeof(JobSlot)));
    ck(cudaMalloc(&pairs, sizeof(PairDesc)));
    ck(cudaMalloc(&made, sizeof(int)));
    ck(cudaMemcpy(A, a.data(), n, cudaMemcpyHostToDevice));
    ck(cudaMemcpy(B, b.data(), n, cudaMemcpyHostToDevice));
    PairDesc pd{};
    pd.A = A;
    pd.B = B;
    pd.n = pd.m = n;
    ck(cudaMemcpy(pairs, &pd, sizeof(pd), cudaMemcpyHostToDevice));
    std::vector<JobSlot> s(1);
    std::memset((void *)s.data(), 0, sizeof(JobSlot));
    s[0].claim = id;
    s[0].xt = tag | 2;
    s[0].yt = tag | 3;
    s[0].lt = tag | (uint32_t)lim;
    s[0].pt = tag | (uint32_t)small << 31;
    s[0].result = tag | (uint32_t)~(uint32_t)lim;
    ck(cudaMemcpy(slot, s.data(), sizeof(JobSlot), cudaMemcpyHostToDevice));
    const size_t smem = lv_tiles_smem_bytes(GRID_SMAX, 0, 2);
    ck(cudaFuncSetAttribute(probe_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    probe_kernel<<<1, CTA_THREADS, smem>>>(slot, pairs, loop, made);
    ck(cudaGetLastError());
    ck(cudaDeviceSynchronize());
    int m = 0;
    ck(cudaMemcpy(&m, made, sizeof(int), cudaMemcpyDeviceToHost));
    ck(cudaMemcpy(s.data(), slot, sizeof(JobSlot), cudaMemcpyDeviceToHost));
    std::printf("made %d\n", m);
    for (int c = 0; c < JOB_MAX_CHUNKS; c++)
        if (s[0].ans[c])
            std::printf("%d %u %u\n", c, (unsigned)(s[0].ans[c] >> 32), (unsigned)s[0].ans[c]);
    return 0;
}
