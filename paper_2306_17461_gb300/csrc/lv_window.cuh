// lv_window.cuh -- rounds of Algorithm 1 (Sec. 3.1, Appendix A) with the
// frontier and the strings' bytes at it held in registers, along the waves
// the frontier moves in.
//
// Off the alignment path the row of a diagonal is (nearly always) the row of
// the neighbour nearer to the path one round before: a cell reached from the
// path by one more insertion (diagonals above the path: the row of A stays,
// the row of B moves on by 1) or deletion (below it: the row of B stays).  A
// slot therefore holds not a fixed diagonal but a wave: the diagonal one
// further from the path every round.  Written for the diagonals above the
// path, with u the row of A and v = u + delta the row of B:
//
//     slot s holds diagonal delta = base + s + t in round t;
//     u_t[s] = max(u_{t-1}[s]        from delta - 1 (insertion),
//                  u_{t-1}[s + 1] + 1 from delta     (substitution),
//                  u_{t-1}[s + 2] + 1 from delta + 1 (deletion)),
//     clamped to the diagonal's last cell, then the slide.
//
// Below the path the same holds with the strings (and u, v) exchanged and
// delta = -d.  A slot's rows thus move on by a byte or two a round, and three
// aligned 4-byte words of each string kept from round to round (a window)
// serve its slides: about 0.4 loads of 4 bytes per diagonal and round.  With
// a slot per diagonal, the rows of successive rounds lie n / k bytes apart:
// four loads a round, each an L1 line of its own, of which the L1 serves one
// a cycle (4 to 9 cycles a diagonal and SM).
#pragma once
#include "ed_device.cuh"

namespace edg {

// A string as the windows read it: X4 = X rounded down to 4 bytes, s = X -
// X4, end = length + s.  A word is named by its byte offset from X4 and is
// loaded only when it overlaps the string (it then cannot fault).  A row r
// with r + s below `inner` (as unsigned numbers: no negative row is) has 31
// bytes or more after it: its window's words need no check of their own.
struct WinString {
    const uint8_t *x4;
    uint32_t s, end, inner;
};
__device__ __forceinline__ WinString win_string(const uint8_t *X, int32_t len)
{
    const uint32_t s = (uint32_t)((uintptr_t)X & 3u);
    return WinString{X - s, s, len > 0 ? (uint32_t)len + s : 0u, len > 31 ? (uint32_t)len + s - 31u : 0u};
}
__device__ __forceinline__ uint32_t win_word(const WinString &X, uint32_t off)
{
    return __ldg(reinterpret_cast<const uint32_t *>(X.x4 + off));
}

// E slots: their rows, and for each string the window's words and the offset
// of the first (WIN_NONE: no window).
constexpr uint32_t WIN_NONE = 0x80000000u;
template <int E>
struct Win {
    int32_t u[E];
    uint32_t a0[E], a1[E], a2[E], ba[E], b0[E], b1[E], b2[E], bb[E];
};

// w = the word at global address at + PLUS where p holds (a predicated load:
// no branch, so that several slots' instructions interleave).
template <int PLUS>
__device__ __forceinline__ void win_word_if(size_t at, bool p, uint32_t &w)
{
    asm("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.global.nc.u32 %0, [%1 + %3];\n\t}"
        : "+r"(w)
        : "l"(at), "r"((uint32_t)p), "n"(PLUS));
}

__device__ __forceinline__ uint32_t first_byte(uint32_t x) // index of the lowest nonzero byte; large for 0
{
    uint32_t tz;
    asm("bfind.shiftamt.u32 %0, %1;" : "=r"(tz) : "r"(__brev(x)));
    return tz >> 3;
}

// One round for the thread's slots, all of them inside their strings and far
// from their ends: x1, x2 the rows of the two slots after the thread's last.
// delta: the first slot's diagonal.  Returns false, with nothing changed,
// when a slot of the warp is not (careful_round then takes the round).
// slide: the bytes matched; open: the slots whose first eight bytes all
// matched (their row is the start row + 8 so far).  The whole warp calls it.
//
// No clamp, no bound and no band test here: a row this far from both ends
// cannot be clamped, and a slot outside the band has a negative row.  About
// 35 integer operations a slot (what bounds the rounds: lv_wide.cu).
template <int E>
__device__ __forceinline__ bool fast_round(Win<E> &w, int32_t x1, int32_t x2, const WinString &U, const WinString &V,
                                           int32_t delta, uint32_t &slide, uint32_t &open)
{
    int32_t c[E];
    uint32_t far = 0;
    bool ok = true;
    const uint32_t sv = (uint32_t)delta + V.s;
#pragma unroll
    for (int j = 0; j < E; j++) {
        const int32_t r1 = j + 1 < E ? w.u[j + 1 < E ? j + 1 : 0] : x1;
        const int32_t r2 = j + 2 < E ? w.u[j + 2 < E ? j + 2 : 0] : (j + 2 == E ? x1 : x2);
        c[j] = __viaddmax_s32(r2, 1, __viaddmax_s32(r1, 1, w.u[j]));
        const uint32_t ua = (uint32_t)c[j] + U.s, ub = (uint32_t)c[j] + (sv + j);
        ok = ok && ua < U.inner && ub < V.inner;
        if ((ua & ~3u) - w.ba[j] > 4u)
            far |= 1u << j;
        if ((ub & ~3u) - w.bb[j] > 4u)
            far |= 0x10000u << j;
    }
    if (__any_sync(0xffffffffu, !ok || far != 0)) {
        if (!__all_sync(0xffffffffu, ok))
            return false;
        // windows to load anew (a wave changed hands, or a long slide)
#pragma unroll
        for (int j = 0; j < E; j++) {
            const uint32_t wa = ((uint32_t)c[j] + U.s) & ~3u, wb = ((uint32_t)c[j] + (sv + j)) & ~3u;
            const bool fa = (far >> j) & 1u, fb = (far >> (16 + j)) & 1u;
            const size_t pa = __cvta_generic_to_global(U.x4) + wa, pb = __cvta_generic_to_global(V.x4) + wb;
            win_word_if<0>(pa, fa, w.a0[j]);
            win_word_if<4>(pa, fa, w.a1[j]);
            win_word_if<8>(pa, fa, w.a2[j]);
            win_word_if<0>(pb, fb, w.b0[j]);
            win_word_if<4>(pb, fb, w.b1[j]);
            win_word_if<8>(pb, fb, w.b2[j]);
            w.ba[j] = fa ? wa : w.ba[j];
            w.bb[j] = fb ? wb : w.bb[j];
        }
    }
    uint32_t four = 0, sum = 0;
#pragma unroll
    for (int j = 0; j < E; j++) {
        const uint32_t ua = (uint32_t)c[j] + U.s, ub = (uint32_t)c[j] + (sv + j);
        const uint32_t wa = ua & ~3u, wb = ub & ~3u;
        // the window moves on by a word or not at all
        const bool na = wa != w.ba[j], nb = wb != w.bb[j];
        w.a0[j] = na ? w.a1[j] : w.a0[j];
        w.a1[j] = na ? w.a2[j] : w.a1[j];
        w.b0[j] = nb ? w.b1[j] : w.b0[j];
        w.b1[j] = nb ? w.b2[j] : w.b1[j];
        win_word_if<8>(__cvta_generic_to_global(U.x4) + wa, na, w.a2[j]);
        win_word_if<8>(__cvta_generic_to_global(V.x4) + wb, nb, w.b2[j]);
        w.ba[j] = wa;
        w.bb[j] = wb;
        // (the funnel shift takes the amount modulo 32)
        const uint32_t x = __funnelshift_r(w.a0[j], w.a1[j], 8u * ua) ^ __funnelshift_r(w.b0[j], w.b1[j], 8u * ub);
        const uint32_t l = min(first_byte(x), 4u);
        w.u[j] = c[j] + (int32_t)l;
        sum += l;
        if (x == 0u)
            four |= 1u << j;
    }
    open = 0;
    if (__any_sync(0xffffffffu, four != 0)) {
#pragma unroll
        for (int j = 0; j < E; j++) {
            const uint32_t ua = (uint32_t)c[j] + U.s, ub = (uint32_t)c[j] + (sv + j);
            const uint32_t y = __funnelshift_r(w.a1[j], w.a2[j], 8u * ua) ^ __funnelshift_r(w.b1[j], w.b2[j], 8u * ub);
            if ((four >> j) & 1u) {
                const uint32_t l = min(first_byte(y), 4u);
                w.u[j] += (int32_t)l;
                sum += l;
                if (y == 0u)
                    open |= 1u << j;
            }
            // the windows of these rows, for the next round (nothing waits for
            // them in this one; 12 bytes from a row 8 further are inside)
            const bool f = (four >> j) & 1u;
            const uint32_t wa = ((uint32_t)w.u[j] + U.s) & ~3u, wb = ((uint32_t)w.u[j] + (sv + j)) & ~3u;
            const size_t pa = __cvta_generic_to_global(U.x4) + wa, pb = __cvta_generic_to_global(V.x4) + wb;
            win_word_if<0>(pa, f, w.a0[j]);
            win_word_if<4>(pa, f, w.a1[j]);
            win_word_if<8>(pa, f, w.a2[j]);
            win_word_if<0>(pb, f, w.b0[j]);
            win_word_if<4>(pb, f, w.b1[j]);
            win_word_if<8>(pb, f, w.b2[j]);
            w.ba[j] = f ? wa : w.ba[j];
            w.bb[j] = f ? wb : w.bb[j];
        }
    }
    slide = sum;
    return true;
}

// The first eight bytes of string X from row r on (r >= 0, inside the
// string); bytes past its end are unspecified, the caller's bound masks them.
__device__ __forceinline__ uint64_t win_eight(const WinString &X, int32_t r)
{
    const uint32_t u = (uint32_t)r + X.s, o = u & ~3u;
    const uint32_t w0 = o < X.end ? win_word(X, o) : 0u;
    const uint32_t w1 = o + 4u < X.end ? win_word(X, o + 4u) : 0u;
    const uint32_t w2 = o + 8u < X.end ? win_word(X, o + 8u) : 0u;
    return ((uint64_t)__funnelshift_r(w1, w2, 8u * u) << 32) | __funnelshift_r(w0, w1, 8u * u);
}

// The same round with every bound tested: slots at the band's edges [lo, hi]
// (outside: minus infinity) and near the strings' ends; only the first kmax
// slots of the thread slide (the others are not needed any more).  mism: the
// slides that ended on a mismatch; open as in fast_round.
template <int E>
__device__ __forceinline__ void careful_round(Win<E> &w, int32_t x1, int32_t x2, const WinString &U,
                                              const WinString &V, int32_t N, int32_t M, int32_t delta, int32_t lo,
                                              int32_t hi, int32_t kmax, uint32_t &slide, uint32_t &mism,
                                              uint32_t &open)
{
    slide = mism = open = 0;
    const int32_t u0 = w.u[0];
    int32_t r0 = u0;
#pragma unroll
    for (int j = 0; j < E; j++) {
        const int32_t r1 = j + 1 < E ? w.u[j + 1 < E ? j + 1 : 0] : x1;
        const int32_t r2 = j + 2 < E ? w.u[j + 2 < E ? j + 2 : 0] : (j + 2 == E ? x1 : x2);
        const int32_t dl = delta + j, lim = min(N, M - dl);
        const int32_t c = min(max(r0, max(r1, r2) + 1), lim), full = lim - c;
        r0 = r1; // (slot j + 1's own row, before it is overwritten)
        w.ba[j] = w.bb[j] = WIN_NONE;
        w.u[j] = NEG;
        if (dl >= lo && dl <= hi && c >= 0 && c + dl >= 0) {
            int32_t l = 0;
            if (j < kmax && full > 0) {
                const uint64_t z = win_eight(U, c) ^ win_eight(V, c + dl);
                l = min(z ? (__ffsll((long long)z) - 1) >> 3 : 8, full);
                if (l == 8 && full > 8)
                    open |= 1u << j;
                slide += (uint32_t)l;
                mism += l < full;
            }
            w.u[j] = c + l;
        }
    }
}

} // namespace edg
