// lv_wide.cu -- Algorithm 1 (Sec. 3.1, Appendix A) for wide bands, in one
// persistent cooperative launch: rounds over many diagonals a CTA, with the
// frontier and the strings' bytes at it in registers (lv_window.cuh).
//
// The single-pair kernel of lv_tiles.cu is built for narrow bands: rounds
// bound by their latency, long slides spread over idle CTAs.  Batched and
// served pairs whose band has outgrown one CTA of the batch kernel go on here
// from its frontier; single pairs stay there, however wide (n = 10^8, k = 10^5
// handed over at 386 diagonals a CTA: 303 to 308 ms against 288).
//
// What bounds these rounds: the warps wait for one another.  152 pairs of
// 40 thousand characters, k = 6400, one CTA each (45 ms, 2.5 cycles a diagonal
// and SM; 1.8 in the rounds of a batch of 4096, on groups of CTAs): 42 % of a warp's time at the
// CTA's barriers (a warp with the path's slide or a checked round holds up the
// other 15, by the code), 20 % for its own last instruction; a scheduler of
// four warps issues in 42 % of its cycles, the integer pipe is busy 43 %, L1
// 17 %, and HBM not at all.  With the halo, the warps' overlap and the checked
// rounds a diagonal takes 123 instructions.
//
// GB300 mapping.
//  * A group of CTAs splits the diagonals [-R, R] into one tile per CTA; R (the
//    epoch radius) grows by an eighth and the tiles are then cut again through
//    a global buffer.
//  * Temporal blocking: a CTA runs h rounds on its tile plus h halo diagonals
//    a side, then trades h edge values with its neighbours through global
//    memory, each in one 8-byte word with its round (no fence, no flag).
//  * Within a block the diagonals below and above the alignment path run
//    through their h rounds in registers, 512 threads holding 1 to 4 waves
//    each (win_block; several passes when the tile is wider).  Warps run 8
//    rounds at a time without a barrier; the long slide of the alignment path
//    stalls its warps alone meanwhile.
//  * Every wait is bounded by %globaltimer and reports ST_TIMEOUT.
#include "ed_device.cuh"
#include "lv_kernels.cuh"
#include "lv_window.cuh"

namespace edg {

constexpr int WT = WIDE_THREADS;
constexpr int NWARP = WT / 32;
constexpr int SEG_MAX = 8;  // rounds between the warps' exchanges, at most
constexpr int OCAP = 256;   // slides of a round listed for the whole CTA

struct WideSmem {
    int32_t ex[2][NWARP][2 * SEG_MAX]; // the warps' first rows, by segment parity
    // slides that outran their warp: diagonal, row reached, final row
    int32_t ld[OCAP], lc[OCAP], lr[OCAP];
    int32_t nl;
    int32_t kf;  // the round that reached row n on d = m - n, or INT32_MAX
    int32_t bc[4];
    unsigned long long smin, lead;
    unsigned long long slide, mism, opens; // of the pair, this CTA's share
    int32_t *tile; // this CTA's frontier buffers
    // the pair
    const uint8_t *A, *B;
    int32_t n, m;
    int32_t cap; // bytes one warp compares before the whole CTA takes a slide
};

// The CTA's tile between blocks lies in global memory (read and written once
// a block of h rounds; it stays in L2), so that the L1 keeps the strings'
// bytes: two frontier buffers, read and written in turn; index d - a + h + 1.
size_t lv_wide_tile_words(int smax) { return 2 * ((size_t)smax + 2 * HMAX + 2); }

extern __shared__ __align__(16) unsigned char wide_raw[];
__device__ __forceinline__ WideSmem &wsm() { return *reinterpret_cast<WideSmem *>(wide_raw); }
__device__ __forceinline__ int32_t *wbuf(int i, int smax) { return wsm().tile + i * (smax + 2 * HMAX + 2); }

// The listed slides through the whole CTA, 16 KiB of each string a step; the
// same slide listed twice (by a warp that holds it in its halo) runs once.
// Every thread must call it, after a barrier; the final rows are visible to
// every thread when it returns.
__device__ __noinline__ void wide_slides(int nl)
{
    WideSmem &S = wsm();
    const int tid = threadIdx.x;
    constexpr int64_t STEP = (int64_t)WT * 16 * 2;
    for (int j = 0; j < nl; j++) {
        const int32_t d = S.ld[j], c = S.lc[j];
        int i = 0;
        while (S.ld[i] != d || S.lc[i] != c)
            i++;
        if (i < j) {
            if (tid == 0)
                S.lr[j] = S.lr[i];
            continue;
        }
        const int64_t lim = min((int64_t)S.n, (int64_t)S.m - d) - c;
        int64_t l = lim;
        for (int64_t off = 0; off < lim; off += STEP) {
            const int64_t r = cta_scan<2>(S.A, S.n, S.B, S.m, c, (int64_t)c + d, off, min(STEP, lim - off), &S.smin);
            if (r >= 0) {
                l = r;
                break;
            }
        }
        if (tid < 32)
            prefetch_next(S.A, S.n, S.B, S.m, c + l, c + l + d);
        if (tid == 0) {
            S.lr[j] = c + (int32_t)l;
            S.slide += (unsigned long long)l;
            S.mism += l < lim;
        }
    }
    __syncthreads();
}

// The slides of a warp's diagonals that eight equal bytes left open, one
// diagonal (d, row p reached) per lane that wants it; the whole warp calls
// it.  A lane compares 16 more bytes in one round trip (chance matches end
// there), unless the warp's last slide was a long one (hot: the alignment
// path's, every round); the warp then takes each slide still open, up to
// S.cap bytes, and lists one that outruns it for the whole CTA.  Returns the
// lane's row; *listed is set when it is not final yet.
__device__ __noinline__ int32_t wide_open(int32_t p, int32_t d, bool want, bool own, bool hot, bool *listed)
{
    WideSmem &S = wsm();
    const int lane = threadIdx.x & 31;
    const uint8_t *A = S.A, *B = S.B;
    const int64_t n = S.n, m = S.m;
    const int32_t lim = (int32_t)min(n, m - d), full = lim - p;
    const int32_t p0 = p;
    bool still = want;
    *listed = false;
    if (want && !hot) {
        const uintptr_t pa = (uintptr_t)(A + p), pb = (uintptr_t)(B + ((int64_t)p + d));
        const uintptr_t qa = pa & ~(uintptr_t)15, qb = pb & ~(uintptr_t)15;
        const uint4 a0 = ld_blk_nb(A, n, qa), a1 = ld_blk_nb(A, n, qa + 16);
        const uint4 b0 = ld_blk_nb(B, m, qb), b1 = ld_blk_nb(B, m, qb + 16);
        const int32_t f = min(full, (int32_t)first_diff16(shift_bytes(a0, a1, (uint32_t)(pa & 15)),
                                                          shift_bytes(b0, b1, (uint32_t)(pb & 15))));
        still = f == 16 && full > 16;
        p += f;
    }
    unsigned int st = __ballot_sync(0xffffffffu, still);
    while (st) {
        const int src = __ffs((int)st) - 1;
        st &= st - 1;
        const int32_t c = __shfl_sync(0xffffffffu, p, src), e = __shfl_sync(0xffffffffu, d, src);
        const int64_t left = __shfl_sync(0xffffffffu, lim, src) - c;
        bool open;
        int64_t l = slide_warp<2>(A, n, B, m, c, (int64_t)c + e, 0, left, S.cap, &open);
        if (open) { // to the list; when it is full the warp goes on alone
            int slot = 0;
            if (lane == 0)
                slot = atomicAdd(&S.nl, 1);
            slot = __shfl_sync(0xffffffffu, slot, 0);
            if (slot < OCAP) {
                if (lane == src) {
                    S.ld[slot] = e;
                    S.lc[slot] = c;
                    *listed = true;
                }
                l = 0;
            } else {
                l = slide_warp<2>(A, n, B, m, c, (int64_t)c + e, l, left, INT64_MAX / 4, &open);
            }
        }
        if (l >= PREFETCH_MIN) // a long slide: the next round starts past it
            prefetch_next(A, n, B, m, c + l, c + l + e);
        if (lane == src)
            p = c + (int32_t)l;
    }
    if (own) { // (the round counted eight bytes and a mismatch)
        atomicAdd(&S.opens, 1ull);
        if (p > p0)
            atomicAdd(&S.slide, (unsigned long long)(p - p0));
        if (*listed || p == lim)
            atomicAdd(&S.mism, ~0ull);
    }
    return p;
}

// A pass: one or two strips of the tile, each on warps of its own.  Strip 0
// ([a0, b0), warps 0 .. n0-1) lies below the alignment path and runs with the
// strings exchanged, strip 1 ([a1, b1), the next n1 warps) above it.
struct Pass {
    int32_t a0, b0, n0, a1, b1, n1;
};

// Slots a warp owns: 32 * E less 2 * G, which overlap the next warp's.
__host__ __device__ constexpr int seg_rounds(int E) { return E == 1 ? 4 : 8; }
__host__ __device__ constexpr int warp_slots(int E) { return 32 * E - 2 * seg_rounds(E); }

// Rounds t .. t+h-1 on the strips of a pass, each with its halo: a strip's
// slots are the waves that end the block on its diagonals (lv_window.cuh),
// and 2h more at the far end, whose diagonals the strip leaves; E slots a
// thread.  src and dst are the frontiers of rounds t-1 and t+h-1
// (indexed d - off; only the strips' diagonals are written).
//
// A warp's last 2G slots are the first of the next warp's: it runs segments
// of G rounds with no barrier, each round's slots reaching two less far, then
// the warps hand on those rows through shared memory at one CTA barrier.  That
// barrier also tells whether any thread found k or listed a slide; the whole
// CTA then runs the listed slides, and the warps that listed them go on with
// their segment.  Returns the round at which d = m - n reached row n, or -1.
template <int E>
__device__ __noinline__ int32_t win_block(const int32_t *src, int32_t *dst, int32_t off, int32_t t, int32_t h,
                                          const Pass Q)
{
    constexpr int G = seg_rounds(E), OWN = warp_slots(E), HT = 2 * G / E;
    WideSmem &S = wsm();
    const int lane = threadIdx.x & 31;
    int warp = threadIdx.x >> 5;
    const int wex = warp; // the warp's place in the exchange
    const bool above = warp >= Q.n0, idle = warp >= Q.n0 + Q.n1;
    const bool last = warp == Q.n0 - 1 || warp >= Q.n0 + Q.n1 - 1;
    warp -= above ? Q.n0 : 0;
    const int32_t N = above ? S.n : S.m, M = above ? S.m : S.n;
    const WinString U = win_string(above ? S.A : S.B, N), V = win_string(above ? S.B : S.A, M);
    // the strip as diagonals delta = d (above) or -d: [a, b); the thread's
    // slots are s0 .. s0 + E - 1 of the strip's
    const int32_t a = above ? Q.a1 : 1 - Q.b0, b = above ? Q.b1 : 1 - Q.a0;
    const int32_t s0 = warp * OWN + lane * E;
    const bool own_lane = lane < 32 - HT;
    Win<E> w;
#pragma unroll
    for (int j = 0; j < E; j++) {
        // slots past the halo are never needed: any row will do
        const int32_t dl = min(a - h + s0 + j, b + h - 1), d = above ? dl : -dl;
        int32_t x = NEG;
        if (!idle) {
            x = src[d - off];
            if (!above && x >= 0)
                x += d;
            if (t == 0 && d == 0)
                x = -1; // the start cell comes by "substitution" from before the strings
        }
        w.u[j] = x;
        w.a0[j] = w.a1[j] = w.a2[j] = w.b0[j] = w.b1[j] = w.b2[j] = 0u;
        w.ba[j] = w.bb[j] = WIN_NONE;
    }
    // The slots across a call: written out and read back by hand, so that in
    // the rounds' own loop they stay in registers (a register allocated across
    // a call anywhere was spilled in that loop too: 46 local accesses a round).
    volatile uint32_t kept[9 * E];
    auto keep = [&]() {
#pragma unroll
        for (int j = 0; j < E; j++) {
            kept[j] = (uint32_t)w.u[j];
            kept[E + j] = w.ba[j];
            kept[2 * E + j] = w.bb[j];
            kept[3 * E + j] = w.a0[j];
            kept[4 * E + j] = w.a1[j];
            kept[5 * E + j] = w.a2[j];
            kept[6 * E + j] = w.b0[j];
            kept[7 * E + j] = w.b1[j];
            kept[8 * E + j] = w.b2[j];
        }
    };
    auto back = [&]() {
#pragma unroll
        for (int j = 0; j < E; j++) {
            w.u[j] = (int32_t)kept[j];
            w.ba[j] = kept[E + j];
            w.bb[j] = kept[2 * E + j];
            w.a0[j] = kept[3 * E + j];
            w.a1[j] = kept[4 * E + j];
            w.a2[j] = kept[5 * E + j];
            w.b0[j] = kept[6 * E + j];
            w.b1[j] = kept[7 * E + j];
            w.b2[j] = kept[8 * E + j];
        }
    };
    bool hot = false;
    uint32_t slide = 0, mism = 0, opens = 0;
    int32_t kfound = -1;
    for (int r0 = 0; r0 < h; r0 += G) {
        const int re = min(h, r0 + G);
        int r = idle ? re : r0;
        bool found = false; // a slot of the warp holds the end cell
        for (;;) {
            uint32_t pend = 0; // slots whose slide is listed
            int32_t dl = 0, kmax = 0; // of the round that listed them: the first slot's diagonal, slots needed
            while (r < re && !found) {
                uint32_t sl = 0, mi = 0, om = 0;
                int what = 0; // 0 go on, 1 outside the band, 2 careful, 3 open slides
                // the fast rounds, a loop of their own: nothing else competes
                // for its registers
                do {
                    const int32_t tau = t + r;
                    dl = a - h + s0 + r + 1;
                    const int32_t dw = dl - lane * E; // the warp's first diagonal
                    if (dw > min(tau, M) || dw + 32 * E - 1 < max(-tau, -N)) {
                        what = 1;
                        break;
                    }
                    const int32_t x1 = __shfl_down_sync(0xffffffffu, w.u[0], 1);
                    const int32_t x2 = __shfl_down_sync(0xffffffffu, w.u[E > 1 ? 1 : 0], E > 1 ? 1 : 2);
                    if (tau == 0 || !fast_round<E>(w, x1, x2, U, V, dl, sl, om)) {
                        what = 2;
                        break;
                    }
                    // the slots whose diagonal is the strip's count here (a
                    // thread across its edge counts all of its slots, or none)
                    const int32_t j0 = own_lane ? a - dl : E, j1 = b - dl;
                    if (2 * (min(j1, E) - max(j0, 0)) > E) {
                        slide += sl;
                        mism += E;
                    }
                    if (__any_sync(0xffffffffu, om != 0)) {
                        // slots whose first eight bytes matched: the warp takes
                        // each at once, 512 bytes a step (the alignment path's
                        // slide, nearly every round of its warp)
                        kmax = min(OWN + 2 * (re - 1 - r) - lane * E, b - a + 2 * (h - 1 - r) - s0);
                        om &= kmax >= E ? 0xffffffffu : (kmax > 0 ? (1u << kmax) - 1u : 0u);
                        unsigned int bal;
                        while ((bal = __ballot_sync(0xffffffffu, om != 0)) != 0) {
                            const int from = __ffs((int)bal) - 1, jl = __ffs((int)om) - 1;
                            int32_t p = 0;
#pragma unroll
                            for (int q = 0; q < E; q++)
                                p = q == jl ? w.u[q] : p;
                            const int32_t u0 = __shfl_sync(0xffffffffu, p, from);
                            const int32_t v0 = __shfl_sync(0xffffffffu, p + dl + jl, from);
                            const int64_t lim = min(N - u0, M - v0);
                            const uint8_t *X = above ? S.A : S.B, *Y = above ? S.B : S.A;
                            bool open;
                            const int64_t l = slide_warp<1>(X, N, Y, M, u0, v0, 0, lim, S.cap, &open);
                            if (open || l == lim) { // longer, or at a string's end
                                what = 3;
                                break;
                            }
                            if (l >= PREFETCH_MIN) // a long slide: the next round starts past it
                                prefetch_next(X, N, Y, M, u0 + l, v0 + l);
                            if (lane == from) {
                                const int32_t e = dl + jl, u = u0 + (int32_t)l;
                                if (jl >= j0 && jl < j1) {
                                    slide += (uint32_t)l;
                                    opens++;
                                }
                                const uint32_t wa = ((uint32_t)u + U.s) & ~3u, wb = ((uint32_t)(u + e) + V.s) & ~3u;
                                const size_t pa = __cvta_generic_to_global(U.x4) + wa,
                                             pb = __cvta_generic_to_global(V.x4) + wb;
                                const bool in = (uint32_t)u + U.s < U.inner && (uint32_t)(u + e) + V.s < V.inner;
#pragma unroll
                                for (int q = 0; q < E; q++)
                                    if (q == jl) {
                                        w.u[q] = u;
                                        win_word_if<0>(pa, in, w.a0[q]);
                                        win_word_if<4>(pa, in, w.a1[q]);
                                        win_word_if<8>(pa, in, w.a2[q]);
                                        win_word_if<0>(pb, in, w.b0[q]);
                                        win_word_if<4>(pb, in, w.b1[q]);
                                        win_word_if<8>(pb, in, w.b2[q]);
                                        w.ba[q] = in ? wa : WIN_NONE;
                                        w.bb[q] = in ? wb : WIN_NONE;
                                    }
                                om &= om - 1;
                            }
                        }
                        if (what)
                            break;
                    }
                } while (++r < re);
                if (what == 0)
                    break;
                if (what == 1) {
#pragma unroll
                    for (int j = 0; j < E; j++)
                        w.u[j] = NEG;
                    r++;
                    continue;
                }
                const int32_t tau = t + r;
                // slots still needed: of the segment, and of the strip
                kmax = min(OWN + 2 * (re - 1 - r) - lane * E, b - a + 2 * (h - 1 - r) - s0);
                const int32_t j0 = own_lane ? a - dl : E, j1 = b - dl;
                if (what == 2) {
                    const int32_t x1 = __shfl_down_sync(0xffffffffu, w.u[0], 1);
                    const int32_t x2 = __shfl_down_sync(0xffffffffu, w.u[E > 1 ? 1 : 0], E > 1 ? 1 : 2);
                    careful_round<E>(w, x1, x2, U, V, N, M, dl, max(-tau, -N), min(tau, M), kmax, sl, mi, om);
                    if (2 * (min(j1, E) - max(j0, 0)) > E) {
                        slide += sl;
                        mism += mi;
                    }
                }
                om &= kmax >= E ? 0xffffffffu : (kmax > 0 ? (1u << kmax) - 1u : 0u);
                if (__any_sync(0xffffffffu, om != 0)) {
                    keep();
                    do {
                        const int j = om ? __ffs((int)om) - 1 : 0;
                        const int32_t e = dl + j, d = above ? e : -e, p = (int32_t)kept[j], x = above ? p : p + e;
                        bool listed;
                        const unsigned int gb = __ballot_sync(0xffffffffu, om != 0);
                        const int32_t y = wide_open(x, d, om != 0, om != 0 && j >= j0 && j < j1,
                                                    hot && (gb & (gb - 1)) == 0, &listed);
                        hot = __any_sync(0xffffffffu, om != 0 && (y - x > 64 || listed));
                        if (om) {
                            kept[j] = (uint32_t)(p + (y - x));
                            kept[E + j] = kept[2 * E + j] = WIN_NONE;
                            pend |= listed ? 1u << j : 0u;
                        }
                        om &= om - 1;
                    } while (__any_sync(0xffffffffu, om != 0));
                    back();
                }
                if (__any_sync(0xffffffffu, pend != 0))
                    break;
                // (a row at its string's end is careful_round's, or a long slide's)
                bool f = false;
#pragma unroll
                for (int j = 0; j < E; j++)
                    f = f || (j < kmax && dl + j == M - N && w.u[j] == N);
                if (f)
                    atomicMin(&S.kf, tau);
                found = __any_sync(0xffffffffu, f);
                r++;
            }
            if (r == re && lane < HT) {
#pragma unroll
                for (int j = 0; j < E; j++)
                    S.ex[(r0 / G) & 1][wex][lane * E + j] = w.u[j];
            }
            if (!__syncthreads_or(r < re || found))
                break;
            const int nl = min(S.nl, OCAP), kf = S.kf;
            __syncthreads(); // every thread has read the words above
            if (threadIdx.x == 0)
                S.nl = 0;
            if (nl == 0 && kf != INT32_MAX) { // (no warp is behind the round it was found in)
                kfound = kf;
                break;
            }
            const bool waits = __any_sync(0xffffffffu, pend != 0);
            if (nl > 0) {
                keep();
                wide_slides(nl);
                for (int i = 0; i < nl; i++) {
                    const int32_t d = S.ld[i], e = above ? d : -d, u = above ? S.lc[i] : S.lc[i] + d, j = e - dl;
                    if (j >= 0 && j < E && ((pend >> j) & 1u) && (int32_t)kept[j] == u) {
                        kept[j] = (uint32_t)(u + S.lr[i] - S.lc[i]);
                        kept[E + j] = kept[2 * E + j] = WIN_NONE;
                        pend &= ~(1u << j);
                    }
                }
                back();
                __syncthreads(); // every thread has read the list
            }
            if (waits) { // round r is final for this warp now
                bool f = false;
#pragma unroll
                for (int j = 0; j < E; j++)
                    f = f || (j < kmax && dl + j == M - N && w.u[j] == N);
                if (f)
                    atomicMin(&S.kf, t + r);
                found = __any_sync(0xffffffffu, f);
                r++;
            }
        }
        if (kfound >= 0)
            break;
        if (lane >= 32 - HT && !last) { // the next warp's first rows
#pragma unroll
            for (int j = 0; j < E; j++)
                w.u[j] = S.ex[(r0 / G) & 1][wex + 1][(lane - (32 - HT)) * E + j];
        }
        __syncwarp();
    }
    // the block's last round (all reads of src lie before the first barrier)
#pragma unroll
    for (int j = 0; j < E; j++) {
        const int32_t s = s0 + j, e = a + s;
        if (own_lane && !idle && s < b - a)
            dst[(above ? e : -e) - off] = w.u[j] < 0 ? NEG : (above ? w.u[j] : w.u[j] + e);
    }
    slide = __reduce_add_sync(0xffffffffu, slide);
    mism = __reduce_add_sync(0xffffffffu, mism);
    opens = __reduce_add_sync(0xffffffffu, opens);
    if (lane == 0) {
        atomicAdd(&S.opens, (unsigned long long)opens);
        atomicAdd(&S.slide, (unsigned long long)slide);
        atomicAdd(&S.mism, (unsigned long long)mism);
    }
    __syncthreads();
    return kfound;
}

// The diagonal of the tile's furthest row (the alignment path's, or the end
// nearest to it): b when it lies in the last PATH_MARGIN diagonals, a in the
// first (the tile is then on one side of the path).
constexpr int32_t PATH_MARGIN = 16;
__device__ __forceinline__ int32_t path_of(const int32_t *src, int32_t off, int32_t a, int32_t b)
{
    WideSmem &S = wsm();
    if (threadIdx.x == 0)
        S.lead = 0;
    __syncthreads();
    unsigned long long best = 0;
    for (int32_t d = a + (int32_t)threadIdx.x; d < b; d += WT) {
        const int32_t x = src[d - off];
        if (x >= 0) // the row summed over both strings: 2x + d
            best = max(best, ((unsigned long long)(2ll * x + d + (1ll << 31)) << 28) | (uint32_t)(d - a));
    }
#pragma unroll
    for (int o = 16; o; o >>= 1)
        best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
    if ((threadIdx.x & 31) == 0)
        atomicMax(&S.lead, best);
    __syncthreads();
    const int32_t p = a + (int32_t)(S.lead & 0xfffffffull);
    return p < a + PATH_MARGIN ? a : (p >= b - PATH_MARGIN ? b : p);
}

// Rounds t .. t+h-1 on the tile [a, b), from src to dst: the diagonals below
// and above the path in one pass, with as few slots a thread as hold them (1,
// 2 or 4), or, past 1792 slots, in several.
__device__ __forceinline__ int32_t wide_rounds(const int32_t *src, int32_t *dst, int32_t t, int32_t h, int32_t a,
                                               int32_t b)
{
    const int32_t off = a - h - 1, hh = 2 * h - 2;
    const int32_t p = path_of(src, off, a, b);
    // warps that hold a strip of w diagonals
    auto warps = [&](int32_t w, int E) { return w > 0 ? (w + hh + warp_slots(E) - 1) / warp_slots(E) : 0; };
    auto run = [&](int32_t a0, int32_t b0, int32_t a1, int32_t b1, int E) {
        const Pass Q = {a0, b0, warps(b0 - a0, E), a1, b1, warps(b1 - a1, E)};
        return E == 1 ? win_block<1>(src, dst, off, t, h, Q)
                      : (E == 2 ? win_block<2>(src, dst, off, t, h, Q) : win_block<4>(src, dst, off, t, h, Q));
    };
    for (int E = 1; E <= 4; E *= 2)
        if (warps(p - a, E) + warps(b - p, E) <= NWARP)
            return run(a, p, p, b, E);
    const int32_t room = NWARP * warp_slots(4) - hh;
    int32_t kf = -1, al = a, br = b;
    // full strips from both ends, then what is left around the path
    for (; p - al > room && kf < 0; al += room)
        kf = run(al, al + room, b, b, 4);
    for (; br - p > room && kf < 0; br -= room)
        kf = run(a, a, br - room, br, 4);
    if (kf >= 0)
        return kf;
    if (warps(p - al, 4) + warps(br - p, 4) <= NWARP)
        return run(al, p, p, br, 4);
    kf = run(al, p, b, b, 4);
    return kf >= 0 ? kf : run(a, a, p, br, 4);
}

// ------------------------------------------------------------------ group
__device__ __forceinline__ unsigned long long ld_word(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_word(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// A wait gave up: the first one records where (for the host's error text).
__device__ __noinline__ void wide_wait_failed(LaunchCtl *ctl, unsigned long long site, unsigned long long t,
                                              unsigned long long want, unsigned long long seen)
{
    if (atomicCAS(&ctl->error, 0u, ST_TIMEOUT) == 0u) {
        ctl->diag[0] = site;
        ctl->diag[1] = blockIdx.x;
        ctl->diag[2] = t;
        ctl->diag[3] = want;
        ctl->diag[4] = seen;
        __threadfence();
    }
}

// Bounded barrier over the G CTAs of a group, on (count, gen).  Returns 1
// when all arrived, 0 on error or timeout, 2 when `abandon` is set and the
// group's k became known meanwhile.
__device__ __noinline__ int wide_barrier(const LvArgs &P, GroupCtl *gc, uint32_t *count, uint32_t *gen_p, int G,
                                         bool abandon)
{
    WideSmem &S = wsm();
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        const uint32_t gen = ld_acquire(gen_p);
        __threadfence();
        if (atomicAdd(count, 1u) == (uint32_t)G - 1) {
            atomicExch(count, 0u);
            __threadfence();
            st_release(gen_p, gen + 1);
        } else {
            const uint64_t t0 = gtimer();
            while (ld_acquire(gen_p) == gen) {
                if (ld_acquire(&P.ctl->error) != 0) {
                    ok = 0;
                    break;
                }
                if (abandon && *(volatile unsigned long long *)&gc->done_k != ~0ull) {
                    ok = 2;
                    break;
                }
                if (gtimer() - t0 > P.idle_ns) {
                    wide_wait_failed(P.ctl, abandon ? 5 : 2, 0, gen, ld_acquire(count));
                    ok = 0;
                    break;
                }
            }
        }
        S.bc[0] = ok;
    }
    __syncthreads();
    const int ok = S.bc[0];
    __syncthreads();
    return ok;
}

// The largest radius whose band [max(-R, -n), min(R, m)] fits in cap
// diagonals.
__device__ int64_t wide_fit_radius(int64_t n, int64_t m, int64_t cap)
{
    int64_t lo = 0, hi = max(n, m);
    while (lo < hi) {
        const int64_t mid = lo + (hi - lo + 1) / 2;
        if (min(mid, m) + min(mid, n) + 1 <= cap)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// Ends the pair for the whole group without a distance (ST_WIDE, ST_LIMIT):
// the first CTA here records the status.
__device__ void wide_stop(unsigned long long *res, GroupCtl *gc, uint32_t status)
{
    if (threadIdx.x == 0 && atomicCAS(&gc->done_k, ~0ull, DONE_STOPPED) == ~0ull)
        res[R_STATUS] = status;
}

// One pair on the group; kc is the radius its re-tiling buffers hold.  Returns
// false if the launch must stop.  tm: cycles in rounds, neighbour waits and
// epoch changes.
__device__ __forceinline__ bool wide_pair(const LvArgs &P, const PairDesc &D, GroupCtl *gc, int gi, int G, int c0,
                                          int32_t *gfb, int64_t kc, uint64_t deadline, unsigned long long *tm,
                                          uint32_t *blocks)
{
    WideSmem &S = wsm();
    const int tid = threadIdx.x, h = P.h, smax = P.smax;
    const int64_t n = D.n, m = D.m, nm = max(n, m), gstride = 2 * kc + 5;
    const bool can_suspend = P.budget_ns != 0 && D.keep != nullptr;
    int64_t R = min(max(min((int64_t)P.s0 * G / 2, (int64_t)P.kcap), (int64_t)h - 1), nm);
    int64_t t = 0;
    if (D.keep && D.t0 > 0) {
        t = D.t0;
        R = D.R0;
    } else if (D.init) {
        t = D.init_t;
        R = min(max(R, t + 16 * h), nm); // some room before the first epoch change
        R = min(R, max(t + h - 1, wide_fit_radius(n, m, (int64_t)G * smax)));
        R = min(R, (int64_t)P.kcap);
    }
    // the tile of radius R: [a, b), S.. wide; none when it lies past the band
    int64_t lo_all, hi_all, ts;
    int32_t a, b;
    auto cut = [&]() {
        lo_all = max(-R, -n);
        hi_all = min(R, m);
        ts = max((int64_t)h, (hi_all - lo_all + G) / G);
        a = (int32_t)min(hi_all + 1, lo_all + (int64_t)gi * ts);
        b = (int32_t)min(hi_all + 1, lo_all + (int64_t)(gi + 1) * ts);
    };
    if (tid == 0) {
        S.A = D.A;
        S.B = D.B;
        S.n = (int32_t)n;
        S.m = (int32_t)m;
        S.cap = P.t2_cap;
        S.nl = 0;
        S.kf = INT32_MAX;
        S.slide = S.mism = S.opens = 0;
    }
    cut();
    if (ts > smax || (D.keep && R > D.keep_r)) {
        wide_stop(D.res, gc, ST_WIDE);
        if (tid == 0 && gi == 0 && D.t0 > 0) { // the saved state is still good
            D.res[R_RESUME_T] = (unsigned long long)t;
            D.res[R_RESUME_R] = (unsigned long long)R;
        }
        return true;
    }
    int cur = 0; // the buffer that holds round t - 1
    // round t - 1 of the tile and its halo
    auto fill = [&](const int32_t *from, int64_t zero) {
        const int64_t plo = max(-(t - 1), -n), phi = min(t - 1, m);
        int32_t *dst = wbuf(cur, smax);
        for (int32_t i = tid; i < b - a + 2 * h; i += WT) {
            const int64_t d = (int64_t)a - h + i;
            dst[i + 1] = from && d >= plo && d <= phi ? __ldcg(from + d + zero) : NEG;
        }
        __syncthreads();
    };
    if (a < b)
        fill(t == 0 ? nullptr : (D.keep && D.t0 > 0 ? D.keep : D.init),
             D.keep && D.t0 > 0 ? D.keep_r + 2 : D.init_zero);
    __syncthreads();
    uint32_t epoch = 0;
    int64_t t_ep = t;
    for (;;) {
        // ---------------------------------------------- stop / epoch checks
        if (tid == 0)
            S.bc[1] = *(volatile unsigned long long *)&gc->done_k != ~0ull ? 1 : (ld_acquire(&P.ctl->error) != 0 ? 2 : 0);
        __syncthreads();
        const int stop0 = S.bc[1];
        __syncthreads();
        if (stop0)
            return stop0 == 1;
        auto grows = [&](int64_t x) { return x + h - 1 > R && R < nm; };
        auto due = [&](int64_t x) { return grows(x) || (can_suspend && x >= t_ep + P.sync_rounds); };
        if (a >= b && !due(t)) {
            // no tile: on to the group's next epoch change (every CTA finds the
            // same round; none: the pair ends before one, wait for that)
            int64_t x = t + h;
            const int64_t need = max((int64_t)0, R - h + 2 - t); // rounds until grows(), by whole blocks
            int64_t nb = R < nm ? (need + h - 1) / h : INT64_MAX / (4 * h);
            if (can_suspend)
                nb = min(nb, (max((int64_t)0, t_ep + P.sync_rounds - t) + h - 1) / h);
            x = t + nb * h;
            if (nb >= INT64_MAX / (4 * h)) {
                if (tid == 0) {
                    const uint64_t w0 = gtimer();
                    int st = 0;
                    while (st == 0) {
                        if (*(volatile unsigned long long *)&gc->done_k != ~0ull)
                            st = 1;
                        else if (ld_acquire(&P.ctl->error) != 0)
                            st = 2;
                        else if (gtimer() - w0 > P.idle_ns) {
                            wide_wait_failed(P.ctl, 3, t, epoch, 0);
                            st = 2;
                        }
                    }
                    S.bc[1] = st;
                }
                __syncthreads();
                return S.bc[1] == 1;
            }
            t = x;
        }
        if (due(t)) {
            // ------------------------------------------ epoch change
            const uint64_t te0 = clock64();
            int64_t Rn = R;
            bool wide = false; // the band outgrew the tiles: save it for wider ones
            uint32_t stop = 0; // decided once every CTA of the group is here without k
            if (grows(t)) {
                Rn = min(max(R * 9 / 8, t + h - 1), min(nm, (int64_t)P.kcap));
                if (t + h - 1 > Rn && Rn < nm)
                    stop = ST_LIMIT;
                Rn = min(Rn, wide_fit_radius(n, m, (int64_t)G * smax));
                if (D.keep)
                    Rn = min(Rn, D.keep_r);
                if (!stop && t + h - 1 > Rn && Rn < nm) {
                    if (!D.keep)
                        stop = ST_WIDE;
                    else {
                        wide = true;
                        Rn = R;
                    }
                }
            }
            int32_t *buf = gfb + ((epoch + 1) & 1) * gstride;
            const int32_t *src = wbuf(cur, smax);
            for (int32_t i = tid; i < b - a; i += WT)
                __stcg(buf + (int64_t)a + i + kc + 2, src[i + h + 1]);
            if (gi == 0 && tid == 0) // the leader alone decides whether the launch leaves the pair here
                *(volatile uint32_t *)&gc->susp[(epoch + 1) & 1] =
                    (wide || (can_suspend && gtimer() >= deadline)) ? 1u : 0u;
            __threadfence();
            const int eb = wide_barrier(P, gc, &gc->ebar_count, &gc->ebar_gen, G, true);
            if (eb == 0)
                return false;
            if (eb == 2)
                return true; // k is known: the pair is over
            if (stop) {
                wide_stop(D.res, gc, stop);
                return true;
            }
            epoch++;
            if (*(volatile uint32_t *)&gc->susp[epoch & 1]) {
                // save round t - 1 of the band for the next launch, then leave
                const int64_t plo = max(-(t - 1), -n), phi = min(t - 1, m);
                for (int64_t d = plo + (int64_t)gi * WT + tid; d <= phi; d += (int64_t)G * WT)
                    D.keep[d + D.keep_r + 2] = __ldcg(buf + d + kc + 2);
                if (gi == 0 && tid == 0) {
                    D.res[R_STATUS] = wide ? ST_WIDE : ST_SUSPENDED;
                    D.res[R_RESUME_T] = (unsigned long long)t;
                    D.res[R_RESUME_R] = (unsigned long long)Rn;
                }
                return true;
            }
            t_ep = t;
            R = Rn;
            cut();
            if (a < b)
                fill(buf, kc + 2);
            tm[2] += clock64() - te0;
            if (a >= b)
                continue;
        }
        // ---------------------------------------------- h rounds
        const uint64_t tr0 = clock64();
        const int32_t kf = wide_rounds(wbuf(cur, smax), wbuf(cur ^ 1, smax), (int32_t)t, h, a, b);
        cur ^= 1;
        tm[0] += clock64() - tr0;
        if (kf >= 0) {
            if (tid == 0) {
                D.res[R_K] = (unsigned long long)kf;
                __threadfence();
                atomicMin(&gc->done_k, (unsigned long long)kf);
            }
            return true;
        }
        t += h;
        ++*blocks;
        // ---------------------------------------------- halo exchange
        // one word per edge value, (round << 32) | L: a word of round t is
        // the value of round t - 1.  The parity of t / h alternates the
        // buffers: a tile is one block ahead of a neighbour at most.
        const uint64_t tw0 = clock64();
        const int parity = (int)((t / h) & 1);
        int32_t *edge = wbuf(cur, smax) + h + 1; // index d - a
        auto words = [&](int cta, int side) { return P.halo + ((int64_t)(cta * 2 + parity) * 2 + side) * HMAX; };
        const bool hl = gi > 0, hr = b <= hi_all; // neighbours
        for (int i = tid; i < 2 * h; i += WT) {
            const int side = i >= h, j = side ? i - h : i;
            const int32_t x = side ? b - a - h + j : j;
            const int32_t v = x >= 0 && x < b - a ? edge[x] : NEG;
            st_word(words(blockIdx.x, side) + j, ((unsigned long long)(uint32_t)t << 32) | (uint32_t)v);
        }
        // 2h threads (whole warps) read one word each
        if (tid < 2 * HMAX) {
            const int side = tid >= HMAX, j = tid - side * HMAX;
            const bool has = j < h && (side ? hr : hl);
            const unsigned long long *wp = words(side ? c0 + gi + 1 : c0 + gi - 1, side ? 0 : 1) + j;
            const uint64_t w0 = gtimer();
            int st = 0;
            unsigned long long v = 0;
            while (st == 0) {
                bool ok = true;
                if (has) {
                    v = ld_word(wp);
                    ok = (uint32_t)(v >> 32) >= (uint32_t)t;
                }
                if (ok)
                    st = 3;
                else if (*(volatile unsigned long long *)&gc->done_k != ~0ull)
                    st = 1;
                else if (*(volatile uint32_t *)&P.ctl->error != 0)
                    st = 2;
                else if (gtimer() - w0 > P.idle_ns) {
                    wide_wait_failed(P.ctl, 4, (unsigned long long)t, (unsigned long long)t, v);
                    st = 2;
                }
            }
            if (j < h)
                edge[side ? b - a + j : j - h] = has ? (int32_t)(uint32_t)v : NEG;
            if (st != 3)
                atomicMax(&S.bc[2], 4 - st); // 3: k is known, 2: an error
        }
        __syncthreads();
        const int bad = S.bc[2];
        __syncthreads();
        tm[1] += clock64() - tw0;
        if (bad) {
            if (tid == 0)
                S.bc[2] = 0;
            return bad == 3;
        }
    }
}

__global__ void __launch_bounds__(WT, WIDE_PER_SM) lv_wide_kernel(const __grid_constant__ LvArgs P)
{
    WideSmem &S = wsm();
    const uint64_t deadline = gtimer() + P.budget_ns;
    if (threadIdx.x == 0) {
        S.bc[2] = 0;
        S.tile = P.wide + (size_t)blockIdx.x * (2 * ((size_t)P.smax + 2 * HMAX + 2));
    }
    int cls = 0;
    while (cls + 1 < P.ncls && (int)blockIdx.x >= P.cls_c0[cls + 1])
        cls++;
    const int G = P.cls_G[cls];
    const int rel = (int)blockIdx.x - P.cls_c0[cls];
    const int gi = rel % G, c0 = (int)blockIdx.x - gi;
    GroupCtl *gc = &P.gctl[P.cls_g0[cls] + rel / G];
    const int64_t kc = P.cls_kc[cls];
    int32_t *gfb = P.gf + P.cls_gf[cls] + (int64_t)(rel / G) * 2 * (2 * kc + 5);
    for (;;) {
        // the CTA's edge words start each pair cleared (round 0): every CTA
        // of the group has left the pair before, and the barrier below orders
        // the clear before the first read of the next pair
        for (int i = threadIdx.x; i < 4 * HMAX; i += WT)
            st_word(P.halo + (size_t)blockIdx.x * 4 * HMAX + i, 0ull);
        if (gi == 0 && threadIdx.x == 0) {
            // the class's own queue first, then the classes below it
            int32_t q = -1;
            for (int c = cls; c >= 0 && q < 0; c--) {
                const uint32_t cnt = (uint32_t)(P.cls_p0[c + 1] - P.cls_p0[c]);
                if (*(volatile uint32_t *)&P.ctl->queue[c] >= cnt)
                    continue;
                const uint32_t i = atomicAdd(&P.ctl->queue[c], 1u);
                if (i < cnt)
                    q = P.cls_p0[c] + (int32_t)i;
            }
            gc->pair = q;
            gc->done_k = ~0ull;
            gc->ebar_count = 0; // no CTA is inside the epoch barrier here
        }
        __threadfence();
        if (wide_barrier(P, gc, &gc->bar_count, &gc->bar_gen, G, false) != 1)
            break;
        const int q = *(volatile int32_t *)&gc->pair;
        if (q < 0)
            break;
        const PairDesc D = P.pairs[q];
        unsigned long long tm[3] = {0, 0, 0};
        uint32_t blocks = 0;
        const bool ok = wide_pair(P, D, gc, gi, G, c0, gfb, kc, deadline, tm, &blocks);
        __syncthreads();
        if (threadIdx.x == 0) {
            if (S.slide)
                atomicAdd(&D.res[R_SLIDE], S.slide);
            if (S.mism)
                atomicAdd(&D.res[R_MISMATCH], S.mism);
            if (S.opens)
                atomicAdd(&D.res[R_OPEN], S.opens);
            if (gi == 0)
                D.res[R_WIDE] = blocks;
            atomicMax(&D.res[R_T0], tm[0]);
            atomicMax(&D.res[R_T0 + 2], tm[1]);
            atomicMax(&D.res[R_T0 + 3], tm[2]);
            atomicAdd(&D.res[R_T0 + 4], tm[0]);
            atomicAdd(&D.res[R_T0 + 5], 1ull);
        }
        if (!ok)
            break;
        __threadfence();
        if (wide_barrier(P, gc, &gc->bar_count, &gc->bar_gen, G, false) != 1)
            break;
    }
}

cudaError_t launch_lv_wide(const LvArgs &P, int grid, cudaStream_t s)
{
    LvArgs Pc = P;
    void *args[] = {&Pc};
    return cudaLaunchCooperativeKernel((const void *)lv_wide_kernel, dim3(grid), dim3(WT), args,
                                       sizeof(WideSmem), s);
}

} // namespace edg
