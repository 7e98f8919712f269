// hash.cu -- the prefix-hash table of Sec. 3.2 on the device.
//
//   T[i] = h(X[0..i)) = sum_{j<i} (X[j] + 1) * p^(i-1-j)   mod q = 2^61 - 1
//
// Prefix hashes compose by the concatenation rule of Sec. 2,
//   h([S1, S2]) = h(S1) * p^|S2| + h(S2),
// so T is a scan; all segments but the last have fixed lengths, so that only
// hashes are scanned and every power is known beforehand.  Three passes: the
// hashes of tiles of TILE_CHARS characters (16 characters a thread and row:
// their codes times the split powers, summed in 64 bits and reduced once), one
// CTA's scan of those (8 bytes per 16 KiB), and the output, in which each
// thread extends its prefix over its characters.  The characters are read
// twice, which costs a ninth of the output's traffic and saves every wait
// between tiles: a single pass with a look-back chain spent two thirds of its
// cycles at the barrier behind it (480 us for 10^8 characters).
//
// Reads 1 byte (twice) and writes 8 bytes per character, through shared memory
// in whole lines; with an output stride b > 1 it writes only the prefixes of
// whole blocks, T[j] = h(X[0..jb)), the blocked table of Sec. 3.3 (Alg. 2),
// 8/b bytes per character.
//
// Bound: the bytes, and one modular product per character for its output
// (about 35 instructions in all).  The first form took three products per
// character and wrote at a 128-byte stride: 1057 us for 10^8 characters,
// 370 us now (2430 GB/s of the 9 bytes a character).
#include <algorithm>

#include "ed_device.cuh"
#include "lv_kernels.cuh"

namespace edg {

constexpr int HT = 256;                 // threads per CTA
constexpr int HW = HT / 32;             // its warps
constexpr int HITEMS = 16;              // characters hashed, and written, at a time
constexpr int HPARTS = 2;               // such parts a thread holds of a row
constexpr int THREAD_CHARS = HPARTS * HITEMS;
constexpr int ROW_CHARS = HT * THREAD_CHARS; // 8192
constexpr int HROWS = 2;                // rows per tile
constexpr int TILE_CHARS = HROWS * ROW_CHARS;
constexpr int HPAD = HITEMS + 1;        // words between threads' outputs in shared memory
constexpr int HPER_SM = 4;              // CTAs per SM (64 registers a thread, 35 KB each)
constexpr int ST = 1024;                // threads of the tiles' scan

size_t prefix_hash_state_bytes(int64_t len)
{
    const int64_t tiles = (len + TILE_CHARS - 1) / TILE_CHARS + 1;
    return 2 * sizeof(uint64_t) * (size_t)tiles; // each tile's hash, and the prefix before it
}

int prefix_hash_launches(int64_t len) { return len > TILE_CHARS ? 3 : 1; }

// A multiplier b as mul61 takes it: b and b * 2^32 mod q, each hi * 2^31 + lo.
struct Mul61 {
    uint32_t c0l, c0h, c1l, c1h;
};

// The powers a launch uses.
struct HashPowers {
    uint32_t lo[HITEMS], hi[HITEMS]; // p^k = hi * 2^31 + lo, k < 16
    uint64_t ones;                   // the hash of 16 characters of code 0, plus 1 each
    Mul61 base;                      // p
    Mul61 pow16[11];                 // p^(16 * 2^k): up to p^TILE_CHARS
};

// a * b mod q, below 2^62 + 2^34 (not reduced further), for a < 2^63: with
// a = a1 2^32 + a0 it is a0 b + a1 (b 2^32), both split at 31 bits; 2^61 = 1.
__device__ __forceinline__ uint64_t mul61(uint64_t a, const Mul61 &b)
{
    const uint32_t a0 = (uint32_t)a, a1 = (uint32_t)(a >> 32);
    const uint64_t sl = (uint64_t)a0 * b.c0l + (uint64_t)a1 * b.c1l; // < 2^63 + 2^62
    const uint64_t sh = (uint64_t)a0 * b.c0h + (uint64_t)a1 * b.c1h; // < 2^62 + 2^61
    return (sl & Q61) + (sl >> 61) + (sh >> 30) + ((sh & 0x3fffffffull) << 31);
}
__device__ __forceinline__ uint64_t fold61(uint64_t r) { return (r & Q61) + (r >> 61); } // below 2^61 + 8
__device__ __forceinline__ uint64_t canon61(uint64_t r) // the residue below q, for r < 2^64
{
    r = (r & Q61) + (r >> 61);
    return r >= Q61 ? r - Q61 : r;
}
__device__ __forceinline__ Mul61 mul_of(uint64_t b) // b < q
{
    // b * 2^32 mod q: b's upper 32 bits pass 2^61
    const uint64_t c1 = canon61(((b << 32) & Q61) + (b >> 29));
    return Mul61{(uint32_t)b & 0x7fffffffu, (uint32_t)(b >> 31), (uint32_t)c1 & 0x7fffffffu, (uint32_t)(c1 >> 31)};
}

__device__ __forceinline__ uint32_t code_at(const uint4 &v, int i) // character i of 16
{
    const uint32_t w = i < 4 ? v.x : (i < 8 ? v.y : (i < 12 ? v.z : v.w));
    return __byte_perm(w, 0, 0x4440 + (i & 3));
}

// The hash of 16 characters, below 2^61 + 8.
__device__ __forceinline__ uint64_t hash16(const HashPowers &P, const uint4 &v)
{
    uint64_t lo = 0, hi = 0; // below 2^45
#pragma unroll
    for (int i = 0; i < HITEMS; i++) {
        const uint32_t c = code_at(v, i);
        lo += (uint64_t)c * P.lo[HITEMS - 1 - i];
        hi += (uint64_t)c * P.hi[HITEMS - 1 - i];
    }
    return fold61(lo + ((hi & 0x3fffffffull) << 31) + (hi >> 30) + P.ones);
}
// ... and of a thread's 32.
__device__ __forceinline__ uint64_t hash32(const HashPowers &P, const uint4 (&v)[HPARTS])
{
    return fold61(mul61(hash16(P, v[0]), P.pow16[0]) + hash16(P, v[1]));
}

// The hash of every whole tile (one CTA each).
__global__ void __launch_bounds__(HT) tile_hash_kernel(const uint8_t *X, int64_t len, uint64_t *agg,
                                                       const __grid_constant__ HashPowers P)
{
    __shared__ uint64_t s_warp[HW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t s0 = blockIdx.x * (int64_t)TILE_CHARS + (int64_t)tid * THREAD_CHARS;
    uint4 v[HROWS][HPARTS];
#pragma unroll
    for (int r = 0; r < HROWS; r++)
#pragma unroll
        for (int q = 0; q < HPARTS; q++)
            v[r][q] = load16(X, len, s0 + r * ROW_CHARS + q * HITEMS);
    uint64_t h = 0;
#pragma unroll
    for (int r = 0; r < HROWS; r++)
        h = fold61(mul61(h, P.pow16[9]) + hash32(P, v[r]));
    // the threads' hashes (32 characters of each row) left to right
#pragma unroll
    for (int k = 0; k < 5; k++) {
        const uint64_t o = __shfl_down_sync(0xffffffffu, h, 1 << k);
        h = fold61(mul61(h, P.pow16[1 + k]) + o);
    }
    if (lane == 0)
        s_warp[warp] = h;
    __syncthreads();
    if (tid < 32) {
        h = tid < HW ? s_warp[tid] : 0ull;
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const uint64_t o = __shfl_down_sync(0xffffffffu, h, 1 << k);
            h = fold61(mul61(h, P.pow16[6 + k]) + o);
        }
        if (tid == 0)
            agg[blockIdx.x] = canon61(h);
    }
}

// pre[t] = the hash of everything before tile t, t = 0 .. cnt, from the hashes
// of tiles 0 .. cnt-1.  One CTA: every thread takes `per` consecutive tiles.
__global__ void __launch_bounds__(ST) tile_scan_kernel(const uint64_t *agg, uint64_t *pre, int64_t cnt, int per,
                                                       const __grid_constant__ HashPowers P)
{
    __shared__ uint64_t s_warp[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const Mul61 &tile = P.pow16[10];
    const int64_t t0 = (int64_t)tid * per;
    uint64_t h = 0, step = 1; // this thread's tiles; p^(TILE_CHARS * per)
    for (int i = 0; i < per; i++) {
        h = mul61(h, tile) + (t0 + i < cnt ? agg[t0 + i] : 0ull);
        step = mul61(step, tile);
    }
    h = canon61(h);
    step = canon61(step);
    uint64_t over = 1; // p^(TILE_CHARS * per * lane)
#pragma unroll
    for (int k = 0; k < 5; k++) {
        const uint64_t o = __shfl_up_sync(0xffffffffu, h, 1 << k);
        const Mul61 ms = mul_of(step);
        if (lane >= 1 << k)
            h = canon61(mul61(o, ms) + h);
        if ((lane >> k) & 1)
            over = canon61(mul61(over, ms));
        step = canon61(mul61(step, ms));
    }
    if (lane == 31)
        s_warp[warp] = h;
    uint64_t excl = __shfl_up_sync(0xffffffffu, h, 1);
    if (lane == 0)
        excl = 0;
    __syncthreads();
    if (warp == 0) {
        uint64_t w = s_warp[lane];
#pragma unroll
        for (int k = 0; k < 5; k++) {
            const uint64_t o = __shfl_up_sync(0xffffffffu, w, 1 << k);
            const Mul61 ms = mul_of(step);
            if (lane >= 1 << k)
                w = canon61(mul61(o, ms) + w);
            step = canon61(mul61(step, ms));
        }
        const uint64_t wx = __shfl_up_sync(0xffffffffu, w, 1);
        s_warp[lane] = lane > 0 ? wx : 0ull;
    }
    __syncthreads();
    // what is before this thread's first tile: the warps before, carried over
    // the lanes before, and those lanes
    uint64_t t = canon61(mul61(s_warp[warp], mul_of(over)) + excl);
    for (int i = 0; i < per; i++) {
        if (t0 + i <= cnt)
            pre[t0 + i] = t;
        t = canon61(mul61(t, tile) + (t0 + i < cnt ? agg[t0 + i] : 0ull));
    }
}

__global__ void __launch_bounds__(HT, HPER_SM) prefix_hash_kernel(const uint8_t *X, int64_t len, uint64_t *T,
                                                                  int64_t stride, const uint64_t *pre,
                                                                  const __grid_constant__ HashPowers P)
{
    __shared__ uint64_t s_out[HT * HPAD];
    __shared__ uint64_t s_warp[2][HW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t t0 = blockIdx.x * (int64_t)TILE_CHARS;
    uint64_t before = pre ? pre[blockIdx.x] : 0ull; // everything before the row
    if (blockIdx.x == 0 && tid == 0)
        T[0] = 0;
    // p^(32 lane), and the power that carries warp `lane`'s hash to the end of
    // the row: p^(1024 (7 - lane))
    uint64_t pl = 1, pe = 1;
#pragma unroll
    for (int k = 0; k < 5; k++)
        if ((lane >> k) & 1)
            pl = canon61(mul61(pl, P.pow16[1 + k]));
#pragma unroll
    for (int k = 0; k < 3; k++)
        if (((HW - 1 - lane) >> k) & 1)
            pe = canon61(mul61(pe, P.pow16[6 + k]));
    const Mul61 mlane = mul_of(pl), mend = mul_of(pe);
    for (int r = 0; r < HROWS; r++) {
        const int64_t r0 = t0 + r * ROW_CHARS;
        if (r0 >= len)
            break;
        // 1. this thread's 32 characters and their hash (a thread with fewer
        // ends the string: no thread reads its hash)
        const int64_t s0 = r0 + (int64_t)tid * THREAD_CHARS;
        uint4 v[HPARTS];
#pragma unroll
        for (int q = 0; q < HPARTS; q++)
            v[q] = s0 + q * HITEMS < len ? load16(X, len, s0 + q * HITEMS) : make_uint4(0u, 0u, 0u, 0u);
        // 2. inclusive scan across the warp, then every warp its own prefix
        uint64_t h = hash32(P, v);
#pragma unroll
        for (int k = 0; k < 5; k++) {
            const uint64_t o = __shfl_up_sync(0xffffffffu, h, 1 << k);
            if (lane >= 1 << k)
                h = fold61(mul61(o, P.pow16[1 + k]) + h);
        }
        if (lane == 31)
            s_warp[r & 1][warp] = h;
        uint64_t excl = __shfl_up_sync(0xffffffffu, h, 1);
        if (lane == 0)
            excl = 0;
        __syncthreads(); // (also: the last row's outputs have been read)
        uint64_t w = before; // everything before the warp
        for (int q = 0; q < warp; q++)
            w = fold61(mul61(w, P.pow16[6]) + s_warp[r & 1][q]);
        // everything before the next row: the warps' hashes carried to the
        // row's end, summed over lanes 0 .. 7
        if (r + 1 < HROWS) {
            uint64_t e = lane < HW ? fold61(mul61(s_warp[r & 1][lane], mend)) : 0ull;
            // (they fit in 64 bits: lane 7's multiplier is 1 and its value below
            // 2^61; the others are at most 2^61, as fold61 takes values below
            // 2^62 + 2^34 to at most that)
#pragma unroll
            for (int o = 4; o; o >>= 1)
                e += __shfl_xor_sync(0xffffffffu, e, o);
            before = fold61(mul61(before, P.pow16[9]) + fold61(__shfl_sync(0xffffffffu, e, 0)));
        }
        // ... and before this thread
        uint64_t t = mul61(w, mlane) + excl;
        // 3. T for each character
        if (stride == 1) {
#pragma unroll
            for (int q = 0; q < HPARTS; q++) {
#pragma unroll
                for (int i = 0; i < HITEMS; i++) {
                    t = mul61(t, P.base) + code_at(v[q], i) + 1u;
                    s_out[tid * HPAD + i] = canon61(t);
                }
                __syncthreads();
                const int64_t q0 = r0 + q * HITEMS;
                if (r0 + ROW_CHARS <= len) {
#pragma unroll 8
                    for (int i = 0; i < HITEMS; i++) {
                        const int e = i * HT + tid, u = e / HITEMS, j = e % HITEMS;
                        T[q0 + u * THREAD_CHARS + j + 1] = s_out[u * HPAD + j];
                    }
                } else {
                    for (int e = tid; e < HT * HITEMS; e += HT) {
                        const int u = e / HITEMS, j = e % HITEMS;
                        if (q0 + u * THREAD_CHARS + j < len)
                            T[q0 + u * THREAD_CHARS + j + 1] = s_out[u * HPAD + j];
                    }
                }
                __syncthreads();
            }
        } else {
            // only the prefixes that end a whole block
            int64_t next = (s0 / stride + 1) * stride; // first block end after s0
#pragma unroll
            for (int i = 0; i < THREAD_CHARS; i++) {
                t = mul61(t, P.base) + code_at(v[i / HITEMS], i % HITEMS) + 1u;
                if (s0 + i + 1 == next && next <= len) {
                    T[next / stride] = canon61(t);
                    next += stride;
                }
            }
        }
    }
}

cudaError_t launch_prefix_hash(const uint8_t *X, int64_t len, uint64_t base, uint64_t *T, int64_t stride,
                               void *scan_state, cudaStream_t s)
{
    const int64_t tiles = len == 0 ? 1 : (len + TILE_CHARS - 1) / TILE_CHARS;
    // the powers, by exact 128-bit products
    auto mul = [](uint64_t x, uint64_t y) {
        const unsigned __int128 z = (unsigned __int128)x * y;
        uint64_t r = (uint64_t)(z & Q61) + (uint64_t)(z >> 61);
        return r >= Q61 ? r - Q61 : r;
    };
    auto split = [&](uint64_t x) {
        const uint64_t y = mul(x, 1ull << 32);
        return Mul61{(uint32_t)(x & 0x7fffffffu), (uint32_t)(x >> 31), (uint32_t)(y & 0x7fffffffu), (uint32_t)(y >> 31)};
    };
    HashPowers P;
    P.base = split(base);
    uint64_t pw = 1;
    for (int k = 0; k < HITEMS; k++, pw = mul(pw, base)) {
        P.lo[k] = (uint32_t)(pw & 0x7fffffffu);
        P.hi[k] = (uint32_t)(pw >> 31);
        P.ones = (k ? P.ones : 0) + pw;
        P.ones = P.ones >= Q61 ? P.ones - Q61 : P.ones;
    }
    for (int k = 0; k < 11; k++, pw = mul(pw, pw))
        P.pow16[k] = split(pw);
    uint64_t *agg = static_cast<uint64_t *>(scan_state), *pre = agg + tiles;
    if (tiles > 1) { // (the last tile's hash is not needed)
        tile_hash_kernel<<<(unsigned)(tiles - 1), HT, 0, s>>>(X, len, agg, P);
        tile_scan_kernel<<<1, ST, 0, s>>>(agg, pre, tiles - 1, (int)((tiles + ST - 1) / ST), P);
    }
    prefix_hash_kernel<<<(unsigned)tiles, HT, 0, s>>>(X, len, T, stride < 1 ? 1 : stride, tiles > 1 ? pre : nullptr,
                                                      P);
    return cudaGetLastError();
}

} // namespace edg

// ---------------------------------------------------------------------------
// Allocation-free prefix hash (see ed_prefix_hash_noalloc in include/ed.h).
//
// The tiles' hashes and prefixes live in this file-scope device array
// instead of memory the caller or a context allocates.  Every GPU that loads
// the library holds it until the process exits.  Host code only ever uses
// the array's device address, obtained once per device with
// cudaGetSymbolAddress (the name itself is a host-side stand-in).
#include <mutex>

#include "../../include/ed.h"

namespace {

constexpr size_t NOALLOC_SCRATCH_BYTES = 1u << 20; // 1 MiB
constexpr int NOALLOC_MAX_DEVICES = 64;

static __device__ __align__(256) unsigned char g_noalloc_scan[NOALLOC_SCRATCH_BYTES];

std::mutex g_noalloc_mu;
void *g_noalloc_addr[NOALLOC_MAX_DEVICES] = {};

} // namespace

extern "C" int ed_prefix_hash_noalloc(const uint8_t *X, size_t len, uint64_t base, uint64_t *T,
                                      void *stream)
{
    if (!T || (len && !X) || base < 2 || base >= ((1ull << 61) - 1))
        return ED_EINVAL;
    if (len > ED_NOALLOC_MAX_LEN)
        return ED_EINVAL;
    static_assert((ED_NOALLOC_MAX_LEN / edg::TILE_CHARS + 2) * 16 <= NOALLOC_SCRATCH_BYTES, "the tiles' words fit");
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES)
        return ED_ECUDA;
    void *scratch = nullptr;
    {
        // first call on this device: look up the array's device address
        std::lock_guard<std::mutex> g(g_noalloc_mu);
        if (!g_noalloc_addr[dev]) {
            void *p = nullptr;
            if (cudaGetSymbolAddress(&p, g_noalloc_scan) != cudaSuccess || !p) {
                cudaGetLastError();
                return ED_ECUDA;
            }
            g_noalloc_addr[dev] = p;
        }
        scratch = g_noalloc_addr[dev];
    }
    cudaStream_t s = (cudaStream_t)stream;
    if (edg::launch_prefix_hash(X, (int64_t)len, base, T, 1, scratch, s) != cudaSuccess)
        return ED_ECUDA;
    return cudaStreamSynchronize(s) == cudaSuccess ? ED_OK : ED_ECUDA;
}
