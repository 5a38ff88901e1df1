// Pair-count kernels of libwtheta and the entry points that launch them.
//
// The computation is Sec. 2 of arXiv:1208.3658: every pair's angular
// separation (App. A) is binned (Sec. 2.1); auto counts take each unordered
// pair i < j once, cross counts every (i, j).  The paper splits the pair
// matrix into sub-matrices, one kernel launch each, with per-block shared
// histograms summed on the host.  Here one persistent launch walks the whole
// (triangular or rectangular) space of tile pairs from a device work cursor:
//   - RA/Dec -> FP64 unit vectors once per point (kept in the caller's order
//     for the rare FP64 recheck);
//   - the points are put in spatial order (cube-map face, then a Hilbert curve
//     on the face; a radix sort of 31-bit keys) so that a tile of consecutive
//     points is a compact patch of sky and a warp's pairs mostly share one
//     fate (all beyond the top edge, or all in range);
//   - tile pairs whose bounding caps lie wholly beyond the top edge are
//     skipped (their pairs are overflow); inside a tile pair, a sub-tile of 256
//     A points or a group of 8 and a chunk of 32 B points are settled in one
//     slot, or by counting the pairs below each edge between them, when their
//     bounding spheres allow it;
//   - FP32 float4 copies (x, y, z, original index) padded to whole tiles with
//     far-away sentinel points that never land in a bin, and planar FP32
//     coordinates relative to the centre of each point's chunk;
//   - a CTA stages the B tile in shared memory, negated and duplicated for
//     packed FP32x2 arithmetic, and a lane keeps R A points in registers; against
//     an edge two pairs cost 3 fma.f32x2 in those local coordinates, and a squared
//     chord 3 add.f32x2 + 1 mul.f32x2 + 2 fma.f32x2;
//   - s is screened against the top edge: pairs beyond it are overflow and
//     cost nothing more (Sec. 2.2: separations outside the bin range can be
//     skipped); the overflow slot is filled at the end as total minus the rest;
//   - in-range pairs are binned by a table lookup on the bits of s, the FP32
//     comparison being final outside a rigorous guard band around each edge;
//     inside it the pair is recomputed in FP64 exactly as the definition says;
//   - counts go to 32-bit shared histogram columns, a few per warp (or private
//     to a thread or a warp), flushed into uint64 global counts before any can
//     wrap.
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <mutex>

#include "wtheta_internal.h"

namespace wtheta {

// ---------------------------------------------------------------------------
// device error word and helpers
// ---------------------------------------------------------------------------
__device__ unsigned int g_device_error;

static std::atomic<unsigned long long> g_launches{0};
static inline void count_launch(unsigned n = 1) { g_launches.fetch_add(n, std::memory_order_relaxed); }

static constexpr float kSentinel = 1.0e10f;  // sentinel offset; (1e10)^2 >> 4

__host__ __device__ constexpr int ilog2(int x) { return x <= 1 ? 0 : 1 + ilog2(x / 2); }

__device__ __forceinline__ float min3f(float a, float b, float c) {
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// two FP32 values packed in one 64-bit register, for the sm_100-family
// packed FP32x2 instructions (each lane rounds exactly like its scalar op)
typedef unsigned long long f2_t;
__device__ __forceinline__ f2_t pack2(float lo, float hi) {
    f2_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f2_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f2_t add2(f2_t a, f2_t b) {
    f2_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2_t mul2(f2_t a, f2_t b) {
    f2_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2_t fma2(f2_t a, f2_t b, f2_t c) {
    f2_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Shared-memory accesses of the hot loops, through 32-bit shared-window
// addresses (so no generic 64-bit address arithmetic on the way).
__device__ __forceinline__ unsigned smem_addr(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void lds_f2x2(unsigned a, f2_t& x, f2_t& y) {
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "r"(a));
}
__device__ __forceinline__ void sts_f2x2(unsigned a, f2_t x, f2_t y) {
    asm volatile("st.shared.v2.b64 [%0], {%1, %2};" :: "r"(a), "l"(x), "l"(y) : "memory");
}
__device__ __forceinline__ uint2 lds_u2(unsigned a) {
    uint2 v;
    asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ f2_t lds_f2(unsigned a) {
    f2_t z;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(z) : "r"(a));
    return z;
}
// n += sign bit of d, as one shift-and-add (written this way: as plain C++ the
// adds of two values are combined first, into three operations instead of two)
__device__ __forceinline__ void add_sign(unsigned& n, float d) {
    asm("{\n\t.reg .u32 t;\n\tshr.u32 t, %1, 31;\n\tadd.u32 %0, %0, t;\n\t}"
        : "+r"(n) : "r"(__float_as_uint(d)));
}
__device__ __forceinline__ uint4 lds_u4(unsigned a) {
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ double lds_f64(unsigned a) {
    double v;
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ long long lds_s64(unsigned a) {
    long long v;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ unsigned lds_u32(unsigned a) {
    unsigned v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts_u32(unsigned a, unsigned v) {
    asm volatile("st.shared.b32 [%0], %1;" :: "r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void sts_u32_if(bool p, unsigned a, unsigned v) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q st.shared.b32 [%0], %1;\n\t}"
                 :: "r"(a), "r"(v), "r"((unsigned)p) : "memory");
}
__device__ __forceinline__ void red_add_shared(unsigned a, unsigned v) {
    asm volatile("red.shared.add.u32 [%0], %1;" :: "r"(a), "r"(v) : "memory");
}

// ---------------------------------------------------------------------------
// conversion kernels
// ---------------------------------------------------------------------------
__device__ __forceinline__ void radec_unit(double ra, double dec, double& x, double& y, double& z) {
    const double d2r = 3.14159265358979323846 / 180.0;
    if (!isfinite(ra) || !isfinite(dec)) atomicOr(&g_device_error, WTHETA_DERR_NONFINITE);
    else if (fabs(dec) > 90.0) atomicOr(&g_device_error, WTHETA_DERR_DEC_RANGE);
    const double a = ra * d2r, d = dec * d2r;
    const double cd = cos(d), sd = sin(d), ca = cos(a), sa = sin(a);
    x = __dmul_rn(cd, ca);
    y = __dmul_rn(cd, sa);
    z = sd;
}

__device__ __forceinline__ void check_unit(double x, double y, double z) {
    if (!isfinite(x) || !isfinite(y) || !isfinite(z)) {
        atomicOr(&g_device_error, WTHETA_DERR_NONFINITE);
    } else {
        const double r2 = x * x + y * y + z * z;
        if (fabs(r2 - 1.0) > 1e-6) atomicOr(&g_device_error, WTHETA_DERR_NOT_UNIT);
    }
}

__device__ __forceinline__ float4 point32(double x, double y, double z, long long idx) {
    return make_float4(__double2float_rn(x), __double2float_rn(y), __double2float_rn(z),
                       __int_as_float((int)idx));
}

// Padding point k of catalogue tag t: far from the unit sphere and from the
// padding of any other tag, (+-S (k+1), S t, 0) with the sign of t's parity;
// its squared chord with anything else is at least S^2 >> 4, so it never
// lands in a bin.
__device__ __forceinline__ float4 sentinel32(int tag, long long k) {
    const float sign = (tag & 1) ? -1.f : 1.f;
    return make_float4(sign * kSentinel * (float)(k + 1), kSentinel * (float)tag, 0.f, 0.f);
}

__device__ __forceinline__ bool is_sentinel(const float4& q) {
    return q.x * q.x + q.y * q.y + q.z * q.z > 4.f;
}

// RA/Dec degrees -> FP64 unit vectors (SoA with stride xyz_stride).
__global__ void k_radec_to_xyz(const double* __restrict__ rd, long long n,
                               double* __restrict__ xyz, long long xyz_stride) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        double x, y, z;
        radec_unit(rd[2 * i], rd[2 * i + 1], x, y, z);
        xyz[i] = x;
        xyz[xyz_stride + i] = y;
        xyz[2 * xyz_stride + i] = z;
    }
}

// Caller's FP64 SoA unit vectors -> FP32 float4 copies in the same order
// (w = index), then sentinels up to n_pad.
__global__ void k_xyz_to_f32(const double* __restrict__ xyz, long long n, long long n_pad,
                             float4* __restrict__ p32, int tag) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n_pad;
         i += (long long)gridDim.x * blockDim.x) {
        if (i < n) {
            const double x = xyz[i], y = xyz[n + i], z = xyz[2 * n + i];
            check_unit(x, y, z);
            p32[i] = point32(x, y, z, i);
        } else {
            p32[i] = sentinel32(tag, i - n);
        }
    }
}

// ---------------------------------------------------------------------------
// spatial order: cube-map face + Hilbert index of a 2^L x 2^L grid on it
// ---------------------------------------------------------------------------
// Position along the Hilbert curve of cell (x, y) in an S x S grid (S a power
// of two): descend the quadrants from the largest, adding each quadrant's
// offset along the curve and reflecting/transposing the remaining coordinates
// into that quadrant's orientation.
__device__ __forceinline__ unsigned hilbert_index(unsigned S, unsigned x, unsigned y) {
    unsigned d = 0;
    for (unsigned h = S >> 1; h > 0; h >>= 1) {
        const unsigned rx = (x & h) ? 1u : 0u, ry = (y & h) ? 1u : 0u;
        d += h * h * ((3u * rx) ^ ry);
        if (ry == 0) {
            if (rx == 1) {
                x = S - 1 - x;
                y = S - 1 - y;
            }
            const unsigned t = x;
            x = y;
            y = t;
        }
    }
    return d;
}

__device__ __forceinline__ unsigned cell_key(double x, double y, double z, int L) {
    const double ax = fabs(x), ay = fabs(y), az = fabs(z);
    unsigned face;
    double u, v, m;
    if (ax >= ay && ax >= az) { face = x >= 0 ? 0u : 1u; u = y; v = z; m = ax; }
    else if (ay >= az)        { face = y >= 0 ? 2u : 3u; u = x; v = z; m = ay; }
    else                      { face = z >= 0 ? 4u : 5u; u = x; v = y; m = az; }
    const unsigned S = 1u << L;
    if (!(m > 0.0)) return face * S * S;  // not a unit vector; any cell will do
    const double fu = (u / m + 1.0) * 0.5 * (double)S, fv = (v / m + 1.0) * 0.5 * (double)S;
    const unsigned iu = (unsigned)fmin(fmax(fu, 0.0), (double)(S - 1));
    const unsigned iv = (unsigned)fmin(fmax(fv, 0.0), (double)(S - 1));
    return face * S * S + hilbert_index(S, iu, iv);
}

// Spatial order of a catalogue: a 31-bit key per point (cube-map face, then
// the Hilbert index of its cell on a 2^14 x 2^14 grid of the face, cells of
// about 20 arcsec), sorted by a stable least-significant-digit radix sort
// (4 passes of 8 bits: per-block digit counts, a scan of each digit's counts
// across the blocks, a stable scatter).  Consecutive points of the order are then close on the sky down
// to the scale of a few points, which the per-tile culling and the
// per-chunk settling of pairs both rely on.
constexpr int kSortLevel = 14;
constexpr int kSortThreads = 256;
// Rounds of 256 keys per block of the sort: enough blocks for about two per
// SM of a large GPU (at most 16 rounds), so that a small catalogue's passes
// are short, one round each, instead of a few blocks looping over 16 rounds.
static inline int sort_rounds(long long n) {
    const long long r = (n + 256LL * 304 - 1) / (256LL * 304);
    return (int)std::min<long long>(std::max<long long>(r, 1), 16);
}

__global__ void k_sort_keys(const double* __restrict__ xyz, long long stride, long long n,
                            int check, unsigned* __restrict__ key, unsigned* __restrict__ idx) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const double x = xyz[i], y = xyz[stride + i], z = xyz[2 * stride + i];
        if (check) check_unit(x, y, z);
        key[i] = cell_key(x, y, z, kSortLevel);
        idx[i] = (unsigned)i;
    }
}

// hist[d * n_blocks + b] = keys of block b whose digit is d.
__global__ void __launch_bounds__(kSortThreads) k_digit_hist(const unsigned* __restrict__ key,
                                                             long long n, int shift, int rounds,
                                                             unsigned* __restrict__ hist) {
    __shared__ unsigned cnt[256];
    const int t = threadIdx.x;
    cnt[t] = 0;
    __syncthreads();
    const long long tile = (long long)kSortThreads * rounds;
    const long long lo = blockIdx.x * tile, hi = min(lo + tile, n);
    for (long long i = lo + t; i < hi; i += kSortThreads) atomicAdd(&cnt[(key[i] >> shift) & 255u], 1u);
    __syncthreads();
    hist[(long long)t * gridDim.x + blockIdx.x] = cnt[t];
}

// Per digit d, the keys of digit d in blocks before b: hist[d * n_blocks + b]
// becomes that count (an exclusive scan along the digit's row, which is
// contiguous: coalesced), and tot[d] the digit's total.  One warp per digit,
// 8 digits per block of 256 threads.
__global__ void __launch_bounds__(256) k_digit_rows(unsigned* __restrict__ hist, int n_blocks,
                                                    unsigned* __restrict__ tot) {
    const int lane = threadIdx.x & 31;
    const int d = blockIdx.x * 8 + (threadIdx.x >> 5);
    unsigned* row = hist + (long long)d * n_blocks;
    unsigned run = 0;
#pragma unroll 4
    for (int b0 = 0; b0 < n_blocks; b0 += 32) {
        const int b = b0 + lane;
        const unsigned v = b < n_blocks ? row[b] : 0u;
        unsigned incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        if (b < n_blocks) row[b] = run + incl - v;
        run += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) tot[d] = run;
}

// Stable scatter of one pass: block b writes its keys of digit d from the
// keys of smaller digits (the exclusive scan of tot, done here by every
// block) plus rows[d * n_blocks + b] (k_digit_rows) on, in index order
// (rounds of 256 keys; inside a round, warps in order and lanes in order).
__global__ void __launch_bounds__(kSortThreads) k_digit_scatter(
    const unsigned* __restrict__ key_in, const unsigned* __restrict__ idx_in, long long n,
    int shift, int rounds, const unsigned* __restrict__ rows, const unsigned* __restrict__ tot,
    unsigned* __restrict__ key_out, unsigned* __restrict__ idx_out) {
    static_assert(kSortThreads == 256, "one thread per digit");
    __shared__ unsigned base[256];
    __shared__ unsigned wcnt[kSortThreads / 32][256];
    __shared__ unsigned wsum[kSortThreads / 32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    {
        const unsigned x = tot[t];
        unsigned incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        if (lane == 31) wsum[w] = incl;
        __syncthreads();
        unsigned pre = incl - x;
        for (int q = 0; q < w; ++q) pre += wsum[q];
        base[t] = pre + rows[(long long)t * gridDim.x + blockIdx.x];
    }
    const long long lo = blockIdx.x * (long long)kSortThreads * rounds;
    for (int r = 0; r < rounds; ++r) {
#pragma unroll
        for (int q = 0; q < kSortThreads / 32; ++q) wcnt[q][t] = 0;
        __syncthreads();
        const long long i = lo + (long long)r * kSortThreads + t;
        const bool valid = i < n;
        const unsigned k = valid ? key_in[i] : 0u;
        const unsigned d = valid ? (k >> shift) & 255u : 256u;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const unsigned rank = __popc(peers & ((1u << lane) - 1u));
        if (valid && rank == 0) wcnt[w][d] = __popc(peers);
        __syncthreads();
        {
            unsigned acc = base[t];
#pragma unroll
            for (int q = 0; q < kSortThreads / 32; ++q) {
                const unsigned c = wcnt[q][t];
                wcnt[q][t] = acc;
                acc += c;
            }
            base[t] = acc;
        }
        __syncthreads();
        if (valid) {
            const unsigned pos = wcnt[w][d] + rank;
            key_out[pos] = k;
            idx_out[pos] = idx_in[i];
        }
        __syncthreads();
    }
}

// One whole pass of a small sort (at most kSmallSort keys) in one launch: block
// b holds keys [1024 b, 1024 (b + 1)), one per thread.  hist[b' * 256 + d] are
// the digit counts of every block, which each block sums up itself (256
// threads a row, four rows at a time; at most 64 blocks), so no launch counts
// or scans them: the kernel before has counted this pass's digits, and this one
// counts the next pass's (next_hist, zeroed) while it scatters.  Stable: inside
// a block, warps in order and lanes in order.
//
// Bound by the latency of a launch and of about six dependent memory accesses:
// a w(theta) of 1k + 1k points took 96 us instead of 117 with three launches a
// pass, one of 10k + 10k 271 us instead of 300 (with the host copies), in the build
// that it came with (75 and 217 us now).
constexpr int kSmallThreads = 1024;
constexpr long long kSmallSort = 65536;
__global__ void __launch_bounds__(kSmallThreads) k_small_pass(
    const unsigned* __restrict__ key_in, const unsigned* __restrict__ idx_in, int n, int shift,
    const unsigned* __restrict__ hist, unsigned* __restrict__ next_hist,
    unsigned* __restrict__ key_out, unsigned* __restrict__ idx_out) {
    constexpr int NW = kSmallThreads / 32;
    __shared__ unsigned wcnt[NW][256];
    __shared__ unsigned tot[4][256], pre[4][256], wsum[8];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, b = blockIdx.x;
    const int i = b * kSmallThreads + t;
    const bool valid = i < n;
    const unsigned k = valid ? key_in[i] : 0u, ix = valid ? idx_in[i] : 0u;
    {
        const int d = t & 255, g = t >> 8, G = gridDim.x;
        unsigned all = 0, before = 0;
#pragma unroll 4
        for (int q = g; q < G; q += 4) {
            const unsigned c = hist[q * 256 + d];
            all += c;
            before += q < b ? c : 0u;
        }
        tot[g][d] = all;
        pre[g][d] = before;
    }
#pragma unroll
    for (int q = 0; q < NW * 256 / kSmallThreads; ++q) (&wcnt[0][0])[q * kSmallThreads + t] = 0u;
    __syncthreads();
    const unsigned d = valid ? (k >> shift) & 255u : 256u;
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    const unsigned rank = __popc(peers & ((1u << lane) - 1u));
    if (valid && rank == 0) wcnt[w][d] = __popc(peers);
    unsigned x = 0, incl = 0;
    if (t < 256) {
        x = tot[0][t] + tot[1][t] + tot[2][t] + tot[3][t];
        incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        if (lane == 31) wsum[w] = incl;
    }
    __syncthreads();
    if (t < 256) {
        unsigned acc = incl - x + pre[0][t] + pre[1][t] + pre[2][t] + pre[3][t];
        for (int q = 0; q < w; ++q) acc += wsum[q];
#pragma unroll 8
        for (int q = 0; q < NW; ++q) {
            const unsigned c = wcnt[q][t];
            wcnt[q][t] = acc;
            acc += c;
        }
    }
    __syncthreads();
    if (valid) {
        const unsigned pos = wcnt[w][d] + rank;
        key_out[pos] = k;
        idx_out[pos] = ix;
        if (next_hist)
            atomicAdd(next_hist + (pos / kSmallThreads) * 256 + ((k >> (shift + 8)) & 255u), 1u);
    }
}

// The one or two catalogues of a count, prepared together: both into one
// FP64 SoA array x (stride N = na + nb), converted from RA/Dec or copied from
// unit vectors (then checked), each point with its sort key (the cell key,
// with the catalogue in bit 31 so that b's points sort after a's) and its
// position.  hist (zeroed; or null): the first digit counts of a small sort's
// blocks.  FP64 work: launched in blocks of 64 threads, so that a small
// catalogue still spreads over every SM.
__global__ void __launch_bounds__(64) k_joint_keys(const double* __restrict__ a, long long na,
                                                   const double* __restrict__ b, long long nb,
                                                   int is_xyz, double* __restrict__ x,
                                                   unsigned* __restrict__ key,
                                                   unsigned* __restrict__ idx,
                                                   unsigned* __restrict__ hist) {
    const long long N = na + nb;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N;
         i += (long long)gridDim.x * blockDim.x) {
        const bool in_b = i >= na;
        const double* src = in_b ? b : a;
        const long long j = in_b ? i - na : i, n = in_b ? nb : na;
        double px, py, pz;
        if (is_xyz) {
            px = src[j];
            py = src[n + j];
            pz = src[2 * n + j];
            check_unit(px, py, pz);
        } else {
            radec_unit(src[2 * j], src[2 * j + 1], px, py, pz);
        }
        x[i] = px;
        x[N + i] = py;
        x[2 * N + i] = pz;
        const unsigned kv = cell_key(px, py, pz, kSortLevel) | (in_b ? 0x80000000u : 0u);
        key[i] = kv;
        idx[i] = (unsigned)i;
        if (hist) atomicAdd(hist + (i / kSmallThreads) * 256 + (kv & 255u), 1u);
    }
}

// One chunk of 32 consecutive positions of the spatial order, one point per
// lane (q its FP32 copy, (px, py, pz) its FP64 one): the bounding spheres of
// the chunk and of its groups of 8 points, and the points' coordinates relative
// to the chunk's centre c.
//   - Spheres (small_sphere): radius = the largest FP32 distance of a point from
//     the centre, enlarged by a relative 1e-6 for the few roundings of that
//     arithmetic.
//   - Local coordinates b' = fl32(b - c), from the FP64 points: the rounding is
//     relative to |b'|, so a chunk's own geometry is kept to 2^-24 of its size.
//   - For the pair kernel's local form (one_edge_step) the chunk keeps
//     kappa = |b|^2 - |c|^2 (for unit vectors the same for every point of the
//     chunk; the middle of its range here) and half the slack that the form
//     adds to an edge's guard band for this chunk: the deviation of kappa from
//     that middle, and u (12 r + 80 r^2 + 5 |kappa|) for the roundings that
//     grow with the chunk's radius r (u = 2^-24; derived at local_guard in the
//     host sources), times 1.05.
// A chunk holding a padding sentinel gets radius -1 and one wider than 0.5 gets
// radius 3, so that their pairs are never settled per chunk; both keep the
// origin as their centre (b' = the FP32 copy).
struct LocalChunks {
    float* xyz;       // planar local coordinates, stride apart
    long long stride;
    float4* caps;     // per chunk: centre, radius
    float4* groups;   // the same per group of 8 points
    float2* kap;      // per chunk: kappa, half the slack
};
// Bounding sphere of the points q of W adjacent lanes (8 or 32), nearly the
// smallest one: from the middle of their bounding box (c), eight steps towards
// the farthest point by 1/3, 1/4, ... of the distance (Badoiu and Clarkson), the
// best centre kept.  Against spheres around the mean, radii shrink by 13% (8
// points) and 8% (32) for uniform points and by a quarter for clustered ones,
// and with them the number of spans that hold an edge.
template <int W>
__device__ __forceinline__ float4 small_sphere(const float4& q, float3 c) {
    const unsigned lane = threadIdx.x & 31u;
    auto most = [](unsigned v) {
        if constexpr (W == 32) {
            return __reduce_max_sync(0xffffffffu, v);
        } else {
#pragma unroll
            for (int o = 1; o < W; o <<= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
            return v;
        }
    };
    float3 b = c;
    float best = __int_as_float(0x7f800000);
#pragma unroll 1
    for (int it = 0; it < 9; ++it) {
        const float dx = q.x - c.x, dy = q.y - c.y, dz = q.z - c.z;
        // the farthest lane, from the squared distance without its last bits
        const unsigned far =
            most((__float_as_uint(dx * dx + dy * dy + dz * dz) & ~31u) | lane);
        const float m = __uint_as_float(far & ~31u);
        if (m < best) {
            best = m;
            b = c;
        }
        const float st = 1.f / (float)(it + 3);
        c.x += st * (__shfl_sync(0xffffffffu, q.x, far & 31u) - c.x);
        c.y += st * (__shfl_sync(0xffffffffu, q.y, far & 31u) - c.y);
        c.z += st * (__shfl_sync(0xffffffffu, q.z, far & 31u) - c.z);
    }
    const float dx = q.x - b.x, dy = q.y - b.y, dz = q.z - b.z;
    const float r2 = __uint_as_float(most(__float_as_uint(dx * dx + dy * dy + dz * dz)));
    return make_float4(b.x, b.y, b.z, sqrtf(r2) * (1.f + 1e-6f));
}

__device__ __forceinline__ void write_chunk(long long i, const float4& q, double px, double py,
                                            double pz, const LocalChunks& L) {
    const int lane = threadIdx.x & 31;
    float3 lo = make_float3(q.x, q.y, q.z), hi = lo;
    auto widen = [&](int o) {
        lo.x = fminf(lo.x, __shfl_xor_sync(0xffffffffu, lo.x, o));
        lo.y = fminf(lo.y, __shfl_xor_sync(0xffffffffu, lo.y, o));
        lo.z = fminf(lo.z, __shfl_xor_sync(0xffffffffu, lo.z, o));
        hi.x = fmaxf(hi.x, __shfl_xor_sync(0xffffffffu, hi.x, o));
        hi.y = fmaxf(hi.y, __shfl_xor_sync(0xffffffffu, hi.y, o));
        hi.z = fmaxf(hi.z, __shfl_xor_sync(0xffffffffu, hi.z, o));
    };
    auto middle = [&] {
        return make_float3(0.5f * (lo.x + hi.x), 0.5f * (lo.y + hi.y), 0.5f * (lo.z + hi.z));
    };
    widen(1);
    widen(2);
    widen(4);
    const float4 group = small_sphere<8>(q, middle());
    if ((lane & 7) == 0) L.groups[i / 8] = group;
    widen(8);
    widen(16);
    const float4 sphere = small_sphere<32>(q, middle());
    float cx = sphere.x, cy = sphere.y, cz = sphere.z;
    const float r = sphere.w;
    // padding; NaN coordinates (which fminf and fmaxf pass over, but not r)
    const bool pad = __any_sync(0xffffffffu, is_sentinel(q));
    const bool nan = __any_sync(0xffffffffu, !(q.x + q.y + q.z == q.x + q.y + q.z));
    const bool wide = nan || !(r <= 0.5f && cx * cx + cy * cy + cz * cz <= 4.f);
    if (pad || wide) cx = cy = cz = 0.f;
    const double ex = px - (double)cx, ey = py - (double)cy, ez = pz - (double)cz;
    const double kb = ex * (px + (double)cx) + ey * (py + (double)cy) + ez * (pz + (double)cz);
    double k0 = kb, k1 = kb;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        k0 = fmin(k0, __shfl_xor_sync(0xffffffffu, k0, o));
        k1 = fmax(k1, __shfl_xor_sync(0xffffffffu, k1, o));
    }
    L.xyz[i] = pad ? q.x : (float)ex;
    L.xyz[L.stride + i] = pad ? q.y : (float)ey;
    L.xyz[2 * L.stride + i] = pad ? q.z : (float)ez;
    if (lane == 0) {
        const float kappa = (float)(0.5 * (k0 + k1));
        const float dev = (float)fmax(k1 - (double)kappa, (double)kappa - k0);
        const float rr = r + 2.4e-7f;
        const float slack = 1.05f * (dev + 5.9604645e-8f * (12.f * rr + 80.f * rr * rr +
                                                            5.f * fabsf(kappa)));
        L.caps[i / 32] = make_float4(cx, cy, cz, pad ? -1.f : wide ? 3.f : r);
        L.kap[i / 32] = make_float2(kappa, 0.5f * slack);
    }
}

// FP32 copies of both catalogues in the joint order (order: the sorted
// positions of x, a's points first): a's points at [0, na)
// and sentinels up to pa, b's at [pa, pa + nb) and sentinels up to pa + pb
// (tags tag0 and tag0 + 1), each point keeping in w its index within its own
// catalogue, and the chunks' spheres and local coordinates.  One warp per chunk
// (pa and pb are multiples of 32).  L.xyz may lie where the sort kept its keys.
__global__ void __launch_bounds__(256) k_gather_joint(const double* __restrict__ x, long long na,
                                                      long long pa, long long nb, long long pb,
                                                      const unsigned* __restrict__ order, int tag0,
                                                      float4* __restrict__ p32,
                                                      LocalChunks L) {
    const long long N = na + nb, P = pa + pb;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < P;
         i += (long long)gridDim.x * blockDim.x) {
        const bool in_b = i >= pa;
        const long long j = in_b ? i - pa : i, n = in_b ? nb : na;
        double px, py, pz;
        float4 q;
        if (j < n) {
            const long long k = order[(in_b ? na : 0) + j];
            px = x[k];
            py = x[N + k];
            pz = x[2 * N + k];
            q = point32(px, py, pz, in_b ? k - na : k);
        } else {
            q = sentinel32(tag0 + (in_b ? 1 : 0), j - n);
            px = q.x;
            py = q.y;
            pz = q.z;
        }
        p32[i] = q;
        write_chunk(i, q, px, py, pz, L);
    }
}

// Labels in sorted order (the digit of one more radix pass); a label outside
// [0, n_labels) sets WTHETA_DERR_LABEL and counts as 0.
__global__ void k_sorted_labels(const unsigned* __restrict__ order, const int* __restrict__ labels,
                                long long n, int n_labels, unsigned* __restrict__ out) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        int l = labels[order[i]];
        if (l < 0 || l >= n_labels) {
            atomicOr(&g_device_error, WTHETA_DERR_LABEL);
            l = 0;
        }
        out[i] = (unsigned)l;
    }
}

// sizes[l] = number of points with label l (labels sorted or not).
__global__ void k_count_labels(const unsigned* __restrict__ lab, long long n, int n_labels,
                               unsigned long long* __restrict__ sizes) {
    __shared__ unsigned c[256];
    for (int q = threadIdx.x; q < 256; q += blockDim.x) c[q] = 0;
    __syncthreads();
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        atomicAdd(&c[lab[i] & 255u], 1u);
    __syncthreads();
    for (int q = threadIdx.x; q < n_labels; q += blockDim.x)
        if (c[q]) atomicAdd(sizes + q, (unsigned long long)c[q]);
}

// FP32 copies with every region starting on a tile boundary: region r's
// points (sorted positions src[r] .. src[r+1]-1) go to dst[r] .., the rest of
// its last tile holds sentinels; with the chunks' spheres and local
// coordinates, one warp per chunk.  dst[R] = n_pad, a multiple of 32.  A sentinel is numbered
// within its region (below the tile size) and tagged by its region and
// array, so that no two sentinels a count can pair coincide in FP32 (numbered
// by their position in a long array, sentinels more than 2^24 points in would
// round onto one another).
__global__ void __launch_bounds__(256) k_gather_regions(const double* __restrict__ xyz,
                                                        long long stride,
                                                        const unsigned* __restrict__ order,
                                                        const long long* __restrict__ src,
                                                        const long long* __restrict__ dst, int R,
                                                        long long n_pad, float4* __restrict__ p32,
                                                        int tag, LocalChunks L) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n_pad;
         i += (long long)gridDim.x * blockDim.x) {
        int lo = 0, hi = R - 1;  // last region with dst <= i
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (dst[mid] <= i) lo = mid; else hi = mid - 1;
        }
        const long long j = i - dst[lo], n_lo = src[lo + 1] - src[lo];
        double px, py, pz;
        float4 q;
        if (j < n_lo) {
            const long long k = order[src[lo] + j];
            px = xyz[k];
            py = xyz[stride + k];
            pz = xyz[2 * stride + k];
            q = point32(px, py, pz, k);
        } else {
            q = sentinel32(2 * lo + tag, j - n_lo);
            px = q.x;
            py = q.y;
            pz = q.z;
        }
        p32[i] = q;
        write_chunk(i, q, px, py, pz, L);
    }
}

// The catalogues of a batch into one FP64 SoA array (stride N) with a label
// per point (its catalogue): catalogue c's points go to positions
// [off[c], off[c + 1]), converted from RA/Dec or copied from unit vectors.
struct BatchCat {
    const double* src;   // interleaved RA/Dec degrees, or SoA unit vectors (3 n)
    long long n;
};
__global__ void k_batch_gather(const BatchCat* __restrict__ cats, const long long* __restrict__ off,
                               int n_cats, int is_xyz, long long N, double* __restrict__ x,
                               int* __restrict__ lab) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N;
         i += (long long)gridDim.x * blockDim.x) {
        int lo = 0, hi = n_cats - 1;  // last catalogue with off <= i
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (off[mid] <= i) lo = mid; else hi = mid - 1;
        }
        const BatchCat c = cats[lo];
        const long long j = i - off[lo];
        double px, py, pz;
        if (is_xyz) {
            px = c.src[j];
            py = c.src[c.n + j];
            pz = c.src[2 * c.n + j];
        } else {
            radec_unit(c.src[2 * j], c.src[2 * j + 1], px, py, pz);
        }
        x[i] = px;
        x[N + i] = py;
        x[2 * N + i] = pz;
        lab[i] = lo;
    }
}

// acc[k] += add[k] for the K+2 slots (combining two counts of one shard).
__global__ void k_add_counts(unsigned long long* acc, const unsigned long long* add, int n) {
    for (int k = threadIdx.x; k < n; k += blockDim.x) acc[k] += add[k];
}

// counts[K+1] = total - sum(counts[0..K]): the overflow slot.
__global__ void k_finalize(unsigned long long* counts, int K, unsigned long long total) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        unsigned long long s = 0;
        for (int k = 0; k <= K; ++k) s += counts[k];
        counts[K + 1] = total - s;
    }
}

// ---------------------------------------------------------------------------
// the pair-count kernel
// ---------------------------------------------------------------------------
// kHistLane: one private uint32 column per thread, plain read-modify-write;
// kHistWarp: one column per warp, lanes with equal slots merged by
//            __match_any_sync and added by one shared atomic;
// kHistLaneAtomic: updated by a shared atomic add (one instruction instead of
//            load, add, store): four columns per warp in builds with span jobs,
//            one per thread in those without;
// kHistWarpRed: one column per warp, shared atomic add.

// Tile-pair index -> (I, J).  Auto: upper triangle I <= J, row-major.
__device__ __forceinline__ void item_to_tiles(long long t, long long T_a, long long T_b,
                                              int is_auto, long long* I, long long* J) {
    if (!is_auto) {
        *I = t < (1LL << 32) && T_b < (1LL << 32) ? (long long)((unsigned)t / (unsigned)T_b) : t / T_b;
        *J = t - *I * T_b;
        return;
    }
    if (T_a < (1 << 15)) {
        // as below in 32 bits: t < 2^29, so FP32 finds the row to within a few
        // and the exact comparisons settle it
        const int T = (int)T_a, k = (int)t;
        const float b = 2.f * (float)T + 1.f;
        int i = (int)((b - sqrtf(fmaxf(b * b - 8.f * (float)k, 0.f))) * 0.5f);
        i = min(max(i, 0), T - 1);
        while (i > 0 && i * T - i * (i - 1) / 2 > k) --i;
        while (i + 1 < T && (i + 1) * T - (i + 1) * i / 2 <= k) ++i;
        *I = i;
        *J = i + (k - (i * T - i * (i - 1) / 2));
        return;
    }
    const long long T = T_a;
    // rows 0..I-1 hold off(I) = I T - I (I - 1) / 2 items
    const double b = 2.0 * (double)T + 1.0;
    long long i = (long long)floor((b - sqrt(fmax(b * b - 8.0 * (double)t, 0.0))) * 0.5);
    if (i < 0) i = 0;
    if (i > T - 1) i = T - 1;
    while (i > 0 && i * T - i * (i - 1) / 2 > t) --i;
    while (i + 1 < T && (i + 1) * T - (i + 1) * i / 2 <= t) ++i;
    *I = i;
    *J = i + (t - (i * T - i * (i - 1) / 2));
}

// Bounding cap of each tile of T spatially ordered FP32 points (positions
// [0, n); padding sentinels, far off the unit sphere, are left out):
// centre = normalised FP64 sum, radius = the largest angle from the centre,
// plus 1e-6 rad for the FP32 rounding of the points (a point moves by at most
// ~1.1e-7 rad from its FP64 position).
__global__ void __launch_bounds__(128) k_tile_caps(const float4* __restrict__ p32, long long n,
                                                   int T, TileCap* __restrict__ caps) {
    __shared__ double red[4][4];
    __shared__ int cnt[4];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long t0 = (long long)blockIdx.x * T;
    const long long t1 = min(t0 + (long long)T, n);
    double sx = 0, sy = 0, sz = 0;
    int c = 0;
    for (long long i = t0 + tid; i < t1; i += blockDim.x) {
        const float4 q = p32[i];
        if (is_sentinel(q)) continue;
        sx += q.x; sy += q.y; sz += q.z;
        ++c;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sx += __shfl_xor_sync(0xffffffffu, sx, o);
        sy += __shfl_xor_sync(0xffffffffu, sy, o);
        sz += __shfl_xor_sync(0xffffffffu, sz, o);
        c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    if (lane == 0) { red[warp][0] = sx; red[warp][1] = sy; red[warp][2] = sz; cnt[warp] = c; }
    __syncthreads();
    sx = red[0][0] + red[1][0] + red[2][0] + red[3][0];
    sy = red[0][1] + red[1][1] + red[2][1] + red[3][1];
    sz = red[0][2] + red[1][2] + red[2][2] + red[3][2];
    c = cnt[0] + cnt[1] + cnt[2] + cnt[3];
    const double nrm = sqrt(sx * sx + sy * sy + sz * sz);
    const bool empty = c == 0;
    const bool spread = !(nrm > 1e-3 * (double)c);  // centre ill-defined: no skipping
    const double cx = spread ? 1.0 : sx / nrm, cy = spread ? 0.0 : sy / nrm,
                 cz = spread ? 0.0 : sz / nrm;
    double m = 0;
    for (long long i = t0 + tid; i < t1; i += blockDim.x) {
        const float4 q = p32[i];
        if (is_sentinel(q)) continue;
        const double dx = cx - q.x, dy = cy - q.y, dz = cz - q.z;
        m = fmax(m, dx * dx + dy * dy + dz * dz);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    __syncthreads();
    if (lane == 0) red[warp][3] = m;
    __syncthreads();
    if (tid == 0) {
        m = fmax(fmax(red[0][3], red[1][3]), fmax(red[2][3], red[3][3]));
        TileCap cap;
        cap.x = cx; cap.y = cy; cap.z = cz;
        cap.rho = empty ? -1.0
                        : (spread ? 4.0 : 2.0 * asin(fmin(1.0, 0.5 * sqrt(m))) + 1e-6);
        caps[blockIdx.x] = cap;
    }
}

// Whether two tiles may hold a pair below the top edge theta_top (radians):
// their caps' centres are closer than theta_top + both radii (+ 3e-6 rad of
// slack for the FP64 arithmetic here).  Empty tiles hold no pair.
__device__ __forceinline__ bool caps_may_meet(const TileCap& A, const TileCap& B,
                                              double theta_top) {
    if (!(A.rho >= 0.0 && B.rho >= 0.0)) return false;
    const double dx = A.x - B.x, dy = A.y - B.y, dz = A.z - B.z;
    const double chord = sqrt(dx * dx + dy * dy + dz * dz);
    const double theta_c = 2.0 * asin(fmin(1.0, 0.5 * chord));
    return theta_c - A.rho - B.rho - 3e-6 <= theta_top;
}

// Keeps the tile pairs that may hold a pair below the top edge: those whose
// caps are closer than theta_top + margin.  The skipped ones hold only
// overflow pairs (and empty tiles none), which the overflow slot (total minus
// the other slots) accounts for; counts stay exact.  Kept items are appended
// in any order (the counts do not depend on it).
__global__ void k_cull_items(const TileCap* __restrict__ ca, const TileCap* __restrict__ cb,
                             long long tiles_a, long long tiles_b, int is_auto, long long n_items,
                             double theta_top, unsigned* __restrict__ list,
                             unsigned long long* __restrict__ n_list,
                             unsigned long long* __restrict__ stats) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long n_round = (n_items + 31) / 32 * 32;
    const int lane = threadIdx.x & 31;
    unsigned long long skipped = 0;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n_round; t += stride) {
        bool keep = false;
        if (t < n_items) {
            long long I, J;
            item_to_tiles(t, tiles_a, tiles_b, is_auto, &I, &J);
            keep = caps_may_meet(ca[I], cb[J], theta_top);
            skipped += keep ? 0 : 1;
        }
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        unsigned long long base = 0;
        if (lane == 0 && m) base = atomicAdd(n_list, (unsigned long long)__popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (keep) list[base + __popc(m & ((1u << lane) - 1u))] = (unsigned)t;
    }
    if (stats) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) skipped += __shfl_xor_sync(0xffffffffu, skipped, o);
        if (lane == 0 && skipped) atomicAdd(stats + WTHETA_STAT_SKIPPED, skipped);
    }
}

// The same skipping for a batch's work table.  cs holds every count's items
// in the full table (begin, n), its tiles' caps and its list; each kept
// item's index within its count is appended to that count's list (in any
// order), kept[seg] counting them.
__global__ void k_cull_batch(const CullSeg* __restrict__ cs, int n_segs, long long total,
                             double theta_top, unsigned long long* __restrict__ kept,
                             unsigned long long* __restrict__ stats) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long n_round = (total + 31) / 32 * 32;
    const int lane = threadIdx.x & 31;
    unsigned long long skipped = 0;
    for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < n_round; g += stride) {
        bool keep = false;
        int seg = -1;
        long long local = 0;
        if (g < total) {
            int lo = 0, hi = n_segs - 1;  // last count with begin <= g
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (cs[mid].begin <= g) lo = mid; else hi = mid - 1;
            }
            seg = lo;
            local = g - cs[seg].begin + cs[seg].offset;
            long long I, J;
            item_to_tiles(local, cs[seg].ta, cs[seg].tb, cs[seg].is_auto, &I, &J);
            keep = caps_may_meet(cs[seg].ca[I], cs[seg].cb[J], theta_top);
            skipped += keep ? 0 : 1;
        }
        const unsigned peers = __match_any_sync(0xffffffffu, keep ? seg : -1);
        const int leader = __ffs(peers) - 1;
        unsigned long long base = 0;
        if (keep && lane == leader) base = atomicAdd(kept + seg, (unsigned long long)__popc(peers));
        base = __shfl_sync(0xffffffffu, base, leader);
        if (keep) cs[seg].list[base + __popc(peers & ((1u << lane) - 1u))] = (unsigned)local;
    }
    if (stats) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) skipped += __shfl_xor_sync(0xffffffffu, skipped, o);
        if (lane == 0 && skipped) atomicAdd(stats + WTHETA_STAT_SKIPPED, skipped);
    }
}

// Kept tile pairs per tile row of every count (rows[cs_row0[seg] + I]), for
// splitting the rows of each count among shards by their work.
__global__ void k_cull_rows(const CullSeg* __restrict__ cs, int n_segs, long long total,
                            double theta_top, const long long* __restrict__ row0,
                            unsigned long long* __restrict__ rows) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < total; g += stride) {
        int lo = 0, hi = n_segs - 1;  // last count with begin <= g
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (cs[mid].begin <= g) lo = mid; else hi = mid - 1;
        }
        const long long local = g - cs[lo].begin + cs[lo].offset;
        long long I, J;
        item_to_tiles(local, cs[lo].ta, cs[lo].tb, cs[lo].is_auto, &I, &J);
        if (caps_may_meet(cs[lo].ca[I], cs[lo].cb[J], theta_top)) atomicAdd(rows + row0[lo] + I, 1ull);
    }
}

// After k_cull_batch: each count's kept items become a contiguous range of
// the launch's items, in the table's order; *total receives their number.  One
// block scans the counts 1024 at a time (the region pairs of 64 regions are 8256
// counts: 0.03 ms; one thread walking them took about 0.75 of 12.1 ms).
constexpr int kPrefixThreads = 1024;
__global__ void __launch_bounds__(kPrefixThreads) k_cull_prefix(
    Segment* __restrict__ segs, const CullSeg* __restrict__ cs,
    const unsigned long long* __restrict__ kept, int n_segs,
    unsigned long long* __restrict__ total) {
    __shared__ unsigned long long wsum[kPrefixThreads / 32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    unsigned long long run = 0;
    for (int i0 = 0; i0 < n_segs; i0 += kPrefixThreads) {
        const int i = i0 + t;
        const unsigned long long x = i < n_segs ? kept[i] : 0ull;
        unsigned long long incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        if (lane == 31) wsum[w] = incl;
        __syncthreads();
        unsigned long long pre = run;
        for (int q = 0; q < kPrefixThreads / 32; ++q) {
            if (q < w) pre += wsum[q];
            run += wsum[q];
        }
        if (i < n_segs) {
            segs[i].item_begin = (long long)(pre + incl - x);
            segs[i].item_offset = 0;
            segs[i].item_list = cs[i].list;
        }
        __syncthreads();
    }
    if (t == 0) *total = run;
}

// sqrt within 2^-22 relative
__device__ __forceinline__ float sqrt_approx(float x) {
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// Edges at or below x (FP64 edges at shared address c64).
__device__ __forceinline__ unsigned edges_below(double x, unsigned c64, int K) {
    unsigned lo = 0, hi = (unsigned)K + 1;
    while (lo < hi) {
        const unsigned mid = (lo + hi) >> 1;
        if (lds_f64(c64 + 8u * mid) <= x) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// The definition's squared chord, in FP64, of the pair of sorted positions (ia, jb),
// read from the FP64 arrays through the original indices kept in the FP32 copies.
__device__ __forceinline__ double pair_chord2(const Segment& S, long long ia, long long jb) {
    const long long i = __float_as_int(S.a32[ia].w), j = __float_as_int(S.b32[jb].w);
    const double* a = S.a64;
    const double* b = S.b64;
    const long long as = S.a64_stride, bs = S.b64_stride;
    const double dx = __dsub_rn(a[i], b[j]);
    const double dy = __dsub_rn(a[as + i], b[bs + j]);
    const double dz = __dsub_rn(a[2 * as + i], b[2 * bs + j]);
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// FP64 recheck: the slot of that squared chord; c64 is the shared address of the
// FP64 edges.  hint >= 0: the slot just below the one edge whose guard band held the
// FP32 value (checked, else the edges are searched).
__device__ __forceinline__ unsigned recheck_slot(const Segment& S, long long ia, long long jb,
                                                 unsigned c64, int K, int hint = -1) {
    const double s = pair_chord2(S, ia, jb);
    if (hint >= 0 && hint <= K) {
        // the FP32 value lay in the guard band of edge `hint` alone: the slot
        // is hint or hint + 1, confirmed against the neighbouring edges
        if (s < lds_f64(c64 + 8u * (unsigned)hint)) {
            if (hint == 0 || lds_f64(c64 + 8u * (unsigned)(hint - 1)) <= s) return (unsigned)hint;
        } else if (hint == K || s < lds_f64(c64 + 8u * (unsigned)(hint + 1))) {
            return (unsigned)hint + 1u;
        }
    }
    return edges_below(s, c64, K);  // (K + 1: overflow)
}

// The staged B tile: per point its three coordinates, negated and duplicated
// for the packed FP32 arithmetic (24 B), so that two consecutive points are
// three 16-byte loads.  For span jobs a chunk of 32 points takes 16 B more, so
// that lanes on different chunks read different banks (PAD); without them all
// lanes read the same point, and a step's address is one addition.
constexpr unsigned kPointB = 24, kChunkB = 32 * kPointB + 16;
template <bool PAD>
__device__ __forceinline__ unsigned point_addr(unsigned tile, int j) {
    if (!PAD) return tile + (unsigned)j * kPointB;
    return tile + (unsigned)(j >> 5) * kChunkB + (unsigned)(j & 31) * kPointB;
}

// Items are taken in parts until there are this many per block.
constexpr int kPartWaves = 4;

template <int NT, int R, int JU, int HM, int DEF>
struct PairKernel {
    static constexpr int TA = NT * R;   // A points per tile
    static constexpr int TB = NT * R;   // B points per tile (equal: auto needs square tiles)
    static constexpr int NW = NT / 32;
    // Columns of the private histograms and the words from one slot's row to
    // the next.  With span jobs (kHistLaneAtomic, not deferred) the lanes of a
    // warp share CPW = 4 columns updated by shared reductions: most updates are
    // one or two per job, so sharing costs nothing measurable, and the columns
    // take an eighth of the memory (17.4 -> 2.3 KB at 32 bins), which keeps five
    // blocks on an SM and leaves the L1 room for their A tiles.  Rows lie an
    // odd number of words apart, so that lanes adding to different rows of one
    // column hit different banks.
    static constexpr int CPW = (HM == kHistWarp || HM == kHistWarpRed) ? 1
                               : HM == kHistLaneAtomic && DEF == 0     ? 4
                                                                       : 32;
    static constexpr int HCOLS = NW * CPW;
    static constexpr int HSTRIDE = CPW == 4 || HM == kHistWarpRed ? (HCOLS | 1) : HCOLS;
    __device__ static int column() {
        return (int)(threadIdx.x >> 5) * CPW + (int)(threadIdx.x & (CPW - 1));
    }
    static constexpr unsigned ROWB = 4u * HSTRIDE;
    static constexpr bool SPANS = DEF == 0 && HM != kHistWarp;  // has span jobs
    // Bytes of a screening-table entry in shared memory (lut_entry).
    static constexpr unsigned LUTB = SPANS ? 8 : 16;
    static constexpr unsigned TILEB = SPANS ? TB / 32 * kChunkB : TB * kPointB;

    // log2 of the most parts an item is taken in: eighths of the B tile (one unit
    // per sub-tile), or single chunks in a one-warp block.  With quarters at most,
    // 20k points without sorting were 840 parts for 760 blocks, almost two waves:
    // 245 us against 201 us
    static constexpr int MAXLP = NW == 1 ? ilog2(TB / 32) : 3;

    static size_t smem_bytes(int K, int n_lut) {
        size_t b = TILEB;                       // B tile
        b += (size_t)n_lut * LUTB;              // screening table
        b += (size_t)(K + 2) * 8;               // FP64 edges (+ pad)
        if (SPANS) {
            b += (size_t)TB / 32 * 16;          // bounding spheres of its 32-point chunks
            b += (size_t)TA / 8 * 16;           // bounding spheres of A's groups of 8
            b += (size_t)(K + 2) * 8;           // middle and half slack of every edge
        }
        b += (size_t)(K + 2) * ROWB;            // histograms, row K+1 a trash row
        return b;
    }
};

template <int NT, int HCOLS, int HSTRIDE = HCOLS>
__device__ __forceinline__ void flush_hist(unsigned* hist, int K,
                                           unsigned long long* __restrict__ counts) {
    if constexpr (HCOLS <= 32) {
        // few columns: a thread per row
        for (int b = threadIdx.x; b <= K + 1; b += NT) {
            unsigned long long sum = 0;
#pragma unroll 4
            for (int q = 0; q < HCOLS; ++q) {
                sum += (unsigned long long)(long long)(int)hist[b * HSTRIDE + q];
                hist[b * HSTRIDE + q] = 0;
            }
            if (sum && b <= K) atomicAdd(counts + b, sum);  // row K+1 is trash
        }
        return;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int b = warp; b <= K + 1; b += NT / 32) {
        unsigned long long sum = 0;
        for (int q = lane; q < HCOLS; q += 32) {
            // signed: an edge's counts go to a column as +n below and -n above it
            sum += (unsigned long long)(long long)(int)hist[b * HSTRIDE + q];
            hist[b * HSTRIDE + q] = 0;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0 && sum && b <= K) atomicAdd(counts + b, sum);  // row K+1 is trash
    }
}

template <int HM>
__device__ __forceinline__ void hist_add(unsigned cell, unsigned v) {
    if (HM == kHistLane) {
        unsigned c;
        asm volatile("ld.shared.b32 %0, [%1];" : "=r"(c) : "r"(cell) : "memory");
        asm volatile("st.shared.b32 [%0], %1;" :: "r"(cell), "r"(c + v) : "memory");
    } else {
        red_add_shared(cell, v);
    }
}

// Table entry of an FP32 squared chord's bucket (bits >= 0: non-negative).
// Builds with span jobs keep the 8 bytes of BinTable (LUTB = 8): their pairs are
// mostly told apart by edges, and the table leaves the L1 its room.  Builds that
// bin every pair through the table keep 16 bytes: the band's bounds and the byte
// offsets of the rows below and above it (both the trash row in a bucket with
// several edges, whose values are a band all over), four operations fewer per pair.
// 200k + 200k survey points without span binning: 10.6 ms with 8 bytes and a step's
// address by chunk, 9.2 in an earlier kernel, 9.0 with 16 bytes and point_addr<false>.
template <unsigned LUTB>
__device__ __forceinline__ auto lut_entry(unsigned bits, unsigned lut, int shift, int base,
                                          int top_idx) {
    const int idx = min(max((int)(bits >> shift) - base, 0), top_idx);
    if constexpr (LUTB == 8) return lds_u2(lut + 8u * (unsigned)idx);
    else return lds_u4(lut + 16u * (unsigned)idx);
}
// The entry's parts: whether bits lie below the edge's band, or inside it, the
// row they go to if not inside (provisionally, if inside, the row above), and the
// slot below the edge (-1: several edges).
__device__ __forceinline__ bool lut_below(uint2 e, unsigned bits) { return bits < e.x; }
__device__ __forceinline__ bool lut_band(uint2 e, unsigned bits, bool) {
    return bits - e.x <= e.y >> kLutWidthShift;  // below: the difference wraps
}
__device__ __forceinline__ unsigned lut_slot(uint2 e) { return e.y & kLutSlot; }
template <unsigned ROWB>
__device__ __forceinline__ unsigned lut_row(uint2 e, bool below) {
    return (lut_slot(e) + (below ? 0u : 1u)) * ROWB;
}
template <unsigned ROWB>
__device__ __forceinline__ int lut_hint(uint2 e) {
    return (e.y & kLutSeveral) ? -1 : (int)lut_slot(e);
}
__device__ __forceinline__ bool lut_below(uint4 e, unsigned bits) { return bits < e.x; }
// (from the comparison that is made anyway: with both made here, the compiler kept
// the entries of all of a step's values to the end, 254 registers against 174 at
// 16 A points a thread)
__device__ __forceinline__ bool lut_band(uint4 e, unsigned bits, bool below) {
    return !below && bits <= e.y;
}
template <unsigned ROWB>
__device__ __forceinline__ unsigned lut_row(uint4 e, bool below) {
    return below ? e.z : e.w;
}
template <unsigned ROWB>
__device__ __forceinline__ int lut_hint(uint4 e) {
    return e.w == e.z ? -1 : (int)(e.z / ROWB);
}
// The 16-byte entry of BinTable's entry (x, y).
template <unsigned ROWB>
__device__ __forceinline__ uint4 lut_wide(unsigned x, unsigned y, int K) {
    const unsigned slot = y & kLutSlot, row = slot * ROWB;
    if (x == 0xFFFFFFFFu) return make_uint4(x, x, row, row + ROWB);  // no edge: all below
    if (y & kLutSeveral) {
        const unsigned trash = ((unsigned)K + 1u) * ROWB;
        return make_uint4(x, x + (y >> kLutWidthShift), trash, trash);
    }
    return make_uint4(x, x + (y >> kLutWidthShift), row, row + ROWB);
}

// Bins NV screened values s[h R + r] (pairs of A point r and B point j + h)
// into the thread's private histogram column at shared address col (rows ROWB
// bytes apart).  The table gives the slot below the bucket's edge; a value
// beyond the top edge (or masked with +inf) lands in the trash row K+1.  A value
// inside a band is counted, for now, in the row above it; the function returns
// true if the step held any such value, and the caller then settles them
// (recount_band_values).  No branch.
template <int NV, int HM, unsigned ROWB, unsigned LUTB>
__device__ __forceinline__ bool bin_values(const float (&s)[NV], unsigned col, unsigned lut,
                                           int shift, int base, int top_idx) {
    bool any_band = false;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const unsigned bits = __float_as_uint(s[v]);
        const auto e = lut_entry<LUTB>(bits, lut, shift, base, top_idx);
        const bool below = lut_below(e, bits);
        any_band |= lut_band(e, bits, below);
        hist_add<HM>(col + lut_row<ROWB>(e, below), 1u);
    }
    return any_band;
}

// Bounds of edge k's guard band, a little outside the table's: its half-width
// (guard_half_width in the host sources) is at most u (11.4 sqrt(c) + 22.1 c)
// plus 6e-13, u = 2^-24.
__device__ __forceinline__ float guard_half(float c) {
    return 5.9604645e-8f * (12.f * sqrt_approx(c) + 24.f * c) + 1e-12f;
}
__device__ __forceinline__ bool outside_guard(float s, unsigned c64, unsigned k) {
    const float c = (float)lds_f64(c64 + 8u * k);
    return fabsf(s - c) > 1.1f * guard_half(c);
}

// A step's NV squared chords, passed by value.
template <int NV>
struct StepValues {
    float v[NV];
};

// Rare: the step held values inside a guard band.  Given the step's values
// again, take back their provisional counts and add each to the row its FP64
// recheck gives (one copy of the recheck code, in a loop over a bitmask);
// returns the number of values rechecked.  Kept out of line: its FP64
// registers then do not weigh on the loops that call it.  Where the first value
// lies in one edge's band, so does nearly always every other one, and FP64
// settles them without a search in FP32 before (10k + 10k points in 36 arcsec, 16
// bins 0.1 - 10 arcsec, 1.8e7 rechecks: 4.38 ms with it, 3.74 without; with a hint
// for each value 3.85, and 0.5% on every other workload, in spilled registers).
template <int NT, int R, int NV, int HM, unsigned ROWB, unsigned LUTB>
__device__ __noinline__ unsigned recount_band_values(const StepValues<NV> sv, unsigned col,
                                                     unsigned lut, int shift, int base,
                                                     int top_idx, int K, const Segment& S,
                                                     long long a0, long long bj, unsigned sC) {
    const float (&s)[NV] = sv.v;
    unsigned n_recheck = 0;
    unsigned mask = 0;
    int hint_v = -1, hint = -1;  // the first such value and its edge's lower slot
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const unsigned bits = __float_as_uint(s[v]);
        const auto e = lut_entry<LUTB>(bits, lut, shift, base, top_idx);
        if (lut_band(e, bits, lut_below(e, bits))) {
            mask |= 1u << v;
            hist_add<HM>(col + lut_row<ROWB>(e, false), 0xFFFFFFFFu);  // -1
            if (hint_v < 0) {
                hint_v = v;
                hint = lut_hint<ROWB>(e);
            }
        }
    }
    while (mask) {
        const int v = __ffs(mask) - 1;
        mask &= mask - 1;
        unsigned slot = 0;
        bool sure = false;
        if (hint < 0) {
            // the step met a bucket with several edges: the edges searched in FP32
            // first, and FP64 only within a guard band of the edges next to it
            float x;
            if constexpr (LUTB == 8) {
                x = s[v];
            } else {
                x = s[0];  // s[v] without an index: s stays in registers
#pragma unroll
                for (int w = 1; w < NV; ++w) x = v == w ? s[w] : x;
            }
            slot = edges_below(x, sC, K);
            sure = (slot == 0u || outside_guard(x, sC, slot - 1u)) &&
                   (slot > (unsigned)K || outside_guard(x, sC, slot));
        }
        if (!sure) {
            slot = recheck_slot(S, a0 + v % R, bj + v / R, sC, K, v == hint_v ? hint : -1);
            ++n_recheck;
        }
        hist_add<HM>(col + slot * ROWB, 1u);
    }
    return n_recheck;
}

// Squared chords of JU consecutive B points (from tile position j, at shared
// address b) with the thread's R A points: s[h R + r].  On a diagonal tile,
// pairs with i >= j get +inf, i being a_first + r (the thread's first A point's
// position in the tile).
template <int R, int JU, bool DIAG>
__device__ __forceinline__ void chords(float (&s)[JU * R], unsigned b, const f2_t (&ax)[R / 2],
                                       const f2_t (&ay)[R / 2], const f2_t (&az)[R / 2], int j,
                                       int a_first) {
    static_assert(JU <= 2, "");
    f2_t bx[JU], by[JU], bz[JU];
    if (JU == 2) {
        lds_f2x2(b, bx[0], by[0]);
        lds_f2x2(b + 16u, bz[0], bx[JU - 1]);
        lds_f2x2(b + 32u, by[JU - 1], bz[JU - 1]);
    } else {
        bx[0] = lds_f2(b);
        by[0] = lds_f2(b + 8u);
        bz[0] = lds_f2(b + 16u);
    }
#pragma unroll
    for (int h = 0; h < JU; ++h) {
#pragma unroll
        for (int q = 0; q < R / 2; ++q) {
            const f2_t dx = add2(ax[q], bx[h]);
            const f2_t dy = add2(ay[q], by[h]);
            const f2_t dz = add2(az[q], bz[h]);
            const f2_t t = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
            unpack2(t, s[h * R + 2 * q], s[h * R + 2 * q + 1]);
        }
    }
    if (DIAG) {
#pragma unroll
        for (int h = 0; h < JU; ++h)
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (j + h <= a_first + r) s[h * R + r] = __int_as_float(0x7f800000);
    }
}

template <int NV>
__device__ __forceinline__ float min_of(const float (&s)[NV]) {
    float m = s[0];
#pragma unroll
    for (int v = 1; v + 1 < NV; v += 2) m = min3f(m, s[v], s[v + 1]);
    if (NV % 2 == 0) m = fminf(m, s[NV - 1]);
    return m;
}

// The FP32 steps [j0, j1) of a B tile for the thread's R A points, each pair
// binned through the table (values inside a guard band settled in FP64).
template <int NT, int R, int JU, int HM, unsigned ROWB, bool DIAG>
__device__ __forceinline__ void exact_steps(int j0, int j1, unsigned tile, unsigned lut,
                                            unsigned sC, unsigned col, const f2_t (&ax)[R / 2],
                                            const f2_t (&ay)[R / 2], const f2_t (&az)[R / 2],
                                            float hf, int shift, int base, int top_idx, int K,
                                            const Segment& S, long long a0, long long b0,
                                            int a_first, unsigned long long& n_recheck) {
    constexpr int NV = JU * R;
    constexpr unsigned LUTB = 16;  // (builds without span jobs)
    unsigned b = point_addr<false>(tile, j0);
#pragma unroll 1
    for (int j = j0; j < j1; b += JU * kPointB, j += JU) {
        float s[NV];
        chords<R, JU, DIAG>(s, b, ax, ay, az, j, a_first);
        const float m = min_of(s);
        if (!(m <= hf)) continue;
        if (bin_values<NV, HM, ROWB, LUTB>(s, col, lut, shift, base, top_idx)) {
            StepValues<NV> s2;
            chords<R, JU, DIAG>(s2.v, b, ax, ay, az, j, a_first);
            n_recheck += recount_band_values<NT, R, NV, HM, ROWB, LUTB>(
                s2, col, lut, shift, base, top_idx, K, S, a0, b0 + j, sC);
        }
    }
}

// How the pairs of a group of A points (sphere ga) with a chunk of B points
// (sphere gb) can be settled.  By the triangle inequality every FP32 pair
// distance lies within |ca - cb| -/+ (ra + rb); the FP64 unit vectors are
// within 1.2e-7 of their FP32 copies and the FP32 arithmetic here errs by a
// few units in the last place, all covered by the 1e-6 absolute and relative
// slack, so every pair's FP64 squared chord lies in [slo, shi].  The table
// gives the lowest slot rlo and the highest slot rhi that the interval can
// touch (an end inside an edge's guard band takes the edge in; a bucket with
// several edges has them searched, their FP32 values being far closer to the
// FP64 ones than the slack).  Returns the number of edges between them:
//   0        every pair is in slot rlo (a span wholly above h_top, the top
//            edge's band, is the overflow slot K + 1 at once);
//   1 .. kMaxEdges  the counts of the slots follow from the number of pairs
//            below each of those edges (up to kMaxEdgesFar if the span reaches
//            beyond 60 degrees);
//   -1       more edges, or padding: bin pair by pair.
// Two edges cost a job about a quarter of the table's lookups and shared
// atomics for its 256 pairs.  kMaxEdges 4, 6, 8: 256 log bins to 20 deg (200k + 200k
// points) 7.80, 7.67, 7.87 ms; 24 bins (30k x 48k) 446, 444, 444 us with the host's
// part; 32 bins (1M + 1M) 29.26, 29.26, 29.29 ms; 60 linear bins to 60 deg (100k +
// 100k) 7.14, 7.26, 7.32 ms.
// Beyond 60 degrees the line is 16, because values in a bucket with several edges
// are recounted out of line, one by one, and linear bins have such buckets there
// (the table's buckets are steps of the logarithm).  The span's ends do not tell:
// 36 linear bins have only one, just below 180 deg, and the spans across it end in
// the next.  6 everywhere / a line of 16 where an end meets such a bucket / this / 16
// everywhere, full sky: 36 bins (100k + 100k) 12.3, 12.5, 8.2, 8.2 ms (4.7e7 values
// recounted with 6, 1.1e6 with this), 256 bins (100k + 100k) 203, 166, 134, 134, 90
// bins (300k + 300k) 175, 154, 104, 104, 20 bins from 60 deg 6.0, 6.0, 6.2, 6.2; the
// 256 log bins to 20 deg 7.6, 7.7, 7.7, 9.0.
constexpr int kMaxEdges = 6, kMaxEdgesFar = 16;
__device__ __forceinline__ int span_edges(float4 ga, float4 gb, unsigned lut, unsigned c64,
                                          int shift, int base, int top_idx, int K, unsigned h_top,
                                          unsigned& rlo, unsigned& rhi) {
    const float dx = ga.x - gb.x, dy = ga.y - gb.y, dz = ga.z - gb.z;
    const float dc = sqrt_approx(dx * dx + dy * dy + dz * dz);
    const float rr = (ga.w + gb.w) * (1.f + 1e-6f) + 1e-6f;
    const float lo = fmaxf(dc * (1.f - 1e-6f) - rr, 0.f), hi = dc * (1.f + 1e-6f) + rr;
    const float slo = lo * lo * (1.f - 1e-5f);
    const float shi = hi * hi * (1.f + 1e-5f);
    const unsigned bl = __float_as_uint(slo), bh = __float_as_uint(shi);
    // padding (a group's radius far above 2, a chunk's -1), a wide chunk, NaN
    const bool real = (ga.w <= 2.f) & (gb.w >= 0.f) & (gb.w <= 2.f);
    if (__all_sync(0xffffffffu, real && bl > h_top)) {  // the whole warp beyond the top edge
        rlo = rhi = (unsigned)K + 1u;
        return 0;
    }
    const uint2 el = lut_entry<8>(bl, lut, shift, base, top_idx);
    const uint2 eh = lut_entry<8>(bh, lut, shift, base, top_idx);
    rlo = lut_slot(el) + ((lut_below(el, bl) | lut_band(el, bl, false)) ? 0u : 1u);
    rhi = lut_slot(eh) + (lut_below(eh, bh) ? 0u : 1u);
    if ((el.y | eh.y) & kLutSeveral) {
        rlo = edges_below(slo, c64, K);
        rhi = edges_below(shi, c64, K);
    }
    const int most = shi >= 1.f ? kMaxEdgesFar : kMaxEdges;
    if (bl > h_top) rlo = rhi = (unsigned)K + 1u;
    const int n = (int)(rhi - rlo);
    return real && n <= most ? n : -1;
}

// The local form of a pair's squared chord: with the chunk's centre c, b = c +
// b', and a' = a - c,
//     s = |a'|^2 + kappa - 2 a.b',   kappa = |b|^2 - |c|^2,
// where kappa is one number for the whole chunk when b is a unit vector.  So
// per pair d = (s - mid) / 2 is three fused multiply-adds from
// A0 = (|a'|^2 + (kappa - mid)) / 2, which each A point has once per job, and
// the three subtractions of |a - b|^2 fall away.  The products are small (|b'|
// is at most the chunk's radius), so the roundings stay below those of the
// difference form; |d| > G, G the edge's half slack plus the chunk's
// (local_guard, write_chunk), settles the side of the FP64 squared chord.
//
// A one-edge step is 12 packed fmas per B point and 8 A points.
//
// One step: two B points (staged negated, at shared address b) and the
// thread's R A points.  neg[q]
// counts the values with d < 0 and mb[q] keeps the smallest |d|, one
// accumulator per A pair q so that the steps' dependency chains interleave.
template <int R>
__device__ __forceinline__ void one_edge_step(unsigned b, const f2_t (&ax)[R / 2],
                                              const f2_t (&ay)[R / 2], const f2_t (&az)[R / 2],
                                              const f2_t (&a0)[R / 2], unsigned (&neg)[R / 2],
                                              float (&mb)[R / 2]) {
    f2_t bx[2], by[2], bz[2];
    lds_f2x2(b, bx[0], by[0]);
    lds_f2x2(b + 16u, bz[0], bx[1]);
    lds_f2x2(b + 32u, by[1], bz[1]);
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int q = 0; q < R / 2; ++q) {
            float d0, d1;
            unpack2(fma2(ax[q], bx[h], fma2(ay[q], by[h], fma2(az[q], bz[h], a0[q]))), d0, d1);
            mb[q] = min3f(mb[q], fabsf(d0), fabsf(d1));
            add_sign(neg[q], d0);
            add_sign(neg[q], d1);
        }
}

// One step against two edges, the second's
// value from the first's by one more subtraction of half their distance
// (ndel = -(mid2 - mid1) / 2).
template <int R>
__device__ __forceinline__ void two_edge_step(unsigned b, const f2_t (&ax)[R / 2],
                                              const f2_t (&ay)[R / 2], const f2_t (&az)[R / 2],
                                              const f2_t (&a0)[R / 2], f2_t ndel, unsigned& neg1,
                                              unsigned& neg2, float& mb1, float& mb2) {
    f2_t bx[2], by[2], bz[2];
    lds_f2x2(b, bx[0], by[0]);
    lds_f2x2(b + 16u, bz[0], bx[1]);
    lds_f2x2(b + 32u, by[1], bz[1]);
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int q = 0; q < R / 2; ++q) {
            const f2_t t = fma2(ax[q], bx[h], fma2(ay[q], by[h], fma2(az[q], bz[h], a0[q])));
            float d0, d1, e0, e1;
            unpack2(t, d0, d1);
            unpack2(add2(t, ndel), e0, e1);
            mb1 = min3f(mb1, fabsf(d0), fabsf(d1));
            mb2 = min3f(mb2, fabsf(e0), fabsf(e1));
            add_sign(neg1, d0);
            add_sign(neg1, d1);
            add_sign(neg2, e0);
            add_sign(neg2, e1);
        }
}

// The pairs of the thread's R A points (tile positions a_first ..) with the
// B points [j_begin, j_end) of the staged tile.
template <int NT, int R, int JU, int HM, int DEF, bool DIAG>
__device__ __forceinline__ void tile_pass(unsigned tile, unsigned lut, unsigned sC, unsigned hist,
                                          const f2_t (&ax)[R / 2], const f2_t (&ay)[R / 2],
                                          const f2_t (&az)[R / 2], const PairParams& p,
                                          const Segment& S, long long I, long long J, int a_first,
                                          int j_begin, int j_end,
                                          unsigned long long& n_recheck) {
    using PK = PairKernel<NT, R, JU, HM, DEF>;
    constexpr int TA = PK::TA, TB = PK::TB;
    constexpr int NV = JU * R;
    const int lane = threadIdx.x & 31;
    const unsigned h_top = p.tab.h_top;
    const float hf = __uint_as_float(h_top);
    const int shift = p.tab.shift, base = p.tab.base, K = p.tab.K, top_idx = p.tab.n_lut - 1;
    constexpr unsigned ROWB = PK::ROWB, LUTB = PK::LUTB;
    const unsigned col = hist + 4u * (unsigned)PK::column();
    const long long a0 = I * TA + a_first, b0 = J * TB;

    if (DEF == 1) {
        // Deferred binning: the screening loop only notes, one bit per step,
        // which of 32 consecutive steps hold an in-range value; those steps
        // are then recomputed and binned.  The screening loop stays small.
        static_assert(DEF != 1 || TB % (8 * 32 * JU) == 0, "an eighth holds whole 32-step blocks");
#pragma unroll 1
        for (int jb = j_begin; jb < j_end; jb += 32 * JU) {
            unsigned mask = 0;
#pragma unroll 1
            for (int st = 0; st < 32; ++st) {
                float s[NV];
                chords<R, JU, DIAG>(s, point_addr<false>(tile, jb + st * JU), ax, ay, az,
                                    jb + st * JU, a_first);
                mask |= (min_of(s) <= hf ? 1u : 0u) << st;
            }
            while (mask) {
                const int st = __ffs(mask) - 1;
                mask &= mask - 1;
                const int j = jb + st * JU;
                StepValues<NV> s;
                chords<R, JU, DIAG>(s.v, point_addr<false>(tile, j), ax, ay, az, j, a_first);
                if (bin_values<NV, HM, ROWB, LUTB>(s.v, col, lut, shift, base, top_idx))
                    n_recheck += recount_band_values<NT, R, NV, HM, ROWB, LUTB>(
                        s, col, lut, shift, base, top_idx, K, S, a0, b0 + j, sC);
            }
        }
        return;
    } else if (HM == kHistWarp) {
#pragma unroll 1
        for (int j = j_begin; j < j_end; j += JU) {
            float s[NV];
            chords<R, JU, DIAG>(s, point_addr<false>(tile, j), ax, ay, az, j, a_first);
            const float m = min_of(s);
            if (!__any_sync(0xffffffffu, m <= hf)) continue;
            unsigned amb_mask = 0;
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const unsigned bits = __float_as_uint(s[v]);
                const auto e = lut_entry<LUTB>(bits, lut, shift, base, top_idx);
                const bool below = lut_below(e, bits), amb = lut_band(e, bits, below);
                amb_mask |= amb ? (1u << v) : 0u;
                const unsigned off =
                    amb ? ((unsigned)K + 1u) * ROWB : lut_row<ROWB>(e, below);
                const unsigned peers = __match_any_sync(0xffffffffu, off);
                if (lane == __ffs(peers) - 1) red_add_shared(col + off, (unsigned)__popc(peers));
            }
            while (amb_mask) {
                const int v = __ffs(amb_mask) - 1;
                amb_mask &= amb_mask - 1;
                const unsigned slot = recheck_slot(S, a0 + v % R, b0 + j + v / R, sC, K);
                ++n_recheck;
                red_add_shared(col + slot * ROWB, 1u);
            }
        }
        return;
    }
    // pair by pair as screened
    exact_steps<NT, R, JU, HM, ROWB, DIAG>(j_begin, j_end, tile, lut, sC, col, ax, ay, az, hf, shift,
                                           base, top_idx, K, S, a0, b0, a_first, n_recheck);
}

// The thread's R A points, R consecutive points of the spatial order (a
// compact group: see write_chunk), packed two by two for the FP32x2
// instructions.  Each value goes through an explicit add of +0 (exact; it
// only turns -0 into +0, which leaves every squared chord unchanged): the
// packed operands then get registers of their own instead of being formed in
// place from the vector-load destinations, a layout measured to cost about a
// quarter of the screening loop's throughput.
template <int R>
__device__ __forceinline__ void load_group(const float4* __restrict__ gA, f2_t (&ax)[R / 2],
                                           f2_t (&ay)[R / 2], f2_t (&az)[R / 2]) {
#pragma unroll
    for (int q = 0; q < R / 2; ++q) {
        const float4 a = gA[2 * q];
        const float4 b = gA[2 * q + 1];
        ax[q] = pack2(__fadd_rn(a.x, 0.f), __fadd_rn(b.x, 0.f));
        ay[q] = pack2(__fadd_rn(a.y, 0.f), __fadd_rn(b.y, 0.f));
        az[q] = pack2(__fadd_rn(a.z, 0.f), __fadd_rn(b.z, 0.f));
    }
}

// The R consecutive points from position pos on (R | pos) of the planar local
// coordinates p, packed two by two: relative to the centre of their own chunk.
// A warp that reads 32 groups of one sub-tile touches 8 lines per load (lanes
// 32 B apart) where float4 points, 128 B apart, touch 32: the reads of the
// jobs' A points had been over half of the L1 data pipe's wavefronts, which
// bounded the kernel (69% of their peak rate, FMA and ALU pipes at 40%).
template <int R>
__device__ __forceinline__ void load_local(const float* __restrict__ p, long long stride,
                                           long long pos, f2_t (&ax)[R / 2], f2_t (&ay)[R / 2],
                                           f2_t (&az)[R / 2]) {
#pragma unroll
    for (int q = 0; q < R / 4; ++q) {
        const float4 x = *reinterpret_cast<const float4*>(p + pos + 4 * q);
        const float4 y = *reinterpret_cast<const float4*>(p + stride + pos + 4 * q);
        const float4 z = *reinterpret_cast<const float4*>(p + 2 * stride + pos + 4 * q);
        ax[2 * q] = pack2(x.x, x.y);
        ax[2 * q + 1] = pack2(x.z, x.w);
        ay[2 * q] = pack2(y.x, y.y);
        ay[2 * q + 1] = pack2(y.z, y.w);
        az[2 * q] = pack2(z.x, z.y);
        az[2 * q + 1] = pack2(z.z, z.w);
    }
}

// The group's points, given relative to centre a, relative to centre b (b = 0:
// the points themselves).  b - a is rounded relative to itself and the sum
// relative to itself, so a coordinate difference against a point b' of b's
// chunk errs by about 2 u |a - b| + u (ra + rb) instead of the 2 u of
// differences of the FP32 copies.  A squared chord of such differences errs by
// at most u (10 s + sqrt(s) (6 r + 4 ra)), r and ra <= 0.5 (write_chunk): inside the
// guard band derived for the FP32 copies, u (11.3 sqrt(c) + 22 c).
template <int R>
__device__ __forceinline__ void recentre(const float4& a, const float4& b, const f2_t (&ax)[R / 2],
                                         const f2_t (&ay)[R / 2], const f2_t (&az)[R / 2],
                                         f2_t (&lx)[R / 2], f2_t (&ly)[R / 2], f2_t (&lz)[R / 2]) {
    const float x = a.x - b.x, y = a.y - b.y, z = a.z - b.z;
    const f2_t dx = pack2(x, x), dy = pack2(y, y), dz = pack2(z, z);
#pragma unroll
    for (int q = 0; q < R / 2; ++q) {
        lx[q] = add2(ax[q], dx);
        ly[q] = add2(ay[q], dy);
        lz[q] = add2(az[q], dz);
    }
}

// Sphere c of the staged chunks or groups (caps: shared address).
__device__ __forceinline__ float4 chunk_sphere(unsigned caps, int c) {
    const uint4 g = lds_u4(caps + 16u * (unsigned)c);
    return make_float4(__uint_as_float(g.x), __uint_as_float(g.y), __uint_as_float(g.z),
                       __uint_as_float(g.w));
}

// ---------------------------------------------------------------------------
// Span jobs.  A (group, chunk) pair whose span needs its pairs computed is one
// or more jobs: for every edge inside the span the number of pairs below it is
// counted, two edges to a job (kJobTwo) and the last of an odd number alone
// (kJobOne); a span with too many edges is one job binned pair by pair
// (kJobExact).  Every pair of a span of edges goes to its highest slot at
// first, and an edge with n pairs below it then moves n of them one slot down
// (+n below, -n above), so the jobs of a span are independent of one another.
// Each warp keeps one ring of jobs per kind in shared memory and runs 32 of
// them as one round, one job per lane: a lane computes only pairs whose slot
// is not known from the spheres, whatever its own group's spans, and the lanes
// of a round run the same loop.
// ---------------------------------------------------------------------------
constexpr int kJobOne = 0, kJobTwo = 1, kJobExact = 2, kJobKinds = 3, kChunk = 32;
constexpr int kRing = 64;  // words of a ring: fewer than 32 waiting, at most 32 pushed at once

// Bits 0-4 lane, 5-7 sub-tile, 8-15 chunk, 16-24 the (first) edge.  While a
// lane still has jobs of a span to push, bits 25-30 of its word hold the number
// of edges left, or kExact for one job pair by pair.
constexpr unsigned kExact = 32u, kJobBits = (1u << 25) - 1u;
__device__ __forceinline__ unsigned job_word(int lane, int sub, int chunk, unsigned slot) {
    return (unsigned)lane | ((unsigned)sub << 5) | ((unsigned)chunk << 8) | (slot << 16);
}

__device__ __forceinline__ unsigned atom_add_shared(unsigned a, unsigned v) {
    unsigned old;
    asm volatile("atom.shared.add.u32 %0, [%1], %2;" : "=r"(old) : "r"(a), "r"(v) : "memory");
    return old;
}

// A job's R A points (the owner lane's group), relative to the centre ca of
// their own chunk.
template <int NT, int R, int JU, int HM>
__device__ __forceinline__ int job_points(unsigned job, unsigned sIJ, const Segment& S, float4& ca,
                                          f2_t (&ax)[R / 2], f2_t (&ay)[R / 2],
                                          f2_t (&az)[R / 2]) {
    constexpr int TA = PairKernel<NT, R, JU, HM, 0>::TA, SA = 32 * R;
    const int a_first = (int)((job >> 5) & 7u) * SA + (int)(job & 31u) * R;
    const long long pos = lds_s64(sIJ) * TA + a_first;
    ca = __ldg(S.a_caps + pos / kChunk);
    load_local<R>(S.al, S.al_stride, pos, ax, ay, az);
    return a_first;
}

// The pairs of a group of R A points (relative to chunk c's centre; positions
// a0 .. of the catalogue, a_first .. of the tile) with the chunk's points t0, t0 +
// ts, ... (positions b0 + t) binned through the table, values inside a guard
// band settled in FP64.  One B point per step: fewer live values.  DIAG: only
// pairs i < j.
template <int NT, int R, int HM, unsigned ROWB, bool DIAG>
__device__ __forceinline__ void exact_chunk(unsigned tile, int c, int t0, int ts, unsigned lut,
                                            unsigned sC, unsigned col, const f2_t (&ax)[R / 2],
                                            const f2_t (&ay)[R / 2], const f2_t (&az)[R / 2],
                                            const PairParams& p, const Segment& S, long long a0,
                                            long long b0, int a_first, unsigned& n_recheck) {
    const float hf = __uint_as_float(p.tab.h_top);
    const int shift = p.tab.shift, base = p.tab.base, top_idx = p.tab.n_lut - 1;
#pragma unroll 1
    for (int t = t0; t < kChunk; t += ts) {
        const unsigned b = tile + (unsigned)c * kChunkB + (unsigned)t * kPointB;
        const int j = c * kChunk + t;
        float s[R];
        chords<R, 1, DIAG>(s, b, ax, ay, az, j, a_first);
        if (!(min_of(s) <= hf)) continue;
        if (bin_values<R, HM, ROWB, 8>(s, col, lut, shift, base, top_idx)) {
            StepValues<R> s2;
            chords<R, 1, DIAG>(s2.v, b, ax, ay, az, j, a_first);
            n_recheck += recount_band_values<NT, R, R, HM, ROWB, 8>(
                s2, col, lut, shift, base, top_idx, p.tab.K, S, a0, b0 + t, sC);
        }
    }
}

// A job of the pair-by-pair kind.
template <int NT, int R, int JU, int HM>
__device__ __forceinline__ void exact_job(unsigned job, int t0, int ts, unsigned sIJ, unsigned tile,
                                          unsigned lut, unsigned caps, unsigned sC, unsigned col,
                                          const PairParams& p, const Segment& S,
                                          unsigned& n_recheck) {
    using PK = PairKernel<NT, R, JU, HM, 0>;
    f2_t ax[R / 2], ay[R / 2], az[R / 2];
    float4 ca;
    const int a_first = job_points<NT, R, JU, HM>(job, sIJ, S, ca, ax, ay, az);
    const int c = (int)((job >> 8) & 255u);
    recentre<R>(ca, chunk_sphere(caps, c), ax, ay, az, ax, ay, az);
    exact_chunk<NT, R, HM, PK::ROWB, false>(tile, c, t0, ts, lut, sC, col, ax, ay, az, p, S,
                                            lds_s64(sIJ) * PK::TA + a_first,
                                            lds_s64(sIJ + 8u) * PK::TB + c * kChunk, a_first,
                                            n_recheck);
}

// The middle of edge k (edge table at shared address band) and half its slack
// for the local form.
__device__ __forceinline__ float edge_mid(unsigned band, unsigned k, float& G) {
    float mid;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(mid), "=f"(G) : "r"(band + 8u * k));
    return mid;
}

// A job of kind T (one or two edges) over the chunk's steps t0, t0 + ts, ...
// (two points each).  neg1 and neg2 count the values below the first and second
// edge (neg2 = 0 for one), mb1 and mb2 return the smallest |d| less the slack:
// at most zero if some value may be on either side.
template <int NT, int R, int JU, int HM>
__device__ __forceinline__ void span_part(int T, unsigned job, int t0, int ts, unsigned sIJ,
                                          unsigned tile, unsigned caps, unsigned band,
                                          const Segment& S, unsigned& neg1, unsigned& neg2,
                                          float& mb1, float& mb2) {
    constexpr int CPT = PairKernel<NT, R, JU, HM, 0>::TB / kChunk;
    const int c = (int)((job >> 8) & 255u);
    const float2 kap = __ldg(S.b_kap + lds_s64(sIJ + 8u) * CPT + c);
    f2_t ax[R / 2], ay[R / 2], az[R / 2], a0[R / 2];
    float4 ca;
    job_points<NT, R, JU, HM>(job, sIJ, S, ca, ax, ay, az);
    const unsigned edge = (job >> 16) & 511u;
    float G, G2 = 0.f;
    const float mid = edge_mid(band, edge, G);
    {
        f2_t lx[R / 2], ly[R / 2], lz[R / 2];
        recentre<R>(ca, chunk_sphere(caps, c), ax, ay, az, lx, ly, lz);
        recentre<R>(ca, make_float4(0.f, 0.f, 0.f, 0.f), ax, ay, az, ax, ay, az);
        const float km = kap.x - mid;
        const f2_t km2 = pack2(km, km), half = pack2(0.5f, 0.5f);
#pragma unroll
        for (int q = 0; q < R / 2; ++q)
            a0[q] = mul2(half, fma2(lx[q], lx[q], fma2(ly[q], ly[q], fma2(lz[q], lz[q], km2))));
    }
    unsigned b = tile + (unsigned)c * kChunkB;
    const unsigned end = b + kChunk * kPointB, step = (unsigned)ts * (2 * kPointB);
    b += (unsigned)t0 * (2 * kPointB);
    neg1 = neg2 = 0;
    mb1 = mb2 = __int_as_float(0x7f800000);
    if (T == kJobOne) {
        unsigned negq[R / 2];
        float mbq[R / 2];
#pragma unroll
        for (int q = 0; q < R / 2; ++q) {
            negq[q] = 0;
            mbq[q] = __int_as_float(0x7f800000);
        }
#pragma unroll 1
        for (; b < end; b += step) one_edge_step<R>(b, ax, ay, az, a0, negq, mbq);
#pragma unroll
        for (int q = 0; q < R / 2; ++q) {
            neg1 += negq[q];
            mb1 = fminf(mb1, mbq[q]);
        }
    } else {
        const float mid2 = edge_mid(band, edge + 1u, G2);
        const float ndel = 0.5f * (mid - mid2);
#pragma unroll 1
        for (; b < end; b += step)
            two_edge_step<R>(b, ax, ay, az, a0, pack2(ndel, ndel), neg1, neg2, mb1, mb2);
        mb2 -= G2 + kap.y;
    }
    mb1 -= G + kap.y;
}

// Rare: a job found a value within the slack of edge k.  The warp counts the
// job's pairs below the edge again, one B point per lane, and settles each
// value within the slack by its FP64 squared chord.  Returns that count, with
// the number of values rechecked above bit 16.  Out of line: its FP64
// registers do not weigh on the loops.
template <int NT, int R>
__device__ __noinline__ unsigned recount_edge(unsigned job, unsigned k, unsigned sIJ, unsigned band,
                                              unsigned sC, const Segment& S) {
    constexpr int TA = NT * R, TB = NT * R, SA = 32 * R;
    const int lane = threadIdx.x & 31;
    const long long pa = lds_s64(sIJ) * TA + (int)((job >> 5) & 7u) * SA + (int)(job & 31u) * R;
    const long long pb = lds_s64(sIJ + 8u) * TB + (int)((job >> 8) & 255u) * kChunk + lane;
    const float4 ca = __ldg(S.a_caps + pa / kChunk), cb = __ldg(S.b_caps + pb / kChunk);
    const float2 kap = __ldg(S.b_kap + pb / kChunk);
    const float bx = -S.bl[pb], by = -S.bl[S.bl_stride + pb], bz = -S.bl[2 * S.bl_stride + pb];
    float G;
    const float mid = edge_mid(band, k, G);
    G += kap.y;
    const float km = kap.x - mid, dx = ca.x - cb.x, dy = ca.y - cb.y, dz = ca.z - cb.z;
    const double c = lds_f64(sC + 8u * k);
    unsigned n = 0;
#pragma unroll 1
    for (int r = 0; r < R; ++r) {
        const float ax = S.al[pa + r], ay = S.al[S.al_stride + pa + r],
                    az = S.al[2 * S.al_stride + pa + r];
        const float lx = __fadd_rn(ax, dx), ly = __fadd_rn(ay, dy), lz = __fadd_rn(az, dz);
        const float a0 = 0.5f * fmaf(lx, lx, fmaf(ly, ly, fmaf(lz, lz, km)));
        const float d = fmaf(__fadd_rn(ax, ca.x), bx,
                             fmaf(__fadd_rn(ay, ca.y), by, fmaf(__fadd_rn(az, ca.z), bz, a0)));
        if (fabsf(d) > G) {
            n += d < 0.f ? 1u : 0u;
        } else {
            n += (pair_chord2(S, pa + r, pb) < c ? 1u : 0u) + (1u << 16);
        }
    }
    return __reduce_add_sync(0xffffffffu, n);
}

// Adds a warp's count (lanes with flag set, times w) to a 64-bit shared
// counter at address a (statistics only).
__device__ __forceinline__ void warp_stat(unsigned a, bool flag, unsigned w) {
    const unsigned m = __ballot_sync(0xffffffffu, flag);
    if ((threadIdx.x & 31) == 0 && m)
        asm volatile("red.shared.add.u64 [%0], %1;" ::"r"(a),
                     "l"((unsigned long long)__popc(m) * w)
                     : "memory");
}

// One round of jobs of kind T: this lane's share of job `run` (active: the
// lane has one; ts = 2^lts adjacent lanes share a job, this one taking steps
// t0, t0 + ts, ...).  The first lane of each job moves the counts, summed
// over the ts lanes, below the job's edges.
template <int NT, int R, int JU, int HM, bool ST>
__device__ __forceinline__ void job_round(int T, unsigned run, bool active, int t0, int ts,
                                          unsigned sIJ, unsigned tile, unsigned lut, unsigned caps,
                                          unsigned band, unsigned sC, unsigned col,
                                          const PairParams& p, const Segment& S, bool stats,
                                          unsigned stat) {
    constexpr unsigned row_bytes = PairKernel<NT, R, JU, HM, 0>::ROWB;
    const int lane = threadIdx.x & 31;
    unsigned n_recheck = 0;
    if (T == kJobExact) {
        if (active)
            exact_job<NT, R, JU, HM>(run, t0, ts, sIJ, tile, lut, caps, sC, col, p, S, n_recheck);
    } else {
        unsigned neg1 = 0, neg2 = 0;
        float mb1 = __int_as_float(0x7f800000), mb2 = mb1;
        if (active)
            span_part<NT, R, JU, HM>(T, run, t0, ts, sIJ, tile, caps, band, S, neg1, neg2, mb1,
                                     mb2);
#pragma unroll 1
        for (int o = ts >> 1; o > 0; o >>= 1) {
            neg1 += __shfl_xor_sync(0xffffffffu, neg1, o);
            neg2 += __shfl_xor_sync(0xffffffffu, neg2, o);
            mb1 = fminf(mb1, __shfl_xor_sync(0xffffffffu, mb1, o));
            mb2 = fminf(mb2, __shfl_xor_sync(0xffffffffu, mb2, o));
        }
        const bool first = active && t0 == 0;
        const unsigned edge = (run >> 16) & 511u;
        // jobs with a value within the slack of their first or second edge
        unsigned b1 = __ballot_sync(0xffffffffu, first && !(mb1 > 0.f));
        unsigned b2 = __ballot_sync(0xffffffffu, first && !(mb2 > 0.f));
#pragma unroll 1
        while (b1 | b2) {
            const bool second = b1 == 0u;
            const int src = __ffs(second ? b2 : b1) - 1;
            if (second) b2 &= b2 - 1u; else b1 &= b1 - 1u;
            const unsigned j = __shfl_sync(0xffffffffu, run, src);
            const unsigned v = recount_edge<NT, R>(j, ((j >> 16) & 511u) + (second ? 1u : 0u),
                                                   sIJ, band, sC, S);
            if (lane == src) {
                if (second) neg2 = v & 0xFFFFu; else neg1 = v & 0xFFFFu;
                n_recheck += v >> 16;
            }
        }
        if (first) {
            const unsigned row = col + edge * row_bytes;
            hist_add<HM>(row, neg1);
            hist_add<HM>(row + row_bytes, neg2 - neg1);
            if (T == kJobTwo) hist_add<HM>(row + 2u * row_bytes, 0u - neg2);
        }
    }
    if (ST && stats) {
        if (__any_sync(0xffffffffu, n_recheck != 0)) {
            unsigned long long v = n_recheck;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0)
                asm volatile("red.shared.add.u64 [%0], %1;" ::"r"(stat), "l"(v) : "memory");
        }
    }
}

// log2 of the lanes per job for a round of m < 32 jobs: the largest power of
// two with m ts <= 32 (edge jobs: at most the chunk's 16 steps).
__device__ __forceinline__ int round_share(int T, int m) {
    const int l = __clz(m - 1) - 27;  // m in (2^(4-l), 2^(5-l)]
    return m == 1 ? (T == kJobExact ? 5 : 4) : l;
}

// Before an item's units: every sub-tile of A (32 R = 256 points, the sphere
// around its 8 chunks' spheres) against every chunk of B, one pair per lane.
// Where all 8192 pairs are in one slot, or beyond the top edge, they are
// counted here and the chunk drops out of the sub-tile's list (a word of chunk
// bits at todo + 4 sub), instead of 32 lanes finding that out one group each.
// Not in a diagonal tile pair.
template <int NT, int R, int JU, int HM, bool ST>
__device__ __forceinline__ void settle_chunks(unsigned todo, unsigned lut, unsigned sC, unsigned hist,
                                              const PairParams& p, const Segment& S, long long I,
                                              long long J, bool diag, int part, int lp,
                                              unsigned stat) {
    using PK = PairKernel<NT, R, JU, HM, 0>;
    constexpr int CPT = PK::TB / kChunk, SA = 32 * R;
    static_assert(SA / kChunk == 8 && CPT <= 32, "8 chunks a sub-tile, a word of chunk bits");
    const int lane = threadIdx.x & 31, sub = threadIdx.x >> 5;
    const float4 own = __ldg(S.a_caps + (I * PK::TA + sub * SA) / kChunk + (lane & 7));
    const float4 gb = __ldg(S.b_caps + J * CPT + min(lane, CPT - 1));
    float4 ga = own;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        ga.x += __shfl_xor_sync(0xffffffffu, ga.x, o);
        ga.y += __shfl_xor_sync(0xffffffffu, ga.y, o);
        ga.z += __shfl_xor_sync(0xffffffffu, ga.z, o);
    }
    ga.x *= 0.125f; ga.y *= 0.125f; ga.z *= 0.125f;
    const float dx = own.x - ga.x, dy = own.y - ga.y, dz = own.z - ga.z;
    // (the factor and the term cover the roundings of this arithmetic; a chunk
    // with padding or too wide a one leaves the sub-tile to its groups)
    ga.w = own.w >= 0.f && own.w <= 0.5f
               ? (sqrt_approx(dx * dx + dy * dy + dz * dz) + own.w) * (1.f + 4e-6f) + 2e-7f
               : 3.f;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) ga.w = fmaxf(ga.w, __shfl_xor_sync(0xffffffffu, ga.w, o));
    unsigned rlo = 0, rhi = 0;
    const int n = span_edges(ga, gb, lut, sC, p.tab.shift, p.tab.base, p.tab.n_lut - 1, p.tab.K,
                             p.tab.h_top, rlo, rhi);
    const bool here = lane < CPT && lane >= (part * CPT) >> lp && lane < ((part + 1) * CPT) >> lp;
    const bool settled = here && !diag && n == 0;
    hist_add<HM>(hist + 4u * (unsigned)PK::column() +
                     (settled ? rhi : (unsigned)p.tab.K + 1u) * PK::ROWB,
                 (unsigned)(SA * kChunk));
    const unsigned left = __ballot_sync(0xffffffffu, here && !settled);
    if (lane == 0) sts_u32(todo + 4u * (unsigned)sub, left);
    if (ST && p.stats != nullptr) {
        warp_stat(stat + 8u, settled, (unsigned)(SA * kChunk));
        warp_stat(stat + 16u, settled, (unsigned)(SA * kChunk));
    }
}

// A warp's share of one item with span binning: units of its own sub-tile
// first, then those left of the others (shared counters at address units, one
// per sub-tile).  Each lane classifies its group against every chunk of a
// unit that settle_chunks left; a chunk in one slot is counted at once, the others become jobs (the
// warp's rings in the block's ring array at shared address rings, kRing words
// per kind) and 32 jobs of a kind run as one round.  When every unit is taken,
// the jobs left in all the warps' rings are pooled and shared out evenly (a
// warp would otherwise run its own leftovers in partial rounds while the
// others wait at the next item's barrier), each job of a partial round shared
// among several lanes.
// In a diagonal tile pair of an auto count (pairs i < j) a group skips the
// chunks before its own and takes those after it like any other; its own
// chunk goes pair by pair with the i < j mask, every warp its own sub-tile.
// The tile pair (I, J) stays in shared memory (sIJ) and the statistics go to
// the block's shared counters (stat: rechecks, span pairs, skipped pairs), so
// that the rounds run with few live registers.  Every thread of the block
// calls this once per item (it holds block barriers).
template <int NT, int R, int JU, int HM, bool ST>
__device__ __forceinline__ void span_item(unsigned units, unsigned rings, unsigned sIJ,
                                          unsigned tile, unsigned lut, unsigned caps,
                                          unsigned groups, unsigned band, unsigned sC, unsigned hist,
                                          const PairParams& p, const Segment& S, bool diag,
                                          int part, int lp, unsigned stat) {
    using PK = PairKernel<NT, R, JU, HM, 0>;
    constexpr int TA = PK::TA, TB = PK::TB;
    constexpr int NW = NT / 32, SA = 32 * R, UPS = 8, UB = TB / UPS, CPU = UB / kChunk;
    constexpr unsigned row_bytes = PK::ROWB;
    constexpr unsigned NP = (unsigned)(R * kChunk);
    constexpr unsigned RING = 4u * kRing, RINGS = RING * kJobKinds;  // bytes: a ring, a warp's
    constexpr unsigned FULL = 0x202020u;  // some fill (8 bits per kind) is 32 or more
    static_assert(R == 8, "groups of write_chunk");
    static_assert(NW <= 8 && TB / kChunk <= 32 && UB % kChunk == 0 && CPU <= 8 && kChunk % JU == 0 &&
                      (NW > 1 || TB / kChunk <= 8),
                  "job fields, a unit's chunk bits");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned ring = rings + RINGS * (unsigned)warp;
    const unsigned col = hist + 4u * (unsigned)PK::column();
    const bool stats = ST && p.stats != nullptr;
    // the part's chunks
    const int c_begin = (part * (TB / kChunk)) >> lp, c_end = ((part + 1) * (TB / kChunk)) >> lp;
    unsigned fills = 0;   // jobs waiting per kind, 8 bits each; bit 24 + T: ring T starts at 32
    unsigned word = 0;    // this lane's next job (of the chunk it has classified)
    // the current unit: its first chunk, bits of the chunks left, its sub-tile,
    // sub-tiles done (from bits 0, 8, 16, 20): one register across the rounds
    unsigned at_unit = 0;
    int pool = -1;        // kind of the pooled leftovers being run
#pragma unroll 1
    for (;;) {
        int T, m = 32, lts = 0;
        unsigned at = 0;  // shared address of this lane's job
        if (pool < 0 && (fills & FULL) == 0u) {
            if (!__any_sync(0xffffffffu, (word >> 25) != 0u)) {
                // the next chunk
#pragma unroll 1
                while ((at_unit & 0xFF00u) == 0u && (at_unit >> 20) < (unsigned)NW) {
                    const unsigned k = at_unit >> 20, sub = ((unsigned)warp + k) & (NW - 1);
                    unsigned u = 0;
                    if (lane == 0) u = atom_add_shared(units + 4u * sub, 1u);
                    u = __shfl_sync(0xffffffffu, u, 0);
                    // (a one-warp block takes its part of the tile as one unit)
                    const int cn = NW == 1 ? c_begin : (int)u * CPU;
                    const int ce = NW == 1 ? c_end : cn + CPU;
                    if (NW == 1 ? u != 0u : cn >= c_end) {
                        at_unit = (k + 1u) << 20;
                        continue;
                    }
                    // (in a diagonal tile pair: every pair of the unit has i >= j)
                    if (diag && ce * kChunk <= (int)sub * SA) continue;
                    const unsigned bits = (lds_u32(units + 4u * (unsigned)NW + 4u * sub) >> cn) &
                                          ((1u << (ce - cn)) - 1u);
                    at_unit = (unsigned)cn | (bits << 8) | (sub << 16) | (k << 20);
                }
                if ((at_unit >> 20) == (unsigned)NW) {
                    pool = 0;  // every unit taken: the leftovers
                    __syncthreads();  // the rings are quiescent
                    if (lane == 0) sts_u32(units + 4u * (unsigned)warp, fills);
                    __syncthreads();
                    continue;
                }
                const unsigned bit = at_unit & 0xFF00u & (0u - (at_unit & 0xFF00u));
                const int c = (int)(at_unit & 255u) + 23 - __clz(bit), sub = (int)((at_unit >> 16) & 7u);
                at_unit ^= bit;
                unsigned rlo = 0, rhi = 0;
                const int n = span_edges(chunk_sphere(groups, sub * 32 + lane), chunk_sphere(caps, c),
                                         lut, sC, p.tab.shift, p.tab.base, p.tab.n_lut - 1, p.tab.K,
                                         p.tab.h_top, rlo, rhi);
                const int own = diag ? (sub * SA + lane * R) / kChunk : -1;
                const bool mine = c > own;
                // (to the trash row if nothing is settled: no branch)
                hist_add<HM>(col + (mine && n >= 0 ? rhi : (unsigned)p.tab.K + 1u) * row_bytes, NP);
                word = job_word(lane, sub, c, rlo) |
                       ((!mine ? 0u : n < 0 ? kExact : (unsigned)n) << 25);
                if (stats) {
                    warp_stat(stat + 8u, mine && n >= 0, NP);
                    warp_stat(stat + 16u, mine ? n == 0 : c < own, NP);
                }
            }
            // push one job of every lane that has some left: the odd edge alone,
            // then the others by twos
            const unsigned left = word >> 25;
            const bool one = (left & 1u) != 0u, exact = left == kExact;
            const unsigned m1 = __ballot_sync(0xffffffffu, one);
            const unsigned m3 = __ballot_sync(0xffffffffu, exact);
            const unsigned m2 = __ballot_sync(0xffffffffu, left != 0u) & ~(m1 | m3);
            const int Tp = one ? kJobOne : exact ? kJobExact : kJobTwo;
            const unsigned mk = one ? m1 : exact ? m3 : m2;
            const unsigned pos = (fills >> (8 * Tp)) + ((fills >> (24 + Tp)) << 5) +
                                 (unsigned)__popc(mk & ((1u << lane) - 1u));
            sts_u32_if(left != 0u, ring + RING * (unsigned)Tp + ((4u * pos) & (RING - 4u)),
                       word & kJobBits);
            const unsigned by = left == 0u ? 0u : one ? 1u : 2u;
            word += exact ? 0u - (kExact << 25) : (by << 16) - (by << 25);
            fills += (unsigned)__popc(m1) + ((unsigned)__popc(m2) << 8) + ((unsigned)__popc(m3) << 16);
            if ((fills & FULL) == 0u) continue;
        }
        if (pool < 0) {
            // a full round of the first kind that has one
            T = (fills & 0x20u) ? kJobOne : (fills & 0x2000u) ? kJobTwo : kJobExact;
            at = ring + RING * (unsigned)T +
                 4u * ((((fills >> (24 + T)) & 1u) * 32u + (unsigned)lane));
            fills = (fills - (32u << (8 * T))) ^ (1u << (24 + T));
        } else {
            // The leftovers of every warp, pooled: each warp published its fills
            // in its unit counter (no longer claimed), and the jobs of each
            // kind, the rings taken in warp order, are shared out in contiguous
            // slices of about n / NW jobs, each slice one round with the lanes
            // of a job adjacent.
            if (pool == kJobKinds) break;
            T = pool++;
            int n = 0;
#pragma unroll
            for (int q = 0; q < NW; ++q) n += (int)((lds_u32(units + 4u * (unsigned)q) >> (8 * T)) & 255u);
            const int lo = warp * n / NW;
            m = (warp + 1) * n / NW - lo;
            if (m == 0) continue;
            lts = round_share(T, m);
            // job lo + lane / ts of the pool: position i of warp q's ring
            int i = lo + min(lane >> lts, m - 1), q = 0;
            unsigned f = lds_u32(units);
#pragma unroll
            for (int w = 0; w < NW - 1; ++w) {
                const int fw = (int)((f >> (8 * T)) & 255u);
                if (q == w && i >= fw) {
                    i -= fw;
                    ++q;
                    f = lds_u32(units + 4u * (unsigned)q);
                }
            }
            at = rings + RINGS * (unsigned)q + RING * (unsigned)T +
                 4u * (((((f >> (24 + T)) & 1u) * 32u) + (unsigned)i) & (kRing - 1));
        }
        __syncwarp();
        const unsigned run = lds_u32(at);
        __syncwarp();
        job_round<NT, R, JU, HM, ST>(T, run, (lane >> lts) < m, lane & ((1 << lts) - 1), 1 << lts,
                                     sIJ, tile, lut, caps, band, sC, col, p, S, stats, stat);
    }
    if (diag) {
        // every group of the warp's sub-tile against its own chunk, pair by pair,
        // i < j: the groups whose chunk is in this part (4 per chunk), each
        // shared among 32 / m lanes
        constexpr int GPC = kChunk / R, CPS = SA / kChunk;
        const int g0 = max(c_begin, warp * CPS) * GPC;
        const int m = min(c_end, (warp + 1) * CPS) * GPC - g0;  // a power of two, or none
        if (m > 0) {
            const int lts = 5 - (31 - __clz(m));
            const int a_first = (g0 + (lane >> lts)) * R, c = a_first / kChunk;
            const long long a0 = lds_s64(sIJ) * TA + a_first;
            const long long b0 = lds_s64(sIJ + 8u) * TB + c * kChunk;
            f2_t ax[R / 2], ay[R / 2], az[R / 2];
            load_local<R>(S.al, S.al_stride, a0, ax, ay, az);
            recentre<R>(__ldg(S.a_caps + a0 / kChunk), chunk_sphere(caps, c), ax, ay, az, ax, ay, az);
            unsigned nr = 0;
            exact_chunk<NT, R, HM, row_bytes, true>(tile, c, lane & ((1 << lts) - 1), 1 << lts, lut,
                                                    sC, col, ax, ay, az, p, S, a0, b0, a_first, nr);
            if (stats) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) nr += __shfl_xor_sync(0xffffffffu, nr, o);
                if (lane == 0 && nr)
                    asm volatile("red.shared.add.u64 [%0], %1;" ::"r"(stat),
                                 "l"((unsigned long long)nr) : "memory");
            }
        }
    }
    __syncwarp();
}

// The overflow slots of a launch's counts, total minus the other slots, one warp
// per count: by the last block to finish, after all others' counts.  Out of
// line, as its registers would weigh on the kernel's.
__device__ __noinline__ void fill_overflow(const PairParams& p) {
    __threadfence();
    const int K = p.tab.K;
    for (int q = threadIdx.x >> 5; q < max(p.n_segs, 1); q += blockDim.x >> 5) {
        const Segment& g = p.n_segs > 0 ? p.segs[q] : p.seg0;
        unsigned long long sum = 0;
        for (int k = threadIdx.x & 31; k <= K; k += 32) sum += __ldcg(g.counts + k);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if ((threadIdx.x & 31) == 0) g.counts[K + 1] = g.total - sum;
    }
}

// ST: with the span path's statistics code (a launch with p.stats set); the
// build without it is the one launched when no statistics are asked for.
// Registers: 96 at 8 A points a thread (20 warps an SM), 168 at 16 (12 warps; left to
// itself the compiler took 174, one block less: 16 points, deferred, 200k + 200k
// survey points 17.9 ms against 14.7).
template <int NT, int R, int JU, int HM, int DEF, bool ST>
__global__ void __launch_bounds__(NT, (R == 8 ? 640 : 384) / NT) k_pairs(const __grid_constant__ PairParams p) {
    using PK = PairKernel<NT, R, JU, HM, DEF>;
    constexpr int TA = PK::TA, TB = PK::TB, HCOLS = PK::HCOLS, HSTRIDE = PK::HSTRIDE;
    constexpr int NW = NT / 32, SA = 32 * R, UPS = 8, UB = TB / UPS;
    static_assert(TA == NW * SA && TB % UPS == 0, "units tile the item");
    __shared__ unsigned s_units[2 * NW];  // units taken; chunks left per sub-tile (spans)
    // span job rings (one per kind and warp) for the shapes that bin spans
    __shared__ unsigned s_ring[PK::SPANS ? NW * kJobKinds * kRing : 1];
    extern __shared__ __align__(16) unsigned char smem[];
    const int K = p.tab.K;
    // (the spheres and edge middles only where there are span jobs)
    float4* sCap = reinterpret_cast<float4*>(smem + PK::TILEB);
    float4* sGroup = sCap + (PK::SPANS ? TB / 32 : 0);  // spheres of A's groups
    unsigned char* sLut = reinterpret_cast<unsigned char*>(sGroup + (PK::SPANS ? TA / 8 : 0));
    double* sC = reinterpret_cast<double*>(sLut + PK::LUTB * (unsigned)p.tab.n_lut);
    float2* sBand = reinterpret_cast<float2*>(sC + (K + 2));
    unsigned* hist = reinterpret_cast<unsigned*>(sBand + (PK::SPANS ? K + 2 : 0));
    // the item and its tile pair (I, J), in two buffers by the parity of the
    // block's item count: thread 0 writes the next item's while other warps may
    // still be in the current one
    __shared__ long long s_item[2], s_IJ[2][2];
    __shared__ int s_part[2], s_seg[2];
    __shared__ unsigned long long s_stat[3];  // span-path rechecks, span pairs, skipped pairs

    const int tid = threadIdx.x;
    // the parameter block through its generic address: lanes that index the
    // constant bank each at their own place are served one by one
    const PairParams* gp = &p;
    asm volatile("" : "+l"(gp));
    for (int q = tid; q < p.tab.n_lut; q += NT) {
        const unsigned x = gp->tab.lut[q][0], y = gp->tab.lut[q][1];
        if constexpr (PK::LUTB == 8) reinterpret_cast<uint2*>(sLut)[q] = make_uint2(x, y);
        else reinterpret_cast<uint4*>(sLut)[q] = lut_wide<PK::ROWB>(x, y, K);
    }
    for (int q = tid; q <= K; q += NT) {
        sC[q] = gp->tab.c64[q];
        if constexpr (PK::SPANS) sBand[q] = make_float2(gp->tab.edge[q][0], gp->tab.edge[q][1]);
    }
    for (int q = tid; q < (K + 2) * HSTRIDE; q += NT) hist[q] = 0u;
    if (tid < 3) s_stat[tid] = 0ull;

    // the current count lives in shared memory; thread 0 switches it when an
    // item of another count is claimed, after the block flushed its columns
    __shared__ Segment sSeg;
    // items of this launch: p.n_items, or fewer when a device-side pass kept
    // only some of them (tile pairs wholly beyond the top edge are skipped)
    // Few items are taken in 2^lp parts of the B tile each: without that a small
    // count is as long as one tile pair takes one block, on a chip mostly idle.
    const long long n_tile_pairs =
        p.n_items_dev ? min(p.n_items, (long long)*p.n_items_dev) : p.n_items;
    int lp = 0;
    while (lp < PK::MAXLP && (n_tile_pairs << lp) < (long long)kPartWaves * gridDim.x) ++lp;
    const long long n_launch = n_tile_pairs << lp, n_end = p.n_items << lp;
    unsigned long long n_recheck = 0;
    unsigned n_items = 0, n_tiles = 0;
    int since_flush = 0, cur_seg = -2;
    // Claims an item into buffer w (one thread: an atomic, the item's count and
    // its tile pair).  (Claimed while the block still works on the item before,
    // a claim's latency went but blocks sat on claimed items at the tail: survey
    // 32.4 -> 32.3 ms, 30k x 48k 424 -> 429 us.)
    auto claim = [&](int w) {
        const long long tp = (long long)atomicAdd(p.cursor, 1ull), t = tp >> lp;
        s_item[w] = tp < n_launch ? tp : n_end;
        s_part[w] = (int)(tp & ((1 << lp) - 1));
        if (tp >= n_launch) return;
        int seg = -1;
        if (p.n_segs > 0) {
            const long long g = p.item_begin + t;
            int lo = 0, hi = p.n_segs - 1;  // last segment with item_begin <= g
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (p.segs[mid].item_begin <= g) lo = mid; else hi = mid - 1;
            }
            seg = lo;
        }
        s_seg[w] = seg;
        // tile pair of the item
        const Segment* G = seg < 0 ? &p.seg0 : p.segs + seg;
        long long local = p.item_begin + t - G->item_begin + G->item_offset;
        if (G->item_list) local = G->item_list[local];
        long long I, J;
        item_to_tiles(local, G->tiles_a, G->tiles_b, G->is_auto, &I, &J);
        s_IJ[w][0] = I;
        s_IJ[w][1] = J;
    };
    for (;;) {
        if (tid == 0) claim(n_items & 1);
        __syncthreads();  // the claim visible; previous item's shared reads finished
        if (s_item[n_items & 1] >= n_end) break;
        const int seg = s_seg[n_items & 1];
        if (seg != cur_seg) {
            if (cur_seg != -2 && since_flush > 0) {
                flush_hist<NT, HCOLS, HSTRIDE>(hist, K, sSeg.counts);
                since_flush = 0;
            }
            __syncthreads();  // flush done before the segment is replaced
            if (tid == 0) sSeg = seg < 0 ? p.seg0 : p.segs[seg];
            cur_seg = seg;
            __syncthreads();
        }
        const Segment& S = sSeg;
        const long long I = s_IJ[n_items & 1][0], J = s_IJ[n_items & 1][1];
        // the part of the B tile that this item takes
        const int part = s_part[n_items & 1], b_len = TB >> lp, b_begin = part * b_len;
        n_tiles += part == 0 ? 1 : 0;
        // with span jobs the tile holds local coordinates (relative to each chunk's
        // centre), otherwise the FP32 copies
        const unsigned a_tile = smem_addr(smem);
        // two points at a time: three 16-byte stores
        auto stage2 = [&](int j, float x0, float y0, float z0, float x1, float y1, float z1) {
            const unsigned b = point_addr<PK::SPANS>(a_tile, j);
            sts_f2x2(b, pack2(-x0, -x0), pack2(-y0, -y0));
            sts_f2x2(b + 16u, pack2(-z0, -z0), pack2(-x1, -x1));
            sts_f2x2(b + 32u, pack2(-y1, -y1), pack2(-z1, -z1));
        };
        if constexpr (PK::SPANS) {
            const float* gL = S.bl + J * TB;
            const long long ls = S.bl_stride;
#pragma unroll 4
            for (int j = b_begin + 2 * tid; j < b_begin + b_len; j += 2 * NT) {
                const float2 x = *reinterpret_cast<const float2*>(gL + j);
                const float2 y = *reinterpret_cast<const float2*>(gL + ls + j);
                const float2 z = *reinterpret_cast<const float2*>(gL + 2 * ls + j);
                stage2(j, x.x, y.x, z.x, x.y, y.y, z.y);
            }
            for (int q = tid; q < TB / 32; q += NT) sCap[q] = S.b_caps[J * (TB / 32) + q];
            for (int q = tid; q < TA / 8; q += NT) sGroup[q] = S.a_groups[I * (TA / 8) + q];
        } else {
            const float4* gB = S.b32 + J * TB;
#pragma unroll 4
            for (int j = b_begin + 2 * tid; j < b_begin + b_len; j += 2 * NT) {
                const float4 a = gB[j], b = gB[j + 1];
                stage2(j, a.x, a.y, a.z, b.x, b.y, b.z);
            }
        }
        if (tid < NW) s_units[tid] = NW == 1 ? 0 : (part * UPS) >> lp;
        if constexpr (PK::SPANS)
            settle_chunks<NT, R, JU, HM, ST>(smem_addr(s_units + NW), smem_addr(sLut), smem_addr(sC),
                                             smem_addr(hist), p, S, I, J, S.is_auto && I == J, part,
                                             lp, smem_addr(s_stat));
        __syncthreads();  // B tile staged, unit counters reset
        const unsigned a_lut = smem_addr(sLut), a_cap = smem_addr(sCap), a_group = smem_addr(sGroup), a_band = smem_addr(sBand),
                       a_hist = smem_addr(hist), a_c = smem_addr(sC);
        // The item is split into units of one warp's worth of A points (SA =
        // 32 R consecutive points, a sub-tile) by an eighth of the B tile (the
        // warps of a block end an item within less of one another than with
        // quarters: survey 33.3 -> 32.9 ms, 200k + 200k binned after screening
        // 15.3 -> 12.3 ms).  A warp takes the units of its own sub-tile first, then
        // those left of the others, so the warps of the block finish the item
        // together whatever the mix of cheap and costly units.
        const bool diag = S.is_auto && I == J;
        if constexpr (PK::SPANS) {
            span_item<NT, R, JU, HM, ST>(smem_addr(s_units), smem_addr(s_ring),
                                         smem_addr(s_IJ[n_items & 1]), a_tile, a_lut, a_cap, a_group,
                                         a_band, a_c, a_hist, p, S, diag, part, lp, smem_addr(s_stat));
        } else {
            const int lane = tid & 31, warp = tid >> 5;
            int cur = -1;
            f2_t ax[R / 2], ay[R / 2], az[R / 2];
#pragma unroll 1
            for (int k = 0; k < NW; ++k) {
                const int sub = (warp + k) % NW;
#pragma unroll 1
                for (;;) {
                    unsigned u = 0;
                    if (lane == 0) u = atomicAdd(&s_units[sub], 1u);
                    u = __shfl_sync(0xffffffffu, u, 0);
                    // (one-warp blocks: the part of the tile as one unit)
                    const int jb = NW == 1 ? b_begin : (int)u * UB;
                    const int je = NW == 1 ? b_begin + b_len : jb + UB;
                    if (NW == 1 ? u != 0u : jb >= b_begin + b_len) break;
                    const int a_first = sub * SA + lane * R;
                    if (diag && je <= sub * SA) continue;  // every pair has i >= j
                    if (sub != cur) {
                        load_group<R>(S.a32 + I * TA + a_first, ax, ay, az);
                        cur = sub;
                    }
                    if (diag && jb < (sub + 1) * SA)
                        tile_pass<NT, R, JU, HM, DEF, true>(a_tile, a_lut, a_c, a_hist, ax, ay, az, p,
                                                            S, I, J, a_first, jb, je, n_recheck);
                    else
                        tile_pass<NT, R, JU, HM, DEF, false>(a_tile, a_lut, a_c, a_hist, ax, ay, az, p,
                                                             S, I, J, a_first, jb, je, n_recheck);
                }
            }
        }
        ++n_items;
        if (++since_flush == p.items_per_flush) {
            __syncthreads();
            flush_hist<NT, HCOLS, HSTRIDE>(hist, K, sSeg.counts);
            __syncthreads();
            since_flush = 0;
        }
    }
    // all threads left the loop after the same barrier
    if (cur_seg != -2) flush_hist<NT, HCOLS, HSTRIDE>(hist, K, sSeg.counts);
    if (p.done) {
        __threadfence();  // this block's counts before its mark
        __syncthreads();
        if (tid == 0) s_part[0] = atomicAdd(p.done, 1ull) + 1ull == gridDim.x ? 1 : 0;
        __syncthreads();
        if (s_part[0]) fill_overflow(p);
    }
    if (p.stats) {
        unsigned long long v = n_recheck;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((tid & 31) == 0 && v) atomicAdd(p.stats + WTHETA_STAT_RECHECK, v);
        if (tid == 0) {
            // the span path's counts (the loop's last barrier ordered them)
            if (s_stat[0]) atomicAdd(p.stats + WTHETA_STAT_RECHECK, s_stat[0]);
            if (s_stat[1]) atomicAdd(p.stats + WTHETA_STAT_SPAN, s_stat[1]);
            // pairs of chunks settled in one slot were never computed
            if (s_stat[2]) atomicAdd(p.stats + WTHETA_STAT_PAIRS, 0ull - s_stat[2]);
        }
        if (tid == 0 && n_items) {
            if (n_tiles) atomicAdd(p.stats + WTHETA_STAT_TILES, (unsigned long long)n_tiles);
            atomicAdd(p.stats + WTHETA_STAT_PAIRS, n_items * (unsigned long long)(TA * TB >> lp));
        }
    }
}

// The device tables of a w(theta) launch (its counts' segments and culling
// table), written by one small kernel from its parameters before anything else
// of the count; it also zeroes what the later kernels add to (counts, launch
// cursor, kept counters, the digit counts of a small sort), one launch instead
// of a copy from pageable memory and three memsets.
struct CountTables {
    Segment segs[3];
    CullSeg cs[3];
    int n_segs;
    int with_cull;
    unsigned* zero[4];   // words to zero
    long long n_zero[4];
};
__global__ void __launch_bounds__(256) k_begin_count(const __grid_constant__ CountTables t,
                                                     Segment* __restrict__ segs,
                                                     CullSeg* __restrict__ cs) {
    const long long i = blockIdx.x * 256LL + threadIdx.x;
    if (i < t.n_segs) {
        segs[i] = t.segs[i];
        if (t.with_cull) cs[i] = t.cs[i];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
        for (long long j = i; j < t.n_zero[q]; j += 256LL * gridDim.x) t.zero[q][j] = 0u;
}
static int launch_begin_count(const CountTables& t, Segment* segs, CullSeg* cs, cudaStream_t st) {
    long long n = 1;
    for (int q = 0; q < 4; ++q) n = std::max(n, t.n_zero[q]);
    const unsigned g = (unsigned)std::min<long long>((n + 255) / 256, 128);
    k_begin_count<<<g, 256, 0, st>>>(t, segs, cs);
    count_launch();
    return check_cuda(cudaGetLastError());
}

// counts[K+1] = total - sum(counts[0..K]) for every count of a batch.
__global__ void k_finalize_segments(const Segment* __restrict__ segs, int n_segs, int K) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_segs; i += gridDim.x * blockDim.x) {
        unsigned long long* c = segs[i].counts;
        unsigned long long s = 0;
        for (int k = 0; k <= K; ++k) s += c[k];
        c[K + 1] = segs[i].total - s;
    }
}

// ---------------------------------------------------------------------------
// launch plumbing
// ---------------------------------------------------------------------------
template <int NT, int R, int JU, int HM, int DEF>
static Variant make_variant() {
    constexpr bool spans = PairKernel<NT, R, JU, HM, DEF>::SPANS;  // only the span path has ST code
    return Variant{NT, R, JU, HM, DEF, PairKernel<NT, R, JU, HM, DEF>::MAXLP, &k_pairs<NT, R, JU, HM, DEF, true>,
                   spans ? &k_pairs<NT, R, JU, HM, DEF, false> : &k_pairs<NT, R, JU, HM, DEF, true>,
                   &PairKernel<NT, R, JU, HM, DEF>::smem_bytes};
}

// The build of v's kernel for a launch with these parameters.
static void (*pair_kernel(const Variant* v, const PairParams& prm))(PairParams) {
    return prm.stats ? v->kernel : v->kernel_fast;
}

constexpr int kMaxVariants = 32;

// Instantiated shapes (tile = threads x points_per_thread).  Per-warp
// histograms (mode 2) need the whole warp in step, so they bin inline.
const Variant* variants(int* n) {
    static const Variant v[] = {
        make_variant<128, 8, 2, kHistLaneAtomic, 0>(), make_variant<128, 8, 2, kHistLaneAtomic, 1>(),
        make_variant<128, 8, 2, kHistLane, 1>(),       make_variant<128, 8, 2, kHistWarp, 0>(),
        make_variant<128, 8, 1, kHistLaneAtomic, 1>(), make_variant<64, 16, 2, kHistLaneAtomic, 1>(),
        make_variant<64, 16, 2, kHistWarp, 0>(),       make_variant<128, 16, 2, kHistLaneAtomic, 1>(),
        make_variant<256, 8, 2, kHistLaneAtomic, 1>(), make_variant<256, 8, 2, kHistWarp, 0>(),
        make_variant<64, 8, 2, kHistLaneAtomic, 0>(),  make_variant<128, 8, 2, kHistWarpRed, 0>(),
        make_variant<64, 8, 2, kHistWarpRed, 0>(),     make_variant<32, 8, 2, kHistLaneAtomic, 0>(),
        make_variant<128, 8, 2, kHistLaneAtomic, 2>(), make_variant<64, 8, 2, kHistLaneAtomic, 2>(),
        make_variant<32, 8, 2, kHistLaneAtomic, 2>(), make_variant<128, 8, 2, kHistWarpRed, 2>(),
        make_variant<64, 8, 2, kHistWarpRed, 2>(),
    };
    static_assert(sizeof(v) / sizeof(v[0]) <= kMaxVariants, "grid_for's table");
    *n = (int)(sizeof(v) / sizeof(v[0]));
    return v;
}

int device_info(DeviceInfo* out) {
    static std::mutex mu;
    static DeviceInfo cache[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return WTHETA_ECUDA;
    std::lock_guard<std::mutex> g(mu);
    if (cache[dev].sm_count == 0) {
        if (cudaDeviceGetAttribute(&cache[dev].sm_count, cudaDevAttrMultiProcessorCount, dev) !=
                cudaSuccess ||
            cudaDeviceGetAttribute(&cache[dev].max_smem_optin,
                                   cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
            return WTHETA_ECUDA;
        // keep freed scratch in this process's stream-ordered pool between calls
        cudaMemPool_t pool;
        if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
            unsigned long long keep = ~0ull;
            cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
        }
    }
    *out = cache[dev];
    return WTHETA_OK;
}

// The default shape for one call by the larger catalogue's size: tiles of 256
// points (one warp) up to 4096, of 512 points (64 threads) up to 32768, else of
// 1024.  w(theta) of n + n points on a 10 deg patch (16 bins) / a 15 deg patch (24) /
// a 60 deg cap (32), with 32, 64, 128 threads, us per call on the device:
//    1k  101 107 125 / 106 111 125 /  99 105 122
//    4k  112 118 136 / 118 119 136 / 109 121 129
//    8k  143 142 146 / 158 151 164 / 135 133 140
//   16k  241 230 234 / 272 265 271 / 200 198 204
//   32k  421 441 457 / 531 541 575 / 304 326 357
//   48k  686 694 700 / 899 892 898 / 454 473 492
//   64k  979 970 981 / 1319 1288 1300 / 603 605 641
// and cross counts n x n: 4k 99 112 129 / 104 109 129 / 98 103 125, 32k 284 306 305 /
// 355 359 350 / 213 226 244, 48k 460 483 474 / 571 597 577 / 315 330 343.  The lines
// were drawn with 32 and 64 threads level from 5k on and 64 ahead of 128 up to 32k
// (32k 455 461 486 on the 10 deg patch); since the span builds spill nothing, 32
// threads are ahead by up to 7% at 32k and level or ahead to 64k.
const Variant* pick_for_size(const wtheta_tune* tune, long long n_max, int K, int n_lut,
                             int max_smem) {
    if (!tune && n_max <= 32768) {
        wtheta_tune small = {};
        small.threads = n_max <= 4096 ? 32 : 64;
        small.points_per_thread = 8;
        const Variant* v = pick_variant(&small, K, n_lut, max_smem);
        if (v) return v;
    }
    return pick_variant(tune, K, n_lut, max_smem);
}

const Variant* pick_variant(const wtheta_tune* tune, int K, int n_lut, int max_smem) {
    int nv = 0;
    const Variant* v = variants(&nv);
    const int want_nt = tune && tune->threads ? tune->threads : 128;
    const int want_r = tune && tune->points_per_thread ? tune->points_per_thread : 8;
    const int want_ju = tune && tune->j_per_screen ? tune->j_per_screen : 2;
    int want_hm = tune && tune->hist_mode ? tune->hist_mode : 0;
    int want_def = tune && tune->deferred ? (tune->deferred == 2 ? 1 : 0) : -1;
    auto fits = [&](const Variant& x) { return x.smem(K, n_lut) <= (size_t)max_smem; };
    auto shape = [&](const Variant& x) {
        return x.nt == want_nt && x.r == want_r && x.ju == want_ju;
    };
    auto find = [&](int hm, int def) -> const Variant* {
        for (int i = 0; i < nv; ++i)
            if (shape(v[i]) && v[i].hm == hm && v[i].def == def && fits(v[i])) return &v[i];
        return nullptr;
    };
    // every pair through the table (span binning off): the builds without span
    // code, with a column per thread (four per warp contend: 100k x 100k points, 16
    // bins, hist_mode 3: 4.53 ms against 4.46) or per warp
    const bool no_spans = tune && tune->span_bins == 2;
    if (no_spans && want_def != 1) {
        const Variant* x = find(want_hm == 0 ? (int)kHistLaneAtomic : want_hm, 2);
        if (x && (want_hm != 0 || x->smem(K, n_lut) <= 100 * 1024)) return x;
        x = want_hm == 0 ? find(kHistWarpRed, 2) : nullptr;
        if (x) return x;
    }
    if (want_hm == 0) {
        want_hm = find(kHistWarpRed, 0) ? kHistWarpRed : kHistWarp;
        for (int i = 0; i < nv; ++i)
            if (shape(v[i]) && v[i].hm == kHistLaneAtomic && v[i].def != 2 &&
                v[i].smem(K, n_lut) <= 100 * 1024)
                want_hm = kHistLaneAtomic;
        // four columns per warp while five blocks of 128 threads fit an SM; one
        // column per warp beyond (200k + 200k points, 256 bins: 9.2 ms against
        // 9.9 ms)
        const Variant* four = find(kHistLaneAtomic, 0);
        if (want_def != 1 && four && find(kHistWarpRed, 0) &&
            four->smem(K, n_lut) > (size_t)44 * 1024 * (size_t)want_nt / 128)
            want_hm = kHistWarpRed;
    }
    if (want_def < 0) want_def = 0;  // inline binning measured faster once in-range pairs matter
    for (int i = 0; i < nv; ++i)
        if (shape(v[i]) && v[i].hm == want_hm && v[i].def == want_def && fits(v[i])) return &v[i];
    // fall back: same tile size, per-warp histograms (shared atomics first)
    for (int hm : {(int)kHistWarpRed, (int)kHistWarp})
        for (int i = 0; i < nv; ++i)
            if (v[i].nt * v[i].r == want_nt * want_r && v[i].hm == hm &&
                v[i].def == (no_spans && hm == kHistWarpRed ? 2 : 0) && fits(v[i]))
                return &v[i];
    return nullptr;
}

int grid_for(const Variant* v, size_t smem, long long n_items, int sm_count, int want_per_sm,
                    int* grid) {
    // The limit of a kernel's dynamic shared memory only rises: a server, a plan or
    // another thread may launch the same kernel with the size it asked for before.
    static std::mutex mu;
    static size_t most[64][kMaxVariants];
    int dev = 0, nv = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return WTHETA_ECUDA;
    {
        std::lock_guard<std::mutex> g(mu);
        size_t& kept = most[dev][v - variants(&nv)];
        const size_t limit = std::max(kept, smem);
        if (cudaFuncSetAttribute((const void*)v->kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)limit) != cudaSuccess ||
            cudaFuncSetAttribute((const void*)v->kernel_fast,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)limit) != cudaSuccess)
            return WTHETA_ECUDA;
        kept = limit;
    }
    int per_sm = 0;
    int per_sm_fast = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void*)v->kernel, v->nt,
                                                      smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_fast, (const void*)v->kernel_fast,
                                                      v->nt, smem) != cudaSuccess)
        return WTHETA_ECUDA;
    per_sm = std::min(per_sm, per_sm_fast);  // one grid size for both builds
    per_sm = std::max(per_sm, 1);
    if (want_per_sm > 0) per_sm = std::min(per_sm, want_per_sm);
    long long g = (long long)per_sm * sm_count;
    // (a small count's items are taken in up to 2^max_parts parts)
    g = std::min(g, n_items << v->max_parts);
    *grid = (int)std::max(g, 1LL);
    return WTHETA_OK;
}

long long round_up(long long x, long long m) { return (x + m - 1) / m * m; }

int check_cuda(cudaError_t e) {
    if (e == cudaSuccess) return WTHETA_OK;
    if (e == cudaErrorMemoryAllocation) return WTHETA_ENOMEM;
    return WTHETA_ECUDA;
}

static int launch_grid(long long n, int sm_count) {
    const long long g = (n + 255) / 256;
    return (int)std::min<long long>(std::max<long long>(g, 1), (long long)sm_count * 16);
}

static long long sort_blocks(long long n) {
    const long long tile = (long long)kSortThreads * sort_rounds(n);
    return std::max<long long>(1, (n + tile - 1) / tile);
}

// Blocks of one launch per pass for a sort of n keys.
static long long small_blocks(long long n) { return (n + kSmallThreads - 1) / kSmallThreads; }

size_t order_bytes(long long n, int with_labels) {
    const size_t a4 = ((size_t)n * 4 + 255) / 256 * 256;
    // digit counts per block: of one pass, or of the four of a small sort
    long long rows = sort_blocks(n);
    if (n <= kSmallSort) rows = std::max(rows, 4 * small_blocks(n));
    return (4 + (with_labels ? 1 : 0)) * a4 +        // keys, indices (x2), labels
           ((size_t)rows * 256 * 4 + 255) / 256 * 256 +  // digit counts
           256 * 4;                                  // digit totals
}

// The buffers of a sort's scratch (order_bytes(n, with_labels) bytes): keys
// and indices twice (passes alternate), labels, per-block digit counts and
// the digit totals.
struct SortBufs {
    unsigned* key[2];
    unsigned* idx[2];
    unsigned* lab;
    unsigned* hist;
    unsigned* tot;
    long long G;
    int rounds;
};
static SortBufs sort_bufs(unsigned char* scratch, long long n, int with_labels) {
    const size_t a4 = ((size_t)n * 4 + 255) / 256 * 256;
    SortBufs B;
    B.G = sort_blocks(n);
    B.rounds = sort_rounds(n);
    B.idx[0] = (unsigned*)scratch;  // first: what follows it is free once it is sorted
    B.idx[1] = (unsigned*)(scratch + a4);
    B.key[0] = (unsigned*)(scratch + 2 * a4);
    B.key[1] = (unsigned*)(scratch + 3 * a4);
    B.lab = (unsigned*)(scratch + 4 * a4);
    B.hist = (unsigned*)(scratch + (4 + (with_labels ? 1 : 0)) * a4);
    B.tot = B.hist + ((size_t)B.G * 256 + 63) / 64 * 64;
    return B;
}

// One stable pass on the byte of key_in at shift.
static void digit_pass(const SortBufs& B, const unsigned* key_in, const unsigned* idx_in,
                       long long n, int shift, unsigned* key_out, unsigned* idx_out,
                       cudaStream_t st) {
    k_digit_hist<<<(unsigned)B.G, kSortThreads, 0, st>>>(key_in, n, shift, B.rounds, B.hist);
    k_digit_rows<<<256 / 8, 256, 0, st>>>(B.hist, (int)B.G, B.tot);
    k_digit_scatter<<<(unsigned)B.G, kSortThreads, 0, st>>>(key_in, idx_in, n, shift, B.rounds,
                                                            B.hist, B.tot, key_out, idx_out);
    count_launch(3);
}

// The four passes over 32-bit keys in B.key[0] (indices in B.idx[0]); the
// sorted keys and indices come back in the same buffers.
static void key_passes(const SortBufs& B, long long n, cudaStream_t st) {
    for (int pass = 0; pass < 4; ++pass) {
        const int in = pass & 1, o = in ^ 1;
        digit_pass(B, B.key[in], B.idx[in], n, 8 * pass, B.key[o], B.idx[o], st);
    }
}

// The same for at most kSmallSort keys, one launch a pass: hist has the four
// passes' digit counts, zeroed but for the first's, which is complete.
static void small_passes(const SortBufs& B, long long n, cudaStream_t st) {
    const unsigned G = (unsigned)small_blocks(n);
    for (int pass = 0; pass < 4; ++pass) {
        const int in = pass & 1, o = in ^ 1;
        unsigned* h = B.hist + (size_t)pass * G * 256;
        k_small_pass<<<G, kSmallThreads, 0, st>>>(B.key[in], B.idx[in], (int)n, 8 * pass, h,
                                                  pass < 3 ? h + (size_t)G * 256 : nullptr,
                                                  B.key[o], B.idx[o]);
    }
    count_launch(4);
}

int spatial_order(const double* x64, long long stride, long long n, int check,
                  const int* labels, int n_labels, unsigned char* scratch, int sm_count,
                  cudaStream_t st, const unsigned** order, const unsigned** sorted_labels) {
    const SortBufs B = sort_bufs(scratch, n, labels != nullptr);
    *order = B.idx[0];
    if (sorted_labels) *sorted_labels = nullptr;
    if (n <= 0) return WTHETA_OK;
    k_sort_keys<<<launch_grid(n, sm_count), 256, 0, st>>>(x64, stride, n, check, B.key[0],
                                                          B.idx[0]);
    count_launch();
    key_passes(B, n, st);
    if (labels) {
        // one more stable pass per byte of the label (two above 256 labels):
        // regions in label order, each in spatial order
        int cur = 0;
        for (int shift = 0; shift == 0 || (shift < 16 && (n_labels - 1) >> shift); shift += 8) {
            k_sorted_labels<<<launch_grid(n, sm_count), 256, 0, st>>>(B.idx[cur], labels, n,
                                                                      n_labels, B.lab);
            count_launch();
            digit_pass(B, B.lab, B.idx[cur], n, shift, B.key[cur ^ 1], B.idx[cur ^ 1], st);
            cur ^= 1;
        }
        *order = B.idx[cur];
        if (sorted_labels) *sorted_labels = B.key[cur];
    }
    return check_cuda(cudaGetLastError());
}

// The FP32 part of a prepared set of P padded positions: points, then the
// spheres of chunks and groups; and the part that may lie where the sort kept its buffers: local
// coordinates and the chunks' kappa and slack.
static size_t a256(size_t b) { return (b + 255) / 256 * 256; }
static size_t sphere_bytes(long long P) { return a256((size_t)P / 32 * 16) + a256((size_t)P / 8 * 16); }
static size_t local_bytes(long long P) { return a256((size_t)P * 12) + (size_t)P / 32 * 8; }

size_t prepare_joint_bytes(long long na, long long pa, long long nb, long long pb) {
    const long long N = na + nb, P = pa + pb;
    size_t b = a256((size_t)P * 16);              // FP32 points
    b += sphere_bytes(P);                         // bounding spheres
    b += a256((size_t)N * 24);                    // FP64, input order
    // the sort; once the order is known its other buffers become the local
    // coordinates
    b += std::max(order_bytes(N, 0), a256((size_t)N * 4) + local_bytes(P));
    return b;
}

void prepare_layout(long long na, long long pa, long long nb, long long pb, unsigned char* scratch,
                    Prepared* A, Prepared* B) {
    const long long N = na + nb, P = pa + pb;
    unsigned char* sp = scratch;
    A->p32 = (const float4*)sp;
    sp += a256((size_t)P * 16);
    A->c32 = (const float4*)sp;
    A->groups = (const float4*)(sp + a256((size_t)P / 32 * 16));
    sp += sphere_bytes(P);
    A->x64 = (const double*)sp;
    A->stride = N;
    sp += a256((size_t)N * 24) + a256((size_t)N * 4);  // and the sorted order
    A->l32 = (const float*)sp;
    A->l_stride = P;
    A->kap = (const float2*)(sp + a256((size_t)P * 12));
    *B = tile_view(*A, pa);
    B->x64 = A->x64 + na;
}

void prepare_zero(long long na, long long pa, long long nb, long long pb, unsigned char* scratch,
                  unsigned** words, long long* n) {
    const long long N = na + nb, P = pa + pb;
    unsigned char* sort = scratch + a256((size_t)P * 16) + sphere_bytes(P) + a256((size_t)N * 24);
    *words = sort_bufs(sort, N, 0).hist;
    *n = N <= kSmallSort ? small_blocks(N) * 4 * 256 : 0;
}

int prepare_joint(const double* a, long long na, long long pa, const double* b, long long nb,
                  long long pb, int is_xyz, int tag0, unsigned char* scratch, int sm_count,
                  cudaStream_t st, Prepared* A, Prepared* B, bool zeroed) {
    TraceRange trace("prepare");
    const long long N = na + nb, P = pa + pb;
    if (N >= (1LL << 32) - 1) return WTHETA_EINVAL;  // 32-bit positions in the sort
    prepare_layout(na, pa, nb, pb, scratch, A, B);
    double* x = (double*)A->x64;
    const SortBufs S = sort_bufs((unsigned char*)x + a256((size_t)N * 24), N, 0);
    LocalChunks L;
    L.xyz = (float*)A->l32;
    L.stride = P;
    L.caps = (float4*)A->c32;
    L.groups = (float4*)A->groups;
    L.kap = (float2*)A->kap;
    if (N > 0) {
        const long long g = std::min<long long>((N + 63) / 64, (long long)sm_count * 32);
        const bool small = N <= kSmallSort;
        if (small && !zeroed) {
            const int rc = check_cuda(
                cudaMemsetAsync(S.hist, 0, (size_t)small_blocks(N) * 4 * 256 * 4, st));
            if (rc) return rc;
        }
        k_joint_keys<<<(unsigned)g, 64, 0, st>>>(a, na, b, nb, is_xyz, x, S.key[0], S.idx[0],
                                                 small ? S.hist : nullptr);
        count_launch();
        if (small) small_passes(S, N, st);
        else key_passes(S, N, st);
    }
    if (P > 0) {
        k_gather_joint<<<launch_grid(P, sm_count), 256, 0, st>>>(x, na, pa, nb, pb, S.idx[0], tag0,
                                                                 (float4*)A->p32, L);
        count_launch();
    }
    return check_cuda(cudaGetLastError());
}

int launch_radec_to_xyz(const double* coords, long long n, double* xyz, int sm_count,
                        cudaStream_t st) {
    if (n <= 0) return WTHETA_OK;
    k_radec_to_xyz<<<launch_grid(n, sm_count), 256, 0, st>>>(coords, n, xyz, n);
    count_launch();
    return check_cuda(cudaGetLastError());
}

int launch_count_labels(const unsigned* lab, long long n, int n_labels,
                        unsigned long long* sizes, int sm_count, cudaStream_t st) {
    if (n <= 0) return WTHETA_OK;
    k_count_labels<<<launch_grid(n, sm_count), 256, 0, st>>>(lab, n, n_labels, sizes);
    count_launch();
    return check_cuda(cudaGetLastError());
}

int launch_gather_regions(const double* x64, long long stride, const unsigned* order,
                          const long long* src, const long long* dst, int R, long long n_pad,
                          int tag, int sm_count, cudaStream_t st, const Prepared& out) {
    if (n_pad <= 0) return WTHETA_OK;
    LocalChunks L;
    L.xyz = (float*)out.l32;
    L.stride = out.l_stride;
    L.caps = (float4*)out.c32;
    L.groups = (float4*)out.groups;
    L.kap = (float2*)out.kap;
    k_gather_regions<<<launch_grid(n_pad, sm_count), 256, 0, st>>>(
        x64, stride, order, src, dst, R, n_pad, (float4*)out.p32, tag, L);
    count_launch();
    return check_cuda(cudaGetLastError());
}

size_t regions_bytes(long long n_pad) {
    return a256((size_t)n_pad * 16) + a256((size_t)n_pad / 32 * 16);
}
size_t regions_group_bytes(long long n_pad) { return a256((size_t)n_pad / 8 * 16); }
size_t regions_sort_bytes(long long n, long long n_pad) {
    return std::max(a256(order_bytes(n, 1)), 2 * a256((size_t)n * 4) + a256(local_bytes(n_pad)));
}

Prepared regions_layout(unsigned char* p, unsigned char* groups, unsigned char* sort, long long n,
                        long long n_pad) {
    Prepared q;
    q.p32 = (const float4*)p;
    q.c32 = (const float4*)(p + a256((size_t)n_pad * 16));
    q.groups = (const float4*)groups;
    unsigned char* local = sort + 2 * a256((size_t)n * 4);  // past both index buffers
    q.l32 = (const float*)local;
    q.l_stride = n_pad;
    q.kap = (const float2*)(local + a256((size_t)n_pad * 12));
    return q;
}

PlanLayout plan_scratch(int n_cats2, long long n, long long n_pad) {
    PlanLayout Y;
    size_t b = 256;  // the cursor
    Y.cats = b;
    b += a256((size_t)n_cats2 * sizeof(BatchCat));
    Y.offs = b;
    b += a256((size_t)2 * (n_cats2 + 1) * 8);
    Y.x = b;
    b += a256((size_t)n * 24);
    Y.lab = b;  // the labels; once sorted, the groups' spheres
    b += std::max(a256((size_t)n * 4), regions_group_bytes(n_pad));
    Y.sort = b;
    b += regions_sort_bytes(n, n_pad);
    Y.all = b;
    b += regions_bytes(n_pad);
    Y.bytes = b;
    return Y;
}

Prepared tile_view(const Prepared& A, long long pos) {
    Prepared q = A;
    q.p32 += pos;
    q.c32 += pos / 32;
    q.groups += pos / 8;
    q.kap += pos / 32;
    q.l32 += pos;
    return q;
}

int launch_cull_batch(const CullSeg* cs, int n_segs, long long total, double theta_top,
                      unsigned long long* kept, Segment* segs, unsigned long long* n_kept,
                      int sm_count, cudaStream_t st, unsigned long long* stats) {
    if (n_segs <= 0) return WTHETA_OK;
    k_cull_batch<<<launch_grid(std::max(total, 1LL), sm_count), 256, 0, st>>>(
        cs, n_segs, total, theta_top, kept, stats);
    k_cull_prefix<<<1, kPrefixThreads, 0, st>>>(segs, cs, kept, n_segs, n_kept);
    count_launch(2);
    return check_cuda(cudaGetLastError());
}

unsigned long long per_item_bound(const Variant* v) {
    // A thread bins (or settles by chunk) R x TB pairs per unit of its own
    // sub-tile and may take the units of every other sub-tile of the item
    // (NT/32 of them): own = NT/32 x R TB pairs of its own groups.  With span
    // jobs it also runs at most one job (R x 32 pairs, counted up or down in a
    // word) per round of its warp; the warp's jobs are at most
    // (kMaxEdgesFar + 1) / 2 per lane and chunk, so its full rounds add at most
    // that many times own; before them come its chunk's pairs with a whole
    // sub-tile (at most own), after them at most three pooled rounds and the
    // pairs of its own chunk of a diagonal tile pair.  A per-warp column
    // gains 32 times as much, one shared by eight lanes eight times.
    const unsigned long long own = (unsigned long long)(v->nt / 32) * (unsigned long long)v->r *
                                   (unsigned long long)v->nt * (unsigned long long)v->r;
    return (v->hm == kHistWarp || v->hm == kHistWarpRed ? 32ull : 8ull) *
           ((2ull + (kMaxEdgesFar + 1) / 2) * own + 4ull * 32ull * (unsigned)v->r);
}

Segment make_segment(const Prepared& A, const Prepared& B, long long ta, long long tb,
                            int is_auto, long long item_begin, unsigned long long* counts,
                            unsigned long long total) {
    Segment g;
    std::memset(&g, 0, sizeof(g));
    g.a32 = A.p32; g.b32 = B.p32; g.a64 = A.x64; g.b64 = B.x64;
    g.a_caps = A.c32;
    g.a_groups = A.groups;
    g.al = A.l32;
    g.al_stride = A.l_stride;
    g.b_caps = B.c32;
    g.b_kap = B.kap;
    g.bl = B.l32;
    g.bl_stride = B.l_stride;
    g.a64_stride = A.stride; g.b64_stride = B.stride;
    g.tiles_a = ta; g.tiles_b = tb;
    g.item_begin = item_begin;
    g.n_items = is_auto ? ta * (ta + 1) / 2 : ta * tb;
    g.counts = counts;
    g.total = total;
    g.is_auto = is_auto;
    return g;
}

PairParams make_params(const Variant* v, const BinTable& tab, const Segment* seg0,
                              const Segment* segs, int n_segs, long long item_begin,
                              long long n_items, unsigned long long* cursor,
                              unsigned long long* stats) {
    PairParams prm;
    std::memset(&prm, 0, sizeof(prm));
    if (seg0) prm.seg0 = *seg0;
    prm.segs = segs;
    prm.n_segs = n_segs;
    prm.item_begin = item_begin;
    prm.n_items = n_items;
    // the words of the private columns are signed sums
    prm.items_per_flush = (int)std::min<unsigned long long>(0x7FFFFFFFull / per_item_bound(v),
                                                            1ull << 30);
    prm.cursor = cursor;
    prm.stats = stats;
    std::memcpy(&prm.tab, &tab, sizeof(tab));
    return prm;
}

// Core of wtheta_count / wtheta_count_xyz / wtheta_count_ex.
static int count_impl(const double* ca, long long n_a, const double* cb, long long n_b,
                      int is_xyz, const double* edges, int K, int is_auto,
                      unsigned long long* counts, const wtheta_tune* tune,
                      unsigned long long* stats, cudaStream_t st) {
    TraceRange trace("wtheta_count");
    if (!counts || n_a < 0 || n_b < 0 || (is_auto != 0 && is_auto != 1) ||
        (is_xyz != 0 && is_xyz != 1))
        return WTHETA_EINVAL;
    if (n_a > 0 && !ca) return WTHETA_EINVAL;
    if (is_auto) {
        if (cb && cb != ca) return WTHETA_EINVAL;
        if (n_b != n_a && !(cb == nullptr && n_b == 0)) return WTHETA_EINVAL;
        cb = ca;
        n_b = n_a;
    } else if (n_b > 0 && !cb) {
        return WTHETA_EINVAL;
    }
    if (tune && (tune->threads < 0 || tune->points_per_thread < 0 || tune->hist_mode < 0 ||
                 tune->hist_mode > 4 || tune->j_per_screen < 0 || tune->j_per_screen > 2 ||
                 tune->deferred < 0 || tune->deferred > 2 || tune->blocks_per_sm < 0 ||
                 tune->skip_far < 0 || tune->skip_far > 2 || tune->span_bins < 0 ||
                 tune->span_bins > 2))
        return WTHETA_EINVAL;
    static thread_local BinTable tab;  // large; built per call on the host
    int rc = build_table(edges, K, &tab);
    if (rc) return rc;
    DeviceInfo di;
    if ((rc = device_info(&di))) return rc;

    const unsigned long long total =
        is_auto ? (unsigned long long)n_a * (unsigned long long)(n_a > 0 ? n_a - 1 : 0) / 2ull
                : (unsigned long long)n_a * (unsigned long long)n_b;
    const bool empty = is_auto ? n_a < 2 : (n_a == 0 || n_b == 0);
    if (empty) {
        if ((rc = check_cuda(cudaMemsetAsync(counts, 0, sizeof(unsigned long long) * (K + 2), st))))
            return rc;
        k_finalize<<<1, 1, 0, st>>>(counts, K, total);
        count_launch();
        return check_cuda(cudaGetLastError());
    }

    const Variant* v = pick_for_size(tune, std::max(n_a, n_b), K, tab.n_lut, di.max_smem_optin);
    if (!v) return WTHETA_EINVAL;  // no instantiated shape matches the tuning request
    const long long T = (long long)v->nt * v->r;  // TA == TB
    const long long pa = round_up(n_a, T), pb = is_auto ? pa : round_up(n_b, T);

    const long long ta = pa / T, tb = pb / T;
    const long long n_items = is_auto ? ta * (ta + 1) / 2 : ta * tb;
    const size_t smem = v->smem(K, tab.n_lut);
    const int want_per_sm = tune && tune->blocks_per_sm ? tune->blocks_per_sm : 0;
    int resident = 0;  // blocks resident at once
    if ((rc = grid_for(v, smem, 1LL << 36, di.sm_count, want_per_sm, &resident))) return rc;
    // skip tile pairs wholly beyond the top edge (their pairs are overflow),
    // unless the items fill at most two waves of the launch: the caps and the
    // culling launches then cost about what they could save
    const bool skip_far = (!tune || tune->skip_far != 2) && edges[K] < 180.0 && n_items > 0 &&
                          n_items < (1LL << 32) &&
                          (n_items > 2LL * resident || (tune && tune->skip_far == 1));

    // scratch: the cursor and the kept count, both catalogues prepared
    // together, then the tile caps and the kept list
    const size_t bp = prepare_joint_bytes(n_a, pa, is_auto ? 0 : n_b, is_auto ? 0 : pb);
    const size_t off_caps = 256 + (bp + 255) / 256 * 256;
    const size_t off_list = off_caps + (skip_far ? ((size_t)(ta + tb) * sizeof(TileCap) + 255) / 256 * 256 : 0);
    const size_t bytes = off_list + (skip_far ? (size_t)n_items * 4 : 0);
    void* scratch = nullptr;
    if ((rc = dev_malloc_async(&scratch, bytes, st))) return rc;
    unsigned char* sp = (unsigned char*)scratch;
    unsigned long long* cursor = (unsigned long long*)sp;  // cursor, kept count, blocks done
    Prepared A, B;
    CountTables begin;
    std::memset(&begin, 0, sizeof(begin));
    begin.zero[0] = (unsigned*)counts;
    begin.n_zero[0] = 2LL * (K + 2);
    begin.zero[1] = (unsigned*)cursor;
    begin.n_zero[1] = 2 * 3;
    prepare_zero(n_a, pa, is_auto ? 0 : n_b, is_auto ? 0 : pb, sp + 256, &begin.zero[2],
                 &begin.n_zero[2]);
    rc = launch_begin_count(begin, nullptr, nullptr, st);
    if (!rc)
        rc = prepare_joint(ca, n_a, pa, is_auto ? nullptr : cb, is_auto ? 0 : n_b,
                           is_auto ? 0 : pb, is_xyz, 0, sp + 256, di.sm_count, st, &A, &B, true);
    if (is_auto) B = A;

    unsigned* list = nullptr;
    unsigned long long* n_list = nullptr;
    if (!rc && skip_far) {
        n_list = cursor + 1;
        TileCap* caps_a = (TileCap*)(sp + off_caps);
        TileCap* caps_b = is_auto ? caps_a : caps_a + ta;
        list = (unsigned*)(sp + off_list);
        // one launch over both catalogues (b's tiles follow a's)
        k_tile_caps<<<(unsigned)(is_auto ? ta : ta + tb), 128, 0, st>>>(A.p32, is_auto ? pa : pa + pb,
                                                                     (int)T, caps_a);
        const double theta_top = edges[K] * (3.14159265358979323846 / 180.0);
        k_cull_items<<<launch_grid(n_items, di.sm_count), 256, 0, st>>>(
            caps_a, caps_b, ta, tb, is_auto, n_items, theta_top, list, n_list, stats);
        count_launch(2);
        rc = check_cuda(cudaGetLastError());
    }
    int grid = 0;
    if (!rc) rc = grid_for(v, smem, n_items, di.sm_count, want_per_sm, &grid);
    if (!rc) {
        Segment seg = make_segment(A, B, ta, tb, is_auto, 0, counts, total);
        seg.item_list = list;
        PairParams prm = make_params(v, tab, &seg, nullptr, 0, 0, n_items, cursor, stats);
        prm.n_items_dev = n_list;
        prm.done = cursor + 2;
        rc = launch_pairs(v, prm, grid, smem, st);
    }
    const cudaError_t fe = cudaFreeAsync(scratch, st);
    if (!rc) rc = check_cuda(fe);
    return rc;
}

// Pairs (i < j) of an auto count of n points whose first point i is in the
// sorted rows [r0, r1).
static unsigned long long auto_pairs_in_rows(long long n, long long r0, long long r1) {
    if (r1 <= r0) return 0ull;
    const unsigned long long a = (unsigned long long)r0, b = (unsigned long long)r1;
    return (b - a) * (unsigned long long)(n - 1) - (b * (b - 1) / 2 - (a ? a * (a - 1) / 2 : 0ull));
}

// First item (tile pair) of tile row I: auto counts enumerate the upper
// triangle row by row (row I holds t - I items), cross counts the rectangle.
static long long row_item(long long I, long long ta, long long tb, int is_auto) {
    return is_auto ? I * ta - I * (I - 1) / 2 : I * tb;
}

// A w(theta)'s device scratch: cursor, kept total and blocks done, segments,
// culling table and kept counts, both catalogues prepared together, tile caps
// (n_caps of them: for the skipping, and for a shard split's kept items per row,
// which reads them whether far tile pairs are skipped or not), kept items per
// row with the first row of every count, kept lists.
WthetaLayout wtheta_layout(long long nd, long long pd, long long nr, long long pr, long long T,
                           bool cull, int n_shards, long long total_items) {
    const long long td = pd / T, tr = pr / T;
    WthetaLayout Y;
    size_t b = 256 + 1024 + 1024 + 256;
    Y.prep = b;
    b += a256(prepare_joint_bytes(nd, pd, nr, pr));
    Y.caps = b;
    Y.n_caps = cull || n_shards > 1 ? td + tr : 0;
    b += a256((size_t)Y.n_caps * sizeof(TileCap));
    Y.rows = b;
    if (n_shards > 1) b += a256((size_t)(2 * td + tr) * 8);
    Y.row0 = b;
    if (n_shards > 1) b += 256;
    Y.lists = b;
    if (cull) b += (size_t)total_items * 4;
    Y.bytes = b;
    return Y;
}

// The three counts of one w(theta) (DD, DR, RR) in one persistent launch:
// each catalogue is prepared once, far tile pairs of each count are skipped
// on the device, and the counts are three segments of one work table, so
// there is one launch tail instead of three.  counts: device, 3 x (K+2).
//
// With n_shards > 1 only shard `shard` of each count is counted: the tile
// rows of the count (points of its first catalogue in the spatial order) are
// split into n_shards contiguous ranges holding equal numbers of kept tile
// pairs (one synchronisation brings the kept tile pairs per row to the host),
// and the shard counts the pairs whose first point lies in its rows, overflow
// slot included; the shards' counts add up to the whole count.
static int count_wtheta_impl(const double* cd, long long nd, const double* cr, long long nr,
                             int is_xyz, const double* edges, int K,
                             unsigned long long* counts, const wtheta_tune* tune,
                             unsigned long long* stats, cudaStream_t st, int shard = 0,
                             int n_shards = 1) {
    TraceRange trace("wtheta_count_wtheta");
    if (!counts || nd < 0 || nr < 0 || (nd > 0 && !cd) || (nr > 0 && !cr) ||
        (is_xyz != 0 && is_xyz != 1) || n_shards < 1 || shard < 0 || shard >= n_shards)
        return WTHETA_EINVAL;
    if (tune && (tune->threads < 0 || tune->points_per_thread < 0 || tune->hist_mode < 0 ||
                 tune->hist_mode > 4 || tune->j_per_screen < 0 || tune->j_per_screen > 2 ||
                 tune->deferred < 0 || tune->deferred > 2 || tune->blocks_per_sm < 0 ||
                 tune->skip_far < 0 || tune->skip_far > 2 || tune->span_bins < 0 ||
                 tune->span_bins > 2))
        return WTHETA_EINVAL;
    static thread_local BinTable tab;
    int rc = build_table(edges, K, &tab);
    if (rc) return rc;
    DeviceInfo di;
    if ((rc = device_info(&di))) return rc;
    const size_t K2 = (size_t)K + 2;
    const Variant* v = pick_for_size(tune, std::max(nd, nr), K, tab.n_lut, di.max_smem_optin);
    if (!v) return WTHETA_EINVAL;
    const long long T = (long long)v->nt * v->r;
    const long long pd = round_up(nd, T), pr = round_up(nr, T);
    const long long td = pd / T, tr = pr / T;
    const unsigned long long ndd = (unsigned long long)nd * (unsigned long long)(nd > 0 ? nd - 1 : 0) / 2;
    const unsigned long long ndr = (unsigned long long)nd * (unsigned long long)nr;
    const unsigned long long nrr = (unsigned long long)nr * (unsigned long long)(nr > 0 ? nr - 1 : 0) / 2;
    // the counts with work, biggest first
    struct Cnt {
        int kind;
        long long items;            // tile pairs of the count (of the shard's rows)
        unsigned long long total;   // pairs of the count (of the shard's rows)
        long long offset;           // first item of the shard's rows
    };
    Cnt all[3] = {{0, td * (td + 1) / 2, ndd, 0}, {1, td * tr, ndr, 0}, {2, tr * (tr + 1) / 2, nrr, 0}};
    std::vector<Cnt> cnts;
    for (const Cnt& c : all)
        if (c.total > 0) cnts.push_back(c);
    std::stable_sort(cnts.begin(), cnts.end(),
                     [](const Cnt& a, const Cnt& b) { return a.items > b.items; });
    const int n_segs = (int)cnts.size();
    long long total_items = 0;
    for (const Cnt& c : cnts) total_items += c.items;
    const size_t smem = v->smem(K, tab.n_lut);
    const int want_per_sm = tune && tune->blocks_per_sm ? tune->blocks_per_sm : 0;
    int resident = 0;  // blocks resident at once
    if ((rc = grid_for(v, smem, 1LL << 36, di.sm_count, want_per_sm, &resident))) return rc;
    // skip far tile pairs unless the items fill at most two waves of the
    // launch (the caps and the culling launches then cost about what they
    // could save) or a shard split needs the kept items per row
    const bool cull = (!tune || tune->skip_far != 2) && edges[K] < 180.0 && td * td < (1LL << 32) &&
                      td * tr < (1LL << 32) && tr * tr < (1LL << 32) &&
                      (total_items > 2LL * resident || n_shards > 1 || (tune && tune->skip_far == 1));
    const WthetaLayout Y = wtheta_layout(nd, pd, nr, pr, T, cull, n_shards, total_items);
    unsigned char* m = nullptr;
    if ((rc = dev_malloc_async((void**)&m, Y.bytes, st))) return rc;
    unsigned long long* cursor = (unsigned long long*)m;  // cursor, kept count, blocks done
    unsigned long long* n_kept = cursor + 1;
    Segment* d_segs = (Segment*)(m + 256);
    CullSeg* d_cull = (CullSeg*)(m + 256 + 1024);
    unsigned long long* d_kept = (unsigned long long*)(m + 256 + 2048);
    static_assert(3 * sizeof(Segment) <= 1024 && 3 * sizeof(CullSeg) <= 1024, "tables fit");
    Prepared D, R;
    CountTables tbl;  // without tables yet if the shard's rows are still to be chosen
    std::memset(&tbl, 0, sizeof(tbl));
    tbl.zero[0] = (unsigned*)counts;
    tbl.n_zero[0] = 6LL * (long long)K2;
    tbl.zero[1] = (unsigned*)cursor;
    tbl.n_zero[1] = 2 * 3;
    prepare_zero(nd, pd, nr, pr, m + Y.prep, &tbl.zero[2], &tbl.n_zero[2]);
    if (cull) {
        tbl.zero[3] = (unsigned*)d_kept;
        tbl.n_zero[3] = 2 * 3;
    }
    tbl.with_cull = cull ? 1 : 0;
    prepare_layout(nd, pd, nr, pr, m + Y.prep, &D, &R);
    TileCap* caps_d = (TileCap*)(m + Y.caps);
    TileCap* caps_r = caps_d + td;  // R's tiles follow D's in the joint copies
    const double theta_top = edges[K] * (3.14159265358979323846 / 180.0);
    auto cull_seg = [&](int i, long long begin) {
        const int k = cnts[i].kind;
        CullSeg c;
        std::memset(&c, 0, sizeof(CullSeg));
        c.begin = begin;
        c.n = cnts[i].items;
        c.offset = cnts[i].offset;
        c.ta = k == 2 ? tr : td;
        c.tb = k == 0 ? td : tr;
        c.is_auto = k != 1;
        c.ca = k == 2 ? caps_r : caps_d;
        c.cb = k == 0 ? caps_d : caps_r;
        return c;
    };
    auto prepare_both = [&] {
        int e = prepare_joint(cd, nd, pd, cr, nr, pr, is_xyz, 0, m + Y.prep, di.sm_count, st, &D,
                              &R, true);
        if (!e && Y.n_caps > 0)
            e = launch_tile_caps(D.p32, pd + pr, (int)T, td + tr, caps_d, st);
        return e;
    };
    if (n_shards > 1) {
        rc = launch_begin_count(tbl, d_segs, d_cull, st);
        if (!rc) rc = prepare_both();
        for (long long& z : tbl.n_zero) z = 0;
    }
    if (!rc && n_shards > 1 && n_segs > 0) {
        // kept tile pairs per tile row of every count (all tile pairs count when
        // nothing is skipped), then this shard's rows of each count
        long long row0[3], nrow[3], item = 0;
        CullSeg cs[3];
        for (int i = 0; i < n_segs; ++i) {
            cs[i] = cull_seg(i, item);
            item += cnts[i].items;
            row0[i] = i == 0 ? 0 : row0[i - 1] + nrow[i - 1];
            nrow[i] = cnts[i].kind == 2 ? tr : td;
        }
        unsigned long long* d_rows = (unsigned long long*)(m + Y.rows);
        long long* d_row0 = (long long*)(m + Y.row0);
        const long long n_rows = row0[n_segs - 1] + nrow[n_segs - 1];
        std::vector<unsigned long long> rows(n_rows);
        rc = check_cuda(cudaMemsetAsync(d_rows, 0, (size_t)n_rows * 8, st));
        if (!rc) rc = check_cuda(cudaMemcpyAsync(d_cull, cs, sizeof(CullSeg) * n_segs,
                                                 cudaMemcpyHostToDevice, st));
        if (!rc) rc = check_cuda(cudaMemcpyAsync(d_row0, row0, sizeof(row0), cudaMemcpyHostToDevice, st));
        if (!rc) {
            k_cull_rows<<<launch_grid(total_items, di.sm_count), 256, 0, st>>>(
                d_cull, n_segs, total_items, cull ? theta_top : 4.0, d_row0, d_rows);
            count_launch();
            rc = check_cuda(cudaGetLastError());
        }
        if (!rc) rc = check_cuda(cudaMemcpyAsync(rows.data(), d_rows, (size_t)n_rows * 8,
                                                 cudaMemcpyDeviceToHost, st));
        if (!rc) rc = check_cuda(cudaStreamSynchronize(st));
        for (int i = 0; i < n_segs && !rc; ++i) {
            const int k = cnts[i].kind;
            const int aut = k != 1;
            long long I0 = 0, I1 = 0;
            rc = wtheta_shard_weights((const uint64_t*)rows.data() + row0[i], nrow[i], shard, n_shards,
                                      (int64_t*)&I0, (int64_t*)&I1);
            const long long ta = k == 2 ? tr : td, tb = k == 0 ? td : tr;
            const long long n_a = k == 2 ? nr : nd, n_b = k == 0 ? nd : nr;
            const long long r0 = std::min(I0 * T, n_a), r1 = std::min(I1 * T, n_a);
            cnts[i].offset = row_item(I0, ta, tb, aut);
            cnts[i].items = row_item(I1, ta, tb, aut) - cnts[i].offset;
            cnts[i].total = aut ? auto_pairs_in_rows(n_a, r0, r1)
                                : (unsigned long long)(r1 - r0) * (unsigned long long)n_b;
        }
        total_items = 0;
        for (const Cnt& c : cnts) total_items += c.items;
    }
    Segment segs[3];
    CullSeg cs[3];
    long long item = 0;
    for (int i = 0; i < n_segs; ++i) {
        const int k = cnts[i].kind;
        const Prepared& A = k == 2 ? R : D;
        const Prepared& B = k == 0 ? D : R;
        const long long ta = k == 2 ? tr : td, tb = k == 0 ? td : tr;
        segs[i] = make_segment(A, B, ta, tb, k != 1, item, counts + (size_t)k * K2, cnts[i].total);
        segs[i].n_items = cnts[i].items;
        segs[i].item_offset = cnts[i].offset;
        cs[i] = cull_seg(i, item);
        cs[i].list = (unsigned*)(m + Y.lists) + item;
        item += cnts[i].items;
    }
    for (int i = 0; i < n_segs; ++i) {
        tbl.segs[i] = segs[i];
        tbl.cs[i] = cs[i];
    }
    tbl.n_segs = n_segs;
    if (!rc) rc = launch_begin_count(tbl, d_segs, d_cull, st);
    if (!rc && n_shards == 1) rc = prepare_both();
    if (!rc && n_segs > 0) {
        if (!rc && cull)
            rc = launch_cull_batch(d_cull, n_segs, total_items, theta_top, d_kept, d_segs, n_kept,
                                   di.sm_count, st, stats);
        int grid = 0;
        if (!rc) rc = grid_for(v, smem, std::max(total_items, 1LL), di.sm_count, want_per_sm, &grid);
        if (!rc && total_items > 0) {
            PairParams prm = make_params(v, tab, nullptr, d_segs, n_segs, 0, total_items, cursor,
                                         stats);
            if (cull) prm.n_items_dev = n_kept;
            prm.done = cursor + 2;
            rc = launch_pairs(v, prm, grid, smem, st);
        } else if (!rc) {
            rc = launch_finalize_segments(d_segs, n_segs, K, st);
        }
    }
    const cudaError_t fe = cudaFreeAsync(m, st);
    if (!rc) rc = check_cuda(fe);
    return rc;
}

int launch_pairs(const Variant* v, const PairParams& prm, int grid, size_t smem,
                 cudaStream_t st) {
    pair_kernel(v, prm)<<<grid, v->nt, smem, st>>>(prm);
    count_launch();
    return check_cuda(cudaGetLastError());
}

int launch_finalize_segments(const Segment* d_segs, int n_segs, int K, cudaStream_t st) {
    if (n_segs <= 0) return WTHETA_OK;
    k_finalize_segments<<<(n_segs + 127) / 128, 128, 0, st>>>(d_segs, n_segs, K);
    count_launch();
    return check_cuda(cudaGetLastError());
}

int launch_tile_caps(const float4* p32, long long n, int T, long long tiles, TileCap* caps,
                     cudaStream_t st) {
    if (tiles <= 0) return WTHETA_OK;
    k_tile_caps<<<(unsigned)tiles, 128, 0, st>>>(p32, n, T, caps);
    count_launch();
    return check_cuda(cudaGetLastError());
}

int launch_cull_items(const TileCap* ca, const TileCap* cb, long long ta, long long tb,
                      int is_auto, long long n_items, double theta_top, unsigned* list,
                      unsigned long long* n_list, int sm_count, cudaStream_t st) {
    if (n_items <= 0) return WTHETA_OK;
    k_cull_items<<<launch_grid(n_items, sm_count), 256, 0, st>>>(ca, cb, ta, tb, is_auto, n_items,
                                                                   theta_top, list, n_list, nullptr);
    count_launch();
    return check_cuda(cudaGetLastError());
}

void add_launches(long long n) { g_launches.fetch_add((unsigned long long)n); }

// -1: no injected failure; n >= 0: the allocation after n more succeed fails
static std::atomic<long long> g_fail_alloc{-1};

static bool injected_failure() {
    long long v = g_fail_alloc.load();
    while (v >= 0) {
        if (g_fail_alloc.compare_exchange_weak(v, v - 1)) return v == 0;
    }
    return false;
}

int dev_malloc(void** p, size_t bytes) {
    if (injected_failure()) return WTHETA_ENOMEM;
    const cudaError_t e = cudaMalloc(p, bytes);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        return WTHETA_ENOMEM;
    }
    return check_cuda(e);
}

int dev_malloc_async(void** p, size_t bytes, cudaStream_t st) {
    if (injected_failure()) return WTHETA_ENOMEM;
    const cudaError_t e = cudaMallocAsync(p, bytes, st);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        return WTHETA_ENOMEM;
    }
    return check_cuda(e);
}

TraceRange::TraceRange(const char* name) { nvtxRangePushA(name); }
TraceRange::~TraceRange() { nvtxRangePop(); }

// ---------------------------------------------------------------------------
// allocation-free variant of the xyz count
// ---------------------------------------------------------------------------
// The fixed scratch of wtheta_count_xyz_noalloc: a 256-byte head holding the
// work cursor, then FP32 float4 copies of catalogue a and (cross counts)
// catalogue b, each padded to whole tiles.  It is loaded with the library's
// module on every device that uses it and lives until the process exits.
static __device__ __align__(256) unsigned char
    g_noalloc_scratch[256 + 16 * (size_t)WTHETA_NOALLOC_MAX_POINTS];

// Device address of g_noalloc_scratch on the current device.  In host code
// the symbol names a host-side stand-in, not device memory, so the address is
// looked up once per device (with that device current) and cached.
static int noalloc_scratch(unsigned char** out) {
    static std::mutex mu;
    static void* addr[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return WTHETA_ECUDA;
    std::lock_guard<std::mutex> g(mu);
    if (!addr[dev]) {
        void* p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || p == nullptr) return WTHETA_ECUDA;
        addr[dev] = p;
    }
    *out = (unsigned char*)addr[dev];
    return WTHETA_OK;
}

static int count_xyz_noalloc_impl(const double* ca, long long n_a, const double* cb,
                                  long long n_b, const double* edges, int K, int is_auto,
                                  unsigned long long* counts, cudaStream_t st) {
    if (!counts || n_a < 0 || n_b < 0 || (is_auto != 0 && is_auto != 1)) return WTHETA_EINVAL;
    if (n_a > 0 && !ca) return WTHETA_EINVAL;
    if (is_auto) {
        if (cb && cb != ca) return WTHETA_EINVAL;
        if (n_b != n_a && !(cb == nullptr && n_b == 0)) return WTHETA_EINVAL;
        cb = ca;
        n_b = n_a;
    } else if (n_b > 0 && !cb) {
        return WTHETA_EINVAL;
    }
    const long long T = WTHETA_NOALLOC_TILE;
    // each size alone first, so that the rounding below cannot overflow
    if (n_a > (long long)WTHETA_NOALLOC_MAX_POINTS || n_b > (long long)WTHETA_NOALLOC_MAX_POINTS)
        return WTHETA_ESIZE;
    const long long pa = round_up(n_a, T), pb = is_auto ? 0 : round_up(n_b, T);
    if (pa + pb > (long long)WTHETA_NOALLOC_MAX_POINTS) return WTHETA_ESIZE;
    static thread_local BinTable tab;
    int rc = build_table(edges, K, &tab);
    if (rc) return rc;
    DeviceInfo di;
    if ((rc = device_info(&di))) return rc;
    unsigned char* base = nullptr;
    if ((rc = noalloc_scratch(&base))) return rc;

    if ((rc = check_cuda(cudaMemsetAsync(counts, 0, sizeof(unsigned long long) * (K + 2), st))))
        return rc;
    const unsigned long long total =
        is_auto ? (unsigned long long)n_a * (unsigned long long)(n_a > 0 ? n_a - 1 : 0) / 2ull
                : (unsigned long long)n_a * (unsigned long long)n_b;
    const bool empty = is_auto ? n_a < 2 : (n_a == 0 || n_b == 0);
    if (empty) {
        k_finalize<<<1, 1, 0, st>>>(counts, K, total);
        count_launch();
        return check_cuda(cudaGetLastError());
    }
    wtheta_tune fixed = {128, 8, 0, 0, 0, 0, 2, 2};  // the tile of WTHETA_NOALLOC_TILE points
    const Variant* v = pick_variant(&fixed, K, tab.n_lut, di.max_smem_optin);
    // (without spheres: only a build without span jobs)
    if (!v || (long long)v->nt * v->r != T || has_spans(v)) return WTHETA_EINVAL;

    unsigned long long* cursor = (unsigned long long*)base;
    float4* a32 = (float4*)(base + 256);
    float4* b32 = is_auto ? a32 : a32 + pa;
    const int cvt_threads = 256;
    auto cvt_grid = [&](long long n) {
        long long g = (n + cvt_threads - 1) / cvt_threads;
        return (int)std::min<long long>(std::max<long long>(g, 1), (long long)di.sm_count * 16);
    };
    // every word the kernels read is rewritten here: both padded copies and the cursor
    k_xyz_to_f32<<<cvt_grid(pa), cvt_threads, 0, st>>>(ca, n_a, pa, a32, 0);
    count_launch();
    if (!is_auto) {
        k_xyz_to_f32<<<cvt_grid(pb), cvt_threads, 0, st>>>(cb, n_b, pb, b32, 1);
        count_launch();
    }
    // (cursor, a word unused here, blocks done)
    if ((rc = check_cuda(cudaMemsetAsync(cursor, 0, 3 * sizeof(unsigned long long), st)))) return rc;
    const long long ta = pa / T, tb = is_auto ? ta : pb / T;
    const long long n_items = is_auto ? ta * (ta + 1) / 2 : ta * tb;
    const size_t smem = v->smem(K, tab.n_lut);
    int grid = 0;
    if ((rc = grid_for(v, smem, n_items, di.sm_count, 0, &grid))) return rc;
    Prepared A, B;
    A.p32 = a32; A.x64 = ca; A.stride = n_a;
    B.p32 = b32; B.x64 = cb; B.stride = n_b;
    const Segment seg = make_segment(A, B, ta, tb, is_auto, 0, counts, total);
    PairParams prm = make_params(v, tab, &seg, nullptr, 0, 0, n_items, cursor, nullptr);
    prm.done = cursor + 2;
    return launch_pairs(v, prm, grid, smem, st);
}

}  // namespace wtheta

// ---------------------------------------------------------------------------
// batched counts: one work queue over many catalogue pairs, one graph
// ---------------------------------------------------------------------------

struct wtheta_plan {
    int dev = 0;
    int K = 0;
    int n_cats = 0;
    int is_xyz = 0;                        // catalogues are SoA unit vectors, not RA/Dec
    wtheta::BinTable tab;
    const wtheta::Variant* v = nullptr;
    wtheta_tune tune = {};
    int autotuned = 0;
    float autotune_ms = 0.f;
    std::vector<wtheta_catalog_pair> cats;
    void* scratch = nullptr;               // prepared copies of every catalogue
    std::vector<wtheta::Prepared> prep;    // 2 per catalogue pair
    std::vector<long long> n_pad;
    // all catalogues (data 2m, randoms 2m + 1) are prepared together: one FP64
    // array of every point, one sort by (catalogue, spatial key), FP32 copies
    // with every catalogue starting on a tile boundary
    std::vector<long long> src_off, dst_off;  // 2 n_cats + 1 each
    long long n_all = 0, n_all_pad = 0;
    wtheta::BatchCat* d_cats = nullptr;
    long long* d_src_off = nullptr;         // src_off, then dst_off (for the gather)
    double* x_all = nullptr;
    int* lab_all = nullptr;
    unsigned char* sort_scratch = nullptr;
    wtheta::Prepared all;                   // the copies of every catalogue
    wtheta::TileCap* caps_all = nullptr;
    wtheta::Segment* d_segs = nullptr;
    int n_segs = 0;
    long long total_items = 0;
    long long pairs = 0;
    unsigned long long* d_counts = nullptr;  // internal: [cat][kind][K+2]
    unsigned long long* d_cursor = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    int graph_kernels = 0;
    int grid = 0;
    size_t smem = 0;
    long long runs = 0;
    // skipping of far tile pairs, done in the graph on every run
    int cull = 0;
    double theta_top = 0.0;
    void* cull_mem = nullptr;
    wtheta::CullSeg* d_cull = nullptr;        // per count, in the work table's order
    unsigned long long* d_kept = nullptr;     // per count
    unsigned long long* d_total = nullptr;    // kept items of the run
    unsigned long long* d_stats = nullptr;    // WTHETA_NSTATS of the last run
    std::vector<wtheta::TileCap*> caps;       // per catalogue
    int sm_count = 0;
};

namespace wtheta {

// Autotuner cache: the shape picked for batches of similar work on a device
// of this size, keyed by (SM count, K, log2 of the batch's pair count).
struct TuneKey {
    int sm, K, size_bucket;
};
static std::mutex g_tune_mu;
static std::vector<std::pair<TuneKey, int>> g_tune_cache;

static int lookup_tuned(const TuneKey& k) {
    std::lock_guard<std::mutex> g(g_tune_mu);
    for (auto& e : g_tune_cache)
        if (e.first.sm == k.sm && e.first.K == k.K && e.first.size_bucket == k.size_bucket)
            return e.second;
    return -1;
}

static void store_tuned(const TuneKey& k, int idx) {
    std::lock_guard<std::mutex> g(g_tune_mu);
    g_tune_cache.push_back({k, idx});
}

// Preparation of every catalogue of a plan, as one pipeline over all of them
// (a constant number of launches whatever the number of catalogues):
// conversion into one FP64 array with a catalogue label per point, one
// spatial sort by (catalogue, key), FP32 copies with every catalogue starting
// on a tile boundary (sentinels in the rest of its last tile), chunk spheres
// and, when far tile pairs are skipped, tile caps.  Reads the catalogues'
// current contents (the graph replays it on every run).
static int batch_prepare(wtheta_plan* P, int T, cudaStream_t st) {
    const int nc2 = 2 * P->n_cats;
    if (P->n_all <= 0) return WTHETA_OK;
    k_batch_gather<<<launch_grid(P->n_all, P->sm_count), 256, 0, st>>>(
        P->d_cats, P->d_src_off, nc2, P->is_xyz, P->n_all, P->x_all, P->lab_all);
    count_launch();
    const unsigned* order = nullptr;
    int rc = spatial_order(P->x_all, P->n_all, P->n_all, P->is_xyz, P->lab_all, nc2,
                           P->sort_scratch, P->sm_count, st, &order, nullptr);
    if (!rc)
        rc = launch_gather_regions(P->x_all, P->n_all, order, P->d_src_off, P->d_src_off + nc2 + 1,
                                   nc2, P->n_all_pad, 0, P->sm_count, st, P->all);
    if (!rc && P->cull)
        rc = launch_tile_caps(P->all.p32, P->n_all_pad, T, P->n_all_pad / T, P->caps_all, st);
    return rc;
}

// Lays out the plan's scratch and work table for one kernel shape (its tile
// T = threads x points_per_thread), prepares every catalogue on stream st.
static int plan_layout(wtheta_plan* P, const Variant* v, int sm_count, cudaStream_t st) {
    const long long T = (long long)v->nt * v->r;
    const int nc = P->n_cats, nc2 = 2 * nc;
    P->sm_count = sm_count;
    P->n_pad.assign(nc2, 0);
    P->src_off.assign(nc2 + 1, 0);
    P->dst_off.assign(nc2 + 1, 0);
    std::vector<BatchCat> hc(nc2);
    for (int c = 0; c < nc2; ++c) {
        const wtheta_catalog_pair& q = P->cats[c / 2];
        hc[c].src = c % 2 ? q.rand : q.data;
        hc[c].n = c % 2 ? q.n_rand : q.n_data;
        P->n_pad[c] = round_up(hc[c].n, T);
        P->src_off[c + 1] = P->src_off[c] + hc[c].n;
        P->dst_off[c + 1] = P->dst_off[c] + P->n_pad[c];
    }
    P->n_all = P->src_off[nc2];
    P->n_all_pad = P->dst_off[nc2];
    const long long N = P->n_all, NP = P->n_all_pad;
    const PlanLayout Y = plan_scratch(nc2, N, NP);
    if (P->scratch) cudaFree(P->scratch);
    P->scratch = nullptr;
    int rc = dev_malloc(&P->scratch, Y.bytes);
    if (rc) return rc;
    unsigned char* base = (unsigned char*)P->scratch;
    P->d_cursor = (unsigned long long*)base;
    P->d_cats = (BatchCat*)(base + Y.cats);
    P->d_src_off = (long long*)(base + Y.offs);
    P->x_all = (double*)(base + Y.x);
    P->lab_all = (int*)(base + Y.lab);
    P->sort_scratch = base + Y.sort;
    P->all = regions_layout(base + Y.all, base + Y.lab, base + Y.sort, N, NP);
    P->all.x64 = P->x_all;
    P->all.stride = N;
    std::vector<long long> offs(P->src_off);
    offs.insert(offs.end(), P->dst_off.begin(), P->dst_off.end());
    rc = check_cuda(cudaMemcpyAsync(P->d_cats, hc.data(), sizeof(BatchCat) * nc2,
                                    cudaMemcpyHostToDevice, st));
    if (!rc) rc = check_cuda(cudaMemcpyAsync(P->d_src_off, offs.data(), offs.size() * 8,
                                             cudaMemcpyHostToDevice, st));
    if (rc) return rc;
    // every catalogue's view of the shared copies (FP64 in the caller's order:
    // the FP32 copies carry each point's position in the FP64 array)
    P->prep.assign(nc2, Prepared());
    for (int c = 0; c < nc2; ++c) P->prep[c] = tile_view(P->all, P->dst_off[c]);
    // the work table: DD, DR, RR of every pair, biggest count first
    std::vector<Segment> segs;
    std::vector<int> seg_cat_a, seg_cat_b;  // prepared catalogue of each side
    P->pairs = 0;
    for (int m = 0; m < nc; ++m) {
        const long long nd = P->cats[m].n_data, nr = P->cats[m].n_rand;
        const long long td = P->n_pad[2 * m] / T, tr = P->n_pad[2 * m + 1] / T;
        unsigned long long* c = P->d_counts + (size_t)3 * m * (P->K + 2);
        const unsigned long long ndd = (unsigned long long)nd * (unsigned long long)(nd - 1) / 2;
        const unsigned long long ndr = (unsigned long long)nd * (unsigned long long)nr;
        const unsigned long long nrr = (unsigned long long)nr * (unsigned long long)(nr - 1) / 2;
        P->pairs += (long long)(ndd + ndr + nrr);
        segs.push_back(make_segment(P->prep[2 * m], P->prep[2 * m], td, td, 1, 0, c, ndd));
        segs.push_back(make_segment(P->prep[2 * m], P->prep[2 * m + 1], td, tr, 0, 0,
                                    c + (P->K + 2), ndr));
        segs.push_back(make_segment(P->prep[2 * m + 1], P->prep[2 * m + 1], tr, tr, 1, 0,
                                    c + 2 * (P->K + 2), nrr));
        seg_cat_a.insert(seg_cat_a.end(), {2 * m, 2 * m, 2 * m + 1});
        seg_cat_b.insert(seg_cat_b.end(), {2 * m, 2 * m + 1, 2 * m + 1});
    }
    std::vector<int> order(segs.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
    std::stable_sort(order.begin(), order.end(),
                     [&](int a, int b) { return segs[a].n_items > segs[b].n_items; });
    std::vector<Segment> sorted;
    std::vector<CullSeg> cull(segs.size());
    long long items = 0;
    for (size_t i = 0; i < order.size(); ++i) {
        Segment g = segs[order[i]];
        g.item_begin = items;
        CullSeg& q = cull[i];
        std::memset(&q, 0, sizeof(q));
        q.begin = items;
        q.n = g.n_items;
        q.ta = g.tiles_a;
        q.tb = g.tiles_b;
        q.is_auto = g.is_auto;
        items += g.n_items;
        sorted.push_back(g);
    }
    P->total_items = items;
    P->n_segs = (int)sorted.size();
    if (P->d_segs) cudaFree(P->d_segs);
    P->d_segs = nullptr;
    if (P->cull_mem) cudaFree(P->cull_mem);
    P->cull_mem = nullptr;
    P->caps.assign(2 * nc, nullptr);
    if ((rc = dev_malloc((void**)&P->d_segs, sizeof(Segment) * sorted.size()))) return rc;
    if (P->cull) {
        // kept counters, total, the count table, the tile caps of all the
        // catalogues' tiles, and one list of item indices per count
        size_t cb = ((size_t)P->n_segs * 8 + 8 + 255) / 256 * 256;
        const size_t off_cs = cb;
        cb += (sizeof(CullSeg) * P->n_segs + 255) / 256 * 256;
        const size_t off_caps = cb;
        cb += ((size_t)(NP / T) * sizeof(TileCap) + 255) / 256 * 256;
        const size_t off_lists = cb;
        cb += (size_t)items * 4;
        if ((rc = dev_malloc(&P->cull_mem, cb))) return rc;
        unsigned char* cm = (unsigned char*)P->cull_mem;
        P->d_kept = (unsigned long long*)cm;
        P->d_total = P->d_kept + P->n_segs;
        P->d_cull = (CullSeg*)(cm + off_cs);
        P->caps_all = (TileCap*)(cm + off_caps);
        for (int c = 0; c < nc2; ++c) P->caps[c] = P->caps_all + P->dst_off[c] / T;
        unsigned* lists = (unsigned*)(cm + off_lists);
        for (size_t i = 0; i < order.size(); ++i) {
            cull[i].ca = P->caps[seg_cat_a[order[i]]];
            cull[i].cb = P->caps[seg_cat_b[order[i]]];
            cull[i].list = lists + cull[i].begin;
        }
        rc = check_cuda(cudaMemcpyAsync(P->d_cull, cull.data(), sizeof(CullSeg) * cull.size(),
                                        cudaMemcpyHostToDevice, st));
        if (rc) return rc;
    }
    rc = check_cuda(cudaMemcpyAsync(P->d_segs, sorted.data(), sizeof(Segment) * sorted.size(),
                                    cudaMemcpyHostToDevice, st));
    // the catalogues, prepared once now (for the autotuner's timing); the
    // graph prepares them again on every run
    if (!rc) rc = batch_prepare(P, (int)T, st);
    return rc;
}

static int launch_batch_pairs(wtheta_plan* P, const Variant* v, long long item_begin,
                              long long n_items, int grid, size_t smem, cudaStream_t st,
                              const unsigned long long* n_items_dev = nullptr,
                              unsigned long long* stats = nullptr) {
    PairParams prm = make_params(v, P->tab, nullptr, P->d_segs, P->n_segs, item_begin,
                                 n_items, P->d_cursor, stats);
    prm.n_items_dev = n_items_dev;
    pair_kernel(v, prm)<<<grid, v->nt, smem, st>>>(prm);
    count_launch();
    return check_cuda(cudaGetLastError());
}

// Times each candidate shape on the first items of the queue (the biggest
// counts) and keeps the fastest per pair.  Candidates share a tile size per
// layout; a different tile size re-lays the plan out.
static int autotune(wtheta_plan* P, const DeviceInfo& di, cudaStream_t st, int* best_idx) {
    int nv = 0;
    const Variant* vs = variants(&nv);
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
        return WTHETA_ECUDA;
    float best = 1e30f;
    int rc = WTHETA_OK;
    long long cur_T = -1;
    for (int i = 0; i < nv && !rc; ++i) {
        const Variant* v = &vs[i];
        if (v->def == 2) continue;  // spans are never worth leaving out here
        const size_t smem = v->smem(P->K, P->tab.n_lut);
        if (smem > (size_t)di.max_smem_optin) continue;
        const long long T = (long long)v->nt * v->r;
        if (T != cur_T) {
            if ((rc = plan_layout(P, v, di.sm_count, st))) break;
            cur_T = T;
        }
        int grid = 0;
        if ((rc = grid_for(v, smem, P->total_items, di.sm_count, 0, &grid))) break;
        // a sample of several items per CTA, from the front of the queue
        const long long n_sample =
            std::min<long long>(P->total_items, std::max<long long>(8LL * grid, P->total_items / 64));
        float ms = 0.f;
        for (int rep = 0; rep < 2 && !rc; ++rep) {  // first pass warms up
            rc = check_cuda(cudaMemsetAsync(P->d_cursor, 0, 8, st));
            if (!rc) rc = check_cuda(cudaEventRecord(e0, st));
            if (!rc) rc = launch_batch_pairs(P, v, 0, n_sample, grid, smem, st);
            if (!rc) rc = check_cuda(cudaEventRecord(e1, st));
            if (!rc) rc = check_cuda(cudaEventSynchronize(e1));
            if (!rc) rc = check_cuda(cudaEventElapsedTime(&ms, e0, e1));
        }
        if (rc) break;
        const float per = ms / ((float)n_sample * (float)T * (float)T);  // per pair
        if (per < best) {
            best = per;
            *best_idx = i;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return rc;
}

static int plan_capture(wtheta_plan* P, const DeviceInfo& di) {
    cudaStream_t cs;
    int rc = check_cuda(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    if (rc) return rc;
    const unsigned long long launches0 = g_launches.load();
    rc = check_cuda(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
    if (!rc) {
        // re-prepare every catalogue from its current coordinates (one
        // pipeline over all of them, tile caps included), then count
        const int T = P->v->nt * P->v->r;
        rc = batch_prepare(P, T, cs);
        if (!rc && P->cull) {
            // the kept tile pairs of every count, and the launch's item ranges
            if (!rc) rc = check_cuda(cudaMemsetAsync(P->d_kept, 0, (size_t)P->n_segs * 8, cs));
            if (!rc) {
                k_cull_batch<<<launch_grid(P->total_items, di.sm_count), 256, 0, cs>>>(
                    P->d_cull, P->n_segs, P->total_items, P->theta_top, P->d_kept, nullptr);
                k_cull_prefix<<<1, kPrefixThreads, 0, cs>>>(P->d_segs, P->d_cull, P->d_kept, P->n_segs,
                                                P->d_total);
                count_launch(2);
                rc = check_cuda(cudaGetLastError());
            }
        }
        const size_t nbytes = (size_t)P->n_cats * 3 * (P->K + 2) * sizeof(unsigned long long);
        if (!rc) rc = check_cuda(cudaMemsetAsync(P->d_counts, 0, nbytes, cs));
        if (!rc) rc = check_cuda(cudaMemsetAsync(P->d_cursor, 0, 8, cs));
        if (!rc) rc = check_cuda(cudaMemsetAsync(P->d_stats, 0, 8 * WTHETA_NSTATS, cs));
        if (!rc)
            rc = launch_batch_pairs(P, P->v, 0, P->total_items, P->grid, P->smem, cs,
                                    P->cull ? P->d_total : nullptr, P->d_stats);
        if (!rc) {
            k_finalize_segments<<<(P->n_segs + 127) / 128, 128, 0, cs>>>(P->d_segs, P->n_segs,
                                                                        P->K);
            count_launch();
            rc = check_cuda(cudaGetLastError());
        }
        cudaGraph_t g = nullptr;
        const cudaError_t ce = cudaStreamEndCapture(cs, &g);
        if (!rc) rc = check_cuda(ce);
        if (!rc) {
            P->graph = g;
            rc = check_cuda(cudaGraphInstantiate(&P->exec, g, 0));
        } else if (g) {
            cudaGraphDestroy(g);
        }
    }
    // launches recorded during capture are replayed, not launched: uncount them
    P->graph_kernels = (int)(g_launches.load() - launches0);
    g_launches.fetch_sub(P->graph_kernels);
    cudaStreamDestroy(cs);
    return rc;
}

static void plan_release(wtheta_plan* P) {
    if (P->exec) cudaGraphExecDestroy(P->exec);
    if (P->graph) cudaGraphDestroy(P->graph);
    if (P->scratch) cudaFree(P->scratch);
    if (P->d_segs) cudaFree(P->d_segs);
    if (P->d_counts) cudaFree(P->d_counts);
    if (P->cull_mem) cudaFree(P->cull_mem);
    if (P->d_stats) cudaFree(P->d_stats);
    delete P;
}

static int batch_plan_impl(const wtheta_catalog_pair* cats, int n_cats, int is_xyz,
                           const double* edges, int K, const wtheta_tune* tune, cudaStream_t st,
                           wtheta_plan** out) {
    // catalogues are labelled by 16-bit index in the shared sort
    if (!out || !cats || n_cats < 1 || n_cats > 32768 || (is_xyz != 0 && is_xyz != 1))
        return WTHETA_EINVAL;
    for (int m = 0; m < n_cats; ++m) {
        const wtheta_catalog_pair& c = cats[m];
        if (c.n_data < 2 || c.n_rand < 2 || !c.data || !c.rand) return WTHETA_EINVAL;
    }
    if (tune && (tune->threads < 0 || tune->points_per_thread < 0 || tune->hist_mode < 0 ||
                 tune->hist_mode > 4 || tune->j_per_screen < 0 || tune->j_per_screen > 2 ||
                 tune->deferred < 0 || tune->deferred > 2 || tune->blocks_per_sm < 0 ||
                 tune->skip_far < 0 || tune->skip_far > 2 || tune->span_bins < 0 ||
                 tune->span_bins > 2))
        return WTHETA_EINVAL;
    wtheta_plan* P = new wtheta_plan();
    P->K = K;
    P->n_cats = n_cats;
    P->is_xyz = is_xyz;
    P->cats.assign(cats, cats + n_cats);
    int rc = build_table(edges, K, &P->tab);
    if (!rc) {
        P->cull = (!tune || tune->skip_far != 2) && edges[K] < 180.0;
        P->theta_top = edges[K] * (3.14159265358979323846 / 180.0);
        // list entries are 32-bit item indices within a count
        for (int m = 0; m < n_cats; ++m) {
            const long long t = (std::max(cats[m].n_data, cats[m].n_rand) + 255) / 256;
            if (t * t >= (1LL << 32)) P->cull = 0;
        }
    }
    DeviceInfo di;
    if (!rc) rc = device_info(&di);
    if (!rc) rc = check_cuda(cudaGetDevice(&P->dev));
    if (!rc)
        rc = dev_malloc((void**)&P->d_counts, (size_t)n_cats * 3 * (K + 2) * sizeof(unsigned long long));
    if (!rc) rc = dev_malloc((void**)&P->d_stats, 8 * WTHETA_NSTATS);
    if (rc) {
        plan_release(P);
        return rc;
    }
    int nv = 0;
    const Variant* vs = variants(&nv);
    if (tune) {
        P->v = pick_variant(tune, K, P->tab.n_lut, di.max_smem_optin);
        if (!P->v) rc = WTHETA_EINVAL;
    } else {
        // size bucket: log2 of the batch's pairs
        long long pairs = 0;
        for (int m = 0; m < n_cats; ++m)
            pairs += cats[m].n_data * cats[m].n_data / 2 + cats[m].n_data * cats[m].n_rand +
                     cats[m].n_rand * cats[m].n_rand / 2;
        int bucket = 0;
        while ((1LL << (bucket + 1)) <= pairs && bucket < 62) ++bucket;
        const TuneKey key{di.sm_count, K, bucket};
        int idx = lookup_tuned(key);
        if (idx < 0) {
            cudaEvent_t t0, t1;
            cudaEventCreate(&t0);
            cudaEventCreate(&t1);
            cudaEventRecord(t0, st);
            rc = autotune(P, di, st, &idx);
            cudaEventRecord(t1, st);
            cudaEventSynchronize(t1);
            cudaEventElapsedTime(&P->autotune_ms, t0, t1);
            cudaEventDestroy(t0);
            cudaEventDestroy(t1);
            if (!rc && idx >= 0) store_tuned(key, idx);
        }
        if (!rc && idx < 0) rc = WTHETA_EINVAL;
        if (!rc) {
            P->v = &vs[idx];
            P->autotuned = 1;
        }
    }
    if (!rc) {
        P->tune.threads = P->v->nt;
        P->tune.points_per_thread = P->v->r;
        P->tune.j_per_screen = P->v->ju;
        P->tune.hist_mode = P->v->hm;
        P->tune.deferred = P->v->def == 1 ? 2 : 1;
        P->tune.skip_far = P->cull ? 1 : 2;
        P->tune.span_bins = tune && tune->span_bins == 2 ? 2 : 1;
        P->smem = P->v->smem(K, P->tab.n_lut);
        rc = plan_layout(P, P->v, di.sm_count, st);
    }
    if (!rc) rc = grid_for(P->v, P->smem, P->total_items, di.sm_count,
                           tune && tune->blocks_per_sm ? tune->blocks_per_sm : 0, &P->grid);
    if (!rc) {
        P->tune.blocks_per_sm = (P->grid + di.sm_count - 1) / di.sm_count;
        rc = check_cuda(cudaStreamSynchronize(st));
    }
    if (!rc) rc = plan_capture(P, di);
    if (rc) {
        cudaStreamSynchronize(st);
        plan_release(P);
        return rc;
    }
    *out = P;
    return WTHETA_OK;
}

}  // namespace wtheta

using namespace wtheta;

extern "C" {

int wtheta_count(const double* a, int64_t n_a, const double* b, int64_t n_b, const double* edges,
                 int32_t K, int32_t is_auto, uint64_t* counts, void* stream) {
    return count_impl(a, n_a, b, n_b, 0, edges, K, is_auto, (unsigned long long*)counts, nullptr,
                      nullptr, (cudaStream_t)stream);
}

int wtheta_count_xyz(const double* a, int64_t n_a, const double* b, int64_t n_b,
                     const double* edges, int32_t K, int32_t is_auto, uint64_t* counts,
                     void* stream) {
    return count_impl(a, n_a, b, n_b, 1, edges, K, is_auto, (unsigned long long*)counts, nullptr,
                      nullptr, (cudaStream_t)stream);
}

int wtheta_count_ex(const double* a, int64_t n_a, const double* b, int64_t n_b, int32_t is_xyz,
                    const double* edges, int32_t K, int32_t is_auto, uint64_t* counts,
                    const wtheta_tune* tune, uint64_t* stats, void* stream) {
    return count_impl(a, n_a, b, n_b, is_xyz, edges, K, is_auto, (unsigned long long*)counts, tune,
                      (unsigned long long*)stats, (cudaStream_t)stream);
}

int wtheta_radec_to_xyz(const double* rd, int64_t n, double* xyz, void* stream) {
    if (n < 0 || (n > 0 && (!rd || !xyz))) return WTHETA_EINVAL;
    if (n == 0) return WTHETA_OK;
    const int threads = 256;
    const int grid = (int)std::min<long long>((n + threads - 1) / threads, 1 << 20);
    k_radec_to_xyz<<<grid, threads, 0, (cudaStream_t)stream>>>(rd, n, xyz, n);
    count_launch();
    return check_cuda(cudaGetLastError());
}

int wtheta_count_xyz_noalloc(const double* a, int64_t n_a, const double* b, int64_t n_b,
                             const double* edges, int32_t K, int32_t is_auto, uint64_t* counts,
                             void* stream) {
    return count_xyz_noalloc_impl(a, n_a, b, n_b, edges, K, is_auto, (unsigned long long*)counts,
                                  (cudaStream_t)stream);
}

int wtheta_batch_plan(const wtheta_catalog_pair* cats, int32_t n_cats, const double* edges,
                      int32_t K, const wtheta_tune* tune, void* stream, wtheta_plan** plan) {
    return batch_plan_impl(cats, n_cats, 0, edges, K, tune, (cudaStream_t)stream, plan);
}

int wtheta_batch_plan_ex(const wtheta_catalog_pair* cats, int32_t n_cats, int32_t coords_are_xyz,
                         const double* edges, int32_t K, const wtheta_tune* tune, void* stream,
                         wtheta_plan** plan) {
    return batch_plan_impl(cats, n_cats, coords_are_xyz, edges, K, tune, (cudaStream_t)stream,
                           plan);
}

int wtheta_batch_run(wtheta_plan* P, uint64_t* counts, void* stream) {
    if (!P || !counts) return WTHETA_EINVAL;
    TraceRange trace("wtheta_batch_run");
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return WTHETA_ECUDA;
    if (dev != P->dev) return WTHETA_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    int rc = check_cuda(cudaGraphLaunch(P->exec, st));
    if (rc) return rc;
    count_launch((unsigned)P->graph_kernels);
    ++P->runs;
    const size_t bytes = (size_t)P->n_cats * 3 * (P->K + 2) * sizeof(unsigned long long);
    return check_cuda(cudaMemcpyAsync(counts, P->d_counts, bytes, cudaMemcpyDeviceToDevice, st));
}

int wtheta_batch_info(const wtheta_plan* P, wtheta_batch_info_t* info) {
    if (!P || !info) return WTHETA_EINVAL;
    std::memset(info, 0, sizeof(*info));
    info->tune = P->tune;
    info->n_items = P->total_items;
    info->pairs = P->pairs;
    const long long T = (long long)P->v->nt * P->v->r;
    info->evaluated_pairs = P->total_items * T * T;
    if (P->runs > 0) {
        // pairs whose squared chord the last run computed (it must have finished)
        unsigned long long st[WTHETA_NSTATS];
        if (cudaDeviceSynchronize() != cudaSuccess ||
            cudaMemcpy(st, P->d_stats, sizeof(st), cudaMemcpyDeviceToHost) != cudaSuccess)
            return WTHETA_ECUDA;
        info->evaluated_pairs = (long long)st[WTHETA_STAT_PAIRS];
    }
    info->n_counts = 3 * P->n_cats;
    info->graph_kernels = P->graph_kernels;
    info->autotune_ms = P->autotune_ms;
    info->autotuned = P->autotuned;
    return WTHETA_OK;
}

int wtheta_batch_free(wtheta_plan* P) {
    if (!P) return WTHETA_EINVAL;
    cudaDeviceSynchronize();
    plan_release(P);
    return WTHETA_OK;
}

int wtheta_count_shard(const double* a, int64_t n_a, const double* b, int64_t n_b,
                       const double* edges, int32_t K, int32_t is_auto, int32_t shard,
                       int32_t n_shards, uint64_t* counts, void* stream) {
    int64_t r0 = 0, r1 = 0;
    if (is_auto) {
        if (b && b != a) return WTHETA_EINVAL;
        if (n_b != n_a && !(b == nullptr && n_b == 0)) return WTHETA_EINVAL;
    }
    int rc = wtheta_shard_rows(n_a, is_auto ? n_a : n_b, is_auto, shard, n_shards, &r0, &r1);
    if (rc) return rc;
    if (!counts || (n_a > 0 && !a) || (!is_auto && n_b > 0 && !b)) return WTHETA_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    const double* rows = a ? a + 2 * r0 : nullptr;
    if (!is_auto)
        return count_impl(rows, r1 - r0, b, n_b, 0, edges, K, 0, (unsigned long long*)counts,
                          nullptr, nullptr, st);
    // rows [r0, r1) of an auto count: the pairs inside the rows, plus the rows
    // against every later point
    rc = count_impl(rows, r1 - r0, nullptr, 0, 0, edges, K, 1, (unsigned long long*)counts,
                    nullptr, nullptr, st);
    if (rc || r1 >= n_a || r1 == r0) return rc;
    unsigned long long* tmp = nullptr;
    if ((rc = dev_malloc_async((void**)&tmp, sizeof(unsigned long long) * (K + 2), st)))
        return rc;
    rc = count_impl(rows, r1 - r0, a + 2 * r1, n_a - r1, 0, edges, K, 0, tmp, nullptr, nullptr,
                    st);
    if (!rc) {
        k_add_counts<<<1, 64, 0, st>>>((unsigned long long*)counts, tmp, K + 2);
        count_launch();
        rc = check_cuda(cudaGetLastError());
    }
    const cudaError_t fe = cudaFreeAsync(tmp, st);
    return rc ? rc : check_cuda(fe);
}

uint64_t wtheta_kernel_launches(void) { return g_launches.load(std::memory_order_relaxed); }

int wtheta_get_error(void* stream, uint32_t* code) {
    if (!code) return WTHETA_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    int rc = check_cuda(cudaStreamSynchronize(st));
    if (rc) return rc;
    unsigned int v = 0, zero = 0;
    if ((rc = check_cuda(cudaMemcpyFromSymbol(&v, g_device_error, sizeof(v))))) return rc;
    if ((rc = check_cuda(cudaMemcpyToSymbol(g_device_error, &zero, sizeof(zero))))) return rc;
    *code = v;
    return WTHETA_OK;
}

int wtheta_inject_alloc_failure(int32_t after) {
    if (after < -1) return WTHETA_EINVAL;
    g_fail_alloc.store(after);
    return WTHETA_OK;
}

int wtheta_count_wtheta(const double* coords_d, int64_t n_d, const double* coords_r,
                        int64_t n_r, int32_t coords_are_xyz, const double* bin_edges_deg,
                        int32_t n_bins, uint64_t* counts, const wtheta_tune* tune,
                        uint64_t* stats, void* stream) {
    return count_wtheta_impl(coords_d, n_d, coords_r, n_r, coords_are_xyz, bin_edges_deg, n_bins,
                             (unsigned long long*)counts, tune, (unsigned long long*)stats,
                             (cudaStream_t)stream);
}

int wtheta_count_wtheta_shard(const double* coords_d, int64_t n_d, const double* coords_r,
                              int64_t n_r, int32_t coords_are_xyz, const double* bin_edges_deg,
                              int32_t n_bins, int32_t shard, int32_t n_shards, uint64_t* counts,
                              const wtheta_tune* tune, uint64_t* stats, void* stream) {
    return count_wtheta_impl(coords_d, n_d, coords_r, n_r, coords_are_xyz, bin_edges_deg, n_bins,
                             (unsigned long long*)counts, tune, (unsigned long long*)stats,
                             (cudaStream_t)stream, shard, n_shards);
}

int wtheta_correlate(const double* data, int64_t n_d, const double* rand, int64_t n_r,
                     const double* edges, int32_t K, uint64_t* counts_out, double* w_out,
                     void* stream) {
    if (n_d < 0 || n_r < 0 || (n_d > 0 && !data) || (n_r > 0 && !rand)) return WTHETA_EINVAL;
    int rc = validate_edges(edges, K);
    if (rc) return rc;
    if (w_out && (n_d < 2 || n_r < 2)) return WTHETA_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t nslot = (size_t)K + 2;
    void* buf = nullptr;
    const size_t bytes = 256 + (size_t)(n_d + n_r) * 16 + 3 * nslot * 8;
    if ((rc = dev_malloc_async(&buf, bytes, st))) return rc;
    unsigned long long* dc = (unsigned long long*)buf;  // 3 (K+2) counts
    double* dd = (double*)((unsigned char*)buf + ((3 * nslot * 8 + 255) / 256) * 256);
    double* dr = dd + 2 * n_d;
    rc = check_cuda(cudaMemcpyAsync(dd, data, (size_t)n_d * 16, cudaMemcpyHostToDevice, st));
    if (!rc) rc = check_cuda(cudaMemcpyAsync(dr, rand, (size_t)n_r * 16, cudaMemcpyHostToDevice, st));
    if (!rc) rc = count_wtheta_impl(dd, n_d, dr, n_r, 0, edges, K, dc, nullptr, nullptr, st);
    uint64_t host_counts[3 * (kMaxBins + 2)];
    if (!rc)
        rc = check_cuda(cudaMemcpyAsync(host_counts, dc, 3 * nslot * 8, cudaMemcpyDeviceToHost, st));
    cudaError_t fe = cudaFreeAsync(buf, st);
    cudaError_t se = cudaStreamSynchronize(st);
    if (!rc) rc = check_cuda(fe);
    if (!rc) rc = check_cuda(se);
    if (rc) return rc;
    if (counts_out) std::memcpy(counts_out, host_counts, 3 * nslot * 8);
    if (w_out)
        rc = wtheta_ls(host_counts, host_counts + nslot, host_counts + 2 * nslot, n_d, n_r, K, w_out);
    return rc;
}

}  // extern "C"
