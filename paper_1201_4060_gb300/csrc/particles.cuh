// Shared definitions of the particle kernels: workspace layout, weights, gather.
// Included by particles.cu (binning, sort, dispatch) and by the gather_*.cu
// translation units that instantiate the gather for each coefficient type and
// order range (split only to compile in parallel).
#pragma once
#include <cuda.h>

#include <cstring>

#include "fixed.cuh"
#include "internal.h"

namespace bs {
namespace gather_impl {

// Tensor map of the coefficient array [3][N][N][N] (FP32, or BF16 with
// elem_bytes = 2) for TMA tile loads: box (z, y, x, component) = (box_z,
// box_y, box_x, 1).  Defined in particles.cu; BSPLINE_OK, or an error if the
// driver's encoder is missing or refuses (the caller then stages with cp.async).
int encode_coef_tmap(CUtensorMap* map, const void* coef, int N, int box_z, int box_y, int box_x, int elem_bytes = 4);

constexpr int kAnchorBits = 10;          // N <= 1024

// One particle's located record: packed first stencil node
// (ax << 20 | ay << 10 | az), the local variable t per axis and the
// particle's original index.  Exactly one 32-byte sector: the placement pass
// writes records to scattered slots, and a record that filled only part of a
// sector would cost a read-modify-write of it in DRAM.
template <typename TR> struct Rec;
template <> struct __align__(32) Rec<float> {
    unsigned cell;
    float t[3];
    unsigned idx;
    unsigned pad[3];    // written as zeros, so that every store covers the whole sector
};
template <> struct __align__(32) Rec<double> {
    unsigned cell;
    unsigned idx;
    double t[3];
};
static_assert(sizeof(Rec<float>) == 32 && sizeof(Rec<double>) == 32, "one sector per record");

// Particles per gather work item: a brick with more particles is split into
// several items, each staging the brick's tile, so no CTA serialises a clump.
constexpr unsigned kChunk = 2048;
// FP64 plans' evaluation: 512, or 42 (three components of 42 particles are the 126 units of a 128-thread CTA;
// gather_fixed).  512 where the call has as many such items as fill the SMs, and the bricks hold so many particles that
// staging and converting a tile for each 42 of them costs more than the long form's idle threads.  Measured, us a call
// with items of 42 / 512, uniform particles, at 128^3 (4096 bricks), particles a brick in brackets: order 2 [8] 64 / 78,
// [48] 127 / 116, [96] 199 / 176; order 4 [30] 149 / 196, [48] 224 / 216, [96] 352 / 258; order 6 [64] 476 / 487, [96] 666 / 530,
// [256] 1487 / 1108; order 8 [64] 917 / 996, [96] 1293 / 1074; clustered, order 4 [64] 245 / 276, [128] 419 / 352.  At 32^3 (64
// bricks), by the call's particles: order 4 65536 74 / 87, 131072 115 / 111, 200000 161 / 116; order 8 131072 372 / 307, 163840
// 452 / 512, 262144 708 / 581.  At 64^3, order 6: 65536 129 / 135, 200000 299 / 273, clustered 129 / 195, 299 / 293.  Both give
// the same bits.
constexpr unsigned kFixedLong = 512, kFixedShort = 42, kFixedLongItems = 384;
inline unsigned item_particles(int dtype, int order, int64_t P, unsigned NB) {
    if (dtype != BSPLINE_F64) return kChunk;
    const int64_t dense = order == 2 ? 32 : (order <= 4 ? 48 : 96);
    return P >= (int64_t)kFixedLong * kFixedLongItems && P >= dense * NB ? kFixedLong : kFixedShort;
}
// The shortest items of a type: what the workspace holds places for, so that a call of fewer particles never needs a
// larger one because its items are of 42 instead of 512.
constexpr unsigned shortest_item(int dtype) { return dtype == BSPLINE_F64 ? kFixedShort : kChunk; }

// Particles of a run of the count pass, and whether it goes by runs, which give each particle its place within its
// brick (launch_bin says why).  Both grow with P: a call of fewer particles needs no larger workspace.
constexpr int64_t kHistLeast = 8192, kHistPerBrick = 64;     // particles in all, particles a brick
inline unsigned count_run_length(int64_t P, int sms) {
    return (unsigned)std::min<int64_t>(8192, std::max<int64_t>(1024, (P / (2 * sms) + 255) / 256 * 256));
}
inline bool counts_by_runs(int64_t P, unsigned NB, int sms) {
    return NB <= std::max(count_run_length(P, sms), 4096u) && P >= std::max<int64_t>(kHistLeast, kHistPerBrick * NB);
}

template <typename TR> struct Ws {
    unsigned* count;    // [NB + 2]  particles per brick; slot NB = invalid positions; NB + 1 = *unsorted
    unsigned* unsorted; // nonzero if positions passed as sorted were not in brick order (count pass)
    unsigned* offset;   // [NB + 3]  start of each brick's sorted segment; [NB] end of the valid
                        //           particles, [NB + 1] end of all, [NB + 2] start of the sparse range
    unsigned* cursor;   // [NB + 1]  next free sorted slot of each brick (starts at offset), without ranks
    unsigned* rank;     // [P]       each particle's place within its brick (count pass by runs; else none)
    unsigned* chunk;    // [NB + 1]  exclusive prefix sum of ceil(count / chunk_len): first work item of a brick
    unsigned* item;     // [NB + ceil(P / shortest)]  brick of each work item (the first chunk[NB] are set)
    long long P;        // particles
    Rec<TR>* s_rec;     // [P]       located records sorted by brick
};

constexpr size_t align_up(size_t v) { return (v + 255) & ~(size_t)255; }

template <typename TR> size_t carve(Ws<TR>* w, void* base, unsigned NB, int64_t P, bool ranks, unsigned shortest = kChunk) {
    size_t off = 0;
    auto take = [&](size_t bytes) {
        void* ptr = base ? (void*)((char*)base + off) : nullptr;
        off += align_up(bytes);
        return ptr;
    };
    w->P = P;
    w->count = (unsigned*)take(sizeof(unsigned) * (NB + 2));
    w->unsorted = base ? w->count + NB + 1 : nullptr;
    w->offset = (unsigned*)take(sizeof(unsigned) * (NB + 3));
    w->cursor = (unsigned*)take(sizeof(unsigned) * (NB + 1));
    w->rank = (unsigned*)take(ranks ? sizeof(unsigned) * P : 0);
    w->chunk = (unsigned*)take(sizeof(unsigned) * (NB + 1));
    w->item = (unsigned*)take(sizeof(unsigned) * (NB + (P + shortest - 1) / shortest));
    w->s_rec = (Rec<TR>*)take(sizeof(Rec<TR>) * P);
    return off;
}

// Periodic grid index of i >= 0 (a single subtraction in the common case i < 2N).
__device__ __forceinline__ int wrap_index(int i, int N) { return i < N ? i : (i < 2 * N ? i - N : i % N); }

// ------------------------------------------------------------------ locate
// For 0 <= s < 2^52: base = floor(s - n/2) and t = (s - n/2) - base rounded to
// float, computed exactly from the bits of s with integer operations (GB300's
// FP64 pipe is narrow: only s = x N / L stays in FP64).  s = fl + fr 2^-sa
// with integer fl and an sa-bit fraction fr; for odd n the half is folded
// into the fraction.  Returns false outside that range.
__device__ __forceinline__ float pow2f(int k) { return __int_as_float((127 + k) << 23); }   // -126 <= k <= 127

__device__ __forceinline__ bool locate_nonneg(double s, int n, long long* base, float* t) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(s);
    if (b >> 63) return false;                                 // negative
    const int e = (int)(b >> 52) - 1023;                       // unbiased exponent
    if (e >= 52) return false;                                 // >= 2^52, Inf or NaN
    const unsigned long long m = (b & ((1ULL << 52) - 1)) | (1ULL << 52);
    const long long hfl = n >> 1;                              // floor(n / 2)
    if (e < 0) {                                               // s in [0, 1)
        // below 2^-60 (or subnormal) s is 0 to the FP32 accuracy of the weights
        const float sf = (e < -60) ? 0.f : __ull2float_rn(m) * pow2f(e - 52);
        if (!(n & 1)) {
            *base = -hfl;
            *t = sf;
        } else if (e == -1) {                                  // s in [0.5, 1): s - 1/2 = (m - 2^52) 2^-53
            *base = -hfl;
            *t = __ull2float_rn(m - (1ULL << 52)) * pow2f(-53);
        } else {                                               // s in [0, 0.5)
            *base = -hfl - 1;
            *t = sf + 0.5f;
        }
        return true;
    }
    const int sa = 52 - e;                                     // fraction bits, 1..52
    const long long fl = (long long)(m >> sa);
    const unsigned long long fr = m & ((1ULL << sa) - 1);
    if (!(n & 1)) {
        *base = fl - hfl;
        *t = __ull2float_rn(fr) * pow2f(-sa);
    } else {
        const unsigned long long hb = 1ULL << (sa - 1);        // one half in the fraction's units
        if (fr >= hb) {
            *base = fl - hfl;
            *t = __ull2float_rn(fr - hb) * pow2f(-sa);
        } else {
            *base = fl - hfl - 1;
            *t = __ull2float_rn(fr + hb) * pow2f(-sa);
        }
    }
    return true;
}

// First stencil node modulo N (N a power of two, or 3 times one).
__device__ __forceinline__ unsigned wrap_anchor(long long a, int N) {
    if ((N & (N - 1)) == 0) return (unsigned)(a & (long long)(N - 1));
    long long r = a % N;
    return (unsigned)(r < 0 ? r + N : r);
}

// One axis of Eq. alg-int-6: the first stencil node modulo N and t, from s = x N / L; false for a
// non-finite s or one with no fractional bits left.
template <typename TR>
__device__ __forceinline__ bool locate_axis(double s, int N, int order, unsigned* anchor, TR* t) {
    if constexpr (sizeof(TR) == 4) {
        long long base;
        if (locate_nonneg(s, order, &base, t)) {
            *anchor = wrap_anchor(base + 1, N);
            return true;
        }
    }
    const double sh = s - 0.5 * order;
    if (!(fabs(sh) < 4.0e15)) {          // NaN, Inf, or no fractional bits left
        *anchor = 0;
        *t = 0;
        return false;
    }
    const double f = floor(sh);
    *t = (TR)(sh - f);
    *anchor = wrap_anchor((long long)f + 1, N);
    return true;
}

// Locate one particle (Eq. alg-int-6): its brick key and record; the key is NB
// for a non-finite position or one with no fractional bits left.
template <typename TR>
__device__ __forceinline__ unsigned locate_particle(const double* __restrict__ x, long long p, int N, double scale,
                                                    int order, const BrickGrid& g, Rec<TR>* r) {
    const unsigned NB = g.NB;
    unsigned anc[3];
    TR tt[3];
    bool ok = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) ok = locate_axis<TR>(x[3 * p + a] * scale, N, order, &anc[a], &tt[a]) && ok;
    if (!ok) return NB;
    r->cell = (anc[0] << (2 * kAnchorBits)) | (anc[1] << kAnchorBits) | anc[2];
    r->t[0] = tt[0];
    r->t[1] = tt[1];
    r->t[2] = tt[2];
    return ((anc[0] >> g.bshift) * (unsigned)g.nby + anc[1] / (unsigned)g.by) * (unsigned)g.nbz + (anc[2] >> g.bshift);
}

// Count pass of a run of n particles by one CTA through a shared-memory histogram: key(i) gives the brick of
// the run's i-th particle (each warp calls it for 32 consecutive i, all lanes; i >= n must return any key
// and is not counted), count[] receives the run's counts, and rank[i] each particle's place within its
// brick.  A global atomic per brick and run, on consecutive addresses, replaces one per particle and pass at
// random ones: the placement pass then needs none.  s: NB + 1 + n words.
constexpr unsigned kHistKeyBits = 14;                   // NB < 2^14, n <= 2^14
template <typename Key>
__device__ __forceinline__ void count_run(unsigned* s, unsigned NB, unsigned n, unsigned* __restrict__ count,
                                          unsigned* __restrict__ rank, Key key) {
    unsigned* s_key = s + NB + 1;
    for (unsigned b = threadIdx.x; b <= NB; b += blockDim.x) s[b] = 0;
    __syncthreads();
    for (unsigned i = threadIdx.x; i < ((n + 31u) & ~31u); i += blockDim.x) {
        const unsigned k = key(i);
        if (i < n) s_key[i] = (atomicAdd(&s[k], 1u) << kHistKeyBits) | k;
    }
    __syncthreads();
    for (unsigned b = threadIdx.x; b <= NB; b += blockDim.x) {
        const unsigned h = s[b];
        if (h) s[b] = atomicAdd(&count[b], h);
    }
    __syncthreads();
    for (unsigned i = threadIdx.x; i < n; i += blockDim.x) {
        const unsigned v = s_key[i];
        rank[i] = s[v & ((1u << kHistKeyBits) - 1u)] + (v >> kHistKeyBits);
    }
    __syncthreads();
}

// ------------------------------------------------------------------ weights
// v[m] = M_k(t + m), m = 0..k-1, for the cardinal B-spline of order k.
// Node j (0-based, j = 0 leftmost) of an order-n stencil has weight
// B(t + n/2 - 1 - j) = M_n(t + n - 1 - j) and derivative
// M_{n-1}(t + n - 1 - j) - M_{n-1}(t + n - 2 - j).
template <int n, typename A>
__device__ __forceinline__ void bspline_weights(A t, A (&w)[n], A (&dw)[n]) {
    A v[n];
    v[0] = A(1);
#pragma unroll
    for (int m = 1; m < n; ++m) v[m] = A(0);
#pragma unroll
    for (int k = 2; k <= n - 1; ++k) {
        const A inv = A(1) / A(k - 1);
#pragma unroll
        for (int m = k - 1; m >= 0; --m) {
            const A left = (m > 0) ? v[m - 1] : A(0);
            v[m] = ((t + A(m)) * v[m] + (A(k - m) - t) * left) * inv;
        }
    }
    // v = order n-1 values; one more step for order n, derivative by differencing
    const A inv = A(1) / A(n - 1);
#pragma unroll
    for (int j = 0; j < n; ++j) {
        const int m = n - 1 - j;
        const A vm = (m <= n - 2) ? v[m] : A(0);
        const A vl = (m >= 1) ? v[m - 1] : A(0);
        w[j] = ((t + A(m)) * vm + (A(n - m) - t) * vl) * inv;
        dw[j] = vm - vl;
    }
}

// ------------------------------------------------------------------ gather
// Coefficient tile of one brick: (BX + ORD - 1) x (BY + ORD - 1) x (BZ + ORD - 1)
// nodes per component, [c][x][y][z] with z fastest and z rows of PZ entries
// (FP32/BF16: padded to a multiple of 4 so every row starts 16-byte
// aligned), periodic wrap of the grid indices on staging.  FP32 and BF16
// coefficients are staged as FP32 (BF16 widened on load).
template <typename CT> struct TileT { using T = float; };
template <> struct TileT<double> { using T = double; };

template <typename CT> __device__ __forceinline__ typename TileT<CT>::T widen(CT v) { return v; }
template <> __device__ __forceinline__ float widen<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

// BYO: brick y extent other than the plan's default (batches tune it; 0 = brick_y).
template <typename CT, int ORD, int BYO = 0> struct Shape {
    static constexpr bool F64 = sizeof(CT) == 8;
    static constexpr int BX = brick_x(F64 ? BSPLINE_F64 : BSPLINE_F32);
    static constexpr int BY = BYO ? BYO : brick_y(F64 ? BSPLINE_F64 : BSPLINE_F32, ORD);
    static constexpr int BZ = BX;
    static constexpr int EX = BX + ORD - 1, EY = BY + ORD - 1, EZ = BZ + ORD - 1;
    static constexpr int PZ = F64 ? EZ : ((EZ + 3) & ~3);
    // strides of y, x and the component; FP32 tiles pad the component to 128 bytes (TMA destinations)
    static constexpr int SY = PZ, SX = EY * PZ, TS = F64 ? EX * SX : ((EX * SX + 31) & ~31);
};

template <int ORD, typename CT, int BYO = 0>
constexpr size_t tile_bytes() {
    return sizeof(typename TileT<CT>::T) * 3 * (size_t)Shape<CT, ORD, BYO>::TS;
}

// Brick index -> first cell of the brick.
template <int BX, int BY, int BZ>
__device__ __forceinline__ void brick_origin(unsigned brick, const BrickGrid& g, int* x0, int* y0, int* z0) {
    const unsigned bz = brick % (unsigned)g.nbz, t = brick / (unsigned)g.nbz;
    *z0 = (int)bz * BZ;
    *y0 = (int)(t % (unsigned)g.nby) * BY;
    *x0 = (int)(t / (unsigned)g.nby) * BX;
}


__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}
// 16 bytes, cached in L2 only (each tile is read once per work item).
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// ---- TMA tile loads completing on a shared-memory mbarrier
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");   // visible to the async proxy
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_test(unsigned long long* bar, unsigned parity) {
    unsigned done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0u;
}
// Box at coordinates (z, y, x, c) of `map` into shared memory at dst (128-byte aligned).
__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int z, int y, int x, int c,
                                            unsigned long long* bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5}], [%6];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<unsigned long long>(map)), "r"(z), "r"(y), "r"(x), "r"(c), "r"(smem_u32(bar))
        : "memory");
}
// Bounded wait for phase `parity` of the mbarrier (about a second of polls): false if it ran out.
__device__ __forceinline__ bool mbar_wait_bounded(unsigned long long* bar, unsigned parity) {
    for (long long it = 0; it < (1LL << 22); ++it) {
        if (mbar_test(bar, parity)) return true;
        __nanosleep(64);
    }
    return false;
}

// Copy the brick's tile into shared memory, one z-row per warp step: lane =
// z offset (lanes >= EZ idle).  Rows are walked in (c, ix, iy) order; indices
// wrap periodically.  Same-type coefficients go through cp.async (no register
// round trip); BF16 is widened to FP32 through registers.  The caller
// synchronises the CTA after cp_async_wait_all.
template <int ORD, typename CT, int BYO = 0>
__device__ __forceinline__ void stage_tile(typename TileT<CT>::T* tile, const CT* __restrict__ coef, int N, int x0,
                                           int y0, int z0) {
    using TT = typename TileT<CT>::T;
    using S = Shape<CT, ORD, BYO>;
    static_assert(S::EZ <= 32, "one z-row per warp step");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (lane >= S::EZ) return;
    const int gz = wrap_index(z0 + lane, N);
    // planes (c, ix): 3 EX of them, each EY rows along y; warps take planes round-robin
    for (int pl = warp; pl < 3 * S::EX; pl += nw) {
        const int c = pl / S::EX, ix = pl - c * S::EX;
        const CT* plane = coef + ((size_t)c * N + wrap_index(x0 + ix, N)) * (size_t)N * N + gz;
        TT* dst = tile + (size_t)c * S::TS + (size_t)ix * S::SX + lane;
        auto copy = [&](int iy, const CT* s) {
            if constexpr (sizeof(CT) == sizeof(TT)) {
                if constexpr (sizeof(CT) == 4) cp_async4(dst + iy * S::SY, s);
                else cp_async8(dst + iy * S::SY, s);
            } else {
                dst[iy * S::SY] = widen<CT>(*s);
            }
        };
        if (N >= S::EY) {
            // rows y0.. up to the end of the period advance by N; the rest wrap to row 0
            const int nrun = min(S::EY, N - y0);
            const CT* s = plane + (size_t)y0 * N;
#pragma unroll 7
            for (int iy = 0; iy < nrun; ++iy, s += N) copy(iy, s);
            s = plane;
            for (int iy = nrun; iy < S::EY; ++iy, s += N) copy(iy, s);
        } else {
            for (int iy = 0; iy < S::EY; ++iy) copy(iy, plane + (size_t)wrap_index(y0 + iy, N) * N);
        }
    }
}

// FP32 tiles with 16-byte copies: a tile row is PZ / 4 chunks of 4
// coefficients, 16-byte aligned in both memories (z0 and N are multiples of
// 4, so a chunk never straddles the periodic wrap).  Within a (c, ix) plane
// the lane -> (row, chunk) assignment and its offsets are the same for every
// plane, so they are computed once.
template <int ORD, int BYO = 0>
__device__ __forceinline__ void stage_tile16(float* tile, const float* __restrict__ coef, int N, int x0, int y0,
                                             int z0) {
    using S = Shape<float, ORD, BYO>;
    constexpr int CH = S::PZ / 4;                     // chunks per row
    constexpr int PER = S::EY * CH;                   // chunks per plane
    constexpr int NI = (PER + 31) / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int goff[NI], soff[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int f = lane + 32 * i;
        const int iy = f / CH, ch = f - iy * CH;
        goff[i] = f < PER ? wrap_index(y0 + iy, N) * N + wrap_index(z0 + 4 * ch, N) : -1;
        soff[i] = iy * S::SY + 4 * ch;
    }
    for (int pl = warp; pl < 3 * S::EX; pl += nw) {
        const int c = pl / S::EX, ix = pl - c * S::EX;
        const float* plane = coef + ((size_t)c * N + wrap_index(x0 + ix, N)) * (size_t)N * N;
        float* dst = tile + (size_t)c * S::TS + (size_t)ix * S::SX;
#pragma unroll
        for (int i = 0; i < NI; ++i)
            if (goff[i] >= 0) cp_async16(dst + soff[i], plane + goff[i]);
    }
}

// BF16 coefficients: 16-byte loads of 8 values (rows start at z0, a multiple
// of 16, and N is a multiple of 8, so a chunk never straddles the wrap),
// widened to FP32 in registers and stored as two 16-byte words.  All of a
// lane's loads of a plane are issued together, and the next plane's before
// this plane's stores (registers stand in for the asynchronous copy).
template <int ORD, int BYO = 0>
__device__ __forceinline__ void stage_tile_bf16(float* tile, const __nv_bfloat16* __restrict__ coef, int N, int x0,
                                                int y0, int z0) {
    using S = Shape<__nv_bfloat16, ORD, BYO>;
    constexpr int CH = (S::PZ + 7) / 8;               // chunks of 8 per row (the last may overhang the pitch)
    constexpr int PER = S::EY * CH;
    constexpr int NI = (PER + 31) / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int goff[NI], soff[NI], nst[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int f = lane + 32 * i;
        const int iy = f / CH, ch = f - iy * CH;
        goff[i] = f < PER ? wrap_index(y0 + iy, N) * N + wrap_index(z0 + 8 * ch, N) : -1;
        soff[i] = iy * S::SY + 8 * ch;
        nst[i] = (S::PZ - 8 * ch) >= 8 ? 2 : 1;       // 16-byte stores that stay inside the row pitch
    }
    // a warp's planes (c, ix) in turn, the next plane's loads in flight while this one is widened and stored
    auto load = [&](int pl, uint4 (&v)[NI]) {
        const int c = pl / S::EX, ix = pl - c * S::EX;
        const __nv_bfloat16* plane = coef + ((size_t)c * N + wrap_index(x0 + ix, N)) * (size_t)N * N;
#pragma unroll
        for (int i = 0; i < NI; ++i)
            if (goff[i] >= 0) v[i] = __ldg(reinterpret_cast<const uint4*>(plane + goff[i]));
    };
    uint4 v[NI], vn[NI];
    if (warp < 3 * S::EX) load(warp, vn);
    for (int pl = warp; pl < 3 * S::EX; pl += nw) {
#pragma unroll
        for (int i = 0; i < NI; ++i) v[i] = vn[i];
        if (pl + nw < 3 * S::EX) load(pl + nw, vn);
        const int c = pl / S::EX, ix = pl - c * S::EX;
        float* dst = tile + (size_t)c * S::TS + (size_t)ix * S::SX;
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            if (goff[i] < 0) continue;
            const unsigned w4[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
            float f[8];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                f[2 * q] = __uint_as_float(w4[q] << 16);             // bf16 -> fp32: the high half of the word
                f[2 * q + 1] = __uint_as_float(w4[q] & 0xffff0000u);
            }
            *reinterpret_cast<float4*>(dst + soff[i]) = make_float4(f[0], f[1], f[2], f[3]);
            if (nst[i] == 2) *reinterpret_cast<float4*>(dst + soff[i] + 4) = make_float4(f[4], f[5], f[6], f[7]);
        }
    }
}

// BF16 coefficients stay BF16 in shared memory, in two copies of the tile
// ([c][x][y][z], rows of PZ elements, 16-byte aligned): copy A holds element
// z of a row at z, copy B holds element z + 1 at z.  A stencil line of ORD
// values starting at tile z = oz is then ceil(ORD / 2) aligned 32-bit words:
// copy A from word oz / 2 if oz is even, copy B from word (oz - 1) / 2 if it
// is odd.  Each word carries two consecutive values (the lower z in its low
// half), widened to FP32 in registers, so the contraction reads half the
// shared-memory bytes of an FP32 tile with the same FP32 arithmetic.
template <int ORD, int BYO = 0> struct Bf16Pair {
    using S = Shape<__nv_bfloat16, ORD, BYO>;
    static constexpr int EX = S::EX, EY = S::EY, EZ = S::EZ;
    static constexpr int PZ = (EZ + 7) & ~7;            // elements per row: 16-byte rows
    static constexpr int SYW = PZ / 2, SXW = EY * SYW;  // words per row, per x-plane
    static constexpr int TSW = (EX * SXW + 31) & ~31;   // words per component
    static constexpr int COPYW = 3 * TSW;               // words per copy
    static constexpr int NWL = (ORD + 1) / 2;           // words per stencil line
    static constexpr size_t bytes = 2 * sizeof(unsigned) * (size_t)COPYW;
};

// Copy A of a brick: 16-byte cp.async chunks of 8 values (z0 is a multiple of
// 16 and N of 8, so no chunk straddles the periodic wrap); element by element
// below N = 16.  The caller waits for the copies and synchronises.
template <int ORD, int BYO>
__device__ __forceinline__ void stage_bf16_copy_a(unsigned* words, const __nv_bfloat16* __restrict__ coef, int N,
                                                  int x0, int y0, int z0) {
    using T = Bf16Pair<ORD, BYO>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (N >= 16) {
        constexpr int CH = T::PZ / 8;                   // chunks per row
        constexpr int PER = T::EY * CH;                 // chunks per (c, x) plane
        constexpr int NI = (PER + 31) / 32;
        int goff[NI], soff[NI];
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const int f = lane + 32 * i;
            const int iy = f / CH, ch = f - iy * CH;
            goff[i] = f < PER ? wrap_index(y0 + iy, N) * N + wrap_index(z0 + 8 * ch, N) : -1;
            soff[i] = iy * T::SYW + 4 * ch;
        }
        for (int pl = warp; pl < 3 * T::EX; pl += nw) {
            const int c = pl / T::EX, ix = pl - c * T::EX;
            const __nv_bfloat16* plane = coef + ((size_t)c * N + wrap_index(x0 + ix, N)) * (size_t)N * N;
            unsigned* dst = words + (size_t)c * T::TSW + (size_t)ix * T::SXW;
#pragma unroll
            for (int i = 0; i < NI; ++i)
                if (goff[i] >= 0) cp_async16(dst + soff[i], plane + goff[i]);
        }
    } else {
        __nv_bfloat16* e = reinterpret_cast<__nv_bfloat16*>(words);
        for (int k = threadIdx.x; k < 3 * T::EX * T::EY * T::PZ; k += blockDim.x) {
            const int z = k % T::PZ, r = k / T::PZ, iy = r % T::EY, ix = (r / T::EY) % T::EX, c = r / (T::EY * T::EX);
            e[2 * ((size_t)c * T::TSW + (size_t)ix * T::SXW + (size_t)iy * T::SYW) + z] =
                coef[(((size_t)c * N + wrap_index(x0 + ix, N)) * N + wrap_index(y0 + iy, N)) * N + wrap_index(z0 + z, N)];
        }
    }
}

// Copy B from copy A: word j = (A[2j + 1], A[2j + 2]), four words per
// thread and step (16-byte accesses).  The upper value of a row's last word
// comes from the next row (or is zero at the end of the copy): it is never
// part of a stencil line.  Call after copy A is complete and visible; ends
// with a barrier.
template <int ORD, int BYO>
__device__ __forceinline__ void build_bf16_copy_b(unsigned* words) {
    using T = Bf16Pair<ORD, BYO>;
    static_assert(T::COPYW % 4 == 0, "16-byte steps");
    const uint4* a4 = reinterpret_cast<const uint4*>(words);
    uint4* b4 = reinterpret_cast<uint4*>(words + T::COPYW);
    for (int v = threadIdx.x; v < T::COPYW / 4; v += blockDim.x) {
        const uint4 a = a4[v];
        const unsigned nx = (4 * v + 4 < T::COPYW) ? words[4 * v + 4] : 0u;
        b4[v] = make_uint4(__byte_perm(a.x, a.y, 0x5432), __byte_perm(a.y, a.z, 0x5432), __byte_perm(a.z, a.w, 0x5432),
                           __byte_perm(a.w, nx, 0x5432));
    }
    __syncthreads();
}


__device__ __forceinline__ float bf16_lo(unsigned w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(unsigned w) { return __uint_as_float(w & 0xffff0000u); }

// TMA staging of an FP32 brick away from the periodic seams: thread 0 arms the
// mbarrier and issues one box (PZ, EY, EX, 1) per component; the boxes never
// leave the grid there (z0 <= N - 32 when z0 + EZ <= N), and the padding z
// rows beyond EZ are never read.  Returns whether the brick was staged this
// way (the caller stages the others with cp.async).  use_tma: 0 = never,
// kTmaOn = interior bricks, kTmaArmOnly = arm the barrier for the tile's bytes
// but issue no copy (test hook: the wait then runs out with nothing in flight).
constexpr int kTmaOn = 1, kTmaArmOnly = 2;
template <int ORD, typename CT, int BYO = 0>
__device__ __forceinline__ bool stage_tile_tma(float* tile, const CUtensorMap* map, unsigned long long* bar, int N,
                                               int x0, int y0, int z0, int use_tma) {
    using S = Shape<CT, ORD, BYO>;
    const bool tma = sizeof(CT) == 4 && use_tma && x0 + S::EX <= N && y0 + S::EY <= N && z0 + S::EZ <= N;
    if (tma && threadIdx.x == 0) {
        mbar_init(bar, 1);
        mbar_expect_tx(bar, 3u * S::PZ * S::EY * S::EX * (unsigned)sizeof(float));
        if (use_tma != kTmaArmOnly) {
#pragma unroll
            for (int c = 0; c < 3; ++c) tma_load_4d(tile + c * S::TS, map, z0, y0, x0, c, bar);
        }
    }
    return tma;
}

// TMA staging of copy A of a BF16 pair tile away from the periodic seams (as
// stage_tile_tma: one box (PZ, EY, EX, 1) per component, into the component's
// 128-byte aligned words); returns whether the brick was staged this way.
template <int ORD, int BYO>
__device__ __forceinline__ bool stage_bf16_tma(unsigned* words, const CUtensorMap* map, unsigned long long* bar,
                                               int N, int x0, int y0, int z0, int use_tma) {
    using T = Bf16Pair<ORD, BYO>;
    const bool tma = use_tma && x0 + T::EX <= N && y0 + T::EY <= N && z0 + T::EZ <= N;
    if (tma && threadIdx.x == 0) {
        mbar_init(bar, 1);
        mbar_expect_tx(bar, 3u * T::PZ * T::EY * T::EX * 2u);
        if (use_tma != kTmaArmOnly) {
#pragma unroll
            for (int c = 0; c < 3; ++c) tma_load_4d(words + c * T::TSW, map, z0, y0, x0, c, bar);
        }
    }
    return tma;
}

// Every thread waits for the TMA tile (observing the barrier's phase makes the
// bytes visible to it).  A wait that runs out (about a second) sets *flag,
// waits once more for the copies in flight, and returns false for the whole
// CTA, which then abandons its item.  Call after a barrier that follows the
// mbarrier's initialisation.
__device__ __forceinline__ bool tma_tile_wait(unsigned long long* bar, unsigned long long* flag) {
    const bool timed_out = __syncthreads_or(mbar_wait_bounded(bar, 0) ? 0 : 1) != 0;
    if (timed_out) {
        if (threadIdx.x == 0) atomicOr(flag, 1ULL);
        mbar_wait_bounded(bar, 0);
        return false;
    }
    return true;
}

// Outputs of an abandoned work item: NaN for each of its particles, so that a
// time-out never leaves stale values behind (the status word says why).
template <typename TR, typename AT>
__device__ __forceinline__ void fill_nan_item(const Ws<TR>& w, unsigned c0, unsigned n, AT* __restrict__ out_u,
                                              AT* __restrict__ out_grad, int ncomp_u) {
    const AT nan = (AT)NAN;
    for (unsigned i = threadIdx.x; i < n; i += blockDim.x) {
        const size_t idx = w.s_rec[c0 + i].idx;
        if (out_u) {
            for (int k = 0; k < ncomp_u; ++k) out_u[(size_t)ncomp_u * idx + k] = nan;
        }
        if (out_grad) {
#pragma unroll
            for (int k = 0; k < 9; ++k) out_grad[9 * idx + k] = nan;
        }
    }
}

template <int ORD, typename CT, int BYO = 0>
__device__ __forceinline__ void stage_brick(typename TileT<CT>::T* tile, const CT* __restrict__ coef, int N, int x0,
                                            int y0, int z0) {
    if constexpr (sizeof(CT) == 4) {
        if (N >= 16) {
            stage_tile16<ORD, BYO>(tile, coef, N, x0, y0, z0);
            return;
        }
    } else if constexpr (sizeof(CT) == 2) {
        if (N >= 16) {
            stage_tile_bf16<ORD, BYO>(tile, coef, N, x0, y0, z0);
            return;
        }
    }
    stage_tile<ORD, CT, BYO>(tile, coef, N, x0, y0, z0);
}

// Packed two-way FP32 contraction (fma.rn.f32x2) of one component:
// adjacent y-lines jy, jy + 1 are contracted along z together (their loads
// form the pair, the z weight is duplicated), and their y-sums are kept as
// (even, odd) pairs that are added at the end of each x-plane.  The
// sums are grouped by parity of jy.
// ld(jx, jy, jz) gives the coefficient at stencil node (jx, jy, jz): the
// staged gather reads its shared-memory tile, the direct gather global
// memory, with the same arithmetic in the same order, so the two agree bit
// for bit.
template <int ORD> struct PairWeights {
    static constexpr int NP = ORD / 2;                // pairs of y-lines
    float2 wz2[ORD], dwz2[ORD], wyp[NP > 0 ? NP : 1], dwyp[NP > 0 ? NP : 1];
    __device__ __forceinline__ PairWeights(const float (&wz)[ORD], const float (&dwz)[ORD], const float (&wy)[ORD],
                                           const float (&dwy)[ORD]) {
#pragma unroll
        for (int j = 0; j < ORD; ++j) {
            wz2[j] = make_float2(wz[j], wz[j]);
            dwz2[j] = make_float2(dwz[j], dwz[j]);
        }
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            wyp[p] = make_float2(wy[2 * p], wy[2 * p + 1]);
            dwyp[p] = make_float2(dwy[2 * p], dwy[2 * p + 1]);
        }
    }
};

// One x-row of the contraction: ldr(jy, jz) gives the coefficient at
// (jy, jz) of the row; returns the row's sums s00 = sum_y wy sum_z wz c, s10
// with dwy, s01 with dwz.
template <int ORD, bool GRAD, typename LDR>
__device__ __forceinline__ void row_x2(LDR ldr, const PairWeights<ORD>& pw, const float (&wy)[ORD],
                                       const float (&dwy)[ORD], const float (&wz)[ORD], const float (&dwz)[ORD],
                                       float* s00, float* s10, float* s01) {
    constexpr int NP = ORD / 2;
    float2 y00 = make_float2(0.f, 0.f), y10 = y00, y01 = y00;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        float2 z0 = make_float2(0.f, 0.f), z1 = z0;
#pragma unroll
        for (int jz = 0; jz < ORD; ++jz) {
            const float2 a = make_float2(ldr(2 * p, jz), ldr(2 * p + 1, jz));
            z0 = __ffma2_rn(pw.wz2[jz], a, z0);
            if (GRAD) z1 = __ffma2_rn(pw.dwz2[jz], a, z1);
        }
        y00 = __ffma2_rn(pw.wyp[p], z0, y00);
        if (GRAD) {
            y10 = __ffma2_rn(pw.dwyp[p], z0, y10);
            y01 = __ffma2_rn(pw.wyp[p], z1, y01);
        }
    }
    if constexpr (ORD % 2 == 1) {                   // the unpaired last line
        float z0 = 0.f, z1 = 0.f;
#pragma unroll
        for (int jz = 0; jz < ORD; ++jz) {
            const float a = ldr(ORD - 1, jz);
            z0 = fmaf(wz[jz], a, z0);
            if (GRAD) z1 = fmaf(dwz[jz], a, z1);
        }
        y00.x = fmaf(wy[ORD - 1], z0, y00.x);
        if (GRAD) {
            y10.x = fmaf(dwy[ORD - 1], z0, y10.x);
            y01.x = fmaf(wy[ORD - 1], z1, y01.x);
        }
    }
    *s00 = y00.x + y00.y;
    *s10 = y10.x + y10.y;
    *s01 = y01.x + y01.y;
}

// row_x2 on a BF16 pair tile: line jy of the x-row starts at word row0 + jy
// SYW; the same terms in the same order as row_x2 (pairs of y-lines, z
// ascending), each value the exact FP32 value of its BF16 coefficient.
template <int ORD, bool GRAD, int SYW>
__device__ __forceinline__ void row_x2_words(const unsigned* __restrict__ row0, const PairWeights<ORD>& pw,
                                             const float (&wy)[ORD], const float (&dwy)[ORD], const float (&wz)[ORD],
                                             const float (&dwz)[ORD], float* s00, float* s10, float* s01) {
    constexpr int NP = ORD / 2, NWL = (ORD + 1) / 2;
    float2 y00 = make_float2(0.f, 0.f), y10 = y00, y01 = y00;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        const unsigned* l0 = row0 + (2 * p) * SYW;
        const unsigned* l1 = l0 + SYW;
        float2 z0 = make_float2(0.f, 0.f), z1 = z0;
#pragma unroll
        for (int k = 0; k < NWL; ++k) {
            const unsigned a = l0[k], b = l1[k];
            const float2 v0 = make_float2(bf16_lo(a), bf16_lo(b));
            z0 = __ffma2_rn(pw.wz2[2 * k], v0, z0);
            if (GRAD) z1 = __ffma2_rn(pw.dwz2[2 * k], v0, z1);
            if (2 * k + 1 < ORD) {
                const float2 v1 = make_float2(bf16_hi(a), bf16_hi(b));
                z0 = __ffma2_rn(pw.wz2[2 * k + 1], v1, z0);
                if (GRAD) z1 = __ffma2_rn(pw.dwz2[2 * k + 1], v1, z1);
            }
        }
        y00 = __ffma2_rn(pw.wyp[p], z0, y00);
        if (GRAD) {
            y10 = __ffma2_rn(pw.dwyp[p], z0, y10);
            y01 = __ffma2_rn(pw.wyp[p], z1, y01);
        }
    }
    if constexpr (ORD % 2 == 1) {                   // the unpaired last line
        const unsigned* l = row0 + (ORD - 1) * SYW;
        float z0 = 0.f, z1 = 0.f;
#pragma unroll
        for (int k = 0; k < NWL; ++k) {
            const unsigned a = l[k];
            z0 = fmaf(wz[2 * k], bf16_lo(a), z0);
            if (GRAD) z1 = fmaf(dwz[2 * k], bf16_lo(a), z1);
            if (2 * k + 1 < ORD) {
                z0 = fmaf(wz[2 * k + 1], bf16_hi(a), z0);
                if (GRAD) z1 = fmaf(dwz[2 * k + 1], bf16_hi(a), z1);
            }
        }
        y00.x = fmaf(wy[ORD - 1], z0, y00.x);
        if (GRAD) {
            y10.x = fmaf(dwy[ORD - 1], z0, y10.x);
            y01.x = fmaf(wy[ORD - 1], z1, y01.x);
        }
    }
    *s00 = y00.x + y00.y;
    *s10 = y10.x + y10.y;
    *s01 = y01.x + y01.y;
}

// Accumulation of one x-row's sums into u and the gradient.
template <bool GRAD>
__device__ __forceinline__ void add_row(float wxj, float dwxj, float s00, float s10, float s01, float* u, float* gx,
                                        float* gy, float* gz) {
    *u = fmaf(wxj, s00, *u);
    if (GRAD) {
        *gx = fmaf(dwxj, s00, *gx);
        *gy = fmaf(wxj, s10, *gy);
        *gz = fmaf(wxj, s01, *gz);
    }
}

template <int ORD, bool GRAD, typename LD>
__device__ __forceinline__ void contract_x2(LD ld, const PairWeights<ORD>& pw, const float (&wx)[ORD],
                                            const float (&dwx)[ORD], const float (&wy)[ORD], const float (&dwy)[ORD],
                                            const float (&wz)[ORD], const float (&dwz)[ORD], float dscale,
                                            float* __restrict__ out_u, float* __restrict__ out_grad) {
    float u = 0.f, gx = 0.f, gy = 0.f, gz = 0.f;
#pragma unroll
    for (int jx = 0; jx < ORD; ++jx) {
        float s00, s10, s01;
        row_x2<ORD, GRAD>([&](int jy, int jz) { return ld(jx, jy, jz); }, pw, wy, dwy, wz, dwz, &s00, &s10, &s01);
        add_row<GRAD>(wx[jx], dwx[jx], s00, s10, s01, &u, &gx, &gy, &gz);
    }
    *out_u = u;
    if (GRAD) {
        out_grad[0] = gx * dscale;
        out_grad[1] = gy * dscale;
        out_grad[2] = gz * dscale;
    }
}

// All three components of one particle from the staged tile (weights once).
template <int ORD, bool GRAD, int SX, int SY, int TS>
__device__ __forceinline__ void eval_particle_x2(const float* __restrict__ base, float tx, float ty, float tz,
                                                 float dscale, float* __restrict__ out_u,
                                                 float* __restrict__ out_grad) {
    float wx[ORD], dwx[ORD], wy[ORD], dwy[ORD], wz[ORD], dwz[ORD];
    bspline_weights<ORD, float>(tx, wx, dwx);
    bspline_weights<ORD, float>(ty, wy, dwy);
    bspline_weights<ORD, float>(tz, wz, dwz);
    const PairWeights<ORD> pw(wz, dwz, wy, dwy);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float* tc = base + c * TS;
        contract_x2<ORD, GRAD>([&](int jx, int jy, int jz) { return tc[jx * SX + jy * SY + jz]; }, pw, wx, dwx, wy,
                               dwy, wz, dwz, dscale, &out_u[c], &out_grad[3 * c]);
    }
}

// One component of eval_particle_x2; base points at the component's first stencil node.
template <int ORD, bool GRAD, int SX, int SY>
__device__ __forceinline__ void eval_component_x2(const float* __restrict__ base, float tx, float ty, float tz,
                                                  float dscale, float* __restrict__ out_u,
                                                  float* __restrict__ out_grad) {
    float wx[ORD], dwx[ORD], wy[ORD], dwy[ORD], wz[ORD], dwz[ORD];
    bspline_weights<ORD, float>(tx, wx, dwx);
    bspline_weights<ORD, float>(ty, wy, dwy);
    bspline_weights<ORD, float>(tz, wz, dwz);
    const PairWeights<ORD> pw(wz, dwz, wy, dwy);
    contract_x2<ORD, GRAD>([&](int jx, int jy, int jz) { return base[jx * SX + jy * SY + jz]; }, pw, wx, dwx, wy,
                           dwy, wz, dwz, dscale, out_u, out_grad);
}

// Components c0..c0+NC-1 of one particle from a BF16 pair tile (weights once);
// base = the particle's first stencil word of component 0 in its copy.
template <int ORD, bool GRAD, typename T, int NC>
__device__ __forceinline__ void eval_bf16(const unsigned* __restrict__ base, int c0, float tx, float ty, float tz,
                                          float dscale, float* __restrict__ out_u, float* __restrict__ out_grad) {
    float wx[ORD], dwx[ORD], wy[ORD], dwy[ORD], wz[ORD], dwz[ORD];
    bspline_weights<ORD, float>(tx, wx, dwx);
    bspline_weights<ORD, float>(ty, wy, dwy);
    bspline_weights<ORD, float>(tz, wz, dwz);
    const PairWeights<ORD> pw(wz, dwz, wy, dwy);
#pragma unroll
    for (int q = 0; q < NC; ++q) {
        const unsigned* cb = base + (c0 + q) * T::TSW;
        float u = 0.f, gx = 0.f, gy = 0.f, gz = 0.f;
#pragma unroll
        for (int jx = 0; jx < ORD; ++jx) {
            float s00, s10, s01;
            row_x2_words<ORD, GRAD, T::SYW>(cb + jx * T::SXW, pw, wy, dwy, wz, dwz, &s00, &s10, &s01);
            add_row<GRAD>(wx[jx], dwx[jx], s00, s10, s01, &u, &gx, &gy, &gz);
        }
        out_u[q] = u;
        if (GRAD) {
            out_grad[3 * q + 0] = gx * dscale;
            out_grad[3 * q + 1] = gy * dscale;
            out_grad[3 * q + 2] = gz * dscale;
        }
    }
}

// u and grad u of one component of one particle in FP64 arithmetic, its stencil read from global memory
// (comp: the component's [N][N][N] coefficients), for the particles whose stencil the fixed-point form below does
// not hold: by one thread, or by a warp, with the same operations in the same order.  An FP64 instruction takes an
// SM's quarter 75 cycles whatever its active lanes, so that one particle by one thread takes 15 (order 4) to 60 us
// (order 8), as long as a small call's whole gather; a warp spreads the weights and the stencil's lines over its lanes.

// One value of the recurrence of bspline_weights: M_k(t + m) from a = M_{k-1}(t + m), b = M_{k-1}(t + m - 1).
template <int k> __device__ __forceinline__ double weight_f64(double t, int m, double a, double b) {
    return fma(t + m, a, ((k - m) - t) * b) * (1.0 / (k - 1));
}
template <int n, int k = 2> __device__ __forceinline__ void weights_f64(double t, double (&v)[n], double (&w)[n], double (&dw)[n]) {
    if constexpr (k == 2) {
        v[0] = 1.0;
#pragma unroll
        for (int m = 1; m < n; ++m) v[m] = 0.0;
    }
    if constexpr (k < n) {
#pragma unroll
        for (int m = k - 1; m >= 0; --m) v[m] = weight_f64<k>(t, m, v[m], m > 0 ? v[m - 1] : 0.0);
        weights_f64<n, k + 1>(t, v, w, dw);
    } else {
#pragma unroll
        for (int m = 0; m < n; ++m) {
            const double b = m > 0 ? v[m - 1] : 0.0;
            w[n - 1 - m] = weight_f64<n>(t, m, v[m], b);
            dw[n - 1 - m] = v[m] - b;
        }
    }
}
template <int ORD, bool GRAD>
__device__ __noinline__ void eval_f64_thread(const double* __restrict__ comp, int N, unsigned cell, double tx,
                                             double ty, double tz, double dscale, double* __restrict__ out_u,
                                             double* __restrict__ out_grad) {
    const int ax = (int)(cell >> (2 * kAnchorBits)), ay = (int)((cell >> kAnchorBits) & 1023u), az = (int)(cell & 1023u);
    double wx[ORD], dwx[ORD], wy[ORD], dwy[ORD], wz[ORD], dwz[ORD];
    {
        double v[ORD];
        weights_f64<ORD>(tx, v, wx, dwx);
        weights_f64<ORD>(ty, v, wy, dwy);
        weights_f64<ORD>(tz, v, wz, dwz);
    }
    double u = 0, gx = 0, gy = 0, gz = 0;
#pragma unroll 1
    for (int jx = 0; jx < ORD; ++jx) {
        double y00 = 0, y10 = 0, y01 = 0;
#pragma unroll 1
        for (int jy = 0; jy < ORD; ++jy) {
            const double* line = comp + ((size_t)wrap_index(ax + jx, N) * N + wrap_index(ay + jy, N)) * N;
            double z0 = 0, z1 = 0;
#pragma unroll
            for (int jz = 0; jz < ORD; ++jz) {
                const double v = line[wrap_index(az + jz, N)];
                z0 = fma(wz[jz], v, z0);
                if (GRAD) z1 = fma(dwz[jz], v, z1);
            }
            y00 = fma(wy[jy], z0, y00);
            if (GRAD) {
                y10 = fma(dwy[jy], z0, y10);
                y01 = fma(wy[jy], z1, y01);
            }
        }
        u = fma(wx[jx], y00, u);
        if (GRAD) {
            gx = fma(dwx[jx], y00, gx);
            gy = fma(wx[jx], y10, gy);
            gz = fma(wx[jx], y01, gz);
        }
    }
    *out_u = u;
    if (GRAD) {
        out_grad[0] = gx * dscale;
        out_grad[1] = gy * dscale;
        out_grad[2] = gz * dscale;
    }
}

// The recurrence with lane (axis, m) holding v[m]: after step k < n, M_k(t + m); then the node's two weights.
template <int n, int k = 2> __device__ __forceinline__ void weights_f64_warp(double t, int m, double v, double* w, double* dw) {
    double b = __shfl_up_sync(0xffffffffu, v, 1);
    if (m == 0) b = 0.0;
    if constexpr (k < n) {
        weights_f64_warp<n, k + 1>(t, m, m < k ? weight_f64<k>(t, m, v, b) : 0.0, w, dw);
    } else {
        *w = weight_f64<n>(t, m, v, b);
        *dw = v - b;
    }
}
// Sums by lane, each in the order of eval_f64_thread: along z, chain 2 line + s (s = 0: w, 1: w'); along y, lane
// s ORD + jx (s = 0: Y00, 1: Y10, 2: Y01); along x, lanes 0 to 3 (u and the three derivatives).
template <int ORD, bool GRAD>
__device__ __noinline__ void eval_f64_warp(const double* __restrict__ comp, int N, unsigned cell, double tx,
                                           double ty, double tz, double dscale, double* __restrict__ out_u,
                                           double* __restrict__ out_grad) {
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int C = 2 * ORD * ORD, R = (C + 31) / 32;  // chains, and those of a lane
    const int lane = threadIdx.x & 31;
    const int ax = (int)(cell >> (2 * kAnchorBits)), ay = (int)((cell >> kAnchorBits) & 1023u), az = (int)(cell & 1023u);
    double v[R][ORD];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int l = min(lane + 32 * r, C - 1) >> 1, jx = l / ORD, jy = l % ORD;
        const double* line = comp + ((size_t)wrap_index(ax + jx, N) * N + wrap_index(ay + jy, N)) * N;
#pragma unroll
        for (int jz = 0; jz < ORD; ++jz) v[r][jz] = line[wrap_index(az + jz, N)];
    }
    double w, dw;                                        // lane a ORD + m: node ORD - 1 - m of axis a
    const int a = lane / ORD;
    weights_f64_warp<ORD>(a == 0 ? tx : (a == 1 ? ty : tz), lane % ORD, lane % ORD == 0 ? 1.0 : 0.0, &w, &dw);
    const auto weight = [&](int axis, int j, bool derivative) {
        const double wj = __shfl_sync(kAll, w, (axis + 1) * ORD - 1 - j), dj = __shfl_sync(kAll, dw, (axis + 1) * ORD - 1 - j);
        return derivative ? dj : wj;
    };
    double z[R], y = 0, x = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) z[r] = 0.0;
#pragma unroll
    for (int jz = 0; jz < ORD; ++jz) {
        const double wj = weight(2, jz, lane & 1);
#pragma unroll
        for (int r = 0; r < R; ++r) z[r] = fma(wj, v[r][jz], z[r]);
    }
    const int sy = min(lane / ORD, 2), jx0 = lane % ORD;
#pragma unroll
    for (int jy = 0; jy < ORD; ++jy) {
        const int chain = 2 * (jx0 * ORD + jy) + (sy == 2 ? 1 : 0);
        double b = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const double br = __shfl_sync(kAll, z[r], chain & 31);
            if ((chain >> 5) == r) b = br;
        }
        y = fma(weight(1, jy, sy == 1), b, y);
    }
    const int sx = lane < 2 ? 0 : min(lane - 1, 2);      // lanes 0, 1: Y00, 2: Y10, 3: Y01
#pragma unroll
    for (int jx = 0; jx < ORD; ++jx) x = fma(weight(0, jx, lane == 1), __shfl_sync(kAll, y, sx * ORD + jx), x);
    if (lane == 0) *out_u = x;
    else if (GRAD && lane < 4) out_grad[lane - 1] = x * dscale;
}

// FP64 plans: one CTA per work item, the brick's coefficients staged and turned into 60-bit fixed point
// (fixed.cuh) at one scale per component, the largest magnitude in the tile; weights, contraction and
// derivatives are integer multiply-adds, and only the twelve results are FP64 again.  Bound: integer issue.
// The FP64 pipe took 1900 operations a particle at order 6: 5.36 ms for 10^6 particles on 256^3; the fixed
// form's 5100 wide multiply-adds, with the tile's conversion (216 values a particle there), take 1.72 ms.
// The error of a fixed-point result is a unit or two whatever the stencil holds (rms 0.7, largest 2.5 for u; a unit is
// 2^-59 to 2^-60 of the tile's largest value from order 4 on, twice that at order 3), that of FP64 arithmetic a
// multiple of 2^-53 sum w |a| (rms 0.8 to 2.5 at order 4, 0.9 to 4 at order 8, for smooth, white and steep
// coefficients; the sums that the gradients are rounded against are no smaller).  So a component is taken from the
// fixed form where sum w |a| is at least 2^53 units (fixed::contract gives a lower estimate); the others, and every
// particle of a component whose tile holds a NaN or an infinity or nothing above 2^-895, are evaluated in FP64
// from global memory (eval_f64_thread, eval_f64_warp): the low flanks of steep or localised fields, one particle
// in 10^4 or fewer of a turbulent one, 1 to 8 % of a product of Fourier modes (where its nodal planes meet).  That choice
// depends on the coefficients and the position alone, so every route to the evaluation gives the same bits.
// Order 2 stays in FP64: with eight nodes a component the conversion costs more than it saves (256^3, 10^6
// particles, a call 0.48 ms in FP64, 0.50 ms in fixed point).
// NC = 3: a thread takes a particle's components in turn; NC = 1 (items of up to 42 particles): a thread
// takes one component of a particle, the axes' weights being shared: with the 30 particles a brick of the
// case above three of the four warps would idle otherwise (2.99 ms).
constexpr unsigned kFixedSize = 1u << (53 - 34);       // 2^53 units in those of fixed::contract
template <int ORD, int NC> constexpr int fixed_threads() { return NC == 3 && ORD >= 7 ? 192 : 128; }
template <int ORD, typename TR, bool GRAD, int NC>
__global__ void __launch_bounds__(fixed_threads<ORD, NC>(), ORD >= 7 ? 2 : (ORD <= 4 ? 4 : 3))
gather_fixed(const double* __restrict__ coef, int N, BrickGrid bg, Ws<TR> w, unsigned chunk_len,
             double* __restrict__ out_u, double* __restrict__ out_grad, double dscale,
             unsigned long long* __restrict__ status) {
    using S = Shape<double, ORD>;
    constexpr int T = fixed_threads<ORD, NC>(), kBits = fixed::value_bits<ORD>();
    if (blockIdx.x >= w.chunk[bg.NB]) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned s_top[3], s_any[3], s_left;
    __shared__ unsigned short s_pair[3 * (NC == 3 ? kFixedLong : kFixedShort)];      // 3 particle + component
    const unsigned brick = w.item[blockIdx.x];
    const unsigned beg = w.offset[brick] + (blockIdx.x - w.chunk[brick]) * chunk_len;
    const unsigned n = min(chunk_len, w.offset[brick] + w.count[brick] - beg);
    int x0, y0, z0;
    brick_origin<S::BX, S::BY, S::BZ>(brick, bg, &x0, &y0, &z0);
    // the tile, 16 lanes a z-row
    static_assert(S::EZ <= 16 && T % 16 == 0 && T / 16 <= 2 * S::EY, "16 lanes a row");
    uint2* words = reinterpret_cast<uint2*>(smem_raw);
    {
        const int z = threadIdx.x & 15;
        int ix = 0, iy = threadIdx.x >> 4;
        const double* col = coef + wrap_index(z0 + z, N);
        for (int r = iy; r < S::EX * S::EY; r += T / 16) {
            while (iy >= S::EY) {
                iy -= S::EY;
                ++ix;
            }
            const double* src = col + ((size_t)wrap_index(x0 + ix, N) * N + wrap_index(y0 + iy, N)) * N;
            if (z < S::EZ) {
#pragma unroll
                for (int c = 0; c < 3; ++c) cp_async8(words + c * S::TS + r * S::PZ + z, src + (size_t)c * N * N * N);
            }
            iy += T / 16;
        }
    }
    if (threadIdx.x < 3) s_top[threadIdx.x] = s_any[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_left = 0;
    cp_async_wait_all();
    __syncthreads();
    if constexpr (ORD == 2) {
        // eight nodes a component: FP64 arithmetic on the staged values costs less than converting them
        const double* tile = reinterpret_cast<const double*>(smem_raw);
        const unsigned units2 = NC == 3 ? n : 3 * n;
        for (unsigned i = threadIdx.x; i < units2; i += T) {
            const unsigned c0 = NC == 3 ? 0u : i / n, q = NC == 3 ? i : i - c0 * n;
            const Rec<TR> rc = w.s_rec[beg + q];
            const int ox = (int)(rc.cell >> (2 * kAnchorBits)) - x0, oy = (int)((rc.cell >> kAnchorBits) & 1023u) - y0;
            const int oz = (int)(rc.cell & 1023u) - z0;
            const size_t idx = rc.idx;
            if (!BS_CHECK_OK(ox >= 0 && ox < S::BX && oy >= 0 && oy < S::BY && oz >= 0 && oz < S::BZ &&
                                 (long long)idx < w.P,
                             status + kStatusBounds))
                continue;
            double wx[ORD], dwx[ORD], wy[ORD], dwy[ORD], wz[ORD], dwz[ORD];
            bspline_weights<ORD, double>(rc.t[0], wx, dwx);
            bspline_weights<ORD, double>(rc.t[1], wy, dwy);
            bspline_weights<ORD, double>(rc.t[2], wz, dwz);
            const double* base = tile + ox * S::SX + oy * S::SY + oz;
#pragma unroll 1
            for (int c = (int)c0; c < (int)c0 + NC; ++c) {
                const double* tc = base + c * S::TS;
                double u = 0, gx = 0, gy = 0, gz = 0;
#pragma unroll
                for (int jx = 0; jx < ORD; ++jx) {
                    double y00 = 0, y10 = 0, y01 = 0;
#pragma unroll
                    for (int jy = 0; jy < ORD; ++jy) {
                        const double a0 = tc[jx * S::SX + jy * S::SY], a1 = tc[jx * S::SX + jy * S::SY + 1];
                        const double v0 = fma(wz[1], a1, wz[0] * a0);
                        y00 = fma(wy[jy], v0, y00);
                        if (GRAD) {
                            y10 = fma(dwy[jy], v0, y10);
                            y01 = fma(wy[jy], fma(dwz[1], a1, dwz[0] * a0), y01);
                        }
                    }
                    u = fma(wx[jx], y00, u);
                    if (GRAD) {
                        gx = fma(dwx[jx], y00, gx);
                        gy = fma(wx[jx], y10, gy);
                        gz = fma(wx[jx], y01, gz);
                    }
                }
                out_u[3 * idx + c] = u;
                if (GRAD) {
                    out_grad[9 * idx + 3 * c + 0] = gx * dscale;
                    out_grad[9 * idx + 3 * c + 1] = gy * dscale;
                    out_grad[9 * idx + 3 * c + 2] = gz * dscale;
                }
            }
        }
        return;
    }
    // each component's largest high word and any bit but signs
#pragma unroll 1
    for (int c = 0; c < 3; ++c) {
        unsigned top = 0, any = 0;
        for (int k = threadIdx.x; k < S::TS; k += T) {
            const uint2 d = words[c * S::TS + k];
            top = max(top, d.y & 0x7fffffffu);
            any |= d.x;
        }
        top = __reduce_max_sync(0xffffffffu, top);
        any = __reduce_or_sync(0xffffffffu, any) | top;
        if ((threadIdx.x & 31) == 0) {
            atomicMax(&s_top[c], top);
            atomicOr(&s_any[c], any);
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int c = 0; c < 3; ++c) {
        const int emax = (int)(s_top[c] >> 20);
        for (int k = threadIdx.x; k < S::TS; k += T) {
            const uint2 d = words[c * S::TS + k];
            const fixed::Limbs l = fixed::limbs(fixed::from_double(d.y, d.x, emax, kBits));
            words[c * S::TS + k] = make_uint2((unsigned)l.lo, (unsigned)l.hi);
        }
    }
    __syncthreads();
    int4* ws = reinterpret_cast<int4*>(smem_raw + align_up(tile_bytes<ORD, double>()));
    // components c0 .. c0 + NC - 1 of the item's particle i; wx(j): the x weights of node j
    auto evaluate = [&](const Rec<TR>& rc, unsigned i, int c0, auto wx, const fixed::Limbs (&wy)[ORD],
                        const fixed::Limbs (&dwy)[ORD], const fixed::Limbs (&wz)[ORD], const fixed::Limbs (&dwz)[ORD]) {
        const int ax = (int)(rc.cell >> (2 * kAnchorBits)), ay = (int)((rc.cell >> kAnchorBits) & 1023u);
        const int az = (int)(rc.cell & 1023u);
        const size_t idx = rc.idx;
        const uint2* base = words + (ax - x0) * S::SX + (ay - y0) * S::SY + (az - z0);
#pragma unroll 1
        for (int c = c0; c < c0 + NC; ++c) {
            long long f[4];
            unsigned size = 0;
            const uint2* tc = base + c * S::TS;
            fixed::contract<ORD, GRAD>(
                [&](int jx, int jy, int jz) {
                    const uint2 v = tc[jx * S::SX + jy * S::SY + jz];
                    return fixed::Limbs{(int)v.y, (int)v.x};
                },
                wx, wy, dwy, wz, dwz, f, &size);
            const int emax = (int)(s_top[c] >> 20);
            if (!s_any[c]) {
                f[0] = f[1] = f[2] = f[3] = 0;           // a component that is zero in the whole tile
            } else if (emax < fixed::kMinExponent || emax == 2047 || size < kFixedSize) {
                s_pair[atomicAdd(&s_left, 1u)] = (unsigned short)(3 * i + c);       // not held by the fixed form
                continue;
            }
            // V 2^(emax - 1022 - kBits), in two exact steps (one of them may leave the normal range)
            const int k = emax - 1022 - kBits, k1 = k / 2;
            const double s1 = __hiloint2double((1023 + k1) << 20, 0), s2 = __hiloint2double((1023 + k - k1) << 20, 0);
            out_u[3 * idx + c] = ((double)f[0] * s1) * s2;
            if (GRAD) {
#pragma unroll
                for (int e = 0; e < 3; ++e) out_grad[9 * idx + 3 * c + e] = (((double)f[1 + e] * s1) * s2) * dscale;
            }
        }
    };
    auto record_ok = [&](const Rec<TR>& rc) {
        const int ox = (int)(rc.cell >> (2 * kAnchorBits)) - x0, oy = (int)((rc.cell >> kAnchorBits) & 1023u) - y0;
        const int oz = (int)(rc.cell & 1023u) - z0;
        return BS_CHECK_OK(ox >= 0 && ox < S::BX && oy >= 0 && oy < S::BY && oz >= 0 && oz < S::BZ &&
                               (long long)rc.idx < w.P,
                           status + kStatusBounds);
    };
    const auto fixed_t = [](double t) { return __double2ll_rn(t * 1152921504606846976.0); };     // t 2^60
    fixed::Limbs wy[ORD], dwy[ORD], wz[ORD], dwz[ORD];
    if constexpr (NC == 1) {
        // thread (a, q): the weights of particle q along axis a, then its component a
        const unsigned a = threadIdx.x / n, q = threadIdx.x - a * n;
        const bool on = threadIdx.x < 3 * n;
        Rec<TR> rc;
        if (on) {
            rc = w.s_rec[beg + q];
            fixed::weights<ORD>(fixed_t(a == 0 ? rc.t[0] : (a == 1 ? rc.t[1] : rc.t[2])), wy, dwy);
#pragma unroll
            for (int j = 0; j < ORD; ++j)
                ws[(a * ORD + j) * kFixedShort + q] = make_int4(wy[j].hi, wy[j].lo, dwy[j].hi, dwy[j].lo);
        }
        __syncthreads();
        if (on && record_ok(rc)) {
#pragma unroll
            for (int j = 0; j < ORD; ++j) {
                const int4 y = ws[(ORD + j) * kFixedShort + q], v = ws[(2 * ORD + j) * kFixedShort + q];
                wy[j] = {y.x, y.y};
                dwy[j] = {y.z, y.w};
                wz[j] = {v.x, v.y};
                dwz[j] = {v.z, v.w};
            }
            evaluate(rc, q, (int)a, [&](int j) { return ws[j * kFixedShort + q]; }, wy, dwy, wz, dwz);
        }
    } else {
        for (unsigned i = threadIdx.x; i < n; i += T) {
            const Rec<TR> rc = w.s_rec[beg + i];
            if (!record_ok(rc)) continue;
            fixed::weights<ORD>(fixed_t(rc.t[0]), wy, dwy);
#pragma unroll
            for (int j = 0; j < ORD; ++j)                // the x weights wait in shared memory
                ws[j * T + threadIdx.x] = make_int4(wy[j].hi, wy[j].lo, dwy[j].hi, dwy[j].lo);
            fixed::weights<ORD>(fixed_t(rc.t[1]), wy, dwy);
            fixed::weights<ORD>(fixed_t(rc.t[2]), wz, dwz);
            evaluate(rc, i, 0, [&](int j) { return ws[j * T + threadIdx.x]; }, wy, dwy, wz, dwz);
        }
    }
    // those left over, in FP64: few of them a warp each, many a thread each (a warp's form takes 30 to 80 FP64
    // instructions a pair, a thread's 340 to 1700 for up to 32 pairs).  10^4 particles on 32^3 in one product of modes (4 to
    // 8 % left over, gathered in the bricks of its nodal lines), up to 8 / 12 / 20 pairs a warp: order 4 55 / 61 / 61 us,
    // order 8 152 / 148 / 142; a narrow Gaussian, nearly all left over, order 4 63 / 67 / 80, order 8 180 / 179 / 211
    __syncthreads();
    const unsigned left = s_left;
    const bool by_warp = left <= 8 * (T / 32);
    for (unsigned e = by_warp ? threadIdx.x >> 5 : threadIdx.x; e < left; e += by_warp ? T / 32 : T) {
        const unsigned pair = s_pair[e], i = pair / 3, c = pair - 3 * i;
        const Rec<TR> rc = w.s_rec[beg + i];
        const double* comp = coef + (size_t)c * N * N * N;
        double* u = out_u + 3 * (size_t)rc.idx + c;
        double* g = GRAD ? out_grad + 9 * (size_t)rc.idx + 3 * c : nullptr;
        if (by_warp) eval_f64_warp<ORD, GRAD>(comp, N, rc.cell, rc.t[0], rc.t[1], rc.t[2], dscale, u, g);
        else eval_f64_thread<ORD, GRAD>(comp, N, rc.cell, rc.t[0], rc.t[1], rc.t[2], dscale, u, g);
    }
}

// A particle's outputs go to its original index, scattered: u (12 bytes) and
// grad u (36 bytes) are written with 8-byte stores where they are 8-byte
// aligned and one 4-byte store for the odd word, chosen by the index's
// parity with selects (no divergence): 2 + 5 store instructions instead of
// 3 + 9, since the load/store queue, not the bytes, is what the scattered
// stores occupy.  Needs 8-byte aligned output arrays (the caller checks).
__device__ __forceinline__ void store_u3(float* p, unsigned odd, const float (&u)[3]) {
    // even index: (u0, u1) at p, u2 at p + 2; odd: u0 at p, (u1, u2) at p + 1
    float* s = odd ? p : p + 2;
    float* v = odd ? p + 1 : p;
    *s = odd ? u[0] : u[2];
    *reinterpret_cast<float2*>(v) = odd ? make_float2(u[1], u[2]) : make_float2(u[0], u[1]);
}
__device__ __forceinline__ void store_g9(float* p, unsigned odd, const float (&g)[9]) {
    // even index: four pairs from p, g8 at p + 8; odd: g0 at p, four pairs from p + 1
    float* s = odd ? p : p + 8;
    float* v = odd ? p + 1 : p;
    *s = odd ? g[0] : g[8];
#pragma unroll
    for (int k = 0; k < 4; ++k)
        *reinterpret_cast<float2*>(v + 2 * k) =
            odd ? make_float2(g[2 * k + 1], g[2 * k + 2]) : make_float2(g[2 * k], g[2 * k + 1]);
}

// Threads of a gather CTA: 384, two CTAs on an SM; 256 and three where three tiles fit (FP32 up to order 4):
// with the couple of hundred particles that a brick often holds, half of twelve warps would have no job, and
// a third tile's copy is in flight.  Order 4, 256^3, 178 particles a brick: 155 -> 105 us (64-field batch 3.50 -> 3.28 ms).
template <int ORD, typename CT, int BYO = 0> constexpr bool three_tiles() {
    return 3 * ((sizeof(CT) == 2 ? Bf16Pair<ORD, BYO>::bytes : tile_bytes<ORD, CT, BYO>()) + 7 * 1024) <= 227 * 1024;
}
template <int ORD, typename CT, int BYO = 0> constexpr int gather_threads() { return three_tiles<ORD, CT, BYO>() ? 256 : 384; }
template <int ORD, typename CT, int BYO = 0> constexpr int gather_ctas() { return three_tiles<ORD, CT, BYO>() ? 3 : 2; }

// Bank order of an item's particles.  Particles are bucketed by bank (bucket[0..31]: their counts) and
// ordered rank-major, bank-minor: particle (bank r, rank k within it) comes after all of smaller rank and
// after those of its rank in smaller banks.  tab[k] (k < kRankTable): the banks holding more than k
// particles as a mask, and the particles of smaller rank; the warps of the CTA fill it, then synchronise.
// Deeper ranks (a clump within one bank) are counted bank by bank.  Counting every particle that way took
// 160 instructions each: 5 % of the quintic gather's, 8 % of the cubic position gradient's.
constexpr unsigned kRankTable = 128;
__device__ __forceinline__ void fill_rank_table(const unsigned* bucket, uint2* tab) {
    const unsigned lane = threadIdx.x & 31, b = bucket[lane];
    const unsigned top = min(__reduce_max_sync(0xffffffffu, b), kRankTable);
    for (unsigned k = threadIdx.x >> 5; k < top; k += blockDim.x >> 5) {
        const unsigned mask = __ballot_sync(0xffffffffu, b > k), below = __reduce_add_sync(0xffffffffu, min(b, k));
        if (lane == 0) tab[k] = make_uint2(mask, below);
    }
}
__device__ __forceinline__ unsigned bank_position(const unsigned* bucket, const uint2* tab, unsigned r, unsigned k) {
    if (k < kRankTable) {
        const uint2 t = tab[k];
        return t.y + (unsigned)__popc(t.x & ((1u << r) - 1u));
    }
    unsigned pos = 0;
#pragma unroll 8
    for (unsigned q = 0; q < 32; ++q) {
        const unsigned bq = bucket[q];
        pos += min(bq, k) + ((q < r && bq > k) ? 1u : 0u);
    }
    return pos;
}

// FP32 accumulation (FP32 or BF16 coefficients).  Each particle reads
// 3 ORD^3 tile values from shared memory, and a warp load costs one cycle per
// distinct address in the busiest of the 32 banks; random stencil origins
// would make most loads 3-4 way conflicted.  Within a chunk, particles are
// therefore bucketed by the bank of their stencil origin (residue mod 32),
// ranked within their bucket, and ordered rank-major, bank-minor: a warp
// that takes 32 consecutive particles of that order sees each bank at most
// once per rank it spans.
// One CTA per work item: item i is chunk i - chunk[b] of the brick b with
// chunk[b] <= i < chunk[b + 1] (at most kChunk particles); the grid is an
// upper bound on the number of items and surplus CTAs return at once.
// Two CTAs per SM (80 registers): orders 7 and 8 would otherwise take 84 and
// 102 registers and run one CTA per SM, 22 % and 16 % slower at 256^3.
// gather_f32_item evaluates work item `item` (at most chunk_len <= kChunk
// particles of one brick); the kernel gather_f32 runs one item per CTA, the
// batch kernel many per CTA (BYO: its brick y extent).  The caller has
// checked item < w.chunk[NB] and keeps every thread of the CTA here.
template <int ORD, typename CT, typename TR, bool GRAD, int BYO = 0>
__device__ __forceinline__ void gather_f32_item(unsigned item, unsigned chunk_len, const CT* __restrict__ coef, int N,
                                                const BrickGrid& bg, const Ws<TR>& w, float* __restrict__ out_u,
                                                float* __restrict__ out_grad, float dscale, const CUtensorMap* tmap,
                                                int use_tma, unsigned long long* __restrict__ status) {
    using S = Shape<CT, ORD, BYO>;
    constexpr int T = gather_threads<ORD, CT, BYO>(), NW = T / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // the tile 128-byte aligned (TMA destinations; the launch adds 128 bytes of slack), offset from the
    // shared array itself so that its loads stay shared-memory loads (an address rebuilt from an integer
    // would be a generic one)
    float* tile = reinterpret_cast<float*>(smem_raw + ((0u - smem_u32(smem_raw)) & 127u));
    __shared__ unsigned s_bucket[32];
    __shared__ uint2 s_rank[kRankTable];
    __shared__ unsigned short s_order[kChunk];
    __shared__ __align__(8) unsigned long long s_mbar;
    const unsigned brick = w.item[item];
    const unsigned c0 = w.offset[brick] + (item - w.chunk[brick]) * chunk_len;
    const unsigned end = w.offset[brick] + w.count[brick];
    int x0, y0, z0;
    brick_origin<S::BX, S::BY, S::BZ>(brick, bg, &x0, &y0, &z0);
    // BF16: the pair tile (copy A now, asynchronously; copy B after the bucketing)
    constexpr bool kBf16 = sizeof(CT) == 2;
    using T2 = Bf16Pair<ORD, BYO>;
    unsigned* words = reinterpret_cast<unsigned*>(tile);
    // bricks away from the periodic seams by TMA, the others with cp.async
    bool tma;
    if constexpr (kBf16) tma = stage_bf16_tma<ORD, BYO>(words, tmap, &s_mbar, N, x0, y0, z0, use_tma);
    else tma = stage_tile_tma<ORD, CT, BYO>(tile, tmap, &s_mbar, N, x0, y0, z0, use_tma);
    if (tma) {
    } else if constexpr (kBf16) {
        stage_bf16_copy_a<ORD, BYO>(words, reinterpret_cast<const __nv_bfloat16*>(coef), N, x0, y0, z0);
    } else {
        stage_brick<ORD, CT, BYO>(tile, coef, N, x0, y0, z0);
    }
    // shared-memory bank (word index mod 32) of a particle's first stencil value
    auto bank_of = [&](int ox, int oy, int oz) -> unsigned {
        if constexpr (kBf16)
            return (unsigned)(((oz & 1) ? T2::COPYW : 0) + (ox * T2::EY + oy) * T2::SYW + (oz >> 1)) & 31u;
        else
            return (unsigned)(ox * S::SX + oy * S::SY + oz) & 31u;
    };
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool vec_out = ((reinterpret_cast<uintptr_t>(out_u) | (GRAD ? reinterpret_cast<uintptr_t>(out_grad) : 0u)) &
                          7u) == 0u;
    // checks build: the stencil inside the staged tile, the output index inside the arrays
    auto origin_ok = [&](int ox, int oy, int oz, unsigned idx) {
        return BS_CHECK_OK(ox >= 0 && ox < S::BX && oy >= 0 && oy < S::BY && oz >= 0 && oz < S::BZ &&
                               (long long)idx < w.P,
                           status + kStatusBounds);
    };
    {
        const int n = (int)min(chunk_len, end - c0);
        if (threadIdx.x < 32) s_bucket[threadIdx.x] = 0;
        __syncthreads();                                  // the tile copies stay in flight while bucketing
        // bucket (bank residue of the stencil origin) and rank within it, kept in registers
        constexpr int KT = (kChunk + T - 1) / T;
        unsigned packed[KT];
#pragma unroll
        for (int k = 0; k < KT; ++k) {
            const int i = threadIdx.x + k * T;
            if (i < n) {
                const unsigned cp = w.s_rec[c0 + i].cell;
                const int ox = (int)(cp >> (2 * kAnchorBits)) - x0;
                const int oy = (int)((cp >> kAnchorBits) & 1023u) - y0;
                const int oz = (int)(cp & 1023u) - z0;
                const unsigned r = bank_of(ox, oy, oz);
                packed[k] = (atomicAdd(&s_bucket[r], 1u) << 5) | r;
            }
        }
        __syncthreads();
        fill_rank_table(s_bucket, s_rank);
        __syncthreads();
#pragma unroll
        for (int k = 0; k < KT; ++k) {
            const int i = threadIdx.x + k * T;
            if (i < n) {
                const unsigned pos = bank_position(s_bucket, s_rank, packed[k] & 31u, packed[k] >> 5);
                if (BS_CHECK_OK(pos < (unsigned)n, status + kStatusBounds)) s_order[pos] = (unsigned short)i;
            }
        }
        cp_async_wait_all();
        if (tma && !tma_tile_wait(&s_mbar, status + kStatusParticleTimeout)) {
            fill_nan_item<TR, float>(w, c0, (unsigned)n, out_u, GRAD ? out_grad : nullptr, 3);
            return;
        }
        __syncthreads();                                  // tile and order ready
        if constexpr (kBf16) build_bf16_copy_b<ORD, BYO>(words);
        // Warp jobs over that order.  Rank j holds #{banks with more than j
        // particles} particles, non-increasing in j.  While a rank holds at
        // least 16 particles it is one job (every load conflict-free); the
        // sparse tail ranks are packed 32 to a job: a job spanning k ranks
        // costs k-way conflicts, as k separate jobs would, in one instruction
        // stream instead of k.
        const unsigned my_bucket = s_bucket[lane];
        unsigned above = 0;                               // buckets ordered before this lane's
#pragma unroll
        for (int q = 0; q < 32; ++q) {
            const unsigned bq = __shfl_sync(0xffffffffu, my_bucket, q);
            above += (bq > my_bucket || (bq == my_bucket && q < lane)) ? 1u : 0u;
        }
        const unsigned src16 = __ffs(__ballot_sync(0xffffffffu, above == 15u)) - 1;
        const unsigned j16 = __shfl_sync(0xffffffffu, my_bucket, src16);   // ranks j < j16 hold >= 16
        const unsigned pos16 = __reduce_add_sync(0xffffffffu, min(my_bucket, j16));
        const unsigned njobs = j16 + ((unsigned)n - pos16 + 31u) / 32u;
        auto job_range = [&](unsigned j, unsigned* lo, unsigned* hi) {
            if (j < j16) {
                *lo = __reduce_add_sync(0xffffffffu, min(my_bucket, j));
                *hi = __reduce_add_sync(0xffffffffu, min(my_bucket, j + 1));
            } else {
                *lo = pos16 + 32u * (j - j16);
                *hi = min((unsigned)n, *lo + 32u);
            }
        };
        // the next job's record is loaded while the current one is evaluated
        Rec<TR> rc_n;
        bool v_n = false;
        auto fetch = [&](unsigned j) {
            unsigned lo, hi;
            job_range(j, &lo, &hi);
            const unsigned pos = lo + (unsigned)lane;
            v_n = pos < hi;
            if (v_n) {
                const unsigned i = c0 + s_order[pos];
                rc_n = w.s_rec[i];
            }
        };
        // Jobs are dealt to the NW warps in rounds.  A last, partly filled round
        // of m <= 2 NW / 3 jobs is run per component instead: 3 m shorter warp
        // tasks (one component of the job's 32 particles each), so the item
        // does not wait a whole job time on a few warps.
        const unsigned m_tail = njobs % NW;
        const unsigned jfull = (m_tail != 0 && 3 * m_tail <= 2 * NW) ? njobs - m_tail : njobs;
        if ((unsigned)warp < jfull) fetch(warp);
        for (unsigned j = warp; j < jfull; j += NW) {
            const Rec<TR> rc = rc_n;
            const unsigned idx = rc.idx;
            const bool v = v_n;
            v_n = false;
            if (j + NW < jfull) fetch(j + NW);
            if (v) {
                const int ox = (int)(rc.cell >> (2 * kAnchorBits)) - x0;
                const int oy = (int)((rc.cell >> kAnchorBits) & 1023u) - y0;
                const int oz = (int)(rc.cell & 1023u) - z0;
                if (!origin_ok(ox, oy, oz, idx)) continue;
                float u[3], g[9];
                if constexpr (kBf16)
                    eval_bf16<ORD, GRAD, T2, 3>(words + ((oz & 1) ? T2::COPYW : 0) + (ox * T2::EY + oy) * T2::SYW +
                                                    (oz >> 1),
                                                0, (float)rc.t[0], (float)rc.t[1], (float)rc.t[2], dscale, u, g);
                else
                    eval_particle_x2<ORD, GRAD, S::SX, S::SY, S::TS>(tile + ox * S::SX + oy * S::SY + oz,
                                                                      (float)rc.t[0], (float)rc.t[1], (float)rc.t[2],
                                                                      dscale, u, g);
                if (vec_out) {
                    store_u3(out_u + 3 * (size_t)idx, idx & 1u, u);
                    if (GRAD) store_g9(out_grad + 9 * (size_t)idx, idx & 1u, g);
                } else {
#pragma unroll
                    for (int c = 0; c < 3; ++c) out_u[3 * (size_t)idx + c] = u[c];
                    if (GRAD) {
#pragma unroll
                        for (int k = 0; k < 9; ++k) out_grad[9 * (size_t)idx + k] = g[k];
                    }
                }
            }
        }
        for (unsigned q = warp; q < 3 * (njobs - jfull); q += NW) {
            const unsigned c = q % 3;
            unsigned lo, hi;
            job_range(jfull + q / 3, &lo, &hi);
            const unsigned pos = lo + (unsigned)lane;
            if (pos < hi) {
                const unsigned i = c0 + s_order[pos];
                const Rec<TR> rc = w.s_rec[i];
                const unsigned idx = rc.idx;
                const int ox = (int)(rc.cell >> (2 * kAnchorBits)) - x0;
                const int oy = (int)((rc.cell >> kAnchorBits) & 1023u) - y0;
                const int oz = (int)(rc.cell & 1023u) - z0;
                if (!origin_ok(ox, oy, oz, idx)) continue;
                float u, g[3];
                if constexpr (kBf16)
                    eval_bf16<ORD, GRAD, T2, 1>(words + ((oz & 1) ? T2::COPYW : 0) + (ox * T2::EY + oy) * T2::SYW +
                                                    (oz >> 1),
                                                (int)c, (float)rc.t[0], (float)rc.t[1], (float)rc.t[2], dscale, &u, g);
                else
                    eval_component_x2<ORD, GRAD, S::SX, S::SY>(tile + c * S::TS + ox * S::SX + oy * S::SY + oz,
                                                               (float)rc.t[0], (float)rc.t[1], (float)rc.t[2], dscale,
                                                               &u, g);
                out_u[3 * (size_t)idx + c] = u;
                if (GRAD) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) out_grad[9 * (size_t)idx + 3 * c + k] = g[k];
                }
            }
        }
    }
}

template <int ORD, typename CT, typename TR, bool GRAD>
__global__ void __launch_bounds__(gather_threads<ORD, CT>(), gather_ctas<ORD, CT>())
gather_f32(const CT* __restrict__ coef, int N, BrickGrid bg, Ws<TR> w, float* __restrict__ out_u,
           float* __restrict__ out_grad, float dscale, const __grid_constant__ CUtensorMap tmap, int use_tma,
           unsigned long long* __restrict__ status) {
    if (blockIdx.x >= w.chunk[bg.NB]) return;
    gather_f32_item<ORD, CT, TR, GRAD>(blockIdx.x, kChunk, coef, N, bg, w, out_u, out_grad, dscale, &tmap, use_tma,
                                       status);
}

// Direct gather: particles evaluated from global memory, without a staged brick.  SORTED: those of the
// bricks holding fewer than the split (placed by the scan in one contiguous range after the dense bricks);
// otherwise every particle, in the caller's order, straight from its position (calls whose particles are
// too few for a sort to pay: run_points).
// A CTA takes G particles through four steps: thread (particle, axis) locates it and computes the axis'
// weights; thread (particle, y-line, piece) copies the stencil lines' aligned 16-byte pieces to shared memory
// (the pieces of a line are neighbouring threads', so a copy touches few cache lines, and a CTA's whole
// input is in flight at once); thread (particle, component, x-row) contracts its row; thread (particle, component) adds the
// rows up and stores.  Same contraction in the same order as the staged gather (row_x2, add_row), so the
// results are the same bits.  Bound: DRAM sectors and latency; a thread per particle, which read each of its
// 3 n^3 values through L1 by itself, cost 6 times as many L1 lookups.  Measured: 2^18 particles on 512^3, order 6, in brick order 386 -> 296 us;
// 10^3 particles on 64^3, order 4, one launch instead of five, 35 -> 12 us a call.
template <int ORD, typename CT> struct Points {
    static constexpr int T = 128;
    static constexpr int G = ORD == 8 ? 4 : T / (3 * ORD);   // particles of a CTA (order 8: 48 KB of shared memory)
    static constexpr int V = 16 / (int)sizeof(CT);      // values of a piece
    static constexpr int NQ = (ORD + 2 * V - 2) / V;    // pieces a line can touch
    static constexpr int LINE = 4 * NQ;                 // words of a line
    // words of an x-row; the skew spreads the rows' common offsets over the banks
    static constexpr int ROW = ORD * LINE + ((ORD * LINE) % 8 == 0 ? 4 : 0);
    static constexpr int WORDS = G * 3 * ORD * ROW;
    static_assert(G * ORD * NQ <= T && G * 3 * ORD <= T, "one round of threads per step");
};
template <int ORD, typename CT, typename TR, bool GRAD, bool SORTED>
__global__ void __launch_bounds__(Points<ORD, CT>::T)
gather_points(const CT* __restrict__ coef, int N, const double* __restrict__ x, long long P, double scale, unsigned NB,
              Ws<TR> w, float* __restrict__ out_u, float* __restrict__ out_grad, float dscale,
              unsigned long long* __restrict__ status) {
    using K = Points<ORD, CT>;
    constexpr int T = K::T, G = K::G;
    __shared__ __align__(16) unsigned s_line[K::WORDS];
    __shared__ float s_w[G][3][2][ORD], s_sum[G][3 * ORD][3];
    __shared__ int s_anchor[G][3];
    __shared__ long long s_idx[G];
    const long long beg = SORTED ? w.offset[NB + 2] : 0, end = SORTED ? w.offset[NB] : P;
    const int tid = threadIdx.x;
    for (long long i0 = beg + (long long)blockIdx.x * G; i0 < end; i0 += (long long)gridDim.x * G) {
        if (tid < 3 * G) {
            const int q = tid / 3, a = tid - 3 * q;
            const long long i = i0 + q;
            unsigned anchor = 0;
            float t = 0.f;
            bool ok = false;
            if (i < end) {
                if constexpr (SORTED) {
                    const Rec<TR> rc = w.s_rec[i];
                    anchor = (rc.cell >> (kAnchorBits * (2 - a))) & 1023u;
                    t = a == 0 ? rc.t[0] : (a == 1 ? rc.t[1] : rc.t[2]);
                    ok = BS_CHECK_OK((int)anchor < N && (long long)rc.idx < w.P, status + kStatusBounds);
                    if (a == 0) s_idx[q] = rc.idx;
                } else {
                    ok = locate_axis<float>(x[3 * i + a] * scale, N, ORD, &anchor, &t);
                    if (a == 0) s_idx[q] = i;
                }
            }
            s_anchor[q][a] = ok ? (int)anchor : -1;
            float wt[ORD], dwt[ORD];
            bspline_weights<ORD, float>(t, wt, dwt);
#pragma unroll
            for (int j = 0; j < ORD; ++j) {
                s_w[q][a][0][j] = wt[j];
                s_w[q][a][1][j] = dwt[j];
            }
        }
        __syncthreads();
        const auto good = [&](int q) { return (s_anchor[q][0] | s_anchor[q][1] | s_anchor[q][2]) >= 0; };
        // thread (particle, y-line, piece) copies that piece of every component and x-row: everything but the
        // x index is the thread's own
        if (tid < G * ORD * K::NQ) {
            const int q = tid / (ORD * K::NQ), e = tid - q * (ORD * K::NQ), jy = e / K::NQ, k = e - jy * K::NQ;
            const int ax = s_anchor[q][0], az = s_anchor[q][2];
            if (good(q) && K::V * k < (az & (K::V - 1)) + ORD) {
                const size_t NN = (size_t)N * N;
                const CT* src = coef + (size_t)wrap_index(s_anchor[q][1] + jy, N) * N +
                                wrap_index((az & ~(K::V - 1)) + K::V * k, N);
                unsigned* dst = s_line + q * (3 * ORD) * K::ROW + jy * K::LINE + 4 * k;
#pragma unroll
                for (int jx = 0; jx < ORD; ++jx) {
                    const CT* at = src + (size_t)wrap_index(ax + jx, N) * NN;
#pragma unroll
                    for (int c = 0; c < 3; ++c) cp_async16(dst + (c * ORD + jx) * K::ROW, at + (size_t)c * N * NN);
                }
            }
        }
        cp_async_wait_all();
        __syncthreads();
        if (tid < G * 3 * ORD) {
            const int q = tid / (3 * ORD), r = tid - q * 3 * ORD;
            if (good(q)) {
                float wy[ORD], dwy[ORD], wz[ORD], dwz[ORD];
#pragma unroll
                for (int j = 0; j < ORD; ++j) {
                    wy[j] = s_w[q][1][0][j];
                    dwy[j] = s_w[q][1][1][j];
                    wz[j] = s_w[q][2][0][j];
                    dwz[j] = s_w[q][2][1][j];
                }
                const PairWeights<ORD> pw(wz, dwz, wy, dwy);
                const CT* line = reinterpret_cast<const CT*>(s_line + tid * K::ROW) + (s_anchor[q][2] & (K::V - 1));
                float s00, s10, s01;
                row_x2<ORD, GRAD>([&](int jy, int jz) { return widen<CT>(line[jy * K::NQ * K::V + jz]); }, pw, wy, dwy, wz,
                                  dwz, &s00, &s10, &s01);
                s_sum[q][r][0] = s00;
                s_sum[q][r][1] = s10;
                s_sum[q][r][2] = s01;
            }
        }
        __syncthreads();
        if (tid < 3 * G && i0 + tid / 3 < end) {
            const int q = tid / 3, c = tid - 3 * q;
            const size_t idx = (size_t)s_idx[q];
            const bool ok = good(q);
            float u = 0.f, gx = 0.f, gy = 0.f, gz = 0.f;
            if (ok) {
#pragma unroll
                for (int jx = 0; jx < ORD; ++jx) {
                    const float* v = s_sum[q][c * ORD + jx];
                    add_row<GRAD>(s_w[q][0][0][jx], s_w[q][0][1][jx], v[0], v[1], v[2], &u, &gx, &gy, &gz);
                }
            } else if (!SORTED) {
                u = gx = gy = gz = NAN;
                if (c == 0) atomicAdd(status + kStatusNonfinite, 1ULL);
            }
            if (ok || !SORTED) {                         // a sorted record fails only its check (checks builds)
                out_u[3 * idx + c] = u;
                if (GRAD) {
                    out_grad[9 * idx + 3 * c + 0] = gx * dscale;
                    out_grad[9 * idx + 3 * c + 1] = gy * dscale;
                    out_grad[9 * idx + 3 * c + 2] = gz * dscale;
                }
            }
        }
        __syncthreads();
    }
}

template <typename K> int set_smem(K kernel, size_t bytes) {
    if (bytes > 32 * 1024) {           // static shared memory counts against the 48 KB default too
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) return set_cuda_error(e);
    }
    return BSPLINE_OK;
}

template <int ORD, typename CT, typename AT, typename TR>
int run_gather(bspline_plan_s* p, const void* coeffs, Ws<TR> w, BrickGrid g, void* out_u, void* out_grad,
               bool grad, unsigned below) {
    const unsigned NB = g.NB;
    const size_t sm = tile_bytes<ORD, CT>();
    const AT dscale = (AT)((double)p->N / p->L);
    int rc;
    if constexpr (sizeof(AT) == 8) {
        const unsigned len = item_particles(p->dtype, ORD, w.P, NB);
        const bool whole = len == kFixedLong;
        auto k = whole ? (grad ? gather_fixed<ORD, TR, true, 3> : gather_fixed<ORD, TR, false, 3>)
                       : (grad ? gather_fixed<ORD, TR, true, 1> : gather_fixed<ORD, TR, false, 1>);
        const int threads = whole ? fixed_threads<ORD, 3>() : fixed_threads<ORD, 1>();
        // the tile and the weights of the particles in work
        const size_t sm_x = align_up(sm) + sizeof(int4) * ORD * (whole ? threads : 3 * kFixedShort);
        if ((rc = set_smem(k, sm_x))) return rc;
        const long long items = (long long)NB + (w.P + len - 1) / len;
        k<<<(unsigned)items, threads, sm_x, p->stream>>>(
            reinterpret_cast<const double*>(coeffs), p->N, g, w, len, (double*)out_u, grad ? (double*)out_grad : nullptr,
            dscale, p->d_status);
    } else {
        auto k = grad ? gather_f32<ORD, CT, TR, true> : gather_f32<ORD, CT, TR, false>;
        // room to align the tile to 128 bytes; BF16: the two copies of the pair tile
        const size_t sm_aligned = (sizeof(CT) == 2 ? Bf16Pair<ORD>::bytes : sm) + 128;
        if ((rc = set_smem(k, sm_aligned))) return rc;
        // FP32 coefficients: a TMA tensor map for the interior bricks (cp.async if it cannot be made)
        using S = Shape<CT, ORD>;
        CUtensorMap tmap;
        std::memset(&tmap, 0, sizeof tmap);
        int use_tma = 0;
        if (p->N >= 16 && !(p->test_hooks & BSPLINE_TEST_NO_TMA)) {
            const int box_z = sizeof(CT) == 2 ? Bf16Pair<ORD>::PZ : S::PZ;
            use_tma = encode_coef_tmap(&tmap, coeffs, p->N, box_z, S::EY, S::EX, (int)sizeof(CT)) == BSPLINE_OK
                          ? kTmaOn : 0;
        }
        if (use_tma && (p->test_hooks & BSPLINE_TEST_SKIP_TMA_ISSUE)) use_tma = kTmaArmOnly;
        // work items: at most one partial chunk per staged brick plus P / kChunk full ones; with a split a
        // staged brick holds at least `below` particles (2^18 particles on 512^3: 44160 -> 8320 CTAs, of
        // which most find no item, 43 -> 8 us)
        const long long bricks = below ? std::min<long long>(NB, w.P / below) : NB;
        const long long items = bricks + (w.P + kChunk - 1) / kChunk;
        k<<<(unsigned)items, gather_threads<ORD, CT>(), sm_aligned, p->stream>>>(
            reinterpret_cast<const CT*>(coeffs), p->N, g, w, (float*)out_u, grad ? (float*)out_grad : nullptr, dscale,
            tmap, use_tma, p->d_status);
    }
    return BSPLINE_OK;
}

// The direct gather (FP32 accumulation only): with x, of all P particles at their positions; without, of the
// sorted particles of the bricks below the plan's split.
template <int ORD, typename CT, typename AT, typename TR>
int run_gather_points(bspline_plan_s* p, const void* coeffs, const double* x, int64_t P, Ws<TR> w, unsigned NB,
                      void* out_u, void* out_grad, bool grad) {
    if constexpr (sizeof(AT) == 8) {
        return BSPLINE_OK;
    } else {
        const double scale = (double)p->N / p->L;
        auto k = x ? (grad ? gather_points<ORD, CT, TR, true, false> : gather_points<ORD, CT, TR, false, false>)
                   : (grad ? gather_points<ORD, CT, TR, true, true> : gather_points<ORD, CT, TR, false, true>);
        // the sparse range's length is known on the device only: a few waves, grid-striding beyond
        constexpr int G = Points<ORD, CT>::G;
        const long long want = (P + G - 1) / G;
        const unsigned blocks = (unsigned)std::min(want, x ? 1LL << 30 : 32LL * p->sms);
        k<<<blocks, Points<ORD, CT>::T, 0, p->stream>>>(reinterpret_cast<const CT*>(coeffs), p->N, x, P, scale, NB, w,
                                                        (float*)out_u, grad ? (float*)out_grad : nullptr, (float)scale,
                                                        p->d_status);
        return BSPLINE_OK;
    }
}

}  // namespace gather_impl

#define BS_GATHER_EXTERN(ORD, CT, AT, TR)                                                                 \
    extern template int gather_impl::run_gather<ORD, CT, AT, TR>(bspline_plan_s*, const void*,               \
                                                                  gather_impl::Ws<TR>, BrickGrid, void*,     \
                                                                  void*, bool, unsigned);                              \
    extern template int gather_impl::run_gather_points<ORD, CT, AT, TR>(                                     \
        bspline_plan_s*, const void*, const double*, int64_t, gather_impl::Ws<TR>, unsigned, void*, void*, bool);
#define BS_GATHER_INSTANTIATE(ORD, CT, AT, TR)                                                          \
    template int gather_impl::run_gather<ORD, CT, AT, TR>(bspline_plan_s*, const void*, gather_impl::Ws<TR>, \
                                                           BrickGrid, void*, void*, bool, unsigned);        \
    template int gather_impl::run_gather_points<ORD, CT, AT, TR>(                                            \
        bspline_plan_s*, const void*, const double*, int64_t, gather_impl::Ws<TR>, unsigned, void*, void*, bool);

}  // namespace bs
