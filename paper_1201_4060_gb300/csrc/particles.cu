// Particle side of the path: locate, bin/sort, and evaluate u and grad u.
//
// Locate (Eq. alg-int-6): s = x N / L in FP64; the stencil nodes are
// floor(s - n/2) + j, j = 1..n; the local variable is t = (s - n/2) - floor(s - n/2).
// The first node (the "anchor") picks a brick of 16^3 (FP64: 8^3) cells; particles are
// counting-sorted by brick so that one CTA stages the brick's coefficients
// (plus the n-1 halo) in shared memory once and evaluates all of its particles.
//
// Weights: per axis, the n node weights B(t + n/2 - j) and their derivatives
// come from the Cox-de Boor recurrence of the cardinal B-spline
// (M_k(x) = (x M_{k-1}(x) + (k - x) M_{k-1}(x - 1)) / (k - 1)), in registers.
// They equal the columns of M x_bar and M^(1) x_bar of Section 4.
//
// Contraction (Table 1, reordered to contract the contiguous z axis first):
// per component, Z0 = sum_z w_z a, Z1 = sum_z w'_z a (2 n^3), then
// Y00 = sum_y w_y Z0, Y10 = sum_y w'_y Z0, Y01 = sum_y w_y Z1 (3 n^2), then
// u = sum_x w_x Y00, du/dx = sum_x w'_x Y00, du/dy = sum_x w_x Y10,
// du/dz = sum_x w_x Y01 (4 n), derivatives scaled by N / L.
#include "adjoint.cuh"

namespace bs {

#define BS_ORDERS(M, CT, AT, TR) M(2, CT, AT, TR) M(3, CT, AT, TR) M(4, CT, AT, TR) M(5, CT, AT, TR) \
    M(6, CT, AT, TR) M(7, CT, AT, TR) M(8, CT, AT, TR)
BS_ORDERS(BS_GATHER_EXTERN, double, double, double)
BS_ORDERS(BS_GATHER_EXTERN, float, float, float)
BS_ORDERS(BS_GATHER_EXTERN, __nv_bfloat16, float, float)
#define BS_ADJ_ORDERS(M, CT, TR) M(2, CT, TR) M(3, CT, TR) M(4, CT, TR) M(5, CT, TR) M(6, CT, TR) M(7, CT, TR) \
    M(8, CT, TR)
BS_ADJ_ORDERS(BS_ADJOINT_EXTERN, double, double)
BS_ADJ_ORDERS(BS_ADJOINT_EXTERN, float, float)
BS_ADJ_ORDERS(BS_ADJOINT_EXTERN, __nv_bfloat16, float)

namespace gather_impl {

// cuTensorMapEncodeTiled, looked up once through the runtime (no link against the driver library).
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_tiled() {
    static const EncodeTiledFn fn = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            return (EncodeTiledFn) nullptr;
        }
        return reinterpret_cast<EncodeTiledFn>(f);
    }();
    return fn;
}

int encode_coef_tmap(CUtensorMap* map, const void* coef, int N, int box_z, int box_y, int box_x, int elem_bytes) {
    const EncodeTiledFn fn = encode_tiled();
    if (!fn) return BSPLINE_ERR_CUDA;
    const cuuint64_t n = (cuuint64_t)N, eb = (cuuint64_t)elem_bytes;
    const cuuint64_t dims[4] = {n, n, n, 3};                               // z, y, x, component
    const cuuint64_t strides[3] = {n * eb, n * n * eb, n * n * n * eb};  // bytes, dims 1..3
    const cuuint32_t box[4] = {(cuuint32_t)box_z, (cuuint32_t)box_y, (cuuint32_t)box_x, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUtensorMapDataType t = elem_bytes == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
    const CUresult r = fn(map, t, 4, const_cast<void*>(coef), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? BSPLINE_OK : BSPLINE_ERR_CUDA;
}

}  // namespace gather_impl

namespace {
using namespace gather_impl;

// ------------------------------------------------------------------ bin
// Warp-aggregated increment of counter[key] for the lanes of `active`: one
// atomic per distinct key in the warp (positions in brick order).
__device__ __forceinline__ void warp_increment(unsigned* counter, unsigned key, unsigned active) {
    const unsigned peers = __match_any_sync(active, key);
    if ((threadIdx.x & 31u) == __ffs(peers) - 1) atomicAdd(&counter[key], (unsigned)__popc(peers));
}

// Counting sort, pass 1: particles per brick (slot NB: invalid positions, also
// counted in the status word).  HIST: runs of `run` particles, counted in shared
// memory, which also gives each particle's place within its brick (count_run);
// else one atomic a particle, and the placement pass draws the places.  Both
// loops run warp-uniformly.  SORTED: the
// caller passed the positions grouped by brick, so position p is also the
// particle's sorted slot: its record is written there (coalesced, its own
// index as the original one), each key is checked against its predecessor's
// (the lane below, or located again at a warp's first lane) and *w.unsorted is
// set if the order is broken anywhere, in which case the placement pass
// rewrites every record; invalid positions get their NaN outputs here.
template <typename TR, bool SORTED, bool HIST, typename OT>
__global__ void __launch_bounds__(256)
bin_kernel(const double* __restrict__ x, long long P, int N, double scale, int order, BrickGrid g, Ws<TR> w,
           unsigned long long* __restrict__ status, unsigned run, OT* __restrict__ out_u, OT* __restrict__ out_grad) {
    const unsigned NB = g.NB;
    const long long lane = threadIdx.x & 31;
    auto key = [&](long long p) -> unsigned {            // every lane of the warp, consecutive p
        const bool valid = p < P;
        unsigned k = 0;
        if (valid) {
            Rec<TR> r;
            k = locate_particle<TR>(x, p, N, scale, order, g, &r);
            if (k == NB) atomicAdd(status, 1ULL);
            if (SORTED && k < NB) {
                r.idx = (unsigned)p;
                if constexpr (sizeof(TR) == 4) r.pad[0] = r.pad[1] = r.pad[2] = 0u;
                w.s_rec[p] = r;
            }
        }
        if constexpr (SORTED) {
            unsigned prev = __shfl_up_sync(0xffffffffu, k, 1);
            if (lane == 0 && valid && p > 0) {
                Rec<TR> r;
                prev = locate_particle<TR>(x, p - 1, N, scale, order, g, &r);
            }
            const bool broken = valid && p > 0 && prev > k;
            if (__any_sync(0xffffffffu, broken) && lane == 0) atomicOr(w.unsorted, 1u);
            if (valid && k == NB) {
                const OT nan = (OT)NAN;
                if (out_u) {
#pragma unroll
                    for (int i = 0; i < 3; ++i) out_u[3 * p + i] = nan;
                }
                if (out_grad) {
#pragma unroll
                    for (int i = 0; i < 9; ++i) out_grad[9 * p + i] = nan;
                }
            }
        }
        return k;
    };
    if constexpr (HIST) {
        extern __shared__ unsigned s_bin[];
        for (long long p0 = (long long)blockIdx.x * run; p0 < P; p0 += (long long)gridDim.x * run)
            count_run(s_bin, NB, (unsigned)min((long long)run, P - p0), w.count, w.rank + p0,
                      [&](unsigned i) { return key(p0 + i); });
    } else {
        const long long stride = (long long)gridDim.x * blockDim.x;
        for (long long pw = (long long)blockIdx.x * blockDim.x + threadIdx.x - lane; pw < P; pw += stride) {
            const long long p = pw + lane;
            const bool valid = p < P;
            const unsigned k = key(p);
            if constexpr (SORTED) {                      // a warp's particles share bricks
                const unsigned active = __ballot_sync(0xffffffffu, valid);
                if (valid) warp_increment(w.count, k, active);
            } else if (valid) {
                atomicAdd(&w.count[k], 1u);
            }
        }
    }
}

// ------------------------------------------------------------------ scan (single CTA)
// Places the bricks' segments in the sorted order and counts the staged
// gather's work items.  Bricks holding at least `below` particles ("dense":
// every brick when below = 0) come first, in brick order; the bricks below
// it ("sparse", evaluated by the direct gather) follow, placed from the end
// of the valid particles downwards (so that no pass has to total the dense
// ones first), and the direct gather runs flat over one contiguous range; the
// invalid bin NB comes last.  Writes offset[b] (and its copy cursor[b] for the placement
// pass), offset[NB] = the end of the valid particles, offset[NB + 1] = the
// end of all, offset[NB + 2] = the start of the sparse range; chunk[] (dense
// bricks only) the exclusive prefix sum of the work items, ceil(count /
// kChunk), chunk[NB] their total, and item[] each item's brick.
__device__ __forceinline__ unsigned warp_inclusive(unsigned v, unsigned lane) {
#pragma unroll
    for (unsigned d = 1; d < 32; d <<= 1) {
        const unsigned a = __shfl_up_sync(0xffffffffu, v, d);
        if (lane >= d) v += a;
    }
    return v;
}

// SPLIT = false (below = 0: every brick dense) skips the sparse bookkeeping.
// Bound: one CTA's latency per tile.  A thread takes RUN consecutive bricks (4: 16-byte loads and stores), the next
// tile's counts requested before this tile is scanned.  Measured with runs of 1 / 2 / 4 / 8: 96 bricks 6.2 / 6.4 / 7.6 /
// 8.5 us, 5632 11.1 / 10.4 / 10.3 / 11.9, 18432 23.6 / 22.4 / 18.8 / 24.6, 44032 48 / 45 / 35 / 52: 1 where one tile of it
// holds the bricks, else 4.
template <bool SPLIT, unsigned RUN>
__global__ void __launch_bounds__(1024) scan_kernel(const unsigned* __restrict__ count, unsigned* __restrict__ offset,
                                                    unsigned* __restrict__ cursor, unsigned* __restrict__ chunk,
                                                    unsigned* __restrict__ item, unsigned NB, unsigned below,
                                                    unsigned chunk_len, long long P) {
    __shared__ unsigned wd[32], wsp[32], wc[32];
    const unsigned t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const unsigned V = (unsigned)P - count[NB];           // valid particles
    unsigned v[RUN], nx[RUN];
    auto load = [&](unsigned b0) {                        // the run's counts, zero beyond the bricks
        const unsigned i = b0 + t * RUN;
        if constexpr (RUN == 4) {
            if (i + RUN <= NB) {
                const uint4 q = *reinterpret_cast<const uint4*>(count + i);
                nx[0] = q.x;
                nx[1] = q.y;
                nx[2] = q.z;
                nx[3] = q.w;
                return;
            }
        }
#pragma unroll
        for (unsigned k = 0; k < RUN; ++k) nx[k] = i + k < NB ? count[i + k] : 0u;
    };
    unsigned cd = 0, cs = 0, cc = 0;                      // carries: dense, sparse, items
    // tiles of 1024 runs: sums of the runs, warp scans of those, then a scan of the 32 warp totals
    load(0);
    for (unsigned b0 = 0; b0 < NB; b0 += 1024 * RUN) {
        unsigned sd = 0, ss = 0, sc = 0;
#pragma unroll
        for (unsigned k = 0; k < RUN; ++k) {
            v[k] = nx[k];
            const bool dense = !SPLIT || v[k] >= below;
            sd += dense ? v[k] : 0u;
            ss += dense ? 0u : v[k];
            sc += dense ? (v[k] + chunk_len - 1) / chunk_len : 0u;
        }
        if (b0 + 1024 * RUN < NB) load(b0 + 1024 * RUN);
        const unsigned vd = warp_inclusive(sd, lane), vc = warp_inclusive(sc, lane);
        const unsigned vs = SPLIT ? warp_inclusive(ss, lane) : 0u;
        if (lane == 31) {
            wd[warp] = vd;
            wsp[warp] = vs;
            wc[warp] = vc;
        }
        __syncthreads();
        if (warp == 0) {
            wd[lane] = warp_inclusive(wd[lane], lane);
            if (SPLIT) wsp[lane] = warp_inclusive(wsp[lane], lane);
            wc[lane] = warp_inclusive(wc[lane], lane);
        }
        __syncthreads();
        unsigned exd = cd + (warp ? wd[warp - 1] : 0u) + vd - sd;                 // exclusive
        unsigned exs = V - cs - (warp ? wsp[warp - 1] : 0u) - vs + ss;              // end of the run's segments
        unsigned exc = cc + (warp ? wc[warp - 1] : 0u) + vc - sc;
        const unsigned i = b0 + t * RUN;
        unsigned o[RUN], c[RUN];
#pragma unroll
        for (unsigned k = 0; k < RUN; ++k) {
            const bool dense = !SPLIT || v[k] >= below;
            exs -= dense ? 0u : v[k];
            o[k] = dense ? exd : exs;
            c[k] = exc;
            const unsigned nc = dense ? (v[k] + chunk_len - 1) / chunk_len : 0u;
            for (unsigned q = 0; q < nc; ++q) item[exc + q] = i + k;
            exd += dense ? v[k] : 0u;
            exc += nc;
        }
        bool stored = false;
        if constexpr (RUN == 4) {
            if (i + RUN <= NB) {
                const uint4 a = make_uint4(o[0], o[1], o[2], o[3]);
                *reinterpret_cast<uint4*>(offset + i) = a;
                *reinterpret_cast<uint4*>(cursor + i) = a;
                *reinterpret_cast<uint4*>(chunk + i) = make_uint4(c[0], c[1], c[2], c[3]);
                stored = true;
            }
        }
        if (!stored) {
#pragma unroll
            for (unsigned k = 0; k < RUN; ++k)
                if (i + k < NB) {
                    offset[i + k] = o[k];
                    cursor[i + k] = o[k];
                    chunk[i + k] = c[k];
                }
        }
        cd += wd[31];
        cs += wsp[31];
        cc += wc[31];
        __syncthreads();                                  // the totals are read before the next tile
    }
    if (t == 0) {
        offset[NB] = V;                                   // the invalid bin
        cursor[NB] = V;
        offset[NB + 1] = (unsigned)P;
        offset[NB + 2] = cd;
        chunk[NB] = cc;
    }
}

template <typename TR>
void launch_scan(const Ws<TR>& w, unsigned NB, unsigned below, unsigned chunk_len, long long P, cudaStream_t st) {
    const auto k = NB <= 1024u ? (below ? scan_kernel<true, 1> : scan_kernel<false, 1>)
                               : (below ? scan_kernel<true, 4> : scan_kernel<false, 4>);
    k<<<1, 1024, 0, st>>>(w.count, w.offset, w.cursor, w.chunk, w.item, NB, below, chunk_len, P);
}

// ------------------------------------------------------------------ place
// Counting sort, pass 2: locate again (cheaper than storing and re-reading the
// records) and write each record and its original index to its brick's segment:
// at the place the count pass gave it (ranked), else at the next free slot.  Invalid positions get NaN outputs.  SORTED: nothing to do
// unless the count pass found the order broken.  PERM (bspline_sort_order):
// every particle, invalid ones included (bin NB, last), gets a slot, and only
// its original index is written there, to perm.  cot (the adjoint of FP32
// types): each placed particle's cotangents g_u (or zeros) and g_grad (or
// zeros) also go to its slot, 16 floats (64 bytes: two whole sectors) a slot,
// so that the adjoint kernels read them in sorted order; a warp reads its 32
// particles' cotangents as whole lines into 12 * 32 floats of dynamic shared
// memory (the launch gives 12 * 32 * 4 bytes per warp).
template <typename TR, typename OT, bool SORTED = false, bool PERM = false>
__global__ void scatter_kernel(const double* __restrict__ x, long long P, int N, double scale, int order,
                               BrickGrid g, Ws<TR> w, OT* __restrict__ out_u, OT* __restrict__ out_grad,
                               int ranked, unsigned long long* __restrict__ status, int* __restrict__ perm = nullptr,
                               const float* __restrict__ cu = nullptr, const float* __restrict__ cg = nullptr,
                               float4* __restrict__ cot = nullptr) {
    const unsigned NB = g.NB;
    if constexpr (SORTED) {
        if (*w.unsorted == 0u) return;
    }
    if constexpr (PERM) {
        const long long stride = (long long)gridDim.x * blockDim.x;
        for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < P; p += stride) {
            Rec<TR> r;
            const unsigned k = locate_particle<TR>(x, p, N, scale, order, g, &r);
            const unsigned d = ranked ? w.offset[k] + w.rank[p] : atomicAdd(&w.cursor[k], 1u);
            if (BS_CHECK_OK(d < (unsigned)P, status + kStatusBounds)) perm[d] = (int)p;
        }
        return;
    }
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long lane = threadIdx.x & 31;
    extern __shared__ float s_cot_stage[];
    float* sw = s_cot_stage + (threadIdx.x >> 5) * (12 * 32);
    for (long long pw = (long long)blockIdx.x * blockDim.x + threadIdx.x - lane; pw < P; pw += stride) {
        const long long p = pw + lane;
        Rec<TR> r;
        unsigned k = NB;
        if (p < P) k = locate_particle<TR>(x, p, N, scale, order, g, &r);
        if (p < P && k >= NB) {
            const OT nan = (OT)NAN;
            if (out_u) {
#pragma unroll
                for (int i = 0; i < 3; ++i) out_u[3 * p + i] = nan;
            }
            if (out_grad) {
#pragma unroll
                for (int i = 0; i < 9; ++i) out_grad[9 * p + i] = nan;
            }
        }
        const bool place = p < P && k < NB;
        if (cot) {                                      // the warp's cotangents, coalesced
            const int nq = (int)min(32LL, P - pw);
            __syncwarp();                               // the previous iteration's reads are done
            for (int i = (int)lane; i < 3 * nq; i += 32) sw[i] = cu ? cu[3 * pw + i] : 0.f;
            for (int i = (int)lane; i < 9 * nq; i += 32) sw[96 + i] = cg ? cg[9 * pw + i] : 0.f;
            __syncwarp();
        }
        const unsigned d = !place ? 0u : (ranked ? w.offset[k] + w.rank[p] : atomicAdd(&w.cursor[k], 1u));
        if (place && BS_CHECK_OK(d < w.offset[k] + w.count[k], status + kStatusBounds)) {
            r.idx = (unsigned)p;
            if constexpr (sizeof(TR) == 4) r.pad[0] = r.pad[1] = r.pad[2] = 0u;
            w.s_rec[d] = r;                             // one whole 32-byte sector
            if (cot) {
                float v[12];
#pragma unroll
                for (int i = 0; i < 3; ++i) v[i] = sw[3 * lane + i];
#pragma unroll
                for (int i = 0; i < 9; ++i) v[3 + i] = sw[96 + 9 * lane + i];
                float4* dst = cot + 4 * (size_t)d;
                dst[0] = make_float4(v[0], v[1], v[2], v[3]);
                dst[1] = make_float4(v[4], v[5], v[6], v[7]);
                dst[2] = make_float4(v[8], v[9], v[10], v[11]);
                dst[3] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
    }
}

template <typename CT, typename AT, typename TR>
int dispatch_order(bspline_plan_s* p, const void* coeffs, Ws<TR> w, BrickGrid g, void* out_u,
                   void* out_grad, bool grad, unsigned below) {
    switch (p->order) {
        case 2: return run_gather<2, CT, AT, TR>(p, coeffs, w, g, out_u, out_grad, grad, below);
        case 3: return run_gather<3, CT, AT, TR>(p, coeffs, w, g, out_u, out_grad, grad, below);
        case 4: return run_gather<4, CT, AT, TR>(p, coeffs, w, g, out_u, out_grad, grad, below);
        case 5: return run_gather<5, CT, AT, TR>(p, coeffs, w, g, out_u, out_grad, grad, below);
        case 6: return run_gather<6, CT, AT, TR>(p, coeffs, w, g, out_u, out_grad, grad, below);
        case 7: return run_gather<7, CT, AT, TR>(p, coeffs, w, g, out_u, out_grad, grad, below);
        case 8: return run_gather<8, CT, AT, TR>(p, coeffs, w, g, out_u, out_grad, grad, below);
    }
    return BSPLINE_ERR_UNSUPPORTED_ORDER;
}

template <typename CT, typename AT, typename TR>
int dispatch_points(bspline_plan_s* p, const void* coeffs, const double* x, int64_t P, Ws<TR> w, unsigned NB,
                    void* out_u, void* out_grad, bool grad) {
    switch (p->order) {
        case 2: return run_gather_points<2, CT, AT, TR>(p, coeffs, x, P, w, NB, out_u, out_grad, grad);
        case 3: return run_gather_points<3, CT, AT, TR>(p, coeffs, x, P, w, NB, out_u, out_grad, grad);
        case 4: return run_gather_points<4, CT, AT, TR>(p, coeffs, x, P, w, NB, out_u, out_grad, grad);
        case 5: return run_gather_points<5, CT, AT, TR>(p, coeffs, x, P, w, NB, out_u, out_grad, grad);
        case 6: return run_gather_points<6, CT, AT, TR>(p, coeffs, x, P, w, NB, out_u, out_grad, grad);
        case 7: return run_gather_points<7, CT, AT, TR>(p, coeffs, x, P, w, NB, out_u, out_grad, grad);
        case 8: return run_gather_points<8, CT, AT, TR>(p, coeffs, x, P, w, NB, out_u, out_grad, grad);
    }
    return BSPLINE_ERR_UNSUPPORTED_ORDER;
}

inline unsigned grid_for(long long P, int threads) {
    long long g = (P + threads - 1) / threads;
    if (g > (1LL << 30)) g = 1LL << 30;
    return (unsigned)(g < 1 ? 1 : g);
}

// The count pass; returns whether it ranked the particles.  Through shared-memory histograms where the bricks
// are no more than a run's particles (the run, up to 8192, shrinks with P so that every SM gets two) or so few
// that clustered particles queue for their counters: 2^22
// particles, count + placement, 86 + 220 -> 63 + 223 us on 256^3 in the adjoint (5632 bricks, the cotangents'
// copies bound the placement), 455 + 465 -> 55 + 76 us clustered on 128^3 (704 bricks, whose counters the
// warps queued for).  Else an atomic a particle and pass: at 512^3 (44032 bricks, 2^24 particles) places
// returned by the count's atomics made the step 1.5 % slower; at 5632 bricks and 10^6 particles the runs
// (3328) gain nothing.  Few particles do not repay the zeroing and flushing of the bins (FP64 u at order 2, atomics /
// histogram, us a call: 64 bricks, 4000 particles 30.2 / 33.1, 16000 37.2 / 35.5, and 10^4 beside the transform at order 4
// 45.9 / 44.2; 512 bricks, 16000 36.8 / 38.6, 64000 58.5 / 49.3; 4096 bricks, 64000 54.6 / 63.0, 256000 109.6 / 110.3, 10^6 310 / 293).  Never for sorted input: a warp's
// particles share a brick or two, one atomic each, and nothing is placed afterwards (FP32, 64^3 in brick order,
// histogram / warp: 2000 particles, order 4, 34.6 / 29.3 us a call; 50000 41.7 / 36.3; 10^6, order 2, 111 / 103).
template <typename TR, bool SORTED, typename OT>
bool launch_bin(bspline_plan_s* p, const double* x, int64_t P, const BrickGrid& g, const Ws<TR>& w, OT* ou, OT* og,
                unsigned grid, unsigned long long* status, cudaStream_t st) {
    const double scale = (double)p->N / p->L;
    if constexpr (!SORTED) {
        if (counts_by_runs(P, g.NB, p->sms)) {
            const unsigned run = count_run_length(P, p->sms);
            const size_t sm = sizeof(unsigned) * (g.NB + 1 + run);
            auto k = bin_kernel<TR, false, true, OT>;
            if (set_smem(k, sm) == BSPLINE_OK) {
                const unsigned runs = (unsigned)((P + run - 1) / run);
                k<<<std::min(runs, grid), 256, sm, st>>>(x, P, p->N, scale, p->order, g, w, status, run, ou, og);
                return true;
            }
        }
    }
    bin_kernel<TR, SORTED, false, OT><<<grid, 256, 0, st>>>(x, P, p->N, scale, p->order, g, w, status, 0u, ou, og);
    return false;
}

// Whether a call evaluates its particles in the caller's order, each straight from global memory
// (gather_points), instead of sorting them.  The direct gather costs about 0.0035 n^3 ns a particle while
// the coefficients stay in L2 and two to three times that beyond; the sorted calls cost 25 to 100 us of
// launches and passes and then 0.3 ns a particle.  Measured (us, unsorted / sorted, FP32): 64^3 order 4,
// 10^3 particles 13 / 26; 128^3 order 6, 16000 20 / 41, 64000 56 / 59, 256000 197 / 124; 256^3 order 4,
// 64000 46 / 63, 256000 161 / 138; 512^3 order 6, 64000 157 / 179; 256^3 order 2, 10^6 161 / 224.
// Beside a transform (bspline_eval, bspline_run_host) the sort hides behind it and only the two gathers
// compare: a quarter of the bound (96^3 order 5 BF16, 64312 particles, eval: sorted 65, unsorted 73).
constexpr long long kUnsortedNodes = 12LL << 20;        // particles times n^3
bool unsorted_call(const bspline_plan_s* p, int64_t P, int flags, bool beside) {
    if (p->dtype == BSPLINE_F64 || (flags & BSPLINE_INTERP_SORTED)) return false;
    if (p->direct_below != BSPLINE_GATHER_SPLIT_AUTO && p->direct_below != 0xffffffffu) return false;
    return P * p->order * p->order * p->order <= (beside ? kUnsortedNodes / 4 : kUnsortedNodes);
}

// The automatic split: a staged brick costs as much as about 4096 / n^3 particles of the direct gather; a
// call whose bricks hold fewer than that on average is split there, a denser one is staged throughout.
// Measured (us, every brick direct / staged, FP32): 512^3, 24 particles a brick: order 2 296 / 667, order 4
// 481 / 763, order 6 956 / 888; 256^3, 45 a brick: order 3 100 / 130, order 4 129 / 138, order 6 268 / 171.
unsigned auto_split(int64_t P, unsigned NB, int n) {
    const unsigned below = 4096u / (unsigned)(n * n * n);
    return P < (long long)below * NB ? below : 0u;
}

// The evaluation of such a call: the direct gather on the plan's stream, no workspace.
template <typename CT, typename AT, typename TR>
int run_points(bspline_plan_s* p, const void* coeffs, const double* x, int64_t P, void* out_u, void* out_grad,
               int flags) {
    const cudaError_t e = cudaMemsetAsync(p->d_status, 0, sizeof(unsigned long long) * kStatusParticleWords, p->stream);
    if (e != cudaSuccess) return set_cuda_error(e);
    StageTimer tm(p, BSPLINE_STAGE_GATHER_DIRECT);
    const int rc = dispatch_points<CT, AT, TR>(p, coeffs, x, P, Ws<TR>{}, 0u, out_u, out_grad,
                                               !(flags & BSPLINE_INTERP_NO_GRAD));
    return rc ? rc : set_cuda_error(cudaGetLastError());
}

// The sort (bin, scan, scatter) runs on sort_stream when one is given (it
// needs only the positions) and the gather on the plan's stream after `sorted`.
template <typename CT, typename AT, typename TR>
int run_interp(bspline_plan_s* p, const void* coeffs, const double* x, int64_t P, void* out_u, void* out_grad,
               int flags, cudaStream_t sort_stream, cudaEvent_t sorted) {
    if (unsorted_call(p, P, flags, sort_stream != nullptr)) {
        if (sort_stream) {                              // the positions may arrive on that stream
            cudaError_t e = cudaEventRecord(sorted, sort_stream);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(p->stream, sorted, 0);
            if (e != cudaSuccess) return set_cuda_error(e);
        }
        return run_points<CT, AT, TR>(p, coeffs, x, P, out_u, out_grad, flags);
    }
    const BrickGrid g = brick_grid(p->N, p->dtype, p->order);
    const unsigned NB = g.NB;
    Ws<TR> w;
    const unsigned len = item_particles(p->dtype, p->order, P, NB);
    const bool ranks = counts_by_runs(P, NB, p->sms);
    const size_t need = carve<TR>(&w, nullptr, NB, P, ranks, shortest_item(p->dtype));
    int rc = p->pws.grow(need);
    if (rc) return rc;
    carve<TR>(&w, p->pws.ptr, NB, P, ranks, shortest_item(p->dtype));
    const cudaStream_t main_stream = p->stream;
    cudaStream_t st = sort_stream ? sort_stream : main_stream;
    p->stream = st;                                     // stage timers follow the sort's stream
    struct Restore {
        bspline_plan_s* p;
        cudaStream_t s;
        ~Restore() { p->stream = s; }
    } restore{p, main_stream};
    cudaError_t e;
    if ((e = cudaMemsetAsync(w.count, 0, sizeof(unsigned) * (NB + 2), st)) != cudaSuccess) return set_cuda_error(e);
    if ((e = cudaMemsetAsync(p->d_status, 0, sizeof(unsigned long long) * kStatusParticleWords, st)) != cudaSuccess)
        return set_cuda_error(e);                       // non-finite count, tile-wait flag, checks
    const bool grad = !(flags & BSPLINE_INTERP_NO_GRAD);
    const bool presorted = (flags & BSPLINE_INTERP_SORTED) != 0;
    const double scale = (double)p->N / p->L;
    AT* ou = (AT*)out_u;
    AT* og = grad ? (AT*)out_grad : nullptr;
    // Beside the transform (sort_stream given), the locate passes run as a small grid-stride grid, two
    // 256-thread CTAs per SM: they then share the SMs with the transform's CTAs instead of taking them in
    // turn, and use the HBM bandwidth the transform leaves (512^3, 2^24 particles: 5.33 -> 5.04 ms per
    // step; one CTA per SM or more than three were slower).  Alone, the full grid is faster.
    unsigned sort_grid = grid_for(P, 256);
    if (sort_stream && 2LL * p->sms < (long long)sort_grid) sort_grid = (unsigned)(2 * p->sms);
    // bricks with fewer particles than this go to the direct gather (FP32 accumulation only)
    unsigned below = p->direct_below;
    if (below == BSPLINE_GATHER_SPLIT_AUTO) below = auto_split(P, NB, p->order);
    if (sizeof(AT) == 8 || presorted) below = 0u;       // sorted input: bricks stay in input order
    bool ranked;
    {
        StageTimer tm(p, BSPLINE_STAGE_BIN);
        ranked = presorted ? launch_bin<TR, true, AT>(p, x, P, g, w, ou, og, sort_grid, p->d_status, st)
                           : launch_bin<TR, false, AT>(p, x, P, g, w, ou, og, sort_grid, p->d_status, st);
    }
    {
        StageTimer tm(p, BSPLINE_STAGE_SCAN);
        launch_scan<TR>(w, NB, below, len, P, st);
    }
    {
        StageTimer tm(p, BSPLINE_STAGE_SCATTER);
        if (presorted)
            scatter_kernel<TR, AT, true><<<sort_grid, 256, 0, st>>>(x, P, p->N, scale, p->order, g, w, ou, og,
                                                                    ranked, p->d_status);
        else
            scatter_kernel<TR, AT><<<sort_grid, 256, 0, st>>>(x, P, p->N, scale, p->order, g, w, ou, og, ranked, p->d_status);
    }
    if (sort_stream) {
        if ((e = cudaEventRecord(sorted, sort_stream)) != cudaSuccess) return set_cuda_error(e);
        if ((e = cudaStreamWaitEvent(main_stream, sorted, 0)) != cudaSuccess) return set_cuda_error(e);
    }
    p->stream = main_stream;
    {
        StageTimer tm(p, BSPLINE_STAGE_GATHER);
        rc = dispatch_order<CT, AT, TR>(p, coeffs, w, g, out_u, out_grad, grad, below);
    }
    if (rc) return rc;
    if (below > 0) {
        StageTimer tm(p, BSPLINE_STAGE_GATHER_DIRECT);
        rc = dispatch_points<CT, AT, TR>(p, coeffs, nullptr, P, w, NB, out_u, out_grad, grad);
    }
    if (rc) return rc;
    return set_cuda_error(cudaGetLastError());
}

// Same launch sequence as run_interp, with the workspace and the status word
// supplied by the caller instead of the plan.
template <typename CT, typename AT, typename TR>
int run_interp_ws(bspline_plan_s* p, void* ws, unsigned long long* status, const void* coeffs, const double* x,
                  int64_t P, void* out_u, void* out_grad, int flags) {
    if (unsorted_call(p, P, flags, false)) return run_points<CT, AT, TR>(p, coeffs, x, P, out_u, out_grad, flags);
    const BrickGrid g = brick_grid(p->N, p->dtype, p->order);
    const unsigned NB = g.NB;
    Ws<TR> w;
    const unsigned len = item_particles(p->dtype, p->order, P, NB);
    carve<TR>(&w, ws, NB, P, counts_by_runs(P, NB, p->sms), shortest_item(p->dtype));
    cudaStream_t st = p->stream;
    cudaError_t e;
    if ((e = cudaMemsetAsync(w.count, 0, sizeof(unsigned) * (NB + 2), st)) != cudaSuccess) return set_cuda_error(e);
    if ((e = cudaMemsetAsync(status, 0, sizeof(unsigned long long) * kStatusParticleWords, st)) != cudaSuccess)
        return set_cuda_error(e);                       // non-finite count, tile-wait flag, checks
    const bool grad = !(flags & BSPLINE_INTERP_NO_GRAD);
    const bool ranked = launch_bin<TR, false, AT>(p, x, P, g, w, nullptr, nullptr, grid_for(P, 256), status, st);
    launch_scan<TR>(w, NB, 0u, len, P, st);
    scatter_kernel<TR, AT><<<grid_for(P, 256), 256, 0, st>>>(x, P, p->N, (double)p->N / p->L, p->order, g, w, (AT*)out_u, grad ? (AT*)out_grad : nullptr,
                                                             ranked, status);
    int rc = dispatch_order<CT, AT, TR>(p, coeffs, w, g, out_u, out_grad, grad, 0u);
    if (rc) return rc;
    return set_cuda_error(cudaGetLastError());
}

template <typename CT, typename TR>
int adjoint_order(bspline_plan_s* p, const void* coeffs, Ws<TR> w, BrickGrid g, long long items,
                  const void* g_u, const void* g_grad, void* g_coef, double* g_x, const float4* cot) {
    using adjoint_impl::run_adjoint;
    switch (p->order) {
        case 2: return run_adjoint<2, CT, TR>(p, coeffs, w, g, items, g_u, g_grad, g_coef, g_x, cot);
        case 3: return run_adjoint<3, CT, TR>(p, coeffs, w, g, items, g_u, g_grad, g_coef, g_x, cot);
        case 4: return run_adjoint<4, CT, TR>(p, coeffs, w, g, items, g_u, g_grad, g_coef, g_x, cot);
        case 5: return run_adjoint<5, CT, TR>(p, coeffs, w, g, items, g_u, g_grad, g_coef, g_x, cot);
        case 6: return run_adjoint<6, CT, TR>(p, coeffs, w, g, items, g_u, g_grad, g_coef, g_x, cot);
        case 7: return run_adjoint<7, CT, TR>(p, coeffs, w, g, items, g_u, g_grad, g_coef, g_x, cot);
        case 8: return run_adjoint<8, CT, TR>(p, coeffs, w, g, items, g_u, g_grad, g_coef, g_x, cot);
    }
    return BSPLINE_ERR_UNSUPPORTED_ORDER;
}

// Adjoint of the particle side: the same bin / scan / scatter as run_interp,
// then the spread into g_coef and the position gradient g_x (either may be
// skipped).  Non-finite positions contribute nothing and get NaN in g_x.
template <typename CT, typename TR>
int run_adjoint_particles(bspline_plan_s* p, const void* coeffs, const double* x, int64_t P, const void* g_u,
                          const void* g_grad, void* g_coef, double* g_x) {
    const BrickGrid g = brick_grid(p->N, p->dtype, p->order);
    const unsigned NB = g.NB;
    Ws<TR> w;
    const bool ranks = counts_by_runs(P, NB, p->sms);
    const size_t need = carve<TR>(&w, nullptr, NB, P, ranks);
    int rc = p->pws.grow(need);
    if (rc) return rc;
    carve<TR>(&w, p->pws.ptr, NB, P, ranks);
    // FP32 types: the placement pass also copies each particle's cotangents to its sorted slot, which the
    // spread and the position gradients then read in order instead of gathering them from random indices
    float4* cot = nullptr;
    if (sizeof(TR) == 4 && (g_u || g_grad) && (g_coef || g_x)) {
        if ((rc = p->cot.grow(sizeof(float4) * 4 * (size_t)P))) return rc;
        cot = reinterpret_cast<float4*>(p->cot.ptr);
    }
    cudaStream_t st = p->stream;
    cudaError_t e;
    if ((e = cudaMemsetAsync(w.count, 0, sizeof(unsigned) * (NB + 2), st)) != cudaSuccess) return set_cuda_error(e);
    if ((e = cudaMemsetAsync(p->d_status, 0, sizeof(unsigned long long) * kStatusParticleWords, st)) != cudaSuccess)
        return set_cuda_error(e);                       // non-finite count, tile-wait flag, checks
    bool ranked;
    {
        StageTimer tm(p, BSPLINE_STAGE_BIN);
        ranked = launch_bin<TR, false, double>(p, x, P, g, w, nullptr, nullptr, grid_for(P, 256), p->d_status, st);
    }
    {
        StageTimer tm(p, BSPLINE_STAGE_SCAN);
        launch_scan<TR>(w, NB, 0u, kChunk, P, st);
    }
    {
        StageTimer tm(p, BSPLINE_STAGE_SCATTER);
        const size_t cot_smem = cot ? sizeof(float) * 12 * 256 : 0;   // 12 * 32 floats per warp
        scatter_kernel<TR, double><<<grid_for(P, 256), 256, cot_smem, st>>>(x, P, p->N, (double)p->N / p->L, p->order, g, w, g_x, nullptr, ranked,
                                                                     p->d_status, nullptr, (const float*)g_u,
                                                                     (const float*)g_grad, cot);
    }
    const long long items = (long long)NB + (P + kChunk - 1) / kChunk;
    if (g_coef && p->deterministic && sizeof(TR) == 4) {
        // the fixed-point accumulator of the deterministic spread and its bound word
        if ((rc = p->det.grow(sizeof(long long) * 3 * (size_t)p->N * p->N * p->N + 16))) return rc;
    }
    if (g_coef) {
        StageTimer tm(p, BSPLINE_STAGE_SPREAD);
        rc = adjoint_order<CT, TR>(p, coeffs, w, g, items, g_u, g_grad, g_coef, nullptr, cot);
        if (rc) return rc;
    }
    if (g_x) {
        StageTimer tm(p, BSPLINE_STAGE_GRAD_X);
        rc = adjoint_order<CT, TR>(p, coeffs, w, g, items, g_u, g_grad, nullptr, g_x, cot);
        if (rc) return rc;
    }
    return set_cuda_error(cudaGetLastError());
}

// Brick order of the particles (bspline_sort_order): count, scan, then each
// particle's original index written to its sorted slot.
template <typename TR>
int run_sort_order(bspline_plan_s* p, const double* x, int64_t P, int* perm) {
    const BrickGrid g = brick_grid(p->N, p->dtype, p->order);
    const unsigned NB = g.NB;
    Ws<TR> w;
    const bool ranks = counts_by_runs(P, NB, p->sms);
    const size_t need = carve<TR>(&w, nullptr, NB, P, ranks);
    int rc = p->pws.grow(need);
    if (rc) return rc;
    carve<TR>(&w, p->pws.ptr, NB, P, ranks);
    cudaStream_t st = p->stream;
    cudaError_t e;
    if ((e = cudaMemsetAsync(w.count, 0, sizeof(unsigned) * (NB + 2), st)) != cudaSuccess) return set_cuda_error(e);
    if ((e = cudaMemsetAsync(p->d_status, 0, sizeof(unsigned long long) * kStatusParticleWords, st)) != cudaSuccess)
        return set_cuda_error(e);
    const double scale = (double)p->N / p->L;
    const bool ranked = launch_bin<TR, false, float>(p, x, P, g, w, nullptr, nullptr, grid_for(P, 256), p->d_status, st);
    launch_scan<TR>(w, NB, 0u, kChunk, P, st);
    scatter_kernel<TR, float, false, true><<<grid_for(P, 256), 256, 0, st>>>(x, P, p->N, scale, p->order, g, w,
                                                                            (float*)nullptr, (float*)nullptr,
                                                                            ranked, p->d_status, perm);
    return set_cuda_error(cudaGetLastError());
}

}  // namespace

int launch_sort_order(bspline_plan_s* p, const double* x, int64_t P, int* perm) {
    if (p->dtype == BSPLINE_F64) return run_sort_order<double>(p, x, P, perm);
    return run_sort_order<float>(p, x, P, perm);
}

int launch_adjoint_particles(bspline_plan_s* p, const void* coeffs, const double* x, int64_t P, const void* g_u,
                             const void* g_grad, void* g_coef, double* g_x) {
    switch (p->dtype) {
        case BSPLINE_F64:
            return run_adjoint_particles<double, double>(p, coeffs, x, P, g_u, g_grad, g_coef, g_x);
        case BSPLINE_F32:
            return run_adjoint_particles<float, float>(p, coeffs, x, P, g_u, g_grad, g_coef, g_x);
        case BSPLINE_BF16:
            return run_adjoint_particles<__nv_bfloat16, float>(p, coeffs, x, P, g_u, g_grad, g_coef, g_x);
    }
    return BSPLINE_ERR_INVALID_ARG;
}

int launch_interp_ws(bspline_plan_s* p, void* ws, unsigned long long* status, const void* coeffs, const double* x,
                     int64_t P, void* out_u, void* out_grad, int flags) {
    switch (p->dtype) {
        case BSPLINE_F64:
            return run_interp_ws<double, double, double>(p, ws, status, coeffs, x, P, out_u, out_grad, flags);
        case BSPLINE_F32:
            return run_interp_ws<float, float, float>(p, ws, status, coeffs, x, P, out_u, out_grad, flags);
        case BSPLINE_BF16:
            return run_interp_ws<__nv_bfloat16, float, float>(p, ws, status, coeffs, x, P, out_u, out_grad, flags);
    }
    return BSPLINE_ERR_INVALID_ARG;
}

size_t interp_workspace_bytes(const bspline_plan_s* p, int64_t P) {
    const BrickGrid g = brick_grid(p->N, p->dtype, p->order);
    const unsigned NB = g.NB;
    const bool ranks = counts_by_runs(P, NB, p->sms);
    if (p->dtype == BSPLINE_F64) {
        Ws<double> w;
        return carve<double>(&w, nullptr, NB, P, ranks, shortest_item(p->dtype));
    }
    Ws<float> w;
    return carve<float>(&w, nullptr, NB, P, ranks, shortest_item(p->dtype));
}

int launch_interp_split(bspline_plan_s* p, const void* coeffs, const double* x, int64_t P, void* out_u,
                        void* out_grad, int flags, cudaStream_t sort_stream, cudaEvent_t sorted) {
    switch (p->dtype) {
        case BSPLINE_F64:
            return run_interp<double, double, double>(p, coeffs, x, P, out_u, out_grad, flags, sort_stream, sorted);
        case BSPLINE_F32:
            return run_interp<float, float, float>(p, coeffs, x, P, out_u, out_grad, flags, sort_stream, sorted);
        case BSPLINE_BF16:
            return run_interp<__nv_bfloat16, float, float>(p, coeffs, x, P, out_u, out_grad, flags, sort_stream,
                                                           sorted);
    }
    return BSPLINE_ERR_INVALID_ARG;
}

bool interp_sorts(const bspline_plan_s* p, int64_t P, int flags) { return !unsorted_call(p, P, flags, false); }
bool eval_sorts(const bspline_plan_s* p, int64_t P, int flags) { return !unsorted_call(p, P, flags, true); }

int launch_interp(bspline_plan_s* p, const void* coeffs, const double* x, int64_t P, void* out_u, void* out_grad,
                  int flags) {
    return launch_interp_split(p, coeffs, x, P, out_u, out_grad, flags, nullptr, nullptr);
}

}  // namespace bs
