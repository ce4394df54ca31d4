// Fixed-point complex arithmetic of the FP64 transform (fixed.cuh: GB300 runs integer multiply-adds 17
// times as fast as FP64 operations, and 64-bit adds, two instructions, more than 20 times).
//
// A line's values are held as integers T = v 2^p in block floating point.  A value that has summed m of the line's
// modes is, in magnitude, at most m sqrt 2 times the largest component, and at most the line's L1 norm
// sum (|re| + |im|).  The first stage's p keeps the first bound within 2^60.5; p then falls from stage to stage by
// the bits of the radix, until it is the one that keeps the norm within 1.375 2^60 (the first p, where that is
// smaller).  A component that a butterfly forms on the way is at most sqrt 2 times such a value, or half of the first
// bound, so limbs stay below 2^31.  The last stage's unit is then 2^-60.5 to 2^-59.5 of the norm, the earlier ones' are
// finer by what a stage's rounding grows on its way to the result, and the error of a result is a unit or two,
// where a norm is at most sqrt(2 N) times the result's rms.  rms error over rms result of white lines, in 1e-16, by this
// code on a host against 128-bit arithmetic, FP64 stages in brackets: kx and ky pass, N = 64 0.6 (1.6), 256
// 0.8 (2.0), 1024 1.0 (2.2); kz pass 0.7 (1.7), 0.8 (2.0), 1.0 (2.3); lines that fall as k^(-11/6) 0.5 to 1.3 (1.2 to 2.0).
// With the last p from the first stage on, as it was before, a line of comparable modes lost log2 N bits at the
// input: 0.6, 1.6, 5.7 and 1.4, 4.3, 17.7.
// Lines whose largest magnitude is not in 2^[-895, 977], or that hold a NaN or an infinity, make their tile
// take the FP64 stages (the caller).  p depends on the line's values alone.
//
// Bound: integer issue (64-bit adds and the limbs' shifts; the ky/kz pass also by missing instructions).  Measured at
// 256^3, FP64 stages / one scale a line / block floating point: X pass 1.31 / 0.33 / 0.35 ms, ky/kz pass 2.70 / 0.90 / 0.94.
#pragma once
#include "fft_core.cuh"
#include "fixed.cuh"

namespace bs {
namespace fftc {

struct __align__(16) Fx {
    long long x, y;
};

template <long long C> __device__ __forceinline__ long long mul_const(long long v) {
    constexpr long long r = C + fixed::kHalfLimb;
    const fixed::Limbs c = {(int)(r >> 30), (int)(r & 0x3fffffff) - (int)fixed::kHalfLimb};
    fixed::Acc a;
    a.clear();
    a.add(fixed::limbs(v), c);
    return a.value();
}
// round(2^60 / sqrt 2), round(2^60 sqrt(3) / 2)
template <> __device__ __forceinline__ long long mul_sqrt_half(long long v) { return mul_const<815238614083298888LL>(v); }
template <> __device__ __forceinline__ long long mul_half_sqrt3(long long v) { return mul_const<998459311558907194LL>(v); }
template <> __device__ __forceinline__ long long sub_half(long long a, long long s) { return a - ((s + 1) >> 1); }

// A stage's step: a division by 2^bits, rounded to nearest (bits 0 to 3).
struct Step {
    int bits, half;
    __device__ __forceinline__ explicit Step(int b) : bits(b), half((1 << b) >> 1) {}
};
__device__ __forceinline__ Fx rescaled(Fx a, Step s) { return {(a.x + s.half) >> s.bits, (a.y + s.half) >> s.bits}; }
// a times the twiddle w = (re.hi, re.lo, im.hi, im.lo) 2^-60, stepped
__device__ __forceinline__ Fx twiddled(Fx a, int4 w, Step s) {
    const fixed::Limbs ax = fixed::limbs(a.x), ay = fixed::limbs(a.y);
    fixed::Acc re, im;
    re.clear();
    im.clear();
    re.add(ax, {w.x, w.y});
    re.add(ay, {-w.z, -w.w});
    im.add(ax, {w.z, w.w});
    im.add(ay, {w.x, w.y});
    const int bias = s.half - (int)fixed::kHalfLimb;                         // clear() is half a limb
    return {(re.biased() + bias) >> s.bits, (im.biased() + bias) >> s.bits};
}
__device__ __forceinline__ Fx twiddled(Fx a, int4 w) { return twiddled(a, w, Step(0)); }

// Bits that a stage can add: ceil(log2 RADIX).
constexpr int stage_bits(int radix) { return radix == 8 ? 3 : (radix == 2 ? 1 : 2); }
constexpr int steps_between(int L, int from, int to) {
    int bits = 0;
    for (int ns = from; ns < to; ns *= radix_for(L / ns)) bits += stage_bits(radix_for(L / ns));
    return bits;
}
// The steps of a line: `left` bits to go, taken as early as the bounds ask.
struct Steps {
    int left;
    template <int RADIX> __device__ __forceinline__ Step next() {
        const int b = min(left, stage_bits(RADIX));
        left -= b;
        return Step(b);
    }
};

// Scale of a line: emax its largest biased exponent, S an upper bound of its L1 norm in units of
// 2^(emax - 1041) (norm_part summed over its values).
__device__ __forceinline__ unsigned norm_part(unsigned hi32, int emax) {
    const unsigned m = (((hi32 & 0xfffffu) | 0x100000u) >> 2) + 1;
    return (hi32 << 1) ? (m >> min(emax - fixed::exponent_bits(hi32), 31)) + 1 : 0;     // zeros do not count
}
struct LineScale {
    int top = 0;                                         // emax - 20 + ceil(log2(S / 1.375)): the last p is 1081 - top
    int spare = 0;                                       // bits by which the first stage's p is larger
    LineScale() = default;
    __device__ __forceinline__ explicit LineScale(int packed) : top(packed & 0xfff), spare(packed >> 12) {}
    __device__ __forceinline__ int packed() const { return top | (spare << 12); }
    // 2^bits: what a value after the first stage can be over sqrt 2 times the largest component; most: the bits of
    // all later stages
    __device__ __forceinline__ LineScale(int emax, unsigned S, int bits, int most) {
        const int z = __clz((int)S);
        top = S ? emax - 20 + (32 - z) - ((S << z) < 0xb0000000u ? 1 : 0) : 0;
        spare = min(max(top - emax + 1 - bits, 0), most);
    }
    __device__ __forceinline__ Steps steps() const { return {spare}; }
    // its steps that stages of `taken` bits have left over
    __device__ __forceinline__ Steps steps_after(int taken) const { return {max(spare - taken, 0)}; }
    // v 2^(1081 - top + spare), rounded to nearest; emax >= 128, or v = 0
    __device__ __forceinline__ long long in(double v) const {
        const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
        const int e = fixed::exponent_bits(hi);
        const long long m = (long long)(((unsigned long long)((hi & 0xfffffu) | (e ? 0x100000u : 0u)) << 42) |
                                        ((unsigned long long)lo << 10));
        const long long sign = (long long)((int)hi >> 31);
        const int sh = min(top - spare - e + 3, 63);                         // one less than the shift
        return ((((m ^ sign) - sign) >> sh) + 1) >> 1;
    }
    // t 2^-p as a double, rounded to nearest (ties away from zero)
    __device__ __forceinline__ double out(long long t) const {
        const unsigned sign = (unsigned)(t >> 32) & 0x80000000u;
        const unsigned long long a = (unsigned long long)(t < 0 ? -t : t);
        const int z = __clzll((long long)a);
        const unsigned long long n = a << (z & 63);                          // the leading bit at 63
        // the leading bit adds one to the exponent field below it
        const unsigned long long b = ((unsigned long long)(unsigned)(top + 4 - z) << 52) + (n >> 11) + ((n >> 10) & 1u);
        return a ? __hiloint2double((int)((unsigned)(b >> 32) | sign), (int)(unsigned)b) : 0.0;
    }
};

// Reductions over the threads of one line (thread t works on line t % NLINES); red: T / 32 * NLINES words.
// The result is the line's in every one of its threads, in an order that never changes.
template <int NLINES, int T, typename Op> __device__ __forceinline__ unsigned line_reduce(unsigned v, unsigned* red, Op op) {
    static_assert((NLINES & (NLINES - 1)) == 0 && T % 32 == 0, "lines");
#pragma unroll
    for (int d = NLINES; d < 32; d <<= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, d));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int NL = NLINES < 32 ? NLINES : 32;
    if (lane < NL) red[warp * NL + lane] = v;
    __syncthreads();
    v = red[lane % NL];
#pragma unroll
    for (int w = 1; w < T / 32; ++w) v = op(v, red[w * NL + lane % NL]);
    return v;
}

// A line's scale from the high words and low words of its values, which each() hands over one by one, twice
// (the thread's own values of its line).  gain: what the line's L1 norm can be over that of those values (and
// 2^gain_bits what a value of the line can be over their largest component times sqrt 2).  L: its length.
// False, for the whole CTA, if the tile has to take the FP64 stages.  tops[line]: the scales, visible after
// the caller's next barrier.
template <int L, int NLINES, int T, typename Each>
__device__ __forceinline__ bool line_scale(Each each, unsigned gain, int gain_bits, unsigned* red, int* tops, LineScale* scale) {
    unsigned top = 0, low = 0;
    each([&](unsigned hi, unsigned lo) {
        top = max(top, hi & 0x7fffffffu);
        low |= lo;
    });
    top = line_reduce<NLINES, T>(top, red, [](unsigned a, unsigned b) { return max(a, b); });
    const int emax = (int)(top >> 20);
    // a high word of zero may still belong to a subnormal
    const int bad = top ? (emax < fixed::kMinExponent || emax > 2000) : low != 0;
    if (__syncthreads_or(bad)) return false;
    unsigned S = 0;
    each([&](unsigned hi, unsigned) { S += norm_part(hi, emax); });
    S = line_reduce<NLINES, T>(S, red, [](unsigned a, unsigned b) { return a + b; });
    *scale = LineScale(emax, gain * S, stage_bits(radix_for(L)) + gain_bits, steps_between(L, radix_for(L), L));
    if (threadIdx.x < NLINES) tops[threadIdx.x] = scale->packed();
    return true;
}

// stage_first (fft_core.cuh) in fixed point, its values ld(position, line) from global memory held in
// registers while the scale is found.
template <int L, int NLINES, int T, int QS, typename Ld>
__device__ __forceinline__ bool stage_first_fixed(Fx* s, unsigned* red, int* tops, Ld ld, LineScale* scale) {
    constexpr int RADIX = radix_for(L);
    constexpr int NB = (L / RADIX) * NLINES;
    constexpr int BPT = (NB + T - 1) / T;
    static_assert(T % NLINES == 0, "a thread stays on its line");
    const int t = threadIdx.x;
    double2 v[BPT][RADIX];
#pragma unroll
    for (int i = 0; i < BPT; ++i) {
        const int u = t + i * T;
#pragma unroll
        for (int r = 0; r < RADIX; ++r)
            v[i][r] = (NB % T == 0 || u < NB) ? ld(u / NLINES + r * (L / RADIX), u % NLINES) : make_double2(0.0, 0.0);
    }
    const auto each = [&](auto f) {
#pragma unroll
        for (int i = 0; i < BPT; ++i)
#pragma unroll
            for (int r = 0; r < RADIX; ++r) {
                f((unsigned)__double2hiint(v[i][r].x), (unsigned)__double2loint(v[i][r].x));
                f((unsigned)__double2hiint(v[i][r].y), (unsigned)__double2loint(v[i][r].y));
            }
    };
    if (!line_scale<L, NLINES, T>(each, 1, 0, red, tops, scale)) return false;
#pragma unroll
    for (int i = 0; i < BPT; ++i) {
        const int u = t + i * T;
        if (NB % T == 0 || u < NB) {
            const int b = u % NLINES, j = u / NLINES;
            Fx f[RADIX];
#pragma unroll
            for (int r = 0; r < RADIX; ++r) f[r] = {scale->in(v[i][r].x), scale->in(v[i][r].y)};
            butterfly<RADIX>(f);
#pragma unroll
            for (int r = 0; r < RADIX; ++r) s[(j * RADIX + r) * QS + b] = f[r];
        }
    }
    __syncthreads();
    return true;
}

}  // namespace fftc
}  // namespace bs
