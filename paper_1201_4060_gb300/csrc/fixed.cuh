// 60-bit fixed-point arithmetic of the FP64 evaluation.
//
// GB300 sustains 527 G FP64 operations a second (1.7 per clock per SM; measured, fma or add alike) but
// 9000 G 32 x 32 -> 64-bit integer multiply-adds.  The stencil contraction of an FP64 plan is therefore
// done on integers: a number v is held as the integer V = v 2^60 (weights) or v 2^(B - E) (values, 2^E the
// power of two above the largest one of a tile), rounded to nearest, in two limbs
//     V = hi 2^30 + lo,  lo in [-2^29, 2^29),
// and a product sum  sum a b / 2^60  as  H + M 2^-30  with
//     H = sum a.hi b.hi,  M = sum (a.hi b.lo + a.lo b.hi)
// in 64-bit accumulators: three multiply-adds a term.  The omitted lo lo terms are below 2^-2 of the last
// place each.  Bounds that keep every accumulator inside 63 bits and every limb inside 31: weights |b| <= 2^60,
// node weights non-negative with sum 1, derivative weights with sum |b| <= D: 2 at order 3, at most 1.5 from order 4
// on.  Values |a| <= 2^B, sums after the derivative weights <= D 2^B: with B = 60 from order 4 on |hi| <= 1.5 2^30 and, for
// up to 8 terms, |H| <= 1.5 2^60, |M| <= 8 (1.5 2^30) 2^29 + 2^29 (1.5 2^30) < 2^63; B = 59 at order 3.
#pragma once

namespace bs {
namespace fixed {

#define BS_HD __host__ __device__ __forceinline__

constexpr long long kOne = 1LL << 60;
constexpr long long kHalfLimb = 1LL << 29;

struct Limbs {
    int hi, lo;
};

BS_HD Limbs limbs(long long v) {
    const long long r = v + kHalfLimb;
    return {(int)(r >> 30), (int)((unsigned)r & 0x3fffffffu) - (int)kHalfLimb};
}
BS_HD long long value(Limbs a) { return ((long long)a.hi << 30) + a.lo; }

// acc + a b: one 32 x 32 + 64-bit multiply-add.  Written out for the device: from the C expression the
// compiler, which sees the 64-bit origin of the limbs, forms 64-bit products of several instructions.
BS_HD long long mad_wide(int a, int b, long long acc) {
#ifdef __CUDA_ARCH__
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
    return acc;
#else
    return acc + (long long)a * b;
#endif
}

// Accumulator of a product sum.  H starts at half a limb, which is what limbs() adds, and M at the
// rounding of its shift.
struct Acc {
    long long H, M;
    BS_HD void clear() { H = M = kHalfLimb; }
    BS_HD void add(Limbs a, Limbs b) {
        H = mad_wide(a.hi, b.hi, H);
        M = mad_wide(a.hi, b.lo, M);
        M = mad_wide(a.lo, b.hi, M);
    }
    BS_HD long long biased() const { return H + (M >> 30); }          // value + half a limb
    BS_HD long long value() const { return biased() - kHalfLimb; }
    BS_HD Limbs limbs() const {
        const long long r = biased();
        return {(int)(r >> 30), (int)((unsigned)r & 0x3fffffffu) - (int)kHalfLimb};
    }
};

// round(2^60 a / b), 0 <= a <= 7
constexpr long long ratio(int a, int b) { return (((long long)a << 60) + b / 2) / b; }
BS_HD constexpr Limbs ratio_limbs(int a, int b) {
    const long long r = ratio(a, b) + kHalfLimb;
    return {(int)(r >> 30), (int)(r & 0x3fffffff) - (int)kHalfLimb};
}

// Node weights and derivative weights of an order-n stencil at t = T 2^-60 in [0, 1], node 0 leftmost: the
// Cox-de Boor recurrence of bspline_weights (particles.cuh), each step's division by k - 1 folded into its
// three factors,  v[m] <- (t / (k - 1)) (v[m] - v[m - 1]) + (m / (k - 1)) v[m] + ((k - m) / (k - 1)) v[m - 1].
template <int n> BS_HD void weights(long long T, Limbs (&w)[n], Limbs (&dw)[n]) {
    long long v[n];
    Limbs lv[n];
    v[0] = kOne;
    lv[0] = {1 << 30, 0};
    const Limbs lt = limbs(T);
    long long nv[n];
#pragma unroll
    for (int k = 2; k <= n; ++k) {
        Limbs tk = lt;
        if (k > 2) {
            Acc a;
            a.clear();
            a.add(lt, ratio_limbs(1, k - 1));
            tk = a.limbs();
        }
        if (k == n) {
#pragma unroll
            for (int j = 0; j < n; ++j) {
                const int m = n - 1 - j;
                dw[j] = limbs((m < n - 1 ? v[m] : 0) - (m > 0 ? v[m - 1] : 0));
            }
        }
#pragma unroll
        for (int m = 0; m < k; ++m) {
            Acc a;
            a.clear();
            const Limbs z = {0, 0}, vm = m < k - 1 ? lv[m] : z, vl = m > 0 ? lv[m - 1] : z;
            a.add(tk, {vm.hi - vl.hi, vm.lo - vl.lo});
            if (m > 0 && m < k - 1) a.add(ratio_limbs(m, k - 1), vm);
            if (m > 0) a.add(ratio_limbs(k - m, k - 1), vl);
            nv[m] = a.value();
        }
#pragma unroll
        for (int m = 0; m < k; ++m) {
            v[m] = nv[m];
            lv[m] = limbs(nv[m]);
        }
    }
#pragma unroll
    for (int j = 0; j < n; ++j) w[j] = lv[n - 1 - j];
}

BS_HD int exponent_bits(unsigned hi32) { return (int)((hi32 >> 20) & 0x7ffu); }

// Bits of a tile's largest value.
template <int n> constexpr int value_bits() { return n >= 4 ? 60 : 59; }

// The fixed value, rounded to nearest, of the double with words hi32, lo32 when the tile's largest biased
// exponent is emax: v 2^(1022 + bits - emax), |result| <= 2^bits.  emax >= kMinExponent: zeros and subnormals, whose
// implicit significand bit is not zeroed here, are then shifted out.
constexpr int kMinExponent = 128;
BS_HD long long from_double(unsigned hi32, unsigned lo32, int emax, int bits) {
    const int sh = emax - exponent_bits(hi32) + 62 - bits;   // from a significand of 63 bits; one less than the shift
    const long long m = (long long)(((unsigned long long)((hi32 & 0xfffffu) | 0x100000u) << 42) |
                                    ((unsigned long long)lo32 << 10));
    const long long sign = (long long)((int)hi32 >> 31);
    return ((((m ^ sign) - sign) >> (sh < 63 ? sh : 63)) + 1) >> 1;
}

BS_HD unsigned mul_hi(unsigned a, unsigned b) { return (unsigned)(((unsigned long long)a * b) >> 32); }

// One component's sums over the stencil: the value and the three first derivatives in grid units, on the
// values' scale.  at(jx, jy, jz) gives the limbs of a stencil value, wx(jx) the x weight of node jx and its
// derivative weight (hi, lo, hi, lo).  *size: a lower estimate of the weighted sum of magnitudes
// sum w |a| that the results are rounded against, in units of 2^34: the y and x sums of |sum_z w a|, each
// product rounded down.  It does not depend on GRAD.
template <int n, bool GRAD, typename At, typename WX>
BS_HD void contract(At at, WX wx, const Limbs (&wy)[n], const Limbs (&dwy)[n], const Limbs (&wz)[n],
                    const Limbs (&dwz)[n], long long (&out)[4], unsigned* size) {
    Acc u, gx, gy, gz;
    u.clear();
    gx.clear();
    gy.clear();
    gz.clear();
    unsigned sx = 0;
#pragma unroll 1
    for (int jx = 0; jx < n; ++jx) {
        Acc y00, y10, y01;
        y00.clear();
        y10.clear();
        y01.clear();
        unsigned sy = 0;
#pragma unroll
        for (int jy = 0; jy < n; ++jy) {
            Acc z0, z1;
            z0.clear();
            z1.clear();
#pragma unroll
            for (int jz = 0; jz < n; ++jz) {
                const Limbs a = at(jx, jy, jz);
                z0.add(a, wz[jz]);
                if (GRAD) z1.add(a, dwz[jz]);
            }
            const Limbs l0 = z0.limbs();
            y00.add(l0, wy[jy]);
            sy += mul_hi((unsigned)(l0.hi < 0 ? -l0.hi : l0.hi), (unsigned)wy[jy].hi);
            if (GRAD) {
                y10.add(l0, dwy[jy]);
                y01.add(z1.limbs(), wy[jy]);
            }
        }
        const Limbs l00 = y00.limbs();
        const int4 x = wx(jx);
        const Limbs w = {x.x, x.y};
        u.add(l00, w);
        sx += mul_hi(sy, (unsigned)w.hi);
        if (GRAD) {
            gx.add(l00, {x.z, x.w});
            gy.add(y10.limbs(), w);
            gz.add(y01.limbs(), w);
        }
    }
    out[0] = u.value();
    if (GRAD) {
        out[1] = gx.value();
        out[2] = gy.value();
        out[3] = gz.value();
    }
    *size = sx;
}

}  // namespace fixed
}  // namespace bs
