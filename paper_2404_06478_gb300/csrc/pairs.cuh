// pairs.cuh — shared pieces of the pair passes (Sinkhorn, M-step, adjoint):
// the packed pair evaluation, the online log-sum-exp, the dustbin scalars and
// the cone bounds of the exact skipping.
#pragma once

#include "common.cuh"
#include "kernels.h"

namespace laue {

constexpr int kGran = kConeGran;  // pairs per cone granule of the exact skipping
constexpr int kGroup = 4;     // staged pairs per max-then-sum group
constexpr float kPadFar = 1.0e6f;

struct DustPtrs {
    float *F0, *F0n, *G0, *log2U, *log2O, *Fmax, *Gmax, *err;
};

__device__ __forceinline__ DustPtrs dust_ptrs(float* base, int T) {
    DustPtrs d;
    d.F0 = base;
    d.F0n = base + T;
    d.G0 = base + 2 * T;
    d.log2U = base + 3 * T;
    d.log2O = base + 4 * T;
    d.Fmax = base + 5 * T;  // per-angle max of F (row potentials)
    d.Gmax = base + 6 * T;  // per-angle max of G (column potentials)
    d.err = base + 7 * T;
    return d;
}

// Packed pair value base + K |(p - c)/|p - c| - r|^2 for two pairs at once;
// nc = -c, nr = -r.  13 packed instructions and 2 MUFU rsqrt.
__device__ __forceinline__ f2 pair_v2(f2 px, f2 py, f2 pz, f2 ncx, f2 ncy, f2 ncz, f2 nrx, f2 nry, f2 nrz,
                                      f2 K2, f2 base) {
    f2 dx = add2(px, ncx), dy = add2(py, ncy), dz = add2(pz, ncz);
    f2 q = mul2(dx, dx);
    q = fma2(dy, dy, q);
    q = fma2(dz, dz, q);
    f2 s = pk(rsq(lo(q)), rsq(hi(q)));
    f2 ex = fma2(dx, s, nrx), ey = fma2(dy, s, nry), ez = fma2(dz, s, nrz);
    f2 e2 = mul2(ex, ex);
    e2 = fma2(ey, ey, e2);
    e2 = fma2(ez, ez, e2);
    return fma2(e2, K2, base);
}

// Online base-2 log-sum-exp state of one row: running max m and two packed
// partial sums S (relative to m).
struct RowLse {
    float m;
    f2 S;
    f2 nm;  // {-m, -m}
    __device__ __forceinline__ void init(float v) {
        m = v;
        S = pk(1.0f, 0.0f);
        nm = dup(-v);
    }
    // fold 8 values (4 packed) in: one max / rescale, 8 MUFU ex2
    __device__ __forceinline__ void add4(const f2 (&v)[kGroup]) {
        float c1 = max3(lo(v[0]), hi(v[0]), lo(v[1]));
        float c2 = max3(hi(v[1]), lo(v[2]), hi(v[2]));
        float cm = max3(c1, c2, fmaxf(lo(v[3]), hi(v[3])));
        if (cm > m) {
            float sc = ex2(m - cm);
            S = mul2(S, dup(sc));
            m = cm;
            nm = dup(-cm);
        }
#pragma unroll
        for (int g = 0; g < kGroup; ++g) {
            f2 t = add2(v[g], nm);
            S = add2(S, pk(ex2(lo(t)), ex2(hi(t))));
        }
    }
    __device__ __forceinline__ void add1(f2 v) {
        float cm = fmaxf(lo(v), hi(v));
        if (cm > m) {
            float sc = ex2(m - cm);
            S = mul2(S, dup(sc));
            m = cm;
            nm = dup(-cm);
        }
        f2 t = add2(v, nm);
        S = add2(S, pk(ex2(lo(t)), ex2(hi(t))));
    }
    __device__ __forceinline__ float value() const { return m + lg2(lo(S) + hi(S)); }
};

// Angle block of element k of a list with offsets off[T+1] (binary search).
__device__ __forceinline__ int block_of(const int* __restrict__ off, int T, int k) {
    int lo_ = 0, hi_ = T;
    while (hi_ - lo_ > 1) {
        int mid = (lo_ + hi_) >> 1;
        if (off[mid] <= k) lo_ = mid;
        else hi_ = mid;
    }
    return lo_;
}

// ------------------------------------- exact underflow skipping (cone bounds)
// A granule is kGran pairs of one angle block, a sub-granule kSubGran of them; a
// cone bounds the directions of their spots: for observed spots
// the unit vectors p / |p| and the smallest |p|, for model spots the rays r
// and the largest |c|.  For an observed cone O and a model cone M, every pair
// has an angle between rhat = (p - c)/|p - c| and r of at least
//   th = angle(a_O, a_M) - beta_O - beta_M - asin(c_max / p_min)
// (the direction of p seen from c differs from p/|p| by at most
// asin(|c| / |p|)), so its cost is at least D^2 (2 sin(th/2))^2.
struct Cone {
    float ax, ay, az, beta, ext;  // axis, half-angle (rad), p_min or c_max
};

__device__ __forceinline__ Cone load_cone(const float4* cone, const float* ext, int g) {
    float4 c = cone[g];
    return Cone{c.x, c.y, c.z, c.w, ext[g]};
}

__device__ __forceinline__ float angle_between(float ax, float ay, float az, float bx, float by, float bz) {
    float c = ax * bx + ay * by + az * bz;
    return acosf(fminf(1.0f, fmaxf(-1.0f, c)));
}

// Lower bound of K |rhat - r|^2 (K = D^2 log2(e) / eps) over the pairs of an
// observed cone and a model cone; 0 when the cones may overlap.
__device__ __forceinline__ float min_scaled_cost(const Cone& O, const Cone& M, float K) {
    float sep = angle_between(O.ax, O.ay, O.az, M.ax, M.ay, M.az);
    float off = O.ext > M.ext ? asinf(M.ext / O.ext) : 1.6f;
    float th = sep - O.beta - M.beta - off - 1e-4f;
    if (!(th > 0.0f)) return 0.0f;
    float s = sinf(0.5f * fminf(th, 3.14159f));
    return K * 4.0f * s * s;
}

// Every plan entry of a pair whose shifted exponent is below -kSkipLog2 is
// flushed to exactly 0 by ex2.approx.ftz (below 2^-126), so the sums are
// bit-identical with or without the pair.
constexpr float kSkipLog2 = 130.0f;

__device__ __forceinline__ void lse_merge_into(float& m, float& s, float m2, float s2) {
    Lse2 L;
    L.m = m;
    L.s = s;
    L.merge(m2, s2);
    m = L.m;
    s = L.s;
}

// Column pair (two model spots): negated centres and rays, packed duplicates.
struct ColPair {
    f2 ncxa, ncya, ncza, nrxa, nrya, nrza;
    f2 ncxb, ncyb, nczb, nrxb, nryb, nrzb;
    f2 ka, kb;  // {-K_a, -K_a}, {-K_b, -K_b}: cost factors of the two model spots
};

__device__ __forceinline__ void load_col_pair(const SkArgs& a, int q, ColPair& C) {
    float4 X = a.modX[q], Y = a.modY[q], Z = a.modZ[q], W = a.modW[q];
    C.ncxa = dup(X.x);
    C.ncya = dup(X.z);
    C.ncza = dup(Y.x);
    C.nrxa = dup(Z.x);
    C.nrya = dup(Z.z);
    C.nrza = dup(W.x);
    C.ncxb = dup(X.y);
    C.ncyb = dup(X.w);
    C.nczb = dup(Y.y);
    C.nrxb = dup(Z.y);
    C.nryb = dup(Z.w);
    C.nrzb = dup(W.y);
    C.ka = dup(W.z);
    C.kb = dup(W.w);
}

}  // namespace laue
