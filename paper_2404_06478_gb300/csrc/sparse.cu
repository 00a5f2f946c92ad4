// sparse.cu — the E-step on a sparse plan (paper Section "Working with
// sparse assignment matrices": only the rho nearest neighbours of each spot
// carry assignment weight, so a Sinkhorn update costs rho |J| instead of
// |I| |J|).
//
// Support: each model spot j keeps the rho observed spots of its angle block
// with the smallest pair cost C_ij = D_j^2 |rhat_ij - r_j|^2 (D_j the cost
// length of the spot's detector; ties to the lower observed index); every
// other observed-model entry of the plan is 0, the outlier column and the
// unmatched-model row stay dense.  The records hold
// e2_ij = (D_j / D)^2 |rhat_ij - r_j|^2.  The neighbour lists
// are built once per call from the model list's rays and centres, then
// transposed into rows (CSR by observed spot, ascending model index).  The
// updates are those of the dense passes restricted to the support, in base 2
// with K = D^2 log2(e)/eps and kc = c_out log2(e)/eps:
//   F_i = -LSE2({G_j - K e2_ij : i in N(j)} u {G_0 - kc})
//   G_j = -LSE2({F_i - K e2_ij : i in N(j)} u {F_0})
// and the dustbin updates in the same order as the dense passes.
//
// Work split: the spots of each angle block are cut into tiles of kSpTile;
// one CTA per tile, eight lanes per spot (8-byte {index, e2} records read
// coalesced), sums shifted by the angle block's largest potential.  The
// per-tile partial log-sum-exps of a pass are merged into the dustbin
// potentials by the first blocks of the pass after it, which does not need
// them yet (as for the dense passes), and passes overlap their launches.
#include <algorithm>

#include "api_internal.h"
#include "slices.cuh"

namespace laue {

constexpr int kSpThreads = 256;
constexpr int kSpWarps = kSpThreads / 32;
constexpr int kSpTile = 512;  // spots per tile
constexpr int kKnnThreads = 256;

struct SpDust {
    float *F0, *F0n, *G0, *log2U, *log2O, *err;
};

__device__ __forceinline__ SpDust sp_dust(float* base, int nd) {
    SpDust d;
    d.F0 = base;
    d.F0n = base + nd;
    d.G0 = base + 2 * nd;
    d.log2U = base + 3 * nd;
    d.log2O = base + 4 * nd;
    d.err = base + 5 * nd;
    return d;
}

// running-maximum log-sum-exp accumulation of one term
__device__ __forceinline__ void acc_lse(float& m, float& s, float v) {
    if (v > m) {
        s = s * ex2(m - v) + 1.0f;
        m = v;
    } else {
        s += ex2(v - m);
    }
}

// |rhat - r|^2 for one pair (the scalar form of the dense passes' cost)
__device__ __forceinline__ float sp_e2(float4 p, float4 c, float4 r) {
    float dx = p.x - c.x, dy = p.y - c.y, dz = p.z - c.z;
    float s = rsq(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
    float ex = fmaf(dx, s, -r.x), ey = fmaf(dy, s, -r.y), ez = fmaf(dz, s, -r.z);
    return fmaf(ex, ex, fmaf(ey, ey, ez * ez));
}

// ---------------------------------------------------------------- schedule
// One CTA: tiles of every angle (rt_base / ct_base their prefix).
__global__ void __launch_bounds__(1024) sp_schedule_kernel(SpArgs a) {
    __shared__ int warp_sum[2][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int base[2] = {0, 0};
    for (int t0 = 0; t0 < a.T; t0 += 1024) {
        const int t = t0 + threadIdx.x;
        int incl[2], c[2];
        for (int k = 0; k < 2; ++k) {
            const int* off = k ? a.J_off : a.I_off;
            c[k] = t < a.T ? (off[t + 1] - off[t] + kSpTile - 1) / kSpTile : 0;
            incl[k] = c[k];
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl[k], o);
                if (lane >= o) incl[k] += y;
            }
            if (lane == 31) warp_sum[k][w] = incl[k];
        }
        __syncthreads();
        for (int k = 0; k < 2; ++k) {
            int before = base[k], all = 0;
            for (int u = 0; u < 32; ++u) {
                if (u < w) before += warp_sum[k][u];
                all += warp_sum[k][u];
            }
            if (t < a.T) (k ? a.ct_base : a.rt_base)[t] = before + incl[k] - c[k];
            base[k] += all;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        a.rt_base[a.T] = base[0];
        a.ct_base[a.T] = base[1];
    }
    __syncthreads();
    for (int k = 0; k < 2; ++k) {
        const int *off = k ? a.J_off : a.I_off, *tb = k ? a.ct_base : a.rt_base;
        int4* tile = k ? a.ctile : a.rtile;
        for (int q = threadIdx.x; q < base[k]; q += 1024) {
            const int t = block_of(tb, a.T, q), s = off[t] + (q - tb[t]) * kSpTile;
            tile[q] = make_int4(t, s, min(s + kSpTile, off[t + 1]), 0);
        }
    }
}

// ------------------------------------------------------------- neighbours
// Inserts (i, v) into the sorted list L of n <= rho entries (an equal e2 goes
// after: its index is larger); worst becomes the largest kept e2 once the list
// is full.
__device__ __forceinline__ void knn_insert(int2* L, int rho, int& n, float& worst, int i, float v) {
    int q = n < rho ? n++ : rho - 1;
    while (q > 0 && __int_as_float(L[q - 1].y) > v) {
        L[q] = L[q - 1];
        --q;
    }
    L[q] = make_int2(i, __float_as_int(v));
    if (n == rho) worst = __int_as_float(L[rho - 1].y);
}

// One thread per model spot (column tiles): the rho smallest e2 over its
// block's observed spots in shared memory, kept sorted by (e2, index).
__global__ void __launch_bounds__(kKnnThreads) sp_knn_kernel(SpArgs a) {
    extern __shared__ int2 sp_heap[];
    if ((int)blockIdx.x >= a.ct_base[a.T]) return;
    const int4 td = a.ctile[blockIdx.x];
    const int i0 = a.I_off[td.x], i1 = a.I_off[td.x + 1];
    int2* L = sp_heap + (size_t)threadIdx.x * a.rho;
    for (int j = td.y + threadIdx.x; j < td.z; j += kKnnThreads) {
        const float4 c = a.c[j], r = a.r[j];
        int n = 0;
        float worst = 3.0e38f;  // the list's largest e2 once it holds rho entries
        int i = i0;
        for (; i + 4 <= i1; i += 4) {  // four independent costs, then the rare insertions in index order
            float v0 = sp_e2(a.p[i], c, r), v1 = sp_e2(a.p[i + 1], c, r);
            float v2 = sp_e2(a.p[i + 2], c, r), v3 = sp_e2(a.p[i + 3], c, r);
            if (v0 < worst) knn_insert(L, a.rho, n, worst, i, v0);
            if (v1 < worst) knn_insert(L, a.rho, n, worst, i + 1, v1);
            if (v2 < worst) knn_insert(L, a.rho, n, worst, i + 2, v2);
            if (v3 < worst) knn_insert(L, a.rho, n, worst, i + 3, v3);
        }
        for (; i < i1; ++i) {
            float v = sp_e2(a.p[i], c, r);
            if (v < worst) knn_insert(L, a.rho, n, worst, i, v);
        }
        const int det = a.s ? (int)a.s[j].w : -1;
        const float kd = (det >= 0 && det < a.n_det) ? a.kdet[det] : 1.0f;
        int2* out = a.cent + (size_t)j * a.rho;
        for (int k = 0; k < a.rho; ++k)
            out[k] = k < n ? make_int2(L[k].x, __float_as_int(__int_as_float(L[k].y) * kd)) : make_int2(-1, 0);
        if (a.nbr_out)
            for (int k = 0; k < a.rho; ++k) a.nbr_out[(size_t)j * a.rho + k] = k < n ? L[k].x : -1;
    }
}

// The same lists where the workspace has room for the direction order and the
// cones of the dense passes (k: a warp's 32 model spots of one granule): only
// the observed sub-granules that the granule can see within an angle are
// searched, an angle that should hold about twice rho spots at the block's
// density; a warp with a spot that has fewer than rho neighbours inside it
// searches again with a wider one.  The pairs come in the order of directions,
// so an insertion compares (e2, index) and the lists are those of the search
// over every pair.
struct KnnStage {
    float4 p[2][32];  // observed spots of a batch: x, y, z, caller's index
};

__global__ void __launch_bounds__(128) sp_knn_cone_kernel(SpArgs a, SkArgs k) {
    extern __shared__ __align__(16) char knn_smem[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    KnnStage& S = ((KnnStage*)knn_smem)[w];
    int2* L = (int2*)(knn_smem + 4 * sizeof(KnnStage)) + (size_t)w * 32 * a.rho + lane;  // entry q at L[32 q]
    const int half = blockIdx.x * 4 + w, g = half >> 1;
    if (g >= k.mod_gbase[a.T]) return;
    const int t = block_of(k.mod_gbase, a.T, g);
    const int rank = 64 * (g - k.mod_gbase[t]) + 32 * (half & 1) + lane;
    const int nj = a.J_off[t + 1] - a.J_off[t], i0 = a.I_off[t], ni = a.I_off[t + 1] - i0;
    const bool valid = rank < nj;
    if (!__any_sync(0xffffffffu, valid)) return;
    const int j = valid ? k.mod_perm[a.J_off[t] + rank] : k.mod_perm[a.J_off[t]];
    const float4 c = a.c[j], r = a.r[j];
    const Cone own = load_cone(k.mod_cone, k.mod_ext, g);
    const float4* sub = k.obs_sub + (size_t)kSubs * k.obs_gbase[t];
    const float* ext = k.obs_subext + (size_t)kSubs * k.obs_gbase[t];
    const int np = k.I2_off[t + 1] - k.I2_off[t];
    const int want = min(a.rho, ni);
    // two detectors see about 2 sr
    float th = sqrtf(2.0f * 2.0f * (float)a.rho / (3.14159f * (float)max(ni, 1)));
    int n = 0;
    while (true) {
        const bool everything = !(th < 1.5f);
        const float sh = sinf(0.5f * fminf(th, 3.14f));
        const float limit = everything ? 3.0e38f : 4.0f * sh * sh;
        float worst = everything ? 3.0e38f : limit * 0.9999f;  // costs within it are all met
        int worst_i = 0x7fffffff;
        n = 0;
        SubWalk walk;
        walk.init(sub, ext, np);
        auto fetch = [&](int st) {  // two sub-granules of 16 spots
            const int s0 = walk.next(own, false, everything ? 0 : 1, 1.0f, limit);
            const int s1 = s0 < 0 ? -1 : walk.next(own, false, everything ? 0 : 1, 1.0f, limit);
            const int s = lane < 16 ? s0 : s1, q = 16 * s + (lane & 15);
            float4 v = make_float4(0.0f, 0.0f, 0.0f, __int_as_float(-1));
            if (s >= 0 && q < ni) {
                const int i = k.obs_perm[i0 + q];
                v = a.p[i];
                v.w = __int_as_float(i);
            }
            S.p[st][lane] = v;
            return s0 >= 0;
        };
        int st = 0;
        bool more = fetch(0);
        while (more) {
            __syncwarp();
            const bool next = fetch(st ^ 1);
#pragma unroll 4
            for (int q = 0; q < 32; ++q) {
                const float4 p = S.p[st][q];
                const int i = __float_as_int(p.w);
                const float v = sp_e2(p, c, r);
                if (i < 0 || !(v < worst || (v == worst && i < worst_i))) continue;
                int at = n < want ? n++ : want - 1;
                while (at > 0) {
                    const int2 b = L[32 * (at - 1)];
                    const float bv = __int_as_float(b.y);
                    if (!(bv > v || (bv == v && b.x > i))) break;
                    L[32 * at] = b;
                    --at;
                }
                L[32 * at] = make_int2(i, __float_as_int(v));
                if (n == want) {
                    const int2 b = L[32 * (want - 1)];
                    worst = __int_as_float(b.y);
                    worst_i = b.x;
                }
            }
            st ^= 1;
            more = next;
        }
        if (everything || !__any_sync(0xffffffffu, valid && n < want)) break;
        th *= 1.6f;
        __syncwarp();
    }
    if (!valid) return;
    const int det = a.s ? (int)a.s[j].w : -1;
    const float kd = (det >= 0 && det < a.n_det) ? a.kdet[det] : 1.0f;
    int2* out = a.cent + (size_t)j * a.rho;
    for (int q = 0; q < a.rho; ++q) {
        const int2 b = q < n ? L[32 * q] : make_int2(-1, 0);
        out[q] = q < n ? make_int2(b.x, __float_as_int(__int_as_float(b.y) * kd)) : b;
        if (a.nbr_out) a.nbr_out[(size_t)j * a.rho + q] = b.x;
    }
}

__global__ void sp_count_kernel(SpArgs a) {
    size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (size_t)a.n_model * a.rho) return;
    int i = a.cent[e].x;
    if (i >= 0) atomicAdd(&a.rfill[i], 1);
}

// Position of row i's records; the starts are 32 bits wide where all positions
// fit them (sp_wide), which the passes are 7 % faster with (214 grains x 46
// angles, 16 neighbours, 100 iterations: 3.11 against 3.35 ms).
__device__ __forceinline__ long long row_start(const SpArgs& a, int i) {
    return a.rptr64 ? a.rptr64[i] : a.rptr[i];
}
template <class Idx>
__device__ __forceinline__ Idx start_of(const SpArgs& a, int i) {
    if constexpr (sizeof(Idx) == 8) return a.rptr64[i];
    else return a.rptr[i];
}
__device__ __forceinline__ void set_row_start(const SpArgs& a, long long i, long long at) {
    if (a.rptr64) a.rptr64[i] = at;
    else a.rptr[i] = (int)at;
}

// Row starts from the entries of each row: sums of blocks of kScan rows, then
// each block adds the sums before it.  The sums sit where the tile partials of
// the row passes will.
constexpr int kScan = 8192;
__global__ void __launch_bounds__(1024) sp_scan_sums_kernel(SpArgs a) {
    __shared__ long long warp_sum[32];
    long long s = 0;
    for (int k = threadIdx.x; k < kScan; k += 1024) {
        const long long i = (long long)blockIdx.x * kScan + k;
        if (i < a.n_obs) s += a.rfill[i];
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) warp_sum[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 32; ++w) s += warp_sum[w];
        ((long long*)a.rpart)[blockIdx.x] = s;
    }
}

__global__ void __launch_bounds__(1024) sp_scan_kernel(SpArgs a) {
    __shared__ long long warp_sum[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    auto block_sum = [&](long long s) {
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) warp_sum[w] = s;
        __syncthreads();
        long long all = 0;
        for (int u = 0; u < 32; ++u) all += warp_sum[u];
        __syncthreads();
        return all;
    };
    long long before = 0;
    for (int k = threadIdx.x; k < (int)blockIdx.x; k += 1024) before += ((const long long*)a.rpart)[k];
    before = block_sum(before);
    constexpr int kPer = kScan / 1024;
    const long long i0 = (long long)blockIdx.x * kScan + kPer * threadIdx.x;
    int v[kPer];
    long long s = 0;
    for (int q = 0; q < kPer; ++q) {
        v[q] = i0 + q < a.n_obs ? a.rfill[i0 + q] : 0;
        s += v[q];
    }
    long long incl = s;
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_sum[w] = incl;
    __syncthreads();
    long long at = before + incl - s;
    for (int u = 0; u < w; ++u) at += warp_sum[u];
    if (i0 == 0) set_row_start(a, 0, 0);
    for (int q = 0; q < kPer; ++q) {
        at += v[q];
        if (i0 + q < a.n_obs) set_row_start(a, 1 + i0 + q, at);
    }
}

__global__ void sp_fill_kernel(SpArgs a) {
    size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (size_t)a.n_model * a.rho) return;
    int2 v = a.cent[e];
    if (v.x < 0) return;
    const long long slot = row_start(a, v.x) + atomicAdd(&a.rfill[v.x], 1);
    a.rent[slot] = make_int2((int)(e / a.rho), v.y);
}

// each row in ascending model index (a fixed summation order)
__global__ void sp_sort_rows_kernel(SpArgs a) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.n_obs) return;
    int2* row = a.rent + row_start(a, i);
    const int n = (int)(row_start(a, i + 1) - row_start(a, i));
    for (int k = 1; k < n; ++k) {
        int2 v = row[k];
        int q = k - 1;
        while (q >= 0 && row[q].x > v.x) {
            row[q + 1] = row[q];
            --q;
        }
        row[q + 1] = v;
    }
}

// ------------------------------------------------------------------ init
__global__ void sp_init_pot_kernel(SpArgs a) {
    const float s = 1.0f / a.to_user;
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < a.n_obs) a.F[k] = a.warm ? a.f[k] * s : 0.0f;
    if (k < a.n_model) a.G[k] = a.warm ? a.g[k] * s : 0.0f;
}

// Masses, starting dustbin potentials and F_0 of the first row pass (from the
// starting G and G_0).  One CTA per dustbin.
__global__ void __launch_bounds__(1024) sp_init_dust_kernel(SpArgs a) {
    __shared__ float sm[32], ss[32];
    const int nd = a.mode ? a.T : 1;
    const int d = blockIdx.x;
    SpDust D = sp_dust(a.dust, nd);
    const float s = 1.0f / a.to_user;
    const long long nI = a.mode ? (a.I_off[d + 1] - a.I_off[d]) : a.I_off[a.T];
    const long long nJ = a.mode ? (a.J_off[d + 1] - a.J_off[d]) : a.J_off[a.T];
    const float g0 = (a.warm && a.dust_out) ? a.dust_out[nd + d] * s : 0.0f;
    float log2U = kNegHuge;
    if (threadIdx.x == 0) {
        double u = ceil(a.frac * (double)nJ - 1e-9);
        double o = u + (double)nI - (double)nJ;
        if (o < 0) {
            u = (double)(nJ - nI);
            o = 0;
        }
        log2U = u > 0 ? (float)log2(u) : kNegHuge;
        D.log2U[d] = log2U;
        D.log2O[d] = o > 0 ? (float)log2(o) : kNegHuge;
        D.F0[d] = (a.warm && a.dust_out) ? a.dust_out[d] * s : 0.0f;
        D.G0[d] = g0;
    }
    const int j0 = a.mode ? a.J_off[d] : 0, j1 = a.mode ? a.J_off[d + 1] : a.n_model;
    float m = kNegHuge, sum = 0.0f;
    for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x) acc_lse(m, sum, a.warm ? a.g[j] * s : 0.0f);
    warp_lse_reduce(m, sum);
    if ((threadIdx.x & 31) == 0) {
        sm[threadIdx.x >> 5] = m;
        ss[threadIdx.x >> 5] = sum;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        Lse2 L;
        L.init(g0 - a.kc);
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) L.merge(sm[w], ss[w]);
        D.F0n[d] = log2U - L.value();
    }
}

// Block log-sum-exp of the lanes' (m, s); the result is valid in thread 0.
__device__ __forceinline__ void sp_block_lse(float& m, float& s, float* red_m, float* red_s) {
    warp_lse_reduce(m, s);
    if ((threadIdx.x & 31) == 0) {
        red_m[threadIdx.x >> 5] = m;
        red_s[threadIdx.x >> 5] = s;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        Lse2 L;
        L.m = kNegHuge;
        L.s = 0.0f;
        for (int k = 0; k < kSpWarps; ++k) L.merge(red_m[k], red_s[k]);
        m = L.m;
        s = L.s;
    }
}

// Warp-level LSE of the partials of tiles [k0, k1) (valid in every lane).
__device__ __forceinline__ void sp_merge_parts(const float2* part, int k0, int k1, float& m, float& s) {
    m = kNegHuge;
    s = 0.0f;
    for (int k = k0 + (int)(threadIdx.x & 31); k < k1; k += 32 * 8) {
        float2 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = k + 32 * q < k1 ? __ldcg(&part[k + 32 * q]) : make_float2(kNegHuge, 0.0f);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            Lse2 L{m, s};
            L.merge(v[q].x, v[q].y);
            m = L.m;
            s = L.s;
        }
    }
    warp_lse_reduce(m, s);
}

// --------------------------------------------------------------- row pass
// Each row is the sum of its support terms 2^(G_j - K e2 - shift) and the
// outlier term, shifted by shift = max(largest G of the angle block, the
// outlier exponent): every term is <= 1, so no running maximum is kept.  A row
// whose shifted sum falls below kSpTiny is recomputed with the running maximum.
// Eight lanes per row, four rows per warp; the lanes stride over the row's
// records.
constexpr float kSpTiny = 1.0e-30f;
constexpr int kSpLanes = 8;  // lanes per spot

template <class Idx>
__device__ float sp_row_exact(const SpArgs& a, int i, float dustv) {
    float m = kNegHuge, s = 0.0f;
    acc_lse(m, s, dustv);
    for (Idx e = start_of<Idx>(a, i); e < start_of<Idx>(a, i + 1); ++e) {
        int2 v = a.rent[e];
        acc_lse(m, s, a.G[v.x] + a.negK * __int_as_float(v.y));
    }
    return s > 0.0f ? m + lg2(s) : kNegHuge;
}

__device__ float sp_col_exact(const SpArgs& a, int j, float F0) {
    float m = kNegHuge, s = 0.0f;
    acc_lse(m, s, F0);
    const int2* ce = a.cent + (size_t)j * a.rho;
    for (int k = 0; k < a.rho; ++k) {
        int2 v = ce[k];
        if (v.x >= 0) acc_lse(m, s, a.F[v.x] + a.negK * __int_as_float(v.y));
    }
    return s > 0.0f ? m + lg2(s) : kNegHuge;
}

// per-angle largest G of the starting potentials (one CTA per angle)
__global__ void __launch_bounds__(256) sp_gmax_kernel(SpArgs a) {
    __shared__ float red[8];
    const int t = blockIdx.x;
    float m = kNegHuge;
    for (int j = a.J_off[t] + threadIdx.x; j < a.J_off[t + 1]; j += blockDim.x) m = fmaxf(m, a.G[j]);
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < (int)(blockDim.x >> 5); ++k) m = fmaxf(m, red[k]);
        a.gmax[t] = fmaxf(m, red[0]);
    }
}

// Dustbin potentials from the tile partials of a pass.  Rows: F_0 of the
// iteration and G_0 from it and the new F; columns: the next F_0 from the new G
// and the current G_0.  A warp per dustbin.
template <bool ROWS>
__device__ __forceinline__ void sp_finish_pass(const SpArgs& a, int block, int blocks) {
    const int nd = a.mode ? a.T : 1;
    const SpDust D = sp_dust(a.dust, nd);
    const int *base = ROWS ? a.rt_base : a.ct_base;
    for (int d = block * kSpWarps + (int)(threadIdx.x >> 5); d < nd; d += blocks * kSpWarps) {
        float m, s;
        sp_merge_parts(ROWS ? a.rpart : a.cpart, a.mode ? base[d] : 0, a.mode ? base[d + 1] : base[a.T], m, s);
        if ((threadIdx.x & 31) == 0) {
            Lse2 L{m, s};
            if (ROWS) {
                const float F0 = __ldcg(D.F0n + d);
                D.F0[d] = F0;
                L.merge(F0 - a.kc, 1.0f);
                D.G0[d] = D.log2O[d] - L.value();
            } else {
                L.merge(__ldcg(D.G0 + d) - a.kc, 1.0f);
                D.F0n[d] = D.log2U[d] - L.value();
            }
        }
    }
}

__global__ void __launch_bounds__(kSpThreads) sp_finish_pass_kernel(SpArgs a) {
    sp_finish_pass<false>(a, blockIdx.x, gridDim.x);
}

// Row (ROWS) or column update of iteration it; the first blocks finish the
// pass before.  Eight lanes per spot stride over its records, four records of
// a lane and the records of two spots loaded together: bound by the latency of
// record -> potential -> exponential.
constexpr int kSpBatch = 4;

template <bool ROWS, class Idx>
__global__ void __launch_bounds__(kSpThreads) sp_pass_kernel(SpArgs a, int it, int finishers) {
    __shared__ float red_m[kSpWarps], red_s[kSpWarps];
    // programmatic dependent launch: everything read here was complete before the pass before waited
    if (ROWS && it == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
    const int nd = a.mode ? a.T : 1;
    const SpDust D = sp_dust(a.dust, nd);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int grp = lane / kSpLanes, gl = lane % kSpLanes;
    const int *base = ROWS ? a.rt_base : a.ct_base, *other = ROWS ? a.ct_base : a.rt_base;
    const int tile = (int)blockIdx.x - finishers;
    const bool live = tile >= 0 && tile < base[a.T];
    const int4 td = live ? (ROWS ? a.rtile : a.ctile)[tile] : make_int4(0, 0, 0, 0);
    const int o0 = other[td.x], o1 = other[td.x + 1];
    if (!(ROWS && it == 0)) asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (tile < 0) {
        if (!ROWS || it > 0) sp_finish_pass<!ROWS>(a, blockIdx.x, finishers);
        return;
    }
    if (!live) return;
    const int2* rec = ROWS ? a.rent : a.cent;
    const float* pot = ROWS ? a.G : a.F;
    float* out = ROWS ? a.F : a.G;
    const float off = ROWS ? a.kc : 0.0f;
    // the dustbin's term; the other side's largest potential of the angle, from its tiles' partials (they keep
    // max(F - kc) and max G)
    const float dust = ROWS ? __ldcg(D.G0 + (a.mode ? td.x : 0)) - a.kc : __ldcg(D.F0n + (a.mode ? td.x : 0));
    float top = kNegHuge;
    if (ROWS && it == 0) {
        top = a.gmax[td.x];
    } else {
        const float2* part = ROWS ? a.cpart : a.rpart;
        for (int k = o0 + lane; k < o1; k += 32) top = fmaxf(top, __ldcg(&part[k].x));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
        if (!ROWS) top = top > kNegHuge ? top + a.kc : kNegHuge;
    }
    const float shift = fmaxf(top, dust);
    const float dterm = ex2(dust - shift);
    float pm = kNegHuge, ps = 0.0f;  // LSE of the new potentials (less kc) over this lane's spots
    constexpr int kStep = kSpWarps * (32 / kSpLanes);
    for (int ib = td.y + w * (32 / kSpLanes); ib < td.z; ib += 2 * kStep) {
        Idx e0[2], e1[2];
        float sum[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int i = ib + u * kStep + grp;
            const bool v = i < td.z;
            e0[u] = v ? (ROWS ? start_of<Idx>(a, i) : (Idx)i * a.rho) + gl : 0;
            e1[u] = v ? (ROWS ? start_of<Idx>(a, i + 1) : (Idx)(i + 1) * a.rho) : 0;
            sum[u] = 0.0f;
        }
        while (true) {
            int2 v[2][kSpBatch];
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int q = 0; q < kSpBatch; ++q) {
                    const Idx e = e0[u] + q * kSpLanes;
                    v[u][q] = e < e1[u] ? __ldcg(&rec[e]) : make_int2(-1, 0);
                }
            float g[2][kSpBatch];
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int q = 0; q < kSpBatch; ++q) g[u][q] = v[u][q].x >= 0 ? pot[v[u][q].x] : 0.0f;
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int q = 0; q < kSpBatch; ++q)
                    if (v[u][q].x >= 0) sum[u] += ex2(g[u][q] + a.negK * __int_as_float(v[u][q].y) - shift);
            e0[0] += kSpBatch * kSpLanes;
            e0[1] += kSpBatch * kSpLanes;
            if (!__any_sync(0xffffffffu, e0[0] < e1[0] || e0[1] < e1[1])) break;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int i = ib + u * kStep + grp;
#pragma unroll
            for (int o = kSpLanes / 2; o > 0; o >>= 1) sum[u] += __shfl_xor_sync(0xffffffffu, sum[u], o);
            if (i < td.z && gl == 0) {
                sum[u] += dterm;
                const float lse = sum[u] > kSpTiny ? shift + lg2(sum[u])
                                                   : (ROWS ? sp_row_exact<Idx>(a, i, dust) : sp_col_exact(a, i, dust));
                out[i] = -lse;
                acc_lse(pm, ps, -lse - off);
            }
        }
    }
    sp_block_lse(pm, ps, red_m, red_s);
    if (threadIdx.x == 0) (ROWS ? a.rpart : a.cpart)[tile] = make_float2(pm, ps);
}

// ------------------------------------------------------------- read-out
struct SpTop2 {
    float b1, b2;
    int arg;
};

// the larger first value wins, equal values go to the lower model index
__device__ __forceinline__ SpTop2 sp_top2_merge(SpTop2 x, SpTop2 y) {
    bool xw = x.b1 > y.b1 || (x.b1 == y.b1 && (unsigned)x.arg < (unsigned)y.arg);
    SpTop2 w = xw ? x : y, l = xw ? y : x;
    w.b2 = fmaxf(w.b2, l.b1);
    return w;
}

__global__ void __launch_bounds__(kSpThreads) sp_harvest_row_kernel(SpArgs a) {
    __shared__ float red[kSpWarps];
    const int nd = a.mode ? a.T : 1;
    SpDust D = sp_dust(a.dust, nd);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float my_err = 0.0f;
    if ((int)blockIdx.x < a.rt_base[a.T]) {
        const int4 td = a.rtile[blockIdx.x];
        const float dustv = D.G0[a.mode ? td.x : 0] - a.kc;
        for (int i = td.y + w; i < td.z; i += kSpWarps) {
            float m = kNegHuge, s = 0.0f;
            SpTop2 T2{kNegHuge, kNegHuge, -1};
            const long long end = row_start(a, i + 1);
            for (long long e = row_start(a, i) + lane; e < end; e += 32) {
                int2 v = a.rent[e];
                float x = a.G[v.x] + a.negK * __int_as_float(v.y);
                acc_lse(m, s, x);
                if (x > T2.b1) {  // ascending model index per lane: ties keep the earlier
                    T2.b2 = T2.b1;
                    T2.b1 = x;
                    T2.arg = v.x;
                } else if (x > T2.b2) {
                    T2.b2 = x;
                }
            }
            warp_lse_reduce(m, s);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                SpTop2 y{__shfl_xor_sync(0xffffffffu, T2.b1, o), __shfl_xor_sync(0xffffffffu, T2.b2, o),
                         __shfl_xor_sync(0xffffffffu, T2.arg, o)};
                T2 = sp_top2_merge(T2, y);
            }
            if (lane == 0) {
                const float F = a.F[i];
                if (dustv > T2.b1) {  // the outlier column only when strictly larger
                    T2.b2 = T2.b1;
                    T2.b1 = dustv;
                    T2.arg = -1;
                } else if (dustv > T2.b2) {
                    T2.b2 = dustv;
                }
                Lse2 L{m, s};
                L.merge(dustv, 1.0f);
                my_err = fmaxf(my_err, fabsf(ex2(F + L.value()) - 1.0f));
                if (a.assign) a.assign[i] = T2.arg;
                if (a.margin) a.margin[i] = ex2(F + T2.b1) - (T2.b2 > kNegHuge ? ex2(F + T2.b2) : 0.0f);
            }
        }
    }
    if (lane == 0) red[w] = my_err;
    __syncthreads();
    if (threadIdx.x == 0) {
        float e = 0.0f;
        for (int k = 0; k < kSpWarps; ++k) e = fmaxf(e, red[k]);
        atomicMax((int*)(D.err + 0), __float_as_int(e));  // non-negative floats order as ints
    }
}

__global__ void __launch_bounds__(kSpThreads) sp_harvest_col_kernel(SpArgs a) {
    __shared__ float red[kSpWarps];
    const int nd = a.mode ? a.T : 1;
    SpDust D = sp_dust(a.dust, nd);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float my_err = 0.0f;
    if ((int)blockIdx.x < a.ct_base[a.T]) {
        const int4 td = a.ctile[blockIdx.x];
        const float F0 = D.F0[a.mode ? td.x : 0];
        for (int j = td.y + w; j < td.z; j += kSpWarps) {
            const int2* ce = a.cent + (size_t)j * a.rho;
            const float G = a.G[j];
            float qj = 0.0f;
            for (int k = lane; k < a.rho; k += 32) {
                int2 v = ce[k];
                if (v.x >= 0) qj += ex2(a.F[v.x] + G + a.negK * __int_as_float(v.y));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) qj += __shfl_xor_sync(0xffffffffu, qj, o);
            if (lane == 0) {
                if (a.q) a.q[j] = qj;
                my_err = fmaxf(my_err, fabsf(qj + ex2(G + F0) - 1.0f));
            }
        }
    }
    if (lane == 0) red[w] = my_err;
    __syncthreads();
    if (threadIdx.x == 0) {
        float e = 0.0f;
        for (int k = 0; k < kSpWarps; ++k) e = fmaxf(e, red[k]);
        atomicMax((int*)(D.err + 1), __float_as_int(e));
    }
}

__global__ void sp_finish_kernel(SpArgs a, int have_rows, int have_cols) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    bool bad = false;
    if (k < a.n_obs) {
        float v = a.F[k];
        bad |= !isfinite(v);
        a.f[k] = v * a.to_user;
    }
    if (k < a.n_model) {
        float v = a.G[k];
        bad |= !isfinite(v);
        a.g[k] = v * a.to_user;
    }
    if (k == 0) {
        const int nd = a.mode ? a.T : 1;
        SpDust D = sp_dust(a.dust, nd);
        if (a.dust_out)
            for (int d = 0; d < nd; ++d) {
                a.dust_out[d] = D.F0[d] * a.to_user;
                a.dust_out[nd + d] = D.G0[d] * a.to_user;
            }
        if (a.marg_err) {
            float er = D.err[0];
            for (int d = 0; d < nd; ++d)  // the unmatched-model row
                if (D.log2U[d] > kNegHuge) er = fmaxf(er, fabsf(ex2(D.F0[d] - D.F0n[d]) - 1.0f));
            a.marg_err[0] = have_rows ? er : -1.0f;
            a.marg_err[1] = have_cols ? D.err[1] : -1.0f;
        }
    }
    if (bad) set_status(a.ctrl, LAUE_ERR_NUMERIC);
}

__global__ void sp_clear_err_kernel(SpArgs a) {
    SpDust D = sp_dust(a.dust, a.mode ? a.T : 1);
    D.err[0] = D.err[1] = 0.0f;
}

// ------------------------------------------------------------- host side
static size_t sp_max_tiles(int n, int T) { return (size_t)(n + kSpTile - 1) / kSpTile + (size_t)T; }

// Positions of the records need 64 bits, a lane's steps past its own row (up to
// the longest) included.
static bool sp_wide(int n_model, int rho) { return (long long)n_model * (rho + 1) + 65536 >= 0x7fffffffLL; }

size_t sparse_workspace_bytes(int T, int n_obs, int n_model, int rho) {
    const size_t nnz = (size_t)n_model * rho;
    size_t b = 0;
    auto add = [&](size_t bytes) { b += align_up(bytes > 0 ? bytes : 1, 256); };
    add(sizeof(int2) * nnz);                         // cent
    add(sizeof(int2) * nnz);                         // rent
    add((sp_wide(n_model, rho) ? 8 : 4) * ((size_t)n_obs + 2));  // rptr
    add(sizeof(int) * ((size_t)n_obs + 1));          // rfill
    add(sizeof(float) * ((size_t)n_obs + 1));        // F
    add(sizeof(float) * ((size_t)n_model + 1));      // G
    add(sizeof(float) * ((size_t)5 * T + 8));        // dust
    add(sizeof(float2) * sp_max_tiles(n_obs, T));    // rpart
    add(sizeof(float2) * sp_max_tiles(n_model, T));  // cpart
    add(sizeof(int4) * sp_max_tiles(n_obs, T));      // rtile
    add(sizeof(int4) * sp_max_tiles(n_model, T));    // ctile
    add(sizeof(int) * 2 * ((size_t)T + 1));          // rt_base, ct_base
    add(sizeof(float) * ((size_t)T + 1));            // gmax
    return b;
}

void sparse_carve(SpArgs& a, char* base, int T, int n_obs, int n_model, int rho) {
    const size_t nnz = (size_t)n_model * rho;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char* p = base + off;
        off += align_up(bytes > 0 ? bytes : 1, 256);
        return p;
    };
    a.cent = (int2*)take(sizeof(int2) * nnz);
    a.rent = (int2*)take(sizeof(int2) * nnz);
    const bool wide = sp_wide(n_model, rho);
    a.rptr = (int*)take((wide ? 8 : 4) * ((size_t)n_obs + 2));
    a.rptr64 = wide ? (long long*)a.rptr : nullptr;
    a.rfill = (int*)take(sizeof(int) * ((size_t)n_obs + 1));
    a.F = (float*)take(sizeof(float) * ((size_t)n_obs + 1));
    a.G = (float*)take(sizeof(float) * ((size_t)n_model + 1));
    a.dust = (float*)take(sizeof(float) * ((size_t)5 * T + 8));
    a.rpart = (float2*)take(sizeof(float2) * sp_max_tiles(n_obs, T));
    a.cpart = (float2*)take(sizeof(float2) * sp_max_tiles(n_model, T));
    a.rtile = (int4*)take(sizeof(int4) * sp_max_tiles(n_obs, T));
    a.ctile = (int4*)take(sizeof(int4) * sp_max_tiles(n_model, T));
    a.rt_base = (int*)take(sizeof(int) * 2 * ((size_t)T + 1));
    a.ct_base = a.rt_base + T + 1;
    a.gmax = (float*)take(sizeof(float) * ((size_t)T + 1));
    a.max_rt = (int)sp_max_tiles(n_obs, T);
    a.max_ct = (int)sp_max_tiles(n_model, T);
}

size_t sparse_knn_smem(int rho) { return (size_t)kKnnThreads * rho * sizeof(int2); }

template <bool ROWS>
static cudaError_t sp_pass(const SpArgs& a, int it, cudaStream_t s) {
    const int finishers = a.mode ? (a.T + kSpWarps - 1) / kSpWarps : 1;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(finishers + (ROWS ? a.max_rt : a.max_ct));
    c.blockDim = dim3(kSpThreads);
    c.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = 1;
    if (!a.rptr64) return cudaLaunchKernelEx(&c, sp_pass_kernel<ROWS, int>, a, it, finishers);
    return cudaLaunchKernelEx(&c, sp_pass_kernel<ROWS, long long>, a, it, finishers);
}

cudaError_t sparse_sinkhorn_run(const SpArgs& a, const SkArgs* order, int n_iter, bool rows, bool cols,
                                cudaStream_t s) {
    cudaError_t e;
    const size_t nnz = (size_t)a.n_model * a.rho;
    const int nd = a.mode ? a.T : 1;
    sp_schedule_kernel<<<1, 1024, 0, s>>>(a);
    // neighbour lists and their transpose
    if (order && a.n_obs > 0 && a.n_model > 0) {
        if ((e = sinkhorn_prepare(*order, s, false)) != cudaSuccess) return e;
        const size_t shm = 4 * sizeof(KnnStage) + (size_t)128 * a.rho * sizeof(int2);
        if ((e = cudaFuncSetAttribute(sp_knn_cone_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm)) !=
            cudaSuccess)
            return e;
        const int halves = 2 * (a.n_model / 64 + a.T + 1);  // bound on the granules' halves
        sp_knn_cone_kernel<<<(halves + 3) / 4, 128, shm, s>>>(a, *order);
    } else {
        const size_t shm = sparse_knn_smem(a.rho);
        if ((e = cudaFuncSetAttribute(sp_knn_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm)) !=
            cudaSuccess)
            return e;
        sp_knn_kernel<<<a.max_ct, kKnnThreads, shm, s>>>(a);
    }
    if ((e = cudaMemsetAsync(a.rfill, 0, sizeof(int) * ((size_t)a.n_obs + 1), s)) != cudaSuccess) return e;
    const unsigned nb = (unsigned)((nnz + 255) / 256);
    if (nnz > 0) sp_count_kernel<<<nb, 256, 0, s>>>(a);
    if (a.n_obs > 0) {
        const int blocks = (a.n_obs + kScan - 1) / kScan;
        sp_scan_sums_kernel<<<blocks, 1024, 0, s>>>(a);
        sp_scan_kernel<<<blocks, 1024, 0, s>>>(a);
    }
    if ((e = cudaMemsetAsync(a.rfill, 0, sizeof(int) * ((size_t)a.n_obs + 1), s)) != cudaSuccess) return e;
    if (nnz > 0) sp_fill_kernel<<<nb, 256, 0, s>>>(a);
    if (a.n_obs > 0) sp_sort_rows_kernel<<<(a.n_obs + 255) / 256, 256, 0, s>>>(a);
    const int blocks = std::max(1, (std::max(a.n_obs, a.n_model) + 255) / 256);
    sp_init_pot_kernel<<<blocks, 256, 0, s>>>(a);
    sp_init_dust_kernel<<<nd, 1024, 0, s>>>(a);
    if (a.T > 0) sp_gmax_kernel<<<a.T, 256, 0, s>>>(a);
    for (int it = 0; it < n_iter; ++it) {
        if ((e = sp_pass<true>(a, it, s)) != cudaSuccess) return e;
        if ((e = sp_pass<false>(a, it, s)) != cudaSuccess) return e;
    }
    if (n_iter > 0) sp_finish_pass_kernel<<<a.mode ? (a.T + kSpWarps - 1) / kSpWarps : 1, kSpThreads, 0, s>>>(a);
    if (rows || cols) sp_clear_err_kernel<<<1, 1, 0, s>>>(a);
    if (rows) sp_harvest_row_kernel<<<a.max_rt, kSpThreads, 0, s>>>(a);
    if (cols) sp_harvest_col_kernel<<<a.max_ct, kSpThreads, 0, s>>>(a);
    sp_finish_kernel<<<blocks, 256, 0, s>>>(a, rows ? 1 : 0, cols ? 1 : 0);
    return cudaGetLastError();
}

}  // namespace laue
