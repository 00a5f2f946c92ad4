// sinkhorn.cu — fused pair cost + log-domain balanced Sinkhorn with dustbins
// (paper Eqs. update_L, elbo, estep_obj; Algorithm BalancedOT), blocked by
// rotation angle.
//
// Extended plan: observed rows i plus the unmatched-model row 0 (mass U),
// model columns j plus the outlier column 0 (mass O); costs C_ij (same angle
// only), C_i0 = c_out, C_0j = 0, C_00 = c_out.  In base-2 units with
// F = f log2(e)/eps, G = g log2(e)/eps and K = D^2 log2(e)/eps:
//   row    F_i = -LSE2({G_j - K e2_ij}_{j in J_t} u {G_0 - kc})
//   dust   F_0 = log2 U - LSE2({G_j}_j u {G_0 - kc})
//   column G_j = -LSE2({F_i - K e2_ij}_{i in I_t} u {F_0})
//   dust   G_0 = log2 O - LSE2({F_i - kc}_i u {F_0 - kc})
// with e2_ij = |rhat_ij - r_j|^2 and kc = c_out log2(e)/eps.  The cost matrix
// is never stored: the passes keep e2 of the pairs whose plan entry can be
// nonzero for one E-step, and recompute it from the spot coordinates elsewhere.
//
// Unbalanced mode (Appendix "Optimal transport variants", Algorithm
// UnbalancedOT): no dustbins, and each balanced update is scaled by
// tau_row = kappa / (kappa + eps) (rows) or tau_col = lambda / (lambda + eps)
// (columns), the log-domain form of the exponents of the scaling updates.
//
// Layout.  The workspace holds the spots as pairs: each angle block is padded
// to an even count and element pairs (a, b) are interleaved into float4 rows
// such as {x_a, x_b, y_a, y_b}, so one 16-byte shared-memory load yields two
// packed operands for the f32x2 FMA/ADD/MUL instructions.  Model centres and
// rays are stored negated (d = p + (-c), e = d/|d| + (-r)).  Padding entries
// carry a potential of -3e38, which makes their plan entries exactly 0.
//
// Passes (passes.cu).  Every pass is one launch over the tiles of all angle
// blocks; its tiles' partial log-sum-exps become the dustbin potentials
// beside the next pass:
//   end of a row pass:    F_0 <- F_0(next), then G_0 from the new F and F_0
//   end of a column pass: F_0(next) from the new G and G_0
// which reproduces the sequential order of the algorithm exactly.
#include "pairs.cuh"

namespace laue {

// ---------------------------------------------------------------- scheduler
// Exclusive prefix of get(i), i < n, by a CTA of 1024 threads: put(i, prefix);
// returns the sum.
template <class Get, class Put>
__device__ int block_prefix(int n, int* warp_sum, Get get, Put put) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int base = 0;
    for (int i0 = 0; i0 < n; i0 += 1024) {
        const int i = i0 + threadIdx.x;
        const int c = i < n ? get(i) : 0;
        int incl = c;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) warp_sum[w] = incl;
        __syncthreads();
        if (w == 0) {
            int v = warp_sum[lane];
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += y;
            }
            warp_sum[lane] = v;
        }
        __syncthreads();
        if (i < n) put(i, base + (w ? warp_sum[w - 1] : 0) + incl - c);
        base += warp_sum[31];
        __syncthreads();
    }
    return base;
}

// Slots among the pairs [0, n) that warp w of 1024 threads reads (pair q is
// thread q % 1024's).
__device__ __forceinline__ int warp_share(int n, int w) {
    return 2 * (n / 1024 * 32 + min(32, max(0, n % 1024 - 32 * w)));
}

// One CTA.  Pair offsets of the padded blocks, row and column tile queues
// (angles by descending work, tiles of one angle contiguous), per-angle tile
// ranges, log2 masses of the dustbins; clears the counters.  A cold start's
// potentials are all 0, so its maxima and first F_0 need no pass over them:
// the sums of sk_init_dust_kernel are then counts of spots.
constexpr int kSchedAngles = 1024;  // angles whose offsets fit in shared memory
__global__ void __launch_bounds__(1024) sk_schedule_kernel(SkArgs a, int dustbins) {
    __shared__ int sI[kSchedAngles + 1], sJ[kSchedAngles + 1], warp_sum[32], pads[32];
    const int T = a.T;
    const int *I = a.I_off, *J = a.J_off;
    if (T <= kSchedAngles) {
        for (int t = threadIdx.x; t <= T; t += blockDim.x) {
            sI[t] = I[t];
            sJ[t] = J[t];
        }
        __syncthreads();
        I = sI;
        J = sJ;
    }
    int* order_r = (int*)a.row_part;  // scratch until the passes run
    int* order_c = (int*)a.col_part;
    for (int t = threadIdx.x; t < T; t += blockDim.x) {
        const int wr = J[t + 1] - J[t], wc = I[t + 1] - I[t];
        int rr = 0, rc = 0;
        for (int u = 0; u < T; ++u) {
            const int ur = J[u + 1] - J[u], uc = I[u + 1] - I[u];
            rr += (ur > wr) || (ur == wr && u < t);
            rc += (uc > wc) || (uc == wc && u < t);
        }
        order_r[rr] = t;
        order_c[rc] = t;
    }
    auto pairs_i = [&](int t) { return (I[t + 1] - I[t] + 1) / 2; };
    auto pairs_j = [&](int t) { return (J[t + 1] - J[t] + 1) / 2; };
    auto granules = [](int n) { return (n + kGran - 1) / kGran; };
    const int ni2 = block_prefix(T, warp_sum, pairs_i, [&](int t, int v) { a.I2_off[t] = v; });
    const int nj2 = block_prefix(T, warp_sum, pairs_j, [&](int t, int v) { a.J2_off[t] = v; });
    const int ngi = block_prefix(T, warp_sum, [&](int t) { return granules(pairs_i(t)); },
                                 [&](int t, int v) { a.obs_gbase[t] = v; });
    const int ngj = block_prefix(T, warp_sum, [&](int t) { return granules(pairs_j(t)); },
                                 [&](int t, int v) { a.mod_gbase[t] = v; });
    auto tiles_r = [&](int k) { return (pairs_i(order_r[k]) + a.tile_rows - 1) / a.tile_rows; };
    auto tiles_c = [&](int k) { return (pairs_j(order_c[k]) + a.tile_cols - 1) / a.tile_cols; };
    int nr = block_prefix(T, warp_sum, tiles_r, [&](int k, int v) {
        int4& at = a.ang_tiles[order_r[k]];
        at.x = v;
        at.y = tiles_r(k);
    });
    int nc = block_prefix(T, warp_sum, tiles_c, [&](int k, int v) {
        int4& at = a.ang_tiles[order_c[k]];
        at.z = v;
        at.w = tiles_c(k);
    });
    if (threadIdx.x == 0) {
        a.I2_off[T] = ni2;
        a.J2_off[T] = nj2;
        a.obs_gbase[T] = ngi;
        a.mod_gbase[T] = ngj;
        if (nr > a.max_row_tiles || nc > a.max_col_tiles) {
            set_status(a.ctrl, LAUE_ERR_CAPACITY);
            nr = min(nr, a.max_row_tiles);
            nc = min(nc, a.max_col_tiles);
        }
        a.ctrl[CTRL_N_ROW_TILES] = nr;
        a.ctrl[CTRL_N_COL_TILES] = nc;
        a.ctrl[CTRL_HRV_DONE] = a.ctrl[CTRL_HCOL_DONE] = 0;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < T; t += blockDim.x) {
        int4 at = a.ang_tiles[t];
        int i0 = a.I2_off[t], ni = a.I2_off[t + 1] - i0;
        for (int k = 0; k < at.y; ++k) {
            int idx = at.x + k;
            if (idx < a.max_row_tiles)
                a.row_tiles[idx] = make_int4(t, i0 + k * a.tile_rows, min(a.tile_rows, ni - k * a.tile_rows), 0);
        }
        int j0 = a.J2_off[t], nj = a.J2_off[t + 1] - j0;
        for (int k = 0; k < at.w; ++k) {
            int idx = at.z + k;
            if (idx < a.max_col_tiles)
                a.col_tiles[idx] = make_int4(t, j0 + k * a.tile_cols, min(a.tile_cols, nj - k * a.tile_cols), 0);
        }
    }
    if (!a.warm)
        for (int t = threadIdx.x; t < T; t += blockDim.x) {
            DustPtrs D = dust_ptrs(a.dust, T);
            D.Gmax[t] = J[t + 1] > J[t] ? 0.0f : kNegHuge;
            D.Fmax[t] = I[t + 1] > I[t] ? 0.0f : kNegHuge;
        }
    if (!dustbins) return;
    // dustbin masses (paper: T_a = T_b - b^T 1 + a^T 1), in double precision
    DustPtrs D = dust_ptrs(a.dust, T);
    const int nd = a.mode ? T : 1;
    if (threadIdx.x < 32) pads[threadIdx.x] = 0;
    __syncthreads();
    if (!a.mode)
        for (int t = threadIdx.x; t < T; t += blockDim.x)
            if ((J[t + 1] - J[t]) & 1) atomicAdd(&pads[(a.J2_off[t] + pairs_j(t) - 1) % 1024 / 32], 1);
    __syncthreads();
    for (int d = threadIdx.x; d < nd; d += blockDim.x) {
        long long nI = a.mode ? (I[d + 1] - I[d]) : I[T];
        long long nJ = a.mode ? (J[d + 1] - J[d]) : J[T];
        double u = ceil(a.frac * (double)nJ - 1e-9);
        double o = u + (double)nI - (double)nJ;
        if (o < 0) {
            u = (double)(nJ - nI);
            o = 0;
        }
        const float log2U = u > 0 ? (float)log2(u) : kNegHuge;
        D.log2U[d] = log2U;
        D.log2O[d] = o > 0 ? (float)log2(o) : kNegHuge;
        if (!a.warm && a.mode != 2) {
            // F_0(next) = log2 U - LSE2({0}_j u {-kc}), in the order of sk_init_dust_kernel
            const int n = a.mode ? pairs_j(d) : nj2;
            Lse2 L;
            L.init(0.0f - a.kc);
            for (int w = 0; w < 32; ++w) {
                int c = warp_share(n, w);
                if (!a.mode) c -= pads[w];
                else if ((nJ & 1) && (n - 1) % 1024 / 32 == w) --c;
                L.merge(c > 0 ? 0.0f : kNegHuge, (float)c);
            }
            D.F0n[d] = log2U - L.value();
        }
    }
}

// ------------------------------------------------------- spatial order
// Within each angle block the spots are ranked by a 23-bit key of their
// direction (observed: p / |p|, model: the ray r): the cube-map face of the
// direction and the Morton interleave of its two in-face coordinates at 10
// bits each.  Spots close on a detector get close ranks, so runs of kGran
// pairs are spatially compact and their cones are narrow.  One CTA sorts one
// block (LSD radix sort, 4-bit digits, stable: ties keep the caller's order).
__device__ __forceinline__ unsigned spread10(unsigned v) {
    v &= 1023u;
    v = (v | (v << 8)) & 0x00FF00FFu;
    v = (v | (v << 4)) & 0x0F0F0F0Fu;
    v = (v | (v << 2)) & 0x33333333u;
    v = (v | (v << 1)) & 0x55555555u;
    return v;
}

__device__ __forceinline__ unsigned direction_key(float x, float y, float z) {
    float ax = fabsf(x), ay = fabsf(y), az = fabsf(z);
    int face;
    float m, u, v;
    if (ax >= ay && ax >= az) {
        face = x < 0.0f;
        m = ax;
        u = y;
        v = z;
    } else if (ay >= az) {
        face = 2 + (y < 0.0f);
        m = ay;
        u = x;
        v = z;
    } else {
        face = 4 + (z < 0.0f);
        m = az;
        u = x;
        v = y;
    }
    if (!(m > 0.0f)) return 0u;
    unsigned qu = (unsigned)fminf(1023.0f, fmaxf(0.0f, (u / m + 1.0f) * 512.0f));
    unsigned qv = (unsigned)fminf(1023.0f, fmaxf(0.0f, (v / m + 1.0f) * 512.0f));
    return ((unsigned)face << 20) | spread10(qu) | (spread10(qv) << 1);
}

constexpr int kSortThreads = 1024;
constexpr int kRankSort = 512;

// Blocks 0..T-1 sort the observed blocks, T..2T-1 the model blocks.
__global__ void __launch_bounds__(kSortThreads) sk_sort_kernel(SkArgs a) {
    __shared__ int cnt[kSortThreads / 32][16];
    __shared__ int dbase[16];
    const bool mod = (int)blockIdx.x >= a.T;
    const int t = mod ? blockIdx.x - a.T : blockIdx.x;
    const int* off = mod ? a.J_off : a.I_off;
    const int b0 = off[t], n = off[t + 1] - b0;
    const size_t nsp = (size_t)a.n_obs + a.n_model + 2;
    const size_t side0 = mod ? (size_t)a.n_obs + 1 : 0;
    unsigned* kbuf[2] = {a.sort_key + side0 + b0, a.sort_key + nsp + side0 + b0};
    int* ibuf[2] = {a.sort_idx + side0 + b0, a.sort_idx + nsp + side0 + b0};
    int* perm = (mod ? a.mod_perm : a.obs_perm) + b0;
    int* pos = (mod ? a.mod_pos : a.obs_pos) + b0;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (n <= kRankSort) {
        // a small block: every thread counts the keys before its own, n / 4 steps of the warps that hold keys
        // against six passes of five barriers
        __shared__ __align__(16) unsigned key[kRankSort];
        const int l = threadIdx.x;
        unsigned mine = 0xffffffffu;
        if (l < n) {
            float4 v = mod ? a.mod_r[b0 + l] : a.obs_p[b0 + l];
            mine = direction_key(v.x, v.y, v.z);
        }
        if (l < kRankSort) key[l] = mine;
        __syncthreads();
        if (32 * w >= n) return;
        int before = 0;
        const int before_own = l / 4 * 4;  // whole groups of four keys before the own one
        for (int u = 0; u < n; u += 4) {
            const uint4 k = *(const uint4*)&key[u];
            if (u < before_own)
                before += (k.x <= mine) + (k.y <= mine) + (k.z <= mine) + (k.w <= mine);
            else if (u > before_own)
                before += (k.x < mine) + (k.y < mine) + (k.z < mine) + (k.w < mine);
            else
                before += (k.x < mine || (k.x == mine && u < l)) + (k.y < mine || (k.y == mine && u + 1 < l)) +
                          (k.z < mine || (k.z == mine && u + 2 < l)) + (k.w < mine);
        }
        if (l < n) {
            perm[before] = b0 + l;
            pos[l] = before;
        }
        return;
    }
    for (int l = threadIdx.x; l < n; l += kSortThreads) {
        float4 v = mod ? a.mod_r[b0 + l] : a.obs_p[b0 + l];
        kbuf[0][l] = direction_key(v.x, v.y, v.z);
        ibuf[0][l] = l;
    }
    __syncthreads();
    for (int pass = 0; pass < 6; ++pass) {
        const unsigned* sk = kbuf[pass & 1];
        const int* si = ibuf[pass & 1];
        unsigned* dk = kbuf[(pass + 1) & 1];
        int* di = ibuf[(pass + 1) & 1];
        const int shift = 4 * pass;
        if (threadIdx.x < 16) dbase[threadIdx.x] = 0;
        __syncthreads();
        for (int l = threadIdx.x; l < n; l += kSortThreads) atomicAdd(&dbase[(sk[l] >> shift) & 15u], 1);
        __syncthreads();
        if (threadIdx.x == 0) {
            int acc = 0;
            for (int d = 0; d < 16; ++d) {
                int c = dbase[d];
                dbase[d] = acc;
                acc += c;
            }
        }
        __syncthreads();
        for (int c0 = 0; c0 < n; c0 += kSortThreads) {
            int l = c0 + threadIdx.x;
            bool valid = l < n;
            unsigned key = valid ? sk[l] : 0u;
            int idx = valid ? si[l] : 0;
            int d = valid ? (int)((key >> shift) & 15u) : 16;
            unsigned mine = 0u;
            for (int v = 0; v < 16; ++v) {
                unsigned b = __ballot_sync(0xffffffffu, d == v);
                if (d == v) mine = b;
                if (lane == 0) cnt[w][v] = __popc(b);
            }
            __syncthreads();
            if (threadIdx.x < 16) {
                int acc = dbase[threadIdx.x];
                for (int ww = 0; ww < kSortThreads / 32; ++ww) {
                    int c = cnt[ww][threadIdx.x];
                    cnt[ww][threadIdx.x] = acc;
                    acc += c;
                }
                dbase[threadIdx.x] = acc;
            }
            __syncthreads();
            if (valid) {
                int p = cnt[w][d] + __popc(mine & ((1u << lane) - 1u));
                dk[p] = key;
                di[p] = idx;
            }
            __syncthreads();
        }
    }
    // six passes: the sorted order is back in buffer 0
    for (int l = threadIdx.x; l < n; l += kSortThreads) {
        int idx = ibuf[0][l];
        perm[l] = b0 + idx;
        pos[idx] = l;
    }
}

// Cone of each granule (kGran pairs of one block), one warp per granule:
// axis = normalised mean direction, half-angle = largest angle from it, and
// the smallest |p| (observed) or largest |c| (model).
__global__ void __launch_bounds__(256) sk_cone_kernel(SkArgs a) {
    int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    int n_go = a.obs_gbase[a.T], n_gm = a.mod_gbase[a.T];
    if (warp >= n_go + n_gm) return;
    const bool mod = warp >= n_go;
    const int g = mod ? warp - n_go : warp;
    const int* gb = mod ? a.mod_gbase : a.obs_gbase;
    const int t = block_of(gb, a.T, g);
    const int* off = mod ? a.J_off : a.I_off;
    const int* poff = mod ? a.J2_off : a.I2_off;
    const int nspots = off[t + 1] - off[t];
    const int l0 = 2 * kGran * (g - gb[t]);            // first spot rank of the granule
    const int l1 = min(nspots, l0 + 2 * kGran);
    float d[2 * kGran / 32][3], dx[2 * kGran / 32];
    float sx = 0.f, sy = 0.f, sz = 0.f, ext = mod ? 0.0f : 3.0e38f;
    for (int k = 0; k < 2 * kGran / 32; ++k) {
        int l = l0 + lane + 32 * k;
        d[k][0] = d[k][1] = d[k][2] = 0.0f;
        dx[k] = mod ? 0.0f : 3.0e38f;
        if (l >= l1) continue;
        int q = poff[t] + (l >> 1), ln = l & 1;
        float x, y, z;
        if (mod) {
            float4 Z = a.modZ[q], W = a.modW[q], X = a.modX[q], Y = a.modY[q];
            x = -(ln ? Z.y : Z.x);
            y = -(ln ? Z.w : Z.z);
            z = -(ln ? W.y : W.x);
            float cx = ln ? X.y : X.x, cy = ln ? X.w : X.z, cz = ln ? Y.y : Y.x;
            dx[k] = sqrtf(cx * cx + cy * cy + cz * cz);
            ext = fmaxf(ext, dx[k]);
        } else {
            float4 X = a.obsX[q], Y = a.obsY[q];
            x = ln ? X.y : X.x;
            y = ln ? X.w : X.z;
            z = ln ? Y.y : Y.x;
            float r = sqrtf(x * x + y * y + z * z);
            dx[k] = r;
            ext = fminf(ext, r);
        }
        float r = rsqrtf(fmaxf(x * x + y * y + z * z, 1e-30f));
        d[k][0] = x * r;
        d[k][1] = y * r;
        d[k][2] = z * r;
        sx += d[k][0];
        sy += d[k][1];
        sz += d[k][2];
    }
    // cones of the sub-granules: 2 kSubGran = 16 spots, half a warp
    for (int k = 0; k < 2 * kGran / 32; ++k) {
        const bool have = l0 + lane + 32 * k < l1;
        float mx = d[k][0], my = d[k][1], mz = d[k][2], e = dx[k];
        for (int o = 8; o > 0; o >>= 1) {
            mx += __shfl_xor_sync(0xffffffffu, mx, o);
            my += __shfl_xor_sync(0xffffffffu, my, o);
            mz += __shfl_xor_sync(0xffffffffu, mz, o);
            float y = __shfl_xor_sync(0xffffffffu, e, o);
            e = mod ? fmaxf(e, y) : fminf(e, y);
        }
        const float m2 = mx * mx + my * my + mz * mz;
        const bool none = !(m2 > 1e-12f);  // no axis (or a spot that is not a number): no bound
        const float r = rsqrtf(fmaxf(m2, 1e-30f));
        mx = none ? 0.0f : mx * r;
        my = none ? 0.0f : my * r;
        mz = none ? 1.0f : mz * r;
        float beta = have ? angle_between(mx, my, mz, d[k][0], d[k][1], d[k][2]) : 0.0f;
        for (int o = 8; o > 0; o >>= 1) beta = fmaxf(beta, __shfl_xor_sync(0xffffffffu, beta, o));
        const int sub = 2 * k + (lane >> 4);
        if ((lane & 15) == 0) {
            (mod ? a.mod_sub : a.obs_sub)[kSubs * (size_t)g + sub] = make_float4(mx, my, mz, none ? 3.2f : beta + 1e-5f);
            (mod ? a.mod_subext : a.obs_subext)[kSubs * (size_t)g + sub] = e;
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        sx += __shfl_xor_sync(0xffffffffu, sx, o);
        sy += __shfl_xor_sync(0xffffffffu, sy, o);
        sz += __shfl_xor_sync(0xffffffffu, sz, o);
        ext = mod ? fmaxf(ext, __shfl_xor_sync(0xffffffffu, ext, o)) : fminf(ext, __shfl_xor_sync(0xffffffffu, ext, o));
    }
    float n2 = sx * sx + sy * sy + sz * sz;
    float ax = 0.f, ay = 0.f, az = 1.f;
    bool degenerate = !(n2 > 1e-12f);
    if (!degenerate) {
        float r = rsqrtf(n2);
        ax = sx * r;
        ay = sy * r;
        az = sz * r;
    }
    float beta = 0.0f;
    for (int k = 0; k < 2 * kGran / 32; ++k) {
        int l = l0 + lane + 32 * k;
        if (l >= l1) continue;
        beta = fmaxf(beta, angle_between(ax, ay, az, d[k][0], d[k][1], d[k][2]));
    }
    for (int o = 16; o > 0; o >>= 1) beta = fmaxf(beta, __shfl_xor_sync(0xffffffffu, beta, o));
    if (lane == 0) {
        if (degenerate) beta = 3.2f;  // no bound
        float4* cone = mod ? a.mod_cone : a.obs_cone;
        float* ex = mod ? a.mod_ext : a.obs_ext;
        cone[g] = make_float4(ax, ay, az, beta + 1e-5f);
        ex[g] = ext;
    }
}

// ------------------------------------------------------------------- pack
// Pair-interleaved workspace copies; F, G from the caller's potentials on a
// warm start, else 0.  The thread of the last element of an odd block also
// writes the padding slot.
__global__ void sk_pack_kernel(SkArgs a) {
    const float s = 1.0f / a.to_user;  // mm^2 -> base-2 internal units
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    for (int u = k; u < 4 * a.T; u += gridDim.x * blockDim.x) a.pmax[u] = 0u;
    if (k == 0) {  // the lists are built next
        a.ctrl[CTRL_POOL_NEXT] = 0;
        for (int u = CTRL_ROW_EVAL; u < CTRL_COL_EVAL + 2; ++u) a.ctrl[u] = 0;
    }
    if (k < a.n_obs) {
        int t = block_of(a.I_off, a.T, k);
        int l = a.obs_pos[k];  // rank of the spot in its block's spatial order
        int q = a.I2_off[t] + (l >> 1), lane = l & 1;
        float4 p = a.obs_p[k];
        float* X = (float*)&a.obsX[q];
        float* Y = (float*)&a.obsY[q];
        X[lane] = p.x;
        X[2 + lane] = p.y;
        Y[lane] = p.z;
        const float F = a.warm ? a.f[k] * s : 0.0f;
        Y[2 + lane] = F;
        a.Fc[2 * q + lane] = F;
        if (lane == 0 && l + 1 == a.I_off[t + 1] - a.I_off[t]) {
            X[1] = 0.0f;
            X[3] = 0.0f;
            Y[1] = kPadFar;
            Y[3] = kNegHuge;
            a.Fc[2 * q + 1] = kNegHuge;
        }
    }
    if (k < a.n_model) {
        int t = block_of(a.J_off, a.T, k);
        int l = a.mod_pos[k];
        int q = a.J2_off[t] + (l >> 1), lane = l & 1;
        float4 c = a.mod_c[k];
        float4 r = a.mod_r[k];
        float* X = (float*)&a.modX[q];
        float* Y = (float*)&a.modY[q];
        float* Z = (float*)&a.modZ[q];
        float* W = (float*)&a.modW[q];
        X[lane] = -c.x;
        X[2 + lane] = -c.y;
        Y[lane] = -c.z;
        const float G = a.warm ? a.g[k] * s : 0.0f;
        Y[2 + lane] = G;
        a.Gc[2 * q + lane] = G;
        Z[lane] = -r.x;
        Z[2 + lane] = -r.y;
        W[lane] = -r.z;
        int det = a.mod_s ? (int)a.mod_s[k].w : -1;
        W[2 + lane] = (det >= 0 && det < a.n_det) ? a.negK_det[det] : a.negKD2;
        if (lane == 0 && l + 1 == a.J_off[t + 1] - a.J_off[t]) {
            X[1] = 0.0f;
            X[3] = 0.0f;
            Y[1] = 0.0f;
            Y[3] = kNegHuge;
            a.Gc[2 * q + 1] = kNegHuge;
            Z[1] = 0.0f;
            Z[3] = 0.0f;
            W[1] = -1.0f;
            W[3] = 0.0f;
        }
    }
    if (k == 0) {
        DustPtrs D = dust_ptrs(a.dust, a.T);
        int nd = a.mode ? a.T : 1;
        for (int d = 0; d < nd; ++d) {
            D.F0[d] = (a.warm && a.dust_out) ? a.dust_out[d] * s : 0.0f;
            D.G0[d] = (a.warm && a.dust_out) ? a.dust_out[nd + d] * s : 0.0f;
        }
    }
}

// One CTA: F_0(next) = log2 U - LSE2({G_j} u {G_0 - kc}) for the starting G of a
// warm start.
__global__ void __launch_bounds__(1024) sk_init_dust_kernel(SkArgs a) {
    __shared__ float sm[32], ss[32];
    DustPtrs D = dust_ptrs(a.dust, a.T);
    int nd = a.mode ? a.T : 1;
    for (int d = 0; d < nd; ++d) {
        int q0 = a.mode ? a.J2_off[d] : 0, q1 = a.mode ? a.J2_off[d + 1] : a.J2_off[a.T];
        float m = kNegHuge, s = 0.0f;
        for (int q = q0 + threadIdx.x; q < q1; q += blockDim.x) {
            float4 y = a.modY[q];
            for (int lane = 0; lane < 2; ++lane) {
                float v = lane ? y.w : y.z;
                if (v <= kNegHuge) continue;  // padding
                if (v > m) {
                    s = s * ex2(m - v) + 1.0f;
                    m = v;
                } else {
                    s += ex2(v - m);
                }
            }
        }
        warp_lse_reduce(m, s);
        if ((threadIdx.x & 31) == 0) {
            sm[threadIdx.x >> 5] = m;
            ss[threadIdx.x >> 5] = s;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            Lse2 L;
            L.init(D.G0[d] - a.kc);
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) L.merge(sm[w], ss[w]);
            D.F0n[d] = D.log2U[d] - L.value();
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------- finish
__global__ void sk_finish_kernel(SkArgs a, int have_rows, int have_cols) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    bool bad = false;
    if (k < a.n_obs) {
        int t = block_of(a.I_off, a.T, k);
        int l = a.obs_pos[k];
        float v = a.Fc[2 * a.I2_off[t] + l];
        bad |= !isfinite(v);
        a.f[k] = v * a.to_user;
    }
    if (k < a.n_model) {
        int t = block_of(a.J_off, a.T, k);
        int l = a.mod_pos[k];
        float v = a.Gc[2 * a.J2_off[t] + l];
        bad |= !isfinite(v);
        a.g[k] = v * a.to_user;
    }
    if (k == 0) {
        DustPtrs D = dust_ptrs(a.dust, a.T);
        int nd = a.mode ? a.T : 1;
        if (a.dust_out) {
            for (int d = 0; d < nd; ++d) {
                a.dust_out[d] = D.F0[d] * a.to_user;
                a.dust_out[nd + d] = D.G0[d] * a.to_user;
            }
        }
        if (a.marg_err) {
            a.marg_err[0] = have_rows ? D.err[0] : -1.0f;
            a.marg_err[1] = have_cols ? D.err[1] : -1.0f;
        }
    }
    if (bad) set_status(a.ctrl, LAUE_ERR_NUMERIC);
}

__global__ void sk_clear_err_kernel(SkArgs a) {
    DustPtrs D = dust_ptrs(a.dust, a.T);
    D.err[0] = D.err[1] = D.err[2] = D.err[3] = 0.0f;
}

// Per-angle maxima of the starting G (for the first row pass) and F (for the
// M-step's skipping bound), padding excluded.
__global__ void __launch_bounds__(256) sk_init_gmax_kernel(SkArgs a) {
    __shared__ float red[8], redf[8];
    int t = blockIdx.x;
    float m = kNegHuge, f = kNegHuge;
    for (int q = a.J2_off[t] + threadIdx.x; q < a.J2_off[t + 1]; q += blockDim.x) {
        float4 y = a.modY[q];
        m = fmaxf(m, fmaxf(y.z, y.w));
    }
    for (int q = a.I2_off[t] + threadIdx.x; q < a.I2_off[t + 1]; q += blockDim.x) {
        float4 y = a.obsY[q];
        f = fmaxf(f, fmaxf(y.z, y.w));
    }
    for (int o = 16; o > 0; o >>= 1) {
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        f = fmaxf(f, __shfl_xor_sync(0xffffffffu, f, o));
    }
    if ((threadIdx.x & 31) == 0) {
        red[threadIdx.x >> 5] = m;
        redf[threadIdx.x >> 5] = f;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < 8; ++k) {
            m = fmaxf(m, red[k]);
            f = fmaxf(f, redf[k]);
        }
        DustPtrs D = dust_ptrs(a.dust, a.T);
        D.Gmax[t] = m;
        D.Fmax[t] = f;  // the M-step's skipping bound
    }
}

cudaError_t sinkhorn_prepare(const SkArgs& a, cudaStream_t s, bool dustbins, bool sorted) {
    int nmax = a.n_obs > a.n_model ? a.n_obs : a.n_model;
    int blocks = (nmax + 255) / 256;
    if (blocks < 1) blocks = 1;
    if (!sorted) {
        sk_schedule_kernel<<<1, 1024, 0, s>>>(a, dustbins ? 1 : 0);
        sk_sort_kernel<<<2 * a.T, kSortThreads, 0, s>>>(a);
    }
    sk_pack_kernel<<<blocks, 256, 0, s>>>(a);
    if (!sorted) {
        int max_gran = (a.n_obs + a.n_model) / (2 * kGran) + 2 * a.T + 2;  // bound on the granule count
        sk_cone_kernel<<<(max_gran * 32 + 255) / 256, 256, 0, s>>>(a);
    }
    if (a.warm) {
        if (a.mode != 2 && dustbins) sk_init_dust_kernel<<<1, 1024, 0, s>>>(a);
        sk_init_gmax_kernel<<<a.T, 256, 0, s>>>(a);
    }
    return cudaGetLastError();
}

cudaError_t sinkhorn_finish(const SkArgs& a, const SkLaunch& l, int n_iter, bool want_rows, bool want_cols,
                            cudaStream_t s) {
    int nmax = a.n_obs > a.n_model ? a.n_obs : a.n_model;
    int blocks = (nmax + 255) / 256;
    if (blocks < 1) blocks = 1;
    if (want_rows || want_cols) sk_clear_err_kernel<<<1, 1, 0, s>>>(a);
    cudaError_t e = sinkhorn_harvest(a, l, n_iter, want_rows, want_cols, s);
    if (e != cudaSuccess) return e;
    sk_finish_kernel<<<blocks, 256, 0, s>>>(a, want_rows ? 1 : 0, want_cols ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t sinkhorn_run(const SkArgs& a0, const SkLaunch& l, int n_iter, bool want_rows, bool want_cols,
                         cudaStream_t s) {
    SkArgs a = a0;
    // listing the pairs costs about as much as one sweep of each side
    if (n_iter < 2) a.pool_chunks = 0;
    a.list_share = list_share_of(a, n_iter);
    cudaError_t e = sinkhorn_prepare(a, s);
    if (e != cudaSuccess) return e;
    e = sinkhorn_build_lists(a, l, s);
    if (e != cudaSuccess) return e;
    e = sinkhorn_iterate(a, l, n_iter, s);
    if (e != cudaSuccess) return e;
    return sinkhorn_finish(a, l, n_iter, want_rows, want_cols, s);
}

}  // namespace laue
