// slices.cuh — slices of the pair passes (passes.cu, mstep.cu): the walk over
// the sub-granules that a slice can see, the staging of streamed spots, and
// the entries of listed slices.
#pragma once

#include "pairs.cuh"

namespace laue {

// CTA of a pass over tiles of `tile` pairs that finishes a pass over tiles of `other`
constexpr __host__ __device__ int pass_threads(int tile, int other = 0) {
    return tile > 128 || other > 128 ? 256 : 128;
}

constexpr float kListLog2 = 127.0f;   // K e2 beyond which ex2.approx.ftz gives exactly 0 (potentials <= shift)
constexpr float kQSkip = -40.0f;      // log2 of the smallest plan entry the M-step's sums keep

// Walk over the sub-granules of a streamed block that a slice's cone can see,
// in order; every call is warp-uniform.
struct SubWalk {
    const float4* sub;
    const float* ext;
    int nsub, s0;
    unsigned mask;
    __device__ __forceinline__ void init(const float4* sub_, const float* ext_, int n_pairs) {
        sub = sub_;
        ext = ext_;
        nsub = (n_pairs + kSubGran - 1) / kSubGran;
        s0 = -32;
        mask = 0u;
    }
    // next sub-granule, -1 past the end
    __device__ __forceinline__ int next(const Cone& own, bool own_obs, int skip, float K, float limit) {
        while (!mask) {
            s0 += 32;
            if (s0 >= nsub) return -1;
            const int s = s0 + (threadIdx.x & 31);
            bool need = s < nsub;
            if (need && skip) {
                const Cone c = load_cone(sub, ext, s);
                need = (own_obs ? min_scaled_cost(own, c, K) : min_scaled_cost(c, own, K)) <= limit;
            }
            mask = __ballot_sync(0xffffffffu, need);
        }
        const int s = s0 + __ffs(mask) - 1;
        mask &= mask - 1;
        return s;
    }
};

// What a slice has to do.  pairs: those of the sub-granules that it can see
// (whose cost bound is at most limit).  near (if asked for): about how many
// streamed spots lie within a lane's own angle of its direction d (least: the
// angle's cosine), summed over the lanes, from the axes of the sub-granules.
struct SliceCount {
    int pairs, near;
};
template <bool NEAR>
__device__ __forceinline__ SliceCount count_pairs(const Cone& own, bool own_obs, const float4* sub, const float* ext,
                                                  int n_pairs, int n_spots, int skip, float K, float limit,
                                                  const float (&d)[3], float least) {
    SliceCount n{0, 0};
    const int nsub = (n_pairs + kSubGran - 1) / kSubGran;
    for (int s0 = 0; s0 < nsub; s0 += 32) {
        const int s = s0 + (threadIdx.x & 31);
        Cone c{0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        bool need = s < nsub;
        if (need) {
            c = load_cone(sub, ext, s);
            if (skip) need = (own_obs ? min_scaled_cost(own, c, K) : min_scaled_cost(c, own, K)) <= limit;
        }
        if (need) n.pairs += min(kSubGran, n_pairs - s * kSubGran);
        if (!NEAR) continue;
        for (unsigned m = __ballot_sync(0xffffffffu, need); m; m &= m - 1) {
            const int l = __ffs(m) - 1;
            const float dot = __shfl_sync(0xffffffffu, c.ax, l) * d[0] + __shfl_sync(0xffffffffu, c.ay, l) * d[1] +
                              __shfl_sync(0xffffffffu, c.az, l) * d[2];
            if (dot >= least) n.near += min(2 * kSubGran, n_spots - 2 * (s0 + l) * kSubGran);
        }
    }
    n.pairs = __reduce_add_sync(0xffffffffu, n.pairs);
    if (NEAR) n.near = __reduce_add_sync(0xffffffffu, n.near);
    return n;
}

// One of the first pairs of a batch's four sub-granules.
__device__ __forceinline__ int nth(const int4& f, int g) { return g == 0 ? f.x : g == 1 ? f.y : g == 2 ? f.z : f.w; }

// A warp's staging buffer: two batches of 32 streamed pairs (four
// sub-granules) that cp.async fills while the other is evaluated.
struct WarpStage {
    float4 X[2][32];         // {-cx, -cy} or {px, py} of a pair
    float4 Z[2][32], W[2][32];  // model pairs: {-rx, -ry}, {-rz, -K}
    float2 Y[2][32], P[2][32];  // {-cz} or {pz}; the potentials
};

__device__ __forceinline__ void cp16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp8(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// Streams the pairs of the sub-granules that the slice can see (skip = 0: of
// the whole block) through the warp's buffer; per batch fn(stage, pairs,
// first pair of each of its sub-granules).  The streamed block: n_pairs pairs
// from pair b0 of the model spots (MODEL) or the observed spots; pot their
// potentials (nullptr: not staged).
template <bool MODEL, bool DENSE, class Fn>
__device__ __forceinline__ void sweep(const SkArgs& a, WarpStage& S, const Cone& own, const float4* sub, const float* ext,
                                      int b0, int n_pairs, int skip, float limit, const float* pot, Fn fn) {
    const int lane = threadIdx.x & 31;
    SubWalk walk;
    walk.init(sub, ext, n_pairs);
    auto fetch = [&](int st, int4& first) {  // issues the copies of the next batch; its pairs
        int n = 0;
        int f[4] = {0, 0, 0, 0};
        if (DENSE && __popc(walk.mask) >= 4) {  // without the search for more
            unsigned m = walk.mask;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                f[c] = (walk.s0 + __ffs(m) - 1) * kSubGran;
                m &= m - 1;
            }
            walk.mask = m;
            n = 3 * kSubGran + min(kSubGran, n_pairs - f[3]);
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int s = walk.next(own, MODEL, skip, a.skipK, limit);
                if (s < 0) break;
                f[c] = s * kSubGran;
                n = c * kSubGran + min(kSubGran, n_pairs - f[c]);
            }
        }
        first = make_int4(f[0], f[1], f[2], f[3]);
        if (lane < n) {
            const int g = lane / kSubGran;
            const int q = b0 + (g == 0 ? f[0] : g == 1 ? f[1] : g == 2 ? f[2] : f[3]) + lane % kSubGran;
            cp16(&S.X[st][lane], (MODEL ? a.modX : a.obsX) + q);
            cp8(&S.Y[st][lane], (MODEL ? a.modY : a.obsY) + q);
            if (MODEL) {
                cp16(&S.Z[st][lane], a.modZ + q);
                cp16(&S.W[st][lane], a.modW + q);
            }
            if (pot) cp8(&S.P[st][lane], pot + 2 * (size_t)q);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        return n;
    };
    int4 first, first_n;
    int st = 0, n = fetch(0, first);
    while (n > 0) {
        const int n_next = fetch(st ^ 1, first_n);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();
        fn(st, n, first);
        __syncwarp();
        st ^= 1;
        n = n_next;
        first = first_n;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
}

// |rhat - r|^2 of two packed pairs, the arithmetic of pair_v2.
__device__ __forceinline__ f2 pair_e2(f2 px, f2 py, f2 pz, f2 ncx, f2 ncy, f2 ncz, f2 nrx, f2 nry, f2 nrz) {
    f2 dx = add2(px, ncx), dy = add2(py, ncy), dz = add2(pz, ncz);
    f2 q = mul2(dx, dx);
    q = fma2(dy, dy, q);
    q = fma2(dz, dz, q);
    f2 s = pk(rsq(lo(q)), rsq(hi(q)));
    f2 ex = fma2(dx, s, nrx), ey = fma2(dy, s, nry), ez = fma2(dz, s, nrz);
    f2 e2 = mul2(ex, ex);
    e2 = fma2(ey, ey, e2);
    return fma2(ez, ez, e2);
}

// What a pass needs to know of a slice, written with the lists and kept for
// the iterations.
struct __align__(32) SliceDesc {
    int t, q, nspot;  // angle, first pair of its own, its spots (0: no slice)
    int nch;          // chunks of its lists, -1: swept
    int s0, ns;       // first pair and pairs of the streamed block
    int pad;          // 0
    float cut;        // cost bound beyond which the M-step's sweep skips
};
static_assert(sizeof(SliceDesc) == kSliceDescBytes, "laid out by the host");

// A warp's slice; the lanes' own pairs.
struct Slice {
    int id, t, q, lane, nch;
    int s0, ns;
    float cut;
    bool valid, vb;  // the lane's spots a and b exist
    bool any;
};

__device__ __forceinline__ Slice load_slice(const SliceDesc* desc, int id) {
    Slice s;
    s.id = id;
    s.lane = threadIdx.x & 31;
    const int4 d0 = __ldcg((const int4*)&desc[id]), d1 = __ldcg((const int4*)&desc[id] + 1);
    s.t = d0.x;
    s.q = d0.y + s.lane;
    s.nch = d0.z > 0 ? d0.w : 0;
    s.s0 = d1.x;
    s.ns = d1.y;
    s.cut = __int_as_float(d1.w);
    s.any = d0.z > 0;
    s.valid = 2 * s.lane < d0.z;
    s.vb = 2 * s.lane + 1 < d0.z;
    return s;
}

// Number of slices of a side: kW per tile.
template <int TILE>
__device__ __forceinline__ int slice_count(const SkArgs& a, bool rows) {
    return __ldcg(a.ctrl + (rows ? CTRL_N_ROW_TILES : CTRL_N_COL_TILES)) * (TILE / 32);
}

// Observed pair of a lane, duplicated for the packed arithmetic.
struct RowPair {
    f2 pxa, pya, pza, pxb, pyb, pzb;
};

__device__ __forceinline__ RowPair load_row_pair(const SkArgs& a, int q, bool valid) {
    float4 X = valid ? a.obsX[q] : make_float4(0.f, 0.f, 0.f, 0.f);
    float2 Y = valid ? *(const float2*)&a.obsY[q] : make_float2(kPadFar, kPadFar);
    return RowPair{dup(X.x), dup(X.z), dup(Y.x), dup(X.y), dup(X.w), dup(Y.y)};
}


// ---------------------------------------------------- entries of a listed slice
// A chunk in memory: the costs of 8 entries of each of the 64 spots, then their slots.
struct Chunk {
    float2 e2[kListDepth][32];      // of the lane's spots a and b
    unsigned slot[kListDepth][32];  // a in the low half, b in the high half
};
static_assert(sizeof(Chunk) == kListChunkBytes, "laid out by the host");

// A warp's ring of chunks in shared memory, filled by cp.async: the lists are
// read once per pass, from HBM at the 1000-grain density, so the next chunks
// are in flight while one is used.  The first ones are asked for before the
// pass waits for the one before it.
constexpr int kRing = 3;
struct Ring {
    Chunk c[kRing];
};

// The lane's share of a slice's chunk numbers [32 k, 32 k + 32).
__device__ __forceinline__ int chunk_numbers(const SkArgs& a, const int* tab, int id, int lane, int k) {
    return a.pool_chunks > 0 ? __ldcg(tab + (size_t)kListChunks * id + 32 * k + lane) : 0;
}

__device__ __forceinline__ void ring_fill(const SkArgs& a, Ring& R, int c, int nch, int number, int lane) {
    if (c < nch) {
        const char* src = a.pool + (size_t)number * kListChunkBytes + 16 * lane;
        char* dst = (char*)&R.c[c % kRing] + 16 * lane;
#pragma unroll
        for (int k = 0; k < (int)kListChunkBytes / 512; ++k) cp16(dst + 512 * k, src + 512 * k);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// numbers: the lane's share of the first 32 chunk numbers
__device__ __forceinline__ void ring_start(const SkArgs& a, Ring& R, const Slice& sl, int numbers) {
#pragma unroll
    for (int c = 0; c < kRing - 1; ++c) ring_fill(a, R, c, sl.nch, __shfl_sync(0xffffffffu, numbers, c), sl.lane);
}

// fn(chunk) for every chunk of the slice, in order.
template <class Fn>
__device__ __forceinline__ void for_each_chunk(const SkArgs& a, Ring& R, const int* tab, const Slice& sl, int numbers,
                                               Fn fn) {
    for (int c = 0; c < sl.nch; ++c) {
        const int ahead = c + kRing - 1;
        if ((ahead & 31) == 0 && ahead < sl.nch) numbers = chunk_numbers(a, tab, sl.id, sl.lane, ahead >> 5);
        ring_fill(a, R, ahead, sl.nch, __shfl_sync(0xffffffffu, numbers, ahead & 31), sl.lane);
        asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 1) : "memory");
        __syncwarp();
        fn(R.c[c % kRing]);
        __syncwarp();
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// ------------------------------------------------------------ swept slices
__device__ __forceinline__ void row_pair_v(const RowPair& R, const WarpStage& S, int st, int j, f2 base, f2& va, f2& vb) {
    const ulonglong2 X = *(const ulonglong2*)&S.X[st][j], Z = *(const ulonglong2*)&S.Z[st][j],
                     W = *(const ulonglong2*)&S.W[st][j];
    const f2 ncz = *(const f2*)&S.Y[st][j];
    va = pair_v2(R.pxa, R.pya, R.pza, X.x, X.y, ncz, Z.x, Z.y, W.x, W.y, base);
    vb = pair_v2(R.pxb, R.pyb, R.pzb, X.x, X.y, ncz, Z.x, Z.y, W.x, W.y, base);
}

__device__ __forceinline__ void col_pair_v(const ColPair& C, const WarpStage& S, int st, int j, f2 base, f2& va, f2& vb) {
    const ulonglong2 X = *(const ulonglong2*)&S.X[st][j];
    const f2 pz = *(const f2*)&S.Y[st][j];
    va = pair_v2(X.x, X.y, pz, C.ncxa, C.ncya, C.ncza, C.nrxa, C.nrya, C.nrza, C.ka, base);
    vb = pair_v2(X.x, X.y, pz, C.ncxb, C.ncyb, C.nczb, C.nrxb, C.nryb, C.nrzb, C.kb, base);
}

// What the slices of either side need to sweep the other.
struct Sweep {
    Cone own;
    const float4* sub;
    const float* ext;
    int b0, n;
};

template <bool ROWS>
__device__ __forceinline__ Sweep sweep_of(const SkArgs& a, const Slice& sl) {
    const int first = sl.q - sl.lane, t = sl.t;
    Sweep w;
    if (ROWS) {
        w.own = load_cone(a.obs_cone, a.obs_ext, a.obs_gbase[t] + (first - a.I2_off[t]) / kGran);
        w.sub = a.mod_sub + (size_t)kSubs * a.mod_gbase[t];
        w.ext = a.mod_subext + (size_t)kSubs * a.mod_gbase[t];
    } else {
        w.own = load_cone(a.mod_cone, a.mod_ext, a.mod_gbase[t] + (first - a.J2_off[t]) / kGran);
        w.sub = a.obs_sub + (size_t)kSubs * a.obs_gbase[t];
        w.ext = a.obs_subext + (size_t)kSubs * a.obs_gbase[t];
    }
    w.b0 = sl.s0;
    w.n = sl.ns;
    return w;
}

// fn(stage, pair of the stage, pair of the block) over the slice's sweep, whose
// staged potentials are less `shift`; skip = 0: over the whole block.
template <bool ROWS, class Fn>
__device__ __forceinline__ void for_each_swept(const SkArgs& a, WarpStage& S, const Slice& sl, int skip, float shift,
                                               Fn fn) {
    const Sweep w = sweep_of<ROWS>(a, sl);
    sweep<ROWS, true>(a, S, w.own, w.sub, w.ext, w.b0, w.n, skip, kSkipLog2, ROWS ? a.Gc : a.Fc,
                      [&](int st, int n, const int4& f) {
        float2& P = S.P[st][sl.lane];
        if (sl.lane < n) P = make_float2(P.x - shift, P.y - shift);
        __syncwarp();
#pragma unroll 4
        for (int j = 0; j < n; ++j) fn(st, j, nth(f, j / kSubGran) + j % kSubGran);
    });
}

// A warp's shared memory: its slice is listed or swept.
union WarpBuffer {
    WarpStage stage;
    Ring ring;
};

}  // namespace laue
