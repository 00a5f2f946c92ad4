// passes.cu — the pair passes of the fused E-step (see sinkhorn.cu): the pair
// lists, the row and column updates, and the plan read-out.
//
// A pass runs one warp per SLICE: 32 consecutive spot pairs of a tile, each
// lane holding the two spots a and b of its pair.  A slice is either LISTED
// (see sk_list_kernel: the pairs whose plan entry can be nonzero, with their
// costs) or SWEPT: the warp walks the sub-granules of the block that its cone
// can see, stages their spots in shared memory and evaluates every pair of
// them.
//
// Both forms add the same nonzero terms in the same order (ascending slot of
// the other side, even and odd slots in two accumulators), and every term
// they leave out is exactly 0, so a potential has the same bits either way.
//
// A pass has no serial end: the tiles' partial sums are merged into the dustbin
// potentials by CTAs of the NEXT pass (see finish_pass), which does not need
// them yet: the row update takes G_0 of the column pass before the last row
// update, the column update F_0 of the column update before.  So CTAs are
// small (four slices), and end as soon as their longest slice does.
#include <algorithm>
#include <type_traits>

#include "slices.cuh"

namespace laue {

constexpr float kTinySum = 1.0e-30f;  // below ~2^-100 the fast sum is recomputed exactly
constexpr float kFarLog2 = 60.0f;     // see the read-out kernels
constexpr float kListAlways = 1.0e30f;  // list_share of slices that need not look

// ------------------------------------------------------------- pair lists
// For fixed poses and temperature the pairs whose plan entry can be nonzero
// do not change over the iterations of an E-step: with the potentials at most
// the shift, a term is 2^(G_j - shift - K e2) <= 2^(-K e2), which
// ex2.approx.ftz flushes to 0 beyond K e2 = 126.  So each slice's pairs with
// K e2 <= kListLog2 are listed once per E-step, with the cost e2 that the
// passes would recompute: 0.44 % of the 9.2e9 same-angle pairs of the
// 1000-grain configuration at 1 mm^2, where the passes used to evaluate
// 28.9 %.  A pass then streams 6 bytes per entry (HBM) instead of spending 13
// packed instructions and two MUFU per evaluated pair.  Measured at that size:
// listing 1.70 + 1.48 ms once, a pass 1.57 / 1.50 ms before and 0.063 ms now.
// A single iteration is not worth listing for: one sweep of both sides takes
// about as long (sinkhorn_run).
//
// One warp lists one slice; chunks come from the pool as the longest of the
// slice's 64 lists grows (a chunk's place in the pool is not reproducible, its
// contents are).  A slice is left to the sweep when its chunks run out, when a
// block has more than 65536 spots (16-bit slots), or when more than half of
// the pairs it evaluates would be listed: a listed entry costs about as much
// as two swept pairs.
//
// A list that is given up halfway is lost time (up to fifteen swept passes of
// the slice), so a slice first estimates its entries: how many of the streamed
// spots' sub-granules lie, by their axes, within the listed angle of its own
// spots.  It is left to the sweep if they exceed a list, or list_share of its
// evaluated pairs (list_share_of).  The cost of listing is 1.4 swept iterations at
// an entry per 30 evaluated pairs, 3 at one in 6, 4 to 11 at one in 3, so the share
// grows with the iterations that a list is used for.  90 angles of 13300 x 7744
// spots, 20 iterations at 100 mm^2: 91.6 ms when every slice tried, 77.7 now (at
// 21 mm^2, where the pool holds a part of the entries: 48.0 and 46.4); 60 angles
// of 1020 x 776 spots, 2 and 5 iterations at 100 mm^2: 0.90 and 1.06 ms, now 0.52
// and 0.79; at 1 mm^2 the same slices are listed.
//
// Most of the pairs that the cones let through are still too far apart, so a
// cheap test comes first: the angle between p (seen from the origin) and r is
// at most the angle of the cost bound plus the parallax asin(|c| / |p|), three
// packed multiply-adds per two pairs against thirteen and two MUFU.  Only the
// pairs that pass it (a bit mask per spot and batch) have their cost taken.
struct ListStage {
    WarpStage S;
    float2 nx[32], ny[32], nz[32];  // unit directions of the streamed pairs
    int tab[kListChunks];
};

constexpr int kListWarps = 4;

// PLAN (columns of the M-step): the entries are the pairs whose plan entry
// 2^v, v = F_i + G_j - K e2, is at least 2^kQSkip, and hold that entry instead
// of the cost; the cut-off of the cost is then what the angle's largest F and
// the slice's largest G leave.
template <int TILE, bool ROWS, bool PLAN>
__global__ void __launch_bounds__(32 * kListWarps) sk_list_kernel(SkArgs a) {
    static_assert(!(ROWS && PLAN), "the M-step sums over columns");
    __shared__ __align__(16) ListStage stage[kListWarps];
    constexpr int kW = TILE / 32;
    const int lane = threadIdx.x & 31;
    const int id = blockIdx.x * kListWarps + (threadIdx.x >> 5);
    const int tile = id / kW, w = id % kW;
    if (tile >= a.ctrl[ROWS ? CTRL_N_ROW_TILES : CTRL_N_COL_TILES]) return;
    ListStage& L = stage[threadIdx.x >> 5];
    const int4 td = (ROWS ? a.row_tiles : a.col_tiles)[tile];
    const int t = td.x, first = td.y + 32 * w, n_own = min(32, max(0, td.z - 32 * w));
    SliceDesc& desc = ((SliceDesc*)(ROWS ? a.row_desc : a.col_desc))[id];
    if (n_own == 0) {
        if (lane < 8) ((int*)&desc)[lane] = 0;  // no spots, no chunks
        return;
    }
    const int q = first + lane;
    const bool valid = lane < n_own;
    const int o0 = (ROWS ? a.I2_off : a.J2_off)[t], b0 = (ROWS ? a.J2_off : a.I2_off)[t];
    const int np = (ROWS ? a.J2_off : a.I2_off)[t + 1] - b0;
    const int* own_off = ROWS ? a.I_off : a.J_off;
    const int* str_off = ROWS ? a.J_off : a.I_off;
    const int n_str = str_off[t + 1] - str_off[t];
    const bool vb = valid && 2 * (q - o0) + 1 < own_off[t + 1] - own_off[t];
    const int* own_g = ROWS ? a.obs_gbase : a.mod_gbase;
    const int* str_g = ROWS ? a.mod_gbase : a.obs_gbase;
    const Cone own = load_cone(ROWS ? a.obs_cone : a.mod_cone, ROWS ? a.obs_ext : a.mod_ext,
                               own_g[t] + (first - o0) / kGran);
    const float4* sub = (ROWS ? a.mod_sub : a.obs_sub) + (size_t)kSubs * str_g[t];
    const float* subext = (ROWS ? a.mod_subext : a.obs_subext) + (size_t)kSubs * str_g[t];
    float2 G = make_float2(kNegHuge, kNegHuge);
    float cut = kListLog2, cone_cut = kSkipLog2;
    if (PLAN) {
        if (valid) G = *(const float2*)&a.Gc[2 * (size_t)q];
        float top = fmaxf(G.x, G.y);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
        cut = cone_cut = dust_ptrs(a.dust, a.T).Fmax[t] + top - kQSkip + 1.0f;
    }
    RowPair R{};
    ColPair C;
    if (ROWS) R = load_row_pair(a, q, valid);
    else load_col_pair(a, valid ? q : first, C);
    // unit directions of the lane's spots
    float da[3], db[3];
    if (ROWS) {
        const float x[6] = {lo(R.pxa), lo(R.pya), lo(R.pza), lo(R.pxb), lo(R.pyb), lo(R.pzb)};
        const float ra = rsqrtf(x[0] * x[0] + x[1] * x[1] + x[2] * x[2]);
        const float rb = rsqrtf(x[3] * x[3] + x[4] * x[4] + x[5] * x[5]);
        for (int k = 0; k < 3; ++k) {
            da[k] = x[k] * ra;
            db[k] = x[3 + k] * rb;
        }
    } else {
        da[0] = -lo(C.nrxa), da[1] = -lo(C.nrya), da[2] = -lo(C.nrza);
        db[0] = -lo(C.nrxb), db[1] = -lo(C.nryb), db[2] = -lo(C.nrzb);
    }
    // the angle of a cost of `most` in units of 1 / K, K 4 sin^2(th / 2) = most
    auto angle_of = [](float most, float K) {
        const float h = fmaxf(most, 0.0f) / (4.0f * K);
        return h < 1.0f ? 2.0f * asinf(sqrtf(h)) : 7.0f;
    };
    bool fail = a.pool_chunks == 0 || n_str > 65536;
    int evaluated;
    if (fail || a.list_share >= kListAlways) {
        evaluated = count_pairs<false>(own, ROWS, sub, subext, np, n_str, a.skip, a.skipK, cone_cut, da, 2.0f).pairs;
    } else {
        // the entries that the lanes' first spots will have, on average: too many to list, or to be worth it?
        const float far = angle_of(PLAN ? dust_ptrs(a.dust, a.T).Fmax[t] + G.x - kQSkip : cut, a.listK);
        const SliceCount n = count_pairs<true>(own, ROWS, sub, subext, np, n_str, a.skip, a.skipK, cone_cut, da,
                                               !valid ? 2.0f : far < 3.1f ? cosf(far) : -3.0f);
        evaluated = n.pairs;
        const float mean = (float)n.near / (float)n_own;
        fail = mean > (float)(kListDepth * kListChunks) || mean > a.list_share * (float)evaluated;
    }
    int ca = 0, cb = 0, nch = 0;
    if (!fail) {
        const float th = angle_of(cut, a.skipK);  // of the largest listed cost of any spot
        const f2 dax = dup(da[0]), day = dup(da[1]), daz = dup(da[2]);
        const f2 dbx = dup(db[0]), dby = dup(db[1]), dbz = dup(db[2]);
        auto put = [&](int& cnt, int ab, float e2, int slot) {
            char* p = a.pool + (size_t)L.tab[cnt / kListDepth] * kListChunkBytes;
            const int at = (cnt % kListDepth) * 64 + 2 * lane + ab;
            ((float*)p)[at] = e2;
            ((unsigned short*)(p + kListDepth * 64 * 4))[at] = (unsigned short)slot;
            ++cnt;
        };
        sweep<ROWS, false>(a, L.S, own, sub, subext, b0, np, a.skip, cone_cut, PLAN ? a.Fc : nullptr,
                    [&](int st, int n, const int4& f) {
            if (fail || kListDepth * nch > evaluated) {
                fail = true;  // mostly nonzero: the sweep is as good
                return;
            }
            // the batch's unit directions; the largest parallax of the slice with it
            float ext = ROWS ? 0.0f : 3.0e38f;
            {
                const float4 X = L.S.X[st][lane];
                const float2 Y = L.S.Y[st][lane];
                float2 ux = make_float2(X.x, X.y), uy = make_float2(X.z, X.w), uz = Y;
                if (ROWS) {
                    const float4 Z = L.S.Z[st][lane], W = L.S.W[st][lane];
                    ux = make_float2(-Z.x, -Z.y), uy = make_float2(-Z.z, -Z.w), uz = make_float2(-W.x, -W.y);
                } else {
                    const float r0 = rsqrtf(ux.x * ux.x + uy.x * uy.x + uz.x * uz.x);
                    const float r1 = rsqrtf(ux.y * ux.y + uy.y * uy.y + uz.y * uz.y);
                    ux = make_float2(ux.x * r0, ux.y * r1);
                    uy = make_float2(uy.x * r0, uy.y * r1);
                    uz = make_float2(uz.x * r0, uz.y * r1);
                }
                L.nx[lane] = ux;
                L.ny[lane] = uy;
                L.nz[lane] = uz;
                if (lane < n) ext = subext[(nth(f, lane / kSubGran)) / kSubGran];
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float y = __shfl_xor_sync(0xffffffffu, ext, o);
                ext = ROWS ? fmaxf(ext, y) : fminf(ext, y);
            }
            const float cmax = ROWS ? ext : own.ext, pmin = ROWS ? own.ext : ext;
            const float reach = th + (pmin > cmax ? asinf(cmax / pmin) : 7.0f) + 1e-4f;
            const float least = reach < 3.1f ? cosf(reach) - 4e-6f : -3.0f;
            __syncwarp();
            unsigned ma[2] = {0u, 0u}, mb[2] = {0u, 0u};
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                const int j1 = min(16, n - 16 * hf);
#pragma unroll 4
                for (int j = 0; j < j1; ++j) {
                    const f2 x = *(const f2*)&L.nx[16 * hf + j], y = *(const f2*)&L.ny[16 * hf + j],
                             z = *(const f2*)&L.nz[16 * hf + j];
                    const f2 ta = fma2(daz, z, fma2(day, y, mul2(dax, x)));
                    const f2 tb = fma2(dbz, z, fma2(dby, y, mul2(dbx, x)));
                    // not less, so that a spot that is not a number stays
                    ma[hf] |= (!(lo(ta) < least) ? 1u : 0u) << (2 * j) | (!(hi(ta) < least) ? 2u : 0u) << (2 * j);
                    mb[hf] |= (!(lo(tb) < least) ? 1u : 0u) << (2 * j) | (!(hi(tb) < least) ? 2u : 0u) << (2 * j);
                }
            }
            for (int hf = 0; hf < 2; ++hf) {
                unsigned m0 = valid ? ma[hf] : 0u, m1 = vb ? mb[hf] : 0u;
                // room for the half batch
                while (!fail && __any_sync(0xffffffffu, max(ca + __popc(m0), cb + __popc(m1)) > kListDepth * nch)) {
                    int c = a.pool_chunks;
                    if (nch < kListChunks) {
                        if (lane == 0) c = atomicAdd(a.ctrl + CTRL_POOL_NEXT, 1);
                        c = __shfl_sync(0xffffffffu, c, 0);
                    }
                    fail = c >= a.pool_chunks;
                    if (!fail) {
                        if (lane == 0) L.tab[nch] = c;
                        __syncwarp();
                        ++nch;
                    }
                }
                if (fail) return;
                while (__any_sync(0xffffffffu, m0 | m1)) {
#pragma unroll
                    for (int ab = 0; ab < 2; ++ab) {
                        unsigned& m = ab ? m1 : m0;
                        if (!m) continue;
                        const int bit = __ffs(m) - 1;
                        m &= m - 1;
                        const int j = 16 * hf + (bit >> 1);
                        const int slot = 2 * (nth(f, j / kSubGran) + j % kSubGran) + (bit & 1);
                        const ulonglong2 X = *(const ulonglong2*)&L.S.X[st][j];
                        const f2 Y = *(const f2*)&L.S.Y[st][j];
                        f2 e;
                        float k;
                        if (ROWS) {
                            const ulonglong2 Z = *(const ulonglong2*)&L.S.Z[st][j], W = *(const ulonglong2*)&L.S.W[st][j];
                            e = pair_e2(ab ? R.pxb : R.pxa, ab ? R.pyb : R.pya, ab ? R.pzb : R.pza, X.x, X.y, Y, Z.x, Z.y,
                                        W.x);
                            k = bit & 1 ? hi(W.y) : lo(W.y);
                        } else {
                            e = pair_e2(X.x, X.y, Y, ab ? C.ncxb : C.ncxa, ab ? C.ncyb : C.ncya, ab ? C.nczb : C.ncza,
                                        ab ? C.nrxb : C.nrxa, ab ? C.nryb : C.nrya, ab ? C.nrzb : C.nrza);
                            k = lo(ab ? C.kb : C.ka);
                        }
                        float e2 = bit & 1 ? hi(e) : lo(e);
                        bool in;
                        if (PLAN) {
                            const float2 F = L.S.P[st][j];
                            const float v = fmaf(e2, k, bit & 1 ? F.y : F.x) + (ab ? G.y : G.x);
                            in = !(v < kQSkip);
                            e2 = ex2(v);
                        } else {
                            in = !(e2 * k < -kListLog2);
                        }
                        // the padding spot of an odd block is no entry
                        if (in && slot < n_str) put(ab ? cb : ca, ab, e2, slot);
                    }
                }
            }
        });
    }
    int most = max(ca, cb);
    for (int o = 16; o > 0; o >>= 1) most = max(most, __shfl_xor_sync(0xffffffffu, most, o));
    nch = fail ? 0 : (most + kListDepth - 1) / kListDepth;
    // entries of the slice (with padding) against the spot pairs of the sweep
    if (!fail && nch * kListDepth > evaluated) fail = true;
    if (!fail) {
        int* to = (ROWS ? a.row_tab : a.col_tab) + (size_t)kListChunks * id;
        for (int c = lane; c < nch; c += 32) to[c] = L.tab[c];
        // pad every list to the slice's depth (2^-inf adds nothing)
        for (int ab = 0; ab < 2; ++ab)
            for (int c = ab ? cb : ca; c < kListDepth * nch; ++c) {
                char* p = a.pool + (size_t)L.tab[c / kListDepth] * kListChunkBytes;
                const int at = (c % kListDepth) * 64 + 2 * lane + ab;
                ((float*)p)[at] = PLAN ? 0.0f : 3.0e38f;
                ((unsigned short*)(p + kListDepth * 64 * 4))[at] = 0;
            }
    }
    if (lane == 0) {
        desc.t = t;
        desc.q = first;
        desc.nspot = min(64, own_off[t + 1] - own_off[t] - 2 * (first - o0));
        desc.nch = fail ? -1 : nch;
        desc.s0 = b0;
        desc.ns = np;
        desc.cut = cone_cut;
        desc.pad = 0;
        const long long n = fail ? 4LL * n_own * evaluated : 64LL * kListDepth * nch;
        atomicAdd((unsigned long long*)(a.ctrl + (ROWS ? CTRL_ROW_EVAL : CTRL_COL_EVAL)), (unsigned long long)n);
        if (PLAN && a.pool_chunks > 0)  // the pairs that listing the plan visits
            atomicAdd((unsigned long long*)(a.ctrl + CTRL_MS_PAIRS), (unsigned long long)(4LL * n_own * evaluated));
    }
}

// Sums of 2^(pot_slot - shift - K e2) over a listed slice's entries for the
// lane's two spots: even slots into e, odd slots into o.  GATHER_K: -K comes
// with the slot's model spot (rows of a geometry with several cost lengths).
struct ListSum {
    float ea, oa, eb, ob;
};

template <bool GATHER_K>
__device__ __forceinline__ void list_sum(const SkArgs& a, Ring& R, const int* tab, const Slice& sl, int numbers,
                                         const float* pot, float shift, float ka, float kb, const float4* modW,
                                         ListSum& S) {
    for_each_chunk(a, R, tab, sl, numbers, [&](const Chunk& C) {
        float pa[kListDepth], pb[kListDepth];
#pragma unroll
        for (int k = 0; k < kListDepth; ++k) {
            const unsigned s = C.slot[k][sl.lane];
            pa[k] = pot[s & 0xffffu];
            pb[k] = pot[s >> 16];
        }
#pragma unroll
        for (int k = 0; k < kListDepth; ++k) {
            const unsigned s = C.slot[k][sl.lane];
            const float2 e2 = C.e2[k][sl.lane];
            if (GATHER_K) {
                const unsigned ja = s & 0xffffu, jb = s >> 16;
                const float2 wa = *((const float2*)&modW[ja >> 1] + 1), wb = *((const float2*)&modW[jb >> 1] + 1);
                ka = ja & 1u ? wa.y : wa.x;
                kb = jb & 1u ? wb.y : wb.x;
            }
            const float ta = ex2(fmaf(e2.x, ka, pa[k] - shift)), tb = ex2(fmaf(e2.y, kb, pb[k] - shift));
            const bool oa = s & 1u, ob = s & 0x10000u;
            S.ea += oa ? 0.0f : ta;
            S.oa += oa ? ta : 0.0f;
            S.eb += ob ? 0.0f : tb;
            S.ob += ob ? tb : 0.0f;
        }
    });
}

// Shifted sums over a swept slice.
template <bool ROWS>
__device__ __forceinline__ void swept_sum(const SkArgs& a, WarpStage& S, const Slice& sl, float shift, ListSum& out) {
    f2 Sa = pk(out.ea, out.oa), Sb = pk(out.eb, out.ob);
    auto add = [&](f2 va, f2 vb) {
        Sa = add2(Sa, pk(ex2(lo(va)), ex2(hi(va))));
        Sb = add2(Sb, pk(ex2(lo(vb)), ex2(hi(vb))));
    };
    if (ROWS) {
        const RowPair R = load_row_pair(a, sl.q, sl.valid);
        for_each_swept<ROWS>(a, S, sl, a.skip, shift, [&](int st, int j, int) {
            f2 va, vb;
            row_pair_v(R, S, st, j, *(const f2*)&S.P[st][j], va, vb);
            add(va, vb);
        });
    } else {
        ColPair C;
        load_col_pair(a, sl.valid ? sl.q : sl.q - sl.lane, C);
        for_each_swept<ROWS>(a, S, sl, a.skip, shift, [&](int st, int j, int) {
            f2 va, vb;
            col_pair_v(C, S, st, j, *(const f2*)&S.P[st][j], va, vb);
            add(va, vb);
        });
    }
    out = ListSum{lo(Sa), hi(Sa), lo(Sb), hi(Sb)};
}

// Exact log-sum-exps (running maximum) of the lanes' two spots over part
// `part` of PARTS of the block (dust: the starting value), where a shifted sum
// underflowed: four streamed pairs to a group.
template <bool ROWS, int PARTS>
__device__ __forceinline__ void exact_sums(const SkArgs& a, WarpStage& S, const Slice& sl, float dust, int part,
                                           RowLse& A, RowLse& B) {
    A.init(dust);
    B.init(dust);
    RowPair R{};
    ColPair C;
    if (ROWS) R = load_row_pair(a, sl.q, sl.valid);
    else load_col_pair(a, sl.valid ? sl.q : sl.q - sl.lane, C);
    const Sweep w = sweep_of<ROWS>(a, sl);
    int from = 0, to = w.n;
    if (PARTS > 1) {
        const int subs = (w.n + kSubGran - 1) / kSubGran;
        from = subs * part / PARTS * kSubGran;
        to = min(subs * (part + 1) / PARTS * kSubGran, w.n);
    }
    sweep<ROWS, true>(a, S, w.own, w.sub, w.ext, w.b0 + from, to - from, 0, kSkipLog2, ROWS ? a.Gc : a.Fc,
                [&](int st, int n, const int4&) {
        auto pair = [&](int j, f2& va, f2& vb) {
            const f2 base = *(const f2*)&S.P[st][j];
            if (ROWS) row_pair_v(R, S, st, j, base, va, vb);
            else col_pair_v(C, S, st, j, base, va, vb);
        };
        int j = 0;
        for (; j + kGroup <= n; j += kGroup) {
            f2 va[kGroup], vb[kGroup];
#pragma unroll
            for (int g = 0; g < kGroup; ++g) pair(j + g, va[g], vb[g]);
            A.add4(va);
            B.add4(vb);
        }
        for (; j < n; ++j) {
            f2 va, vb;
            pair(j, va, vb);
            A.add1(va);
            B.add1(vb);
        }
    });
}

template <bool ROWS>
__device__ __noinline__ void exact_lse(const SkArgs& a, WarpStage& S, const Slice& sl, float dust, float& va_out,
                                       float& vb_out) {
    RowLse A, B;
    exact_sums<ROWS, 1>(a, S, sl, dust, 0, A, B);
    va_out = A.value();
    vb_out = B.value();
}

// One of several parts: {max a, sum a, max b, sum b}.
template <bool ROWS, int PARTS>
__device__ __noinline__ float4 exact_part(const SkArgs& a, WarpStage& S, const Slice& sl, float dust, int part) {
    RowLse A, B;
    exact_sums<ROWS, PARTS>(a, S, sl, dust, part, A, B);
    return make_float4(A.m, lo(A.S) + hi(A.S), B.m, lo(B.S) + hi(B.S));
}

// ----------------------------------------------------- ends of the passes
// Largest potential of each angle block, kept by the passes as the maximum of
// the tile partials in an order-preserving code (0: none yet).  Rows and
// columns have two sets each: pass `it` fills set it & 1, and clears the other
// side's set that the next pass fills, whose readers are done.
__device__ __forceinline__ unsigned max_code(float v) {
    const unsigned b = __float_as_uint(v);
    return b & 0x80000000u ? ~b : b | 0x80000000u;
}
__device__ __forceinline__ float angle_max(const unsigned* set, int t, float add) {
    const unsigned k = __ldcg(set + t);
    const float m = k == 0u ? kNegHuge : __uint_as_float(k & 0x80000000u ? k & 0x7fffffffu : ~k);
    return m > kNegHuge ? m + add : kNegHuge;
}
__device__ __forceinline__ unsigned* row_max(const SkArgs& a, int it) { return a.pmax + (it & 1) * a.T; }
__device__ __forceinline__ unsigned* col_max(const SkArgs& a, int it) { return a.pmax + (2 + (it & 1)) * a.T; }
// after n_iter iterations (0: the maxima of the starting potentials)
__device__ __forceinline__ float final_row_max(const SkArgs& a, const DustPtrs& D, int t, int n_iter) {
    return n_iter > 0 ? angle_max(row_max(a, n_iter - 1), t, a.kc) : D.Fmax[t];
}
__device__ __forceinline__ float final_col_max(const SkArgs& a, const DustPtrs& D, int t, int n_iter) {
    return n_iter > 0 ? angle_max(col_max(a, n_iter - 1), t, 0.0f) : D.Gmax[t];
}

// Lanes' partial log-sum-exps of a tile into part[tile], its warps in order,
// and the angle's maximum.  Only the tile's own warps meet here.
template <int TILE>
__device__ __forceinline__ void store_part(float m, float s, int tile, int t, float2* part, unsigned* maxima, float* sm,
                                           float* ss) {
    constexpr int kW = TILE / 32;
    const int warp = threadIdx.x >> 5;
    warp_lse_reduce(m, s);
    if ((threadIdx.x & 31) == 0) {
        sm[warp] = m;
        ss[warp] = s;
    }
    asm volatile("bar.sync %0, %1;" ::"r"(1 + warp / kW), "n"(TILE) : "memory");
    if ((int)threadIdx.x % TILE == 0) {
        Lse2 L;
        L.m = kNegHuge;
        L.s = 0.0f;
        for (int k = 0; k < kW; ++k) L.merge(sm[warp + k], ss[warp + k]);
        part[tile] = make_float2(L.m, L.s);
        if (L.m > kNegHuge) atomicMax(maxima + t, max_code(L.m));
    }
}

// True in exactly one CTA, the last one to get here.
__device__ __forceinline__ bool last_block(int* done, int* flag) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        *flag = atomicAdd(done, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    const bool last = *flag != 0;
    if (last) __threadfence();
    return last;
}

// Log-sum-exp of the n tile partials by one CTA: TILE chains (chain c
// takes the tiles c, c + TILE, ... in order), then the chains by warp and the
// warps in order.  A chain's running maxima are known before its sum (a prefix
// maximum), so every exponential is taken in parallel and only the sum's
// multiply-adds are serial: the CTA's segments of a chain hold their
// elements in registers and hand the sum on.  Thread 0 gets (m, s).
template <int TILE, int THREADS>
__device__ void merge_parts(const float2* part, int n, float& m_out, float& s_out, float* sm, float* ss,
                            float (*segmax)[TILE], float* cm, float* cs) {
    constexpr int kSeg = THREADS / TILE, kR = 8;
    const int c = threadIdx.x % TILE, seg = threadIdx.x / TILE;
    if (seg == 0) {
        cm[c] = kNegHuge;
        cs[c] = 0.0f;
    }
    for (int r0 = 0; r0 * TILE < n; r0 += kSeg * kR) {
        float2 v[kR];
        float top = kNegHuge;
#pragma unroll
        for (int i = 0; i < kR; ++i) {
            const int k = c + TILE * (r0 + seg * kR + i);
            v[i] = k < n ? __ldcg(&part[k]) : make_float2(kNegHuge, 0.0f);
            if (v[i].y != 0.0f) top = fmaxf(top, v[i].x);
        }
        segmax[seg][c] = top;
        __syncthreads();
        float m = cm[c];
        for (int g = 0; g < seg; ++g) m = fmaxf(m, segmax[g][c]);
        float e[kR];
        unsigned fresh = 0u;
#pragma unroll
        for (int i = 0; i < kR; ++i) {
            const bool nw = v[i].y != 0.0f && v[i].x > m;
            e[i] = nw ? ex2(m - v[i].x) : ex2(v[i].x - m);
            if (nw) {
                fresh |= 1u << i;
                m = v[i].x;
            }
        }
        for (int g = 0; g < kSeg; ++g) {
            if (seg == g) {
                float s = cs[c];
#pragma unroll
                for (int i = 0; i < kR; ++i)
                    if (v[i].y != 0.0f) s = (fresh >> i) & 1u ? fmaf(s, e[i], v[i].y) : fmaf(v[i].y, e[i], s);
                cs[c] = s;
                if (g == kSeg - 1) cm[c] = m;
            }
            __syncthreads();
        }
    }
    __syncthreads();
    if (threadIdx.x < TILE) {
        float m = cm[c], s = cs[c];
        warp_lse_reduce(m, s);
        if ((threadIdx.x & 31) == 0) {
            sm[threadIdx.x >> 5] = m;
            ss[threadIdx.x >> 5] = s;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        Lse2 L;
        L.m = kNegHuge;
        L.s = 0.0f;
        for (int k = 0; k < TILE / 32; ++k) L.merge(sm[k], ss[k]);
        m_out = L.m;
        s_out = L.s;
    }
}

// (m, s) merged with the partials [first, first + cnt) in order, by one warp:
// the exponentials in parallel, the sum's multiply-adds in order.
__device__ __forceinline__ void warp_merge_parts(const float2* part, int first, int cnt, float& m, float& s) {
    const int lane = threadIdx.x & 31;
    for (int k0 = 0; k0 < cnt; k0 += 32) {
        const float2 p = k0 + lane < cnt ? __ldcg(&part[first + k0 + lane]) : make_float2(kNegHuge, 0.0f);
        const bool live = p.y != 0.0f;
        float top = live ? p.x : kNegHuge;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float y = __shfl_up_sync(0xffffffffu, top, o);
            if (lane >= o) top = fmaxf(top, y);
        }
        float before = __shfl_up_sync(0xffffffffu, top, 1);
        before = lane == 0 ? m : fmaxf(m, before);
        const bool nw = live && p.x > before;
        const float e = nw ? ex2(before - p.x) : ex2(p.x - before);
        const unsigned lives = __ballot_sync(0xffffffffu, live), fresh = __ballot_sync(0xffffffffu, nw);
        for (int l = 0; l < min(32, cnt - k0); ++l) {
            const float el = __shfl_sync(0xffffffffu, e, l), yl = __shfl_sync(0xffffffffu, p.y, l);
            if ((lives >> l) & 1u) s = (fresh >> l) & 1u ? fmaf(s, el, yl) : fmaf(yl, el, s);
        }
        m = fmaxf(m, __shfl_sync(0xffffffffu, top, 31));
    }
}


template <int TILE, int THREADS = pass_threads(TILE)>
struct PassShared {
    WarpBuffer w[THREADS / 32];
    float sm[THREADS / 32], ss[THREADS / 32];
    float segmax[THREADS / TILE][TILE];
    float cm[TILE], cs[TILE];
    int last;
};

// A split pass (see sk_pass_kernel): for each slice kExactParts - 1 more warps,
// that read their parts of the block when its sums underflowed.
constexpr int kExactParts = 4;
template <int THREADS>
struct ExactShared {
    WarpStage stage[kExactParts - 1][THREADS / 32];
    float4 lse[kExactParts - 1][THREADS];
    unsigned low[THREADS / 32];
};
template <int TILE, int OTHER>
constexpr __host__ __device__ size_t pass_smem_bytes() {
    constexpr int thr = pass_threads(TILE, OTHER);
    constexpr size_t own = sizeof(PassShared<TILE, thr>), other = sizeof(PassShared<OTHER, thr>);
    return ((own > other ? own : other) + 127) / 128 * 128;
}
// The warps of a slice.
__device__ __forceinline__ void slice_barrier(int warp) {
    asm volatile("bar.sync %0, %1;" ::"r"(5 + warp), "n"(32 * kExactParts) : "memory");
}

// Dustbin potentials from the partials of a pass: rows (of iteration it): F_0
// of the iteration and G_0 from it and the new F; columns: the next F_0 from
// the new G and the current G_0.  Block `block` of `blocks`; also clears the
// maxima set `clear` and counts the pass's pairs.
template <int TILE, int THREADS, bool ROWS>
__device__ void finish_pass(const SkArgs& a, PassShared<TILE, THREADS>& H, int block, int blocks, unsigned* clear) {
    const DustPtrs D = dust_ptrs(a.dust, a.T);
    const int lane = threadIdx.x & 31;
    const float2* part = ROWS ? a.row_part : a.col_part;
    if (a.mode == 1) {
        constexpr int warps = THREADS / 32;
        for (int u = block * warps + (threadIdx.x >> 5); u < a.T; u += blocks * warps) {
            const int4 at = a.ang_tiles[u];
            const float v0 = __ldcg((ROWS ? D.F0n : D.G0) + u);
            float m = v0 - a.kc, s = 1.0f;
            warp_merge_parts(part, ROWS ? at.x : at.z, ROWS ? at.y : at.w, m, s);
            if (lane == 0) {
                const float v = (ROWS ? D.log2O : D.log2U)[u] - (m + lg2(s));
                if (ROWS) {
                    D.F0[u] = v0;
                    D.G0[u] = v;
                } else {
                    D.F0n[u] = v;
                }
            }
        }
    } else if (a.mode == 0 && block == 0) {
        float m, s;
        const float v0 = threadIdx.x == 0 ? __ldcg(ROWS ? D.F0n : D.G0) : 0.0f;
        merge_parts<TILE, THREADS>(part, __ldcg(a.ctrl + (ROWS ? CTRL_N_ROW_TILES : CTRL_N_COL_TILES)), m, s, H.sm, H.ss,
                          H.segmax, H.cm, H.cs);
        if (threadIdx.x == 0) {
            Lse2 L;
            L.init(v0 - a.kc);
            L.merge(m, s);
            const float v = (ROWS ? D.log2O[0] : D.log2U[0]) - L.value();
            if (ROWS) {
                D.F0[0] = v0;
                D.G0[0] = v;
            } else {
                D.F0n[0] = v;
            }
        }
    }
    if (block == 0) {
        if (clear)
            for (int u = threadIdx.x; u < a.T; u += THREADS) clear[u] = 0u;
        if (threadIdx.x == 0)
            *(unsigned long long*)(a.ctrl + CTRL_SK_PAIRS) +=
                __ldcg((const unsigned long long*)(a.ctrl + (ROWS ? CTRL_ROW_EVAL : CTRL_COL_EVAL)));
    }
}

// Blocks that finish the pass before: a warp per angle for per-angle dustbins.
__host__ __device__ inline int finish_blocks(int mode, int T, int threads) {
    return mode == 1 ? (T + threads / 32 - 1) / (threads / 32) : 1;
}

// The last column pass.
template <int TILE>
__global__ void __launch_bounds__(pass_threads(TILE)) sk_finish_pass_kernel(SkArgs a) {
    extern __shared__ __align__(128) char pass_smem[];
    finish_pass<TILE, pass_threads(TILE), false>(a, *(PassShared<TILE>*)pass_smem, blockIdx.x, gridDim.x, nullptr);
}

// Programmatic dependent launch: a pass starts while the one before it ends.
// What it reads before pass_wait is what the list kernels and the scheduler
// left, and those were complete before the pass before it (which waited for
// its own predecessor before it let this one start) went on.
__device__ __forceinline__ void pass_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pass_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// --------------------------------------------------- row and column passes
// Iteration `it` of the row (ROWS) or column update.  What bounds it: at the
// 1000-grain density the lists (324 MB a pass, 48 us at the copy rate, 63 us
// measured), below that the chain of a pass: launch, gathers of the potentials,
// partial sums (100 grains: 53 / 43 us a pass when it evaluated pairs, 4.1 us
// now; 5 grains: 11 and 3.0 us).  The other side's tile width, for the partials
// that the first blocks merge, is OTHER.
//
// Without dustbins (unbalanced OT) a shifted sum underflows for most spots:
// the potentials of spots far from any partner are the largest, and shift all
// the others.  Their slices read the whole block with a running maximum, a
// serial chain, so a pass over few slices has PARTS warps to a slice that read a
// part of the block each; part 0's warp merges.  23 grains x 17 angles at 4 mm^2:
// 17 us a pass with one warp, 13 us with four.
//
// Registers: 128 a thread, 512 threads to an SM.  No more are resident anyway:
// a named barrier whose id is not a constant takes all 16 of a CTA, four CTAs to
// an SM.  With 64 registers the sums over swept pairs spilled: 90 angles of
// 13300 x 7744 spots at 100 mm^2 without lists 5.8 ms an iteration, now 4.6; one
// block of 200000 x 8000 spots 11.1 ms, now 6.3; split, 23 grains x 60 angles at 4
// and 100 mm^2, 50 iterations, 1.24 and 2.32 ms, now 1.14 and 1.82.
constexpr int kPassThreadsPerSm = 512;
template <int TILE, int OTHER, bool ROWS, int PARTS>
__global__ void __launch_bounds__(PARTS* pass_threads(TILE, OTHER),
                                  kPassThreadsPerSm / pass_threads(TILE, OTHER) / PARTS > 0
                                      ? kPassThreadsPerSm / pass_threads(TILE, OTHER) / PARTS
                                      : 1)
    sk_pass_kernel(SkArgs a, int it, int finishers) {
    extern __shared__ __align__(128) char pass_smem[];
    constexpr int kThreads = pass_threads(TILE, OTHER);
    PassShared<TILE, kThreads>& H = *(PassShared<TILE, kThreads>*)pass_smem;
    ExactShared<kThreads>& X = *(ExactShared<kThreads>*)(pass_smem + pass_smem_bytes<TILE, OTHER>());
    const int part = PARTS > 1 ? threadIdx.x / kThreads : 0, own = threadIdx.x - part * kThreads;
    const int warp = own >> 5;
    if (ROWS && it == 0) pass_wait();  // the first pass follows the kernels that write the lists
    if ((int)blockIdx.x < finishers) {
        if (PARTS > 1 && part > 0) return;
        if (!(ROWS && it == 0)) pass_wait();
        pass_release();
        unsigned* clear = ROWS ? col_max(a, it) : row_max(a, it + 1);
        if (!ROWS || it > 0)
            finish_pass<OTHER, kThreads, !ROWS>(a, *(PassShared<OTHER, kThreads>*)pass_smem, blockIdx.x, finishers, clear);
        return;
    }
    const SliceDesc* desc = (const SliceDesc*)(ROWS ? a.row_desc : a.col_desc);
    const int* tab = ROWS ? a.row_tab : a.col_tab;
    constexpr int kW = TILE / 32;
    // (starting the tiles by descending length measured no faster: 11.9 against 12.0 ms at 317 grains and 21 mm^2,
    // 31.4 against 30.0 ms at 1000 grains, where neighbouring tiles' gathers share L1 and L2)
    const int tile = (blockIdx.x - finishers) * (kThreads / TILE) + own / TILE;
    if (tile >= __ldcg(a.ctrl + (ROWS ? CTRL_N_ROW_TILES : CTRL_N_COL_TILES))) return;
    const int id = tile * kW + warp % kW;
    int numbers = 0;
    if (part == 0) numbers = chunk_numbers(a, tab, id, threadIdx.x & 31, 0);
    const Slice sl = load_slice(desc, id);
    if (PARTS > 1 && part > 0) {
        if (!(ROWS && it == 0)) pass_wait();
        pass_release();
        if (!sl.any) return;
        slice_barrier(warp);
        if (!X.low[warp]) return;
        X.lse[part - 1][own] = exact_part<ROWS, PARTS>(a, X.stage[part - 1][warp], sl, kNegHuge, part);
        slice_barrier(warp);
        return;
    }
    WarpBuffer& M = H.w[warp];
    ring_start(a, M.ring, sl, numbers);
    const int t = sl.t, lane = sl.lane;
    float2 K = make_float2(a.negKD2, a.negKD2);  // -K of the lane's own spots (columns)
    if (!ROWS && sl.valid) K = *((const float2*)&a.modW[sl.q] + 1);
    if (!sl.vb) K.y = -1.0f;
    const DustPtrs D = dust_ptrs(a.dust, a.T);
    const float* pot = ROWS ? a.Gc : a.Fc;
    float* out = ROWS ? a.Fc : a.Gc;
    if (!(ROWS && it == 0)) pass_wait();
    pass_release();
    const bool ub = a.mode == 2;  // unbalanced OT: no dustbins, scaled update
    const int d = a.mode ? t : 0;
    float pm = kNegHuge, ps = 0.0f;
    if (sl.any) {
        // the dustbin's term: the outlier column (rows), the unmatched-model row with C_0j = 0 (columns)
        const float dust = ub ? kNegHuge : ROWS ? __ldcg(D.G0 + d) - a.kc : __ldcg(D.F0n + d);
        const float top = ROWS ? (it > 0 ? angle_max(col_max(a, it - 1), t, 0.0f) : D.Gmax[t])
                               : angle_max(row_max(a, it), t, a.kc);
        const float shift = ub ? top : fmaxf(top, dust);
        const float e0 = ub ? 0.0f : ex2(dust - shift);
        ListSum S{e0, 0.0f, e0, 0.0f};
        if (sl.nch < 0)
            swept_sum<ROWS>(a, M.stage, sl, shift, S);
        else if (!ROWS || a.uniK)
            list_sum<false>(a, M.ring, tab, sl, numbers, pot + 2 * sl.s0, shift, K.x, ROWS ? a.negKD2 : K.y, nullptr, S);
        else
            list_sum<ROWS>(a, M.ring, tab, sl, numbers, pot + 2 * sl.s0, shift, 0.0f, 0.0f, a.modW + sl.s0, S);
        const float sa = S.ea + S.oa, sb = S.eb + S.ob;
        float va = -(shift + lg2(sa)), vv = sl.vb ? -(shift + lg2(sb)) : 0.0f;
        const unsigned low_a = __ballot_sync(0xffffffffu, sl.valid && !(sa > kTinySum));
        const unsigned low_b = __ballot_sync(0xffffffffu, sl.vb && !(sb > kTinySum));
        if (PARTS > 1) {
            if (lane == 0) X.low[warp] = low_a | low_b;
            slice_barrier(warp);
        }
        if (low_a | low_b) {
            float xa, xb;
            if (PARTS == 1) {
                exact_lse<ROWS>(a, M.stage, sl, dust, xa, xb);
            } else {
                float4 x = exact_part<ROWS, PARTS>(a, M.stage, sl, dust, 0);
                slice_barrier(warp);
                for (int p = 0; p < PARTS - 1; ++p) {
                    const float4 y = X.lse[p][own];
                    lse_merge_into(x.x, x.y, y.x, y.y);
                    lse_merge_into(x.z, x.w, y.z, y.w);
                }
                xa = x.x + lg2(x.y);
                xb = x.z + lg2(x.w);
            }
            if ((low_a >> lane) & 1u) va = -xa;
            if ((low_b >> lane) & 1u) vv = -xb;
            if (lane == 0)
                atomicAdd((unsigned*)a.ctrl + (ROWS ? CTRL_EXACT_ROWS : CTRL_EXACT_COLS),
                          (unsigned)(__popc(low_a) + __popc(low_b)));
        }
        if (sl.valid) {
            if (ub) {  // Algorithm UnbalancedOT: the balanced update raised to kappa / (kappa + eps)
                const float tau = ROWS ? a.tau_row : a.tau_col;
                va = sl.ns > 0 ? tau * va : 0.0f;
                vv = sl.ns > 0 ? tau * vv : 0.0f;
            }
            *(float2*)&out[2 * (size_t)sl.q] = make_float2(va, sl.vb ? vv : kNegHuge);
            // tile partial of LSE2(F_i - kc) for the outlier column, of LSE2(G_j) for the unmatched row
            const float off = ROWS ? a.kc : 0.0f;
            pm = va - off;
            ps = 1.0f;
            if (sl.vb) lse_merge_into(pm, ps, vv - off, 1.0f);
        }
    }
    // the tile's first slice is never empty: its angle is the tile's
    store_part<TILE>(pm, ps, tile, t, ROWS ? a.row_part : a.col_part, ROWS ? row_max(a, it) : col_max(a, it), H.sm, H.ss);
}

// ------------------------------------------------------------- read-out
// Largest of the CTA's non-negative values into *out.
__device__ __forceinline__ void block_err(float v, float* red, int* out) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < (int)(blockDim.x >> 5); ++k) v = fmaxf(v, red[k]);
        atomicMax(out, __float_as_int(v));
    }
}

// Plan read-out per observed spot with the final potentials: argmax over the
// block's model spots and the outlier column (ties to the lowest index, the
// outlier column only when strictly larger), top1 - top2 margin in plan
// units, and the row-marginal error.  Once per E-step.
//
// Listed slices read their lists, swept ones the sub-granules that their
// cones see.  A pair left out has an exponent of at most the largest
// potential less kListLog2; a row whose best entry (the outlier column
// included) does not stand kFarLog2 above that is read again over its whole
// block, the lanes of the warp sharing its pairs, so the ranking and the sums
// are those of every pair.
struct Top2 {
    float m, s, b1, b2;
    int arg;
    __device__ __forceinline__ void init() {
        m = kNegHuge;
        s = 0.0f;
        b1 = kNegHuge;
        b2 = kNegHuge;
        arg = -1;
    }
    // j: the spot's slot in the spatial order; perm maps slots to the caller's
    // indices, and ties go to the lowest caller index
    __device__ __forceinline__ void add(float v, int j, const int* perm) {
        if (v > m) {
            s = s * ex2(m - v) + 1.0f;
            m = v;
        } else {
            s += ex2(v - m);
        }
        if (v > b1 || (v == b1 && v > kNegHuge && perm[j] < perm[arg])) {
            b2 = b1;
            b1 = v;
            arg = j;
        } else if (v > b2) {
            b2 = v;
        }
    }
    // the same of two disjoint sets of entries
    __device__ __forceinline__ void merge(const Top2& o, const int* perm) {
        const float top = fmaxf(m, o.m);
        s = (s == 0.0f ? 0.0f : s * ex2(m - top)) + (o.s == 0.0f ? 0.0f : o.s * ex2(o.m - top));
        m = top;
        b2 = fmaxf(fminf(b1, o.b1), fmaxf(b2, o.b2));
        if (o.b1 > b1 || (o.b1 == b1 && o.b1 > kNegHuge && perm[o.arg] < perm[arg])) {
            b1 = o.b1;
            arg = o.arg;
        }
    }
};

// Top2 of one observed spot over its whole block, by the warp together.
__device__ __noinline__ Top2 whole_row(const SkArgs& a, int t, float px, float py, float pz) {
    const int lane = threadIdx.x & 31, j0 = a.J2_off[t], nj = a.J2_off[t + 1] - j0, jbase = a.J_off[t];
    const f2 x = dup(px), y = dup(py), z = dup(pz);
    Top2 P;
    P.init();
    for (int k = lane; k < nj; k += 32) {
        const ulonglong2 X = *(const ulonglong2*)&a.modX[j0 + k], Z = *(const ulonglong2*)&a.modZ[j0 + k],
                         W = *(const ulonglong2*)&a.modW[j0 + k];
        const f2 v = pair_v2(x, y, z, X.x, X.y, *(const f2*)&a.modY[j0 + k], Z.x, Z.y, W.x, W.y,
                             *(const f2*)&a.Gc[2 * (size_t)(j0 + k)]);
        P.add(lo(v), jbase + 2 * k, a.mod_perm);
        P.add(hi(v), jbase + 2 * k + 1, a.mod_perm);  // padding slots have -3e38 and never win
    }
    for (int o = 16; o > 0; o >>= 1) {
        Top2 Q;
        Q.m = __shfl_xor_sync(0xffffffffu, P.m, o);
        Q.s = __shfl_xor_sync(0xffffffffu, P.s, o);
        Q.b1 = __shfl_xor_sync(0xffffffffu, P.b1, o);
        Q.b2 = __shfl_xor_sync(0xffffffffu, P.b2, o);
        Q.arg = __shfl_xor_sync(0xffffffffu, P.arg, o);
        P.merge(Q, a.mod_perm);
    }
    return P;
}

// Log-sum-exp of one model spot's column over its whole block, by the warp together.
__device__ __noinline__ Lse2 whole_col(const SkArgs& a, int t, int q, int odd) {
    const int lane = threadIdx.x & 31, i0 = a.I2_off[t], ni = a.I2_off[t + 1] - i0;
    ColPair C;
    load_col_pair(a, q, C);
    Lse2 L;
    L.m = kNegHuge;
    L.s = 0.0f;
    for (int k = lane; k < ni; k += 32) {
        const ulonglong2 X = *(const ulonglong2*)&a.obsX[i0 + k];
        const f2 pz = *(const f2*)&a.obsY[i0 + k], F = *(const f2*)&a.Fc[2 * (size_t)(i0 + k)];
        const f2 v = odd ? pair_v2(X.x, X.y, pz, C.ncxb, C.ncyb, C.nczb, C.nrxb, C.nryb, C.nrzb, C.kb, F)
                         : pair_v2(X.x, X.y, pz, C.ncxa, C.ncya, C.ncza, C.nrxa, C.nrya, C.nrza, C.ka, F);
        L.merge(lo(v), 1.0f);
        L.merge(hi(v), 1.0f);
    }
    warp_lse_reduce(L.m, L.s);
    return L;
}

// Padding entries of a list (their cost is 3e38; a spot that is not a number stays an entry).
__device__ __forceinline__ bool is_entry(float e2) { return !(e2 > 2.0e38f); }

template <int TILE>
__global__ void __launch_bounds__(pass_threads(TILE), kPassThreadsPerSm / pass_threads(TILE))
    sk_harvest_row_kernel(SkArgs a, int n_iter) {
    extern __shared__ __align__(128) char pass_smem[];
    PassShared<TILE>& H = *(PassShared<TILE>*)pass_smem;
    DustPtrs D = dust_ptrs(a.dust, a.T);
    const SliceDesc* desc = (const SliceDesc*)a.row_desc;
    const int at = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    Slice sl{};
    if (at < slice_count<TILE>(a, true)) sl = load_slice(desc, at);
    const int t = sl.t, lane = sl.lane;
    float my_err = 0.0f;
    if (sl.any) {
        WarpBuffer& M = H.w[threadIdx.x >> 5];
        const int lrow = 2 * (sl.q - a.I2_off[t]);
        const bool vb = sl.vb;
        const int jbase = a.J_off[t], j0 = a.J2_off[t];
        const float dustv = a.mode == 2 ? kNegHuge : D.G0[a.mode ? t : 0] - a.kc;
        Top2 A, B;
        A.init();
        B.init();
        const RowPair R = load_row_pair(a, sl.q, sl.valid);
        auto sweep_all = [&](int skip) {
            for_each_swept<true>(a, M.stage, sl, skip, 0.0f, [&](int st, int j, int k) {
                f2 va, vv;
                row_pair_v(R, M.stage, st, j, *(const f2*)&M.stage.P[st][j], va, vv);
                const int at = jbase + 2 * k;
                if (!sl.valid) return;
                A.add(lo(va), at, a.mod_perm);
                A.add(hi(va), at + 1, a.mod_perm);  // padding slots have -3e38 and never win
                B.add(lo(vv), at, a.mod_perm);
                B.add(hi(vv), at + 1, a.mod_perm);
            });
        };
        if (sl.nch >= 0) {
            const float* pot = a.Gc + 2 * j0;
            const int numbers = chunk_numbers(a, a.row_tab, sl.id, lane, 0);
            ring_start(a, M.ring, sl, numbers);
            for_each_chunk(a, M.ring, a.row_tab, sl, numbers, [&](const Chunk& E) {
                for (int k = 0; k < kListDepth; ++k) {
                    const int ja = E.slot[k][lane] & 0xffffu, jb = E.slot[k][lane] >> 16;
                    const float2 e2 = E.e2[k][lane];
                    float ka = a.negKD2, kb = a.negKD2;
                    if (!a.uniK) {
                        ka = ((const float*)&a.modW[j0 + (ja >> 1)])[2 + (ja & 1)];
                        kb = ((const float*)&a.modW[j0 + (jb >> 1)])[2 + (jb & 1)];
                    }
                    if (is_entry(e2.x)) A.add(fmaf(e2.x, ka, pot[ja]), jbase + ja, a.mod_perm);
                    if (is_entry(e2.y)) B.add(fmaf(e2.y, kb, pot[jb]), jbase + jb, a.mod_perm);
                }
            });
        } else {
            sweep_all(a.skip);
        }
        const float far = final_col_max(a, D, t, n_iter) - kListLog2 + kFarLog2;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            unsigned low = __ballot_sync(0xffffffffu, e ? vb && !(fmaxf(B.b1, dustv) >= far)
                                                        : sl.valid && !(fmaxf(A.b1, dustv) >= far));
            for (; low; low &= low - 1) {
                const int l = __ffs(low) - 1;
                const Top2 P = whole_row(a, t, __shfl_sync(0xffffffffu, e ? lo(R.pxb) : lo(R.pxa), l),
                                         __shfl_sync(0xffffffffu, e ? lo(R.pyb) : lo(R.pya), l),
                                         __shfl_sync(0xffffffffu, e ? lo(R.pzb) : lo(R.pza), l));
                if (lane == l) (e ? B : A) = P;
            }
        }
        if (sl.valid) {
            int i = a.I_off[t] + lrow;
            const float2 Fp = *(const float2*)&a.Fc[2 * (size_t)sl.q];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                if (e == 1 && !vb) break;
                Top2& P = e ? B : A;
                float F = e ? Fp.y : Fp.x;
                if (dustv > P.b1) {  // outlier column last, only when strictly larger
                    P.b2 = P.b1;
                    P.b1 = dustv;
                    P.arg = -1;
                } else if (dustv > P.b2) {
                    P.b2 = dustv;
                }
                Lse2 L;
                L.m = P.m;
                L.s = P.s;
                L.merge(dustv, 1.0f);
                float rs = ex2(F + L.value());
                my_err = fmaxf(my_err, fabsf(rs - 1.0f));
                // unbalanced plan: a spot that keeps most of its mass is an outlier
                if (a.mode == 2 && !(rs >= 0.5f)) P.arg = -1;
                int ic = a.obs_perm[i + e];  // the caller's index of this observed spot
                if (a.assign) a.assign[ic] = P.arg >= 0 ? a.mod_perm[P.arg] : -1;
                if (a.margin) a.margin[ic] = ex2(F + P.b1) - (P.b2 > kNegHuge ? ex2(F + P.b2) : 0.0f);
            }
        }
    }
    block_err(my_err, H.sm, (int*)(D.err + 2));
    if (!last_block(a.ctrl + CTRL_HRV_DONE, &H.last)) return;
    if (threadIdx.x == 0) {
        float err = __int_as_float(__ldcg((const int*)(D.err + 2)));
        int nd = a.mode == 2 ? 0 : (a.mode ? a.T : 1);
        for (int d = 0; d < nd; ++d) {
            if (D.log2U[d] > kNegHuge) err = fmaxf(err, fabsf(ex2(D.F0[d] - D.F0n[d]) - 1.0f));
        }
        D.err[0] = err;
        a.ctrl[CTRL_HRV_DONE] = 0;
    }
}

// Column mass q_j = sum_i Q_ij over observed rows and the column-marginal
// error with the final potentials, in base 2 with a running maximum.  Pairs
// are left out, and columns read again, as for the rows.
template <int TILE>
__global__ void __launch_bounds__(pass_threads(TILE), kPassThreadsPerSm / pass_threads(TILE))
    sk_harvest_col_kernel(SkArgs a, int n_iter) {
    extern __shared__ __align__(128) char pass_smem[];
    PassShared<TILE>& H = *(PassShared<TILE>*)pass_smem;
    DustPtrs D = dust_ptrs(a.dust, a.T);
    const SliceDesc* desc = (const SliceDesc*)a.col_desc;
    const int at = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    Slice sl{};
    if (at < slice_count<TILE>(a, false)) sl = load_slice(desc, at);
    const int t = sl.t, lane = sl.lane;
    float my_err = 0.0f;
    if (sl.any) {
        WarpBuffer& M = H.w[threadIdx.x >> 5];
        const int lcol = 2 * (sl.q - a.J2_off[t]);
        const bool vb = sl.vb;
        const int i0 = a.I2_off[t];
        const float F0 = a.mode == 2 ? kNegHuge : D.F0[a.mode ? t : 0];
        Lse2 A, B;
        A.m = B.m = kNegHuge;
        A.s = B.s = 0.0f;
        auto add = [](Lse2& L, float v) {
            if (v > L.m) {
                L.s = L.s * ex2(L.m - v) + 1.0f;
                L.m = v;
            } else {
                L.s += ex2(v - L.m);
            }
        };
        ColPair C;
        load_col_pair(a, sl.valid ? sl.q : sl.q - lane, C);
        auto sweep_all = [&](int skip) {
            for_each_swept<false>(a, M.stage, sl, skip, 0.0f, [&](int st, int j, int) {
                f2 va, vv;
                col_pair_v(C, M.stage, st, j, *(const f2*)&M.stage.P[st][j], va, vv);
                add(A, lo(va));
                add(A, hi(va));
                add(B, lo(vv));
                add(B, hi(vv));
            });
        };
        if (sl.nch >= 0) {
            const float* pot = a.Fc + 2 * i0;
            const float ka = lo(C.ka), kb = lo(C.kb);
            const int numbers = chunk_numbers(a, a.col_tab, sl.id, lane, 0);
            ring_start(a, M.ring, sl, numbers);
            for_each_chunk(a, M.ring, a.col_tab, sl, numbers, [&](const Chunk& E) {
                for (int k = 0; k < kListDepth; ++k) {
                    const unsigned s = E.slot[k][lane];
                    const float2 e2 = E.e2[k][lane];
                    if (is_entry(e2.x)) add(A, fmaf(e2.x, ka, pot[s & 0xffffu]));
                    if (is_entry(e2.y)) add(B, fmaf(e2.y, kb, pot[s >> 16]));
                }
            });
        } else {
            sweep_all(a.skip);
        }
        const float far = final_row_max(a, D, t, n_iter) - kListLog2 + kFarLog2;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            unsigned low = __ballot_sync(0xffffffffu, e ? vb && !(B.m >= far) : sl.valid && !(A.m >= far));
            for (; low; low &= low - 1) {
                const int l = __ffs(low) - 1;
                const Lse2 P = whole_col(a, t, sl.q - lane + l, e);
                if (lane == l) (e ? B : A) = P;
            }
        }
        if (sl.valid) {
            const float2 Gp = *(const float2*)&a.Gc[2 * (size_t)sl.q];
            for (int e = 0; e < 2; ++e) {
                if (e == 1 && !vb) break;
                const Lse2& L = e ? B : A;
                const float G = e ? Gp.y : Gp.x;
                const float qj = L.s > 0.0f ? ex2(G + L.m + lg2(L.s)) : 0.0f;
                if (a.q) a.q[a.mod_perm[a.J_off[t] + lcol + e]] = qj;
                my_err = fmaxf(my_err, fabsf(qj + ex2(G + F0) - 1.0f));
            }
        }
    }
    block_err(my_err, H.sm, (int*)(D.err + 3));
    if (!last_block(a.ctrl + CTRL_HCOL_DONE, &H.last)) return;
    if (threadIdx.x == 0) {
        D.err[1] = __int_as_float(__ldcg((const int*)(D.err + 3)));
        a.ctrl[CTRL_HCOL_DONE] = 0;
    }
}

// ------------------------------------------------------------ launches
// Launch shapes of the pair passes the autotuner chooses from: the pairs of a
// tile.  (Shapes 1 and 2 are the same kernels.)
int sk_variant_threads(int v) { return v == 0 ? 256 : (v == 3 ? 64 : 128); }

// Entries that a spot can expect for costs of `most` in units of 1 / K (two
// detectors see about 2 sr).
static float expected_entries(const SkArgs& a, float most, int n_streamed) {
    return (float)n_streamed / (float)a.T * 3.14159f * (most / a.skipK) / 2.0f;
}

// Largest entries per spot, as a share of the slice's swept pairs, that are
// worth listing for n_iter iterations: where the cost of listing (see above) is
// made up by passes over lists (0.03 to 0.5 of a swept one).  From 40 iterations
// on every list is that fits, and where the entries are few the slices need not
// look (kListAlways).
float list_share_of(const SkArgs& a, int n_iter) {
    const float share = (n_iter - 1.0f) / (15.0f + 0.6f * n_iter);
    if (share < 1.0f) return share;
    return expected_entries(a, kListLog2, std::max(a.n_obs, a.n_model)) <= 128.0f ? kListAlways : 1.0f;
}

// The same for n_pass passes of an M-step (entries of at least 2^-40 at the usual
// potentials).  A single pass is listed for, whole, or swept, whole: listed slices
// beside swept ones only add up.  The line lies at 20 entries of a spot.
// Gradients, listed against swept: 1 mm^2, 1020 observed spots an angle (1 entry)
// 0.171 and 0.183 ms, 13300 (16) 1.84 and 1.96; 21 mm^2, 1020 (26) 0.224 and 0.198,
// 3700 (95) 0.75 and 0.57; 100 mm^2, 13300: 19.2 and 3.8.
float plan_share_of(const SkArgs& a, int n_pass) {
    const float entries = expected_entries(a, 4.0f - kQSkip, a.n_obs);
    if (entries <= (n_pass > 1 ? 128.0f : 20.0f)) return kListAlways;
    return n_pass > 1 ? n_pass / (n_pass + 4.0f) : 0.0f;
}

namespace {

// Calls fn(tile width as an integral constant) for shape v.
template <class Fn>
cudaError_t with_tile(int v, Fn fn) {
    if (v == 0) return fn(std::integral_constant<int, 256>{});
    if (v == 3) return fn(std::integral_constant<int, 64>{});
    return fn(std::integral_constant<int, 128>{});
}

// Both tile widths as integral constants.
template <class Fn>
cudaError_t with_tiles(const SkLaunch& l, Fn fn) {
    return with_tile(l.row_variant, [&](auto row) { return with_tile(l.col_variant, [&](auto col) { return fn(row, col); }); });
}

// Once per device (the current one), before the first launch.
template <int A, int B>
cudaError_t allow_smem() {
    constexpr int thr = pass_threads(A, B);
    const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const int n1 = (int)pass_smem_bytes<A, B>(), n4 = n1 + (int)sizeof(ExactShared<thr>);
    cudaError_t e = cudaFuncSetAttribute(sk_pass_kernel<A, B, true, 1>, at, n1);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(sk_pass_kernel<A, B, false, 1>, at, n1);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(sk_pass_kernel<A, B, true, kExactParts>, at, n4);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(sk_pass_kernel<A, B, false, kExactParts>, at, n4);
    if (A != B || e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(sk_harvest_row_kernel<A>, at, n1);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(sk_harvest_col_kernel<A>, at, n1);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(sk_finish_pass_kernel<A>, at, n1);
    return e;
}

template <class... Params, class... Args>
cudaError_t launch_pass(void (*k)(Params...), int ctas, int threads, size_t smem, bool overlap, cudaStream_t s,
                        Args... args) {
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(ctas);
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&c, k, args...);
}

// CTAs that hold a side's slices.
int slice_ctas(int T, int n_spots, int tile, int threads) {
    const int per = threads / 32;
    return ((int)list_slices(T, n_spots, tile) + per - 1) / per;
}

template <int TILE, int OTHER, bool ROWS>
cudaError_t run_pass(const SkArgs& a, int it, bool split, cudaStream_t s) {
    constexpr int thr = pass_threads(TILE, OTHER);
    constexpr size_t smem = pass_smem_bytes<TILE, OTHER>();
    const int fin = finish_blocks(a.mode, a.T, thr);
    const int ctas = fin + slice_ctas(a.T, ROWS ? a.n_obs : a.n_model, TILE, thr);
    if (split)
        return launch_pass(sk_pass_kernel<TILE, OTHER, ROWS, kExactParts>, ctas, kExactParts * thr,
                           smem + sizeof(ExactShared<thr>), true, s, a, it, fin);
    return launch_pass(sk_pass_kernel<TILE, OTHER, ROWS, 1>, ctas, thr, smem, true, s, a, it, fin);
}

}  // namespace

cudaError_t sinkhorn_setup() {
    cudaError_t e = cudaSuccess;
    for (int r = 0; r < kSkVariants && e == cudaSuccess; ++r)
        for (int c = 0; c < kSkVariants && e == cudaSuccess; ++c)
            e = with_tile(r, [&](auto row) {
                return with_tile(c, [&](auto col) { return allow_smem<decltype(row)::value, decltype(col)::value>(); });
            });
    return e;
}

cudaError_t sinkhorn_row_pass(const SkArgs& a, const SkLaunch& l, int it, cudaStream_t s) {
    return with_tiles(l, [&](auto row, auto col) {
        return run_pass<decltype(row)::value, decltype(col)::value, true>(a, it, l.split, s);
    });
}

cudaError_t sinkhorn_col_pass(const SkArgs& a, const SkLaunch& l, int it, cudaStream_t s) {
    return with_tiles(l, [&](auto row, auto col) {
        return run_pass<decltype(col)::value, decltype(row)::value, false>(a, it, l.split, s);
    });
}

cudaError_t sinkhorn_iterate(const SkArgs& a, const SkLaunch& l, int n_iter, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    for (int it = 0; it < n_iter && e == cudaSuccess; ++it) {
        e = sinkhorn_row_pass(a, l, it, s);
        if (e == cudaSuccess) e = sinkhorn_col_pass(a, l, it, s);
    }
    if (e != cudaSuccess || n_iter == 0) return e;
    return with_tile(l.col_variant, [&](auto tile) {
        constexpr int t = decltype(tile)::value;
        sk_finish_pass_kernel<t><<<finish_blocks(a.mode, a.T, pass_threads(t)), pass_threads(t), sizeof(PassShared<t>), s>>>(
            a);
        return cudaGetLastError();
    });
}

cudaError_t sinkhorn_build_lists(const SkArgs& a, const SkLaunch& l, cudaStream_t s) {
    const int rg = (l.row_slices + kListWarps - 1) / kListWarps, cg = (l.col_slices + kListWarps - 1) / kListWarps;
    return with_tiles(l, [&](auto row, auto col) {
        constexpr int rt = decltype(row)::value, ct = decltype(col)::value;
        sk_list_kernel<rt, true, false><<<rg, 32 * kListWarps, 0, s>>>(a);
        sk_list_kernel<ct, false, false><<<cg, 32 * kListWarps, 0, s>>>(a);
        return cudaGetLastError();
    });
}

// The M-step's columns: slices, and the plan entries of those that are listed.
cudaError_t sinkhorn_list_plan(const SkArgs& a, const SkLaunch& l, cudaStream_t s) {
    return with_tile(l.col_variant, [&](auto tile) {
        sk_list_kernel<decltype(tile)::value, false, true>
            <<<(l.col_slices + kListWarps - 1) / kListWarps, 32 * kListWarps, 0, s>>>(a);
        return cudaGetLastError();
    });
}

cudaError_t sinkhorn_harvest(const SkArgs& a, const SkLaunch& l, int n_iter, bool want_rows, bool want_cols,
                             cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    if (want_rows)
        e = with_tile(l.row_variant, [&](auto tile) {
            constexpr int t = decltype(tile)::value;
            return launch_pass(sk_harvest_row_kernel<t>, slice_ctas(a.T, a.n_obs, t, pass_threads(t)), pass_threads(t),
                               sizeof(PassShared<t>), false, s, a, n_iter);
        });
    if (e == cudaSuccess && want_cols)
        e = with_tile(l.col_variant, [&](auto tile) {
            constexpr int t = decltype(tile)::value;
            return launch_pass(sk_harvest_col_kernel<t>, slice_ctas(a.T, a.n_model, t, pass_threads(t)), pass_threads(t),
                               sizeof(PassShared<t>), false, s, a, n_iter);
        });
    return e;
}

}  // namespace laue
