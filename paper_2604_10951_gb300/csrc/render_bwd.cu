// Backward render for sm_103a: vector-Jacobian product of the forward
// render (Eq. 2, Eq. 7) with the Top-K set, skips, stops and clamps held
// fixed.  The paper trains through the differentiable renderer end to end
// (Sec. 3.1, Sec. 3.5) but prints no gradients; these are the chain
// rule of the forward:
//   s_j    = rgb_j . dL/dRGB + [j in K-set] c_j . dL/dF
//   dL/da_j = T_j (s_j - S_j),  S_j = sum_{i>j} w_i s_i / T_{j+1} + bg.dL/dRGB + dL/dT
//   S_{j-1} = a_j s_j + (1 - a_j) S_j,  T_j = T_{j+1} / (1 - a_j)
// replayed back to front from the saved traversal length and final T.
//
// k_bwd_feat  (Top-K, except where k_bwd_geo_topk does it) one CTA per tile: for every selected (pixel, k) the
//             dot c_i . dL/dF(x) and the feature gradient sum w_i dL/dF(x),
//             grouped by surfel in shared memory first, so each surfel's
//             feature row is read once and costs one row of 16-byte vector
//             reductions per tile.
// k_bwd_geo_topk one warp per 8 x 4 pixel block: back-to-front replay; per
//             surfel the warp reduce-scatters its 13 partial derivatives
//             (adjugate rows 9, opacity 1, colour 3) and adds them to the
//             surfel's gradient row.
// k_bwd_geo_full (K = 0, and Top-K with many channels x K) the same, with c_j . dL/dF
//             and the feature gradients as products shared by the warp's lanes.
// k_bwd_project one thread per surfel: adjugate-row gradients -> homography
//             columns -> means, scales, quaternions; sums the views.
// k_feat_out  writes every row of the feature gradient (zeros for surfels
//             culled in every view).
#include "color.cuh"
#include "fss_internal.cuh"
#include "kernels.cuh"
#include "render_common.cuh"
#include "render_full.cuh"

#include <algorithm>
#include <climits>
#include <type_traits>

namespace fss {

namespace {

constexpr int BWD_FEAT_THREADS = 256;

// reduce-scatter of V values (power of two, 2..32 per lane...) across a warp:
// afterwards lane l holds the warp sum of values (V/32)*l + i for V >= 32, or
// of value l >> (5 - log2 V) for V < 32 (lanes sharing it hold equal sums).
template <int V>
__device__ __forceinline__ void reduce_scatter(float* v) {
    const int lane = threadIdx.x & 31;
    int n = V;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        if (n > 1) {
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int i = 0; i < V / 2; ++i) {
                if (i < n / 2) {
                    const float send = up ? v[i] : v[i + n / 2];
                    const float keep = up ? v[i + n / 2] : v[i];
                    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
            }
            n >>= 1;
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
        }
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// k_bwd_feat (Top-K): per selected (pixel x, k) with surfel i, the dot
// c_i . dL/dF(x) (read by k_bwd_geo_topk) and the feature gradient sum over x of
// w_i(x) dL/dF(x), grouped per tile
//
// Per tile (and per chunk of at most ECAP (pixel, k) entries):
//  1. the chunk's dL/dF rows are staged in shared memory (rows padded by
//     16 bytes); each thread keeps EPT entries (list position, weight) in
//     registers;
//  2. the selected list positions get dense slot numbers (mark + scan) and
//     a counting sort groups the entries by slot (shared-memory atomics)
//     into 8-byte records (slot, dL/dF row offset; weight);
//  3. the selected surfels' feature rows are staged in shared memory in one
//     parallel pass (over the counting-sort tables, which are dead by then);
//  4. the slot-grouped records are split into equal contiguous ranges, one
//     per group of G lanes (G = 16-byte chunks per row, rounded up to a
//     power of two).  A group takes four records per step.  When, for every
//     group of the warp, all four continue the group's current surfel (the
//     common case: about 30 entries per surfel and chunk), the warp takes
//     them without further checks; otherwise each record is checked, and a
//     group flushes one row of 16-byte vector reductions whenever its range
//     moves on to the next surfel.  The four partial dots are
//     reduce-scattered over the group, so each sum costs one shuffle per
//     lane and halving; packed FP32 FMAs (two products per instruction)
//     form the dots and w dL/dF.
// Shared memory holds everything the inner loop reads, so it runs without
// global-memory latency; the equal ranges keep the warps balanced.
// ---------------------------------------------------------------------------
constexpr int ECAP = 1024;  // (pixel, k) entries per pass
constexpr int PTAB = 2048;  // list positions per pass
constexpr int EPT = ECAP / BWD_FEAT_THREADS;  // entries per thread
constexpr int FEAT_UNION_BYTES = (PTAB + 2 * ECAP + 1) * 4;  // counting-sort tables, then feature rows
constexpr int MAX_ROW_PASSES = 64;

// entry record .x: slot << REC_ROW_BITS | offset of the entry's dL/dF row in
// 16-byte units (slot < PTAB = 2^11, offset < 2^17: 28 bits); .y: weight bits
constexpr int REC_ROW_BITS = 17;
constexpr int REC_ROW_MASK = (1 << REC_ROW_BITS) - 1;
constexpr int DOT_UNSET = 0x7fa00001;  // signalling-NaN payload: a dot not formed

// Sums of four values v[0..3] over the G lanes of a group (G a power of two,
// groups aligned in the warp), scattered: lanes swap halves of what is left
// and add, so each halving costs one shuffle per value kept.  Afterwards the
// lane holds the sums of the entries given by group_sum4_owned.
template <int G>
__device__ __forceinline__ void group_sum4(float (&v)[4], int sub) {
    constexpr unsigned ALL = 0xffffffffu;
    if constexpr (G >= 16) {
#pragma unroll
        for (int o = G >> 1; o >= 8; o >>= 1) {
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] += __shfl_xor_sync(ALL, v[j], o);
        }
    }
    if constexpr (G >= 2) {  // four values -> two: lanes with the offset bit keep entries 2, 3
        constexpr int o = G >= 8 ? 4 : G >> 1;
        const bool up = (sub & o) != 0;
        const float s0 = up ? v[0] : v[2], s1 = up ? v[1] : v[3];
        const float k0 = up ? v[2] : v[0], k1 = up ? v[3] : v[1];
        v[0] = k0 + __shfl_xor_sync(ALL, s0, o);
        v[1] = k1 + __shfl_xor_sync(ALL, s1, o);
    }
    if constexpr (G >= 4) {  // two -> one: lanes with the offset bit keep the second
        constexpr int o = G >= 8 ? 2 : 1;
        const bool up = (sub & o) != 0;
        const float sd = up ? v[0] : v[1], kp = up ? v[1] : v[0];
        v[0] = kp + __shfl_xor_sync(ALL, sd, o);
    }
    if constexpr (G >= 8) v[0] += __shfl_xor_sync(ALL, v[0], 1);
}

// rows of zeros after the chunk's dL/dF rows: at least G 16-byte chunks, so
// a lane without a record (or past the row) reads zeros
__host__ __device__ constexpr int zero_rows(int G, int rowb) { return (G * 16 + rowb - 1) / rowb; }

// (first entry, count) whose sums the lane stores after group_sum4: one
// lane per entry (G >= 4), two entries per lane (G = 2), all four (G = 1)
template <int G>
__device__ __forceinline__ int2 group_sum4_owned(int sub) {
    if constexpr (G >= 8) return make_int2((sub >> 1) & 3, (sub & 1) == 0 && sub < 8 ? 1 : 0);
    else if constexpr (G == 4) return make_int2(sub, 1);
    else if constexpr (G == 2) return make_int2(2 * sub, 2);
    else return make_int2(0, 4);
}

template <typename FT, int G>
__global__ void __launch_bounds__(BWD_FEAT_THREADS, 4) k_bwd_feat(const __grid_constant__ Cams cams,
                                                              const __grid_constant__ RParams P, const BwdArgs a,
                                                              int pch, int rowe, int ucap) {
    constexpr int E = FeatVec<FT>::E;
    constexpr int gpw = 32 / G, ngroups = (BWD_FEAT_THREADS / 32) * gpw;  // groups of G lanes
    extern __shared__ __align__(16) unsigned char smem[];
    const int rowb = rowe * (int)sizeof(FT), zr = zero_rows(G, rowb);
    FT* s_df = reinterpret_cast<FT*>(smem);  // [pch + zr][rowe]: the chunk's dL/dF rows, then zeros
    int2* s_rec = reinterpret_cast<int2*>(smem + (((size_t)(pch + zr) * rowb + 15) & ~(size_t)15));  // [ECAP]
    int* s_inv = reinterpret_cast<int*>(s_rec + ECAP);      // [ECAP] slot -> list position
    float* s_dot = reinterpret_cast<float*>(s_inv + ECAP);  // [ECAP] dots by entry (pixel * K + k)
    unsigned short* s_e = reinterpret_cast<unsigned short*>(s_dot + ECAP);  // [ECAP] record position -> entry
    int* s_gs = reinterpret_cast<int*>(s_e + ECAP);         // [ucap] slot -> gradient slot (this row pass)
    unsigned char* uni = reinterpret_cast<unsigned char*>(s_gs + ((ucap + 3) & ~3));
    int* s_tab = reinterpret_cast<int*>(uni);  // [PTAB] position -> slot
    int* s_off = s_tab + PTAB;                 // [ECAP + 1] per-slot counts -> offsets
    int* s_cur = s_off + ECAP + 1;             // [ECAP] scatter cursors
    FT* s_rows = reinterpret_cast<FT*>(uni);   // [ucap][rowe] feature rows (after the counting sort)
    __shared__ int s_red[33];
    __shared__ int s_tile;
    __shared__ int s_pass[MAX_ROW_PASSES + 1];

    if (a.st->err) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int TS = P.ts, lts = TS == 8 ? 3 : TS == 16 ? 4 : 5, npx = TS * TS;
    const int K = P.K, C = P.C, nvec = C / E;
    const int row16 = rowb / 16, zoff16 = pch * row16;  // padded row, first zero row (16-byte units)
    const FastDiv divK(K), divV(nvec);
    // chunk pixel of entry e = tid + i * BLOCK: a constant step when K divides the block
    const bool kdiv = BWD_FEAT_THREADS % K == 0;
    const int q0 = divK.div(tid), qstep = BWD_FEAT_THREADS / K;
    auto entry_q = [&](int i, int e) { return kdiv ? q0 + i * qstep : divK.div(e); };
    const int rv = BWD_FEAT_THREADS / nvec, r0v = tid / nvec, v0 = tid - r0v * nvec;  // row-chunk mapping
    const int sub = lane & (G - 1), gid = warp * gpw + lane / G;
    const bool chunk_live = sub < nvec;
    const int2 own = group_sum4_owned<G>(sub);
    const unsigned char* dfl = reinterpret_cast<const unsigned char*>(s_df) + sub * 16;  // this lane's chunk
    const FT* __restrict__ feats = reinterpret_cast<const FT*>(a.feats);
    const FT* __restrict__ dF = reinterpret_cast<const FT*>(a.d_feat);
    for (int i = tid; i < zr * rowb / 16; i += BWD_FEAT_THREADS)
        reinterpret_cast<uint4*>(s_df + (size_t)pch * rowe)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    for (int t = next_tile_q(a.persistent, &a.st->work_feat, &s_tile, true, cams); t < cams.total_tiles;
         t = next_tile_q(a.persistent, &a.st->work_feat, &s_tile, false, cams)) {
        const int view = view_of_tile(cams, t);
        const CamDev& cam = cams.c[view];
        const int lt = t - cam.tile_off;
        const int tx = lt % cam.tiles_x, ty = lt / cam.tiles_x;
        const int2 rg = checked_range(a.ranges, t, P.pair_cap, a.st);
        const int64_t vbase = (int64_t)view * P.N;

        for (int pc0 = 0; pc0 < npx; pc0 += pch) {
            const int np = min(pch, npx - pc0), ne = np * K;
            // dots not yet formed read as a sentinel (a NaN payload that arithmetic does
            // not produce), so the write-back needs no per-entry state
            for (int e = tid; e < ne; e += BWD_FEAT_THREADS) s_dot[e] = __int_as_float(DOT_UNSET);
            // list positions in passes of PTAB (one pass unless the tile's list is longer)
            const int L = rg.y - rg.x;
            for (int p0 = 0; p0 < L; p0 += PTAB) {
                // 1. this thread's entries (e = tid + i * BLOCK) in this pass: list position
                // and weight (the chunk pixel q and k follow from e)
                int epos[EPT];
                float ew[EPT];
#pragma unroll
                for (int i = 0; i < EPT; ++i) {
                    const int e = tid + i * BWD_FEAT_THREADS;
                    epos[i] = -1;
                    ew[i] = 0.0f;
                    if (e < ne) {
                        const int q = entry_q(i, e), k = e - q * K, p = pc0 + q;
                        const int px = tx * TS + (p & (TS - 1)), py = ty * TS + (p >> lts);
                        if (px < cam.W && py < cam.H) {
                            const int64_t pix = cam.pix_off + (int64_t)py * cam.W + px;
                            int pos = a.saved_pos[pix * K + k];
                            if (pos >= 0 && !in_bounds(a.st, SITE_LIST_POS, pos, L)) pos = -1;
                            if (pos >= p0 && pos < p0 + PTAB) {
                                epos[i] = pos - p0;
                                ew[i] = a.saved_w[pix * K + k];
                                if (P.renorm) {  // dL/dc = (w / W) dL/dF, W the selected weights' sum
                                    float ws = 0.0f;
                                    for (int k2 = 0; k2 < K; ++k2) ws += a.saved_w[pix * K + k2];
                                    ew[i] = ws > 0.0f ? ew[i] / ws : 0.0f;
                                }
                            }
                        }
                    }
                }
                if (p0 == 0) {
                    // the chunk's dL/dF rows (zeros outside the image), copied asynchronously
                    // once this thread's entries have arrived (issued first, they queued
                    // the entry loads behind them) and waited for just before the inner loop
                    if (r0v < rv) {
                        for (int q = r0v; q < np; q += rv) {
                            const int p = pc0 + q, px = tx * TS + (p & (TS - 1)), py = ty * TS + (p >> lts);
                            const bool in = px < cam.W && py < cam.H;
                            const FT* src = in ? dF + (cam.pix_off + (int64_t)py * cam.W + px) * C + v0 * E : dF;
                            cp_async16(s_df + (size_t)q * rowe + v0 * E, src, in ? 16 : 0);
                        }
                    }
                    cp_async_commit();
                }
                // 2. slots of the selected positions, then the entries grouped by slot: the
                // entries per position are counted, and one exclusive scan of
                // (count << 16 | count > 0) over the positions gives each position both its
                // first record (high half) and its slot (low half: selected positions
                // before it); counts <= ECAP and positions <= PTAB fit 16 bits each
                const int nt = min(PTAB, L - p0);  // positions in use (U <= nt)
                for (int i = tid; i < nt; i += BWD_FEAT_THREADS) s_tab[i] = 0;
                __syncthreads();
#pragma unroll
                for (int i = 0; i < EPT; ++i)
                    if (epos[i] >= 0) atomicAdd(&s_tab[epos[i]], 1 << 16);
                __syncthreads();
                const int tot = block_exscan_marked(s_tab, nt, s_red);
                const int U = tot & 0xffff, nsel = tot >> 16;
                if (U == 0) continue;
                for (int i = tid; i < nt; i += BWD_FEAT_THREADS) {
                    const int pre = s_tab[i], nxt = i + 1 < nt ? s_tab[i + 1] : tot;
                    if ((nxt & 0xffff) - (pre & 0xffff) == 1) {  // a selected position: its slot
                        s_inv[pre & 0xffff] = i;
                        s_off[pre & 0xffff] = pre >> 16;
                        s_cur[pre & 0xffff] = pre >> 16;
                    }
                }
                if (tid == 0) s_off[U] = nsel;
                int eslot[EPT];
#pragma unroll
                for (int i = 0; i < EPT; ++i) eslot[i] = epos[i] >= 0 ? s_tab[epos[i]] & 0xffff : -1;
                __syncthreads();
#pragma unroll
                for (int i = 0; i < EPT; ++i) {
                    if (eslot[i] >= 0) {
                        const int at = atomicAdd(&s_cur[eslot[i]], 1);
                        const int e = tid + i * BWD_FEAT_THREADS;
                        s_rec[at] = make_int2((eslot[i] << REC_ROW_BITS) | (entry_q(i, e) * row16), __float_as_int(ew[i]));
                        s_e[at] = (unsigned short)e;
                    }
                }
                const int npass = (U + ucap - 1) / ucap;  // <= MAX_ROW_PASSES (checked by the launcher)
                if (tid <= npass) s_pass[tid] = s_off[min(tid * ucap, U)];
                __syncthreads();
                for (int pi = 0; pi < npass; ++pi) {
                    const int u0 = pi * ucap, nu = min(ucap, U - u0);
                    const int eb = s_pass[pi], ee = s_pass[pi + 1];
                    // 3. feature rows of slots [u0, u0 + nu) (over the counting-sort tables),
                    // copied asynchronously like the dL/dF rows
                    for (int idx = tid; idx < nu * nvec; idx += BWD_FEAT_THREADS) {
                        const int u = divV.div(idx), v = idx - u * nvec;
                        const int64_t sp = (int64_t)a.list[rg.x + p0 + s_inv[u0 + u]] - vbase;
                        const bool ok = in_bounds(a.st, SITE_ITEM, sp, P.N);  // check build: a zero row, no slot
                        cp_async16(s_rows + (size_t)u * rowe + v * E, ok ? feats + sp * C + v * E : feats, ok ? 16 : 0);
                        if (v == 0) {
                            const int sl = ok ? a.splat_slot[sp] : -1;
                            s_gs[u] = in_bounds(a.st, SITE_SLOT, sl, P.N) ? sl : -1;
                        }
                    }
                    cp_async_commit();
                    cp_async_wait_all();
                    __syncthreads();
                    // 4. equal contiguous record ranges per group, starting at an even record
                    // (records are read two at a time), four records per step (warp-uniform
                    // trip count)
                    const int ea = eb & ~1;
                    const int len = (((ee - ea + ngroups - 1) / ngroups) + 3) & ~3;
                    const int i0 = ea + gid * len, i1 = min(ee, i0 + len);
                    int cur = -1;  // the group's current slot
                    float2 f2[E / 2], acc2[E / 2];
#pragma unroll
                    for (int e = 0; e < E / 2; ++e) { f2[e] = make_float2(0.0f, 0.0f); acc2[e] = f2[e]; }
                    // flush the current slot's w dL/dF, then move to `slot`
                    auto next_slot = [&](int slot) {
                        if (chunk_live) {
                            if (cur >= 0 && FSS_CHECKED(s_gs[cur - u0] >= 0)) {
                                float* dst = a.feat_acc + (int64_t)s_gs[cur - u0] * C + sub * E;
#pragma unroll
                                for (int e = 0; e < E / 2; e += 2)
                                    red_add_v4(dst + 2 * e, acc2[e].x, acc2[e].y, acc2[e + 1].x, acc2[e + 1].y);
                            }
                            if (slot >= 0) {
                                float fv[E];
                                FeatVec<FT>::lds(s_rows + (size_t)(slot - u0) * rowe + sub * E, fv);
#pragma unroll
                                for (int e = 0; e < E / 2; ++e) f2[e] = make_float2(fv[2 * e], fv[2 * e + 1]);
                            }
#pragma unroll
                            for (int e = 0; e < E / 2; ++e) acc2[e] = make_float2(0.0f, 0.0f);
                        }
                        cur = slot;
                    };
                    // one record of the current slot: returns the lane's partial dot
                    // (no record: the zero row and weight 0, so the code has no branch)
                    auto take = [&](int2 r, bool live) {
                        const bool on = chunk_live && live;
                        float g[E];
                        FeatVec<FT>::lds(reinterpret_cast<const FT*>(dfl + (size_t)(on ? r.x & REC_ROW_MASK : zoff16) * 16), g);
                        const float w = on ? __int_as_float(r.y) : 0.0f;
                        const float2 w2 = make_float2(w, w);
                        float2 d = make_float2(0.0f, 0.0f);
#pragma unroll
                        for (int e = 0; e < E / 2; ++e) {
                            const float2 g2 = make_float2(g[2 * e], g[2 * e + 1]);
                            d = __ffma2_rn(f2[e], g2, d);
                            acc2[e] = __ffma2_rn(w2, g2, acc2[e]);
                        }
                        return d.x + d.y;
                    };
                    for (int st = 0; st < len; st += 4) {
                        const int i = i0 + st;
                        int4 ra = make_int4(-1, 0, -1, 0), rb = ra;
                        if (i < i1) ra = *reinterpret_cast<const int4*>(s_rec + i);
                        if (i + 2 < i1) rb = *reinterpret_cast<const int4*>(s_rec + i + 2);
                        const int2 r[4] = {make_int2(ra.x, ra.y), make_int2(ra.z, ra.w), make_int2(rb.x, rb.y),
                                           make_int2(rb.z, rb.w)};
                        float v[4];
                        // steady: all four records continue the group's current slot (sorted
                        // records: the fourth decides), or the group's range is used up
                        const bool done = i >= i1;
                        const bool steady = done || (i >= eb && i + 3 < i1 && (rb.z >> REC_ROW_BITS) == cur);
                        if (__all_sync(0xffffffffu, steady)) {  // warp-uniform: no per-record checks
#pragma unroll
                            for (int j = 0; j < 4; ++j) v[j] = take(r[j], !done);
                        } else {
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const bool live = i + j >= eb && i + j < i1;
                                const int slot = r[j].x >> REC_ROW_BITS;
                                if (live && slot != cur) next_slot(slot);
                                v[j] = take(r[j], live);
                            }
                        }
                        group_sum4<G>(v, sub);
#pragma unroll
                        for (int j = 0; j < (G >= 4 ? 1 : 4 / G); ++j) {
                            const int at = i + own.x + j;
                            if (j < own.y && at >= eb && at < i1) s_dot[s_e[at]] = v[j];
                        }
                    }
                    next_slot(-1);
                    __syncthreads();
                }
            }
            // the dots, written back in (pixel, k) order
#pragma unroll
            for (int i = 0; i < EPT; ++i) {
                const int e = tid + i * BWD_FEAT_THREADS;
                const float d = e < ne ? s_dot[e] : __int_as_float(DOT_UNSET);
                if (__float_as_int(d) != DOT_UNSET) {
                    const int q = entry_q(i, e), p = pc0 + q;
                    const int64_t pix = cam.pix_off + (int64_t)(ty * TS + (p >> lts)) * cam.W + tx * TS + (p & (TS - 1));
                    a.dots[pix * K + (e - q * K)] = d;
                }
            }
            cp_async_wait_all();  // (a chunk without selected entries never waited)
            __syncthreads();
        }
    }
}

// ---------------------------------------------------------------------------
// k_bwd_geo_topk: back-to-front replay of the Top-K render, one warp per 8 x 4
// pixel block, each warp on its own
// ---------------------------------------------------------------------------
// The warp walks its tile's list backwards 32 positions at a time (stage_chunk,
// with the surfels' gradient slots beside the records); per surfel its lanes'
// 13 partial derivatives are reduce-scattered over the warp, and 13 lanes add
// the sums to the surfel's gradient row in L2 (64 consecutive bytes, one
// request).  Partial sums used to be gathered per tile in shared memory, behind
// the barriers of the staging (1.8 cycles per issued instruction there): 98 us for a
// 640 x 480 frame of 500k surfels, 88 here; 1296 x 968 with K = 24 324 / 305.
// Bound by instruction issue: about 40 of a warp evaluation's instructions are
// the record, the ray and the derivatives, 55 the reduce-scatter.
constexpr int GEO_THREADS = 128;  // threads per CTA (64 for 8 x 8 tiles): parts of a tile

// CF > 0 instances (16 or 32: channels, rounded up; which path: feat_path) also
// take the feature gradients: the dot c_j . dL/dF from the surfel's staged row
// and the pixel's gradient in registers, and one more reduce-scatter of w dL/dF
// per surfel that any of the warp's pixels selected.  The feature kernel, which
// groups K entries per pixel by surfel in shared memory first, and its dots in
// memory are then not needed: 1296 x 968, 16 channels, K = 24 FP32 geometry and
// features 860 us before, 546 with H = 1 (step 1573 / 1264).  Bound by
// instruction issue: 16 selects and multiplies and 17 shuffles per surfel and
// warp for 16 channels.
// H = 2: a lane has a pixel of each of two blocks, one above the other, so a
// surfel that meets both is read once and its sums go through one reduce-scatter
// (1296 x 968, 500k surfels, 16 channels, K = 24: step FP32 1265 -> 1193 us, BF16
// 1174 -> 1141; 640 x 480, K = 16 244 -> 237, BF16 level).  A warp then has twice the
// work, which small images lose by (256 x 200 146 -> 170, 128 x 128 171 -> 215):
// taken from 48 blocks an SM on.  Without the feature gradients it gains less than
// it loses elsewhere: 1.2M surfels 1295 -> 1249, but six views of 1M 3206 -> 3217,
// 640 x 480 328 -> 340.
template <int CF, typename FT>
struct GeoStage {
    WarpStage st[2];
    int32_t slot[2][32];
    FT row[CF ? 2 : 1][CF ? 32 : 1][CF ? CF + 16 / (int)sizeof(FT) : 1];  // feature rows, padded by 16 bytes
};

// threads per CTA: 64 where the stages of four warps are above 48 KB
template <int TS, int CF, typename FT, int H>
constexpr int geo_threads() {
    const int nt = CF && 4 * sizeof(GeoStage<CF, FT>) > 47 * 1024 ? GEO_THREADS / 2 : GEO_THREADS;
    return TS * TS / H < nt ? TS * TS / H : nt;
}

// warp sums of v[0..12]: afterwards an even lane l < 26 holds the sum of v[l >> 1]
__device__ __forceinline__ void reduce_scatter13(float (&v)[13]) {
    const int lane = threadIdx.x & 31;
    const bool up = (lane & 16) != 0;
    // values i and 8 + i in pairs for i < 5, values 5..7 summed by both halves
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const float send = up ? v[i] : v[i + 8];
        const float keep = up ? v[i + 8] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
    for (int i = 5; i < 8; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], 16);
#pragma unroll
    for (int o = 8, n = 8; o > 1; o >>= 1, n >>= 1) {
        const bool u = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < n / 2; ++i) {
            const float send = u ? v[i] : v[i + n / 2];
            const float keep = u ? v[i + n / 2] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
}

template <int TS, bool VAR, int CF = 0, typename FT = float, int H = 1>
__global__ void __launch_bounds__(geo_threads<TS, CF, FT, H>(),
                                  (CF == 0 ? 1024 : CF == 16 && H == 1 ? 768 : 512) / geo_threads<TS, CF, FT, H>())
    k_bwd_geo_topk(const __grid_constant__ Cams cams, const __grid_constant__ RParams P, const BwdArgs a) {
    constexpr int NT = geo_threads<TS, CF, FT, H>(), NW = NT / 32, PARTS = TS * TS / H / NT, WX = TS / 8;
    constexpr unsigned ALL = 0xffffffffu;
    static_assert(!VAR || CF == 0, "the variants take the feature gradients from their own kernel");
    __shared__ __align__(16) GeoStage<CF, FT> s_stage[NW];
    __shared__ int s_work;
    if (a.st->err) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    GeoStage<CF, FT>& G = s_stage[warp];
    constexpr int E = FeatVec<FT>::E;
    const FT* __restrict__ feats = reinterpret_cast<const FT*>(a.feats);
    if constexpr (CF > 0) {  // channels past C: zeros, once
        for (int i = lane; i < 2 * 32 * CF; i += 32)
            if (i % CF >= P.C) G.row[i / (32 * CF)][(i / CF) % 32][i % CF] = FT(0.0f);
        __syncwarp();
    }
    const int K = P.K, total = cams.total_tiles * PARTS;
    for (bool first = true;; first = false) {
        int u;  // this CTA's next part of a tile (heavy tiles first)
        if (!a.persistent) {
            u = first ? (int)blockIdx.x : INT_MAX;
        } else {
            __syncthreads();
            if (threadIdx.x == 0) s_work = (int)atomicAdd(&a.st->work_geo, 1u);
            __syncthreads();
            u = s_work;
        }
        if (u >= total) return;
        const int t = cams.tile_order ? cams.tile_order[u / PARTS] : u / PARTS;
        // this warp's block of the tile, or (H = 2) the upper one of two
        const int wu = (u % PARTS) * NW + warp, wb = H == 2 ? 2 * WX * (wu / WX) + wu % WX : wu;
        const uint32_t wbit = H == 2 ? (1u | 1u << WX) << wb : 1u << wb;
        const int view = view_of_tile(cams, t);
        const CamDev& cam = cams.c[view];
        const int lt = t - cam.tile_off;
        const int tx = lt % cam.tiles_x, ty = lt / cam.tiles_x;
        const int px = tx * TS + 8 * (wb % WX) + (lane & 7), py = ty * TS + 4 * (wb / WX) + (lane >> 3);
        const float pxf = (float)px + 0.5f, pyf = (float)py + 0.5f;
        const int2 rg = checked_range(a.ranges, t, P.pair_cap, a.st);
        const int64_t vbase = (int64_t)view * P.N;
        // VAR instances carry the variants (renormalised Top-K, spherical-harmonic
        // item colours, low-pass filter), read from the parameters
        const float* __restrict__ rgbv = a.rgb + (VAR && P.color_sh ? 3 * vbase : 0);
        const int64_t pix0 = cam.pix_off + (int64_t)py * cam.W + px;
        const uint32_t* list = a.list + rg.x;
        const uint32_t* masks = a.masks + rg.x;
        float* grows = a.grad_item + vbase * GRAD_STRIDE;  // this view's gradient rows

        int nstop[H], kk[H], next_pos[H], top = 0;
        float T[H], gr[H], gg[H], gb[H], Sh[H];
        float next_dot[H];  // (CF: that surfel's weight)
        // a selected surfel adds rn_a * dot + rn_b to what its weight multiplies:
        // the dot itself, or (dot - F.dL/dF) / W for the renormalised variant
        float rn_a[H], rn_b[H];
        float2 dfr[H][CF ? CF / 2 : 1];  // the pixels' dL/dF
#pragma unroll
        for (int i = 0; i < H; ++i) {
            const int64_t pix = pix0 + (int64_t)(4 * i) * cam.W;
            const bool inside = px < cam.W && py + 4 * i < cam.H;
            nstop[i] = 0;
            T[i] = 1.0f;
            gr[i] = gg[i] = gb[i] = Sh[i] = next_dot[i] = rn_b[i] = 0.0f;
            rn_a[i] = 1.0f;
            kk[i] = next_pos[i] = -1;
            if (inside) {
                nstop[i] = min(a.saved_nstop[pix], rg.y - rg.x);
                T[i] = a.out_T[pix];
                gr[i] = a.d_rgb[3 * pix];
                gg[i] = a.d_rgb[3 * pix + 1];
                gb[i] = a.d_rgb[3 * pix + 2];
                Sh[i] = P.bg[0] * gr[i] + P.bg[1] * gg[i] + P.bg[2] * gb[i] + (a.d_T ? a.d_T[pix] : 0.0f);
                int k = K - 1;
                for (; k >= 0; --k)
                    if (a.saved_pos[pix * K + k] >= 0) break;
                kk[i] = k;
                if (k >= 0) {
                    next_pos[i] = a.saved_pos[pix * K + k];
                    next_dot[i] = (CF == 0 ? a.dots : a.saved_w)[pix * K + k];
                }
                if (VAR && P.renorm) {  // entries 0..k are the selected ones, front to back
                    float ws = 0.0f, wd = 0.0f;
                    for (int k2 = 0; k2 <= k; ++k2) {
                        const float wv = a.saved_w[pix * K + k2];
                        ws += wv;
                        wd = fmaf(wv, a.dots[pix * K + k2], wd);
                    }
                    rn_a[i] = ws > 0.0f ? 1.0f / ws : 0.0f;
                    rn_b[i] = -wd * rn_a[i] * rn_a[i];
                }
            }
            if constexpr (CF > 0) {
#pragma unroll
                for (int v = 0; v < CF / E; ++v) {
                    float f[E];
#pragma unroll
                    for (int e = 0; e < E; ++e) f[e] = 0.0f;
                    if (inside && v * E < P.C) FeatVec<FT>::load(reinterpret_cast<const FT*>(a.d_feat) + pix * P.C + v * E, f);
#pragma unroll
                    for (int e = 0; e < E / 2; ++e) dfr[i][v * (E / 2) + e] = make_float2(f[2 * e], f[2 * e + 1]);
                }
            }
            top = max(top, nstop[i]);
        }
        const int L = __reduce_max_sync(ALL, top);

        // one chunk's records and gradient slots, and the lane mask of those the warp meets
        auto stage = [&](int buf, const ListEntry& e) {
            const int64_t sp = (int64_t)e.item - vbase;
            if ((e.mask & wbit) && FSS_CHECKED(sp >= 0 && sp < P.N)) {
                cp_async4(&G.slot[buf][lane], a.splat_slot + sp);
                if constexpr (CF > 0) {
#pragma unroll
                    for (int v = 0; v < CF / E; ++v)
                        if (v * E < P.C) cp_async16(&G.row[buf][lane][v * E], feats + sp * P.C + v * E, 16);
                }
            }
            return stage_chunk(G.st[buf], e, wbit, a.rec, rgbv, vbase, P.N, a.st);
        };
        // chunk b0 is worked on while the one before it is copied and the list entries of the next are read
        int b0 = ((L - 1) >> 5) << 5;  // (L = 0: the loop does not run)
        ListEntry e1 = list_entry(list, masks, b0 + lane, L);
        uint32_t word = stage((b0 >> 5) & 1, e1), met[H] = {}, met_next[H] = {};  // (H = 2: those that each block meets)
        auto blocks = [&](uint32_t (&m)[H]) {
#pragma unroll
            for (int i = 0; i < H; ++i) m[i] = __ballot_sync(ALL, (e1.mask & (1u << WX * i << wb)) != 0u);
        };
        if (H == 2) blocks(met);
        e1 = list_entry(list, masks, b0 - 32 + lane, L);
        for (; b0 >= 0 && L > 0; b0 -= 32) {
            const int buf = (b0 >> 5) & 1;
            const WarpStage& S = G.st[buf];
            const uint32_t next = stage(buf ^ 1, e1);
            if (H == 2) blocks(met_next);
            e1 = list_entry(list, masks, b0 - 64 + lane, L);
            cp_async_wait_prev();  // this chunk's copies
            __syncwarp();
            for (uint32_t bits = word; bits != 0u; bits ^= 0x80000000u >> __clz(bits)) {
                const int j = 31 - __clz(bits), pos = b0 + j;
                float g[VAR ? 16 : 13];
#pragma unroll
                for (int k = 0; k < (VAR ? 16 : 13); ++k) g[k] = 0.0f;
                bool contrib = false, sel[H];  // CF: this pixel selected the surfel, with the forward's weight
                float wsel[H];
                const float4 oc = S.oc[j];
#pragma unroll
                for (int i = 0; i < H; ++i) {
                    sel[i] = false;
                    wsel[i] = 0.0f;
                    Hit h;
                    if (H == 2 && !((met[i] >> j) & 1u)) continue;  // as the forward, block by block
                    if (pos < nstop[i] &&
                        eval_splat<VAR>(S.r0[j], S.r1[j], S.r2[j], oc.x, pxf, pyf + (float)(4 * i), P.alpha_min, cam.near_plane, h,
                                        P.lowpass)) {
                        contrib = true;
                        const float alpha = fminf(h.alpha_raw, P.alpha_max);
                        const float Tj = T[i] * rcp_approx(1.0f - alpha);
                        const float w = alpha * Tj;
                        float s = oc.y * gr[i] + oc.z * gg[i] + oc.w * gb[i];
                        if (pos == next_pos[i]) {
                            if constexpr (CF > 0) {
                                float d[CF / E];  // by 16-byte chunk, summed as k_bwd_feat's lanes sum them
#pragma unroll
                                for (int v = 0; v < CF / E; ++v) {
                                    float f[E];
                                    FeatVec<FT>::lds(&G.row[buf][j][v * E], f);
                                    float2 p = make_float2(0.0f, 0.0f);
#pragma unroll
                                    for (int e = 0; e < E / 2; ++e)
                                        p = __ffma2_rn(make_float2(f[2 * e], f[2 * e + 1]), dfr[i][v * (E / 2) + e], p);
                                    d[v] = p.x + p.y;
                                }
#pragma unroll
                                for (int o = CF / E / 2; o > 0; o >>= 1)
#pragma unroll
                                    for (int v = 0; v < o; ++v) d[v] += d[v + o];
                                s += d[0];
                                sel[i] = true;
                                wsel[i] = next_dot[i];
                            } else {
                                s += VAR ? fmaf(next_dot[i], rn_a[i], rn_b[i]) : next_dot[i];
                            }
                            const int k = --kk[i];
                            const int64_t at = (pix0 + (int64_t)(4 * i) * cam.W) * K + k;
                            next_pos[i] = k >= 0 ? a.saved_pos[at] : -1;
                            next_dot[i] = k >= 0 ? (CF == 0 ? a.dots : a.saved_w)[at] : 0.0f;
                        }
                        const float dal = Tj * (s - Sh[i]);
                        Sh[i] = fmaf(alpha, s - Sh[i], Sh[i]);  // a s + (1 - a) S
                        g[10] = i ? fmaf(w, gr[i], g[10]) : w * gr[i];
                        g[11] = i ? fmaf(w, gg[i], g[11]) : w * gg[i];
                        g[12] = i ? fmaf(w, gb[i], g[12]) : w * gb[i];
                        if (h.alpha_raw < P.alpha_max) {
                            g[9] = i ? fmaf(dal, h.G, g[9]) : dal * h.G;
                            const float drho = -0.5f * alpha * dal;
                            if (VAR && h.scr) {  // low-pass screen term: rho = 2 |x - c|^2, d rho / d c = -4 (X, Y)
                                g[VAR ? 13 : 0] += -4.0f * h.X * drho;
                                g[VAR ? 14 : 0] += -4.0f * h.Y * drho;
                            } else {
                                const float du = 2.0f * h.u * drho, dv = 2.0f * h.v * drho;
                                const float gc0 = du * h.inv, gc1 = dv * h.inv, gc2 = -(du * h.u + dv * h.v) * h.inv;
                                if (i == 0) {
                                    g[0] = gc0 * h.X; g[1] = gc0 * h.Y; g[2] = gc0;
                                    g[3] = gc1 * h.X; g[4] = gc1 * h.Y; g[5] = gc1;
                                    g[6] = gc2 * h.X; g[7] = gc2 * h.Y; g[8] = gc2;
                                } else {
                                    g[0] = fmaf(gc0, h.X, g[0]); g[1] = fmaf(gc0, h.Y, g[1]); g[2] += gc0;
                                    g[3] = fmaf(gc1, h.X, g[3]); g[4] = fmaf(gc1, h.Y, g[4]); g[5] += gc1;
                                    g[6] = fmaf(gc2, h.X, g[6]); g[7] = fmaf(gc2, h.Y, g[7]); g[8] += gc2;
                                }
                            }
                        }
                        T[i] = Tj;
                    }
                }
                if (__any_sync(ALL, contrib)) {
                    if constexpr (VAR) reduce_scatter<16>(g);  // lane l holds value l >> 1
                    else reduce_scatter13(g);
                    const int slot = G.slot[buf][j];
                    if ((lane & 1) == 0 && (lane >> 1) < (VAR ? 15 : 13) && in_bounds(a.st, SITE_SLOT, slot, P.N))
                        atomicAdd(grows + (int64_t)slot * GRAD_STRIDE + (lane >> 1), g[0]);
                    if constexpr (CF > 0) {
                        if (__any_sync(ALL, sel[0] || sel[H - 1])) {
                            float gf[CF];
#pragma unroll
                            for (int c = 0; c < CF / 2; ++c) {
                                gf[2 * c] = sel[0] ? wsel[0] * dfr[0][c].x : 0.0f;  // (dL/dF may be infinite where not selected)
                                gf[2 * c + 1] = sel[0] ? wsel[0] * dfr[0][c].y : 0.0f;
                                if (H == 2 && sel[H - 1]) {
                                    gf[2 * c] = fmaf(wsel[H - 1], dfr[H - 1][c].x, gf[2 * c]);
                                    gf[2 * c + 1] = fmaf(wsel[H - 1], dfr[H - 1][c].y, gf[2 * c + 1]);
                                }
                            }
                            reduce_scatter<CF>(gf);  // lane l holds channel l (CF = 32) or l >> 1
                            const int c = CF == 32 ? lane : lane >> 1;
                            if ((CF == 32 || (lane & 1) == 0) && c < P.C && in_bounds(a.st, SITE_SLOT, slot, P.N))
                                atomicAdd(a.feat_acc + (int64_t)slot * P.C + c, gf[0]);
                        }
                    }
                }
            }
            word = next;
#pragma unroll
            for (int i = 0; i < H; ++i) met[i] = met_next[i];
            __syncwarp();  // every lane has read this half before the next copies into it
        }
        cp_async_wait_all();
        __syncwarp();  // before the warp's next block
    }
}

// ---------------------------------------------------------------------------
// k_bwd_geo_full: the same replay for the full accumulation (K = 0)
// ---------------------------------------------------------------------------
// (TOPK: only the selected contributors, with the forward's weights; a surfel that none
// of the warp's pixels selected costs no products.)
// Every contributor takes the dot c_j . dL/dF and gives w dL/dF to its row.  The
// block's dL/dF stays in registers for the whole walk, as PX pixels x 4 NQ channels
// per lane (FullLanes: 8 x 8 at 64 channels), and serves both products: a lane's
// partial dots of its PX pixels are reduce-scattered over the CL lanes that share
// them, which leaves each lane its own pixel's dot (7 shuffles for 8 pixels); with the
// block's weights from shared memory a lane's channel sums are reduce-scattered over the
// pixel groups and added to the surfel's row in L2 (256 consecutive bytes a warp at 64
// channels).  The next surfel's row is read ahead.  A dL/dF that is not finite would reach
// the surfels that only other pixels of its block met, as -0 times it: such a block leaves
// those products out.  640 x 480, 500k surfels, 64 channels
// FP32: 481 us with a CTA per tile, all channels of a pixel in its lane and 95
// shuffles per surfel for the sums, 246 here; the step with 16 channels 421 -> 339, 128
// channels (spilled there) 2609 -> 811.  Bound by instruction issue.
struct FullGeoStage {
    WarpStage st[2];
    int32_t slot[2][32], sp[2][32];  // gradient slots and ids of the staged surfels
    float4 w[2][8];                  // the block's weights of a surfel, two surfels in turn
};

__device__ __forceinline__ void red_add_v2(float* addr, float a, float b) {
    asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(addr), "f"(a), "f"(b) : "memory");
}

template <int TS, int CMAX, typename FT, bool VAR, bool TOPK = false>
__global__ void __launch_bounds__(full_threads<TS>(), (CMAX <= 64 ? 512 : 256) / full_threads<TS>())
    k_bwd_geo_full(const __grid_constant__ Cams cams, const __grid_constant__ RParams P, const BwdArgs a) {
    using L = FullLanes<CMAX>;
    constexpr int NT = full_threads<TS>(), NW = NT / 32, PARTS = TS * TS / NT, PX = L::PX, NQ = L::NQ, CL = L::CL;
    constexpr unsigned ALL = 0xffffffffu;
    __shared__ __align__(16) FullGeoStage s_stage[NW];
    __shared__ int s_work;
    if (a.st->err) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cl = lane % CL, pg = lane / CL;  // this lane's channels and pixels of the products
    FullGeoStage& G = s_stage[warp];
    const FT* __restrict__ feats = reinterpret_cast<const FT*>(a.feats);
    const int C = P.C, total = cams.total_tiles * PARTS;
    for (bool first = true;; first = false) {
        int u;  // this CTA's next part of a tile (heavy tiles first)
        if (!a.persistent) {
            u = first ? (int)blockIdx.x : INT_MAX;
        } else {
            __syncthreads();
            if (threadIdx.x == 0) s_work = (int)atomicAdd(&a.st->work_geo, 1u);
            __syncthreads();
            u = s_work;
        }
        if (u >= total) return;
        const int t = cams.tile_order ? cams.tile_order[u / PARTS] : u / PARTS;
        const int wb = (u % PARTS) * NW + warp;  // this warp's block of the tile
        const uint32_t wbit = 1u << wb;
        const int view = view_of_tile(cams, t);
        const CamDev& cam = cams.c[view];
        const int lt = t - cam.tile_off;
        const int tx = lt % cam.tiles_x, ty = lt / cam.tiles_x;
        const int bx = tx * TS + 8 * (wb % (TS / 8)), by = ty * TS + 4 * (wb / (TS / 8));
        const int px = bx + (lane & 7), py = by + (lane >> 3);
        const bool inside = px < cam.W && py < cam.H;
        const float pxf = (float)px + 0.5f, pyf = (float)py + 0.5f;
        const int2 rg = checked_range(a.ranges, t, P.pair_cap, a.st);
        const int64_t vbase = (int64_t)view * P.N;
        // VAR instances carry the variants (spherical-harmonic item colours, low-pass filter)
        const float* __restrict__ rgbv = a.rgb + (VAR && P.color_sh ? 3 * vbase : 0);
        const int64_t pix = cam.pix_off + (int64_t)py * cam.W + px;
        const uint32_t* list = a.list + rg.x;
        const uint32_t* masks = a.masks + rg.x;
        float* grows = a.grad_item + vbase * GRAD_STRIDE;  // this view's gradient rows

        const int K = P.K;
        int kk = -1, next_pos = -1;  // TOPK: the pixel's next selected surfel ...
        float next_w = 0.0f;         // ... and the forward's weight of it
        int nstop = 0;
        float T = 1.0f, gr = 0.0f, gg = 0.0f, gb = 0.0f, Sh = 0.0f;
        if (inside) {
            nstop = min(a.saved_nstop[pix], rg.y - rg.x);
            T = a.out_T[pix];
            gr = a.d_rgb[3 * pix];
            gg = a.d_rgb[3 * pix + 1];
            gb = a.d_rgb[3 * pix + 2];
            Sh = P.bg[0] * gr + P.bg[1] * gg + P.bg[2] * gb + (a.d_T ? a.d_T[pix] : 0.0f);
            if constexpr (TOPK) {
                for (kk = K - 1; kk >= 0; --kk)
                    if (a.saved_pos[pix * K + kk] >= 0) break;
                if (kk >= 0) {
                    next_pos = a.saved_pos[pix * K + kk];
                    next_w = a.saved_w[pix * K + kk];
                }
            }
        }
        const int len = __reduce_max_sync(ALL, nstop);
        if (len == 0) continue;
        float2 df[PX][NQ][2];  // the lane's pixels x channels of dL/dF
#pragma unroll
        for (int p = 0; p < PX; ++p) {
            const int i = pg * PX + p, qx = bx + (i & 7), qy = by + (i >> 3);
            float4 f[NQ];
            L::load_row(reinterpret_cast<const FT*>(a.d_feat) + (cam.pix_off + (int64_t)qy * cam.W + qx) * C, cl,
                        qx < cam.W && qy < cam.H ? C : 0, f);
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                df[p][q][0] = make_float2(f[q].x, f[q].y);
                df[p][q][1] = make_float2(f[q].z, f[q].w);
            }
        }
        float2 z = make_float2(0.0f, 0.0f);  // NaN when some dL/dF is not finite
#pragma unroll
        for (int p = 0; p < PX; ++p)
#pragma unroll
            for (int q = 0; q < NQ; ++q)
#pragma unroll
                for (int k = 0; k < 2; ++k) z = __ffma2_rn(df[p][q][k], make_float2(0.0f, 0.0f), z);
        const bool careful = __any_sync(ALL, !(z.x + z.y == 0.0f));

        // one chunk's records and gradient slots, and the lane mask of those the warp meets
        auto stage = [&](int buf, const ListEntry& e) {
            const int64_t sp = (int64_t)e.item - vbase;
            if ((e.mask & wbit) && FSS_CHECKED(sp >= 0 && sp < P.N)) {
                cp_async4(&G.slot[buf][lane], a.splat_slot + sp);
                G.sp[buf][lane] = (int32_t)sp;
            }
            return stage_chunk(G.st[buf], e, wbit, a.rec, rgbv, vbase, P.N, a.st);
        };
        // chunk b0 is worked on while the one before it is copied and the list entries of the next are read
        int b0 = ((len - 1) >> 5) << 5;
        ListEntry e1 = list_entry(list, masks, b0 + lane, len);
        uint32_t word = stage((b0 >> 5) & 1, e1);
        e1 = list_entry(list, masks, b0 - 32 + lane, len);
        int par = 0;
        for (; b0 >= 0; b0 -= 32) {
            const int buf = (b0 >> 5) & 1;
            const WarpStage& S = G.st[buf];
            const uint32_t next = stage(buf ^ 1, e1);
            e1 = list_entry(list, masks, b0 - 64 + lane, len);
            cp_async_wait_prev();  // this chunk's copies
            __syncwarp();
            float4 nf[NQ];
            if (word) L::load_row(feats + (int64_t)G.sp[buf][31 - __clz(word)] * C, cl, C, nf);
            for (uint32_t bits = word; bits != 0u;) {
                const int j = 31 - __clz(bits), pos = b0 + j;
                bits ^= 0x80000000u >> __clz(bits);
                float4 f[NQ];
#pragma unroll
                for (int q = 0; q < NQ; ++q) f[q] = nf[q];
                if (bits) L::load_row(feats + (int64_t)G.sp[buf][31 - __clz(bits)] * C, cl, C, nf);
                Hit h;
                const float4 oc = S.oc[j];
                const bool contrib = pos < nstop && eval_splat<VAR>(S.r0[j], S.r1[j], S.r2[j], oc.x, pxf, pyf, P.alpha_min,
                                                                    cam.near_plane, h, P.lowpass);
                if (!__any_sync(ALL, contrib)) continue;
                const bool sel = TOPK ? contrib && pos == next_pos : contrib;
                const bool feat = TOPK ? __any_sync(ALL, sel) : true;
                // c_j . dL/dF, this lane's pixel
                float dot[PX];
                if (feat) {
#pragma unroll
                for (int p = 0; p < PX; ++p) {
                    float2 d = make_float2(0.0f, 0.0f);
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        d = __ffma2_rn(make_float2(f[q].x, f[q].y), df[p][q][0], d);
                        d = __ffma2_rn(make_float2(f[q].z, f[q].w), df[p][q][1], d);
                    }
                    dot[p] = d.x + d.y;
                }
#pragma unroll
                for (int o = CL / 2, n = PX / 2; o > 0; o >>= 1, n >>= 1) {
                    const bool up = (lane & o) != 0;
#pragma unroll
                    for (int i = 0; i < n; ++i) {
                        const float send = up ? dot[i] : dot[i + n];
                        const float keep = up ? dot[i + n] : dot[i];
                        dot[i] = keep + __shfl_xor_sync(ALL, send, o);
                    }
                }
                }
                float g[VAR ? 16 : 13];
#pragma unroll
                for (int k = 0; k < (VAR ? 16 : 13); ++k) g[k] = 0.0f;
                float w = 0.0f, wf = -0.0f;  // wf: the weight on dL/dF (-0: not one of its pixels)
                if (contrib) {
                    const float alpha = fminf(h.alpha_raw, P.alpha_max);
                    const float Tj = T * rcp_approx(1.0f - alpha);
                    w = alpha * Tj;
                    float s = oc.y * gr + oc.z * gg + oc.w * gb;
                    if (sel) s += dot[0];
                    if constexpr (TOPK) {
                        if (sel) {
                            wf = next_w;
                            --kk;
                            next_pos = kk >= 0 ? a.saved_pos[pix * K + kk] : -1;
                            next_w = kk >= 0 ? a.saved_w[pix * K + kk] : 0.0f;
                        }
                    } else {
                        wf = w;
                    }
                    const float dal = Tj * (s - Sh);
                    Sh = fmaf(alpha, s - Sh, Sh);  // a s + (1 - a) S
                    g[10] = w * gr;
                    g[11] = w * gg;
                    g[12] = w * gb;
                    if (h.alpha_raw < P.alpha_max) {
                        g[9] = dal * h.G;
                        const float drho = -0.5f * alpha * dal;
                        if (VAR && h.scr) {  // low-pass screen term: rho = 2 |x - c|^2, d rho / d c = -4 (X, Y)
                            g[VAR ? 13 : 0] = -4.0f * h.X * drho;
                            g[VAR ? 14 : 0] = -4.0f * h.Y * drho;
                        } else {
                            const float du = 2.0f * h.u * drho, dv = 2.0f * h.v * drho;
                            const float gc0 = du * h.inv, gc1 = dv * h.inv, gc2 = -(du * h.u + dv * h.v) * h.inv;
                            g[0] = gc0 * h.X; g[1] = gc0 * h.Y; g[2] = gc0;
                            g[3] = gc1 * h.X; g[4] = gc1 * h.Y; g[5] = gc1;
                            g[6] = gc2 * h.X; g[7] = gc2 * h.Y; g[8] = gc2;
                        }
                    }
                    T = Tj;
                }
                if (feat) reinterpret_cast<float*>(G.w[par])[lane] = wf;
                if constexpr (VAR) reduce_scatter<16>(g);  // lane l holds value l >> 1
                else reduce_scatter13(g);
                const int slot = G.slot[buf][j];
                const bool slot_ok = in_bounds(a.st, SITE_SLOT, slot, P.N);
                if ((lane & 1) == 0 && (lane >> 1) < (VAR ? 15 : 13) && slot_ok)
                    atomicAdd(grows + (int64_t)slot * GRAD_STRIDE + (lane >> 1), g[0]);
                if (!feat) continue;
                // w dL/dF: the sum over the lane's pixels, then over the pixel groups
                __syncwarp();
                float wp[PX], gf[4 * NQ];
                L::load_weights(reinterpret_cast<const float*>(G.w[par]) + pg * PX, wp);
                par ^= 1;
                {
                    float2 sum[NQ][2];
#pragma unroll
                    for (int q = 0; q < NQ; ++q) sum[q][0] = sum[q][1] = make_float2(0.0f, 0.0f);
                    auto pixels = [&](auto select) {
#pragma unroll
                        for (int p = 0; p < PX; ++p) {
                            if (decltype(select)::value && __float_as_uint(wp[p]) == 0x80000000u) continue;
#pragma unroll
                            for (int q = 0; q < NQ; ++q)
#pragma unroll
                                for (int k = 0; k < 2; ++k)
                                    sum[q][k] = __ffma2_rn(make_float2(wp[p], wp[p]), df[p][q][k], sum[q][k]);
                        }
                    };
                    if (careful) pixels(std::true_type{});
                    else pixels(std::false_type{});
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        gf[4 * q] = sum[q][0].x;
                        gf[4 * q + 1] = sum[q][0].y;
                        gf[4 * q + 2] = sum[q][1].x;
                        gf[4 * q + 3] = sum[q][1].y;
                    }
                }
                int n = 4 * NQ;
#pragma unroll
                for (int o = 16; o >= CL; o >>= 1) {
                    if (n > 1) {
                        const bool up = (lane & o) != 0;
#pragma unroll
                        for (int i = 0; i < 2 * NQ; ++i) {
                            if (i < n / 2) {
                                const float send = up ? gf[i] : gf[i + n / 2];
                                const float keep = up ? gf[i + n / 2] : gf[i];
                                gf[i] = keep + __shfl_xor_sync(ALL, send, o);
                            }
                        }
                        n >>= 1;
                    } else {
                        gf[0] += __shfl_xor_sync(ALL, gf[0], o);
                    }
                }
                // the lane's NQ sums are those of its values (lane >> 3) NQ on, consecutive channels
                const int v0 = (lane >> 3) * NQ, c = 4 * (cl + CL * (v0 >> 2)) + (v0 & 3);
                if (c < C && slot_ok && (CL == 8 || (lane & 4) == 0)) {
                    float* dst = a.feat_acc + (int64_t)slot * C + c;
                    if constexpr (NQ == 4) red_add_v4(dst, gf[0], gf[1], gf[2], gf[3]);
                    else if constexpr (NQ == 2) red_add_v2(dst, gf[0], gf[1]);
                    else atomicAdd(dst, gf[0]);
                }
            }
            word = next;
            __syncwarp();  // every lane has read this half before the next copies into it
        }
        cp_async_wait_all();
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// k_bwd_project: per surfel, d(adjugate rows) -> d(means, scales, quats)
// ---------------------------------------------------------------------------
// gradients of surfel s from its slot's per-view rows (slot < 0: zeros).
// VAR instances carry the variants, read from the parameters:
//  - spherical-harmonic colours: each view's colour gradient goes to the
//    coefficients (g_rgb [N, B, 3], accumulated in place by the surfel's own
//    thread) and, through the view direction d = (p - o) / |p - o|, to the
//    means: dd/dp = (I - d d^T) / |p - o|; a clamped channel passes nothing;
//  - low-pass filter: the rows' projected-centre gradient (entries 13, 14)
//    goes to the means through xc = fx pc_x / pc_z + cx, yc = fy pc_y / pc_z + cy.
template <bool VAR>
__device__ __forceinline__ void project_grad(const Cams& cams, const RParams& P, const BwdArgs& a, const float* sh,
                                             int64_t s, int slot) {
    float gm[3] = {0, 0, 0}, gs[2] = {0, 0}, gq[4] = {0, 0, 0, 0}, go = 0.0f, gc[3] = {0, 0, 0};
    const int nb = (P.sh_deg + 1) * (P.sh_deg + 1);
    const bool SH = VAR && P.color_sh;
    float* gsh = SH && a.g_rgb ? a.g_rgb + s * nb * 3 : nullptr;  // zeroed before the launch
    if (slot >= 0) {
        const float q0 = a.quats[4 * s], q1 = a.quats[4 * s + 1], q2 = a.quats[4 * s + 2], q3 = a.quats[4 * s + 3];
        const float qn = sqrtf(q0 * q0 + q1 * q1 + q2 * q2 + q3 * q3);
        const float w = q0 / qn, x = q1 / qn, y = q2 / qn, z = q3 / qn;
        const float tu[3] = {1.f - 2.f * (y * y + z * z), 2.f * (x * y + w * z), 2.f * (x * z - w * y)};
        const float tv[3] = {2.f * (x * y - w * z), 1.f - 2.f * (x * x + z * z), 2.f * (y * z + w * x)};
        const float su = a.scales[2 * s], sv = a.scales[2 * s + 1];
        const float pm[3] = {a.means[3 * s], a.means[3 * s + 1], a.means[3 * s + 2]};
        float dtu[3] = {0, 0, 0}, dtv[3] = {0, 0, 0};
        for (int v = 0; v < cams.n; ++v) {
            const float* gv = a.grad_item + ((int64_t)v * P.N + slot) * GRAD_STRIDE;
            const float4 g0 = *reinterpret_cast<const float4*>(gv);
            const float4 g1 = *reinterpret_cast<const float4*>(gv + 4);
            const float4 g2 = *reinterpret_cast<const float4*>(gv + 8);
            const float g12 = gv[12];
            go += g2.y;
            gc[0] += g2.z; gc[1] += g2.w; gc[2] += g12;
            if (SH && (g2.z != 0.f || g2.w != 0.f || g12 != 0.f)) {
                float ox, oy, oz;
                cam_centre(cams.c[v], ox, oy, oz);
                const float vx = a.means[3 * s] - ox, vy = a.means[3 * s + 1] - oy, vz = a.means[3 * s + 2] - oz;
                const float ir = rsqrtf(vx * vx + vy * vy + vz * vz);
                const float dx = vx * ir, dy = vy * ir, dz = vz * ir;
                float Y[16];
                sh_basis(P.sh_deg, dx, dy, dz, Y);
                const float* k = sh + s * nb * 3;
                float gd[3] = {0.f, 0.f, 0.f};
                for (int ch = 0; ch < 3; ++ch) {
                    const float g = ch == 0 ? g2.z : (ch == 1 ? g2.w : g12);
                    float c = 0.5f;
                    for (int b = 0; b < nb; ++b) c = fmaf(k[3 * b + ch], Y[b], c);
                    if (!(c > 0.0f) || g == 0.0f) continue;
                    if (gsh)
                        for (int b = 0; b < nb; ++b) gsh[3 * b + ch] = fmaf(Y[b], g, gsh[3 * b + ch]);
                    float gx, gy, gz;
                    sh_grad_dot(P.sh_deg, dx, dy, dz, k + ch, 3, gx, gy, gz);
                    gd[0] = fmaf(g, gx, gd[0]);
                    gd[1] = fmaf(g, gy, gd[1]);
                    gd[2] = fmaf(g, gz, gd[2]);
                }
                const float dd = dx * gd[0] + dy * gd[1] + dz * gd[2];
                gm[0] += (gd[0] - dx * dd) * ir;
                gm[1] += (gd[1] - dy * dd) * ir;
                gm[2] += (gd[2] - dz * dd) * ir;
            }
            const CamDev& cam = cams.c[v];
            if (VAR && P.lowpass && (gv[13] != 0.f || gv[14] != 0.f)) {
                float pc[3];
#pragma unroll
                for (int r = 0; r < 3; ++r)
                    pc[r] = cam.R[3 * r] * pm[0] + cam.R[3 * r + 1] * pm[1] + cam.R[3 * r + 2] * pm[2] + cam.t[r];
                const float iz = 1.0f / pc[2], gx = gv[13] * cam.fx * iz, gy = gv[14] * cam.fy * iz;
                const float dpc[3] = {gx, gy, -(gx * pc[0] + gy * pc[1]) * iz};
#pragma unroll
                for (int k = 0; k < 3; ++k) gm[k] += cam.R[k] * dpc[0] + cam.R[3 + k] * dpc[1] + cam.R[6 + k] * dpc[2];
            }
            if (g0.x == 0.f && g0.y == 0.f && g0.z == 0.f && g0.w == 0.f && g1.x == 0.f && g1.y == 0.f &&
                g1.z == 0.f && g1.w == 0.f && g2.x == 0.f)
                continue;
            const float4 r0 = a.rec[4 * ((int64_t)v * P.N + s)], r1 = a.rec[4 * ((int64_t)v * P.N + s) + 1];
            const float4 r3 = a.rec[4 * ((int64_t)v * P.N + s) + 3];
            const float xc = r0.w, yc = r1.w, sc = r3.w;
            // gradient of the unshifted adjugate: sc * G S^T
            const float G[3][3] = {{g0.x, g0.y, g0.z}, {g0.w, g1.x, g1.y}, {g1.z, g1.w, g2.x}};
            float gA[3][3];
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                gA[r][0] = sc * (G[r][0] + xc * G[r][2]);
                gA[r][1] = sc * (G[r][1] + yc * G[r][2]);
                gA[r][2] = sc * G[r][2];
            }
            // homography columns c0 = K Rv r_u t_u, c1 = K Rv r_v t_v, c2 = K (Rv p + t)
            float eu[3], ev[3], pc[3];
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                eu[r] = cam.R[3 * r] * tu[0] + cam.R[3 * r + 1] * tu[1] + cam.R[3 * r + 2] * tu[2];
                ev[r] = cam.R[3 * r] * tv[0] + cam.R[3 * r + 1] * tv[1] + cam.R[3 * r + 2] * tv[2];
                pc[r] = cam.R[3 * r] * pm[0] + cam.R[3 * r + 1] * pm[1] + cam.R[3 * r + 2] * pm[2] + cam.t[r];
            }
            float c[3][3];
            const float src[3][3] = {{su * eu[0], su * eu[1], su * eu[2]}, {sv * ev[0], sv * ev[1], sv * ev[2]},
                                     {pc[0], pc[1], pc[2]}};
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                c[j][0] = cam.fx * src[j][0] + cam.cx * src[j][2];
                c[j][1] = cam.fy * src[j][1] + cam.cy * src[j][2];
                c[j][2] = src[j][2];
            }
            // adjugate rows a0 = c1 x c2, a1 = c2 x c0, a2 = c0 x c1;
            // d/dp (p x q).g = q x g, d/dq (p x q).g = g x p
            auto cross = [](const float* p, const float* q, float* o) {
                o[0] = p[1] * q[2] - p[2] * q[1];
                o[1] = p[2] * q[0] - p[0] * q[2];
                o[2] = p[0] * q[1] - p[1] * q[0];
            };
            float dc[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}}, tmp[3];
            cross(c[2], gA[0], tmp); for (int k = 0; k < 3; ++k) dc[1][k] += tmp[k];
            cross(gA[0], c[1], tmp); for (int k = 0; k < 3; ++k) dc[2][k] += tmp[k];
            cross(c[0], gA[1], tmp); for (int k = 0; k < 3; ++k) dc[2][k] += tmp[k];
            cross(gA[1], c[2], tmp); for (int k = 0; k < 3; ++k) dc[0][k] += tmp[k];
            cross(c[1], gA[2], tmp); for (int k = 0; k < 3; ++k) dc[0][k] += tmp[k];
            cross(gA[2], c[0], tmp); for (int k = 0; k < 3; ++k) dc[1][k] += tmp[k];
            // columns -> camera-space vectors (K^T), then world (Rv^T)
            float da[3][3];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                da[j][0] = cam.fx * dc[j][0];
                da[j][1] = cam.fy * dc[j][1];
                da[j][2] = cam.cx * dc[j][0] + cam.cy * dc[j][1] + dc[j][2];
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float rtu = cam.R[k] * da[0][0] + cam.R[3 + k] * da[0][1] + cam.R[6 + k] * da[0][2];
                const float rtv = cam.R[k] * da[1][0] + cam.R[3 + k] * da[1][1] + cam.R[6 + k] * da[1][2];
                gm[k] += cam.R[k] * da[2][0] + cam.R[3 + k] * da[2][1] + cam.R[6 + k] * da[2][2];
                dtu[k] += su * rtu;
                dtv[k] += sv * rtv;
            }
            gs[0] += eu[0] * da[0][0] + eu[1] * da[0][1] + eu[2] * da[0][2];
            gs[1] += ev[0] * da[1][0] + ev[1] * da[1][1] + ev[2] * da[1][2];
        }
        // t_u, t_v -> normalised quaternion -> raw quaternion
        const float Ju[4][3] = {{0, 2 * z, -2 * y}, {0, 2 * y, 2 * z}, {-4 * y, 2 * x, -2 * w}, {-4 * z, 2 * w, 2 * x}};
        const float Jv[4][3] = {{-2 * z, 0, 2 * x}, {2 * y, -4 * x, 2 * w}, {2 * x, 0, 2 * z}, {-2 * w, -4 * z, 2 * y}};
        float dqh[4];
        const float qh[4] = {w, x, y, z};
        float dot = 0.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            dqh[k] = Ju[k][0] * dtu[0] + Ju[k][1] * dtu[1] + Ju[k][2] * dtu[2] + Jv[k][0] * dtv[0] +
                     Jv[k][1] * dtv[1] + Jv[k][2] * dtv[2];
            dot += dqh[k] * qh[k];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) gq[k] = (dqh[k] - dot * qh[k]) / qn;
    }
    if (a.g_means) { a.g_means[3 * s] = gm[0]; a.g_means[3 * s + 1] = gm[1]; a.g_means[3 * s + 2] = gm[2]; }
    if (a.g_scales) { a.g_scales[2 * s] = gs[0]; a.g_scales[2 * s + 1] = gs[1]; }
    if (a.g_quats) for (int k = 0; k < 4; ++k) a.g_quats[4 * s + k] = gq[k];
    if (a.g_opac) a.g_opac[s] = go;
    if (!(VAR && P.color_sh) && a.g_rgb) { a.g_rgb[3 * s] = gc[0]; a.g_rgb[3 * s + 1] = gc[1]; a.g_rgb[3 * s + 2] = gc[2]; }
}

// Zeros for surfels culled in every view (one thread each), then the chain
// rule for the surfels that have a slot, densely over the slots (a few
// percent of the surfels are visible, so a thread per surfel would leave
// most lanes of a warp idle through the long path).
template <bool VAR>
__global__ void __launch_bounds__(256) k_bwd_project(const __grid_constant__ Cams cams, const __grid_constant__ RParams P,
                                                     const BwdArgs a, const float* __restrict__ sh) {
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t gstride = (int64_t)gridDim.x * blockDim.x;
    const bool err = a.st->err != 0;
    for (int64_t s = gtid; s < P.N; s += gstride)
        if (err || a.splat_slot[s] < 0) project_grad<VAR>(cams, P, a, sh, s, -1);
    int64_t ns = err ? 0 : (int64_t)a.st->nslot;
    if (ns > 0 && !in_bounds(a.st, SITE_SLOT, ns - 1, P.N)) ns = 0;
    for (int64_t sl = gtid; sl < ns; sl += gstride) {
        const int32_t s = a.slot_surf[sl];
        if (in_bounds(a.st, SITE_SLOT, s, P.N)) project_grad<VAR>(cams, P, a, sh, s, (int)sl);
    }
}

// ---------------------------------------------------------------------------
// k_feat_out: g_feat[s] = slot >= 0 ? feat_acc[slot] : 0 (16-byte chunks)
// ---------------------------------------------------------------------------
template <typename FT>
__global__ void __launch_bounds__(256) k_feat_out(const __grid_constant__ RParams P, const BwdArgs a) {
    constexpr int E = FeatVec<FT>::E;
    const int nvec = P.C / E;
    const int64_t total = P.N * nvec;
    const bool err = a.st->err != 0;
    const bool pow2 = (nvec & (nvec - 1)) == 0;  // the usual widths: a shift instead of a 64-bit division
    const int sh = __ffs(nvec) - 1;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t s = pow2 ? (i >> sh) : i / nvec;
        const int vv = (int)(i - s * nvec);
        int slot = err ? -1 : a.splat_slot[s];
        if (slot >= 0 && !in_bounds(a.st, SITE_SLOT, slot, P.N)) slot = -1;
        float v[E];
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = 0.0f;
        if (slot >= 0) {
            const float4* src = reinterpret_cast<const float4*>(a.feat_acc + (int64_t)slot * P.C + vv * E);
#pragma unroll
            for (int k = 0; k < E / 4; ++k) {
                const float4 q = src[k];
                v[4 * k] = q.x; v[4 * k + 1] = q.y; v[4 * k + 2] = q.z; v[4 * k + 3] = q.w;
            }
        }
        store_vec<E>(a.g_feat, s * P.C + vv * E, v, P.feat_dtype);
    }
}

// zero the gradient slots in use: grad rows (all views) and feature rows
__global__ void __launch_bounds__(256) k_bwd_clear(const __grid_constant__ Cams cams, const __grid_constant__ RParams P,
                                                   const BwdArgs a) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.st->work_feat = 0u;
        a.st->work_geo = 0u;
    }
    int64_t ns = a.st->nslot;
    if (ns > 0 && !in_bounds(a.st, SITE_SLOT, ns - 1, P.N)) ns = 0;
    const int64_t g4 = ns * (GRAD_STRIDE / 4);
    const int64_t f4 = ns * (P.C / 4);
    const int64_t total = g4 * cams.n + f4;
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        if (i < g4 * cams.n) {
            const int64_t v = cams.n == 1 ? 0 : i / g4, r = i - v * g4;
            reinterpret_cast<float4*>(a.grad_item + v * P.N * GRAD_STRIDE)[r] = z;
        } else {
            reinterpret_cast<float4*>(a.feat_acc)[i - g4 * cams.n] = z;
        }
    }
}

// ---------------------------------------------------------------------------
// launcher
// ---------------------------------------------------------------------------
namespace {

// (the 48 KB that need no attribute include the kernel's static shared memory, under 1 KB)
cudaError_t set_smem(const void* k, size_t smem) { return smem + 1024 > 48 * 1024 ? open_smem(k) : cudaSuccess; }

// one resident wave: CTAs per SM times SMs, capped by the number of tiles
cudaError_t persistent_grid(const void* k, int threads, size_t smem, int& grid) {
    int per_sm = 0, dev = 0, sms = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, smem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    grid = std::max(1, std::min(grid, std::max(1, per_sm) * sms));
    return cudaSuccess;
}

template <typename FT>
cudaError_t launch_feat(const Cams& cams, const RParams& P, const BwdArgs& a, cudaStream_t s) {
    const int nvec = P.C / FeatVec<FT>::E;
    int G = 1;  // lanes per entry: 16-byte chunks of a feature row, padded to a power of two
    while (G < nvec) G <<= 1;
    if (G > 32) return cudaErrorInvalidValue;  // C too large (checked by the ABI)
    const int rowe = P.C + 16 / (int)sizeof(FT);  // padded row, elements
    const size_t rowb = (size_t)rowe * sizeof(FT);
    const int ucap = (int)(FEAT_UNION_BYTES / rowb);  // feature rows per pass
    // row passes per chunk: ceil(U / ucap), U <= ECAP (every slot has an entry)
    if (ucap < 1 || (ECAP + ucap - 1) / ucap > MAX_ROW_PASSES) return cudaErrorInvalidValue;
    const int npx = P.ts * P.ts;
    int pch = std::min(npx, ECAP / std::max(1, P.K));
    pch = (int)std::min<size_t>((size_t)pch, std::max<size_t>(32, (24 * 1024) / rowb));
    const size_t smem = (((size_t)(pch + zero_rows(G, (int)rowb)) * rowb + 15) & ~(size_t)15) + (size_t)4 * ECAP * 4 +
                        (size_t)2 * ECAP +
                        (size_t)((ucap + 3) & ~3) * 4 + FEAT_UNION_BYTES;
    auto go = [&](auto kern) {
        cudaError_t e2 = set_smem((const void*)kern, smem);
        if (e2 != cudaSuccess) return e2;
        int grid = cams.total_tiles;
        if (a.persistent && (e2 = persistent_grid((const void*)kern, BWD_FEAT_THREADS, smem, grid)) != cudaSuccess)
            return e2;
        kern<<<grid, BWD_FEAT_THREADS, smem, s>>>(cams, P, a, pch, rowe, ucap);
        e2 = cudaGetLastError();
        if (e2 == cudaSuccess) kernel_mark(s);
        return e2;
    };
    switch (G) {
        case 1: return go(k_bwd_feat<FT, 1>);
        case 2: return go(k_bwd_feat<FT, 2>);
        case 4: return go(k_bwd_feat<FT, 4>);
        case 8: return go(k_bwd_feat<FT, 8>);
        case 16: return go(k_bwd_feat<FT, 16>);
        default: return go(k_bwd_feat<FT, 32>);
    }
}

template <int TS, int CMAX, typename FT, bool VAR, bool TOPK = false>
cudaError_t launch_geo_full(const Cams& cams, const RParams& P, const BwdArgs& a, cudaStream_t s) {
    constexpr int NT = full_threads<TS>();
    int64_t units = (int64_t)cams.total_tiles * (TS * TS / NT);
    if (a.persistent) {
        int wave = (int)std::min<int64_t>(units, INT_MAX);
        const cudaError_t e = persistent_grid((const void*)k_bwd_geo_full<TS, CMAX, FT, VAR, TOPK>, NT, 0, wave);
        if (e != cudaSuccess) return e;
        units = wave;
    }
    k_bwd_geo_full<TS, CMAX, FT, VAR, TOPK><<<(unsigned)units, NT, 0, s>>>(cams, P, a);
    const cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) kernel_mark(s);
    return e;
}

// Who takes the feature gradients of a Top-K backward.  The feature kernel's work
// grows with K, the replay kernels' little, and theirs does not shrink with BF16 as the
// feature kernel's does.  Training steps, us, feature kernel / replay:
// k_bwd_geo_topk (16 and, BF16, 32 channels), 640 x 480: 16 channels FP32 K = 8 196 /
//   187 (but the feature rows then no longer run beside the replay when launched
//   eagerly: level), K = 9 242 / 222, K = 32 401 / 300; 32 channels BF16 K = 8 207 /
//   215, K = 9 254 / 247, K = 32 425 / 327.
// k_bwd_geo_full (instances of 32, 64 and 128 channels, whose cost does not fall with fewer):
//   640 x 480 FP32: 64 channels K = 4 268 / 244, K = 8 307 / 264, K = 32 568 / 420; 128
//   channels K = 8 463 / 395, K = 32 798 / 634, but 72 channels K = 4 345 / 368; BF16 64
//   channels K = 8 243 / 249, K = 24 434 / 351, but 128 channels K = 16 464 / 473.  With
//   more and smaller surfels (800k, 1280 x 720, exact stop): FP32 40 channels K = 4 691 /
//   711, 64 K = 4 776 / 762 (640 x 360, tiles of 8: 349 / 353), K = 8 955 / 906, 72 K = 8
//   1154 / 1219 (K = 16 605 / 628), 112 K = 12 1845 / 1775; BF16 64 K = 16 1249 / 1285, 48 K = 24 1722 / 1621.  So by channels x K.  Against
//   k_bwd_geo_topk: FP32 32 channels K = 24 337 / 303, 24 K = 12 985 / 960, 16 channels
//   level; BF16 16 channels 248 / 261, 32 298 / 288 but on small images 220 / 241.
//   A warp on its own has a long chain per surfel: with few 8 x 4 blocks an SM the feature
//   kernel's more threads are ahead (tiles of 8: 128 x 128, 64 channels K = 8 FP32 172 /
//   188, 200 x 150 117 / 116; of 16: 64 x 48 533 / 548, 128 x 128 FP32 197 / 189, BF16
//   183 / 199; of 32: 128 x 128 443 / 334).
// Neither with a renormalised selection, which needs every dot before the first, nor with
// the other variants.
enum FeatPath { FEAT_KERNEL, FEAT_REPLAY, FEAT_REPLAY_TWO, FEAT_PRODUCTS };
FeatPath feat_path(const Cams& cams, const RParams& P, int num_sms) {
    if (P.K == 0 || P.renorm || P.color_sh || P.lowpass) return FEAT_KERNEL;
    const bool half = P.feat_dtype == FSS_BF16;
    const int64_t blocks = (int64_t)cams.total_tiles * (P.ts * P.ts / 32);
    if (P.K > 8 && P.C <= 16) return blocks >= (int64_t)num_sms * 48 ? FEAT_REPLAY_TWO : FEAT_REPLAY;
    if (P.K > 8 && P.C <= 32 && half) return FEAT_REPLAY;
    if (blocks >= (int64_t)num_sms * (P.ts == 8 ? 8 : P.ts == 16 ? (half ? 4 : 2) : 0) &&
        (half ? P.C > 32 && P.C <= 64 && P.C * P.K >= 1152
              : P.C > 16 && P.C <= 128 && P.C * P.K >= (P.C <= 64 ? 288 : 1200) && (P.C > 32 || P.K > 8)))
        return FEAT_PRODUCTS;
    return P.K > 8 && P.C <= 32 ? FEAT_REPLAY : FEAT_KERNEL;
}

template <int TS, typename FT>
cudaError_t launch_geo_topk(const Cams& cams, const RParams& P, const BwdArgs& a, FeatPath feat, cudaStream_t s) {
    auto go = [&](auto kern, int nt, int h = 1) {
        int64_t units = (int64_t)cams.total_tiles * (TS * TS / h / nt);
        if (a.persistent) {
            int wave = (int)std::min<int64_t>(units, INT_MAX);
            const cudaError_t e = persistent_grid((const void*)kern, nt, 0, wave);
            if (e != cudaSuccess) return e;
            units = wave;
        }
        kern<<<(unsigned)units, nt, 0, s>>>(cams, P, a);
        const cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) kernel_mark(s);
        return e;
    };
    if (feat == FEAT_PRODUCTS) {
        if (P.C <= 32) {
            if constexpr (sizeof(FT) == 4) return launch_geo_full<TS, 32, FT, false, true>(cams, P, a, s);
        }
        if (P.C <= 64) return launch_geo_full<TS, 64, FT, false, true>(cams, P, a, s);
        if constexpr (sizeof(FT) == 4) return launch_geo_full<TS, 128, FT, false, true>(cams, P, a, s);
    }
    if (feat != FEAT_KERNEL) {
        if (feat == FEAT_REPLAY_TWO) return go(k_bwd_geo_topk<TS, false, 16, FT, 2>, geo_threads<TS, 16, FT, 2>(), 2);
        return P.C <= 16 ? go(k_bwd_geo_topk<TS, false, 16, FT>, geo_threads<TS, 16, FT, 1>())
                         : go(k_bwd_geo_topk<TS, false, 32, FT>, geo_threads<TS, 32, FT, 1>());
    }
    if (P.renorm || P.color_sh || P.lowpass) return go(k_bwd_geo_topk<TS, true>, geo_threads<TS, 0, float, 1>());
    return go(k_bwd_geo_topk<TS, false>, geo_threads<TS, 0, float, 1>());
}

template <int TS, typename FT>
cudaError_t launch_geo(const Cams& cams, const RParams& P, const BwdArgs& a, FeatPath feat, cudaStream_t s) {
    // the variants (renormalised Top-K, spherical-harmonic colours, low-pass
    // filter) have their own instances: no cost on the plain paths
    if (P.K > 0) return launch_geo_topk<TS, FT>(cams, P, a, feat, s);
    const bool var = P.color_sh || P.lowpass;
    if (P.C <= 16) return var ? launch_geo_full<TS, 16, FT, true>(cams, P, a, s) : launch_geo_full<TS, 16, FT, false>(cams, P, a, s);
    if (P.C <= 32) return var ? launch_geo_full<TS, 32, FT, true>(cams, P, a, s) : launch_geo_full<TS, 32, FT, false>(cams, P, a, s);
    if (P.C <= 64) return var ? launch_geo_full<TS, 64, FT, true>(cams, P, a, s) : launch_geo_full<TS, 64, FT, false>(cams, P, a, s);
    return var ? launch_geo_full<TS, 128, FT, true>(cams, P, a, s) : launch_geo_full<TS, 128, FT, false>(cams, P, a, s);
}

template <typename FT>
cudaError_t launch_all(const Cams& cams, const RParams& P, const BwdArgs& a, const float* sh, int num_sms,
                       cudaStream_t s) {
    cudaError_t e;
    k_bwd_clear<<<num_sms * 4, 256, 0, s>>>(cams, P, a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    kernel_mark(s);
    const FeatPath feat = feat_path(cams, P, num_sms);
    if (P.K > 0 && feat != FEAT_KERNEL) {
        kernel_mark(s);  // the feature gradients' place among the events: nothing runs there
    } else if (P.K > 0) {
        if ((e = launch_feat<FT>(cams, P, a, s)) != cudaSuccess) return e;
    }
    // Once the feature gradients are complete their output pass (memory bound)
    // runs in a second stream, launched eagerly, beside the geometry replay
    // (issue bound; 10 us less per 500k-surfel frame of 64 channels) or, where the
    // replay took them, beside the projection (4 us), and joins before the call
    // returns.  Below 48 MB of rows it costs the host more than it saves (four
    // calls, 10 us: autograd steps that the host bounds, 100k surfels 407 -> 399
    // us without it, 300k 421 -> 413; 1296 x 968 with 32 MB 1032 -> 1035).  A graph
    // being captured keeps one stream: replayed, the branch measured 3 us slower
    // than the chain.
    constexpr int64_t FORK_BYTES = 48 << 20;
    cudaStream_t side = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if ((e = cudaStreamIsCapturing(s, &cap)) != cudaSuccess) return e;
    const bool fork = a.g_feat && P.N * P.C * (int64_t)sizeof(FT) >= FORK_BYTES && cap == cudaStreamCaptureStatusNone && !kernel_marks_armed() &&
                      side_stream(s, side, ev_fork, ev_join);
    bool forked = false;
    auto rows_beside = [&]() {
        if ((e = cudaEventRecord(ev_fork, s)) != cudaSuccess) return e;
        if ((e = cudaStreamWaitEvent(side, ev_fork, 0)) != cudaSuccess) return e;
        k_feat_out<FT><<<num_sms * 8, 256, 0, side>>>(P, a);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if ((e = cudaEventRecord(ev_join, side)) != cudaSuccess) {
            (void)cudaStreamSynchronize(side);  // no join event: wait for the side stream's kernel here
            return e;
        }
        forked = true;
        return e;
    };
    const bool before = P.K > 0 && feat == FEAT_KERNEL;  // complete before the replay
    if (fork && before && (e = rows_beside()) != cudaSuccess) return e;
    // from here on every return joins the side stream first, so that no work of
    // this call is left running after it returns, even on an error
    auto joined = [&](cudaError_t err) {
        if (forked) {
            const cudaError_t ej = cudaStreamWaitEvent(s, ev_join, 0);
            if (err == cudaSuccess) err = ej;
        }
        return err;
    };
    if (P.ts == 8) e = launch_geo<8, FT>(cams, P, a, feat, s);
    else if (P.ts == 16) e = launch_geo<16, FT>(cams, P, a, feat, s);
    else e = launch_geo<32, FT>(cams, P, a, feat, s);
    if (e != cudaSuccess) return joined(e);
    if (fork && !before && (e = rows_beside()) != cudaSuccess) return e;
    const int64_t nb = (P.N + 255) / 256;
    // the coefficient gradients' zeros as one memset: written by each surfel's
    // thread, 4 bytes at a time and a row apart, they took 70 of the projection's
    // 90 us (300k surfels, degree 3); the visible surfels' threads add to them
    if (P.color_sh && a.g_rgb &&
        (e = cudaMemsetAsync(a.g_rgb, 0, (size_t)P.N * (P.sh_deg + 1) * (P.sh_deg + 1) * 12, s)) != cudaSuccess)
        return joined(e);
    if (P.color_sh || P.lowpass)
        k_bwd_project<true><<<(unsigned)std::max<int64_t>(1, nb), 256, 0, s>>>(cams, P, a, sh);
    else
        k_bwd_project<false><<<(unsigned)std::max<int64_t>(1, nb), 256, 0, s>>>(cams, P, a, nullptr);
    if ((e = cudaGetLastError()) != cudaSuccess) return joined(e);
    kernel_mark(s);
    if (fork) {
        if ((e = joined(cudaSuccess)) != cudaSuccess) return e;
    } else if (a.g_feat) {
        k_feat_out<FT><<<num_sms * 8, 256, 0, s>>>(P, a);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        kernel_mark(s);
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_render_backward(const Cams& cams, const RParams& P, const BwdArgs& a, const float* sh, int num_sms,
                                   cudaStream_t stream) {
    if (P.feat_dtype == FSS_BF16) return launch_all<__nv_bfloat16>(cams, P, a, sh, num_sms, stream);
    return launch_all<float>(cams, P, a, sh, num_sms, stream);
}

}  // namespace fss
