// Top-K forward render for K > 16 (variants: K > 8; included by one translation unit per
// feature type): the traversal, selection rule and outputs of render_topk.cuh,
// with the K-set of a pixel in shared memory instead of registers.
//
// Why: in registers a set of 32 slots takes 220 registers per thread, so one
// CTA of eight warps per SM, and every insertion runs a 32-slot compare-
// exchange chain (160 instructions) although most pixels meet little more
// than K contributors.  Here
//   - the set is two columns of shared memory per pixel (weight, list
//     position), filled in order: the first K contributors cost two stores;
//   - after that a weight enters only if it exceeds the smallest one, which
//     is kept in a register beside the minima of the groups of eight slots:
//     the new entry takes the smallest one's slot and one group is rescanned;
//   - slots that were refilled are marked: every refilled slot holds a later
//     list position than every other one, so the front-to-back order is the
//     unmarked slots in slot order, then the marked ones by position;
//   - a warp owns its 8 x 4 pixel block from the list to the stored features
//     and never waits for another warp (stage_chunk), so no barrier stalls
//     and a light block's warp does not wait for the tile's heaviest one;
//   - ids, positions and weights go out with consecutive lanes on
//     consecutive entries (a thread per pixel would write 4 K bytes apart).
// 1296 x 968, K = 24, C = 16 FP32, 500k surfels: 1400 us with the set in
// registers (8 warps per SM, 1.49 instructions per cycle), 558 us here (20
// warps, 2.04); now bound by the shared-memory path (76 % busy: four 16-byte
// record reads per evaluation, the set, three reads per selected row chunk).
#pragma once

#include "fss_internal.cuh"
#include "kernels.cuh"
#include "render_common.cuh"

#include <algorithm>
#include <climits>

namespace fss {

constexpr int WIDE_THREADS = 128;  // threads per CTA (64 for 8 x 8 tiles): parts of a tile

// shared memory of one warp: two staging halves, (AUX: normals and argmax
// keys,) the K-set, the selection's order and the pixels' counts
inline __host__ __device__ size_t wide_warp_smem(int K, bool aux) {
    return 2 * sizeof(WarpStage) + (aux ? 32 * (16 + 8) : 0) + (size_t)K * 32 * 8 + (size_t)((K * 32 + 15) & ~15) + 128;
}

// Which of several equal smallest weights leaves.  Sets of up to CHAIN_K entries follow the
// insertion chain of render_topk.cuh, which keeps those of the plain frames: the outputs
// asked for must not change the selection.  Larger sets drop the entry at the latest position.
//
// In the chain an insertion turns every run of equal smaller weights by one (its first entry
// goes behind its last: equal ones stay in their slots) and the last run loses its first.  So
// a run's order when its first entry leaves follows from the set as it is then: taken by
// position, an entry of the run joins it behind the others, a larger one turns it.  (Smaller ones have
// left, and larger ones cannot have.)  From then on entries only leave it, first to last, and
// none joins: a weight enters only above the smallest.  The order is formed once per run,
// into s_ord (free until the traversal ends; `tied` holds the run's weight), and the first of
// it that is still in the set leaves.  Ties are rare: none of this runs otherwise.
constexpr int CHAIN_K = 16;  // the largest set of render_topk.cuh
__device__ __forceinline__ int chain_leaver(const float* s_kw, const int32_t* s_kp, unsigned char* s_ord, int32_t* tied,
                                            int K, float wmin) {
    const int lane = threadIdx.x & 31;
    if (*tied != __float_as_int(wmin)) {
        *tied = __float_as_int(wmin);
        unsigned long long run = 0ull;  // its slots, first in the low bits, 4 bits each
        int n = 0;
        for (int i = 0, last = -1; i < K; ++i) {  // the entries by position
            int s = 0, at = INT_MAX;
            for (int j = 0; j < K; ++j) {
                const int p = s_kp[j * 32 + lane];
                if (p > last && p < at) {
                    at = p;
                    s = j;
                }
            }
            last = at;
            if (s_kw[s * 32 + lane] == wmin) run |= (unsigned long long)s << (4 * n++);
            else if (n > 1) run = (run >> 4) | ((run & 15ull) << (4 * (n - 1)));
        }
        for (int i = 0; i < K; ++i) s_ord[i * 32 + lane] = (unsigned char)((run >> (4 * i)) & 15ull);  // (zeros behind it)
    }
    int i = 0;  // (entries that have left hold larger weights now)
    while (i < K - 1 && s_kw[s_ord[i * 32 + lane] * 32 + lane] != wmin) ++i;
    return s_ord[i * 32 + lane];
}

// the minimum of group g takes w in (scalars: an indexed array would go to local memory)
__device__ __forceinline__ void group_min(int g, float w, float& m0, float& m1, float& m2, float& m3) {
    m0 = g == 0 ? fminf(m0, w) : m0;
    m1 = g == 1 ? fminf(m1, w) : m1;
    m2 = g == 2 ? fminf(m2, w) : m2;
    m3 = g == 3 ? fminf(m3, w) : m3;
}

template <int TS, typename FT, bool AUX>
__global__ void __launch_bounds__(TS * TS < WIDE_THREADS ? TS * TS : WIDE_THREADS) k_render_topk_wide(
    const __grid_constant__ Cams cams, const __grid_constant__ RParams P, const FwdArgs a,
    const __grid_constant__ AuxOut x) {
    constexpr int NT = TS * TS < WIDE_THREADS ? TS * TS : WIDE_THREADS;
    constexpr int PARTS = TS * TS / NT, WPP = NT / 32;
    constexpr unsigned ALL = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_work;
    if (a.st->err) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int K = P.K;
    const bool front = P.select == FSS_SELECT_FRONT;
    unsigned char* base = smem + warp * wide_warp_smem(K, AUX);
    WarpStage* s_st = reinterpret_cast<WarpStage*>(base);  // [2]
    float4* s_nrm = reinterpret_cast<float4*>(s_st + 2);   // AUX: [32] facing normals, centre depths
    unsigned long long* s_lab = reinterpret_cast<unsigned long long*>(s_nrm + 32);  // AUX: [32] argmax keys
    float* s_kw = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(s_st + 2) + (AUX ? 32 * 24 : 0));  // [K][32]
    int32_t* s_kp = reinterpret_cast<int32_t*>(s_kw + K * 32);           // [K][32] list positions, then surfel ids
    unsigned char* s_ord = reinterpret_cast<unsigned char*>(s_kp + K * 32);  // [K][32] rank -> slot
    int32_t* s_n = reinterpret_cast<int32_t*>(s_ord + ((K * 32 + 15) & ~15));  // [32] selected entries
    const FT* __restrict__ feats = reinterpret_cast<const FT*>(a.feats);
    constexpr int E = FeatVec<FT>::E;
    const int nvec = P.C / E;
    const FastDiv divK(K), divV(nvec);
    const int total = cams.total_tiles * PARTS;

    for (bool first = true;; first = false) {
        int u;  // this CTA's next part of a tile (heavy tiles first)
        if (!a.persistent) {
            u = first ? (int)blockIdx.x : INT_MAX;
        } else {
            __syncthreads();
            if (threadIdx.x == 0) s_work = (int)atomicAdd(&a.st->work, 1u);
            __syncthreads();
            u = s_work;
        }
        if (u >= total) return;
        const int t = cams.tile_order ? cams.tile_order[u / PARTS] : u / PARTS;
        const int wb = (u % PARTS) * WPP + warp;  // this warp's block of the tile
        const uint32_t wbit = 1u << wb;
        const int view = view_of_tile(cams, t);
        const CamDev& cam = cams.c[view];
        const int lt = t - cam.tile_off;
        const int tx = lt % cam.tiles_x, ty = lt / cam.tiles_x;
        const int2 lp = pixel_of<TS>(wb * 32 + lane);
        const int px = tx * TS + lp.x, py = ty * TS + lp.y;
        const bool inside = px < cam.W && py < cam.H;
        const float pxf = (float)px + 0.5f, pyf = (float)py + 0.5f;
        const int2 rg = checked_range(a.ranges, t, P.pair_cap, a.st);
        const int n = rg.y - rg.x;
        const int64_t vbase = (int64_t)view * P.N;
        const float* __restrict__ rgbv = a.rgb + (P.color_sh ? 3 * vbase : 0);  // SH: item colours
        const uint32_t* list = a.list + rg.x;
        const uint32_t* masks = a.masks + rg.x;

        float T = 1.0f, cr = 0.0f, cg = 0.0f, cb = 0.0f;
        bool done = !inside;
        int last = -1, n_sel = 0;
        uint32_t rep = 0u;                                      // refilled slots
        float gm0 = INFINITY, gm1 = INFINITY, gm2 = INFINITY, gm3 = INFINITY;  // minima of the slot groups
        float wmin = -INFINITY;                                 // smallest selected weight once K are selected
        if (AUX) s_n[lane] = -1;                                // until the outputs: chain_leaver's run (none yet: a NaN)
        uint32_t n_eval = 0, n_contrib = 0;
        float zs = 0.0f, zmed = 0.0f, nx = 0.0f, ny = 0.0f, nz = 0.0f;  // AUX sums
        bool med = false;

        // chunk i is worked on while chunk i + 1 is copied and the list entries of chunk i + 2 are read
        ListEntry e0 = list_entry(list, masks, lane, n), e1 = list_entry(list, masks, 32 + lane, n);
        uint32_t word = stage_chunk(s_st[0], e0, wbit, a.rec, rgbv, vbase, P.N, a.st);
        for (int b0 = 0; b0 < n; b0 += 32) {
            if (__all_sync(ALL, done)) break;
            const int buf = (b0 >> 5) & 1;
            const WarpStage& S = s_st[buf];
            const uint32_t next = stage_chunk(s_st[buf ^ 1], e1, wbit, a.rec, rgbv, vbase, P.N, a.st);
            e1 = list_entry(list, masks, b0 + 64 + lane, n);
            cp_async_wait_prev();  // this chunk's copies (the next one's stay in flight)
            __syncwarp();
            if (AUX) {  // facing normals, and the centre depths for the low-pass screen term
                if ((word >> lane) & 1u) {
                    const float4 nf = facing_normal(S.r2[lane], S.r0[lane].w, S.r1[lane].w, cam);
                    s_nrm[lane] = make_float4(nf.x, nf.y, nf.z, a.rec[4 * (size_t)list[b0 + lane] + 3].y);
                }
                __syncwarp();
            }
            if (!done) {
                for (uint32_t bits = word; bits != 0u; bits &= bits - 1u) {
                    const int j = __ffs(bits) - 1;
                    ++n_eval;
                    Hit h;
                    const float4 oc = S.oc[j];
                    if (!eval_splat<AUX>(S.r0[j], S.r1[j], S.r2[j], oc.x, pxf, pyf, P.alpha_min, cam.near_plane, h, P.lowpass))
                        continue;
                    const float alpha = fminf(h.alpha_raw, P.alpha_max);
                    const float Tn = T * (1.0f - alpha);
                    if (Tn < P.T_min) { done = true; break; }
                    const float w = alpha * T;
                    cr = fmaf(w, oc.y, cr);
                    cg = fmaf(w, oc.z, cg);
                    cb = fmaf(w, oc.w, cb);
                    ++n_contrib;
                    if (AUX) {
                        const float4 nv = s_nrm[j];
                        const float zh = h.scr ? nv.w : S.r2[j].w * h.inv;  // hit depth, as in the near-plane test
                        zs = fmaf(w, zh, zs);
                        nx = fmaf(w, nv.x, nx);
                        ny = fmaf(w, nv.y, ny);
                        nz = fmaf(w, nv.z, nz);
                        if (!med && Tn < 0.5f) { zmed = zh; med = true; }
                    }
                    if (n_sel < K) {
                        s_kw[n_sel * 32 + lane] = w;
                        s_kp[n_sel * 32 + lane] = b0 + j;
                        group_min(n_sel >> 3, w, gm0, gm1, gm2, gm3);
                        if (++n_sel == K) wmin = fminf(fminf(gm0, gm1), fminf(gm2, gm3));
                    } else if (w > wmin && !front) {
                        // the smallest entry's slot: in the one group whose minimum it is
                        const bool q0 = gm0 == wmin, q1 = gm1 == wmin, q2 = gm2 == wmin, q3 = gm3 == wmin;
                        const int g = q3 ? 3 : (q2 ? 2 : (q1 ? 1 : 0));
                        const int ng = (q0 ? 1 : 0) + (q1 ? 1 : 0) + (q2 ? 1 : 0) + (q3 ? 1 : 0);
                        int slot = 0, ns = 0;
                        float gn = w;  // the group's minimum with the new entry in the slot
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const int s = 8 * g + i;
                            const float v = s < K ? s_kw[s * 32 + lane] : INFINITY;
                            const bool is = v == wmin;
                            slot = is ? s : slot;
                            ns += is ? 1 : 0;
                            gn = is ? gn : fminf(gn, v);
                        }
                        if (ng + ns == 2) {
                            gm0 = g == 0 ? gn : gm0;
                            gm1 = g == 1 ? gn : gm1;
                            gm2 = g == 2 ? gn : gm2;
                            gm3 = g == 3 ? gn : gm3;
                            s_kw[slot * 32 + lane] = w;
                            s_kp[slot * 32 + lane] = b0 + j;
                        } else {  // equal weights (see chain_leaver)
                            if (AUX && K <= CHAIN_K) {
                                slot = chain_leaver(s_kw, s_kp, s_ord, s_n + lane, K, wmin);
                            } else {
                                int pl = -1;
                                for (int s = 0; s < K; ++s) {
                                    const int p = s_kp[s * 32 + lane];
                                    if (s_kw[s * 32 + lane] == wmin && p > pl) { pl = p; slot = s; }
                                }
                            }
                            s_kw[slot * 32 + lane] = w;
                            s_kp[slot * 32 + lane] = b0 + j;
                            gm0 = gm1 = gm2 = gm3 = INFINITY;
                            for (int s = 0; s < K; ++s) group_min(s >> 3, s_kw[s * 32 + lane], gm0, gm1, gm2, gm3);
                        }
                        rep |= 1u << slot;
                        wmin = fminf(fminf(gm0, gm1), fminf(gm2, gm3));
                    }
                    T = Tn;
                    last = b0 + j;
                    if (P.stop_rule == FSS_STOP_EXACT_TOPK && n_sel == K && (front || P.alpha_max * T <= wmin)) {
                        done = true;
                        break;
                    }
                }
            }
            word = next;
            __syncwarp();  // every lane has read this half before the next copies into it
        }
        cp_async_wait_all();
        __syncwarp();

        // per-pixel outputs; the selection's front-to-back order
        const uint32_t used = n_sel >= 32 ? ALL : (1u << n_sel) - 1u, orig = used & ~rep;
        for (int s = 0; s < n_sel; ++s) {
            int rank;
            if ((rep >> s) & 1u) {
                rank = __popc(orig);
                const int p = s_kp[s * 32 + lane];
                for (uint32_t m = rep; m != 0u; m &= m - 1u) rank += s_kp[(__ffs(m) - 1) * 32 + lane] < p ? 1 : 0;
            } else {
                rank = __popc(orig & ((1u << s) - 1u));
            }
            s_ord[rank * 32 + lane] = (unsigned char)s;
        }
        s_n[lane] = inside ? n_sel : 0;
        if (AUX) s_lab[lane] = 0ull;
        if (inside) {
            const int64_t pix = cam.pix_off + (int64_t)py * cam.W + px;
            if (a.out_rgb) {
                a.out_rgb[3 * pix] = fmaf(T, P.bg[0], cr);
                a.out_rgb[3 * pix + 1] = fmaf(T, P.bg[1], cg);
                a.out_rgb[3 * pix + 2] = fmaf(T, P.bg[2], cb);
            }
            if (a.out_T) a.out_T[pix] = T;
            if (a.saved_nstop) a.saved_nstop[pix] = last + 1;
            if (AUX) {
                if (x.depth) x.depth[pix] = zs;
                if (x.depth_med) x.depth_med[pix] = zmed;
                if (x.normal) {
                    x.normal[3 * pix] = nx;
                    x.normal[3 * pix + 1] = ny;
                    x.normal[3 * pix + 2] = nz;
                }
            }
        }
        __syncwarp();
        // the K entries of every pixel, consecutive lanes on consecutive entries of a block row (8 pixels)
        const int bx = tx * TS + 8 * (wb % (TS / 8)), by = ty * TS + 4 * (wb / (TS / 8));  // the block's first pixel
        for (int r = 0; r < 4 && by + r < cam.H; ++r) {
            const int64_t o0 = (cam.pix_off + (int64_t)(by + r) * cam.W + bx) * K;
            const int ne = min(8, cam.W - bx) * K;
            for (int e = lane; e < ne; e += 32) {
                const int c = divK.div(e), k = e - c * K, q = 8 * r + c;
                int pos = -1, id = -1;
                float w = 0.0f;
                if (k < s_n[q]) {
                    const int at = s_ord[k * 32 + q] * 32 + q;
                    pos = s_kp[at];
                    w = s_kw[at];
                    id = (int32_t)((int64_t)list[pos] - vbase);
                    s_kp[at] = id;  // for the feature gather below
                }
                if (a.out_ids) a.out_ids[o0 + e] = id;
                if (a.saved_pos) a.saved_pos[o0 + e] = pos;
                if (a.saved_w) a.saved_w[o0 + e] = w;
            }
        }
        __syncwarp();
        warp_count(&a.st->counters[0], n_eval);
        warp_count(&a.st->counters[1], n_contrib);

        // the selected feature rows, weighted in the selection's front-to-back order (AUX: and their argmax)
        if (a.out_feat || (AUX && x.label)) {
            if (P.renorm) {
                float ws = 0.0f;
                for (int s = 0; s < n_sel; ++s) ws += s_kw[s * 32 + lane];
                const float wsc = ws > 0.0f ? __frcp_rn(ws) : 0.0f;
                for (int s = 0; s < n_sel; ++s) s_kw[s * 32 + lane] *= wsc;
                __syncwarp();
            }
            for (int i = lane; i < 32 * nvec; i += 32) {
                const int q = divV.div(i), vv = i - q * nvec;  // pixel of the block, 16-byte chunk of the row
                const int qx = bx + (q & 7), qy = by + (q >> 3);
                if (qx >= cam.W || qy >= cam.H) continue;
                float2 acc2[E / 2];
#pragma unroll
                for (int e = 0; e < E / 2; ++e) acc2[e] = make_float2(0.0f, 0.0f);
                const int c = s_n[q];
                for (int k = 0; k < c; ++k) {
                    const int at = s_ord[k * 32 + q] * 32 + q;
                    const int id = s_kp[at];
                    const float w = s_kw[at];
                    if (!in_bounds(a.st, SITE_FEAT_ROW, id, P.N)) continue;
                    float2 f2[E / 2];
                    FeatVec<FT>::unpack2(FeatVec<FT>::raw(feats + (size_t)id * P.C + vv * E), f2);
                    const float2 w2 = make_float2(w, w);
#pragma unroll
                    for (int e = 0; e < E / 2; ++e) acc2[e] = __ffma2_rn(w2, f2[e], acc2[e]);
                }
                const int64_t qpix = cam.pix_off + (int64_t)qy * cam.W + qx;
                float acc[E];
#pragma unroll
                for (int e = 0; e < E / 2; ++e) {
                    acc[2 * e] = acc2[e].x;
                    acc[2 * e + 1] = acc2[e].y;
                }
                if (a.out_feat) store_vec<E>(a.out_feat, qpix * P.C + vv * E, acc, P.out_dtype);
                if (AUX && x.label) {
                    int eb = 0;
                    float bv = acc[0];
#pragma unroll
                    for (int e = 1; e < E; ++e) {
                        eb = acc[e] > bv ? e : eb;
                        bv = acc[e] > bv ? acc[e] : bv;
                    }
                    atomicMax(&s_lab[q], argmax_key(bv, vv * E + eb));
                }
            }
            if (AUX && x.label) {
                __syncwarp();
                if (inside)
                    x.label[cam.pix_off + (int64_t)py * cam.W + px] = s_n[lane] > 0 ? argmax_channel(s_lab[lane]) : -1;
            }
        }
        __syncwarp();  // before the warp's next block reuses its shared memory
    }
}

template <int TS, typename FT>
cudaError_t launch_topk_wide(const Cams& cams, const RParams& P, const FwdArgs& a, const AuxOut& x, int num_sms,
                             cudaStream_t s) {
    constexpr int NT = TS * TS < WIDE_THREADS ? TS * TS : WIDE_THREADS;
    constexpr int PARTS = TS * TS / NT;
    const bool aux = x.any() || P.lowpass;  // the variant instance also carries the low-pass filter
    const size_t smem = NT / 32 * wide_warp_smem(P.K, aux);
    return aux ? launch_tiles(k_render_topk_wide<TS, FT, true>, NT, smem, cams, P, a, x, num_sms, s, PARTS)
               : launch_tiles(k_render_topk_wide<TS, FT, false>, NT, smem, cams, P, a, x, num_sms, s, PARTS);
}

}  // namespace fss
