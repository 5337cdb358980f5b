// Top-K forward render (included by one translation unit per feature type,
// so that the two sets of template instances compile in parallel).
//
// Front-to-back alpha compositing of the depth-sorted tile lists (Sec. 3.1,
// Eq. 2) with Top-K Hard Selection before the C-channel feature
// accumulation (Sec. 3.4, Eq. 7).  One thread per pixel, one warp per 8 x 4
// pixel block; a warp goes from its tile's list to the stored features on its
// own, without waiting for the tile's other warps.
// Phase 1: the warp stages the records that its block meets 32 list positions
//   at a time (stage_chunk: asynchronous copies into its own double buffer);
//   every lane intersects its pixel ray with each staged surfel, composites
//   colour and transmittance and keeps its K largest blending weights in
//   registers (ties: see the K-set below).  The warp leaves the loop as
//   soon as all its pixels have stopped.
// Phase 2: the warp gathers only the K selected feature rows per pixel
//   (16-byte loads: 8 bf16 or 4 f32 channels), weights them in FP32 and writes
//   channel-last output with consecutive lanes on consecutive 16-byte chunks.
// It is bound by instruction issue (2.8 of 4 per cycle and SM; about 75 warp
// instructions per evaluation in phase 1 and 14 per selected row chunk in
// phase 2).  Staging by the whole CTA, 256 records at a time behind barriers,
// spent 1.4 to 2 cycles per issued instruction at the barriers and took 101 us
// for a 640 x 480 frame of 500k surfels (C = 64 FP32, K = 8) where this takes
// 93; with the sort and the loss (BF16) 108 against 102.
// Variants: FRONT takes the first K contributors instead of the K largest
// weights; AUX also accumulates the sensor outputs (expected and median
// depth, facing normal) over every contributor and applies the low-pass
// filter when the parameters ask for it; LOSS evaluates the training loss
// (L2 on the features, L1 on the colour) and its gradients where F and rgb
// are formed; SORT (with LOSS) first depth-sorts the CTA's own tile list
// (sort_tile), so that no sort kernel runs before it.
//
// The accumulation is a sparse gather-weighted sum, not a dense contraction,
// so no tensor cores are involved.
#pragma once

#include "fss_internal.cuh"
#include "kernels.cuh"
#include "render_common.cuh"
#include "render_topk_wide.cuh"
#include "sort.cuh"

#include <algorithm>
#include <climits>

namespace fss {

// ---------------------------------------------------------------------------
// Top-K kernel
// ---------------------------------------------------------------------------
// The K-set of a pixel lives in registers as an array sorted by decreasing
// weight.  A new weight x takes its place and each one behind it moves on by a slot:
// the weight carried into slot k is min(slot k - 1, x), known for all slots at once,
// and it stays there if it exceeds the slot's, so only the positions pass from slot
// to slot.  An equal weight in a slot stays and the carried one goes on behind it: a new
// weight never displaces an equal one, and of several equal smallest ones the first in the
// chain's order falls off, which need not be the latest (chain_leaver in render_topk_wide.cuh
// follows this for the variants' sets of the same size).  (Positions all at once as well, which drops
// another one of several equal smallest weights: 2 to 3 us less of a 640 x 480 frame,
// 9 of 423 at 1.5M surfels, 1280 x 720.)  For K < KCAP
// the first KCAP - K slots hold +inf and never move, so the K-th largest
// weight is always slot KCAP - 1.  With the first-K selection the K slots
// after the padding take the first K contributors in order.
//
// PAIR: the intersections of two surfels do not depend on each other, so the
// sets of 4 and 16 slots, which have the registers for it, start them together
// (1.2M surfels, 1280 x 720: K = 3 335 -> 327 us, K = 12 520 -> 488; 3,000 in
// 100 x 90: 97 -> 90 and 103 -> 97).  With 8 slots the 64 registers that 32
// resident warps leave make it slower (406 -> 427 us).
// Sets of 9 to 16 entries take 123 registers, 16 warps per SM, and are still
// ahead of the set in shared memory (render_topk_wide.cuh) throughout: K = 12
// above 488 us against 490, K = 16 with C = 48 561 / 630, small scenes 97 / 119.
//
// CTAs: TOPK_THREADS threads (parts of a tile), so that a block's registers
// are free for the next one soon after it ends; the SORT instances keep a
// tile's warps together, which sort its list first.
constexpr int TOPK_THREADS = 128;
template <int TS, bool SORT>
constexpr int topk_threads() {
    return SORT || TS * TS < TOPK_THREADS ? TS * TS : TOPK_THREADS;
}
// shared memory of one warp: the two staging halves, whose place the selected
// entries (32 rows of KCAP + 1 pairs) take afterwards, and (AUX) the normals
// and argmax keys
constexpr size_t topk_warp_smem(int kcap, bool aux) {
    const size_t stage = 2 * sizeof(WarpStage), sel = (size_t)32 * (kcap + 1) * 8 + 128;
    return (sel > stage ? sel : stage) + (aux ? 32 * (16 + 8) : 0);
}

template <int TS, int KCAP, typename FT, bool FRONT, bool AUX, bool LOSS = false, bool SORT = false>
__global__ void __launch_bounds__(topk_threads<TS, SORT>(), (KCAP <= 8 ? 1024 : 512) / topk_threads<TS, SORT>()) k_render_topk(
    const __grid_constant__ Cams cams, const __grid_constant__ RParams P, const FwdArgs a,
    const __grid_constant__ AuxOut x) {
    constexpr int NT = topk_threads<TS, SORT>(), NW = NT / 32, PARTS = TS * TS / NT;
    constexpr bool PAIR = KCAP != 8;  // two surfels' intersections at a time (see above)
    constexpr int ROW = KCAP + 1;  // padded row of a pixel's selected entries (bank conflicts)
    constexpr unsigned ALL = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_work;
    __shared__ float s_loss[LOSS ? NW : 1];  // LOSS: the warps' sums of a tile (part)
    __shared__ int s_arrived;                // ... and how many have arrived

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (a.st->err) return;
    unsigned char* base = smem + warp * topk_warp_smem(KCAP, AUX);
    WarpStage* s_st = reinterpret_cast<WarpStage*>(base);     // [2]
    float4* s_nrm = reinterpret_cast<float4*>(base + topk_warp_smem(KCAP, false));  // AUX: [32] facing normals, centre depths
    unsigned long long* s_lab = reinterpret_cast<unsigned long long*>(s_nrm + 32);    // AUX: [32] argmax keys
    int2* s_sel = reinterpret_cast<int2*>(base);              // phase 2: [32][ROW] (list position, then surfel id; weight)
    int32_t* s_n = reinterpret_cast<int32_t*>(s_sel + 32 * ROW);  // [32] selected entries
    const int K = P.K;
    const FT* __restrict__ feats = reinterpret_cast<const FT*>(a.feats);
    constexpr int E = FeatVec<FT>::E;
    const int nvec = P.C / E;
    const FastDiv divV(nvec);
    const int total = cams.total_tiles * PARTS;
    if (LOSS && threadIdx.x == 0) s_arrived = 0;
    if (LOSS && !SORT && !a.persistent) __syncthreads();
    for (bool first = true;; first = false) {
        int u;  // this CTA's next tile, or part of one (heavy tiles first)
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
        if constexpr (SORT) {  // this tile's depth sort first, in the staging area
            __syncthreads();   // (the previous tile's last reads of the area)
            sort_tile(cams, P, x.sort.binrec, a.ranges, x.sort.list, x.sort.unb_list, x.sort.scratch,
                      x.sort.masks, a.st, t, smem);
            __syncthreads();  // the sorted list and masks (global, written by this CTA) before staging
        }
        const int wb = (u % PARTS) * NW + warp;  // this warp's block of the tile
        const uint32_t wbit = 1u << wb;
        const int view = view_of_tile(cams, t);
        const CamDev& cam = cams.c[view];
        const int lt = t - cam.tile_off;
        const int tx = lt % cam.tiles_x, ty = lt / cam.tiles_x;
        const int bx = tx * TS + 8 * (wb % (TS / 8)), by = ty * TS + 4 * (wb / (TS / 8));  // the block's first pixel
        const int px = bx + (lane & 7), py = by + (lane >> 3);
        const bool inside = px < cam.W && py < cam.H;
        const float pxf = (float)px + 0.5f, pyf = (float)py + 0.5f;
        const int2 rg = checked_range(a.ranges, t, P.pair_cap, a.st);
        const int n = rg.y - rg.x;
        const int64_t vbase = (int64_t)view * P.N;
        const float* __restrict__ rgbv = a.rgb + (P.color_sh ? 3 * vbase : 0);  // SH: item colours
        const uint32_t* list = a.list + rg.x;
        const uint32_t* masks = a.masks + rg.x;
        if (LOSS && inside) {  // the pixel's targets, into L2 while phase 1 runs
            const int64_t pix = cam.pix_off + (int64_t)py * cam.W + px;
            const char* ft = reinterpret_cast<const char*>(x.loss.Ft) + pix * P.C * (int64_t)sizeof(FT);
            for (int off = 0; off < P.C * (int)sizeof(FT); off += 128)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(ft + off));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(x.loss.rgbt + 3 * pix));
        }

        float T = 1.0f, cr = 0.0f, cg = 0.0f, cb = 0.0f;
        bool done = !inside;
        int last = -1;
        float hw[KCAP];
        int hp[KCAP];
#pragma unroll
        for (int k = 0; k < KCAP; ++k) {
            hw[k] = k < KCAP - K ? INFINITY : -INFINITY;
            hp[k] = -1;
        }
        uint32_t n_eval = 0, n_contrib = 0;
        int n_sel = 0;  // FRONT: contributors taken so far
        float zs = 0.0f, zmed = 0.0f, nx = 0.0f, ny = 0.0f, nz = 0.0f;  // AUX sums
        bool med = false;

        // chunk i is worked on while chunk i + 1 is copied and the list entries of chunk i + 2 are read
        ListEntry e1 = list_entry(list, masks, lane, n);
        uint32_t word = stage_chunk(s_st[0], e1, wbit, a.rec, rgbv, vbase, P.N, a.st);
        e1 = list_entry(list, masks, 32 + lane, n);
        for (int b0 = 0; b0 < n; b0 += 32) {
            if (__all_sync(ALL, done)) break;
            const WarpStage& S = s_st[(b0 >> 5) & 1];
            const uint32_t next = stage_chunk(s_st[((b0 >> 5) & 1) ^ 1], e1, wbit, a.rec, rgbv, vbase, P.N, a.st);
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
            // one surfel: true when the pixel stops
            auto composite = [&](int j, const float4& oc, const Hit& h) {
                const float alpha = fminf(h.alpha_raw, P.alpha_max);
                const float Tn = T * (1.0f - alpha);
                if (Tn < P.T_min) return true;
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
                if (FRONT) {
                    // the first K contributors, in the K slots after the padding
                    if (n_sel < K) {
                        const int slot = KCAP - K + n_sel;
#pragma unroll
                        for (int k = 0; k < KCAP; ++k) {
                            hw[k] = k == slot ? w : hw[k];
                            hp[k] = k == slot ? b0 + j : hp[k];
                        }
                        ++n_sel;
                    }
                } else if (w > hw[KCAP - 1]) {
                    float in[KCAP];
                    int cp = b0 + j;  // the position carried into slot k, with weight min(slot k - 1, w)
#pragma unroll
                    for (int k = KCAP - 1; k >= 0; --k) in[k] = k > 0 ? fminf(hw[k > 0 ? k - 1 : 0], w) : w;
#pragma unroll
                    for (int k = 0; k < KCAP; ++k) {
                        const bool gt = in[k] > hw[k];
                        const int np = gt ? cp : hp[k];
                        cp = gt ? hp[k] : cp;
                        hp[k] = np;
                        hw[k] = fmaxf(hw[k], in[k]);
                    }
                }
                T = Tn;
                last = b0 + j;
                return P.stop_rule == FSS_STOP_EXACT_TOPK && (FRONT ? n_sel == K : P.alpha_max * T <= hw[KCAP - 1]);
            };
            if (!done) {
                if constexpr (PAIR) {
                    for (uint32_t bits = word; bits != 0u;) {
                        const int j0 = __ffs(bits) - 1;
                        bits &= bits - 1u;
                        const bool two = bits != 0u;
                        const int j1 = two ? __ffs(bits) - 1 : j0;
                        bits &= bits - 1u;
                        Hit h0, h1;
                        const bool hit0 = eval_splat<AUX>(S.r0[j0], S.r1[j0], S.r2[j0], S.oc[j0].x, pxf, pyf, P.alpha_min,
                                                          cam.near_plane, h0, P.lowpass);
                        const bool hit1 = eval_splat<AUX>(S.r0[j1], S.r1[j1], S.r2[j1], S.oc[j1].x, pxf, pyf, P.alpha_min,
                                                          cam.near_plane, h1, P.lowpass) && two;
                        ++n_eval;
                        if (hit0 && composite(j0, S.oc[j0], h0)) { done = true; break; }
                        n_eval += two ? 1u : 0u;
                        if (hit1 && composite(j1, S.oc[j1], h1)) { done = true; break; }
                    }
                } else {
                    for (uint32_t bits = word; bits != 0u; bits &= bits - 1u) {
                        const int j = __ffs(bits) - 1;
                        ++n_eval;
                        Hit h;
                        const float4 oc = S.oc[j];
                        if (eval_splat<AUX>(S.r0[j], S.r1[j], S.r2[j], oc.x, pxf, pyf, P.alpha_min, cam.near_plane, h, P.lowpass) &&
                            composite(j, oc, h)) {
                            done = true;
                            break;
                        }
                    }
                }
            }
            word = next;
            __syncwarp();  // every lane has read this half before the next copies into it
        }
        cp_async_wait_all();
        __syncwarp();

        // per-pixel outputs; the K-set in front-to-back order, through shared memory
        float lsum = 0.0f;  // LOSS: this lane's weighted loss terms (nothing live in phase 1)
        float rt[3] = {0.0f, 0.0f, 0.0f};  // LOSS: the colour target, loaded ahead of the ranks
        if (LOSS && inside) {
            const float* r = x.loss.rgbt + 3 * (cam.pix_off + (int64_t)py * cam.W + px);
#pragma unroll
            for (int c = 0; c < 3; ++c) rt[c] = __ldcs(r + c);
        }
        int hc = 0;
#pragma unroll
        for (int k = 0; k < KCAP; ++k) {
            hc += hp[k] >= 0 ? 1 : 0;
            int r = 0;
#pragma unroll
            for (int j = 0; j < KCAP; ++j) r += (hp[j] >= 0 && hp[j] < hp[k]) ? 1 : 0;
            if (hp[k] >= 0) s_sel[lane * ROW + r] = make_int2(hp[k], __float_as_int(hw[k]));
        }
        s_n[lane] = inside ? hc : 0;
        if (AUX) s_lab[lane] = 0ull;
        if (inside) {
            const int64_t pix = cam.pix_off + (int64_t)py * cam.W + px;
            if (a.out_rgb) {
                const float c3[3] = {fmaf(T, P.bg[0], cr), fmaf(T, P.bg[1], cg), fmaf(T, P.bg[2], cb)};
#pragma unroll
                for (int c = 0; c < 3; ++c) a.out_rgb[3 * pix + c] = c3[c];
                if (LOSS) {  // the colour term: |rgb - rgb_t| and its sign
                    float s1 = 0.0f;
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        const float d = c3[c] - rt[c];
                        s1 += fabsf(d);
                        x.loss.drgb[3 * pix + c] = d > 0.0f ? x.loss.sc : (d < 0.0f ? -x.loss.sc : 0.0f);
                    }
                    lsum = fmaf(x.loss.sc, s1, lsum);
                }
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
        {
            const FastDiv divK(K);
            const int ne = min(8, cam.W - bx) * K;
            for (int r = 0; r < 4 && by + r < cam.H; ++r) {
                const int64_t o0 = (cam.pix_off + (int64_t)(by + r) * cam.W + bx) * K;
                for (int e = lane; e < ne; e += 32) {
                    const int c = K == KCAP ? e / KCAP : divK.div(e), k = e - c * K, q = 8 * r + c;
                    int pos = -1, id = -1;
                    float w = 0.0f;
                    if (k < s_n[q]) {
                        const int2 v = s_sel[q * ROW + k];
                        pos = v.x;
                        w = __int_as_float(v.y);
                        id = (int32_t)((int64_t)list[pos] - vbase);
                        s_sel[q * ROW + k].x = id;  // for the feature gather below
                    }
                    if (a.out_ids) a.out_ids[o0 + e] = id;
                    if (a.saved_pos) a.saved_pos[o0 + e] = pos;
                    if (a.saved_w) a.saved_w[o0 + e] = w;
                }
            }
        }
        __syncwarp();
        warp_count(&a.st->counters[0], n_eval);
        warp_count(&a.st->counters[1], n_contrib);

        // phase 2: gather-accumulate the selected feature rows (AUX: and their argmax)
        if (a.out_feat || (AUX && x.label)) {
            if (P.renorm) {  // renormalised variant: weights over the selected weights' sum
                float ws = 0.0f;
                for (int k = 0; k < s_n[lane]; ++k) ws += __int_as_float(s_sel[lane * ROW + k].y);
                const float wsc = ws > 0.0f ? __frcp_rn(ws) : 0.0f;
                for (int k = 0; k < s_n[lane]; ++k)
                    s_sel[lane * ROW + k].y = __float_as_int(__int_as_float(s_sel[lane * ROW + k].y) * wsc);
                __syncwarp();
            }
            for (int i = lane; i < 32 * nvec; i += 32) {
                const int q = divV.div(i), vv = i - q * nvec;  // pixel of the block, 16-byte chunk of the row
                const int qx = bx + (q & 7), qy = by + (q >> 3);
                if (qx >= cam.W || qy >= cam.H) continue;
                const int64_t qpix = cam.pix_off + (int64_t)qy * cam.W + qx;
                typename FeatVec<FT>::Raw ft{};  // LOSS: the target chunk, loaded during the gathers
                if (LOSS) ft = FeatVec<FT>::raw_cs(reinterpret_cast<const FT*>(x.loss.Ft) + qpix * P.C + vv * E);
                // the selected rows' chunks, weighted with packed FP32 pairs (lane for
                // lane fmaf) in the selection's front-to-back order
                float2 acc2[E / 2];
#pragma unroll
                for (int e = 0; e < E / 2; ++e) acc2[e] = make_float2(0.0f, 0.0f);
                const int c = s_n[q];
                for (int k = 0; k < c; ++k) {
                    const int2 v = s_sel[q * ROW + k];
                    if (!in_bounds(a.st, SITE_FEAT_ROW, v.x, P.N)) continue;
                    float2 f2[E / 2];
                    FeatVec<FT>::unpack2(FeatVec<FT>::raw(feats + (size_t)v.x * P.C + vv * E), f2);
                    const float2 w2 = make_float2(__int_as_float(v.y), __int_as_float(v.y));
#pragma unroll
                    for (int e = 0; e < E / 2; ++e) acc2[e] = __ffma2_rn(w2, f2[e], acc2[e]);
                }
                if constexpr (LOSS) {
                    // F as stored (output type = feature type), then the feature term:
                    // d = F - F_t (an FMA with -1: one rounding, as the subtraction),
                    // sum d^2, dL/dF = sf d rounded once to the output type
                    // (F with an evict-first store: the step does not read it again)
                    using Raw = typename FeatVec<FT>::Raw;
                    const Raw fr = FeatVec<FT>::pack(acc2);
                    __stcs(reinterpret_cast<Raw*>(reinterpret_cast<FT*>(a.out_feat) + qpix * P.C + vv * E), fr);
                    float2 f2[E / 2], t2[E / 2], g2[E / 2];
                    FeatVec<FT>::unpack2(fr, f2);
                    FeatVec<FT>::unpack2(ft, t2);
                    const float2 m1 = make_float2(-1.0f, -1.0f), sf2 = make_float2(x.loss.sf, x.loss.sf);
                    float2 q2 = make_float2(0.0f, 0.0f);
#pragma unroll
                    for (int e = 0; e < E / 2; ++e) {
                        const float2 d2 = __ffma2_rn(t2[e], m1, f2[e]);
                        q2 = __ffma2_rn(d2, d2, q2);
                        g2[e] = __fmul2_rn(sf2, d2);
                    }
                    FeatVec<FT>::st(reinterpret_cast<FT*>(x.loss.dF) + qpix * P.C + vv * E, FeatVec<FT>::pack(g2));
                    lsum = fmaf(x.loss.lf, q2.x + q2.y, lsum);
                } else {
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
            }
            if (AUX && x.label) {
                __syncwarp();
                if (inside)
                    x.label[cam.pix_off + (int64_t)py * cam.W + px] = s_n[lane] > 0 ? argmax_channel(s_lab[lane]) : -1;
            }
        }
        if constexpr (LOSS) {  // the CTA's share of the loss: the last warp to arrive adds it, one double atomic
            float v = lsum;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(ALL, v, o);
            if (lane == 0) {
                s_loss[warp] = v;
                __threadfence_block();
                if (atomicAdd(&s_arrived, 1) == NW - 1) {
                    __threadfence_block();
                    double t = 0.0;
                    for (int w = 0; w < NW; ++w) t += *(volatile float*)&s_loss[w];
                    s_arrived = 0;
                    atomicAdd(x.loss.loss, t);
                }
            }
        }
        __syncwarp();  // before the warp's next block reuses its shared memory
    }
}

template <int TS, typename FT>
cudaError_t launch_topk(const Cams& cams, const RParams& P, const FwdArgs& a, const AuxOut& x, int num_sms,
                        cudaStream_t s) {
    constexpr int NT = topk_threads<TS, false>(), PARTS = TS * TS / NT;
    const bool aux = x.any() || P.lowpass;  // the variant instances also carry the low-pass filter
    auto smem = [aux](int kcap) { return NT / 32 * topk_warp_smem(kcap, aux); };
    // the fused loss (and sort): the plain selection with K <= 8, no sensor outputs (checked by the caller)
    if (x.loss.loss && x.sort.list)
        return launch_tiles(k_render_topk<TS, 8, FT, false, false, true, true>, TS * TS,
                            std::max(TS * TS / 32 * topk_warp_smem(8, false), SORT_SMEM_BYTES), cams, P, a, x, num_sms, s);
    if (x.loss.loss)
        return launch_tiles(k_render_topk<TS, 8, FT, false, false, true>, NT, smem(8), cams, P, a, x, num_sms, s, PARTS);
    // larger sets live in shared memory (render_topk_wide.cuh): those of more than
    // 16 entries, and more than 8 for the variants, which need the registers
    const bool plain = !aux && P.select != FSS_SELECT_FRONT;
    if (P.K > (plain ? CHAIN_K : 8)) return launch_topk_wide<TS, FT>(cams, P, a, x, num_sms, s);
    auto go = [&](auto kern, int kcap = 8) { return launch_tiles(kern, NT, smem(kcap), cams, P, a, x, num_sms, s, PARTS); };
    if (P.select == FSS_SELECT_FRONT)
        return aux ? go(k_render_topk<TS, 8, FT, true, true>) : go(k_render_topk<TS, 8, FT, true, false>);
    if (aux) return go(k_render_topk<TS, 8, FT, false, true>);
    if (P.K <= 4) return go(k_render_topk<TS, 4, FT, false, false>, 4);
    if (P.K <= 8) return go(k_render_topk<TS, 8, FT, false, false>);
    return go(k_render_topk<TS, 16, FT, false, false>, 16);
}

template <typename FT>
cudaError_t launch_topk_dtype(const Cams& cams, const RParams& P, const FwdArgs& a, const AuxOut& x, int num_sms,
                              cudaStream_t s) {
    if (P.ts == 8) return launch_topk<8, FT>(cams, P, a, x, num_sms, s);
    if (P.ts == 16) return launch_topk<16, FT>(cams, P, a, x, num_sms, s);
    return launch_topk<32, FT>(cams, P, a, x, num_sms, s);
}

}  // namespace fss
