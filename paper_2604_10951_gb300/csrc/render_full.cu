// Full-accumulation forward render (K = 0, the plain path of Eq. 2): every
// contributor adds w c_i over all C channels.  Two kernels: with few channels
// the products are few beside the compositing, and k_render_full forms them as it
// goes; with more k_render_full_warp shares them among a warp's lanes.
#include "fss_internal.cuh"
#include "kernels.cuh"
#include "render_common.cuh"
#include "render_full.cuh"

#include <algorithm>
#include <climits>
#include <type_traits>

namespace fss {

namespace {

__device__ __forceinline__ int next_tile(const Cams& cams, const FwdArgs& a, int* s_tile, bool first) {
    return next_tile_q(a.persistent, &a.st->work, s_tile, first, cams);
}

}  // namespace

// ---------------------------------------------------------------------------
// k_render_full: a CTA per tile stages records and feature rows 64 at a time,
// and a contributor's lane adds w c_i over all channels from shared memory
// ---------------------------------------------------------------------------
template <int TS, int CMAX, typename FT, bool AUX>
__global__ void __launch_bounds__(TS * TS) k_render_full(const __grid_constant__ Cams cams,
                                                         const __grid_constant__ RParams P, const FwdArgs a,
                                                         const __grid_constant__ AuxOut x) {
    constexpr int NT = TS * TS;
    constexpr int E = FeatVec<FT>::E;
    extern __shared__ __align__(16) unsigned char smem[];
    float4* s_r0 = reinterpret_cast<float4*>(smem);
    float4* s_r1 = s_r0 + FBATCH;
    float4* s_r2 = s_r1 + FBATCH;
    float4* s_oc = s_r2 + FBATCH;                                   // (o, r, g, b)
    uint32_t* s_wm = reinterpret_cast<uint32_t*>(s_oc + FBATCH);    // warps the footprint reaches
    float* s_f = reinterpret_cast<float*>(s_wm + 2 * FBATCH);       // [FBATCH][C] f32 (16-byte aligned)
    float4* s_nrm = reinterpret_cast<float4*>(s_f + (size_t)FBATCH * P.C);  // AUX: facing normals
    __shared__ int s_tile;

    const int tid = threadIdx.x;
    if (a.st->err) return;
    const int C = P.C;
    const FT* __restrict__ feats = reinterpret_cast<const FT*>(a.feats);
    const uint32_t wbit = 1u << (tid >> 5);
    const int nv = C / E;
    const int rpi = NT / nv;                         // staged rows per sweep
    const int r0 = tid / nv, vv0 = tid - r0 * nv;    // this thread's row offset and 16-byte chunk
    for (int t = next_tile(cams, a, &s_tile, true); t < cams.total_tiles; t = next_tile(cams, a, &s_tile, false)) {
        const int view = view_of_tile(cams, t);
        const CamDev& cam = cams.c[view];
        const int lt = t - cam.tile_off;
        const int tx = lt % cam.tiles_x, ty = lt / cam.tiles_x;
        const int2 lp = pixel_of<TS>(tid);
        const int px = tx * TS + lp.x, py = ty * TS + lp.y;
        const bool inside = px < cam.W && py < cam.H;
        const float pxf = (float)px + 0.5f, pyf = (float)py + 0.5f;
        const int2 rg = checked_range(a.ranges, t, P.pair_cap, a.st);
        const int n = rg.y - rg.x;
        const int64_t vbase = (int64_t)view * P.N;
        const float* __restrict__ rgbv = a.rgb + (P.color_sh ? 3 * vbase : 0);  // SH: item colours

        float T = 1.0f, cr = 0.0f, cg = 0.0f, cb = 0.0f;
        float acc[CMAX];
#pragma unroll
        for (int c = 0; c < CMAX; ++c) acc[c] = 0.0f;
        bool done = !inside;
        int last = -1;
        uint32_t n_eval = 0, n_contrib = 0;
        float zs = 0.0f, zmed = 0.0f, nx = 0.0f, ny = 0.0f, nz = 0.0f;  // AUX sums
        bool med = false;

        for (int b0 = 0; b0 < n; b0 += FBATCH) {
            if (__syncthreads_and(done)) break;
            const int cnt = min(FBATCH, n - b0);
            for (int j = tid; j < cnt; j += NT) {
                const uint32_t item = a.list[rg.x + b0 + j];
                if (!in_bounds(a.st, SITE_ITEM, (int64_t)item - vbase, P.N)) {  // check build: a dead record
                    s_oc[j] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    s_wm[j] = 0u;
                    continue;
                }
                const float4* r = a.rec + 4 * (size_t)item;
                s_r0[j] = r[0];
                s_r1[j] = r[1];
                s_r2[j] = r[2];
                const int64_t sp = (int64_t)item - vbase;
                s_oc[j] = make_float4(r[3].x, rgbv[3 * sp], rgbv[3 * sp + 1], rgbv[3 * sp + 2]);
                s_wm[j] = a.masks[rg.x + b0 + j];
                if (AUX) {  // facing normal, and the centre depth for the low-pass screen term
                    const float4 nf = facing_normal(r[2], r[0].w, r[1].w, cam);
                    s_nrm[j] = make_float4(nf.x, nf.y, nf.z, r[3].y);
                }
            }
            if (r0 < rpi) {
                for (int j = r0; j < cnt; j += rpi) {
                    const int64_t sp = (int64_t)a.list[rg.x + b0 + j] - vbase;
                    if (!FSS_CHECKED(sp >= 0 && sp < P.N)) continue;  // recorded by the staging loop
                    float f[E];
                    FeatVec<FT>::load(feats + (size_t)sp * C + vv0 * E, f);
#pragma unroll
                    for (int e = 0; e < E; ++e) s_f[j * C + vv0 * E + e] = f[e];
                }
            }
            __syncthreads();
            if (done) continue;
            for (int j = 0; j < cnt; ++j) {
                if (!(s_wm[j] & wbit)) continue;  // warp-uniform
                ++n_eval;
                Hit h;
                const float4 oc = s_oc[j];
                if (!eval_splat<AUX>(s_r0[j], s_r1[j], s_r2[j], oc.x, pxf, pyf, P.alpha_min, cam.near_plane, h, P.lowpass))
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
                    const float zh = h.scr ? nv.w : s_r2[j].w * h.inv;  // hit depth, as in the near-plane test
                    zs = fmaf(w, zh, zs);
                    nx = fmaf(w, nv.x, nx);
                    ny = fmaf(w, nv.y, ny);
                    nz = fmaf(w, nv.z, nz);
                    if (!med && Tn < 0.5f) { zmed = zh; med = true; }
                }
                const float4* fr = reinterpret_cast<const float4*>(s_f + j * C);
#pragma unroll
                for (int c4 = 0; c4 < CMAX / 4; ++c4) {
                    if (4 * c4 < C) {
                        const float4 f = fr[c4];
                        acc[4 * c4] = fmaf(w, f.x, acc[4 * c4]);
                        acc[4 * c4 + 1] = fmaf(w, f.y, acc[4 * c4 + 1]);
                        acc[4 * c4 + 2] = fmaf(w, f.z, acc[4 * c4 + 2]);
                        acc[4 * c4 + 3] = fmaf(w, f.w, acc[4 * c4 + 3]);
                    }
                }
                T = Tn;
                last = b0 + j;
            }
        }
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
                if (x.label) {  // argmax over the channels, lowest index on ties
                    int cb = 0;
                    float bv = acc[0];
#pragma unroll
                    for (int c = 1; c < CMAX; ++c) {
                        const bool gt = c < C && acc[c] > bv;
                        cb = gt ? c : cb;
                        bv = gt ? acc[c] : bv;
                    }
                    x.label[pix] = n_contrib > 0 ? cb : -1;
                }
            }
            if (a.out_feat) {
#pragma unroll
                for (int c4 = 0; c4 < CMAX / 4; ++c4)
                    if (4 * c4 < C) store_vec<4>(a.out_feat, pix * C + 4 * c4, &acc[4 * c4], P.out_dtype);
            }
        }
        warp_count(&a.st->counters[0], n_eval);
        warp_count(&a.st->counters[1], n_contrib);
    }
}

// ---------------------------------------------------------------------------
// k_render_full_warp: one warp per 8 x 4 pixel block, each on its own (the walk
// of render_topk.cuh)
// ---------------------------------------------------------------------------
// The lanes composite their pixels and leave the weights of each surfel that any of
// them meets in shared memory, with the surfel's feature row copied beside them; eight
// rows at a time the warp adds weights x rows as a small matrix product, in which a
// lane holds PX pixels x 4 NQ channels of F in registers (FullLanes: 8 x 8 at 64
// channels) and reads 8 weights and 8 channels per surfel for 64 multiply-adds, where a
// lane with its own pixel reads all 64 channels.  A pixel's channels are still summed
// front to back.  Each product runs when the next eight rows are full, so that its
// copies have arrived (rows read straight from memory, one ahead: 13 to 44 us slower).
// 640 x 480, 500k surfels, forward: 64 channels FP32 196 -> 166 us, 128 channels 795
// -> 260 (the row in a lane's registers spilled there).
// A lane's pixels multiply rows that they did not meet by -0 (a contributor's
// weight is never that): an infinite or NaN feature would reach them, so a block
// whose sums are not all finite is done again with those products left out.
namespace {

// one warp's shared memory
constexpr int FULL_ROWS = 8;  // rows of a product
template <int CMAX, typename FT, bool AUX>
struct FullStage {
    WarpStage st[2];
    int32_t sp[2][32];                          // the staged surfels
    float4 w[2][FULL_ROWS][8];                  // weights [row][pixel], two products in turn
    __align__(16) FT f[2][FULL_ROWS][CMAX];     // ... and the feature rows
    float4 nrm[AUX ? 32 : 1];                   // AUX: facing normals, centre depths
};

}  // namespace

template <int TS, int CMAX, typename FT, bool AUX>
__global__ void __launch_bounds__(full_threads<TS>(), (CMAX <= 64 ? 512 : 256) / full_threads<TS>()) k_render_full_warp(
    const __grid_constant__ Cams cams, const __grid_constant__ RParams P, const FwdArgs a,
    const __grid_constant__ AuxOut x) {
    using L = FullLanes<CMAX>;
    constexpr int NT = full_threads<TS>(), NW = NT / 32, PARTS = TS * TS / NT, PX = L::PX, NQ = L::NQ;
    constexpr unsigned ALL = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_work;
    using Stage = FullStage<CMAX, FT, AUX>;

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cg = lane % L::CL, pg = lane / L::CL;  // this lane's channels and pixels of the product
    if (a.st->err) return;
    Stage& G = reinterpret_cast<Stage*>(smem)[warp];
    const int C = P.C;
    const FT* __restrict__ feats = reinterpret_cast<const FT*>(a.feats);
    constexpr int E = FeatVec<FT>::E;
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
        const int n = rg.y - rg.x;
        const int64_t vbase = (int64_t)view * P.N;
        const float* __restrict__ rgbv = a.rgb + (P.color_sh ? 3 * vbase : 0);  // SH: item colours
        const uint32_t* list = a.list + rg.x;
        const uint32_t* masks = a.masks + rg.x;

        float T, cr, cgr, cb;
        bool done, med;
        int last;
        uint32_t n_eval, n_contrib;
        float zs, zmed, nx, ny, nz;  // AUX sums
        float2 acc[PX][NQ][2];

        // F += weights x rows of one half; careful: without the products of pixels that did not meet the surfel
        auto product = [&](int half, int rows, auto careful) {
#pragma unroll(NQ > 1 ? 1 : 2)
            for (int r = 0; r < rows; ++r) {
                float4 f[NQ];
                float w[PX];
                L::lds_row(G.f[half][r], cg, f);
                L::load_weights(reinterpret_cast<const float*>(G.w[half][r]) + pg * PX, w);
#pragma unroll
                for (int p = 0; p < PX; ++p) {
                    const float2 ww = make_float2(w[p], w[p]);
                    if (decltype(careful)::value && __float_as_uint(w[p]) == 0x80000000u) continue;
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        acc[p][q][0] = __ffma2_rn(ww, make_float2(f[q].x, f[q].y), acc[p][q][0]);
                        acc[p][q][1] = __ffma2_rn(ww, make_float2(f[q].z, f[q].w), acc[p][q][1]);
                    }
                }
            }
        };
        for (bool careful = false;; careful = true) {
            T = 1.0f;
            cr = cgr = cb = 0.0f;
            done = !inside;
            med = false;
            last = -1;
            n_eval = n_contrib = 0;
            zs = zmed = nx = ny = nz = 0.0f;
#pragma unroll
            for (int p = 0; p < PX; ++p)
#pragma unroll
                for (int q = 0; q < NQ; ++q) acc[p][q][0] = acc[p][q][1] = make_float2(0.0f, 0.0f);
            auto stage = [&](int buf, const ListEntry& e) {
                G.sp[buf][lane] = (int32_t)((int64_t)e.item - vbase);
                return stage_chunk(G.st[buf], e, wbit, a.rec, rgbv, vbase, P.N, a.st);
            };
            int rows = 0, half = 0;  // rows in the half being filled; the other one is full from the first change on
            bool full = false;
            // chunk i is worked on while chunk i + 1 is copied and the list entries of chunk i + 2 are read
            ListEntry e1 = list_entry(list, masks, lane, n);
            uint32_t word = stage(0, e1);
            e1 = list_entry(list, masks, 32 + lane, n);
            for (int b0 = 0; b0 < n; b0 += 32) {
                if (__all_sync(ALL, done)) break;
                const int buf = (b0 >> 5) & 1;
                const WarpStage& S = G.st[buf];
                const uint32_t next = stage(buf ^ 1, e1);
                e1 = list_entry(list, masks, b0 + 64 + lane, n);
                cp_async_wait_prev();  // this chunk's copies (the next one's stay in flight)
                __syncwarp();
                if constexpr (AUX) {  // facing normals, and the centre depths for the low-pass screen term
                    if ((word >> lane) & 1u) {
                        const float4 nf = facing_normal(S.r2[lane], S.r0[lane].w, S.r1[lane].w, cam);
                        G.nrm[lane] = make_float4(nf.x, nf.y, nf.z, a.rec[4 * (size_t)list[b0 + lane] + 3].y);
                    }
                    __syncwarp();
                }
                for (uint32_t bits = word; bits != 0u; bits &= bits - 1u) {
                    const int j = __ffs(bits) - 1;
                    float w = -0.0f;
                    if (!done) {
                        ++n_eval;
                        Hit h;
                        const float4 oc = S.oc[j];
                        if (eval_splat<AUX>(S.r0[j], S.r1[j], S.r2[j], oc.x, pxf, pyf, P.alpha_min, cam.near_plane, h, P.lowpass)) {
                            const float alpha = fminf(h.alpha_raw, P.alpha_max);
                            const float Tn = T * (1.0f - alpha);
                            if (Tn < P.T_min) {
                                done = true;
                            } else {
                                w = alpha * T;
                                cr = fmaf(w, oc.y, cr);
                                cgr = fmaf(w, oc.z, cgr);
                                cb = fmaf(w, oc.w, cb);
                                ++n_contrib;
                                if constexpr (AUX) {
                                    const float4 nv = G.nrm[j];
                                    const float zh = h.scr ? nv.w : S.r2[j].w * h.inv;  // hit depth, as in the near-plane test
                                    zs = fmaf(w, zh, zs);
                                    nx = fmaf(w, nv.x, nx);
                                    ny = fmaf(w, nv.y, ny);
                                    nz = fmaf(w, nv.z, nz);
                                    if (!med && Tn < 0.5f) { zmed = zh; med = true; }
                                }
                                T = Tn;
                                last = b0 + j;
                            }
                        }
                    }
                    if (__any_sync(ALL, __float_as_uint(w) != 0x80000000u)) {  // a row of the product
                        reinterpret_cast<float*>(G.w[half][rows])[lane] = w;
                        const FT* src = feats + (int64_t)G.sp[buf][j] * C;
                        if (lane * E < C) cp_async16(&G.f[half][rows][lane * E], src + lane * E, 16);
                        if (++rows == FULL_ROWS) {  // the half before this one, whose copies have long arrived
                            cp_async_commit();
                            cp_async_wait_prev();
                            __syncwarp();
                            if (full && !careful) product(half ^ 1, FULL_ROWS, std::false_type{});
                            if (full && careful) product(half ^ 1, FULL_ROWS, std::true_type{});
                            __syncwarp();  // read by every lane before it is filled again
                            full = true;
                            half ^= 1;
                            rows = 0;
                        }
                    }
                }
                word = next;
                __syncwarp();  // every lane has read this half and the weights before they are written again
            }
            cp_async_commit();
            cp_async_wait_all();
            __syncwarp();
#pragma unroll 1
            for (int k = full ? 0 : 1; k < 2; ++k) {
                if (!careful) product(half ^ 1 ^ k, k ? rows : FULL_ROWS, std::false_type{});
                else product(half ^ 1 ^ k, k ? rows : FULL_ROWS, std::true_type{});
            }
            __syncwarp();
            if (careful) break;
            float2 z = make_float2(0.0f, 0.0f);  // NaN when a sum is not finite
#pragma unroll
            for (int p = 0; p < PX; ++p)
#pragma unroll
                for (int q = 0; q < NQ; ++q)
                    if (4 * (cg + L::CL * q) < C) {
                        z = __ffma2_rn(acc[p][q][0], make_float2(0.0f, 0.0f), z);
                        z = __ffma2_rn(acc[p][q][1], make_float2(0.0f, 0.0f), z);
                    }
            if (!__any_sync(ALL, !(z.x + z.y == 0.0f))) break;
        }

        if (inside) {
            const int64_t pix = cam.pix_off + (int64_t)py * cam.W + px;
            if (a.out_rgb) {
                a.out_rgb[3 * pix] = fmaf(T, P.bg[0], cr);
                a.out_rgb[3 * pix + 1] = fmaf(T, P.bg[1], cgr);
                a.out_rgb[3 * pix + 2] = fmaf(T, P.bg[2], cb);
            }
            if (a.out_T) a.out_T[pix] = T;
            if (a.saved_nstop) a.saved_nstop[pix] = last + 1;
            if constexpr (AUX) {
                if (x.depth) x.depth[pix] = zs;
                if (x.depth_med) x.depth_med[pix] = zmed;
                if (x.normal) {
                    x.normal[3 * pix] = nx;
                    x.normal[3 * pix + 1] = ny;
                    x.normal[3 * pix + 2] = nz;
                }
            }
        }
#pragma unroll
        for (int p = 0; p < PX; ++p) {
            const int i = pg * PX + p, qx = bx + (i & 7), qy = by + (i >> 3);  // the lane's p-th pixel of the product
            const bool ok = qx < cam.W && qy < cam.H;
            const int64_t pix = cam.pix_off + (int64_t)qy * cam.W + qx;
            if (a.out_feat && ok) {
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const int c = 4 * (cg + L::CL * q);
                    const float v[4] = {acc[p][q][0].x, acc[p][q][0].y, acc[p][q][1].x, acc[p][q][1].y};
                    if (c < C) store_vec<4>(a.out_feat, pix * C + c, v, P.out_dtype);
                }
            }
            if constexpr (AUX) {
                if (x.label) {
                    const uint32_t met = __shfl_sync(ALL, n_contrib, i);
                    L::label(acc[p], cg, C, met > 0, ok ? x.label + pix : nullptr);
                }
            }
        }
        warp_count(&a.st->counters[0], n_eval);
        warp_count(&a.st->counters[1], n_contrib);
    }
}

namespace {

// 640 x 480, 500k surfels, forward, k_render_full / k_render_full_warp: 16 channels FP32
// 110 / 121 us, 32 channels 155 / 155, 64 196 / 166, 128 795 / 260, BF16 the same; with
// sensor outputs (200k) 64 channels 117 / 119, 128 207 / 187.
constexpr int FULL_WARP_C = 32, FULL_WARP_AUX_C = 64;  // channels above which the warps' kernel is taken

template <int TS, typename FT>
cudaError_t launch_full(const Cams& cams, const RParams& P, const FwdArgs& a, const AuxOut& x, int num_sms, cudaStream_t s) {
    const bool aux = x.any() || P.lowpass;  // the variant instances also carry the low-pass filter
    if (P.C > (aux ? FULL_WARP_AUX_C : FULL_WARP_C)) {
        constexpr int NT = full_threads<TS>(), PARTS = TS * TS / NT;
        auto go = [&](auto kern, size_t warp_smem) {
            return launch_tiles(kern, NT, NT / 32 * warp_smem, cams, P, a, x, num_sms, s, PARTS);
        };
        if (aux) return go(k_render_full_warp<TS, 128, FT, true>, sizeof(FullStage<128, FT, true>));
        if (P.C <= 64) return go(k_render_full_warp<TS, 64, FT, false>, sizeof(FullStage<64, FT, false>));
        return go(k_render_full_warp<TS, 128, FT, false>, sizeof(FullStage<128, FT, false>));
    }
    const size_t smem = (size_t)FBATCH * (4 * 16 + 8) + (size_t)FBATCH * P.C * 4 +
                        (aux ? (size_t)FBATCH * 16 : 0);  // staging, masks, rows (+ normals)
    auto go = [&](auto kern) { return launch_tiles(kern, TS * TS, smem, cams, P, a, x, num_sms, s); };
    if (P.C <= 16) return aux ? go(k_render_full<TS, 16, FT, true>) : go(k_render_full<TS, 16, FT, false>);
    if (P.C <= 32) return aux ? go(k_render_full<TS, 32, FT, true>) : go(k_render_full<TS, 32, FT, false>);
    return go(k_render_full<TS, 64, FT, true>);
}

template <typename FT>
cudaError_t launch_full_dtype(const Cams& cams, const RParams& P, const FwdArgs& a, const AuxOut& x, int num_sms,
                              cudaStream_t s) {
    if (P.ts == 8) return launch_full<8, FT>(cams, P, a, x, num_sms, s);
    if (P.ts == 16) return launch_full<16, FT>(cams, P, a, x, num_sms, s);
    return launch_full<32, FT>(cams, P, a, x, num_sms, s);
}

}  // namespace

cudaError_t launch_render_full(const Cams& cams, const RParams& P, const FwdArgs& a, const AuxOut& x, int num_sms,
                               cudaStream_t s) {
    if (P.feat_dtype == FSS_BF16) return launch_full_dtype<__nv_bfloat16>(cams, P, a, x, num_sms, s);
    return launch_full_dtype<float>(cams, P, a, x, num_sms, s);
}

}  // namespace fss
