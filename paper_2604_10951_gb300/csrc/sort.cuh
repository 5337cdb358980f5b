// Per-tile depth sort (the paper composites the surfels in depth order,
// Sec. 3.1), as a CTA-wide device function: the sort kernel runs it with one
// CTA per tile, and the Top-K forward's SORT instances run it on their own
// tile before rendering it.
//
// Binning leaves every tile's range of the pair list filled in arbitrary
// order (bounded items first, then the view's unbounded items are appended
// here).  The CTA sorts its range by the 64-bit key
//   (binary32 bits of the item's camera depth) << 32 | item index,
// which is unique, so the order is total and deterministic.  Depths are
// positive, so their bit patterns order like the numbers.
//   - up to SORT_CAP keys: a counting sort into SORT_BUCKETS depth intervals
//     and a rank within the bucket; lists of at most SORT_SMALL keys, and ones
//     whose depths crowd in a bucket, as 32-key chunks sorted by one warp each
//     in registers, then merged by rank (place in the chunk plus a binary
//     search in every other chunk).  The buckets take the forward of 1.5M surfels at
//     1280 x 720 (220 pairs per tile) from 430 to 421 us; what is left of the
//     kernel's 46 us is the gathers of the records and the warp masks;
//   - longer lists: stable LSD radix sort (8-bit digits) by the same CTA
//     in a global scratch range of the same offsets.
// With the sorted item, each pair gets the mask of the tile's warps (8 x 4
// pixel blocks) that its footprint reaches, which the render passes use
// to skip a surfel warp by warp.
#pragma once

#include "fss_internal.cuh"
#include "kernels.cuh"
#include "render_common.cuh"

namespace fss {

constexpr int SORT_BUCKETS = 512;
constexpr int SORT_SMALL = 128;  // keys: up to these, four chunks are as quick as the histogram
constexpr int SORT_CROWD = 32;  // keys in a bucket

// shared memory of sort_tile: keys, masks (by list position), places in the
// bucket or chunk order, bucket order, histogram
constexpr size_t SORT_SMEM_BYTES = (size_t)SORT_CAP * (8 + 4 + 2 + 2) + (size_t)SORT_BUCKETS * 4;

namespace {

// (the depth from the binning record, whose sectors the warp mask reads too)
__device__ __forceinline__ uint64_t sort_key(const BinRec* __restrict__ binrec, uint32_t item) {
    return ((uint64_t)__float_as_uint(__ldg(&binrec[item].z)) << 32) | item;
}

// stable radix sort of keys[0, n) by one CTA (a multiple of 32 threads);
// result in keys
__device__ __noinline__ void block_radix_sort_global(uint64_t* keys, uint64_t* tmp, int n) {
    __shared__ uint32_t hist[256];
    __shared__ uint32_t offs[256];
    __shared__ int skip;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nt = blockDim.x, nw = nt >> 5;
    uint64_t* src = keys;
    uint64_t* dst = tmp;
    for (int pass = 0; pass < 8; ++pass) {
        const int shift = pass * 8;
        for (int d = tid; d < 256; d += nt) hist[d] = 0;
        __syncthreads();
        for (int i = tid; i < n; i += nt) atomicAdd(&hist[(src[i] >> shift) & 255u], 1u);
        __syncthreads();
        if (tid == 0) {
            uint32_t run = 0;
            skip = 0;
            for (int d = 0; d < 256; ++d) {
                if (hist[d] == (uint32_t)n) skip = 1;
                offs[d] = run;
                run += hist[d];
            }
        }
        __syncthreads();
        if (skip) continue;  // every key has the same digit: order unchanged
        for (int base = 0; base < n; base += nt) {
            const int i = base + tid;
            const bool ok = i < n;
            const uint64_t k = ok ? src[i] : 0ull;
            const uint32_t d = ok ? (uint32_t)((k >> shift) & 255u) : 256u + (uint32_t)lane;
            const unsigned peers = __match_any_sync(0xffffffffu, d);
            const int rank = __popc(peers & ((1u << lane) - 1u));
            const int leader = __ffs(peers) - 1;
            for (int w = 0; w < nw; ++w) {  // warps in order keep the sort stable
                if (wid == w && ok) {
                    dst[offs[d] + rank] = k;
                }
                __syncwarp();
                if (wid == w && ok && lane == leader) offs[d] += __popc(peers);
                __syncthreads();
            }
        }
        __syncthreads();
        uint64_t* t = src; src = dst; dst = t;
    }
    if (src != keys)
        for (int i = tid; i < n; i += nt) keys[i] = src[i];
    __syncthreads();
}

}  // namespace

// Sorts tile t's list in place and writes its warp masks.  Called by every
// thread of the CTA (any multiple of 32 threads, at least 64); `area`:
// SORT_SMEM_BYTES of shared memory, 16-byte aligned.  Returns with the list and masks in
// global memory written by this CTA (the caller synchronises before reading
// them back).
static __device__ __noinline__ void sort_tile(const Cams& cams, const RParams& P, const BinRec* __restrict__ binrec,
                                          const int2* __restrict__ ranges,
                                          uint32_t* list, const uint32_t* __restrict__ unb_list,
                                          uint64_t* __restrict__ scratch, uint32_t* masks, Status* stw, int t,
                                          unsigned char* area) {
    uint64_t* sk = reinterpret_cast<uint64_t*>(area);
    uint32_t* smask = reinterpret_cast<uint32_t*>(area + (size_t)SORT_CAP * 8);
    int* hist = reinterpret_cast<int*>(area + (size_t)SORT_CAP * 12);
    uint16_t* spos = reinterpret_cast<uint16_t*>(area + (size_t)SORT_CAP * 12 + SORT_BUCKETS * 4);
    uint16_t* sord = spos + SORT_CAP;
    const int2 rg = checked_range(ranges, t, P.pair_cap, stw);
    const int n = rg.y - rg.x;
    if (n <= 0) return;
    const int view = view_of_tile(cams, t);
    const CamDev& cam = cams.c[view];
    const int lt = t - cam.tile_off;
    const int tx0 = (lt % cam.tiles_x) * P.ts, ty0 = (lt / cam.tiles_x) * P.ts;
    const int nu = (int)stw->unb_cnt[view];
    if (!in_bounds(stw, SITE_VIS_LIST, nu, ((int64_t)n < P.N ? (int64_t)n : P.N) + 1)) return;
    const int nb = n - nu;
    const uint32_t* ul = unb_list + (int64_t)view * P.N;
    const int tid = threadIdx.x, nt = blockDim.x;
    // the i-th item of the tile (bounded items, then the view's unbounded ones), checked
    auto item_at = [&](int i) -> uint32_t {
        const uint32_t it = i < nb ? list[rg.x + i] : ul[i - nb];
        return in_bounds(stw, SITE_ITEM, it, P.n_items) ? it : 0u;
    };
    if (n <= SORT_CAP) {
        // A. each pair's key and warp mask (the mask does not depend on the
        //    order, so it is formed here, beside the key's gather), and the
        //    smallest and largest depth
        const int n32 = (n + 31) & ~31;  // padded with ~0 keys, larger than every key (depth bits < 0x7f800000)
        uint32_t zlo = 0xffffffffu, zhi = 0u;
        __shared__ uint32_t s_lo, s_hi, s_most;
        __shared__ int s_red[33];
        const bool buckets = n > SORT_SMALL;
        if (buckets) {
            for (int i = tid; i < SORT_BUCKETS; i += nt) hist[i] = 0;
            if (tid == 0) {
                s_lo = 0xffffffffu;
                s_hi = 0u;
                s_most = 0u;
            }
            __syncthreads();
        }
#pragma unroll 2
        for (int i = tid; i < n32; i += nt) {
            uint64_t k = ~0ull;
            if (i < n) {
                const uint32_t item = item_at(i);
                k = sort_key(binrec, item);
                smask[i] = P.lowpass ? warp_block_mask<true>(binrec + item, P.ts, tx0, ty0)
                                     : warp_block_mask<false>(binrec + item, P.ts, tx0, ty0);
                zlo = min(zlo, (uint32_t)(k >> 32));
                zhi = max(zhi, (uint32_t)(k >> 32));
            }
            sk[i] = k;
        }
        if (buckets) {
            // Buckets of equal depth intervals between the two: a key's bucket
            // grows with its depth, so its rank is the bucket's first place plus
            // the smaller keys of its own bucket (the keys are unique).  With
            // 512 buckets a tile's list has one or two keys in most; where the
            // depths crowd (more than SORT_CROWD keys in a bucket), the chunks
            // below sort it instead.
            zlo = __reduce_min_sync(0xffffffffu, zlo);
            zhi = __reduce_max_sync(0xffffffffu, zhi);
            if ((tid & 31) == 0) {
                atomicMin(&s_lo, zlo);
                atomicMax(&s_hi, zhi);
            }
            __syncthreads();
            const float z0 = __uint_as_float(s_lo), dz = __uint_as_float(s_hi) - z0;
            const float sc = dz > 0.0f ? fminf((float)SORT_BUCKETS / dz, 3e38f) : 0.0f;
            auto bucket = [&](uint64_t k) {
                return min((int)((__uint_as_float((uint32_t)(k >> 32)) - z0) * sc), SORT_BUCKETS - 1);
            };
            uint32_t most = 0u;
            for (int i = tid; i < n; i += nt) {
                const uint32_t at = (uint32_t)atomicAdd(&hist[bucket(sk[i])], 1);
                spos[i] = (uint16_t)at;
                most = max(most, at);
            }
            most = __reduce_max_sync(0xffffffffu, most);
            if ((tid & 31) == 0) atomicMax(&s_most, most);
            __syncthreads();
            if (s_most < SORT_CROWD) {
                block_exscan(hist, SORT_BUCKETS, s_red);
                for (int i = tid; i < n; i += nt) sord[hist[bucket(sk[i])] + spos[i]] = (uint16_t)i;
                __syncthreads();
                for (int q = tid; q < n; q += nt) {
                    const int i = sord[q];
                    const uint64_t k = sk[i];
                    const int bk = bucket(k), first = hist[bk], end = bk + 1 < SORT_BUCKETS ? hist[bk + 1] : n;
                    int rank = first;
                    for (int j = first; j < end; ++j) rank += sk[sord[j]] < k ? 1 : 0;
                    list[rg.x + rank] = (uint32_t)k;
                    masks[rg.x + rank] = smask[i];
                }
                return;
            }
        } else {
            __syncthreads();
        }
        // B. short or crowded lists in 32-key chunks: each warp sorts its chunks
        //    in registers (bitonic network over the lanes), carrying each key's
        //    position in the list;
        // C. a key's rank is its place in its chunk plus, per other chunk, the
        //    number of smaller keys there (a 32-way binary search).
        const int nch = (n + 31) >> 5, lane = tid & 31, w = tid >> 5;
        for (int c = w; c < nch; c += nt >> 5) {
            uint64_t k = sk[(c << 5) + lane];
            int pos = (c << 5) + lane;
#pragma unroll
            for (int kk = 2; kk <= 32; kk <<= 1) {
#pragma unroll
                for (int j = kk >> 1; j > 0; j >>= 1) {
                    const uint64_t ok = __shfl_xor_sync(0xffffffffu, k, j);
                    const int op = __shfl_xor_sync(0xffffffffu, pos, j);
                    const bool keep_min = ((lane & kk) == 0) == ((lane & j) == 0);  // ascending runs
                    const bool take = keep_min ? ok < k : ok > k;
                    k = take ? ok : k;
                    pos = take ? op : pos;
                }
            }
            sk[(c << 5) + lane] = k;
            spos[(c << 5) + lane] = (uint16_t)pos;
        }
        __syncthreads();
        for (int q = tid; q < n; q += nt) {
            const uint64_t k = sk[q];
            const int c = q >> 5;
            int rank = q & 31;
            for (int c2 = 0; c2 < nch; ++c2) {
                if (c2 == c) continue;
                const uint64_t* a = sk + (c2 << 5);
                int cnt = a[31] < k ? 32 : 0;
#pragma unroll
                for (int step = 16; step > 0; step >>= 1) cnt += (cnt < 32 && a[cnt + step - 1] < k) ? step : 0;
                rank += cnt;
            }
            list[rg.x + rank] = (uint32_t)k;
            masks[rg.x + rank] = smask[spos[q]];
        }
        return;
    }
    uint64_t* keys = scratch + rg.x;
    uint64_t* tmp = scratch + P.pair_cap + rg.x;
    for (int i = tid; i < n; i += nt) keys[i] = sort_key(binrec, item_at(i));
    __syncthreads();
    block_radix_sort_global(keys, tmp, n);
    for (int i = tid; i < n; i += nt) {
        const uint32_t item = (uint32_t)keys[i];
        list[rg.x + i] = item;
        masks[rg.x + i] = (P.lowpass ? warp_block_mask<true>(binrec + item, P.ts, tx0, ty0)
                                     : warp_block_mask<false>(binrec + item, P.ts, tx0, ty0));
    }
}

}  // namespace fss
