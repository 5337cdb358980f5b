// Query-guided instance labels (Sec. 3.3) on the 5th-generation tensor cores,
// for many queries or wide instance features (query.cu has the definition's
// entry and the kernel for the rest).
//
// For every scene Gaussian g and instance query q:
//   S = sigmoid(f_q . f_ins(g)),  D = exp(-1/2 d^T Sigma_q^-1 d), d = p_g - p_q,
//   A = S D,  l_ins(g) = softmax over q of A.
// The similarity logits f_ins F_q^T are a dense [N, dim] x [dim, nq]
// contraction, so they run as tcgen05 MMAs: one CTA of 8 warps takes QB
// blocks of 128 Gaussians at a time (per block M = 128, N = nq, K = dim in
// steps of 16, BF16 operands, FP32 accumulators in tensor memory).  The
// epilogue reads the accumulators back with tcgen05.ld, one TMEM lane (= one
// Gaussian) per thread and block; warps 0-3 take the first half of the
// queries and warps 4-7 the second, so the softmax needs one exchange of two
// partial sums.  Pass 1 turns each logit into exp(A) and writes it back to
// tensor memory while summing; pass 2 reads exp(A) again, scales it by 1 / sum
// and stores it through a shared-memory transpose.
//
// What bounds it (1.2M Gaussians, 112 queries, 64-d, FP32 labels: 207 us =
// 3.4 TB/s of the 706 MB it must move, 50 % of the measured copy rate; the
// kernel of query.cu takes 280 us): without the reads of the queries' parameters
// it takes 151 us, without pass 2 157 us, without MUFU operations 191 us.
//   - The nine proximity parameters of a query are read from shared memory by
//     every thread (a broadcast 16-byte load still writes 512 bytes of
//     registers): two Gaussians per thread share each read, and two queries sit
//     side by side so that the arithmetic runs on FP32 pairs.
//   - A thread's row of labels is 16-byte pieces nq * s bytes apart from its
//     neighbours', 32 L2 lines per store instruction; transposed through shared
//     memory an instruction writes 8 rows' whole 64-byte pieces.
//   - The next 8 logits are read from tensor memory, and the next tile's
//     operand and centres from global memory, while the current ones are worked
//     on.
// Measured and not kept: exp(A) as a polynomial on the FMA pipe (seven more
// instructions per label, MUFU is not the limit), four Gaussians per thread
// (one CTA per SM: 242 us), 512-thread CTAs (219 us), one Gaussian per thread
// (the same 207 us here, slower for fewer queries).
//
// Shared-memory operands use the no-swizzle K-major layout of 8 x 16-byte
// core matrices: element (r, k) of a [rows, dim] operand sits at byte
// ((r / 8) * (dim / 8) + k / 8) * 128 + (r % 8) * 16 + (k % 8) * 2, i.e. a
// leading-dimension (K) step of 128 bytes between core matrices and a
// stride-dimension (row-group) step of dim * 16 bytes.
//
// Every wait on the MMA's mbarrier is bounded: on expiry the kernel raises
// the caller's error word, stops taking tiles, frees its tensor memory and
// returns.
#include "query_common.cuh"

#include <algorithm>
#include <type_traits>

namespace fss {

namespace {

constexpr int QTHREADS = 256;  // warp w: TMEM lanes 32 (w % 4) on, query half w / 4
template <typename OT>
constexpr int QCOLS = 64 / (int)sizeof(OT);  // columns per pass-2 transpose: 64 bytes
constexpr int QROW = 64 + 16;                // its padded row

// Reads of this thread's TMEM lane.  tmem_ld8 starts a read of 8 columns;
// its registers hold the values after tmem_wait8, which they pass through, so
// that no use moves ahead of the wait.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait8(uint32_t (&r)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]));
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const float (&v)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr),
                 "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
                 "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
                 "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])));
}

// Operand staging in the core-matrix layout, asynchronously: rows [0, nrows)
// (nrows a multiple of 8; rows past `valid` are zero) of a row-major BF16
// matrix of KC 16-byte chunks per row.  A warp takes 8-row groups; the 8
// threads of a shared-memory store phase write the 8 rows of one core matrix
// (128 consecutive bytes, no bank conflict).
__device__ __forceinline__ void copy_rows(unsigned char* dst, const __nv_bfloat16* __restrict__ src, int KC, int nrows,
                                          int64_t valid) {
    const int lane = threadIdx.x & 31, r = lane & 7;
    const unsigned char* base = reinterpret_cast<const unsigned char*>(src);
    for (int g = threadIdx.x >> 5; g < nrows >> 3; g += QTHREADS >> 5) {
        const bool in = 8 * g + r < valid;
        const unsigned char* s = base + (8 * g + r) * (16 * KC);
        unsigned char* d = dst + (g * KC << 7) + (r << 4);
        for (int c = lane >> 3; c < KC; c += 4) cp_async16(d + (c << 7), in ? s + 16 * c : base, in ? 16 : 0);
    }
    cp_async_commit();
}

// CW labels (a multiple of 8) of each of the warp's 32 rows, from tensor
// memory columns `taddr` on, scaled by the row's `inv` and stored through the
// warp's transpose area: CW * s / 16 consecutive lanes
// write one row's piece.  `rows`: the rows that exist; `row`: bytes per row.
template <int CW, typename OT>
__device__ __forceinline__ void store_piece(uint32_t taddr, float inv, unsigned char* s_tr, unsigned char* out,
                                            int64_t row, int rows) {
    const int lane = threadIdx.x & 31;
    uint32_t t[CW / 8][8];
#pragma unroll
    for (int h = 0; h < CW; h += 8) tmem_ld8(taddr + (uint32_t)h, t[h / 8]);
#pragma unroll
    for (int h = 0; h < CW; h += 8) {
        tmem_wait8(t[h / 8]);  // (the first one waits for all)
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(t[h / 8][i]);
        if constexpr (sizeof(OT) == 2) {
            uint32_t w[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const __nv_bfloat162 b2 = __floats2bfloat162_rn(v[2 * i] * inv, v[2 * i + 1] * inv);
                w[i] = *reinterpret_cast<const uint32_t*>(&b2);
            }
            *reinterpret_cast<uint4*>(s_tr + lane * QROW + h * 2) = make_uint4(w[0], w[1], w[2], w[3]);
        } else {
            float4* o = reinterpret_cast<float4*>(s_tr + lane * QROW + h * 4);
            o[0] = make_float4(v[0] * inv, v[1] * inv, v[2] * inv, v[3] * inv);
            o[1] = make_float4(v[4] * inv, v[5] * inv, v[6] * inv, v[7] * inv);
        }
    }
    __syncwarp();
    constexpr int LPR = CW * (int)sizeof(OT) / 16, RPS = 32 / LPR;  // lanes per row, rows per step
    const int r = lane / LPR, part = lane % LPR;
    const unsigned char* src = s_tr + r * QROW + part * 16;
    unsigned char* dst = out + r * row + part * 16;
    const int64_t step = RPS * row;
#pragma unroll
    for (int i = 0; i < LPR; ++i) {
        const uint4 q = *reinterpret_cast<const uint4*>(src + i * RPS * QROW);
        if (r + i * RPS < rows) *reinterpret_cast<uint4*>(dst) = q;
        dst += step;
    }
    __syncwarp();  // before the area's next piece
}

// proximity parameters of two queries, pairwise: (-p_q), then with
// h = -log2(e)/2 and f = -log2(e) the entries h xx, h yy, h zz, f xy, f xz,
// f yz of Sigma_q^-1, so that D = 2^(quadratic form in d)
struct alignas(16) QPair {
    float2 nx, ny, nz, xx, yy, zz, xy, xz, yz, pad;
};
static_assert(sizeof(QPair) == 80, "five 16-byte loads");

template <int QB, typename OT>
__global__ void __launch_bounds__(QTHREADS, QB == 2 ? 2 : 3) k_query_wide(int64_t N, int nq, int KC, int ncols, int nbuf,
                                                           const __nv_bfloat16* __restrict__ f_ins,
                                                           const float* __restrict__ means,
                                                           const __nv_bfloat16* __restrict__ f_q,
                                                           const float* __restrict__ p_q,
                                                           const float* __restrict__ prec, OT* __restrict__ out,
                                                           int32_t* __restrict__ err) {
    constexpr int QT = QM * QB;  // Gaussians per tile
    const int dim = 8 * KC;
    extern __shared__ __align__(1024) unsigned char smem[];
    const uint32_t abytes = (uint32_t)(QT * dim * 2);
    unsigned char* sA = smem;                                  // nbuf x [QT x dim] core matrices, tiles in turn
    unsigned char* sB = sA + nbuf * (size_t)abytes;              // [nq x dim] core matrices
    QPair* s_qp = reinterpret_cast<QPair*>(sB + (size_t)nq * dim * 2);  // [nq / 2]
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    __shared__ float s_sum[2][QT];  // the query halves' sums of exp(A)

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // this warp's transpose area: 32 rows of 64 bytes, padded by 16
    unsigned char* s_tr = reinterpret_cast<unsigned char*>(s_qp + nq / 2) + warp * 32 * QROW;
    const int64_t ntiles = (N + QT - 1) / QT;

    int64_t tile = blockIdx.x;
    // queries: operand B and the per-query proximity parameters, once per CTA
    copy_rows(sB, f_q, KC, nq, nq);
    if (tile < ntiles) copy_rows(sA, f_ins + tile * QT * dim, KC, QT, N - tile * QT);
    for (int q = tid; q < nq; q += blockDim.x) {
        const float h = -0.5f * QLOG2E, f = -QLOG2E;
        const float* P = prec + 6 * q;
        float* d = reinterpret_cast<float*>(s_qp + (q >> 1)) + (q & 1);
        d[0] = -p_q[3 * q]; d[2] = -p_q[3 * q + 1]; d[4] = -p_q[3 * q + 2];
        d[6] = h * P[0]; d[8] = h * P[1]; d[10] = h * P[2];
        d[12] = f * P[3]; d[14] = f * P[4]; d[16] = f * P[5];
    }
    if (tid == 0) {
        s_abort = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");  // visible to the MMA's arrive
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(QB * ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;
    const int half = warp >> 2, ql = (warp & 3) * 32 + lane;  // query half and TMEM lane
    const int cb = half * (nq >> 1), ce = cb + (nq >> 1);     // this thread's queries (a multiple of 8)
    const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16);  // this warp's lanes, column 0
    const uint32_t bar = smem_u32(&s_bar);
    const uint32_t idesc = mma_idesc(nq);
    uint32_t phase = 0;

    // this thread's Gaussians of the tile (TMEM lane ql of each block), loaded a tile ahead
    float np[QB][3];
    auto load_centres = [&](int64_t t) {
#pragma unroll
        for (int b = 0; b < QB; ++b) {
            const int64_t g = t * QT + b * QM + ql;
#pragma unroll
            for (int i = 0; i < 3; ++i) np[b][i] = g < N ? __ldg(means + 3 * g + i) : 0.0f;
        }
    };
    load_centres(tile);
    uint32_t buf = 0;
    for (; tile < ntiles; tile += gridDim.x, buf ^= (uint32_t)(nbuf - 1)) {
        const int64_t g0 = tile * QT, nt = tile + gridDim.x;
        cp_async_wait_all();  // this thread's part of the tile
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // shared-memory writes -> tensor core reads
        __syncthreads();
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int b = 0; b < QB; ++b)
                for (int s = 0; s < KC / 2; ++s) {  // K = 16 per MMA: two 16-byte chunks
                    const uint64_t da = smem_desc(smem_u32(sA) + buf * abytes + (uint32_t)(b * QM * dim * 2) + 256u * s, 128u, KC * 128u);
                    const uint64_t db = smem_desc(smem_u32(sB) + 256u * s, 128u, KC * 128u);
                    asm volatile(
                        "{\n\t.reg .pred p;\n\t"
                        "setp.ne.b32 p, %4, 0;\n\t"
                        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem + (uint32_t)(b * ncols)),
                        "l"(da), "l"(db), "r"(idesc), "r"(s)
                        : "memory");
                }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                         : "memory");
        }
        // the next tile's rows: into the other buffer from here on (its last MMAs
        // were waited for a tile ago), or into the only one once it has been read
        if (nbuf == 2 && nt < ntiles) copy_rows(sA + (buf ^ 1u) * abytes, f_ins + nt * QT * dim, KC, QT, N - nt * QT);
        float2 px[QB], py[QB], pz[QB], sum2[QB];
#pragma unroll
        for (int b = 0; b < QB; ++b) {
            px[b] = make_float2(np[b][0], np[b][0]);
            py[b] = make_float2(np[b][1], np[b][1]);
            pz[b] = make_float2(np[b][2], np[b][2]);
            sum2[b] = make_float2(0.0f, 0.0f);
        }
        load_centres(nt);
        if (!mbar_wait(bar, phase)) s_abort = 1;
        phase ^= 1u;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        __syncthreads();
        if (s_abort) break;
        if (nbuf == 1 && nt < ntiles) copy_rows(sA, f_ins + nt * QT * dim, KC, QT, N - nt * QT);

        uint32_t r[QB][8];  // the next 8 columns, read while the current ones are worked on
#pragma unroll
        for (int b = 0; b < QB; ++b) tmem_ld8(tlane + (uint32_t)(b * ncols + cb), r[b]);
        for (int c0 = cb; c0 < ce; c0 += 8) {
            float v[QB][8];
#pragma unroll
            for (int b = 0; b < QB; ++b) {
                tmem_wait8(r[b]);
#pragma unroll
                for (int i = 0; i < 8; ++i) v[b][i] = __uint_as_float(r[b][i]);
            }
            if (c0 + 8 < ce) {
#pragma unroll
                for (int b = 0; b < QB; ++b) tmem_ld8(tlane + (uint32_t)(b * ncols + c0 + 8), r[b]);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const QPair Q = s_qp[(c0 >> 1) + i];
#pragma unroll
                for (int b = 0; b < QB; ++b) {
                    const float2 dx = __fadd2_rn(px[b], Q.nx), dy = __fadd2_rn(py[b], Q.ny), dz = __fadd2_rn(pz[b], Q.nz);
                    // log2 D = -log2(e)/2 d^T Sigma^-1 d
                    const float2 t = __ffma2_rn(Q.xx, dx, __ffma2_rn(Q.xy, dy, __fmul2_rn(Q.xz, dz)));
                    const float2 u = __ffma2_rn(__ffma2_rn(Q.yy, dy, __fmul2_rn(Q.yz, dz)), dy,
                                                __fmul2_rn(__fmul2_rn(Q.zz, dz), dz));
                    const float2 l = __ffma2_rn(t, dx, u);
                    // log2(e) A = log2(e) S D, S = 1 / (1 + e^-logit) the sigmoid
                    // (scalar: the constants are immediates)
                    const float wx = fmaf(ex2_approx(-QLOG2E * v[b][2 * i]), QLN2, QLN2);
                    const float wy = fmaf(ex2_approx(-QLOG2E * v[b][2 * i + 1]), QLN2, QLN2);
                    v[b][2 * i] = ex2_approx(rcp_approx(wx) * ex2_approx(l.x));  // exp(A)
                    v[b][2 * i + 1] = ex2_approx(rcp_approx(wy) * ex2_approx(l.y));
                }
            }
#pragma unroll
            for (int b = 0; b < QB; ++b) {
#pragma unroll
                for (int i = 0; i < 8; i += 2) {
                    sum2[b].x += v[b][i];
                    sum2[b].y += v[b][i + 1];
                }
                tmem_st8(tlane + (uint32_t)(b * ncols + c0), v[b]);
            }
        }
#pragma unroll
        for (int b = 0; b < QB; ++b) s_sum[half][b * QM + ql] = sum2[b].x + sum2[b].y;
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // pass 2: 32 rows of one block (QB = 2: all its queries; QB = 1: this
        // half of them), in pieces of 64 bytes per row, then 16 and 8 columns
        {
            const int b = QB == 2 ? half : 0, e0 = QB == 2 ? 0 : cb, e1 = QB == 2 ? nq : ce;
            const int64_t r0 = g0 + b * QM + (warp & 3) * 32;
            const int rows = (int)min((int64_t)32, max((int64_t)0, N - r0)), sl = b * QM + ql;
            const float inv = 1.0f / (s_sum[0][sl] + s_sum[1][sl]);
            const uint32_t ta = tlane + (uint32_t)(b * ncols);
            unsigned char* o = reinterpret_cast<unsigned char*>(out + r0 * nq);
            const int64_t row = (int64_t)nq * sizeof(OT);
            int c0 = e0;
            for (; c0 + QCOLS<OT> <= e1; c0 += QCOLS<OT>)
                store_piece<QCOLS<OT>, OT>(ta + c0, inv, s_tr, o + c0 * sizeof(OT), row, rows);
            if (QCOLS<OT> > 16 && c0 + 16 <= e1) {
                store_piece<16, OT>(ta + c0, inv, s_tr, o + c0 * sizeof(OT), row, rows);
                c0 += 16;
            }
            if (c0 < e1) store_piece<8, OT>(ta + c0, inv, s_tr, o + c0 * sizeof(OT), row, rows);
        }
        // every lane's reads of the accumulators are done before the next
        // tile's MMAs (issued after the barrier at the loop's head)
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
    cp_async_wait_all();  // (a tile being copied when the loop was left early)
    if (s_abort && tid == 0) atomicExch(err, 1);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(QB * ncols) : "memory");
}

// operands A and B, the queries' parameters and the warps' transpose areas
size_t query_smem(int qb, int nbuf, int nq, int dim) {
    return (size_t)QM * qb * nbuf * dim * 2 + (size_t)nq * dim * 2 + (size_t)nq / 2 * sizeof(QPair) + (size_t)QTHREADS * QROW;
}

template <int QB, typename OT>
cudaError_t launch_qb(int64_t N, int nq, int dim, int ncols, int nbuf, const void* f_ins, const float* means, const void* f_q,
                      const float* p_q, const float* prec, void* out, int32_t* err, int num_sms, cudaStream_t stream) {
    size_t smem = query_smem(QB, nbuf, nq, dim);
    auto kern = k_query_wide<QB, OT>;
    // resident CTAs per SM: by the registers (the launch bounds), the SM's
    // tensor memory (512 columns) and shared memory.  The request is raised until
    // no more than these fit: a CTA beyond them would wait for tensor memory until
    // another one has done all its tiles (865k x 144 x 32 in FP32: 306 us, 195.02 without)
    const int per_sm = std::max(1, std::min({QB == 2 ? 2 : 3, 512 / (QB * ncols), (int)(227 * 1024 / (smem + 4 * 1024))}));
    smem = std::max(smem, (size_t)(227 * 1024 / (per_sm + 1)));
    cudaError_t e = open_smem((const void*)kern);
    if (e != cudaSuccess) return e;
    const int64_t ntiles = (N + QM * QB - 1) / (QM * QB);
    const int grid = (int)std::min<int64_t>(ntiles, (int64_t)per_sm * num_sms);
    kern<<<grid, QTHREADS, smem, stream>>>(N, nq, dim / 8, ncols, nbuf, static_cast<const __nv_bfloat16*>(f_ins), means,
                                           static_cast<const __nv_bfloat16*>(f_q), p_q, prec, static_cast<OT*>(out),
                                           err);
    e = cudaGetLastError();
    if (e == cudaSuccess) kernel_mark(stream);
    return e;
}

}  // namespace

cudaError_t launch_query_wide(int64_t N, int nq, int dim, const void* f_ins, const float* means, const void* f_q,
                                const float* p_q, const float* prec, void* out, int out_bf16, int32_t* err,
                                int num_sms, cudaStream_t stream) {
    int ncols = 32;  // tensor-memory columns of one accumulator
    while (ncols < nq) ncols <<= 1;
    // two Gaussians per thread where two CTAs of them fit an SM (with two
    // operand buffers, else with one) and N leaves each a tile
    auto fit2 = [&](int nbuf) { return 2 * (query_smem(2, nbuf, nq, dim) + 4 * 1024) <= 227 * 1024; };
    const bool two = 4 * ncols <= 512 && fit2(1) && N > (int64_t)4 * QM * num_sms;
    const int nbuf = two && !fit2(2) ? 1 : 2;
    auto go = [&](auto qb) {
        constexpr int QB = decltype(qb)::value;
        return out_bf16 ? launch_qb<QB, __nv_bfloat16>(N, nq, dim, ncols, nbuf, f_ins, means, f_q, p_q, prec, out, err, num_sms, stream)
                        : launch_qb<QB, float>(N, nq, dim, ncols, nbuf, f_ins, means, f_q, p_q, prec, out, err, num_sms, stream);
    };
    return two ? go(std::integral_constant<int, 2>{}) : go(std::integral_constant<int, 1>{});
}

}  // namespace fss
