// fp32 path of the TTL step, state upkeep kernels and the memory read.
//
// When d_in + d_out <= 512 the fp32 path runs every segment of a call in one launch with
// the rows resident on chip (ttl_resident_f32_kernel, below).  Otherwise it runs two
// kernels a segment (three with the squared-error pre-pass): register-tiled FFMA
// contractions in fp32 throughout (nt_tile, tn_tile), computing the same two phases as the
// bf16 tensor-core path:
//   phase A  H = U W1^T, R = Y W2^T (Y = [K || V]); A = SiLU(H);
//            dH = c_t R * SiLU'(H), At = c_t A with c_t = -eta_t / T'   (Eq. 10)
//   phase B  G1 = dH^T U, G2 = At^T Y; mu = beta mu + G; W = s W_raw - mu  (Eq. 8)
// where s is the pending row renormalisation scale of the previous segment
// (App. A), applied lazily so that no extra pass over the weights is needed.
// The loss L_s = -(1/T') sum_t sum_h A_th R_th equals Eq. 7's segment mean
// because sum_h A_th R_th = y_t . (A_t W2) = y_t . M(u_t).
#include <mutex>
#include <type_traits>

#include "mone_common.cuh"
#include "per_device.h"

namespace mone {

namespace {

constexpr int TM = 64, TN = 64, TK = 64;

// acc[i][j] += sum_k A(m0 + ty*MR + i, k) * B(n0 + tx*4 + j, k) for one (16 MR) x 64 tile.
// A(m, k) = A[m*sam + k*sak]; rows m >= m_valid and k >= k_valid read as 0.
template <int MR>
__device__ __forceinline__ void simt_tile(float (&acc)[MR][4], const float* A, long long sam, long long sak,
                                          const float* B, long long sbn, long long sbk, int K, int m_valid,
                                          int k_valid, float (*As)[16 * MR + 4], float (*Bs)[TN + 4]) {
    constexpr int TMR = 16 * MR;  // rows of the tile
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    for (int k0 = 0; k0 < K; k0 += TK) {
        // TMR x TK elements of A and 64 x TK of B, TK consecutive along the contiguous dimension
        float av[TMR * TK / 256], bv[TN * TK / 256];
#pragma unroll
        for (int r = 0; r < TMR * TK / 256; ++r) {
            const int e = tid + 256 * r;
            int m, k;
            if (sak == 1) { m = e / TK; k = e % TK; } else { m = e % TMR; k = e / TMR; }
            av[r] = (m < m_valid && k0 + k < k_valid) ? A[m * sam + (k0 + k) * sak] : 0.0f;
        }
#pragma unroll
        for (int r = 0; r < TN * TK / 256; ++r) {
            const int e = tid + 256 * r;
            int n, kb;
            if (sbk == 1) { n = e / TK; kb = e % TK; } else { n = e % TN; kb = e / TN; }
            bv[r] = (k0 + kb < k_valid) ? B[n * sbn + (k0 + kb) * sbk] : 0.0f;
        }
#pragma unroll
        for (int r = 0; r < TMR * TK / 256; ++r) {
            const int e = tid + 256 * r;
            int m, k;
            if (sak == 1) { m = e / TK; k = e % TK; } else { m = e % TMR; k = e / TMR; }
            As[k][m] = av[r];
        }
#pragma unroll
        for (int r = 0; r < TN * TK / 256; ++r) {
            const int e = tid + 256 * r;
            int n, kb;
            if (sbk == 1) { n = e / TK; kb = e % TK; } else { n = e % TN; kb = e / TN; }
            Bs[kb][n] = bv[r];
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < TK; ++k) {
            float a[MR], b[4];
#pragma unroll
            for (int i = 0; i < MR; ++i) a[i] = As[k][ty * MR + i];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = Bs[k][tx * 4 + j];
#pragma unroll
            for (int i = 0; i < MR; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
}

__device__ __forceinline__ void cp_async16(float* dst, const float* src, int src_bytes) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(float* dst, const float* src, int src_bytes) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ---- tiled contractions of the fp32 phases: threads as TY (ty) x 16 (tx), TM x TN outputs each, slabs of the
// contraction through a ring of cp.async stages.  (TM + TN) 16-byte shared-memory loads feed 4 TM TN
// multiply-adds a thread; a warp is 4 (ty) x 8 (tx) threads, so a half warp's load is at most 128
// distinct bytes, one wavefront (2 x 16 threads: two for the tx operand).  Multiply-adds are packed pairs: of
// even and odd k in nt_tile, of neighbouring columns in tn_tile.
__device__ __forceinline__ int tile_tx() { return (threadIdx.x & 7) | ((threadIdx.x >> 5 & 1) << 3); }
__device__ __forceinline__ int tile_ty() { return (threadIdx.x >> 3 & 3) | (threadIdx.x >> 6 << 2); }

// Both operands with k contiguous: acc[i][j] += sum_k A[ty + TY i][k] B[tx + 16 j][k], rows of A from
// m_valid on read as 0.  K a multiple of 32; rows 36 floats apart, so the 8 rows of a quarter warp start
// in 8 bank groups.
constexpr int NT_K = 32, NT_LD = NT_K + 4, NT_ST = 3;
template <int TM, int TN, int TY> constexpr size_t nt_smem() { return sizeof(float) * NT_ST * (TY * TM + 16 * TN) * NT_LD; }

template <int TM, int TN, int TY>
__device__ __forceinline__ void nt_tile(float (&acc)[TM][TN], const float* A, long long lda, const float* B, long long ldb,
                                        int K, int m_valid, float* sm) {
    constexpr int BM = TY * TM, BN = 16 * TN, STAGE = (BM + BN) * NT_LD;
    const int tid = threadIdx.x, tx = tile_tx(), ty = tile_ty(), n = K / NT_K;
    // the thread's 16-byte pieces of a slab: rows r0 + 2 TY u (of A, then of B), columns p0
    const int r0 = tid >> 3, p0 = 4 * (tid & 7);
    const float *ga = A + r0 * lda + p0, *gb = B + r0 * ldb + p0;
    auto load = [&](int s) {
        float* d = sm + (s % NT_ST) * STAGE + r0 * NT_LD + p0;
#pragma unroll
        for (int u = 0; u < BM / (2 * TY); ++u) {
            const bool v = r0 + 2 * TY * u < m_valid;
            cp_async16(d + 2 * TY * u * NT_LD, v ? ga + 2 * TY * u * lda + s * NT_K : A, v ? 16 : 0);
        }
#pragma unroll
        for (int u = 0; u < BN / (2 * TY); ++u)
            cp_async16(d + (BM + 2 * TY * u) * NT_LD, gb + 2 * TY * u * ldb + s * NT_K, 16);
    };
    uint64_t p[TM][TN] = {};  // sums over even and odd k
    // the ring may still be read from an earlier contraction of this kernel
    __syncthreads();
#pragma unroll
    for (int s = 0; s < NT_ST - 1; ++s) {
        if (s < n) load(s);
        cp_async_commit();
    }
    for (int s = 0; s < n; ++s) {
        cp_async_wait<NT_ST - 2>();
        __syncthreads();
        if (s + NT_ST - 1 < n) load(s + NT_ST - 1);
        cp_async_commit();
        const float* As = sm + (s % NT_ST) * STAGE + ty * NT_LD;
        const float* Bs = sm + (s % NT_ST) * STAGE + (BM + tx) * NT_LD;
#pragma unroll
        for (int k = 0; k < NT_K; k += 4) {
            ulonglong2 a[TM], b[TN];  // two packed pairs of k each
#pragma unroll
            for (int i = 0; i < TM; ++i) a[i] = *reinterpret_cast<const ulonglong2*>(As + TY * i * NT_LD + k);
#pragma unroll
            for (int j = 0; j < TN; ++j) b[j] = *reinterpret_cast<const ulonglong2*>(Bs + 16 * j * NT_LD + k);
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) p[i][j] = fma_f32x2(a[i].x, b[j].x, p[i][j]);
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) p[i][j] = fma_f32x2(a[i].y, b[j].y, p[i][j]);
        }
    }
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const float2 v = unpack_f32x2(p[i][j]);
            acc[i][j] += v.x + v.y;
        }
}

// Both operands with the output dimension contiguous: acc[i][j] += sum_k A[k][m(i)] B[k][n(j)] with
// m(i) = 4 ty + 4 TY (i / 4) + i % 4 and n(j) = 4 tx + 64 (j / 4) + j % 4 (tile TY TM x 16 TN).  Rows k >= kv read as 0.
constexpr int TN_K = 16, TN_ST = 3;
template <int TM, int TN, int TY> constexpr size_t tn_smem() { return sizeof(float) * TN_ST * TN_K * (TY * TM + 16 * TN); }

template <int TM, int TN, int TY>
__device__ __forceinline__ void tn_tile(float (&acc)[TM][TN], const float* A, long long lda, const float* B, long long ldb,
                                        int K, int kv, float* sm) {
    static_assert(TM % 4 == 0 && TN % 4 == 0, "outputs in groups of four");
    constexpr int BM = TY * TM, BN = 16 * TN, LD = BM + BN, STAGE = TN_K * LD;
    const int tid = threadIdx.x, tx = tile_tx(), ty = tile_ty(), n = (K + TN_K - 1) / TN_K;
    auto load = [&](int s) {
        float* d = sm + (s % TN_ST) * STAGE;
#pragma unroll
        for (int u = 0; u < STAGE / 4 / (16 * TY); ++u) {
            const int e = tid + 16 * TY * u, r = e / (LD / 4), c = 4 * (e % (LD / 4)), k = s * TN_K + r;
            const float* src = c < BM ? A + k * lda + c : B + k * ldb + (c - BM);
            cp_async16(d + r * LD + c, k < kv ? src : A, k < kv ? 16 : 0);
        }
    };
#pragma unroll
    for (int s = 0; s < TN_ST - 1; ++s) {
        if (s < n) load(s);
        cp_async_commit();
    }
    for (int s = 0; s < n; ++s) {
        cp_async_wait<TN_ST - 2>();
        __syncthreads();
        if (s + TN_ST - 1 < n) load(s + TN_ST - 1);
        cp_async_commit();
        const float* S = sm + (s % TN_ST) * STAGE;
#pragma unroll
        for (int k = 0; k < TN_K; ++k) {
            float a[TM], b[TN];
#pragma unroll
            for (int i = 0; i < TM; i += 4)
                *reinterpret_cast<float4*>(a + i) = *reinterpret_cast<const float4*>(S + k * LD + 4 * ty + TY * i);
#pragma unroll
            for (int j = 0; j < TN; j += 4)
                *reinterpret_cast<float4*>(b + j) = *reinterpret_cast<const float4*>(S + k * LD + BM + 4 * tx + 16 * j);
#pragma unroll
            for (int i = 0; i < TM; ++i) {  // pairs of columns: half the issue slots of single multiply-adds
                const uint64_t aa = pack_f32x2(a[i], a[i]);
#pragma unroll
                for (int j = 0; j < TN; j += 2) {
                    const float2 v = unpack_f32x2(fma_f32x2(aa, pack_f32x2(b[j], b[j + 1]), pack_f32x2(acc[i][j], acc[i][j + 1])));
                    acc[i][j] = v.x;
                    acc[i][j + 1] = v.y;
                }
            }
        }
    }
}

struct F32SegArgs {
    int d_in, d_hid, d_out, T, Tp, c0, paper, momentum, renorm_pending, parity, C;
    long long tok0;           // per-token tables: entry of token t of chain cs is [cs * win + tok0 + t]
    int win;
    float lr;
    const float *U;           // base of the memory input rows of this segment for chain cz (see below)
    long long u_cstride;      // element stride between chains of U
    const float *K, *V;
    long long y_cstride;
    long long row_avail;      // input rows available from the segment start
    const float* eta_in;      // plain mode caller rates (already offset to the segment) or null
    long long eta_cstride;
    const float* eta;         // paper mode rates [C][T] (state chain index)
    const float* dbeta;       // [C][T]
    const float* b_beta;
    float *W1, *W2, *mu1, *mu2;
    const float *n1, *n2;
    float* sumsq;             // [2][2][C][d_hid]
    float *dH, *At;           // [C][T][d_hid]
    float* loss;
    float* step_sq;           // [nc] squared norm of this segment's Eq. 8 step, or null
    int* status;
};

__device__ __forceinline__ const float* ss_ptr(const F32SegArgs& a, int parity, int which) {
    return a.sumsq + ((size_t)(parity * 2 + which) * a.C) * a.d_hid;
}

// Phase A: TY TM tokens x 16 TN hidden units a CTA, H over d_in and R over d_out in turn.  Bound by shared
// memory (TM = 4) or FMA issue (TM = 8) and the last wave: 4 chains of 1024 -> 1024 -> 1024, T = 256 (256
// tiles of 64 x 64) take 123 us, 35 TFLOP/s (with 256 threads of 4 x 4 outputs: single multiply-adds 126 us,
// paired 130; 32 x 64 tiles with a slab read, waited for and then multiplied: 250 us; 64 x 128 tiles, one CTA an
// SM: 152 us).
template <int TM, int TN, int TY>
__global__ void __launch_bounds__(16 * TY, 2) phase_a_f32_kernel(const F32SegArgs a) {
    extern __shared__ float4 f32_smem[];
    __shared__ float red[8];
    float* sm = reinterpret_cast<float*>(f32_smem);
    constexpr int BM = TY * TM, BN = 16 * TN;
    const int tid = threadIdx.x, tx = tile_tx(), ty = tile_ty();
    const int t0 = blockIdx.x * BM, h0 = blockIdx.y * BN, cz = blockIdx.z, cs = a.c0 + cz;
    int m_valid = (int)min((long long)min(BM, a.Tp - t0), a.row_avail - t0);
    if (m_valid < 0) m_valid = 0;
    // zero this segment's row sums of squares (read by phase B of this segment)
    if (blockIdx.x == 0 && tid < BN) {
        float* cur = a.sumsq + ((size_t)(a.parity * 2) * a.C + cs) * a.d_hid + h0 + tid;
        cur[0] = 0.f;
        cur[(size_t)a.C * a.d_hid] = 0.f;
    }
    float accH[TM][TN] = {}, accR[TM][TN] = {};
    if (m_valid > 0) {
        const int dh = a.d_out / 2;
        const float* W2 = a.W2 + ((size_t)cs * a.d_hid + h0) * a.d_out;
        nt_tile<TM, TN, TY>(accH, a.U + cz * a.u_cstride + (long long)t0 * a.d_in, a.d_in, a.W1 + ((size_t)cs * a.d_hid + h0) * a.d_in,
                a.d_in, a.d_in, m_valid, sm);
        nt_tile<TM, TN, TY>(accR, a.K + cz * a.y_cstride + (long long)t0 * dh, dh, W2, a.d_out, dh, m_valid, sm);
        nt_tile<TM, TN, TY>(accR, a.V + cz * a.y_cstride + (long long)t0 * dh, dh, W2 + dh, a.d_out, dh, m_valid, sm);
    }
    const float* prev1 = ss_ptr(a, a.parity ^ 1, 0) + (size_t)cs * a.d_hid;
    const float* prev2 = ss_ptr(a, a.parity ^ 1, 1) + (size_t)cs * a.d_hid;
    float ct[TM];
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int t = t0 + ty + TY * i;
        ct[i] = 0.f;
        if (t < a.Tp && t - t0 < m_valid) {
            const float e = a.paper ? a.eta[(size_t)cs * a.win + a.tok0 + t]
                                    : (a.eta_in ? a.eta_in[cz * a.eta_cstride + t] : a.lr);
            ct[i] = -e / (float)a.Tp;
        }
    }
    float lsum = 0.f;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
        const int h = h0 + tx + 16 * j;
        const float s1 = a.renorm_pending ? renorm_scale(a.n1[(size_t)cs * a.d_hid + h], prev1[h]) : 1.f;
        const float s2 = a.renorm_pending ? renorm_scale(a.n2[(size_t)cs * a.d_hid + h], prev2[h]) : 1.f;
#pragma unroll
        for (int i = 0; i < TM; ++i) {
            const size_t o = ((size_t)cs * a.T + t0 + ty + TY * i) * a.d_hid + h;
            const float hv = accH[i][j] * s1;
            const float rv = accR[i][j] * s2;
            const float sg = sigmoidf_(hv);
            const float av = hv * sg;
            const float dsilu = sg * (1.f + hv * (1.f - sg));
            lsum += av * rv;
            a.dH[o] = ct[i] * rv * dsilu;
            a.At[o] = ct[i] * av;
        }
    }
    if (a.loss) {
        lsum = warp_sum(lsum);
        if ((tid & 31) == 0) red[tid >> 5] = lsum;
        __syncthreads();
        if (tid == 0) {
            float tot = 0.f;
            for (int w = 0; w < TY / 2; ++w) tot += red[w];
            atomicAdd(&a.loss[cz], -tot / (float)a.Tp);
        }
    }
}

// Phase B: TY TM hidden rows x 16 TN columns of W1, or of the K or V half of W2, a CTA.  The same 4
// chains: 105 us, 41 TFLOP/s, with 128 x 128 tiles and paired multiply-adds (single ones 122 us; 64 x 64
// tiles 133 us; the 32 x 64 tiles before them 344 us).
template <int TM, int TN, int TY>
__global__ void __launch_bounds__(16 * TY, 32 / TY) phase_b_f32_kernel(const F32SegArgs a) {
    extern __shared__ float4 f32_smem[];
    __shared__ float red[8];
    __shared__ float s_beta;
    constexpr int BM = TY * TM, BN = 16 * TN;
    const int tid = threadIdx.x, tx = tile_tx(), ty = tile_ty();
    const int col0 = blockIdx.x * BN, h0 = blockIdx.y * BM, cz = blockIdx.z, cs = a.c0 + cz;
    const bool isW1 = col0 < a.d_in;
    const int kv = (int)min((long long)a.Tp, a.row_avail);
    // momentum decay beta_s = sigmoid(mean_t w_beta . x_t + b_beta)
    if (a.momentum) {
        float v = 0.f;
        for (int t = tid; t < a.Tp; t += 16 * TY) v += a.dbeta[(size_t)cs * a.win + a.tok0 + t];
        v = warp_sum(v);
        if ((tid & 31) == 0) red[tid >> 5] = v;
        __syncthreads();
        if (tid == 0) {
            float tot = 0.f;
            for (int w = 0; w < TY / 2; ++w) tot += red[w];
            s_beta = sigmoidf_(tot / (float)a.Tp + a.b_beta[cs]);
        }
    }
    float acc[TM][TN] = {};
    {
        const int dh = a.d_out / 2, o0 = col0 - a.d_in;
        const float* A = (isW1 ? a.dH : a.At) + (size_t)cs * a.T * a.d_hid + h0;
        const float* B = isW1 ? a.U + cz * a.u_cstride + col0 : (o0 < dh ? a.K + o0 : a.V + (o0 - dh)) + cz * a.y_cstride;
        tn_tile<TM, TN, TY>(acc, A, a.d_hid, B, isW1 ? a.d_in : dh, a.Tp, kv, reinterpret_cast<float*>(f32_smem));
    }
    const float beta = a.momentum ? s_beta : 0.f;  // tn_tile's first barrier has published it
    const int which = isW1 ? 0 : 1;
    const int width = isW1 ? a.d_in : a.d_out;
    const int c_local = isW1 ? col0 : col0 - a.d_in;
    const float* n0 = (isW1 ? a.n1 : a.n2) + (size_t)cs * a.d_hid;
    const float* prev = ss_ptr(a, a.parity ^ 1, which) + (size_t)cs * a.d_hid;
    float* cur = a.sumsq + ((size_t)(a.parity * 2 + which) * a.C + cs) * a.d_hid;
    bool finite = true;
    float step = 0.f;  // sum of mu_s^2 over this thread's elements
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int h = h0 + 4 * ty + 4 * TY * (i / 4) + i % 4;
        const float s = a.renorm_pending ? renorm_scale(n0[h], prev[h]) : 1.f;
        const size_t row = ((size_t)cs * a.d_hid + h) * width + c_local + 4 * tx;
        float* wrow = (isW1 ? a.W1 : a.W2) + row;
        float* mrow = a.momentum ? (isW1 ? a.mu1 : a.mu2) + row : nullptr;
        float ss = 0.f;
#pragma unroll
        for (int j = 0; j < TN; j += 4) {
            float4 w = *reinterpret_cast<const float4*>(wrow + 16 * j);
            float4 m = make_float4(acc[i][j], acc[i][j + 1], acc[i][j + 2], acc[i][j + 3]);
            if (mrow) {
                const float4 o = *reinterpret_cast<const float4*>(mrow + 16 * j);
                m = make_float4(fmaf(beta, o.x, m.x), fmaf(beta, o.y, m.y), fmaf(beta, o.z, m.z), fmaf(beta, o.w, m.w));
                *reinterpret_cast<float4*>(mrow + 16 * j) = m;
            }
            w = make_float4(s * w.x - m.x, s * w.y - m.y, s * w.z - m.z, s * w.w - m.w);
            *reinterpret_cast<float4*>(wrow + 16 * j) = w;
            finite = finite && isfinite(w.x) && isfinite(w.y) && isfinite(w.z) && isfinite(w.w);
            ss = fmaf(w.x, w.x, fmaf(w.y, w.y, fmaf(w.z, w.z, fmaf(w.w, w.w, ss))));
            step = fmaf(m.x, m.x, fmaf(m.y, m.y, fmaf(m.z, m.z, fmaf(m.w, m.w, step))));
        }
        ss += __shfl_xor_sync(0xffffffffu, ss, 4);
        ss += __shfl_xor_sync(0xffffffffu, ss, 2);
        ss += __shfl_xor_sync(0xffffffffu, ss, 1);
        if ((tx & 7) == 0) atomicAdd(&cur[h], ss);
    }
    if (a.step_sq) {
        step = warp_sum(step);
        if ((tid & 31) == 0) atomicAdd(&a.step_sq[cz], step);
    }
    if (!finite) atomicOr(a.status, DEV_NONFINITE);
}

F32SegArgs make_f32_args(const DevState& s, const SegWork& w) {
    F32SegArgs a{};
    a.d_in = s.d_in; a.d_hid = s.d_hid; a.d_out = s.d_out; a.T = s.T; a.Tp = w.Tp; a.c0 = w.c0;
    a.paper = s.mode == 1; a.momentum = s.momentum; a.renorm_pending = w.renorm_pending;
    a.tok0 = w.u_off; a.win = s.win_rows;
    a.parity = w.parity; a.C = s.C; a.lr = s.lr;
    const int dh = s.d_out / 2;
    if (a.paper) {
        a.U = reinterpret_cast<const float*>(s.U) + ((size_t)w.c0 * s.win_rows + w.u_off) * s.d_in;
        a.u_cstride = (long long)s.win_rows * s.d_in;
    } else {
        a.U = reinterpret_cast<const float*>(w.X) + w.row0 * s.d_in;
        a.u_cstride = w.x_cstride;
    }
    if (w.y_scratch) {  // squared error: the residual targets of this segment, rows from 0
        a.K = s.Kres32 + (size_t)w.c0 * s.T * dh;
        a.V = s.Vres32 + (size_t)w.c0 * s.T * dh;
        a.y_cstride = (long long)s.T * dh;
    } else {
        a.K = reinterpret_cast<const float*>(w.K) + w.row0 * dh;
        a.V = reinterpret_cast<const float*>(w.V) + w.row0 * dh;
        a.y_cstride = w.y_cstride;
    }
    a.row_avail = w.n_rows - w.row0;
    a.eta_in = w.eta_in ? w.eta_in + w.row0 : nullptr;
    a.eta_cstride = w.eta_cstride;
    a.eta = s.eta; a.dbeta = s.dbeta; a.b_beta = s.b_beta;
    a.W1 = s.W1; a.W2 = s.W2; a.mu1 = s.mu1; a.mu2 = s.mu2; a.n1 = s.n1; a.n2 = s.n2;
    a.sumsq = s.sumsq;
    a.dH = reinterpret_cast<float*>(s.dHt);
    a.At = reinterpret_cast<float*>(s.Att);
    a.loss = w.loss;
    a.step_sq = w.step_sq;
    a.status = s.status;
    return a;
}

// ------------------------------------------------------------------ squared-error pre-pass (fp32)
//
// Under the squared-error loss dL/dO = eta (M(u) - y) / T' = -eta (y - M(u)) / T', so the
// residual target y - M(u), with M(u) at the segment's starting weights, takes the place of
// y in both phases.  Two kernels: A' = SiLU(s1 H) s2 with the pending row scales folded in
// (so A' W2raw = A W2), written to the At scratch, which phase A overwrites only after
// the second kernel has read it; then the residual y - A' W2raw into the residual scratch
// and 1/2 |y - M(u)|^2 / T' into the loss.

// Tiles of 32 tokens x 64 outputs (2 x 4 per thread): short segments would leave most SMs idle on 64 x 64.
constexpr int A_MR = 2, A_TM = 16 * A_MR;

__global__ void __launch_bounds__(256) mse_hidden_f32_kernel(const F32SegArgs a) {
    __shared__ float As[TK][A_TM + 4], Bs[TK][TN + 4];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int t0 = blockIdx.x * A_TM, h0 = blockIdx.y * TN, cz = blockIdx.z, cs = a.c0 + cz;
    int m_valid = (int)min((long long)min(A_TM, a.Tp - t0), a.row_avail - t0);
    if (m_valid < 0) m_valid = 0;
    float acc[A_MR][4] = {};
    simt_tile(acc, a.U + cz * a.u_cstride + (long long)t0 * a.d_in, a.d_in, 1,
              a.W1 + ((size_t)cs * a.d_hid + h0) * a.d_in, a.d_in, 1, a.d_in, m_valid, a.d_in, As, Bs);
    const float* prev1 = ss_ptr(a, a.parity ^ 1, 0) + (size_t)cs * a.d_hid;
    const float* prev2 = ss_ptr(a, a.parity ^ 1, 1) + (size_t)cs * a.d_hid;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int h = h0 + tx * 4 + j;
        const float s1 = a.renorm_pending ? renorm_scale(a.n1[(size_t)cs * a.d_hid + h], prev1[h]) : 1.f;
        const float s2 = a.renorm_pending ? renorm_scale(a.n2[(size_t)cs * a.d_hid + h], prev2[h]) : 1.f;
#pragma unroll
        for (int i = 0; i < A_MR; ++i) {
            const int t = t0 + ty * A_MR + i;
            const float x = acc[i][j] * s1;
            a.At[((size_t)cs * a.T + t) * a.d_hid + h] = x * sigmoidf_(x) * s2;
        }
    }
}

__global__ void __launch_bounds__(256) mse_out_f32_kernel(const F32SegArgs a, float* Kres, float* Vres) {
    __shared__ float As[TK][A_TM + 4], Bs[TK][TN + 4];
    __shared__ float red[8];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int t0 = blockIdx.x * A_TM, o0 = blockIdx.y * TN, cz = blockIdx.z, cs = a.c0 + cz;
    const int dh = a.d_out / 2;
    float acc[A_MR][4] = {};
    simt_tile(acc, a.At + ((size_t)cs * a.T + t0) * a.d_hid, a.d_hid, 1, a.W2 + (size_t)cs * a.d_hid * a.d_out + o0,
              1, a.d_out, a.d_hid, min(A_TM, a.T - t0), a.d_hid, As, Bs);
    const bool kpart = o0 < dh;  // dh is a multiple of 64: a tile is all K or all V
    const int col0 = (kpart ? o0 : o0 - dh) + tx * 4;
    const float* Y = (kpart ? a.K : a.V) + cz * a.y_cstride + col0;
    float* R = (kpart ? Kres : Vres) + (size_t)cs * a.T * dh + col0;
    float lsum = 0.f;
#pragma unroll
    for (int i = 0; i < A_MR; ++i) {
        const int t = t0 + ty * A_MR + i;
        const bool live = t < a.Tp && t < a.row_avail;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float r = live ? Y[(long long)t * dh + j] - acc[i][j] : 0.f;
            R[(size_t)t * dh + j] = r;
            lsum = fmaf(r, r, lsum);
        }
    }
    if (a.loss) {
        lsum = warp_sum(lsum);
        if ((tid & 31) == 0) red[tid >> 5] = lsum;
        __syncthreads();
        if (tid == 0) {
            float tot = 0.f;
            for (int w = 0; w < 8; ++w) tot += red[w];
            atomicAdd(&a.loss[cz], 0.5f * tot / (float)a.Tp);
        }
    }
}

// ------------------------------------------------------------------ resident chains (fp32)
//
// When a chain's rows fit on chip, a whole call runs in one launch with the fast
// weights resident.  A CTA owns RB hidden units of one chain: their rows of W1 and
// W2, kept side by side as [W1 | W2] (width D = d_in + d_out) in shared memory, and
// their momentum too, with the gradient in registers.  Hidden units do not interact within a
// step: H[:, r] = U W1[r]^T and R[:, r] = Y W2[r]^T use only row r, dL/dO does not
// depend on W (Eq. 10), the gradient rows dW1[r] = dH[:, r]^T U and dW2[r] =
// At[:, r]^T Y use only column r of dH and At, and Eq. 8's renormalisation is per
// row.  So a CTA takes its rows through every segment of the call without waiting
// for any other CTA, and the weights cross HBM once per call instead of once per
// segment.  Each segment streams its rows [U | K | V] once, RC tokens at a time,
// into a double buffer (three bulk copies a chunk): forward (H, R), the backward epilogue
// (dH, At), then the gradient accumulation from the same staged rows.  At the end
// of the segment the update (momentum, W -= mu) and the row renormalisation are
// applied in place.
//
// 512 threads.  Forward: a warp takes two tokens of a chunk, lane l the columns 4 l + 128 i of [U | Y], with
// the W values of these columns in registers (RB = 4; from shared memory for RB = 8) and even and odd columns
// as packed pairs; the partial sums of H and R over the lanes are added by a transpose-reduction (16 shuffles
// for 16 sums), and the same warp finishes the epilogue.  Narrow chains with RB = 8 give each token 16 lanes instead.  Backward: a thread takes two columns of [W1 | W2]
// for all RB rows and one half of the chunk's tokens.  So a staged value is read from shared memory once in
// each direction.  The two phases of a chunk, each a chain of shared-memory and shuffle latencies between
// barriers with four warps a scheduler, bound it (49% of the issue slots used, 44% of the shared-memory rate).
// 4096 tokens of 256 -> 512 -> 256, T = 128: 406 us with the rows staged by a 16-byte copy a thread and scalar
// FFMA (16,500 warp instructions a chunk), 336 so (10,400).  Eight warps that take two tokens through both
// directions with the gradient of all four rows in registers, added up once a segment: 364 us.
constexpr int RES_RC = 32;                                             // tokens per streamed chunk
__host__ __device__ constexpr int res_ld(int D) { return (D + 31) / 32 * 32 + 16; }  // row pitch, floats

struct ResArgs {
    int d_in, d_out, d_hid, T, c0, win, paper, momentum, renorm, n_seg;
    long long n_tok;             // tokens of this launch, from its first row
    const float* U;              // first row of the launch, chain cz at U + cz * u_cstride
    long long u_cstride;
    const float *K, *V;          // first row of the launch
    long long y_cstride;
    const float* eta;            // paper mode: rates [C][win] at the launch's first row (state chain index)
    const float* dbeta;          // paper mode: w_beta . x_t, same layout
    const float* eta_in;         // plain mode: caller rates at the launch's first row, or null
    long long eta_cstride;
    float lr;
    const float* b_beta;
    float *W1, *W2, *mu1, *mu2;
    const float *n1, *n2;
    float* loss;                 // loss of segment seg of chain cz at loss[seg * m_sstride + cz], or null
    float* step_sq;              // squared norm of the Eq. 8 step, same layout, or null
    long long m_sstride;         // stride between segments of loss and step_sq (0: one accumulator)
    int* status;
};

constexpr int RES_NT = 512, RES_NW = RES_NT / 32;  // threads and warps of a resident CTA

// Sum of v over the CTA; every thread gets the total.  red: RES_NW floats.
__device__ __forceinline__ float block_sum_res(float v, float* red) {
    v = warp_sum(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < RES_NW; ++w) t += red[w];
    return t;
}

// LPT: lanes to a token of the forward, 32 (two tokens a lane) or 16 (one); widths up to DMAX.
template <int RB, int LPT, int DMAX>
__global__ void __launch_bounds__(RES_NT, 1) ttl_resident_f32_kernel(const ResArgs a) {
    // tokens of a lane, sums of a lane (H and R), 16-byte column pieces of a lane
    constexpr int RC = RES_RC, NW = RES_NW, TPL = LPT / 16, NV = 2 * TPL * RB, NI = DMAX / (4 * LPT);
    static_assert(LPT == 32 || (LPT == 16 && RB == 8), "lanes to a token");
    static_assert(RB == 4 || RB == 8, "rows per CTA");
    static_assert(RC == 2 * NW, "two tokens a warp");
    extern __shared__ float4 res_smem[];
    const int D = a.d_in + a.d_out, LD = res_ld(D), dh = a.d_out / 2;
    float* Ws = reinterpret_cast<float*>(res_smem);  // [RB][LD]
    float* Ps = Ws + RB * LD;                        // [RB][LD]: gradient rows from the second token half
    float* Ms = Ps + RB * LD;                        // [RB][LD]: momentum
    float* Xs = Ms + RB * LD;                        // [2][RC][D]: a chunk's U [RC][d_in], K and V [RC][dh]
    float* Gs = Xs + 2 * RC * D;                     // [RC][2][RB][2]: c dH, c A of the chunk, each twice (a packed pair)
    float* red = Gs + RC * 4 * RB;                   // [NW][2 RB]
    float* scl = red + NW * 2 * RB;                  // [2 RB] row scales, then beta
    float* etaS = scl + 2 * RB + 4;                  // [2][RC] rates of the chunk's tokens
    float* dbS = etaS + 2 * RC;                      // [2][RC] w_beta . x of the chunk's tokens
    float* nS = dbS + 2 * RC;                        // [2 RB] renormalisation targets
    __shared__ alignas(8) uint64_t bars[2];          // a chunk's rows have landed in buffer b
    const uint32_t full = smem_u32(bars);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int h0 = blockIdx.x * RB, cz = blockIdx.y, cs = a.c0 + cz;
    const float* Uc = a.U + cz * a.u_cstride;
    const float* Kc = a.K + cz * a.y_cstride;
    const float* Vc = a.V + cz * a.y_cstride;

    // stage up to RC token rows of segment seg, chunk ch into buffer b: three copies of whole rows
    // (thread 0 of the last warp), and the tokens' rates and w_beta . x terms.  Rows past the
    // segment keep what the buffer held: their rate is 0 and no gradient sum reads them
    auto issue = [&](int seg, int ch, int b) {
        const long long t_seg = (long long)seg * a.T;
        const int Tp = (int)min((long long)a.T, a.n_tok - t_seg);
        const int nvalid = min(RC, Tp - ch * RC);
        const long long r0 = t_seg + ch * RC;
        if (tid == RES_NT - 32) {
            float* d = Xs + b * RC * D;
            mbar_expect_tx(full + 8 * b, (uint32_t)(nvalid * D * 4));
            bulk_load(smem_u32(d), Uc + r0 * a.d_in, (uint32_t)(nvalid * a.d_in * 4), full + 8 * b);
            bulk_load(smem_u32(d + RC * a.d_in), Kc + r0 * dh, (uint32_t)(nvalid * dh * 4), full + 8 * b);
            bulk_load(smem_u32(d + RC * (a.d_in + dh)), Vc + r0 * dh, (uint32_t)(nvalid * dh * 4), full + 8 * b);
        }
        if (tid < 2 * RC) {
            const int t = tid & (RC - 1);
            const bool v = t < nvalid;
            const long long r = r0 + (v ? t : 0);
            if (tid < RC) {
                float* d = etaS + b * RC + t;
                if (a.paper)
                    cp_async4(d, a.eta + (size_t)cs * a.win + r, v ? 4 : 0);
                else if (a.eta_in)
                    cp_async4(d, a.eta_in + cz * a.eta_cstride + r, v ? 4 : 0);
                else
                    *d = v ? a.lr : 0.f;
            } else if (a.momentum) {
                cp_async4(dbS + b * RC + t, a.dbeta + (size_t)cs * a.win + r, v ? 4 : 0);
            }
        }
    };

    if (tid == 0) {
        mbar_init(full, 1);
        mbar_init(full + 8, 1);
        fence_mbar_init();
    }
    __syncthreads();
    issue(0, 0, 0);
    cp_async_commit();
    // resident rows
    for (int i = tid; i < RB * (D / 4); i += RES_NT) {
        const int r = i / (D / 4), c = 4 * (i - r * (D / 4));
        const size_t row = (size_t)cs * a.d_hid + h0 + r;
        const size_t o = c < a.d_in ? row * a.d_in + c : row * a.d_out + (c - a.d_in);
        *reinterpret_cast<float4*>(Ws + r * LD + c) = *reinterpret_cast<const float4*>((c < a.d_in ? a.W1 : a.W2) + o);
        if (a.momentum) *reinterpret_cast<float4*>(Ms + r * LD + c) = *reinterpret_cast<const float4*>((c < a.d_in ? a.mu1 : a.mu2) + o);
    }
    if (tid < 2 * RB) nS[tid] = (tid < RB ? a.n1 : a.n2)[(size_t)cs * a.d_hid + h0 + tid % RB];
    const float b_beta = a.momentum ? a.b_beta[cs] : 0.f;
    const int cb = 2 * (tid & 255), th = tid >> 8;  // backward: columns cb, cb + 1, tokens 16 th .. + 15 of a chunk
    const bool own = cb < D;                        // widths are even: both columns or none
    const int kind = cb < a.d_in ? 0 : 1;           // both in one matrix
    // the columns' place in a staged chunk: offset of token 0, and the floats between tokens
    auto x_col = [&](int c, int& stride) {
        stride = c < a.d_in ? a.d_in : dh;
        return c < a.d_in ? c : c < a.d_in + dh ? RC * a.d_in + (c - a.d_in) : RC * (a.d_in + dh) + (c - a.d_in - dh);
    };
    int bs;
    int bo = x_col(cb, bs);
    bo += th * (RC / 2) * bs;
    uint64_t acc[RB];  // packed pairs
#pragma unroll
    for (int r = 0; r < RB; ++r) acc[r] = 0;
    __syncthreads();
    // forward: LPT lanes to a token, a lane's columns 4 (lane % LPT) + 4 LPT i
    int fo[NI];
    const int fl = 4 * (lane % LPT);
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        int stride;
        fo[i] = x_col(fl + 4 * LPT * i, stride);
        fo[i] += (2 * warp + lane / LPT) * stride;
    }
    ulonglong2 w[RB == 4 ? NI : 1][RB == 4 ? RB : 1];  // two packed pairs each
    auto load_w = [&]() {
        if constexpr (RB == 4) {
#pragma unroll
            for (int i = 0; i < NI; ++i)
                if (fl + 4 * LPT * i < D)
#pragma unroll
                    for (int r = 0; r < RB; ++r) w[i][r] = *reinterpret_cast<const ulonglong2*>(Ws + r * LD + fl + 4 * LPT * i);
        }
    };
    load_w();

    bool finite = true;
    int buf = 0;
    uint32_t phase = 0;  // a buffer is filled every second chunk
    for (int seg = 0; seg < a.n_seg; ++seg) {
        const long long t_seg = (long long)seg * a.T;
        const int Tp = (int)min((long long)a.T, a.n_tok - t_seg);
        const int nch = (Tp + RC - 1) / RC;
        float lsum = 0.f, dbsum = 0.f;
        for (int ch = 0; ch < nch; ++ch) {
            cp_async_wait<0>();
            const bool landed = mbar_wait(full + 8 * buf, phase, a.status);
            if (!__syncthreads_and(landed)) {  // the chunk has landed; everyone is done with the other buffer and Gs
                drain_copies();
                return;
            }
            if (ch + 1 < nch)
                issue(seg, ch + 1, buf ^ 1);
            else if (seg + 1 < a.n_seg)
                issue(seg + 1, 0, buf ^ 1);
            cp_async_commit();
            const float* Xb = Xs + buf * RC * D;
            {   // ---- forward of tokens 2 warp, 2 warp + 1: v[(matrix TPL + token) RB + row]
                uint64_t p[NV] = {};  // even and odd columns packed
#pragma unroll
                for (int i = 0; i < NI; ++i) {
                    const int c = fl + 4 * LPT * i;
                    if (c >= D) continue;
                    const ulonglong2 xa = *reinterpret_cast<const ulonglong2*>(Xb + fo[i]);
                    ulonglong2 xb;
                    if constexpr (TPL == 2) xb = *reinterpret_cast<const ulonglong2*>(Xb + fo[i] + (c < a.d_in ? a.d_in : dh));
                    auto add = [&](auto mat) {
                        constexpr int o = decltype(mat)::value * TPL * RB;
#pragma unroll
                        for (int r = 0; r < RB; ++r) {
                            ulonglong2 wr;
                            if constexpr (RB == 4)
                                wr = w[i][r];
                            else
                                wr = *reinterpret_cast<const ulonglong2*>(Ws + r * LD + c);
                            p[o + r] = fma_f32x2(xa.y, wr.y, fma_f32x2(xa.x, wr.x, p[o + r]));
                            if constexpr (TPL == 2) p[o + RB + r] = fma_f32x2(xb.y, wr.y, fma_f32x2(xb.x, wr.x, p[o + RB + r]));
                        }
                    };
                    if (c < a.d_in)
                        add(std::integral_constant<int, 0>{});
                    else
                        add(std::integral_constant<int, 1>{});
                }
                float v[NV];
#pragma unroll
                for (int u = 0; u < NV; ++u) {
                    const float2 f = unpack_f32x2(p[u]);
                    v[u] = f.x + f.y;
                }
                // add the token's lanes' sums: afterwards the lanes whose top bits (of LPT) spell j hold sum j
#pragma unroll
                for (int n = NV, sft = LPT / 2; n > 1; n >>= 1, sft >>= 1) {
                    const bool upper = (lane & sft) != 0;
#pragma unroll
                    for (int u = 0; u < n / 2; ++u) {
                        const float send = upper ? v[u] : v[u + n / 2], keep = upper ? v[u + n / 2] : v[u];
                        v[u] = keep + __shfl_xor_sync(0xffffffffu, send, sft);
                    }
                }
                if (NV < LPT) v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
                // epilogue of output (token, row): c_t = -eta_t / T' (Eq. 10), A = SiLU(H); H is in the
                // lower half of the token's lanes, R LPT / 2 above
                const float rv = __shfl_down_sync(0xffffffffu, v[0], LPT / 2);
                constexpr int LPV = LPT / NV;  // lanes holding a sum
                const int j = lane % LPT / LPV, t = 2 * warp + j / RB + lane / LPT, r = j % RB, ts = ch * RC + t;
                if (lane % LPT < LPT / 2 && lane % LPV == 0) {
                    const float hv = v[0];
                    const float ct = ts < Tp ? -etaS[buf * RC + t] / (float)Tp : 0.f;
                    const float sg = sigmoidf_(hv);
                    const float av = hv * sg;
                    const float ds = sg * (1.f + hv * (1.f - sg));
                    if (ts < Tp) lsum = fmaf(av, rv, lsum);
                    const float gh = ct * rv * ds, ga = ct * av;
                    *reinterpret_cast<float2*>(Gs + 2 * ((t * 2 + 0) * RB + r)) = make_float2(gh, gh);
                    *reinterpret_cast<float2*>(Gs + 2 * ((t * 2 + 1) * RB + r)) = make_float2(ga, ga);
                }
            }
            if (a.momentum && warp == 0) dbsum += warp_sum(lane < Tp - ch * RC ? dbS[buf * RC + lane] : 0.f);
            __syncthreads();
            // ---- gradient rows: acc[r] += sum_t G[t][kind][r] * X[t][cb, cb + 1] over the thread's token half
            if (own) {
                const int nv = min(RC / 2, Tp - ch * RC - th * (RC / 2));
                const float* gk = Gs + 2 * (th * (RC / 2) * 2 + kind) * RB;
                const float* xk = Xb + bo;
                auto add = [&](int t) {
                    const uint64_t x = *reinterpret_cast<const uint64_t*>(xk + t * bs);
#pragma unroll
                    for (int r = 0; r < RB; r += 2) {
                        const ulonglong2 g = *reinterpret_cast<const ulonglong2*>(gk + t * 4 * RB + 2 * r);
                        acc[r] = fma_f32x2(g.x, x, acc[r]);
                        acc[r + 1] = fma_f32x2(g.y, x, acc[r + 1]);
                    }
                };
                if (nv == RC / 2) {
#pragma unroll
                    for (int t = 0; t < RC / 2; ++t) add(t);
                } else {
                    for (int t = 0; t < nv; ++t) add(t);
                }
            }
            phase ^= buf;
            buf ^= 1;
        }
        // ---- end of segment: the token halves' gradients together, the Eq. 8 update, then the row
        //      renormalisation to the norms of W_0
        if (own && th == 1) {
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                *reinterpret_cast<uint64_t*>(Ps + r * LD + cb) = acc[r];
                acc[r] = 0;
            }
        }
        if (a.momentum && tid == 0)  // beta_s = sigmoid(mean_t w_beta . x_t + b_beta); warp 0 holds the sum
            scl[2 * RB] = sigmoidf_(dbsum / (float)Tp + b_beta);
        __syncthreads();
        const float beta = a.momentum ? scl[2 * RB] : 0.f;
        if (a.loss) {
            const float tot = block_sum_res(lsum, red);
            if (tid == 0) atomicAdd(&a.loss[seg * a.m_sstride + cz], -tot / (float)Tp);
        }
        float2 wn[RB];
        float step = 0.f;
        const bool upd = own && th == 0;
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            wn[r] = make_float2(0.f, 0.f);
            if (upd) {
                const float2 p = *reinterpret_cast<const float2*>(Ps + r * LD + cb), wo = *reinterpret_cast<const float2*>(Ws + r * LD + cb);
                const float2 g = unpack_f32x2(acc[r]);
                float2 m = make_float2(g.x + p.x, g.y + p.y);
                if (a.momentum) {
                    float2* mu = reinterpret_cast<float2*>(Ms + r * LD + cb);
                    m = make_float2(fmaf(beta, mu->x, m.x), fmaf(beta, mu->y, m.y));
                    *mu = m;
                }
                acc[r] = 0;
                wn[r] = make_float2(wo.x - m.x, wo.y - m.y);
                step = fmaf(m.x, m.x, fmaf(m.y, m.y, step));
            }
        }
        if (a.step_sq) {
            __syncthreads();  // red may still be read by block_sum_res above
            const float tot = block_sum_res(step, red);
            if (tid == 0) atomicAdd(&a.step_sq[seg * a.m_sstride + cz], tot);
        }
        if (a.renorm) {
            // row sums of squares per (matrix, row); a warp may hold columns of both matrices
            __syncthreads();  // red may still be read by block_sum_res above
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int r = 0; r < RB; ++r) {
                    const float v = warp_sum(kind == k ? fmaf(wn[r].x, wn[r].x, wn[r].y * wn[r].y) : 0.f);
                    if (lane == 0) red[warp * 2 * RB + k * RB + r] = v;
                }
            __syncthreads();
            if (tid < 2 * RB) {
                float tot = 0.f;
                for (int i = 0; i < NW; ++i) tot += red[i * 2 * RB + tid];
                scl[tid] = renorm_scale(nS[tid], tot);
            }
            __syncthreads();
        }
        if (upd) {
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                const float sc = a.renorm ? scl[kind * RB + r] : 1.f;
                const float2 wv = make_float2(wn[r].x * sc, wn[r].y * sc);
                finite = finite && isfinite(wv.x) && isfinite(wv.y);
                *reinterpret_cast<float2*>(Ws + r * LD + cb) = wv;
            }
        }
        if (RB == 4 || seg + 1 == a.n_seg) __syncthreads();  // eight rows: the next chunk's barrier, before W is read
        load_w();
    }
    cp_async_wait<0>();
    // write the rows and the momentum back (the CTA's rows lie inside the chain: index check of
    // MONE_DEBUG builds)
    if (!MONE_DCHECK(h0 + RB <= a.d_hid, a.status, DS_RESIDENT_ROWS)) return;
    for (int i = tid; i < RB * (D / 4); i += RES_NT) {
        const int r = i / (D / 4), c = 4 * (i - r * (D / 4));
        const size_t row = (size_t)cs * a.d_hid + h0 + r;
        const size_t o = c < a.d_in ? row * a.d_in + c : row * a.d_out + (c - a.d_in);
        *reinterpret_cast<float4*>((c < a.d_in ? a.W1 : a.W2) + o) = *reinterpret_cast<const float4*>(Ws + r * LD + c);
        if (a.momentum) *reinterpret_cast<float4*>((c < a.d_in ? a.mu1 : a.mu2) + o) = *reinterpret_cast<const float4*>(Ms + r * LD + c);
    }
    if (!finite) atomicOr(a.status, DEV_NONFINITE);
}

template <int RB> constexpr size_t res_smem_bytes(int D) {
    return sizeof(float) * ((size_t)3 * RB * res_ld(D) + (size_t)2 * RES_RC * D + RES_RC * 4 * RB + RES_NW * 2 * RB + 2 * RB + 4 +
                            4 * RES_RC + 2 * RB);
}

// ------------------------------------------------------------------ state upkeep

// Apply the pending renormalisation of the last segment (when asked) and refresh
// the bf16 operand copies.  One warp per (row, chain, matrix), 8 rows a CTA; each lane
// moves 16-byte vectors, four of them in flight at a time (widths are multiples of 64).
__global__ void __launch_bounds__(256) finalize_kernel(DevState s, int c0, int parity, int apply_scale) {
    const int h = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int cs = c0 + blockIdx.y, which = blockIdx.z;
    pdl_wait();
    pdl_trigger();
    if (h >= s.d_hid) return;
    const int width = which ? s.d_out : s.d_in;
    float* w = (which ? s.W2 : s.W1) + ((size_t)cs * s.d_hid + h) * width;
    bf16* wb = s.dtype == 1 ? (which ? s.W2b : s.W1b) + ((size_t)cs * s.d_hid + h) * width : nullptr;
    float sc = 1.f;
    if (apply_scale) {
        const float* ss = s.sumsq + ((size_t)(parity * 2 + which) * s.C + cs) * s.d_hid;
        const float* n0 = (which ? s.n2 : s.n1) + (size_t)cs * s.d_hid;
        sc = renorm_scale(n0[h], ss[h]);
    }
    for (int base = lane * 4; base < width; base += 4 * 128) {
        float4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (base + u * 128 < width) v[u] = *reinterpret_cast<const float4*>(w + base + u * 128);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = base + u * 128;
            if (i >= width) break;
            const float4 x = make_float4(v[u].x * sc, v[u].y * sc, v[u].z * sc, v[u].w * sc);
            if (apply_scale) *reinterpret_cast<float4*>(w + i) = x;
            if (wb) {
                uint2 p;
                p.x = pack_bf16(x.x, x.y);
                p.y = pack_bf16(x.z, x.w);
                *reinterpret_cast<uint2*>(wb + i) = p;
            }
        }
    }
}

__global__ void __launch_bounds__(256) row_norms_kernel(DevState s) {
    const int h = blockIdx.x, cs = blockIdx.y, which = blockIdx.z;
    const int width = which ? s.d_out : s.d_in;
    const float* w = (which ? s.W2 : s.W1) + ((size_t)cs * s.d_hid + h) * width;
    __shared__ float red[8];
    float v = 0.f;
    for (int i = threadIdx.x; i < width; i += 256) v = fmaf(w[i], w[i], v);
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        float tot = 0.f;
        for (int i = 0; i < 8; ++i) tot += red[i];
        (which ? s.n2 : s.n1)[(size_t)cs * s.d_hid + h] = sqrtf(tot);
    }
}

// ------------------------------------------------------------------ output-channel renormalisation
//
// The other reading of App. A's channel-wise renormalisation: a channel is an output
// channel of each matrix, so W1 keeps its rows (hidden units, renormalised inside the
// phase kernels) and every column of W2 (an output feature) is rescaled to its norm in
// W_0 after each update.  A column spans all hidden units, which the phase kernels tile
// apart, so this is a pass of its own over W2: partial column sums of squares over
// kColRowSlices row slices, then the rescale.  Warps cover 32 consecutive columns.

// 64 columns a CTA as 16 float4 column quads x 16 row groups: a warp reads 256 contiguous bytes
// of each of two rows.
__global__ void __launch_bounds__(256) col_partial_kernel(DevState s, int c0) {
    __shared__ float4 red[16][16];
    const int cq = threadIdx.x & 15, rg = threadIdx.x >> 4;
    const int col = blockIdx.x * 64 + 4 * cq, rs = blockIdx.y, cs = c0 + blockIdx.z;
    const int per = (s.d_hid + kColRowSlices - 1) / kColRowSlices;
    const int r1 = min(s.d_hid, (rs + 1) * per);
    const float* w = s.W2 + (size_t)cs * s.d_hid * s.d_out + col;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int r = rs * per + rg; r < r1; r += 16) {
        const float4 x = *reinterpret_cast<const float4*>(w + (size_t)r * s.d_out);
        v.x = fmaf(x.x, x.x, v.x);
        v.y = fmaf(x.y, x.y, v.y);
        v.z = fmaf(x.z, x.z, v.z);
        v.w = fmaf(x.w, x.w, v.w);
    }
    red[rg][cq] = v;
    __syncthreads();
    if (rg == 0) {
        float4 t = red[0][cq];
        for (int g = 1; g < 16; ++g) {
            t.x += red[g][cq].x; t.y += red[g][cq].y; t.z += red[g][cq].z; t.w += red[g][cq].w;
        }
        *reinterpret_cast<float4*>(s.colpart + ((size_t)rs * s.C + cs) * s.d_out + col) = t;
    }
}

__device__ __forceinline__ float col_sumsq(const DevState& s, int cs, int col) {
    float ss = 0.f;
    for (int rs = 0; rs < kColRowSlices; ++rs) ss += s.colpart[((size_t)rs * s.C + cs) * s.d_out + col];
    return ss;
}

// 64 rows x 64 columns a CTA (float4 column quads): W2[:, col] *= nc2[col] / |W2[:, col]|, and
// the bf16 copy.
__global__ void __launch_bounds__(256) col_scale_kernel(DevState s, int c0) {
    __shared__ float sc[64];
    const int cq = threadIdx.x & 15, rg = threadIdx.x >> 4;
    const int cs = c0 + blockIdx.z;
    if (threadIdx.x < 64) {
        const int col = blockIdx.x * 64 + threadIdx.x;
        sc[threadIdx.x] = renorm_scale(s.nc2[(size_t)cs * s.d_out + col], col_sumsq(s, cs, col));
    }
    __syncthreads();
    const float4 f = make_float4(sc[4 * cq], sc[4 * cq + 1], sc[4 * cq + 2], sc[4 * cq + 3]);
    const size_t base = (size_t)cs * s.d_hid * s.d_out + blockIdx.x * 64 + 4 * cq;
    const int r1 = min(s.d_hid, (int)blockIdx.y * 64 + 64);
    for (int r = blockIdx.y * 64 + rg; r < r1; r += 16) {
        const size_t i = base + (size_t)r * s.d_out;
        float4 x = *reinterpret_cast<const float4*>(s.W2 + i);
        x.x *= f.x; x.y *= f.y; x.z *= f.z; x.w *= f.w;
        *reinterpret_cast<float4*>(s.W2 + i) = x;
        if (s.dtype == 1) {
            uint2 p;
            p.x = pack_bf16(x.x, x.y);
            p.y = pack_bf16(x.z, x.w);
            *reinterpret_cast<uint2*>(s.W2b + i) = p;
        }
    }
}

__global__ void __launch_bounds__(256) col_targets_kernel(DevState s) {
    const int col = blockIdx.x * 256 + threadIdx.x, cs = blockIdx.y;
    if (col < s.d_out) s.nc2[(size_t)cs * s.d_out + col] = sqrtf(col_sumsq(s, cs, col));
    for (int h = col; h < s.d_hid; h += gridDim.x * 256) s.n2[(size_t)cs * s.d_hid + h] = -1.f;
}

__global__ void __launch_bounds__(256) gate_silu_kernel(float* g, size_t n, int from_one) {
    const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (i < n) {
        const float v = from_one ? 1.f : g[i];
        g[i] = v * sigmoidf_(v);
    }
}

// ------------------------------------------------------------------ memory read (Eq. 4)

__global__ void __launch_bounds__(256) read_hidden_kernel(DevState s, int Q) {
    __shared__ float As[TK][TM + 4], Bs[TK][TN + 4];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int q0 = blockIdx.x * TM, h0 = blockIdx.y * TN, c = blockIdx.z;
    float acc[4][4] = {};
    simt_tile(acc, s.Uq + ((size_t)c * Q + q0) * s.d_in, s.d_in, 1, s.W1 + ((size_t)c * s.d_hid + h0) * s.d_in,
              s.d_in, 1, s.d_in, min(TM, Q - q0), s.d_in, As, Bs);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int q = q0 + ty * 4 + i;
        if (q >= Q) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float hv = acc[i][j];
            s.Aq[((size_t)c * Q + q) * s.d_hid + h0 + tx * 4 + j] = hv * sigmoidf_(hv);
        }
    }
}

__global__ void __launch_bounds__(256) read_out_kernel(DevState s, int Q) {
    __shared__ float As[TK][TM + 4], Bs[TK][TN + 4];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int q0 = blockIdx.x * TM, o0 = blockIdx.y * TN, c = blockIdx.z;
    float acc[4][4] = {};
    simt_tile(acc, s.Aq + ((size_t)c * Q + q0) * s.d_hid, s.d_hid, 1, s.W2 + (size_t)c * s.d_hid * s.d_out + o0, 1,
              s.d_out, s.d_hid, min(TM, Q - q0), s.d_hid, As, Bs);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int q = q0 + ty * 4 + i;
        if (q >= Q) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) s.Oq[((size_t)c * Q + q) * s.d_out + o0 + tx * 4 + j] = acc[i][j];
    }
}

// Per output head: gate_h * o_h / sqrt(mean(o_h^2) + eps), written with caller strides.
template <typename Tout>
__global__ void __launch_bounds__(256) read_norm_kernel(DevState s, int Q, Tout* Kout, Tout* Vout, long long s0,
                                                        long long s1, long long s2, long long s3, int L) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nh = 2 * s.n_kv;
    const long long job = (long long)blockIdx.x * 8 + warp;  // (c, q, head)
    if (job >= (long long)s.C * Q * nh) return;
    const int head = (int)(job % nh);
    const int q = (int)((job / nh) % Q);
    const int c = (int)(job / ((long long)nh * Q));
    const float* o = s.Oq + ((size_t)c * Q + q) * s.d_out + head * s.hd;
    float v = 0.f;
    for (int i = lane; i < s.hd; i += 32) v = fmaf(o[i], o[i], v);
    v = warp_sum(v);
    const float g = s.gate ? s.gate[(size_t)c * nh + head] : 1.f;
    const float sc = g / sqrtf(v / (float)s.hd + s.rms_eps);
    Tout* out = head < s.n_kv ? Kout : Vout;
    const int kvh = head < s.n_kv ? head : head - s.n_kv;
    out += (long long)(c / L) * s0 + (long long)(c % L) * s1 + (long long)kvh * s2 + (long long)q * s3;
    for (int i = lane; i < s.hd; i += 32) out[i] = from_f<Tout>(o[i] * sc);
}

}  // namespace

namespace {
// Launch a phase kernel of the fp32 path.
template <typename K>
cudaError_t launch_f32_tiles(K kernel, int threads, size_t smem, PerDevice<SmemOptIn>& once, dim3 grid, const F32SegArgs& a,
                             cudaStream_t st) {
    const cudaError_t e = smem_opt_in(reinterpret_cast<const void*>(kernel), smem, once);
    if (e != cudaSuccess) return e;
    kernel<<<grid, threads, smem, st>>>(a);
    return cudaGetLastError();
}
template <int TM, int TN, int TY>
cudaError_t phase_a_f32(const DevState& s, const SegWork& w, const F32SegArgs& a, cudaStream_t st) {
    static PerDevice<SmemOptIn> once;
    return launch_f32_tiles(phase_a_f32_kernel<TM, TN, TY>, 16 * TY, nt_smem<TM, TN, TY>(), once,
                            dim3(s.T / (TY * TM), s.d_hid / (16 * TN), w.nc), a, st);
}
template <int TM, int TN, int TY>
cudaError_t phase_b_f32(const DevState& s, const SegWork& w, const F32SegArgs& a, cudaStream_t st) {
    static PerDevice<SmemOptIn> once;
    return launch_f32_tiles(phase_b_f32_kernel<TM, TN, TY>, 16 * TY, tn_smem<TM, TN, TY>(), once,
                            dim3((s.d_in + s.d_out) / (16 * TN), s.d_hid / (TY * TM), w.nc), a, st);
}
}  // namespace

cudaError_t launch_phase_a_f32(const DevState& s, const SegWork& w, cudaStream_t st) {
    const F32SegArgs a = make_f32_args(s, w);
    const long long g64 = (long long)(s.T / 64) * (s.d_hid / 64) * w.nc;  // 64 x 64 tiles (T, d_hid multiples of 64)
    // 32 x 64 tiles, but 64 x 64 (8 x 4 outputs a thread) where halving the tiles saves nothing of the last wave.
    // 1024 -> 1024 -> 1024, T = 256, 32 x 64 and 64 x 64 tiles: one chain (64 tiles of 64 x 64) 48 and 73 us,
    // three 102 and 123, four (256) 135 and 123, five 163 and 180, eight 223 and 234
    const auto waves = [&](long long tiles) { return (tiles + s.sms - 1) / s.sms; };
    if (g64 > s.sms && waves(2 * g64) == 2 * waves(g64)) return phase_a_f32<8, 4, 8>(s, w, a, st);
    return phase_a_f32<4, 4, 8>(s, w, a, st);
}

cudaError_t launch_phase_b_f32(const DevState& s, const SegWork& w, cudaStream_t st) {
    const F32SegArgs a = make_f32_args(s, w);
    // a tile lies in W1 or in one half of W2: widths are multiples of 64, for the large tile of 128, which
    // is taken from two thirds of the SMs on
    const bool wide = s.d_in % 128 == 0 && (s.d_out / 2) % 128 == 0 && s.d_hid % 128 == 0;
    if (wide && (long long)(s.d_hid / 128) * ((s.d_in + s.d_out) / 128) * w.nc >= s.sms * 2 / 3)
        return phase_b_f32<8, 8, 16>(s, w, a, st);
    // 64 x 64 tiles from two to an SM on (2 chains of 1024 -> 512 -> 512, T = 512: 49 us, 32 x 64 tiles 53), else 32 x
    // 64 (one chain, T = 64: 13.9 and 11.9 us); with 256 threads of 4 x 4 outputs 64 x 64 tiles take 55 and 12.2
    if ((long long)(s.d_hid / 64) * ((s.d_in + s.d_out) / 64) * w.nc > 2 * s.sms) return phase_b_f32<8, 4, 8>(s, w, a, st);
    return phase_b_f32<4, 4, 8>(s, w, a, st);
}

bool resident_f32_fits(const DevState& s) {
    return s.dtype == 0 && s.memory == 0 && s.loss == 0 && !s.col_renorm && s.d_in + s.d_out <= 512 && s.d_in % 4 == 0 &&
           s.d_out % 8 == 0 && s.d_hid % 8 == 0;
}

cudaError_t launch_resident_f32(const DevState& s, const SegWork& w, long long n_tok, cudaStream_t st) {
    ResArgs a{};
    a.d_in = s.d_in; a.d_out = s.d_out; a.d_hid = s.d_hid; a.T = s.T; a.c0 = w.c0; a.win = s.win_rows;
    a.paper = s.mode == 1; a.momentum = s.momentum; a.renorm = s.renorm;
    a.n_tok = n_tok;
    a.n_seg = (int)((n_tok + s.T - 1) / s.T);
    const int dh = s.d_out / 2;
    if (a.paper) {
        a.U = reinterpret_cast<const float*>(s.U) + ((size_t)w.c0 * s.win_rows + w.u_off) * s.d_in;
        a.u_cstride = (long long)s.win_rows * s.d_in;
        a.eta = s.eta + w.u_off;
        a.dbeta = s.dbeta + w.u_off;
    } else {
        a.U = reinterpret_cast<const float*>(w.X) + w.row0 * s.d_in;
        a.u_cstride = w.x_cstride;
    }
    a.K = reinterpret_cast<const float*>(w.K) + w.row0 * dh;
    a.V = reinterpret_cast<const float*>(w.V) + w.row0 * dh;
    a.y_cstride = w.y_cstride;
    a.eta_in = w.eta_in ? w.eta_in + w.row0 : nullptr;
    a.eta_cstride = w.eta_cstride;
    a.lr = s.lr;
    a.b_beta = s.b_beta;
    a.W1 = s.W1; a.W2 = s.W2; a.mu1 = s.mu1; a.mu2 = s.mu2; a.n1 = s.n1; a.n2 = s.n2;
    a.loss = w.loss0 ? w.loss0 : w.loss;
    a.step_sq = w.step0;
    a.m_sstride = w.loss0 || w.step0 ? w.mstride : 0;
    a.status = s.status;
    // four rows a CTA while that still fits the chains in one wave, else eight (less re-streaming)
    const int D = s.d_in + s.d_out;
    auto launch = [&](auto kernel, int rows, size_t most, size_t smem, PerDevice<SmemOptIn>& once) {
        const cudaError_t e = smem_opt_in(reinterpret_cast<const void*>(kernel), most, once);
        if (e != cudaSuccess) return e;
        kernel<<<dim3(s.d_hid / rows, w.nc), RES_NT, smem, st>>>(a);
        return cudaGetLastError();
    };
    static PerDevice<SmemOptIn> once[3];
    if ((long long)w.nc * (s.d_hid / 4) <= s.sms)
        return launch(ttl_resident_f32_kernel<4, 32, 512>, 4, res_smem_bytes<4>(512), res_smem_bytes<4>(D), once[0]);
    // Eight rows: the 32 sums of two tokens cost a lane 31 shuffles and their selects; 16 lanes to a token halve them and read
    // W twice, which is the better form for a narrow chain whose columns leave some of 32 lanes idle. 1500 tokens, 32 and
    // 16 lanes: D = 192 (8 chains of 64 -> 320 -> 128) 444 and 386 us, 256 (8 of 128 -> 448 -> 128) 735 and 758, 320 (4 of 192 ->
    // 448 -> 128) 408 and 388, 384 (256 -> 768 -> 128) 234 and 252, 512 814 and 925
    if (D <= 320 && D % 128)
        return launch(ttl_resident_f32_kernel<8, 16, 320>, 8, res_smem_bytes<8>(320), res_smem_bytes<8>(D), once[1]);
    return launch(ttl_resident_f32_kernel<8, 32, 512>, 8, res_smem_bytes<8>(512), res_smem_bytes<8>(D), once[2]);
}

cudaError_t launch_mse_f32(const DevState& s, const SegWork& w, cudaStream_t st) {
    F32SegArgs a = make_f32_args(s, w);
    mse_hidden_f32_kernel<<<dim3((s.T + A_TM - 1) / A_TM, s.d_hid / TN, w.nc), 256, 0, st>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    mse_out_f32_kernel<<<dim3((s.T + A_TM - 1) / A_TM, s.d_out / TN, w.nc), 256, 0, st>>>(a, s.Kres32, s.Vres32);
    return cudaGetLastError();
}

cudaError_t launch_finalize(const DevState& s, int c0, int nc, int parity, int apply_scale, cudaStream_t st, bool pdl) {
    return launch_kernel(finalize_kernel, dim3((s.d_hid + 7) / 8, nc, 2), 256, 0, st, pdl, 1, s, c0, parity, apply_scale);
}

cudaError_t launch_col_renorm(const DevState& s, int c0, int nc, cudaStream_t st) {
    col_partial_kernel<<<dim3(s.d_out / 64, kColRowSlices, nc), 256, 0, st>>>(s, c0);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    col_scale_kernel<<<dim3(s.d_out / 64, (s.d_hid + 63) / 64, nc), 256, 0, st>>>(s, c0);
    return cudaGetLastError();
}

cudaError_t launch_col_targets(const DevState& s, cudaStream_t st) {
    col_partial_kernel<<<dim3(s.d_out / 64, kColRowSlices, s.C), 256, 0, st>>>(s, 0);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    col_targets_kernel<<<dim3((s.d_out + 255) / 256, s.C), 256, 0, st>>>(s);
    return cudaGetLastError();
}

cudaError_t launch_gate_silu(float* gate, size_t n, int from_one, cudaStream_t st) {
    gate_silu_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(gate, n, from_one);
    return cudaGetLastError();
}

cudaError_t launch_row_norms(const DevState& s, cudaStream_t st) {
    row_norms_kernel<<<dim3(s.d_hid, s.C, 2), 256, 0, st>>>(s);
    return cudaGetLastError();
}

cudaError_t launch_read_norm(const DevState& s, int Q, int n_layers, void* K_out, void* V_out,
                             const long long* strides, cudaStream_t st) {
    const long long jobs = (long long)s.C * Q * 2 * s.n_kv;
    dim3 grid((unsigned)((jobs + 7) / 8));
    if (s.dtype == 0)
        read_norm_kernel<float><<<grid, 256, 0, st>>>(s, Q, (float*)K_out, (float*)V_out, strides[0], strides[1],
                                                      strides[2], strides[3], n_layers);
    else
        read_norm_kernel<bf16><<<grid, 256, 0, st>>>(s, Q, (bf16*)K_out, (bf16*)V_out, strides[0], strides[1],
                                                     strides[2], strides[3], n_layers);
    return cudaGetLastError();
}

cudaError_t launch_read(const DevState& s, int Q, int n_layers, void* K_out, void* V_out,
                        const long long* strides, cudaStream_t st) {
    read_hidden_kernel<<<dim3((Q + TM - 1) / TM, s.d_hid / TN, s.C), 256, 0, st>>>(s, Q);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    read_out_kernel<<<dim3((Q + TM - 1) / TM, s.d_out / TN, s.C), 256, 0, st>>>(s, Q);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const long long jobs = (long long)s.C * Q * 2 * s.n_kv;
    dim3 grid((unsigned)((jobs + 7) / 8));
    if (s.dtype == 0)
        read_norm_kernel<float><<<grid, 256, 0, st>>>(s, Q, (float*)K_out, (float*)V_out, strides[0], strides[1],
                                                      strides[2], strides[3], n_layers);
    else
        read_norm_kernel<bf16><<<grid, 256, 0, st>>>(s, Q, (bf16*)K_out, (bf16*)V_out, strides[0], strides[1],
                                                     strides[2], strides[3], n_layers);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ allocation-free memory read
//
// Scratch of mone_mem_generate_kv_noalloc: a fixed file-scope device array that
// every GPU loading the library holds until the process exits.  Host code cannot
// use the array's name as a device address (it is a host-side stand-in), so the
// address is resolved with cudaGetSymbolAddress, once per device, with that
// device current.

static __device__ __align__(256) float g_noalloc_scratch[kNoAllocScratchFloats];

namespace {
std::mutex g_noalloc_mu;
float* g_noalloc_ptr[64] = {};  // per device ordinal
}  // namespace

cudaError_t noalloc_scratch(float** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        g_noalloc_ptr[dev] = static_cast<float*>(p);
    }
    *out = g_noalloc_ptr[dev];
    return cudaSuccess;
}

cudaError_t launch_read_noalloc(const DevState& s, const TcMaps* tc, const void* Xq, int Q, int n_layers,
                                void* K_out, void* V_out, const long long* strides, cudaStream_t st) {
    float* base = nullptr;
    cudaError_t e = noalloc_scratch(&base);
    if (e != cudaSuccess) return e;
    // the same kernels as the allocating read, pointed at the fixed scratch; every
    // element of the regions is written before it is read, so nothing needs clearing
    // between calls
    DevState t = s;
    t.Uq = base;
    t.Aq = t.Uq + (size_t)s.C * Q * s.d_in;
    t.Oq = t.Aq + (size_t)s.C * Q * s.d_hid;
    if (tc) return launch_read_tc(t, *tc, Xq, t.Uq, t.Aq, t.Oq, Q, n_layers, K_out, V_out, strides, st);
    e = launch_query_transform(t, Xq, Q, t.Uq, false, st);
    return e != cudaSuccess ? e : launch_read(t, Q, n_layers, K_out, V_out, strides, st);
}

}  // namespace mone
