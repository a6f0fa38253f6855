// bf16 tensor-core path of one TTL segment step (tcgen05 + TMEM + TMA, sm_103a).
//
// A segment step of the SiLU-MLP memory M(u) = SiLU(u W1^T) W2 (Eq. 3 form) on
// T tokens is four dense contractions (Eq. 10), done in two persistent kernels:
//
//   phase A, tile = (chain, 128 tokens, 128 hidden units), two TMEM accumulators
//       H = U W1^T            K = d_in      (memory forward)
//       R = Y W2^T            K = d_out     (Y = [K || V], the targets of Eq. 7)
//     fused epilogue: A = SiLU(H), dH = c_t R * SiLU'(H), At = c_t A with
//     c_t = -eta_t / T'.  Eq. 7's loss is linear in M, so dL/dO = -eta Y / T'
//     does not depend on W and the raw target tile is the right operand.
//     Writes dH and At row-major (bf16 [token][hidden]) and the loss partial
//     sum_t sum_h A_th R_th = sum_t y_t . M(u_t).
//
//   phase B, tile = (chain, 128 hidden units, 256 columns of W1 or of W2)
//       G1 = dH^T U           K = T'        (gradient of W1)
//       G2 = At^T Y           K = T'        (gradient of W2)
//     Both operands are read MN-major straight from the row-major buffers.
//     TMEM lane = hidden unit, so in the fused update epilogue (Eq. 8, App. A) a
//     lane owns a row of the fp32 state: mu = beta mu + G; W = s W_raw - mu
//     (s = the previous segment's pending row renormalisation); it writes W,
//     mu, the bf16 operand copy and the new row sums of squares.
//
// Both kernels: one CTA per SM, persistent over a static tile schedule, 10 warps (phase B two more, which move
// the fp32 state).
// Warp 0 lane 0 streams operand tiles with TMA into a shared-memory ring
// (128-byte swizzle), warp 1 lane 0 issues tcgen05.mma into one of two TMEM
// accumulator buffers, warps 2..9 drain the other buffer, so the epilogue of
// tile i overlaps the main loop of tile i+1.  Every mbarrier wait is bounded
// (kWaitLimitNs); a timeout latches DEV_TIMEOUT and the kernel winds down.
#include <mutex>

#include "mone_common.cuh"
#include "per_device.h"

namespace mone {

// What the launches need to know of a device.
struct TcDevice {
    int sms;
    int pair_clusters;   // co-resident CTA pairs of the phase A pair kernel (0: use the one-CTA kernel)
    int pairb_clusters;  // the same for the phase B pair kernel
    int split4, split2;  // co-resident clusters of the phase A split kernels
};

namespace {

constexpr int BK = 64;                    // 64 bf16 = one 128-byte swizzle row
constexpr int EPI_WARPS = 8;
constexpr int THREADS = 64 + EPI_WARPS * 32;
constexpr int EPI_THREADS = EPI_WARPS * 32;
constexpr uint32_t EPI_BAR = 1;           // named barrier among the epilogue warps

// phase A
constexpr int A_BM = 128, A_BN = 128, A_STAGES = 6;
constexpr int A_STAGE = (A_BM + A_BN) * BK * 2;           // 32 KB
// phase B
constexpr int B_BM = 128, B_BN = 256;
constexpr int BOX = 64 * BK * 2;                          // one 64 x 64 MN-major box, 8 KB

template <int STAGES, int STAGE, int TABLE>
struct Layout {
    static constexpr int RING = STAGES * STAGE;
    static constexpr int BARS = RING;                     // full[S], empty[S], tfull[2], tempty[2]
    static constexpr int SLOT = BARS + (2 * STAGES + 4) * 8;
    static constexpr int FLAG = SLOT + 16;
    static constexpr int TAB = FLAG + 16;
    static constexpr int END = TAB + TABLE * 4;
    static constexpr int DYN = END + 1024;                // + alignment slack
};
// table: [2 parity][2 matrix][A_BN] scales
using LA = Layout<A_STAGES, A_STAGE, 4 * A_BN>;
static_assert(LA::DYN <= 227 * 1024, "shared memory budget");

struct TcArgs {
    int d_in, d_out, d_hid, T, Tp, c0, nc, C, paper, momentum, renorm_pending, parity;
    int u_row0, u_chain0, y_row0;
    long long tok0;             // per-token tables: entry of token t of chain cs is [cs * win + tok0 + t]
    int win;
    float lr;
    const float* eta_in;        // plain-mode caller rates, offset to the segment start, or null
    long long eta_cstride;
    const float* eta;           // paper-mode rates [C][T]
    const float* dbeta;         // [C][T]
    const float* zinv;          // [C][T] 1/|z_t| (paper mode), or null
    const float* b_beta;        // [C]
    bf16 *W1b, *W2b;
    const float *n1, *n2;
    float* sumsq;               // [2 parity][2 matrix][C][d_hid]
    bf16 *dH, *At;              // [C][T][d_hid]
    float* loss;                // [nc] or null
    float* step_sq;             // [nc] squared norm of this segment's Eq. 8 step (phase B), or null
    int* status;
    int r_only;                 // phase A pairs: At and c SiLU'(x) / |z| come from the squared-error
                                // pre-pass (the latter in dH); accumulate R only and form dH in place
    int store_mode;             // phase B: when the state ring's slots are handed back (S_PAIRS1, ..)
    unsigned long long wait_ns; // limit of every mbarrier wait of the launch (kWaitLimitNs)
    int stall;                  // test knob (phase A): the producer issues no loads, so the first
                                // wait for a full stage runs out; nothing is in flight when it does
};

__device__ __forceinline__ float* ss_row(const TcArgs& a, int parity, int which, int cs) {
    return a.sumsq + ((size_t)(parity * 2 + which) * a.C + cs) * a.d_hid;
}

struct Ctl {
    uint8_t* base;
    uint32_t bars;
    __device__ uint32_t full(int s) const { return bars + 8 * s; }
    __device__ uint32_t empty(int s, int S) const { return bars + 8 * (S + s); }
    __device__ uint32_t tfull(int b, int S) const { return bars + 8 * (2 * S + b); }
    __device__ uint32_t tempty(int b, int S) const { return bars + 8 * (2 * S + 2 + b); }
};

template <class L, int STAGES>
__device__ __forceinline__ Ctl setup(uint8_t* raw) {
    Ctl c;
    c.base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
    c.bars = smem_u32(c.base + L::BARS);
    if (threadIdx.x == 0) {
        for (int i = 0; i < STAGES; ++i) {
            mbar_init(c.full(i), 1);
            mbar_init(c.empty(i, STAGES), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(c.tfull(b, STAGES), 1);
            mbar_init(c.tempty(b, STAGES), EPI_WARPS);
        }
        fence_mbar_init();
    }
    if (threadIdx.x / 32 == 0) {
        tmem_alloc(smem_u32(c.base + L::SLOT), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    return c;
}


// ------------------------------------------------------------------ phase A

// Epilogue of one phase A tile (chain cs, token rows trow.., hidden columns h0..h0+BN)
// held in TMEM at `tmem` (H in columns [0, BN), R in [BN, 2 BN), one token per lane), run
// by the EPI_WARPS epilogue warps (warp = TMEM lane quarter x column half).  Builds the
// tile's renormalisation scales, zeroes the segment's row sums of squares when `zero_ss`,
// waits for the accumulators, then writes dH and At and adds the loss partial.
// `release` is called by every epilogue warp once its last TMEM read of the tile is
// done.  Returns false if the accumulator wait timed out.
template <int BN, class Release>
__device__ __forceinline__ bool phase_a_epilogue(const TcArgs& a, uint32_t tmem, uint32_t tfull_bar, int parity_bit,
                                                 float* tab, int* flag, int cz, int cs, int h0, int trow,
                                                 bool zero_ss, uint8_t* stg, Release&& release) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int e = warp - 2, q = warp & 3, ch = e >> 2, et = threadIdx.x - 64;
    static_assert(BN <= EPI_THREADS && BN % 64 == 0, "one scale per epilogue thread, 32-column chunks");
    // the tile's rows of dH / At lie inside the [C][T][d_hid] scratch (index check of MONE_DEBUG builds)
    const bool wr = MONE_DCHECK(cs < a.C && trow + 128 <= a.T && h0 + BN <= a.d_hid, a.status, DS_PHASE_A_TILE);
    if (et < BN) {
        const int h = h0 + et;
        float s1 = 1.f, s2 = 1.f;
        if (a.renorm_pending) {
            s1 = renorm_scale(a.n1[(size_t)cs * a.d_hid + h], ss_row(a, a.parity ^ 1, 0, cs)[h]);
            s2 = renorm_scale(a.n2[(size_t)cs * a.d_hid + h], ss_row(a, a.parity ^ 1, 1, cs)[h]);
        }
        tab[et] = s1;
        tab[BN + et] = s2;
        if (zero_ss) {
            ss_row(a, a.parity, 0, cs)[h] = 0.f;
            ss_row(a, a.parity, 1, cs)[h] = 0.f;
        }
    }
    if (et == 0) *flag = mbar_wait(tfull_bar, parity_bit, a.status, a.wait_ns) ? 1 : 0;
    __syncwarp();
    named_bar_sync(EPI_BAR, EPI_THREADS);
    if (!*flag) return false;
    tc_fence_after();
    const int row = q * 32 + lane;
    const int t = trow + row;
    float ct = 0.f, zi = 1.f;
    if (t < a.Tp) {
        const float ev = a.paper ? a.eta[(size_t)cs * a.win + a.tok0 + t]
                                 : (a.eta_in ? a.eta_in[cz * a.eta_cstride + t] : a.lr);
        ct = -ev / (float)a.Tp;
        if (a.zinv) zi = a.zinv[(size_t)cs * a.win + a.tok0 + t];
    }
    const float czi = ct * zi;
    const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16);
    bf16* dHrow = a.dH + ((size_t)cs * a.T + t) * a.d_hid + h0;
    bf16* Arow = a.At + ((size_t)cs * a.T + t) * a.d_hid + h0;
    float lsum = 0.f;
    constexpr int CHUNKS = BN / 64;  // 32-column chunks per warp (each warp holds BN / 2 columns)
#pragma unroll 1
    for (int cc = 0; cc < CHUNKS; ++cc) {
        const int c0 = ch * (BN / 2) + cc * 32;
        float hv[32], rv[32];
        tmem_ld32(lane_base + c0, hv);
        tmem_ld32(lane_base + BN + c0, rv);
        if (cc == CHUNKS - 1) {
            tc_fence_before();
            __syncwarp();
            release();
        }
        uint32_t pd[16], pa[16];
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
            const float4 s1v = *reinterpret_cast<const float4*>(tab + c0 + j);
            const float4 s2v = *reinterpret_cast<const float4*>(tab + BN + c0 + j);
            const float s1a[4] = {s1v.x, s1v.y, s1v.z, s1v.w};
            const float s2a[4] = {s2v.x, s2v.y, s2v.z, s2v.w};
            float dv[4], av4[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float x = hv[j + u] * s1a[u] * zi;
                const float r = rv[j + u] * s2a[u];
                const float sg = sigmoid_tanh(x);
                const float av = x * sg;
                lsum = fmaf(av, r, lsum);
                dv[u] = czi * r * (sg * fmaf(x, 1.f - sg, 1.f));  // c_t (dL/dA) SiLU'(x), scaled by 1/|z_t|
                av4[u] = ct * av;
            }
            pd[j / 2] = pack_bf16(dv[0], dv[1]);
            pd[j / 2 + 1] = pack_bf16(dv[2], dv[3]);
            pa[j / 2] = pack_bf16(av4[0], av4[1]);
            pa[j / 2 + 1] = pack_bf16(av4[2], av4[3]);
        }
        if (!wr) {
        } else if (stg) {
            // rows trow + q*32 .. +31 of this warp, columns h0 + c0 .. +31
            const size_t r0 = ((size_t)cs * a.T + trow + q * 32) * a.d_hid + h0 + c0;
            store_rows_coalesced(stg, pd, a.dH + r0, a.d_hid, lane);
            store_rows_coalesced(stg, pa, a.At + r0, a.d_hid, lane);
        } else {
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                *reinterpret_cast<uint4*>(dHrow + c0 + v * 8) =
                    make_uint4(pd[4 * v], pd[4 * v + 1], pd[4 * v + 2], pd[4 * v + 3]);
                *reinterpret_cast<uint4*>(Arow + c0 + v * 8) =
                    make_uint4(pa[4 * v], pa[4 * v + 1], pa[4 * v + 2], pa[4 * v + 3]);
            }
        }
    }
    if (a.loss) {
        lsum = warp_sum(lsum);
        if (lane == 0) atomicAdd(&a.loss[cz], -lsum / (float)a.Tp);
    }
    return true;
}

// The same epilogue split in two for a tile whose H accumulator (over d_in) completes before
// its R accumulator (over d_out), the order phase A issues them in.  At = c SiLU(x) needs only
// H, so once `hfull_bar` fires (H done, R still accumulating) the epilogue writes At and leaves
// s' = c (1/|z|) SiLU'(x) in H's TMEM columns; once `tfull_bar` fires it forms dH = R s2 s'.
// Only the second part runs after the main loop.  No loss partial (the caller uses
// phase_a_epilogue when a loss is requested).
template <int BN, class Release>
__device__ __forceinline__ bool phase_a_epilogue_split(const TcArgs& a, uint32_t tmem, uint32_t hfull_bar,
                                                       uint32_t tfull_bar, int parity_bit, float* tab, int* flag,
                                                       int cz, int cs, int h0, int trow, bool zero_ss, uint8_t* stg,
                                                       Release&& release) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int e = warp - 2, q = warp & 3, ch = e >> 2, et = threadIdx.x - 64;
    static_assert(BN <= EPI_THREADS && BN % 64 == 0, "one scale per epilogue thread, 32-column chunks");
    // the tile's rows of dH / At lie inside the [C][T][d_hid] scratch (index check of MONE_DEBUG builds)
    const bool wr = MONE_DCHECK(cs < a.C && trow + 128 <= a.T && h0 + BN <= a.d_hid, a.status, DS_PHASE_A_TILE);
    if (et < BN) {
        const int h = h0 + et;
        float s1 = 1.f, s2 = 1.f;
        if (a.renorm_pending) {
            s1 = renorm_scale(a.n1[(size_t)cs * a.d_hid + h], ss_row(a, a.parity ^ 1, 0, cs)[h]);
            s2 = renorm_scale(a.n2[(size_t)cs * a.d_hid + h], ss_row(a, a.parity ^ 1, 1, cs)[h]);
        }
        tab[et] = s1;
        tab[BN + et] = s2;
        if (zero_ss) {
            ss_row(a, a.parity, 0, cs)[h] = 0.f;
            ss_row(a, a.parity, 1, cs)[h] = 0.f;
        }
    }
    if (et == 0) *flag = mbar_wait(hfull_bar, parity_bit, a.status, a.wait_ns) ? 1 : 0;
    __syncwarp();
    named_bar_sync(EPI_BAR, EPI_THREADS);
    if (!*flag) return false;
    tc_fence_after();
    const int row = q * 32 + lane;
    const int t = trow + row;
    float ct = 0.f, zi = 1.f;
    if (t < a.Tp) {
        const float ev = a.paper ? a.eta[(size_t)cs * a.win + a.tok0 + t]
                                 : (a.eta_in ? a.eta_in[cz * a.eta_cstride + t] : a.lr);
        ct = -ev / (float)a.Tp;
        if (a.zinv) zi = a.zinv[(size_t)cs * a.win + a.tok0 + t];
    }
    const float czi = ct * zi;
    const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16);
    const size_t r0 = ((size_t)cs * a.T + trow + q * 32) * a.d_hid + h0;  // this warp's first row
    constexpr int CHUNKS = BN / 64;  // 32-column chunks per warp (each warp holds BN / 2 columns)
    // ---- part 1, overlapping the R main loop: At, and s' into H's columns
#pragma unroll 1
    for (int cc = 0; cc < CHUNKS; ++cc) {
        const int c0 = ch * (BN / 2) + cc * 32;
        float hv[32];
        tmem_ld32(lane_base + c0, hv);
        uint32_t pa[16];
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
            const float4 s1v = *reinterpret_cast<const float4*>(tab + c0 + j);
            const float s1a[4] = {s1v.x, s1v.y, s1v.z, s1v.w};
            float av4[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float x = hv[j + u] * s1a[u] * zi;
                const float sg = sigmoid_tanh(x);
                av4[u] = ct * (x * sg);
                hv[j + u] = czi * (sg * fmaf(x, 1.f - sg, 1.f));  // c_t SiLU'(x), scaled by 1/|z_t|
            }
            pa[j / 2] = pack_bf16(av4[0], av4[1]);
            pa[j / 2 + 1] = pack_bf16(av4[2], av4[3]);
        }
        tmem_st32(lane_base + c0, hv);
        if (wr) store_rows_coalesced(stg, pa, a.At + r0 + c0, a.d_hid, lane);
    }
    tmem_wait_st();
    // ---- part 2, after the main loop: dH = R s2 s'
    if (et == 0) flag[2] = mbar_wait(tfull_bar, parity_bit, a.status, a.wait_ns) ? 1 : 0;
    __syncwarp();
    named_bar_sync(EPI_BAR, EPI_THREADS);
    if (!flag[2]) return false;
    tc_fence_after();
#pragma unroll 1
    for (int cc = 0; cc < CHUNKS; ++cc) {
        const int c0 = ch * (BN / 2) + cc * 32;
        float sp[32], rv[32];
        tmem_ld32(lane_base + c0, sp);
        tmem_ld32(lane_base + BN + c0, rv);
        if (cc == CHUNKS - 1) {
            tc_fence_before();
            __syncwarp();
            release();
        }
        uint32_t pd[16];
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
            const float4 s2v = *reinterpret_cast<const float4*>(tab + BN + c0 + j);
            pd[j / 2] = pack_bf16(rv[j] * s2v.x * sp[j], rv[j + 1] * s2v.y * sp[j + 1]);
            pd[j / 2 + 1] = pack_bf16(rv[j + 2] * s2v.z * sp[j + 2], rv[j + 3] * s2v.w * sp[j + 3]);
        }
        if (wr) store_rows_coalesced(stg, pd, a.dH + r0 + c0, a.d_hid, lane);
    }
    return true;
}

// Epilogue of a phase A pair tile in the R-only form (squared-error loss): At and
// s' = c_t SiLU'(x) / |z_t| were written by the pre-pass (s' in dH), so dH = R s2 s' in place.
template <int BN, class Release>
__device__ __forceinline__ bool phase_a_epilogue_r_only(const TcArgs& a, uint32_t tmem, uint32_t tfull_bar,
                                                        int parity_bit, float* tab, int* flag, int cs, int h0,
                                                        int trow, bool zero_ss, uint8_t* stg, Release&& release) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int e = warp - 2, q = warp & 3, ch = e >> 2, et = threadIdx.x - 64;
    // the tile's rows of dH lie inside the [C][T][d_hid] scratch (index check of MONE_DEBUG builds)
    const bool wr = MONE_DCHECK(cs < a.C && trow + 128 <= a.T && h0 + BN <= a.d_hid, a.status, DS_PHASE_A_TILE);
    if (et < BN) {
        const int h = h0 + et;
        float s2 = 1.f;
        if (a.renorm_pending)
            s2 = renorm_scale(a.n2[(size_t)cs * a.d_hid + h], ss_row(a, a.parity ^ 1, 1, cs)[h]);
        tab[BN + et] = s2;
        if (zero_ss) {
            ss_row(a, a.parity, 0, cs)[h] = 0.f;
            ss_row(a, a.parity, 1, cs)[h] = 0.f;
        }
    }
    if (et == 0) *flag = mbar_wait(tfull_bar, parity_bit, a.status, a.wait_ns) ? 1 : 0;
    __syncwarp();
    named_bar_sync(EPI_BAR, EPI_THREADS);
    if (!*flag) return false;
    tc_fence_after();
    const int row = q * 32 + lane;
    const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16);
    const size_t r0 = ((size_t)cs * a.T + trow + q * 32) * a.d_hid + h0;  // this warp's first row
    const bf16* sp_row = a.dH + ((size_t)cs * a.T + trow + row) * a.d_hid + h0;
    constexpr int CHUNKS = BN / 64;
#pragma unroll 1
    for (int cc = 0; cc < CHUNKS; ++cc) {
        const int c0 = ch * (BN / 2) + cc * 32;
        float rv[32];
        tmem_ld32(lane_base + BN + c0, rv);
        if (cc == CHUNKS - 1) {
            tc_fence_before();
            __syncwarp();
            release();
        }
        uint4 sv[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) sv[v] = *reinterpret_cast<const uint4*>(sp_row + c0 + v * 8);
        uint32_t pd[16];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const __nv_bfloat162* sb = reinterpret_cast<const __nv_bfloat162*>(&sv[v]);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float2 sf = __bfloat1622float2(sb[u]);
                const int j = v * 8 + 2 * u;
                pd[j / 2] = pack_bf16(rv[j] * tab[BN + c0 + j] * sf.x, rv[j + 1] * tab[BN + c0 + j + 1] * sf.y);
            }
        }
        if (wr) store_rows_coalesced(stg, pd, a.dH + r0 + c0, a.d_hid, lane);  // in place: every lane has read its row
    }
    return true;
}

__global__ void __launch_bounds__(THREADS, 1)
tc_phase_a_kernel(const __grid_constant__ CUtensorMap tmU, const __grid_constant__ CUtensorMap tmK,
                  const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmW1,
                  const __grid_constant__ CUtensorMap tmW2, const TcArgs a) {
    extern __shared__ uint8_t smem_raw[];
    const Ctl c = setup<LA, A_STAGES>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t tmem = *reinterpret_cast<uint32_t*>(c.base + LA::SLOT);
    pdl_wait();
    pdl_trigger();
    const int n_tt = a.T / A_BM, n_ht = a.d_hid / A_BN;
    const int ntiles = a.nc * n_ht * n_tt;
    const int KB1 = a.d_in / BK, KB = KB1 + a.d_out / BK, half = (a.d_out / 2) / BK;

    if (warp == 0) {
        if (lane == 0) {
            tma_prefetch_map(&tmU);
            tma_prefetch_map(&tmK);
            tma_prefetch_map(&tmV);
            tma_prefetch_map(&tmW1);
            tma_prefetch_map(&tmW2);
            const uint64_t wpol = l2_evict_last_policy();  // the bf16 W copy phase B wrote
            uint32_t kc = 0;
            bool ok = true;
            for (int tile = blockIdx.x; tile < ntiles && ok && !a.stall; tile += gridDim.x) {
                const int cz = tile / (n_ht * n_tt), ht = (tile / n_tt) % n_ht, tt = tile % n_tt;
                const int cs = a.c0 + cz, h0 = ht * A_BN, trow = tt * A_BM;
                for (int kb = 0; kb < KB; ++kb, ++kc) {
                    const int s = kc % A_STAGES;
                    if (kc >= A_STAGES && !mbar_wait(c.empty(s, A_STAGES), ((kc / A_STAGES) - 1) & 1, a.status, a.wait_ns)) {
                        ok = false;
                        break;
                    }
                    const uint32_t sa = smem_u32(c.base + s * A_STAGE), sb = sa + A_BM * BK * 2, fb = c.full(s);
                    mbar_expect_tx(fb, A_STAGE);
                    if (kb < KB1) {
                        tma_load_3d(sa, &tmU, fb, kb * BK, a.u_row0 + trow, a.u_chain0 + cz);
                        tma_load_3d_hint(sb, &tmW1, fb, kb * BK, h0, cs, wpol);
                    } else {
                        const int k2 = kb - KB1;
                        if (k2 < half)
                            tma_load_3d(sa, &tmK, fb, k2 * BK, a.y_row0 + trow, cz);
                        else
                            tma_load_3d(sa, &tmV, fb, (k2 - half) * BK, a.y_row0 + trow, cz);
                        tma_load_3d_hint(sb, &tmW2, fb, k2 * BK, h0, cs, wpol);
                    }
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = idesc_bf16_f32(A_BM, A_BN, false, false);
            uint32_t kc = 0;
            int local = 0;
            bool ok = true;
            for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, ++local) {
                const int b = local & 1;
                if (local >= 2 && !mbar_wait(c.tempty(b, A_STAGES), ((local >> 1) - 1) & 1, a.status, a.wait_ns)) break;
                tc_fence_after();
                const uint32_t dH = tmem + b * 256, dR = dH + A_BN;
                for (int kb = 0; kb < KB; ++kb, ++kc) {
                    const int s = kc % A_STAGES;
                    if (!mbar_wait(c.full(s), (kc / A_STAGES) & 1, a.status, a.wait_ns)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t sa = smem_u32(c.base + s * A_STAGE);
                    const uint64_t da = sdesc_sw128(sa, 16), db = sdesc_step(da, A_BM * BK * 2);
                    const bool first = (kb == 0 || kb == KB1);
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)
                        umma_bf16(kb < KB1 ? dH : dR, sdesc_step(da, k * 32), sdesc_step(db, k * 32), idesc,
                                  (first && k == 0) ? 0u : 1u);
                    umma_commit(c.empty(s, A_STAGES));
                }
                umma_commit(c.tfull(b, A_STAGES));
            }
        }
        __syncwarp();
    } else {
        float* table = reinterpret_cast<float*>(c.base + LA::TAB);
        int* flag = reinterpret_cast<int*>(c.base + LA::FLAG);
        int local = 0;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++local) {
            const int cz = tile / (n_ht * n_tt), ht = (tile / n_tt) % n_ht, tt = tile % n_tt;
            const int b = local & 1;
            const uint32_t tempty = c.tempty(b, A_STAGES);
            if (!phase_a_epilogue<A_BN>(a, tmem + b * 256, c.tfull(b, A_STAGES), (local >> 1) & 1, table + b * 2 * A_BN,
                                  flag + b, cz, a.c0 + cz, ht * A_BN, tt * A_BM, tt == 0, nullptr, [&] {
                                      if (lane == 0) mbar_arrive(tempty);
                                  }))
                break;
        }
    }
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------ phase A on CTA pairs
//
// The same tile step on a cluster of two CTAs that share each tcgen05.mma
// (cta_group::2): M = 256 tokens, 128 in each CTA, x N = 256 hidden units, whose W
// rows are split between the pair (128 rows staged in each CTA).  Each CTA's TMEM
// holds the H and R rows of its own tokens (256 + 256 columns: one accumulator
// buffer).  A TMA tensor load costs the SM about the same whether its box has 64 or
// 128 rows, and phase A is bounded by those loads: here an SM issues two 128-row
// boxes per 64-deep k-block for a 128 x 256 accumulator, twice the work per load of
// the one-CTA kernel's 128 x 128 tile.  Rank 0 of the pair issues the MMAs: both
// CTAs' loads complete on rank 0's full barrier (a relay, with each CTA's loads on
// its own barrier and one remote arrive per stage, measured 1.7x slower), each MMA
// commit arrives on the empty and accumulator-full barriers of both CTAs, and all 16
// epilogue warps of the pair release the accumulator on rank 0's tempty barrier.  The
// epilogue stores dH and At through per-warp transpose buffers (coalesced rows).
constexpr int P_BN = 256;
constexpr int P_STAGES = 6;
constexpr int P_A = A_BM * BK * 2;                  // 16 KB: this CTA's 128 token rows
constexpr int P_STAGE = P_A + (P_BN / 2) * BK * 2;  // + 16 KB: this CTA's 128 W rows
struct LP {
    static constexpr int RING = P_STAGES * P_STAGE;
    static constexpr int BARS = RING;  // full[S] empty[S] tfull[2] tempty[2]
    static constexpr int NBARS = 2 * P_STAGES + 4;
    static constexpr int SLOT = BARS + NBARS * 8;
    static constexpr int FLAG = SLOT + 16;              // 2 tiles x 4 flags
    static constexpr int TAB = FLAG + 32;               // scale tables of two consecutive tiles
    static constexpr int STG = TAB + 4 * P_BN * 4;      // per epilogue warp: 32 x 64 B transpose buffer
    static constexpr int END = STG + EPI_WARPS * 2048;
    static constexpr int DYN = END + 1024;
};
static_assert(LP::DYN <= 227 * 1024, "shared memory budget");
static_assert(LP::STG % 16 == 0, "staging buffers hold 16-byte pieces");

__global__ void __launch_bounds__(THREADS, 1)
tc_phase_a_pair_kernel(const __grid_constant__ CUtensorMap tmU, const __grid_constant__ CUtensorMap tmK,
                       const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmW1,
                       const __grid_constant__ CUtensorMap tmW2, const TcArgs a) {
    extern __shared__ uint8_t smem_raw[];
    Ctl c;
    c.base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    c.bars = smem_u32(c.base + LP::BARS);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    if (threadIdx.x == 0) {
        for (int i = 0; i < P_STAGES; ++i) {
            mbar_init(c.full(i), 1);
            mbar_init(c.empty(i, P_STAGES), 1);
        }
        mbar_init(c.tfull(0, P_STAGES), 1);
        mbar_init(c.tfull(1, P_STAGES), 1);  // H accumulator complete (R still accumulating)
        mbar_init(c.tempty(0, P_STAGES), 2 * EPI_WARPS);
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc_pair(smem_u32(c.base + LP::SLOT), 512);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    cluster_sync();  // barriers of both CTAs initialised, TMEM of the pair allocated
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<uint32_t*>(c.base + LP::SLOT);
    pdl_wait();
    pdl_trigger();
    const int n_tp = a.T / (2 * A_BM), n_ht = a.d_hid / P_BN;
    const int npairs = a.nc * n_ht * n_tp;
    const int cluster = blockIdx.x >> 1, nclusters = gridDim.x >> 1;
    // the R-only form (squared-error loss) takes no H k-blocks
    const int KB1 = a.r_only ? 0 : a.d_in / BK, KB = KB1 + a.d_out / BK, half = (a.d_out / 2) / BK;

    if (warp == 0) {
        if (lane == 0) {
            tma_prefetch_map(&tmU);
            tma_prefetch_map(&tmK);
            tma_prefetch_map(&tmV);
            tma_prefetch_map(&tmW1);
            tma_prefetch_map(&tmW2);
            const uint64_t wpol = l2_evict_last_policy();  // the bf16 W copy phase B wrote
            uint32_t kc = 0;
            bool ok = true;
            for (int pt = cluster; pt < npairs && ok && !a.stall; pt += nclusters) {
                const int cz = pt / (n_ht * n_tp), ht = (pt / n_tp) % n_ht, tp = pt % n_tp;
                const int cs = a.c0 + cz, hrow = ht * P_BN + (int)rank * (P_BN / 2);
                const int trow = tp * 2 * A_BM + (int)rank * A_BM;
                for (int kb = 0; kb < KB; ++kb, ++kc) {
                    const int s = kc % P_STAGES;
                    if (kc >= P_STAGES && !mbar_wait(c.empty(s, P_STAGES), ((kc / P_STAGES) - 1) & 1, a.status, a.wait_ns)) {
                        ok = false;
                        break;
                    }
                    // both CTAs' loads complete on rank 0's full barrier
                    const uint32_t sa = smem_u32(c.base + s * P_STAGE), sb = sa + P_A;
                    const uint32_t fb = map_to_cta(c.full(s), 0);
                    if (rank == 0) mbar_expect_tx(c.full(s), 2 * P_STAGE);
                    if (kb < KB1) {
                        tma_load_3d_pair(sa, &tmU, fb, kb * BK, a.u_row0 + trow, a.u_chain0 + cz);
                        tma_load_3d_pair_hint(sb, &tmW1, fb, kb * BK, hrow, cs, wpol);
                    } else {
                        const int k2 = kb - KB1;
                        if (k2 < half)
                            tma_load_3d_pair(sa, &tmK, fb, k2 * BK, a.y_row0 + trow, cz);
                        else
                            tma_load_3d_pair(sa, &tmV, fb, (k2 - half) * BK, a.y_row0 + trow, cz);
                        tma_load_3d_pair_hint(sb, &tmW2, fb, k2 * BK, hrow, cs, wpol);
                    }
                }
            }
            if (!ok) drain_copies();
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {
            const uint32_t idesc = idesc_bf16_f32(2 * A_BM, P_BN, false, false);
            uint32_t kc = 0;
            int local = 0;
            bool ok = true;
            for (int pt = cluster; pt < npairs && ok; pt += nclusters, ++local) {
                // one accumulator buffer: wait until both CTAs' epilogues have read the last tile
                if (local >= 1 && !mbar_wait(c.tempty(0, P_STAGES), (local - 1) & 1, a.status, a.wait_ns)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t dH = tmem, dR = tmem + P_BN;
                for (int kb = 0; kb < KB; ++kb, ++kc) {
                    const int s = kc % P_STAGES;
                    if (!mbar_wait(c.full(s), (kc / P_STAGES) & 1, a.status, a.wait_ns)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t sa = smem_u32(c.base + s * P_STAGE);
                    const uint64_t da = sdesc_sw128(sa, 16), db = sdesc_step(da, P_A);
                    const bool first = (kb == 0 || kb == KB1);
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)
                        umma_bf16_pair(kb < KB1 ? dH : dR, sdesc_step(da, k * 32), sdesc_step(db, k * 32), idesc,
                                       (first && k == 0) ? 0u : 1u);
                    umma_commit_pair(c.empty(s, P_STAGES), 0x3);
                    if (kb == KB1 - 1) umma_commit_pair(c.tfull(1, P_STAGES), 0x3);  // H complete
                }
                if (!ok) break;
                umma_commit_pair(c.tfull(0, P_STAGES), 0x3);
            }
            if (!ok) drain_copies();
        }
        __syncwarp();
    } else {
        float* table = reinterpret_cast<float*>(c.base + LP::TAB);
        int* flag = reinterpret_cast<int*>(c.base + LP::FLAG);
        const uint32_t tempty0 = map_to_cta(c.tempty(0, P_STAGES), 0);
        int local = 0;
        for (int pt = cluster; pt < npairs; pt += nclusters, ++local) {
            const int cz = pt / (n_ht * n_tp), ht = (pt / n_tp) % n_ht, tp = pt % n_tp;
            const int tt = tp * 2 + (int)rank;
            // the scale table and flag alternate between tiles: a warp may start the next
            // tile while another still reads this one's table
            auto release = [&] {
                if (lane == 0) mbar_arrive_remote(tempty0);
            };
            float* tab = table + (local & 1) * 2 * P_BN;
            int* fl = flag + (local & 1) * 4;
            uint8_t* stg = c.base + LP::STG + (warp - 2) * 2048;
            const bool ok =
                a.r_only ? phase_a_epilogue_r_only<P_BN>(a, tmem, c.tfull(0, P_STAGES), local & 1, tab, fl, a.c0 + cz,
                                                         ht * P_BN, tt * A_BM, tt == 0, stg, release)
                : a.loss ? phase_a_epilogue<P_BN>(a, tmem, c.tfull(0, P_STAGES), local & 1, tab, fl, cz, a.c0 + cz,
                                                  ht * P_BN, tt * A_BM, tt == 0, stg, release)
                         : phase_a_epilogue_split<P_BN>(a, tmem, c.tfull(1, P_STAGES), c.tfull(0, P_STAGES), local & 1,
                                                        tab, fl, cz, a.c0 + cz, ht * P_BN, tt * A_BM, tt == 0, stg,
                                                        release);
            if (!ok) break;
        }
    }
    tc_fence_before();
    cluster_sync();  // every MMA of the pair has completed and every TMEM read is done
    tc_fence_after();
    if (warp == 0) tmem_dealloc_pair(tmem, 512);
}

// ------------------------------------------------------------------ phase A on few tiles
//
// A launch of few tiles (one chain of a streamed segment: 32 tiles of 128 x 128) leaves most SMs
// idle and runs at the pace of one tile's 48 k-blocks.  Here a cluster of S CTAs shares a tile: CTA r
// accumulates its share of the k-blocks of H and of R, each CTA writes its partial sums to shared
// memory as S column parts, and CTA r adds up part r from all of them through distributed shared
// memory and runs the epilogue on it.  One tile per cluster.  One chain of 2048 -> 1024 -> 1024, T = 512
// (caches cold): 21.8 us with four CTAs a tile, 28.4 us on the CTA pairs of larger launches.
template <int S>
struct LSplit {
    static constexpr int RING = A_STAGES * A_STAGE;       // partial sums: [S parts][H, R][128 rows][128 / S] in its place
    static constexpr int BARS = RING;                     // full[S], empty[S], tfull[2], tempty[2]
    static constexpr int SLOT = BARS + (2 * A_STAGES + 4) * 8;
    static constexpr int FLAG = SLOT + 16;
    static constexpr int TAB = FLAG + 16;                 // scales s1, s2 of the part's columns
    static constexpr int END = TAB + 2 * (A_BN / S) * 4;
    static constexpr int DYN = END + 1024;
};
static_assert(LSplit<2>::DYN <= 227 * 1024 && 2 * A_BM * A_BN * 4 <= LSplit<2>::RING, "shared memory budget");

__device__ __forceinline__ float4 ld_cluster_f32x4(uint32_t cluster_addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(cluster_addr)
                 : "memory");
    return v;
}

template <int S>
__global__ void __launch_bounds__(THREADS, 1)
tc_phase_a_split_kernel(const __grid_constant__ CUtensorMap tmU, const __grid_constant__ CUtensorMap tmK,
                        const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmW1,
                        const __grid_constant__ CUtensorMap tmW2, const TcArgs a) {
    using L = LSplit<S>;
    constexpr int PC = A_BN / S;  // columns of a part
    extern __shared__ uint8_t smem_raw[];
    const Ctl c = setup<L, A_STAGES>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t tmem = *reinterpret_cast<uint32_t*>(c.base + L::SLOT);
    const int r = (int)cluster_ctarank(), tile = blockIdx.x / S;
    const int n_tt = a.T / A_BM, n_ht = a.d_hid / A_BN;
    const int cz = tile / (n_ht * n_tt), h0 = (tile / n_tt) % n_ht * A_BN, trow = tile % n_tt * A_BM, cs = a.c0 + cz;
    // this CTA's k-blocks: [b1, e1) of H over d_in, [b2, e2) of R over d_out (neither empty: the launch sees to it)
    const int KB1 = a.d_in / BK, KB2 = a.d_out / BK, half = KB2 / 2;
    const int b1 = KB1 * r / S, e1 = KB1 * (r + 1) / S, b2 = KB2 * r / S, e2 = KB2 * (r + 1) / S;
    const int n1 = e1 - b1, n = n1 + e2 - b2;
    int* flag = reinterpret_cast<int*>(c.base + L::FLAG);
    pdl_wait();
    pdl_trigger();
    if (warp == 0) {
        if (lane == 0) {
            const uint64_t wpol = l2_evict_last_policy();  // the bf16 W copy phase B wrote
            for (int i = 0; i < n && !a.stall; ++i) {
                const int s = i % A_STAGES;
                if (i >= A_STAGES && !mbar_wait(c.empty(s, A_STAGES), ((i / A_STAGES) - 1) & 1, a.status, a.wait_ns)) {
                    drain_copies();
                    break;
                }
                const uint32_t sa = smem_u32(c.base + s * A_STAGE), sb = sa + A_BM * BK * 2, fb = c.full(s);
                mbar_expect_tx(fb, A_STAGE);
                if (i < n1) {
                    tma_load_3d(sa, &tmU, fb, (b1 + i) * BK, a.u_row0 + trow, a.u_chain0 + cz);
                    tma_load_3d_hint(sb, &tmW1, fb, (b1 + i) * BK, h0, cs, wpol);
                } else {
                    const int k2 = b2 + i - n1;
                    if (k2 < half)
                        tma_load_3d(sa, &tmK, fb, k2 * BK, a.y_row0 + trow, cz);
                    else
                        tma_load_3d(sa, &tmV, fb, (k2 - half) * BK, a.y_row0 + trow, cz);
                    tma_load_3d_hint(sb, &tmW2, fb, k2 * BK, h0, cs, wpol);
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = idesc_bf16_f32(A_BM, A_BN, false, false);
            bool ok = true;
            for (int i = 0; i < n; ++i) {
                const int s = i % A_STAGES;
                if (!mbar_wait(c.full(s), (i / A_STAGES) & 1, a.status, a.wait_ns)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint64_t da = sdesc_sw128(smem_u32(c.base + s * A_STAGE), 16), db = sdesc_step(da, A_BM * BK * 2);
#pragma unroll
                for (int k = 0; k < BK / 16; ++k)
                    umma_bf16(i < n1 ? tmem : tmem + A_BN, sdesc_step(da, k * 32), sdesc_step(db, k * 32), idesc,
                              ((i == 0 || i == n1) && k == 0) ? 0u : 1u);
                umma_commit(c.empty(s, A_STAGES));
            }
            if (ok)
                umma_commit(c.tfull(0, A_STAGES));
            else
                drain_copies();
        }
        __syncwarp();
    } else {
        // ---- this CTA's partial sums: row = TMEM lane, 64 columns of H and of R a warp
        const int q = warp & 3, ch = (warp - 2) >> 2, row = q * 32 + lane;
        const bool ok = __all_sync(0xffffffffu, mbar_wait(c.tfull(0, A_STAGES), 0, a.status, a.wait_ns));
        if (threadIdx.x == 64) *flag = ok ? 1 : 0;
        if (ok) {
            tc_fence_after();
            const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16);
#pragma unroll 1
            for (int i = 0; i < 4; ++i) {  // 32 columns of H or R each
                const int acc = i >> 1, col = ch * 64 + (i & 1) * 32;
                float v[32];
                tmem_ld32(lane_base + acc * A_BN + col, v);
                uint8_t* dst = c.base + (((size_t)(col / PC) * 2 + acc) * A_BM + row) * (PC * 4);
#pragma unroll
                for (int p = 0; p < 8; ++p) {  // 16-byte pieces, exchanged within 128 bytes by row: conflict-free
                    const int piece = (col % PC) / 4 + p;
                    *reinterpret_cast<float4*>(dst + (((piece & ~7) | ((piece ^ row) & 7)) << 4)) =
                        make_float4(v[4 * p], v[4 * p + 1], v[4 * p + 2], v[4 * p + 3]);
                }
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    cluster_sync();  // every CTA's partial sums are in its shared memory
    if (warp >= 2) {
        // ---- epilogue of part r: a thread takes one row's PC / 2 columns
        const int et = threadIdx.x - 64, row = et & (A_BM - 1), hc = et >> 7, t = trow + row;
        float* tab = reinterpret_cast<float*>(c.base + L::TAB);
        if (et < PC) {
            const int h = h0 + r * PC + et;
            float s1 = 1.f, s2 = 1.f;
            if (a.renorm_pending) {
                s1 = renorm_scale(a.n1[(size_t)cs * a.d_hid + h], ss_row(a, a.parity ^ 1, 0, cs)[h]);
                s2 = renorm_scale(a.n2[(size_t)cs * a.d_hid + h], ss_row(a, a.parity ^ 1, 1, cs)[h]);
            }
            tab[et] = s1;
            tab[PC + et] = s2;
            if (trow == 0) {  // this segment's row sums of squares start from zero
                ss_row(a, a.parity, 0, cs)[h] = 0.f;
                ss_row(a, a.parity, 1, cs)[h] = 0.f;
            }
        }
        bool ok = true;  // every CTA's accumulators were in
        for (int k = 0; k < S; ++k) {
            uint32_t f;
            asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(f) : "r"(map_to_cta(smem_u32(flag), k)) : "memory");
            ok = ok && f != 0;
        }
        // the tile's rows of dH / At lie inside the [C][T][d_hid] scratch (index check of MONE_DEBUG builds)
        ok = ok && MONE_DCHECK(cs < a.C && trow + A_BM <= a.T && h0 + A_BN <= a.d_hid, a.status, DS_PHASE_A_TILE);
        named_bar_sync(EPI_BAR, EPI_THREADS);
        float ct = 0.f, zi = 1.f;
        if (t < a.Tp) {
            const float ev = a.paper ? a.eta[(size_t)cs * a.win + a.tok0 + t]
                                     : (a.eta_in ? a.eta_in[cz * a.eta_cstride + t] : a.lr);
            ct = -ev / (float)a.Tp;
            if (a.zinv) zi = a.zinv[(size_t)cs * a.win + a.tok0 + t];
        }
        const float czi = ct * zi;
        float lsum = 0.f;
        const uint32_t part = smem_u32(c.base + ((size_t)r * 2 * A_BM + row) * (PC * 4));
        const size_t o = ((size_t)cs * a.T + t) * a.d_hid + h0 + r * PC + hc * (PC / 2);
#pragma unroll
        for (int b = 0; b < PC / 2; b += 16) {
            float hv[16], rv[16];
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const int piece = (hc * (PC / 2) + b) / 4 + p;
                const uint32_t off = part + (((piece & ~7) | ((piece ^ row) & 7)) << 4);
                float4 x[S], y[S];  // all loads of the piece before any sum
#pragma unroll
                for (int k = 0; k < S; ++k) {
                    const uint32_t ad = map_to_cta(off, k);
                    x[k] = ld_cluster_f32x4(ad);
                    y[k] = ld_cluster_f32x4(ad + A_BM * PC * 4);
                }
                float4 h4 = x[0], r4 = y[0];
#pragma unroll
                for (int k = 1; k < S; ++k) {
                    h4.x += x[k].x; h4.y += x[k].y; h4.z += x[k].z; h4.w += x[k].w;
                    r4.x += y[k].x; r4.y += y[k].y; r4.z += y[k].z; r4.w += y[k].w;
                }
                hv[4 * p] = h4.x; hv[4 * p + 1] = h4.y; hv[4 * p + 2] = h4.z; hv[4 * p + 3] = h4.w;
                rv[4 * p] = r4.x; rv[4 * p + 1] = r4.y; rv[4 * p + 2] = r4.z; rv[4 * p + 3] = r4.w;
            }
            uint32_t pd[8], pa[8];
#pragma unroll
            for (int j = 0; j < 16; j += 2) {
                float dv[2], av[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int col = hc * (PC / 2) + b + j + u;
                    const float x = hv[j + u] * tab[col] * zi, rr = rv[j + u] * tab[PC + col];
                    const float sg = sigmoid_tanh(x), act = x * sg;
                    lsum = fmaf(act, rr, lsum);
                    dv[u] = czi * rr * (sg * fmaf(x, 1.f - sg, 1.f));  // c_t (dL/dA) SiLU'(x), scaled by 1/|z_t|
                    av[u] = ct * act;
                }
                pd[j / 2] = pack_bf16(dv[0], dv[1]);
                pa[j / 2] = pack_bf16(av[0], av[1]);
            }
            if (ok) {
                st_32b(a.dH + o + b, pd);
                st_32b(a.At + o + b, pa);
            }
        }
        if (a.loss && ok) {
            lsum = warp_sum(lsum);
            if (lane == 0) atomicAdd(&a.loss[cz], -lsum / (float)a.Tp);
        }
    }
    tc_fence_before();
    cluster_sync();  // no CTA leaves while another reads its shared memory
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------ phase B
//
// Tile = 128 hidden rows x 256 weight columns of W1 or of W2 (128 columns of W1 where d_in leaves that
// remainder), accumulated with TMEM lane = hidden row: D = dH^T U or
// At^T Y, both operands MN-major, per 64-token k-block one TMA box of dH or At and of U, two of Y (a tile of W2 may
// take 128 columns from K and 128 from V).
//
// Warps: 0 operand producer (TMA), 1 MMA issuer, 2..9 update, 10 state producer, 11 store warp.
// The fp32 state of a tile moves in chunks of 32 rows x 64 columns of W and mu (16 KB, one TMA box)
// through an 8-slot shared-memory ring.  A chunk belongs to one update warp: its rows are the warp's
// TMEM lane quarter, so a lane owns one hidden row of the chunk.  It holds the row's
// renormalisation scale in a register, reads and writes its part of the row 16 bytes at a time
// (128-byte swizzle: conflict-free), sums the row's squares without a shuffle, and writes the bf16
// copy in whole 32-byte sectors.  No barrier joins the update warps; each waits for its own chunks.
//
// What bounds it: with many chains the state's HBM traffic (18 B per parameter: 128 chains of
// 2048 -> 1024 -> 1024 at T = 256 run at 0.97 of the HBM copy rate), with one chain the latency of a tile.
// The lane-per-row form replaced one with lane = weight column, whose update (scalar shared-memory
// accesses, a 31-shuffle row reduction, 2-byte stores, two barriers a chunk) took a one-chain launch
// (96 tiles, one a CTA) from 18.4 to 21.2 us; merging its six operand boxes a k-block into two changed nothing.
//
// PAIR: clusters of 2 CTAs run tcgen05.mma.cta_group::2 over 256 hidden rows x 256 columns.  CTA r
// stages its own 128 hidden rows of dH (or At) and columns r*128 .. +127 of U (or Y) per k-block,
// so each SM takes in 32 KB of operands a k-block instead of 48 KB for the same 128 x 256
// accumulator.  Both CTAs' loads complete on rank 0's full barrier, rank 0 issues the MMAs, each
// commit arrives on both CTAs' barriers, and the 16 update warps of the pair release an
// accumulator buffer on rank 0's tempty barrier.

constexpr int S_ROWS = 32, S_COLS = 64;                    // state chunk: hidden rows x weight columns
constexpr int S_SLOTS = 8;
// when the store warp hands slots back to the loads: by twos one store later, one by one three stores later, by twos
// three stores later, by fours two stores later (each leaves fewer loads in flight than the one before)
enum { S_PAIRS1, S_LAG3, S_PAIRS3, S_QUADS2 };
constexpr int S_F32 = S_ROWS * S_COLS * 4;                 // 8 KB
constexpr int S_SLOT = 2 * S_F32;                          // W and mu: 16 KB
constexpr int B_THREADS = 12 * 32;
constexpr int B_STATE_WARP = 10;          // TMA loads of state chunks
constexpr int B_STORE_WARP = 11;          // TMA stores of updated chunks, slot release

template <bool PAIR>
struct LayoutBT {
    // operand stages: one CTA 48 KB (128 hidden rows + 256 columns); a pair member 32 KB (its 128
    // hidden rows + 128 columns), three of them in the same space as two
    static constexpr int A_BYTES = B_BM * BK * 2;
    static constexpr int STAGE = A_BYTES + (PAIR ? B_BN / 2 : B_BN) * BK * 2;
    static constexpr int STAGES = PAIR ? 3 : 2;
    static constexpr int RING = STAGES * STAGE;
    static constexpr int STATE = RING;
    static constexpr int BARS = STATE + S_SLOTS * S_SLOT;  // full[S] empty[S] tfull[2] tempty[2] sfull/sdone/sempty[N]
    static constexpr int NBARS = 2 * STAGES + 4 + 3 * S_SLOTS;
    static constexpr int SLOT = BARS + NBARS * 8;
    static constexpr int END = SLOT + 16;
    static constexpr int DYN = END + 1024;
};
using LayoutB = LayoutBT<false>;
using LayoutB2 = LayoutBT<true>;
static_assert(LayoutB::DYN <= 227 * 1024 && LayoutB2::DYN <= 227 * 1024, "phase B shared memory budget");

// Column tiles of [W1 | W2]: each lies in W1 or in W2 (a tile of W2 may take half its columns from K and half
// from V: d_out is a multiple of 256, its half of 128).
__host__ __device__ constexpr int b_col_tiles(int d_in, int d_out) { return (d_in + B_BN - 1) / B_BN + d_out / B_BN; }

// The tiles one CTA of phase B walks: t = first, first + step, ... < count.  The narrow tiles (128 columns, one to a
// stripe of hidden rows where d_in leaves that remainder) come after all others: in their place between them they
// would all fall to the same CTAs wherever step and the stripe's tiles share a factor, and the launch would take as
// long as with whole tiles (1000 tokens of 56 chains of 640 -> 1536 -> 1792, T = 128: 7.04 ms so, 6.90 with them last).
template <bool PAIR>
struct BTiles {
    int first, step, count, n_ht, n_ct, n1, n_wide, rank, d_in;
    __device__ BTiles(const TcArgs& a) {
        d_in = a.d_in;
        n_ht = a.d_hid / (PAIR ? 2 * B_BM : B_BM);
        n1 = (d_in + B_BN - 1) / B_BN;
        n_ct = b_col_tiles(a.d_in, a.d_out);
        count = a.nc * n_ht * n_ct;
        rank = PAIR ? (int)cluster_ctarank() : 0;
        first = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
        step = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
        n_wide = n_ct;
        if (!PAIR && d_in % B_BN) {
            n1 -= 1;  // wide tiles of W1
            n_wide -= 1;
        }
    }
    // tile t: chain of the launch, this CTA's first hidden row, matrix (0: U, W1; 1: Y, W2), first column within
    // it, live columns
    struct Tile {
        int cz, h0, m, col, ncol;
    };
    __device__ Tile decode(int t) const {
        Tile x;
        const int wide = n_wide * (count / n_ct);  // count / n_ct: stripes of hidden rows over all chains
        const bool narrow = !PAIR && t >= wide;
        const int stripe = narrow ? t - wide : t / n_wide, c = narrow ? n1 : t - stripe * n_wide;
        x.cz = stripe / n_ht;
        x.h0 = (stripe - x.cz * n_ht) * (PAIR ? 2 * B_BM : B_BM) + rank * B_BM;
        x.m = c < n1 || narrow ? 0 : 1;
        x.col = (x.m ? c - n1 : c) * B_BN;
        x.ncol = narrow ? B_BN / 2 : B_BN;
        return x;
    }
};

// STEP: also sum |mu_s|^2 per chain (the per-segment metrics); a separate instance, so the update
// loop of the ordinary one keeps its registers
template <bool PAIR, bool STEP>
__global__ void __launch_bounds__(B_THREADS, 1)
tc_phase_b_kernel(const __grid_constant__ CUtensorMap tmUb, const __grid_constant__ CUtensorMap tmKb,
                  const __grid_constant__ CUtensorMap tmVb, const __grid_constant__ CUtensorMap tmDH,
                  const __grid_constant__ CUtensorMap tmAT, const __grid_constant__ CUtensorMap tmW1s,
                  const __grid_constant__ CUtensorMap tmW2s, const TcArgs a) {
    extern __shared__ uint8_t smem_raw[];
    using L = LayoutBT<PAIR>;
    constexpr int NS = L::STAGES;
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t bars = smem_u32(base + L::BARS);
    auto full = [&](int s) { return bars + 8 * s; };
    auto empty = [&](int s) { return bars + 8 * (NS + s); };
    auto tfull = [&](int b) { return bars + 8 * (2 * NS + b); };
    auto tempty = [&](int b) { return bars + 8 * (2 * NS + 2 + b); };
    auto sfull = [&](int k) { return bars + 8 * (2 * NS + 4 + k); };
    auto sempty = [&](int k) { return bars + 8 * (2 * NS + 4 + S_SLOTS + k); };
    auto sdone = [&](int k) { return bars + 8 * (2 * NS + 4 + 2 * S_SLOTS + k); };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const BTiles<PAIR> tl(a);
    using Tile = typename BTiles<PAIR>::Tile;
    if (threadIdx.x == 0) {
        for (int i = 0; i < NS; ++i) {
            mbar_init(full(i), 1);
            mbar_init(empty(i), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(tfull(b), 1);
            mbar_init(tempty(b), PAIR ? 16 : 8);  // every update warp (of both CTAs of a pair)
        }
        for (int k = 0; k < S_SLOTS; ++k) {
            mbar_init(sfull(k), 1);
            mbar_init(sempty(k), 1);
            mbar_init(sdone(k), 1);  // the update warp that owns the chunk
        }
        fence_mbar_init();
    }
    if (warp == 0) {
        if constexpr (PAIR) {
            tmem_alloc_pair(smem_u32(base + L::SLOT), 512);
            tmem_relinquish_pair();
        } else {
            tmem_alloc(smem_u32(base + L::SLOT), 512);
            tmem_relinquish();
        }
    }
    tc_fence_before();
    if constexpr (PAIR)
        cluster_sync();  // barriers of both CTAs initialised, TMEM of the pair allocated
    else
        __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<uint32_t*>(base + L::SLOT);

    const int KB = (a.Tp + BK - 1) / BK;  // tokens beyond T' carry zero dH / At
    const int chunk_bytes = a.momentum ? 2 * S_F32 : S_F32;
    // chunk i of a tile: columns (i >> 3) * 128 + (i & 1) * 64, rows ((i >> 1) & 3) * 32.  A chunk is
    // updated by the warp of that quarter and column half, so every warp takes one chunk of eight in
    // a row and a ring slot always belongs to the same warp; two consecutive boxes cover 512
    // contiguous bytes of each row (with 256 bytes at a time the 128-chain step lost 5% to DRAM).
    auto chunk_col = [](int i) { return (i >> 3) * 128 + (i & 1) * S_COLS; };
    auto chunk_row = [](int i) { return ((i >> 1) & 3) * S_ROWS; };

    if (warp == 0) {
        if (lane == 0) {
            tma_prefetch_map(&tmUb);
            tma_prefetch_map(&tmKb);
            tma_prefetch_map(&tmVb);
            tma_prefetch_map(&tmDH);
            tma_prefetch_map(&tmAT);
            pdl_wait();  // dH and At come from the kernel before
            uint32_t kc = 0;
            bool ok = true;
            for (int t = tl.first; t < tl.count && ok; t += tl.step) {
                const Tile x = tl.decode(t);
                const CUtensorMap* ma = x.m ? &tmAT : &tmDH;
                // this CTA's share of the columns: all 256, or 128 of a pair; of W2 128 at a time from K or V
                const int col = x.col + (PAIR ? tl.rank * (B_BN / 2) : 0), dhalf = a.d_out / 2;
                auto load_y = [&](int c, auto&& load) {
                    const bool v = c >= dhalf;
                    load(v ? &tmVb : &tmKb, (v ? c - dhalf : c) / 64);
                };
                for (int kb = 0; kb < KB; ++kb, ++kc) {
                    const int s = kc % NS;
                    if (kc >= NS && !mbar_wait(empty(s), ((kc / NS) - 1) & 1, a.status, a.wait_ns)) {
                        ok = false;
                        break;
                    }
                    const uint32_t sa = smem_u32(base + s * L::STAGE), sb = sa + L::A_BYTES;
                    if constexpr (PAIR) {
                        const uint32_t fb = map_to_cta(full(s), 0);  // both CTAs' loads complete on rank 0's barrier
                        if (tl.rank == 0) mbar_expect_tx(full(s), 2 * L::STAGE);
                        tma_load_4d_pair(sa, ma, fb, 0, kb * BK, x.h0 / 64, a.c0 + x.cz);
                        if (x.m)
                            load_y(col, [&](const CUtensorMap* mb, int blk) {
                                tma_load_4d_pair(sb, mb, fb, 0, a.y_row0 + kb * BK, blk, x.cz);
                            });
                        else
                            tma_load_4d_pair(sb, &tmUb, fb, 0, a.u_row0 + kb * BK, col / 64, a.u_chain0 + x.cz);
                    } else {
                        mbar_expect_tx(full(s), L::STAGE);
                        tma_load_4d(sa, ma, full(s), 0, kb * BK, x.h0 / 64, a.c0 + x.cz);
                        if (x.m) {
#pragma unroll
                            for (int hb = 0; hb < 2; ++hb)
                                load_y(col + hb * 128, [&](const CUtensorMap* mb, int blk) {
                                    tma_load_4d(sb + hb * 2 * BOX, mb, full(s), 0, a.y_row0 + kb * BK, blk, x.cz);
                                });
                        } else {  // blocks past d_in read as zeros
                            tma_load_4d(sb, &tmUb, full(s), 0, a.u_row0 + kb * BK, col / 64, a.u_chain0 + x.cz);
                        }
                    }
                }
            }
            if (PAIR && !ok) drain_copies();
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0 && (!PAIR || tl.rank == 0)) {
            const uint32_t idesc = idesc_bf16_f32(PAIR ? 2 * B_BM : B_BM, B_BN, true, true);
            uint32_t kc = 0;
            int local = 0;
            bool ok = true;
            for (int t = tl.first; t < tl.count && ok; t += tl.step, ++local) {
                const int b = local & 1;
                if (local >= 2 && !mbar_wait(tempty(b), ((local >> 1) - 1) & 1, a.status, a.wait_ns)) break;
                tc_fence_after();
                const uint32_t d = tmem + b * B_BN;
                for (int kb = 0; kb < KB; ++kb, ++kc) {
                    const int s = kc % NS;
                    if (!mbar_wait(full(s), (kc / NS) & 1, a.status, a.wait_ns)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint64_t da0 = sdesc_sw128(smem_u32(base + s * L::STAGE), BOX), db0 = sdesc_step(da0, L::A_BYTES);
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k) {
                        const uint64_t da = sdesc_step(da0, k * 16 * 128), db = sdesc_step(db0, k * 16 * 128);
                        if constexpr (PAIR)
                            umma_bf16_pair(d, da, db, idesc, (kb == 0 && k == 0) ? 0u : 1u);
                        else
                            umma_bf16(d, da, db, idesc, (kb == 0 && k == 0) ? 0u : 1u);
                    }
                    if constexpr (PAIR)
                        umma_commit_pair(empty(s), 0x3);
                    else
                        umma_commit(empty(s));
                }
                if (!ok) break;
                if constexpr (PAIR)
                    umma_commit_pair(tfull(b), 0x3);
                else
                    umma_commit(tfull(b));
            }
            if (PAIR && !ok) drain_copies();
        }
        __syncwarp();
    } else if (warp == B_STATE_WARP) {
        // ---- state producer: W (and mu) chunks of every tile, in update order.  It does not wait for the
        //      kernel before this one (phase A), which writes neither; what wrote them is complete.
        if (lane == 0) {
            tma_prefetch_map(&tmW1s);
            tma_prefetch_map(&tmW2s);
            uint32_t seq = 0;
            bool ok = true;
            for (int t = tl.first; t < tl.count && ok; t += tl.step) {
                const Tile x = tl.decode(t);
                for (int i = 0; i < x.ncol / 16; ++i, ++seq) {
                    const int k = seq % S_SLOTS;
                    if (seq >= S_SLOTS && !mbar_wait(sempty(k), ((seq / S_SLOTS) - 1) & 1, a.status, a.wait_ns)) {
                        ok = false;
                        break;
                    }
                    const int col = x.col + chunk_col(i);
                    // the chunk lies inside the matrix (a tiled copy's block coordinate counts 32 columns)
                    if (!MONE_DCHECK((col & 31) == 0 && col + S_COLS <= (x.m ? a.d_out : a.d_in), a.status, DS_TMA_X)) {
                        ok = false;
                        break;
                    }
                    mbar_expect_tx(sfull(k), chunk_bytes);
                    tma_load_5d(smem_u32(base + L::STATE + k * S_SLOT), x.m ? &tmW2s : &tmW1s, sfull(k), 0,
                                x.h0 + chunk_row(i), col / 32, a.c0 + x.cz, 0);
                }
            }
        }
        __syncwarp();
    } else if (warp == B_STORE_WARP) {
        // ---- store warp: write every updated chunk back with TMA, then free its slot
        if (lane == 0) {
            uint32_t seq = 0;
            bool ok = true;
            for (int t = tl.first; t < tl.count && ok; t += tl.step) {
                const Tile x = tl.decode(t);
                for (int i = 0; i < x.ncol / 16; ++i, ++seq) {
                    const int k = seq % S_SLOTS;
                    if (!mbar_wait(sdone(k), (seq / S_SLOTS) & 1, a.status, a.wait_ns)) {
                        ok = false;
                        break;
                    }
                    tma_store_5d(x.m ? &tmW2s : &tmW1s, smem_u32(base + L::STATE + k * S_SLOT), 0,
                                 x.h0 + chunk_row(i), (x.col + chunk_col(i)) / 32, a.c0 + x.cz, 0);
                    bulk_commit();
                    // hand slots back whose stores have read them: `done` is the last such chunk, `n` of them at once
                    auto hand_back = [&](uint32_t done, int n) {
                        for (int u = n - 1; u >= 0; --u) mbar_arrive(sempty((done - u) % S_SLOTS));
                    };
                    if (a.store_mode == S_LAG3) {
                        bulk_wait_read<3>();
                        if (seq >= 3) hand_back(seq - 3, 1);
                    } else if (a.store_mode == S_QUADS2) {
                        if ((seq & 3) == 1 && seq > 1) {
                            bulk_wait_read<2>();
                            hand_back(seq - 2, 4);
                        }
                    } else if (!(seq & 1) && seq) {
                        if (a.store_mode == S_PAIRS3) {
                            bulk_wait_read<3>();
                            if (seq > 3) hand_back(seq - 3, 2);
                        } else {
                            bulk_wait_read<1>();
                            hand_back(seq - 1, 2);
                        }
                    }
                }
            }
            bulk_wait_all();
        }
        __syncwarp();
    } else {
        // ---- update warps 2..9: TMEM lane quarter q (32 hidden rows, one per lane), column half
        const int q = warp & 3, half = (warp - 2) >> 2;
        const uint32_t tempty_rank0 = PAIR ? map_to_cta(tempty(0), 0) : tempty(0);
        const uint64_t wpol = l2_evict_last_policy();  // phase A of the next segment reads the copy
        pdl_wait();  // the row sums of squares were zeroed by the kernel before
        pdl_trigger();
        bool finite = true;
        uint32_t tile_seq0 = 0;  // chunk sequence number of the current tile's first chunk
        int local = 0;
        for (int t = tl.first; t < tl.count; t += tl.step, ++local) {
            const Tile x = tl.decode(t);
            const int cs = a.c0 + x.cz, which = x.m ? 1 : 0, width = x.m ? a.d_out : a.d_in;
            const int b = local & 1, row = x.h0 + q * 32 + lane;
            // the tile's rows and columns lie inside the chain's W (index check of MONE_DEBUG builds)
            const bool wr = MONE_DCHECK(cs < a.C && row < a.d_hid && x.col + x.ncol <= width, a.status, DS_PHASE_B_TILE);
            float sc = 1.f, beta = 0.f;
            if (a.renorm_pending && wr)
                sc = renorm_scale((x.m ? a.n2 : a.n1)[(size_t)cs * a.d_hid + row], ss_row(a, a.parity ^ 1, which, cs)[row]);
            if (a.momentum) {  // beta_s = sigmoid(mean_t w_beta . x_t + b_beta)
                const float* db = a.dbeta + (size_t)cs * a.win + a.tok0;
                float v = 0.f;
#pragma unroll 4
                for (int tk = lane; tk < a.Tp; tk += 32) v += db[tk];
                beta = sigmoidf_(warp_sum(v) / (float)a.Tp + a.b_beta[cs]);
            }
            const int ncg = x.ncol / 128;
            bool ok = __all_sync(0xffffffffu, mbar_wait(tfull(b), (local >> 1) & 1, a.status, a.wait_ns));
            if (!ok) break;
            tc_fence_after();
            const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16) + b * B_BN + half * S_COLS;
            float ss = 0.f, step = 0.f;  // sums of squares of this lane's part of its row of W, and of mu
            bf16* wrow = (x.m ? a.W2b : a.W1b) + ((size_t)cs * a.d_hid + row) * width + x.col + half * S_COLS;
#pragma unroll 1
            for (int cg = 0; cg < ncg; ++cg) {
                const uint32_t seq = tile_seq0 + cg * S_SLOTS + q * 2 + half;
                const int k = seq % S_SLOTS;
                ok = __all_sync(0xffffffffu, mbar_wait(sfull(k), (seq / S_SLOTS) & 1, a.status, a.wait_ns));
                if (!ok) break;
                uint8_t* slot = base + L::STATE + k * S_SLOT + lane * 128;
#pragma unroll
                for (int blk = 0; blk < S_COLS / 32; ++blk) {
                    float g[32];
                    tmem_ld32(lane_base + cg * 128 + blk * 32, g);
                    if (cg == ncg - 1 && blk == S_COLS / 32 - 1) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) {
                            if constexpr (PAIR)
                                mbar_arrive_remote(tempty_rank0 + 8 * b);
                            else
                                mbar_arrive(tempty(b));
                        }
                    }
                    uint8_t* wp = slot + blk * 4096;
                    uint32_t pk[16];
#pragma unroll
                    for (int p = 0; p < 8; ++p) {
                        const int off = (p ^ (lane & 7)) << 4;
                        float4 w = *reinterpret_cast<const float4*>(wp + off);
                        float4 m = make_float4(g[4 * p], g[4 * p + 1], g[4 * p + 2], g[4 * p + 3]);
                        if (a.momentum) {
                            float4* mp = reinterpret_cast<float4*>(wp + S_F32 + off);
                            const float4 mo = *mp;
                            m.x = fmaf(beta, mo.x, m.x);
                            m.y = fmaf(beta, mo.y, m.y);
                            m.z = fmaf(beta, mo.z, m.z);
                            m.w = fmaf(beta, mo.w, m.w);
                            *mp = m;
                        }
                        w.x = fmaf(sc, w.x, -m.x);
                        w.y = fmaf(sc, w.y, -m.y);
                        w.z = fmaf(sc, w.z, -m.z);
                        w.w = fmaf(sc, w.w, -m.w);
                        *reinterpret_cast<float4*>(wp + off) = w;
                        ss = fmaf(w.x, w.x, fmaf(w.y, w.y, fmaf(w.z, w.z, fmaf(w.w, w.w, ss))));
                        if constexpr (STEP)
                            step = fmaf(m.x, m.x, fmaf(m.y, m.y, fmaf(m.z, m.z, fmaf(m.w, m.w, step))));
                        pk[2 * p] = pack_bf16(w.x, w.y);
                        pk[2 * p + 1] = pack_bf16(w.z, w.w);
                    }
                    if (wr) {
                        st_32b_hint(wrow + cg * 128 + blk * 32, pk, wpol);
                        st_32b_hint(wrow + cg * 128 + blk * 32 + 16, pk + 8, wpol);
                    }
                }
                // make this warp's shared-memory writes visible to the TMA store, then tell the store warp
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(sdone(k));
            }
            if (!ok) break;
            finite = finite && isfinite(ss);  // a NaN or Inf weight makes its row's sum non-finite
            if (wr) atomicAdd(&ss_row(a, a.parity, which, cs)[row], ss);
            if constexpr (STEP) {  // per-segment metric: the tile's share of |mu_s|^2
                step = warp_sum(step);
                if (lane == 0) atomicAdd(&a.step_sq[x.cz], step);
            }
            tile_seq0 += x.ncol / 16;
        }
        if (!finite) atomicOr(a.status, DEV_NONFINITE);
    }
    tc_fence_before();
    if constexpr (PAIR)
        cluster_sync();  // every MMA of the pair has completed and every TMEM read is done
    else
        __syncthreads();
    tc_fence_after();
    if (warp == 0) {
        if constexpr (PAIR)
            tmem_dealloc_pair(tmem, 512);
        else
            tmem_dealloc(tmem, 512);
    }
}

TcArgs make_args(const DevState& s, const SegWork& w) {
    TcArgs a{};
    a.d_in = s.d_in; a.d_out = s.d_out; a.d_hid = s.d_hid; a.T = s.T; a.Tp = w.Tp; a.c0 = w.c0; a.nc = w.nc;
    a.C = s.C;
    a.paper = s.mode == 1; a.momentum = s.momentum; a.renorm_pending = w.renorm_pending; a.parity = w.parity;
    a.u_row0 = a.paper ? (int)w.u_off : (int)w.row0;
    a.tok0 = w.u_off;
    a.win = s.win_rows;
    a.u_chain0 = a.paper ? w.c0 : 0;
    a.y_row0 = w.y_scratch ? 0 : (int)w.row0;
    a.lr = s.lr;
    a.eta_in = w.eta_in ? w.eta_in + w.row0 : nullptr;
    a.eta_cstride = w.eta_cstride;
    a.eta = s.eta; a.dbeta = s.dbeta; a.b_beta = s.b_beta;
    a.zinv = a.paper ? s.zinv : nullptr;
    a.W1b = s.W1b; a.W2b = s.W2b;
    a.n1 = s.n1; a.n2 = s.n2; a.sumsq = s.sumsq;
    a.dH = reinterpret_cast<bf16*>(s.dHt); a.At = reinterpret_cast<bf16*>(s.Att);
    a.loss = w.loss; a.step_sq = w.step_sq; a.status = s.status;
    a.wait_ns = kWaitLimitNs;
    return a;
}

// ------------------------------------------------------------------ memory read (Eq. 4)
//
// The read of generate_kv on the bf16 path, on the tensor cores, in two kernels:
//   hidden:  A_q = SiLU(Z_q W1^T / |z_q|)  tile = (128 queries, 128 hidden units, chain), K = d_in
//   out:     O = A_q W2, then per output head h of width hd: g_h o_h / sqrt(mean(o_h^2) + eps)
//            written into the caller's K / V layout   tile = (128 queries, 128 outputs, chain), K = d_hid
// One tile per CTA: warp 0 streams the query rows and the bf16 weight copy with TMA,
// warp 1 issues tcgen05.mma into a 128-column TMEM accumulator, warps 2..5 (one per TMEM
// lane quarter, lane = query) run the epilogue.  Each weight tile is read by ceil(Q/128)
// CTAs; query rows >= Q arrive as TMA zero fill and are never stored.  W2 is [hidden][out],
// so in the out kernel the weight operand is MN-major (64-column boxes, as in phase B).
// A launch with more tiles than SMs runs two CTAs per SM (three 32 KB stages each), so one
// CTA's epilogue overlaps the other's loads; a launch that fits in one wave runs one CTA per
// SM with six stages, twice the operand bytes in flight for its single K loop.  Reads of more tiles
// than one wave of two CTAs an SM run on CTA pairs (tc_read_pair_kernel).
constexpr int R_STAGE = 2 * 128 * BK * 2;  // 32 KB: 128 query rows + 128 weight rows / columns
constexpr int R_THREADS = 6 * 32;
constexpr uint32_t R_EPI_BAR = 1;
template <int NST>
struct LRT {
    static constexpr int CTAS_PER_SM = NST <= 3 ? 2 : 1;
    static constexpr int RING = NST * R_STAGE;
    static constexpr int BARS = RING;  // full[S] empty[S] tfull
    static constexpr int NBARS = 2 * NST + 1;
    static constexpr int SLOT = BARS + (NBARS * 8 + 15) / 16 * 16;
    static constexpr int FLAG = SLOT + 16;
    static constexpr int TAB = FLAG + 16;  // MSE_HIDDEN: renorm scales s1, s2 of the tile's rows
    static constexpr int STG = TAB + 256 * 4;  // 4 epilogue warps x 2 KB transpose buffers
    static constexpr int END = STG + 4 * 2048;
    static constexpr int DYN = END + 1024;
};
using LR = LRT<3>;   // several waves
using LR6 = LRT<6>;  // one wave
static_assert(LR::CTAS_PER_SM * (LR::DYN + 1024) <= 228 * 1024, "read kernel CTAs per SM");
static_assert(LR6::DYN <= 227 * 1024, "read kernel shared memory");
static_assert(LR::STG % 16 == 0, "staging buffers hold 16-byte pieces");

struct ReadArgs {
    int Q, d_in, d_hid, d_out, n_kv, L;
    float eps;
    const float* gate;     // [C][2 n_kv] per-head gates, or null (gate 1)
    bf16* Aq;              // [C][Q][d_hid]
    bf16 *Kout, *Vout;     // caller's K / V, element strides s0 (context), s1 (layer), s2 (head), s3 (query)
    long long s0, s1, s2, s3;
    int* status;
    // operand coordinates: A rows start at a_row0 + 128 * blockIdx.x of chain a_chain0 + blockIdx.z,
    // weights of chain b_chain0 + blockIdx.z
    int a_row0, a_chain0, b_chain0;
    // squared-error loss pre-pass (MSE_* modes): one segment of chains b_chain0 + blockIdx.z
    int C, T, Tp, win, parity, renorm_pending;
    long long tok0, row0, n_rows, y_cstride;
    const float *zinv, *n1, *n2, *sumsq;  // as in TcArgs
    const bf16 *K, *V;     // caller's targets of the group (chain z at z * y_cstride)
    bf16 *Kres, *Vres;     // [C][T][d_out/2] residual targets y - M(u)
    float* loss;           // [nc] or null
    // MSE_HIDDEN, when phase A runs in its R-only form: also write At = c_t SiLU(x) and
    // c_t SiLU'(x) / |z_t| (into dH), with c_t = -eta_t / T'
    bf16 *At, *Sp;         // [C][T][d_hid] or null
    int paper;
    float lr;
    const float *eta, *eta_in;
    long long eta_cstride;
    const float* qzinv;    // read: 1/|z| per query [C][Q] (paper mode), or null
};

enum { READ_HIDDEN = 0, MSE_HIDDEN = 1, MSE_OUT = 2 };  // other MODEs: read out with heads of width MODE

// Epilogue of N hidden units n0 .. of a warp's 32 queries qw .. of chain c (lane = query, accumulator at
// lane_base): A_q = SiLU(H / |z_q|).
template <int N>
__device__ __forceinline__ void read_hidden_epilogue(const ReadArgs& a, uint32_t lane_base, int c, int qw, int n0, int lane,
                                                     uint8_t* stg) {
    bf16* row0 = a.Aq + ((size_t)c * a.Q + qw) * a.d_hid + n0;
    // the tile's columns of A_q lie inside [Q][d_hid] (index check of MONE_DEBUG builds)
    const bool wr = MONE_DCHECK(n0 + N <= a.d_hid, a.status, DS_READ_TILE);
    const float zi = a.qzinv && qw + lane < a.Q ? a.qzinv[(size_t)c * a.Q + qw + lane] : 1.f;
#pragma unroll 1
    for (int cc = 0; cc < N / 32; ++cc) {
        float hv[32];
        tmem_ld32(lane_base + cc * 32, hv);
#pragma unroll
        for (int j = 0; j < 32; ++j) hv[j] *= zi;
        uint32_t pk[16];
#pragma unroll
        for (int j = 0; j < 16; ++j)
            pk[j] = pack_bf16(hv[2 * j] * sigmoidf_(hv[2 * j]), hv[2 * j + 1] * sigmoidf_(hv[2 * j + 1]));
        if (wr) store_rows_coalesced(stg, pk, row0 + cc * 32, a.d_hid, lane, a.Q - qw);
    }
}

// The same of N outputs n0 .. (heads of width HD): normalised, gated and written to the caller's K / V.
template <int N, int HD>
__device__ __forceinline__ void read_out_epilogue(const ReadArgs& a, uint32_t lane_base, int c, int qw, int n0, int lane) {
    const int qi = qw + lane;
    const int nh = 2 * a.n_kv;
#pragma unroll 1
    for (int hh = 0; hh < N / HD; ++hh) {
        float v[HD];
#pragma unroll
        for (int cc = 0; cc < HD / 32; ++cc)
            tmem_ld32(lane_base + hh * HD + cc * 32, *reinterpret_cast<float(*)[32]>(v + cc * 32));
        float ss = 0.f;
#pragma unroll
        for (int i = 0; i < HD; ++i) ss = fmaf(v[i], v[i], ss);
        const int head = n0 / HD + hh;
        const bool wr = MONE_DCHECK(head < nh, a.status, DS_READ_TILE);
        const float g = a.gate && wr ? a.gate[(size_t)c * nh + head] : 1.f;
        const float sc = g / sqrtf(ss / (float)HD + a.eps);
        if (qi < a.Q && wr) {
            const int kvh = head < a.n_kv ? head : head - a.n_kv;
            bf16* out = (head < a.n_kv ? a.Kout : a.Vout) + (long long)(c / a.L) * a.s0 + (long long)(c % a.L) * a.s1 +
                        (long long)kvh * a.s2 + (long long)qi * a.s3;
            if ((reinterpret_cast<uintptr_t>(out) & 15u) == 0) {
#pragma unroll
                for (int i = 0; i < HD; i += 8)
                    *reinterpret_cast<uint4*>(out + i) =
                        make_uint4(pack_bf16(v[i] * sc, v[i + 1] * sc), pack_bf16(v[i + 2] * sc, v[i + 3] * sc),
                                   pack_bf16(v[i + 4] * sc, v[i + 5] * sc), pack_bf16(v[i + 6] * sc, v[i + 7] * sc));
            } else {
#pragma unroll
                for (int i = 0; i < HD; ++i) out[i] = __float2bfloat16_rn(v[i] * sc);
            }
        }
    }
}

// MODE READ_HIDDEN: A_q = SiLU(Z_q W1^T / |z_q|).  MODE 64 / 128: the read's out kernel with heads
// of that width.  MODE MSE_HIDDEN: A' = SiLU(s1 (1/|z_t|) H) s2, the segment's activations
// with the pending renorm scales (s2 folded in, so A' W2raw = A W2).  MODE MSE_OUT: the
// residual target y_t - M(u_t) = y_t - A'_t W2raw (and the segment's squared-error loss).
template <int MODE, int NST>
__global__ void __launch_bounds__(R_THREADS, LRT<NST>::CTAS_PER_SM)
tc_read_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const ReadArgs a) {
    constexpr bool OUT = MODE != READ_HIDDEN && MODE != MSE_HIDDEN;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t bars = smem_u32(base + LRT<NST>::BARS);
    auto full = [&](int s) { return bars + 8 * s; };
    auto empty = [&](int s) { return bars + 8 * (NST + s); };
    const uint32_t tfull = bars + 8 * (2 * NST);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < NST; ++s) {
            mbar_init(full(s), 1);
            mbar_init(empty(s), 1);
        }
        mbar_init(tfull, 1);
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(smem_u32(base + LRT<NST>::SLOT), 128);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<uint32_t*>(base + LRT<NST>::SLOT);
    const int q0 = blockIdx.x * 128, n0 = blockIdx.y * 128, c = blockIdx.z;
    const int KB = (OUT ? a.d_hid : a.d_in) / BK;
    float* table = reinterpret_cast<float*>(base + LRT<NST>::TAB);

    if (warp == 0) {
        if (lane == 0) {
            tma_prefetch_map(&tmA);
            tma_prefetch_map(&tmB);
            for (int kb = 0; kb < KB; ++kb) {
                const int s = kb % NST;
                if (kb >= NST && !mbar_wait(empty(s), ((kb / NST) - 1) & 1, a.status)) break;
                const uint32_t sa = smem_u32(base + s * R_STAGE), sb = sa + 128 * BK * 2, fb = full(s);
                mbar_expect_tx(fb, R_STAGE);
                tma_load_3d(sa, &tmA, fb, kb * BK, a.a_row0 + q0, a.a_chain0 + c);
                if (OUT) {
                    tma_load_3d(sb, &tmB, fb, n0, kb * BK, a.b_chain0 + c);
                    tma_load_3d(sb + BOX, &tmB, fb, n0 + 64, kb * BK, a.b_chain0 + c);
                } else {
                    tma_load_3d(sb, &tmB, fb, kb * BK, n0, a.b_chain0 + c);
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = idesc_bf16_f32(128, 128, false, OUT);
            bool ok = true;
            for (int kb = 0; kb < KB; ++kb) {
                const int s = kb % NST;
                if (!mbar_wait(full(s), (kb / NST) & 1, a.status)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t sa = smem_u32(base + s * R_STAGE);
                const uint64_t da = sdesc_sw128(sa, 16), db = sdesc_sw128(sa + 128 * BK * 2, OUT ? BOX : 16);
#pragma unroll
                for (int k = 0; k < BK / 16; ++k)
                    umma_bf16(tmem, sdesc_step(da, k * 32), sdesc_step(db, OUT ? k * 16 * 128 : k * 32), idesc,
                              (kb == 0 && k == 0) ? 0u : 1u);
                umma_commit(empty(s));
            }
            if (ok) umma_commit(tfull);
        }
        __syncwarp();
    } else {
        const int q = warp & 3;  // TMEM lane quarter of this warp
        int* flag = reinterpret_cast<int*>(base + LRT<NST>::FLAG);
        if constexpr (MODE == MSE_HIDDEN) {
            // renorm scales of this tile's 128 hidden rows (one per epilogue thread)
            const int h = n0 + (int)threadIdx.x - 64, cs = a.b_chain0 + c;
            float s1 = 1.f, s2 = 1.f;
            if (a.renorm_pending) {
                // row sums of squares of the last update: [2 parity][2 matrix][C][d_hid]
                const float* ss1 = a.sumsq + ((size_t)((a.parity ^ 1) * 2 + 0) * a.C + cs) * a.d_hid;
                const float* ss2 = a.sumsq + ((size_t)((a.parity ^ 1) * 2 + 1) * a.C + cs) * a.d_hid;
                s1 = renorm_scale(a.n1[(size_t)cs * a.d_hid + h], ss1[h]);
                s2 = renorm_scale(a.n2[(size_t)cs * a.d_hid + h], ss2[h]);
            }
            table[threadIdx.x - 64] = s1;
            table[128 + threadIdx.x - 64] = s2;
        }
        if (threadIdx.x == 64) *flag = mbar_wait(tfull, 0, a.status) ? 1 : 0;
        __syncwarp();
        named_bar_sync(R_EPI_BAR, 128);
        if (*flag) {
            tc_fence_after();
            const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16);
            const int qw = q0 + q * 32;  // first query row of this warp
            if constexpr (MODE == MSE_HIDDEN) {
                const int cs = a.b_chain0 + c, t = qw + lane;
                const float zi = (t < a.Tp) ? (a.zinv ? a.zinv[(size_t)cs * a.win + a.tok0 + t] : 1.f) : 0.f;
                float ct = 0.f;  // c_t = -eta_t / T' (R-only outputs)
                if (a.At && t < a.Tp) {
                    const float ev = a.paper ? a.eta[(size_t)cs * a.win + a.tok0 + t]
                                             : (a.eta_in ? a.eta_in[c * a.eta_cstride + t] : a.lr);
                    ct = -ev / (float)a.Tp;
                }
                const float czi = ct * zi;
                uint8_t* stg = base + LRT<NST>::STG + (warp - 2) * 2048;
                const size_t roff = ((size_t)cs * a.T + qw) * a.d_hid + n0;
#pragma unroll 1
                for (int cc = 0; cc < 4; ++cc) {
                    float hv[32];
                    tmem_ld32(lane_base + cc * 32, hv);
                    uint32_t pk[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const int k0 = cc * 32 + 2 * j;
                        const float x0 = hv[2 * j] * table[k0] * zi, x1 = hv[2 * j + 1] * table[k0 + 1] * zi;
                        pk[j] = pack_bf16(x0 * sigmoidf_(x0) * table[128 + k0], x1 * sigmoidf_(x1) * table[128 + k0 + 1]);
                    }
                    store_rows_coalesced(stg, pk, a.Aq + roff + cc * 32, a.d_hid, lane);
                    if (a.At) {  // the R-only form of phase A takes At and c SiLU'(x) / |z| from here
                        uint32_t pa[16], ps[16];
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const int k0 = cc * 32 + 2 * j;
                            const float x0 = hv[2 * j] * table[k0] * zi, x1 = hv[2 * j + 1] * table[k0 + 1] * zi;
                            const float g0 = sigmoid_tanh(x0), g1 = sigmoid_tanh(x1);
                            pa[j] = pack_bf16(ct * x0 * g0, ct * x1 * g1);
                            ps[j] = pack_bf16(czi * (g0 * fmaf(x0, 1.f - g0, 1.f)), czi * (g1 * fmaf(x1, 1.f - g1, 1.f)));
                        }
                        store_rows_coalesced(stg, pa, a.At + roff + cc * 32, a.d_hid, lane);
                        store_rows_coalesced(stg, ps, a.Sp + roff + cc * 32, a.d_hid, lane);
                    }
                }
            } else if constexpr (MODE == MSE_OUT) {
                const int cs = a.b_chain0 + c, t = qw + lane, dh = a.d_out / 2;
                const bool kpart = n0 < dh;
                const int col0 = kpart ? n0 : n0 - dh;
                const bool live = t < a.Tp && a.row0 + t < a.n_rows;
                const bf16* yrow = (kpart ? a.K : a.V) + (size_t)c * a.y_cstride + (size_t)(a.row0 + t) * dh + col0;
                uint8_t* stg = base + LRT<NST>::STG + (warp - 2) * 2048;
                bf16* row0 = (kpart ? a.Kres : a.Vres) + ((size_t)cs * a.T + qw) * dh + col0;
                float lsum = 0.f;
#pragma unroll 1
                for (int cc = 0; cc < 4; ++cc) {
                    float ov[32];
                    tmem_ld32(lane_base + cc * 32, ov);
                    uint32_t pk[16];
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        uint4 y = make_uint4(0, 0, 0, 0);
                        if (live) y = *reinterpret_cast<const uint4*>(yrow + cc * 32 + v * 8);
                        const __nv_bfloat162* yb = reinterpret_cast<const __nv_bfloat162*>(&y);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const float2 yf = __bfloat1622float2(yb[u]);
                            const int j = v * 8 + 2 * u;
                            const float r0 = live ? yf.x - ov[j] : 0.f, r1 = live ? yf.y - ov[j + 1] : 0.f;
                            lsum = fmaf(r0, r0, fmaf(r1, r1, lsum));
                            pk[v * 4 + u] = pack_bf16(r0, r1);
                        }
                    }
                    store_rows_coalesced(stg, pk, row0 + cc * 32, dh, lane);
                }
                if (a.loss) {
                    lsum = warp_sum(lsum);
                    if (lane == 0) atomicAdd(&a.loss[c], 0.5f * lsum / (float)a.Tp);
                }
            } else if constexpr (!OUT) {
                read_hidden_epilogue<128>(a, lane_base, c, qw, n0, lane, base + LRT<NST>::STG + (warp - 2) * 2048);
            } else {
                read_out_epilogue<128, MODE>(a, lane_base, c, qw, n0, lane);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 128);
}

// ------------------------------------------------------------------ memory read of many tiles
//
// The hidden and out kernels on CTA pairs that share each tcgen05.mma: tile = (256 queries, 128 in each CTA,
// 256 hidden units or outputs, of whose weights each CTA stages 128), one pair per two SMs running through the
// tiles, two accumulators in TMEM so that a tile's epilogue overlaps the next tile's MMAs.  The 128 x 128 tiles
// of tc_read_kernel take 128 bytes of operands a clock from L2 at the full MMA rate and are bound by that at
// half of it; these tiles take 64.  1000 queries of 28 chains of 3072 -> 2048 -> 2048 (587 GFLOP): 580 us for
// the two kernels on 128 x 128 tiles, 380 on the pairs (1.5 PFLOP/s, of 1.9 measured in large GEMMs), 435 with
// four epilogue warps instead of eight.
constexpr int RP_STAGES = 6, RP_BN = 256;
constexpr int RP_EPI = 8, RP_THREADS = (2 + RP_EPI) * 32;  // epilogue warps: two to a TMEM lane quarter, half the columns each
struct LRP {
    static constexpr int RING = RP_STAGES * R_STAGE;  // a stage: 128 query rows + 128 weight rows / columns
    static constexpr int BARS = RING;                 // full[S] empty[S] tfull[2] tempty[2]
    static constexpr int NBARS = 2 * RP_STAGES + 4;
    static constexpr int SLOT = BARS + NBARS * 8;
    static constexpr int STG = SLOT + 16;             // per epilogue warp: 2 KB transpose buffer
    static constexpr int END = STG + RP_EPI * 2048;
    static constexpr int DYN = END + 1024;
};
static_assert(LRP::DYN <= 227 * 1024 && LRP::STG % 16 == 0, "shared memory budget");

template <int MODE>
__global__ void __launch_bounds__(RP_THREADS, 1)
tc_read_pair_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const ReadArgs a) {
    constexpr bool OUT = MODE != READ_HIDDEN;
    extern __shared__ uint8_t smem_raw[];
    Ctl c;
    c.base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    c.bars = smem_u32(c.base + LRP::BARS);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    if (threadIdx.x == 0) {
        for (int i = 0; i < RP_STAGES; ++i) {
            mbar_init(c.full(i), 1);
            mbar_init(c.empty(i, RP_STAGES), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(c.tfull(b, RP_STAGES), 1);
            mbar_init(c.tempty(b, RP_STAGES), 2 * RP_EPI);
        }
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc_pair(smem_u32(c.base + LRP::SLOT), 512);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    cluster_sync();  // barriers of both CTAs initialised, TMEM of the pair allocated
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<uint32_t*>(c.base + LRP::SLOT);
    const int n_q = (a.Q + 255) / 256, n_n = (OUT ? a.d_out : a.d_hid) / RP_BN;
    const int ntiles = a.C * n_n * n_q, cluster = blockIdx.x >> 1, nclusters = gridDim.x >> 1;
    const int KB = (OUT ? a.d_hid : a.d_in) / BK;

    if (warp == 0) {
        if (lane == 0) {
            tma_prefetch_map(&tmA);
            tma_prefetch_map(&tmB);
            uint32_t kc = 0;
            bool ok = true;
            for (int t = cluster; t < ntiles && ok; t += nclusters) {
                const int cz = t / (n_n * n_q), n0 = (t / n_q) % n_n * RP_BN + (int)rank * 128;
                const int q0 = t % n_q * 256 + (int)rank * 128;
                for (int kb = 0; kb < KB; ++kb, ++kc) {
                    const int s = kc % RP_STAGES;
                    if (kc >= RP_STAGES && !mbar_wait(c.empty(s, RP_STAGES), ((kc / RP_STAGES) - 1) & 1, a.status)) {
                        ok = false;
                        break;
                    }
                    // both CTAs' loads complete on rank 0's full barrier
                    const uint32_t sa = smem_u32(c.base + s * R_STAGE), sb = sa + 128 * BK * 2;
                    const uint32_t fb = map_to_cta(c.full(s), 0);
                    if (rank == 0) mbar_expect_tx(c.full(s), 2 * R_STAGE);
                    tma_load_3d_pair(sa, &tmA, fb, kb * BK, q0, cz);
                    if (OUT) {
                        tma_load_3d_pair(sb, &tmB, fb, n0, kb * BK, cz);
                        tma_load_3d_pair(sb + BOX, &tmB, fb, n0 + 64, kb * BK, cz);
                    } else {
                        tma_load_3d_pair(sb, &tmB, fb, kb * BK, n0, cz);
                    }
                }
            }
            if (!ok) drain_copies();
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {
            const uint32_t idesc = idesc_bf16_f32(256, RP_BN, false, OUT);
            uint32_t kc = 0;
            int local = 0;
            bool ok = true;
            for (int t = cluster; t < ntiles && ok; t += nclusters, ++local) {
                const int b = local & 1;
                if (local >= 2 && !mbar_wait(c.tempty(b, RP_STAGES), ((local >> 1) - 1) & 1, a.status)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                for (int kb = 0; kb < KB; ++kb, ++kc) {
                    const int s = kc % RP_STAGES;
                    if (!mbar_wait(c.full(s), (kc / RP_STAGES) & 1, a.status)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t sa = smem_u32(c.base + s * R_STAGE);
                    const uint64_t da = sdesc_sw128(sa, 16), db = sdesc_sw128(sa + 128 * BK * 2, OUT ? BOX : 16);
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)
                        umma_bf16_pair(tmem + b * RP_BN, sdesc_step(da, k * 32), sdesc_step(db, OUT ? k * 16 * 128 : k * 32),
                                       idesc, (kb == 0 && k == 0) ? 0u : 1u);
                    umma_commit_pair(c.empty(s, RP_STAGES), 0x3);
                }
                if (!ok) break;
                umma_commit_pair(c.tfull(b, RP_STAGES), 0x3);
            }
            if (!ok) drain_copies();
        }
        __syncwarp();
    } else {
        const int q = warp & 3;  // TMEM lane quarter of this warp
        const int col = (warp - 2) / 4 * (RP_BN / 2);
        int local = 0;
        for (int t = cluster; t < ntiles; t += nclusters, ++local) {
            const int b = local & 1;
            const int cz = t / (n_n * n_q), n0 = (t / n_q) % n_n * RP_BN + col;
            const int qw = t % n_q * 256 + (int)rank * 128 + q * 32;
            const bool ok = mbar_wait(c.tfull(b, RP_STAGES), (local >> 1) & 1, a.status);
            if (!__all_sync(0xffffffffu, ok)) break;
            tc_fence_after();
            const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16) + b * RP_BN + col;
            if constexpr (OUT)
                read_out_epilogue<RP_BN / 2, MODE>(a, lane_base, cz, qw, n0, lane);
            else
                read_hidden_epilogue<RP_BN / 2>(a, lane_base, cz, qw, n0, lane, c.base + LRP::STG + (warp - 2) * 2048);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_remote(map_to_cta(c.tempty(b, RP_STAGES), 0));
        }
    }
    tc_fence_before();
    cluster_sync();  // every MMA of the pair has completed and every TMEM read is done
    tc_fence_after();
    if (warp == 0) tmem_dealloc_pair(tmem, 512);
}

// ------------------------------------------------------------------ memory read, weights as the MMA rows
//
// For a query of Q <= 256 tokens the read runs with the operands the other way round: the
// weight tile is the tcgen05 A operand (M = 128 weight rows) and the queries are the B
// operand (N = NT = Q rounded up to 32), so neither an MMA row nor a staged query row is
// padding and each CTA takes in half the query bytes of the 128-query form.
//   hidden (HD = 0):  D[h][q] = W1[h] . z_q;  A_q[q][h] = SiLU(D[h][q] / |z_q|) (paper mode; the
//                     unnormalised z_q = SiLU(alpha x_q + gamma) comes from query_z_kernel, and
//                     the row scale commutes with the contraction), bf16 [C][Q][d_hid], stored
//                     through a per-warp 32 x 32 transpose so each row leaves as 64 contiguous bytes
//   out (HD = 64/128): D[o][q] = sum_h W2[h][o] A_q[q][h] (W2 MN-major); per head of HD
//                     features the RMS of each query's HD values is a reduction across the
//                     head's TMEM lanes (warp transpose-sums, then shared memory), then the
//                     gate, then the store into the caller's K / V (lanes = contiguous features)
// Warp 0 streams the weight tile and the query rows with TMA (2 to 8 stages), warp 1 issues
// the MMAs into one NT-column TMEM accumulator, warps 2..5 (one TMEM lane quarter each) run
// the epilogue.  Query rows >= Q arrive as TMA zero fill and are never stored.
// Both kernels are launched with programmatic stream serialisation: a CTA may start while the
// kernel before it (the query transform, or the hidden kernel) is still running, loads the
// weight tiles of its first stages, which that kernel does not write, and only then waits for
// that kernel's completion (griddepcontrol.wait) before it loads the query rows it produced.
constexpr int RT_THREADS = 6 * 32;
constexpr int RT_MAX_NT = 256;
constexpr int RT_A = 128 * BK * 2;  // 16 KB: the weight tile of one k-block
// Ring budget: 192 KB (one CTA per SM) when the grid fits in one wave; 96 KB (two CTAs per SM,
// one's epilogue overlapping the other's loads) when it takes several.
constexpr int RT_RING_1 = 192 * 1024, RT_RING_2 = 96 * 1024;
// A stage holds two k-blocks, each operand's in one TMA box (d_in and d_hid are multiples of 128), where
// three such stages fit the ring, else one.  A box costs the SM nearly the same at half the size, and
// with one CTA an SM the boxes set its pace: 64 queries of 16 chains of 2048 -> 1024 -> 1024 went from
// 41.3 to 38.8 us, of one chain from 36.2 to 30.8, of 4 chains of 3072 -> 2048 -> 2048 from 51.3 to 43.0 (200
// queries, where two of the larger stages fit: 66.3 to 67.7).
__host__ __device__ constexpr int rt_kblocks(int nt, int ring) { return ring / (2 * (RT_A + nt * BK * 2)) >= 3 ? 2 : 1; }
__host__ __device__ constexpr int rt_stage(int nt, int ring) { return rt_kblocks(nt, ring) * (RT_A + nt * BK * 2); }
__host__ __device__ constexpr int rt_stages(int nt, int ring = RT_RING_1) {
    return ring / rt_stage(nt, ring) < 8 ? ring / rt_stage(nt, ring) : 8;
}
// shared memory after the ring: barriers, TMEM slot and flag, then the epilogue's buffers:
// 4 warps x 2 KB transposes and the queries' 1/|z| (hidden), or 4 x NT column partial sums +
// 2 x NT scales (out)
__host__ __device__ constexpr int rt_bars(int nt, int ring = RT_RING_1) { return rt_stages(nt, ring) * rt_stage(nt, ring); }
__host__ __device__ constexpr int rt_epi(int nt, int ring = RT_RING_1) { return rt_bars(nt, ring) + 256; }
__host__ __device__ constexpr int rt_dyn(int nt, int ring = RT_RING_1) {
    return rt_epi(nt, ring) + (4 * 2048 + RT_MAX_NT * 4 > 6 * nt * 4 ? 4 * 2048 + RT_MAX_NT * 4 : 6 * nt * 4) + 1024;
}
static_assert(rt_dyn(RT_MAX_NT) <= 227 * 1024 && rt_dyn(32) <= 227 * 1024, "read shared memory budget");
static_assert(rt_dyn(RT_MAX_NT, RT_RING_2) <= 113 * 1024 && rt_dyn(32, RT_RING_2) <= 113 * 1024,
              "two read CTAs per SM");
static_assert(rt_stages(RT_MAX_NT, RT_RING_2) >= 2, "read pipeline depth");

template <int HD>
__global__ void __launch_bounds__(RT_THREADS, 2)
tc_read_t_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmQ, const ReadArgs a,
                 int NT, int ring) {
    constexpr bool OUT = HD != 0;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int NST = rt_stages(NT, ring), STAGE = rt_stage(NT, ring), KPS = rt_kblocks(NT, ring);
    const uint32_t bars = smem_u32(base + rt_bars(NT, ring));
    auto full = [&](int s) { return bars + 8 * s; };
    auto empty = [&](int s) { return bars + 8 * (8 + s); };
    const uint32_t tfull = bars + 8 * 16;
    uint32_t* slot = reinterpret_cast<uint32_t*>(base + rt_bars(NT, ring) + 8 * 17);
    int* flag = reinterpret_cast<int*>(base + rt_bars(NT, ring) + 8 * 17 + 8);
    uint8_t* epi = base + rt_epi(NT, ring);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < NST; ++s) {
            mbar_init(full(s), 1);
            mbar_init(empty(s), 1);
        }
        mbar_init(tfull, 1);
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(smem_u32(slot), RT_MAX_NT);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *slot;
    const int q0 = blockIdx.x * NT, n0 = blockIdx.y * 128, c = blockIdx.z;
    const int KB = (OUT ? a.d_hid : a.d_in) / BK;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // the out kernel may start

    if (warp == 0) {
        if (lane == 0) {
            tma_prefetch_map(&tmW);
            tma_prefetch_map(&tmQ);
            // stage i: k-blocks KPS i ..; W1 as [k-block][128 rows], W2 (MN-major) as [64 outputs][KPS 64 hidden rows]
            auto load_w = [&](int i, uint32_t sa, uint32_t fb) {
                if (OUT)
                    tma_load_4d(sa, &tmW, fb, 0, i * KPS * BK, n0 / 64, a.b_chain0 + c);
                else
                    tma_load_4d(sa, &tmW, fb, 0, n0, i * KPS, a.b_chain0 + c);
            };
            // the first stages' weight tiles, then the wait for the kernel that writes the queries
            const int n = KB / KPS, pre = n < NST ? n : NST;
            for (int i = 0; i < pre; ++i) {
                mbar_expect_tx(full(i), STAGE);
                load_w(i, smem_u32(base + i * STAGE), full(i));
            }
            asm volatile("griddepcontrol.wait;" ::: "memory");
            for (int i = 0; i < n; ++i) {
                const int s = i % NST;
                const uint32_t sa = smem_u32(base + s * STAGE), fb = full(s);
                if (i >= pre) {
                    if (!mbar_wait(empty(s), ((i / NST) - 1) & 1, a.status)) break;
                    mbar_expect_tx(fb, STAGE);
                    load_w(i, sa, fb);
                }
                tma_load_4d(sa + KPS * RT_A, &tmQ, fb, 0, a.a_row0 + q0, i * KPS, a.a_chain0 + c);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = idesc_bf16_f32(128, NT, OUT, false);
            bool ok = true;
            for (int i = 0; i < KB / KPS; ++i) {
                const int s = i % NST;
                if (!mbar_wait(full(s), (i / NST) & 1, a.status)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t sa = smem_u32(base + s * STAGE);
                const uint64_t da0 = sdesc_sw128(sa, OUT ? KPS * BOX : 16), db0 = sdesc_sw128(sa + KPS * RT_A, 16);
                for (int kb = 0; kb < KPS; ++kb) {
                    // the k-block's weights: 64 further rows of both output blocks (W2), or the next tile (W1)
                    const uint64_t da = sdesc_step(da0, kb * (OUT ? BOX : RT_A)), db = sdesc_step(db0, kb * NT * BK * 2);
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)
                        umma_bf16(tmem, sdesc_step(da, OUT ? k * 16 * 128 : k * 32), sdesc_step(db, k * 32), idesc,
                                  (i | kb | k) ? 1u : 0u);
                }
                umma_commit(empty(s));
            }
            if (ok) umma_commit(tfull);
        }
        __syncwarp();
    } else {
        const int q = warp & 3;  // TMEM lane quarter: weight rows n0 + 32 q .. + 31
        const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16);
        float* zs = reinterpret_cast<float*>(epi + 4 * 2048);  // hidden: 1/|z| of the tile's queries
        if constexpr (!OUT) {
            asm volatile("griddepcontrol.wait;" ::: "memory");  // zinv comes from the kernel before
            for (int j = threadIdx.x - 64; j < NT; j += 128)
                zs[j] = (a.qzinv && q0 + j < a.Q) ? a.qzinv[(size_t)c * a.Q + q0 + j] : 1.f;
        }
        if (threadIdx.x == 64) *flag = mbar_wait(tfull, 0, a.status) ? 1 : 0;
        __syncwarp();
        named_bar_sync(R_EPI_BAR, 128);
        if (*flag) {
            tc_fence_after();
            const int nch = NT / 32;
            if constexpr (!OUT) {
                // the tile's columns of A_q lie inside [Q][d_hid] (index check of MONE_DEBUG builds)
                const bool wr = MONE_DCHECK(n0 + 128 <= a.d_hid, a.status, DS_READ_TILE);
                uint16_t* stg = reinterpret_cast<uint16_t*>(epi + (warp - 2) * 2048);  // [32 queries][32 rows]
                const int h = n0 + q * 32;
#pragma unroll 1
                for (int cc = 0; cc < nch; ++cc) {
                    float v[32];
                    tmem_ld32(lane_base + cc * 32, v);
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const float x = v[j] * zs[cc * 32 + j];
                        const bf16 b = __float2bfloat16_rn(x * sigmoidf_(x));
                        stg[j * 32 + lane] = *reinterpret_cast<const uint16_t*>(&b);
                    }
                    __syncwarp();
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int r = 8 * k + (lane >> 2), i = lane & 3;
                        const int qi = q0 + cc * 32 + r;
                        const uint4 val = *reinterpret_cast<const uint4*>(stg + r * 32 + i * 8);
                        if (qi < a.Q && wr)
                            *reinterpret_cast<uint4*>(a.Aq + ((size_t)c * a.Q + qi) * a.d_hid + h + i * 8) = val;
                    }
                    __syncwarp();
                }
            } else {
                // per-column sums of squares of this warp's 32 features, then the head's total
                float* part = reinterpret_cast<float*>(epi);  // [4 warps][NT]
                float* scl = part + 4 * NT;                   // [2 heads of the tile][NT]
                constexpr int HPT = 128 / HD;                 // heads per 128-feature tile
                constexpr int WPH = HD / 32;                  // warps per head
#pragma unroll 1
                for (int cc = 0; cc < nch; ++cc) {
                    float v[32];
                    tmem_ld32(lane_base + cc * 32, v);
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] *= v[j];
                    // transpose-reduce: afterwards lane j holds the sum over the warp's lanes of column j
#pragma unroll
                    for (int sft = 16; sft >= 1; sft >>= 1) {
                        const bool upper = (lane & sft) != 0;
#pragma unroll
                        for (int u = 0; u < sft; ++u) {
                            const float send = upper ? v[u] : v[u + sft];
                            const float keep = upper ? v[u + sft] : v[u];
                            v[u] = keep + __shfl_xor_sync(0xffffffffu, send, sft);
                        }
                    }
                    part[q * NT + cc * 32 + lane] = v[0];
                }
                named_bar_sync(R_EPI_BAR, 128);
                const int nh = 2 * a.n_kv;
                for (int i = threadIdx.x - 64; i < HPT * NT; i += 128) {
                    const int hl = i / NT, j = i - hl * NT;
                    float ss = 0.f;
#pragma unroll
                    for (int w = 0; w < WPH; ++w) ss += part[(hl * WPH + w) * NT + j];
                    const int head = n0 / HD + hl;
                    const float g = a.gate && head < nh ? a.gate[(size_t)c * nh + head] : 1.f;
                    scl[hl * NT + j] = g / sqrtf(ss / (float)HD + a.eps);
                }
                named_bar_sync(R_EPI_BAR, 128);
                const int o = n0 + q * 32 + lane;  // this thread's output feature
                const int hl = (q * 32) / HD, head = n0 / HD + hl, d = o - head * HD;
                const bool wr = MONE_DCHECK(head < nh, a.status, DS_READ_TILE);
                const int kvh = head < a.n_kv ? head : head - a.n_kv;
                bf16* outp = (head < a.n_kv ? a.Kout : a.Vout) + (long long)(c / a.L) * a.s0 +
                             (long long)(c % a.L) * a.s1 + (long long)kvh * a.s2 + d;
#pragma unroll 1
                for (int cc = 0; cc < nch; ++cc) {
                    float v[32];
                    tmem_ld32(lane_base + cc * 32, v);
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const int qi = q0 + cc * 32 + j;
                        if (qi < a.Q && wr)
                            outp[(long long)qi * a.s3] = __float2bfloat16_rn(v[j] * scl[hl * NT + cc * 32 + j]);
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, RT_MAX_NT);
}

// Launch a read-structured kernel with the stage count that suits its grid (see LRT).
template <int MODE>
cudaError_t launch_read_kernel(const TcDevice& dev, dim3 grid, const CUtensorMap& A, const CUtensorMap& B, const ReadArgs& a,
                               cudaStream_t st) {
    if ((long long)grid.x * grid.y * grid.z <= dev.sms)
        tc_read_kernel<MODE, 6><<<grid, R_THREADS, LR6::DYN, st>>>(A, B, a);
    else
        tc_read_kernel<MODE, 3><<<grid, R_THREADS, LR::DYN, st>>>(A, B, a);
    return cudaGetLastError();
}

// A read kernel over `grid` tiles of 128 x 128: on CTA pairs when the tiles are more than one wave of two CTAs
// an SM.  Chains of 2048 -> 1024 -> 1024 (whole reads, CTA pairs and one-CTA tiles): 64 tiles 42.5 and 36.9 us,
// 288 tiles 53.2 and 53.5, 352 tiles 71.6 and 85.2; 288 tiles of 512 -> 256 -> 256 45.7 and 43.1.
template <int MODE>
cudaError_t launch_read_many(const TcDevice& dev, dim3 grid, const CUtensorMap& A, const CUtensorMap& B, const ReadArgs& a,
                             cudaStream_t st) {
    if ((long long)grid.x * grid.y * grid.z <= 2 * dev.sms) return launch_read_kernel<MODE>(dev, grid, A, B, a, st);
    const long long tiles = (long long)((grid.x + 1) / 2) * (grid.y / 2) * grid.z;
    return launch_kernel(tc_read_pair_kernel<MODE>, dim3(2 * (unsigned)std::min<long long>(tiles, dev.sms / 2)), dim3(RP_THREADS),
                         LRP::DYN, st, false, 2, A, B, a);
}

// Whether phase A runs on CTA pairs (256-token x 256-hidden tiles) for this handle's shape.
bool phase_a_pairs(const DevState& s, const TcDevice& dev) {
    return (s.T / A_BM) % 2 == 0 && s.d_hid % P_BN == 0 && dev.pair_clusters > 0;
}

}  // namespace

cudaError_t tc_device(const TcDevice** out) {
    static PerDevice<TcDevice> devices;
    return devices.get(out, [](TcDevice& d) {
        cudaError_t e = sm_count(&d.sms);
        auto opt_in = [&](auto kernel, int dyn) {
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);
        };
        opt_in(tc_phase_a_kernel, LA::DYN);
        opt_in(tc_phase_a_pair_kernel, LP::DYN);
        opt_in(tc_phase_a_split_kernel<4>, LSplit<4>::DYN);
        opt_in(tc_phase_a_split_kernel<2>, LSplit<2>::DYN);
        opt_in(tc_phase_b_kernel<false, false>, LayoutB::DYN);
        opt_in(tc_phase_b_kernel<false, true>, LayoutB::DYN);
        opt_in(tc_phase_b_kernel<true, false>, LayoutB2::DYN);
        opt_in(tc_phase_b_kernel<true, true>, LayoutB2::DYN);
        for (auto fn : {tc_read_kernel<0, 3>, tc_read_kernel<64, 3>, tc_read_kernel<128, 3>, tc_read_kernel<MSE_HIDDEN, 3>,
                        tc_read_kernel<MSE_OUT, 3>})
            opt_in(fn, LR::DYN);
        for (auto fn : {tc_read_kernel<0, 6>, tc_read_kernel<64, 6>, tc_read_kernel<128, 6>, tc_read_kernel<MSE_HIDDEN, 6>,
                        tc_read_kernel<MSE_OUT, 6>})
            opt_in(fn, LR6::DYN);
        for (auto fn : {tc_read_pair_kernel<READ_HIDDEN>, tc_read_pair_kernel<64>, tc_read_pair_kernel<128>}) opt_in(fn, LRP::DYN);
        for (auto fn : {tc_read_t_kernel<0>, tc_read_t_kernel<64>, tc_read_t_kernel<128>}) opt_in(fn, rt_dyn(RT_MAX_NT));
        if (e != cudaSuccess) return e;
        // the forms on clusters are left out where they cannot run
        auto clusters = [&](auto kernel, int size, int threads, int dyn, int& n) {
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = size;
            at[0].val.clusterDim.y = 1;
            at[0].val.clusterDim.z = 1;
            cfg.gridDim = dim3(size * (d.sms / size));
            cfg.blockDim = dim3(threads);
            cfg.dynamicSmemBytes = dyn;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
                cudaGetLastError();
                n = 0;
            }
        };
        clusters(tc_phase_a_pair_kernel, 2, THREADS, LP::DYN, d.pair_clusters);
        clusters(tc_phase_b_kernel<true, false>, 2, B_THREADS, LayoutB2::DYN, d.pairb_clusters);
        clusters(tc_phase_a_split_kernel<4>, 4, THREADS, LSplit<4>::DYN, d.split4);
        clusters(tc_phase_a_split_kernel<2>, 2, THREADS, LSplit<2>::DYN, d.split2);
        return cudaSuccess;
    });
}

cudaError_t launch_phase_a_tc(const DevState& s, const TcMaps& m, const TcInputMaps& in, const SegWork& w,
                              cudaStream_t st) {
    const TcDevice& dev = *s.tc;
    TcArgs a = make_args(s, w);
    if (s.fault_stall > 0) {  // test knob: this launch's waits run out after 1 ms with nothing in flight
        --s.fault_stall;
        a.stall = 1;
        a.wait_ns = 1000000ull;
    }
    const CUtensorMap& U = s.mode == 1 ? m.Ua : in.Xa;
    const bool pdl = w.single && !w.first;
    // few tiles of a call on one stream (its other kernels leave the SMs to this one): clusters of 4 or 2 a tile
    const int tiles = w.nc * (s.T / A_BM) * (s.d_hid / A_BN);
    if (w.single && s.loss == 0) {
        if (tiles <= dev.split4 && s.d_in >= 4 * BK && s.d_out >= 4 * BK)
            return launch_kernel(tc_phase_a_split_kernel<4>, dim3(4 * tiles), dim3(THREADS), LSplit<4>::DYN, st, pdl, 4, U,
                                 in.Ka, in.Va, m.W1b, m.W2b, a);
        if (tiles <= dev.split2)
            return launch_kernel(tc_phase_a_split_kernel<2>, dim3(2 * tiles), dim3(THREADS), LSplit<2>::DYN, st, pdl, 2, U,
                                 in.Ka, in.Va, m.W1b, m.W2b, a);
    }
    if (phase_a_pairs(s, dev)) {
        // squared-error segments: the pre-pass wrote At and c SiLU'(x) / |z|, only R is left
        a.r_only = (s.loss == 1) ? 1 : 0;  // 1: MONE_LOSS_MSE
        // CTA pairs over 256-token x 256-hidden tiles
        const int npairs = w.nc * (s.T / (2 * A_BM)) * (s.d_hid / P_BN);
        const int maxc = dev.pair_clusters - (s.reserve_sms + 1) / 2;  // leave reserved SMs free
        const int clusters = npairs < maxc ? npairs : maxc;
        return launch_kernel(tc_phase_a_pair_kernel, dim3(2 * clusters), dim3(THREADS), LP::DYN, st, pdl && !a.r_only, 2, U,
                             in.Ka, in.Va, m.W1b, m.W2b, a);
    }
    const int sms = dev.sms - s.reserve_sms;
    const int grid = tiles < sms ? tiles : sms;
    return launch_kernel(tc_phase_a_kernel, dim3(grid), dim3(THREADS), LA::DYN, st, pdl && s.loss == 0, 1, U, in.Ka, in.Va,
                         m.W1b, m.W2b, a);
}

cudaError_t launch_phase_b_tc(const DevState& s, const TcMaps& m, const TcInputMaps& in, const SegWork& w,
                              cudaStream_t st) {
    const TcDevice& dev = *s.tc;
    TcArgs a = make_args(s, w);
    // CTA pairs over 256-hidden x 256-column tiles (a tile's columns all live) from T = 1024 on:
    // there a tile's operand stream (768 KB a CTA) rivals its state stream, and the pair takes a
    // third off it.  At T = 512 the pair's coupled loads and accumulator release cost more than they save.
    constexpr int PAIR_MIN_T = 1024;
    const bool pairs = s.T >= PAIR_MIN_T && s.d_in % B_BN == 0 && dev.pairb_clusters > 0;
    // When the state ring's slots are handed back, that is how many of its loads are in flight. A launch of few tiles a CTA
    // is mostly ramp, and without momentum a slot carries half the bytes: hand back at once. The longer a launch runs
    // (tiles a CTA) and the more operands stream beside the state (T), the fewer state loads in flight serve it best: they
    // queue before the operands' and the stores. Measured over 70 contexts of 8 to 224 chains, the steps where the
    // faster of two neighbours changes; whole contexts, ms, with S_PAIRS1, S_LAG3, S_PAIRS3, S_QUADS2: 8 chains of 2048 -> 1024 ->
    // 1024, T = 128 (T * tiles 323): 1.75 1.79 1.86 1.92; 28 of 2432 -> 1280 -> 768, T = 128 (1533): 6.99 6.77 7.02 7.35; 64 of
    // 2048 -> 1024 -> 1024, T = 512 (10,348): 5.15 5.16 4.78 4.93; 20 of 3072 -> 2048 -> 2048, T = 768 (16,168): 4.56 4.54 4.54 4.42.
    const auto store_mode = [&](int tiles, int ctas) {
        const double per_cta = (double)tiles / ctas, run = per_cta * s.T;
        if (!s.momentum || per_cta <= 4) return S_PAIRS1;
        return run < 4400 ? S_LAG3 : run < 16000 ? S_PAIRS3 : S_QUADS2;
    };
    const CUtensorMap& U = s.mode == 1 ? m.Ub : in.Xb;
    const CUtensorMap& U2 = s.mode == 1 ? m.Ub2 : in.Xb2;
    const int col_tiles = b_col_tiles(s.d_in, s.d_out);
    if (pairs) {
        const int npairs = w.nc * col_tiles * (s.d_hid / (2 * B_BM));
        const int maxc = dev.pairb_clusters - (s.reserve_sms + 1) / 2;
        const int clusters = npairs < maxc ? npairs : maxc;
        // on pairs the operand streams are smaller; by twos one store later was within 1% of the best nearly everywhere
        a.store_mode = S_PAIRS1;
        return launch_kernel(a.step_sq ? tc_phase_b_kernel<true, true> : tc_phase_b_kernel<true, false>, dim3(2 * clusters),
                             dim3(B_THREADS), LayoutB2::DYN, st, w.single != 0, 2, U2, in.Kb, in.Vb, m.dH, m.At, m.W1s,
                             m.W2s, a);
    }
    const int ntiles = w.nc * col_tiles * (s.d_hid / B_BM);
    const int sms = dev.sms - s.reserve_sms;
    const int grid = ntiles < sms ? ntiles : sms;
    a.store_mode = store_mode(ntiles, grid);
    return launch_kernel(a.step_sq ? tc_phase_b_kernel<false, true> : tc_phase_b_kernel<false, false>, dim3(grid),
                         dim3(B_THREADS), LayoutB::DYN, st, w.single != 0, 1, U, in.Kb, in.Vb, m.dH, m.At, m.W1s, m.W2s, a);
}

cudaError_t launch_mse_tc(const DevState& s, const TcMaps& m, const TcInputMaps& in, const SegWork& w,
                          cudaStream_t st) {
    const TcDevice& dev = *s.tc;
    const bool paper = s.mode == 1;
    ReadArgs a{};
    a.d_in = s.d_in; a.d_hid = s.d_hid; a.d_out = s.d_out; a.n_kv = s.n_kv;
    a.status = s.status;
    a.C = s.C; a.T = s.T; a.Tp = w.Tp; a.win = s.win_rows; a.parity = w.parity; a.renorm_pending = w.renorm_pending;
    a.tok0 = w.u_off; a.row0 = w.row0; a.n_rows = w.n_rows; a.y_cstride = w.y_cstride;
    a.zinv = paper ? s.zinv : nullptr;
    a.n1 = s.n1; a.n2 = s.n2; a.sumsq = s.sumsq;
    a.K = static_cast<const bf16*>(w.K); a.V = static_cast<const bf16*>(w.V);
    a.Kres = s.Kres; a.Vres = s.Vres;
    a.loss = w.loss;
    a.Aq = s.Amse;
    if (phase_a_pairs(s, dev)) {  // phase A runs in its R-only form: write At and c SiLU'(x) / |z| here
        a.At = reinterpret_cast<bf16*>(s.Att);
        a.Sp = reinterpret_cast<bf16*>(s.dHt);
        a.paper = paper ? 1 : 0;
        a.lr = s.lr;
        a.eta = s.eta;
        a.eta_in = w.eta_in ? w.eta_in + w.row0 : nullptr;
        a.eta_cstride = w.eta_cstride;
    }
    // hidden: U rows of the segment (paper: the transformed window, absolute chain; plain: the
    // caller's X of the group), W1 of chain c0 + z
    a.a_row0 = paper ? (int)w.u_off : (int)w.row0;
    a.a_chain0 = paper ? w.c0 : 0;
    a.b_chain0 = w.c0;
    cudaError_t e = launch_read_kernel<MSE_HIDDEN>(dev, dim3(s.T / 128, s.d_hid / 128, w.nc), paper ? m.Ua : in.Xa, m.W1b, a, st);
    if (e != cudaSuccess) return e;
    // out: the activations of the same chains (absolute), W2 MN-major
    a.a_row0 = 0;
    a.a_chain0 = w.c0;
    return launch_read_kernel<MSE_OUT>(dev, dim3(s.T / 128, s.d_out / 128, w.nc), m.Amse, m.W2m, a, st);
}

cudaError_t launch_read_tc(const DevState& s, const TcMaps& m, const void* Xq, void* Uq, void* Aq, float* zq, int Q,
                           int n_layers, void* K_out, void* V_out, const long long* strides, cudaStream_t st) {
    const TcDevice& dev = *s.tc;
    if (s.hd != 64 && s.hd != 128) return cudaErrorInvalidValue;
    // the query side: unnormalised z and 1/|z|, which the hidden kernel applies
    cudaError_t e = launch_query_z(s, Xq, Q, Uq, zq, st);
    if (e != cudaSuccess) return e;
    ReadArgs a{};
    a.Q = Q; a.d_in = s.d_in; a.d_hid = s.d_hid; a.d_out = s.d_out; a.n_kv = s.n_kv; a.L = n_layers;
    a.eps = s.rms_eps;
    a.gate = s.gate;
    a.Aq = static_cast<bf16*>(Aq);
    a.Kout = static_cast<bf16*>(K_out);
    a.Vout = static_cast<bf16*>(V_out);
    a.s0 = strides[0]; a.s1 = strides[1]; a.s2 = strides[2]; a.s3 = strides[3];
    a.status = s.status;
    a.qzinv = s.mode == 1 ? zq : nullptr;
    if (Q <= RT_MAX_NT) {  // weights as the 128-row operand, the queries as N
        const int NT = (Q + 31) / 32 * 32;
        // one CTA per SM with the deep ring when a kernel's tiles fit in one wave, else two
        const int ring1 = (long long)(s.d_hid / 128) * s.C <= dev.sms ? RT_RING_1 : RT_RING_2;
        const int ring2 = (long long)(s.d_out / 128) * s.C <= dev.sms ? RT_RING_1 : RT_RING_2;
        const int k1 = rt_kblocks(NT, ring1), k2 = rt_kblocks(NT, ring2);
        CUtensorMap tu, ta;
        if (!encode_map_bf16_blocks(&tu, Uq, s.d_in, Q, s.C, NT, k1) || !encode_map_bf16_blocks(&ta, Aq, s.d_hid, Q, s.C, NT, k2))
            return cudaErrorInvalidValue;
        // programmatic stream serialisation: each kernel may start before the one it follows ends
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.blockDim = dim3(RT_THREADS);
        cfg.stream = st;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        cfg.gridDim = dim3(1, s.d_hid / 128, s.C);
        cfg.dynamicSmemBytes = rt_dyn(NT, ring1);
        if ((e = cudaLaunchKernelEx(&cfg, tc_read_t_kernel<0>, m.W1r[k1 - 1], tu, a, NT, ring1)) != cudaSuccess) return e;
        cfg.gridDim = dim3(1, s.d_out / 128, s.C);
        cfg.dynamicSmemBytes = rt_dyn(NT, ring2);
        if (s.hd == 64) return cudaLaunchKernelEx(&cfg, tc_read_t_kernel<64>, m.W2r[k2 - 1], ta, a, NT, ring2);
        return cudaLaunchKernelEx(&cfg, tc_read_t_kernel<128>, m.W2r[k2 - 1], ta, a, NT, ring2);
    }
    a.C = s.C;
    CUtensorMap mu, ma;
    if (!encode_map_bf16_3d(&mu, Uq, s.d_in, Q, s.C, 64, 128) || !encode_map_bf16_3d(&ma, Aq, s.d_hid, Q, s.C, 64, 128))
        return cudaErrorInvalidValue;
    const int nq = (Q + 127) / 128;
    if ((e = launch_read_many<READ_HIDDEN>(dev, dim3(nq, s.d_hid / 128, s.C), mu, m.W1b, a, st)) != cudaSuccess) return e;
    if (s.hd == 64) return launch_read_many<64>(dev, dim3(nq, s.d_out / 128, s.C), ma, m.W2m, a, st);
    return launch_read_many<128>(dev, dim3(nq, s.d_out / 128, s.C), ma, m.W2m, a, st);
}

// ------------------------------------------------------------------ tensor maps

namespace {
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
typedef CUresult (*ReplaceAddressFn)(CUtensorMap*, void*);
EncodeTiledFn g_encode = nullptr;
ReplaceAddressFn g_replace = nullptr;
std::once_flag g_encode_once;

void* driver_entry(const char* name) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    return cudaGetDriverEntryPointByVersion(name, &fn, 12000, cudaEnableDefault, &q) == cudaSuccess &&
                   q == cudaDriverEntryPointSuccess
               ? fn
               : nullptr;
}

EncodeTiledFn encoder() {
    std::call_once(g_encode_once, [] {
        g_encode = reinterpret_cast<EncodeTiledFn>(driver_entry("cuTensorMapEncodeTiled"));
        g_replace = reinterpret_cast<ReplaceAddressFn>(driver_entry("cuTensorMapReplaceAddress"));
    });
    return g_encode;
}
}  // namespace

bool encode_map_bf16_3d(CUtensorMap* map, const void* base, uint64_t inner, uint64_t rows, uint64_t chains,
                        uint32_t box_inner, uint32_t box_rows) {
    if (!encoder() || !map) return false;
    const cuuint64_t dims[3] = {inner, rows, chains};
    const cuuint64_t strides[2] = {inner * 2, inner * rows * 2};
    const cuuint32_t box[3] = {box_inner, box_rows, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    return g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool encode_map_bf16_blocks(CUtensorMap* map, const void* base, uint64_t inner, uint64_t rows, uint64_t chains,
                            uint32_t box_rows, uint32_t box_blocks) {
    const uint64_t dims[4] = {64, rows, inner / 64, chains}, strides[3] = {inner * 2, 128, inner * rows * 2};
    const uint32_t box[4] = {64, box_rows, box_blocks, 1};
    return encode_map_bf16_4d(map, base, dims, strides, box);
}

bool encode_map_state(CUtensorMap* map, const float* W, const float* mu, uint64_t inner, uint64_t rows,
                      uint64_t chains) {
    if (!encoder() || !map || (mu && mu <= W)) return false;
    const cuuint64_t dims[5] = {32, rows, inner / 32, chains, mu ? 2u : 1u};
    const cuuint64_t strides[4] = {inner * 4, 128, inner * rows * 4,
                                   mu ? (cuuint64_t)(mu - W) * 4 : (cuuint64_t)(inner * rows * chains * 4)};
    const cuuint32_t box[5] = {32, 32, 2, 1, mu ? 2u : 1u};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return g_encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, const_cast<float*>(W), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool encode_map_bf16_4d(CUtensorMap* map, const void* base, const uint64_t dims[4], const uint64_t strides[3],
                        const uint32_t box[4]) {
    if (!encoder() || !map) return false;
    const cuuint64_t d[4] = {dims[0], dims[1], dims[2], dims[3]};
    const cuuint64_t st[3] = {strides[0], strides[1], strides[2]};
    const cuuint32_t b[4] = {box[0], box[1], box[2], box[3]};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), d, st, b, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool encode_map_bf16_5d(CUtensorMap* map, const void* base, const uint64_t dims[5], const uint64_t strides[4],
                        const uint32_t box[5]) {
    if (!encoder() || !map) return false;
    const cuuint64_t d[5] = {dims[0], dims[1], dims[2], dims[3], dims[4]};
    const cuuint64_t st[4] = {strides[0], strides[1], strides[2], strides[3]};
    const cuuint32_t b[5] = {box[0], box[1], box[2], box[3], box[4]};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base), d, st, b, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool retarget_map(CUtensorMap* map, const void* base) {
    return encoder() && g_replace && g_replace(map, const_cast<void*>(base)) == CUDA_SUCCESS;
}

bool encode_map_plain_3d(CUtensorMap* map, const void* base, bool f32, uint64_t inner, uint64_t rows,
                         uint64_t chains, uint32_t box_inner, uint32_t box_rows) {
    if (!encoder() || !map) return false;
    const uint64_t es = f32 ? 4 : 2;
    const cuuint64_t dims[3] = {inner, rows, chains};
    const cuuint64_t strides[2] = {inner * es, inner * rows * es};
    const cuuint32_t box[3] = {box_inner, box_rows, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    return g_encode(map, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
                    const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace mone
