// Consumer attention of the read (Eq. 5, with Eq. 2 per head): the query tokens attend
// over [memory tokens || their own keys], softmax(q k^T / sqrt(hd)) v, with the memory
// tokens visible to every query token and the query tokens causal among themselves;
// query head h reads key/value head h / (n_q / n_kv) (grouped heads).
//
// Three forms.  bf16 with 16-byte-aligned rows runs on the tensor cores: many query rows in
// attention_prefill_kernel (S = Q K^T and O = P V as tcgen05 MMAs with TMEM accumulators, the
// softmax one row per thread in between), few in attention_decode_kernel (the keys split over
// warps and a cluster of CTAs).  fp32, and bf16 caches with other strides, run
// on the CUDA cores in flash-decode form: a CTA takes one (chain, key/value head, tile of
// query tokens) and stages the cache rows its tokens can see through shared memory in
// chunks of KC = 64 positions (converted to fp32 once, shared by every query head of the
// group).  Each warp owns up to MAXI (query head, token) items: per chunk, lane l scores
// keys l and l + 32 against every item (queries in shared memory), the chunk's max and sum
// are reduced once per item, and the probabilities pass through shared memory into the
// value accumulation, where a lane owns hd / 32 dimensions.
#include <algorithm>
#include <cfloat>
#include <mutex>

#include "mone_common.cuh"
#include "per_device.h"

namespace mone {

namespace {

constexpr int ATT_WARPS = 8;
constexpr int ATT_ITEMS = 64;                 // (query head, token) items per CTA
constexpr int MAXI = ATT_ITEMS / ATT_WARPS;   // items per warp
constexpr int KC = 64;                        // cache positions per shared-memory chunk

struct AttnArgs {
    const void* Q;          // [C][n_q][Lq][hd]
    const void *K, *V;      // caches, element strides s0 (context), s1 (layer), s2 (head), s3 (position)
    void* out;              // [C][n_q][Lq][hd]
    long long s0, s1, s2, s3;
    int L, n_q, n_kv, group, Lq, n_mem, rows;  // rows: query tokens per CTA (group * rows <= ATT_ITEMS)
    float scale;            // 1 / sqrt(hd)
    int tile_tok, per_block;  // decode form: tokens of a block, 16-row tiles that cut it
    int group_inv;            // decode form: 65536 / group + 1
    int vec;                // caches 16-byte aligned (base and every stride): stage with 16-byte loads
    int* status;            // device status word (bounded waits of the prefill form)
};

// Stage cache positions [j0, j0 + nk) of one head into shared memory as fp32 rows of HD
// values, `pitch` floats apart.
template <typename T, int HD>
__device__ __forceinline__ void stage_rows(float* dst, const T* src, long long s3, int j0, int nk, bool vec,
                                           int pitch) {
    if (vec) {
        constexpr int PER = 16 / sizeof(T);   // elements per 16-byte load
        constexpr int VPR = HD / PER;         // loads per row
        const int nv = nk * VPR;
#pragma unroll 4
        for (int e = threadIdx.x; e < nv; e += ATT_WARPS * 32) {
            const int j = e / VPR, v = e % VPR;
            const uint4 r = *reinterpret_cast<const uint4*>(src + (long long)(j0 + j) * s3 + v * PER);
            float f[PER];
            if constexpr (sizeof(T) == 2) {
                const __nv_bfloat162* b = reinterpret_cast<const __nv_bfloat162*>(&r);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float2 x = __bfloat1622float2(b[u]);
                    f[2 * u] = x.x;
                    f[2 * u + 1] = x.y;
                }
            } else {
                f[0] = __uint_as_float(r.x); f[1] = __uint_as_float(r.y);
                f[2] = __uint_as_float(r.z); f[3] = __uint_as_float(r.w);
            }
#pragma unroll
            for (int u = 0; u < PER; ++u) dst[j * pitch + v * PER + u] = f[u];
        }
    } else {
        for (int e = threadIdx.x; e < nk * HD; e += ATT_WARPS * 32) {
            const int j = e / HD, d = e % HD;
            dst[j * pitch + d] = to_f<T>(src[(long long)(j0 + j) * s3 + d]);
        }
    }
}

template <typename T, int HD>
struct AttnSmem {
    // key rows padded by 4 floats: a lane reads its key row 16 bytes at a time, and the 8 lanes of a
    // quarter warp (one shared-memory wavefront of 128-bit loads) start 68 / 132 floats apart: 8 bank groups
    static constexpr int KP = HD + 4;
    static constexpr int K_OFF = 0;                          // [KC][KP] keys (fp32)
    static constexpr int V_OFF = K_OFF + KC * KP;            // [KC][HD] values
    static constexpr int Q_OFF = V_OFF + KC * HD;            // [warp][MAXI][HD] scaled queries
    static constexpr int P_OFF = Q_OFF + ATT_WARPS * MAXI * HD;  // [warp][MAXI][KC] probabilities of a chunk
    static constexpr int FLOATS = P_OFF + ATT_WARPS * MAXI * KC;
};

template <typename T, int HD>
__global__ void __launch_bounds__(ATT_WARPS * 32, 2) attention_kernel(const AttnArgs a) {
    using SM = AttnSmem<T, HD>;
    constexpr int D = HD / 32;  // value / accumulator dimensions per lane
    extern __shared__ float sh[];
    float* Ks = sh + SM::K_OFF;
    float* Vs = sh + SM::V_OFF;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* Qs = sh + SM::Q_OFF + warp * MAXI * HD;
    float* Ps = sh + SM::P_OFF + warp * MAXI * KC;
    const int c = blockIdx.z, g = blockIdx.y, r0 = blockIdx.x * a.rows;
    const long long kv_off = (long long)(c / a.L) * a.s0 + (long long)(c % a.L) * a.s1 + (long long)g * a.s2;
    const T* Kc = static_cast<const T*>(a.K) + kv_off;
    const T* Vc = static_cast<const T*>(a.V) + kv_off;

    // this warp's items: item = warp + ATT_WARPS * k -> (head in group, token row); the running
    // softmax (max, sum) is kept identical in every lane, the accumulator split over lanes by dimension
    float acc[MAXI][D], mx[MAXI], sum[MAXI];
    int vis[MAXI];  // keys item k sees (0: no item)
#pragma unroll
    for (int k = 0; k < MAXI; ++k) {
        const int it = warp + ATT_WARPS * k;
        const int hg = it / a.rows, i = r0 + it % a.rows;
        vis[k] = 0;
        mx[k] = -INFINITY;
        sum[k] = 0.f;
#pragma unroll
        for (int d = 0; d < D; ++d) acc[k][d] = 0.f;
        float qv[D];
#pragma unroll
        for (int d = 0; d < D; ++d) qv[d] = 0.f;
        if (hg < a.group && i < a.Lq) {
            vis[k] = a.n_mem + i + 1;
            const int h = g * a.group + hg;
            const T* qr = static_cast<const T*>(a.Q) + (((size_t)c * a.n_q + h) * a.Lq + i) * HD;
#pragma unroll
            for (int d = 0; d < D; ++d) qv[d] = to_f<T>(qr[lane + 32 * d]) * a.scale;
        }
#pragma unroll
        for (int d = 0; d < D; ++d) Qs[k * HD + lane + 32 * d] = qv[d];
    }
    const int last = min(a.Lq, r0 + a.rows) - 1;
    const int keys = a.n_mem + last + 1;  // positions the tile's last token sees
    for (int j0 = 0; j0 < keys; j0 += KC) {
        const int nk = min(KC, keys - j0);
        __syncthreads();
        stage_rows<T, HD>(Ks, Kc, a.s3, j0, nk, a.vec, SM::KP);
        stage_rows<T, HD>(Vs, Vc, a.s3, j0, nk, a.vec, HD);
        // value rows up to the next multiple of 4 are read with probability 0: make them finite
        for (int e = threadIdx.x; e < (((nk + 3) & ~3) - nk) * HD; e += ATT_WARPS * 32) Vs[nk * HD + e] = 0.f;
        __syncthreads();
        // scores: lane owns keys j0 + lane and j0 + lane + 32 of the chunk; keys and the (broadcast)
        // queries are read 4 dimensions at a time
        float z0[MAXI], z1[MAXI];
#pragma unroll
        for (int k = 0; k < MAXI; ++k) z0[k] = z1[k] = 0.f;
        const float4* k0 = reinterpret_cast<const float4*>(Ks + lane * SM::KP);
        const float4* k1 = reinterpret_cast<const float4*>(Ks + (lane + 32) * SM::KP);
        const float4* q4 = reinterpret_cast<const float4*>(Qs);
#pragma unroll 2
        for (int d4 = 0; d4 < HD / 4; ++d4) {
            const float4 a0 = k0[d4], a1 = k1[d4];
#pragma unroll
            for (int k = 0; k < MAXI; ++k) {
                const float4 qd = q4[k * (HD / 4) + d4];
                z0[k] = fmaf(qd.x, a0.x, fmaf(qd.y, a0.y, fmaf(qd.z, a0.z, fmaf(qd.w, a0.w, z0[k]))));
                z1[k] = fmaf(qd.x, a1.x, fmaf(qd.y, a1.y, fmaf(qd.z, a1.z, fmaf(qd.w, a1.w, z1[k]))));
            }
        }
#pragma unroll
        for (int k = 0; k < MAXI; ++k) {
            // causal / chunk masks; an item with no visible key in this chunk keeps its state
            const bool v0 = lane < nk && j0 + lane < vis[k], v1 = lane + 32 < nk && j0 + lane + 32 < vis[k];
            const float cm = warp_max(fmaxf(v0 ? z0[k] : -INFINITY, v1 ? z1[k] : -INFINITY));
            float p0 = 0.f, p1 = 0.f;
            if (cm != -INFINITY) {
                const float mn = fmaxf(mx[k], cm);
                const float corr = __expf(mx[k] - mn);
                p0 = v0 ? __expf(z0[k] - mn) : 0.f;
                p1 = v1 ? __expf(z1[k] - mn) : 0.f;
                sum[k] = fmaf(sum[k], corr, warp_sum(p0 + p1));
#pragma unroll
                for (int d = 0; d < D; ++d) acc[k][d] *= corr;
                mx[k] = mn;
            }
            Ps[k * KC + lane] = p0;
            Ps[k * KC + lane + 32] = p1;
        }
        __syncwarp();
        // values: lane owns dimensions lane + 32 d; the probabilities are read 4 keys at a time
        // (positions of the chunk past nk hold p = 0 and finite staged values)
        const float4* p4 = reinterpret_cast<const float4*>(Ps);
        for (int j = 0; j < nk; j += 4) {
            float vd[4][D];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int d = 0; d < D; ++d) vd[u][d] = Vs[(j + u) * HD + lane + 32 * d];
#pragma unroll
            for (int k = 0; k < MAXI; ++k) {
                const float4 p = p4[(k * KC + j) / 4];
#pragma unroll
                for (int d = 0; d < D; ++d)
                    acc[k][d] = fmaf(p.x, vd[0][d], fmaf(p.y, vd[1][d], fmaf(p.z, vd[2][d], fmaf(p.w, vd[3][d], acc[k][d]))));
            }
        }
        __syncwarp();
    }
#pragma unroll
    for (int k = 0; k < MAXI; ++k) {
        if (!vis[k]) continue;
        const int it = warp + ATT_WARPS * k;
        const int h = g * a.group + it / a.rows, i = r0 + it % a.rows;
        T* o = static_cast<T*>(a.out) + (((size_t)c * a.n_q + h) * a.Lq + i) * HD;
        const float inv = 1.f / sum[k];
#pragma unroll
        for (int d = 0; d < D; ++d) o[lane + 32 * d] = from_f<T>(acc[k][d] * inv);
    }
}

// 2^x on the special-function unit (PTX ex2.approx), whose error is far below the bf16
// rounding of the probabilities it feeds (the parity tests bound the result at 1e-2).
__device__ __forceinline__ float at_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// ---------------------------------------------------------------- prefill form (bf16, tcgen05)
// One CTA per (chain, key/value head, tile of query tokens), two CTAs an SM.  A tile's 128 MMA rows are
// (query head of the group, token) pairs, rt = 128 / group tokens of each of the group's heads, so
// the group's heads share every staged key and value row.
//
// Warps 0-7: the softmax, two threads per row (= TMEM lane), one for each half of a chunk's keys.
// Warp 8: the loader; keys and values arrive in chunks of NK positions, in the order they are consumed,
// through a ring of NS slots, by TMA with the caller's strides (positions past the last key read as
// zeros).  Warp 9: the MMA issuer.  Per chunk: S = Q K^T into one of two TMEM buffers; the softmax
// takes the row max (exchanged between a row's two threads), writes its bf16 probabilities over the
// scores, where P V takes its A operand from, and keeps the row sum; O += P V accumulates in TMEM over all
// chunks.  The next chunk's S is there before the softmax asks for it.  O is rescaled in TMEM whenever the
// max of one of a warp's rows has grown, so that the largest probability of a row is 1, which bf16 holds
// exactly: rescaled only on growth by more than 2^8 the kernel takes 8% less time, but the error against 64
// bits is 2 to 9% larger (2.26e-3 for 2.16e-3 of 2048 queries, hd 128).
//
// What bounds it: the softmax's instructions (scale, ex2, bf16, and the sum of the rounded values: about
// five an element), at 55% of the issue slots; the max exchange and the waits around it leave the rest.
// 16 chains x 8 heads x 4, 2048 + 64 keys, hd 64: 471 us, 2.23 M visible pairs a head at 620 TFLOP/s (the
// one-CTA form it replaced, which took S, the softmax and P V of a 256-key chunk in turn: 1140 us); 4 chains,
// hd 128: 185 us (389).  Measured on the way, with the rarer rescaling (437 us): P through shared memory,
// two tiles a CTA 699 us; P in TMEM 565; loads by TMA instead of cp.async 490; one thread per row with two S
// buffers of 64 keys 463.

template <int HD>
struct FaSmem {
    static constexpr int LOAD_WARP = 8, MMA_WARP = 9, THREADS = 10 * 32;
    static constexpr int NK = HD == 64 ? 96 : 64;          // key positions per chunk: 2 NK + HD TMEM columns
    static constexpr int TMEM = 256;                       // two CTAs an SM
    static constexpr int Q_SLAB = 128 * 128;               // 128 query rows x 64 bf16
    static constexpr int SLAB = NK * 128;                  // NK keys x 64 bf16
    static constexpr int TILE = (HD / 64) * SLAB;          // NK keys x HD
    static constexpr int NS = HD == 64 ? 7 : 4;            // ring slots, one K or V chunk each
    static constexpr int Q_OFF = 0;
    static constexpr int KV_OFF = Q_OFF + (HD / 64) * Q_SLAB;
    static constexpr int X_OFF = KV_OFF + NS * TILE;       // [2][2][128] floats: row max (or sum) of each half
    static constexpr int BAR_OFF = X_OFF + 2 * 2 * 128 * 4;  // qfull full[NS] empty[NS] sfull[2] odone[2] pready[2] vlast
    static constexpr int SLOT_OFF = BAR_OFF + (2 * NS + 8) * 8;
    static constexpr int DYN = SLOT_OFF + 16 + 1024;       // + TMEM slot, + alignment slack
};
static_assert(2 * (FaSmem<64>::DYN + 1024) <= 228 * 1024 && 2 * (FaSmem<128>::DYN + 1024) <= 228 * 1024,
              "two attention CTAs an SM");

// N probabilities 2^(v k2 + moff) of a row in bf16 to N / 2 TMEM columns at `tp`.  Returns their sum as
// the MMA sees them (bf16-rounded).
template <int N>
__device__ __forceinline__ float fa_probs(const float (&v)[N], uint64_t k2, uint64_t moff, uint32_t tp) {
    uint64_t sum[2] = {0, 0};
#pragma unroll
    for (int b = 0; b < N; b += 16) {
        uint32_t pk[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float2 x = unpack_f32x2(fma_f32x2(pack_f32x2(v[b + 2 * j], v[b + 2 * j + 1]), k2, moff));
            pk[j] = pack_bf16(at_exp2(x.x), at_exp2(x.y));
            sum[j & 1] = add_f32x2(sum[j & 1], pack_f32x2(__uint_as_float(pk[j] << 16), __uint_as_float(pk[j] & 0xffff0000u)));
        }
        tmem_st8(tp + b / 2, pk);
    }
    const float2 s = unpack_f32x2(add_f32x2(sum[0], sum[1]));
    return s.x + s.y;
}

template <int HD>
__global__ void __launch_bounds__(FaSmem<HD>::THREADS, 2)
attention_prefill_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                         const __grid_constant__ CUtensorMap tmV, const AttnArgs a) {
    using SM = FaSmem<HD>;
    constexpr int NS = SM::NS, NK = SM::NK, NE = NK / 2;  // NE: keys of a chunk per softmax thread
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t bars = smem_u32(base + SM::BAR_OFF);
    const uint32_t qfull = bars;
    auto full = [&](int s) { return bars + 8 * (1 + s); };
    auto empty = [&](int s) { return bars + 8 * (1 + NS + s); };
    // of chunk j, phase j >> 1: two of each, since the softmax may be a chunk ahead of the issuer's P V
    auto sfull = [&](int j) { return bars + 8 * (1 + 2 * NS + (j & 1)); };
    auto odone = [&](int j) { return bars + 8 * (3 + 2 * NS + (j & 1)); };
    auto pready = [&](int j) { return bars + 8 * (5 + 2 * NS + (j & 1)); };
    const uint32_t vlast = bars + 8 * (7 + 2 * NS);
    uint32_t* slot = reinterpret_cast<uint32_t*>(base + SM::SLOT_OFF);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        mbar_init(qfull, 1);
        mbar_init(vlast, 1);
        for (int s = 0; s < NS; ++s) {
            mbar_init(full(s), 1);
            mbar_init(empty(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(sfull(b), 1);
            mbar_init(odone(b), 1);
            mbar_init(pready(b), 8);  // the eight softmax warps
        }
        fence_mbar_init();
    }
    if (warp == SM::MMA_WARP) {
        tmem_alloc(smem_u32(slot), SM::TMEM);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *slot, t_out = tmem + 2 * NK;  // two S (and P) buffers, then O

    // token tiles: the last first (causal: it has the most keys)
    const int c = blockIdx.z, g = blockIdx.y, rt = a.rows, r0 = (gridDim.x - 1 - blockIdx.x) * rt;
    const int keys = a.n_mem + min(a.Lq, r0 + rt), n = (keys + NK - 1) / NK;  // keys the tile's last token sees, in chunks
    // The last chunk may hold later tokens' rows (past the cache's last row TMA writes zeros). No probability of theirs is
    // added up, but 0 times a non-finite value would be: their value rows are cleared.
    const bool clear = keys < a.n_mem + a.Lq && keys < n * NK;

    if (warp == SM::LOAD_WARP) {
        bool landed = false;
        if (lane == 0) {
            tma_prefetch_map(&tmQ);
            tma_prefetch_map(&tmK);
            tma_prefetch_map(&tmV);
            mbar_expect_tx(qfull, (HD / 64) * a.group * rt * 128);
#pragma unroll
            for (int kb = 0; kb < HD / 64; ++kb)  // the query rows, [head of the group][token]
                tma_load_4d(smem_u32(base + SM::Q_OFF) + kb * SM::Q_SLAB, &tmQ, qfull, 64 * kb, r0, g * a.group, c);
            // a dimension that the caches share (stride 0) has one element in the maps
            const int ctx = a.s0 ? c / a.L : 0, layer = a.s1 ? c % a.L : 0, head = a.s2 ? g : 0;
            int s = 0, ph = 1;  // slot, and the phase of its release (the first round passes)
            auto load = [&](const CUtensorMap* m, int j) {
                if (!mbar_wait(empty(s), ph, a.status)) return false;
                const uint32_t dst = smem_u32(base + SM::KV_OFF + s * SM::TILE);
                mbar_expect_tx(full(s), SM::TILE);
#pragma unroll
                for (int kb = 0; kb < HD / 64; ++kb)
                    tma_load_5d(dst + kb * SM::SLAB, m, full(s), 64 * kb, j * NK, head, layer, ctx);
                if (++s == NS) {
                    s = 0;
                    ph ^= 1;
                }
                return true;
            };
            // K0 K1 V0 K2 V1 .. K(n-1) V(n-2) V(n-1)
            bool ok = load(&tmK, 0);
            for (int j = 0; ok && j < n - 1; ++j) ok = load(&tmK, j + 1) && load(&tmV, j);
            if (!clear) {
                ok = ok && load(&tmV, n - 1);
            } else if (ok && mbar_wait(empty(s), ph, a.status)) {  // on a barrier of its own: it counts as loaded once cleared
                mbar_expect_tx(vlast, SM::TILE);
#pragma unroll
                for (int kb = 0; kb < HD / 64; ++kb)
                    tma_load_5d(smem_u32(base + SM::KV_OFF + s * SM::TILE) + kb * SM::SLAB, &tmV, vlast, 64 * kb, (n - 1) * NK, head,
                                layer, ctx);
                landed = mbar_wait(vlast, 0, a.status);
            }
        }
        __syncwarp();
        if (clear && __shfl_sync(0xffffffffu, landed, 0)) {
            const int slot_v = (2 * n - 1) % NS;  // of the last of the 2 n loads
            uint8_t* v = base + SM::KV_OFF + slot_v * SM::TILE;
#pragma unroll 1
            for (int e = (keys - (n - 1) * NK) * 8 + lane; e < NK * 8; e += 32)  // 16-byte pieces, exchanged within a row
#pragma unroll
                for (int kb = 0; kb < HD / 64; ++kb) *reinterpret_cast<uint4*>(v + kb * SM::SLAB + e * 16) = make_uint4(0, 0, 0, 0);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(full(slot_v));
        }
    } else if (warp == SM::MMA_WARP) {
        if (lane == 0) {
            const uint32_t id_s = idesc_bf16_f32(128, NK, false, false), id_o = idesc_bf16_f32(128, HD, false, true);
            // descriptors of the queries and of the ring's first slot as K and as V
            const uint64_t dq = sdesc_sw128(smem_u32(base + SM::Q_OFF), 16), dk0 = sdesc_sw128(smem_u32(base + SM::KV_OFF), 16),
                           dv0 = sdesc_sw128(smem_u32(base + SM::KV_OFF), SM::SLAB);
            int s = 0, ph = 0;  // the ring's next slot and its phase
            auto next = [&]() {
                if (++s == NS) {
                    s = 0;
                    ph ^= 1;
                }
            };
            auto issue_s = [&](int j) {  // S = Q K^T over HD (K-major both)
                if (!mbar_wait(full(s), ph, a.status)) return false;
                tc_fence_after();
                const uint64_t dk = sdesc_step(dk0, s * SM::TILE);
#pragma unroll
                for (int kb = 0; kb < HD / 64; ++kb)
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        umma_bf16(tmem + (j & 1) * NK, sdesc_step(dq, kb * SM::Q_SLAB + u * 32),
                                  sdesc_step(dk, kb * SM::SLAB + u * 32), id_s, (kb | u) ? 1u : 0u);
                umma_commit(sfull(j));
                umma_commit(empty(s));
                next();
                return true;
            };
            bool ok = mbar_wait(qfull, 0, a.status) && issue_s(0) && (n < 2 || issue_s(1));
            for (int j = 0; ok && j < n; ++j) {
                // P of chunk j is in TMEM
                ok = mbar_wait(full(s), ph, a.status) && mbar_wait(pready(j), (j >> 1) & 1, a.status);
                if (!ok) break;
                tc_fence_after();
                const uint64_t dv = sdesc_step(dv0, s * SM::TILE);
#pragma unroll
                for (int kk = 0; kk < NK / 16; ++kk)  // O += P V over the chunk's keys (P in TMEM, V MN-major)
                    umma_bf16_ta(t_out, tmem + (j & 1) * NK + kk * 8, sdesc_step(dv, kk * 16 * 128), id_o, (j | kk) ? 1u : 0u);
                umma_commit(odone(j));
                umma_commit(empty(s));
                next();
                // S of chunk j + 2 goes over the P that P V has to have read
                if (j + 2 < n) ok = mbar_wait(odone(j), (j >> 1) & 1, a.status) && issue_s(j + 2);
            }
            if (!ok) drain_copies();
        }
        __syncwarp();
    } else {
        // ---- softmax: row = TMEM lane, half = keys NE half .. of every chunk
        const int quarter = warp & 3, half = warp >> 2, row = quarter * 32 + lane;
        const int hr = row / rt, i = r0 + row % rt;
        const bool live = hr < a.group && i < a.Lq;
        const int vis = a.n_mem + (live ? i : r0) + 1;   // keys the row sees (a row of padding: any)
        const float k2 = a.scale * 1.4426950408889634f;  // softmax scale in base 2: exp(s x) = 2^(s log2(e) x)
        const uint32_t lane_off = (uint32_t)(quarter * 32) << 16, t_o = t_out + lane_off + half * (HD / 2);
        float* xch = reinterpret_cast<float*>(base + SM::X_OFF);
        float m_run = -INFINITY, l = 0.f;
        bool ok = true;
        for (int j = 0; j < n; ++j) {
            const uint32_t t_s = tmem + lane_off + (j & 1) * NK;
            ok = __all_sync(0xffffffffu, mbar_wait(sfull(j), (j >> 1) & 1, a.status));
            tc_fence_after();
            float v[NE];
            if constexpr (NE == 48)
                tmem_ld48(t_s + half * NE, v);
            else
                tmem_ld32(t_s + half * NE, v);
            if ((j + 1) * NK > a.n_mem + r0 + 1) {      // some row does not see the whole chunk:
                const int nv = vis - j * NK - half * NE;  // a hidden key's score of -inf gives it a probability of 0
#pragma unroll
                for (int u = 0; u < NE; ++u) v[u] = u < nv ? v[u] : -INFINITY;
            }
            float c4[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
            for (int u = 4; u < NE; u += 4)
#pragma unroll
                for (int k = 0; k < 4; ++k) c4[k] = fmaxf(c4[k], v[u + k]);
            float cm = fmaxf(fmaxf(c4[0], c4[1]), fmaxf(c4[2], c4[3]));
            float* x = xch + (j & 1) * 256;
            x[half * 128 + row] = cm;
            // The two warps of the rows meet, all their scores read (P goes over them); after a wait that ran
            // out both leave here.
            tc_fence_before();
            ok = named_bar_and(1 + quarter, 64, ok);
            if (!ok) break;
            tc_fence_after();
            cm = fmaxf(cm, x[(half ^ 1) * 128 + row]);
            if (j == 0) {
                m_run = fmaxf(cm, -FLT_MAX);  // finite: where every key so far scores -inf, probabilities of 0
            } else {
                const bool grown = cm > m_run;
                if (__any_sync(0xffffffffu, grown)) {  // the same in both warps: each rescales its half of O
                    // O up to the last chunk (on this barrier the phase before is done: S of this chunk waited for it)
                    const bool in = __all_sync(0xffffffffu, mbar_wait(odone(j - 1), ((j - 1) >> 1) & 1, a.status));
                    tc_fence_after();
                    const float corr = grown ? at_exp2((m_run - cm) * k2) : 1.f;
                    if (grown) m_run = cm;
                    l *= corr;
#pragma unroll 1
                    for (int cb = 0; in && cb < HD / 2; cb += 16) {
                        float ov[16];
                        uint32_t on[16];
                        tmem_ld16(t_o + cb, ov);
#pragma unroll
                        for (int u = 0; u < 16; ++u) on[u] = __float_as_uint(ov[u] * corr);
                        tmem_st16(t_o + cb, on);
                    }
                }
            }
            const float moff = -m_run * k2;
            l += fa_probs(v, pack_f32x2(k2, k2), pack_f32x2(moff, moff), t_s + half * (NE / 2));
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(pready(j));
        }
        float* x = xch + (n & 1) * 256;
        x[half * 128 + row] = l;
        if (ok) ok = __all_sync(0xffffffffu, mbar_wait(odone(n - 1), ((n - 1) >> 1) & 1, a.status));
        ok = named_bar_and(1 + quarter, 64, ok);
        if (ok) {
            tc_fence_after();
            const float inv = 1.f / (l + x[(half ^ 1) * 128 + row]);
            bf16* orow = static_cast<bf16*>(a.out) +
                         (((size_t)c * a.n_q + g * a.group + (live ? hr : 0)) * a.Lq + (live ? i : 0)) * HD + half * (HD / 2);
#pragma unroll
            for (int cb = 0; cb < HD / 2; cb += 32) {
                float v[32];
                tmem_ld32(t_o + cb, v);
                if (live) {
#pragma unroll
                    for (int u = 0; u < 32; u += 8)
                        *reinterpret_cast<uint4*>(orow + cb + u) =
                            make_uint4(pack_bf16(v[u] * inv, v[u + 1] * inv), pack_bf16(v[u + 2] * inv, v[u + 3] * inv),
                                       pack_bf16(v[u + 4] * inv, v[u + 5] * inv), pack_bf16(v[u + 6] * inv, v[u + 7] * inv));
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == SM::MMA_WARP) tmem_dealloc(tmem, SM::TMEM);
}

// ---------------------------------------------------------------- decode form (bf16, few rows)
// Few (query head, token) rows per key/value head: the caches are read once and little is computed,
// so the kernel is a stream over keys and values, bound by HBM, or at short caches by latency.  A
// cluster of `splits` CTAs takes (chain, key/value head, 16 rows); the keys' blocks of 32 (hd 128: 16)
// positions are split over the CTAs and their warps.  Each warp runs an online softmax of its own with
// mma.m16n8k16 on operands loaded from global memory straight into fragment order (a 128-row
// tcgen05 tile would be 1/8 to 1/32 full, and its staging would cost more than the arithmetic): the
// contraction over hd and the order of output columns are free, so they are permuted to let every
// thread load 16 contiguous bytes (K: dims 32 p + 8 t .. + 7 of key g; V: dims 64 p + 8 g .. + 7 of keys
// 2 t, 2 t + 1, 2 t + 8, 2 t + 9; lane = 4 g + t).  The warps' partial results meet in shared memory, the
// CTAs' through distributed shared memory.
constexpr int DE_WARPS = 4, DE_ROWS = 16;
// This form is taken up to 16 rows per key/value head, and beyond that while its row tiles over all
// heads stay few: it re-reads the caches for each 16 rows but splits the keys, the prefill form does
// neither.  1 chain x 8 heads x 4, 4000 keys: 16 / 64 / 128 rows take 7.9 / 9.5 / 14.0 us here and 37 us
// in the prefill form; 16 chains, 1000 keys: 16 rows 10.4 us here, 20 rows 14.9; 32 rows 13.2 in the prefill form.
constexpr int DE_MAX_TILES = 128;

template <int HD>
struct DeSmem {
    // per warp, then once for the CTA: O [16][HD], then max and sum per row
    static constexpr int PART = DE_ROWS * HD + 2 * DE_ROWS;
    static constexpr int FLOATS = (DE_WARPS + 1) * PART;
};

// Row tiles of the decode form.  The tokens go in blocks of 128 / group, the tokens of a tile of the prefill form,
// whose (token, head of the group) rows, heads innermost, are cut into tiles of 16: a tile sees the keys up to its
// last token's only, and a non-finite value row reaches (as 0 times it) no token outside the later one's block.
struct DeTile {
    int rr0, tok0, ntok, keys;  // first row within the block; the block's tokens; keys the tile's last token sees
    static int count(int group, int Lq) {
        const int bt = 128 / group, per = (bt * group + DE_ROWS - 1) / DE_ROWS;
        return Lq / bt * per + (Lq % bt * group + DE_ROWS - 1) / DE_ROWS;
    }
    // r / group for 0 <= r < 1024 and group <= 64: the factor's error adds less than r / 65536 < 1 / group
    static __device__ int over_group(const AttnArgs& a, int r) { return (r * a.group_inv) >> 16; }
    __device__ DeTile(const AttnArgs& a, int t) {
        const int b = a.Lq > a.tile_tok ? t / a.per_block : 0;
        rr0 = (t - b * a.per_block) * DE_ROWS;
        tok0 = b * a.tile_tok;
        ntok = min(a.tile_tok, a.Lq - tok0);
        keys = a.n_mem + tok0 + min(over_group(a, rr0 + DE_ROWS - 1), ntok - 1) + 1;
    }
    // row r of the tile; false past its last (the others then point at some valid row)
    __device__ bool row(const AttnArgs& a, int r, int& head, int& tok) const {
        const int i = over_group(a, rr0 + r);
        head = (rr0 + r) - i * a.group;
        tok = tok0 + min(i, ntok - 1);
        return i < ntok;
    }
};

__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&A)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(A[0]), "r"(A[1]), "r"(A[2]), "r"(A[3]), "r"(b0), "r"(b1));
}

// fp32 of CTA `rank` of the cluster at the place of `p` in this one
__device__ __forceinline__ float ld_cluster_f32(const float* p, uint32_t rank) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(map_to_cta(smem_u32(p), rank)) : "memory");
    return v;
}

template <int HD>
__global__ void __launch_bounds__(DE_WARPS * 32, HD == 64 ? 4 : 3) attention_decode_kernel(const AttnArgs a, int splits) {
    constexpr int NP = HD / 32, NV = HD / 64;  // 16-byte pieces of a key per thread; of a value
    constexpr int KB = HD == 64 ? 32 : 16;     // keys per step
    extern __shared__ float de_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gq = lane >> 2, t = lane & 3;
    const int c = blockIdx.z, g = blockIdx.y, rank = (int)cluster_ctarank();
    const DeTile tile(a, (int)cluster_id_x());
    const int keys = __shfl_sync(0xffffffffu, tile.keys, 0);  // the same in every lane, and known to be
    const long long kv_off = (long long)(c / a.L) * a.s0 + (long long)(c % a.L) * a.s1 + (long long)g * a.s2;
    const bf16* Kc = static_cast<const bf16*>(a.K) + kv_off + 8 * t;
    const bf16* Vc = static_cast<const bf16*>(a.V) + kv_off + 8 * gq;
    // rows gq and gq + 8 of the tile
    uint32_t qa[HD / 16][4];
    int vis[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        int head, tok;
        const bool live = tile.row(a, gq + 8 * h, head, tok);
        vis[h] = live ? a.n_mem + tok + 1 : 0;
        const bf16* q = static_cast<const bf16*>(a.Q) + (((size_t)c * a.n_q + (size_t)g * a.group + head) * a.Lq + tok) * HD + 8 * t;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const uint4 v = live ? *reinterpret_cast<const uint4*>(q + 32 * p) : make_uint4(0, 0, 0, 0);
            qa[2 * p][h] = v.x;
            qa[2 * p][2 + h] = v.y;
            qa[2 * p + 1][h] = v.z;
            qa[2 * p + 1][2 + h] = v.w;
        }
    }
    const float k2 = a.scale * 1.4426950408889634f;
    float o[8 * NV][4], m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
#pragma unroll
    for (int j = 0; j < 8 * NV; ++j) o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.f;
    const int nb = (keys + KB - 1) / KB;
    const int b1 = (int)((long long)nb * (rank + 1) / splits);
    for (int b = (int)((long long)nb * rank / splits) + warp; b < b1; b += DE_WARPS) {
        const int j0 = b * KB;
        uint4 kr[KB / 8][NP], vr[KB / 16][4][NV];
#pragma unroll
        for (int nt = 0; nt < KB / 8; ++nt) {
            const int key = j0 + 8 * nt + gq;
#pragma unroll
            for (int p = 0; p < NP; ++p)
                kr[nt][p] = key < keys ? __ldg(reinterpret_cast<const uint4*>(Kc + (long long)key * a.s3 + 32 * p))
                                       : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int kk = 0; kk < KB / 16; ++kk)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int key = j0 + 16 * kk + 2 * t + (u & 1) + 8 * (u >> 1);
#pragma unroll
                for (int p = 0; p < NV; ++p)
                    vr[kk][u][p] = key < keys ? __ldg(reinterpret_cast<const uint4*>(Vc + (long long)key * a.s3 + 64 * p))
                                              : make_uint4(0, 0, 0, 0);
            }
        float s[KB / 8][4];
        float cm[2] = {-INFINITY, -INFINITY};
#pragma unroll
        for (int nt = 0; nt < KB / 8; ++nt) {
            s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                mma_16816(s[nt], qa[2 * p], kr[nt][p].x, kr[nt][p].y);
                mma_16816(s[nt], qa[2 * p + 1], kr[nt][p].z, kr[nt][p].w);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {  // e: row half e >> 1, key 2 t + (e & 1)
                const bool in = j0 + 8 * nt + 2 * t + (e & 1) < vis[e >> 1];
                cm[e >> 1] = in ? fmaxf(cm[e >> 1], s[nt][e]) : cm[e >> 1];
            }
        }
        float moff[2], corr[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            cm[h] = fmaxf(cm[h], __shfl_xor_sync(0xffffffffu, cm[h], 1));
            cm[h] = fmaxf(cm[h], __shfl_xor_sync(0xffffffffu, cm[h], 2));
            const float mn = fmaxf(m[h], cm[h]);
            corr[h] = mn == -INFINITY ? 1.f : at_exp2((m[h] - mn) * k2);
            moff[h] = mn == -INFINITY ? 0.f : -mn * k2;
            m[h] = mn;
            l[h] *= corr[h];
        }
#pragma unroll
        for (int j = 0; j < 8 * NV; ++j) {
            o[j][0] *= corr[0];
            o[j][1] *= corr[0];
            o[j][2] *= corr[1];
            o[j][3] *= corr[1];
        }
#pragma unroll
        for (int kk = 0; kk < KB / 16; ++kk) {
            uint32_t pa[4];  // rows g / g + 8 x keys (2t, 2t + 1), then the same of the next eight keys
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int nt = 2 * kk + (q >> 1), h = q & 1, key = j0 + 8 * nt + 2 * t;
                const float e0 = key < vis[h] ? at_exp2(fmaf(s[nt][2 * h], k2, moff[h])) : 0.f;
                const float e1 = key + 1 < vis[h] ? at_exp2(fmaf(s[nt][2 * h + 1], k2, moff[h])) : 0.f;
                pa[q] = pack_bf16(e0, e1);
                // the sum takes the probabilities the MMA sees
                l[h] += __uint_as_float(pa[q] << 16) + __uint_as_float(pa[q] & 0xffff0000u);
            }
#pragma unroll
            for (int p = 0; p < NV; ++p) {
                const uint32_t* v0 = reinterpret_cast<const uint32_t*>(&vr[kk][0][p]);
                const uint32_t* v1 = reinterpret_cast<const uint32_t*>(&vr[kk][1][p]);
                const uint32_t* v2 = reinterpret_cast<const uint32_t*>(&vr[kk][2][p]);
                const uint32_t* v3 = reinterpret_cast<const uint32_t*>(&vr[kk][3][p]);
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    mma_16816(o[8 * p + 2 * w], pa, __byte_perm(v0[w], v1[w], 0x5410), __byte_perm(v2[w], v3[w], 0x5410));
                    mma_16816(o[8 * p + 2 * w + 1], pa, __byte_perm(v0[w], v1[w], 0x7632), __byte_perm(v2[w], v3[w], 0x7632));
                }
            }
        }
    }
    // partial results of the warps: column n of output tile j of piece p is dimension 64 p + 8 n + j
    float* part = de_smem + warp * DeSmem<HD>::PART;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        l[h] += __shfl_xor_sync(0xffffffffu, l[h], 1);
        l[h] += __shfl_xor_sync(0xffffffffu, l[h], 2);
        const int r = gq + 8 * h;
        if (t == 0) {
            part[DE_ROWS * HD + r] = m[h];
            part[DE_ROWS * HD + DE_ROWS + r] = l[h];
        }
#pragma unroll
        for (int p = 0; p < NV; ++p)
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int j = 0; j < 8; j += 4)
                    *reinterpret_cast<float4*>(part + r * HD + 64 * p + 8 * (2 * t + e) + j) =
                        make_float4(o[8 * p + j][2 * h + e], o[8 * p + j + 1][2 * h + e], o[8 * p + j + 2][2 * h + e],
                                    o[8 * p + j + 3][2 * h + e]);
    }
    __syncthreads();
    // the CTA's result: max, sum and O over its warps
    float* sum = de_smem + DE_WARPS * DeSmem<HD>::PART;
    const float* ml = de_smem + DE_ROWS * HD;
    for (int e = threadIdx.x; e < DE_ROWS * HD; e += DE_WARPS * 32) {
        const int r = e / HD;
        float mx = -INFINITY, lt = 0.f, ot = 0.f;
#pragma unroll
        for (int w = 0; w < DE_WARPS; ++w) mx = fmaxf(mx, ml[w * DeSmem<HD>::PART + r]);
#pragma unroll
        for (int w = 0; w < DE_WARPS; ++w) {
            const float mw = ml[w * DeSmem<HD>::PART + r];
            const float f = mw == -INFINITY ? 0.f : at_exp2((mw - mx) * k2);
            lt = fmaf(f, ml[w * DeSmem<HD>::PART + DE_ROWS + r], lt);
            ot = fmaf(f, de_smem[w * DeSmem<HD>::PART + e], ot);
        }
        sum[e] = ot;
        if (e % HD == 0) {
            sum[DE_ROWS * HD + r] = mx;
            sum[DE_ROWS * HD + DE_ROWS + r] = lt;
        }
    }
    if (splits > 1)
        cluster_sync();
    else
        __syncthreads();
    const DeTile tile_o(a, (int)cluster_id_x());  // made again: kept over the loop it costs registers that the loop needs
    // every CTA of the cluster finishes a share of the rows' outputs, two dimensions a thread
    for (int e = 2 * (rank * DE_WARPS * 32 + threadIdx.x); e < DE_ROWS * HD; e += 2 * splits * DE_WARPS * 32) {
        const int r = e / HD, d = e - r * HD;
        int head, tok;
        if (!tile_o.row(a, r, head, tok)) break;
        float mx = -INFINITY, lt = 0.f, o0 = 0.f, o1 = 0.f;
        for (int k = 0; k < splits; ++k) mx = fmaxf(mx, ld_cluster_f32(sum + DE_ROWS * HD + r, k));
        for (int k = 0; k < splits; ++k) {
            const float mk = ld_cluster_f32(sum + DE_ROWS * HD + r, k);
            const float f = mk == -INFINITY ? 0.f : at_exp2((mk - mx) * k2);
            lt = fmaf(f, ld_cluster_f32(sum + DE_ROWS * HD + DE_ROWS + r, k), lt);
            o0 = fmaf(f, ld_cluster_f32(sum + e, k), o0);
            o1 = fmaf(f, ld_cluster_f32(sum + e + 1, k), o1);
        }
        const float inv = 1.f / lt;
        bf16* out = static_cast<bf16*>(a.out) + (((size_t)c * a.n_q + (size_t)g * a.group + head) * a.Lq + tok) * HD + d;
        *reinterpret_cast<uint32_t*>(out) = pack_bf16(o0 * inv, o1 * inv);
    }
    if (splits > 1) cluster_sync();  // no CTA leaves while another reads its shared memory
}

template <typename T, int HD>
cudaError_t launch_t(const AttnArgs& a, int C, cudaStream_t st) {
    const size_t smem = AttnSmem<T, HD>::FLOATS * sizeof(float);
    static PerDevice<SmemOptIn> once;
    cudaError_t e = smem_opt_in(reinterpret_cast<const void*>(attention_kernel<T, HD>), smem, once);
    if (e != cudaSuccess) return e;
    dim3 grid((a.Lq + a.rows - 1) / a.rows, a.n_kv, C);
    attention_kernel<T, HD><<<grid, ATT_WARPS * 32, smem, st>>>(a);
    return cudaGetLastError();
}

template <int HD>
cudaError_t launch_prefill(AttnArgs a, int n_ctx, int C, cudaStream_t st) {
    static PerDevice<SmemOptIn> once;
    cudaError_t e = smem_opt_in(reinterpret_cast<const void*>(attention_prefill_kernel<HD>), FaSmem<HD>::DYN, once);
    if (e != cudaSuccess) return e;
    // The maps of the last call's shape, of which a call only sets the addresses: three maps encoded anew are 0.5 us of
    // the 9 us that a short call takes on the host
    struct Plan {
        long long key[10];
        CUtensorMap q, kv;
    };
    static thread_local Plan plan = {};
    const int rows = 128 / a.group;  // tokens per tile: the group's heads x rows fill the 128 MMA rows
    const long long key[10] = {n_ctx, a.L, a.n_q, a.n_kv, a.Lq, a.n_mem, a.s0, a.s1, a.s2, a.s3};
    if (!std::equal(key, key + 10, plan.key)) {
        const uint64_t Lq = a.Lq, keys = (uint64_t)a.n_mem + Lq;
        const uint64_t qd[4] = {HD, Lq, (uint64_t)a.n_q, (uint64_t)C}, qs[3] = {HD * 2, Lq * HD * 2, a.n_q * Lq * HD * 2};
        const uint32_t qb[4] = {64, (uint32_t)rows, (uint32_t)a.group, 1};
        // the caller's strides; a dimension that the caches share (stride 0) has one element, which takes any stride
        const uint64_t kd[5] = {HD, keys, a.s2 ? (uint64_t)a.n_kv : 1, a.s1 ? (uint64_t)a.L : 1, a.s0 ? (uint64_t)n_ctx : 1};
        const uint64_t s3 = a.s3 * 2;
        const uint64_t ks[4] = {s3, kd[2] > 1 ? a.s2 * 2 : s3, kd[3] > 1 ? a.s1 * 2 : s3, kd[4] > 1 ? a.s0 * 2 : s3};
        const uint32_t kb[5] = {64, FaSmem<HD>::NK, 1, 1, 1};
        plan.key[0] = 0;
        if (!encode_map_bf16_4d(&plan.q, a.Q, qd, qs, qb) || !encode_map_bf16_5d(&plan.kv, a.K, kd, ks, kb))
            return launch_t<bf16, HD>(a, C, st);  // strides past a tensor map's range (2^40 bytes): the CUDA-core form
        std::copy(key, key + 10, plan.key);
    }
    CUtensorMap mq = plan.q, mk = plan.kv, mv = plan.kv;
    if (!retarget_map(&mq, a.Q) || !retarget_map(&mk, a.K) || !retarget_map(&mv, a.V)) return cudaErrorInvalidValue;
    a.rows = rows;
    dim3 grid((a.Lq + a.rows - 1) / a.rows, a.n_kv, C);
    attention_prefill_kernel<HD><<<grid, FaSmem<HD>::THREADS, FaSmem<HD>::DYN, st>>>(mq, mk, mv, a);
    return cudaGetLastError();
}

template <int HD>
cudaError_t launch_decode(AttnArgs a, int C, int sms, cudaStream_t st) {
    a.tile_tok = 128 / a.group;
    a.per_block = (a.tile_tok * a.group + DE_ROWS - 1) / DE_ROWS;
    a.group_inv = 65536 / a.group + 1;
    static PerDevice<SmemOptIn> once;
    constexpr size_t smem = DeSmem<HD>::FLOATS * sizeof(float);
    cudaError_t e = smem_opt_in(reinterpret_cast<const void*>(attention_decode_kernel<HD>), smem, once);
    if (e != cudaSuccess) return e;
    const int row_tiles = DeTile::count(a.group, a.Lq);
    // split the keys over a cluster until the grid fills the SMs' CTA slots, or a CTA's warps would
    // have no block of keys each
    const long long ctas = (long long)row_tiles * a.n_kv * C;
    const int blocks = (a.n_mem + a.Lq + 31) / 32;
    const int slots = (HD == 64 ? 4 : 3) * sms;
    const int splits = (int)std::max(1ll, std::min({8ll, slots / ctas, (long long)blocks / DE_WARPS}));
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = splits;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(splits * row_tiles, a.n_kv, C);
    cfg.blockDim = dim3(DE_WARPS * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, attention_decode_kernel<HD>, a, splits);
}

}  // namespace

cudaError_t launch_attention(const DevState& s, int n_layers, const void* Q, int n_q, int Lq, const void* K,
                             const void* V, const long long* strides, int n_mem, void* out, cudaStream_t st) {
    AttnArgs a{};
    a.Q = Q; a.K = K; a.V = V; a.out = out;
    a.s0 = strides[0]; a.s1 = strides[1]; a.s2 = strides[2]; a.s3 = strides[3];
    a.L = n_layers; a.n_q = n_q; a.n_kv = s.n_kv; a.group = n_q / s.n_kv; a.Lq = Lq; a.n_mem = n_mem;
    a.rows = std::max(1, ATT_ITEMS / a.group);
    a.scale = 1.0f / sqrtf((float)s.hd);
    const long long el = s.dtype == 0 ? 4 : 2;
    a.vec = ((reinterpret_cast<uintptr_t>(K) | reinterpret_cast<uintptr_t>(V)) & 15u) == 0 && (a.s0 * el) % 16 == 0 &&
            (a.s1 * el) % 16 == 0 && (a.s2 * el) % 16 == 0 && (a.s3 * el) % 16 == 0;
    a.status = s.status;
    if (s.dtype == 0)
        return s.hd == 64 ? launch_t<float, 64>(a, s.C, st) : launch_t<float, 128>(a, s.C, st);
    // bf16 on the tensor cores when every row it stages is 16-byte aligned (the queries and the
    // output are dense rows of hd elements); other cache layouts take the CUDA-core kernel
    if (a.vec && ((reinterpret_cast<uintptr_t>(Q) | reinterpret_cast<uintptr_t>(out)) & 15u) == 0) {
        const long long row_tiles = ((long long)a.group * Lq + DE_ROWS - 1) / DE_ROWS;
        if (row_tiles == 1 || row_tiles * a.n_kv * s.C <= DE_MAX_TILES)
            return s.hd == 64 ? launch_decode<64>(a, s.C, s.sms, st) : launch_decode<128>(a, s.C, s.sms, st);
        return s.hd == 64 ? launch_prefill<64>(a, s.C / n_layers, s.C, st) : launch_prefill<128>(a, s.C / n_layers, s.C, st);
    }
    return s.hd == 64 ? launch_t<bf16, 64>(a, s.C, st) : launch_t<bf16, 128>(a, s.C, st);
}

}  // namespace mone
