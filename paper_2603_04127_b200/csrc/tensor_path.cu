// Tensor-core path of libdarkattn: bf16 operands, fp32 accumulation, tcgen05.mma with TMEM accumulators,
// operands staged by TMA (128-byte swizzle), exponentials fused into the TMEM read-out.
//
// Work decomposition. Features are cut into slabs of 128; one CTA owns one (batch, head, slab). Every
// quantity of the attention is a sum over features, so a slab CTA produces, for its 128 features, the
// partial numerator rows, the partial normaliser and the exponent its rows were scaled by; a small
// combine kernel adds the slabs. Per 128-token tile a slab CTA computes
//     U = X Omega_slab^T            Omega = log2(e) s W M folded once per call (u = w.(sMx) = (sM^T w).x), kept as the
//                                   sum of two bf16 matrices (its rounding and what the rounding left out), so that the
//                                   exponent's argument is as accurate as its fp32 accumulation
//     phi(Q) = 2^(U - rowmax U)     any per-row factor cancels in O, including exp(-|Mq|^2/2)
//     phi(K) = 2^(U - n - c)        n = log2(e) |sMk|^2/2 per key (from the norms kernel), c per slab
// and then, causal:   P = tril(phi(Q) phi(K)^T),  O = P V + phi(Q) S_prev,  S += phi(K)^T V,  z += phi(K)^T 1
// with the state S (128 x dv, fp32) resident in TMEM across the chunks of the sequence;
// non-causal: a key pass accumulates S and z over all keys, a query pass applies them.
#include "common.cuh"
#include "tc_common.cuh"

#include <math.h>
#include <string.h>

namespace darkattn {

using namespace tc;

namespace {

constexpr float kLog2e = 1.4426950408889634f;
// The key features are scaled so that the largest one of a (batch, head, slab) is 2^kShiftHeadroom rather than 1: fp32 and
// bf16 reach down to 2^-126, so keys up to 190 binary orders below the largest keep a nonzero feature (causal prefixes see
// only some of the keys), while sums over 2^17 keys of products with values and query features (<= 1) stay far from 2^127.
constexpr float kShiftHeadroom = 64.f;

// ------------------------------------------------------------------ small helpers

// ------------------------------------------------------------------ prologue kernels (SIMT, tiny)
// Omega[h,l,c] = log2(e) * s * sum_a W[l,a] M[h,a,c], stored as its bf16 rounding Om and the bf16 rounding Oml of what
// that left out (Om + Oml carries 16 bits of Omega). One block per (head, 16 rows l); its four warps split the sum over a and add up through
// shared memory; d / 32 columns per lane: a thread's 16 x d/32 tile of outputs takes one broadcast load of four W values per
// 4 d/32 products.
template <int TC>
__global__ void __launch_bounds__(128) fold_omega_kernel(const __nv_bfloat16 *W, const __nv_bfloat16 *M, __nv_bfloat16 *Om, __nv_bfloat16 *Oml,
                                                         int m, int r, int w_per_head, float coef, int *cs, int ncs, int *status, float4 *zero,
                                                         long long nzero)
{
    constexpr int R = 16, d = 32 * TC;
    __shared__ __align__(16) float sw[R][128];
    __shared__ float part[3][R * TC][32];           // the partial sums of warps 1..3
    const int h = blockIdx.y, l0 = blockIdx.x * R, lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
    pdl_wait();
    const __nv_bfloat16 *w = W + ((size_t)(w_per_head ? h : 0) * m + l0) * r;
    for (int i = threadIdx.x; i < R * r; i += 128) sw[i / r][i % r] = __bfloat162float(w[i]);
    {   // what the call's later kernels expect: a clear status word, the key shifts (which the prepass raises to the maximum over
        // the keys) at the smallest order key, the sums of the non-causal state at zero
        const int nb = gridDim.x * gridDim.y, b = blockIdx.y * gridDim.x + blockIdx.x;
        if (b == 0 && threadIdx.x == 0) *status = 0;
        for (int i = b * 128 + threadIdx.x; i < ncs; i += nb * 128) cs[i] = (int)0x80000000u;
        for (long long i = b * 128 + threadIdx.x; i < nzero; i += nb * 128) zero[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    const __nv_bfloat16 *Mh = M + (size_t)h * r * d + lane;
    float acc[R][TC];
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int q = 0; q < TC; ++q) acc[i][q] = 0.f;
#pragma unroll 2
    for (int a0 = 4 * wq; a0 < r; a0 += 16) {       // r is a multiple of 16: warp wq takes a = 4 wq .. 4 wq + 3 of every 16
        float x[4][TC];
#pragma unroll
        for (int jj = 0; jj < 4; ++jj)
#pragma unroll
            for (int q = 0; q < TC; ++q) x[jj][q] = __bfloat162float(Mh[(size_t)(a0 + jj) * d + 32 * q]);
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const float4 wv = *reinterpret_cast<const float4 *>(&sw[i][a0]);
#pragma unroll
            for (int q = 0; q < TC; ++q)
                acc[i][q] = fmaf(wv.x, x[0][q], fmaf(wv.y, x[1][q], fmaf(wv.z, x[2][q], fmaf(wv.w, x[3][q], acc[i][q]))));
        }
    }
    if (wq > 0) {
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
            for (int q = 0; q < TC; ++q) part[wq - 1][i * TC + q][lane] = acc[i][q];
    }
    __syncthreads();
    if (wq == 0) {
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
            for (int q = 0; q < TC; ++q) {
                const float om = coef * (acc[i][q] + part[0][i * TC + q][lane] + part[1][i * TC + q][lane] + part[2][i * TC + q][lane]);
                const __nv_bfloat16 hi = __float2bfloat16_rn(om);
                const size_t o = ((size_t)h * m + l0 + i) * d + lane + 32 * q;
                Om[o] = hi;
                Oml[o] = __float2bfloat16_rn(om - __bfloat162float(hi));
            }
    }
}

// ------------------------------------------------------------------ key prepass: norms and key-side shifts in one pass over K
//   n[bh,j]     = coef * |M_h k_j|^2                                   (log2 units; written by the CTAs of the first slab pair)
//   c[bh,slab]  = max_j max_{l in slab} (u_jl - n_j) - kShiftHeadroom   u = K Omega_hi^T
// The stabiliser of the key features is the largest exponent any key of the (batch, head) reaches in the slab, taken
// from the data (with it the largest key feature is 2^kShiftHeadroom, whatever the norms of the keys); being one constant per
// (batch, head, slab) it cancels in O. One CTA per (batch, head, pair of slabs, piece of the sequence): K tiles by TMA into
// two buffers, x~ = K M^T and U = K Omega_slab^T on the tensor cores, squared norms and row maxima read out of tensor memory
// by four warps (x~ of tile t + 1 is computed while U of tile t is read), the piece's maxima by atomicMax on order keys.
struct PrepassParams {
    CUtensorMap mapK, mapM, mapOm;
    float *nK;           // [BH, N] key norms, log2 units
    int *cs;             // [BH, nslab] order keys of the shifts
    int *status;
    int N, H, Hkv, T, m, r, nslab, npair, nsplit;
    float coef;          // log2(e) * s^2 / 2
};

enum PBars { PB_M, PB_K0, PB_K1, PMX, PMU, PEX, PEU, PNBARS };

template <int D>
__global__ void __launch_bounds__(160, 1) tc_key_prepass_kernel(const __grid_constant__ PrepassParams p)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    constexpr int kTile = 128 * D * 2;
    unsigned char *sM = smem, *sOm = smem + kTile, *sK = smem + 3 * kTile;       // M, two slabs of Omega, two K buffers
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + 5 * kTile);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + PNBARS);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(bars + PNBARS + 1);
    const int tid = threadIdx.x, warp = uniform(tid >> 5);
    const int unit = blockIdx.x / p.nsplit, split = blockIdx.x % p.nsplit;
    const int bh = unit / p.npair, pair = unit % p.npair, h = bh % p.H;
    const int slab0 = 2 * pair, ns = (slab0 + 1 < p.nslab) ? 2 : 1;           // this CTA's one or two slabs
    const int t0 = (int)((long long)p.T * split / p.nsplit), t1 = (int)((long long)p.T * (split + 1) / p.nsplit);
    const int rowk0 = kv_row0(bh, p.H, p.Hkv, p.N);
    if (tid == 0) {
        for (int i = 0; i < PEX; ++i) mbar_init(bars + i, 1);
        mbar_init(bars + PEX, 128); mbar_init(bars + PEU, 128);
        *abort_flag = (smem_u32(smem) & 1023u) ? 1 : 0;
        fence_mbar_init();
    }
    if (warp == 4) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_wait_tma();
    const uint32_t tmem = uniform(*tmem_slot);
    constexpr uint32_t kColX = 0, kColU = 128;      // x~ at 0, U of the two slabs at 128 and 256
    if (*abort_flag) { if (tid == 0) atomicExch(p.status, (int)DARKATTN_ERR_CUDA); }
    else if (warp == 4) {
        if (t1 > t0) {
            auto load_k = [&](int t) {
                const int b = (t - t0) & 1;
                mbar_expect_tx(bars + PB_K0 + b, kTile);
                for (int a = 0; a < D / 64; ++a) tma_load_2d(sK + b * kTile + a * 16384, &p.mapK, bars + PB_K0 + b, a * 64, rowk0 + t * 128);
            };
            if (elect_one()) {
                mbar_expect_tx(bars + PB_M, kTile * (1 + ns));
                for (int a = 0; a < D / 64; ++a) {
                    tma_load_2d(sM + a * 16384, &p.mapM, bars + PB_M, a * 64, h * p.r);
                    for (int s = 0; s < ns; ++s) tma_load_2d(sOm + s * kTile + a * 16384, &p.mapOm, bars + PB_M, a * 64, h * p.m + (slab0 + s) * 128);
                }
                load_k(t0);
                if (t0 + 1 < t1) load_k(t0 + 1);
            }
            const TileDesc tM(sM), tOm0(sOm), tOm1(sOm + kTile), tK0(sK), tK1(sK + kTile);
            const uint32_t id_x = make_idesc(128, p.r, 0, 0), id_u = make_idesc(128, 128, 0, 0);
            bool ok = warp_wait(bars + PB_M, 0, p.status, abort_flag);
            for (int t = t0; t < t1 && ok; ++t) {
                const int i = t - t0, b = i & 1;
                const uint32_t ph = i & 1, phk = (i >> 1) & 1;
                const TileDesc &tK = b ? tK1 : tK0;
                ok = warp_wait(bars + PB_K0 + b, phk, p.status, abort_flag);
                if (ok && i > 0) ok = warp_wait(bars + PEX, ph ^ 1, p.status, abort_flag);       // x~ of the tile before has been read
                if (!ok) break;
                tc_fence_after();
                if (elect_one()) {
                    _Pragma("unroll") for (int k = 0; k < D / 16; ++k) mma_ss(tmem + kColX, kdesc(tK, k), kdesc(tM, k), id_x, k > 0);
                    mma_commit(bars + PMX);
                }
                if (i > 0) { ok = warp_wait(bars + PEU, ph ^ 1, p.status, abort_flag); if (!ok) break; }      // U of the tile before has been read
                tc_fence_after();
                if (elect_one()) {
                    _Pragma("unroll") for (int k = 0; k < D / 16; ++k) mma_ss(tmem + kColU, kdesc(tK, k), kdesc(tOm0, k), id_u, k > 0);
                    if (ns == 2)
                        _Pragma("unroll") for (int k = 0; k < D / 16; ++k) mma_ss(tmem + kColU + 128, kdesc(tK, k), kdesc(tOm1, k), id_u, k > 0);
                    mma_commit(bars + PMU);
                }
                if (t + 2 < t1) {       // this tile's buffer is free once its MMAs are done
                    ok = warp_wait(bars + PMU, ph, p.status, abort_flag);
                    if (!ok) break;
                    if (elect_one()) load_k(t + 2);
                }
            }
        }
    } else {
        const uint32_t lane_addr = tmem + ((uint32_t)(warp * 32) << 16);
        float best0 = -INFINITY, best1 = -INFINITY;
        bool ok = true;
        for (int t = t0; t < t1; ++t) {
            const uint32_t ph = (t - t0) & 1;
            ok = __all_sync(0xffffffffu, wait_or_abort(bars + PMX, ph, p.status, abort_flag));
            if (!ok) break;
            tc_fence_after();
            float acc = 0.f;
            for (int c0 = 0; c0 < p.r; c0 += 16) {
                uint32_t v[16];
                tmem_ld16(lane_addr + kColX + c0, v);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 16; ++j) { const float x = __uint_as_float(v[j]); acc = fmaf(x, x, acc); }
            }
            tc_fence_before();
            mbar_arrive(bars + PEX);
            const float nk = p.coef * acc;
            if (pair == 0) p.nK[(size_t)bh * p.N + (size_t)t * 128 + tid] = nk;
            ok = __all_sync(0xffffffffu, wait_or_abort(bars + PMU, ph, p.status, abort_flag));
            if (!ok) break;
            tc_fence_after();
            float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
            for (int c0 = 0; c0 < 128; c0 += 32) {
                uint32_t v[32];
                tmem_ld32(lane_addr + kColU + c0, v);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 32; ++j) mx0 = fmaxf(mx0, __uint_as_float(v[j]));
            }
            if (ns == 2) {
#pragma unroll
                for (int c0 = 0; c0 < 128; c0 += 32) {
                    uint32_t v[32];
                    tmem_ld32(lane_addr + kColU + 128 + c0, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 32; ++j) mx1 = fmaxf(mx1, __uint_as_float(v[j]));
                }
            }
            tc_fence_before();
            mbar_arrive(bars + PEU);
            best0 = fmaxf(best0, mx0 - nk);
            best1 = fmaxf(best1, mx1 - nk);
        }
        if (ok && t1 > t0) {
            for (int o = 16; o; o >>= 1) {
                best0 = fmaxf(best0, __shfl_xor_sync(0xffffffffu, best0, o));
                best1 = fmaxf(best1, __shfl_xor_sync(0xffffffffu, best1, o));
            }
            if ((tid & 31) == 0) {
                atomicMax(p.cs + bh * p.nslab + slab0, float_order_key(best0 - kShiftHeadroom));
                if (ns == 2) atomicMax(p.cs + bh * p.nslab + slab0 + 1, float_order_key(best1 - kShiftHeadroom));
            }
        }
    }
    if (*abort_flag) __nanosleep(200000);
    tc_fence_before();
    __syncthreads();
    if (warp == 4) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------ the main kernel
struct MainParams {
    CUtensorMap mapQ, mapK, mapV, mapOm, mapOml, mapSb, mapPN;
    CUtensorMap mapSst;  // causal, when stash_S: S before every chunk as [BH*T*m, dv] bf16, for the backward pass
    CUtensorMap mapBf;   // causal, when stash_S: the key features as [BH*N, m] bf16, for the backward pass
    int stash_S;
    const float *nK;     // [BH, N]      key norms in log2 units
    const float *cs;     // [BH, nslab]  key-side shift per slab (log2 units)
    float *pdr;          // [nslab, BH*N, 8]  partial normalisers of the four column groups (0..3), exponent the partial is scaled by (4)
    // Key pass: sums over all keys, [BH, m, DV] and [BH, m, 4 parts]; with segments (npiece > 0) the states of the pieces,
    // [BH, npiece, m, DV] and [BH, npiece, m, 4].
    float *Sacc, *zacc;
    const float *zq;     // [BH, m]  z for the query pass
    // causal scan cut into nsplit segments of the sequence: the causal kernel of segment s > 0 starts from the state
    // before it, Sseg[bh, s] and zseg[bh, s] ([BH, nsplit, ...]; the bf16 copy comes through mapSb).
    const float *Sseg, *zseg;
    int npiece;          // pieces the key pass cuts the nsplit - 1 segments of a (batch, head) into, 0 without segments
    float *zc;           // causal: z before chunk t for the backward pass, [BH, T, m] (row 0 not written)
    int *status;
    int N, H, Hkv, BH, m, nslab, T, nsplit;
    // Sum of the slabs beside the causal scan (done != null): slabs that have stored a tile's rows, [BH, T]; the CTAs from
    // scan_ctas on add them up and normalise.
    int *done;
    int scan_ctas, cut;  // cut: chunks of each segment that are summed there (the kernel behind sums the rest)
    const __nv_bfloat16 *pnum;
    __nv_bfloat16 *O;
    float2 *sv;
};

enum { MODE_CAUSAL = 0, MODE_KEYS = 1, MODE_QUERIES = 2 };

// ------------------------------------------------------------------ causal forward kernel
// 16 epilogue warps (warp w: TMEM lanes 32 (w % 4) .. +31, columns 32 (w / 4) .. +31), one control warp whose first lane issues
// the TMA loads and the MMAs, and one that stores the output. phi(Q) and the masked kernel tile P are only ever the A operand of an
// MMA whose rows are tokens, so they are packed to bf16 in tensor memory and read by the MMA from there; phi(K) also serves
// transposed and as a B operand and goes to shared memory. (The passes over keys and queries further down have roles of their own.)

__device__ __forceinline__ void store_row_f32x32_bf16(const uint32_t (&v)[32], unsigned char *tile, int row, int col0)
{
#pragma unroll
    for (int q = 0; q < 4; ++q) *reinterpret_cast<uint4 *>(tile_chunk(tile, row, col0 / 8 + q)) = pack8(v + 8 * q);
}

// phi(Q) of one row segment: row maximum over the slab's 128 features (exchanged with the three other warps
// of the lane quarter through red[4][128]), 2^(u - max) packed to bf16 into TMEM columns fq + col0/2.
// rmax receives the row maximum. Returns sum_l phi(Q)_l z_l over the segment.
__device__ __forceinline__ float query_features_to_tmem(uint32_t u_addr, uint32_t fq_addr, float *red, const float *z, int q4,
                                                        int g, int r, int col0, float &rmax)
{
    uint32_t v[32], pk[16];
    tmem_ld32(u_addr + col0, v);
    tmem_wait_ld();
    float mx = -INFINITY;
#pragma unroll
    for (int j = 0; j < 32; ++j) mx = fmaxf(mx, __uint_as_float(v[j]));
    red[g * 128 + r] = mx;
    quarter_sync(q4);
    rmax = fmaxf(fmaxf(red[r], red[128 + r]), fmaxf(red[256 + r], red[384 + r]));
    float dz = 0.f;
#pragma unroll
    for (int j = 0; j < 32; j += 2) {
        const float f0 = ex2f(__uint_as_float(v[j]) - rmax), f1 = ex2f(__uint_as_float(v[j + 1]) - rmax);
        const float2 zz = *reinterpret_cast<const float2 *>(z + col0 + j);
        dz = fmaf(f0, zz.x, dz);
        dz = fmaf(f1, zz.y, dz);
        pk[j / 2] = pack_bf16(f0, f1);
    }
    tmem_st16(fq_addr + col0 / 2, pk);
    tmem_wait_st();
    return dz;
}

// (u0, u1) - (n0, n1) - (c, c)
__device__ __forceinline__ void sub2(float &u0, float &u1, float n0, float n1, float c)
{
    asm("{\n\t.reg .b64 a, b, m, d;\n\t"
        "mov.b64 a, {%0, %1};\n\tmov.b64 b, {%2, %3};\n\tmov.b64 d, {%4, %4};\n\tmov.b64 m, {%5, %5};\n\t"
        "fma.rn.f32x2 a, b, m, a;\n\t"
        "fma.rn.f32x2 a, d, m, a;\n\t"
        "mov.b64 {%0, %1}, a;\n\t}"
        : "+f"(u0), "+f"(u1) : "f"(n0), "f"(n1), "f"(c), "f"(-1.f));
}
// 32 rows of the output by one warp: O[row,:] = sum_s num_s[row,:] 2^(rho_s - rho) / sum_s den_s 2^(rho_s - rho),
// rho = max_s rho_s; den_s is the sum of the slab's four partial normalisers. Lane l forms row l's weights; DV / 8 lanes read a
// row, 16 bytes each. The partial rows were written by other SMs a moment ago and come out of L2 (__ldcg: never from this SM's
// L1); what bounds this is that latency, so all loads (up to 16 per lane) are issued before anything is used. The combined
// normaliser and rho are also written to sv for the backward pass; a normaliser that is zero or not finite is reported.
template <int DV, int NS>
__device__ __forceinline__ void combine_rows32_n(const MainParams &p, long long row0, int lane)
{
    const long long rows = (long long)p.BH * p.N, own = row0 + lane;
    constexpr int LPR = DV / 8, RI = 32 / LPR, NIT = 32 / RI;      // lanes of a row, rows and rounds
    constexpr int KS = NS > 0 ? NS : 1, UN = NS > 0 ? (16 / KS < NIT ? 16 / KS : NIT) : 1;      // rounds in flight together
    const int c0 = (lane % LPR) * 8, rl = lane / LPR;
    const __nv_bfloat16 *src = p.pnum + (row0 + rl) * DV + c0;
    __nv_bfloat16 *dst = p.O + (row0 + rl) * DV + c0;
    float rho = -INFINITY, den = 0.f, w[KS];
    float4 d4[KS];
    if constexpr (NS > 0) {
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const float *q = p.pdr + 8 * (s * rows + own);
            d4[s] = __ldcg(reinterpret_cast<const float4 *>(q));
            w[s] = __ldcg(q + 4);
        }
    }
    for (int i0 = 0; i0 < NIT; i0 += UN) {
        uint4 raw[UN][KS];
        if constexpr (NS > 0) {
#pragma unroll
            for (int u = 0; u < UN; ++u)
#pragma unroll
                for (int s = 0; s < NS; ++s) raw[u][s] = __ldcg(reinterpret_cast<const uint4 *>(src + (s * rows + (i0 + u) * RI) * DV));
        }
        if (i0 == 0) {
            if constexpr (NS > 0) {
#pragma unroll
                for (int s = 0; s < NS; ++s) rho = fmaxf(rho, w[s]);
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    w[s] = exp2f(w[s] - rho);
                    den = fmaf((d4[s].x + d4[s].y) + (d4[s].z + d4[s].w), w[s], den);
                }
            } else {
                for (int s = 0; s < p.nslab; ++s) rho = fmaxf(rho, __ldcg(p.pdr + 8 * (s * rows + own) + 4));
                for (int s = 0; s < p.nslab; ++s) {
                    const float *q = p.pdr + 8 * (s * rows + own);
                    const float4 x = __ldcg(reinterpret_cast<const float4 *>(q));
                    den = fmaf((x.x + x.y) + (x.z + x.w), exp2f(__ldcg(q + 4) - rho), den);
                }
            }
            p.sv[own] = make_float2(den, rho);
            if (!(den > 0.f) || !isfinite(den)) atomicCAS(p.status, 0, (int)DARKATTN_ERR_NONFINITE);
        }
        const float inv = 1.f / den;
#pragma unroll
        for (int u = 0; u < UN; ++u) {
            const int r = (i0 + u) * RI + rl;
            const float ir = __shfl_sync(0xffffffffu, inv, r), rr = __shfl_sync(0xffffffffu, rho, r);
            float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
            auto add = [&](const uint4 &x, float ws) {
                float f[8];
                unpack8(x, f);
#pragma unroll
                for (int k = 0; k < 8; k += 2) fma2(acc[k], acc[k + 1], f[k], f[k + 1], ws, ws);
            };
            if constexpr (NS > 0) {
#pragma unroll
                for (int s = 0; s < NS; ++s) add(raw[u][s], __shfl_sync(0xffffffffu, w[s], r));
            } else {
                for (int s = 0; s < p.nslab; ++s)
                    add(__ldcg(reinterpret_cast<const uint4 *>(src + (s * rows + (i0 + u) * RI) * DV)), exp2f(__ldcg(p.pdr + 8 * (s * rows + row0 + r) + 4) - rr));
            }
            uint4 out;
            out.x = pack_bf16(acc[0] * ir, acc[1] * ir); out.y = pack_bf16(acc[2] * ir, acc[3] * ir);
            out.z = pack_bf16(acc[4] * ir, acc[5] * ir); out.w = pack_bf16(acc[6] * ir, acc[7] * ir);
            *reinterpret_cast<uint4 *>(dst + (i0 + u) * RI * DV) = out;
        }
    }
}
template <int DV>
__device__ __forceinline__ void combine_rows32(const MainParams &p, long long row0, int lane)
{
    if (p.nslab == 1) combine_rows32_n<DV, 1>(p, row0, lane);
    else if (p.nslab == 2) combine_rows32_n<DV, 2>(p, row0, lane);
    else if (p.nslab == 4) combine_rows32_n<DV, 4>(p, row0, lane);
    else combine_rows32_n<DV, 0>(p, row0, lane);
}
// A CTA that adds up the slabs beside the scan: groups of four warps take the tiles in the order in which the scan reaches them
// and wait for all slabs of a tile to be stored. (These CTAs come last in the grid and the scan never waits for them.) One SM
// gets 47 GB/s of rows through this; a ring filled by bulk copies did not help (the copies alone, without the sums, ran at 35).
template <int DV>
__device__ void sum_tiles(const MainParams &p)
{
    pdl_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, quarter = warp & 3;
    const int groups = (blockDim.x / 128) * (gridDim.x - p.scan_ctas), g0 = (blockIdx.x - p.scan_ctas) * (blockDim.x / 128) + warp / 4;
    if (warp / 4 >= blockDim.x / 128) return;
    const int lines = p.BH * p.nsplit;
    for (long long k = g0; k < (long long)lines * p.cut; k += groups) {
        const int i = (int)(k / lines), bh = (int)(k % lines) / p.nsplit, seg = (int)(k % lines) % p.nsplit;
        const int t = (int)((long long)p.T * seg / p.nsplit) + i;
        if (t >= (int)((long long)p.T * (seg + 1) / p.nsplit)) continue;
        const int *flag = p.done + (size_t)bh * p.T + t;
        bool ok = true;
        const unsigned long long t0 = global_timer_ns();
        for (;;) {
            int v;
            asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
            if (v >= p.nslab) break;
            const int st = *reinterpret_cast<volatile int *>(p.status);
            if (st == 5 /* DARKATTN_ERR_TIMEOUT */ || st == (int)DARKATTN_ERR_CUDA || global_timer_ns() - t0 > kWaitLimitNs) { ok = false; break; }
            __nanosleep(500);
        }
        if (!__all_sync(0xffffffffu, ok)) {
            if (lane == 0) atomicCAS(p.status, 0, 5 /* DARKATTN_ERR_TIMEOUT */);
            return;
        }
        combine_rows32<DV>(p, (long long)bh * p.N + t * 128 + 32 * quarter, lane);
    }
}

template <int D, int DV>
struct FwdCausalSmem {
    static constexpr int kOm = 0;                          // folded projections of the slab, rounded    [128 l, D]
    static constexpr int kOml = kOm + 128 * D * 2;         // ... and what the rounding left out         [128 l, D]
    static constexpr int kQ = kOml + 128 * D * 2;
    static constexpr int kK = kQ + 128 * D * 2;
    static constexpr int kV = kK + 128 * D * 2;
    static constexpr int kFK = kV + 128 * DV * 2;          // phi(K)                              [128, 128]
    static constexpr int kSb = kFK + 32768;                // bf16 copy of the state              [128 l, DV]
    static constexpr int kRed = kSb + 128 * DV * 2;        // float[4][128]: row maxima exchanged between the warps of a row;
                                                           // mid-chunk the same 2 KB hold the ones operand of z += phi(K)^T 1
    static constexpr int kZ = kRed + 2048;                 // z_prev, float[128]
    static constexpr int kBars = kZ + 512;
    static constexpr int kTotal = kBars + 256;
};

// TMEM columns of the causal kernel: state S at 0 (DV), four partial sums of z at 128 (16 each: consecutive MMAs of
// z += phi(K)^T 1 go to different ones, so that none has to wait for the one before), packed phi(Q) at 192 (64),
// R1 at 256, R2 at 384.
constexpr uint32_t kColS = 0, kColZ = 128, kColFQ = 192, kColR1 = 256, kColR2 = 384;

// 16 epilogue warps, the control warp, the warp that stores the output
constexpr int kCausalThreads = 576;

enum CBars { CB_OM, CB_Q, CB_K, CB_V, CB_ST, CM1, CM2, CM3, CMS, CM4, CE0, CE1, CE2, CE3, CE4, CNBARS };

// Causal: one CTA per (b, h, slab) walks the chunks of the sequence.
//   R1: U_Q -> (phi(Q) read) -> P = phi(Q) phi(K)^T -> packed tril(P) (A operand of P V) -> U_Q of the next chunk
//   R2: U_K -> (phi(K) read) -> O = phi(Q) S_prev + P V -> (O read) -> U_K of the next chunk
// The epilogue warps work in this order: phi(K) of chunk t; the bf16 copy of the state through chunk t - 1 (while P
// runs); tril(P); the output tile and z; phi(Q) of chunk t + 1 (both projections of the next chunk are issued behind
// the output MMAs and run while the output is read). The state tile's buffer doubles as the staging tile of the
// output's TMA store: between the output MMAs of chunk t and the copy of the state through chunk t nobody reads it. One thread
// of another warp issues that store, so that waiting for it does not hold up the MMAs; where the slabs are summed beside the
// scan (p.done) it then counts the tile.
template <int D, int DV>
__global__ void __launch_bounds__(kCausalThreads, 1) tc_fwd_causal_kernel(const __grid_constant__ MainParams p)
{
    using L = FwdCausalSmem<D, DV>;
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char *sOm = smem + L::kOm, *sOml = smem + L::kOml, *sQ = smem + L::kQ, *sK = smem + L::kK, *sV = smem + L::kV;
    unsigned char *sFK = smem + L::kFK, *sSb = smem + L::kSb;
    float *sZ = reinterpret_cast<float *>(smem + L::kZ), *sRed = reinterpret_cast<float *>(smem + L::kRed);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L::kBars);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + CNBARS);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(bars + CNBARS + 1);

    const int tid = threadIdx.x, warp = uniform(tid >> 5);
    if (blockIdx.x >= p.scan_ctas) {                // (takes no tensor memory)
        sum_tiles<DV>(p);
        return;
    }
    const int unit = blockIdx.x / p.nsplit, seg = blockIdx.x % p.nsplit;
    const int bh = unit / p.nslab, slab = unit % p.nslab, h = bh % p.H;
    const int row0 = bh * p.N;
    const int tbeg = (int)((long long)p.T * seg / p.nsplit), tend = (int)((long long)p.T * (seg + 1) / p.nsplit);
    const bool fresh = (seg == 0);                 // the scan state starts at zero (else at the segment's prefix state)
    // the state through the segment's last chunk is also copied (and stored) when the backward pass will start the
    // next segment from it
    const bool copy_last = p.stash_S && tend < p.T;

    if (tid == 0) {
        for (int i = 0; i < CE0; ++i) mbar_init(bars + i, 1);
        for (int i = CE0; i < CNBARS; ++i) mbar_init(bars + i, kEpiWarps);
        *abort_flag = (smem_u32(smem) & 1023u) ? 1 : 0;
        fence_mbar_init();
    }
    if (warp == kEpiWarps) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_wait_tma();
    const uint32_t tmem = uniform(*tmem_slot);
    if (tid < 128) sZ[tid] = fresh ? 0.f : p.zseg[((size_t)bh * p.nsplit + seg) * p.m + slab * 128 + tid];      // (read after the barrier below)
    int *status = p.status;
    if (!fresh && warp < kEpiWarps) {      // the segment's prefix state into the fp32 accumulators in TMEM
        const int lane = tid & 31, q4 = warp & 3, col0 = (warp >> 2) * 32, r = q4 * 32 + lane;
        const uint32_t lane_addr = tmem + ((uint32_t)(q4 * 32) << 16);
        const size_t srow = ((size_t)bh * p.nsplit + seg) * p.m + slab * 128 + r;
        if (col0 < DV) {
            uint32_t v[32];
            const float4 *src = reinterpret_cast<const float4 *>(p.Sseg + srow * DV + col0);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float4 x = src[j];
                v[4 * j] = __float_as_uint(x.x); v[4 * j + 1] = __float_as_uint(x.y);
                v[4 * j + 2] = __float_as_uint(x.z); v[4 * j + 3] = __float_as_uint(x.w);
            }
            tmem_st32(lane_addr + kColS + col0, v);
        }
        {       // z: the prefix into the first partial sum, zero into the three others (one per column group's warp)
            uint32_t v[16];
            const uint32_t zv = (col0 == 0) ? __float_as_uint(p.zseg[srow]) : 0u;
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = zv;
            tmem_st16(lane_addr + kColZ + (col0 / 32) * 16, v);
        }
        tmem_wait_st();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    if (*abort_flag) {
        if (tid == 0) atomicExch(status, (int)DARKATTN_ERR_CUDA);
    } else if (tend <= tbeg) {
    } else if (warp == kEpiWarps) {
        {
            const int rowk0 = kv_row0(bh, p.H, p.Hkv, p.N);       // K and V may be shared by a group of query heads
            auto load_tile = [&](unsigned char *dst, const CUtensorMap *map, uint64_t *bar, int width, int t) {
                const int base = (map == &p.mapQ) ? row0 : rowk0;
                if (elect_one()) {
                    mbar_expect_tx(bar, 128 * width * 2);
                    for (int a = 0; a < width / 64; ++a) tma_load_2d(dst + a * 16384, map, bar, a * 64, base + t * 128);
                }
            };
            auto store_state = [&](int t) {        // the bf16 state before chunk t, for the backward pass
                if (elect_one()) {
                    for (int a = 0; a < DV / 64; ++a) tma_store_2d(&p.mapSst, sSb + a * 16384, a * 64, (bh * p.T + t) * p.m + slab * 128);
                    tma_store_commit();
                }
            };
            const TileDesc tOm(sOm), tOml(sOml), tQ(sQ), tK(sK), tV(sV), tFK(sFK), tSb(sSb);
            const uint64_t ones_desc = make_sdesc(smem_u32(sRed), 16384, 1024);
            const uint32_t id_kk = make_idesc(128, 128, 0, 0);
            const uint32_t id_o = make_idesc(128, DV, 0, 1);
            const uint32_t id_s = make_idesc(128, DV, 1, 1);
            const uint32_t id_z = make_idesc(128, 16, 1, 1);
            const uint32_t R1 = tmem + kColR1, R2 = tmem + kColR2, FQ = tmem + kColFQ;

            if (elect_one()) {
                mbar_expect_tx(bars + CB_OM, 2 * 128 * D * 2 + (fresh ? 0 : 128 * DV * 2));
                for (int a = 0; a < D / 64; ++a) {
                    tma_load_2d(sOm + a * 16384, &p.mapOm, bars + CB_OM, a * 64, h * p.m + slab * 128);
                    tma_load_2d(sOml + a * 16384, &p.mapOml, bars + CB_OM, a * 64, h * p.m + slab * 128);
                }
                if (!fresh)     // bf16 copy of the segment's prefix state
                    for (int a = 0; a < DV / 64; ++a)
                        tma_load_2d(sSb + a * 16384, &p.mapSb, bars + CB_OM, a * 64, (bh * p.nsplit + seg) * p.m + slab * 128);
            }
            load_tile(sQ, &p.mapQ, bars + CB_Q, D, tbeg);
            load_tile(sK, &p.mapK, bars + CB_K, D, tbeg);
            load_tile(sV, &p.mapV, bars + CB_V, DV, tbeg);

#define CWAIT(b, q) do { ok = warp_wait(bars + (b), (q), status, abort_flag); } while (0)
            bool ok = true;
            CWAIT(CB_OM, 0);
            if (ok) CWAIT(CB_Q, 0);
            if (ok) {
                tc_fence_after();
                if (elect_one()) {
                    issue_projection<D>(R1, tQ, tOm, tOml, id_kk);                                                // U_Q of the first chunk
                    mma_commit(bars + CM1);
                }
                CWAIT(CB_K, 0);
            }
            if (ok) {
                tc_fence_after();
                if (elect_one()) {
                    issue_projection<D>(R2, tK, tOm, tOml, id_kk);                                                // U_K of the first chunk
                    mma_commit(bars + CM2);
                }
                CWAIT(CE0, 0);                                                  // phi(Q) packed, Q tile consumed
            }
            if (ok && tbeg + 1 < tend) load_tile(sQ, &p.mapQ, bars + CB_Q, D, tbeg + 1);
            for (int t = tbeg; t < tend && ok; ++t) {
                const uint32_t ph = (t - tbeg) & 1;
                const bool first = (t == tbeg) && fresh, last = (t + 1 == tend);
                CWAIT(CE1, ph); if (!ok) break;                                 // phi(K) and the ones in smem, R2 read, K tile consumed
                if (!last) load_tile(sK, &p.mapK, bars + CB_K, D, t + 1);
                if (p.stash_S && elect_one()) {         // the backward kernels read the key features back instead of forming them again
                    tma_store_2d(&p.mapBf, sFK, slab * 128, row0 + t * 128);
                    tma_store_2d(&p.mapBf, sFK + 16384, slab * 128 + 64, row0 + t * 128);
                    tma_store_commit();
                }
                tc_fence_after();
                if (elect_one()) {
                    _Pragma("unroll") for (int k = 0; k < 8; ++k) mma_ts(R1, FQ + k * 8, kdesc(tFK, k), id_kk, k > 0);            // P = phi(Q) phi(K)^T
                    mma_commit(bars + CM3);
                }
                if (!first) {
                    if (t > tbeg) {                                             // the bf16 state through chunk t - 1 is in smem
                        CWAIT(CE4, ph ^ 1); if (!ok) break;
                        if (p.stash_S) store_state(t);
                    }
                    if (elect_one())
                        _Pragma("unroll") for (int k = 0; k < 8; ++k) mma_ts(R2, FQ + k * 8, mndesc(tSb, k), id_o, k > 0);        // O = phi(Q) S_prev
                }
                if (elect_one())
                    _Pragma("unroll") for (int k = 0; k < 8; ++k)                                                                 // z += phi(K)^T 1
                        mma_ss(tmem + kColZ + 16 * (k & 3), mndesc(tFK, k), ones_desc, id_z, (!first) || k >= 4);
                CWAIT(CB_V, ph); if (!ok) break;
                CWAIT(CE2, ph); if (!ok) break;                                 // tril(P) packed in R1
                tc_fence_after();
                if (elect_one()) {
                    _Pragma("unroll") for (int k = 0; k < 8; ++k) mma_ts(R2, R1 + k * 8, mndesc(tV, k), id_o, (!first) || k > 0); // O += P V
                    if (p.stash_S) tma_store_wait_read();   // the stash copies of the state before this chunk and of phi(K) have left their tiles: the output may be
                                                            // staged in the first, the next phi(K) written to the second
                    mma_commit(bars + CM4);
                }
                if (!last) {        // U_Q of the next chunk, while the epilogue warps read the output tile out
                    CWAIT(CB_Q, ph ^ 1); if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        issue_projection<D>(R1, tQ, tOm, tOml, id_kk);
                        mma_commit(bars + CM1);
                    }
                }
                if (elect_one()) {
                    _Pragma("unroll") for (int k = 0; k < 8; ++k) mma_ss(tmem + kColS, mndesc(tFK, k), mndesc(tV, k), id_s, (!first) || k > 0);   // S += phi(K)^T V
                    mma_commit(bars + CMS);
                }
                CWAIT(CE3, ph); if (!ok) break;                                 // the output tile has been read out of R2 and staged
                if (!last) {
                    CWAIT(CB_K, ph ^ 1); if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        issue_projection<D>(R2, tK, tOm, tOml, id_kk);                                            // U_K of the next chunk
                        mma_commit(bars + CM2);
                    }
                }
                CWAIT(CMS, ph); if (!ok) break;                                 // V tile consumed
                if (!last) {
                    load_tile(sV, &p.mapV, bars + CB_V, DV, t + 1);
                    CWAIT(CE0, ph ^ 1); if (!ok) break;                         // phi(Q) of the next chunk packed, its Q tile consumed
                    if (t + 2 < tend) load_tile(sQ, &p.mapQ, bars + CB_Q, D, t + 2);
                }
            }
            if (ok && copy_last) {      // the state through the segment's last chunk: what the backward pass starts the next segment from
                CWAIT(CE4, (tend - 1 - tbeg) & 1);
                if (ok) store_state(tend);
            }
#undef CWAIT
            if (elect_one()) tma_store_wait_all();
        }
    } else if (warp == kEpiWarps + 1) {
        if ((tid & 31) == 0) {
            const int prow0 = (slab * p.BH + bh) * p.N;
            for (int t = tbeg; t < tend; ++t) {     // this slab's part of the output rows of chunk t, staged in the state tile's buffer
                if (!wait_or_abort(bars + CE3, (t - tbeg) & 1, status, abort_flag)) break;
                for (int a = 0; a < DV / 64; ++a) tma_store_2d(&p.mapPN, sSb + a * 16384, a * 64, prow0 + t * 128);
                tma_store_commit();
                if (t + 1 < tend || copy_last) { tma_store_wait_read(); mbar_arrive(bars + CB_ST); }     // it has left the state tile's buffer
                if (p.done && t - tbeg < p.cut) {       // the rows and (written before the arrivals on CE3) their normalisers are visible to who sees the count
                    tma_store_wait_all();
                    asm volatile("fence.proxy.async;" ::: "memory");
                    __threadfence();
                    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(p.done + (size_t)bh * p.T + t) : "memory");
                }
            }
            tma_store_wait_all();
        }
    } else {
        const int lane = tid & 31, q4 = warp & 3, g = warp >> 2, col0 = g * 32;
        const int r = q4 * 32 + lane;
        const uint32_t lane_addr = tmem + ((uint32_t)(q4 * 32) << 16);
        const uint32_t R1 = lane_addr + kColR1, R2 = lane_addr + kColR2;
        const float cshift = load_key_shift(p.cs, bh * p.nslab + slab);
        const size_t prow0 = ((size_t)slab * p.BH + bh) * p.N;
        uint32_t *sOnes = reinterpret_cast<uint32_t *>(sRed);
        bool ok = true;
        float rmax = 0.f;                           // row maximum of the chunk whose phi(Q) was formed last
// A wait that gave up (here or, seen through the abort flag, in another warp) switches the warp to a dry run: it skips
// every later wait but keeps walking the same chunks, so that every named barrier below still gets all its arrivals and
// no warp is left waiting for one that has gone (what it reads and writes from then on is garbage; the status word says so).
#define EWAIT(b, q) do { ok = ok && __all_sync(0xffffffffu, wait_or_abort(bars + (b), (q), status, abort_flag)); } while (0)
        // phi(K): once the four warps of these rows are done with the exchanged maxima the array is filled with bf16 ones,
        // the B operand of z += phi(K)^T 1
        auto key_features = [&](float nk) {
            tc_fence_after();
            quarter_sync(q4);
            sOnes[g * 128 + r] = 0x3F803F80u;
            features_to_tile(R2 + col0, nk, sFK, r, col0);
            fence_async_smem();
            tc_fence_before();
            mbar_arrive_warp(bars + CE1);
        };
        float dz = 0.f;                             // phi(Q) z_prev over this thread's features, of the chunk whose phi(Q) was formed last
        auto query_features = [&]() {
            tc_fence_after();
            dz = query_features_to_tmem(R1, lane_addr + kColFQ, sRed, sZ, q4, g, r, col0, rmax);
            tc_fence_before();
            mbar_arrive_warp(bars + CE0);
        };
        // the state through chunk t as the bf16 operand of phi(Q) S, once the staged output of chunk t has left the tile
        auto copy_state = [&](int t) {
            const uint32_t q = (t - tbeg) & 1;
            EWAIT(CB_ST, q);
            EWAIT(CMS, q);
            tc_fence_after();
            if (col0 < DV) tmem_row_to_tile(lane_addr + kColS + col0, sSb, r, col0);
            fence_async_smem();
            tc_fence_before();
            mbar_arrive_warp(bars + CE4);
        };
        EWAIT(CM1, 0);
        query_features();
        float nk_next = p.nK[(size_t)row0 + (size_t)tbeg * 128 + r] + cshift;
        for (int t = tbeg; t < tend; ++t) {
            const uint32_t ph = (t - tbeg) & 1;
            const bool last = (t + 1 == tend);
            const size_t prow = prow0 + (size_t)t * 128 + r;
            const float nk = nk_next;
            if (!last) nk_next = p.nK[(size_t)row0 + (size_t)(t + 1) * 128 + r] + cshift;     // needed a chunk from now

            EWAIT(CM2, ph);
            key_features(nk);
            if (t > tbeg) copy_state(t - 1);                // while P runs

            EWAIT(CM3, ph);
            tc_fence_after();
            float rowsum = 0.f;
            {
                uint32_t v[32], pk[16];
                tmem_ld32(R1 + col0, v);
                tmem_wait_ld();
                quarter_sync(q4);                   // every column group has read P before anyone overwrites it
#pragma unroll
                for (int j = 0; j < 32; j += 2) {
                    const float x0 = (col0 + j <= r) ? __uint_as_float(v[j]) : 0.f;
                    const float x1 = (col0 + j + 1 <= r) ? __uint_as_float(v[j + 1]) : 0.f;
                    rowsum += x0 + x1;
                    pk[j / 2] = pack_bf16(x0, x1);
                }
                tmem_st16(R1 + col0 / 2, pk);
                tmem_wait_st();
            }
            tc_fence_before();
            mbar_arrive_warp(bars + CE2);

            EWAIT(CM4, ph);         // the output tile; z through this chunk (its MMAs ran ahead of the output's)
            tc_fence_after();
            if (col0 < DV) {
                uint32_t v[32];
                tmem_ld32(R2 + col0, v);
                tmem_wait_ld();
                store_row_f32x32_bf16(v, sSb, r, col0);
            }
            if (g == 0 && t + 1 < p.T) {            // (also after a segment's last chunk: the next segment's backward needs it)
                const uint32_t z0 = tmem_ld1(lane_addr + kColZ), z1 = tmem_ld1(lane_addr + kColZ + 16);
                const uint32_t z2 = tmem_ld1(lane_addr + kColZ + 32), z3 = tmem_ld1(lane_addr + kColZ + 48);
                tmem_wait_ld();
                const float zv = (__uint_as_float(z0) + __uint_as_float(z1)) + (__uint_as_float(z2) + __uint_as_float(z3));
                sZ[r] = zv;
                p.zc[((size_t)bh * p.T + t + 1) * p.m + slab * 128 + r] = zv;
            }
            p.pdr[8 * prow + g] = rowsum + dz;
            if (g == 0) p.pdr[8 * prow + 4] = rmax + cshift;
            fence_async_smem();
            tc_fence_before();
            mbar_arrive_warp(bars + CE3);
            epi_sync();                             // every z is in place before anyone forms the next chunk's phi(Q)

            if (!last) {
                EWAIT(CM1, ph ^ 1);
                query_features();
            }
        }
        if (copy_last) copy_state(tend - 1);
#undef EWAIT
    }
    if (*abort_flag) __nanosleep(200000);   // error path only: let copies and MMAs in flight drain
    tc_fence_before();
    __syncthreads();
    if (warp == kEpiWarps) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------ key pass: S = phi(K)^T V, z = phi(K)^T 1
// Both passes below run one CTA per SM over a list of pieces (a run of tiles of one (batch, head, slab)); the roles (a warp
// for TMA, warps for the MMAs, the read-out warps) walk the list by themselves, so that one piece's end overlaps the next
// one's start except where the slab's operands change. CTA i works on slab i % nslab, and the line of all (batch, head, tile)
// is cut evenly over the CTAs of a slab: those of different slabs go through the same tiles at the same time and share them
// through L2 (with the slabs one after the other in one line, K and V came from HBM once for each: 537 MB, 82 us of the 104
// the key pass then took at 4 x 16 heads, 8192 tokens, d 128). The states of a line's pieces are added up by atomics; with
// segments (causal) the pieces are fixed and each stores its own state.
struct Piece { int bh, slab, t0, t1, dst; bool whole; };

struct PieceList {
    long long x, end;       // line: tiles [x, end); fixed pieces: index and count
    __device__ __forceinline__ explicit PieceList(const MainParams &p)
    {
        if (p.npiece) { x = blockIdx.x; end = (long long)p.BH * p.nslab * p.npiece; }
        else {
            const int j = blockIdx.x / p.nslab, per = gridDim.x / p.nslab;
            const long long total = (long long)p.BH * p.T;
            x = total * j / per; end = total * (j + 1) / per;
        }
    }
    __device__ __forceinline__ bool next(const MainParams &p, Piece &c)
    {
        if (x >= end) return false;
        if (p.npiece) {
            const int per = p.npiece / (p.nsplit - 1);           // pieces of a segment; the last segment's state is not needed
            c.slab = (int)(x % p.nslab); c.dst = (int)(x / p.nslab % p.npiece); c.bh = (int)(x / p.nslab / p.npiece);
            const int seg = c.dst / per, j = c.dst % per;
            const int b0 = (int)((long long)p.T * seg / p.nsplit), len = (int)((long long)p.T * (seg + 1) / p.nsplit) - b0;
            c.t0 = b0 + (int)((long long)len * j / per); c.t1 = b0 + (int)((long long)len * (j + 1) / per);
            c.whole = true;
            x += gridDim.x;
        } else {
            c.slab = blockIdx.x % p.nslab; c.bh = (int)(x / p.T); c.t0 = (int)(x % p.T); c.dst = 0;
            c.t1 = (int)min((long long)p.T, c.t0 + (end - x));
            c.whole = (c.t0 == 0 && c.t1 == p.T);
            x += c.t1 - c.t0;
        }
        return true;
    }
};

// 16 read-out warps, TMA, MMAs of the projections, MMAs of the second product (a warp each: a thread that issues both kinds
// spends its program order waiting for the one while the other is ready); the key pass has a second TMA warp
constexpr int kPassThreads = 608, kKeysThreads = 640;

// untiled copy of a multiple of 16 bytes (both addresses 16-byte aligned) into shared memory
__device__ __forceinline__ void bulk_load(void *smem_dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(smem_dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void red_add4(float *dst, float a, float b, float c, float d)
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

template <int D, int DV>
struct FwdKeysSmem {
    static constexpr int kNormSlots = 8;       // see the loader: a slot is loaded again long after its tile has been read out
    static constexpr int kFixed = 2 * 128 * D * 2 + kNormSlots * 512 + 512;
    static constexpr int kStages = (kFixed + 4 * 128 * (D + DV) * 2 <= 232448) ? 4 : 2;
    static constexpr int kOm = 0;
    static constexpr int kOml = kOm + 128 * D * 2;
    static constexpr int kK = kOml + 128 * D * 2;
    static constexpr int kV = kK + kStages * 128 * D * 2;
    static constexpr int kNorm = kV + kStages * 128 * DV * 2;
    static constexpr int kBars = kNorm + kNormSlots * 512;
    static constexpr int kTotal = kBars + 512;
};

// Omega loaded / free; K, V rings loaded / free; norms loaded; U ready / state updated / phi(K)^T written (three regions);
// piece's state ready / read
enum KyBars { YB_OM, YB_OMF, YB_K, YB_V = YB_K + 4, YB_KF = YB_V + 4, YB_VF = YB_KF + 4, YB_N = YB_VF + 4, YB_U = YB_N + 8, YB_SD = YB_U + 3, YB_S = YB_SD + 3,
              YB_E, YB_SR = YB_E + 3, YNBARS };

// The tile's exponents are formed transposed, U^T = Omega K^T: a lane of tensor memory is a feature, a column a token. Then
// phi(K)^T, packed to bf16 in place by the warp that read it, is the A operand of S += phi(K)^T V straight from tensor memory
// (no shared-memory tile, no proxy fence), z is a sum along a thread's own columns (no MMAs against ones), and what is left of
// tensor memory holds three tiles: the projections run ahead and eight warps each work on the even and on the odd tiles, so
// that the exponentials of one tile run under the waits, loads and stores of another (in lockstep on one tile a warp spent 1.0 k
// of 2.3 k cycles on those). Bound by the exponentials (16384 per tile, 16 per clock and SM) at d = 64 and by MMA issue (24 per tile)
// at d = 128. Encoder shape 8 x 12 heads, 4096 tokens, d 64, m 256: 101 -> 51 us; 4 x 16 heads, 8192 tokens, d 128: 138 -> 88 us.
template <int D, int DV>
__global__ void __launch_bounds__(kKeysThreads, 1) tc_fwd_keys_kernel(const __grid_constant__ MainParams p)
{
    using L = FwdKeysSmem<D, DV>;
    extern __shared__ __align__(1024) unsigned char smem[];
    constexpr int kXT = 128 * D * 2, kVT = 128 * DV * 2, NST = L::kStages, NN = L::kNormSlots;
    unsigned char *sOm = smem + L::kOm, *sOml = smem + L::kOml, *sK = smem + L::kK, *sV = smem + L::kV;
    float *sNorm = reinterpret_cast<float *>(smem + L::kNorm);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L::kBars);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + YNBARS);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(bars + YNBARS + 1);
    const int tid = threadIdx.x, warp = uniform(tid >> 5);

    if (tid == 0) {
        for (int i = 0; i < YB_E; ++i) mbar_init(bars + i, 1);
        for (int i = YB_E; i < YB_SR; ++i) mbar_init(bars + i, kEpiWarps / 2);
        mbar_init(bars + YB_SR, kEpiWarps);
        *abort_flag = (smem_u32(smem) & 1023u) ? 1 : 0;
        fence_mbar_init();
    }
    if (warp == kEpiWarps) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_wait_tma();
    const uint32_t tmem = uniform(*tmem_slot);
    int *status = p.status;
    PieceList list(p);
    Piece c;

    if (*abort_flag) {
        if (tid == 0) atomicExch(status, (int)DARKATTN_ERR_CUDA);
    } else if (warp == kEpiWarps) {                     // ---- loads
        {
            bool ok = true;
            int it = 0;
            for (int pc = 0; ok && list.next(p, c); ++pc) {
                const int bh = c.bh, slab = c.slab, h = bh % p.H, rowk0 = kv_row0(bh, p.H, p.Hkv, p.N);
                const float *nK = p.nK + (size_t)bh * p.N;
                if (pc > 0) ok = warp_wait(bars + YB_OMF, (pc - 1) & 1, status, abort_flag);      // the piece before is projected
                if (!ok) break;
                if (elect_one()) mbar_expect_tx(bars + YB_OM, 2 * kXT);
                if (elect_one())
                    for (int a = 0; a < D / 64; ++a) {
                        tma_load_2d(sOm + a * 16384, &p.mapOm, bars + YB_OM, a * 64, h * p.m + slab * 128);
                        tma_load_2d(sOml + a * 16384, &p.mapOml, bars + YB_OM, a * 64, h * p.m + slab * 128);
                    }
                for (int t = c.t0; t < c.t1; ++t, ++it) {
                    const int b = it % NST, y = rowk0 + t * 128;
                    if (it >= NST) ok = warp_wait(bars + YB_KF + b, (it / NST - 1) & 1, status, abort_flag);
                    if (!ok) break;
                    if (elect_one()) {
                        mbar_expect_tx(bars + YB_K + b, kXT);
                        for (int a = 0; a < D / 64; ++a) tma_load_2d(sK + b * kXT + a * 16384, &p.mapK, bars + YB_K + b, a * 64, y);
                        // Here tile it - NST is projected, so its region's tile before, it - NST - 3, has been read out, and with it
                        // all tiles before, tile it - 8 (the last user of this slot of norms) among them.
                        static_assert(NST + 3 <= NN, "a slot of norms would be loaded over");
                        mbar_expect_tx(bars + YB_N + it % NN, 512);
                        bulk_load(sNorm + (it % NN) * 128, nK + (size_t)t * 128, 512, bars + YB_N + it % NN);
                        if (NST == 2 && t + 2 < c.t1)        // with a short ring the next loads come out of L2
                            for (int a = 0; a < D / 64; ++a) tma_prefetch_l2_2d(&p.mapK, a * 64, y + 256);
                    }
                }
            }
        }
    } else if (warp == kEpiWarps + 2) {                 // ---- loads of V, whose tiles are held two steps longer than those of K
        {
            bool ok = true;
            int it = 0;
            while (ok && list.next(p, c)) {
                const int rowk0 = kv_row0(c.bh, p.H, p.Hkv, p.N);
                for (int t = c.t0; t < c.t1; ++t, ++it) {
                    const int b = it % NST, y = rowk0 + t * 128;
                    if (it >= NST) ok = warp_wait(bars + YB_VF + b, (it / NST - 1) & 1, status, abort_flag);
                    if (!ok) break;
                    if (elect_one()) {
                        mbar_expect_tx(bars + YB_V + b, kVT);
                        for (int a = 0; a < DV / 64; ++a) tma_load_2d(sV + b * kVT + a * 16384, &p.mapV, bars + YB_V + b, a * 64, y);
                        if (NST == 2 && t + 2 < c.t1)
                            for (int a = 0; a < DV / 64; ++a) tma_prefetch_l2_2d(&p.mapV, a * 64, y + 256);
                    }
                }
            }
        }
    } else if (warp == kEpiWarps + 1) {                 // ---- MMAs: U^T of tile it into region it % 3
        {
            const TileDesc tOm(sOm), tOml(sOml);
            const uint32_t id_u = make_idesc(128, 128, 0, 0);
            bool ok = true;
            int it = 0;
            for (int pc = 0; ok && list.next(p, c); ++pc) {
                ok = warp_wait(bars + YB_OM, pc & 1, status, abort_flag);
                for (int t = c.t0; t < c.t1; ++t, ++it) {
                    const int b = it % NST, q = it % 3;
                    ok = ok && warp_wait(bars + YB_K + b, (it / NST) & 1, status, abort_flag);
                    if (ok && it >= 3) ok = warp_wait(bars + YB_SD + q, (it / 3 - 1) & 1, status, abort_flag);      // the region's last reader is done
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t dst = tmem + 128 + 128 * q;
                    const TileDesc tK(sK + b * kXT);
                    if (elect_one()) {
                        _Pragma("unroll") for (int k = 0; k < D / 16; ++k) mma_ss(dst, kdesc(tOm, k), kdesc(tK, k), id_u, k > 0);
                        _Pragma("unroll") for (int k = 0; k < D / 16; ++k) mma_ss(dst, kdesc(tOml, k), kdesc(tK, k), id_u, 1);
                        mma_commit(bars + YB_U + q);
                        mma_commit(bars + YB_KF + b);
                        if (t + 1 == c.t1) mma_commit(bars + YB_OMF);
                    }
                }
            }
        }
    } else if (warp == kEpiWarps + 3) {                 // ---- MMAs: S += phi(K)^T V
        {
            const uint32_t id_s = make_idesc(128, DV, 0, 1);
            bool ok = true;
            int it = 0;
            for (int pc = 0; ok && list.next(p, c); ++pc) {
                if (pc > 0) ok = warp_wait(bars + YB_SR, (pc - 1) & 1, status, abort_flag);      // the state before has been read out
                for (int t = c.t0; t < c.t1; ++t, ++it) {
                    const int b = it % NST, q = it % 3;
                    ok = ok && warp_wait(bars + YB_V + b, (it / NST) & 1, status, abort_flag);
                    ok = ok && warp_wait(bars + YB_E + q, (it / 3) & 1, status, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t src = tmem + 128 + 128 * q;
                    const TileDesc tV(sV + b * kVT);
                    if (elect_one()) {
                        _Pragma("unroll") for (int k = 0; k < 8; ++k) mma_ts(tmem, src + (k / 2) * 32 + (k % 2) * 8, mndesc(tV, k), id_s, t > c.t0 || k > 0);
                        mma_commit(bars + YB_SD + q);
                        mma_commit(bars + YB_VF + b);
                    }
                }
                if (ok && elect_one()) mma_commit(bars + YB_S);
            }
        }
    } else {                                            // ---- read-out
        const int lane = tid & 31, q4 = warp & 3, g = warp >> 2, col0 = g * 32;
        const int r = q4 * 32 + lane;                   // this thread's feature
        const int grp = warp >> 3, half = 64 * ((warp >> 2) & 1);     // even or odd tiles; which 64 tokens of the tile
        const uint32_t lane_addr = tmem + ((uint32_t)(q4 * 32) << 16);
        bool ok = true;
        int it = 0;
        for (int pc = 0; ok && list.next(p, c); ++pc) {
            const int bh = c.bh, slab = c.slab;
            const float cshift = load_key_shift(p.cs, bh * p.nslab + slab);
            float z0 = 0.f, z1 = 0.f;
            for (int t = c.t0; t < c.t1; ++t, ++it) {
                if ((it & 1) != grp) continue;
                const uint32_t addr = lane_addr + 128 + 128 * (it % 3) + half;
                ok = wait_or_abort(bars + YB_N + it % NN, (it / NN) & 1, status, abort_flag) &&
                     wait_or_abort(bars + YB_U + it % 3, (it / 3) & 1, status, abort_flag);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int c0 = 0; c0 < 64; c0 += 32) {
                    uint32_t v[32], pk[16];
                    tmem_ld32(addr + c0, v);
                    const float4 *nrm = reinterpret_cast<const float4 *>(sNorm + (it % NN) * 128 + half + c0);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float4 nk = nrm[j];
                        float x[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k) x[k] = __uint_as_float(v[4 * j + k]);
                        sub2(x[0], x[1], nk.x, nk.y, cshift);
                        sub2(x[2], x[3], nk.z, nk.w, cshift);
                        pk[2 * j] = pack_bf16(ex2f(x[0]), ex2f(x[1]));
                        pk[2 * j + 1] = pack_bf16(ex2f(x[2]), ex2f(x[3]));
                        // z sums what the MMA multiplies: the rounded features
                        add2(z0, z1, __uint_as_float(pk[2 * j] << 16), __uint_as_float(pk[2 * j] & 0xffff0000u));
                        add2(z0, z1, __uint_as_float(pk[2 * j + 1] << 16), __uint_as_float(pk[2 * j + 1] & 0xffff0000u));
                    }
                    tmem_st16(addr + c0, pk);
                }
                tmem_wait_st();
                tc_fence_before();
                mbar_arrive_warp(bars + YB_E + it % 3);
            }
            if (!ok) break;
            ok = __all_sync(0xffffffffu, wait_or_abort(bars + YB_S, pc & 1, status, abort_flag));
            if (!ok) break;
            tc_fence_after();
            const size_t srow = ((size_t)bh * (p.npiece ? p.npiece : 1) + c.dst) * p.m + slab * 128 + r;
            uint32_t v[32];
            if (col0 < DV) {
                tmem_ld32(lane_addr + col0, v);
                tmem_wait_ld();
            }
            tc_fence_before();
            mbar_arrive_warp(bars + YB_SR);
            if (col0 < DV) {
                float *dst = p.Sacc + srow * DV + col0;
#pragma unroll
                for (int j = 0; j < 32; j += 4) {
                    const float a0 = __uint_as_float(v[j]), a1 = __uint_as_float(v[j + 1]), a2 = __uint_as_float(v[j + 2]), a3 = __uint_as_float(v[j + 3]);
                    if (c.whole) *reinterpret_cast<float4 *>(dst + j) = make_float4(a0, a1, a2, a3);
                    else red_add4(dst + j, a0, a1, a2, a3);
                }
            }
            // z: a part per (tile parity, token half), added up by the kernel that reads the state
            if (c.whole) p.zacc[4 * srow + g] = z0 + z1;
            else atomicAdd(p.zacc + 4 * srow + g, z0 + z1);
        }
    }
    if (*abort_flag) __nanosleep(200000);
    tc_fence_before();
    __syncthreads();
    if (warp == kEpiWarps) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------ non-causal, query pass: partial O = phi(Q) S, den = phi(Q) z
template <int D, int DV>
struct FwdQueriesSmem {
    static constexpr int kGroups = DV == 64 ? 4 : 3;       // groups of four warps, each with a tile of its own in flight
    static constexpr int kStg = kGroups * 4 * 4096;        // a warp's staging: 32 rows of 64 columns
    static constexpr int kFixed = 2 * 128 * D * 2 + 128 * DV * 2 + kStg + 512 + 512;
    static constexpr int kStages = (kFixed + 4 * 128 * D * 2 <= 232448) ? 4 : 2;
    static constexpr int kOm = 0;
    static constexpr int kOml = kOm + 128 * D * 2;
    static constexpr int kQ = kOml + 128 * D * 2;
    static constexpr int kSb = kQ + kStages * 128 * D * 2; // bf16 state of the slab [128 l, DV]
    static constexpr int kStage = kSb + 128 * DV * 2;
    static constexpr int kZ = kStage + kStg;
    static constexpr int kBars = kZ + 512;
    static constexpr int kTotal = kBars + 512;
};

// operands of the slab loaded / free; Q ring loaded / free; U ready, O ready, phi(Q) written, O read (per group)
enum QyBars { UB_OM, UB_OMF, UB_Q, UB_QF = UB_Q + 4, UB_U = UB_QF + 4, UB_O = UB_U + 4, UB_E = UB_O + 4, UB_R = UB_E + 4, UNBARS = UB_R + 4 };

// A tile belongs to a group of four warps, a thread to a row: the row's maximum, its normaliser and its output row need no
// exchange with another warp, and the groups work on different tiles (three or four in flight), so that one's exponentials
// run under another's waits. Tensor memory: dv = 64: per group U (128 columns), phi(Q) packed into its first 64 in place, O into
// the other 64; dv = 128: per group U and then O (128), phi(Q) in one of two 64-column slots. Bound like the key pass.
// Encoder shape (see there) 103 -> 53 us; 4 x 16 heads, 8192 tokens, d 128: 170 -> 117 us.
template <int D, int DV>
__global__ void __launch_bounds__(kPassThreads, 1) tc_fwd_queries_kernel(const __grid_constant__ MainParams p)
{
    using L = FwdQueriesSmem<D, DV>;
    extern __shared__ __align__(1024) unsigned char smem[];
    constexpr int kXT = 128 * D * 2, NST = L::kStages, G = L::kGroups;
    unsigned char *sOm = smem + L::kOm, *sOml = smem + L::kOml, *sQ = smem + L::kQ, *sSb = smem + L::kSb;
    const float *sZ = reinterpret_cast<const float *>(smem + L::kZ);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L::kBars);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + UNBARS);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(bars + UNBARS + 1);
    const int tid = threadIdx.x, warp = uniform(tid >> 5);

    if (tid == 0) {
        for (int i = 0; i < UB_E; ++i) mbar_init(bars + i, 1);
        for (int i = UB_E; i < UNBARS; ++i) mbar_init(bars + i, 4);
        *abort_flag = (smem_u32(smem) & 1023u) ? 1 : 0;
        fence_mbar_init();
    }
    if (warp == kEpiWarps) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_wait_tma();
    const uint32_t tmem = uniform(*tmem_slot);
    int *status = p.status;
    PieceList list(p);
    Piece c;
    // tensor-memory columns of tile it: U; packed phi(Q); O
    auto col_u = [](int it) { return (uint32_t)(128 * (it % G)); };
    auto col_f = [&](int it) { return DV == 64 ? col_u(it) : (uint32_t)(384 + 64 * (it & 1)); };
    auto col_o = [&](int it) { return DV == 64 ? col_u(it) + 64 : col_u(it); };

    if (*abort_flag) {
        if (tid == 0) atomicExch(status, (int)DARKATTN_ERR_CUDA);
    } else if (warp == kEpiWarps) {                     // ---- loads
        {
            bool ok = true;
            int it = 0;
            for (int pc = 0; ok && list.next(p, c); ++pc) {
                const int bh = c.bh, slab = c.slab, h = bh % p.H;
                if (pc > 0) ok = warp_wait(bars + UB_OMF, (pc - 1) & 1, status, abort_flag);     // the piece before is done with its operands
                if (!ok) break;
                if (elect_one()) mbar_expect_tx(bars + UB_OM, 2 * kXT + 128 * DV * 2 + 512);
                if (elect_one())
                    for (int a = 0; a < D / 64; ++a) {
                        tma_load_2d(sOm + a * 16384, &p.mapOm, bars + UB_OM, a * 64, h * p.m + slab * 128);
                        tma_load_2d(sOml + a * 16384, &p.mapOml, bars + UB_OM, a * 64, h * p.m + slab * 128);
                    }
                if (elect_one()) {
                    for (int a = 0; a < DV / 64; ++a) tma_load_2d(sSb + a * 16384, &p.mapSb, bars + UB_OM, a * 64, bh * p.m + slab * 128);
                    bulk_load(smem + L::kZ, p.zq + (size_t)bh * p.m + slab * 128, 512, bars + UB_OM);
                }
                for (int t = c.t0; t < c.t1; ++t, ++it) {
                    const int b = it % NST, y = bh * p.N + t * 128;
                    if (it >= NST) ok = warp_wait(bars + UB_QF + b, (it / NST - 1) & 1, status, abort_flag);
                    if (!ok) break;
                    if (elect_one()) {
                        mbar_expect_tx(bars + UB_Q + b, kXT);
                        for (int a = 0; a < D / 64; ++a) tma_load_2d(sQ + b * kXT + a * 16384, &p.mapQ, bars + UB_Q + b, a * 64, y);
                        if (NST == 2 && t + 2 < c.t1)
                            for (int a = 0; a < D / 64; ++a) tma_prefetch_l2_2d(&p.mapQ, a * 64, y + 256);
                    }
                }
            }
        }
    } else if (warp == kEpiWarps + 1) {                 // ---- MMAs: U of a tile
        {
            const TileDesc tOm(sOm), tOml(sOml);
            const uint32_t id_u = make_idesc(128, 128, 0, 0);
            bool ok = true;
            int it = 0;
            for (int pc = 0; ok && list.next(p, c); ++pc) {
                ok = warp_wait(bars + UB_OM, pc & 1, status, abort_flag);
                for (int t = c.t0; t < c.t1; ++t, ++it) {
                    const int b = it % NST;
                    ok = ok && warp_wait(bars + UB_Q + b, (it / NST) & 1, status, abort_flag);
                    if (ok && it >= G) ok = warp_wait(bars + UB_R + it % G, (it / G - 1) & 1, status, abort_flag);      // the group's last output has been read
                    if (!ok) break;
                    tc_fence_after();
                    const TileDesc tQ(sQ + b * kXT);
                    if (elect_one()) {
                        issue_projection<D>(tmem + col_u(it), tQ, tOm, tOml, id_u);
                        mma_commit(bars + UB_U + it % G);
                        mma_commit(bars + UB_QF + b);
                    }
                }
            }
        }
    } else if (warp == kEpiWarps + 2) {                 // ---- MMAs: O = phi(Q) S
        {
            const TileDesc tSb(sSb);
            const uint32_t id_o = make_idesc(128, DV, 0, 1);
            bool ok = true;
            int it = 0;
            for (int pc = 0; ok && list.next(p, c); ++pc) {
                ok = warp_wait(bars + UB_OM, pc & 1, status, abort_flag);
                for (int t = c.t0; t < c.t1; ++t, ++it) {
                    ok = ok && warp_wait(bars + UB_E + it % G, (it / G) & 1, status, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        _Pragma("unroll") for (int k = 0; k < 8; ++k) mma_ts(tmem + col_o(it), tmem + col_f(it) + 8 * k, mndesc(tSb, k), id_o, k > 0);
                        mma_commit(bars + UB_O + it % G);
                    }
                }
                if (ok && elect_one()) mma_commit(bars + UB_OMF);
            }
        }
    } else if (warp < 4 * G) {                          // ---- read-out
        const int lane = tid & 31, q4 = warp & 3, grp = warp >> 2;
        const uint32_t lane_addr = tmem + ((uint32_t)(q4 * 32) << 16);
        unsigned char *stage = smem + L::kStage + warp * 4096;
        bool ok = true;
        int it = 0;
        for (int pc = 0; ok && list.next(p, c); ++pc) {
            const int bh = c.bh, slab = c.slab;
            const float cshift = load_key_shift(p.cs, bh * p.nslab + slab);
            const size_t prow0 = ((size_t)slab * p.BH + bh) * p.N + q4 * 32;
            bool fresh = true;
            for (int t = c.t0; t < c.t1 && ok; ++t, ++it) {
                if (it % G != grp) continue;
                const uint32_t ph = (it / G) & 1;
                ok = wait_or_abort(bars + UB_U + grp, ph, status, abort_flag);
                if (ok && fresh) ok = wait_or_abort(bars + UB_OM, pc & 1, status, abort_flag);      // z is in place (the piece's first tile of this group)
                fresh = false;
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
                const uint32_t U = lane_addr + col_u(it), F = lane_addr + col_f(it), O = lane_addr + col_o(it);
                float rmax = -INFINITY;
#pragma unroll
                for (int c0 = 0; c0 < 128; c0 += 32) {
                    uint32_t v[32];
                    tmem_ld32(U + c0, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 32; ++j) rmax = fmaxf(rmax, __uint_as_float(v[j]));
                }
                if (DV == 128 && it >= 2) {            // the slot's last reader: the output MMAs of tile it - 2
                    ok = __all_sync(0xffffffffu, wait_or_abort(bars + UB_O + (it - 2) % G, ((it - 2) / G) & 1, status, abort_flag));
                    if (!ok) break;
                    tc_fence_after();
                }
                float d0 = 0.f, d1 = 0.f;
#pragma unroll
                for (int c0 = 0; c0 < 128; c0 += 32) {
                    uint32_t v[32], pk[16];
                    tmem_ld32(U + c0, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 32; j += 4) {
                        const float4 zz = *reinterpret_cast<const float4 *>(sZ + c0 + j);
                        const float f0 = ex2f(__uint_as_float(v[j]) - rmax), f1 = ex2f(__uint_as_float(v[j + 1]) - rmax);
                        const float f2 = ex2f(__uint_as_float(v[j + 2]) - rmax), f3 = ex2f(__uint_as_float(v[j + 3]) - rmax);
                        fma2(d0, d1, f0, f1, zz.x, zz.y);
                        fma2(d0, d1, f2, f3, zz.z, zz.w);
                        pk[j / 2] = pack_bf16(f0, f1);
                        pk[j / 2 + 1] = pack_bf16(f2, f3);
                    }
                    tmem_st16(F + c0 / 2, pk);
                }
                tmem_wait_st();
                tc_fence_before();
                mbar_arrive_warp(bars + UB_E + grp);
                const size_t prow = prow0 + (size_t)t * 128;
                float *dst = p.pdr + 8 * (prow + lane);
                *reinterpret_cast<float4 *>(dst) = make_float4(d0 + d1, 0.f, 0.f, 0.f);
                dst[4] = rmax + cshift;

                ok = __all_sync(0xffffffffu, wait_or_abort(bars + UB_O + grp, ph, status, abort_flag));
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int a = 0; a < DV / 64; ++a) {
                    if (lane == 0) tma_store_wait_read();       // what was staged before has left
                    __syncwarp();
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        uint32_t v[32];
                        tmem_ld32(O + 64 * a + 32 * half, v);
                        tmem_wait_ld();
                        if (a == DV / 64 - 1 && half == 1) {
                            tc_fence_before();
                            mbar_arrive_warp(bars + UB_R + grp);
                        }
#pragma unroll
                        for (int q = 0; q < 4; ++q) *reinterpret_cast<uint4 *>(stage + swz128(lane, 4 * half + q)) = pack8(v + 8 * q);
                    }
                    fence_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        tma_store_2d(&p.mapPN, stage, a * 64, (int)prow);
                        tma_store_commit();
                    }
                }
            }
        }
        if (lane == 0) tma_store_wait_all();
    }
    if (*abort_flag) __nanosleep(200000);
    tc_fence_before();
    __syncthreads();
    if (warp == kEpiWarps) tmem_dealloc(tmem, 512);
}

// Sb = bf16(S), the operand of the query pass, and z from its four parts, for that pass and for the backward pass
__global__ void __launch_bounds__(256) state_to_bf16_kernel(const float *S, __nv_bfloat16 *Sb, long long n4, const float *zparts, float *z, long long nz)
{
    pdl_wait();
    const long long i = blockIdx.x * 256LL + threadIdx.x;
    if (i < n4) {
        const float4 x = reinterpret_cast<const float4 *>(S)[i];
        reinterpret_cast<uint2 *>(Sb)[i] = make_uint2(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w));
    }
    if (i < nz) {
        const float4 x = reinterpret_cast<const float4 *>(zparts)[i];
        z[i] = (x.x + x.y) + (x.z + x.w);
    }
}

// The state before every segment but the first: Sseg[bh, s] = sum of the pieces of the segments before s (in fp32 and, as an
// MMA operand, in bf16), the same for z. One thread per four elements of a (batch, head)'s state; a segment's pieces are
// loaded together. (65536 tokens, 8 heads, m 512, d 64: 25 us when it prefixed in place, a load behind every store.)
__global__ void __launch_bounds__(256) segment_prefix_kernel(const float *__restrict__ Spart, const float *__restrict__ zpart, float *__restrict__ Sseg,
                                                             __nv_bfloat16 *__restrict__ Sb, float *__restrict__ zseg, int nseg, int npiece, int E4, int m, long long total)
{
    pdl_wait();
    const long long i = blockIdx.x * 256LL + threadIdx.x;
    if (i >= total) return;
    const long long bh = i / E4;
    const int e = (int)(i % E4), per = npiece / (nseg - 1);
    float4 run = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s = 1; s < nseg; ++s) {
        const float4 *src = reinterpret_cast<const float4 *>(Spart) + (bh * npiece + (s - 1) * per) * E4 + e;
#pragma unroll 4
        for (int j = 0; j < per; ++j) {
            const float4 x = src[(long long)j * E4];
            run.x += x.x; run.y += x.y; run.z += x.z; run.w += x.w;
        }
        const long long at = (bh * nseg + s) * E4 + e;
        reinterpret_cast<float4 *>(Sseg)[at] = run;
        reinterpret_cast<uint2 *>(Sb)[at] = make_uint2(pack_bf16(run.x, run.y), pack_bf16(run.z, run.w));
    }
    if (e < m) {
        float zr = 0.f;
        for (int s = 1; s < nseg; ++s) {
#pragma unroll 4
            for (int j = 0; j < per; ++j) {
                const float4 x = reinterpret_cast<const float4 *>(zpart)[(bh * npiece + (s - 1) * per + j) * m + e];
                zr += (x.x + x.y) + (x.z + x.w);
            }
            zseg[(bh * nseg + s) * m + e] = zr;
        }
    }
}

// O[row,:] = sum_s num_s[row,:] 2^(rho_s - rho) / sum_s den_s 2^(rho_s - rho), rho = max_s rho_s; den_s is the sum of
// the slab's four partial normalisers. One thread per 8 output columns. The combined normaliser and rho are also
// written to sv for the backward pass; a normaliser that is zero or not finite is reported through the status word.
// NS > 0: the number of slabs at compile time (all loads of a thread are issued before the first use).
template <int NS>
__global__ void combine_kernel(const __nv_bfloat16 *pnum, const float *pdr, __nv_bfloat16 *O, float2 *sv,
                               long long rows, int dv, int nslab_rt, int *status, int T, int nseg, int cut)
{
    pdl_wait();
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const int per_row = dv / 8, seg = blockIdx.y % nseg;
    // blockIdx.y: (batch, head) and segment of the sequence; the first `cut` chunks of a segment have been summed beside the scan
    const int t0 = (int)((long long)T * seg / nseg) + cut, t1 = (int)((long long)T * (seg + 1) / nseg);
    if (i >= (long long)(t1 - t0) * 128 * per_row) return;
    const long long row = ((long long)(blockIdx.y / nseg) * T + t0) * 128 + i / per_row;
    const int c0 = (int)(i % per_row) * 8;
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0}, den = 0.f, rho = -INFINITY;
    auto slab_den = [](const float4 &d4) { return (d4.x + d4.y) + (d4.z + d4.w); };
    if constexpr (NS > 0) {
        float4 d4[NS];
        float rh[NS];
        uint4 raw[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const float *q = pdr + 8 * ((size_t)s * rows + row);
            d4[s] = *reinterpret_cast<const float4 *>(q);
            rh[s] = q[4];
            raw[s] = *reinterpret_cast<const uint4 *>(pnum + ((size_t)s * rows + row) * dv + c0);
        }
#pragma unroll
        for (int s = 0; s < NS; ++s) rho = fmaxf(rho, rh[s]);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const float w = exp2f(rh[s] - rho);
            den = fmaf(slab_den(d4[s]), w, den);
            const __nv_bfloat162 *h2 = reinterpret_cast<const __nv_bfloat162 *>(&raw[s]);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 f = __bfloat1622float2(h2[q]);
                acc[2 * q] = fmaf(f.x, w, acc[2 * q]);
                acc[2 * q + 1] = fmaf(f.y, w, acc[2 * q + 1]);
            }
        }
    } else {
        for (int s = 0; s < nslab_rt; ++s) rho = fmaxf(rho, pdr[8 * ((size_t)s * rows + row) + 4]);
        for (int s = 0; s < nslab_rt; ++s) {
            const float *q = pdr + 8 * ((size_t)s * rows + row);
            const float w = exp2f(q[4] - rho);
            den = fmaf(slab_den(*reinterpret_cast<const float4 *>(q)), w, den);
            const uint4 raw = *reinterpret_cast<const uint4 *>(pnum + ((size_t)s * rows + row) * dv + c0);
            const __nv_bfloat162 *h2 = reinterpret_cast<const __nv_bfloat162 *>(&raw);
#pragma unroll
            for (int q2 = 0; q2 < 4; ++q2) {
                const float2 f = __bfloat1622float2(h2[q2]);
                acc[2 * q2] = fmaf(f.x, w, acc[2 * q2]);
                acc[2 * q2 + 1] = fmaf(f.y, w, acc[2 * q2 + 1]);
            }
        }
    }
    if (c0 == 0) {
        sv[row] = make_float2(den, rho);
        if (!(den > 0.f) || !isfinite(den)) atomicCAS(status, 0, (int)DARKATTN_ERR_NONFINITE);
    }
    const float inv = 1.f / den;
    uint4 out;
    out.x = pack_bf16(acc[0] * inv, acc[1] * inv); out.y = pack_bf16(acc[2] * inv, acc[3] * inv);
    out.z = pack_bf16(acc[4] * inv, acc[5] * inv); out.w = pack_bf16(acc[6] * inv, acc[7] * inv);
    *reinterpret_cast<uint4 *>(O + (size_t)row * dv + c0) = out;
}

size_t take(size_t &off, size_t bytes)
{
    const size_t at = off;
    off += (bytes + 255) / 256 * 256;
    return at;
}

template <int D, int DV, int MODE>
cudaError_t launch_main(const MainParams &P, int grid, cudaStream_t st)
{
    if constexpr (MODE == MODE_CAUSAL) {
        using L = FwdCausalSmem<D, DV>;
        static_assert(L::kTotal <= 232448, "shared memory budget of one CTA exceeded");
        return launch_pdl(tc_fwd_causal_kernel<D, DV>, dim3(grid), dim3(kCausalThreads), L::kTotal, st, P);
    } else if constexpr (MODE == MODE_KEYS) {
        using L = FwdKeysSmem<D, DV>;
        static_assert(L::kTotal <= 232448, "shared memory budget of one CTA exceeded");
        return launch_pdl(tc_fwd_keys_kernel<D, DV>, dim3(grid), dim3(kKeysThreads), L::kTotal, st, P);
    } else {
        using L = FwdQueriesSmem<D, DV>;
        static_assert(L::kTotal <= 232448, "shared memory budget of one CTA exceeded");
        return launch_pdl(tc_fwd_queries_kernel<D, DV>, dim3(grid), dim3(kPassThreads), L::kTotal, st, P);
    }
}

template <int MODE>
cudaError_t launch_main_shape(int d, int dv, const MainParams &P, int grid, cudaStream_t st)
{
    if (d == 64 && dv == 64) return launch_main<64, 64, MODE>(P, grid, st);
    if (d == 128 && dv == 128) return launch_main<128, 128, MODE>(P, grid, st);
    if (d == 64 && dv == 128) return launch_main<64, 128, MODE>(P, grid, st);
    if (d == 128 && dv == 64) return launch_main<128, 64, MODE>(P, grid, st);
    return cudaErrorInvalidValue;
}

}  // namespace

// Shapes the tensor kernels cover: bf16, d and dv in {64, 128}, m and N multiples of 128, chunk 128,
// r a multiple of 16 up to 128.
bool tensor_supported(const darkattn_plan_s *plan)
{
    const Dims &D = plan->dims;
    if (!D.bf16) return false;
    if (!(D.d == 64 || D.d == 128) || !(D.dv == 64 || D.dv == 128)) return false;
    if (D.m % 128 || D.m < 128 || D.N % 128) return false;
    if (D.r % 16 || D.r < 16 || D.r > 128) return false;
    if (D.causal && D.C != 128) return false;
    if ((long long)D.BH * D.N * (D.m / 128) >= (1ll << 31)) return false;
    return true;
}

void tensor_make_layout(darkattn_plan_s *plan)
{
    const Dims &D = plan->dims;
    TensorLayout &Y = plan->tensor;
    const size_t BH = D.BH, N = D.N, m = D.m, d = D.d, dv = D.dv;
    Y.nslab = D.m / 128;
    Y.T = D.N / 128;
    int nsplit = 1;
    const long long units = (long long)BH * Y.nslab;
    if (D.causal && units * 2 <= 148) {
        // few long sequences: cut each into segments (a key pass computes the segment states, the causal
        // kernels of all segments then run side by side), as many as fill the SMs, at least 4 chunks each
        nsplit = (int)(148 / units);
        if (nsplit > Y.T / 4) nsplit = Y.T / 4;
        if (nsplit > 16) nsplit = 16;
        if (nsplit < 1) nsplit = 1;
    }
    Y.nsplit = nsplit;
    // the key pass over all segments but the last, in pieces that fill the SMs (a tile takes 0.8 us, a piece's start and end 3)
    Y.npiece = nsplit > 1 ? (nsplit - 1) * pick_splits(units * (nsplit - 1), Y.T / nsplit, 0.8, 3.0, 8) : 0;
    const size_t nstate = D.causal ? (size_t)nsplit : 1;
    size_t off = 0;
    Y.status = take(off, 256);
    Y.Om = take(off, (size_t)D.H * m * d * 2);
    Y.Oml = take(off, (size_t)D.H * m * d * 2);
    Y.cs = take(off, BH * Y.nslab * 4);
    Y.nK = take(off, BH * N * 4);
    Y.pnum = take(off, (size_t)Y.nslab * BH * N * dv * 2);
    Y.pdr = take(off, (size_t)Y.nslab * BH * N * 32);
    // (states and z of the key pass: sums over all keys, or one per piece; what it adds into is cleared by one run of stores)
    Y.Sacc = take(off, BH * (D.causal ? (size_t)Y.npiece : 1) * m * dv * 4);
    Y.zacc = take(off, BH * (D.causal ? (size_t)Y.npiece : 1) * m * 16);
    Y.done = take(off, BH * (size_t)Y.T * 4);
    Y.Sb = take(off, BH * nstate * m * dv * 2);
    Y.Sseg = take(off, Y.npiece ? BH * nstate * m * dv * 4 : 0);
    Y.zseg = take(off, Y.npiece ? BH * nstate * m * 4 : 0);
    Y.zq = take(off, D.causal ? 0 : BH * m * 4);
    Y.sv = take(off, BH * N * 8);
    Y.zc = take(off, D.causal ? BH * (size_t)Y.T * m * 4 : 0);
    // The causal scan may leave SMs idle, which can add up the slabs meanwhile: 47 GB/s of rows read and written per SM, against
    // 3.6 us (d 64) or 4.2 us (d 128) for a chunk of the scan; of every segment as many chunks as they manage in that time, and not
    // many more CTAs than it takes. 4 x 16 heads, 8192 tokens, d 128, forward calls in a row with 0, 0.5, 0.7, 0.85, 1.0, 1.15, 1.4 of that rate: with a
    // stash 550, 518, 508, 500, 492, 522, 577 us, without 477, 449, 435, 428, 430, 456, 512. Without -> with these sums, no stash: 131 -> 119
    // (2048 tokens), 759 -> 683 (8 heads, 65536 tokens, d 64, m 512), 179 -> 163 (48 heads, 4096 tokens, d 64); with a stash 145 -> 133, 812 -> 740,
    // 189 -> 171. The surplus of 1.6: the same as with all idle SMs (163, 683), and with 1.0 the last tiles are waited for (163 -> 172, with a
    // stash 171 -> 181). Not for scans of fewer than 8 chunks, nor where they would sum less than a fifth.
    const long long scan_ctas = units * nsplit, idle = 148 - scan_ctas;
    Y.summers = Y.cut = 0;
    if (D.causal && Y.T / nsplit >= 8 && idle > 0) {
        const double part = idle * 47e3 * (d == 64 ? 3.6 : 4.2) / ((double)BH * nsplit * (Y.nslab + 1) * 256.0 * dv);
        if (part >= 1.0) { Y.cut = (Y.T + nsplit - 1) / nsplit; Y.summers = (int)(part > 1.6 ? idle * 1.6 / part : idle); if (Y.summers < 1) Y.summers = 1; }
        else if (part >= 0.2) { Y.cut = (int)(part * (Y.T / nsplit)); Y.summers = (int)idle; }
    }
    plan->launches_fwd = (D.causal ? (nsplit > 1 ? 6 : 4) : 6) - (Y.cut >= (Y.T + nsplit - 1) / nsplit ? 1 : 0);
    {
        size_t so = 0;
        Y.sv_sv = take(so, BH * N * 8);
        Y.sv_nK = take(so, BH * N * 4);
        Y.sv_Om = take(so, (size_t)D.H * m * d * 2);
        Y.sv_Oml = take(so, (size_t)D.H * m * d * 2);
        Y.sv_cs = take(so, BH * Y.nslab * 4);
        Y.sv_zc = take(so, D.causal ? BH * (size_t)Y.T * m * 4 : 0);
        Y.sv_Sb = take(so, D.causal ? 0 : BH * m * dv * 2);
        Y.sv_zt = take(so, D.causal ? 0 : BH * m * 4);
        Y.sv_Sst = take(so, D.causal ? BH * (size_t)Y.T * m * dv * 2 : 0);
        Y.sv_Bphi = take(so, D.causal ? BH * N * m * 2 : 0);
        Y.sv_bytes = so;
        plan->saved_bytes = so;
    }
    // backward pass
    Y.Oscr = take(off, BH * N * dv * 2);
    Y.delta = take(off, BH * N * 4);
    Y.rhoc = take(off, D.causal ? BH * (size_t)Y.T * m * 4 : 0);
    Y.espart = take(off, (size_t)4 * Y.nslab * BH * N * 4);
    Y.Tacc = take(off, (size_t)D.H * m * d * 4);
    Y.dMn = take(off, (size_t)D.H * D.r * d * 4);
    Y.dKh = take(off, D.G > 1 ? BH * N * d * 2 : 0);
    Y.dVh = take(off, D.G > 1 ? BH * N * dv * 2 : 0);
    Y.Sst = take(off, D.causal ? BH * (size_t)Y.T * m * dv * 2 : 0);
    Y.Ahat = take(off, D.causal ? BH * N * m * 2 : 0);
    Y.Bphi = take(off, D.causal ? BH * N * m * 2 : 0);
    Y.Racc = take(off, D.causal ? 0 : BH * m * dv * 4);
    Y.rhot = take(off, D.causal ? 0 : BH * m * 4);
    Y.Rb = take(off, D.causal ? 0 : BH * m * dv * 2);
    // with `saved`; without it the forward launches come on top. Causal: delta, two scan kernels, dK finishing, the
    // dM product and the small kernel that adds the norm term's part; non-causal: one more for the rounding of R
    // between the two passes. (With per-kernel timing on, dM is one kernel.)
    plan->launches_bwd = (D.causal ? 6 : 7) + (D.G > 1 ? 2 : 0);      // (+ the two sums over the groups of query heads)
    Y.total_bytes = off;
    plan->workspace_bytes = Y.total_bytes;
}

cudaError_t tensor_prologue(const darkattn_plan_s *plan, const void *K, const void *M, const void *W, char *ws,
                            const Stash &out, cudaStream_t st)
{
    const Dims &D = plan->dims;
    const TensorLayout &Y = plan->tensor;
    const size_t BH = D.BH, N = D.N;
    PrepassParams PP;
    memset(&PP, 0, sizeof(PP));
    const size_t BHkv = (size_t)D.B * D.Hkv;
    if (!make_map(&PP.mapK, K, BHkv * N, D.d, 128) || !make_map(&PP.mapM, M, (size_t)D.H * D.r, D.d, 128) ||
        !make_map(&PP.mapOm, out.Om, (size_t)D.H * D.m, D.d, 128))
        return cudaErrorInvalidValue;
    cudaError_t e = cudaSuccess;
    auto keep = [&](cudaError_t x) { if (x != cudaSuccess && e == cudaSuccess) e = x; };
    timer_mark(plan, st, "fold_omega_kernel");
    // (S and z sums of the non-causal key pass and the counts of the tiles' slabs: adjacent, multiples of 256 bytes)
    const size_t zero_at = D.causal ? Y.done : Y.Sacc;
    float4 *zero = reinterpret_cast<float4 *>(ws + zero_at);
    const long long nzero = (long long)((Y.Sb - zero_at) / 16);
    int *status = reinterpret_cast<int *>(ws + Y.status), *cs = reinterpret_cast<int *>(out.cs);
    const int ncs = (int)(BH * Y.nslab);
    const dim3 fold_grid(D.m / 16, D.H);
    keep(launch_pdl(D.d == 64 ? fold_omega_kernel<2> : fold_omega_kernel<4>, fold_grid, dim3(128), 0, st, (const __nv_bfloat16 *)W, (const __nv_bfloat16 *)M,
                    out.Om, out.Oml, D.m, D.r, D.w_per_head, kLog2e * D.s, cs, ncs, status, zero, nzero));

    // key norms and key-side shifts in one pass over K
    PP.nK = out.nK; PP.cs = reinterpret_cast<int *>(out.cs); PP.status = reinterpret_cast<int *>(ws + Y.status);
    PP.N = D.N; PP.H = D.H; PP.Hkv = D.Hkv; PP.T = Y.T; PP.m = D.m; PP.r = D.r; PP.nslab = Y.nslab; PP.npair = (Y.nslab + 1) / 2;
    PP.coef = kLog2e * 0.5f * D.s * D.s;
    // Each CTA holds all of its SM's tensor memory, so they run one after the other; at d = 64, where two fit the shared memory, the
    // second's start and first loads overlap the first's end. Pieces for 148 or for 296 CTAs at d = 64: the kernel 33.6 and 34.0 us
    // (8 x 12 heads, 4096 tokens), 63.4 and 66.0 (8 heads, 65536 tokens, m 512), the calls around it 183.0 and 183.2, 795 and 744 (the
    // CTAs of what follows land elsewhere), 108.8 and 101.4 (30 heads, 2048 tokens, m 512), 99.2 and 100.9 (32 heads, 8192 tokens, m 128).
    PP.nsplit = pick_splits((long long)BH * PP.npair, Y.T, 1.5, 3.0, 64, D.d == 64 ? 296 : 148);
    const int smem_bytes = 5 * 128 * D.d * 2 + 128;
    timer_mark(plan, st, "tc_key_prepass_kernel");
    keep(launch_pdl(D.d == 64 ? tc_key_prepass_kernel<64> : tc_key_prepass_kernel<128>, dim3((unsigned)(BH * PP.npair * PP.nsplit)), dim3(160), smem_bytes, st, PP));
    return e;
}

darkattn_status_t tensor_forward(const darkattn_plan_s *plan, const void *Q, const void *K, const void *V,
                                 const void *M, const void *W, void *O, void *saved, char *ws, cudaStream_t st, bool stash_states)
{
    const Dims &D = plan->dims;
    const TensorLayout &Y = plan->tensor;
    const size_t BH = D.BH, N = D.N;
    auto bf = [&](size_t off) { return reinterpret_cast<__nv_bfloat16 *>(ws + off); };
    auto fl = [&](size_t off) { return reinterpret_cast<float *>(ws + off); };
    if (!encode_fn()) { set_cuda_error(cudaErrorNotSupported, "tensor_forward: cuTensorMapEncodeTiled unavailable"); return DARKATTN_ERR_CUDA; }

    const Stash stash = saved ? stash_in_saved(Y, saved) : stash_in_workspace(Y, ws);
    MainParams P;
    memset(&P, 0, sizeof(P));
    const size_t BHkv = (size_t)D.B * D.Hkv;
    bool ok = make_map(&P.mapQ, Q, BH * N, D.d, 128) && make_map(&P.mapK, K, BHkv * N, D.d, 128) &&
              make_map(&P.mapV, V, BHkv * N, D.dv, 128) && make_map(&P.mapOm, stash.Om, (size_t)D.H * D.m, D.d, 128) &&
              make_map(&P.mapOml, stash.Oml, (size_t)D.H * D.m, D.d, 128) &&
              make_map(&P.mapSb, D.causal ? bf(Y.Sb) : stash.Sb, BH * (D.causal ? Y.nsplit : 1) * D.m, D.dv, 128) &&
              make_map(&P.mapPN, bf(Y.pnum), (size_t)Y.nslab * BH * N, D.dv, D.causal ? 128 : 32);     // (the query pass stores a warp's 32 rows)
    if (!ok) { set_cuda_error(cudaErrorInvalidValue, "tensor_forward: tensor map encode"); return DARKATTN_ERR_CUDA; }

    cudaError_t e = tensor_prologue(plan, K, M, W, ws, stash, st);
    auto keep = [&](cudaError_t x) { if (x != cudaSuccess && e == cudaSuccess) e = x; };

    P.nK = stash.nK; P.cs = stash.cs; P.zc = stash.zc; P.pdr = fl(Y.pdr); P.Sacc = fl(Y.Sacc); P.zacc = fl(Y.zacc);
    P.status = reinterpret_cast<int *>(ws + Y.status);
    P.N = D.N; P.H = D.H; P.Hkv = D.Hkv; P.BH = D.BH; P.m = D.m; P.nslab = Y.nslab; P.T = Y.T; P.nsplit = Y.nsplit;
    P.stash_S = (D.causal && stash_states) ? 1 : 0;
    if (P.stash_S && !(make_map(&P.mapSst, stash.Sst, BH * Y.T * D.m, D.dv, 128) && make_map(&P.mapBf, stash.Bphi, BH * N, D.m, 128))) {
        set_cuda_error(cudaErrorInvalidValue, "tensor_forward: tensor map encode");
        return DARKATTN_ERR_CUDA;
    }
    const int units = (int)(BH * Y.nslab);
    if (D.causal) {
        if (Y.nsplit > 1) {      // segment states, then their exclusive prefix
            P.npiece = Y.npiece; P.Sseg = fl(Y.Sseg); P.zseg = fl(Y.zseg);
            const int pieces = units * Y.npiece, E4 = D.m * D.dv / 4;
            timer_mark(plan, st, "tc_fwd_keys_kernel");
            keep(launch_main_shape<MODE_KEYS>(D.d, D.dv, P, pieces < 148 ? pieces : 148, st));
            const long long total = (long long)BH * E4;
            timer_mark(plan, st, "segment_prefix_kernel");
            keep(launch_pdl(segment_prefix_kernel, dim3((unsigned)((total + 255) / 256)), dim3(256), 0, st, (const float *)fl(Y.Sacc), (const float *)fl(Y.zacc),
                            fl(Y.Sseg), bf(Y.Sb), fl(Y.zseg), Y.nsplit, Y.npiece, E4, D.m, total));
        }
        timer_mark(plan, st, "tc_fwd_causal_kernel");
        P.cut = Y.cut;
        P.done = Y.summers ? reinterpret_cast<int *>(ws + Y.done) : nullptr;
        P.scan_ctas = units * Y.nsplit; P.pnum = bf(Y.pnum); P.O = (__nv_bfloat16 *)O; P.sv = stash.sv;
        keep(launch_main_shape<MODE_CAUSAL>(D.d, D.dv, P, P.scan_ctas + Y.summers, st));
    } else {
        // one CTA per SM, the same number for every slab; a problem of few tiles gets one CTA for each
        int per = 148 / Y.nslab;
        if (per > (long long)BH * Y.T) per = (int)(BH * Y.T);
        const int grid = Y.nslab * (per > 1 ? per : 1);
        timer_mark(plan, st, "tc_fwd_keys_kernel");
        keep(launch_main_shape<MODE_KEYS>(D.d, D.dv, P, grid, st));
        const long long n4 = (long long)BH * D.m * D.dv / 4;
        timer_mark(plan, st, "state_to_bf16_kernel");
        keep(launch_pdl(state_to_bf16_kernel, dim3((unsigned)((n4 + 255) / 256)), dim3(256), 0, st, (const float *)fl(Y.Sacc), stash.Sb, n4, (const float *)fl(Y.zacc), stash.zt, (long long)BH * D.m));
        P.zq = stash.zt;
        timer_mark(plan, st, "tc_fwd_queries_kernel");
        keep(launch_main_shape<MODE_QUERIES>(D.d, D.dv, P, grid, st));
    }
    const int longest = (Y.T + Y.nsplit - 1) / Y.nsplit;
    if (Y.cut < longest) {
        const long long rows = (long long)BH * N;
        const int nseg = D.causal ? Y.nsplit : 1;
        timer_mark(plan, st, "combine_kernel");
        auto *combine = Y.nslab == 1 ? combine_kernel<1> : Y.nslab == 2 ? combine_kernel<2> : Y.nslab == 4 ? combine_kernel<4> : combine_kernel<0>;
        // (in the second dimension, which is limited to 65535, whole sequences where nothing has been summed yet)
        const bool flat = Y.cut == 0;
        const long long threads = flat ? rows * (D.dv / 8) : (long long)(longest - Y.cut) * 128 * (D.dv / 8);
        keep(launch_pdl(combine, dim3((unsigned)((threads + 255) / 256), flat ? 1 : (unsigned)(BH * nseg)), dim3(256), 0, st, (const __nv_bfloat16 *)bf(Y.pnum),
                        (const float *)fl(Y.pdr), (__nv_bfloat16 *)O, stash.sv, rows, D.dv, Y.nslab, P.status, flat ? (int)(rows / 128) : Y.T, flat ? 1 : nseg, Y.cut));
    }
    if (e != cudaSuccess) { set_cuda_error(e, "tensor_forward"); return DARKATTN_ERR_CUDA; }
    return DARKATTN_OK;
}

}  // namespace darkattn
