// Single-token decode step of causal DARK attention: the recurrent form of the causal scan. Per (batch, head) the
// caller keeps the running state S = sum_j phi(k_j) v_j^T (m x dv) and z = sum_j phi(k_j) (m), both float32; one step
// adds the new token's key and value and reads the new token's query out:
//     S += phi(k) v^T,   z += phi(k),   o = phi(q)^T S / phi(q)^T z          (Section 2's ordering phi(Q) (phi(K)^T V), one row at a time)
// Stabiliser (cancels in o, and is the same at every step, so the state of one step is valid for the next): keys use
// the per-feature shift c_l = |w_l|^2 / 2, i.e. phi(k)_l = exp(u_l - |x~|^2/2 - c_l) = exp(-|x~ - w_l|^2 / 2) <= 1;
// queries use exp(u_l + c_l - max_l(u_l + c_l)).
//
// The step is bound by the traffic of the state (read and written once) when there are many (batch, head) pairs, and by a
// chain of load latencies (q, k -> M -> W -> state) when there are few. Both want the state's loads out of the chain: they
// start first, by asynchronous copies into shared memory (every lane copies what it will use itself, so nothing has to be
// synchronised), and the features are formed while they are on their way. The features of a pair are cut over the CTAs of
// a cluster: each forms x~, then the exponents of its own features, updates its own rows of the state and sends its partial
// numerators and normaliser, scaled by its own maximum, to the first CTA. Measured (m = 256, dv = 128, bf16): 64 pairs
// 14.3 -> 8.1 us, 1024 pairs (134 MB of state) 90.7 -> 63 us, 4.3 TB/s. There seven pairs an SM go through three resident blocks, and a block
// loads the first half of its state, forms features while nothing else of it moves, then streams the rest: not the features' instructions
// (cut by the paired products below: 62.2 -> 61.6 us) but these phases keep it from the copy bandwidth. With few pairs the loads of M and of W stand
// behind the barriers that follow q, k and x~, by the order of this program: their addresses depend on neither.
#include "common.cuh"
#include "tc_common.cuh"

#include <math.h>

namespace darkattn {

namespace {

constexpr int kNT = 256, kWarps = kNT / 32, kGroups = kNT / 8;      // kGroups: rows of M or W in work at a time, eight lanes each
constexpr int kItems = 8, kSlots = 2;                               // 16-byte pieces per lane and slot, slots per warp
constexpr int kRingBytes = kWarps * kSlots * kItems * 32 * 16, kMaxParts = 4, kMaxDv = 512;
constexpr size_t kMaxVectors = 48 * 1024;                           // what a call may need for q, k, x~ and the features
constexpr int kMaxSmem = kRingBytes + (int)kMaxVectors + kMaxParts * (kMaxDv + 2) * 4;

template <typename T>
__device__ __forceinline__ float ldf(const T *p, size_t i)
{
    if constexpr (sizeof(T) == 2) return __bfloat162float(p[i]);
    else return p[i];
}

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void copy16_async(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// stores into the same place of another CTA's shared memory
__device__ __forceinline__ void store_cluster(float *p, uint32_t rank, float v)
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr(p)), "r"(rank));
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

template <typename T>
__device__ __forceinline__ void unpack16(const uint4 &q, float (&w)[16 / sizeof(T)])
{
    const uint32_t u[4] = {q.x, q.y, q.z, q.w};
    if constexpr (sizeof(T) == 2) {                 // eight bf16: the upper half of an fp32 each
#pragma unroll
        for (int j = 0; j < 4; ++j) { w[2 * j] = __uint_as_float(u[j] << 16); w[2 * j + 1] = __uint_as_float(u[j] & 0xffff0000u); }
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = __uint_as_float(u[j]);
    }
}

__device__ __forceinline__ float sum8(float v)
{
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Dot products of the rows of a matrix [nrows, n] with two vectors held in shared memory, and the rows' squared norms. Eight
// lanes share a row: lane `sub` of the eight takes every eighth 16-byte piece of it, so a warp's load covers four rows in
// pieces of 128 contiguous bytes, and three shuffle steps add the eight parts up. put(row, d0, d1, nn) is called by all
// eight lanes. PIECES > 0: rows of exactly 8 PIECES pieces; the lane's share of the vectors stays in registers and
// the loads of 8, 4 or (PIECES = 4: the registers) 1 rows are in flight together (a block is a chain of load latencies). PIECES = 0: any length, rows that
// do not start on 16 bytes element by element.
template <typename T, int PIECES, bool NORM, typename Put>
__device__ __forceinline__ void rows_dots(const T *mat, int nrows, int n, const float *x0, const float *x1, int tid, Put put)
{
    constexpr int V = 16 / (int)sizeof(T);          // elements per 16-byte load
    // Two products to an instruction for bf16: with those of the state update, steps in one graph, d = dv = 128, m 256, five runs a side that differ
    // by 0.01 us: 1 pair 6.08 -> 5.94 us, 32: 7.17 -> 7.06, 64: 7.79 -> 7.63, 128: 13.7 -> 13.3, 256: 17.9 -> 17.4, 512: 26.9 -> 26.3. Not for
    // fp32, whose 16 bytes hold four elements: there the two halves of each sum only add registers (8.29 -> 8.89 us).
    constexpr bool PAIRS = sizeof(T) == 2;
    const int sub = tid & 7, grp = tid >> 3;
    if constexpr (PIECES > 0) {
        constexpr int RB = PIECES == 4 ? 1 : 8 / PIECES;
        float a[PIECES][V], b[PIECES][V];
#pragma unroll
        for (int i = 0; i < PIECES; ++i)
#pragma unroll
            for (int j = 0; j < V; ++j) { a[i][j] = x0[(i * 8 + sub) * V + j]; b[i][j] = x1[(i * 8 + sub) * V + j]; }
        for (int r0 = 0; r0 < nrows; r0 += kGroups * RB) {
            uint4 raw[RB][PIECES];
#pragma unroll
            for (int k = 0; k < RB; ++k) {
                const int row = min(r0 + k * kGroups + grp, nrows - 1);      // (rows past the end: the last one again, not stored)
#pragma unroll
                for (int i = 0; i < PIECES; ++i) raw[k][i] = __ldg(reinterpret_cast<const uint4 *>(mat + (size_t)row * n) + i * 8 + sub);
            }
#pragma unroll
            for (int k = 0; k < RB; ++k) {
                if (r0 + k * kGroups >= nrows) break;
                float d0 = 0.f, d1 = 0.f, nn = 0.f, e0 = 0.f, e1 = 0.f, en = 0.f;      // sums over even and odd elements, two to an instruction
#pragma unroll
                for (int i = 0; i < PIECES; ++i) {
                    float w[V];
                    unpack16<T>(raw[k][i], w);
#pragma unroll
                    for (int j = 0; j < V; j += 2) {
                        if constexpr (PAIRS) {
                            tc::fma2(d0, e0, w[j], w[j + 1], a[i][j], a[i][j + 1]);
                            tc::fma2(d1, e1, w[j], w[j + 1], b[i][j], b[i][j + 1]);
                            if (NORM) tc::fma2(nn, en, w[j], w[j + 1], w[j], w[j + 1]);
                        } else {
                            d0 = fmaf(w[j + 1], a[i][j + 1], fmaf(w[j], a[i][j], d0));
                            d1 = fmaf(w[j + 1], b[i][j + 1], fmaf(w[j], b[i][j], d1));
                            if (NORM) nn = fmaf(w[j + 1], w[j + 1], fmaf(w[j], w[j], nn));
                        }
                    }
                }
                d0 = sum8(d0 + e0); d1 = sum8(d1 + e1);
                if (NORM) nn = sum8(nn + en);
                const int row = r0 + k * kGroups + grp;
                if (row < nrows) put(row, d0, d1, nn);
            }
        }
    } else {
        const bool vec = (n % V == 0) && (reinterpret_cast<uintptr_t>(mat) & 15) == 0;
        for (int r0 = 0; r0 < nrows; r0 += kGroups) {
            const int row = r0 + grp;
            const T *p = mat + (size_t)min(row, nrows - 1) * n;
            float d0 = 0.f, d1 = 0.f, nn = 0.f;
            if (vec) {
#pragma unroll 4
                for (int c = sub * V; c < n; c += 8 * V) {
                    float w[V];
                    unpack16<T>(__ldg(reinterpret_cast<const uint4 *>(p + c)), w);
#pragma unroll
                    for (int j = 0; j < V; ++j) { d0 = fmaf(w[j], x0[c + j], d0); d1 = fmaf(w[j], x1[c + j], d1); nn = fmaf(w[j], w[j], nn); }
                }
            } else {
                for (int c = sub; c < n; c += 8) {
                    const float w = ldf(p, c);
                    d0 = fmaf(w, x0[c], d0); d1 = fmaf(w, x1[c], d1); nn = fmaf(w, w, nn);
                }
            }
            d0 = sum8(d0); d1 = sum8(d1); nn = sum8(nn);
            if (row < nrows) put(row, d0, d1, nn);
        }
    }
}

template <typename T, bool NORM, typename Put>
__device__ __forceinline__ void rows_dots_any(const T *mat, int nrows, int n, const float *x0, const float *x1, int tid, Put put)
{
    constexpr int V = 16 / (int)sizeof(T);
    const bool aligned = (reinterpret_cast<uintptr_t>(mat) & 15) == 0;
    if (aligned && n == 32 * V) rows_dots<T, 4, NORM>(mat, nrows, n, x0, x1, tid, put);            // 256 bf16 or 128 fp32
    else if (aligned && n == 16 * V) rows_dots<T, 2, NORM>(mat, nrows, n, x0, x1, tid, put);       // 128 bf16 or 64 fp32
    else if (aligned && n == 8 * V) rows_dots<T, 1, NORM>(mat, nrows, n, x0, x1, tid, put);   // 64 bf16 or 32 fp32
    else rows_dots<T, 0, NORM>(mat, nrows, n, x0, x1, tid, put);
}

struct DecodeParams {
    const void *q, *k, *v, *M, *W;
    float *S, *z;
    void *o;
    int H, Hkv, d, r, m, dv, w_per_head, parts, mp;      // parts: CTAs per (batch, head); mp: features of each
    float s;
};

// NCB: pieces of 128 columns per row of the state (1, 2 or 4).
template <typename T, int NCB>
__global__ void __launch_bounds__(kNT, 3) decode_step_kernel(const __grid_constant__ DecodeParams p)
{
    extern __shared__ __align__(16) float sm[];
    float4 *ring = reinterpret_cast<float4 *>(sm);                   // [warp][slot][item][lane]; afterwards the partial numerators
    float *vq = sm + kWarps * kSlots * kItems * 32 * 4, *vk = vq + p.d, *xq = vk + p.d, *xk = xq + p.r;
    float2 *fkq = reinterpret_cast<float2 *>(xk + p.r);     // phi(k), phi(q) of every feature
    float *red = reinterpret_cast<float *>(fkq + p.mp);                                         // [kWarps] maxima, [kWarps] normalisers
    float *gather = red + 2 * kWarps;                                // first CTA: [parts][dv + 2] partial numerators, normaliser, maximum
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int part = blockIdx.x % p.parts, bh = blockIdx.x / p.parts, h = bh % p.H;
    const int kvh = (bh / p.H) * p.Hkv + h / (p.H / p.Hkv);           // the key/value head this query head reads (grouped key/value heads)
    const int l0 = part * p.mp, nl = min(p.mp, p.m - l0);             // this CTA's features (the last CTA's may be fewer, never none)
    if (p.parts > 1) cluster_arrive();

    // which piece of the state is the lane's i-th: four columns of a row, a row of dv <= 128 columns to dv / 4 lanes
    // (i = NCB * n + b: columns col0 + 128 b .. + 3 of row row0 + n step; a lane without columns has no rows)
    const int lpr = NCB == 1 ? p.dv / 4 : 32, rpi = 32 / lpr, sub = lane / lpr, col0 = (lane - sub * lpr) * 4;
    const int row0 = warp * rpi + sub, step = kWarps * rpi;
    const int nrows = sub < rpi ? (nl - row0 + step - 1) / step : 0;            // this lane's rows (may be negative)
    const int nslots = ((nl + step - 1) / step * NCB + kItems - 1) / kItems;    // (the same for all lanes)
    float *Sb = p.S + ((size_t)bh * p.m + l0 + row0) * p.dv + col0;
    const size_t rstride = (size_t)step * p.dv;
    float4 *mine = ring + (size_t)warp * kSlots * kItems * 32 + lane;
    auto start_slot = [&](int slot) {
        float4 *dst = mine + (slot % kSlots) * kItems * 32;
#pragma unroll
        for (int j = 0; j < kItems; ++j) {
            const int n = (slot * kItems + j) / NCB, b = j % NCB;
            if (n < nrows && (NCB == 1 || col0 + 128 * b < p.dv)) copy16_async(dst + j * 32, Sb + n * rstride + 128 * b);
        }
        copy_commit();
    };
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    {
        const T *qv = static_cast<const T *>(p.q) + (size_t)bh * p.d, *kv = static_cast<const T *>(p.k) + (size_t)kvh * p.d;
        for (int c = tid; c < p.d; c += kNT) { vk[c] = ldf(kv, c); vq[c] = ldf(qv, c); }
    }
#pragma unroll
    for (int i = 0; i < kSlots; ++i) start_slot(i);
    float *zb = p.z + (size_t)bh * p.m + l0;
    const float z_first = tid < nl ? zb[tid] : 0.f;
    __syncthreads();
    // x~ = s M x for the query and the key
    rows_dots_any<T, false>(static_cast<const T *>(p.M) + (size_t)h * p.r * p.d, p.r, p.d, vq, vk, tid,
                            [&](int row, float a, float b, float) { if ((tid & 7) == 0) { xq[row] = p.s * a; xk[row] = p.s * b; } });
    __syncthreads();
    float nk = 0.f;
    for (int a = lane; a < p.r; a += 32) nk = fmaf(xk[a], xk[a], nk);
    for (int off = 16; off; off >>= 1) nk += __shfl_xor_sync(0xffffffffu, nk, off);
    nk *= 0.5f;
    float mx = -INFINITY;
    rows_dots_any<T, true>(static_cast<const T *>(p.W) + ((size_t)(p.w_per_head ? h : 0) * p.m + l0) * p.r, nl, p.r, xq, xk, tid,
                           [&](int row, float uq, float uk, float nn) {
                               const float c = 0.5f * nn;
                               if ((tid & 7) == 0) fkq[row] = make_float2(__expf(uk - nk - c), uq + c);
                               mx = fmaxf(mx, uq + c);
                           });
    for (int off = 16; off; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    if (lane == 0) red[warp] = mx;
    __syncthreads();
    mx = red[0];
#pragma unroll
    for (int w = 1; w < kWarps; ++w) mx = fmaxf(mx, red[w]);
    // the query's features, the new z and the normaliser phi(q) . z
    float den = 0.f;
    for (int l = tid; l < nl; l += kNT) {
        const float2 fg = fkq[l];
        const float f = __expf(fg.y - mx), zn = (l == tid ? z_first : zb[l]) + fg.x;
        fkq[l].y = f;
        zb[l] = zn;
        den = fmaf(f, zn, den);
    }
    for (int off = 16; off; off >>= 1) den += __shfl_xor_sync(0xffffffffu, den, off);
    if (lane == 0) red[kWarps + warp] = den;
    // the value's columns of this lane
    float4 vv[NCB], num[NCB];
#pragma unroll
    for (int b = 0; b < NCB; ++b) {
        const int c = col0 + 128 * b;
        const T *vr = static_cast<const T *>(p.v) + (size_t)kvh * p.dv;
        num[b] = vv[b] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (c < p.dv) vv[b] = make_float4(ldf(vr, c), ldf(vr, c + 1), ldf(vr, c + 2), ldf(vr, c + 3));
    }
    __syncthreads();

    // state update and read-out
    for (int slot = 0; slot < nslots; ++slot) {
        copy_wait<kSlots - 1>();                    // (each lane reads only what it copied)
        const float4 *src = mine + (slot % kSlots) * kItems * 32;
#pragma unroll
        for (int j = 0; j < kItems; ++j) {
            const int n = (slot * kItems + j) / NCB, b = j % NCB;
            if (n < nrows && (NCB == 1 || col0 + 128 * b < p.dv)) {
                const float4 x = src[j * 32], v4 = vv[b];
                const float2 fg = fkq[row0 + n * step];
                const float f = fg.x, g = fg.y;
                float4 sn = x;
                tc::fma2(sn.x, sn.y, f, f, v4.x, v4.y);
                tc::fma2(sn.z, sn.w, f, f, v4.z, v4.w);
                *reinterpret_cast<float4 *>(Sb + n * rstride + 128 * b) = sn;
                float4 &nm = num[b];
                tc::fma2(nm.x, nm.y, g, g, sn.x, sn.y);
                tc::fma2(nm.z, nm.w, g, g, sn.z, sn.w);
            }
        }
        if (slot + kSlots < nslots) start_slot(slot + kSlots);
        else copy_commit();                         // (an empty group, so that the wait above counts the same)
    }
    copy_wait<0>();
    __syncthreads();                                // the ring becomes the partial numerators: [warp][row of the warp][dv]
    const int npart = kWarps * rpi;
    if (sub < rpi)
#pragma unroll
        for (int b = 0; b < NCB; ++b) {
            const int c = col0 + 128 * b;
            if (c < p.dv) *reinterpret_cast<float4 *>(sm + (size_t)(warp * rpi + sub) * p.dv + c) = num[b];
        }
    __syncthreads();
    if (p.parts > 1) cluster_wait();                // the first CTA runs (all have arrived at their start)
    float *slotp = gather + (size_t)part * (p.dv + 2);
    for (int c = tid; c < p.dv + 2; c += kNT) {
        float x = 0.f;
        if (c < p.dv) for (int g = 0; g < npart; ++g) x += sm[(size_t)g * p.dv + c];
        else if (c == p.dv) {
#pragma unroll
            for (int w = 0; w < kWarps; ++w) x += red[kWarps + w];
        } else x = mx;
        if (p.parts > 1) store_cluster(slotp + c, 0, x);
        else slotp[c] = x;
    }
    if (p.parts > 1) { cluster_arrive(); cluster_wait(); }
    else __syncthreads();
    if (part > 0) return;
    float top = -INFINITY;
    for (int i = 0; i < p.parts; ++i) top = fmaxf(top, gather[(size_t)i * (p.dv + 2) + p.dv + 1]);
    for (int c = tid; c < p.dv; c += kNT) {
        float n = 0.f, dn = 0.f;
        for (int i = 0; i < p.parts; ++i) {
            const float *g = gather + (size_t)i * (p.dv + 2), e = __expf(g[p.dv + 1] - top);
            n = fmaf(e, g[c], n);
            dn = fmaf(e, g[p.dv], dn);
        }
        const float out = n / dn;
        if constexpr (sizeof(T) == 2) static_cast<__nv_bfloat16 *>(p.o)[(size_t)bh * p.dv + c] = __float2bfloat16_rn(out);
        else static_cast<float *>(p.o)[(size_t)bh * p.dv + c] = out;
    }
}

template <typename T>
cudaError_t launch_decode(const DecodeParams &P, int BH, cudaStream_t st)
{
    const size_t smem = kRingBytes + (2 * P.d + 2 * P.r + 2 * P.mp + 2 * kWarps + (size_t)P.parts * (P.dv + 2)) * sizeof(float);
    auto *k = P.dv <= 128 ? decode_step_kernel<T, 1> : P.dv <= 256 ? decode_step_kernel<T, 2> : decode_step_kernel<T, 4>;
    // One limit for all plans of a kernel, set once: another thread's plan must not lower it between this and the launch below.
    const cudaError_t e = allow_smem(reinterpret_cast<const void *>(k), kMaxSmem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)BH * P.parts); cfg.blockDim = dim3(kNT); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // (the kernel waits before it touches memory)
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = P.parts; at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, k, P);
}

}  // namespace

}  // namespace darkattn

using namespace darkattn;

extern "C" darkattn_status_t darkattn_decode_step(darkattn_plan_t plan, const void *q, const void *k, const void *v, const void *M,
                                                  const void *W, float *S, float *z, void *o, void *cuda_stream)
{
    if (!plan || !q || !k || !v || !M || !W || !S || !z || !o) return DARKATTN_ERR_INVALID_ARG;
    const Dims &D = plan->dims;
    if (!D.causal) return DARKATTN_ERR_UNSUPPORTED;          // the recurrent form is the causal one
    if (D.dv % 32) return DARKATTN_ERR_UNSUPPORTED;
    if (D.dv > kMaxDv) return DARKATTN_ERR_UNSUPPORTED;
    if ((size_t)(2 * D.d + 2 * D.r + 2 * D.m + 2048 + 16) * sizeof(float) > kMaxVectors) return DARKATTN_ERR_UNSUPPORTED;
    // CTAs per (batch, head): enough to give most SMs one while the pairs are few; at least 32 features each. In us with one, two and
    // four, bf16, d = dv = 128: m = 256: 1 pair 9.8, 7.6, 6.7; 37 pairs 10.1, 8.2, 8.2; 64 pairs 10.3, 8.4, 10.6; 96 pairs 10.3, 10.4, 10.7; m = 1024:
    // 64 pairs 25.2, 16.3, 19.9; 96 pairs 25.6, 23.5, 19.7; 147 pairs 33.6, 32.3, 36.6. From 75 pairs on two CTAs of some pairs share an SM,
    // which pays for m = 1024 and not for less (m = 256, 147 pairs: 10.9, 13.9, 19.0; d = dv = 64, m = 128: 6.7, 8.3, 14.7); fp32 alike.
    int parts = D.BH <= 37 ? kMaxParts : D.BH < 148 ? 2 : 1;
    while (parts > 1 && D.m < 32 * parts) parts /= 2;
    DecodeParams P{q, k, v, M, W, S, z, o, D.H, D.Hkv, D.d, D.r, D.m, D.dv, D.w_per_head, 0, 0, D.s};
    P.mp = (D.m + parts - 1) / parts;
    P.parts = (D.m + P.mp - 1) / P.mp;
    const cudaError_t e = D.bf16 ? launch_decode<__nv_bfloat16>(P, D.BH, static_cast<cudaStream_t>(cuda_stream))
                                 : launch_decode<float>(P, D.BH, static_cast<cudaStream_t>(cuda_stream));
    if (e != cudaSuccess) { set_cuda_error(e, "decode_step"); return DARKATTN_ERR_CUDA; }
    return DARKATTN_OK;
}
