// FP32 path of libdarkattn: every step of DARK attention with fp32 operands and fp32 accumulation.
//
// This is the path that meets the 1e-4 tolerance (a single bf16 or TF32 operand rounds the argument of the exponential
// too coarsely), and the path that accepts any shape. Its products run on the tensor cores with every fp32 operand split
// into three bf16 numbers (split_gemm.cu); what surrounds them is done on the way into or out of a product, so that the
// intermediates are written once and read by the next product:
//   forward    x~ = s X M^T (both sides; row norms of the keys) | u = x~ W^T (keys: minus the norm; column maxima) |
//              features in place | chunk states and masked kernel tiles | prefix over the chunks | output rows
//   backward   the forward steps with the output rows turned into dO / den and -delta / den | dP and the reverse states |
//              suffix over the chunks | E of both sides and dV | dx~ | dQ, dK and dM | sums over batch and token blocks
// Each line's items between bars are one launch each; all but the first start while the one before drains
// (programmatic dependent launch).
//
// Stabiliser (cancels in O): keys use one shift per (batch, head, feature), c_l = max_j (u_jl - n_j),
// queries use e_il = u_il + c_l - max_l(u_il + c_l); the query's own norm term is a per-row constant
// and is dropped (so is its gradient, which is zero). The product phi(q_i)_l phi(k_j)_l is then the unshifted one times
// a per-row factor.
#include "common.cuh"
#include "split_gemm.cuh"
#include "tc_common.cuh"

#include <math.h>

namespace darkattn {

using sg::launch_pdl;

namespace {

// Features in place, one warp per row: query rows exp(u_l + c_l - max_l(u_l + c_l)), key rows exp(u_l - c_l) (u already
// has the key's norm taken off). V: elements per load. A row is read twice (the second time from L1 or L2).
template <int V>
__global__ void __launch_bounds__(256) features_kernel(float *fQ, float *fK, const int *cK, int N, int m, long long rows)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const long long w = (blockIdx.x * 256LL + threadIdx.x) / 32;
    const int lane = threadIdx.x & 31;
    if (w >= 2 * rows) return;
    const bool keys = w >= rows;
    const long long row = keys ? w - rows : w;
    float *f = (keys ? fK : fQ) + row * m;
    const int *c = cK + row / N * m;
    float mx = 0.f;
    auto load = [&](int l, float (&x)[V], float (&s)[V]) {
        if constexpr (V == 4) {
            const float4 a = *reinterpret_cast<const float4 *>(f + l);
            const int4 k = __ldg(reinterpret_cast<const int4 *>(c + l));
            x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
            s[0] = tc::float_from_order_key(k.x); s[1] = tc::float_from_order_key(k.y); s[2] = tc::float_from_order_key(k.z); s[3] = tc::float_from_order_key(k.w);
        } else { x[0] = f[l]; s[0] = tc::float_from_order_key(__ldg(c + l)); }
    };
    if (!keys) {
        mx = -INFINITY;
        for (int l = lane * V; l < m; l += 32 * V) {
            float x[V], s[V];
            load(l, x, s);
#pragma unroll
            for (int j = 0; j < V; ++j) mx = fmaxf(mx, x[j] + s[j]);
        }
        for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    for (int l = lane * V; l < m; l += 32 * V) {
        float x[V], s[V];
        load(l, x, s);
#pragma unroll
        for (int j = 0; j < V; ++j) x[j] = expf(keys ? x[j] - s[j] : x[j] + s[j] - mx);
        if constexpr (V == 4) *reinterpret_cast<float4 *>(f + l) = make_float4(x[0], x[1], x[2], x[3]);
        else f[l] = x[0];
    }
}

// Over the token blocks of S[pair, block, e] and z[pair, block, l], in place: what came before each block (forward) or
// comes after it (reverse), or the sum over all of them into the first. One thread per V neighbouring elements; eight
// blocks' loads are in flight at a time (the sum is a serial chain, the loads are not).
enum { SCAN_FORWARD = 0, SCAN_REVERSE = 1, SCAN_TOTAL = 2 };
template <int V>
__global__ void __launch_bounds__(256) chunk_scan_kernel(float *S, float *z, int nb, long long E, int m, long long pairs, int mode)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    long long i = (blockIdx.x * 256LL + threadIdx.x) * V;
    float *base;
    long long step;
    if (i < pairs * E) { base = S + i / E * nb * E + i % E; step = E; }
    else {
        i -= pairs * E;
        if (i >= pairs * m) return;
        base = z + i / m * nb * m + i % m;
        step = m;
    }
    float run[V];
#pragma unroll
    for (int j = 0; j < V; ++j) run[j] = 0.f;
    for (int k0 = 0; k0 < nb; k0 += 8) {
        float x[8][V];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int c = mode == SCAN_REVERSE ? nb - 1 - (k0 + k) : k0 + k;
            if (k0 + k < nb) {
                if constexpr (V == 4) { const float4 a = *reinterpret_cast<const float4 *>(base + c * step); x[k][0] = a.x; x[k][1] = a.y; x[k][2] = a.z; x[k][3] = a.w; }
                else x[k][0] = base[c * step];
            }
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (k0 + k >= nb) break;
            const int c = mode == SCAN_REVERSE ? nb - 1 - (k0 + k) : k0 + k;
            if (mode != SCAN_TOTAL) {
                if constexpr (V == 4) *reinterpret_cast<float4 *>(base + c * step) = make_float4(run[0], run[1], run[2], run[3]);
                else base[c * step] = run[0];
            }
#pragma unroll
            for (int j = 0; j < V; ++j) run[j] += x[k][j];
        }
    }
    if (mode == SCAN_TOTAL) {
        if constexpr (V == 4) *reinterpret_cast<float4 *>(base) = make_float4(run[0], run[1], run[2], run[3]);
        else base[0] = run[0];
    }
}

// out[o, e] = sum of src over `n1` outer and `n2` inner slices: src[(i1 * stride1 + o) * n2 + i2, e]. dM sums over the batch
// and the token blocks (o = head), dW also over the heads where they share W (o = 0).
__global__ void __launch_bounds__(256) reduce_kernel(const float *src, float *out, int n1, long long stride1, int n2, long long E, long long total)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const long long t = blockIdx.x * 256LL + threadIdx.x;
    if (t >= total) return;
    const long long o = t / E, e = t % E;
    float acc = 0.f;
    for (int i1 = 0; i1 < n1; ++i1) {
        const float *p = src + (i1 * stride1 + o) * n2 * E + e;
#pragma unroll 8
        for (int i2 = 0; i2 < n2; ++i2) acc += p[i2 * E];
    }
    out[t] = acc;
}

// Grouped key/value heads: out[(b,hk), e] = sum_g src[(b, hk G + g), e]: the gradient of a shared key or value row
// collects the parts of the G query heads that read it.
template <typename T>
__global__ void __launch_bounds__(256) group_sum_f32_kernel(T *out, const float *src, int G, long long E, long long total)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (long long t = blockIdx.x * 256LL + threadIdx.x; t < total; t += gridDim.x * 256LL) {
        const long long kv = t / E, e = t % E;
        float v = 0.f;
        for (int g = 0; g < G; ++g) v += src[(kv * G + g) * E + e];
        if constexpr (sizeof(T) == 2) out[t] = __float2bfloat16_rn(v);
        else out[t] = v;
    }
}

struct Runner {
    const darkattn_plan_s *plan;
    char *ws;
    cudaStream_t st;
    bool dependent = false;         // a kernel of this call has been launched
    cudaError_t err = cudaSuccess;

    const Dims &D() const { return plan->dims; }
    float *f(size_t off) const { return reinterpret_cast<float *>(ws + off); }
    void keep(cudaError_t e) { if (e != cudaSuccess && err == cudaSuccess) err = e; dependent = true; }
    void gemms(sg::Launch &L) { L.status = reinterpret_cast<int *>(ws); keep(sg::run(L, st, dependent)); }
    template <typename... K, typename... A>
    void kernel(void (*k)(K...), long long threads, A... args)
    {
        // (the same division of the SM's memory as the products' kernel: a change between launches costs microseconds)
        keep(cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
        keep(launch_pdl(k, dim3((unsigned)((threads + 255) / 256)), dim3(256), 0, st, dependent, args...));
    }

    // ---- operands
    // tensors [B, H (or H_kv), N, w] in the storage type; cut into blocks of `blk` tokens
    sg::Op input(const void *p, int w, bool kv, int mn, int blk = 0) const
    {
        sg::Op o;
        const long long per = (long long)D().N * w;
        o.p = p; o.sh = per; o.sb = per * (kv ? D().Hkv : D().H); o.kv = kv; o.sc = (long long)blk * w;
        o.ld = w; o.bf16 = D().bf16; o.mn = mn;
        return o;
    }
    // fp32 intermediates [BH, N, w]
    sg::Op rows(size_t off, int w, int mn, int blk = 0) const
    {
        sg::Op o;
        const long long per = (long long)D().N * w;
        o.p = f(off); o.sh = per; o.sb = per * D().H; o.sc = (long long)blk * w; o.ld = w; o.mn = mn;
        return o;
    }
    // fp32 per block [BH, nb, rows, w] (one_block: the first block stands for all)
    sg::Op blocks(size_t off, int nb, long long nrows, int w, int mn, bool one_block = false) const
    {
        sg::Op o;
        const long long per = nrows * w;
        o.p = f(off); o.sh = per * nb; o.sb = per * nb * D().H; o.sc = one_block ? 0 : per; o.ld = w; o.mn = mn;
        return o;
    }
    // parameters M [H, r, d], W [m, r] or [H, m, r]
    sg::Op paramM(const void *M, int mn) const
    {
        sg::Op o; o.p = M; o.sh = (long long)D().r * D().d; o.ld = D().d; o.bf16 = D().bf16; o.mn = mn; return o;
    }
    sg::Op paramW(const void *W, int mn) const
    {
        sg::Op o; o.p = W; o.sh = D().w_per_head ? (long long)D().m * D().r : 0; o.ld = D().r; o.bf16 = D().bf16; o.mn = mn; return o;
    }
    // ---- products over the whole sequence of every (batch, head)
    sg::Prob whole() const
    {
        sg::Prob p;
        p.H = D().H; p.G = D().G; p.batch = D().BH; p.ntok = D().N; p.nblk = 1; p.block = 0;
        return p;
    }
    // ... or over blocks of it
    sg::Prob blocked(int nb, int blk) const
    {
        sg::Prob p = whole();
        p.nblk = nb; p.block = blk;
        return p;
    }
    void out_rows(sg::Prob &p, void *o, int w, bool storage, int blk = 0) const      // [BH, N, w]
    {
        const long long per = (long long)D().N * w;
        p.out = o; p.osh = per; p.osb = per * D().H; p.osc = (long long)blk * w; p.old_ = w; p.obf16 = storage && D().bf16;
    }
    void out_blocks(sg::Prob &p, size_t off, int nb, long long nrows, int w) const
    {
        const long long per = nrows * w;
        p.out = f(off); p.osh = per * nb; p.osb = per * nb * D().H; p.osc = per; p.old_ = w;
    }
};

inline int tiles(int n) { return (n + 127) / 128; }

// Features, states and output rows. With dO given the rows dO / den and -delta / den are formed in place of O.
void run_forward_stages(Runner &R, const void *Q, const void *K, const void *V, const void *M, const void *W, void *O, const void *dO)
{
    const Dims &D = R.D();
    const SimtLayout &Y = R.plan->simt;
    const int N = D.N, d = D.d, r = D.r, m = D.m, dv = D.dv, C = Y.C, nb = Y.nb;
    const long long BH = D.BH;
    {   // x~ = s X M^T
        sg::Launch L;
        for (int side = 0; side < 2; ++side) {
            sg::Prob p = R.whole();
            p.A[0] = R.input(side ? K : Q, d, side, 0); p.B[0] = R.paramM(M, 0); p.K[0] = d;
            p.mtok = 1; p.N = r; p.alpha = D.s;
            R.out_rows(p, R.f(side ? Y.xtK : Y.xtQ), r, false);
            p.chain = 1;                    // (the exponent's argument: the most sensitive)
            if (side) { p.epi = sg::EPI_SQUARES; p.sums = R.f(Y.nK); }
            sg::add(L, p);
        }
        L.init = reinterpret_cast<int *>(R.f(Y.cK)); L.init_n = (int)(BH * m);
        R.gemms(L);
    }
    {   // u = x~ W^T, for the keys minus half the squared norm of x~
        sg::Launch L;
        for (int side = 0; side < 2; ++side) {
            sg::Prob p = R.whole();
            p.A[0] = R.rows(side ? Y.xtK : Y.xtQ, r, 0); p.B[0] = R.paramW(W, 0); p.K[0] = r;
            p.mtok = 1; p.N = m; p.chain = 1;
            R.out_rows(p, R.f(side ? Y.fK : Y.fQ), m, false);
            if (side) {
                p.epi = sg::EPI_KEY_EXPONENT; p.row = {R.f(Y.nK), BH * N, tiles(r), 0.5f};
                p.colmax = reinterpret_cast<int *>(R.f(Y.cK));
            }
            sg::add(L, p);
        }
        R.gemms(L);
    }
    if (m % 4 == 0) R.kernel(features_kernel<4>, 2 * BH * N * 32, R.f(Y.fQ), R.f(Y.fK), reinterpret_cast<const int *>(R.f(Y.cK)), N, m, BH * N);
    else R.kernel(features_kernel<1>, 2 * BH * N * 32, R.f(Y.fQ), R.f(Y.fK), reinterpret_cast<const int *>(R.f(Y.cK)), N, m, BH * N);
    {   // S_c = phi(K_c)^T V_c, z_c = phi(K_c)^T 1 per token block; causal: P_c = tril(phi(Q_c) phi(K_c)^T)
        sg::Launch L;
        sg::Prob p = R.blocked(nb, Y.blk);
        p.A[0] = R.rows(Y.fK, m, 1, Y.blk); p.B[0] = R.input(V, dv, true, 1, Y.blk); p.K[0] = N; p.ktok[0] = 1;
        p.M = m; p.N = dv; p.dot[0] = sg::DOT_ONES; p.dot_out = R.f(Y.zloc);
        R.out_blocks(p, Y.Sloc, nb, m, dv);
        sg::add(L, p);
        if (D.causal) {
            sg::Prob q = R.blocked(nb, C);
            q.A[0] = R.rows(Y.fQ, m, 0, C); q.B[0] = R.rows(Y.fK, m, 0, C); q.K[0] = m;
            q.mtok = q.ntok_dim = 1; q.epi = sg::EPI_MASK;
            R.out_blocks(q, Y.P, nb, C, C);
            sg::add(L, q);
        }
        R.gemms(L);
    }
    const long long E = (long long)m * dv;
    auto scan = [&](size_t S, size_t z, int mode) {
        if (nb == 1 && mode == SCAN_TOTAL) return;
        if (m % 4 == 0) R.kernel(chunk_scan_kernel<4>, BH * (E + m) / 4, R.f(S), R.f(z), nb, E, m, BH, mode);
        else R.kernel(chunk_scan_kernel<1>, BH * (E + m), R.f(S), R.f(z), nb, E, m, BH, mode);
    };
    scan(Y.Sloc, Y.zloc, D.causal ? SCAN_FORWARD : SCAN_TOTAL);
    {   // O = (P V + phi(Q) S_prev) / (P 1 + phi(Q) z_prev)
        sg::Launch L;
        sg::Prob p = D.causal ? R.blocked(nb, C) : R.whole();
        const int s = D.causal ? 1 : 0, blk = D.causal ? C : 0;
        if (D.causal) {
            p.A[0] = R.blocks(Y.P, nb, C, C, 0); p.B[0] = R.input(V, dv, true, 1, C); p.K[0] = C; p.ktok[0] = 1; p.dot[0] = sg::DOT_ONES;
            p.skip2_first = 1;
        }
        p.A[s] = R.rows(Y.fQ, m, 0, blk); p.B[s] = R.blocks(Y.Sloc, nb, m, dv, 1, !D.causal); p.K[s] = m; p.dot[s] = sg::DOT_FEATURES;
        p.dotf = R.f(Y.zloc); p.vec_pair = (long long)nb * m; p.vec_blk = D.causal ? m : 0;
        p.mtok = 1; p.N = dv; p.epi = dO ? sg::EPI_GRAD : sg::EPI_DIVIDE;
        if (dO) {
            p.x = R.input(dO, dv, false, 0, blk); p.sums = R.f(Y.gd);
            R.out_rows(p, R.f(Y.Ga), dv, false, blk);
        } else R.out_rows(p, O, dv, true, blk);
        sg::add(L, p);
        R.gemms(L);
    }
    if (!dO) return;
    const sg::TokVec gd = {R.f(Y.gd), BH * N, tiles(dv), 1.f};
    {   // R_c = phi(Q_c)^T Ga_c, rho_c = phi(Q_c)^T gd_c; causal: dP_c = tril(Ga_c V_c^T + gd_c)
        sg::Launch L;
        sg::Prob p = R.blocked(nb, Y.blk);
        p.A[0] = R.rows(Y.fQ, m, 1, Y.blk); p.B[0] = R.rows(Y.Ga, dv, 1, Y.blk); p.K[0] = N; p.ktok[0] = 1;
        p.M = m; p.N = dv; p.dot[0] = sg::DOT_TOKENS; p.dott = gd; p.dot_out = R.f(Y.rloc);
        R.out_blocks(p, Y.Rloc, nb, m, dv);
        sg::add(L, p);
        if (D.causal) {
            sg::Prob q = R.blocked(nb, C);
            q.A[0] = R.rows(Y.Ga, dv, 0, C); q.B[0] = R.input(V, dv, true, 0, C); q.K[0] = dv;
            q.mtok = q.ntok_dim = 1; q.epi = sg::EPI_MASK; q.row = gd;
            R.out_blocks(q, Y.dP, nb, C, C);
            sg::add(L, q);
        }
        R.gemms(L);
    }
    scan(Y.Rloc, Y.rloc, D.causal ? SCAN_REVERSE : SCAN_TOTAL);
}

size_t take(size_t &off, long long floats)
{
    const size_t at = off;
    off += (((size_t)floats * sizeof(float)) + 255) / 256 * 256;
    return at;
}

// Cuts N tokens into blocks (multiples of 64 tokens) so that `units` products of one block each are at least one wave of
// two CTAs per SM, none shorter than two stages of the contraction.
void cut_tokens(int N, long long units, int most, int &nblk, int &blk)
{
    long long want = (2 * 148 + units - 1) / units;
    if (want > (N + 127) / 128) want = (N + 127) / 128;
    if (want > most) want = most;
    if (want < 1) want = 1;
    blk = (int)(((N + want - 1) / want + 63) / 64 * 64);
    nblk = (N + blk - 1) / blk;
}

}  // namespace

void simt_make_layout(darkattn_plan_s *plan)
{
    const Dims &D = plan->dims;
    SimtLayout &Y = plan->simt;
    const long long BH = D.BH, N = D.N, d = D.d, r = D.r, m = D.m, dv = D.dv;
    if (D.causal) {
        Y.C = (int)(N < D.C ? (N + 3) / 4 * 4 : D.C);
        if (Y.C > D.C) Y.C = D.C;
        Y.blk = Y.C;
        Y.nb = (int)((N + Y.C - 1) / Y.C);
    } else {
        Y.C = 0;
        // (the extra partial states never take more room than two rows of values per token)
        cut_tokens(D.N, BH * tiles(D.m) * tiles(D.dv), (int)(1 + 2 * N / m > 64 ? 64 : 1 + 2 * N / m), Y.nb, Y.blk);
    }
    const long long nb = Y.nb, C = Y.C;
    size_t off = 0;
    Y.status = take(off, 64);
    Y.xtQ = take(off, BH * N * r); Y.xtK = take(off, BH * N * r);
    Y.fQ = take(off, BH * N * m); Y.fK = take(off, BH * N * m);
    Y.cK = take(off, BH * m);
    Y.Sloc = take(off, BH * nb * m * dv); Y.zloc = take(off, BH * nb * m);
    Y.P = D.causal ? take(off, BH * nb * C * C) : 0;
    {   // the key norms are done with before the states are written: they share their place
        size_t end = Y.Sloc;
        Y.nK = take(end, tiles(D.r) * BH * N);
        if (end > off) off = end;
    }
    Y.fwd_bytes = off;
    Y.Ga = take(off, BH * N * dv); Y.gd = take(off, tiles(D.dv) * BH * N);
    Y.dP = D.causal ? take(off, BH * nb * C * C) : 0;
    Y.Rloc = take(off, BH * nb * m * dv); Y.rloc = take(off, BH * nb * m);
    Y.dA = take(off, BH * N * m); Y.dBf = take(off, BH * N * m);
    Y.esK = take(off, tiles(D.m) * BH * N);
    Y.dxtQ = take(off, BH * N * r); Y.dxtK = take(off, BH * N * r);
    Y.dKh = D.G > 1 ? take(off, BH * N * d) : 0; Y.dVh = D.G > 1 ? take(off, BH * N * dv) : 0;
    cut_tokens(D.N, BH * tiles(D.r) * tiles(D.d), 64, Y.nsM, Y.blkM);
    cut_tokens(D.N, BH * tiles(D.m) * tiles(D.r), 64, Y.nsW, Y.blkW);
    Y.dMp = take(off, BH * Y.nsM * r * d);
    Y.dWp = take(off, BH * Y.nsW * m * r);
    Y.total_bytes = off;
}

darkattn_status_t simt_forward(const darkattn_plan_s *plan, const void *Q, const void *K, const void *V,
                               const void *M, const void *W, void *O, char *ws, cudaStream_t st)
{
    Runner R{plan, ws, st};
    run_forward_stages(R, Q, K, V, M, W, O, nullptr);
    if (R.err != cudaSuccess) { set_cuda_error(R.err, "simt_forward"); return DARKATTN_ERR_CUDA; }
    return DARKATTN_OK;
}

darkattn_status_t simt_backward(const darkattn_plan_s *plan, const void *Q, const void *K, const void *V,
                                const void *M, const void *W, const void *dO, void *dQ, void *dK, void *dV,
                                float *dM, char *ws, cudaStream_t st)
{
    const Dims &D = plan->dims;
    const SimtLayout &Y = plan->simt;
    const int N = D.N, d = D.d, r = D.r, m = D.m, dv = D.dv, C = Y.C, nb = Y.nb;
    const long long BH = D.BH;
    Runner R{plan, ws, st};
    run_forward_stages(R, Q, K, V, M, W, nullptr, dO);

    const bool grouped = D.G > 1;
    const sg::TokVec gd = {R.f(Y.gd), BH * N, tiles(dv), 1.f};
    const int blk = D.causal ? C : 0, s = D.causal ? 1 : 0;
    auto per_block = [&]() { return D.causal ? R.blocked(nb, C) : R.whole(); };
    {
        sg::Launch L;
        {   // E_Q = phi(Q) .* (dP phi(K) + Ga S_prev^T + gd z_prev^T)
            sg::Prob p = per_block();
            if (D.causal) { p.A[0] = R.blocks(Y.dP, nb, C, C, 0); p.B[0] = R.rows(Y.fK, m, 1, C); p.K[0] = C; p.ktok[0] = 1; p.skip2_first = 1; }
            p.A[s] = R.rows(Y.Ga, dv, 0, blk); p.B[s] = R.blocks(Y.Sloc, nb, m, dv, 0, !D.causal); p.K[s] = dv;
            p.epi = sg::EPI_RANK1; p.row = gd; p.rank1 = R.f(Y.zloc); p.vec_pair = (long long)nb * m; p.vec_blk = D.causal ? m : 0;
            p.x = R.rows(Y.fQ, m, 0, blk);
            p.mtok = 1; p.N = m;
            R.out_rows(p, R.f(Y.dA), m, false, blk);
            sg::add(L, p);
        }
        {   // E_K = phi(K) .* (dP^T phi(Q) + V R_next^T + rho_next^T), and its row sums
            sg::Prob p = per_block();
            if (D.causal) { p.A[0] = R.blocks(Y.dP, nb, C, C, 1); p.B[0] = R.rows(Y.fQ, m, 1, C); p.K[0] = C; p.ktok[0] = 1; }
            p.A[s] = R.input(V, dv, true, 0, blk); p.B[s] = R.blocks(Y.Rloc, nb, m, dv, 0, !D.causal); p.K[s] = dv;
            p.epi = sg::EPI_RANK1; p.rank1 = R.f(Y.rloc); p.vec_pair = (long long)nb * m; p.vec_blk = D.causal ? m : 0;
            p.x = R.rows(Y.fK, m, 0, blk); p.sums = R.f(Y.esK);
            p.mtok = 1; p.N = m;
            R.out_rows(p, R.f(Y.dBf), m, false, blk);
            sg::add(L, p);
        }
        {   // dV = P^T Ga + phi(K) R_next
            sg::Prob p = per_block();
            if (D.causal) { p.A[0] = R.blocks(Y.P, nb, C, C, 1); p.B[0] = R.rows(Y.Ga, dv, 1, C); p.K[0] = C; p.ktok[0] = 1; }
            p.A[s] = R.rows(Y.fK, m, 0, blk); p.B[s] = R.blocks(Y.Rloc, nb, m, dv, 1, !D.causal); p.K[s] = m;
            p.mtok = 1; p.N = dv;
            if (grouped) R.out_rows(p, R.f(Y.dVh), dv, false, blk);
            else R.out_rows(p, dV, dv, true, blk);
            sg::add(L, p);
        }
        R.gemms(L);
    }
    {   // dx~ = E W, for the keys minus rowsum(E) x~
        sg::Launch L;
        for (int side = 0; side < 2; ++side) {
            sg::Prob p = R.whole();
            p.A[0] = R.rows(side ? Y.dBf : Y.dA, m, 0); p.B[0] = R.paramW(W, 1); p.K[0] = m;
            p.mtok = 1; p.N = r;
            if (side) { p.epi = sg::EPI_SUBX; p.x = R.rows(Y.xtK, r, 0); p.row = {R.f(Y.esK), BH * N, tiles(m), 1.f}; }
            R.out_rows(p, R.f(side ? Y.dxtK : Y.dxtQ), r, false);
            sg::add(L, p);
        }
        R.gemms(L);
    }
    {   // dX = s dx~ M; dM = s sum dx~^T X over the tokens of both sides, per (b,h) and token block
        sg::Launch L;
        for (int side = 0; side < 2; ++side) {
            sg::Prob p = R.whole();
            p.A[0] = R.rows(side ? Y.dxtK : Y.dxtQ, r, 0); p.B[0] = R.paramM(M, 1); p.K[0] = r;
            p.mtok = 1; p.N = d; p.alpha = D.s;
            if (side && grouped) R.out_rows(p, R.f(Y.dKh), d, false);
            else R.out_rows(p, side ? dK : dQ, d, true);
            sg::add(L, p);
        }
        sg::Prob p = R.blocked(Y.nsM, Y.blkM);
        for (int side = 0; side < 2; ++side) {
            p.A[side] = R.rows(side ? Y.dxtK : Y.dxtQ, r, 1, Y.blkM); p.B[side] = R.input(side ? K : Q, d, side, 1, Y.blkM);
            p.K[side] = N; p.ktok[side] = 1;
        }
        p.M = r; p.N = d; p.alpha = D.s;
        R.out_blocks(p, Y.dMp, Y.nsM, r, d);
        sg::add(L, p);
        R.gemms(L);
    }
    const long long E = (long long)r * d;
    R.kernel(reduce_kernel, D.H * E, R.f(Y.dMp), dM, D.B, (long long)D.H, Y.nsM, E, D.H * E);
    if (grouped) {
        const long long BHkv = (long long)D.B * D.Hkv, nv = BHkv * N * dv, nk = BHkv * N * d;
        auto threads = [](long long n) { return n < 148LL * 16 * 256 ? n : 148LL * 16 * 256; };
        if (D.bf16) {
            R.kernel(group_sum_f32_kernel<__nv_bfloat16>, threads(nv), (__nv_bfloat16 *)dV, R.f(Y.dVh), D.G, (long long)N * dv, nv);
            R.kernel(group_sum_f32_kernel<__nv_bfloat16>, threads(nk), (__nv_bfloat16 *)dK, R.f(Y.dKh), D.G, (long long)N * d, nk);
        } else {
            R.kernel(group_sum_f32_kernel<float>, threads(nv), (float *)dV, R.f(Y.dVh), D.G, (long long)N * dv, nv);
            R.kernel(group_sum_f32_kernel<float>, threads(nk), (float *)dK, R.f(Y.dKh), D.G, (long long)N * d, nk);
        }
    }
    if (R.err != cudaSuccess) { set_cuda_error(R.err, "simt_backward"); return DARKATTN_ERR_CUDA; }
    return DARKATTN_OK;
}

// dW_l = sum_i E_il x~_i over queries and keys: E (in the buffers dA, dBf) and x~ are still in the workspace after
// simt_backward. Per (b,h) and token block, then the sum over those (and over the heads when W is shared).
darkattn_status_t simt_backward_dw(const darkattn_plan_s *plan, float *dW, char *ws, cudaStream_t st)
{
    const Dims &D = plan->dims;
    const SimtLayout &Y = plan->simt;
    Runner R{plan, ws, st};
    sg::Launch L;
    sg::Prob p = R.blocked(Y.nsW, Y.blkW);
    for (int side = 0; side < 2; ++side) {
        p.A[side] = R.rows(side ? Y.dBf : Y.dA, D.m, 1, Y.blkW); p.B[side] = R.rows(side ? Y.xtK : Y.xtQ, D.r, 1, Y.blkW);
        p.K[side] = D.N; p.ktok[side] = 1;
    }
    p.M = D.m; p.N = D.r;
    R.out_blocks(p, Y.dWp, Y.nsW, D.m, D.r);
    sg::add(L, p);
    R.gemms(L);
    const long long E = (long long)D.m * D.r;
    if (D.w_per_head) R.kernel(reduce_kernel, D.H * E, R.f(Y.dWp), dW, D.B, (long long)D.H, Y.nsW, E, D.H * E);
    else R.kernel(reduce_kernel, E, R.f(Y.dWp), dW, D.BH, 1LL, Y.nsW, E, E);
    if (R.err != cudaSuccess) { set_cuda_error(R.err, "simt_backward_dw"); return DARKATTN_ERR_CUDA; }
    return DARKATTN_OK;
}

}  // namespace darkattn
