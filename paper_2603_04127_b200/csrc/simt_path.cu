// FP32 path of libdarkattn: every step of DARK attention with fp32 operands and fp32 accumulation.
//
// This is the path that meets the 1e-4 tolerance (a single bf16 or TF32 operand rounds the argument of the exponential
// too coarsely), and the path that accepts any shape. Its products run on the tensor cores with every fp32 operand split
// into three bf16 numbers (split_gemm.cu); what surrounds them is done on the way out of a product, and intermediates are
// written as the bf16 parts that the next product reads:
//   forward    inputs into parts (fp32, or rows that do not start on 16 bytes) | x~ = s X M^T (row norms of the keys) |
//              key shifts c_l = max_j (u_jl - n_j), from the large parts alone | row maxima of the query exponents, likewise
//              (several tiles of features) | features phi = exp(x~ W^T ...) | chunk states and masked kernel tiles |
//              prefix over the chunks | output rows
//   backward   the forward steps with the output rows turned into dO / den and -delta / den | dP and the reverse states |
//              suffix over the chunks | E of both sides and dV | dx~ | dQ, dK and dM | sums over batch and token blocks;
//              with `saved` of the forward pass only x~ is formed again of its steps, and a launch makes the rows from O and the normaliser
// Each line's items between bars are one launch each; each starts while the one before drains
// (programmatic dependent launch). Chunks are 128 tokens, a tile's rows, whatever chunk length the descriptor names (the
// result does not depend on it).
//
// Stabiliser (cancels in O): keys use one shift per (batch, head, feature), c_l = max_j (u_jl - n_j),
// queries use e_il = u_il + c_l - max_l(u_il + c_l); the query's own norm term is a per-row constant
// and is dropped (so is its gradient, which is zero). The product phi(q_i)_l phi(k_j)_l is then the unshifted one times
// a per-row factor. Any constants near these maxima serve, so the maxima are taken from one bf16 product (x~'s and W's large
// parts: off by a few 2^-9 of the terms' size); the features themselves use the whole of both.
#include "common.cuh"
#include "split_gemm.cuh"
#include "tc_common.cuh"

#include <math.h>

namespace darkattn {

using sg::Mat;

namespace {

inline int tiles(int n) { return (n + 127) / 128; }
inline int up4(int n) { return (n + 3) & ~3; }
inline int up8(int n) { return (n + 7) & ~7; }

// Inputs into bf16 planes with rows a multiple of 8 apart: three of an fp32 tensor, one of a bf16 tensor. A thread handles eight
// columns of a row.
struct SplitJob { const void *in; __nv_bfloat16 *out; int w, ld, vec; long long rows, first; };     // first: threads of the jobs before
struct SplitJobs { SplitJob j[5]; int n; long long total; };

template <typename T>
__global__ void __launch_bounds__(256) split_inputs_kernel(const __grid_constant__ SplitJobs J)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    for (long long i = blockIdx.x * 256LL + threadIdx.x; i < J.total; i += gridDim.x * 256LL) {
        int k = 0;
        while (k + 1 < J.n && i >= J.j[k + 1].first) ++k;
        const SplitJob &b = J.j[k];
        const long long e = i - b.first;
        const int per = b.ld / 8, c = (int)(e % per) * 8;
        const long long row = e / per;
        const T *src = static_cast<const T *>(b.in) + row * b.w + c;
        __nv_bfloat16 *dst = b.out + row * b.ld + c;
        if constexpr (sizeof(T) == 2) {
            for (int j = 0; j < 8; ++j) dst[j] = c + j < b.w ? src[j] : __float2bfloat16_rn(0.f);
        } else {
            float x[8];
            if (b.vec) {
                const float4 a = *reinterpret_cast<const float4 *>(src), d = *(reinterpret_cast<const float4 *>(src) + 1);
                x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = d.x; x[5] = d.y; x[6] = d.z; x[7] = d.w;
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) x[j] = c + j < b.w ? src[j] : 0.f;
            }
#pragma unroll
            for (int pl = 0; pl < 3; ++pl) {
                uint32_t u[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    u[j] = tc::pack_bf16(x[2 * j], x[2 * j + 1]);
                    x[2 * j] -= __uint_as_float(u[j] << 16);
                    x[2 * j + 1] -= __uint_as_float(u[j] & 0xffff0000u);
                }
                *reinterpret_cast<uint4 *>(dst + pl * b.rows * b.ld) = make_uint4(u[0], u[1], u[2], u[3]);
            }
        }
    }
}

// Over the token blocks of S[pair, block, row, col]: what came before each block (forward) or comes after it (reverse), or the
// sum over all of them, as bf16 planes Sp [3][pair, block (or one)][m][ld]; z[pair, block, m4] the same in place (the sum into the
// first block). One thread per V neighbouring elements of a row; eight blocks' loads are in flight at a time (the sum is
// a serial chain, the loads are not).
enum { SCAN_FORWARD = 0, SCAN_REVERSE = 1, SCAN_TOTAL = 2 };
template <int V>
__global__ void __launch_bounds__(256) chunk_scan_kernel(const float *S, float *z, __nv_bfloat16 *Sp, int nb, int m, int dv, int ld, int m4, long long pairs, int mode)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const long long E = (long long)m * dv;
    long long i = blockIdx.x * 256LL + threadIdx.x;
    const int nout = mode == SCAN_TOTAL ? 1 : nb;
    if (i < pairs * E / V) {
        const long long pair = i * V / E, e = i * V % E;
        const float *src = S + pair * nb * E + e;
        __nv_bfloat16 *dst = Sp + (pair * nout * m + e / dv) * ld + e % dv;
        const long long dstep = (long long)m * ld, plane = pairs * nout * dstep;
        float run[V];
#pragma unroll
        for (int j = 0; j < V; ++j) run[j] = 0.f;
        auto emit = [&](__nv_bfloat16 *d) {
            float x[V];
#pragma unroll
            for (int j = 0; j < V; ++j) x[j] = run[j];
#pragma unroll
            for (int pl = 0; pl < 3; ++pl, d += plane) {
                if constexpr (V == 4) {
                    const uint32_t u0 = tc::pack_bf16(x[0], x[1]), u1 = tc::pack_bf16(x[2], x[3]);
                    *reinterpret_cast<uint2 *>(d) = make_uint2(u0, u1);
                    x[0] -= __uint_as_float(u0 << 16); x[1] -= __uint_as_float(u0 & 0xffff0000u);
                    x[2] -= __uint_as_float(u1 << 16); x[3] -= __uint_as_float(u1 & 0xffff0000u);
                } else {
                    const __nv_bfloat16 b = __float2bfloat16_rn(x[0]);
                    *d = b;
                    x[0] -= __bfloat162float(b);
                }
            }
        };
        for (int k0 = 0; k0 < nb; k0 += 8) {
            float x[8][V];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int c = mode == SCAN_REVERSE ? nb - 1 - (k0 + k) : k0 + k;
                if (k0 + k < nb) {
                    if constexpr (V == 4) { const float4 a = __ldg(reinterpret_cast<const float4 *>(src + c * E)); x[k][0] = a.x; x[k][1] = a.y; x[k][2] = a.z; x[k][3] = a.w; }
                    else x[k][0] = __ldg(src + c * E);
                }
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (k0 + k >= nb) break;
                const int c = mode == SCAN_REVERSE ? nb - 1 - (k0 + k) : k0 + k;
                if (mode != SCAN_TOTAL && k0 + k > 0) emit(dst + c * dstep);       // (the first one's state is zero and is not read)
#pragma unroll
                for (int j = 0; j < V; ++j) run[j] += x[k][j];
            }
        }
        if (mode == SCAN_TOTAL) emit(dst);
        return;
    }
    i -= pairs * E / V;
    if (i >= pairs * m) return;
    float *base = z + i / m * nb * m4 + i % m;
    float run = 0.f;
    for (int k = 0; k < nb; ++k) {
        float *p = base + (long long)(mode == SCAN_REVERSE ? nb - 1 - k : k) * m4;
        const float x = *p;
        if (mode != SCAN_TOTAL) *p = run;
        run += x;
    }
    if (mode == SCAN_TOTAL) base[0] = run;
}

// out[o, e] = sum of src over `n1` outer and `n2` inner slices: src[(i1 * stride1 + o) * n2 + i2, e]. dM sums over the batch
// and the token blocks (o = head), dW also over the heads where they share W (o = 0). SPLIT: eight warps of a block take every eighth slice
// of the same 32 elements, for few elements and many slices, where a thread for each that adds them up alone is a chain of load latencies
// (dW of m x r = 128 x 64 from 128 slices: 19 us). From 64 k elements on there are threads enough.
template <bool SPLIT>
__global__ void __launch_bounds__(256) reduce_kernel(const float *src, float *out, int n1, long long stride1, int n2, long long E, long long total)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __shared__ float part[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, n = n1 * n2;      // (SPLIT)
    const long long t = SPLIT ? blockIdx.x * 32LL + lane : blockIdx.x * 256LL + threadIdx.x;
    float acc = 0.f;
    if (t < total) {
        const long long o = t / E, e = t % E;
        if constexpr (SPLIT) {
#pragma unroll 4
            for (int k = w; k < n; k += 8) acc += src[(((k / n2) * stride1 + o) * n2 + k % n2) * E + e];
        } else
            for (int i1 = 0; i1 < n1; ++i1) {
                const float *p = src + (i1 * stride1 + o) * n2 * E + e;
#pragma unroll 8
                for (int i2 = 0; i2 < n2; ++i2) acc += p[i2 * E];
            }
    }
    if constexpr (SPLIT) {
        part[w][lane] = acc;
        __syncthreads();
        if (w) return;
        acc = ((part[0][lane] + part[1][lane]) + (part[2][lane] + part[3][lane])) + ((part[4][lane] + part[5][lane]) + (part[6][lane] + part[7][lane]));
    }
    if (t < total) out[t] = acc;
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

// Rows of the output's gradient, from what the forward pass left: Ga = dO / den as bf16 planes (rows `ld` apart, `plane` elements from plane to
// plane) and gd = -(dO . O) / den. A warp per row, one pass over 12 to 14 bytes an element in
// place of the output rows' products.
template <typename T>
__global__ void __launch_bounds__(256) grad_rows_kernel(const T *dO, const float *O, const float *den, __nv_bfloat16 *Ga, float *gd, int dv, int ld, long long plane, long long rows)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const int lane = threadIdx.x & 31;
    const long long row = blockIdx.x * 8LL + (threadIdx.x >> 5);
    if (row >= rows) return;
    const float inv = 1.f / den[row];
    float sum = 0.f;
    for (int c = lane; c < ld; c += 32) {
        float g = 0.f;
        if (c < dv) {
            if constexpr (sizeof(T) == 2) g = __bfloat162float(dO[row * dv + c]);
            else g = dO[row * dv + c];
            sum = fmaf(g, O[row * dv + c], sum);
        }
        float x = g * inv;
        __nv_bfloat16 *dst = Ga + row * ld + c;
#pragma unroll
        for (int pl = 0; pl < 3; ++pl) {
            const __nv_bfloat16 b = __float2bfloat16_rn(x);
            dst[pl * plane] = b;
            x -= __bfloat162float(b);
        }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) gd[row] = -inv * sum;
}

constexpr size_t kInSaved = (size_t)1 << 62;       // an offset into the caller's `saved` buffer instead of the workspace

struct Runner {
    const darkattn_plan_s *plan;
    const SimtLayout &Y;
    char *ws, *saved;
    cudaStream_t st;
    cudaError_t err = cudaSuccess;
    Mat Q, K, V, M, W;

    const Dims &D() const { return plan->dims; }
    char *at(size_t off) const { return off & kInSaved ? saved + (off ^ kInSaved) : ws + off; }
    float *f(size_t off) const { return reinterpret_cast<float *>(at(off)); }
    void keep(cudaError_t e) { if (e != cudaSuccess && err == cudaSuccess) err = e; }
    void gemms(sg::Launch &L) { L.status = reinterpret_cast<int *>(ws); keep(sg::run(L, st)); }
    template <typename... KA, typename... A>
    void kernel(void (*k)(KA...), long long threads, const A &...args)
    {
        keep(launch_pdl(k, dim3((unsigned)((threads + 255) / 256)), dim3(256), 0, st, args...));
    }

    // ---- matrices
    Mat planes(size_t off, long long batch, long long rows, int w) const
    {
        Mat m;
        m.p = reinterpret_cast<__nv_bfloat16 *>(at(off)); m.w = w; m.ld = up8(w); m.rows = rows; m.batch = batch;
        return m;
    }
    Mat tokens(size_t off, int w) const { return planes(off, D().BH, D().N, w); }
    Mat input(int i, const void *p, long long batch, long long rows, int w) const
    {
        Mat m = planes(Y.in[i], batch, rows, w);
        m.planes = D().bf16 ? 1 : 3;
        if (!Y.conv[i]) { m.p = const_cast<__nv_bfloat16 *>(static_cast<const __nv_bfloat16 *>(p)); m.ld = w; }
        return m;
    }
    // ---- operands
    sg::Op op(const Mat &m, int batch, int mn, int tok = 0) const { sg::Op o; o.m = m; o.batch = batch; o.mn = mn; o.tok = tok; return o; }
    sg::Op rows(const Mat &m, int mn) const { return op(m, sg::BATCH_PAIR, mn, 1); }       // token rows of the (batch, head)
    sg::Op kv(const Mat &m, int mn) const { return op(m, sg::BATCH_KV, mn, 1); }           // ... of its key/value head
    sg::Op block(const Mat &m, int mn) const { return op(m, sg::BATCH_BLOCK, mn); }
    sg::Op state(const Mat &m, int mn) const { return op(m, D().causal ? sg::BATCH_BLOCK : sg::BATCH_PAIR, mn); }
    sg::Op opM(int mn) const { return op(M, sg::BATCH_HEAD, mn); }
    sg::Op opW(int mn) const { return op(W, D().w_per_head ? sg::BATCH_HEAD : sg::BATCH_NONE, mn); }
    // ---- products over the whole sequence of every (batch, head), or over blocks of it
    sg::Prob prob(int nb = 1, int blk = 0) const
    {
        sg::Prob p;
        p.H = D().H; p.G = D().G; p.batch = D().BH; p.ntok = D().N; p.nblk = nb; p.block = blk;
        return p;
    }
    sg::Prob per_chunk() const { return D().causal ? prob(Y.nb, 128) : prob(); }
    void product(sg::Launch &L, sg::Prob &p, int s, const sg::Op &A, const sg::Op &B, int K, bool ktok = false, bool hi = false) const
    {
        sg::set_operand(L, p, 2 * s, A, hi);
        sg::set_operand(L, p, 2 * s + 1, B, hi);
        p.K[s] = K; p.ktok[s] = ktok;
    }
    void out_rows(sg::Prob &p, const Mat &m) const          // [BH, N, w]
    {
        p.okind = sg::OUT_PLANES; p.out = m.p; p.old_ = m.ld; p.ops = m.ps(); p.os_pair = m.bs(); p.os_blk = (long long)p.block * m.ld;
    }
    void out_blocks(sg::Prob &p, const Mat &m) const        // [BH, blocks, rows, w]
    {
        p.okind = sg::OUT_PLANES; p.out = m.p; p.old_ = m.ld; p.ops = m.ps(); p.os_blk = m.bs(); p.os_pair = p.nblk * m.bs();
    }
    void plain_rows(sg::Prob &p, void *o, int w, bool storage) const        // [BH, N, w]
    {
        p.out = o; p.old_ = w; p.os_pair = (long long)D().N * w; p.os_blk = (long long)p.block * w;
        p.okind = storage && D().bf16 ? sg::OUT_BF16 : sg::OUT_F32;
    }
    void plain_blocks(sg::Prob &p, size_t off, int nb, long long nrows, int w) const       // [BH, nb, rows, w]
    {
        p.out = f(off); p.old_ = w; p.os_blk = nrows * w; p.os_pair = nb * p.os_blk; p.okind = sg::OUT_F32;
    }
    void x_planes(sg::Prob &p, const Mat &m) const { p.xkind = sg::X_PLANES; p.x = m.p; p.xld = m.ld; p.xps = m.ps(); }
    // whether there are states at all: a causal sequence of one chunk has none
    bool states() const { return !D().causal || Y.nb > 1; }
    void scan(size_t S, size_t z, size_t Sp, int mode)
    {
        const long long E = (long long)D().m * D().dv, BH = D().BH;
        const int ld = up8(D().dv), m4 = up4(D().m);
        __nv_bfloat16 *out = reinterpret_cast<__nv_bfloat16 *>(at(Sp));
        if (D().dv % 4 == 0) kernel(chunk_scan_kernel<4>, BH * (E / 4 + D().m), (const float *)f(S), f(z), out, Y.nb, D().m, D().dv, ld, m4, BH, mode);
        else kernel(chunk_scan_kernel<1>, BH * (E + D().m), (const float *)f(S), f(z), out, Y.nb, D().m, D().dv, ld, m4, BH, mode);
    }
    void sum_slices(size_t src, float *out, int n1, long long stride1, int n2, long long E, long long total)
    {
        if (total < 65536) kernel(reduce_kernel<true>, 8 * total, (const float *)f(src), out, n1, stride1, n2, E, total);
        else kernel(reduce_kernel<false>, total, (const float *)f(src), out, n1, stride1, n2, E, total);
    }
    Mat state_planes(size_t off) const { return planes(off, (long long)D().BH * (D().causal ? Y.nb : 1), D().m, D().dv); }
};

// Inputs into parts (unless they are, in `saved`) and x~, the first two launches of either pass.
void run_projections(Runner &R, const void *Q, const void *K, const void *V, const void *M, const void *W, bool parts_kept)
{
    const Dims &D = R.D();
    const SimtLayout &Y = R.Y;
    const int N = D.N, d = D.d, r = D.r, m = D.m, dv = D.dv, m4 = up4(m);
    const long long BH = D.BH, BHkv = (long long)D.B * D.Hkv;
    R.Q = R.input(0, Q, BH, N, d); R.K = R.input(1, K, BHkv, N, d); R.V = R.input(2, V, BHkv, N, dv);
    R.M = R.input(3, M, D.H, r, d); R.W = R.input(4, W, D.w_per_head ? D.H : 1, m, r);
    const Mat *in[5] = {&R.Q, &R.K, &R.V, &R.M, &R.W};
    const void *src[5] = {Q, K, V, M, W};
    SplitJobs J;
    J.n = 0; J.total = 0;
    for (int i = 0; i < 5; ++i)
        if (Y.conv[i] && !parts_kept) {
            const Mat &x = *in[i];
            J.j[J.n++] = {src[i], x.p, x.w, x.ld, x.w % 8 == 0, x.rows * x.batch, J.total};
            J.total += x.rows * x.batch * (x.ld / 8);
        }
    if (J.n) {
        const long long threads = J.total < 148LL * 8 * 256 ? J.total : 148LL * 8 * 256;
        if (D.bf16) R.kernel(split_inputs_kernel<__nv_bfloat16>, threads, J);
        else R.kernel(split_inputs_kernel<float>, threads, J);
    }
    const Mat xt[2] = {R.tokens(Y.xtQ, r), R.tokens(Y.xtK, r)};
    int *cK = reinterpret_cast<int *>(R.f(Y.cK));
    {   // x~ = s X M^T
        sg::Launch L;
        for (int side = 0; side < 2; ++side) {
            sg::Prob p = R.prob();
            R.product(L, p, 0, side ? R.kv(R.K, 0) : R.rows(R.Q, 0), R.opM(0), d);
            p.mtok = 1; p.N = r; p.alpha = D.s; p.chain = 1;                // (the exponent's argument: the most sensitive)
            if (side) { p.epi = sg::EPI_SQUARES; p.sums = R.f(Y.nK); }
            R.out_rows(p, xt[side]);
            sg::add(L, p);
        }
        L.init = cK; L.init_n = (int)(BH * m4);
        R.gemms(L);
    }
}

// Features, states and output rows. With dO given the rows dO / den and -delta / den are formed in place of O; with `keep` the output in
// fp32 and the normaliser are also left in `saved`.
void run_forward_stages(Runner &R, const void *Q, const void *K, const void *V, const void *M, const void *W, void *O, const void *dO, const SimtSaved *keep)
{
    const Dims &D = R.D();
    const SimtLayout &Y = R.Y;
    const int N = D.N, r = D.r, m = D.m, dv = D.dv, nb = Y.nb, m4 = up4(m);
    const long long BH = D.BH;
    run_projections(R, Q, K, V, M, W, false);
    const Mat xt[2] = {R.tokens(Y.xtQ, r), R.tokens(Y.xtK, r)}, phi[2] = {R.tokens(Y.fQ, m), R.tokens(Y.fK, m)};
    int *cK = reinterpret_cast<int *>(R.f(Y.cK));
    const sg::TokVec norm = {R.f(Y.nK), BH * N, 4 * tiles(r), 0.5f}, rmax = {R.f(Y.rmax), BH * N, 4 * tiles(m), 1.f};
    auto exponents = [&](sg::Launch &L, int side, bool hi) {
        sg::Prob p = R.prob();
        R.product(L, p, 0, R.rows(xt[side], 0), R.opW(0), r, false, hi);
        p.mtok = 1; p.N = m; p.chain = hi ? 2 : 1; p.colmax = cK; p.colkey_ld = m4;
        return p;
    };
    {   // the keys' shifts
        sg::Launch L;
        sg::Prob p = exponents(L, 1, true);
        p.epi = sg::EPI_COLMAX; p.row = norm;
        sg::add(L, p);
        R.gemms(L);
    }
    if (tiles(m) > 1) {     // the rows' maxima of the queries' exponents
        sg::Launch L;
        sg::Prob p = exponents(L, 0, true);
        p.epi = sg::EPI_ROWMAX; p.sums = R.f(Y.rmax);
        sg::add(L, p);
        R.gemms(L);
    }
    {   // phi(Q), phi(K)
        sg::Launch L;
        for (int side = 0; side < 2; ++side) {
            sg::Prob p = exponents(L, side, false);
            p.epi = side ? sg::EPI_PHI_K : sg::EPI_PHI_Q;
            if (side) p.row = norm;
            else if (tiles(m) > 1) p.row = rmax;
            R.out_rows(p, phi[side]);
            sg::add(L, p);
        }
        R.gemms(L);
    }
    const Mat Sp = R.state_planes(Y.Sp), P = R.planes(Y.P, BH * nb, 128, 128);
    {   // S_c = phi(K_c)^T V_c, z_c = phi(K_c)^T 1 per token block; causal: P_c = tril(phi(Q_c) phi(K_c)^T)
        sg::Launch L;
        if (D.causal) {
            sg::Prob q = R.prob(nb, 128);
            R.product(L, q, 0, R.rows(phi[0], 0), R.rows(phi[1], 0), m);
            q.mtok = q.ntok_dim = 1; q.epi = sg::EPI_MASK;
            R.out_blocks(q, P);
            sg::add(L, q);
        }
        if (R.states()) {
            sg::Prob p = R.prob(nb, Y.blk);
            R.product(L, p, 0, R.rows(phi[1], 1), R.kv(R.V, 1), N, true);
            p.M = m; p.N = dv; p.dot[0] = sg::DOT_ONES; p.dot_out = R.f(Y.zloc); p.dot_ld = m4;
            if (!D.causal && nb == 1) R.out_blocks(p, Sp);
            else R.plain_blocks(p, Y.Sloc, nb, m, dv);
            sg::add(L, p);
        }
        R.gemms(L);
    }
    if (nb > 1) R.scan(Y.Sloc, Y.zloc, Y.Sp, D.causal ? SCAN_FORWARD : SCAN_TOTAL);
    {   // O = (P V + phi(Q) S_prev) / (P 1 + phi(Q) z_prev)
        sg::Launch L;
        sg::Prob p = R.per_chunk();
        if (D.causal) { R.product(L, p, 0, R.block(P, 0), R.kv(R.V, 1), 128, true); p.dot[0] = sg::DOT_ONES; p.skip2 = 0; }
        if (R.states()) {
            R.product(L, p, 1, R.rows(phi[0], 0), R.state(Sp, 1), m); p.dot[1] = sg::DOT_FEATURES;
            p.dotf = R.f(Y.zloc); p.vec_pair = (long long)nb * m4; p.vec_blk = D.causal ? m4 : 0;
        }
        p.mtok = 1; p.N = dv; p.epi = dO ? sg::EPI_GRAD : sg::EPI_DIVIDE;
        if (dO) {
            p.xkind = D.bf16 ? sg::X_BF16 : sg::X_F32; p.x = dO; p.xld = dv; p.sums = R.f(Y.gd);
            R.out_rows(p, R.tokens(Y.Ga, dv));
        } else R.plain_rows(p, O, dv, true);
        if (keep) { p.out2 = R.f(kInSaved | keep->O); p.den_out = R.f(kInSaved | keep->den); }
        sg::add(L, p);
        R.gemms(L);
    }
}

size_t take(size_t &off, size_t bytes)
{
    const size_t at = off;
    off += (bytes + 255) / 256 * 256;
    return at;
}

// Cuts N tokens into blocks (multiples of 64 tokens) so that `units` products of one block each are about one per SM, none
// shorter than two stages of the contraction.
void cut_tokens(int N, long long units, int most, int &nblk, int &blk)
{
    long long want = (148 + units - 1) / units;
    if (want > (N + 127) / 128) want = (N + 127) / 128;
    if (want > most) want = most;
    if (want < 1) want = 1;
    blk = (int)(((N + want - 1) / want + 63) / 64 * 64);
    nblk = (N + blk - 1) / blk;
}

// the inputs Q, K, V, M, W: width of a row, bytes as planes
int input_width(const Dims &D, int i) { return i == 2 ? D.dv : i == 4 ? D.r : D.d; }
size_t input_bytes(const Dims &D, int i)
{
    const size_t tokens = (size_t)D.N * (i == 0 ? D.BH : D.B * D.Hkv);
    const size_t rows = i < 3 ? tokens : i == 3 ? (size_t)D.H * D.r : (size_t)(D.w_per_head ? D.H : 1) * D.m;
    return (D.bf16 ? 1 : 3) * rows * up8(input_width(D, i)) * 2;
}

// `stash`: the layout of a call that has `saved`; what the forward pass leaves for the backward pass is there and takes no room in the
// workspace. (A step kept both places before: 17.1 KB of workspace a token and head beside 5.9 KB of stash at d = dv = 128, m = 256, causal,
// bf16, now 10.7; without a stash 17.1 as ever.)
SimtLayout make_layout(const Dims &D, bool backward, const SimtSaved *stash)
{
    SimtLayout Y = {};
    const size_t BH = D.BH, N = D.N, m = D.m, dv = D.dv, m4 = up4(D.m);
    if (D.causal) {
        Y.blk = 128;
        Y.nb = tiles(D.N);
    } else {
        // (the extra partial states never take more room than two rows of values per token)
        cut_tokens(D.N, (long long)BH * tiles(D.m) * tiles(D.dv), (int)(1 + 2 * N / m > 64 ? 64 : 1 + 2 * N / m), Y.nb, Y.blk);
    }
    const size_t nb = Y.nb;
    const bool states = !D.causal || nb > 1;
    auto planes = [](size_t rows, int w) { return 3 * rows * up8(w) * 2; };
    size_t off = 0;
    Y.status = take(off, 256);
    Y.cK = take(off, BH * m4 * 4);
    for (int i = 0; i < 5; ++i) Y.conv[i] = !D.bf16 || input_width(D, i) % 8;
    auto take_x = [&] {
        Y.xtQ = take(off, planes(BH * N, D.r)); Y.xtK = take(off, planes(BH * N, D.r));
        Y.nK = take(off, (size_t)4 * tiles(D.r) * BH * N * 4);
    };
    auto take_rmax = [&] { Y.rmax = tiles(D.m) > 1 ? take(off, (size_t)4 * tiles(D.m) * BH * N * 4) : 0; };
    // what the stash may hold
    auto keep = [&](size_t &at, size_t kept, size_t bytes) { at = stash ? kInSaved | kept : bytes ? take(off, bytes) : 0; };
    auto take_in = [&](int i) { if (Y.conv[i]) keep(Y.in[i], stash ? stash->in[i] : 0, input_bytes(D, i)); };
    auto take_features = [&] {
        keep(Y.fQ, stash ? stash->fQ : 0, planes(BH * N, D.m));
        keep(Y.fK, stash ? stash->fK : 0, planes(BH * N, D.m));
    };
    auto take_states = [&] {
        keep(Y.zloc, stash ? stash->zloc : 0, states ? BH * nb * m4 * 4 : 0);
        Y.Sloc = nb > 1 && !(backward && stash) ? take(off, BH * nb * m * dv * 4) : 0;
        keep(Y.Sp, stash ? stash->Sp : 0, states ? planes(BH * (D.causal ? nb : 1) * m, D.dv) : 0);
        keep(Y.P, stash ? stash->P : 0, D.causal ? planes(BH * nb * 128, 128) : 0);
    };
    if (!backward) {
        take_in(2);
        take_features();
        // What is done with once the features are formed; the states and kernel tiles take its place.
        const size_t mark = off;
        for (int i : {0, 1, 3, 4}) take_in(i);
        take_x();
        take_rmax();
        const size_t end = off;
        off = mark;
        take_states();
        Y.bytes = off < end ? end : off;
        return Y;
    }
    // First what a call with a stash has too, at the same places: dW reads E and x~ whichever call left them.
    take_x();
    Y.Ga = take(off, planes(BH * N, D.dv)); Y.gd = take(off, (size_t)4 * tiles(D.dv) * BH * N * 4);
    Y.dP = D.causal ? take(off, planes(BH * nb * 128, 128)) : 0;
    Y.rloc = states ? take(off, BH * nb * m4 * 4) : 0;
    Y.Rloc = nb > 1 ? take(off, BH * nb * m * dv * 4) : 0;
    Y.Rp = states ? take(off, planes(BH * (D.causal ? nb : 1) * m, D.dv)) : 0;
    Y.dA = take(off, planes(BH * N, D.m)); Y.dBf = take(off, planes(BH * N, D.m));
    Y.esK = take(off, (size_t)4 * tiles(D.m) * BH * N * 4);
    Y.dxtQ = take(off, planes(BH * N, D.r)); Y.dxtK = take(off, planes(BH * N, D.r));
    Y.dKh = D.G > 1 ? take(off, BH * N * D.d * 4) : 0; Y.dVh = D.G > 1 ? take(off, BH * N * dv * 4) : 0;
    cut_tokens(D.N, (long long)BH * tiles(D.r) * tiles(D.d), 64, Y.nsM, Y.blkM);
    cut_tokens(D.N, (long long)BH * tiles(D.m) * tiles(D.r), 64, Y.nsW, Y.blkW);
    Y.dMp = take(off, BH * Y.nsM * D.r * D.d * 4);
    Y.dWp = take(off, BH * Y.nsW * m * D.r * 4);
    if (!stash) take_rmax();
    for (int i = 0; i < 5; ++i) take_in(i);
    take_features();
    take_states();
    Y.bytes = off;
    return Y;
}

}  // namespace

void simt_make_layout(darkattn_plan_s *plan)
{
    const Dims &D = plan->dims;
    plan->simt = make_layout(D, true, nullptr);
    plan->simt_fwd = make_layout(D, false, nullptr);
    const SimtLayout &Y = plan->simt;
    SimtSaved &S = plan->simt_saved;
    const size_t BH = D.BH, N = D.N, nb = Y.nb;
    auto planes = [](size_t rows, int w) { return 3 * rows * up8(w) * 2; };
    const bool states = !D.causal || nb > 1;
    size_t off = 0;
    for (int i = 0; i < 5; ++i) S.in[i] = Y.conv[i] ? take(off, input_bytes(D, i)) : 0;
    S.fQ = take(off, planes(BH * N, D.m)); S.fK = take(off, planes(BH * N, D.m));
    S.P = take(off, D.causal ? planes(BH * nb * 128, 128) : 0);
    S.Sp = take(off, states ? planes(BH * (D.causal ? nb : 1) * D.m, D.dv) : 0);
    S.zloc = take(off, states ? BH * nb * up4(D.m) * 4 : 0);
    S.O = take(off, BH * N * D.dv * 4); S.den = take(off, BH * N * 4);
    S.bytes = off;
    plan->simt_stash = make_layout(D, true, &S);
    plan->simt_fwd_stash = make_layout(D, false, &S);
}

void simt_launches(const darkattn_plan_s *plan, bool saved, int &fwd, int &bwd)
{
    const Dims &D = plan->dims;
    const SimtLayout &Y = plan->simt;
    bool conv = false;
    for (bool c : Y.conv) conv = conv || c;
    const int scan = Y.nb > 1;
    fwd = (conv ? 1 : 0) + 5 + (tiles(D.m) > 1 ? 1 : 0) + scan;
    bwd = (saved ? 2 : fwd) + 1 + scan + 4 + (D.G > 1 ? 2 : 0);
}

// Estimated time in us of a call that fills the SMs: launches one after the other, then per pair the 128 x 128 tiles of all products
// (start and read-out, stages of 64 of the contraction; four fifths of a stage where the inputs are bf16). Fitted like ffma_cost_us.
double simt_cost_us(const darkattn_plan_s *plan, bool backward)
{
    const Dims &D = plan->dims;
    const double N = D.N, d = D.d, r = D.r, m = D.m, dv = D.dv, nb = tiles(D.N), more = nb > 1 ? 1 : 0;
    double count = 0, stages = 0;
    auto product = [&](double M, double Nn, double K, double times = 1) {
        const double t = times * ceil(M / 128) * ceil(Nn / 128);
        count += t;
        stages += t * ceil(K / 64);
    };
    product(N, r, d, 2); product(N, m, r, 3 + (tiles(D.m) > 1 ? 1 : 0));
    if (D.causal) { product(128, 128, m, nb); product(m, dv, 128, more * nb); product(128, dv, 128 + more * m, nb); }
    else { product(m, dv, N); product(N, dv, m); }
    if (backward) {
        if (D.causal) { product(128, 128, dv, nb); product(m, dv, 128, more * nb); product(128, m, 128 + more * dv, 2 * nb); product(128, dv, 128 + more * m, nb); }
        else { product(m, dv, N); product(N, m, dv, 2); product(N, dv, m); }
        product(N, r, m, 2); product(N, d, r, 2); product(r, d, 2 * N);
    }
    const double parts = D.bf16 ? 0.8 : 1.0;
    return backward ? 52 + D.BH * (9.2e-3 * count + 2.04e-2 * parts * stages) : 35 + D.BH * (1.7e-2 * count + 1.48e-2 * parts * stages);
}

darkattn_status_t simt_forward(const darkattn_plan_s *plan, const void *Q, const void *K, const void *V,
                               const void *M, const void *W, void *O, char *saved, char *ws, cudaStream_t st)
{
    const SimtLayout &Y = saved ? plan->simt_fwd_stash : plan->simt_fwd;
    Runner R{plan, Y, ws, saved, st};
    run_forward_stages(R, Q, K, V, M, W, O, nullptr, saved ? &plan->simt_saved : nullptr);
    if (R.err != cudaSuccess) { set_cuda_error(R.err, "simt_forward"); return DARKATTN_ERR_CUDA; }
    return DARKATTN_OK;
}

darkattn_status_t simt_backward(const darkattn_plan_s *plan, const void *Q, const void *K, const void *V,
                                const void *M, const void *W, const void *dO, const char *saved_in, void *dQ, void *dK, void *dV,
                                float *dM, char *ws, cudaStream_t st)
{
    const Dims &D = plan->dims;
    char *saved = const_cast<char *>(saved_in);     // (read only here)
    const SimtLayout &Y = saved ? plan->simt_stash : plan->simt;
    const int N = D.N, d = D.d, r = D.r, m = D.m, dv = D.dv, nb = Y.nb, m4 = up4(m);
    const long long BH = D.BH;
    Runner R{plan, Y, ws, saved, st};
    // With `saved` x~ alone is formed again (it stays in the workspace for dW), dO / den and -delta / den come from the kept output. Forward and
    // backward: fp32, 2 x 8 heads of 1000 tokens, d 64, m 128, with dW 240 -> 197 us; bf16, 12 heads of 1500 tokens, d 64, m 256 306 -> 230;
    // 8 heads of 3001 tokens on 4, d 128, m 256 522 -> 398; no mask, fp32, 2 x 8 heads of 1000 tokens 184 -> 150.
    if (saved) {
        run_projections(R, Q, K, V, M, W, true);
        const Mat ga = R.tokens(Y.Ga, dv);
        const float *O = R.f(kInSaved | plan->simt_saved.O), *den = R.f(kInSaved | plan->simt_saved.den);
        if (D.bf16) R.kernel(grad_rows_kernel<__nv_bfloat16>, BH * N * 32, (const __nv_bfloat16 *)dO, O, den, ga.p, R.f(Y.gd), dv, ga.ld, ga.ps(), BH * N);
        else R.kernel(grad_rows_kernel<float>, BH * N * 32, (const float *)dO, O, den, ga.p, R.f(Y.gd), dv, ga.ld, ga.ps(), BH * N);
    } else run_forward_stages(R, Q, K, V, M, W, nullptr, dO, nullptr);

    const bool grouped = D.G > 1;
    const sg::TokVec gd = {R.f(Y.gd), BH * N, saved ? 1 : 4 * tiles(dv), 1.f}, es = {R.f(Y.esK), BH * N, 4 * tiles(m), 1.f};
    const Mat xtK = R.tokens(Y.xtK, r), fQ = R.tokens(Y.fQ, m), fK = R.tokens(Y.fK, m), Ga = R.tokens(Y.Ga, dv), E[2] = {R.tokens(Y.dA, m), R.tokens(Y.dBf, m)};
    const Mat Sp = R.state_planes(Y.Sp), Rp = R.state_planes(Y.Rp), P = R.planes(Y.P, BH * nb, 128, 128), dP = R.planes(Y.dP, BH * nb, 128, 128);
    const Mat dxt[2] = {R.tokens(Y.dxtQ, r), R.tokens(Y.dxtK, r)};
    {   // R_c = phi(Q_c)^T Ga_c, rho_c = phi(Q_c)^T gd_c; causal: dP_c = tril(Ga_c V_c^T + gd_c)
        sg::Launch L;
        if (D.causal) {
            sg::Prob q = R.prob(nb, 128);
            R.product(L, q, 0, R.rows(Ga, 0), R.kv(R.V, 0), dv);
            q.mtok = q.ntok_dim = 1; q.epi = sg::EPI_MASK; q.row = gd;
            R.out_blocks(q, dP);
            sg::add(L, q);
        }
        if (R.states()) {
            sg::Prob p = R.prob(nb, Y.blk);
            R.product(L, p, 0, R.rows(fQ, 1), R.rows(Ga, 1), N, true);
            p.M = m; p.N = dv; p.dot[0] = sg::DOT_TOKENS; p.dott = gd; p.dot_out = R.f(Y.rloc); p.dot_ld = m4;
            if (!D.causal && nb == 1) R.out_blocks(p, Rp);
            else R.plain_blocks(p, Y.Rloc, nb, m, dv);
            sg::add(L, p);
        }
        R.gemms(L);
    }
    if (nb > 1) R.scan(Y.Rloc, Y.rloc, Y.Rp, D.causal ? SCAN_REVERSE : SCAN_TOTAL);
    {
        sg::Launch L;
        auto vec = [&](sg::Prob &p, size_t v) { if (R.states()) { p.colvec = R.f(v); p.vec_pair = (long long)nb * m4; p.vec_blk = D.causal ? m4 : 0; } };
        {   // E_Q = phi(Q) .* (dP phi(K) + Ga S_prev^T + gd z_prev^T)
            sg::Prob p = R.per_chunk();
            if (D.causal) { R.product(L, p, 0, R.block(dP, 0), R.rows(fK, 1), 128, true); p.skip2 = 0; }
            if (R.states()) R.product(L, p, 1, R.rows(Ga, 0), R.state(Sp, 0), dv);
            p.epi = sg::EPI_RANK1; p.row = gd; vec(p, Y.zloc);
            R.x_planes(p, fQ);
            p.mtok = 1; p.N = m;
            R.out_rows(p, E[0]);
            sg::add(L, p);
        }
        {   // E_K = phi(K) .* (dP^T phi(Q) + V R_next^T + rho_next^T), and its row sums
            sg::Prob p = R.per_chunk();
            if (D.causal) { R.product(L, p, 0, R.block(dP, 1), R.rows(fQ, 1), 128, true); p.skip2 = nb - 1; }
            if (R.states()) R.product(L, p, 1, R.kv(R.V, 0), R.state(Rp, 0), dv);
            p.epi = sg::EPI_RANK1; vec(p, Y.rloc);
            R.x_planes(p, fK); p.sums = R.f(Y.esK);
            p.mtok = 1; p.N = m;
            R.out_rows(p, E[1]);
            sg::add(L, p);
        }
        {   // dV = P^T Ga + phi(K) R_next
            sg::Prob p = R.per_chunk();
            if (D.causal) { R.product(L, p, 0, R.block(P, 1), R.rows(Ga, 1), 128, true); p.skip2 = nb - 1; }
            if (R.states()) R.product(L, p, 1, R.rows(fK, 0), R.state(Rp, 1), m);
            p.mtok = 1; p.N = dv;
            if (grouped) R.plain_rows(p, R.f(Y.dVh), dv, false);
            else R.plain_rows(p, dV, dv, true);
            sg::add(L, p);
        }
        R.gemms(L);
    }
    {   // dx~ = E W, for the keys minus rowsum(E) x~
        sg::Launch L;
        for (int side = 0; side < 2; ++side) {
            sg::Prob p = R.prob();
            R.product(L, p, 0, R.rows(E[side], 0), R.opW(1), m);
            p.mtok = 1; p.N = r;
            if (side) { p.epi = sg::EPI_SUBX; R.x_planes(p, xtK); p.row = es; }
            R.out_rows(p, dxt[side]);
            sg::add(L, p);
        }
        R.gemms(L);
    }
    {   // dX = s dx~ M; dM = s sum dx~^T X over the tokens of both sides, per (b,h) and token block
        sg::Launch L;
        for (int side = 0; side < 2; ++side) {
            sg::Prob p = R.prob();
            R.product(L, p, 0, R.rows(dxt[side], 0), R.opM(1), r);
            p.mtok = 1; p.N = d; p.alpha = D.s;
            if (side && grouped) R.plain_rows(p, R.f(Y.dKh), d, false);
            else R.plain_rows(p, side ? dK : dQ, d, true);
            sg::add(L, p);
        }
        sg::Prob p = R.prob(Y.nsM, Y.blkM);
        R.product(L, p, 0, R.rows(dxt[0], 1), R.rows(R.Q, 1), N, true);
        R.product(L, p, 1, R.rows(dxt[1], 1), R.kv(R.K, 1), N, true);
        p.M = r; p.N = d; p.alpha = D.s;
        R.plain_blocks(p, Y.dMp, Y.nsM, r, d);
        sg::add(L, p);
        R.gemms(L);
    }
    const long long Em = (long long)r * d;
    R.sum_slices(Y.dMp, dM, D.B, D.H, Y.nsM, Em, D.H * Em);
    if (grouped) {
        const long long BHkv = (long long)D.B * D.Hkv, nv = BHkv * N * dv, nk = BHkv * N * d;
        auto threads = [](long long n) { return n < 148LL * 16 * 256 ? n : 148LL * 16 * 256; };
        if (D.bf16) {
            R.kernel(group_sum_f32_kernel<__nv_bfloat16>, threads(nv), (__nv_bfloat16 *)dV, (const float *)R.f(Y.dVh), D.G, (long long)N * dv, nv);
            R.kernel(group_sum_f32_kernel<__nv_bfloat16>, threads(nk), (__nv_bfloat16 *)dK, (const float *)R.f(Y.dKh), D.G, (long long)N * d, nk);
        } else {
            R.kernel(group_sum_f32_kernel<float>, threads(nv), (float *)dV, (const float *)R.f(Y.dVh), D.G, (long long)N * dv, nv);
            R.kernel(group_sum_f32_kernel<float>, threads(nk), (float *)dK, (const float *)R.f(Y.dKh), D.G, (long long)N * d, nk);
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
    Runner R{plan, Y, ws, nullptr, st};
    sg::Launch L;
    sg::Prob p = R.prob(Y.nsW, Y.blkW);
    R.product(L, p, 0, R.rows(R.tokens(Y.dA, D.m), 1), R.rows(R.tokens(Y.xtQ, D.r), 1), D.N, true);
    R.product(L, p, 1, R.rows(R.tokens(Y.dBf, D.m), 1), R.rows(R.tokens(Y.xtK, D.r), 1), D.N, true);
    p.M = D.m; p.N = D.r;
    R.plain_blocks(p, Y.dWp, Y.nsW, D.m, D.r);
    sg::add(L, p);
    R.gemms(L);
    const long long E = (long long)D.m * D.r;
    if (D.w_per_head) R.sum_slices(Y.dWp, dW, D.B, D.H, Y.nsW, E, D.H * E);
    else R.sum_slices(Y.dWp, dW, D.BH, 1, Y.nsW, E, E);
    if (R.err != cudaSuccess) { set_cuda_error(R.err, "simt_backward_dw"); return DARKATTN_ERR_CUDA; }
    return DARKATTN_OK;
}

}  // namespace darkattn
