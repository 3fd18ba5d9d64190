// Batched products of fp32 accuracy on the tensor cores.
//
// An fp32 number is the exact sum of three bf16 numbers (24 = 3 x 8 significant bits): x = x0 + x1 + x2, each the bf16
// rounding of what the ones before left out, so |x1| <= 2^-9 |x| and |x2| <= 2^-18 |x|. The product of two of them is
//     x y = x0 y0 + (x0 y1 + x1 y0) + (x0 y2 + x1 y1 + x2 y0) + (terms below 2^-26 |x y|),
// i.e. six bf16 products that the tensor cores form exactly and add in fp32; what is left out is a quarter of an fp32
// product's own rounding. An operand stored in bf16 is its own first part and needs one plane instead of three (three
// products against an fp32 operand, one against another bf16 operand). Small terms are issued first, so that they are not
// rounded against the large ones one at a time.
//
// One CTA of 256 threads forms a 128 x (up to 128) tile of C, a stage of 64 elements of the contraction at a time: the
// threads read both operands from global memory in their natural layout (16-byte loads along the contiguous index, whichever
// of the product's dimensions that is), split them and write the planes to shared memory in the 128-byte-swizzled K-major
// or MN-major layout that the MMA reads; one thread issues the MMAs. A CTA needs 96 KB of shared memory and 256 columns of
// tensor memory: two share an SM, and one's loads and splits run under the other's MMAs.
//
// The code is one kernel of short loops: operand by operand through the same few hundred instructions, whatever the product.
// Most launches of a short call run each instruction once or twice per CTA, so the time of unrolled and specialised code was
// the time of fetching it (a 128 x 128 x 64 tile: 12 us as a kernel per product with everything unrolled).
//
// Accumulation: the tensor cores round a running sum towards zero at every step, which over a long contraction adds up to
// more than fp32's own rounding. So the large products x0 y0 and the small ones have accumulators of their own, and after
// every second stage (every stage where the exponent's argument is formed) both are added to sums in registers, rounded to nearest, and start from zero again: measured
// against float64 the path's results are closer than with a chain of fp32 FMAs.
//
// What bounds it: a full stage of six products is 24 MMAs of 64 cycles = 1536 cycles of the tensor pipe, but each reads 8 KB
// of shared memory and the planes are written there first: 192 + 96 KB, 2300 cycles of its 128 bytes per clock.
#include "split_gemm.cuh"
#include "tc_common.cuh"

namespace darkattn {
namespace sg {

using namespace tc;

namespace {

constexpr int kNT = 256;
constexpr int kPlane = 16384;                       // one bf16 plane of a 128 x 64 operand tile
constexpr int kOperand = 3 * kPlane;                // A's three planes, then B's
constexpr int kDot = 2 * kOperand;                  // float[128]: the rows' dot products
constexpr int kRow = kDot + 512;                    // float[128]: the rows' values of the epilogue
constexpr int kPart = kRow + 512;                   // float[8][128]: partial sums of MN-major dot products; [2][128]: of the rows' sums
constexpr int kTile = kPart + 4096;                 // the tile and its operands
constexpr int kBar = kTile + 256;                   // MMA barrier, tensor-memory slot
constexpr int kSmem = kBar + 64;
static_assert(2 * (kSmem + 1024) <= 233472, "two CTAs share an SM");
constexpr int kPitch = 72;                          // floats between rows of a warp's 32 x 64 staged piece: conflict-free
static_assert(8 * 32 * kPitch * 4 <= 2 * kOperand, "the staged pieces fit over the operand planes");

// An operand tile: rows of contiguous elements. MN-major: 64 rows along the contraction of 128 elements, else 128 rows of 64.
struct Src {
    const char *p;           // first element of the tile at contraction index 0
    long long ldb;           // bytes from row to row
    int rows, cols;          // of the matrix, counted from p (elements past them read as zero)
    int bf16, mn, vec, K;    // vec: rows start on 16 bytes
};
// where a tile stands
struct Tile {
    int z, pair, blk, b, h, hk, m0, n0, tn, Mlim, Nlim, pb, exists;
    long long tok0;
};
struct Shared { Tile t; Src s[4]; };                // operands A0, B0, A1, B1
static_assert(sizeof(Shared) <= kBar - kTile, "room for the tile");

__device__ __forceinline__ uint32_t fast_div(uint32_t n, const FastDiv &d) { return (__umulhi(n, d.mul) + n) >> d.shr; }

// Works out the CTA's tile and its operands: lane i < 4 of one warp the i-th operand.
__device__ __forceinline__ void decode(const Launch &L, Shared &sh, int lane)
{
    uint32_t w = blockIdx.x;
    int pb = 0;
    while (pb + 1 < L.n && w >= L.p[pb].blocks) { w -= L.p[pb].blocks; ++pb; }
    const Prob &P = L.p[pb];
    Tile t;
    const uint32_t z = fast_div(w, P.dTiles), tl = w - z * P.dTiles.d, tm = fast_div(tl, P.dTilesN), pair = fast_div(z, P.dBlk), b = fast_div(pair, P.dH);
    t.pb = pb;
    t.z = (int)z;
    t.tn = (int)(tl - tm * P.dTilesN.d);
    t.m0 = (int)tm * 128; t.n0 = t.tn * 128;
    t.pair = (int)pair; t.blk = (int)(z - pair * P.dBlk.d); t.b = (int)b; t.h = (int)(pair - b * P.dH.d); t.hk = (int)fast_div((uint32_t)t.h, P.dG);
    const int ntok = P.block ? min(P.block, P.ntok - t.blk * P.block) : P.ntok;       // tokens of this block
    t.tok0 = (long long)t.pair * P.ntok + (long long)t.blk * P.block;                 // first of them, in the per-token vectors
    t.Mlim = P.mtok ? ntok : P.M; t.Nlim = P.ntok_dim ? ntok : P.N;
    t.exists = t.m0 < t.Mlim && t.n0 < t.Nlim;                                        // (false: behind the end of a short last block)
    const int seg = lane >> 1, isB = lane & 1;
    int K = P.ktok[seg] ? min(ntok, P.K[seg]) : P.K[seg];
    if (P.epi == EPI_MASK && t.n0 > t.m0 + 127) K = 0;                                // wholly above the diagonal: nothing to multiply
    if (seg == 1 && P.skip2_first && t.blk == 0) K = 0;
    const Op &o = isB ? P.B[seg] : P.A[seg];
    const int es = o.bf16 ? 2 : 4, mn0 = isB ? t.n0 : t.m0, lim = (isB ? t.Nlim : t.Mlim) - mn0;
    Src s;
    s.K = K; s.bf16 = o.bf16; s.mn = o.mn;
    s.ldb = (long long)o.ld * es;
    s.p = static_cast<const char *>(o.p) + (t.b * o.sb + (o.kv ? t.hk : t.h) * o.sh + t.blk * o.sc) * es + (o.mn ? (long long)mn0 * es : mn0 * s.ldb);
    s.rows = o.mn ? K : lim; s.cols = o.mn ? lim : K;
    s.vec = ((reinterpret_cast<uintptr_t>(s.p) | (uintptr_t)s.ldb) & 15) == 0;
    sh.s[lane] = s;
    if (lane == 0) sh.t = t;
}

// A thread's share of an operand tile: four chunks of 8 contiguous elements per stage. K-major tiles are 128 rows of 8
// chunks (32 rows apart for a thread), MN-major tiles 64 rows of 16 (16 rows apart).
struct Place {
    const char *p; long long step; int row, rows, n, rstep;     // first chunk, bytes and rows to the next; elements of a chunk that exist
    __device__ __forceinline__ Place(const Src &s, int k0, int tid)
    {
        rstep = s.mn ? 16 : 32;
        row = s.mn ? k0 + (tid >> 4) : tid >> 3;
        const int col = s.mn ? (tid & 15) * 8 : k0 + (tid & 7) * 8;
        p = s.p + row * s.ldb + (col << (s.bf16 ? 1 : 2));
        step = rstep * s.ldb;
        rows = s.rows;
        n = s.cols - col;
    }
    __device__ __forceinline__ int count(int i) const { return row + i * rstep < rows ? n : 0; }
};

// Starts the loads. Rows start on 16 bytes and are whole 16-byte pieces apart, so a piece that begins inside the matrix ends
// inside its row; elements past the matrix are cleared afterwards (mend), as rows that start elsewhere are read there.
__device__ __forceinline__ void fetch(const Src &s, int k0, int tid, uint4 (&q)[4][2])
{
    const Place a(s, k0, tid);
    const bool vec = s.vec, second = !s.bf16;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int c = vec ? a.count(i) : 0;
        const uint4 *g = reinterpret_cast<const uint4 *>(a.p + i * a.step);
        q[i][0] = q[i][1] = make_uint4(0, 0, 0, 0);
        if (c > 0) q[i][0] = __ldg(g);
        if (c > 4 && second) q[i][1] = __ldg(g + 1);
    }
}

__device__ __noinline__ void mend_copy(const Src &s, int k0, int tid, uint4 (&q)[4][2])
{
    const Place a(s, k0, tid);
#pragma unroll 1
    for (int i = 0; i < 4; ++i) {
        const int c = a.count(i);
        uint32_t *u = reinterpret_cast<uint32_t *>(q[i]);
        if (!s.vec)
            for (int j = 0; j < 8; ++j) u[j] = 0u;
        for (int j = 0; j < 8; ++j) {
            if (!s.vec && j < c) {
                if (s.bf16) u[j >> 1] |= (uint32_t)__ldg(reinterpret_cast<const unsigned short *>(a.p + i * a.step) + j) << (16 * (j & 1));
                else u[j] = __ldg(reinterpret_cast<const uint32_t *>(a.p + i * a.step) + j);
            }
            if (j >= c) {
                if (s.bf16) u[j >> 1] &= (j & 1) ? 0xffffu : 0u;
                else u[j] = 0u;
            }
        }
    }
}
// chunks that lie partly outside the matrix, and rows that do not start on 16 bytes
__device__ __forceinline__ void mend(const Src &s, int k0, int tid, uint4 (&q)[4][2])
{
    const bool ragged = !s.vec || (s.mn ? (min(s.cols, 128) & 7) != 0 : (min(64, s.K - k0) & 7) != 0);     // (the same for all threads)
    if (!ragged) return;
    uint4 c[4][2];           // (a copy: the rare call must not put the caller's registers into memory)
#pragma unroll
    for (int i = 0; i < 4; ++i) { c[i][0] = q[i][0]; c[i][1] = q[i][1]; }
    mend_copy(s, k0, tid, c);
#pragma unroll
    for (int i = 0; i < 4; ++i) { q[i][0] = c[i][0]; q[i][1] = c[i][1]; }
}

// the three bf16 parts of a pair of fp32 numbers
__device__ __forceinline__ void split2(uint32_t ua, uint32_t ub, uint32_t &p0, uint32_t &p1, uint32_t &p2)
{
    const float a = __uint_as_float(ua), b = __uint_as_float(ub);
    p0 = pack_bf16(a, b);
    const float a1 = a - __uint_as_float(p0 << 16), b1 = b - __uint_as_float(p0 & 0xffff0000u);
    p1 = pack_bf16(a1, b1);
    p2 = pack_bf16(a1 - __uint_as_float(p1 << 16), b1 - __uint_as_float(p1 & 0xffff0000u));
}

// a thread's four chunks into the operand's planes
__device__ __forceinline__ void put(const Src &s, const uint4 (&q)[4][2], unsigned char *planes, int tid)
{
    unsigned char *d = planes + (s.mn ? ((tid & 8) << 10) + swz128(tid >> 4, tid & 7) : swz128(tid >> 3, tid & 7));
    const int step = s.mn ? 16 * 128 : 32 * 128;
    if (s.bf16) {
#pragma unroll
        for (int i = 0; i < 4; ++i) *reinterpret_cast<uint4 *>(d + i * step) = q[i][0];
        return;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i, d += step) {
        uint4 p0, p1, p2;
        split2(q[i][0].x, q[i][0].y, p0.x, p1.x, p2.x);
        split2(q[i][0].z, q[i][0].w, p0.y, p1.y, p2.y);
        split2(q[i][1].x, q[i][1].y, p0.z, p1.z, p2.z);
        split2(q[i][1].z, q[i][1].w, p0.w, p1.w, p2.w);
        *reinterpret_cast<uint4 *>(d) = p0;
        *reinterpret_cast<uint4 *>(d + kPlane) = p1;
        *reinterpret_cast<uint4 *>(d + 2 * kPlane) = p2;
    }
}

__device__ __forceinline__ float tok_value(const TokVec &t, long long at)
{
    float v = 0.f;
    for (int i = 0; i < t.parts; ++i) v += t.p[i * t.stride + at];
    return t.scale * v;
}

// Rows' dot products with a vector along the contraction, from a thread's chunks of an fp32 A on their way to shared memory:
// K-major A has one row and eight contraction indices per chunk (rd[i]), MN-major A eight rows (rd[j]) and one index.
__device__ __forceinline__ void add_dot(const Prob &P, const Tile &t, int kind, const Src &s, const uint4 (&q)[4][2], int k0, int tid, float (&rd)[8])
{
    if (kind == DOT_FEATURES) {
        const float *f = P.dotf + t.pair * P.vec_pair + t.blk * P.vec_blk;
        const int k = k0 + (tid & 7) * 8;
        float w[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) w[j] = __ldg(f + min(k + j, s.K - 1));
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t u[8] = {q[i][0].x, q[i][0].y, q[i][0].z, q[i][0].w, q[i][1].x, q[i][1].y, q[i][1].z, q[i][1].w};
#pragma unroll
            for (int j = 0; j < 8; ++j) rd[i] = fmaf(w[j], __uint_as_float(u[j]), rd[i]);
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t u[8] = {q[i][0].x, q[i][0].y, q[i][0].z, q[i][0].w, q[i][1].x, q[i][1].y, q[i][1].z, q[i][1].w};
        if (s.mn) {
            const float w = kind == DOT_TOKENS ? tok_value(P.dott, t.tok0 + min(k0 + (tid >> 4) + 16 * i, s.K - 1)) : 1.f;
#pragma unroll
            for (int j = 0; j < 8; ++j) rd[j] = fmaf(w, __uint_as_float(u[j]), rd[j]);
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) rd[i] += __uint_as_float(u[j]);
        }
    }
}

// 16 lanes x 32 columns of tensor memory in the fragment shape: v[4 k + 2 i + j] is row lane / 4 + 8 i, column 8 k + 2 (lane % 4) + j
__device__ __forceinline__ void tmem_ld_frag(uint32_t taddr, uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
}

// The accumulators of a warp's 32 rows and 64 columns (the MMAs have been waited for) into its sums.
// acc[c][16 hh + 4 k + 2 i + j]: column 32 c + 8 k + 2 (lane % 4) + j of row 16 hh + 8 i + lane / 4.
__device__ __forceinline__ void collect(uint32_t taddr, int cols, bool small, float (&acc)[2][32])
{
    tc_fence_after();
#pragma unroll
    for (int c = 0; c < 2; ++c)
        if (c * 32 < cols) {
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                uint32_t v[16];
                tmem_ld_frag(taddr + c * 32 + ((uint32_t)(hh * 16) << 16), v);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 16; ++j) acc[c][16 * hh + j] += __uint_as_float(v[j]);
                if (small) {
                    tmem_ld_frag(taddr + 128 + c * 32 + ((uint32_t)(hh * 16) << 16), v);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 16; ++j) acc[c][16 * hh + j] += __uint_as_float(v[j]);
                }
            }
        }
    tc_fence_before();
}

// four consecutive elements of a row; n of them exist (the others read as zero)
__device__ __forceinline__ float4 load4(const char *p, bool bf16, bool vec, int n)
{
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (bf16) {
        const unsigned short *s = reinterpret_cast<const unsigned short *>(p);
        if (vec && n >= 4) {
            const uint2 u = *reinterpret_cast<const uint2 *>(s);
            x = make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
        } else {
            x.x = __uint_as_float((uint32_t)s[0] << 16);
            if (n > 1) x.y = __uint_as_float((uint32_t)s[1] << 16);
            if (n > 2) x.z = __uint_as_float((uint32_t)s[2] << 16);
            if (n > 3) x.w = __uint_as_float((uint32_t)s[3] << 16);
        }
    } else {
        const float *s = reinterpret_cast<const float *>(p);
        if (vec && n >= 4) x = *reinterpret_cast<const float4 *>(s);
        else {
            x.x = s[0];
            if (n > 1) x.y = s[1];
            if (n > 2) x.z = s[2];
            if (n > 3) x.w = s[3];
        }
    }
    return x;
}
__device__ __forceinline__ void store4(char *p, bool bf16, bool vec, int n, float4 x)
{
    if (bf16) {
        __nv_bfloat16 *d = reinterpret_cast<__nv_bfloat16 *>(p);
        if (vec && n >= 4) *reinterpret_cast<uint2 *>(d) = make_uint2(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w));
        else {
            d[0] = __float2bfloat16_rn(x.x);
            if (n > 1) d[1] = __float2bfloat16_rn(x.y);
            if (n > 2) d[2] = __float2bfloat16_rn(x.z);
            if (n > 3) d[3] = __float2bfloat16_rn(x.w);
        }
    } else {
        float *d = reinterpret_cast<float *>(p);
        if (vec && n >= 4) *reinterpret_cast<float4 *>(d) = x;
        else {
            d[0] = x.x;
            if (n > 1) d[1] = x.y;
            if (n > 2) d[2] = x.z;
            if (n > 3) d[3] = x.w;
        }
    }
}

// a / b: the product with the reciprocal of b, corrected by the remainder
__device__ __forceinline__ float quotient(float a, float b, float inv)
{
    const float q = a * inv;
    return fmaf(fmaf(-q, b, a), inv, q);
}

// Writes a warp's 32 rows and 64 columns, staged in shared memory: half a warp per row, four columns per lane.
template <int EPI>
__device__ __forceinline__ void write_rows(const Prob &P, const Tile &t, unsigned char *smem, const float *stage, int warp, int lane)
{
    constexpr bool kX = EPI == EPI_RANK1 || EPI == EPI_SUBX || EPI == EPI_GRAD, kSum = EPI == EPI_RANK1 || EPI == EPI_GRAD || EPI == EPI_SQUARES;
    const float *sDot = reinterpret_cast<const float *>(smem + kDot), *sRow = reinterpret_cast<const float *>(smem + kRow);
    float *sPart = reinterpret_cast<float *>(smem + kPart);
    const int half = warp >> 2, col = t.n0 + half * 64 + (lane & 15) * 4, n = t.Nlim - col;       // this lane's columns (n of them exist)
    const int oes = P.obf16 ? 2 : 4, xes = P.x.bf16 ? 2 : 4;
    const char *xb = nullptr;
    long long xld = 0;
    bool xvec = false;
    if (kX) {
        xb = static_cast<const char *>(P.x.p) + (t.b * P.x.sb + (P.x.kv ? t.hk : t.h) * P.x.sh + t.blk * P.x.sc + col) * xes;
        xld = (long long)P.x.ld * xes;
        xvec = ((reinterpret_cast<uintptr_t>(xb) | (uintptr_t)xld) & (4 * xes - 1)) == 0;
    }
    char *out = static_cast<char *>(P.out) + (t.b * P.osb + t.h * P.osh + t.blk * P.osc + col) * oes;
    const long long oldb = (long long)P.old_ * oes;
    const bool ovec = ((reinterpret_cast<uintptr_t>(out) | (uintptr_t)oldb) & (4 * oes - 1)) == 0, obf = P.obf16;
    float4 f1 = make_float4(0.f, 0.f, 0.f, 0.f), cm = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    if (EPI == EPI_RANK1 && n > 0) f1 = load4(reinterpret_cast<const char *>(P.rank1 + t.pair * P.vec_pair + t.blk * P.vec_blk + col), false, false, n);
    const bool has_row = P.row.p != nullptr;
    const float alpha = P.alpha;
    const int rbase = (warp & 3) * 32;
#pragma unroll 4
    for (int it = 0; it < 16; ++it) {
        const int rp = it * 2 + (lane >> 4), rl = rbase + rp, row = t.m0 + rl;
        const bool live = row < t.Mlim && n > 0;
        float4 x = *reinterpret_cast<const float4 *>(stage + rp * kPitch + (lane & 15) * 4);
        x = make_float4(alpha * x.x, alpha * x.y, alpha * x.z, alpha * x.w);
        const float v = has_row ? sRow[rl] : (EPI == EPI_RANK1 ? 1.f : 0.f);
        float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
        if (kX && live) y = load4(xb + row * xld, P.x.bf16, xvec, n);
        float part = 0.f;                       // this lane's share of the row's sum
        if (EPI == EPI_KEY_EXPONENT) {
            x.x -= v; x.y -= v; x.z -= v; x.w -= v;
            if (live) cm = make_float4(fmaxf(cm.x, x.x), fmaxf(cm.y, x.y), fmaxf(cm.z, x.z), fmaxf(cm.w, x.w));
        }
        if (EPI == EPI_MASK) {
            x.x = col > row ? 0.f : x.x + v; x.y = col + 1 > row ? 0.f : x.y + v;
            x.z = col + 2 > row ? 0.f : x.z + v; x.w = col + 3 > row ? 0.f : x.w + v;
        }
        if (EPI == EPI_DIVIDE) {
            const float den = sDot[rl], inv = 1.f / den;
            x = make_float4(quotient(x.x, den, inv), quotient(x.y, den, inv), quotient(x.z, den, inv), quotient(x.w, den, inv));
        }
        if (EPI == EPI_GRAD) {
            const float inv = 1.f / sDot[rl];
            part = -inv * (fmaf(y.x, x.x * inv, y.y * (x.y * inv)) + fmaf(y.z, x.z * inv, y.w * (x.w * inv)));
            x = make_float4(y.x * inv, y.y * inv, y.z * inv, y.w * inv);
        }
        if (EPI == EPI_RANK1) {
            x = make_float4(y.x * fmaf(v, f1.x, x.x), y.y * fmaf(v, f1.y, x.y), y.z * fmaf(v, f1.z, x.z), y.w * fmaf(v, f1.w, x.w));
            part = (x.x + x.y) + (x.z + x.w);
        }
        if (EPI == EPI_SUBX) x = make_float4(fmaf(-v, y.x, x.x), fmaf(-v, y.y, x.y), fmaf(-v, y.z, x.z), fmaf(-v, y.w, x.w));
        if (EPI == EPI_SQUARES) part = fmaf(x.x, x.x, x.y * x.y) + fmaf(x.z, x.z, x.w * x.w);
        if (live) store4(out + row * oldb, obf, ovec, n, x);
        if (kSum) {
#pragma unroll
            for (int o = 8; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
            if ((lane & 15) == 0) sPart[half * 128 + rl] = part;
        }
    }
    if (EPI == EPI_KEY_EXPONENT) {              // maxima over the warp's rows, then (in memory) over all rows
        float m[4] = {cm.x, cm.y, cm.z, cm.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            m[j] = fmaxf(m[j], __shfl_xor_sync(0xffffffffu, m[j], 16));
            if (lane < 16 && j < n) atomicMax(P.colmax + (long long)t.pair * P.N + col + j, float_order_key(m[j]));
        }
    }
}

__global__ void __launch_bounds__(kNT, 2) split_gemm_kernel(const __grid_constant__ Launch L)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + kBar);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bar + 1);
    Shared &sh = *reinterpret_cast<Shared *>(smem + kTile);
    float *sDot = reinterpret_cast<float *>(smem + kDot), *sRow = reinterpret_cast<float *>(smem + kRow), *sPart = reinterpret_cast<float *>(smem + kPart);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (warp == 0) {
        if (lane == 0) { mbar_init(bar, 1); fence_mbar_init(); }
        tmem_alloc(tmem_slot, 256);
        tmem_relinquish();
    } else if (warp == 1 && lane < 4) decode(L, sh, lane);
    if (L.init) {               // (the first launch of a call: nothing of it runs before)
        if (blockIdx.x == 0 && tid == 0) *L.status = 0;
        for (int i = blockIdx.x * kNT + tid; i < L.init_n; i += gridDim.x * kNT) L.init[i] = (int)0x80000000u;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const Tile &t = sh.t;
    const Prob &P = L.p[t.pb];
    asm volatile("griddepcontrol.wait;" ::: "memory");         // what came before (the index arithmetic did not need it)
    asm volatile("griddepcontrol.launch_dependents;");

    if (t.exists) {
        const int nw = (min(t.Nlim - t.n0, 128) + 15) & ~15;                            // columns of the tile, in the MMA's granularity
        const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (warp >> 2) * 64;
        const int cols = nw - (warp >> 2) * 64;                                         // of which this warp's (may be negative or above 64)
        if (P.row.p && tid < 128) sRow[tid] = t.m0 + tid < t.Mlim ? tok_value(P.row, t.tok0 + t.m0 + tid) : 0.f;
        float acc[2][32], rd[8];
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[0][j] = acc[1][j] = 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j) rd[j] = 0.f;
        bool ok = true;                     // false once a wait gave up (the status word says so)
        int issued = 0, chain = 0, small = 0;       // stages issued; of which in the accumulators; whether the small products' one is in use
        uint4 q[4][2];
        int seg = sh.s[0].K > 0 ? 0 : 1, o = 0, k0 = 0;
        bool more = sh.s[2 * seg].K > 0;
        if (more) fetch(sh.s[2 * seg], 0, tid, q);
        while (more) {                      // one operand of one stage per turn: A, B, A, ...
            const Src &s = sh.s[2 * seg + o];
            if (o == 0 && issued) {
                ok = ok && mbar_wait(bar, (issued - 1) & 1, L.status);                  // the MMAs of the stage before have read the planes
                if (chain >= P.chain) { collect(taddr, cols, small, acc); chain = 0; small = 0; }
            }
            mend(s, k0, tid, q);
            put(s, q, smem + o * kOperand, tid);
            if (o == 0 && P.dot[seg] != DOT_NONE) add_dot(P, t, P.dot[seg], s, q, k0, tid, rd);
            // the next operand's loads
            const int seg0 = seg;
            if (o == 0) o = 1;
            else {
                o = 0;
                k0 += 64;
                if (k0 >= s.K) { k0 = 0; ++seg; }
                more = seg < 2 && sh.s[2 * seg].K > 0;
            }
            if (more) fetch(sh.s[2 * seg + o], k0, tid, q);
            if (o == 1) continue;
            fence_async_smem();
            tc_fence_before();
            __syncthreads();
            const Src &sa = sh.s[2 * seg0], &sb = sh.s[2 * seg0 + 1];
            if (tid == 0) {
                tc_fence_after();
                const uint32_t idesc = make_idesc(128, nw, sa.mn, sb.mn);
                const uint32_t base = smem_u32(smem);
                const uint64_t dA = make_sdesc(base, sa.mn ? 8192 : 16, 1024), dB = make_sdesc(base + kOperand, sb.mn ? 8192 : 16, 1024);
                const uint64_t stA = (sa.mn ? 2048 : 32) >> 4, stB = (sb.mn ? 2048 : 32) >> 4;
                const int pa = sa.bf16 ? 1 : 3, pb = sb.bf16 ? 1 : 3;
                bool again = small;
                for (int i = 0; i < pa; ++i)
                    for (int j = 0; j < pb && i + j < 3; ++j) {
                        const uint32_t d = tmem + (i + j ? 128 : 0);
                        const uint64_t a0 = dA + (uint64_t)((i * kPlane) >> 4), b0 = dB + (uint64_t)((j * kPlane) >> 4);
                        mma_ss(d, a0, b0, idesc, i + j ? again : chain > 0);
                        mma_ss(d, a0 + stA, b0 + stB, idesc, 1);
                        mma_ss(d, a0 + 2 * stA, b0 + 2 * stB, idesc, 1);
                        mma_ss(d, a0 + 3 * stA, b0 + 3 * stB, idesc, 1);
                        again |= i + j > 0;
                    }
                mma_commit(bar);
            }
            small |= !(sa.bf16 && sb.bf16);
            ++issued; ++chain;
        }
        // rows' dot products: sum over the threads that share a row
        if (P.dot_out) {
#pragma unroll
            for (int j = 0; j < 8; ++j) rd[j] += __shfl_xor_sync(0xffffffffu, rd[j], 16);
            if (lane < 16)
#pragma unroll
                for (int j = 0; j < 8; ++j) sPart[warp * 128 + lane * 8 + j] = rd[j];
        } else if (P.epi == EPI_DIVIDE || P.epi == EPI_GRAD) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
#pragma unroll
                for (int f = 4; f; f >>= 1) rd[i] += __shfl_xor_sync(0xffffffffu, rd[i], f);
                if ((tid & 7) == 0) sDot[i * 32 + (tid >> 3)] = rd[i];
            }
        }
        if (issued) {
            ok = ok && mbar_wait(bar, (issued - 1) & 1, L.status);
            collect(taddr, cols, small, acc);
        }
        __syncthreads();                    // (every warp has seen the MMAs done: the planes are free)
        if (P.dot_out && t.tn == 0 && tid < 128 && t.m0 + tid < t.Mlim) {
            float v = 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i) v += sPart[i * 128 + tid];
            P.dot_out[(long long)t.z * P.M + t.m0 + tid] = v;
        }
        float *stage = reinterpret_cast<float *>(smem) + warp * 32 * kPitch;
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int j = 0; j < 32; j += 2) {
                const int row = 16 * (j >> 4) + 8 * ((j >> 1) & 1) + (lane >> 2), cc = 32 * c + 8 * ((j >> 2) & 3) + 2 * (lane & 3);
                // (columns past the tile's last were not written by its MMAs)
                *reinterpret_cast<float2 *>(stage + row * kPitch + cc) = cc < cols ? make_float2(acc[c][j], acc[c][j + 1]) : make_float2(0.f, 0.f);
            }
        __syncwarp();
        switch (P.epi) {
        case EPI_SQUARES: write_rows<EPI_SQUARES>(P, t, smem, stage, warp, lane); break;
        case EPI_KEY_EXPONENT: write_rows<EPI_KEY_EXPONENT>(P, t, smem, stage, warp, lane); break;
        case EPI_MASK: write_rows<EPI_MASK>(P, t, smem, stage, warp, lane); break;
        case EPI_DIVIDE: write_rows<EPI_DIVIDE>(P, t, smem, stage, warp, lane); break;
        case EPI_GRAD: write_rows<EPI_GRAD>(P, t, smem, stage, warp, lane); break;
        case EPI_RANK1: write_rows<EPI_RANK1>(P, t, smem, stage, warp, lane); break;
        case EPI_SUBX: write_rows<EPI_SUBX>(P, t, smem, stage, warp, lane); break;
        default: write_rows<EPI_PLAIN>(P, t, smem, stage, warp, lane); break;
        }
        if (P.sums) {                       // the rows' sums over the tile's columns
            __syncthreads();
            const int row = t.m0 + tid;
            if (tid < 128 && row < t.Mlim) P.sums[(long long)t.tn * P.batch * P.ntok + t.tok0 + row] = sPart[tid] + sPart[128 + tid];
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 256);
}

}  // namespace

// n / d for n < 2^31 as (high word of n mul + n) >> shr
static FastDiv make_div(unsigned d)
{
    FastDiv f;
    f.d = d; f.shr = 0;
    while ((1u << f.shr) < d) ++f.shr;
    f.mul = (unsigned)(((1ull << 32) * ((1ull << f.shr) - d)) / d + 1);
    return f;
}

void add(Launch &L, Prob p)
{
    const int M = p.mtok ? (p.block ? p.block : p.ntok) : p.M, N = p.ntok_dim ? (p.block ? p.block : p.ntok) : p.N;
    const unsigned tilesM = (M + 127) / 128, tilesN = (N + 127) / 128;
    p.blocks = (unsigned)p.batch * p.nblk * tilesM * tilesN;
    p.dTiles = make_div(tilesM * tilesN); p.dTilesN = make_div(tilesN);
    p.dBlk = make_div((unsigned)p.nblk); p.dH = make_div((unsigned)p.H); p.dG = make_div((unsigned)p.G);
    L.total += p.blocks;
    L.p[L.n++] = p;
}

cudaError_t run(const Launch &L, cudaStream_t st, bool dependent)
{
    static_assert(sizeof(Launch) <= 4000, "kernel parameter space");
    cudaError_t e = cudaFuncSetAttribute(split_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(split_gemm_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    return launch_pdl(split_gemm_kernel, dim3(L.total), dim3(kNT), kSmem, st, dependent, L);
}

}  // namespace sg
}  // namespace darkattn
