// Batched products of fp32 accuracy on the tensor cores.
//
// An fp32 number is the exact sum of three bf16 numbers (24 = 3 x 8 significant bits): x = x0 + x1 + x2, each the bf16
// rounding of what the ones before left out, so |x1| <= 2^-9 |x| and |x2| <= 2^-18 |x|. The product of two of them is
//     x y = x0 y0 + (x0 y1 + x1 y0) + (x0 y2 + x1 y1 + x2 y0) + (terms below 2^-26 |x y|),
// i.e. six bf16 products that the tensor cores form exactly and add in fp32; what is left out is a quarter of an fp32
// product's own rounding. An operand stored in bf16 is its own first part and needs one plane instead of three (three
// products against an fp32 operand, one against another bf16 operand).
//
// The parts are formed once, by whoever writes a matrix, and kept as three planes in memory (6 bytes an element instead of 4).
// So the kernel that multiplies has no conversion to do: one persistent CTA per SM whose warps have roles. One thread issues
// TMA loads (all planes of an operand's 64-wide stage in one or two instructions; what lies past a matrix arrives as
// zeros, so no size needs care) into a ring of as many stages as fit, one issues the MMAs, two warps form dot products
// of A's rows with a vector where a product needs them, sixteen warps read finished accumulators, apply what the path does to
// the element, split it again and store the planes, while the next tile is multiplied.
// (Splitting in the consumer, every tile by every CTA that reads it, was bound by the latency and the issue slots of the
// loading threads: 453 us for the forward pass of 2 x 16 heads of 2001 tokens, d = 128, m = 256.)
//
// Accumulation: the tensor cores round a running sum towards zero at every step, which over a long contraction adds up to
// more than fp32's own rounding. So the large products x0 y0 and the small ones have accumulators of their own, and after
// every second stage (every stage where the exponent's argument is formed) both are added to sums in registers, rounded to
// nearest, and start from zero again: measured against float64 the path's results are closer than with a chain of fp32 FMAs.
//
// What bounds it: a launch of few tiles the latencies of one: parameters, loads, MMAs, epilogue, about 5 us. With all SMs busy no unit by
// the counters (2 x 16 heads of 2001 tokens, d 128, m 256, the six launches of a forward call): tensor pipe 5 to 21 % of the time, L2 5 to 8 TB/s in the four
// long ones, which is 21 to 30 % of its peak, DRAM up to 54 %, an instruction issued in 31 to 45 % of the cycles; the sixteen read-out warps mostly
// wait for memory, tensor memory and barriers. The MMA warp runs converged (tc::elect_one): by a lane of its own the 24 MMAs of a stage of six
// products took 97 cycles each, whatever their width. All roles' code passes through every SM's instruction cache, so its size counts (162 -> 136 KB
// by the waits' small loop, 101 by small loops for x and the plain output, 90 by the issue), and so do reads of the launch's parameters (kept in shared
// memory). With all of this 2 x 16 heads of 2001 tokens, d 128, m 256: 380 -> 337 us; training
// step of 2 x 8 heads, 1000 tokens, d 64, fp32: 291 -> 242 us (191 with the stash), mostly by the coalesced loads of x in the backward products.
#include "split_gemm.cuh"
#include "tc_common.cuh"

#include <string.h>

namespace darkattn {
namespace sg {

using namespace tc;

namespace {

constexpr int kEpi = 16, kLoadWarp = 16, kMmaWarp = 17, kDotWarp = 18, kDots = 2, kNT = 640;     // warps 0..15 write out, 18 and 19 form dot products
constexpr int kPlane = 16384;                       // one bf16 plane of a 128 x 64 operand tile
constexpr int kRing = 12;                           // planes
constexpr int kMaxStages = 6;
constexpr int kStg = kRing * kPlane;                // 2 KB per epilogue warp: what is on its way out
constexpr int kDot = kStg + 2 * kPlane;             // float[2][128]: the rows' dot products
constexpr int kWt = kDot + 1024;                    // float[64]: the vector's part of a stage; float[128]: half of the MN-major sums
constexpr int kBar = kWt + 768;
// The products' descriptions: a tile's steps read some forty fields of them, chosen by the tile's product, and an indexed read of
// the launch's parameters takes well over 100 cycles (it misses the constant cache that all roles share).
constexpr int kBody = kBar + 176;
constexpr int kSmem = (kBody + kMaxProbs * (int)sizeof(ProbBody) + 15) / 16 * 16;
static_assert(sizeof(ProbBody) % 8 == 0, "read as words from 8-byte aligned places");
static_assert(kSmem <= 232448, "shared memory budget of one CTA exceeded");
constexpr float kLog2e = 1.4426950408889634f;
// Key features are kept 2^24 times too large (a common factor, it cancels). A causal prefix may hold only keys far below the sequence's
// largest: so their features keep all their digits down to 2^-126 of the largest and do not vanish before 2^-150, the range of an fp32
// number with its subnormals (ex2 flushes those, and the third part of a number below 2^-110 is one). Queries and keys eight times the
// usual size had twice as many undefined rows without it as an fp32 exponential leaves, and errors of 2e-3 in others; now
// fewer and 7e-5. Exponents above the line are multiplied after ex2, not shifted before it: 24 added to an exponent near 0 costs it
// four bits (0.82 -> 0.94e-6 of error in the results). 2 x 16 heads of 2001 tokens, d 128, m 256: 374 -> 380 us.
constexpr float kKeyScale = 16777216.f, kKeyScaleLog2 = 24.f, kKeyScaleLine = -100.f;

struct Tile { int pb, z, pair, blk, h, hk, m0, n0, tn, Mlim, Nlim, K0, K1, total, n0st; };

__device__ __forceinline__ uint32_t fast_div(uint32_t n, const FastDiv &d) { return (__umulhi(n, d.mul) + n) >> d.shr; }

__device__ __forceinline__ void decode(const Launch &L, const ProbBody *body, uint32_t w, Tile &t)
{
    if (w >= L.total) return;
    int pb = 0;
    while (pb + 1 < L.n && w >= body[pb].blocks) { w -= body[pb].blocks; ++pb; }
    const ProbBody &P = body[pb];
    const uint32_t z = fast_div(w, P.dTiles), tl = w - z * P.dTiles.d, tm = fast_div(tl, P.dTilesN), pair = fast_div(z, P.dBlk), b = fast_div(pair, P.dH);
    t.pb = pb;
    t.z = (int)z;
    t.tn = (int)(tl - tm * P.dTilesN.d);
    t.m0 = (int)tm * 128; t.n0 = t.tn * 128;
    t.pair = (int)pair; t.blk = (int)(z - pair * P.dBlk.d);
    t.h = (int)(pair - b * P.dH.d);
    t.hk = (int)(b * (P.dH.d / P.dG.d) + fast_div((uint32_t)t.h, P.dG));                // key/value head, counted over the batch
    const int ntok = P.block ? min(P.block, P.ntok - t.blk * P.block) : P.ntok;         // tokens of this block
    t.Mlim = P.mtok ? ntok : P.M; t.Nlim = P.ntok_dim ? ntok : P.N;
    t.K0 = P.ktok[0] ? min(ntok, P.K[0]) : P.K[0];
    t.K1 = t.blk == P.skip2 ? 0 : (P.ktok[1] ? min(ntok, P.K[1]) : P.K[1]);
    t.n0st = (t.K0 + 63) >> 6;
    t.total = t.n0st + ((t.K1 + 63) >> 6);
}

__device__ __forceinline__ int batch_of(int kind, const Tile &t)
{
    switch (kind) {
    case BATCH_PAIR: return t.pair;
    case BATCH_KV: return t.hk;
    case BATCH_HEAD: return t.h;
    case BATCH_BLOCK: return t.z;
    }
    return 0;
}

__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y, int z, int w)
{
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
                 ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}

// (eight parts' loads in flight at a time: one after the other they took as long as the rest of a tile's epilogue)
template <bool MAX>
__device__ __forceinline__ float tok_value(const TokVec &t, long long at)
{
    float v = MAX ? -INFINITY : 0.f;
    for (int i0 = 0; i0 < t.parts; i0 += 8) {
        float x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = i0 + i < t.parts ? __ldg(t.p + (i0 + i) * t.stride + at) : (MAX ? -INFINITY : 0.f);
#pragma unroll
        for (int i = 0; i < 8; ++i) v = MAX ? fmaxf(v, x[i]) : v + x[i];
    }
    return MAX ? v : t.scale * v;
}

__device__ __forceinline__ void epi_all_sync() { asm volatile("bar.sync 1, 512;" ::: "memory"); }
__device__ __forceinline__ void dot_sync() { asm volatile("bar.sync 2, 64;" ::: "memory"); }

// Sixteen columns of x from `col` on for the warp's 32 rows (`row0`: the first one's token, `rows` of them and `n` columns exist): y gets
// this lane's row. Neighbouring lanes load neighbouring pieces of a row and hand them over through the warp's 2 KB: a row per
// lane, 8 bytes at a time, took 13 k cycles a tile where this takes 3 k. Rows that do not start on 16 bytes go element by element.
__device__ __forceinline__ void load_x16(const ProbBody &P, long long row0, int rows, int col, int n, unsigned char *mine, int lane, float (&y)[16])
{
    const int es = P.xkind == X_F32 ? 4 : 2;
    const char *base = static_cast<const char *>(P.x) + (row0 * P.xld + col) * es;
    const long long ldb = (long long)P.xld * es;
    auto at = [&](int r, int q) { return reinterpret_cast<uint4 *>(mine + r * 64 + ((q ^ ((r >> 1) & 3)) << 4)); };
    __syncwarp();
    if (((reinterpret_cast<uintptr_t>(P.x) | (uintptr_t)ldb) & 15) == 0) {
        const uint4 zero = make_uint4(0, 0, 0, 0);
        if (P.xkind == X_F32) {
            uint4 u[4];
#pragma unroll
            for (int it = 0; it < 4; ++it) {
                const int r = it * 8 + (lane >> 2), q = lane & 3;
                u[it] = r < rows && 4 * q < n ? __ldg(reinterpret_cast<const uint4 *>(base + r * ldb) + q) : zero;
            }
#pragma unroll
            for (int it = 0; it < 4; ++it) *at(it * 8 + (lane >> 2), lane & 3) = u[it];
        } else {
            const int planes = P.xkind == X_PLANES ? 3 : 1;
            uint4 u[2][3];
#pragma unroll
            for (int it = 0; it < 2; ++it)
#pragma unroll
                for (int pl = 0; pl < 3; ++pl) {
                    const int r = it * 16 + (lane >> 1), q = lane & 1;
                    u[it][pl] = pl < planes && r < rows && 8 * q < n ? __ldg(reinterpret_cast<const uint4 *>(base + r * ldb + pl * P.xps * 2) + q) : zero;
                }
#pragma unroll
            for (int it = 0; it < 2; ++it) {
                float f[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) f[j] = 0.f;
#pragma unroll
                for (int pl = 2; pl >= 0; --pl) {   // (small parts first; the sum of the three is exact)
                    const uint32_t v[4] = {u[it][pl].x, u[it][pl].y, u[it][pl].z, u[it][pl].w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) add2(f[2 * j], f[2 * j + 1], __uint_as_float(v[j] << 16), __uint_as_float(v[j] & 0xffff0000u));
                }
                const int r = it * 16 + (lane >> 1), q = lane & 1;
                *reinterpret_cast<float4 *>(at(r, 2 * q)) = make_float4(f[0], f[1], f[2], f[3]);
                *reinterpret_cast<float4 *>(at(r, 2 * q + 1)) = make_float4(f[4], f[5], f[6], f[7]);
            }
        }
    } else {
        const char *p = base + lane * ldb;          // (never planes: those are the path's own)
#pragma unroll 1
        for (int j = 0; j < 16; ++j) {
            float v = 0.f;
            if (lane < rows && j < n) v = es == 4 ? reinterpret_cast<const float *>(p)[j] : __uint_as_float((uint32_t)reinterpret_cast<const unsigned short *>(p)[j] << 16);
            reinterpret_cast<float *>(at(lane, j >> 2))[j & 3] = v;
        }
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float4 v = *reinterpret_cast<const float4 *>(at(lane, q));
        y[4 * q] = v.x; y[4 * q + 1] = v.y; y[4 * q + 2] = v.z; y[4 * q + 3] = v.w;
    }
}

// What the path does to a row's 32 columns: acc (this lane's row, columns n0 + 32 g .. + 31) in place. mine: the warp's staging.
__device__ __forceinline__ void apply(const ProbBody &P, const Tile &t, float (&acc)[32], float den, float rowv, unsigned char *mine, int g, int rl)
{
    const int col0 = t.n0 + g * 32, row = t.m0 + rl, lane = rl & 31;
    const bool live = row < t.Mlim;
    const long long tok = (long long)t.pair * P.ntok + (long long)t.blk * P.block + row;
    float part = 0.f;
    if (P.alpha != 1.f) {
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[j] *= P.alpha;
    }
    switch (P.epi) {
    case EPI_SQUARES:
#pragma unroll
        for (int j = 0; j < 32; ++j) part = fmaf(acc[j], acc[j], part);      // (columns past the end are zero)
        break;
    case EPI_COLMAX: {
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[j] = live ? fmaxf(acc[j] - rowv, -INFINITY) : -INFINITY;        // (NaN: a key that is not a number leaves the other keys' shift alone)
        // maxima over the warp's rows: halve the columns and the lanes that hold them in turn; lane l ends with column l
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            const bool up = lane & o;
#pragma unroll
            for (int j = 0; j < o; ++j) {
                const float keep = up ? acc[j + o] : acc[j], give = up ? acc[j] : acc[j + o];
                acc[j] = fmaxf(keep, __shfl_xor_sync(0xffffffffu, give, o));
            }
        }
        if (col0 + lane < t.Nlim) atomicMax(P.colmax + (long long)t.pair * P.colkey_ld + col0 + lane, float_order_key(acc[0]));
        break;
    }
    case EPI_ROWMAX:
    case EPI_PHI_Q:
    case EPI_PHI_K: {
        // a lane decodes one column's shift; all read them from the warp's staging
        float *skey = reinterpret_cast<float *>(mine);
        skey[lane] = col0 + lane < t.Nlim ? float_from_order_key(__ldg(P.colmax + (long long)t.pair * P.colkey_ld + col0 + lane)) : 0.f;
        __syncwarp();
        if (P.epi == EPI_PHI_K) {
            float low = 0.f;
#pragma unroll
            for (int j = 0; j < 32; j += 2) {
                const float2 k = *reinterpret_cast<const float2 *>(skey + j);
                add2(acc[j], acc[j + 1], -rowv, -rowv);
                add2(acc[j], acc[j + 1], -k.x, -k.y);
                mul2(acc[j], acc[j + 1], kLog2e, kLog2e);
                low = fminf(low, fminf(acc[j], acc[j + 1]));
            }
            __syncwarp();
            if (low < kKeyScaleLine) {
#pragma unroll
                for (int j = 0; j < 32; ++j) { const bool l = acc[j] < kKeyScaleLine; acc[j] = ex2f(l ? acc[j] + kKeyScaleLog2 : acc[j]) * (l ? 1.f : kKeyScale); }
            } else {
#pragma unroll
                for (int j = 0; j < 32; j += 2) { acc[j] = ex2f(acc[j]); acc[j + 1] = ex2f(acc[j + 1]); mul2(acc[j], acc[j + 1], kKeyScale, kKeyScale); }
            }
            break;
        }
        const int n = t.Nlim - col0;
        float mx = -INFINITY;
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
            const float4 k = *reinterpret_cast<const float4 *>(skey + j);
            acc[j] += k.x; acc[j + 1] += k.y; acc[j + 2] += k.z; acc[j + 3] += k.w;
        }
        __syncwarp();
        if (n >= 32) {
#pragma unroll
            for (int j = 0; j < 32; ++j) mx = fmaxf(mx, acc[j]);
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) mx = j < n ? fmaxf(mx, acc[j]) : mx;
        }
        part = mx;
        if (P.epi == EPI_ROWMAX) break;
        if (P.row.p) mx = rowv;
        else {                                      // the row is whole in this tile: its other parts' maxima
            float *xch = reinterpret_cast<float *>(mine) + 32 + lane;       // (behind the shifts)
            *xch = mx;
            epi_all_sync();
            xch -= g * 2048;                        // the other parts: every fourth warp's, 2 KB to a warp
            mx = fmaxf(fmaxf(xch[0], xch[2048]), fmaxf(xch[2 * 2048], xch[3 * 2048]));
            epi_all_sync();
        }
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[j] = ex2f(kLog2e * (acc[j] - mx));
        break;
    }
    case EPI_MASK:
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[j] = col0 + j > row ? 0.f : acc[j] + rowv;
        break;
    case EPI_DIVIDE: {
        const float inv = 1.f / den;
        float f0 = 0.f, f1 = 0.f;
#pragma unroll
        for (int j = 0; j < 32; j += 2) fma2(f0, f1, acc[j], acc[j + 1], 0.f, 0.f);
        if (den > 1e-30f && f0 + f1 == 0.f) {       // quotients: the product with the reciprocal, corrected once by the
                                                    // remainder (Markstein, IBM J. Res. Dev. 34, 1990): within an ulp
#pragma unroll
            for (int j = 0; j < 32; ++j) { const float q = acc[j] * inv; acc[j] = fmaf(fmaf(-q, den, acc[j]), inv, q); }
        } else {                                    // (where the reciprocal may overflow, or a numerator is infinite)
#pragma unroll 1
            for (int j = 0; j < 32; ++j) {
                const float q = acc[0] / den;
#pragma unroll
                for (int i = 0; i < 31; ++i) acc[i] = acc[i + 1];
                acc[31] = q;
            }
        }
        break;
    }
    case EPI_GRAD:
    case EPI_RANK1:
    case EPI_SUBX: {
        if (P.xkind == X_NONE) break;
        const float inv = 1.f / den, v = P.epi == EPI_SUBX || P.row.p ? rowv : 1.f;     // (den: 1 where there is no dot product)
        const float *f = P.colvec + t.pair * P.vec_pair + t.blk * P.vec_blk + col0;     // (padded to a multiple of four)
#pragma unroll
        for (int j0 = 0; j0 < 32; j0 += 16) {
            float y[16];
            const int n = t.Nlim - col0 - j0;
            load_x16(P, tok - lane, t.Mlim - row + lane, col0 + j0, n, mine, lane, y);
            float *a = acc + j0;
            if (P.epi == EPI_GRAD) {
#pragma unroll
                for (int i = 0; i < 16; ++i) { part = fmaf(y[i], a[i] * inv, part); a[i] = y[i] * inv; }
            } else if (P.epi == EPI_SUBX) {
#pragma unroll
                for (int i = 0; i < 16; ++i) a[i] = fmaf(-v, y[i], a[i]);
            } else {
#pragma unroll
                for (int i = 0; i < 16; i += 4) {
                    const float4 c = i < n && P.colvec ? __ldg(reinterpret_cast<const float4 *>(f + j0 + i)) : make_float4(0.f, 0.f, 0.f, 0.f);
                    a[i] = y[i] * fmaf(v, c.x, a[i]); a[i + 1] = i + 1 < n ? y[i + 1] * fmaf(v, c.y, a[i + 1]) : 0.f;
                    a[i + 2] = i + 2 < n ? y[i + 2] * fmaf(v, c.z, a[i + 2]) : 0.f; a[i + 3] = i + 3 < n ? y[i + 3] * fmaf(v, c.w, a[i + 3]) : 0.f;
                    part += (a[i] + a[i + 1]) + (a[i + 2] + a[i + 3]);
                }
            }
        }
        if (P.epi == EPI_GRAD) part *= -inv;
        break;
    }
    }
    if (P.sums && live) P.sums[(long long)(t.tn * 4 + g) * P.batch * P.ntok + tok] = part;
}

__global__ void __launch_bounds__(kNT, 1) split_gemm_kernel(const __grid_constant__ Launch L)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + kBar), *empty = full + kMaxStages;           // a stage's planes have arrived, have been read
    uint64_t *accfull = empty + kMaxStages, *accfree = accfull + 2, *dotfull = accfree + 2, *dotfree = dotfull + 2;     // two of each
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(dotfree + 2);
    float *sDot = reinterpret_cast<float *>(smem + kDot), *sWt = reinterpret_cast<float *>(smem + kWt);
    const int tid = threadIdx.x, warp = uniform(tid >> 5), lane = tid & 31;
    const int stages = min(kMaxStages, kRing / L.stage_planes), stage_bytes = L.stage_planes * kPlane;

    ProbBody *body = reinterpret_cast<ProbBody *>(smem + kBody);
    for (int i = tid; i < L.n * (int)(sizeof(ProbBody) / 4); i += kNT) {
        const int pb = i / (int)(sizeof(ProbBody) / 4), k = i % (int)(sizeof(ProbBody) / 4);
        reinterpret_cast<int *>(body + pb)[k] = reinterpret_cast<const int *>(static_cast<const ProbBody *>(&L.p[pb]))[k];
    }
    if (tid == 0) {
        for (int i = 0; i < kMaxStages; ++i) { mbar_init(full + i, 1); mbar_init(empty + i, 1 + kDots); }
        for (int i = 0; i < 2; ++i) { mbar_init(accfull + i, 1); mbar_init(accfree + i, kEpi); mbar_init(dotfull + i, kDots); mbar_init(dotfree + i, kEpi); }
        fence_mbar_init();
    }
    if (warp == kMmaWarp) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = uniform(*tmem_slot);
    // (the reads of the parameters, none of which is in a cache yet, and the first tile's place run under the kernel before)
    Tile t;
    decode(L, body, blockIdx.x, t);
    pdl_wait_tma();
    if (L.init) {
        if (blockIdx.x == 0 && tid == 0) *L.status = 0;
        for (int i = blockIdx.x * kNT + tid; i < L.init_n; i += gridDim.x * kNT) L.init[i] = (int)0x80000000u;
    }

    // ok: false once a wait gave up: later waits are skipped, the loops run dry (the status word says so)
    bool ok = true;
    auto wait = [&](uint64_t *bar, uint32_t parity) { ok = ok && mbar_wait(bar, parity & 1, L.status); };
    auto warp_wait = [&](uint64_t *bar, uint32_t parity) { wait(bar, parity); ok = __all_sync(0xffffffffu, ok); };       // one answer for the warp
    uint32_t st = 0, sph = 0;       // slot and parity of the next stage
    auto next_stage = [&]() { if (++st == (uint32_t)stages) { st = 0; sph ^= 1; } };

    if (warp == kLoadWarp) {
        // ---------------------------------------------------------------- load
        if (lane == 0) {
            for (uint32_t w = blockIdx.x; w < L.total; w += gridDim.x, decode(L, body, w, t)) {
                const ProbBody &P = body[t.pb];
                for (int i = 0; i < t.total && ok; ++i) {
                    const int s = i >= t.n0st, k0 = (i - (s ? t.n0st : 0)) * 64;
                    wait(empty + st, sph ^ 1);
                    if (!ok) break;
                    unsigned char *dst = smem + st * stage_bytes;
                    const Opnd &a = P.op[2 * s], &b = P.op[2 * s + 1];
                    const int bhalves = b.mn && t.Nlim - t.n0 <= 64 ? 1 : 2;
                    mbar_expect_tx(full + st, a.planes * kPlane + (b.mn ? b.planes * bhalves * (kPlane / 2) : b.planes * kPlane));
                    auto load = [&](const Opnd &o, const CUtensorMap *map, unsigned char *d, int mn0, int halves) {
                        const int rb = o.tok ? t.blk * P.block : 0, bt = batch_of(o.batch, t);
                        if (!o.mn) tma_load_4d(d, map, full + st, k0, rb + mn0, bt, 0);
                        else
                            for (int hh = 0; hh < halves; ++hh) tma_load_4d(d + hh * o.planes * (kPlane / 2), map, full + st, mn0 + hh * 64, rb + k0, bt, 0);
                    };
                    load(a, &L.p[t.pb].map[2 * s], dst, t.m0, 2);
                    load(b, &L.p[t.pb].map[2 * s + 1], dst + a.planes * kPlane, t.n0, bhalves);
                    next_stage();
                }
            }
        }
    } else if (warp == kMmaWarp) {
        // ---------------------------------------------------------------- multiply
        uint32_t unit = 0;
        for (uint32_t w = blockIdx.x; w < L.total; w += gridDim.x, decode(L, body, w, t)) {
            const ProbBody &P = body[t.pb];
            const int nw = uniform((min(t.Nlim - t.n0, 128) + 15) & ~15);               // columns of this tile, in the MMA's granularity
            const int total = uniform(t.total), n0st = uniform(t.n0st), chain = uniform(P.chain);
            const uint32_t planesA0 = uniform(P.op[0].planes), planesB0 = uniform(P.op[1].planes), mnA0 = uniform(P.op[0].mn), mnB0 = uniform(P.op[1].mn);
            const uint32_t planesA1 = uniform(P.op[2].planes), planesB1 = uniform(P.op[3].planes), mnA1 = uniform(P.op[2].mn), mnB1 = uniform(P.op[3].mn);
            for (int i = 0; i < total && ok; ++unit) {
                const uint32_t big = tmem + (unit & 1) * 256, sml = big + 128;
                warp_wait(accfree + (unit & 1), (unit >> 1) ^ 1);
                bool small = false;
                for (int c = 0; c < chain && i < total && ok; ++c, ++i) {
                    const bool s = i >= n0st;
                    const uint32_t planesA = s ? planesA1 : planesA0, planesB = s ? planesB1 : planesB0, mnA = s ? mnA1 : mnA0, mnB = s ? mnB1 : mnB0;
                    const uint32_t base = smem_u32(smem) + st * stage_bytes, baseB = base + planesA * kPlane;
                    const uint32_t idesc = make_idesc(128, nw, mnA, mnB);
                    const uint64_t dA = mnA ? make_sdesc(base, planesA * 8192, 1024) : make_sdesc(base, 16, 1024);
                    const uint64_t dB = mnB ? make_sdesc(baseB, planesB * 8192, 1024) : make_sdesc(baseB, 16, 1024);
                    const uint32_t kA = (mnA ? 2048 : 32) >> 4, kB = (mnB ? 2048 : 32) >> 4, pA = (mnA ? 8192 : kPlane) >> 4, pB = (mnB ? 8192 : kPlane) >> 4;
                    warp_wait(full + st, sph);
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        bool acc = small;
#pragma unroll 1
                        for (uint32_t x = 0; x < planesA; ++x)
#pragma unroll 1
                            for (uint32_t y = 0; y < planesB && x + y < 3; ++y) {
                                const uint32_t d = x + y ? sml : big;
                                const uint64_t a0 = dA + x * pA, b0 = dB + y * pB;
                                mma_ss(d, a0, b0, idesc, x + y ? acc : c > 0);
                                mma_ss(d, a0 + kA, b0 + kB, idesc, 1);
                                mma_ss(d, a0 + 2 * kA, b0 + 2 * kB, idesc, 1);
                                mma_ss(d, a0 + 3 * kA, b0 + 3 * kB, idesc, 1);
                                acc |= x + y > 0;
                            }
                        mma_commit(empty + st);
                    }
                    small |= planesA + planesB > 2;
                    next_stage();
                }
                if (ok && elect_one()) mma_commit(accfull + (unit & 1));
            }
        }
    } else if (warp >= kDotWarp) {
        // ---------------------------------------------------------------- dot products of A's rows
        const int dt = tid - kDotWarp * 32;         // 0..63
        uint32_t nd = 0;
        for (uint32_t w = blockIdx.x; w < L.total; w += gridDim.x, decode(L, body, w, t)) {
            const ProbBody &P = body[t.pb];
            // K-major A: rd[0..3] of row dt, rd[4..7] of row dt + 64; MN-major A: the eight rows of chunk dt % 16, every fourth index
            float rd[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) rd[j] = 0.f;
            for (int i = 0; i < t.total; ++i) {
                const int s = i >= t.n0st, k0 = (i - (s ? t.n0st : 0)) * 64, dk = P.dot[s], K = s ? t.K1 : t.K0;
                float wt = 1.f;                     // the vector's element k0 + dt, on its way while the stage is waited for
                if (dk == DOT_FEATURES) wt = k0 + dt < K ? __ldg(P.dotf + t.pair * P.vec_pair + t.blk * P.vec_blk + k0 + dt) : 0.f;
                if (dk == DOT_TOKENS) wt = k0 + dt < K ? tok_value<false>(P.dott, (long long)t.pair * P.ntok + (long long)t.blk * P.block + k0 + dt) : 0.f;
                wait(full + st, sph);               // (also without a dot product: the arrival below belongs to this use of the stage)
                if (dk != DOT_NONE) {
                    dot_sync();                     // the stage before's vector has been read
                    sWt[dt] = wt;
                    dot_sync();
                    // (on the FMA pipe: mma.sync here waited for the tensor cores that the other MMAs keep busy, 105 -> 170 us a launch)
                    const unsigned char *A = smem + st * stage_bytes;
                    const int planes = P.op[2 * s].planes;
                    if (P.op[2 * s].mn) {
                        const int ch = dt & 15;
                        for (int pl = planes - 1; pl >= 0; --pl) {
                            const unsigned char *Ap = A + (ch >> 3) * planes * 8192 + pl * 8192;
#pragma unroll 8
                            for (int i8 = 0; i8 < 16; ++i8) {
                                const int k = (dt >> 4) + 4 * i8;
                                const uint4 q = *reinterpret_cast<const uint4 *>(Ap + swz128(k, ch & 7));
                                const float v = sWt[k];
                                const uint32_t u[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                                for (int j = 0; j < 4; ++j) {
                                    rd[2 * j] = fmaf(v, __uint_as_float(u[j] << 16), rd[2 * j]);
                                    rd[2 * j + 1] = fmaf(v, __uint_as_float(u[j] & 0xffff0000u), rd[2 * j + 1]);
                                }
                            }
                        }
                    } else {
                        for (int pl = planes - 1; pl >= 0; --pl) {
                            const unsigned char *Ap = A + pl * kPlane;
#pragma unroll 4
                            for (int ch = 0; ch < 8; ++ch) {
                                const uint4 x = *reinterpret_cast<const uint4 *>(Ap + swz128(dt, ch)), y = *reinterpret_cast<const uint4 *>(Ap + swz128(dt + 64, ch));
                                const float4 f0 = *reinterpret_cast<const float4 *>(sWt + ch * 8), f1 = *reinterpret_cast<const float4 *>(sWt + ch * 8 + 4);
                                const float f[8] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w};
                                const uint32_t u[4] = {x.x, x.y, x.z, x.w}, v[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
                                for (int j = 0; j < 4; ++j) {
                                    rd[j] = fmaf(f[2 * j + 1], __uint_as_float(u[j] & 0xffff0000u), fmaf(f[2 * j], __uint_as_float(u[j] << 16), rd[j]));
                                    rd[4 + j] = fmaf(f[2 * j + 1], __uint_as_float(v[j] & 0xffff0000u), fmaf(f[2 * j], __uint_as_float(v[j] << 16), rd[4 + j]));
                                }
                            }
                        }
                    }
                }
                mbar_arrive_warp(empty + st);
                next_stage();
            }
            if (P.dot_out) {                        // MN-major: sum over the threads that share a chunk
#pragma unroll
                for (int j = 0; j < 8; ++j) rd[j] += __shfl_xor_sync(0xffffffffu, rd[j], 16);
                float *mine = sWt + 64 + lane * 8;
                dot_sync();                         // (the tile before's sums have been read)
                if (warp > kDotWarp && lane < 16)
#pragma unroll
                    for (int j = 0; j < 8; ++j) mine[j] = rd[j];
                dot_sync();
                if (t.tn == 0 && warp == kDotWarp && lane < 16)
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (t.m0 + lane * 8 + j < t.Mlim) P.dot_out[(long long)t.z * P.dot_ld + t.m0 + lane * 8 + j] = rd[j] + mine[j];
            }
            if (P.epi == EPI_DIVIDE || P.epi == EPI_GRAD) {
                wait(dotfree + (nd & 1), (nd >> 1) ^ 1);
                sDot[(nd & 1) * 128 + dt] = (rd[0] + rd[1]) + (rd[2] + rd[3]);
                sDot[(nd & 1) * 128 + 64 + dt] = (rd[4] + rd[5]) + (rd[6] + rd[7]);
                mbar_arrive_warp(dotfull + (nd & 1));
                ++nd;
            }
        }
    } else {
        // ---------------------------------------------------------------- add up and write out
        const int q4 = warp & 3, g = warp >> 2, rl = q4 * 32 + lane;                    // 32 rows, 32 columns per warp
        const uint32_t taddr = tmem + ((uint32_t)(q4 * 32) << 16) + g * 32;
        unsigned char *mine = smem + kStg + warp * 2048;
        uint32_t unit = 0, nd = 0;
        for (uint32_t w = blockIdx.x; w < L.total; w += gridDim.x, decode(L, body, w, t)) {
            const ProbBody &P = body[t.pb];
            const int row = t.m0 + rl, cols = t.Nlim - t.n0 - g * 32;                   // this warp's columns (may be negative or above 32)
            float rowv = 0.f;
            if (P.row.p && row < t.Mlim) {
                const long long tok = (long long)t.pair * P.ntok + (long long)t.blk * P.block + row;
                rowv = P.epi == EPI_PHI_Q ? tok_value<true>(P.row, tok) : tok_value<false>(P.row, tok);
            }
            float acc[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) acc[j] = 0.f;
            const int chain = P.chain, n0 = P.small[0] ? t.n0st : 0, n1 = P.small[1] ? t.n0st : t.total;       // small products: stages below n0 and from n1 on
            for (int i = 0; i < t.total; i += chain, ++unit) {
                const bool small = i < n0 || min(i + chain, t.total) > n1;
                ok = ok && __all_sync(0xffffffffu, mbar_wait(accfull + (unit & 1), (unit >> 1) & 1, L.status));
                tc_fence_after();
                if (cols > 0) {
                    uint32_t v[32];
                    tmem_ld32(taddr + (unit & 1) * 256, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 32; j += 2) add2(acc[j], acc[j + 1], __uint_as_float(v[j]), __uint_as_float(v[j + 1]));
                    if (small) {
                        tmem_ld32(taddr + (unit & 1) * 256 + 128, v);
                        tmem_wait_ld();
                        // The parts of an infinite value are inf, NaN and NaN: where the large products are infinite they decide alone
                        // (with the check kept to products of values 382 us at 2 x 16 heads of 2001 tokens, d 128, m 256, for all 379)
                        float top = 0.f;
#pragma unroll
                        for (int j = 0; j < 32; ++j) top = fmaxf(top, fabsf(acc[j]));
                        if (top < INFINITY) {
#pragma unroll
                            for (int j = 0; j < 32; j += 2) add2(acc[j], acc[j + 1], __uint_as_float(v[j]), __uint_as_float(v[j + 1]));
                        } else {
#pragma unroll
                            for (int j = 0; j < 32; ++j) if (fabsf(acc[j]) < INFINITY) acc[j] += __uint_as_float(v[j]);
                        }
                    }
                }
                tc_fence_before();
                mbar_arrive_warp(accfree + (unit & 1));
            }
            // (the MMAs write columns in steps of 16 and the loads above take 32: clear what lies past the tile's last)
            if (cols < 32) {
#pragma unroll
                for (int j = 0; j < 32; ++j) acc[j] = j < cols ? acc[j] : 0.f;
            }
            float den = 1.f;
            if (P.epi == EPI_DIVIDE || P.epi == EPI_GRAD) {
                ok = ok && __all_sync(0xffffffffu, mbar_wait(dotfull + (nd & 1), (nd >> 1) & 1, L.status));
                den = sDot[(nd & 1) * 128 + rl];
                if (P.den_out && t.tn == 0 && g == 0 && t.m0 + rl < t.Mlim) P.den_out[(long long)t.pair * P.ntok + (long long)t.blk * P.block + t.m0 + rl] = den;
                mbar_arrive_warp(dotfree + (nd & 1));
                ++nd;
            }
            apply(P, t, acc, den, rowv, mine, g, rl);
            if (P.okind == OUT_NONE) continue;
            if (P.okind == OUT_PLANES) {
                // plane by plane through the warp's 2 KB: four lanes per row's 64 bytes, eight rows per store (rows are padded to
                // whole 16-byte pieces). The warps need no barrier between them.
                __nv_bfloat16 *out = static_cast<__nv_bfloat16 *>(P.out) + (t.pair * P.os_pair + t.blk * P.os_blk);
                // (kernel tiles are written whole: their rows and columns past a short last chunk are zero and take part in products)
                const int rlim = P.epi == EPI_MASK ? 128 : t.Mlim, clim = P.epi == EPI_MASK ? 128 : t.Nlim;
#pragma unroll 1
                for (int pl = 0; pl < 3; ++pl, out += P.ops) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        uint32_t u[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            float &a = acc[8 * q + 2 * j], &b = acc[8 * q + 2 * j + 1];
                            u[j] = pack_bf16(a, b);
                            a -= __uint_as_float(u[j] << 16);
                            b -= __uint_as_float(u[j] & 0xffff0000u);
                        }
                        *reinterpret_cast<uint4 *>(mine + lane * 64 + ((q ^ ((lane >> 1) & 3)) << 4)) = make_uint4(u[0], u[1], u[2], u[3]);
                    }
                    __syncwarp();
#pragma unroll
                    for (int it = 0; it < 4; ++it) {
                        const int r2 = it * 8 + (lane >> 2), q = lane & 3, orow = t.m0 + q4 * 32 + r2, oc = t.n0 + g * 32 + q * 8;
                        const uint4 x = *reinterpret_cast<const uint4 *>(mine + r2 * 64 + ((q ^ ((r2 >> 1) & 3)) << 4));
                        if (orow < rlim && oc < clim) *reinterpret_cast<uint4 *>(out + (long long)orow * P.old_ + oc) = x;
                    }
                    __syncwarp();
                }
            } else {
                // rows of any width and alignment: 16 columns at a time through the warp's 2 KB, eight rows of 64 bytes per store
#pragma unroll 1
                for (int o = 0; o < 2; ++o) {       // (o = 1: the fp32 copy)
                    if (o && !P.out2) break;
                    const bool bf = !o && P.okind == OUT_BF16;
                    const int es = bf ? 2 : 4;
                    char *out = (o ? reinterpret_cast<char *>(P.out2) : static_cast<char *>(P.out)) + (t.pair * P.os_pair + t.blk * P.os_blk) * es;
                    const long long ldb = (long long)P.old_ * es;
                    const bool vec = ((reinterpret_cast<uintptr_t>(out) | (uintptr_t)ldb) & (4 * es - 1)) == 0;
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        if (c * 16 >= cols) break;
                        __syncwarp();
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            *reinterpret_cast<float4 *>(mine + lane * 64 + ((q ^ ((lane >> 1) & 3)) << 4)) = make_float4(acc[c * 16 + 4 * q], acc[c * 16 + 4 * q + 1], acc[c * 16 + 4 * q + 2], acc[c * 16 + 4 * q + 3]);
                        __syncwarp();
#pragma unroll 1
                        for (int it = 0; it < 4; ++it) {
                            const int r2 = it * 8 + (lane >> 2), q = lane & 3, orow = t.m0 + q4 * 32 + r2, oc = t.n0 + g * 32 + c * 16 + q * 4, n = t.Nlim - oc;
                            const float4 x = *reinterpret_cast<const float4 *>(mine + r2 * 64 + ((q ^ ((r2 >> 1) & 3)) << 4));
                            if (orow >= t.Mlim || n <= 0) continue;
                            char *d = out + orow * ldb + (long long)oc * es;
                            if (vec && n >= 4) {
                                if (bf) *reinterpret_cast<uint2 *>(d) = make_uint2(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w));
                                else *reinterpret_cast<float4 *>(d) = x;
                            } else {
                                const float xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                                for (int j = 0; j < 4; ++j)
                                    if (j < n) {
                                        if (bf) reinterpret_cast<__nv_bfloat16 *>(d)[j] = __float2bfloat16_rn(xs[j]);
                                        else reinterpret_cast<float *>(d)[j] = xs[j];
                                    }
                            }
                        }
                    }
                }
                __syncwarp();
            }
        }
    }
    if (__syncthreads_or(!ok)) __nanosleep(200000);         // error path only: let copies and MMAs in flight drain
    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) tmem_dealloc(tmem, 512);
}

// [planes][batch][rows][w] bf16 with rows ld apart, box 64 columns x box_rows x 1 x box_planes, 128-byte swizzle
bool make_map4(CUtensorMap *map, const Mat &m, int box_rows, int box_planes)
{
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    cuuint64_t dims[4] = {(cuuint64_t)m.w, (cuuint64_t)m.rows, (cuuint64_t)m.batch, (cuuint64_t)m.planes};
    cuuint64_t strides[3] = {(cuuint64_t)m.ld * 2, (cuuint64_t)m.bs() * 2, (cuuint64_t)m.ps() * 2};
    cuuint32_t box[4] = {64, (cuuint32_t)box_rows, 1, (cuuint32_t)box_planes}, es[4] = {1, 1, 1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, m.p, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// n / d for n < 2^31 as (high word of n mul + n) >> shr: division by an invariant with a rounded-up multiplier (Granlund and Montgomery,
// PLDI 1994)
FastDiv make_div(unsigned d)
{
    FastDiv f;
    f.d = d; f.shr = 0;
    while ((1u << f.shr) < d) ++f.shr;
    f.mul = (unsigned)(((1ull << 32) * ((1ull << f.shr) - d)) / d + 1);
    return f;
}

}  // namespace

void set_operand(Launch &L, Prob &p, int i, const Op &o, bool hi_only)
{
    const int planes = hi_only ? 1 : o.m.planes;
    if (!make_map4(&p.map[i], o.m, o.mn ? 64 : 128, planes)) L.bad = 1;
    p.op[i] = {(unsigned char)planes, (unsigned char)o.mn, (unsigned char)o.batch, (unsigned char)o.tok};
}

void add(Launch &L, const Prob &q)
{
    Prob &p = L.p[L.n++];
    p = q;
    const int M = p.mtok ? (p.block ? p.block : p.ntok) : p.M, N = p.ntok_dim ? (p.block ? p.block : p.ntok) : p.N;
    const unsigned tilesM = (M + 127) / 128, tilesN = (N + 127) / 128;
    p.blocks = (unsigned)p.batch * p.nblk * tilesM * tilesN;
    p.dTiles = make_div(tilesM * tilesN); p.dTilesN = make_div(tilesN);
    p.dBlk = make_div((unsigned)p.nblk); p.dH = make_div((unsigned)p.H); p.dG = make_div((unsigned)p.G);
    for (int s = 0; s < 2; ++s) p.small[s] = p.op[2 * s].planes + p.op[2 * s + 1].planes > 2;
    for (int s = 0; s < 2; ++s)
        if (p.K[s] > 0 && p.op[2 * s].planes + p.op[2 * s + 1].planes > L.stage_planes) L.stage_planes = p.op[2 * s].planes + p.op[2 * s + 1].planes;
    L.total += p.blocks;
}

cudaError_t run(const Launch &L, cudaStream_t st)
{
    static_assert(sizeof(Launch) <= 4000, "kernel parameter space");
    if (L.bad) return cudaErrorInvalidValue;
    return launch_pdl(split_gemm_kernel, dim3(L.total < 148 ? L.total : 148), dim3(kNT), kSmem, st, L);
}

}  // namespace sg
}  // namespace darkattn
