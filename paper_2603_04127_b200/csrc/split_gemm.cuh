// Batched products of fp32 accuracy on the tensor cores, the engine of the FP32 path (see split_gemm.cu).
#pragma once

#include "common.cuh"

#include <cuda.h>

namespace darkattn {
namespace sg {

// A matrix [batch][rows][w] of bf16 numbers, or of fp32 numbers kept as `planes` = 3 bf16 parts (plane i holds what the planes
// before it left out). Strides in elements, rows `ld` (a multiple of 8) apart.
struct Mat {
    __nv_bfloat16 *p = nullptr;
    int w = 0, ld = 0, planes = 3;
    long long rows = 0, batch = 0;
    long long bs() const { return rows * ld; }
    long long ps() const { return batch * rows * ld; }
};

// which batch entry of an operand a tile reads
enum Batch { BATCH_PAIR = 0, BATCH_KV, BATCH_HEAD, BATCH_NONE, BATCH_BLOCK };

// An operand of a product on the host: `mn` says which of the product's dimensions runs along the contiguous index: 0 the
// contraction (rows are M or N), 1 M or N (rows are the contraction). tok: the rows are tokens, and start at the token block.
struct Op {
    Mat m;
    int batch = BATCH_PAIR, mn = 0, tok = 0;
};

// One number per token, kept as a few partial sums (or maxima): p[i * stride + token].
struct TokVec {
    const float *p = nullptr;
    long long stride = 0;
    int parts = 1;
    float scale = 1.f;
};

// division by a number that is known when the launch is built
struct FastDiv { unsigned d = 1, mul = 1, shr = 0; };

// dot products of the rows of A with a vector along the contraction
enum DotKind {
    DOT_NONE = 0,
    DOT_ONES,            // the rows' sums
    DOT_FEATURES,        // with dotf
    DOT_TOKENS           // with dott
};
// What happens to the tile on its way out (`x`, `row`, ... below are the Prob's fields; every kind starts from alpha * C).
enum Epi {
    EPI_PLAIN = 0,
    EPI_SQUARES,         // sums (if given): squares of the row's elements
    EPI_COLMAX,          // colmax: maxima over the rows of C - row; nothing is written
    EPI_ROWMAX,          // sums: the rows' maxima of C + colkey; nothing is written
    EPI_PHI_K,           // exp(C - row - colkey)
    EPI_PHI_Q,           // exp(C + colkey - max of row's parts (not given: the row's own maximum, one tile of columns))
    EPI_MASK,            // C + row (if given), 0 where col > row
    EPI_DIVIDE,          // C / the row's dot product
    EPI_GRAD,            // x / den (den: the row's dot product); sums: - x . (C / den) / den
    EPI_RANK1,           // (C + row * colvec) * x (row = 1 if not given, colvec 0); sums (if given): the row's elements
    EPI_SUBX             // C - row * x (x if given)
};
enum OutKind { OUT_NONE = 0, OUT_PLANES, OUT_F32, OUT_BF16 };
enum XKind { X_NONE = 0, X_PLANES, X_F32, X_BF16 };

struct Opnd { unsigned char planes, mn, batch, tok; };

// C = A[0] B[0] (+ A[1] B[1]) for every (batch, head, token block) and what is done with it on the way out; K = 0: no product.
// Dimensions marked as tokens end with the block: their size is min(block, ntok - index * block). Blocks are multiples of 64
// tokens, of 128 where a tile's rows are tokens of a block.
struct ProbBody {
    Opnd op[4];                     // A0, B0, A1, B1
    int K[2] = {0, 0}, ktok[2] = {0, 0};
    int M = 0, N = 0, mtok = 0, ntok_dim = 0;
    int skip2 = -1;                 // the second product is left out for this token block (its state is zero)
    int H = 1, G = 1, nblk = 1, block = 0, ntok = 0, batch = 1;    // batch entries: `batch` (batch, head) pairs times nblk token blocks
    int chain = 2;                  // stages of 64 after which the accumulators are added to the sums
    int dot[2] = {DOT_NONE, DOT_NONE};
    int epi = EPI_PLAIN;
    float alpha = 1.f;
    const float *dotf = nullptr, *colvec = nullptr;  // the vector of (pair, block) starts at pair * vec_pair + block * vec_blk
    long long vec_pair = 0, vec_blk = 0;
    TokVec dott, row;
    int xkind = X_NONE, xld = 0;    // x: [pair][token][xld], planes xps apart
    const void *x = nullptr;
    long long xps = 0;
    float *dot_out = nullptr;       // [batch entry][dot_ld]
    int dot_ld = 0;
    float *sums = nullptr;          // per row and 32 columns: [4 tilesN][tokens]
    int *colmax = nullptr;          // order keys, [pair][colkey_ld]: written by EPI_COLMAX, read as colkey
    int colkey_ld = 0;
    int okind = OUT_NONE, old_ = 0;
    void *out = nullptr;            // element (row, col) at out + pair * os_pair + block * os_blk + row * old_ + col
    long long os_pair = 0, os_blk = 0, ops = 0;     // ops: from plane to plane
    float *out2 = nullptr, *den_out = nullptr;      // EPI_DIVIDE (if given): the quotients in fp32 as well, laid out like `out`; the rows' dot products, [pair][token]
    // derived
    int small[2] = {0, 0};          // whether the products have small parts
    unsigned blocks = 0;
    FastDiv dTiles, dTilesN, dBlk, dH, dG;
};
struct Prob : ProbBody {
    CUtensorMap map[4];             // of the operands
};

constexpr int kMaxProbs = 3;
struct Launch {
    Prob p[kMaxProbs];
    int n = 0;
    unsigned total = 0;                         // tiles of all of them
    int stage_planes = 2;                       // most planes of the two operands of a product
    int bad = 0;                                // a tensor map could not be encoded
    int *status = nullptr;
    int *init = nullptr; int init_n = 0;        // order keys set to the smallest one, and the status word cleared, by this launch
};

// Sets an operand (0..3: A0, B0, A1, B1) of a product. hi_only: the first plane alone.
void set_operand(Launch &L, Prob &p, int i, const Op &o, bool hi_only = false);
// Adds a product to a launch (fills in the derived fields).
void add(Launch &L, const Prob &p);
cudaError_t run(const Launch &L, cudaStream_t st);

}  // namespace sg
}  // namespace darkattn
