// Batched products of fp32 accuracy on the tensor cores, the engine of the FP32 path (see split_gemm.cu).
#pragma once

#include "common.cuh"

namespace darkattn {
namespace sg {

// One matrix operand. Element (row, col) of a batch entry is p[batch offset + row * ld + col]; `mn` says which of the
// product's dimensions runs along the contiguous index: 0 the contraction (rows are M or N), 1 M or N (rows are the contraction).
struct Op {
    const void *p = nullptr;
    long long sb = 0, sh = 0, sc = 0;   // element strides of the batch, the head (kv: the key/value head) and the token block
    int ld = 0, kv = 0, bf16 = 0, mn = 0;
};

// One number per token, kept as a few partial sums: scale * sum_i p[i * stride + token].
struct TokVec {
    const float *p = nullptr;
    long long stride = 0;
    int parts = 1;
    float scale = 1.f;
};

// division by a number that is known when the launch is built
struct FastDiv { unsigned d = 1, mul = 1, shr = 0; };

// dot products of the rows of A with a vector along the contraction, formed by the threads that load A
enum DotKind {
    DOT_NONE = 0,
    DOT_ONES,            // the rows' sums
    DOT_FEATURES,        // with dotf (K-major A)
    DOT_TOKENS           // with dott (MN-major A)
};
// What happens to the tile on its way out (`x`, `row`, ... below are the Prob's fields; every kind starts from alpha * C).
enum Epi {
    EPI_PLAIN = 0,
    EPI_SQUARES,         // sums: squares of the row's elements
    EPI_KEY_EXPONENT,    // - row; colmax: maxima over the rows
    EPI_MASK,            // + row (if given), 0 where col > row
    EPI_DIVIDE,          // / the row's dot product
    EPI_GRAD,            // x / den (den: the row's dot product); sums: - x . (C / den) / den
    EPI_RANK1,           // (C + row * rank1[col]) * x (row = 1 if not given); sums (if given): the row's elements
    EPI_SUBX             // - row * x
};

// C = A[0] B[0] (+ A[1] B[1]) for every (batch, head, token block) and what is done with it on the way out.
// Dimensions marked as tokens end with the block: their size is min(block, ntok - index * block).
struct Prob {
    Op A[2], B[2];
    int K[2] = {0, 0};
    int M = 0, N = 0;
    int mtok = 0, ntok_dim = 0, ktok[2] = {0, 0};
    int skip2_first = 0;            // the second product is left out for the first token block (its state is zero)
    int H = 1, G = 1, nblk = 1, block = 0, ntok = 0, batch = 1;    // batch entries: `batch` (batch, head) pairs times nblk token blocks
    int chain = 2;                  // stages of 64 after which the accumulators are added to the sums
    int dot[2] = {DOT_NONE, DOT_NONE};
    int epi = EPI_PLAIN;
    float alpha = 1.f;
    const float *dotf = nullptr, *rank1 = nullptr;  // the vector of (pair, block) starts at pair * vec_pair + block * vec_blk
    long long vec_pair = 0, vec_blk = 0;
    TokVec dott, row;
    Op x;
    float *dot_out = nullptr;       // [batch entry][M]
    float *sums = nullptr;          // per row and tile of columns: [tilesN][tokens] (needed by the kinds that name it, except RANK1)
    int *colmax = nullptr;          // order keys, [pair][N]
    void *out = nullptr;
    long long osb = 0, osh = 0, osc = 0;
    int old_ = 0, obf16 = 0;
    // derived
    unsigned blocks = 0;
    FastDiv dTiles, dTilesN, dBlk, dH, dG;
};

constexpr int kMaxProbs = 3;
struct Launch {
    Prob p[kMaxProbs];
    int n = 0;
    unsigned total = 0;                         // tiles of all of them
    int *status = nullptr;
    int *init = nullptr; int init_n = 0;        // order keys set to the smallest one by this launch (used by a later one)
};

// Adds a product to a launch (fills in the derived fields).
void add(Launch &L, Prob p);
// Runs the launch; `dependent`: after a kernel of this library in the same stream, whose tail it may overlap.
cudaError_t run(const Launch &L, cudaStream_t st, bool dependent);

// Launches a kernel that starts with griddepcontrol.wait; `dependent` as above.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*k)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool dependent, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, KArgs(args)...);
}

}  // namespace sg
}  // namespace darkattn
