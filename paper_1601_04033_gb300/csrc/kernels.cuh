// Internal interface between the host runtime (runtime.cu) and the kernels
// (dense.cu, select.cu, sparse.cu).  Not part of the public C ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fasgd.h"

namespace fasgd {

// Per-element update rule of a pass: ASGD/SASGD (Eq. 1-2), FASGD (Eq. 4-8),
// or FASGD with v averaging the std and the step divided by it (the prose
// reading of Sec. 2.2).
enum : int { kRuleSgd = 0, kRuleFasgd = 1, kRuleFasgdStd = 2 };

// Hyper-parameters of Eq. 4-6 as the kernels consume them.  one_m_gamma and
// one_m_beta are formed once on the host in fp32 (1 - gamma, 1 - beta).
struct StatParams {
    float gamma, one_m_gamma;
    float beta, one_m_beta;
    float eps;
    float minus_zero;   // -0.0f, a value the compiler does not see (update.cuh, product2)
};

// Block b's share of P (a multiple of 4) parameters of a pass over `blocks`
// blocks in tiles of `tile`: an equal piece (a multiple of 128) of what is left
// over when every block has as many whole tiles as all can have, then those
// tiles, interleaved.  So no block has a tile more than another (a pass over 5M
// parameters has 16.06 tiles per SM), and the short copies come while the
// pipeline fills (25M, K = 1, push + apply + pull: 169.5 us, 170.3 with the piece
// last; eight message rounds 1224 against 1231).
struct BlockShare {
    int64_t tiles;      // this block's tiles, the piece (the first) included
    int64_t whole;      // whole tiles of each block
    int64_t first, step, piece_start;
    int32_t tile, piece;
    __host__ __device__ BlockShare(int64_t P, int32_t tile_, int64_t blocks, int64_t b) : tile(tile_) {
        whole = P / (blocks * tile);
        first = b * tile;
        step = blocks * tile;
        const int64_t rest = P - whole * step;
        const int64_t share = ((rest + blocks - 1) / blocks + 127) / 128 * 128;
        const int64_t from = b * share < rest ? b * share : rest;
        piece = (int32_t)(rest - from < share ? rest - from : share);
        piece_start = whole * step + from;
        tiles = whole + (piece > 0 ? 1 : 0);
    }
    __host__ __device__ int64_t offset(int64_t t) const {
        t -= piece > 0 ? 1 : 0;
        return t >= 0 ? first + t * step : piece_start;
    }
    __host__ __device__ int32_t length(int64_t t) const { return t == 0 && piece > 0 ? piece : tile; }
};

// Blocks of a message push's pass, and float-float sums of v that it leaves: a
// number of its own, one per SM of a GB300, so that the sums' partition, and with
// it every bit of the statistic, is a function of P alone whatever the GPU (no
// block waits for another, so fewer SMs take them in turns).
constexpr int32_t kMessageBlocks = 152;

// A per-message push decided before or inside its pass (FASGD rules): the pass
// reads the decision, or takes it from the statistic's sums (message_decide)
// where they were just formed afresh; if transmitted it applies src and copies
// it into slot (the client's gradient cache slot, which is also grad[0]), else
// it applies grad[0] as it stands.  Either way it leaves its blocks' sums of the
// new v in `partial`, which is not `fresh` (a block may end before another has
// read it).  partial == null: not a message push.
struct PassMessage {
    const uint32_t* decided;        // the decision (1: transmitted), or null
    const float2* fresh;            // if not decided: kMessageBlocks sums of v
    float2* partial;                // out: the sums of the new v
    int32_t nblocks;                // kMessageBlocks
    float c, eps_b;
    uint32_t round_key0[10], round_key1[10];
    uint32_t client_word, n_lo, n_hi;
    const float* src;               // the pushed gradient, fp32[P], 16-byte aligned
    float* slot;                    // == grad[0]
    int32_t* flag_out;              // may be null: 1 transmitted, 0 dropped (if not decided)
};

// One fused pass over the parameters applying K dense pushes in order.
struct DenseArgs {
    float* theta;
    float* n;
    float* b;
    float* v;
    const float* grad[FASGD_KMAX];  // grad[k]: push k's gradient, fp32[P]
    float coef[FASGD_KMAX];         // alpha(tau_k) of push k (Eq. 1 / Eq. 7 without v)
    int64_t P;
    int32_t K;
    StatParams sp;
    int32_t* err;                   // device error flags (bit 3: a pipeline wait expired)
    PassMessage msg;                // K = 1, FASGD rules
};

// One sparse push: idx[i] receives val[i] for i < count.
struct SparseArgs {
    float* theta;
    float* n;
    float* b;
    float* v;
    const int32_t* idx;
    const float* val;
    const int64_t* count_dev;  // may be null: count = count_max
    int64_t count_max;
    int64_t P;
    float coef;
    StatParams sp;
    int32_t* err;              // device error flags (bit 0: count, bit 1: index, bit 2: order)
    int64_t half_below, quarter_below;   // set by the launch: lists shorter than these take
                                         // half, a quarter of the warps
};

// Parameters per tile of the select kernels, and the bit mask words a tile
// owns (one bit per parameter).
constexpr int kSelectTile = 4096;
constexpr int kSelectTileWords = kSelectTile / 32;

struct SelectArgs {
    const float* values;   // copied into val for kept parameters (a push's gradient, or theta)
    const float* v;
    int32_t* idx;
    float* val;
    int64_t* count;      // total number sent (int64, device)
    uint32_t* mask;      // scratch: ntiles * kSelectTileWords words
    uint16_t* tile_count; // scratch: ntiles, 16-byte aligned, readable to a multiple of eight
    int64_t* tile_base;  // scratch: ntiles
    int64_t P;
    int32_t ntiles;
    float c;
    float eps_b;
    uint32_t round_key0[10];       // Philox key schedule: seed advanced by the
    uint32_t round_key1[10];       // Weyl constants, one pair per round
    uint32_t client_word;          // client + 2^31 * stream (0: push, 1: fetch)
    uint32_t push_lo, push_hi;     // the client's count of earlier calls of that stream
};

// Client side of a B-FASGD fetch: theta[idx[i]] = val[i] for i < count.
struct ScatterArgs {
    float* theta;
    const int32_t* idx;
    const float* val;
    const int64_t* count_dev;  // may be null: count = count_max
    int64_t count_max;
    int64_t P;
    int32_t* err;              // may be null; flags 1 (count) and 2 (index)
};

// Copies of up to four of the server's arrays (copy.cu): dst[i] <- src[i],
// P floats each; src 16-byte aligned, dst 4-byte aligned device memory.
struct CopyArgs {
    const float* src[4];
    float* dst[4];
    int32_t count;
    int64_t P;
};

// Closed-loop simulation: stochastic gradient and loss of the synthetic
// quadratic objective (sim.cu).
struct SimGradArgs {
    const float* theta;   // the client's copy, fp32[P], 16-byte aligned
    const float* h;       // curvatures
    const float* star;    // minimiser
    const float* sigma;   // noise scales
    float* grad;          // output
    int64_t P;
    uint32_t round_key0[10];
    uint32_t round_key1[10];
    uint32_t client, n_lo, n_hi;
};

constexpr int kSimLossScratch = 1024;   // doubles of scratch the loss needs

struct SimLossArgs {
    const float* theta;
    const float* h;
    const float* star;
    int64_t P;
    double* partial;      // kSimLossScratch doubles
    double* loss;         // output (device)
};

// Launchers: enqueue on `stream`, return the launch status.
// `launches` is incremented by the number of kernels enqueued.
cudaError_t launch_dense(const DenseArgs& a, int rule, bool exact, int num_sms, cudaStream_t stream,
                         int64_t* launches);
cudaError_t launch_sparse(const SparseArgs& a, int rule, bool exact, int num_sms, cudaStream_t stream,
                          int64_t* launches);
cudaError_t launch_select(const SelectArgs& a, cudaStream_t stream, int64_t* launches);
cudaError_t launch_copy(const CopyArgs& a, int num_sms, cudaStream_t stream);
cudaError_t launch_scatter(const ScatterArgs& a, int num_sms, cudaStream_t stream);
// Self-test: bounded pipeline waits that can never complete (raise flag 8 in err).
cudaError_t launch_wait_expiry(int32_t* err, cudaStream_t stream);
cudaError_t launch_sim_grad(const SimGradArgs& a, int num_sms, cudaStream_t stream);
cudaError_t launch_sim_loss(const SimLossArgs& a, cudaStream_t stream);

inline int32_t select_tiles(int64_t P) {
    return (int32_t)((P + kSelectTile - 1) / kSelectTile);
}

// Fills the Philox key schedule of `a` from the 64-bit seed.
void select_key_schedule(SelectArgs& a, uint64_t seed);

}  // namespace fasgd
