// Forward / data-gradient convolutions on the tensor cores as persistent, warp-specialised launches over whole groups of
// micro-batches, sm_100a.  See conv_pipe.cu.
#pragma once
#include "conv_tc.h"

namespace hpf {

// What a launch may be asked to do besides the convolution: shared memory is planned for it.
struct ConvPipeUse {
    bool addend = false;         // the write-out reads a residual (or, for the sums of a BN+ReLU's backward, its input) beside the accumulator
    bool moments = false;        // it forms BN moments or the sums of a BN+ReLU's backward
    bool bn_in = false;          // a BN+ReLU is applied to the operand
};

// Work split of one convolution.  It depends on the shape of ONE micro-batch, on the precision and on how many micro-batches
// the launches it is planned for cover - never on which of them share a launch - so that every sum is formed in the same order
// whichever micro-batches a planned launch is given.
struct ConvPipeGeom {
    int tiles_per_m;             // tiles of 128 positions of one micro-batch
    int T;                       // tiles per unit (they share every weight tile)
    int units_per_m;             // units of one micro-batch
    int unit_block, blocks_per_m; // consecutive units one CTA takes; blocks of a micro-batch = rows of its BN partial moments
    int slices, n_chunk;         // output channels: slices of n_chunk
    int ksplit;                  // CTAs that share one unit's K loop
    int a_rows, a_stages, b_stages, b_taps, b_resident, acc_bufs;      // b_taps: taps per stage of the weight ring
    unsigned int acc_cols, a_stage_bytes, b_stage_bytes, b_tap_bytes;
    int stacked;
    ConvPipeUse use;
    int flat, box_h;             // operand copies: 128 consecutive pixels, or box_h padded map rows each
    int pos_per_m, Wp, Hp, halo, strips, strip_w, col0;
};
bool conv_pipe_geom(const ConvShape& s, int pass, int passes, int launched, ConvPipeUse use, ConvPipeGeom* g);

// BN work that rides in the forward kernel.
//   out_partials: the output is the input of a BN: per block of units and output channel the mean and the sum of squared
//     deviations of the stored values, [blocks_per_m][2][c_out] floats, then [blocks_per_m] counts and, of a BN without a
//     ReLU (out_plain), [blocks_per_m][c_out] lower parts of the means, conv_pipe_partial_floats() per micro-batch;
//   in_partials: the input x is the input of a BN+ReLU that only this convolution reads: it merges the producer's moments
//     (in_blocks rows), applies y = relu(gamma*(x-mean)*rstd+beta) to its operand, stores y (in_y) and the statistics
//     (in_stats: mean[C], rstd[C] per micro-batch) for the backward pass.
//   bwd_partials (data gradient): the output is the gradient of a BN+ReLU's output that no other kernel adds to: per block of
//     units and channel the sums of dz and of dz * xhat, [blocks_per_m][2][channels] floats in conv_pipe_partial_floats() per
//     micro-batch, from the BN's input (bwd_x), statistics (bwd_stats) and parameters (in_gamma, in_beta).
struct ConvPipeBn {
    float* out_partials = nullptr;
    bool out_plain = false;
    const float* in_partials = nullptr;
    int in_blocks = 0;
    const float* in_gamma = nullptr;
    const float* in_beta = nullptr;
    float* in_stats = nullptr;
    float* in_y = nullptr;
    float in_eps = 0.f;
    float* bwd_partials = nullptr;
    const float* bwd_x = nullptr;
    const float* bwd_stats = nullptr;
};
size_t conv_pipe_partial_floats(int blocks_per_m, int channels);
bool conv_pipe_can_fuse_bn_output(const ConvPipeGeom& g);
// Whether a BN+ReLU may be applied to this convolution's operand on its way to the tensor core.
bool conv_pipe_can_fuse_bn_input(const ConvShape& s);
// Scratch of one micro-batch for launches that split their K loop (0: none does); zeroed once, successive micro-batches follow.
size_t conv_pipe_splitk_bytes(const ConvPipeGeom& g);
size_t conv_pipe_splitk_bytes(const ConvShape& s, int pass, int passes, int launched);

// A prepared launch; the pointers are those of micro-batch 0, whose successors follow contiguously.
struct ConvPipePlan {
    int valid = 0;
    alignas(64) unsigned char storage[960];
};
cudaError_t conv_pipe_init();
// s.N = samples of one micro-batch, M micro-batches in the tensors, `launched` of them in the launches this is planned for.
// in / out / extra as conv_tc_prepare; w_ready: the prepared weights were complete before the kernel that precedes this one in
// its stream was enqueued.
cudaError_t conv_pipe_prepare(ConvPipePlan* plan, const ConvShape& s, int pass, int passes, int M, int launched, const float* in, const float* w_hi,
                              const float* w_lo, float* out, const float* extra, bool accumulate, const ConvPipeBn* bn,
                              void* splitk, size_t splitk_bytes, bool w_ready, ConvPipeUse use);
// Micro-batches m_first .. m_first + m_count - 1 in one launch.
// pdl_late: the successor may be scheduled when a CTA has issued its last MMAs (their operands have arrived), not at its start.
cudaError_t conv_pipe_launch(const ConvPipePlan* plan, int m_first, int m_count, bool pdl_late, DeviceStatus* status, cudaStream_t st, int64_t* n_launch);

// Persistent cells: prepared launches run one after the other by ONE resident grid of `ctas` CTAs with a grid-wide barrier
// between them.  conv_pipe_cell_op writes the device-side record of a launch (conv_pipe_cell_op_bytes() bytes, to be copied
// to 64-byte aligned device memory) and reports what it needs; the list is launched with the largest smem / tmem_cols of its
// records.  d_barrier: two zeroed words per stream of cells.
size_t conv_pipe_cell_op_bytes();
void conv_pipe_cell_op(const ConvPipePlan* plan, DeviceStatus* status, void* dst_host, unsigned int* smem, unsigned int* tmem_cols);
// CTAs that can be resident on the current device at once, those of all cells that run at the same time together.
int conv_pipe_cell_max_ctas();
cudaError_t conv_pipe_cell_launch(const void* d_ops, int n_ops, int m_first, int m_count, int ctas, unsigned int smem, unsigned int tmem_cols,
                                  unsigned int* d_barrier, DeviceStatus* status, cudaStream_t st, int64_t* n_launch);

// y = BN(x) (+ ReLU) and the statistics of m_count micro-batches of `rows` rows, which follow one another, from the partial moments a
// forward kernel left; with add: sum = y + add and, unless null, act = max(sum, 0) beside it.
// (channels beyond what it takes: the BN forms its statistics itself)
bool bn_merge_apply_takes(int C);
cudaError_t bn_merge_apply(const float* partials, int units, const float* gamma, const float* beta, float eps, bool relu, const float* x, float* y, const float* add,
                           float* sum, float* act, float* stats, long long rows, int C, int m_count, cudaStream_t st, int64_t* n_launch);

}  // namespace hpf
