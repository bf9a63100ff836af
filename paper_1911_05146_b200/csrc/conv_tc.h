// Tensor-core (tcgen05 / TMEM / TMA) convolution path, sm_100a.  See conv_tc.cu.
#pragma once
#include "hpf_kernels.h"

namespace hpf {

enum ConvPass { PASS_FWD = 0, PASS_DGRAD = 1, PASS_WGRAD = 2 };

// Whether the tensor-core kernels cover this shape for this pass.
bool conv_tc_supported(const ConvShape& s, int pass);

// Whether a forward or data-gradient convolution without BN work of its own is faster here than as a pipelined launch
// (conv_pipe.h), which covers the same shapes.
bool conv_tc_faster_alone(const ConvShape& s, int pass, int passes);

// Resolves the driver entry point used to encode tensor maps.  Needs a CUDA driver.
cudaError_t conv_tc_init();

// weight-gradient partials of one micro-batch; launched: as in ConvTcHints
size_t conv_tc_scratch_bytes(const ConvShape& s, int launched = 0);

// A prepared launch: tensor maps are encoded once (they bake in the device pointers) and the kernel
// parameters are kept ready in `storage`.
struct ConvTcPlan {
    ConvShape s;
    int pass;
    int valid;
    int direct;          // weight gradient: the kernel that feeds the TMA tiles to the tensor core as they land
    alignas(64) unsigned char storage[896];
};

// What else a launch may be told.
struct ConvTcHints {
    // the model's micro-batches, contiguous in every tensor; for a weight gradient the floats between their outputs and
    // between their partial sums (0: packed)
    int micro_batches = 1;
    int launched = 0;            // how many of them the launches this is planned for cover; 0: a call by itself, not part of a step
    long long slot_stride = 0;
    long long partial_stride = 0;
    // weight gradient only: 1 keeps the kernel that transposes its tiles in shared memory (a cross-check)
    int wgrad_transposing = 0;
    // forward / data gradient: room for splitting a long K loop over several CTAs (conv_tc_splitk_bytes, of one
    // micro-batch; the first kSplitKTicketBytes hold tickets, zero before the first use and left zero).  nullptr: never split.
    void* splitk = nullptr;
    size_t splitk_bytes = 0;
};
constexpr size_t kSplitKTicketBytes = 4096;
// Bytes a forward (or data-gradient) launch of this shape wants for splitting its K loop; 0 when it would not split.
size_t conv_tc_splitk_bytes(const ConvShape& s, int pass, int passes);
// passes = 3: error-compensated (hi*hi + lo*hi + hi*lo); passes = 1: single TF32 pass.
// pass = PASS_FWD:   out = conv(in, w) (+ extra); w_hi / w_lo = split weights [K][R][R][C]
// pass = PASS_DGRAD: out (+)= dgrad(in = dy) (+ extra); w_hi / w_lo = split rearranged weights [C][R][R][K]
// pass = PASS_WGRAD: out = wgrad(in = dy, in2 = x)
cudaError_t conv_tc_prepare(ConvTcPlan* plan, const ConvShape& s, int pass, int passes, const float* in, const float* in2,
                            const float* w_hi, const float* w_lo, float* out, const float* extra, bool accumulate, void* scratch,
                            const ConvTcHints* hints = nullptr);
// m_first, m_count: the micro-batches the launch covers.  pdl_late (forward / data gradient): the successor may be scheduled
// when a CTA's first accumulator is complete, not at its start.
cudaError_t conv_tc_launch(const ConvTcPlan* plan, DeviceStatus* status, cudaStream_t st, int64_t* n_launch, int m_first = 0, int m_count = 1,
                           bool pdl_late = false);

// One convolution's weights inside the flat parameter vector.
struct WeightPrepEntry { long long w_off; int C, K, R, reserved; };
// For every table entry (device memory): w_hi/w_lo = hi/lo split of the weights, wt_hi/wt_lo = split of the weights
// rearranged for the data gradient (wt[c][R-1-r][R-1-s][k] = w[k][r][s][c]); all four use the entry's w_off.
cudaError_t conv_weight_prep(const float* params, float* w_hi, float* w_lo, float* wt_hi, float* wt_lo,
                             const WeightPrepEntry* d_table, int n_entries, int max_tiles, cudaStream_t st, int64_t* n_launch);
// 32 x 32 tiles the preparation kernel walks for one convolution (max_tiles above = the largest of the table)
int conv_weight_prep_tiles(int C, int K, int R);

cudaError_t conv_weight_prep_single(const float* w, float* w_hi, float* w_lo, float* wt_hi, float* wt_lo, int C, int K, int R,
                                    cudaStream_t st, int64_t* n_launch);

}  // namespace hpf
