// Host code of the library that has no entry point of its own, without a GPU: linked with the library's objects, the runtime
// calls that need a device replaced (-Wl,--wrap).  Usage: host_checks NAME; exit status 0 and a line of figures, or 1.
#include "hpf_model.cu"          // the model's plans are its own: this file takes the place of its object

#include <cstdio>
#include <cstring>
#include <map>

static thread_local int g_device = 0;
static std::mutex g_lock;
static std::map<int, int> g_attributes;      // device -> attributes set on it
static int g_fail_on = -1;

extern "C" {
cudaError_t __wrap_cudaGetDevice(int* dev) { *dev = g_device; return cudaSuccess; }
cudaError_t __wrap_cudaFuncSetAttribute(const void*, cudaFuncAttribute, int)
{
    std::lock_guard<std::mutex> hold(g_lock);
    if (g_device == g_fail_on) return cudaErrorInvalidDevice;
    ++g_attributes[g_device];
    return cudaSuccess;
}
cudaError_t __wrap_cudaGetDriverEntryPoint(const char*, void** fn, unsigned long long, cudaDriverEntryPointQueryResult* q)
{
    *fn = reinterpret_cast<void*>(&g_attributes);
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
}

#define CHECK(x) do { if (!(x)) { printf("%s:%d: %s\n", __FILE__, __LINE__, #x); return 1; } } while (0)

// Kernel attributes belong to a device: each device a process drives gets its own, once, whichever thread comes first.
static int attributes_per_device()
{
    CHECK(conv_tc_init() == cudaSuccess && conv_pipe_init() == cudaSuccess);
    const int n = g_attributes[0];
    CHECK(n > 0);
    g_device = 1;
    CHECK(conv_tc_init() == cudaSuccess && conv_pipe_init() == cudaSuccess);
    CHECK(g_attributes[1] == n);
    g_device = 2; g_fail_on = 2;
    CHECK(conv_pipe_init() != cudaSuccess);      // a failure is not remembered as done
    g_fail_on = -1;
    CHECK(conv_tc_init() == cudaSuccess && conv_pipe_init() == cudaSuccess);
    CHECK(g_attributes[2] == n);
    std::vector<std::thread> all;
    for (int t = 0; t < 16; ++t)
        all.emplace_back([t] { g_device = 3 + t % 4; (void)conv_tc_init(); (void)conv_pipe_init(); });
    for (auto& t : all) t.join();
    for (int d = 0; d < 7; ++d) CHECK(g_attributes[d] == n);
    printf("%d attributes on each of 7 devices\n", n);
    return 0;
}

// Two pre-activation bottleneck blocks on H x H maps behind a 3 -> c stem, and a head.
static hpf_model* bottlenecks(int H, int c, int w, int co, int B, int M)
{
    std::vector<hpf_op> ops;
    auto add = [&](int kind, int s0, int s1, int ci, int k, int ks) {
        ops.push_back(hpf_op{kind, s0, s1, ci, k, ks, kind == HPF_OP_CONV || kind == HPF_OP_HEAD ? 1 : 0, kind == HPF_OP_CONV ? ks / 2 : 0, kind == HPF_OP_BNRELU ? 1e-5f : 0.f});
        return (int)ops.size() - 1;
    };
    int t = add(HPF_OP_CONV, -1, -1, 3, c, 3);
    for (int b = 0; b < 2; ++b) {
        int v = add(HPF_OP_CONV, add(HPF_OP_BNRELU, t, -1, c, c, 0), -1, c, w, 1);
        v = add(HPF_OP_CONV, add(HPF_OP_BNRELU, v, -1, w, w, 0), -1, w, w, 3);
        v = add(HPF_OP_CONV, add(HPF_OP_BNRELU, v, -1, w, w, 0), -1, w, co, 1);
        const int shortcut = b ? t : add(HPF_OP_CONV, t, -1, c, co, 1);
        t = add(HPF_OP_ADD, v, shortcut, co, co, 0);
        c = co;
    }
    add(HPF_OP_HEAD, add(HPF_OP_BNRELU, t, -1, c, c, 0), -1, c, 10, 0);
    const int32_t shape[4] = {B, H, H, 3};
    hpf_model* mdl = nullptr;
    size_t bytes = 0;
    if (hpf_model_create(ops.data(), (int32_t)ops.size(), shape, nullptr, 0, M, &mdl) != HPF_OK || hpf_workspace_bytes(mdl, &bytes) != HPF_OK) return nullptr;
    return mdl;
}

// A cell's launches cover one micro-batch: their work is split for that, not for the M micro-batches of a step's launches.
// The busiest CTA has at most a tenth more units than an even split over the GPU leaves it.
static int cells_are_planned_for_one_micro_batch()
{
    const struct { int H, c, w, co, B, M; } nets[] = {{32, 16, 16, 64, 128, 8}, {32, 16, 16, 64, 128, 4}, {16, 64, 32, 128, 128, 4}, {56, 64, 64, 256, 64, 4},
                                                      {14, 512, 256, 1024, 64, 4}, {27, 16, 16, 64, 42, 3}};
    int finer = 0, seen = 0;
    for (const auto& net : nets) {
        hpf_model* mdl = bottlenecks(net.H, net.c, net.w, net.co, net.B, net.M);
        CHECK(mdl);
        const hpf_model::KernelPlan &step = mdl->kernels[0], &cell = mdl->cell_kernels();
        CHECK(step.launched == net.M && cell.launched == 1);
        for (int pass = 0; pass < 2; ++pass)
            for (int i = 0; i < mdl->n_ops; ++i) {
                CHECK(step.use_pipe[pass][i] == cell.use_pipe[pass][i]);
                if (!cell.use_pipe[pass][i] || (pass == PASS_DGRAD && mdl->ops[i].op.src0 < 0)) continue;
                const ConvPipeGeom& g = cell.pipe_geom[pass][i];
                const int ctas = 148 / g.slices > 0 ? 148 / g.slices : 1;
                const int busiest = (g.blocks_per_m * g.ksplit + ctas - 1) / ctas * g.unit_block, even = (g.units_per_m * g.ksplit + ctas - 1) / ctas;
                CHECK(10 * busiest <= 11 * even);
                finer += g.blocks_per_m * g.ksplit > step.pipe_geom[pass][i].blocks_per_m * step.pipe_geom[pass][i].ksplit;
                ++seen;
            }
        hpf_model_destroy(mdl);
    }
    CHECK(seen > 60 && finer > 20);
    // one plan where the step's launches cover one micro-batch anyway
    hpf_model* one = bottlenecks(32, 16, 16, 64, 16, 1);
    CHECK(one && &one->cell_kernels() == &one->kernels[0] && one->kernels[0].launched == 1);
    hpf_model_destroy(one);
    printf("%d launches, %d of them split finer than the step's\n", seen, finer);
    return 0;
}

// What asks for cells of their own makes a step's launches cover one micro-batch; stage lanes, which only order them, do not.
static int launches_cover_all_micro_batches()
{
    const struct { int option, value, covered; } cases[] = {{HPF_OPT_STAGE_LANES, 1, 4}, {HPF_OPT_STAGE_LANES, 2, 4}, {HPF_OPT_STAGE_LANES, 8, 4},
                                                            {HPF_OPT_CELL_TIMES, 1, 1}, {HPF_OPT_KEEP_MESSAGES, 1, 1}, {HPF_OPT_GROUP_LAUNCHES, 0, 1}};
    for (const auto& c : cases) {
        hpf_model* mdl = bottlenecks(32, 16, 16, 64, 128, 4);
        CHECK(mdl && hpf_set_option(mdl, c.option, c.value) == HPF_OK);
        CHECK(mdl->group_size() == c.covered);
        int32_t slots = 0;
        CHECK(hpf_num_stream_slots(mdl, &slots) == HPF_OK && slots == (c.option == HPF_OPT_STAGE_LANES ? std::min(c.value, 4) : 1));
        hpf_model_destroy(mdl);
    }
    printf("ok\n");
    return 0;
}

// Which kernel a convolution that is called by itself runs on.
static int calls_by_themselves()
{
    auto tile = [](int N, int H, int C, int K, int R, int stride, int pass, int passes) {
        return conv_tc_faster_alone(make_conv_shape(N, H, H, C, K, R, stride, R / 2), pass, passes);
    };
    CHECK(tile(16, 32, 64, 16, 1, 1, PASS_FWD, 3) && tile(10, 17, 512, 32, 1, 2, PASS_FWD, 3));
    CHECK(tile(37, 32, 64, 16, 1, 1, PASS_FWD, 3) && !tile(38, 32, 64, 16, 1, 1, PASS_FWD, 3));            // 296 tiles
    CHECK(tile(74, 16, 16, 64, 1, 1, PASS_FWD, 3) && !tile(75, 16, 16, 64, 1, 1, PASS_FWD, 3));            // 148 x 64 outputs
    CHECK(!tile(75, 16, 16, 256, 1, 1, PASS_FWD, 3) && tile(75, 16, 16, 256, 1, 1, PASS_DGRAD, 3));        // the two ways differ
    CHECK(!tile(75, 16, 96, 96, 1, 1, PASS_FWD, 3) && tile(75, 16, 96, 96, 1, 1, PASS_FWD, 1));            // one pass, and not widening
    CHECK(!tile(75, 16, 64, 96, 1, 1, PASS_FWD, 1));
    CHECK(tile(37, 15, 64, 48, 1, 2, PASS_FWD, 3) && tile(74, 15, 48, 64, 1, 2, PASS_FWD, 3) && !tile(74, 15, 128, 48, 1, 2, PASS_DGRAD, 3));
    CHECK(tile(16, 7, 512, 64, 1, 1, PASS_FWD, 3) && !tile(16, 7, 528, 64, 1, 1, PASS_FWD, 3) && tile(16, 7, 528, 64, 1, 1, PASS_DGRAD, 3));
    CHECK(!tile(64, 56, 64, 256, 1, 1, PASS_FWD, 1) && !tile(4, 8, 64, 64, 3, 1, PASS_FWD, 3));
    printf("ok\n");
    return 0;
}

// A step's weight gradients run beside its chain of data gradients whether it has one micro-batch or several: the same limit
// on their CTAs (and so on their partial sums); a call by itself has the GPU.
static int weight_gradients_of_a_step()
{
    const ConvShape s = make_conv_shape(128, 32, 32, 64, 16, 1, 1, 0);
    const size_t slice = (size_t)s.K * s.C * sizeof(float);
    CHECK(conv_tc_scratch_bytes(s, 1) <= 222 * slice && conv_tc_scratch_bytes(s, 1) > 148 * slice);
    CHECK(conv_tc_scratch_bytes(s, 2) <= 111 * slice);
    CHECK(conv_tc_scratch_bytes(s) > 222 * slice);
    printf("ok\n");
    return 0;
}

int main(int argc, char** argv)
{
    if (argc > 1 && !strcmp(argv[1], "weight_gradients_of_a_step")) return weight_gradients_of_a_step();
    if (argc > 1 && !strcmp(argv[1], "calls_by_themselves")) return calls_by_themselves();
    if (argc > 1 && !strcmp(argv[1], "launches_cover_all_micro_batches")) return launches_cover_all_micro_batches();
    if (argc > 1 && !strcmp(argv[1], "cells_are_planned_for_one_micro_batch")) return cells_are_planned_for_one_micro_batch();
    if (argc > 1 && !strcmp(argv[1], "attributes_per_device")) return attributes_per_device();
    printf("unknown check\n");
    return 1;
}
