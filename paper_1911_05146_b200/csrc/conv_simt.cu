// CUDA-core (fp32 FMA) convolution kernels: forward, data gradient, weight gradient for any
// kernel size / stride / padding / channel count.  They serve the 3-channel stem convolution
// (whose reduction length 27 or 147 cannot feed the tensor-core path: a 12-byte pixel is no legal
// TMA row), channel counts that are not multiples of 16, and as an fp32 cross-check of the
// tensor-core kernels.  One kernel, three addressing modes of the same tiled GEMM.
//
// What bounds it: the stem's weight gradient is the last kernel of a backward pass, a few microseconds of arithmetic, so what
// counts is the latency of its k steps.  An element's place in its tensor splits into a part that is fixed per thread and a
// part per k step; only the latter is worked out in the loop, with multiplications for divisions, and the next step's loads are
// under way during this one's arithmetic.  Tiles follow the output: 64 x 64, or 16 / 32 channels wide (a 16-channel stem
// filled a quarter of a 64-wide tile), for a weight gradient of 16 channels 16 x 32 with the block's warps sharing the k steps.
// 3x3 stem, 16 channels, 32 x 32 pixels, batch 128 in four micro-batches: weight gradient 38 + 22 us a micro-batch before.
#include "hpf_kernels.h"

namespace hpf {
namespace {

constexpr int THREADS = 256;

enum { MODE_FWD = 0, MODE_DGRAD = 1, MODE_WGRAD = 2 };

// x / d for 0 <= x < 2^31: the estimate with magic = floor(2^32 / d) + 1 is at most one too large
struct Div { int d; unsigned int magic; };
__device__ __forceinline__ int div_of(const Div& v, int x)
{
    if (v.d == 1) return x;
    const int q = (int)__umulhi((unsigned int)x, v.magic);
    return q * v.d > x ? q - 1 : q;
}
Div make_div(int d) { return Div{d, d <= 1 ? 0u : (unsigned int)((1ull << 32) / (unsigned int)d) + 1u}; }

struct SimtArgs {
    const float* a;        // fwd: x      dgrad: dy     wgrad: dy
    const float* b;        // fwd: w      dgrad: w      wgrad: x
    float* out;            // fwd: y      dgrad: dx     wgrad: partials [splits][K][R*R*C]
    const float* extra;    // fwd: residual, dgrad: addend (nullable)
    int accumulate;        // dgrad: dx += result
    ConvShape s;
    int Md, Nd, Kd;        // GEMM extents (a strided data gradient: of the largest class)
    int k_per_split;       // wgrad: pixels per slice
    int splits;            // wgrad: slices of a micro-batch (grid z = micro-batch * splits + slice)
    long long a_ms, b_ms, out_ms;
    Div dC, dK, dR, dQ, dP, dW, dH;
};

// TM x 4 outputs per thread
template <int MODE, int BM, int BN, int BK, int KS, int TM>
__global__ void __launch_bounds__(THREADS) conv_simt_kernel(const __grid_constant__ SimtArgs g)
{
    static_assert((BM / TM) * (BN / 4) * KS == THREADS && BK % KS == 0, "256 threads");
    constexpr int EA = BM * BK / THREADS, EB = BN * BK / THREADS;
    constexpr int TILE = (BM + 4) * BK + (BN + 4) * BK, RED = KS > 1 ? KS * BM * BN : 0;
    __shared__ __align__(16) float sm[TILE > RED ? TILE : RED];
    float (*As)[BM + 4] = reinterpret_cast<float (*)[BM + 4]>(sm);
    float (*Bs)[BN + 4] = reinterpret_cast<float (*)[BN + 4]>(sm + (BM + 4) * BK);
    const ConvShape& s = g.s;
    const int tid = threadIdx.x;
    const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
    const float *ga = g.a, *gb = g.b;
    int k_begin = 0, k_end = g.Kd, Md = g.Md, slice = 0;
    long long out_off = 0;
    // A strided data gradient is one GEMM per class of output positions (h % stride, w % stride): all positions of a class meet
    // the same taps, and no tap that falls between the samples is multiplied.
    int hp = 0, wp = 0, r0 = 0, s0 = 0, ns = s.R, Hc = s.H, Wc = s.W;
    if (MODE == MODE_WGRAD) {
        const int micro = blockIdx.z / g.splits;
        slice = blockIdx.z - micro * g.splits;
        ga += micro * g.a_ms; gb += micro * g.b_ms; out_off = micro * g.out_ms;
        k_begin = slice * g.k_per_split;
        k_end = k_begin + g.k_per_split < g.Kd ? k_begin + g.k_per_split : g.Kd;
    }
    if (MODE == MODE_DGRAD && s.stride > 1) {
        hp = blockIdx.z / s.stride; wp = blockIdx.z - hp * s.stride;
        r0 = (hp + s.pad) % s.stride; s0 = (wp + s.pad) % s.stride;
        ns = s0 < s.R ? (s.R - s0 + s.stride - 1) / s.stride : 0;
        const int nr = r0 < s.R ? (s.R - r0 + s.stride - 1) / s.stride : 0;
        Hc = (s.H - hp + s.stride - 1) / s.stride; Wc = (s.W - wp + s.stride - 1) / s.stride;
        if (hp >= s.H || wp >= s.W) return;
        Md = s.N * Hc * Wc; k_end = nr * ns * s.K;
        if (m0 >= Md) return;
    }
    // ---- what is fixed per thread ----
    int a_off[MODE == MODE_WGRAD ? 1 : EA], a_y[MODE == MODE_WGRAD ? 1 : EA], a_x[MODE == MODE_WGRAD ? 1 : EA];
    if (MODE != MODE_WGRAD) {
#pragma unroll
        for (int e = 0; e < EA; ++e) {
            const int m = m0 + tid / BK + e * (THREADS / BK);
            a_off[e] = -1; a_y[e] = a_x[e] = 0;
            if (m >= Md) continue;
            if (MODE == MODE_FWD) {                    // m = (n,p,q)
                const int t = div_of(g.dQ, m), q = m - t * s.Q, n = div_of(g.dP, t), p = t - n * s.P;
                a_y[e] = p * s.stride - s.pad; a_x[e] = q * s.stride - s.pad;
                a_off[e] = n;
            } else {                                   // m = (n,h,w) of the class; the sample of tap 0 of the class
                const int t = s.stride > 1 ? m / Wc : div_of(g.dW, m), w = m - t * Wc, n = s.stride > 1 ? t / Hc : div_of(g.dH, t), h = t - n * Hc;
                a_y[e] = (hp + s.stride * h + s.pad - r0) / s.stride; a_x[e] = (wp + s.stride * w + s.pad - s0) / s.stride;
                a_off[e] = n;
            }
        }
    }
    int bc = 0, br = 0, bs = 0;                        // wgrad: n = (r,s,c) of this thread's column of B
    const int bn = n0 + (MODE == MODE_FWD ? 0 : tid % BN);
    if (MODE == MODE_WGRAD) { int t = div_of(g.dC, bn); bc = bn - t * s.C; br = div_of(g.dR, t); bs = t - br * s.R; }

    float ra[EA], rb[EB];
    auto fetch = [&](int k0) {
        if (MODE == MODE_WGRAD) {
            const int m = m0 + tid % BM;
#pragma unroll
            for (int e = 0; e < EA; ++e) {
                const int k = k0 + tid / BM + e * (THREADS / BM);
                ra[e] = m < Md && k < k_end ? __ldg(ga + (int64_t)k * s.K + m) : 0.f;
            }
#pragma unroll
            for (int e = 0; e < EB; ++e) {             // pixel k = (n,p,q): x[n, p*st+r-pad, q*st+s-pad, c]
                const int k = k0 + tid / BN + e * (THREADS / BN);
                const int t = div_of(g.dQ, k), q = k - t * s.Q, img = div_of(g.dP, t), p = t - img * s.P;
                const int ih = p * s.stride + br - s.pad, iw = q * s.stride + bs - s.pad;
                const bool in = k < k_end && bn < g.Nd && (unsigned)ih < (unsigned)s.H && (unsigned)iw < (unsigned)s.W;
                rb[e] = in ? __ldg(gb + (((int64_t)img * s.H + ih) * s.W + iw) * s.C + bc) : 0.f;
            }
        } else {
            const int k = k0 + tid % BK;               // fwd: (r,s,c), dgrad: (r,s,k) over the class's taps
            const int t = div_of(MODE == MODE_FWD ? g.dC : g.dK, k), c = k - t * (MODE == MODE_FWD ? s.C : s.K);
            const int rr = MODE == MODE_FWD || s.stride == 1 ? div_of(g.dR, t) : t / (ns > 0 ? ns : 1), ss = t - rr * ns;
#pragma unroll
            for (int e = 0; e < EA; ++e) {
                const int y = MODE == MODE_FWD ? a_y[e] + rr : a_y[e] - rr, x = MODE == MODE_FWD ? a_x[e] + ss : a_x[e] - ss;
                const int H = MODE == MODE_FWD ? s.H : s.P, W = MODE == MODE_FWD ? s.W : s.Q, C = MODE == MODE_FWD ? s.C : s.K;
                const bool in = k < k_end && a_off[e] >= 0 && (unsigned)y < (unsigned)H && (unsigned)x < (unsigned)W;
                ra[e] = in ? __ldg(ga + (((int64_t)a_off[e] * H + y) * W + x) * C + c) : 0.f;
            }
#pragma unroll
            for (int e = 0; e < EB; ++e) {
                if (MODE == MODE_FWD) {                // w[n][kk]
                    const int n = n0 + tid / BK + e * (THREADS / BK);
                    rb[e] = k < k_end && n < g.Nd ? __ldg(gb + (int64_t)n * g.Kd + k) : 0.f;
                } else {                               // kk = (r,s,k), n = c: w[k][r][s][c]
                    const int kb = k0 + tid / BN + e * (THREADS / BN);
                    const int tb = div_of(g.dK, kb), ch = kb - tb * s.K;
                    const int rb_ = s.stride == 1 ? div_of(g.dR, tb) : tb / (ns > 0 ? ns : 1), sb_ = tb - rb_ * ns;
                    rb[e] = kb < k_end && bn < g.Nd ? __ldg(gb + (((int64_t)ch * s.R + r0 + s.stride * rb_) * s.R + s0 + s.stride * sb_) * s.C + bn) : 0.f;
                }
            }
        }
    };
    constexpr int TX = BN / 4, SLICE = THREADS / KS;
    const int ks = tid / SLICE, lt = tid - ks * SLICE, ty = lt / TX, tx = lt - ty * TX;
    float acc[TM][4];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;

    if (k_begin < k_end) fetch(k_begin);
    for (int k0 = k_begin; k0 < k_end; k0 += BK) {
        __syncthreads();
#pragma unroll
        for (int e = 0; e < EA; ++e) {
            if (MODE == MODE_WGRAD) As[tid / BM + e * (THREADS / BM)][tid % BM] = ra[e];
            else As[tid % BK][tid / BK + e * (THREADS / BK)] = ra[e];
        }
#pragma unroll
        for (int e = 0; e < EB; ++e) {
            if (MODE == MODE_FWD) Bs[tid % BK][tid / BK + e * (THREADS / BK)] = rb[e];
            else Bs[tid / BN + e * (THREADS / BN)][tid % BN] = rb[e];
        }
        __syncthreads();
        if (k0 + BK < k_end) fetch(k0 + BK);
#pragma unroll
        for (int k = 0; k < BK / KS; ++k) {
            const int kk = ks * (BK / KS) + k;
            const float4 b4 = *reinterpret_cast<const float4*>(&Bs[kk][tx * 4]);
            const float bv[4] = {b4.x, b4.y, b4.z, b4.w};
            float av[TM];
#pragma unroll
            for (int i = 0; i < TM; i += 4) {
                const float4 a4 = *reinterpret_cast<const float4*>(&As[kk][ty * TM + i]);
                av[i] = a4.x; av[i + 1] = a4.y; av[i + 2] = a4.z; av[i + 3] = a4.w;
            }
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
    }
    if (KS > 1) {
        // the slices of the k steps, in order
        __syncthreads();
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) sm[(ks * BM + ty * TM + i) * BN + tx * 4 + j] = acc[i][j];
        __syncthreads();
        for (int i = tid; i < BM * BN; i += THREADS) {
            float v = 0.f;
#pragma unroll
            for (int z = 0; z < KS; ++z) v += sm[z * BM * BN + i];
            const int m = m0 + i / BN, n = n0 + i % BN;
            if (m < Md && n < g.Nd) g.out[out_off + ((int64_t)slice * g.Md + m) * g.Nd + n] = v;
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int m = m0 + ty * TM + i;
        if (m >= Md) continue;
        int64_t row = m;
        if (MODE == MODE_DGRAD && s.stride > 1) {
            const int t = m / Wc, w = m - t * Wc, n = t / Hc, h = t - n * Hc;
            row = ((int64_t)n * s.H + hp + s.stride * h) * s.W + wp + s.stride * w;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = n0 + tx * 4 + j;
            if (n >= g.Nd) continue;
            float v = acc[i][j];
            if (MODE == MODE_WGRAD) {
                g.out[out_off + ((int64_t)slice * g.Md + m) * g.Nd + n] = v;
            } else {
                const int64_t o = row * g.Nd + n;
                if (g.extra) v += __ldg(&g.extra[o]);
                if (MODE == MODE_DGRAD && g.accumulate) v += g.out[o];
                g.out[o] = v;
            }
        }
    }
}

// dw[i] = sum over splits (ascending) of partials[z][i]; grid y = micro-batch
__global__ void __launch_bounds__(THREADS)
wgrad_reduce_kernel(const float* __restrict__ partials, float* __restrict__ dw, int64_t n, int splits, long long part_ms, long long dw_ms)
{
    partials += blockIdx.y * part_ms; dw += blockIdx.y * dw_ms;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        float s = 0.f;
#pragma unroll 8
        for (int z = 0; z < splits; ++z) s += __ldcg(&partials[(int64_t)z * n + i]);
        dw[i] = s;
    }
}

// Slices of the pixels of one micro-batch.  Few output tiles (a stem convolution: one to three) leave it to the slices to
// fill the GPU, two blocks per SM over the micro-batches of a launch, down to 128 pixels each.
struct WgradSplit { int splits, k_per_split; };
WgradSplit wgrad_split(const ConvShape& s, int launched)
{
    constexpr int kStep = 64;
    const int64_t pixels = (int64_t)s.N * s.P * s.Q;
    const int64_t outs = (int64_t)s.K * s.R * s.R * s.C;
    int64_t splits = pixels / 1024;                       // >= 1024 pixels per slice
    const int64_t out_tiles = (int64_t)((s.K + 63) / 64) * ((s.R * s.R * s.C + 63) / 64) * launched;
    if (splits * out_tiles < 296) splits = (296 + out_tiles - 1) / out_tiles;
    if (splits * out_tiles > 1184) splits = (1184 + out_tiles - 1) / out_tiles;
    if (splits > pixels / 128) splits = pixels / 128;
    const int64_t cap = (int64_t)(32 << 20) / (outs * 4) ;  // partials <= 32 MiB
    if (splits > cap) splits = cap;
    if (splits > 256) splits = 256;
    if (splits < 1) splits = 1;
    int64_t kps = (pixels + splits - 1) / splits;
    kps = (kps + kStep - 1) / kStep * kStep;
    WgradSplit r;
    r.k_per_split = (int)kps;
    r.splits = (int)((pixels + kps - 1) / kps);
    return r;
}

SimtArgs make_args(const float* a, const float* b, float* out, const float* extra, bool accumulate, const ConvShape& s)
{
    SimtArgs g{};
    g.a = a; g.b = b; g.out = out; g.extra = extra; g.accumulate = accumulate ? 1 : 0; g.s = s; g.splits = 1;
    g.dC = make_div(s.C); g.dK = make_div(s.K); g.dR = make_div(s.R); g.dQ = make_div(s.Q); g.dP = make_div(s.P);
    g.dW = make_div(s.W); g.dH = make_div(s.H);
    return g;
}

template <int MODE, int BM, int BN, int BK, int KS, int TM = 4>
void launch_tiles(const SimtArgs& g, int z, cudaStream_t st)
{
    conv_simt_kernel<MODE, BM, BN, BK, KS, TM><<<dim3((g.Md + BM - 1) / BM, (g.Nd + BN - 1) / BN, z), THREADS, 0, st>>>(g);
}
template <int MODE>
void launch_by_width(const SimtArgs& g, int z, cudaStream_t st)
{
    if (g.Nd <= 16) launch_tiles<MODE, 256, 16, 16, 1>(g, z, st);
    else if (g.Nd <= 32) launch_tiles<MODE, 128, 32, 16, 1>(g, z, st);
    // (eight rows a thread take three shared-memory loads per 32 products instead of four; from two such tiles per SM on)
    else if ((long long)g.Md * ((g.Nd + 63) / 64) * z >= 2 * 148 * 128) launch_tiles<MODE, 128, 64, 16, 1, 8>(g, z, st);
    else launch_tiles<MODE, 64, 64, 16, 1>(g, z, st);
}

inline void count(int64_t* n_launch, int k) { if (n_launch) *n_launch += k; }

}  // namespace

size_t conv_simt_scratch_bytes(const ConvShape& s, int launched)
{
    const WgradSplit w = wgrad_split(s, launched);
    return (size_t)w.splits * s.K * s.R * s.R * s.C * sizeof(float);
}

cudaError_t conv_fwd_simt(const float* x, const float* w, float* y, const float* residual, const ConvShape& s,
                          cudaStream_t st, int64_t* n_launch)
{
    SimtArgs g = make_args(x, w, y, residual, false, s);
    g.Md = s.N * s.P * s.Q; g.Nd = s.K; g.Kd = s.R * s.R * s.C;
    launch_by_width<MODE_FWD>(g, 1, st);
    count(n_launch, 1);
    return cudaGetLastError();
}

cudaError_t conv_dgrad_simt(const float* dy, const float* w, float* dx, const float* addend, bool accumulate,
                            const ConvShape& s, cudaStream_t st, int64_t* n_launch)
{
    SimtArgs g = make_args(dy, w, dx, addend, accumulate, s);
    g.Md = s.N * ((s.H + s.stride - 1) / s.stride) * ((s.W + s.stride - 1) / s.stride); g.Nd = s.C; g.Kd = s.R * s.R * s.K;
    launch_by_width<MODE_DGRAD>(g, s.stride * s.stride, st);
    count(n_launch, 1);
    return cudaGetLastError();
}

cudaError_t conv_wgrad_simt(const float* x, const float* dy, float* dw, const ConvShape& s, void* scratch,
                            cudaStream_t st, int64_t* n_launch, int launched, int m_count, long long scratch_ms, long long dw_ms)
{
    const WgradSplit ws = wgrad_split(s, launched);
    SimtArgs g = make_args(dy, x, reinterpret_cast<float*>(scratch), nullptr, false, s);
    g.Md = s.K; g.Nd = s.R * s.R * s.C; g.Kd = s.N * s.P * s.Q; g.k_per_split = ws.k_per_split; g.splits = ws.splits;
    g.a_ms = (long long)s.N * s.P * s.Q * s.K; g.b_ms = (long long)s.N * s.H * s.W * s.C; g.out_ms = scratch_ms;
    const int z = ws.splits * m_count;
    if (g.Md <= 16 && g.Nd <= 32) launch_tiles<MODE_WGRAD, 16, 32, 64, 8>(g, z, st);
    else if (g.Nd <= 32) launch_tiles<MODE_WGRAD, 64, 32, 32, 2>(g, z, st);
    else launch_tiles<MODE_WGRAD, 64, 64, 16, 1>(g, z, st);
    const int64_t n = (int64_t)s.K * s.R * s.R * s.C;
    int nb = (int)((n + THREADS - 1) / THREADS);
    if (nb > 1184) nb = 1184;
    wgrad_reduce_kernel<<<dim3(nb, m_count), THREADS, 0, st>>>(reinterpret_cast<const float*>(scratch), dw, n, ws.splits, scratch_ms, dw_ms);
    count(n_launch, 2);
    return cudaGetLastError();
}

}  // namespace hpf
