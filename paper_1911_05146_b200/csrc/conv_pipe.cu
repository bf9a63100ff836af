// Forward convolution and data gradient (a forward convolution of dy with rearranged weights), sm_100a: one persistent CTA
// per SM walks units of work, every role of the pipeline on warps of its own.
//
//   D[position, c_out] = sum over channel chunks of 16 and taps  A[position + tap, c] * W[c_out, tap, c]
//
// What bounds these launches.  At 16..256 channels the convolutions of a residual network move far more bytes than the
// tensor core needs time for, so the kernel is built as a stream: loads of the next operand block, the split of this one,
// its MMAs and the write-out of the one before run side by side, and no step of a tile waits for the whole tile before it.
//
// Positions.  A 3x3 window (pad 1) is computed on a padded grid of positions: every map row is followed by ONE zero column
// (it is the right border of its row and the left border of the next), every map by one zero row.  In shared memory the
// positions are consecutive 128-byte rows, so the operand of tap (r, s) is the same block of rows read from
// (r-1)*Wp + (s-1) rows further on: a block is loaded, normalised and split ONCE for its nine taps.  (A K-major operand may
// start at any 128-byte row: the swizzle is a function of the address.)  The padding costs MMA rows (1/17 of them at 16
// pixels, 1/9 at 8) and saves eight of nine copies.  Maps wider than 254 pixels are cut into column strips with a zero or
// neighbour column on either side.  A 1x1 window has no halo: positions are the output pixels.
//
// Operand rows.  A chunk is 16 channels: bytes 0-63 of the 128-byte row hold the value (the tensor core ignores the low 13
// mantissa bits: that is the hi part), bytes 64-127 the lo part of the three-pass form, in the 128-byte swizzle.
//
// Roles (16 warps): warp 0 copies the operand, warp 1 the weights (TMA; kept in shared memory for the whole launch when they
// fit), warp 2 issues the MMAs, warps 4-7 rewrite the operand in place (BN+ReLU, lo part), warps 8-15 read finished
// accumulators from tensor memory, add the residual, store and form the BN moments.
//
// Measured alone, batch 128, three passes, against the tile kernel's one 128-pixel tile per CTA and nine copies per 3x3 tile:
// 3x3 16->16 @32 45 -> 20 us, 64->64 @32 107 -> 68, 128->128 @16 58 -> 48; 1x1 64->64 @32 31 -> 25, 16->64 @32 23 -> 18 (2.3 TB/s),
// but 64->16 @32 18 -> 22 (profiles/conv_sweep_batch128.md).
#include "conv_pipe.h"
#include "tc_ptx.cuh"

#include <algorithm>
#include <string.h>
#include <type_traits>

namespace hpf {

namespace {

constexpr int kSplitWarps = 4, kEpiWarps = 8;
constexpr int kFirstSplit = 4;                        // warps 0..2: operand copies, weight copies, MMAs; 3 idle
constexpr int kSplitThreads = 32 * kSplitWarps, kRowStep = 8 * kSplitWarps;
constexpr int kPipeThreads = 32 * (kFirstSplit + kSplitWarps + kEpiWarps);
constexpr int kMaxBlockRows = 768, kRowBatch = 4;     // operand rows of a block at most; rows a splitter thread has in flight
constexpr uint32_t kPipeSmem = 222 * 1024;            // dynamic shared memory of a CTA
constexpr int kMaxA = 8, kMaxB = 8;

struct PipeScalars {
    const float* in;
    float* out;
    const float* extra;
    DeviceStatus* status;
    long long in_ms, out_ms;                          // floats between micro-batches (extra is laid out like out)
    int accumulate;
    int units_per_m, unit_block, blocks_per_m, tiles_per_m, T, slices, n_chunk, ksplit;
    int R, taps, n_chunks, c_in, c_out;
    int pos_per_m, Wp, img_pos, Hv, W, halo, strips, strip_w, col0;
    uint32_t magic_w, magic_img, magic_strip;
    int in_sw, in_sh, in_sn, os_w, os_h, os_n;
    int zero_fill, out_h, out_w, dense_h, dense_w;
    int a_stages, b_stages, b_taps, b_resident, acc_bufs, split_groups, epi_alternate;
    // how the operand is copied: flat (128 consecutive pixels per box) or blocks of box_h padded rows of one map
    int flat, box_h, box_pos, blocks_per_img;
    uint32_t magic_box, magic_bpi;
    long long pix_ms;                                 // flat: pixels per micro-batch; else maps per micro-batch
    uint32_t a_stage_bytes, b_stage_bytes, b_tap_bytes, acc_cols, tmem_cols, idesc, idesc2;
    uint32_t off_b, off_bn, off_red, off_stat, off_stage;
    int three, stacked, pdl_late, w_ready;
    // BN+ReLU on the way in
    const float* bn_partials;
    const float* bn_gamma;
    const float* bn_beta;
    float* bn_stats;
    float* bn_y;
    int bn_units;
    float bn_eps;
    double bn_inv_rows;
    // BN moments of the output; bn_x (data gradient): the sums of a BN+ReLU's backward instead, whose input bn_x is laid out like out
    float* st_partials;
    const float* bn_x;
    // split K
    char* sk_base;                                    // per micro-batch: tickets, then partial tiles
    long long sk_ms;                                  // bytes between micro-batches
};
struct alignas(64) PipeParams {
    CUtensorMap tm_a, tm_b, tm_b_lo;
    PipeScalars s;
};

// x / d with magic = floor(2^32 / d) + 1: the estimate is at most one too large
__device__ __forceinline__ int div_magic(int x, int d, uint32_t magic)
{
    if (d == 1) return x;
    int q = (int)__umulhi((uint32_t)x, magic);
    return q * d > x ? q - 1 : q;
}
inline uint32_t magic_of(int d) { return d <= 1 ? 0u : (uint32_t)((1ull << 32) / (uint64_t)d) + 1u; }

struct Pixel { int n, y, x; bool in, own; };
// position -> pixel; in: a pixel of the map (padding otherwise), own: an output of this position (not a strip's halo column)
__device__ __forceinline__ Pixel locate(const PipeScalars& p, int pos)
{
    Pixel r;
    const bool some = (unsigned)pos < (unsigned)p.pos_per_m;
    const int q = some ? pos : 0;
    int img = div_magic(q, p.img_pos, p.magic_img);
    const int rem = q - img * p.img_pos;
    r.y = div_magic(rem, p.Wp, p.magic_w);
    const int col = rem - r.y * p.Wp - p.col0;
    int x0 = 0;
    if (p.strips > 1) {
        const int n = div_magic(img, p.strips, p.magic_strip);
        x0 = (img - n * p.strips) * p.strip_w;
        img = n;
    }
    r.n = img; r.x = x0 + col;
    r.in = some && r.y < p.Hv && (unsigned)r.x < (unsigned)p.W;
    r.own = r.in && (unsigned)col < (unsigned)p.strip_w;
    return r;
}

// 16 consecutive floats of one thread: two full sectors
__device__ __forceinline__ void store16(float* d, const float* v)
{
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(d), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]),
                 "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]) : "memory");
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(d + 8), "f"(v[8]), "f"(v[9]), "f"(v[10]), "f"(v[11]),
                 "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15]) : "memory");
}
__device__ __forceinline__ void load16(const float* s, float* v)
{
#pragma unroll
    for (int j = 0; j < 16; j += 4) {
        const float4 t = __ldcg(reinterpret_cast<const float4*>(s + j));
        v[j] = t.x; v[j + 1] = t.y; v[j + 2] = t.z; v[j + 3] = t.w;
    }
}
__device__ __forceinline__ void split_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kSplitThreads) : "memory"); }
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 2, 256;" ::: "memory"); }

__host__ __device__ inline size_t partial_floats(int units, int C) { return (size_t)units * 2 * C + (size_t)((units + 3) & ~3); }

__device__ __forceinline__ float4 lane_sum(float4 v, int o)
{
    v.x += __shfl_xor_sync(0xffffffffu, v.x, o); v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    v.z += __shfl_xor_sync(0xffffffffu, v.z, o); v.w += __shfl_xor_sync(0xffffffffu, v.w, o);
    return v;
}
// Four values at a time with the two-wide fp32 instructions: the same rounding, half the instructions - what the write-out
// and the operand rewrite of a tile cost is instructions issued and fetched.
__device__ __forceinline__ uint64_t pair(float x, float y) { uint64_t r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y)); return r; }
__device__ __forceinline__ void unpair(uint64_t v, float& x, float& y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v)); }
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) { uint64_t r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) { uint64_t r; asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) { uint64_t r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) { uint64_t r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }
__device__ __forceinline__ float4 unpair4(uint64_t lo, uint64_t hi) { float4 r; unpair(lo, r.x, r.y); unpair(hi, r.z, r.w); return r; }
__device__ __forceinline__ float4 add4(float4 a, float4 b) { return unpair4(add2(pair(a.x, a.y), pair(b.x, b.y)), add2(pair(a.z, a.w), pair(b.z, b.w))); }
__device__ __forceinline__ float4 sub4(float4 a, float4 b) { return unpair4(sub2(pair(a.x, a.y), pair(b.x, b.y)), sub2(pair(a.z, a.w), pair(b.z, b.w))); }
__device__ __forceinline__ float4 mul4(float4 a, float4 b) { return unpair4(mul2(pair(a.x, a.y), pair(b.x, b.y)), mul2(pair(a.z, a.w), pair(b.z, b.w))); }
__device__ __forceinline__ float4 fma4(float4 a, float4 b, float4 c)
{
    return unpair4(fma2(pair(a.x, a.y), pair(b.x, b.y), pair(c.x, c.y)), fma2(pair(a.z, a.w), pair(b.z, b.w), pair(c.z, c.w)));
}
// what the tensor core ignores of a value
__device__ __forceinline__ float4 lo_part(float4 v) { return sub4(v, make_float4(tf32_hi(v.x), tf32_hi(v.y), tf32_hi(v.z), tf32_hi(v.w))); }

// Statistics of a BN's input from the partial moments of one micro-batch: rows of (mean[C], M2[C]) with n values each.
//   mean = ref + sum n (mean_u - ref) / N,   M2 = sum M2_u + sum n (mean_u - ref)^2 - N (mean - ref)^2,   ref = row 0's mean:
// no difference of large numbers appears however far a channel's mean is from zero compared with its spread.  Fixed order
// (every CTA of a launch gets the same bits), fp32 terms, the last combination in fp64.  THREADS threads, which share named
// barrier 1; tab: mean[C], rstd[C]; red: 4 x THREADS float4.  First every thread adds its rows of four channels, then one
// thread per channel combines: what this costs is latency and instruction fetches, so nothing is unrolled that need not be.
template <int THREADS>
__device__ __forceinline__ void merge_moments(const float* partials, int rows, int C, double inv_rows, float eps, float* tab, float4* red, int tid)
{
    const float* counts = partials + (size_t)rows * 2 * C;
    const int c4n = C >> 2;
    const int L = c4n <= THREADS ? THREADS / c4n : 1;
#pragma unroll 1
    for (int c0 = 0; c0 < c4n; c0 += THREADS) {
        const int width = c4n - c0 < THREADS ? c4n - c0 : THREADS;       // float4 columns of this pass
        const int ln = L > 1 ? tid / c4n : 0, local = L > 1 ? tid - ln * c4n : tid, col = c0 + local;
        const bool mine = local < width && ln < L;
        float4 sd = make_float4(0.f, 0.f, 0.f, 0.f), sq = sd, m2 = sd, ref = sd;
        if (mine) {
            ref = __ldcg(reinterpret_cast<const float4*>(partials) + col);
#pragma unroll 1
            for (int k0 = ln; k0 < rows; k0 += 4 * L) {
                float4 a[4], b[4];
                float n[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int k = k0 + j * L;
                    const bool have = k < rows;
                    const float4* row = reinterpret_cast<const float4*>(partials + (size_t)(have ? k : 0) * 2 * C);
                    n[j] = have ? __ldcg(counts + k) : 0.f;
                    a[j] = __ldcg(row + col);
                    b[j] = have ? __ldcg(row + c4n + col) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float dx = a[j].x - ref.x, dy = a[j].y - ref.y, dz = a[j].z - ref.z, dw = a[j].w - ref.w;
                    const float nx = n[j] * dx, ny = n[j] * dy, nz = n[j] * dz, nw = n[j] * dw;
                    sd.x += nx; sd.y += ny; sd.z += nz; sd.w += nw;
                    sq.x = fmaf(nx, dx, sq.x); sq.y = fmaf(ny, dy, sq.y); sq.z = fmaf(nz, dz, sq.z); sq.w = fmaf(nw, dw, sq.w);
                    m2 = add4(m2, b[j]);
                }
            }
        }
        int lanes = L, at = tid;                      // row lanes left to add: red[lane * width + local]
        bool put = mine;
        if (c4n <= 16 && (c4n & (c4n - 1)) == 0) {
            // the row lanes of a column inside a warp first: a fixed butterfly
#pragma unroll 1
            for (int o = 16; o >= c4n; o >>= 1) { sd = lane_sum(sd, o); sq = lane_sum(sq, o); m2 = lane_sum(m2, o); }
            lanes = THREADS / 32;
            at = (tid >> 5) * c4n + (tid & 31);
            put = (tid & 31) < c4n;
        }
        if (put) { red[at] = sd; red[THREADS + at] = sq; red[2 * THREADS + at] = m2; }
        if (mine && ln == 0) red[3 * THREADS + local] = ref;
        asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
        const float* r = reinterpret_cast<const float*>(red);
#pragma unroll 1
        for (int c = tid; c < 4 * width; c += THREADS) {
            float d = 0.f, q = 0.f, v = 0.f;
#pragma unroll 2
            for (int l = 0; l < lanes; ++l) { const int i = 4 * l * width + c; d += r[i]; q += r[4 * THREADS + i]; v += r[8 * THREADS + i]; }
            const double dm = (double)d * inv_rows;
            double var = ((double)v + (double)q) * inv_rows - dm * dm;
            if (var < 0.0) var = 0.0;
            tab[4 * c0 + c] = (float)((double)r[12 * THREADS + c] + dm);
            tab[C + 4 * c0 + c] = 1.0f / sqrtf((float)(var + (double)eps));
        }
        if (c0 + THREADS < c4n) asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
    }
}

// Walks the units of this CTA: micro-batch, unit of the micro-batch, part of the K loop.  What a CTA takes are whole blocks of
// `unit_block` consecutive units of a micro-batch, so that the BN moments of a block are formed by one CTA.
struct UnitWalk {
    int m, ul, z, left;          // left: blocks, the current one included
    int end;                     // first unit beyond the current block
    __device__ __forceinline__ UnitWalk(const PipeScalars& p, int m_first, int first, int count) : left(count)
    {
        z = 0;
        if (p.ksplit > 1) { z = first % p.ksplit; first /= p.ksplit; }
        m = first / p.blocks_per_m;
        ul = (first - m * p.blocks_per_m) * p.unit_block;
        m += m_first;
        set_end(p);
    }
    __device__ __forceinline__ void set_end(const PipeScalars& p) { end = ul + p.unit_block < p.units_per_m ? ul + p.unit_block : p.units_per_m; }
    __device__ __forceinline__ void next(const PipeScalars& p)
    {
        if (p.ksplit > 1) {      // (blocks of one unit)
            --left;
            if (++z < p.ksplit) return;
            z = 0;
            if (++ul == p.units_per_m) { ul = 0; ++m; }
            return;
        }
        if (++ul < end) return;
        --left;
        if (ul == p.units_per_m) { ul = 0; ++m; }
        set_end(p);
    }
    __device__ __forceinline__ bool last_of_block() const { return ul + 1 == end; }
    __device__ __forceinline__ bool last(const PipeScalars& p) const { return left == 1 && (p.ksplit > 1 || last_of_block()); }
    __device__ __forceinline__ int tiles(const PipeScalars& p) const { const int n = p.tiles_per_m - ul * p.T; return n < p.T ? n : p.T; }
    __device__ __forceinline__ int kb(const PipeScalars& p) const { return p.ksplit > 1 ? z * p.n_chunks / p.ksplit : 0; }
    __device__ __forceinline__ int ke(const PipeScalars& p) const { return p.ksplit > 1 ? (z + 1) * p.n_chunks / p.ksplit : p.n_chunks; }
};

// The operand block of a unit: whole copy blocks around the positions it needs.
struct Span {
    int block0, blocks;          // copy blocks (block0 may be -1: the zero row above the first map)
    int pos0, rows, lead;        // position of the first row, rows, rows in front of the unit's first halo row
};
__device__ __forceinline__ Span span_of(const PipeScalars& p, const UnitWalk& u)
{
    Span r;
    const int start = u.ul * p.T * kTileM - p.halo, need = u.tiles(p) * kTileM + 2 * p.halo;
    if (p.flat) { r.block0 = start / kTileM; r.blocks = need / kTileM; r.pos0 = start; r.rows = need; r.lead = 0; return r; }
    const int bp = p.box_pos;
    r.block0 = div_magic(start + bp * 2, bp, p.magic_box) - 2;      // halo <= 2 blocks: the dividend is never negative
    r.pos0 = r.block0 * bp;
    r.lead = start - r.pos0;
    r.blocks = div_magic(r.lead + need + bp - 1, bp, p.magic_box);
    r.rows = r.blocks * bp;
    return r;
}

// What one warp does with 32 rows x 32 (or 16) columns of a finished tile, which stand in its patch of shared memory.
struct EmitArgs {
    float* out;                  // this warp's column group
    const float* extra;
    const float4* patch;
    float* moments;              // the warp's k, sum (x - k), sum (x - k)^2 of its columns: three rows of mom_pitch floats, or null
    int mom_pitch;
    bool accumulate, ok;
    int zero_fill, dense_h, dense_w;
    // not null: `extra` is the input x of a BN+ReLU whose output gradient this is: it is not added; the sums are those of
    // dz = dy where the activation was positive, and of dz * xhat
    const float* bn_mean;        // this column group's: mean, rstd (bn_c floats further on), gamma, beta
    const float* bn_gamma;
    const float* bn_beta;
    int bn_c;
};

// The residuals of four row steps, beginning with step b.
__device__ __forceinline__ void emit_residuals(const EmitArgs& a, int ro, int lane, int lsh, int b, float4* e)
{
    const int cq = lane & ((1 << lsh) - 1), r = (lane >> lsh) + ((32 >> lsh) * b);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int so = __shfl_sync(0xffffffffu, ro, r + (32 >> lsh) * i);
        // (not the read-only path: the preceding kernel may have written it)
        e[i] = __ldcg(reinterpret_cast<const float4*>(a.extra + (so >= 0 ? so + 4 * cq : 0)));
    }
}

// 1 << lsh lanes hold a row's 16-byte pieces; ro is this lane's row offset or -1.  Loads, shared-memory reads and stores are
// batched by kind, so that a batch's latencies overlap; there is ONE copy of this code for all widths and forms, since a
// launch of a few microseconds runs it once or twice and would wait for its instructions otherwise (the kernel had grown to
// 200 KB with specialised copies: 4000-8000 clocks for the first tile of a launch).
// Moments are taken about a value of the column: sums of x and x*x themselves would cancel for a channel whose mean is large
// against its spread.
template <bool BNB>
__device__ __forceinline__ void emit_rows(const EmitArgs& a, int ro, int fill, int lane, int lsh, bool have_shift, float4* e)
{
    const int cq = lane & ((1 << lsh) - 1), rq = lane >> lsh, rstep = 32 >> lsh, steps = 1 << lsh;
    const unsigned int who = __ballot_sync(0xffffffffu, ro >= 0);        // lane = row here
    float4 k = make_float4(0.f, 0.f, 0.f, 0.f), sd = k, sq = k;
    const bool moments = a.moments != nullptr && who != 0u;
    float4 rs = k, g = k, bt = k;
    if (BNB) {
        // (statistics are results of the step: not the read-only path)
        k = __ldcg(reinterpret_cast<const float4*>(a.bn_mean + 4 * cq)); rs = __ldcg(reinterpret_cast<const float4*>(a.bn_mean + a.bn_c + 4 * cq));
        g = __ldg(reinterpret_cast<const float4*>(a.bn_gamma + 4 * cq)); bt = __ldg(reinterpret_cast<const float4*>(a.bn_beta + 4 * cq));
    } else if (moments) {
        if (have_shift) k = *reinterpret_cast<const float4*>(a.moments + 4 * cq);
        else {
            const int r0 = __ffs(who) - 1, so = __shfl_sync(0xffffffffu, ro, r0);
            k = a.patch[r0 * 8 + (cq ^ (r0 & 7))];
            if (a.extra) k = add4(k, __ldcg(reinterpret_cast<const float4*>(a.extra + so + 4 * cq)));
        }
    }
#pragma unroll 1
    for (int b = 0; b < steps; b += 4) {
        int so[4];
        float4 v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = rq + rstep * (b + i);
            so[i] = __shfl_sync(0xffffffffu, ro, r);
            v[i] = a.patch[r * 8 + (cq ^ (r & 7))];
        }
        if (BNB) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const bool real = so[i] >= 0;
                const float4 xh = mul4(sub4(e[i], k), rs), z = fma4(g, xh, bt);
                const float4 d = make_float4(real && z.x > 0.f ? v[i].x : 0.f, real && z.y > 0.f ? v[i].y : 0.f, real && z.z > 0.f ? v[i].z : 0.f,
                                             real && z.w > 0.f ? v[i].w : 0.f);
                sd = add4(sd, d);
                sq = fma4(d, xh, sq);
            }
            if (b + 4 < steps) emit_residuals(a, ro, lane, lsh, b + 4, e);
        } else if (a.extra) {
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = add4(v[i], e[i]);
            if (b + 4 < steps) emit_residuals(a, ro, lane, lsh, b + 4, e);
        }
        float* out = a.out + 4 * cq;
        if (a.accumulate) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (so[i] >= 0) v[i] = add4(v[i], __ldcg(reinterpret_cast<const float4*>(out + so[i])));
        }
        if (a.ok) {
#pragma unroll
            for (int i = 0; i < 4; ++i) if (so[i] >= 0) *reinterpret_cast<float4*>(out + so[i]) = v[i];
        }
        if (moments && !BNB) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 d = sub4(so[i] >= 0 ? v[i] : k, k);
                sd = add4(sd, d);
                sq = fma4(d, d, sq);
            }
        }
    }
    if (moments) {
        // the lanes that share a column, then one lane per four columns adds to the block's sums
#pragma unroll 1
        for (int o = 16; o >= steps; o >>= 1) { sd = lane_sum(sd, o); sq = lane_sum(sq, o); }
        if (lane < steps) {
            float4 *pk = reinterpret_cast<float4*>(a.moments + 4 * cq), *pd = reinterpret_cast<float4*>(a.moments + a.mom_pitch + 4 * cq),
                   *pq = reinterpret_cast<float4*>(a.moments + 2 * a.mom_pitch + 4 * cq);
            if (have_shift) { *pd = add4(*pd, sd); *pq = add4(*pq, sq); }
            else { *pk = k; *pd = sd; *pq = sq; }
        }
    }
    if (a.zero_fill == 2) {
        // strided data gradient: the positions between the samples receive no contribution
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
        for (int i = 0; i < steps; ++i) {
            const int so = __shfl_sync(0xffffffffu, ro, rq + rstep * i), f = __shfl_sync(0xffffffffu, fill, rq + rstep * i);
            if (so < 0 || !a.ok) continue;
            float* out = a.out + so + 4 * cq;
            if (f & 1) *reinterpret_cast<float4*>(out + a.dense_w) = zero;
            if (f & 2) *reinterpret_cast<float4*>(out + a.dense_h) = zero;
            if (f & 4) *reinterpret_cast<float4*>(out + a.dense_h + a.dense_w) = zero;
        }
    }
    __syncwarp();
}

// The MMA issuer (one thread).  RESIDENT: the weights of all chunks and taps stand in shared memory; otherwise a ring.
// KIND 0: one pass; 1: hi*hi and hi*lo from one MMA over [B_hi; B_lo]; 2: three MMAs.  Everything that does not change is
// taken out of the loops and nothing in the tap loop waits or branches on loaded values: with the modes told apart inside it
// an MMA took 115 clocks to issue, against 40 (N = 32) the tensor core needs.
struct MmaEnv {
    volatile int* abort_flag;
    uint32_t smem_base, tmem_base, a_full, a_empty, b_full, b_empty, acc_full, acc_empty;
    int m_first, u_first, u_count;
    int *a_used, *b_used;
    bool drain;                  // wait until every barrier has seen its last arrival (they are used again)
};
template <int KIND>
__device__ __forceinline__ void issue_tile(uint32_t acc, uint64_t a, uint64_t b, uint64_t b_half, uint32_t idesc, uint32_t idesc2, uint32_t keep)
{
    // (a: value or hi part, +4: lo part; +2: the chunk's second K step)
    if (KIND == 0) {
        umma_tf32(acc, a, b, idesc, keep);
        umma_tf32(acc, a + 2, b + 2, idesc, 1u);
    } else if (KIND == 1) {
        umma_tf32(acc, a, b, idesc2, keep);
        umma_tf32(acc, a + 4, b, idesc, 1u);
        umma_tf32(acc, a + 2, b + 2, idesc2, 1u);
        umma_tf32(acc, a + 6, b + 2, idesc, 1u);
    } else {
        const uint64_t bl = b + b_half;
        umma_tf32(acc, a, b, idesc, keep);
        umma_tf32(acc, a + 4, b, idesc, 1u);
        umma_tf32(acc, a, bl, idesc, 1u);
        umma_tf32(acc, a + 2, b + 2, idesc, 1u);
        umma_tf32(acc, a + 6, b + 2, idesc, 1u);
        umma_tf32(acc, a + 2, bl + 2, idesc, 1u);
    }
}
template <bool RESIDENT, int KIND>
__device__ __forceinline__ void mma_role(const PipeScalars& p, const MmaEnv& e)
{
    const uint64_t a_desc = smem_desc(0, 16, 1024, 128), b_desc = smem_desc(0, 16, 512, 64);
    const uint32_t idesc = p.idesc, idesc2 = p.idesc2, acc_cols = p.acc_cols, a_step = p.a_stage_bytes >> 4, b_step = p.b_stage_bytes >> 4, b_tap = p.b_tap_bytes >> 4;
    const uint64_t b_half = ((uint32_t)p.n_chunk * 64u) >> 4;
    const int taps = p.taps, group = RESIDENT ? p.taps : p.b_taps, R = p.R, a_stages = p.a_stages, b_stages = p.b_stages, acc_bufs = p.acc_bufs, T = p.T;
    const uint64_t row_step = (uint64_t)((p.Wp - (R - 1)) * 8);      // from a window row's last tap to the next row's first
    const uint64_t a_first = a_desc | (uint64_t)(e.smem_base >> 4), b_first = b_desc | (uint64_t)((e.smem_base + p.off_b) >> 4);
    int s = 0, bs = 0, buf = 0, b_it = 0, a_it = 0;
    uint32_t apar = 0, bpar = 0, cpar = 1u;
    if (RESIDENT) {
        b_it = 1;
        if (!mbar_wait(e.b_full, 0, e.abort_flag)) { report(p.status, 22); return; }
    }
#pragma unroll 1
    for (UnitWalk u(p, e.m_first, e.u_first, e.u_count); u.left > 0; u.next(p)) {
        const int nt = u.tiles(p), kb = u.kb(p), ke = u.ke(p);
        const uint64_t lead = (uint64_t)(span_of(p, u).lead * 8);
        if (!mbar_wait(e.acc_empty + 8 * buf, cpar, e.abort_flag)) { report(p.status, 23); return; }
        tc_fence_after();
        const uint32_t acc0 = e.tmem_base + (uint32_t)(buf * T) * acc_cols;
        uint32_t keep = 0u;
#pragma unroll 1
        for (int c = kb; c < ke; ++c) {
            if (!mbar_wait(e.a_full + 8 * s, apar, e.abort_flag)) { report(p.status, 24); return; }
            uint64_t a = a_first + (uint64_t)((uint32_t)s * a_step) + lead;
            uint64_t b = RESIDENT ? b_first + (uint64_t)((uint32_t)(c * taps) * b_tap) : 0;
            int sx = 0;
#pragma unroll 1
            for (int left = taps; left > 0; left -= group) {
                if (!RESIDENT) {
                    if (!mbar_wait(e.b_full + 8 * bs, bpar, e.abort_flag)) { report(p.status, 25); *e.b_used = b_it; *e.a_used = a_it; return; }
                    b = b_first + (uint64_t)((uint32_t)bs * b_step);
                }
#pragma unroll 1
                for (int k = 0; k < group; ++k) {
#pragma unroll 1
                    for (int t = 0; t < nt; ++t) issue_tile<KIND>(acc0 + (uint32_t)t * acc_cols, a + (uint64_t)(t * 1024), b, b_half, idesc, idesc2, keep);
                    keep = 1u;
                    b += b_tap;
                    a += 8;
                    if (++sx == R) { sx = 0; a += row_step - 8; }
                }
                if (!RESIDENT) {
                    umma_commit(e.b_empty + 8 * bs);
                    ++b_it;
                    if (++bs == b_stages) { bs = 0; bpar ^= 1u; }
                }
            }
            umma_commit(e.a_empty + 8 * s);
            ++a_it;
            if (++s == a_stages) { s = 0; apar ^= 1u; }
        }
        umma_commit(e.acc_full + 8 * buf);
        if (++buf == acc_bufs) { buf = 0; cpar ^= 1u; }
        *e.b_used = b_it; *e.a_used = a_it;
    }
    if (e.drain) {
#pragma unroll 1
        for (int i = 0; i < a_stages && i < a_it; ++i) mbar_wait(e.a_empty + 8 * i, (uint32_t)((a_it - 1 - i) / a_stages) & 1u, e.abort_flag);
        if (!RESIDENT)
#pragma unroll 1
            for (int i = 0; i < b_stages && i < b_it; ++i) mbar_wait(e.b_empty + 8 * i, (uint32_t)((b_it - 1 - i) / b_stages) & 1u, e.abort_flag);
    }
}

struct PipeShared {
    uint64_t bars[3 * kMaxA + 2 * kMaxB + 4];         // a_raw, a_full, a_empty, acc_full[2], acc_empty[2], b_full, b_empty
    uint32_t tmem_slot;
    int abort_flag, b_issued, b_used, a_issued, a_used;
    int last_of_unit;
};
// One warp, a barrier a lane: by one thread, whose first parameters came through a constant cache that a warp had flooded with
// 32 different addresses, the 44 of them took 2.8 us (0.3 us now).  Every launch of a chain waits for that, since its CTAs
// only start when the predecessor's leave: ResNet-29 0.990 -> 0.937 ms, ResNet-110 6.27 -> 5.96, scoring ResNet-182 6.87 -> 6.68.
__device__ __forceinline__ void pipe_init_barriers(const PipeScalars& p, PipeShared& sh, int lane)
{
    const uint32_t bar = smem_u32(&sh.bars[0]), split = (uint32_t)(kSplitWarps / p.split_groups), emit = p.epi_alternate ? kEpiWarps / 2 : kEpiWarps;
#pragma unroll
    for (int s = lane; s < 3 * kMaxA + 2 * kMaxB + 4; s += 32) {
        const bool full = s >= kMaxA && s < 2 * kMaxA, acc_empty = s >= 3 * kMaxA + 2 && s < 3 * kMaxA + 4;
        mbar_init(bar + 8 * s, full ? split : (acc_empty ? emit : 1u));
    }
    if (lane == 0) { sh.abort_flag = 0; sh.b_issued = 0; sh.b_used = 0; sh.a_issued = 0; sh.a_used = 0; }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// The work of one CTA (number bid of nblk) of a launch: the barriers are initialised, tensor memory is allocated.
// FLAT: the operand's positions and the output's pixels are the same consecutive rows (1x1 windows without a stride).
// BNB: a data gradient that forms the sums of a BN+ReLU's backward.
// CELL: inside the persistent cell kernel, which keeps its tensor memory and has no successor to trigger.
template <bool BN_IN, bool FLAT, bool BNB, bool CELL>
__device__ __forceinline__ void pipe_cta(const PipeParams& gp, const PipeScalars& p, PipeShared& sh, uint8_t* smem, const uint32_t tmem_base,
                                         const int m_first, const int m_count, const int bid, const int nblk)
{
    const uint32_t smem_base = smem_u32(smem);
    const int warp = warp_index(), lane = threadIdx.x & 31;
    uint64_t* bars = sh.bars;
    int &abort_flag = sh.abort_flag, &b_issued = sh.b_issued, &b_used = sh.b_used, &a_issued = sh.a_issued, &a_used = sh.a_used, &last_of_unit = sh.last_of_unit;
    const uint32_t a_raw = smem_u32(&bars[0]), a_full = smem_u32(&bars[kMaxA]), a_empty = smem_u32(&bars[2 * kMaxA]),
                   acc_full = smem_u32(&bars[3 * kMaxA]), acc_empty = smem_u32(&bars[3 * kMaxA + 2]), b_full = smem_u32(&bars[3 * kMaxA + 4]),
                   b_empty = smem_u32(&bars[3 * kMaxA + 4 + kMaxB]);
    // a CTA keeps one channel slice and takes consecutive blocks of units: as many as the others or one more
    int slice = 0, cta = bid, ctas = nblk;
    if (p.slices > 1) { slice = cta % p.slices; cta /= p.slices; ctas /= p.slices; }
    const int total = m_count * p.blocks_per_m * p.ksplit;
    const int each = total / ctas, more = total - each * ctas;
    const int u_first = cta * each + (cta < more ? cta : more), u_count = each + (cta < more ? 1 : 0);
    const int co0 = slice * p.n_chunk;

    if (warp == 0) {
        if (elect_one()) {
            // ---- operand copies ----
            if (!CELL) pdl_wait();
            const int S = p.a_stages;
            int s = 0, it = 0;
            uint32_t par = 1u;
            bool live = true;
#pragma unroll 1
            for (UnitWalk u(p, m_first, u_first, u_count); u.left > 0 && live; u.next(p)) {
                const Span sp = span_of(p, u);
                const uint32_t tx = (uint32_t)sp.rows * 64u;
                // first block: map, row within it
                int img0 = 0, h0 = 0, strip0 = 0;
                if (!p.flat) {
                    if (sp.block0 < 0) { img0 = -1; h0 = p.blocks_per_img + sp.block0; if (h0 < 0) h0 = 0; }
                    else { img0 = div_magic(sp.block0, p.blocks_per_img, p.magic_bpi); h0 = sp.block0 - img0 * p.blocks_per_img; }
                    if (p.strips > 1 && img0 >= 0) { const int n = div_magic(img0, p.strips, p.magic_strip); strip0 = img0 - n * p.strips; img0 = n; }
                }
                const int first = (int)((long long)u.m * p.pix_ms);
#pragma unroll 1
                for (int c = u.kb(p), ce = u.ke(p); c < ce; ++c, ++it) {
                    if (!mbar_wait(a_empty + 8 * s, par, &abort_flag)) { report(p.status, 20); live = false; break; }
                    const uint32_t bar = a_raw + 8 * s;
                    uint32_t dst = smem_base + (uint32_t)s * p.a_stage_bytes;
                    mbar_expect_tx(bar, tx);
                    if (p.flat) {
#pragma unroll 1
                        for (int k = 0; k < sp.blocks; ++k, dst += kTileM * 128u) tma_load_2d(dst, &gp.tm_a, bar, 16 * c, first + (sp.block0 + k) * kTileM);
                    } else {
                        int img = img0, h = h0, strip = strip0;
                        const uint32_t step = (uint32_t)p.box_pos * 128u;
#pragma unroll 1
                        for (int k = 0; k < sp.blocks; ++k, dst += step) {
                            // (a block beyond the last row of its map is the zero row: outside the tensor, filled with zeros)
                            tma_load_4d(dst, &gp.tm_a, bar, 16 * c, strip * p.strip_w - p.col0, h * p.box_h, first + (img < 0 ? 0 : img));
                            if (++h == p.blocks_per_img) { h = 0; if (img < 0 || ++strip == p.strips) { strip = 0; ++img; } }
                        }
                    }
                    if (++s == S) { s = 0; par ^= 1u; }
                }
            }
            a_issued = it;
        }
    } else if (warp == 1) {
        if (elect_one()) {
            // ---- weights ----
            if (!CELL && !p.w_ready) pdl_wait();
            const uint32_t half = (uint32_t)p.n_chunk * 64u, tap_bytes = p.b_tap_bytes, dst0 = smem_base + p.off_b;
            const bool three = p.three != 0;
            const uint32_t tx = three ? 2u * half : half;
            const int taps = p.taps, c_in = p.c_in;
            if (p.b_resident) {
                const int n = p.n_chunks * taps;
                mbar_expect_tx(b_full, tx * (uint32_t)n);
                uint32_t dst = dst0;
#pragma unroll 1
                for (int c = 0; c < p.n_chunks; ++c)
#pragma unroll 1
                    for (int tap = 0; tap < taps; ++tap, dst += tap_bytes) {
                        tma_load_2d(dst, &gp.tm_b, b_full, tap * c_in + 16 * c, co0);
                        if (three) tma_load_2d(dst + half, &gp.tm_b_lo, b_full, tap * c_in + 16 * c, co0);
                    }
                b_issued = 1;
            } else {
                int s = 0, it = 0;
                uint32_t par = 1u;
                bool live = true;
#pragma unroll 1
                for (UnitWalk u(p, m_first, u_first, u_count); u.left > 0 && live; u.next(p))
#pragma unroll 1
                    for (int c = u.kb(p), ce = u.ke(p); c < ce && live; ++c)
#pragma unroll 1
                        for (int tap = 0; tap < taps; ++it) {
                            if (!mbar_wait(b_empty + 8 * s, par, &abort_flag)) { report(p.status, 21); live = false; break; }
                            const uint32_t bar = b_full + 8 * s;
                            uint32_t dst = dst0 + (uint32_t)s * p.b_stage_bytes;
                            mbar_expect_tx(bar, tx * (uint32_t)p.b_taps);
#pragma unroll 1
                            for (int e = tap + p.b_taps; tap < e; ++tap, dst += tap_bytes) {
                                tma_load_2d(dst, &gp.tm_b, bar, tap * c_in + 16 * c, co0);
                                if (three) tma_load_2d(dst + half, &gp.tm_b_lo, bar, tap * c_in + 16 * c, co0);
                            }
                            if (++s == p.b_stages) { s = 0; par ^= 1u; }
                        }
                b_issued = it;
            }
        }
    } else if (warp == 2) {
        if (elect_one()) {
            // ---- MMAs ----
            const MmaEnv env{&abort_flag, smem_base, tmem_base, a_full, a_empty, b_full, b_empty, acc_full, acc_empty, m_first, u_first, u_count, &a_used, &b_used, CELL};
            if (p.b_resident) {
                if (!p.three) mma_role<true, 0>(p, env);
                else if (p.stacked) mma_role<true, 1>(p, env);
                else mma_role<true, 2>(p, env);
            } else {
                if (!p.three) mma_role<false, 0>(p, env);
                else if (p.stacked) mma_role<false, 1>(p, env);
                else mma_role<false, 2>(p, env);
            }
        }
    } else if (warp >= kFirstSplit && warp < kFirstSplit + kSplitWarps) {
        // ---- the operand: normalise, split ----
        // The warps work on `split_groups` blocks at a time: what a block costs is a chain of latencies - copy, shared-memory
        // reads, arithmetic, stores, fence, hand-over - and not instructions.  The ring is a multiple of the groups, so that a
        // stage is always the same group's: one that came back to a stage after another group's turn could take the parity of
        // the round before last for this round's.
        const int tid = threadIdx.x - 32 * kFirstSplit;
        const int groups = p.split_groups, wpg = kSplitWarps / groups, my_group = (tid >> 5) / wpg, gw = (tid >> 5) - my_group * wpg;
        // a thread owns one 16-byte quarter of the rows row0 + row_step * j; the eight rows of a warp are taken so that a
        // quarter-warp holds a row and the one four further on: their swizzled quarters cover all banks
        const int row_step = 8 * wpg;
        const int cph = lane & 3, r8 = ((lane >> 2) & 1) * 4 + (lane >> 3), row0 = gw * 8 + r8;
        const uint32_t at_hi = (uint32_t)row0 * 128u + (uint32_t)((cph ^ r8) << 4), at_lo = (uint32_t)row0 * 128u + (uint32_t)(((cph + 4) ^ r8) << 4);
        const uint32_t byte_step = (uint32_t)row_step * 128u;
        const int S = p.a_stages, C = p.c_in, halo = p.halo;
        const bool three = p.three != 0;
        float* tab = reinterpret_cast<float*>(smem + p.off_bn);
        if (BN_IN) {
#pragma unroll 1
            for (int i = tid; i < C; i += kSplitThreads) { tab[2 * C + i] = __ldg(p.bn_gamma + i); tab[3 * C + i] = __ldg(p.bn_beta + i); }
            if (!CELL) pdl_wait();
        }
        // a step of row_step positions in maps, rows and columns of the padded grid
        const int dn = BN_IN && !FLAT ? row_step / p.img_pos : 0, drem = row_step - dn * p.img_pos;
        const int dy = BN_IN && !FLAT ? drem / p.Wp : 0, dx = drem - dy * p.Wp, Hp = BN_IN && !FLAT ? p.img_pos / p.Wp : 1;
        // this group's next block: its chunk within the unit, its place in the ring
        int s = my_group, ahead = my_group, cur_m = -1;
        uint32_t par = 0;
        const bool store_y = BN_IN && slice == 0;
        bool ok = true;
#pragma unroll 1
        for (UnitWalk cu(p, m_first, u_first, u_count); cu.left > 0; cu.next(p)) {
            const int kb = cu.kb(p), ke = cu.ke(p);
            const Span sp = span_of(p, cu);
            const int own_lo = sp.lead + halo, own_hi = own_lo + cu.tiles(p) * kTileM, valid = p.pos_per_m - sp.pos0;
            if (BN_IN) {
                if (cu.m != cur_m) {
                    cur_m = cu.m;
                    split_sync();                     // everybody is done with the table of the micro-batch before
                    merge_moments<kSplitThreads>(p.bn_partials + (size_t)cur_m * partial_floats(p.bn_units, C), p.bn_units, C, p.bn_inv_rows, p.bn_eps, tab,
                                  reinterpret_cast<float4*>(smem + p.off_red), tid);
                    split_sync();
                }
                if (slice == 0 && cu.ul == 0 && cu.z == 0)
#pragma unroll 1
                    for (int i = tid; i < 2 * C; i += kSplitThreads) p.bn_stats[(size_t)cur_m * 2 * C + i] = tab[i];
            }
#pragma unroll 1
            for (int c = kb + ahead; c < ke; c += groups) {
                {
                    ok = mbar_wait(a_raw + 8 * s, par, &abort_flag) && ok;
                    // (after a wait that gave up the warps run through the rest without waiting: they still have to meet at
                    // the named barriers)
                    if (!ok && lane == 0) report(p.status, 26);
                    uint8_t* hi = smem + (uint32_t)s * p.a_stage_bytes + at_hi;
                    uint8_t* lo = smem + (uint32_t)s * p.a_stage_bytes + at_lo;
                    if (BN_IN) {
                        const int ch = 16 * c + 4 * cph;
                        const float4 mu = *reinterpret_cast<const float4*>(tab + ch), rs = *reinterpret_cast<const float4*>(tab + C + ch);
                        const float4 g = *reinterpret_cast<const float4*>(tab + 2 * C + ch), b = *reinterpret_cast<const float4*>(tab + 3 * C + ch);
                        float* ydst = p.bn_y + (long long)cur_m * p.in_ms + 16 * c + 4 * cph;
                        int yo = (sp.pos0 + row0) * C;                   // FLAT: offset of this thread's first row
                        int pn = 0, py = 0, px = 0;                      // otherwise its map, row and column
                        if (!FLAT) {
                            int pos = sp.pos0 + row0;
                            if (pos < 0) { pos += p.img_pos; pn = -1; }
                            const int q = div_magic(pos, p.img_pos, p.magic_img);
                            pn += q; pos -= q * p.img_pos;
                            py = div_magic(pos, p.Wp, p.magic_w); px = pos - py * p.Wp;
                        }
                        // four rows in flight; the block is allocated in whole batches, so the last one needs no bounds
#pragma unroll 1
                        for (int row = row0; row < sp.rows; row += kRowBatch * row_step, hi += kRowBatch * byte_step, lo += kRowBatch * byte_step) {
                            float4 v[kRowBatch];
#pragma unroll
                            for (int j = 0; j < kRowBatch; ++j) v[j] = *reinterpret_cast<const float4*>(hi + byte_step * j);
                            int off[kRowBatch];
                            bool inside[kRowBatch], own[kRowBatch];
#pragma unroll
                            for (int j = 0; j < kRowBatch; ++j) {
                                const int r = row + row_step * j;
                                if (FLAT) {
                                    inside[j] = own[j] = r < valid;
                                    off[j] = yo; yo += row_step * C;
                                } else {
                                    inside[j] = px < p.W && py < p.Hv && pn >= 0 && r < valid;
                                    own[j] = inside[j] && r >= own_lo && r < own_hi;
                                    off[j] = pn * p.in_sn + py * p.in_sh + px * p.in_sw;
                                    px += dx; py += dy; pn += dn;
                                    if (px >= p.Wp) { px -= p.Wp; ++py; }
                                    if (py >= Hp) { py -= Hp; ++pn; }
                                }
                            }
#pragma unroll
                            for (int j = 0; j < kRowBatch; ++j) {
                                const float4 z = fma4(g, mul4(sub4(v[j], mu), rs), b);
                                v[j] = make_float4(fmaxf(z.x, 0.f), fmaxf(z.y, 0.f), fmaxf(z.z, 0.f), fmaxf(z.w, 0.f));
                                if (!inside[j]) v[j] = make_float4(0.f, 0.f, 0.f, 0.f);      // the padding is zero AFTER the activation
                                *reinterpret_cast<float4*>(hi + byte_step * j) = v[j];
                            }
                            if (three)
#pragma unroll
                                for (int j = 0; j < kRowBatch; ++j)
                                    *reinterpret_cast<float4*>(lo + byte_step * j) =
                                        lo_part(v[j]);
                            if (store_y)
#pragma unroll
                                for (int j = 0; j < kRowBatch; ++j) if (own[j]) *reinterpret_cast<float4*>(ydst + off[j]) = v[j];
                        }
                    } else if (three) {
#pragma unroll 1
                        for (int row = row0; row < sp.rows; row += kRowBatch * row_step, hi += kRowBatch * byte_step, lo += kRowBatch * byte_step) {
                            float4 v[kRowBatch];
#pragma unroll
                            for (int j = 0; j < kRowBatch; ++j) v[j] = *reinterpret_cast<const float4*>(hi + byte_step * j);
#pragma unroll
                            for (int j = 0; j < kRowBatch; ++j)
                                *reinterpret_cast<float4*>(lo + byte_step * j) =
                                    lo_part(v[j]);
                        }
                    }
                    fence_async_smem();               // generic-proxy writes -> tensor-core reads
                    __syncwarp();
                    if (lane == 0) mbar_arrive(a_full + 8 * s);
                }
                s += groups;
                if (s >= S) { s -= S; par ^= 1u; }
                ahead += groups;
            }
            ahead -= ke - kb;
        }
    } else if (warp >= kFirstSplit + kSplitWarps) {
        // ---- write-out: tensor memory -> registers -> a 32 x 32 patch of shared memory -> global memory ----
        // A TMEM lane is a position, so stores straight from the registers touch 32 lines per instruction (measured: half a
        // sector per clock and SM); through a warp's own patch eight lanes write a row's 128 bytes, and a thread that keeps
        // four columns forms their moments without crossing lanes.
        const int tid = threadIdx.x - 32 * (kFirstSplit + kSplitWarps), ew = warp - kFirstSplit - kSplitWarps;
        const int quad = warp & 3, half = ew >> 2;    // a warp reads the 32 lanes of its quadrant; two warps share one
        const int n_chunk = p.n_chunk, groups = (n_chunk + 31) >> 5, T = p.T, C_out = p.c_out, ksplit = p.ksplit;
        const bool stacked = p.stacked != 0, stats = p.st_partials != nullptr;
        // Two sets of four warps.  With two accumulator sets and at most 64 channels each takes every other unit, so that the
        // latencies of one unit's write-out run beside the other's; otherwise they share a unit: alternate groups of 32
        // channels, or alternate tiles where there is one group.
        const bool alternate = p.epi_alternate != 0, by_tile = !alternate && groups == 1, whole = alternate || by_tile;
        const int g_first = whole ? 0 : half, g_step = whole ? 1 : 2, t_first = by_tile ? half : 0, t_step = by_tile ? 2 : 1;
        // (alternating sets: a block's first unit always counts as part 0..3, whichever set's turn it is, so that its moments are
        // added in the same order wherever in a CTA's work the block stands)
        const int parts = whole ? 8 : 4;
        int part = whole ? ew : quad;
        int turn = 0;
        float4* patch = reinterpret_cast<float4*>(smem + p.off_stage) + ew * 256;
        if (!CELL) pdl_wait();
        int buf = alternate ? half : 0, flip = 0;
        uint32_t par = 0;
        // the warps' moments of the block so far, twice: those of the block before may still be read
        float* const mom0 = reinterpret_cast<float*>(smem + p.off_stat);
        const int mom_size = parts * (3 * n_chunk + 1);
        bool have = false;
        int count = 0;
#pragma unroll 1
        for (UnitWalk u(p, m_first, u_first, u_count); u.left > 0; u.next(p)) {
            bool finish = true, ok = true;
            if (!alternate || turn == half) {
            const int nt = u.tiles(p);
            float* out = p.out + (long long)u.m * p.out_ms + co0;
            const float* addend = BNB ? p.bn_x : p.extra;
            const float* extra = addend ? addend + (long long)u.m * p.out_ms + co0 : nullptr;
            const float* bnb = BNB ? p.bn_stats + (long long)u.m * 2 * C_out + co0 : nullptr;
            EmitArgs ea{out, extra, patch, nullptr, n_chunk, p.accumulate != 0, true, p.zero_fill, p.dense_h, p.dense_w, nullptr, nullptr, nullptr, C_out};
            // this lane's row of a tile, and which neighbours of a strided data gradient's sample get zeros
            int ro = -1, fill = 0;
            auto place = [&](int t) {
                const int pos = (u.ul * T + t) * kTileM + quad * 32 + lane;
                if (FLAT) { ro = pos < p.pos_per_m ? pos * C_out : -1; return; }
                const Pixel px = locate(p, pos);
                ro = px.own ? px.n * p.os_n + px.y * p.os_h + px.x * p.os_w : -1;
                const bool right = 2 * px.x + 1 < p.out_w, below = 2 * px.y + 1 < p.out_h;
                fill = (right ? 1 : 0) | (below ? 2 : 0) | (right && below ? 4 : 0);
            };
            const uint32_t acc0 = tmem_base + (uint32_t)(buf * T) * p.acc_cols + ((uint32_t)(quad * 32) << 16);
            const size_t sk_tile = (size_t)kTileM * n_chunk;
            const float* sk_all = nullptr;
            // the first residuals travel while the accumulator is formed
            float4 e[4];
            place(t_first);
            if (extra && t_first < nt) { ea.extra = extra + 32 * g_first; emit_residuals(ea, ro, lane, n_chunk - 32 * g_first >= 32 ? 3 : 2, 0, e); }
            ok = mbar_wait(acc_full + 8 * buf, par, &abort_flag);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok && lane == 0) report(p.status, 27);
            if (!CELL && p.pdl_late && u.last(p)) pdl_launch_dependents();
            tc_fence_after();
            // 16 columns of this lane's row, hi and lo products added
            auto accumulator = [&](int t, int col, float* v) {
                const uint32_t at = acc0 + (uint32_t)t * p.acc_cols + (uint32_t)col;
                tmem_ld16_nowait(at, v);
                if (stacked) {
                    float w[16];
                    tmem_ld16_nowait(at + (uint32_t)n_chunk, w);
                    tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 16; j += 2) unpair(add2(pair(v[j], v[j + 1]), pair(w[j], w[j + 1])), v[j], v[j + 1]);
                } else {
                    tmem_ld_wait();
                }
            };
            if (ksplit > 1) {
                // this CTA's partial sums; the CTA that takes the last ticket of the unit adds them in split order
                const size_t key = (size_t)u.ul * p.slices + slice;
                char* base = p.sk_base + u.m * p.sk_ms;
                unsigned int* ticket = reinterpret_cast<unsigned int*>(base) + key;
                float* partials = reinterpret_cast<float*>(base + kSplitKTicketBytes);
                sk_all = partials + key * ksplit * T * sk_tile;
                float* mine = partials + (key * ksplit + u.z) * T * sk_tile;
#pragma unroll 1
                for (int t = t_first; t < nt; t += t_step)
#pragma unroll 1
                    for (int g = g_first; g < groups; g += g_step)
#pragma unroll 1
                        for (int h = 2 * g; h < 2 * g + 2 && 16 * h < n_chunk; ++h) {
                            float v[16];
                            accumulator(t, 16 * h, v);
                            if (ok) store16(mine + t * sk_tile + ((size_t)h * kTileM + quad * 32 + lane) * 16, v);
                        }
                __threadfence();
                epi_sync();
                if (tid == 0) {
                    last_of_unit = atomicAdd(ticket, 1u) == (unsigned int)ksplit - 1u;
                    if (last_of_unit) *ticket = 0u;
                }
                epi_sync();
                finish = last_of_unit != 0;
                if (finish) __threadfence();
            }
            ea.ok = ok;
#pragma unroll 1
            for (int t = t_first; finish && t < nt; t += t_step) {
                if (t > t_first) place(t);
                const int rows = __popc(__ballot_sync(0xffffffffu, ro >= 0));
                count += rows;
#pragma unroll 1
                for (int g = g_first, gi = 0; g < groups; g += g_step, ++gi) {
                    const int left = n_chunk - 32 * g, lsh = left >= 32 ? 3 : 2;
                    ea.out = out + 32 * g;
                    if (BNB) { ea.bn_mean = bnb + 32 * g; ea.bn_gamma = p.bn_gamma + co0 + 32 * g; ea.bn_beta = p.bn_beta + co0 + 32 * g; }
                    if (extra) {
                        ea.extra = extra + 32 * g;
                        if (t > t_first || gi > 0) emit_residuals(ea, ro, lane, lsh, 0, e);
                    }
                    if (stats) ea.moments = mom0 + flip * mom_size + part * 3 * n_chunk + 32 * g;
                    // 16 columns of the row at a time into the patch
#pragma unroll 1
                    for (int h = 0; h < 2 && 16 * h < left; ++h) {
                        float v[16];
                        if (ksplit > 1) {
#pragma unroll
                            for (int j = 0; j < 16; ++j) v[j] = 0.f;
#pragma unroll 1
                            for (int z = 0; z < ksplit; ++z) {
                                float w[16];
                                load16(sk_all + ((size_t)z * T + t) * sk_tile + ((size_t)(2 * g + h) * kTileM + quad * 32 + lane) * 16, w);
#pragma unroll
                                for (int j = 0; j < 16; j += 2) unpair(add2(pair(v[j], v[j + 1]), pair(w[j], w[j + 1])), v[j], v[j + 1]);
                            }
                        } else {
                            accumulator(t, 32 * g + 16 * h, v);
                        }
#pragma unroll
                        for (int j = 0; j < 4; ++j) patch[lane * 8 + ((4 * h + j) ^ (lane & 7))] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                    }
                    __syncwarp();
                    emit_rows<BNB>(ea, ro, fill, lane, lsh, have, e);
                }
                if (rows) have = true;
            }
            // the accumulator is read: the next unit's MMAs may have it
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty + 8 * buf);
            if (alternate) par ^= 1u;                 // (a set of warps always meets its own accumulator set)
            else if (++buf == p.acc_bufs) { buf = 0; par ^= 1u; }
            }
            turn ^= 1;
            if (stats && finish && (ksplit > 1 || u.last_of_block())) {
                // the block's moments: lanes, then the warps' parts, each about its own shift
                float* contrib = mom0 + flip * mom_size;
                float* counts = contrib + (size_t)parts * 3 * n_chunk;
                if (lane == 0 && (whole || half == 0)) counts[part] = (float)count;
                count = 0; have = false;
                if (alternate) part = ew ^ (turn << 2);
                epi_sync();
                if (BNB && tid < n_chunk) {
                    float sum = 0.f, sq = 0.f;
                    const float* c3 = contrib + tid;
#pragma unroll 1
                    for (int w = 0; w < parts; ++w, c3 += 3 * n_chunk)
                        if (counts[w] > 0.f) { sum += c3[n_chunk]; sq += c3[2 * n_chunk]; }
                    float* row = p.st_partials + (size_t)u.m * partial_floats(p.blocks_per_m, C_out) + (size_t)(u.ul / p.unit_block) * 2 * C_out + co0 + tid;
                    if (ok) { row[0] = sum; row[C_out] = sq; }
                } else if (tid < n_chunk) {
                    // parts about their own shifts k_w: sum and squares about the first one's,
                    //   sum (x - k0) = sum_w [d_w + n_w e],  sum (x - k0)^2 = sum_w [q_w + e (2 d_w + n_w e)],  e = k_w - k0
                    float N = 0.f, k0 = 0.f, sum = 0.f, sq = 0.f;
                    const float* c3 = contrib + tid;
#pragma unroll 1
                    for (int w = 0; w < parts; ++w, c3 += 3 * n_chunk) {
                        const float n = counts[w];
                        if (n == 0.f) continue;
                        const float d = c3[n_chunk];
                        if (N == 0.f) k0 = c3[0];
                        const float e = c3[0] - k0;
                        N += n;
                        sum += fmaf(n, e, d);
                        sq += fmaf(e, fmaf(n, e, 2.f * d), c3[2 * n_chunk]);
                    }
                    const float dm = N > 0.f ? sum / N : 0.f, m2 = fmaxf(fmaf(-sum, dm, sq), 0.f);
                    float* dst = p.st_partials + (size_t)u.m * partial_floats(p.blocks_per_m, C_out);
                    const int r = u.ul / p.unit_block;
                    float* row = dst + (size_t)r * 2 * C_out + co0 + tid;
                    if (ok) { row[0] = k0 + dm; row[C_out] = m2; }
                    if (tid == 0 && slice == 0 && ok) dst[(size_t)p.blocks_per_m * 2 * C_out + r] = N;
                }
                flip ^= 1;
            }
        }
    }

    // ---- teardown ----
    tc_fence_before();
    __syncthreads();
    if (abort_flag && threadIdx.x == 0) {
        // copies still in flight must land before the shared memory is given back
        for (int it = a_used; it < a_issued; ++it) {
            const long long t0 = clock64();
            while (!mbar_try_wait(a_raw + 8 * (it % p.a_stages), (uint32_t)(it / p.a_stages) & 1u) && clock64() - t0 < kWaitLimit) {}
        }
        for (int it = b_used; it < b_issued; ++it) {
            const int s = p.b_resident ? 0 : it % p.b_stages;
            const uint32_t parity = p.b_resident ? 0u : (uint32_t)(it / p.b_stages) & 1u;
            const long long t0 = clock64();
            while (!mbar_try_wait(b_full + 8 * s, parity) && clock64() - t0 < kWaitLimit) {}
        }
    }
    __syncthreads();
}

template <bool BN_IN, bool FLAT, bool BNB>
__global__ void __launch_bounds__(kPipeThreads, 1) conv_pipe_kernel(const __grid_constant__ PipeParams gp, const int m_first, const int m_count)
{
    const PipeScalars& p = gp.s;
    {
        // The scalar parameters span several lines of the constant cache: every warp touches one of them, so that the roles do
        // not meet the misses one after the other.  (A warp whose lanes touch different words takes them one at a time.)
        const int at = warp_index() * 16;
        if (at < (int)(sizeof(PipeScalars) / 4)) asm volatile("" ::"r"(reinterpret_cast<const uint32_t*>(&gp.s)[at]));
    }
    extern __shared__ uint8_t smem_raw[];
    __shared__ PipeShared sh;
    uint8_t* smem = smem_raw + (((smem_u32(smem_raw) + 1023u) & ~1023u) - smem_u32(smem_raw));
    if (warp_index() == 3) pipe_init_barriers(p, sh, threadIdx.x & 31);
    if (threadIdx.x == 32) { prefetch_tmap(&gp.tm_a); prefetch_tmap(&gp.tm_b); prefetch_tmap(&gp.tm_b_lo); }
    if (warp_index() == 0) tmem_alloc(smem_u32(&sh.tmem_slot), p.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // The successor may be scheduled from here on: not before this CTA holds its tensor memory, or the successor's CTA could
    // take the columns this one needs and wait for this one to finish.
    if (!p.pdl_late) pdl_launch_dependents();
    const uint32_t tmem_base = sh.tmem_slot;
    pipe_cta<BN_IN, FLAT, BNB, false>(gp, p, sh, smem, tmem_base, m_first, m_count, (int)blockIdx.x, (int)gridDim.x);
    if (warp_index() == 0) tmem_dealloc(tmem_base, p.tmem_cols);
}

// ------------------------------------------------------------------------------------------------
// persistent cells: the forward convolutions of a cell in ONE resident grid
// ------------------------------------------------------------------------------------------------
// A fixed grid stays resident for the whole cell and walks the list of launches: its CTAs take the place of each launch's
// CTAs, run the same code, and meet at a grid-wide barrier before the next launch, whose input the whole grid has just
// produced.  Every CTA must be resident at the same time; the host sizes the grids so that all cells that can run
// concurrently fit the GPU together.  The barrier wait is bounded like every other wait here.
struct CellOp {
    PipeParams p;                // exactly what the stand-alone launch would receive
    int bn_in, flat;             // which kernel it would be
};
struct CellParams {
    const CellOp* ops;           // device memory, written before the launch and read-only for the kernel
    int n_ops;
    unsigned int* barrier;       // {arrivals, generation}: zero before the first use, left with arrivals at zero
    DeviceStatus* status;
    unsigned int tmem_cols;      // the largest accumulators of the list
};

__device__ __forceinline__ unsigned int ld_acquire_gpu(const unsigned int* ptr)
{
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ptr) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_gpu(unsigned int* ptr, unsigned int v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(ptr), "r"(v) : "memory");
}

// All CTAs of the grid arrive; the last one opens the next generation.  What the CTAs wrote before the barrier is visible to
// all of them after it, also to copies issued through the async proxy (TMA).  Returns false when the wait ran out or another
// kernel already reported a failure.
__device__ __forceinline__ bool cell_grid_barrier(unsigned int* bar, DeviceStatus* status, int* stop_flag)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned int gen = ld_acquire_gpu(bar + 1);      // cannot advance before this CTA has arrived
        __threadfence();
        int stop = 0;
        if (atomicAdd(bar, 1u) == gridDim.x - 1) {
            bar[0] = 0u;
            __threadfence();
            st_release_gpu(bar + 1, gen + 1u);
        } else {
            const long long t0 = clock64();
            int polls = 0;
            while (ld_acquire_gpu(bar + 1) == gen) {
                if ((++polls & 63) == 0 && (clock64() - t0 > kWaitLimit || ld_acquire_gpu(&status->code) != 0u)) { report(status, 9); stop = 1; break; }
            }
        }
        *stop_flag = stop;
    }
    __syncthreads();
    asm volatile("fence.proxy.async;" ::: "memory");
    return *stop_flag == 0;
}

__global__ void __launch_bounds__(kPipeThreads, 1) conv_pipe_cell_kernel(const __grid_constant__ CellParams cp, const int m_first, const int m_count)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ PipeShared sh;
    __shared__ PipeScalars p;
    __shared__ int cell_stop;
    constexpr int kWords = (int)(sizeof(PipeScalars) / 4);
    static_assert(sizeof(PipeScalars) % 4 == 0 && kWords <= kPipeThreads, "one parameter word per thread");
    uint8_t* smem = smem_raw + (((smem_u32(smem_raw) + 1023u) & ~1023u) - smem_u32(smem_raw));
    const int tid = threadIdx.x;
    if (warp_index() == 0) tmem_alloc(smem_u32(&sh.tmem_slot), cp.tmem_cols);
    if (tid == 0) { cell_stop = 0; sh.abort_flag = 0; }
    // one word of the parameters per thread: the first launch's now, the next one's while the current one runs
    uint32_t nxt = tid < kWords ? __ldg(reinterpret_cast<const uint32_t*>(&cp.ops[0].p.s) + tid) : 0u;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = sh.tmem_slot;
    bool first = true;
    for (int op = 0; op < cp.n_ops; ++op) {
        if (tid < kWords) reinterpret_cast<uint32_t*>(&p)[tid] = nxt;
        if (op + 1 < cp.n_ops && tid < kWords) nxt = __ldg(reinterpret_cast<const uint32_t*>(&cp.ops[op + 1].p.s) + tid);
        __syncthreads();
        const PipeParams& gp = cp.ops[op].p;
        const int bn_in = __ldg(&cp.ops[op].bn_in), flat = __ldg(&cp.ops[op].flat);
        const int tasks = m_count * p.blocks_per_m * p.ksplit;
        int per_slice = (int)gridDim.x / p.slices;
        if (per_slice < 1) per_slice = 1;
        if (per_slice > tasks) per_slice = tasks;
        const int V = per_slice * p.slices;
        for (int v = blockIdx.x; v < V; v += gridDim.x) {
            // the barriers of the call before have seen their last arrival: they start over
            if (tid < 32) {
                if (!first)
                    for (int i = tid; i < 3 * kMaxA + 2 * kMaxB + 4; i += 32) mbar_inval(smem_u32(&sh.bars[i]));
                __syncwarp();
                pipe_init_barriers(p, sh, tid);
            }
            first = false;
            __syncthreads();
            tc_fence_after();
            if (bn_in) {
                if (flat) pipe_cta<true, true, false, true>(gp, p, sh, smem, tmem_base, m_first, m_count, v, V);
                else pipe_cta<true, false, false, true>(gp, p, sh, smem, tmem_base, m_first, m_count, v, V);
            } else {
                if (flat) pipe_cta<false, true, false, true>(gp, p, sh, smem, tmem_base, m_first, m_count, v, V);
                else pipe_cta<false, false, false, true>(gp, p, sh, smem, tmem_base, m_first, m_count, v, V);
            }
            if (sh.abort_flag) { if (tid == 0) cell_stop = 1; break; }
        }
        if (sh.abort_flag || (op + 1 < cp.n_ops && !cell_grid_barrier(cp.barrier, cp.status, &cell_stop))) break;
    }
    tc_fence_before();
    __syncthreads();
    if (warp_index() == 0) tmem_dealloc(tmem_base, cp.tmem_cols);
}

// Statistics for a BN that runs a kernel of its own although its input came from a convolution that left moments (the formulas
// of merge_moments).  A block takes 128 channels with eight row lanes, grid (channels / 128, micro-batches): latency bound, so the
// rows are spread (one block per micro-batch took 16 us at 1024 channels).
__global__ void __launch_bounds__(256) bn_finalize_kernel(const float* __restrict__ partials, int rows, int C, double inv_rows, float eps, float* stats)
{
    __shared__ float4 red[3][8][32];
    __shared__ float4 refs[32];
    pdl_launch_dependents();
    pdl_wait();
    const int t = threadIdx.x, lane = t & 31, ln = t >> 5, c4n = C >> 2, col = blockIdx.x * 32 + lane;
    partials += (size_t)blockIdx.y * partial_floats(rows, C); stats += (size_t)blockIdx.y * 2 * C;
    const float* counts = partials + (size_t)rows * 2 * C;
    float4 sd = make_float4(0.f, 0.f, 0.f, 0.f), sq = sd, m2 = sd, ref = sd;
    if (col < c4n) {
        ref = __ldcg(reinterpret_cast<const float4*>(partials) + col);
#pragma unroll 4
        for (int k = ln; k < rows; k += 8) {
            const float4* row = reinterpret_cast<const float4*>(partials + (size_t)k * 2 * C);
            const float n = __ldcg(counts + k);
            const float4 d = sub4(__ldcg(row + col), ref), nd = mul4(make_float4(n, n, n, n), d);
            sd = add4(sd, nd);
            sq = fma4(nd, d, sq);
            m2 = add4(m2, __ldcg(row + c4n + col));
        }
    }
    red[0][ln][lane] = sd; red[1][ln][lane] = sq; red[2][ln][lane] = m2;
    if (ln == 0) refs[lane] = ref;
    __syncthreads();
    const int c = blockIdx.x * 128 + t;
    if (t >= 128 || c >= C) return;
    const float* r = reinterpret_cast<const float*>(&red[0][0][0]) + t;
    float d = 0.f, q = 0.f, v = 0.f;
#pragma unroll
    for (int l = 0; l < 8; ++l) { d += r[128 * l]; q += r[128 * (8 + l)]; v += r[128 * (16 + l)]; }
    const double dm = (double)d * inv_rows;
    double var = ((double)v + (double)q) * inv_rows - dm * dm;
    if (var < 0.0) var = 0.0;
    stats[c] = (float)((double)reinterpret_cast<const float*>(refs)[t] + dm);
    stats[C + c] = 1.0f / sqrtf((float)(var + (double)eps));
}

// Forward pass, or the data gradient seen as a forward problem.
struct PipeView {
    int P, Q;                    // output grid of the GEMM
    int c_in, c_out;
    int in_W, in_H;              // input pixels the positions may touch
    int in_sw, in_sh, in_sn, os_w, os_h, os_n, zero_fill, out_h, out_w, dense_h, dense_w;
    long long in_ms, out_ms;
};

bool pipe_view(const ConvShape& s, int pass, PipeView* v)
{
    if (s.C % 16 || s.K % 16) return false;
    if (s.R == 3 ? (s.stride != 1 || s.pad != 1) : (s.R != 1 || s.pad != 0)) return false;
    if (s.stride < 1 || s.stride > 2) return false;
    const long long x = (long long)s.N * s.H * s.W * s.C, y = (long long)s.N * s.P * s.Q * s.K;
    if (x >= (1LL << 31) || y >= (1LL << 31)) return false;        // 32-bit offsets inside a micro-batch
    if (pass == PASS_FWD) {
        v->P = s.P; v->Q = s.Q; v->c_in = s.C; v->c_out = s.K;
        v->in_W = s.Q; v->in_H = s.P;                              // in steps of the stride
        v->in_sw = s.stride * s.C; v->in_sh = s.stride * s.W * s.C; v->in_sn = s.H * s.W * s.C;
        v->os_w = s.K; v->os_h = s.Q * s.K; v->os_n = s.P * s.Q * s.K;
        v->zero_fill = 1; v->out_h = s.P; v->out_w = s.Q; v->dense_h = v->os_h; v->dense_w = v->os_w;
        v->in_ms = x; v->out_ms = y;
    } else {
        v->P = s.P; v->Q = s.Q; v->c_in = s.K; v->c_out = s.C;
        v->in_W = s.Q; v->in_H = s.P;
        v->in_sw = s.K; v->in_sh = s.Q * s.K; v->in_sn = s.P * s.Q * s.K;
        v->dense_w = s.C; v->dense_h = s.W * s.C;
        v->os_w = s.stride * s.C; v->os_h = s.stride * s.W * s.C; v->os_n = s.H * s.W * s.C;
        v->zero_fill = s.stride; v->out_h = s.H; v->out_w = s.W;
        v->in_ms = y; v->out_ms = x;
    }
    return true;
}

int sm_count()
{
    static PerDevice<int> sms;
    int n = 0;
    const cudaError_t e = sms.get(&n, [](int dev, int* v) { return cudaDeviceGetAttribute(v, cudaDevAttrMultiProcessorCount, dev); });
    if (e != cudaSuccess) { (void)cudaGetLastError(); return 148; }
    return n;
}

constexpr int kPlanSms = 148;                         // the split of the work is planned for a whole B200, with or without a device at hand
inline unsigned int stat_bytes(int n_chunk) { return (unsigned int)(2 * (n_chunk <= 64 ? 8 : 4) * (3 * n_chunk + 1) * 4 + 127) & ~127u; }
inline int split_groups_of(int a_stages) { return a_stages % 4 == 0 ? 4 : (a_stages % 2 == 0 ? 2 : 1); }
inline unsigned int bn_bytes(int c_in) { return (unsigned int)(4 * c_in * 4 + 4 * kSplitThreads * 16); }

}  // namespace

size_t conv_pipe_partial_floats(int units_per_m, int channels) { return partial_floats(units_per_m, channels); }

static bool plan_geom(const ConvShape& s, int pass, int passes, int launched, ConvPipeGeom* g)
{
    PipeView v;
    if (pass == PASS_WGRAD || !pipe_view(s, pass, &v)) return false;
    const bool three = passes == 3;
    // Channel slices of 128 beyond 128 channels: a unit of 256 positions x 128 channels reads half as many weight bytes from
    // L2 per MMA as 128 positions x 256 channels do.
    g->n_chunk = v.c_out <= 128 ? v.c_out : (v.c_out % 128 == 0 ? 128 : (v.c_out <= 256 ? v.c_out : 0));
    if (!g->n_chunk) return false;
    g->slices = v.c_out / g->n_chunk;
    g->strips = 1; g->col0 = 0; g->strip_w = v.Q; g->halo = 0; g->Wp = v.Q; g->Hp = v.P;
    if (s.R == 3) {
        g->Wp = v.Q + 1; g->Hp = v.P + 1;
        if (v.Q > 254) {
            g->strips = (v.Q + 251) / 252;
            g->strip_w = (v.Q + g->strips - 1) / g->strips;
            g->Wp = g->strip_w + 2; g->col0 = 1;
        }
        g->halo = g->Wp + 1;
    }
    g->flat = s.R == 1 && (s.stride == 1 || pass == PASS_DGRAD) ? 1 : 0;
    if (!g->flat && g->Wp > 256) return false;
    // one copy per padded map row, or per whole map where that is no more than 40 positions
    g->box_h = g->Wp * g->Hp <= 40 ? g->Hp : 1;
    const int bp = g->flat ? kTileM : g->box_h * g->Wp;
    const long long pos = (long long)s.N * g->strips * g->Wp * g->Hp;
    if (pos >= (1LL << 30)) return false;
    g->pos_per_m = (int)pos;
    g->tiles_per_m = (g->pos_per_m + kTileM - 1) / kTileM;
    const int taps = s.R * s.R, chunks = v.c_in / 16, n = g->n_chunk;
    g->b_tap_bytes = (unsigned int)(three ? 2 : 1) * (unsigned int)n * 64u;
    const unsigned int all_b = g->b_tap_bytes * (unsigned int)(taps * chunks);
    // (the data gradient applies no BN)
    const unsigned int fixed = kEpiWarps * 4096u + stat_bytes(n) + (pass == PASS_FWD ? bn_bytes(v.c_in <= 512 ? v.c_in : 0) : 0u);
    // Tiles per unit, stacked weights (hi*hi and hi*lo from one MMA over [B_hi; B_lo]), accumulator sets and the two rings:
    // the combination with the least modelled time for the busiest CTA, from clocks measured stage by stage.  A chunk takes
    // the longest of: its MMAs (K = 8; at 128 columns an unstacked MMA reads 128 bytes of shared memory per clock, all there
    // is, and pays for every other access) and the waits between them; an operand stage's life (copy, split, MMAs) over the
    // stages of the ring - with two stages of 32 KB a 1x1 convolution waited for that, 1640 clocks a chunk against 870 of
    // MMAs; the same for the weights; the bytes at 20 (operand, mostly from HBM) and 28 (weights, L2) per clock and SM.
    auto clk = [](int c) { return c <= 32 ? 40.0 : (c <= 64 ? 48.0 : (c <= 96 ? 58.0 : (c <= 128 ? 68.0 : 0.5 * c))); };
    double best = 0.0;
    g->T = 0;
    for (int T = 4; T >= 1; T >>= 1)
        for (int stacked = three && 2 * n <= 256 ? 1 : 0; stacked >= 0; --stacked)
            for (int bufs = 2; bufs >= 1; --bufs) {
                const int cols = stacked ? 2 * n : n;
                if (bufs * T * cols > 512) continue;
                const int need = T * kTileM + 2 * g->halo, rows = g->flat ? need : need + 2 * bp - 2;
                const int nj = (rows + kRowStep * kRowBatch - 1) / (kRowStep * kRowBatch) * kRowBatch;
                if (nj * kRowStep > kMaxBlockRows) continue;
                const unsigned int a_stage = (unsigned int)(nj * kRowStep) * 128u;
                const int units = (g->tiles_per_m + T - 1) / T;
                const int per_slice = kPlanSms / g->slices > 0 ? kPlanSms / g->slices : 1;
                const double rounds = (double)(((long long)launched * units + per_slice - 1) / per_slice);
                const double step = !three ? clk(n) : (stacked ? clk(2 * n) + clk(n) : 3.0 * (n == 128 ? 80.0 : clk(n)));
                const double tap_mma = 2.0 * T * step, epi = 1100.0 * T * ((n + 31) / 32) / 2.0;
                // weights: resident, or a ring whose stage holds the taps of a window row (fewer waits) or one tap
                for (int bt = s.R; bt >= 0; bt = bt == 3 ? 1 : bt - 1) {
                    const bool resident = bt == 0;
                    if (resident && all_b > 100u * 1024u) continue;
                    const unsigned int b_stage = resident ? all_b : (unsigned int)bt * g->b_tap_bytes;
                    for (int bs = resident ? 1 : 2; bs <= (resident ? 1 : kMaxB); ++bs) {
                        const unsigned int b_all = (unsigned int)bs * b_stage;
                        if (b_all + fixed + 2 * a_stage > kPipeSmem) break;
                        int as = (int)((kPipeSmem - fixed - b_all) / a_stage);
                        if (as > kMaxA) as = kMaxA;
                        const double mma = resident ? taps * tap_mma + 100.0
                                                    : (double)(taps / bt) * std::max({bt * tap_mma + 100.0, (1000.0 + b_stage / 40.0 + bt * tap_mma) / bs, b_stage / 28.0});
                        // (of the rings that serve the same number of groups the deepest is the best)
                        for (int tried = 0; as >= 2 && tried != 7; --as) {
                        const int groups = split_groups_of(as);
                        if (tried & groups) continue;
                        tried |= groups;
                        const double split = three ? 250.0 + 5.6 * rows * groups / 4.0 : 100.0;
                        const double chunk = std::max({mma, (1200.0 + rows * 1.6 + split + mma) / as, split / groups, rows * 64.0 / 20.0});
                        const double k_loop = chunk * chunks, body = bufs == 2 ? std::max(k_loop, epi) : k_loop + epi;
                        const double cost = rounds * body + chunk + 1000.0 + epi;
                        if (g->T == 0 || cost < best * 0.999) {
                            best = cost;
                            g->T = T; g->units_per_m = units; g->a_rows = nj * kRowStep; g->a_stage_bytes = a_stage; g->a_stages = as;
                            g->b_resident = resident ? 1 : 0; g->b_taps = resident ? taps : bt; g->b_stages = resident ? taps * chunks : bs;
                            g->b_stage_bytes = resident ? g->b_tap_bytes : b_stage;
                            g->stacked = stacked; g->acc_cols = (unsigned int)cols; g->acc_bufs = bufs;
                        }
                        }
                    }
                }
            }
    if (!g->T) return false;
    // Few units with a long K loop: several CTAs share it (partial tiles in L2, added in order by the last to finish).
    g->ksplit = 1;
    const int tasks = launched * g->units_per_m * g->slices, ksteps = 2 * taps * chunks;
    if (2 * tasks <= kPlanSms && ksteps >= 128) {
        int S = kPlanSms / tasks;
        if (S > 8) S = 8;
        if (S > ksteps / 32) S = ksteps / 32;
        if (S > chunks) S = chunks;
        if (S > 1) g->ksplit = S;
    }
    // Blocks of units: the reader of the BN moments merges one row per block, so as few as leave the busiest CTA with at most
    // a tenth more work.
    g->unit_block = 1;
    if (g->ksplit == 1) {
        const int per_slice = kPlanSms / g->slices > 0 ? kPlanSms / g->slices : 1;
        const int most = (launched * g->units_per_m + per_slice - 1) / per_slice;
        for (int u = 2; u <= 16 && u <= most; ++u) {
            const int blocks = launched * ((g->units_per_m + u - 1) / u);
            if (10 * u * ((blocks + per_slice - 1) / per_slice) <= 11 * most) g->unit_block = u;
        }
    }
    g->blocks_per_m = (g->units_per_m + g->unit_block - 1) / g->unit_block;
    return true;
}

// The search takes several microseconds and a single convolution's call asks for its plan and its scratch sizes: as long as the
// convolution itself for a small one (1x1 on 4 x 4 maps, forward and both gradients: 64 us, 32 with the last plans kept).
// Each thread keeps a fixed number of them.
bool conv_pipe_geom(const ConvShape& s, int pass, int passes, int launched, ConvPipeGeom* g)
{
    struct Kept { int key[11]; bool used, ok; ConvPipeGeom g; };
    constexpr int kKept = 64;
    static thread_local Kept kept[kKept];
    const int key[11] = {s.N, s.H, s.W, s.C, s.K, s.R, s.stride, s.pad, pass, passes, launched};
    unsigned int h = 2166136261u;
    for (int k : key) h = (h ^ (unsigned int)k) * 16777619u;
    Kept& e = kept[(h >> 16) % kKept];
    if (!e.used || memcmp(e.key, key, sizeof key) != 0) {
        memcpy(e.key, key, sizeof key);
        e.ok = plan_geom(s, pass, passes, launched, &e.g);
        e.used = true;
    }
    *g = e.g;
    return e.ok;
}

bool conv_pipe_can_fuse_bn_output(const ConvPipeGeom& g) { return g.n_chunk <= 128; }      // a warp keeps the moments of two groups of 32 channels
bool conv_pipe_can_fuse_bn_input(const ConvShape& s) { return s.stride == 1 && s.C % 16 == 0 && s.C <= 512 && s.W <= 254; }      // (no column strips)

size_t conv_pipe_splitk_bytes(const ConvPipeGeom& g)
{
    if (g.ksplit < 2) return 0;
    return (kSplitKTicketBytes + (size_t)g.units_per_m * g.slices * g.ksplit * g.T * kTileM * g.n_chunk * sizeof(float) + 255) & ~(size_t)255;
}
size_t conv_pipe_splitk_bytes(const ConvShape& s, int pass, int passes, int launched)
{
    ConvPipeGeom g;
    return conv_pipe_geom(s, pass, passes, launched, &g) ? conv_pipe_splitk_bytes(g) : 0;
}

struct ConvPipeLaunch { PipeParams p; unsigned int smem; int bn_in; };
static_assert(sizeof(ConvPipeLaunch) <= sizeof(((ConvPipePlan*)0)->storage), "plan storage too small");

cudaError_t conv_pipe_init()
{
    static PerDevice<bool> attributes;
    bool set = false;
    return attributes.get(&set, [](int, bool* done) {
        cudaError_t e = cudaSuccess;
        for (auto kernel : {conv_pipe_kernel<false, false, false>, conv_pipe_kernel<false, true, false>, conv_pipe_kernel<true, false, false>, conv_pipe_kernel<true, true, false>,
                            conv_pipe_kernel<false, false, true>, conv_pipe_kernel<false, true, true>})
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPipeSmem + 1024);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(conv_pipe_cell_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPipeSmem + 1024);
        *done = true;
        return e;
    });
}

namespace {
cudaError_t encode_map(CUtensorMap* tm, const float* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides, const cuuint32_t* box,
                       CUtensorMapSwizzle swizzle)
{
    if (!g_encode) return cudaErrorNotReady;
    const cuuint32_t ones[4] = {1, 1, 1, 1};
    const CUresult r = g_encode(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, (cuuint32_t)rank, const_cast<float*>(base), dims, strides, box, ones,
                                CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}
cudaError_t encode_weights(CUtensorMap* tm, const float* base, long long kdim, int c_out, int n_chunk)
{
    const cuuint64_t dims[2] = {(cuuint64_t)kdim, (cuuint64_t)c_out}, strides[1] = {(cuuint64_t)kdim * 4};
    const cuuint32_t box[2] = {16, (cuuint32_t)n_chunk};
    return encode_map(tm, base, 2, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_64B);
}
unsigned int columns_pow2(unsigned int need)
{
    unsigned int c = 32;
    while (c < need) c <<= 1;
    return c;
}
}  // namespace

cudaError_t conv_pipe_prepare(ConvPipePlan* plan, const ConvShape& s, int pass, int passes, int M, int launched, const float* in, const float* w_hi,
                              const float* w_lo, float* out, const float* extra, bool accumulate, const ConvPipeBn* bn, void* splitk,
                              size_t splitk_bytes, bool w_ready)
{
    plan->valid = 0;
    ConvPipeGeom g;
    PipeView v;
    if ((passes != 1 && passes != 3) || !conv_pipe_geom(s, pass, passes, launched, &g) || !pipe_view(s, pass, &v)) return cudaErrorNotSupported;
    ConvPipeLaunch* L = reinterpret_cast<ConvPipeLaunch*>(plan->storage);
    memset(L, 0, sizeof *L);
    const long long kdim = (long long)s.R * s.R * v.c_in;
    cudaError_t e = encode_weights(&L->p.tm_b, w_hi, kdim, v.c_out, g.n_chunk);
    if (e == cudaSuccess) e = encode_weights(&L->p.tm_b_lo, passes == 3 ? w_lo : w_hi, kdim, v.c_out, g.n_chunk);
    if (e != cudaSuccess) return e;
    PipeScalars& p = L->p.s;
    p.in = in; p.out = out; p.extra = extra; p.in_ms = v.in_ms; p.out_ms = v.out_ms;
    p.accumulate = accumulate ? 1 : 0;
    p.units_per_m = g.units_per_m; p.unit_block = g.unit_block; p.blocks_per_m = g.blocks_per_m; p.tiles_per_m = g.tiles_per_m; p.T = g.T; p.slices = g.slices; p.n_chunk = g.n_chunk; p.ksplit = g.ksplit;
    p.R = s.R; p.taps = s.R * s.R; p.n_chunks = v.c_in / 16; p.c_in = v.c_in; p.c_out = v.c_out;
    p.pos_per_m = g.pos_per_m; p.Wp = g.Wp; p.img_pos = g.Wp * g.Hp; p.Hv = v.P; p.W = v.Q; p.halo = g.halo;
    p.strips = g.strips; p.strip_w = g.strip_w; p.col0 = g.col0;
    p.magic_w = magic_of(g.Wp); p.magic_img = magic_of(p.img_pos); p.magic_strip = magic_of(g.strips);
    p.in_sw = v.in_sw; p.in_sh = v.in_sh; p.in_sn = v.in_sn; p.os_w = v.os_w; p.os_h = v.os_h; p.os_n = v.os_n;
    p.zero_fill = v.zero_fill; p.out_h = v.out_h; p.out_w = v.out_w; p.dense_h = v.dense_h; p.dense_w = v.dense_w;
    p.flat = g.flat; p.box_h = g.box_h; p.box_pos = g.box_h * g.Wp; p.blocks_per_img = g.Hp / g.box_h;
    p.magic_box = magic_of(p.box_pos); p.magic_bpi = magic_of(p.blocks_per_img);
    p.pix_ms = g.flat ? (long long)s.N * v.P * v.Q : s.N;
    if ((long long)M * p.pix_ms >= (1LL << 31)) return cudaErrorNotSupported;
    {
        CUtensorMap* tm = &L->p.tm_a;
        const cuuint64_t fd[2] = {(cuuint64_t)v.c_in, (cuuint64_t)(M * p.pix_ms)}, fs[1] = {(cuuint64_t)v.c_in * 4};
        const cuuint32_t fb[2] = {16, kTileM};
        const cuuint64_t rd[4] = {(cuuint64_t)v.c_in, (cuuint64_t)v.in_W, (cuuint64_t)v.in_H, (cuuint64_t)M * s.N};
        const cuuint64_t rs[3] = {(cuuint64_t)v.in_sw * 4, (cuuint64_t)v.in_sh * 4, (cuuint64_t)v.in_sn * 4};
        const cuuint32_t rb[4] = {16, (cuuint32_t)g.Wp, (cuuint32_t)g.box_h, 1};
        e = g.flat ? encode_map(tm, in, 2, fd, fs, fb, CU_TENSOR_MAP_SWIZZLE_128B) : encode_map(tm, in, 4, rd, rs, rb, CU_TENSOR_MAP_SWIZZLE_128B);
        if (e != cudaSuccess) return e;
    }
    p.a_stages = g.a_stages; p.b_stages = g.b_stages; p.b_taps = g.b_taps; p.b_resident = g.b_resident; p.acc_bufs = g.acc_bufs;
    p.a_stage_bytes = g.a_stage_bytes; p.b_stage_bytes = g.b_stage_bytes; p.b_tap_bytes = g.b_tap_bytes; p.acc_cols = g.acc_cols;
    p.tmem_cols = columns_pow2((unsigned int)(g.acc_bufs * g.T) * g.acc_cols);
    p.idesc = instr_desc(g.n_chunk, false, false);
    p.idesc2 = instr_desc(g.stacked ? 2 * g.n_chunk : g.n_chunk, false, false);
    p.split_groups = split_groups_of(g.a_stages);
    p.epi_alternate = g.acc_bufs == 2 && g.n_chunk <= 64 && g.ksplit == 1 ? 1 : 0;
    p.three = passes == 3 ? 1 : 0; p.stacked = g.stacked; p.w_ready = w_ready ? 1 : 0;
    const unsigned int a_bytes = (unsigned int)g.a_stages * g.a_stage_bytes;
    p.off_b = a_bytes;
    p.off_stage = (p.off_b + (unsigned int)g.b_stages * g.b_stage_bytes + 127u) & ~127u;
    p.off_stat = p.off_stage + kEpiWarps * 4096u;
    p.off_red = p.off_stat + stat_bytes(g.n_chunk);
    p.off_bn = p.off_red + 4 * kSplitThreads * 16;
    L->smem = p.off_red + 1024;
    if (bn && bn->out_partials) {
        if (!conv_pipe_can_fuse_bn_output(g)) return cudaErrorNotSupported;
        p.st_partials = bn->out_partials;
    }
    if (bn && bn->bwd_partials) {
        if (pass != PASS_DGRAD || s.stride != 1 || extra || accumulate || !conv_pipe_can_fuse_bn_output(g)) return cudaErrorNotSupported;
        p.st_partials = bn->bwd_partials; p.bn_x = bn->bwd_x; p.bn_stats = const_cast<float*>(bn->bwd_stats);
        p.bn_gamma = bn->in_gamma; p.bn_beta = bn->in_beta;
    }
    if (bn && bn->in_partials) {
        if (pass != PASS_FWD || !conv_pipe_can_fuse_bn_input(s) || bn->in_blocks < 1) return cudaErrorNotSupported;
        p.bn_partials = bn->in_partials; p.bn_units = bn->in_blocks; p.bn_gamma = bn->in_gamma; p.bn_beta = bn->in_beta;
        p.bn_stats = bn->in_stats; p.bn_y = bn->in_y; p.bn_eps = bn->in_eps;
        p.bn_inv_rows = 1.0 / ((double)s.N * s.H * s.W);
        L->smem = p.off_bn + 4u * (unsigned int)v.c_in * 4u + 1024;
        L->bn_in = 1;
    }
    if (g.ksplit > 1) {
        if (!splitk || conv_pipe_splitk_bytes(g) > splitk_bytes) return cudaErrorInvalidValue;
        p.sk_base = reinterpret_cast<char*>(splitk); p.sk_ms = (long long)splitk_bytes;
    }
    if (L->smem > kPipeSmem + 1024) return cudaErrorNotSupported;
    plan->valid = 1;
    return cudaSuccess;
}

cudaError_t conv_pipe_launch(const ConvPipePlan* plan, int m_first, int m_count, bool pdl_late, DeviceStatus* status, cudaStream_t st, int64_t* n_launch)
{
    if (!plan->valid || m_count < 1) return cudaErrorInvalidValue;
    ConvPipeLaunch L = *reinterpret_cast<const ConvPipeLaunch*>(plan->storage);
    L.p.s.status = status;
    // (a launch that waits for its weights lets its successor start only after that wait: the successor may not wait for them)
    L.p.s.pdl_late = pdl_late || !L.p.s.w_ready ? 1 : 0;
    const PipeScalars& p = L.p.s;
    const int tasks = m_count * p.blocks_per_m * p.ksplit;
    int per_slice = sm_count() / p.slices;
    if (per_slice < 1) per_slice = 1;
    if (per_slice > tasks) per_slice = tasks;
    const bool flat = p.flat && p.zero_fill == 1;
    auto kernel = L.bn_in ? (flat ? conv_pipe_kernel<true, true, false> : conv_pipe_kernel<true, false, false>)
                          : (p.bn_x ? (flat ? conv_pipe_kernel<false, true, true> : conv_pipe_kernel<false, false, true>)
                                    : (flat ? conv_pipe_kernel<false, true, false> : conv_pipe_kernel<false, false, false>));
    // What a CTA has to do decides how its warps share it (the sums are the same either way).  A block of the operand takes one
    // splitter warp about 2000 clocks and all four of them 850, so with one or two blocks in all they share each; with a single unit
    // both halves of the write-out's warps take it.
    const int units = (tasks + per_slice - 1) / per_slice * p.unit_block, blocks = units * ((p.n_chunks + p.ksplit - 1) / p.ksplit);
    if (blocks < 4) L.p.s.split_groups = blocks < 2 || p.split_groups == 1 ? 1 : 2;
    if (units == 1 && p.n_chunk > 32) L.p.s.epi_alternate = 0;      // (each half a group of columns: the partial sums of the moments stay the same)
    launch_pdl(kernel, dim3(per_slice * p.slices), dim3(kPipeThreads), L.smem, st, L.p, m_first, m_count);
    if (n_launch) ++*n_launch;
    return cudaGetLastError();
}

size_t conv_pipe_cell_op_bytes() { return sizeof(CellOp); }

void conv_pipe_cell_op(const ConvPipePlan* plan, DeviceStatus* status, void* dst_host, unsigned int* smem, unsigned int* tmem_cols)
{
    const ConvPipeLaunch* L = reinterpret_cast<const ConvPipeLaunch*>(plan->storage);
    CellOp op;
    memset(&op, 0, sizeof op);
    op.p = L->p;
    op.p.s.status = status;
    op.bn_in = L->bn_in; op.flat = L->p.s.flat && L->p.s.zero_fill == 1;
    memcpy(dst_host, &op, sizeof op);
    *smem = L->smem; *tmem_cols = L->p.s.tmem_cols;
}

int conv_pipe_cell_max_ctas() { return sm_count(); }

cudaError_t conv_pipe_cell_launch(const void* d_ops, int n_ops, int m_first, int m_count, int ctas, unsigned int smem, unsigned int tmem_cols,
                                  unsigned int* d_barrier, DeviceStatus* status, cudaStream_t st, int64_t* n_launch)
{
    if (n_ops < 1 || ctas < 1 || m_count < 1 || tmem_cols < 32 || tmem_cols > 512) return cudaErrorInvalidValue;
    CellParams cp;
    cp.ops = reinterpret_cast<const CellOp*>(d_ops); cp.n_ops = n_ops; cp.barrier = d_barrier; cp.status = status; cp.tmem_cols = tmem_cols;
    // Over half of an SM's shared memory in any case: two cells' CTAs never share an SM, where one could wait for tensor
    // memory that the other holds while it waits for that one's grid.
    if (smem < 120u * 1024u) smem = 120u * 1024u;
    // a plain stream-ordered launch: a resident grid that started early would only hold SM slots while it waits
    conv_pipe_cell_kernel<<<dim3(ctas), dim3(kPipeThreads), smem, st>>>(cp, m_first, m_count);
    if (n_launch) ++*n_launch;
    return cudaGetLastError();
}

cudaError_t bn_finalize_partials(const float* partials, int units, int C, float eps, double rows, float* stats, int m_count, cudaStream_t st,
                                 int64_t* n_launch)
{
    launch_pdl(bn_finalize_kernel, dim3((C + 127) / 128, m_count), dim3(256), 0, st, partials, units, C, 1.0 / rows, eps, stats);
    if (n_launch) ++*n_launch;
    return cudaGetLastError();
}

}  // namespace hpf
