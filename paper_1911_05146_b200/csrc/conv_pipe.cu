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
// Roles (16 warps): warp 0 copies the operand (a 1x1 window's without a stride: warps 0 and 3, 16 bytes a lane), warp 1 the
// weights (TMA; kept in shared memory for the whole launch when they fit), warp 2 issues the MMAs, warps 4-7 rewrite the operand
// in place (BN+ReLU, lo part), warps 8-15 read finished accumulators from tensor memory, add the residual, store and form
// the BN moments.
//
// Measured alone, batch 128, three passes (graph of ten launches), before and since the write-out reads rows (write_out), the MMAs are
// issued in straight lines (mma_role) and the operand of a 1x1 window is copied by lanes: 3x3 16->16 @32 19.8 -> 15.5 us,
// 64->64 @8 15.1 -> 11.6; 1x1 64->16 @32 21.8 -> 13.7, 16->64 @32 17.8 -> 14.3; batch 64: 3x3 64->64 @56 90 -> 74, 256->256 @14 82 -> 73;
// 1x1 64->256 @56 70 -> 71, 256->64 @56 86 -> 69, 512->128 @28 54 -> 43, 1024->256 @14 56 -> 41.
#include "conv_pipe.h"
#include "tc_ptx.cuh"

#include <algorithm>
#include <math.h>
#include <string.h>
#include <type_traits>

namespace hpf {

namespace {

constexpr int kSplitWarps = 4, kEpiWarps = 8;
constexpr int kFirstSplit = 4;                        // warps 0..2: operand copies, weight copies, MMAs; 3: barriers, half of a 1x1 operand's copies
constexpr int kSplitThreads = 32 * kSplitWarps, kRowStep = 8 * kSplitWarps;
constexpr int kPipeThreads = 32 * (kFirstSplit + kSplitWarps + kEpiWarps);
constexpr int kMaxBlockRows = 768, kRowBatch = 2;     // operand rows of a block at most; rows a splitter thread has in flight (code counts: 1 / 2 / 4 / 8: ResNet-110 5.47 / 5.44 / 5.46 / 5.59 ms)
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
    uint32_t magic_w, magic_img, magic_strip, magic_blocks, magic_ksplit;
    int in_sw, in_sh, in_sn, os_w, os_h, os_n;
    int zero_fill, out_h, out_w, dense_h, dense_w;
    int a_stages, b_stages, b_taps, b_resident, acc_bufs, split_groups, epi_alternate;
    // how the operand is copied: flat (128 consecutive pixels per box) or blocks of box_h padded rows of one map
    int flat, box_h, box_pos, blocks_per_img;
    uint32_t magic_box, magic_bpi;
    long long pix_ms;                                 // flat: pixels per micro-batch; else maps per micro-batch
    uint32_t a_stage_bytes, b_stage_bytes, b_tap_bytes, acc_cols, tmem_cols, idesc, idesc2;
    uint32_t off_b, off_bn, off_red, off_stat, off_slots, off_ring, off_bnb, slot_bytes;
    int wide;                                         // a write-out lane has 8 channels of a row (else 4)
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
    int st_plain;                                     // of a plain BN's input: added up in fp64, with the lower parts of the means
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

// W = 4 or 8 consecutive floats of one thread (16 or 32 bytes, aligned).  Reads are ordered ones: the preceding kernel may have
// written what they fetch.
template <int W>
__device__ __forceinline__ void store_vec(float* d, const float* v)
{
    if constexpr (W == 8)
        asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(d), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]),
                     "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]) : "memory");
    else *reinterpret_cast<float4*>(d) = make_float4(v[0], v[1], v[2], v[3]);
}
template <int W>
__device__ __forceinline__ void load_vec(const float* s, float* v)
{
#pragma unroll
    for (int j = 0; j < W; j += 4) {
        const float4 t = __ldcg(reinterpret_cast<const float4*>(s + j));
        v[j] = t.x; v[j + 1] = t.y; v[j + 2] = t.z; v[j + 3] = t.w;
    }
}
// the same in shared memory
template <int W>
__device__ __forceinline__ void read_vec(const float* s, float* v)
{
#pragma unroll
    for (int j = 0; j < W; j += 4) {
        const float4 t = *reinterpret_cast<const float4*>(s + j);
        v[j] = t.x; v[j + 1] = t.y; v[j + 2] = t.z; v[j + 3] = t.w;
    }
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const float* src) { asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory"); }
__device__ __forceinline__ void cp_async16_zfill(uint32_t dst, const float* src, bool real)
{
    asm volatile("cp.async.cg.shared.global.L2::256B [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(real ? 16 : 0) : "memory");
}
// arrives (once a lane) when this lane's copies so far have landed
__device__ __forceinline__ void cp_async_arrive(uint32_t bar) { asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory"); }
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int LEFT>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory"); }
__device__ __forceinline__ void split_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kSplitThreads) : "memory"); }
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 2, 256;" ::: "memory"); }

// partial moments of a micro-batch: rows of [2][C], a count a row, and what rounding takes off the rows' means ([C] a row)
__host__ __device__ inline size_t partial_lo(int units, int C) { return (size_t)units * 2 * C + (size_t)((units + 3) & ~3); }
__host__ __device__ inline size_t partial_floats(int units, int C) { return partial_lo(units, C) + (size_t)units * C; }

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
// acc[0..W) op= ..., two at a time
template <int W>
__device__ __forceinline__ void add_to(float* acc, const float* v)
{
#pragma unroll
    for (int j = 0; j < W; j += 2) unpair(add2(pair(acc[j], acc[j + 1]), pair(v[j], v[j + 1])), acc[j], acc[j + 1]);
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
    constexpr int kRows = 4;                          // rows in flight (six: no faster)
#pragma unroll 1
    for (int c0 = 0; c0 < c4n; c0 += THREADS) {
        const int width = c4n - c0 < THREADS ? c4n - c0 : THREADS;       // float4 columns of this pass
        const int ln = L > 1 ? tid / c4n : 0, local = L > 1 ? tid - ln * c4n : tid, col = c0 + local;
        const bool mine = local < width && ln < L;
        float4 sd = make_float4(0.f, 0.f, 0.f, 0.f), sq = sd, m2 = sd, ref = sd;
        if (mine) {
            ref = __ldcg(reinterpret_cast<const float4*>(partials) + col);
#pragma unroll 1
            for (int k0 = ln; k0 < rows; k0 += kRows * L) {
                float4 a[kRows], b[kRows];
                float n[kRows];
#pragma unroll
                for (int j = 0; j < kRows; ++j) {
                    const int k = k0 + j * L;
                    const bool have = k < rows;
                    const float4* row = reinterpret_cast<const float4*>(partials + (size_t)(have ? k : 0) * 2 * C);
                    n[j] = have ? __ldcg(counts + k) : 0.f;
                    a[j] = __ldcg(row + col);
                    b[j] = have ? __ldcg(row + c4n + col) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
                for (int j = 0; j < kRows; ++j) {
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
    int row;                     // first block's number within its micro-batch
    __device__ __forceinline__ UnitWalk(const PipeScalars& p, int m_first, int first, int count) : left(count)
    {
        z = 0;
        if (p.ksplit > 1) { const int whole = div_magic(first, p.ksplit, p.magic_ksplit); z = first - whole * p.ksplit; first = whole; }
        m = div_magic(first, p.blocks_per_m, p.magic_blocks);
        row = first - m * p.blocks_per_m;
        ul = row * p.unit_block;
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

// The MMA issuer (one thread).
// KIND 0: one pass; 1: hi*hi and hi*lo from one MMA over [B_hi; B_lo]; 2: three MMAs.  Everything that does not change is
// taken out of the loops and nothing in the tap loop waits or branches on loaded values: with the modes told apart inside it
// an MMA took 115 clocks to issue, against 40 (N = 32) the tensor core needs.
struct MmaEnv {
    volatile int* abort_flag;
    uint32_t smem_base, tmem_base, a_full, a_empty, b_full, b_empty, acc_full, acc_empty;
    int *a_used, *b_used;
};
// (Only the low words of the descriptors ever change.)
__device__ __forceinline__ uint64_t desc_at(uint32_t lo, uint32_t hi) { uint64_t r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi)); return r; }
template <int KIND>
__device__ __forceinline__ void issue_tile(uint32_t acc, uint32_t a, uint32_t a_hi, uint32_t b, uint32_t b_hi, uint32_t b_half, uint32_t idesc, uint32_t idesc2, uint32_t keep)
{
    // (a: value or hi part, +4: lo part; +2: the chunk's second K step)
    auto A = [&](uint32_t d) { return desc_at(a + d, a_hi); };
    auto B = [&](uint32_t d) { return desc_at(b + d, b_hi); };
    if (KIND == 0) {
        umma_tf32(acc, A(0), B(0), idesc, keep);
        umma_tf32(acc, A(2), B(2), idesc, 1u);
    } else if (KIND == 1) {
        umma_tf32(acc, A(0), B(0), idesc2, keep);
        umma_tf32(acc, A(4), B(0), idesc, 1u);
        umma_tf32(acc, A(2), B(2), idesc2, 1u);
        umma_tf32(acc, A(6), B(2), idesc, 1u);
    } else {
        umma_tf32(acc, A(0), B(0), idesc, keep);
        umma_tf32(acc, A(4), B(0), idesc, 1u);
        umma_tf32(acc, A(0), B(b_half), idesc, 1u);
        umma_tf32(acc, A(2), B(2), idesc, 1u);
        umma_tf32(acc, A(6), B(2), idesc, 1u);
        umma_tf32(acc, A(2), B(b_half + 2), idesc, 1u);
    }
}
// WINDOW: 3 or 1.  What one MMA of 16 columns costs is 40 clocks; every branch between two of them in this one-thread code about 50 more.
template <bool RESIDENT, int KIND, int WINDOW, bool CELL>
__device__ __forceinline__ void mma_role(const PipeScalars& p, const MmaEnv& e, UnitWalk u)
{
    const uint64_t a_desc = smem_desc(e.smem_base, 16, 1024, 128), b_desc = smem_desc(e.smem_base + p.off_b, 16, 512, 64);
    const uint32_t a_hi = (uint32_t)(a_desc >> 32), b_hi = (uint32_t)(b_desc >> 32), a_first = (uint32_t)a_desc, b_first = (uint32_t)b_desc;
    const uint32_t idesc = p.idesc, idesc2 = p.idesc2, acc_cols = p.acc_cols, a_step = p.a_stage_bytes >> 4, b_step = p.b_stage_bytes >> 4, b_tap = p.b_tap_bytes >> 4;
    const uint32_t b_half = ((uint32_t)p.n_chunk * 64u) >> 4;
    const int a_stages = p.a_stages, b_stages = p.b_stages, acc_bufs = p.acc_bufs, T = p.T;
    const bool by_tap = !RESIDENT && WINDOW > 1 && p.b_taps == 1;    // a stage of the weight ring is one tap, not a window row
    const uint32_t next_row = (uint32_t)p.Wp * 8u;                   // from a window row to the next
    int s = 0, bs = 0, buf = 0, b_it = 0, a_it = 0;
    uint32_t apar = 0, bpar = 0, cpar = 1u;
    if (RESIDENT) {
        b_it = 1;
        if (!mbar_wait(e.b_full, 0, e.abort_flag)) { report(p.status, 22); return; }
    }
#pragma unroll 1
    for (; u.left > 0; u.next(p)) {
        const int nt = u.tiles(p), kb = u.kb(p), ke = u.ke(p);
        const uint32_t skipped = p.flat ? 0u : (uint32_t)(span_of(p, u).lead * 8);
        if (!mbar_wait(e.acc_empty + 8 * buf, cpar, e.abort_flag)) { report(p.status, 23); return; }
        tc_fence_after();
        const uint32_t acc0 = e.tmem_base + (uint32_t)(buf * T) * acc_cols;
        uint32_t keep = 0u;
        uint32_t b = b_first + (uint32_t)(kb * WINDOW * WINDOW) * b_tap;      // RESIDENT: the taps of all chunks stand in a row
#pragma unroll 1
        for (int c = kb; c < ke; ++c) {
            if (!mbar_wait(e.a_full + 8 * s, apar, e.abort_flag)) { report(p.status, 24); return; }
            uint32_t row = a_first + (uint32_t)s * a_step + skipped;
#pragma unroll 1
            for (int r = 0; r < WINDOW; ++r, row += next_row) {
#pragma unroll
                for (int x = 0; x < WINDOW; ++x) {
                    if (!RESIDENT && (by_tap || x == 0)) {
                        if (!mbar_wait(e.b_full + 8 * bs, bpar, e.abort_flag)) { report(p.status, 25); *e.b_used = b_it; *e.a_used = a_it; return; }
                        b = b_first + (uint32_t)bs * b_step;
                    }
                    issue_tile<KIND>(acc0, row + 8u * x, a_hi, b, b_hi, b_half, idesc, idesc2, keep);
                    if (T > 1)
#pragma unroll 1
                        for (int t = 1; t < nt; ++t) issue_tile<KIND>(acc0 + (uint32_t)t * acc_cols, row + 8u * x + (uint32_t)(t * 1024), a_hi, b, b_hi, b_half, idesc, idesc2, keep);
                    keep = 1u;
                    b += b_tap;
                    if (!RESIDENT && (by_tap || x == WINDOW - 1)) {
                        umma_commit(e.b_empty + 8 * bs);
                        ++b_it;
                        if (++bs == b_stages) { bs = 0; bpar ^= 1u; }
                    }
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
    // The late trigger.  Here, where a CTA has one last unit whatever its patches and sets of write-out warps are: tied to the write-out's
    // walk it missed every launch with several patches a unit.  Launches in a row, without it / with it, three passes, batch 128:
    // 3x3 128 -> 128 @16 45.2 / 42.6 us, 32 -> 128 @16 19.0 / 17.6, 64 -> 64 @32 53.3 / 51.4, 1x1 256 -> 64 @8 data gradient 8.0 / 7.4; batch 64: 64 -> 256 @56
    // 72.8 / 70.7; slower 3x3 256 -> 256 @8 73.2 / 76.1 and 16 -> 16 @32 14.9 / 15.3.  Behind the last
    // accumulator of a set instead the same or up to 2 % slower.
    if (!CELL && p.pdl_late) pdl_launch_dependents();
    if (CELL) {                  // wait until every barrier has seen its last arrival: they are used again
#pragma unroll 1
        for (int i = 0; i < a_stages && i < a_it; ++i) mbar_wait(e.a_empty + 8 * i, (uint32_t)((a_it - 1 - i) / a_stages) & 1u, e.abort_flag);
        if (!RESIDENT)
#pragma unroll 1
            for (int i = 0; i < b_stages && i < b_it; ++i) mbar_wait(e.b_empty + 8 * i, (uint32_t)((b_it - 1 - i) / b_stages) & 1u, e.abort_flag);
    }
}
template <int WINDOW, bool CELL>
__device__ __forceinline__ void mma_roles(const PipeScalars& p, const MmaEnv& e, const UnitWalk& u)
{
    if (p.b_resident) {
        if (!p.three) mma_role<true, 0, WINDOW, CELL>(p, e, u);
        else if (p.stacked) mma_role<true, 1, WINDOW, CELL>(p, e, u);
        else mma_role<true, 2, WINDOW, CELL>(p, e, u);
    } else {
        if (!p.three) mma_role<false, 0, WINDOW, CELL>(p, e, u);
        else if (p.stacked) mma_role<false, 1, WINDOW, CELL>(p, e, u);
        else mma_role<false, 2, WINDOW, CELL>(p, e, u);
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
        mbar_init(bar + 8 * s, full ? split : (acc_empty ? emit : (s < kMaxA && p.flat ? 32u : 1u)));
    }
    if (lane == 0) { sh.abort_flag = 0; sh.b_issued = 0; sh.b_used = 0; sh.a_issued = 0; sh.a_used = 0; }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// The end of a block of units in the write-out, for a plain BN: what eight lanes have of a column and what the warps have of it added up in
// fp64, as the kernels that form a BN's statistics themselves add their threads' sums.
__device__ __forceinline__ void lanes_fp64(const float* from, int step, float& sum, float& sq)
{
    double s = 0.0, q = 0.0;
#pragma unroll 1
    for (int j = 0; j < 8; ++j) { s += (double)from[16 * j]; q += (double)from[step + 16 * j]; }
    sum = (float)s; sq = (float)q;
}
__device__ __forceinline__ void parts_fp64(const PipeScalars& p, const float* c3, const float* counts, int parts, int bm, int br, int c)
{
    const int n_chunk = p.n_chunk, C = p.c_out;
    double n = 0.0, k0 = 0.0, sum = 0.0, sq = 0.0;
#pragma unroll 1
    for (int w = 0; w < parts; ++w, c3 += 3 * n_chunk) {
        const double cnt = counts[w];
        if (cnt == 0.0) continue;
        const double d = c3[n_chunk];
        if (n == 0.0) k0 = c3[0];
        const double ek = (double)c3[0] - k0;
        n += cnt;
        sum += fma(cnt, ek, d);
        sq += fma(ek, fma(cnt, ek, 2.0 * d), (double)c3[2 * n_chunk]);
    }
    const double dm = n > 0.0 ? sum / n : 0.0, mean = k0 + dm;
    float* all = p.st_partials + (size_t)bm * partial_floats(p.blocks_per_m, C);
    float* row = all + (size_t)br * 2 * C + c;
    row[0] = (float)mean; row[C] = fmaxf((float)fma(-sum, dm, sq), 0.f);
    all[partial_lo(p.blocks_per_m, C) + (size_t)br * C + c] = (float)(mean - (double)(float)mean);
    if (c == 0) all[(size_t)p.blocks_per_m * 2 * C + br] = (float)n;
}

// ---- write-out: tensor memory -> registers -> global memory ----
// A 16x256b load gives four lanes of a warp a row of the accumulator, two columns of every eight each.  The weights' rows are copied
// in an order (the dimensions of their tensor map) that makes a lane's columns of a group of 4 W output channels W consecutive
// ones: the four lanes have a row of the group between them, residuals are read the same way, and a lane keeps the sums of its
// own channels from row to row, with no transposition and no exchange between lanes until a block of units ends.
// A warp's 32 rows x 32 channels with residual and moments took 3600 clocks through a patch of shared memory, 300 instructions with
// their latencies; now 2000 without and up to 4300 with a residual, which is then the memory's rate (18 bytes a clock and SM).
//
// What a launch of a few microseconds pays here is the first execution of every instruction: 100-150 clocks per 128 bytes of
// code, a first patch took 8600 clocks against 2400 of the following ones.  So there is one loop over patches (32 rows x
// one group of channels), every part of which stands in the code once, and its first, dry round - no rows, nothing waited
// for, nothing stored; what it reads from tensor and shared memory is discarded - runs ahead of the first accumulator.  Everything together: ResNet-110 5.96 -> 5.62 ms, ResNet-11 0.327 -> 0.299.
template <int W, bool FLAT, bool BNB, bool PLAIN, bool CELL>
__device__ __forceinline__ void write_out(const PipeScalars& p, PipeShared& sh, uint8_t* smem, const uint32_t tmem_base,
                                          const uint32_t acc_full, const uint32_t acc_empty, const UnitWalk& u0, const int slice)
{
    constexpr int kCols = 4 * W, H = 2 * W;           // channels of a group; values a lane holds of 16 rows
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int tid = threadIdx.x - 32 * (kFirstSplit + kSplitWarps), ew = warp - kFirstSplit - kSplitWarps;
    const int quad = warp & 3, half = ew >> 2;        // a warp reads the 32 lanes of its quadrant; two warps share one
    const int q = lane & 3, r8 = lane >> 2;           // this lane's quarter of a row; its rows are r8 + 8 i
    const int n_chunk = p.n_chunk, groups = n_chunk / kCols, T = p.T, C_out = p.c_out, ksplit = p.ksplit, co0 = slice * n_chunk;
    const bool stacked = p.stacked != 0, stats = p.st_partials != nullptr, plain = CELL ? p.st_plain != 0 : PLAIN;
    // Two sets of four warps.  Where there is one group of channels they take alternate units (with two accumulator sets) or
    // alternate tiles of a unit; otherwise alternate groups.
    const bool alternate = p.epi_alternate != 0, whole = groups == 1;
    const int g_first = whole ? 0 : half, g_step = whole ? 1 : 2, t_first = whole && !alternate ? half : 0, t_step = whole && !alternate ? 2 : 1;
    const int parts = whole ? 8 : 4;
    int part = whole ? ew : quad;
    float4* const slots = reinterpret_cast<float4*>(smem + p.off_slots + (uint32_t)ew * p.slot_bytes);      // the lanes' sums of the block so far, W / 2 float4 a lane and group
    // residuals of two times 16 rows; 8 (or 4) lanes copy a row's line (piece l % W of row l / W), so that no sector is fetched twice
    uint8_t* const ring = smem + p.off_ring + ew * (W * 512);
    const int copy_row = lane / W, copy_piece = lane % W, copy_step = 32 / W;
    float* const bn_tab = reinterpret_cast<float*>(smem + p.off_bnb) + ew * 256;    // BNB: mean, rstd, gamma, beta of this warp's groups
    float* const mom0 = reinterpret_cast<float*>(smem + p.off_stat);                // the warps' moments of a block, twice: those of the block before may still be read
    const int mom_size = parts * (3 * n_chunk + 1);
    const float* const addend = BNB ? p.bn_x : p.extra;
    const size_t sk_tile = (size_t)kTileM * n_chunk;
    int bn_m = -1, buf = alternate ? half : 0, flip = 0, count = 0;
    uint32_t par = 0;
    bool have = false, ok = true, finish = true, dry = true;
    // blocks of units: the current one's micro-batch, row of partial moments, the number of its first unit within the CTA's work
    const int blocks = u0.left;
    int bm = u0.m, br = u0.row, first_unit = 0;

    // the patch under way and the one after it: unit, tile, group, offsets of this lane's four rows (-1: none), which of the
    // warp's 32 there are, and, three bits a row, which neighbours of a strided data gradient's sample get zeros
    UnitWalk u = u0, nu = u0;
    if (alternate && half == 1) nu.next(p);
    int t = 0, g = g_first, nt = t_first, ng = g_first;
    int off[4], noff[4], fill = 0, nfill = 0;
    unsigned int who = 0, nwho = 0;
    int nrow = -1;                                    // offset of the next patch's row `lane`
    bool first = false, nfirst = true;
#pragma unroll
    for (int i = 0; i < 4; ++i) off[i] = noff[i] = -1;
    bool place = true;
#pragma unroll 1
    while (true) {
        const bool more = nu.left > 0;
        if (place && more) {
            // (a set that shares the tiles of a unit may find none left: no rows then)
            const int pos0 = (nu.ul * T + nt) * kTileM + quad * 32;
            const bool some = nt < nu.tiles(p);
            if (FLAT) {
                const int n = some ? p.pos_per_m - pos0 : 0;
                nwho = n >= 32 ? 0xffffffffu : (n > 0 ? (1u << n) - 1u : 0u);
#pragma unroll
                for (int i = 0; i < 4; ++i) noff[i] = r8 + 8 * i < n ? (pos0 + r8 + 8 * i) * C_out : -1;
                nrow = lane < n ? (pos0 + lane) * C_out : -1;
            } else {
                const Pixel px = locate(p, pos0 + lane);
                const int ro = some && px.own ? px.n * p.os_n + px.y * p.os_h + px.x * p.os_w : -1;
                const bool right = 2 * px.x + 1 < p.out_w, below = 2 * px.y + 1 < p.out_h;
                const int f = (right ? 1 : 0) | (below ? 2 : 0) | (right && below ? 4 : 0);
                nwho = __ballot_sync(0xffffffffu, ro >= 0);
                nrow = ro;
                nfill = 0;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    noff[i] = __shfl_sync(0xffffffffu, ro, r8 + 8 * i);
                    nfill |= __shfl_sync(0xffffffffu, f, r8 + 8 * i) << (3 * i);
                }
            }
        }
        if (!dry && first) {
            ok = mbar_wait(acc_full + 8 * buf, par, &sh.abort_flag);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok && lane == 0) report(p.status, 27);
            tc_fence_after();
        }
        const uint32_t acc0 = tmem_base + (uint32_t)(buf * T) * p.acc_cols + ((uint32_t)(quad * 32) << 16);
        // 16 rows of a group, hi and lo products added
        auto accumulator = [&](int at_t, int at_g, int h, float* v) {
            const uint32_t at = acc0 + (uint32_t)at_t * p.acc_cols + (uint32_t)(kCols * at_g) + ((uint32_t)(16 * h) << 16);
            tmem_ld_rows<W>(at, v);
            if (stacked) {
                float w[H];
                tmem_ld_rows<W>(at + (uint32_t)n_chunk, w);
                tmem_ld_wait();
                add_to<H>(v, w);
            } else {
                tmem_ld_wait();
            }
        };
        float* const sk_all = ksplit > 1 ? reinterpret_cast<float*>(p.sk_base + u.m * p.sk_ms + kSplitKTicketBytes) + ((size_t)u.ul * p.slices + slice) * ksplit * T * sk_tile : nullptr;
        if (ksplit > 1 && !dry && first) {
            // this CTA's partial sums; the CTA that takes the last ticket of the unit adds them in split order
            unsigned int* ticket = reinterpret_cast<unsigned int*>(p.sk_base + u.m * p.sk_ms) + (size_t)u.ul * p.slices + slice;
            float* mine = sk_all + u.z * T * sk_tile;
#pragma unroll 1
            for (int t1 = t_first; t1 < u.tiles(p); t1 += t_step)
#pragma unroll 1
                for (int g1 = g_first; g1 < groups; g1 += g_step)
#pragma unroll 1
                    for (int h = 0; h < 2; ++h) {
                        float v[H];
                        accumulator(t1, g1, h, v);
                        float* d = mine + t1 * sk_tile + ((size_t)((2 * g1 + h) * 4 + quad) * 32 + lane) * H;
                        if (ok) { store_vec<W>(d, v); store_vec<W>(d + W, v + W); }
                    }
            __threadfence();
            epi_sync();
            if (tid == 0) {
                sh.last_of_unit = atomicAdd(ticket, 1u) == (unsigned int)ksplit - 1u;
                if (sh.last_of_unit) *ticket = 0u;
            }
            epi_sync();
            finish = sh.last_of_unit != 0;
            if (finish) __threadfence();
            else {
                who = 0;
#pragma unroll
                for (int i = 0; i < 4; ++i) off[i] = -1;
            }
        }
        if (BNB && !dry && u.m != bn_m) {
            // statistics and parameters of this warp's columns (statistics are results of the step: not the read-only path)
            bn_m = u.m;
            const float* st = p.bn_stats + (long long)u.m * 2 * C_out + co0;
            __syncwarp();
#pragma unroll 1
            for (int g1 = g_first, gi = 0; g1 < groups; g1 += g_step, ++gi)
                if (lane < 4 * W) {
                    const int kind = lane / W;
                    const float* from = kind < 2 ? st + kind * C_out : (kind == 2 ? p.bn_gamma : p.bn_beta) + co0;
                    reinterpret_cast<float4*>(bn_tab + gi * 4 * kCols)[lane] = __ldcg(reinterpret_cast<const float4*>(from + kCols * g1) + lane % W);
                }
            __syncwarp();
        }
        const int gi = whole ? 0 : g >> 1;
        if (g == g_first) count += __popc(who);
        float* const sums = mom0 + flip * mom_size + part * 3 * n_chunk + kCols * g + W * q;      // k, then the block's results
        float4* const slot = slots + gi * (W / 2) * 32 + lane;
        float* const dst = p.out + (long long)u.m * p.out_ms + co0 + kCols * g + W * q;
        const float* const src = addend + (long long)nu.m * p.out_ms + co0 + kCols * ng + 4 * copy_piece;
        float k[W], sd[W], sq[W];
        bool have_k = have;
#pragma unroll
        for (int j = 0; j < W; ++j) k[j] = sd[j] = sq[j] = 0.f;
        if (stats && have) {
            if (!BNB) read_vec<W>(sums, k);
#pragma unroll
            for (int j = 0; j < W; j += 4) { read_vec<4>(reinterpret_cast<const float*>(slot + 8 * j), sd + j); read_vec<4>(reinterpret_cast<const float*>(slot + 8 * (W + j)), sq + j); }
        }
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            const int o[2] = {h ? off[2] : off[0], h ? off[3] : off[1]};
            float v[H];
            if (ksplit > 1 && finish && !dry) {
#pragma unroll
                for (int j = 0; j < H; ++j) v[j] = 0.f;
#pragma unroll 1
                for (int z = 0; z < ksplit; ++z) {
                    float w[H];
                    load_vec<H>(sk_all + ((size_t)z * T + t) * sk_tile + ((size_t)((2 * g + h) * 4 + quad) * 32 + lane) * H, w);
                    add_to<H>(v, w);
                }
            } else {
                accumulator(t, g, h, v);
            }
            // in the order of the rows: tensor memory gives two columns of row 0, two of row 1, the next two of row 0, ...
            float x[2][W], e[H];
#pragma unroll
            for (int j = 0; j < W; ++j) { x[0][j] = v[(j >> 1) * 4 + (j & 1)]; x[1][j] = v[(j >> 1) * 4 + 2 + (j & 1)]; }
            if (addend) {
                if (!dry) { cp_async_wait<1>(); __syncwarp(); }
#pragma unroll
                for (int r = 0; r < 2; ++r)
#pragma unroll
                    for (int j = 0; j < W; j += 4)
                        read_vec<4>(reinterpret_cast<const float*>(ring + h * (W * 256) + (r8 + 8 * r) * (W * 16) + (((q * (W / 4) + j / 4) ^ (W == 8 ? r8 : 0)) << 4)), e + W * r + j);
                if (!BNB) { add_to<W>(x[0], e); add_to<W>(x[1], e + W); }
            }
            if (dry && h == 0 && !CELL) pdl_wait();
            if (addend) {
                // the residual (BNB: the BN's input) of the next patch travels while this one is written out
                __syncwarp();
                if (more) {
                    uint32_t to = smem_u32(ring + h * (W * 256)) + (uint32_t)(copy_row * (W * 16));
#pragma unroll
                    for (int i = 0; i < W / 2; ++i, to += (uint32_t)(copy_step * W * 16)) {
                        const int r = copy_row + copy_step * i;
                        const int no = __shfl_sync(0xffffffffu, nrow, 16 * h + r);
                        cp_async16(to + (uint32_t)((copy_piece ^ (W == 8 ? r & 7 : 0)) << 4), src + (no >= 0 ? no : 0));
                    }
                }
                cp_async_commit();
            }
            if (p.accumulate) {
#pragma unroll
                for (int r = 0; r < 2; ++r)
                    if (o[r] >= 0) { float w[W]; load_vec<W>(dst + o[r], w); add_to<W>(x[r], w); }
            }
            if (BNB) {
                const float* tab = bn_tab + gi * 4 * kCols + W * q;
#pragma unroll
                for (int j = 0; j < W; j += 4) {
                    const float4 mu = *reinterpret_cast<const float4*>(tab + j), rs = *reinterpret_cast<const float4*>(tab + kCols + j),
                                 ga = *reinterpret_cast<const float4*>(tab + 2 * kCols + j), be = *reinterpret_cast<const float4*>(tab + 3 * kCols + j);
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const float* xe = e + W * r + j;
                        const bool real = o[r] >= 0;
                        const float4 xh = mul4(sub4(make_float4(xe[0], xe[1], xe[2], xe[3]), mu), rs), z = fma4(ga, xh, be);
                        const float4 d = make_float4(real && z.x > 0.f ? x[r][j] : 0.f, real && z.y > 0.f ? x[r][j + 1] : 0.f,
                                                     real && z.z > 0.f ? x[r][j + 2] : 0.f, real && z.w > 0.f ? x[r][j + 3] : 0.f);
                        const float4 a = add4(make_float4(sd[j], sd[j + 1], sd[j + 2], sd[j + 3]), d),
                                     b = fma4(d, xh, make_float4(sq[j], sq[j + 1], sq[j + 2], sq[j + 3]));
                        sd[j] = a.x; sd[j + 1] = a.y; sd[j + 2] = a.z; sd[j + 3] = a.w;
                        sq[j] = b.x; sq[j + 1] = b.y; sq[j + 2] = b.z; sq[j + 3] = b.w;
                    }
                }
            } else if (stats) {
                // moments are taken about a value of the column (the first one): sums of x and x * x themselves would cancel for
                // a channel whose mean is large against its spread
                if (!have_k && (((who >> (16 * h)) & 0xffffu) || dry)) {
                    const int r0 = __ffs(who) - 1, from = (r0 & 7) * 4 + q;
#pragma unroll
                    for (int j = 0; j < W; ++j) k[j] = __shfl_sync(0xffffffffu, r0 & 8 ? x[1][j] : x[0][j], from);
                    have_k = true;
                    if (lane < 4)
#pragma unroll
                        for (int j = 0; j < W; j += 4) *reinterpret_cast<float4*>(sums + j) = make_float4(k[j], k[j + 1], k[j + 2], k[j + 3]);
                }
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const bool real = o[r] >= 0;
#pragma unroll
                    for (int j = 0; j < W; j += 2) {
                        const uint64_t kk = pair(k[j], k[j + 1]), d = sub2(real ? pair(x[r][j], x[r][j + 1]) : kk, kk);
                        unpair(add2(pair(sd[j], sd[j + 1]), d), sd[j], sd[j + 1]);
                        unpair(fma2(d, d, pair(sq[j], sq[j + 1])), sq[j], sq[j + 1]);
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < 2; ++r)
                if (o[r] >= 0 && ok) store_vec<W>(dst + o[r], x[r]);
            if (!FLAT && p.zero_fill == 2) {
                // strided data gradient: the positions between the samples receive no contribution
                float zero[W];
#pragma unroll
                for (int j = 0; j < W; ++j) zero[j] = 0.f;
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int f = o[r] >= 0 && ok ? fill >> (3 * (2 * h + r)) : 0;
                    if (f & 1) store_vec<W>(dst + o[r] + p.dense_w, zero);
                    if (f & 2) store_vec<W>(dst + o[r] + p.dense_h, zero);
                    if (f & 4) store_vec<W>(dst + o[r] + p.dense_h + p.dense_w, zero);
                }
            }
        }
        if (stats) {
#pragma unroll
            for (int j = 0; j < W; j += 4) {
                slot[8 * j] = make_float4(sd[j], sd[j + 1], sd[j + 2], sd[j + 3]);
                slot[8 * (W + j)] = make_float4(sq[j], sq[j + 1], sq[j + 2], sq[j + 3]);
            }
            __syncwarp();                             // k is read by the next patch, the sums by the lanes that add them up
        }
        if (nfirst && !dry) {
            // the accumulator is read: the next unit's MMAs may have it
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty + 8 * buf);
            if (alternate) par ^= 1u;                 // (a set of warps always meets its own accumulator set)
            else if (++buf == p.acc_bufs) { buf = 0; par ^= 1u; }
        }
        if (g + g_step >= groups && who) have = true;
        // Ends of blocks between this patch and the next (alternating sets: also of blocks in which this set has no unit): the moments
        // of the lanes, then the warps' parts, each about its own shift.
        const int at_block = blocks - (more ? nu.left : 0);
#pragma unroll 1
        for (int b = dry ? -1 : blocks - u.left; stats && b < at_block; ++b) {
            float* const contrib = mom0 + flip * mom_size;
            float* const counts = contrib + (size_t)parts * 3 * n_chunk;
            // a lane adds what eight lanes have of its column
            const float* from = reinterpret_cast<const float*>(slots) + ((lane % W) >> 2) * 128 + (lane / W) * 4 + (lane & 3);
#pragma unroll 1
            for (int g1 = g_first; g1 < groups; g1 += g_step, from += W * 64) {
                float sum = 0.f, sq1 = 0.f;
                if (plain) lanes_fp64(from, W * 32, sum, sq1);
                else
#pragma unroll
                    for (int j = 0; j < 8; ++j) { sum += from[16 * j]; sq1 += from[W * 32 + 16 * j]; }
                float* to = contrib + part * 3 * n_chunk + kCols * g1 + lane;
                if (lane < kCols) { to[n_chunk] = sum; to[2 * n_chunk] = sq1; }
            }
            if (lane == 0 && (whole || half == 0)) counts[part] = (float)count;
            epi_sync();
            if (plain) {
                if (tid < n_chunk && ok && finish && b >= 0) parts_fp64(p, contrib + tid, counts, parts, bm, br, co0 + tid);
            } else if (tid < n_chunk) {
                // parts about their own shifts k_w: sum and squares about the first one's,
                //   sum (x - k0) = sum_w [d_w + n_w e],  sum (x - k0)^2 = sum_w [q_w + e (2 d_w + n_w e)],  e = k_w - k0
                // (BNB: no shifts, the sums themselves)
                float N = 0.f, k0 = 0.f, sum = 0.f, sq1 = 0.f;
                const float* c3 = contrib + tid;
#pragma unroll 1
                for (int w = 0; w < parts; ++w, c3 += 3 * n_chunk) {
                    const float cnt = counts[w];
                    if (cnt == 0.f) continue;
                    const float d = c3[n_chunk];
                    if (N == 0.f && !BNB) k0 = c3[0];
                    const float ek = BNB ? 0.f : c3[0] - k0;
                    N += cnt;
                    sum += fmaf(cnt, ek, d);
                    sq1 += fmaf(ek, fmaf(cnt, ek, 2.f * d), c3[2 * n_chunk]);
                }
                const float dm = N > 0.f ? sum / N : 0.f, m2 = fmaxf(fmaf(-sum, dm, sq1), 0.f);
                float* all = p.st_partials + (size_t)bm * partial_floats(p.blocks_per_m, C_out);
                float* row = all + (size_t)br * 2 * C_out + co0 + tid;
                if (ok && finish && b >= 0) {
                    row[0] = BNB ? sum : k0 + dm; row[C_out] = BNB ? sq1 : m2;
                    if (!BNB && tid == 0 && slice == 0) all[(size_t)p.blocks_per_m * 2 * C_out + br] = N;
                }
            }
            flip ^= 1;
            count = 0; have = false;
            if (b >= 0 && ksplit == 1) {
                const int start = br * p.unit_block, left = p.units_per_m - start;
                first_unit += left < p.unit_block ? left : p.unit_block;
                if (++br == p.blocks_per_m) { br = 0; ++bm; }
                // (alternating sets: a block's first unit counts as part 0..3, whichever set's turn it is, so that its moments are added in
                // the same order wherever in a CTA's work the block stands)
                if (alternate) part = quad + 4 * (half ^ (first_unit & 1));
            }
        }
        if (!more) break;
        // the next patch is the current one, and what follows it
        u = nu; t = nt < T ? nt : T - 1; g = ng; who = nwho; fill = nfill; first = nfirst;
        if (first) finish = true;
        if (ksplit > 1) { bm = u.m; br = u.ul; }
#pragma unroll
        for (int i = 0; i < 4; ++i) off[i] = finish ? noff[i] : -1;
        if (!finish) who = 0;
        dry = false;
        place = nfirst = false;
        if ((ng += g_step) >= groups) {
            ng = g_first; place = true;
            if ((nt += t_step) >= nu.tiles(p)) {
                nt = t_first; nfirst = true;
                nu.next(p);
                if (alternate && nu.left > 0) nu.next(p);
            }
        }
    }
}

// The work of one CTA (number bid of nblk) of a launch: the barriers are initialised, tensor memory is allocated.
// FLAT: the operand's positions and the output's pixels are the same consecutive rows (1x1 windows without a stride).
// BNB: a data gradient that forms the sums of a BN+ReLU's backward.
// CELL: inside the persistent cell kernel, which keeps its tensor memory and has no successor to trigger.
// W: channels of a row that a write-out lane has.
// PLAIN: the moments it forms are a plain BN's (a kernel of its own: as a branch of the write-out the fp64 sums cost every launch, ResNet-11
// 286 -> 290 us); a persistent cell has the branch.
template <bool BN_IN, bool FLAT, bool BNB, bool PLAIN, int W, bool CELL>
__device__ __forceinline__ void pipe_cta(const PipeParams& gp, const PipeScalars& p, PipeShared& sh, uint8_t* smem, const uint32_t tmem_base,
                                         const int m_first, const int m_count, const int bid, const int nblk)
{
    const uint32_t smem_base = smem_u32(smem);
    const int warp = warp_index(), lane = threadIdx.x & 31;
    uint64_t* bars = sh.bars;
    int &abort_flag = sh.abort_flag, &b_issued = sh.b_issued, &b_used = sh.b_used, &a_issued = sh.a_issued, &a_used = sh.a_used;
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
    const UnitWalk u0(p, m_first, u_first, u_count);

    if (p.flat && (warp == 0 || warp == 3)) {
        // ---- operand copies, consecutive pixels ----
        // Two warps take alternate blocks, 16 bytes a lane straight to their place in the swizzled rows.  A tensor copy takes an SM 6.7
        // clocks for every 64-byte row of its box (copies alone on all SMs: 9.6 bytes a clock and SM, 15 in rows of 128 bytes).
        const int S = p.a_stages, C = p.c_in, row0 = lane >> 2, mine = warp == 0 ? 0 : 1;
        const uint32_t at = smem_base + (uint32_t)row0 * 128u + (uint32_t)(((lane & 3) ^ row0) << 4);
        int s = mine % S, it = 0;
        uint32_t par = mine < S ? 1u : 0u;
        bool live = true, waited = CELL;
#pragma unroll 1
        for (UnitWalk u = u0; u.left > 0 && live; u.next(p)) {
            const int start = u.ul * p.T * kTileM, rows = u.tiles(p) * kTileM, valid = p.pos_per_m - start;
            const float* const unit = p.in + (long long)u.m * p.in_ms + (long long)(start + row0) * C + 4 * (lane & 3);
#pragma unroll 1
            for (int c = u.kb(p), ce = u.ke(p); c < ce; ++c, ++it) {
                if ((it & 1) != mine) continue;
                live = __all_sync(0xffffffffu, mbar_wait(a_empty + 8 * s, par, &abort_flag));
                if (!live) { if (lane == 0) report(p.status, 20); break; }
                if (!waited) { pdl_wait(); waited = true; }
                const float* src = unit + 16 * c;
                uint32_t dst = at + (uint32_t)s * p.a_stage_bytes;
#pragma unroll 4
                for (int row = row0; row < rows; row += 8, src += 8 * C, dst += 1024u) cp_async16_zfill(dst, row < valid ? src : p.in, row < valid);
                cp_async_arrive(a_raw + 8 * s);
                s += 2;
                if (s >= S) { s -= S; par ^= 1u; }
            }
        }
        cp_async_wait<0>();                           // (also after a wait that gave up: nothing may land in shared memory that was given back)
    } else if (warp == 0) {
        if (elect_one()) {
            // ---- operand copies ---- (the first one's coordinates are worked out while the predecessor still runs)
            const int S = p.a_stages;
            int s = 0, it = 0;
            uint32_t par = 1u;
            bool live = true;
#pragma unroll 1
            for (UnitWalk u = u0; u.left > 0 && live; u.next(p)) {
                const Span sp = span_of(p, u);
                const uint32_t tx = (uint32_t)sp.rows * 64u;
                // first block: map, row within it
                int img0 = 0, h0 = 0, strip0 = 0;
                {
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
                    if (!CELL && it == 0) pdl_wait();
                    {
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
            const int taps = p.taps, c_in = p.c_in, block0 = p.wide ? co0 >> 5 : co0 >> 4;
            if (p.b_resident) {
                const int n = p.n_chunks * taps;
                mbar_expect_tx(b_full, tx * (uint32_t)n);
                uint32_t dst = dst0;
#pragma unroll 1
                for (int c = 0; c < p.n_chunks; ++c)
#pragma unroll 1
                    for (int tap = 0; tap < taps; ++tap, dst += tap_bytes) {
                        tma_load_5d(dst, &gp.tm_b, b_full, tap * c_in + 16 * c, 0, 0, 0, block0);
                        if (three) tma_load_5d(dst + half, &gp.tm_b_lo, b_full, tap * c_in + 16 * c, 0, 0, 0, block0);
                    }
                b_issued = 1;
            } else {
                int s = 0, it = 0;
                uint32_t par = 1u;
                bool live = true;
#pragma unroll 1
                for (UnitWalk u = u0; u.left > 0 && live; u.next(p))
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
                                tma_load_5d(dst, &gp.tm_b, bar, tap * c_in + 16 * c, 0, 0, 0, block0);
                                if (three) tma_load_5d(dst + half, &gp.tm_b_lo, bar, tap * c_in + 16 * c, 0, 0, 0, block0);
                            }
                            if (++s == p.b_stages) { s = 0; par ^= 1u; }
                        }
                b_issued = it;
            }
        }
    } else if (warp == 2) {
        if (elect_one()) {
            // ---- MMAs ----
            const MmaEnv env{&abort_flag, smem_base, tmem_base, a_full, a_empty, b_full, b_empty, acc_full, acc_empty, &a_used, &b_used};
            if (FLAT || p.R == 1) mma_roles<1, CELL>(p, env, u0);
            else mma_roles<3, CELL>(p, env, u0);
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
        }
        // a step of row_step positions in maps, rows and columns of the padded grid
        const int dn = BN_IN && !FLAT ? row_step / p.img_pos : 0, drem = row_step - dn * p.img_pos;
        const int dy = BN_IN && !FLAT ? drem / p.Wp : 0, dx = drem - dy * p.Wp, Hp = BN_IN && !FLAT ? p.img_pos / p.Wp : 1;
        // this group's next block: its chunk within the unit, its place in the ring
        int s = my_group, ahead = my_group, cur_m = -1;
        uint32_t par = 0;
        const bool store_y = BN_IN && slice == 0;
        bool ok = true;
        UnitWalk cu = u0;
        // (No dry round here: the merge and the first block are bound by their own latencies, and what the round costs in conditions made
        // ResNet-110 5.46 -> 5.59 ms, scoring ResNet-182 6.03 -> 6.29.)
        if (BN_IN && !CELL) pdl_wait();
#pragma unroll 1
        for (; cu.left > 0; cu.next(p)) {
            const int kb = cu.kb(p), ke = cu.ke(p);
            const Span sp = span_of(p, cu);
            const int own_lo = sp.lead + halo, own_hi = own_lo + cu.tiles(p) * kTileM, valid = p.pos_per_m - sp.pos0;
            if (BN_IN) {
                if (cu.m != cur_m) {
                    cur_m = cu.m;
                    split_sync();                     // everybody is done with the table of the micro-batch before
                    const float* const rows0 = p.bn_partials + (size_t)cur_m * partial_floats(p.bn_units, C);
                    merge_moments<kSplitThreads>(rows0, p.bn_units, C, p.bn_inv_rows, p.bn_eps, tab, reinterpret_cast<float4*>(smem + p.off_red), tid);
                    split_sync();
                }
                if (slice == 0 && cu.ul == 0 && cu.z == 0)
#pragma unroll 1
                    for (int i = tid; i < 2 * C; i += kSplitThreads) p.bn_stats[(size_t)cur_m * 2 * C + i] = tab[i];
            }
#pragma unroll 1
            for (int c = kb + ahead; c < ke; c += groups) {
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
                    float* ydst = p.bn_y + (long long)cu.m * p.in_ms + 16 * c + 4 * cph;
                    int yo = (sp.pos0 + row0) * C;                   // FLAT: offset of this thread's first row
                    int pn = 0, py = 0, px = 0;                      // otherwise its map, row and column
                    if (!FLAT) {
                        int pos = sp.pos0 + row0;
                        if (pos < 0) { pos += p.img_pos; pn = -1; }
                        const int q = div_magic(pos, p.img_pos, p.magic_img);
                        pn += q; pos -= q * p.img_pos;
                        py = div_magic(pos, p.Wp, p.magic_w); px = pos - py * p.Wp;
                    }
                    // two rows in flight; the block is allocated in whole batches, so the last one needs no bounds
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
                                *reinterpret_cast<float4*>(lo + byte_step * j) = lo_part(v[j]);
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
                            *reinterpret_cast<float4*>(lo + byte_step * j) = lo_part(v[j]);
                    }
                }
                fence_async_smem();               // generic-proxy writes -> tensor-core reads
                __syncwarp();
                if (lane == 0) mbar_arrive(a_full + 8 * s);
                s += groups;
                if (s >= S) { s -= S; par ^= 1u; }
                ahead += groups;
            }
            ahead -= ke - kb;
        }
    } else if (warp >= kFirstSplit + kSplitWarps) {
        write_out<W, FLAT, BNB, PLAIN, CELL>(p, sh, smem, tmem_base, acc_full, acc_empty, u0, slice);
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

template <bool BN_IN, bool FLAT, bool BNB, bool PLAIN, int W>
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
    if (threadIdx.x == 32) { if (!p.flat) prefetch_tmap(&gp.tm_a); prefetch_tmap(&gp.tm_b); prefetch_tmap(&gp.tm_b_lo); }
    if (warp_index() == 0) tmem_alloc(smem_u32(&sh.tmem_slot), p.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // The successor may be scheduled from here on: not before this CTA holds its tensor memory, or the successor's CTA could
    // take the columns this one needs and wait for this one to finish.
    if (!p.pdl_late) pdl_launch_dependents();
    const uint32_t tmem_base = sh.tmem_slot;
    pipe_cta<BN_IN, FLAT, BNB, PLAIN, W, false>(gp, p, sh, smem, tmem_base, m_first, m_count, (int)blockIdx.x, (int)gridDim.x);
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
                if (flat) { if (p.wide) pipe_cta<true, true, false, false, 8, true>(gp, p, sh, smem, tmem_base, m_first, m_count, v, V); else pipe_cta<true, true, false, false, 4, true>(gp, p, sh, smem, tmem_base, m_first, m_count, v, V); }
                else { if (p.wide) pipe_cta<true, false, false, false, 8, true>(gp, p, sh, smem, tmem_base, m_first, m_count, v, V); else pipe_cta<true, false, false, false, 4, true>(gp, p, sh, smem, tmem_base, m_first, m_count, v, V); }
            } else {
                if (flat) { if (p.wide) pipe_cta<false, true, false, false, 8, true>(gp, p, sh, smem, tmem_base, m_first, m_count, v, V); else pipe_cta<false, true, false, false, 4, true>(gp, p, sh, smem, tmem_base, m_first, m_count, v, V); }
                else { if (p.wide) pipe_cta<false, false, false, false, 8, true>(gp, p, sh, smem, tmem_base, m_first, m_count, v, V); else pipe_cta<false, false, false, false, 4, true>(gp, p, sh, smem, tmem_base, m_first, m_count, v, V); }
            }
            if (sh.abort_flag) { if (tid == 0) cell_stop = 1; break; }
        }
        if (sh.abort_flag || (op + 1 < cp.n_ops && !cell_grid_barrier(cp.barrier, cp.status, &cell_stop))) break;
    }
    tc_fence_before();
    __syncthreads();
    if (warp_index() == 0) tmem_dealloc(tmem_base, cp.tmem_cols);
}

// A BN that no convolution applies, from the moments the producing convolution left: every block merges them (the same bits in each)
// and normalises its rows, one launch and one reading of x instead of a launch for the statistics and one for
// the rest.  sum, act: the residual sum and the ReLU that follow a plain BN in a post-activation block, sum = y + add, act = max(sum, 0),
// two launches and three trips through memory less.  Bound by memory; grid (blocks, micro-batches).
constexpr int kMergeThreads = 256;
constexpr int kMergeMaxChannels = 24576;              // mean and rstd of every channel in shared memory: 192 KB
constexpr int kMergeStep = kMergeThreads + 4;         // doubles between the values of a thread: the combining threads' banks
// merge_moments in fp64 and with the lower parts of the rows' means: a plain BN is no less precise here than where it forms its
// statistics itself (fp64 sums of fp32 partial sums, a root in fp64).  Mean, in sigma, and 1/sigma, in units of the last place, against fp64
// statistics of the stored values, root mean square over the channels, itself / here: 64 channels @8, 4 maps, 1.7e-8, 0.56 / 1.1e-8, 0.38;
// 32 @16, 32 maps, 1.4e-8, 0.39 / 0.9e-8, 0.27; 64 @56, 16 maps, 1.1e-8, 0.35 / 0.8e-8, 0.31.  In fp32 (as for BN+ReLU) 3.5e-8, 0.88; 1.2e-8,
// 0.58; 1.0e-8, 0.56.  A step of ResNet-110 with post-activation blocks takes 6.06 ms with it and 6.03 in fp32.
// red: 8 x kMergeStep.
__device__ __forceinline__ void merge_moments_fp64(const float* partials, int rows, int C, double inv_rows, float eps, float* tab, double* red, int t)
{
    constexpr int T = kMergeThreads, kRows = 2;
    const float *counts = partials + (size_t)rows * 2 * C, *lower = partials + partial_lo(rows, C);
    const int c4n = C >> 2, L = c4n <= T ? T / c4n : 1;
#pragma unroll 1
    for (int c0 = 0; c0 < c4n; c0 += T) {
        const int width = c4n - c0 < T ? c4n - c0 : T;
        const int ln = L > 1 ? t / c4n : 0, local = L > 1 ? t - ln * c4n : t, col = c0 + local;
        const bool mine = local < width && ln < L;
        double s[8] = {};                             // of four channels sum n (mean_u - ref), sum M2_u + n (mean_u - ref)^2
        if (mine) {
            const float4 r4 = __ldcg(reinterpret_cast<const float4*>(partials) + col);
            const float ref[4] = {r4.x, r4.y, r4.z, r4.w};
#pragma unroll 1
            for (int k0 = ln; k0 < rows; k0 += kRows * L) {
                float mean[kRows][4], lo[kRows][4], m2[kRows][4], n[kRows];
#pragma unroll
                for (int j = 0; j < kRows; ++j) {
                    const bool have = k0 + j * L < rows;
                    const size_t k = have ? k0 + j * L : 0;
                    n[j] = have ? __ldcg(counts + k) : 0.f;
                    load_vec<4>(partials + k * 2 * C + 4 * col, mean[j]);
                    load_vec<4>(partials + (k * 2 + 1) * C + 4 * col, m2[j]);
                    load_vec<4>(lower + k * C + 4 * col, lo[j]);
                }
#pragma unroll
                for (int j = 0; j < kRows; ++j)
                    if (k0 + j * L < rows)
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const double d = (double)mean[j][e] - (double)ref[e] + (double)lo[j][e], nd = (double)n[j] * d;
                            s[e] += nd;
                            s[4 + e] += fma(nd, d, (double)m2[j][e]);
                        }
            }
        }
        int lanes = L, at = t;                        // row lanes left to add
        bool put = mine;
        if (c4n <= 16 && (c4n & (c4n - 1)) == 0) {
            // the row lanes of a column inside a warp first: a fixed butterfly
#pragma unroll 1
            for (int o = 16; o >= c4n; o >>= 1)
#pragma unroll
                for (int e = 0; e < 8; ++e) s[e] += __shfl_xor_sync(0xffffffffu, s[e], o);
            lanes = T / 32;
            at = (t >> 5) * c4n + (t & 31);
            put = (t & 31) < c4n;
        }
        if (put)
#pragma unroll
            for (int e = 0; e < 8; ++e) red[e * kMergeStep + at] = s[e];
        __syncthreads();
#pragma unroll 1
        for (int c = t; c < 4 * width; c += T) {
            const double* r = red + (c & 3) * kMergeStep + (c >> 2);
            double d = 0.0, q = 0.0;
#pragma unroll 4
            for (int l = 0; l < lanes; ++l, r += width) { d += r[0]; q += r[4 * kMergeStep]; }
            const double dm = d * inv_rows;
            double var = q * inv_rows - dm * dm;
            if (var < 0.0) var = 0.0;
            tab[4 * c0 + c] = (float)((double)__ldcg(partials + 4 * c0 + c) + dm);
            tab[C + 4 * c0 + c] = (float)rsqrt(var + (double)eps);
        }
        __syncthreads();
    }
}
struct BnMergeApply {
    const float *partials, *gamma, *beta;
    float* stats;
    const float4 *x, *add;
    float4 *y, *sum, *act;       // add, sum, act: null without
    int units, C;
    double inv_rows;
    float eps;
    long long n4, per_block, ms4;   // float4 of a micro-batch, of a block; between micro-batches
};
template <bool RELU>
__global__ void __launch_bounds__(kMergeThreads, 3) bn_merge_apply_kernel(const BnMergeApply a)
{
    constexpr float floor = RELU ? 0.f : -INFINITY;
    extern __shared__ float tab[];                    // mean, rstd
    __shared__ __align__(16) double red[8 * kMergeStep];
    pdl_launch_dependents();
    pdl_wait();
    const int t = threadIdx.x, C = a.C, c4n = C >> 2;
    const float* partials = a.partials + (size_t)blockIdx.y * partial_floats(a.units, C);
    if constexpr (RELU) {
        merge_moments<kMergeThreads>(partials, a.units, C, a.inv_rows, a.eps, tab, reinterpret_cast<float4*>(red), t);
        __syncthreads();
    } else merge_moments_fp64(partials, a.units, C, a.inv_rows, a.eps, tab, red, t);
    if (blockIdx.x == 0)
        for (int i = t; i < 2 * C; i += kMergeThreads) a.stats[(size_t)blockIdx.y * 2 * C + i] = tab[i];
    const long long first = blockIdx.x * a.per_block + t, end = (blockIdx.x + 1) * a.per_block < a.n4 ? (blockIdx.x + 1) * a.per_block : a.n4;
    const long long ms = blockIdx.y * a.ms4;
    int col = (int)(first % c4n);
    const int step = kMergeThreads % c4n;             // 0: a thread keeps its channels
    const float4 *mean4 = reinterpret_cast<const float4*>(tab), *rstd4 = mean4 + c4n;
    float4 mu = mean4[col], rs = rstd4[col], g = __ldg(reinterpret_cast<const float4*>(a.gamma) + col), b = __ldg(reinterpret_cast<const float4*>(a.beta) + col);
#pragma unroll 1
    for (long long i = first; i < end; i += 4 * kMergeThreads) {
        float4 v[4], e[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (i + j * kMergeThreads < end) {
                v[j] = __ldcg(a.x + ms + i + j * kMergeThreads);
                if (a.add) e[j] = __ldcg(a.add + ms + i + j * kMergeThreads);
            }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (i + j * kMergeThreads < end) {
                const long long at = ms + i + j * kMergeThreads;
                float4 z = fma4(g, mul4(sub4(v[j], mu), rs), b);
                z = make_float4(fmaxf(z.x, floor), fmaxf(z.y, floor), fmaxf(z.z, floor), fmaxf(z.w, floor));
                a.y[at] = z;
                if (a.add) {
                    z = add4(z, e[j]);
                    a.sum[at] = z;
                    if (a.act) a.act[at] = make_float4(fmaxf(z.x, 0.f), fmaxf(z.y, 0.f), fmaxf(z.z, 0.f), fmaxf(z.w, 0.f));
                }
                if (step) {
                    col += step;
                    if (col >= c4n) col -= c4n;
                    mu = mean4[col]; rs = rstd4[col]; g = __ldg(reinterpret_cast<const float4*>(a.gamma) + col); b = __ldg(reinterpret_cast<const float4*>(a.beta) + col);
                }
            }
    }
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
inline unsigned int stat_bytes(int n_chunk) { return (unsigned int)(2 * (n_chunk <= 32 ? 8 : 4) * (3 * n_chunk + 1) * 4 + 127) & ~127u; }
// sums a write-out warp's lanes keep: two values of 32 lanes a channel of its groups (no launch of more than 128 channels forms any)
inline unsigned int slot_bytes(int n_chunk)
{
    if (n_chunk > 128) return 0;
    return n_chunk % 32 == 0 ? (unsigned int)(n_chunk / 32 + 1) / 2 * 2048u : (unsigned int)(n_chunk / 16 + 1) / 2 * 1024u;
}
constexpr unsigned int kBnbBytes = kEpiWarps * 1024u;  // statistics and parameters of a write-out warp's channels (data gradient)
inline int split_groups_of(int a_stages) { return a_stages % 4 == 0 ? 4 : (a_stages % 2 == 0 ? 2 : 1); }
inline unsigned int bn_bytes(int c_in) { return (unsigned int)(4 * c_in * 4 + 4 * kSplitThreads * 16); }

}  // namespace

size_t conv_pipe_partial_floats(int units_per_m, int channels) { return partial_floats(units_per_m, channels); }

static bool plan_geom(const ConvShape& s, int pass, int passes, int launched, ConvPipeUse use, ConvPipeGeom* g)
{
    PipeView v;
    if (pass == PASS_WGRAD || !pipe_view(s, pass, &v)) return false;
    const bool three = passes == 3;
    // Channel slices of 128 beyond 128 channels: a unit of 256 positions x 128 channels reads half as many weight bytes from
    // L2 per MMA as 128 positions x 256 channels do.
    g->n_chunk = v.c_out <= 128 ? v.c_out : (v.c_out % 128 == 0 ? 128 : (v.c_out <= 256 ? v.c_out : 0));
    if (!g->n_chunk) return false;
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
    // Where that leaves more than half the GPU idle, slices of 64: each write-out warp then has one group of 32 channels instead of
    // two, 2400 clocks less of a launch of a few microseconds.
    if (g->n_chunk == 128 && 2LL * launched * g->tiles_per_m * (v.c_out / 128) <= kPlanSms) g->n_chunk = 64;
    g->slices = v.c_out / g->n_chunk;
    const int taps = s.R * s.R, chunks = v.c_in / 16, n = g->n_chunk;
    g->b_tap_bytes = (unsigned int)(three ? 2 : 1) * (unsigned int)n * 64u;
    const unsigned int all_b = g->b_tap_bytes * (unsigned int)(taps * chunks);
    // (the data gradient applies no BN)
    g->use = use;
    const unsigned int fixed = (use.addend ? kEpiWarps * (n % 32 == 0 ? 4096u : 2048u) : 0u) + (use.moments ? kEpiWarps * slot_bytes(n) + stat_bytes(n) : 0u) + 128u +
                               (pass == PASS_DGRAD ? (use.moments ? kBnbBytes : 0u) : (use.bn_in ? bn_bytes(v.c_in) : 0u));
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
                const double tap_mma = 2.0 * T * step, epi = T * (use.addend ? 3600.0 : 2000.0) * (n <= 32 ? 0.5 : (n + 63) / 64);
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
                        const double split = use.bn_in ? 1200.0 + 8.0 * rows * groups / 4.0 : (three ? 250.0 + 5.6 * rows * groups / 4.0 : 100.0);
                        const double chunk = std::max({mma, (1200.0 + rows * 1.6 + split + mma) / as, split / groups, rows * 64.0 / 20.0});
                        const double k_loop = chunk * chunks, body = bufs == 2 ? std::max(k_loop, epi) : k_loop + epi;
                        // (weights that stay leave the memory system to the rest)
                        const double cost = (rounds * body + chunk + 1000.0 + epi) * (resident ? 1.0 : 1.03);
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
bool conv_pipe_geom(const ConvShape& s, int pass, int passes, int launched, ConvPipeUse use, ConvPipeGeom* g)
{
    struct Kept { int key[12]; bool used, ok; ConvPipeGeom g; };
    constexpr int kKept = 256;
    static thread_local Kept kept[kKept];
    const int key[12] = {s.N, s.H, s.W, s.C, s.K, s.R, s.stride, s.pad, pass, passes, launched, (use.addend ? 1 : 0) | (use.moments ? 2 : 0) | (use.bn_in ? 4 : 0)};
    unsigned int h = 2166136261u;
    for (int k : key) h = (h ^ (unsigned int)k) * 16777619u;
    // (keys that differ in the last word only must not share a place: the convolutions of a block take turns)
    h = (h ^ (h >> 15)) * 2246822519u;
    Kept& e = kept[(h >> 16) % kKept];
    if (!e.used || memcmp(e.key, key, sizeof key) != 0) {
        memcpy(e.key, key, sizeof key);
        e.ok = plan_geom(s, pass, passes, launched, use, &e.g);
        e.used = true;
    }
    *g = e.g;
    return e.ok;
}

bool conv_pipe_can_fuse_bn_output(const ConvPipeGeom& g) { return g.n_chunk <= 128; }      // a warp keeps the moments of two groups of 32 channels
// (No column strips.)  Every channel slice of a launch repeats the work on its operand, about 1200 clocks for 128 rows of 16 channels
// instead of 400: with four and more slices of 128 channels of a 1x1 window that is what the launch takes, and BN+ReLU in kernels of their own
// cost less (256->1024 @14 and the like: ResNet-152 35.0 -> 34.1 ms).  Two slices pay: 64->256 @56 would take 16 us to read and write.
// So do four slices of 64 channels, which launches have that leave SMs idle otherwise: ResNet-11 285.8 us, 287.0 with BN kernels there
// instead, ResNet-29 858 and 865.
bool conv_pipe_can_fuse_bn_input(const ConvShape& s) { return s.stride == 1 && s.C % 16 == 0 && s.C <= 512 && s.W <= 254 && (s.R > 1 || s.K <= 256); }

size_t conv_pipe_splitk_bytes(const ConvPipeGeom& g)
{
    if (g.ksplit < 2) return 0;
    return (kSplitKTicketBytes + (size_t)g.units_per_m * g.slices * g.ksplit * g.T * kTileM * g.n_chunk * sizeof(float) + 255) & ~(size_t)255;
}
size_t conv_pipe_splitk_bytes(const ConvShape& s, int pass, int passes, int launched)
{
    ConvPipeGeom g;
    return conv_pipe_geom(s, pass, passes, launched, ConvPipeUse(), &g) ? conv_pipe_splitk_bytes(g) : 0;
}

struct ConvPipeLaunch { PipeParams p; unsigned int smem; int bn_in; };
static_assert(sizeof(ConvPipeLaunch) <= sizeof(((ConvPipePlan*)0)->storage), "plan storage too small");

namespace {
using PipeKernel = void (*)(PipeParams, int, int);
template <int W>
PipeKernel pipe_kernel(bool bn_in, bool flat, bool bnb, bool plain)
{
    if (bnb) return flat ? conv_pipe_kernel<false, true, true, false, W> : conv_pipe_kernel<false, false, true, false, W>;
    if (plain && bn_in) return flat ? conv_pipe_kernel<true, true, false, true, W> : conv_pipe_kernel<true, false, false, true, W>;
    if (plain) return flat ? conv_pipe_kernel<false, true, false, true, W> : conv_pipe_kernel<false, false, false, true, W>;
    if (bn_in) return flat ? conv_pipe_kernel<true, true, false, false, W> : conv_pipe_kernel<true, false, false, false, W>;
    return flat ? conv_pipe_kernel<false, true, false, false, W> : conv_pipe_kernel<false, false, false, false, W>;
}
}  // namespace

cudaError_t conv_pipe_init()
{
    static PerDevice<bool> attributes;
    bool set = false;
    return attributes.get(&set, [](int, bool* done) {
        cudaError_t e = cudaSuccess;
        for (int k = 0; k < 16; ++k)
            for (PipeKernel kernel : {pipe_kernel<8>(k & 1, k & 2, k & 4, k & 8), pipe_kernel<4>(k & 1, k & 2, k & 4, k & 8)})
                if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPipeSmem + 1024);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(conv_pipe_cell_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPipeSmem + 1024);
        for (auto kernel : {bn_merge_apply_kernel<true>, bn_merge_apply_kernel<false>})
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * kMergeMaxChannels * (int)sizeof(float));
        *done = true;
        return e;
    });
}

namespace {
cudaError_t encode_map(CUtensorMap* tm, const float* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides, const cuuint32_t* box,
                       CUtensorMapSwizzle swizzle)
{
    if (!g_encode) return cudaErrorNotReady;
    const cuuint32_t ones[5] = {1, 1, 1, 1, 1};
    const CUresult r = g_encode(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, (cuuint32_t)rank, const_cast<float*>(base), dims, strides, box, ones,
                                CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}
// Rows in the order the write-out wants the accumulator's columns in (write_out): of a group of 4 W channels, columns 2 i and 2 i + 1
// of the c-th eight are channels W i + 2 c and the next.
cudaError_t encode_weights(CUtensorMap* tm, const float* base, long long kdim, int c_out, int n_chunk, int W)
{
    const cuuint64_t row = (cuuint64_t)kdim * 4;
    const cuuint64_t dims[5] = {(cuuint64_t)kdim, 2, 4, (cuuint64_t)W / 2, (cuuint64_t)(c_out / (4 * W))}, strides[4] = {row, W * row, 2 * row, 4 * W * row};
    const cuuint32_t box[5] = {16, 2, 4, (cuuint32_t)W / 2, (cuuint32_t)(n_chunk / (4 * W))};
    return encode_map(tm, base, 5, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_64B);
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
                              size_t splitk_bytes, bool w_ready, ConvPipeUse use)
{
    plan->valid = 0;
    ConvPipeGeom g;
    PipeView v;
    if ((passes != 1 && passes != 3) || !conv_pipe_geom(s, pass, passes, launched, use, &g) || !pipe_view(s, pass, &v)) return cudaErrorNotSupported;
    ConvPipeLaunch* L = reinterpret_cast<ConvPipeLaunch*>(plan->storage);
    memset(L, 0, sizeof *L);
    const long long kdim = (long long)s.R * s.R * v.c_in;
    // (16-byte copies and stores; a tensor map refuses other addresses itself)
    if ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out) | reinterpret_cast<uintptr_t>(extra)) & 15) return cudaErrorInvalidValue;
    // 32-byte pieces of a row where the buffers allow them (a caller's own may start at any 16 bytes)
    const uintptr_t at = reinterpret_cast<uintptr_t>(out) | reinterpret_cast<uintptr_t>(splitk) | (splitk_bytes & 31);
    const bool wide = g.n_chunk % 32 == 0 && at % 32 == 0;
    cudaError_t e = encode_weights(&L->p.tm_b, w_hi, kdim, v.c_out, g.n_chunk, wide ? 8 : 4);
    if (e == cudaSuccess) e = encode_weights(&L->p.tm_b_lo, passes == 3 ? w_lo : w_hi, kdim, v.c_out, g.n_chunk, wide ? 8 : 4);
    if (e != cudaSuccess) return e;
    PipeScalars& p = L->p.s;
    p.in = in; p.out = out; p.extra = extra; p.in_ms = v.in_ms; p.out_ms = v.out_ms;
    p.accumulate = accumulate ? 1 : 0;
    p.units_per_m = g.units_per_m; p.unit_block = g.unit_block; p.blocks_per_m = g.blocks_per_m; p.tiles_per_m = g.tiles_per_m; p.T = g.T; p.slices = g.slices; p.n_chunk = g.n_chunk; p.ksplit = g.ksplit;
    p.R = s.R; p.taps = s.R * s.R; p.n_chunks = v.c_in / 16; p.c_in = v.c_in; p.c_out = v.c_out;
    p.pos_per_m = g.pos_per_m; p.Wp = g.Wp; p.img_pos = g.Wp * g.Hp; p.Hv = v.P; p.W = v.Q; p.halo = g.halo;
    p.strips = g.strips; p.strip_w = g.strip_w; p.col0 = g.col0;
    p.magic_w = magic_of(g.Wp); p.magic_img = magic_of(p.img_pos); p.magic_strip = magic_of(g.strips); p.magic_blocks = magic_of(g.blocks_per_m); p.magic_ksplit = magic_of(g.ksplit);
    p.in_sw = v.in_sw; p.in_sh = v.in_sh; p.in_sn = v.in_sn; p.os_w = v.os_w; p.os_h = v.os_h; p.os_n = v.os_n;
    p.zero_fill = v.zero_fill; p.out_h = v.out_h; p.out_w = v.out_w; p.dense_h = v.dense_h; p.dense_w = v.dense_w;
    p.flat = g.flat; p.box_h = g.box_h; p.box_pos = g.box_h * g.Wp; p.blocks_per_img = g.Hp / g.box_h;
    p.magic_box = magic_of(p.box_pos); p.magic_bpi = magic_of(p.blocks_per_img);
    p.pix_ms = g.flat ? (long long)s.N * v.P * v.Q : s.N;
    if ((long long)M * p.pix_ms >= (1LL << 31)) return cudaErrorNotSupported;
    if (!g.flat) {
        const cuuint64_t rd[4] = {(cuuint64_t)v.c_in, (cuuint64_t)v.in_W, (cuuint64_t)v.in_H, (cuuint64_t)M * s.N};
        const cuuint64_t rs[3] = {(cuuint64_t)v.in_sw * 4, (cuuint64_t)v.in_sh * 4, (cuuint64_t)v.in_sn * 4};
        const cuuint32_t rb[4] = {16, (cuuint32_t)g.Wp, (cuuint32_t)g.box_h, 1};
        e = encode_map(&L->p.tm_a, in, 4, rd, rs, rb, CU_TENSOR_MAP_SWIZZLE_128B);
        if (e != cudaSuccess) return e;
    }
    p.a_stages = g.a_stages; p.b_stages = g.b_stages; p.b_taps = g.b_taps; p.b_resident = g.b_resident; p.acc_bufs = g.acc_bufs;
    p.a_stage_bytes = g.a_stage_bytes; p.b_stage_bytes = g.b_stage_bytes; p.b_tap_bytes = g.b_tap_bytes; p.acc_cols = g.acc_cols;
    p.tmem_cols = columns_pow2((unsigned int)(g.acc_bufs * g.T) * g.acc_cols);
    p.idesc = instr_desc(g.n_chunk, false, false);
    p.idesc2 = instr_desc(g.stacked ? 2 * g.n_chunk : g.n_chunk, false, false);
    p.split_groups = split_groups_of(g.a_stages);
    p.wide = wide ? 1 : 0;
    p.epi_alternate = g.acc_bufs == 2 && g.n_chunk == (wide ? 32 : 16) && g.ksplit == 1 ? 1 : 0;
    p.slot_bytes = slot_bytes(g.n_chunk);
    p.three = passes == 3 ? 1 : 0; p.stacked = g.stacked; p.w_ready = w_ready ? 1 : 0;
    const unsigned int a_bytes = (unsigned int)g.a_stages * g.a_stage_bytes;
    p.off_b = a_bytes;
    p.off_ring = (p.off_b + (unsigned int)g.b_stages * g.b_stage_bytes + 127u) & ~127u;
    p.off_slots = p.off_ring + (g.use.addend ? kEpiWarps * (wide ? 4096u : 2048u) : 0u);
    p.off_stat = p.off_slots + (g.use.moments ? kEpiWarps * p.slot_bytes : 0u);
    p.off_red = p.off_bnb = p.off_stat + (g.use.moments ? stat_bytes(g.n_chunk) : 0u);
    p.off_bn = p.off_red + 4 * kSplitThreads * 16;
    const bool sums = bn && (bn->out_partials || bn->bwd_partials);
    if (((extra || (bn && bn->bwd_partials)) && !use.addend) || (sums && !use.moments) || (bn && bn->in_partials && !use.bn_in)) return cudaErrorInvalidValue;
    L->smem = p.off_red + (pass == PASS_DGRAD && use.moments ? kBnbBytes : 0u) + 1024;
    if (bn && bn->out_partials) {
        if (!conv_pipe_can_fuse_bn_output(g)) return cudaErrorNotSupported;
        p.st_partials = bn->out_partials; p.st_plain = bn->out_plain ? 1 : 0;
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
    auto kernel = p.wide ? pipe_kernel<8>(L.bn_in, flat, p.bn_x != nullptr, p.st_plain) : pipe_kernel<4>(L.bn_in, flat, p.bn_x != nullptr, p.st_plain);
    // What a CTA has to do decides how its warps share it (the sums are the same either way).  A block of the operand takes one
    // splitter warp about 2000 clocks and all four of them 850, so with one or two blocks in all they share each; with a single unit
    // both halves of the write-out's warps take it.
    const int units = (tasks + per_slice - 1) / per_slice * p.unit_block, blocks = units * ((p.n_chunks + p.ksplit - 1) / p.ksplit);
    if (blocks < 4) L.p.s.split_groups = blocks < 2 || p.split_groups == 1 ? 1 : 2;
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

bool bn_merge_apply_takes(int C) { return C <= kMergeMaxChannels; }

cudaError_t bn_merge_apply(const float* partials, int units, const float* gamma, const float* beta, float eps, bool relu, const float* x, float* y, const float* add,
                           float* sum, float* act, float* stats, long long rows, int C, int m_count, cudaStream_t st, int64_t* n_launch)
{
    BnMergeApply a{};
    a.partials = partials; a.gamma = gamma; a.beta = beta; a.stats = stats; a.units = units; a.C = C;
    a.x = reinterpret_cast<const float4*>(x); a.add = reinterpret_cast<const float4*>(add);
    a.y = reinterpret_cast<float4*>(y); a.sum = reinterpret_cast<float4*>(sum); a.act = reinterpret_cast<float4*>(act);
    a.inv_rows = 1.0 / (double)rows; a.eps = eps;
    a.n4 = a.ms4 = rows * C / 4;
    // Every block merges the moments first: eight float4 a thread at least, twice as much of the tensor as of moments, four blocks an SM
    // at most.
    long long blocks = (a.n4 + 8 * kMergeThreads - 1) / (8 * kMergeThreads), most = 4 * kPlanSms / m_count, share = a.n4 / ((long long)units * C);
    if (blocks > share) blocks = share;
    if (blocks > most) blocks = most;
    if (blocks < 1) blocks = 1;
    a.per_block = (a.n4 + blocks - 1) / blocks;
    launch_pdl(relu ? bn_merge_apply_kernel<true> : bn_merge_apply_kernel<false>, dim3((unsigned int)((a.n4 + a.per_block - 1) / a.per_block), m_count), dim3(kMergeThreads), (size_t)2 * C * sizeof(float), st, a);
    if (n_launch) ++*n_launch;
    return cudaGetLastError();
}

}  // namespace hpf
