// Convolution on the tensor cores through windows of the input kept in shared memory (int8, binary and fp32 layers,
// delta and dense; tcgen05.mma kind::i8 and kind::f16).
//
// What bounds a convolution as an implicit GEMM here is not the tensor core but the way of its A operand into shared
// memory: gathered tap by tap, every input pixel is copied kh * kw times.  This kernel copies it once:
//   - the output pixels of all images are numbered in one linear space with row pitch Wq and image pitch Hq * Wq, so
//     much wider than the image that the zero padding of a row is the start of the next one.  In that space the input
//     pixel under tap (ky, kx) of output pixel i is pixel i + shift(ky, kx): an accumulator tile of 128 consecutive
//     output pixels reads 128 consecutive input pixels for every tap, from `shift` on;
//   - the window of input pixels that the tile's taps touch is laid out in shared memory as [16 bytes of K][pixel], the
//     K-major layout without swizzle whose row groups are 128 bytes apart, so a tap's operand is the same window read
//     from a start address 16 * shift bytes further on: no copy per tap at all;
//   - a stride s splits the input into s * s planes (pixels of equal remainders), each with taps of its own that are
//     again shifts within the plane; a block of the K loop is one plane and some channels;
//   - first layers (at most 4 channels) have too few K bytes per pixel: their windows hold, per output column, the kw
//     pixels of a filter row side by side, and the taps are the filter rows.  Where the stride is one or two 16-byte chunks
//     of pixels, neighbouring columns' chunks are the same pixels: the window then is the row itself in one or two arrays,
//     a chunk further right in the filter row being the next slot, instead of a copy of kw pixels per column.
// Pixels that did not change (delta) or lie outside the image are zero in the window.  A tile none of whose projection
// pixels has to be updated leaves at once; there is no compaction of rows below that (a tile's MMAs cost less than
// finding its rows did).
//
// fp32 layers: every operand is split into three bf16 pieces (8 + 8 + 8 bits: all 24 bits of the significand), and six
// of the nine products of pieces are formed; what the other three would add is below 2^-25 of a product, less than the
// rounding of one fp32 multiplication.  The second and third piece are kept 2^9 and 2^18 times as large, so that the pieces
// of small values do not fall below bf16's exponents; the products of equal scale share an accumulator.  The tensor core
// adds in fp32 but truncates, so the leading product has an accumulator that is added to registers (round to nearest)
// after at most WN_PROMOTE K steps of 16, and the five small ones have two of their own.  A value whose first piece is no
// finite number (an infinity, a NaN, or a float above bf16's largest) makes its third piece a NaN, by which a CTA notices
// it: such a CTA forms its sums one by one from the operands instead (wn_exact_row), and a layer with such a filter
// keeps the CUDA cores.  Error against fp64 (2-norm, dense, normal operands; a chain of fmaf): 3x3 of 256 channels 2.5e-7
// (4.1e-7), 5x5 of 96 3.4e-7 (8.3e-7), 11x11 first layer 1.0e-7 (1.6e-7); without the promotion 1.7e-6.
//
// Roles: warps 0-7 fill windows and drain accumulators, warp 8 issues the MMAs, warp 9 the bulk copies of the filters
// (packed at create time as the operand tiles they are).  K can be split over the CTAs of a cluster by blocks: the
// partial tiles are added through distributed shared memory in a fixed order (fp32 results are reproducible bit for bit,
// and a dense pass needs no zeroed projection).  Every wait on an mbarrier is bounded; one that runs out sets
// ERRW_TIMEOUT and the CTA leaves through the common exit.
//
// What bounds it: in a long K loop the MMAs' operand reads from shared memory (an MMA of 128 columns reads 8 KB and takes 97 to
// 118 clocks instead of 64, one of 32 columns 77; fp32: 413 clocks a K step of 16, 384 of them MMAs, 126 bytes of shared memory
// a clock); in a launch of a few tiles a chain (clocks: set-up 1.8 k, first window 2.2 k, MMAs 3 to 6 k, way out 1.2 to 2.3 k, 7 k
// for 64 KB of fp32 rows).  AlexNet-shaped stack at 227 x 227: 8 fp32 streams 187 us, 32 fp32 frames 462, one int8 frame 65, 32
// int8 frames 121; 4 ResNet-18-shaped int8 streams 171.
#include "rrm_common.cuh"
#include "rrm_tc.cuh"
#include "rrm_dev.cuh"
#include <climits>
#include <type_traits>

namespace rrm {

constexpr int WN_FILL = 256;                  // threads that fill windows and drain accumulators: two warpgroups
constexpr int WN_THREADS = WN_FILL + 64;
constexpr int WN_MAX_STAGES = 8, WN_MAX_ABUF = 4, WN_MAX_MT = 2;
constexpr int WN_MAX_SPAN = 1152;             // pixels of one plane of a window
constexpr int WN_TURN = 64;                  // columns of its 32 rows that a warp turns around at a time
constexpr int WN_PROMOTE = 32;                // fp32: K steps the leading product accumulates before it is promoted
constexpr int WN_NARROW = 32;                 // integers: columns of a tile where the wide ones are too few
constexpr size_t WN_SMEM_LIMIT = 227 * 1024;

// One plane's taps: first filter row / column and their numbers, the remainders of its pixels, the first tap's shift.
struct WinPlane { int ky0, kx0, ny, nx, ry, rx, shift0; };
constexpr int WN_MAX_PLANES = 16;

// x / d for 0 <= x < 2^31 as a 64-bit product and a shift
struct WinDiv { unsigned m, sh; };

struct WinParams {
    const void* A;            // int8 / fp32: delta rows (delta) or values (dense); binary: changed bits (delta) / unused
    const void* Anew;         // binary: current sign bits
    const uint32_t* in_act;   // input activity bitmap (delta mode)
    const uint32_t* oact;     // projection pixels to update (delta mode)
    int* ocount;              // their number is added here, and that of the accumulator tiles they lie in behind it
    const unsigned char* Wimg;      // [n tile][tap][group][2][pieces][bn][16 bytes]
    const void* bias;
    void* P;                  // [opixels][c_out]
    int* errw;
    const uint32_t* count_bitmap;   // dense evaluation inside a delta step: the layer's update bitmap, whose bits are counted
    int n, h, w, oh, ow, kh, kw, stride, pad, c_in, c_out;
    int row_units;            // units per input pixel: bytes, words or floats
    int Wq, Hq;               // pitches of the linear output space
    int min_shift, span, L;   // window: first pixel relative to the tile's first, pixels, 16-byte slots per K chunk
    int planes, all_tables;   // (all_tables: the planes' tables have room side by side)
    WinPlane plane[WN_MAX_PLANES];
    WinDiv div_img, div_row;  // by Hq * Wq and by Wq
    int groups, gblk, nchb, nblk;   // 32-byte K groups per tap, groups per block, channel blocks per plane, blocks
    int ks, per;              // CTAs that share a tile's blocks, blocks of each
    int tsplit;               // > 1: a share is one block's taps, cut into so many parts (ks = nblk * tsplit)
    int cluster;              // the shares of a tile form a cluster that adds them up (0: each adds onto the projection by itself)
    int bn, mt;               // columns and accumulator tiles (of 128 rows) per CTA
    int ntiles, narrow;       // column tiles, and whether they are the narrow ones
    int tps, stages, abuf;    // taps per filter stage, stages, window buffers
    int xarr;                 // first layers: arrays of an image row's chunks (0: the chunks of every column side by side)
    unsigned a_step, a_lbo;   // 16-byte slots between a pixel's K groups, and between the two chunks of a group
    unsigned stage_bytes, abytes, tail_off, tmem_cols;    // (tail_off: barriers and tables, behind windows, stages and drained rows)
    unsigned wait_limit;
    int frames;               // several frames in one launch (delta only; gridDim.z = frames x ks), distances as in TcParams
    long long row_stride, arena_stride, p_stride;
    int store;                // delta: the product is stored, not added
    // f in the kernel (dense passes): the layer's output, or what its pool window takes the maximum of, pixel by pixel
    void* X;                  // [opixels][cs] int8, sign words or float
    const void* res;          // shortcut values, laid out like X, or nullptr
    const void* bn_scale;
    const void* bn_shift;
    int cs, bits, shift, act_fn, theta;      // (bits: signs, 32 channels per word)
    int keep_from;            // first projection pixel whose projection is stored (at P); INT_MAX: none
};

struct WinTail {
    unsigned long long afull[WN_MAX_ABUF], aempty[WN_MAX_ABUF], bfull[WN_MAX_STAGES], bempty[WN_MAX_STAGES], dfull[2], dempty[2], done;
    uint32_t tmem_base;
    int fail;
    int exact;                                // fp32: a window holds a value whose pieces are no finite numbers
    alignas(16) int bias[128];                // of the CTA's columns (f in the kernel)
    int q[WN_MAX_MT * TC_M];                  // projection pixel of the row (-1: none, or not to be updated)
    // the windows' tables, one behind the other: per window pixel of a plane its offset in the input in units, -1: zero (first
    // layers: of its image row's first pixel, in pixels; and behind them, in the second half, the first input column under the
    // filter row * 256 + the input rows from the tap's first on, at most 255)
    int tab[2 * WN_MAX_SPAN];
};

// ---- small device helpers
// Low half of an operand descriptor: start address and the distance between the two 16-byte K chunks of an MMA, both in
// units of 16 bytes; the high half is the same for all (row groups 128 bytes apart, no swizzle).
__device__ __forceinline__ uint32_t wn_desc_lo(uint32_t addr, uint32_t k_slots) { return ((addr & 0x3ffffu) >> 4) | k_slots << 16; }
constexpr uint32_t WN_DESC_HI = (128u >> 4) | 1u << 14;
// The MMAs of one K step, issued by the lane with e != 0 in code the whole warp runs.  The descriptors come as 32-bit halves
// of which only the low one changes.
__device__ __forceinline__ void wn_step_i8(uint32_t d, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t accumulate, uint32_t e)
{
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b64 a, b;\n\t"
        "mov.b64 a, {%1, %3};\n\tmov.b64 b, {%2, %3};\n\t"
        "setp.ne.b32 p, %5, 0;\n\tsetp.ne.b32 q, %6, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::i8 [%0], a, b, %4, p;\n\t}"
        ::"r"(d), "r"(a_lo), "r"(b_lo), "r"(WN_DESC_HI), "r"(idesc), "r"(accumulate), "r"(e) : "memory");
}
// fp32: six products of pieces in four MMAs.  A filter tile's pieces lie side by side along the columns, so an MMA of twice
// the width adds one input piece times two filter pieces to the two accumulators of small products, d1 (scale 2^9) and d2
// (2^18) right behind it: a0 * (b1, b2), a1 * (b0, b1), and a2 * b0 to d2; the leading a0 * b0 goes to d0.
__device__ __forceinline__ void wn_step_f32(uint32_t d0, uint32_t d1, uint32_t d2, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t b0, uint32_t b1, uint32_t idesc,
                                            uint32_t idesc2, uint32_t acc0, uint32_t acc1, uint32_t e)
{
    asm volatile(
        "{\n\t.reg .pred p, r, q, t;\n\t.reg .b64 x, y, z, u, v;\n\t"
        "mov.b64 x, {%2, %7};\n\tmov.b64 y, {%3, %7};\n\tmov.b64 z, {%4, %7};\n\tmov.b64 u, {%5, %7};\n\tmov.b64 v, {%6, %7};\n\t"
        "setp.ne.b32 p, %10, 0;\n\tsetp.ne.b32 r, %11, 0;\n\tsetp.ne.b32 q, %12, 0;\n\tsetp.eq.b32 t, 0, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%1], x, v, %9, r;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%1], y, u, %9, t;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%13], z, u, %8, t;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], x, u, %8, p;\n\t}"
        ::"r"(d0), "r"(d1), "r"(a0), "r"(a1), "r"(a2), "r"(b0), "r"(b1), "r"(WN_DESC_HI), "r"(idesc), "r"(idesc2), "r"(acc0), "r"(acc1), "r"(e), "r"(d2) : "memory");
}
// one look at a barrier
__device__ __forceinline__ uint32_t mbar_poll(uint32_t bar, uint32_t parity)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(r) : "r"(bar), "r"(parity) : "memory");
    return r;
}
__device__ __forceinline__ void wn_commit(uint32_t bar, uint32_t e)
{
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar), "r"(e) : "memory");
}
__device__ __forceinline__ uint32_t wn_elect()
{
    uint32_t e;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
    return e;
}
__device__ __forceinline__ void wn_ld32(uint32_t taddr, uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void wn_zero32(uint32_t taddr)
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, "
        "%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1};" ::"r"(taddr), "r"(0u) : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
// the filling warps agree (and meet): true only if all of them say so
__device__ __forceinline__ bool wn_agree(bool ok)
{
    int r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %1, 0;\n\t"
        "barrier.cta.red.and.pred q, 1, 256, p;\n\t"
        "selp.b32 %0, 1, 0, q;\n\t}"
        : "=r"(r) : "r"((int)ok) : "memory");
    return r != 0;
}
__device__ __forceinline__ void wn_meet() { asm volatile("barrier.cta.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ void wn_cluster_meet()
{
    __syncwarp();                                            // (the aligned forms want whole warps)
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint4 wn_ld_remote(uint32_t addr, uint32_t rank)
{
    uint4 v;
    asm volatile(
        "{\n\t.reg .b32 r;\n\t"
        "mapa.shared::cluster.u32 r, %4, %5;\n\t"
        "ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [r];\n\t}"
        : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr), "r"(rank) : "memory");
    return v;
}
// two floats -> their three bf16 pieces, packed (low half: the first float); the second 2^9, the third 2^18 times as large
constexpr float WN_SCALE = 512.f;
__device__ __forceinline__ void wn_split(float a, float b, uint32_t& p0, uint32_t& p1, uint32_t& p2)
{
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p0) : "f"(b), "f"(a));
    a = (a - __uint_as_float(p0 << 16)) * WN_SCALE; b = (b - __uint_as_float(p0 & 0xffff0000u)) * WN_SCALE;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p1) : "f"(b), "f"(a));
    a = (a - __uint_as_float(p1 << 16)) * WN_SCALE; b = (b - __uint_as_float(p1 & 0xffff0000u)) * WN_SCALE;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p2) : "f"(b), "f"(a));
}
// a pair of bf16 sums that a NaN among the addends has made one
__device__ __forceinline__ uint32_t wn_bf16_add(uint32_t a, uint32_t b)
{
    asm("add.rn.bf16x2 %0, %0, %1;" : "+r"(a) : "r"(b));
    return a;
}
__device__ __forceinline__ bool wn_bf16_nan(uint32_t a) { return (a & 0x7fffu) > 0x7f80u || (a >> 16 & 0x7fffu) > 0x7f80u; }
__device__ __forceinline__ uint32_t wn_spread4(uint32_t x) { return ((x & 0xfu) * 0x00204081u) & 0x01010101u; }
__device__ __forceinline__ int wn_div(int x, const WinDiv& d) { return (int)((unsigned long long)(unsigned)x * d.m >> d.sh); }

// The windows' table for one plane: where each window pixel lies in the input.
template <bool DENSE, bool XCOL>
__device__ __forceinline__ void wn_table(const WinParams& p, const uint32_t* in_act, int* tab, int lin0, int plane)
{
    const int ry = p.plane[plane].ry, rx = p.plane[plane].rx;
    const int hwq = p.Hq * p.Wq;
    #pragma unroll 2
    for (int i = threadIdx.x; i < p.span; i += WN_FILL) {
        const int lin = lin0 + p.min_shift + i;
        int off = -1, x0 = 0;
        if (lin >= 0) {
            const int img = wn_div(lin, p.div_img), rem = lin - img * hwq, Y = wn_div(rem, p.div_row), X = rem - Y * p.Wq;
            const int iy = Y * p.stride + ry;
            if (XCOL) {
                // (one table for all planes, which are rows further down: the first one's row, and how many rows are left)
                const int y0 = Y * p.stride, left = min(p.h - y0, 255);
                if (img < p.n && left > 0) off = (img * p.h + y0) * p.w;
                x0 = (X * p.stride - p.pad) * 256 + max(left, 0);
            } else {
                const int ix = X * p.stride + rx;
                if (img < p.n && iy < p.h && ix < p.w) {
                    const int pix = (img * p.h + iy) * p.w + ix;
                    if (DENSE || ((in_act[pix >> 5] >> (pix & 31)) & 1u)) off = pix * p.row_units;
                }
            }
        }
        tab[i] = off;
        if (XCOL) tab[WN_MAX_SPAN + i] = x0;
    }
}

// f without pool window of 4 neighbouring channels (c: channel within the layer; channels beyond the last give zero)
template <int PT, int OT, typename pt>
__device__ __forceinline__ void wn_f(const WinParams& p, int c, const pt (&x)[4], const pt (&res)[4], pt (&y)[4])
{
    const pt v[1][4] = {{x[0], x[1], x[2], x[3]}};
    if (p.bn_scale) epi_f<PT, OT, 1, true, pt>(v, 1u, c, res, p.c_out, p.act_fn, p.shift, p.bn_scale, p.bn_shift, y);
    else epi_f<PT, OT, 1, false, pt>(v, 1u, c, res, p.c_out, p.act_fn, p.shift, nullptr, nullptr, y);
}
// four integers, saturated to int8 each, as one word
__device__ __forceinline__ uint32_t wn_pack4(int y0, int y1, int y2, int y3)
{
    uint32_t hi, w;
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(hi) : "r"(y3), "r"(y2), "r"(0));
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(w) : "r"(y1), "r"(y0), "r"(hi));
    return w;
}
__device__ __forceinline__ void wn_unpack4(uint32_t w, int (&y)[4])
{
    #pragma unroll
    for (int j = 0; j < 4; ++j) y[j] = (int)(int8_t)(w >> (8 * j));
}
// the same with the explicit affine (kept out of line: few layers have one, and the drain's code is fetched once per CTA)
__device__ __noinline__ uint32_t wn_f8_bn(const WinParams& p, int c, int x0, int x1, int x2, int x3, uint32_t res)
{
    const int x[4] = {x0, x1, x2, x3};
    int r[4], y[4];
    wn_unpack4(res, r);
    wn_f<T_I32, T_I8, int>(p, c, x, r, y);
    return wn_pack4(y[0], y[1], y[2], y[3]);
}
// int8 f of 4 neighbouring channels: requantisation (round half up), [+ shortcut], activation; the saturation at 127 is the
// packing's.  Channels beyond the layer's last have zero filters, bias and shortcut.
__device__ __forceinline__ uint32_t wn_f8_plain(const int (&x)[4], uint32_t res, int rnd, int sh, int lo, bool with_res)
{
    int y[4];
    #pragma unroll
    for (int j = 0; j < 4; ++j) y[j] = (x[j] + rnd) >> sh;
    if (with_res) {
        #pragma unroll
        for (int j = 0; j < 4; ++j) y[j] = max(-127, min(127, y[j])) + (int)(int8_t)(res >> (8 * j));
    }
    #pragma unroll
    for (int j = 0; j < 4; ++j) y[j] = max(y[j], lo);
    return wn_pack4(y[0], y[1], y[2], y[3]);
}
__device__ __forceinline__ uint32_t wn_f8(const WinParams& p, int c, const int (&x)[4], uint32_t res)
{
    if (p.bn_scale) return wn_f8_bn(p, c, x[0], x[1], x[2], x[3], res);
    return wn_f8_plain(x, res, p.shift > 0 ? 1 << (p.shift - 1) : 0, p.shift, p.act_fn == RRM_ACT_RELU ? 0 : -127, p.res != nullptr);
}

// fp32 f of 4 neighbouring channels with the explicit affine or a shortcut (out of line like wn_f8_bn)
__device__ __noinline__ float4 wn_f32_slow(const WinParams& p, int ch, int live, size_t at, float4 v)
{
    const float x[4] = {v.x, v.y, v.z, v.w};
    float res[4] = {0.f, 0.f, 0.f, 0.f}, y[4];
    #pragma unroll
    for (int j = 0; j < 4; ++j) if (p.res && j < live) res[j] = reinterpret_cast<const float*>(p.res)[at + j];
    wn_f<T_F32, T_F32, float>(p, ch, x, res, y);
    return make_float4(y[0], y[1], y[2], y[3]);
}

// fp32, the way out of windows with infinities, NaNs or values beyond bf16: one row's share of the sums, columns c_lo to
// c_hi of the tile, from the operands themselves (blocks b0 to b1; a filter value is the sum of its pieces).  lin: the
// row's position, or -1.  Out of line: ordinary data never come here.
template <bool DENSE, bool XCOL>
__device__ __noinline__ void wn_exact_row(const WinParams& p, const float* A, const uint32_t* in_act, int lin, int ntile, int b0, int b1,
                                          int c_lo, int c_hi, float* sums)
{
    for (int c = c_lo; c < c_hi; ++c) sums[c] = 0.f;
    if (lin < 0) return;
    const int hwq = p.Hq * p.Wq;
    const int img = wn_div(lin, p.div_img), rem = lin - img * hwq, oy = wn_div(rem, p.div_row), ox = rem - oy * p.Wq;
    const int row_taps = XCOL ? 1 : p.kw;
    for (int b = b0; b < b1; ++b) {
        const WinPlane& a = p.plane[b / p.nchb];
        const int k_lo = (b % p.nchb) * p.gblk * 16, k_hi = min(k_lo + p.gblk * 16, XCOL ? p.kw * 4 : p.c_in);
        for (int t = 0; t < a.ny * a.nx; ++t) {
            const int ky = a.ky0 + t / a.nx * p.stride, kx0 = a.kx0 + t % a.nx * p.stride;
            const int iy = oy * p.stride - p.pad + ky;
            if (iy < 0 || iy >= p.h) continue;
            const unsigned char* W = p.Wimg + ((size_t)ntile * row_taps * p.kh + (XCOL ? ky : ky * p.kw + kx0)) * p.groups * p.bn * 96;
            for (int k = k_lo; k < k_hi; ++k) {
                const int ix = ox * p.stride - p.pad + (XCOL ? k >> 2 : kx0), ci = XCOL ? k & 3 : k;
                if (ix < 0 || ix >= p.w || ci >= p.c_in) continue;
                const int pix = (img * p.h + iy) * p.w + ix;
                if (!DENSE && !((in_act[pix >> 5] >> (pix & 31)) & 1u)) continue;
                const float x = A[(size_t)pix * p.row_units + ci];
                if (x == 0.f) continue;                      // (the filters are finite)
                for (int c = c_lo; c < c_hi; ++c) {
                    const unsigned short* w = reinterpret_cast<const unsigned short*>(W + (size_t)(k >> 3) * p.bn * 48 + (size_t)c * 16) + (k & 7);
                    float v = __uint_as_float((uint32_t)w[0] << 16);
                    v = fmaf(__uint_as_float((uint32_t)w[p.bn * 8] << 16), 1.f / WN_SCALE, v);
                    v = fmaf(__uint_as_float((uint32_t)w[p.bn * 16] << 16), 1.f / (WN_SCALE * WN_SCALE), v);
                    sums[c] = fmaf(x, v, sums[c]);
                }
            }
        }
    }
}

// DT: T_F32, T_I8 or T_BIN.  XCOL: the first-layer form.  ACT (dense passes): f is applied here and the output written,
// instead of the projection by this kernel and f by another; the projection is stored only where a state needs it.  ASYNC: int8
// windows by asynchronous copies (a kernel of its own for dense passes: every CTA runs the code once, so the other way's
// instructions would cost each launch some 0.15 us).
template <int DT, bool DENSE, bool XCOL, bool ACT, bool ASYNC>
__global__ void __launch_bounds__(WN_THREADS, DT == T_F32 ? 1 : 2) conv_win_kernel(const __grid_constant__ WinParams p)
{
    constexpr int PIECES = DT == T_F32 ? 3 : 1;
    extern __shared__ unsigned char wn_smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // (the same in all lanes, and known to the compiler to be)
    const int tile = blockIdx.x, ntile = blockIdx.y;
    const int frame = (!DENSE && p.frames > 1) ? blockIdx.z / p.ks : 0, split = blockIdx.z - frame * p.ks;
    // (the frame's data; the parameters themselves stay in constant memory)
    const long long row_off = frame * p.row_stride, arena_off = frame * p.arena_stride;
    const char* const A = (const char*)p.A + row_off;
    const char* const Anew = (const char*)p.Anew + row_off;
    const uint32_t* const in_act = shift_bytes(p.in_act, arena_off);
    const uint32_t* const oact = shift_bytes(p.oact, arena_off);
    char* const P = (char*)p.P + frame * p.p_stride * 4;
    unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)wn_smem_raw + 127) & ~(uintptr_t)127);
    const uint32_t base_u32 = smem_u32(base), bstage_u32 = base_u32 + p.abuf * p.abytes;
    WinTail* S = reinterpret_cast<WinTail*>(base + p.tail_off);
    const int lin0 = tile * p.mt * TC_M;
    const int b0 = p.tsplit > 1 ? split / p.tsplit : split * p.per, b1 = min(p.nblk, b0 + p.per);
    const int part = p.tsplit > 1 ? split - b0 * p.tsplit : 0;
    const int plane0 = b0 / p.nchb;
    const uint32_t unit_b = (uint32_t)p.bn * 32u * PIECES;   // filter bytes of one (tap, group)
    bool ok = true;
    int issued = 0;                                          // stages the loader has filled

    pdl_launch_dependents();
    if (tid == 0) {
        for (int s = 0; s < p.abuf; ++s) { mbar_init(smem_u32(&S->afull[s]), WN_FILL); mbar_init(smem_u32(&S->aempty[s]), 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(smem_u32(&S->dfull[s]), 1); mbar_init(smem_u32(&S->dempty[s]), WN_FILL); }
        mbar_init(smem_u32(&S->done), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 8) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&S->tmem_base)), "r"(p.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == WN_FILL + 32) {
        S->fail = 0; S->exact = 0;
        for (int s = 0; s < p.stages; ++s) { mbar_init(smem_u32(&S->bfull[s]), 1); mbar_init(smem_u32(&S->bempty[s]), 1); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // ---- the tile's rows, and the windows' tables.  All that is no predecessor's work comes before the wait for them: a dense
    // pass that overlaps its predecessor's tail then has its barriers, tensor memory, all planes' tables and first filters at
    // hand when the inputs arrive.  Delta tables are made of the input's activity bitmap: here the first plane's, on its way
    // together with the update bitmap, and the others' once the tile has work
    int active = 0;
    auto other_tables = [&] {
        if (!XCOL && p.all_tables) for (int b = plane0 + 1; b * p.nchb < b1; ++b) wn_table<DENSE, XCOL>(p, in_act, S->tab + (b - plane0) * p.span, lin0, b);
    };
    {
        int q = -1;
        uint32_t word = 0;                                   // of the layer's update bitmap
        if (tid < WN_FILL) {
            if (tid < p.mt * TC_M) {
                const int hwq = p.Hq * p.Wq;
                const int lin = lin0 + tid, img = wn_div(lin, p.div_img), rem = lin - img * hwq, oy = wn_div(rem, p.div_row), ox = rem - oy * p.Wq;
                if (img < p.n && oy < p.oh && ox < p.ow) q = (img * p.oh + oy) * p.ow + ox;
                if (DENSE) S->q[tid] = q;
            }
            if (!DENSE) {
                pdl_wait();                                  // bitmaps and inputs are the predecessors' work
                if (q >= 0) word = oact[q >> 5];             // (on its way together with the table's words)
            }
            wn_table<DENSE, XCOL>(p, in_act, S->tab, lin0, plane0);
            if (DENSE) other_tables();
            if (ACT && tid < p.bn) S->bias[tid] = p.bias && ntile * p.bn + tid < p.c_out ? reinterpret_cast<const int*>(p.bias)[ntile * p.bn + tid] : 0;
        }
        if (!DENSE || p.count_bitmap) {
            if (DENSE && tid < WN_FILL) {
                pdl_wait();
                if (q >= 0) word = p.count_bitmap[q >> 5];
            }
            const bool bit = q >= 0 && (word >> (q & 31) & 1u);
            if (!DENSE && tid < p.mt * TC_M) S->q[tid] = bit ? q : -1;
            tc_fence_before();
            active = __syncthreads_count(bit);
        } else {
            tc_fence_before();
            __syncthreads();
            if (warp != 9) pdl_wait();                       // (the filters are constants: their warp waits when the ring is full)
        }
        tc_fence_after();
        if (active && tid == 0 && ntile == 0 && split == 0) {
            int* oc = shift_bytes(p.ocount, arena_off);
            atomicAdd(oc, active);
            atomicAdd(oc + 1, p.mt);                         // accumulator tiles with work (dense inside a delta step: that a delta would have)
        }
    }
    const uint32_t tmem = S->tmem_base;
    if (!DENSE && active == 0) {                             // nothing to update (every share of the tile sees the same)
        if (warp == 8)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(p.tmem_cols) : "memory");
        return;
    }
    // this thread's accumulator rows and columns: with two tiles each warpgroup drains one, else each half of the columns
    const int wg = warp >> 2, m_own = p.mt > 1 ? wg : 0;
    const int c_lo = p.mt > 1 ? 0 : wg * 64, c_hi = p.mt > 1 ? p.bn : min(p.bn, c_lo + 64);
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    float facc[DT == T_F32 ? 64 : 1];                        // fp32 (one tile per CTA): the promoted sums of this thread's half row

    if (warp < 8) {
        // ================= windows
        if (DT == T_F32) {
            #pragma unroll
            for (int j = 0; j < 64; ++j) facc[j] = 0.f;
        }
        auto promote = [&](int ib) -> bool {                 // adds the leading accumulator of block ib to the registers and gives it back
            if (DT != T_F32) return true;
            const int pb = ib & 1;
            bool got = mbar_wait(smem_u32(&S->dfull[pb]), (ib >> 1) & 1, p.wait_limit);
            got = __all_sync(0xffffffffu, got);
            if (!got) return false;
            tc_fence_after();
            #pragma unroll
            for (int c0 = 0; c0 < 64; c0 += 32) {
                if (c_lo + c0 < c_hi) {
                    uint32_t v[32];
                    wn_ld32(tmem + lane_base + (uint32_t)(pb * p.bn + c_lo + c0), v);
                    #pragma unroll
                    for (int j = 0; j < 32; ++j) facc[DT == T_F32 ? c0 + j : 0] += __uint_as_float(v[j]);
                }
            }
            tc_fence_before();
            mbar_arrive(smem_u32(&S->dempty[pb]));
            return true;
        };
        if (!DENSE && !XCOL && p.all_tables && (plane0 + 1) * p.nchb < b1) {   // (now that the tile has work)
            other_tables();
            wn_meet();
        }
        static_assert(!ASYNC || (DT == T_I8 && !XCOL));
        const bool lag = ASYNC && p.abuf > 1;                // asynchronous copies: a block is handed over when the next one is on its way
        const int* src = S->tab;                             // the plane's table
        const int* const xcol0 = S->tab + WN_MAX_SPAN;
        int plane = plane0, chb = b0 - plane0 * p.nchb, ib = 0, buf = -1;
        uint32_t phase = 0;                                  // of aempty: the ring's first filling waits for nobody
        for (int b = b0; b < b1; ++b, ++ib) {
            if (++buf == p.abuf) { buf = 0; phase ^= 1; }
            if (ib >= p.abuf || p.wait_limit == 0) {
                ok = mbar_wait(smem_u32(&S->aempty[buf]), phase ^ 1, p.wait_limit) && *(volatile int*)&S->fail == 0;
                if (!wn_agree(ok)) { ok = false; break; }
            }
            const bool new_plane = ib > 0 && chb == p.nchb;
            if (chb == p.nchb) { chb = 0; ++plane; }
            const int g0 = chb * p.gblk, gn = min(p.gblk, p.groups - g0), ry = XCOL ? p.plane[plane].ry : 0;
            if (!XCOL && new_plane) {
                if (p.all_tables) src += p.span;
                else {
                    wn_meet();                               // (everyone is done with the last plane's)
                    wn_table<DENSE, XCOL>(p, in_act, S->tab, lin0, plane);
                    wn_meet();
                }
            }
            ++chb;
            const uint32_t Ab = base_u32 + buf * p.abytes;
            unsigned char* Ap = base + buf * p.abytes;
            const int arrays = XCOL && p.xarr ? p.xarr : gn * 2;               // of p.L slots each
            const int cl = XCOL && DT == T_I8 && !p.xarr ? (p.kw + 3) >> 2 : arrays;      // 16-byte chunks to copy per pixel
            const uint32_t piece = (uint32_t)(arrays * p.L) * 16u;              // bytes between the fp32 pieces' windows
            const unsigned magic = cl > 1 ? (unsigned)(((1ull << 32) + cl - 1) / cl) : 0u;
            const int items = p.span * cl;
            if (DT == T_I8 && !XCOL && !ASYNC) {
                // Dense blocks are full: through registers, a turn's loads all on their way before its first store.  (Asynchronous
                // copies, handed over when the next block's are on their way, take 2.3 to 3 k clocks a block: 24 AlexNet-shaped
                // keyframes 97.2 -> 93.2 us, 4 ResNet-18-shaped streams 188.9 -> 181.8.)
                const unsigned char* src0 = reinterpret_cast<const unsigned char*>(A) + g0 * 32;
                constexpr int TURN = 6;
                #pragma unroll 1
                for (int idx = tid; idx < items; idx += TURN * WN_FILL) {
                    uint4 v[TURN];
                    #pragma unroll
                    for (int u = 0; u < TURN; ++u) {
                        const int id = idx + u * WN_FILL, i = magic ? (int)__umulhi((unsigned)id, magic) : id, c = id - i * cl;
                        const int off = id < items ? src[i] : -1;
                        v[u] = make_uint4(0, 0, 0, 0);
                        if (off >= 0) v[u] = __ldcg(reinterpret_cast<const uint4*>(src0 + off + c * 16));
                    }
                    #pragma unroll
                    for (int u = 0; u < TURN; ++u) {
                        const int id = idx + u * WN_FILL, i = magic ? (int)__umulhi((unsigned)id, magic) : id, c = id - i * cl;
                        if (id < items) *reinterpret_cast<uint4*>(Ap + (size_t)(c * p.L + i) * 16) = v[u];
                    }
                }
                fence_async_smem();
                mbar_arrive(smem_u32(&S->afull[buf]));
            } else if (DT == T_I8 && !XCOL) {
                // asynchronous copies: delta rows (one frame's steps, one small block per CTA: 64.2 us against 65.8 through
                // registers), and dense passes of many short blocks (win_async_windows)
                const unsigned char* src0 = reinterpret_cast<const unsigned char*>(A) + g0 * 32;
                #pragma unroll 4
                for (int idx = tid; idx < items; idx += WN_FILL) {
                    const int i = magic ? (int)__umulhi((unsigned)idx, magic) : idx, c = idx - i * cl;
                    const int off = src[i];
                    cp_async16(Ab + (uint32_t)(c * p.L + i) * 16u, off >= 0 ? src0 + off + c * 16 : src0, off >= 0 ? 16u : 0u);
                }
                cp_async_commit();
                if (!lag) {
                    cp_async_wait<0>();
                    fence_async_smem();
                    mbar_arrive(smem_u32(&S->afull[buf]));
                } else if (ib > 0) {
                    cp_async_wait<1>();
                    fence_async_smem();
                    mbar_arrive(smem_u32(&S->afull[buf > 0 ? buf - 1 : p.abuf - 1]));
                }
            } else if (DT == T_I8) {
                // first layer, a 4-byte word per pixel: four neighbouring pixels of an image row are one chunk
                const uint32_t* Aw = reinterpret_cast<const uint32_t*>(A);
                auto fetch = [&](int idx, uint32_t (&v)[4]) {
                    const int i = magic ? (int)__umulhi((unsigned)idx, magic) : idx, c = idx - i * cl;
                    const int row0 = src[i], xl = xcol0[i], row = row0 + ry * p.w, x = (xl >> 8) + 4 * c;
                    v[0] = v[1] = v[2] = v[3] = 0u;
                    if (row0 < 0 || ry >= (xl & 255)) return;
                    unsigned bits = 0xfu;                    // which of the four pixels count
                    if (!DENSE) {
                        const int g = max(row + x, 0), sh = g & 31;
                        unsigned long long two = in_act[g >> 5];
                        if (sh > 28 && row + p.w > ((g >> 5) + 1) * 32) two |= (unsigned long long)in_act[(g >> 5) + 1] << 32;
                        bits = (unsigned)(two >> sh);
                        if (row + x < 0) bits <<= -(row + x);
                    }
                    #pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (x + e >= 0 && x + e < p.w && (bits >> e & 1u)) v[e] = Aw[row + x + e];
                };
                // (a turn's loads are all on their way before its first store: the compiler does not move them across)
                for (int idx = tid; idx < items; idx += 2 * WN_FILL) {
                    uint32_t v[2][4];
                    fetch(idx, v[0]);
                    const bool two = idx + WN_FILL < items;
                    if (two) fetch(idx + WN_FILL, v[1]);
                    #pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        if (u > 0 && !two) break;
                        const int id = idx + u * WN_FILL, i = magic ? (int)__umulhi((unsigned)id, magic) : id, c = id - i * cl;
                        *reinterpret_cast<uint4*>(Ap + (size_t)(c * p.L + i) * 16) = make_uint4(v[u][0], v[u][1], v[u][2], v[u][3]);
                    }
                }
                fence_async_smem();
                mbar_arrive(smem_u32(&S->afull[buf]));
            } else if (DT == T_BIN) {
                // bits -> bytes: +2 / -2 per changed channel (dense: +1 / -1), 0 beyond the channels and outside the image
                const uint32_t* Cu = reinterpret_cast<const uint32_t*>(A) + g0;
                const uint32_t* Nu = reinterpret_cast<const uint32_t*>(Anew) + g0;
                // (a turn's loads are all on their way before its first store: the compiler does not move them across)
                for (int idx = tid; idx < items; idx += 4 * WN_FILL) {
                    uint32_t nw[4], cw4[4];
                    int off[4];
                    #pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int id = idx + u * WN_FILL, i = (int)__umulhi((unsigned)id, magic), c = id - i * cl;      // (cl >= 2)
                        off[u] = id < items ? src[i] : -1;
                        if (off[u] >= 0) {
                            nw[u] = Nu[off[u] + (c >> 1)];
                            if (!DENSE) cw4[u] = Cu[off[u] + (c >> 1)];
                        }
                    }
                    #pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int id = idx + u * WN_FILL, i = (int)__umulhi((unsigned)id, magic), c = id - i * cl;
                        if (id >= items) break;
                        uint4 v = make_uint4(0, 0, 0, 0);
                        if (off[u] >= 0) {
                            const int ch0 = (g0 * 2 + c) * 16;
                            const uint32_t valid = ch0 >= p.c_in ? 0u : (ch0 + 16 > p.c_in ? (1u << (p.c_in - ch0)) - 1u : 0xffffu);
                            const int sh = (c & 1) * 16;
                            const uint32_t nb = nw[u] >> sh;
                            uint32_t pos, neg;
                            if (DENSE) { pos = nb & valid; neg = ~nb & valid; }
                            else { const uint32_t ch = (cw4[u] >> sh) & valid; pos = ch & nb; neg = ch & ~nb; }
                            const uint32_t pm = DENSE ? 0x01u : 0x02u, nm = DENSE ? 0xffu : 0xfeu;
                            v.x = wn_spread4(pos) * pm + wn_spread4(neg) * nm;
                            v.y = wn_spread4(pos >> 4) * pm + wn_spread4(neg >> 4) * nm;
                            v.z = wn_spread4(pos >> 8) * pm + wn_spread4(neg >> 8) * nm;
                            v.w = wn_spread4(pos >> 12) * pm + wn_spread4(neg >> 12) * nm;
                        }
                        *reinterpret_cast<uint4*>(Ap + (size_t)(c * p.L + i) * 16) = v;
                    }
                }
                fence_async_smem();
                mbar_arrive(smem_u32(&S->afull[buf]));
            } else {
                const float* Af = reinterpret_cast<const float*>(A);
                const bool vec = (p.row_units & 3) == 0;
                uint32_t thirds = 0;                         // sums of the third pieces
                auto fetch = [&](int idx, float (&x)[8]) {
                    const int i = magic ? (int)__umulhi((unsigned)idx, magic) : idx, c = idx - i * cl;
                    const int off = src[i];
                    #pragma unroll
                    for (int j = 0; j < 8; ++j) x[j] = 0.f;
                    if (XCOL) {
                        // two neighbouring pixels x 4 channels
                        const int xl = xcol0[i], xx = (xl >> 8) + 2 * (g0 * 2 + c);
                        if (off < 0 || ry >= (xl & 255)) return;
                        #pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int pix = off + ry * p.w + xx + e;
                            if (xx + e >= 0 && xx + e < p.w && (DENSE || ((in_act[pix >> 5] >> (pix & 31)) & 1u))) {
                                #pragma unroll
                                for (int ch = 0; ch < 4; ++ch) if (ch < p.c_in) x[e * 4 + ch] = Af[(size_t)pix * p.row_units + ch];
                            }
                        }
                    } else if (off >= 0) {
                        const int ch0 = (g0 * 2 + c) * 8;
                        if (vec) {
                            if (ch0 < p.c_in) { const float4 t = *reinterpret_cast<const float4*>(Af + off + ch0); x[0] = t.x; x[1] = t.y; x[2] = t.z; x[3] = t.w; }
                            if (ch0 + 4 < p.c_in) { const float4 t = *reinterpret_cast<const float4*>(Af + off + ch0 + 4); x[4] = t.x; x[5] = t.y; x[6] = t.z; x[7] = t.w; }
                        } else {
                            #pragma unroll
                            for (int j = 0; j < 8; ++j) if (ch0 + j < p.c_in) x[j] = Af[off + ch0 + j];
                        }
                    }
                };
                auto put = [&](int idx, const float (&x)[8]) {
                    const int i = magic ? (int)__umulhi((unsigned)idx, magic) : idx, c = idx - i * cl;
                    uint32_t s[3][4];
                    #pragma unroll
                    for (int j = 0; j < 4; ++j) wn_split(x[2 * j], x[2 * j + 1], s[0][j], s[1][j], s[2][j]);
                    #pragma unroll
                    for (int j = 0; j < 4; ++j) thirds = wn_bf16_add(thirds, s[2][j]);
                    unsigned char* dst = Ap + (size_t)(c * p.L + i) * 16;
                    #pragma unroll
                    for (int k = 0; k < 3; ++k) *reinterpret_cast<uint4*>(dst + k * piece) = make_uint4(s[k][0], s[k][1], s[k][2], s[k][3]);
                };
                // (a turn's loads are all on their way before its first store: the compiler does not move them across)
                constexpr int TURN = 3;
                for (int idx = tid; idx < items; idx += TURN * WN_FILL) {
                    float x[TURN][8];
                    #pragma unroll
                    for (int u = 0; u < TURN; ++u) if (idx + u * WN_FILL < items) fetch(idx + u * WN_FILL, x[u]);
                    #pragma unroll
                    for (int u = 0; u < TURN; ++u) if (idx + u * WN_FILL < items) put(idx + u * WN_FILL, x[u]);
                }
                fence_async_smem();
                mbar_arrive(smem_u32(&S->afull[buf]));
                if (wn_bf16_nan(thirds)) *(volatile int*)&S->exact = 1;
                if (ib > 0 && !promote(ib - 1)) { *(volatile int*)&S->fail = 1; ok = false; }
                // (a warp whose wait ran out says so when the warps meet at the next block)
            }
        }
        if (ASYNC) {
            cp_async_wait<0>();
            fence_async_smem();
            if (ok && lag && ib > 0) mbar_arrive(smem_u32(&S->afull[buf]));
        }
        if (DT == T_F32 && ok && ib > 0 && !promote(ib - 1)) ok = false;
    } else if (warp == 9) {
        // ================= filters: a stage's taps, one bulk copy each (one thread)
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 1;
            for (int b = b0; b < b1 && ok; ++b) {
                const int plane = b / p.nchb, chb = b - plane * p.nchb;
                const int g0 = chb * p.gblk, gn = min(p.gblk, p.groups - g0);
                const int nx = p.plane[plane].nx, ntap = p.plane[plane].ny * nx;
                const int t_end = p.tsplit > 1 ? (part + 1) * ntap / p.tsplit : ntap;
                int lt = p.tsplit > 1 ? part * ntap / p.tsplit : 0;
                const uint32_t bytes = unit_b * (uint32_t)gn, tap_bytes = (uint32_t)p.groups * unit_b;
                const int row_taps = XCOL ? 1 : p.kw;        // taps of a filter row
                const uint32_t step_x = tap_bytes * (uint32_t)p.stride, step_y = tap_bytes * (uint32_t)(row_taps * p.stride) - step_x * (uint32_t)(nx - 1);
                const int jy = lt / nx;
                int jx = lt - jy * nx;
                const unsigned char* src = p.Wimg + ((size_t)ntile * (row_taps * p.kh) * p.groups + g0) * unit_b +
                                           (size_t)((p.plane[plane].ky0 + jy * p.stride) * row_taps + p.plane[plane].kx0 + jx * p.stride) * tap_bytes;
                while (lt < t_end) {
                    if (DENSE && issued == p.stages) pdl_wait();      // (bounded waits are for this launch's own work, not for its predecessors')
                    if (!mbar_wait(smem_u32(&S->bempty[stage]), phase, p.wait_limit) || *(volatile int*)&S->fail) { ok = false; break; }
                    const int tn = min(p.tps, t_end - lt);
                    const uint32_t bar = smem_u32(&S->bfull[stage]);
                    mbar_arrive_expect_tx(bar, bytes * (uint32_t)tn);
                    uint32_t dst = bstage_u32 + stage * p.stage_bytes;
                    for (int t = 0; t < tn; ++t) {
                        bulk_copy_g2s(dst, src, bytes, bar);
                        dst += bytes;
                        if (++jx == nx) { jx = 0; src += step_y; } else src += step_x;
                    }
                    lt += tn;
                    ++issued;
                    if (++stage == p.stages) { stage = 0; phase ^= 1; }
                }
            }
        }
    } else {
        // ================= MMAs.  The whole warp walks and one elected lane issues.  What the walk costs is what the MMAs of
        // a stage have to be longer than: a step's MMAs are one block of instructions, and the next stage's barrier is polled
        // before this stage's MMAs are issued.
        const uint32_t e = wn_elect();
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
        auto wait = [&](unsigned long long* bar, uint32_t parity) -> bool { return __all_sync(0xffffffffu, mbar_wait(smem_u32(bar), parity, p.wait_limit)); };
        const uint32_t idesc = DT == T_F32 ? (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.bn >> 3) << 17) | ((uint32_t)(TC_M >> 4) << 24)
                                           : tc_instr_desc(p.bn);
        const uint32_t idesc2 = (idesc & ~(0x3fu << 17)) | ((uint32_t)(2 * p.bn >> 3) << 17);     // twice the columns
        // (everything below in 16-byte units)
        const uint32_t a_step = p.a_step, b_unit = unit_b >> 4, bn = (uint32_t)p.bn;
        const uint32_t stage_step = p.stage_bytes >> 4, b_lo0 = wn_desc_lo(bstage_u32, PIECES * bn);
        const uint32_t full0 = smem_u32(&S->bfull[0]), empty0 = smem_u32(&S->bempty[0]);
        int ib = 0, stage = 0, buf = 0;
        uint32_t phase = 0, a_phase = 0, b_stage = b_lo0;
        uint32_t first = 0;                                  // 0 until the CTA's first MMA has been issued
        bool ready = false;                                  // the coming stage has been seen full
        for (int b = b0; b < b1 && ok; ++b, ++ib) {
            const int plane = b / p.nchb, chb = b - plane * p.nchb;
            const int gn = min(p.gblk, p.groups - chb * p.gblk);
            const int nx = p.plane[plane].nx, ntap = p.plane[plane].ny * nx;
            const int t_lo = p.tsplit > 1 ? part * ntap / p.tsplit : 0, t_hi = p.tsplit > 1 ? (part + 1) * ntap / p.tsplit : ntap;
            const int jy = t_lo / nx;
            int j = t_lo - jy * nx;
            if (!wait(&S->afull[buf], a_phase)) { ok = false; break; }
            // fp32: two leading accumulators in turn; this one has to have been drained of the block before the last
            if (DT == T_F32 && !wait(&S->dempty[ib & 1], ((ib >> 1) & 1) ^ 1)) { ok = false; break; }
            const uint32_t a_piece = (uint32_t)((XCOL && p.xarr ? p.xarr : gn * 2) * p.L);
            const uint32_t row_jump = (uint32_t)(p.Wq - nx + 1);
            uint32_t a_tap = wn_desc_lo(base_u32 + buf * p.abytes, p.a_lbo) + (uint32_t)(p.plane[plane].shift0 - p.min_shift + jy * p.Wq + j);
            const uint32_t d0 = tm + (DT == T_F32 ? (uint32_t)(ib & 1) * bn : 0u), d1 = tm + (DT == T_F32 ? 2u * bn : bn);   // (fp32: d1 the small products)
            uint32_t fresh = 0;                              // fp32: 0 until the block's first MMA
            for (int t0 = t_lo; t0 < t_hi; t0 += p.tps) {
                if (!ready && !__all_sync(0xffffffffu, mbar_wait(full0 + 8u * stage, phase, p.wait_limit))) { ok = false; break; }
                tc_fence_after();
                const uint32_t done_bar = empty0 + 8u * stage;
                uint32_t b_lo = b_stage;
                b_stage += stage_step;
                if (++stage == p.stages) { stage = 0; phase ^= 1; b_stage = b_lo0; }
                const uint32_t poll = DT == T_F32 ? mbar_poll(full0 + 8u * stage, phase) : 0u;
                for (int tn = min(p.tps, t_hi - t0); tn > 0; --tn) {
                    uint32_t a_lo = a_tap;
                    #pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        if (g >= gn) break;
                        if (DT == T_F32) wn_step_f32(d0, d1, d1 + bn, a_lo, a_lo + a_piece, a_lo + 2 * a_piece, b_lo, b_lo + bn, idesc, idesc2, fresh, first, e);
                        else {
                            wn_step_i8(d0, a_lo, b_lo, idesc, g == 0 ? first : 1u, e);
                            if (p.mt > 1) wn_step_i8(d1, a_lo + TC_M, b_lo, idesc, g == 0 ? first : 1u, e);
                        }
                        fresh = 1;
                        if (DT == T_F32) first = 1;
                        a_lo += a_step;
                        b_lo += b_unit;
                    }
                    first = 1;
                    if (++j == nx) { j = 0; a_tap += row_jump; } else ++a_tap;
                }
                wn_commit(done_bar, e);
                ready = DT == T_F32 && __all_sync(0xffffffffu, poll != 0);
            }
            if (!ok) break;
            wn_commit(smem_u32(&S->aempty[buf]), e);
            if (DT == T_F32) wn_commit(smem_u32(&S->dfull[ib & 1]), e);
            if (++buf == p.abuf) { buf = 0; a_phase ^= 1; }
        }
        if (ok) wn_commit(smem_u32(&S->done), e);
        else if (first) {
            // giving up with MMAs issued: they must have completed before the tensor memory is freed
            *(volatile int*)&S->fail = 1;
            __threadfence_block();
            wn_commit(smem_u32(&S->done), e);
            mbar_wait(smem_u32(&S->done), 0, WAIT_LIMIT_DEFAULT);
        }
    }
    if (!ok) { *(volatile int*)&S->fail = 1; atomicOr(p.errw, ERRW_TIMEOUT); }

    // ================= accumulators out, through shared memory where rows have to be turned around (the windows are done with)
    const int n0 = ntile * p.bn, ncols = min(p.bn, p.c_out - n0);
    const bool halves = p.mt > 1 && p.bn > 64;               // two tiles: 64 columns at a time, so that both fit
    const int cw = halves ? 64 : p.bn;                       // columns per pass
    const int ldr = cw + 4;                                  // words per staged row (16-byte aligned, staggered over the banks)
    const int ldt = min(p.bn, WN_TURN) + 4;                  // ... where a warp turns its rows around by itself
    const bool vec = (p.c_out & 3) == 0;
    const bool adds = !DENSE && !p.store;                    // delta: onto the stored projection
    const bool bulk_add = adds && vec && !p.cluster;         // ... by the copy engine, a row per thread (exact in any order for integers,
                                                             // one share only for fp32)
    uint32_t* staged = reinterpret_cast<uint32_t*>(base);
    if (warp < 8) {
        if (ok && !mbar_wait(smem_u32(&S->done), 0, p.wait_limit)) { ok = false; *(volatile int*)&S->fail = 1; atomicOr(p.errw, ERRW_TIMEOUT); }
        ok = wn_agree(ok && *(volatile int*)&S->fail == 0);   // nobody stores results of a tile that gave up
        tc_fence_after();
    }
    if (DT == T_F32 && warp < 8 && ok && *(volatile int*)&S->exact) {         // (the same for all of them)
        const int r = (warp & 3) * 32 + lane;
        float* sums = reinterpret_cast<float*>(base) + (size_t)r * (p.bn + 1);   // (odd rows; fewer words than the drained rows')
        wn_exact_row<DENSE, XCOL>(p, reinterpret_cast<const float*>(A), in_act, S->q[r] >= 0 ? lin0 + r : -1, ntile, b0, b1, c_lo, c_hi, sums);
        #pragma unroll
        for (int j = 0; j < 64; ++j) facc[DT == T_F32 ? j : 0] = c_lo + j < c_hi ? sums[c_lo + j] : 0.f;
        __syncwarp();
        #pragma unroll 1
        for (int k = 0; k < 64 && c_lo + k < c_hi; k += 32) {                  // nothing is added to them
            wn_zero32(tmem + lane_base + (uint32_t)(2 * p.bn + c_lo + k));
            wn_zero32(tmem + lane_base + (uint32_t)(3 * p.bn + c_lo + k));
        }
        wn_meet();                                           // everyone has read its sums: the rows may be written over
    }
    const bool direct = ACT && DT != T_F32 && !p.cluster;    // f straight from the accumulator registers
    if (ACT && DT != T_F32 && direct && warp < 8 && ok) {
        const int r = m_own * TC_M + (warp & 3) * 32 + lane;
        const int q = S->q[r];
        const bool keep = q >= p.keep_from;                  // (q >= 0 then)
        uint32_t* mine = staged + (size_t)warp * 32 * ldt;   // (the warp's rows, where projections are kept)
        const bool any_keep = __any_sync(0xffffffffu, keep);
        // (a loop, not unrolled: every CTA runs this code once, so its length is instruction fetches)
        #pragma unroll 1
        for (int cc = c_lo; cc < c_hi; cc += 32) {
            const bool inside = q >= 0 && n0 + cc < (p.bits ? p.cs * 32 : p.cs);
            uint4 rw[2] = {make_uint4(0, 0, 0, 0), make_uint4(0, 0, 0, 0)};
            if (p.res && inside) {
                const uint4* src = reinterpret_cast<const uint4*>(reinterpret_cast<const int8_t*>(p.res) + (size_t)q * p.cs + n0 + cc);
                rw[0] = src[0]; rw[1] = src[1];
            }
            uint32_t v[32];
            __syncwarp();
            wn_ld32(tmem + lane_base + (uint32_t)(m_own * p.bn + cc), v);
            #pragma unroll
            for (int j = 0; j < 32; j += 4) {
                const int4 b = *reinterpret_cast<const int4*>(S->bias + cc + j);
                v[j] += (uint32_t)b.x; v[j + 1] += (uint32_t)b.y; v[j + 2] += (uint32_t)b.z; v[j + 3] += (uint32_t)b.w;
            }
            if (any_keep) {
                // the projection leaves as whole lines, eight lanes a row.  (Row by row through the copy engine, 128 bytes a copy:
                // 9 to 18 clocks each, 4.6 to 9.4 k of a keyframe CTA's 14 to 38 k)
                #pragma unroll
                for (int j = 0; j < 32; j += 4) *reinterpret_cast<uint4*>(mine + lane * ldt + j) = make_uint4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                __syncwarp();
                const int c4 = (lane & 7) * 4, left = ncols - cc - c4;
                #pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int rr = i * 4 + (lane >> 3), qq = __shfl_sync(0xffffffffu, q, rr);
                    if (qq < p.keep_from || left <= 0) continue;
                    const uint4 t = *reinterpret_cast<const uint4*>(mine + rr * ldt + c4);
                    uint32_t* dst = reinterpret_cast<uint32_t*>(P) + (size_t)(qq - p.keep_from) * p.c_out + n0 + cc + c4;
                    if (vec) *reinterpret_cast<uint4*>(dst) = t;
                    else {
                        dst[0] = t.x;
                        if (left > 1) dst[1] = t.y;
                        if (left > 2) dst[2] = t.z;
                        if (left > 3) dst[3] = t.w;
                    }
                }
            }
            if (!inside) continue;
            if (p.bits) {
                uint32_t word = 0;
                #pragma unroll
                for (int j = 0; j < 32; ++j) word |= (uint32_t)((int)v[j] >= p.theta) << j;
                if (ncols - cc < 32) word &= (1u << max(ncols - cc, 0)) - 1u;
                reinterpret_cast<uint32_t*>(p.X)[(size_t)q * p.cs + ((n0 + cc) >> 5)] = word;
            } else {
                const uint32_t rr[8] = {rw[0].x, rw[0].y, rw[0].z, rw[0].w, rw[1].x, rw[1].y, rw[1].z, rw[1].w};
                uint32_t o[8];
                if (!p.bn_scale) {
                    const int rnd = p.shift > 0 ? 1 << (p.shift - 1) : 0, sh = p.shift, lo = p.act_fn == RRM_ACT_RELU ? 0 : -127;
                    if (!p.res) {
                        #pragma unroll
                        for (int j = 0; j < 8; ++j)
                            o[j] = wn_pack4(max(((int)v[4 * j] + rnd) >> sh, lo), max(((int)v[4 * j + 1] + rnd) >> sh, lo),
                                            max(((int)v[4 * j + 2] + rnd) >> sh, lo), max(((int)v[4 * j + 3] + rnd) >> sh, lo));
                    } else {
                        #pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const int x[4] = {(int)v[4 * j], (int)v[4 * j + 1], (int)v[4 * j + 2], (int)v[4 * j + 3]};
                            o[j] = wn_f8_plain(x, rr[j], rnd, sh, lo, true);
                        }
                    }
                } else {
                    #pragma unroll
                    for (int j = 0; j < 8; ++j) o[j] = wn_f8_bn(p, n0 + cc + 4 * j, (int)v[4 * j], (int)v[4 * j + 1], (int)v[4 * j + 2], (int)v[4 * j + 3], rr[j]);
                }
                uint4* dst = reinterpret_cast<uint4*>(reinterpret_cast<int8_t*>(p.X) + (size_t)q * p.cs + n0 + cc);
                dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
                dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
            }
        }
    }
    // one value group of 4 neighbouring channels (c: column of the tile) of projection pixel q leaves: f and the output row
    // (ACT), the projection where it is kept.  Every lane of a warp comes here (signs are put together by shuffles).
    auto emit = [&](int q, int c, const uint32_t (&o)[4]) {
        const int ch = n0 + c;
        if (ACT && DT != T_F32 && p.bits) {
            uint32_t word = 0;
            #pragma unroll
            for (int j = 0; j < 4; ++j) if (c + j < ncols && (int)o[j] >= p.theta) word |= 1u << (4 * (lane & 7) + j);
            word |= __shfl_xor_sync(0xffffffffu, word, 1);
            word |= __shfl_xor_sync(0xffffffffu, word, 2);
            word |= __shfl_xor_sync(0xffffffffu, word, 4);
            if (q >= 0 && (lane & 7) == 0 && c < p.bn && (ch >> 5) < p.cs) reinterpret_cast<uint32_t*>(p.X)[(size_t)q * p.cs + (ch >> 5)] = word;
        } else if (ACT && DT != T_F32) {
            if (q >= 0 && c < p.bn && ch < p.cs) {           // (channels up to the padded width get a value too)
                const size_t at = (size_t)q * p.cs + ch;
                const int x[4] = {(int)o[0], (int)o[1], (int)o[2], (int)o[3]};
                const uint32_t res = p.res ? *reinterpret_cast<const uint32_t*>(reinterpret_cast<const int8_t*>(p.res) + at) : 0u;
                *reinterpret_cast<uint32_t*>(reinterpret_cast<int8_t*>(p.X) + at) = wn_f8(p, ch, x, res);
            }
        } else if (ACT) {
            if (q >= 0 && c < ncols) {
                const size_t at = (size_t)q * p.cs + ch;
                float4 y = make_float4(__uint_as_float(o[0]), __uint_as_float(o[1]), __uint_as_float(o[2]), __uint_as_float(o[3]));
                if (p.bn_scale || p.res) y = wn_f32_slow(p, ch, ncols - c, at, y);
                else if (p.act_fn != RRM_ACT_NONE) {
                    const float leak = 0.1f;
                    const bool relu = p.act_fn == RRM_ACT_RELU;
                    y.x = y.x > 0 ? y.x : (relu ? 0.f : leak * y.x); y.y = y.y > 0 ? y.y : (relu ? 0.f : leak * y.y);
                    y.z = y.z > 0 ? y.z : (relu ? 0.f : leak * y.z); y.w = y.w > 0 ? y.w : (relu ? 0.f : leak * y.w);
                }
                float* dst = reinterpret_cast<float*>(p.X) + at;
                if (vec) *reinterpret_cast<float4*>(dst) = y;
                else {
                    dst[0] = y.x;
                    if (c + 1 < ncols) dst[1] = y.y;
                    if (c + 2 < ncols) dst[2] = y.z;
                    if (c + 3 < ncols) dst[3] = y.w;
                }
            }
        }
        if (q < (ACT ? p.keep_from : 0) || c >= ncols) return;
        uint32_t* dst = reinterpret_cast<uint32_t*>(P) + (size_t)(q - (ACT ? p.keep_from : 0)) * p.c_out + ch;
        if (vec) *reinterpret_cast<uint4*>(dst) = make_uint4(o[0], o[1], o[2], o[3]);
        else {
            #pragma unroll
            for (int j = 0; j < 4; ++j) if (c + j < ncols) dst[j] = o[j];
        }
    };
    auto plus = [](uint32_t a, uint32_t b) -> uint32_t { return DT == T_F32 ? __float_as_uint(__uint_as_float(a) + __uint_as_float(b)) : a + b; };
    // what the sums are added to: the bias (dense), the stored projection (delta)
    auto base_of = [&](int q, int c, uint32_t (&o)[4]) {
        o[0] = o[1] = o[2] = o[3] = 0;
        if (q < 0 || c >= ncols || !(adds || (DENSE && p.bias))) return;
        const uint32_t* from = (adds ? reinterpret_cast<const uint32_t*>(P) + (size_t)q * p.c_out : reinterpret_cast<const uint32_t*>(p.bias)) + n0 + c;
        if (vec) { const uint4 w = *reinterpret_cast<const uint4*>(from); o[0] = w.x; o[1] = w.y; o[2] = w.z; o[3] = w.w; }
        else {
            #pragma unroll
            for (int j = 0; j < 4; ++j) if (c + j < ncols) o[j] = from[j];
        }
    };
    // this thread's accumulator row, up to 64 columns from column cb of the tile on, into shared memory.  (fp32: all of the
    // thread's columns, completed from the promoted sums and the two accumulators of small products)
    auto put_row = [&](int cb, uint32_t* row) {
        #pragma unroll (DT == T_F32 ? 2 : 1)
        for (int k = 0; k < 64; k += 32) {
            const int cc = cb + k;
            if (cc >= c_hi) continue;                        // (the same in all lanes)
            uint32_t v[32];
            __syncwarp();
            if (DT == T_F32) {
                wn_ld32(tmem + lane_base + (uint32_t)(3 * p.bn + cc), v);
                #pragma unroll
                for (int j = 0; j < 32; ++j) facc[DT == T_F32 ? k + j : 0] = fmaf(__uint_as_float(v[j]), 1.f / (WN_SCALE * WN_SCALE), facc[DT == T_F32 ? k + j : 0]);
            }
            wn_ld32(tmem + lane_base + (uint32_t)((DT == T_F32 ? 2 : m_own) * p.bn + cc), v);
            if (DT == T_F32) {
                #pragma unroll
                for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(fmaf(__uint_as_float(v[j]), 1.f / WN_SCALE, facc[DT == T_F32 ? k + j : 0]));
            }
            #pragma unroll
            for (int j = 0; j < 32; j += 4) if (cc + j < c_hi) *reinterpret_cast<uint4*>(row + k + j) = make_uint4(v[j], v[j + 1], v[j + 2], v[j + 3]);
        }
    };
    if (!direct && !p.cluster && !bulk_add) {
        // one share: a warp turns its 32 rows around in shared memory of its own, 64 columns at a time (16 lanes a row, or 8
        // where the tile has no more columns: whole lines), without a barrier of the CTA.  The loop over the rows is short on
        // purpose: every CTA runs this code once, and an unrolled form cost its length in instruction fetches
        if (warp < 8 && ok) {
            uint32_t* mine = staged + (size_t)warp * 32 * ldt;
            const int q_own = S->q[m_own * TC_M + (warp & 3) * 32 + lane];
            const bool narrow = p.bn <= 32;
            const int sub = narrow ? lane >> 3 : lane >> 4, step = narrow ? 4 : 2, c4 = (narrow ? lane & 7 : lane & 15) * 4;
            #pragma unroll 1
            for (int cb = c_lo; cb < c_hi; cb += WN_TURN) {
                put_row(cb, mine + lane * ldt);
                __syncwarp();
                uint32_t base4[4] = {0, 0, 0, 0};
                if (!adds) base_of(0, cb + c4, base4);       // (the bias: the same for every row)
                #pragma unroll 1
                for (int r0 = sub; r0 < 32; r0 += 4 * step) {
                    uint32_t o[4][4];
                    int q[4];
                    #pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        q[i] = __shfl_sync(0xffffffffu, q_own, r0 + i * step);
                        if (cb + c4 >= c_hi) q[i] = -1;
                        if (adds) base_of(q[i], cb + c4, o[i]);
                        else { o[i][0] = base4[0]; o[i][1] = base4[1]; o[i][2] = base4[2]; o[i][3] = base4[3]; }
                    }
                    #pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint4 t = *reinterpret_cast<const uint4*>(mine + (r0 + i * step) * ldt + c4);
                        o[i][0] = plus(o[i][0], t.x); o[i][1] = plus(o[i][1], t.y); o[i][2] = plus(o[i][2], t.z); o[i][3] = plus(o[i][3], t.w);
                        emit(q[i], cb + c4, o[i]);
                    }
                }
                __syncwarp();
            }
        }
    } else if (!direct && !p.cluster) {
        // every share adds its rows onto the projection by itself, through the copy engine
        #pragma unroll 1
        for (int pass = 0; pass < (halves ? 2 : 1); ++pass) {
            const int p0 = pass * 64;                        // first column of the pass
            if (warp < 8 && ok) {
                const int r = m_own * TC_M + (warp & 3) * 32 + lane;
                uint32_t* row = staged + (size_t)r * ldr;
                const int lo = halves ? p0 : c_lo, hi = halves ? min(p0 + 64, c_hi) : c_hi;
                for (int cb = lo; cb < hi; cb += 64) put_row(cb, row + cb - p0);
                const int q = S->q[r], end = min(hi, ncols);
                fence_async_smem();                          // this thread's part of the row -> visible to the copy engine
                if (q >= 0 && end > lo) {
                    char* dst = reinterpret_cast<char*>(P) + ((size_t)q * p.c_out + n0 + lo) * 4;
                    if (DT == T_F32)
                        asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], %2;"
                                     ::"l"(dst), "r"(smem_u32(row + lo - p0)), "r"((uint32_t)(end - lo) * 4u) : "memory");
                    else
                        asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.s32 [%0], [%1], %2;"
                                     ::"l"(dst), "r"(smem_u32(row + lo - p0)), "r"((uint32_t)(end - lo) * 4u) : "memory");
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                }
            }
        }
    } else if (p.cluster) {
        if (warp < 8 && ok) {
            if (c_lo < c_hi) put_row(c_lo, staged + (size_t)((warp & 3) * 32 + lane) * ldr + c_lo);
            // rows split, split + ks, ... of the tile, two at a time per warp (half a warp where the tile has up to 64
            // columns, a quarter up to 32); of four shares' rows at a time all reads are in flight together, added in the
            // order of the shares
            const int lpr = p.bn > 64 ? 5 : (p.bn > 32 ? 4 : 3);                 // (log2 of the lanes of a row)
            const int team = lane >> lpr, c = (lane & ((1 << lpr) - 1)) * 4;
            constexpr int NR = 2, NS = 4;
            uint32_t base4[4] = {0, 0, 0, 0};
            if (!adds) base_of(0, c, base4);                 // (the bias: the same for every row)
            wn_cluster_meet();                               // every share's partial tile is in its shared memory
            #pragma unroll 1
            for (int kb = warp * (32 >> lpr) * NR; split + kb * p.ks < TC_M; kb += 8 * (32 >> lpr) * NR) {
                const int k0 = kb + team * NR;
                uint32_t o[NR][4];
                int q[NR];
                #pragma unroll
                for (int u = 0; u < NR; ++u) {
                    const int r = split + (k0 + u) * p.ks;
                    q[u] = r < TC_M ? S->q[r] : -1;
                    if (adds) base_of(q[u], c, o[u]);
                    else { o[u][0] = base4[0]; o[u][1] = base4[1]; o[u][2] = base4[2]; o[u][3] = base4[3]; }
                }
                #pragma unroll 1
                for (int s0 = 0; s0 < p.ks; s0 += NS) {
                    uint4 t[NS][NR];
                    #pragma unroll
                    for (int s = 0; s < NS; ++s)
                        #pragma unroll
                        for (int u = 0; u < NR; ++u) {
                            t[s][u] = make_uint4(0, 0, 0, 0);
                            if (s0 + s < p.ks && q[u] >= 0 && c < p.bn)
                                t[s][u] = wn_ld_remote(smem_u32(staged + (size_t)(split + (k0 + u) * p.ks) * ldr + c), (uint32_t)(s0 + s));
                        }
                    #pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        if (s0 + s >= p.ks) break;
                        #pragma unroll
                        for (int u = 0; u < NR; ++u) {
                            o[u][0] = plus(o[u][0], t[s][u].x); o[u][1] = plus(o[u][1], t[s][u].y);
                            o[u][2] = plus(o[u][2], t[s][u].z); o[u][3] = plus(o[u][3], t[s][u].w);
                        }
                    }
                }
                #pragma unroll
                for (int u = 0; u < NR; ++u) emit(q[u], c, o[u]);
            }
        } else wn_cluster_meet();
        wn_cluster_meet();                                   // nobody's shared memory goes away while it is read
    }
    tc_fence_before();
    __syncthreads();
    if (tid == WN_FILL + 32 && S->fail) {
        // a role gave up: bulk copies still in flight must land before the CTA's shared memory goes away
        for (int j = max(0, issued - p.stages); j < issued; ++j)
            mbar_wait(smem_u32(&S->bfull[j % p.stages]), (j / p.stages) & 1, WAIT_LIMIT_DEFAULT);
    }
    if (warp == 8)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(p.tmem_cols) : "memory");
}

// Max-pool windows over what the convolution kernel wrote pixel by pixel: bytes (16 channels per thread) or sign words
// (the sign of a maximum is the OR of the signs).  Bound by its reads; the int32 projections it would otherwise read are
// four times as many bytes.
template <int KW, bool BITS>
__global__ void __launch_bounds__(256) pool_window_kernel(const void* A, void* X, int oh, int ow, int th, int tw, int units, int s,
                                                          int pad, int total)
{
    using T = typename std::conditional<BITS, uint32_t, uint4>::type;
    const int i = blockIdx.x * 256 + threadIdx.x;
    pdl_launch_dependents();
    pdl_wait();
    if (i >= total) return;
    const int u = i % units, r = i / units, tx = r % tw, ty = r / tw % th, ns = r / (tw * th);
    const T* src = reinterpret_cast<const T*>(A) + (size_t)ns * oh * ow * units + u;
    T v[KW * KW];
    bool in[KW * KW];
    #pragma unroll
    for (int k = 0; k < KW * KW; ++k) {
        const int y = ty * s - pad + k / KW, x = tx * s - pad + k % KW;
        in[k] = y >= 0 && y < oh && x >= 0 && x < ow;
        if (in[k]) v[k] = src[(size_t)(y * ow + x) * units];
    }
    T o{};
    bool have = false;
    #pragma unroll
    for (int k = 0; k < KW * KW; ++k) {
        if (!in[k]) continue;
        if constexpr (BITS) o |= v[k];
        else if (!have) o = v[k];
        else { o.x = __vmaxs4(o.x, v[k].x); o.y = __vmaxs4(o.y, v[k].y); o.z = __vmaxs4(o.z, v[k].z); o.w = __vmaxs4(o.w, v[k].w); }
        have = true;
    }
    reinterpret_cast<T*>(X)[i] = o;
}

int launch_pool_window(const Layer& L, const Tensor& out, const void* A, void* X, cudaStream_t st)
{
    const rrm_layer_desc& d = L.d;
    const bool bits = out.dtype == T_BIN;
    const int units = bits ? out.cs : out.cs / 16;
    const long long total = (long long)out.pixels() * units;
    const dim3 grid((unsigned)((total + 255) / 256));
    cudaError_t e = cudaSuccess;
    auto go = [&](auto kernel) { e = launch_seq(kernel, dim3(grid), dim3(256), 0, st, A, X, L.oh, L.ow, L.th, L.tw, units, d.pool_s, d.pool_p, (int)total); };
    switch (d.pool_k) {
        case 1: if (bits) go(pool_window_kernel<1, true>); else go(pool_window_kernel<1, false>); break;
        case 2: if (bits) go(pool_window_kernel<2, true>); else go(pool_window_kernel<2, false>); break;
        case 3: if (bits) go(pool_window_kernel<3, true>); else go(pool_window_kernel<3, false>); break;
        default: return RRM_ERR_UNSUPPORTED;
    }
    RRM_CUDA_TRY(e);
    return RRM_OK;
}

// ------------------------------------------------------------------------------------------------
// Filters as operand tiles: [n tile][tap][group][2 chunks][pieces][bn][16 bytes].  One thread per 16 bytes.
// K within a tap: channels (int8 and binary: bytes; fp32: bf16 pieces); first layers: tap = filter row, K = kx * 4 + channel.
// ------------------------------------------------------------------------------------------------
// fp32: *beyond becomes 1 if a filter value's pieces are no finite numbers.
template <int DT, bool XCOL>
__global__ void pack_weights_win_kernel(const void* W, unsigned char* img, int c_in, int c_out, int kh, int kw, int taps, int groups,
                                        int bn, int n_tiles, int* beyond)
{
    const size_t total = (size_t)n_tiles * taps * groups * 2 * bn;
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    const int r = (int)(idx % bn), c = (int)(idx / bn % 2), g = (int)(idx / ((size_t)2 * bn) % groups);
    const int tap = (int)(idx / ((size_t)2 * bn * groups) % taps), nt = (int)(idx / ((size_t)2 * bn * groups * taps));
    const int co = nt * bn + r;
    constexpr int E = DT == T_F32 ? 8 : 16, PIECES = DT == T_F32 ? 3 : 1;
    unsigned char* dst = img + ((((size_t)nt * taps + tap) * groups + g) * 2 + c) * PIECES * bn * 16 + (size_t)r * 16;
    auto at = [&](int e) -> size_t {                          // element e of this chunk, as an index into W ((size_t)-1: none)
        const int k = (g * 2 + c) * E + e;
        int ci, ky, kx;
        if (XCOL) { ky = tap; kx = k >> 2; ci = k & 3; } else { ky = tap / kw; kx = tap - ky * kw; ci = k; }
        if (co >= c_out || ci >= c_in || kx >= kw) return (size_t)-1;
        return (((size_t)co * c_in + ci) * kh + ky) * kw + kx;
    };
    if (DT == T_F32) {
        uint32_t s[3][4];
        #pragma unroll
        for (int j = 0; j < 4; ++j) {
            const size_t a = at(2 * j), b = at(2 * j + 1);
            wn_split(a == (size_t)-1 ? 0.f : reinterpret_cast<const float*>(W)[a], b == (size_t)-1 ? 0.f : reinterpret_cast<const float*>(W)[b],
                     s[0][j], s[1][j], s[2][j]);
            if (wn_bf16_nan(s[2][j])) *beyond = 1;
        }
        for (int k = 0; k < 3; ++k) *reinterpret_cast<uint4*>(dst + (size_t)k * bn * 16) = make_uint4(s[k][0], s[k][1], s[k][2], s[k][3]);
    } else {
        uint32_t v[4] = {0, 0, 0, 0};
        #pragma unroll
        for (int e = 0; e < 16; ++e) {
            const size_t a = at(e);
            const int x = a == (size_t)-1 ? 0 : reinterpret_cast<const int8_t*>(W)[a];
            v[e >> 2] |= ((uint32_t)x & 0xffu) << (8 * (e & 3));
        }
        *reinterpret_cast<uint4*>(dst) = make_uint4(v[0], v[1], v[2], v[3]);
    }
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
static int host_floor_div(int a, int s) { return a >= 0 ? a / s : -((s - 1 - a) / s); }

// The geometry of a layer that does not depend on how it is launched; false: the layer keeps the other kernels.
static bool win_geometry(const rrm_net* net, const Layer& L, WinParams& p)
{
    const rrm_layer_desc& d = L.d;
    const Tensor& in = net->tensors[d.src];
    const bool xcol = d.dtype == RRM_F32 ? d.c_in <= 4 : (d.dtype == RRM_I8 && in.cs == 4);
    if (d.dtype == RRM_I8 && !xcol && in.cs % 32 != 0) return false;
    p.n = d.n; p.h = d.h; p.w = d.w; p.oh = L.oh; p.ow = L.ow; p.kh = d.kh; p.kw = d.kw; p.stride = d.stride; p.pad = d.pad;
    p.c_in = d.c_in; p.c_out = d.c_out; p.row_units = in.cs;
    const int pyn = d.stride < d.kh ? d.stride : d.kh, pxn = xcol ? 1 : (d.stride < d.kw ? d.stride : d.kw);
    p.planes = pyn * pxn;
    if (p.planes > WN_MAX_PLANES) return false;
    const int fy_lo = host_floor_div(-d.pad, d.stride), fy_hi = host_floor_div(d.kh - 1 - d.pad, d.stride);
    const int fx_lo = xcol ? 0 : fy_lo, fx_hi = xcol ? 0 : host_floor_div(d.kw - 1 - d.pad, d.stride);
    auto pitch = [&](int o, int size, int lo, int hi) {      // room for the pixels and for the zeros that taps reach beyond them
        const int last = (size - 1) / d.stride;
        int v = o;
        v = v > o + hi ? v : o + hi;
        v = v > last + 1 - lo ? v : last + 1 - lo;
        return v;
    };
    const int e = d.dtype == RRM_F32 ? 16 : 32;              // K elements of a group
    p.groups = xcol ? ceil_div(d.kw * 4, e) : ceil_div(d.dtype == RRM_I8 ? in.cs : d.c_in, e);
    if (xcol && (p.groups > 4 || d.stride > 128)) return false;                  // (a block holds up to four K groups, a first layer's block all of them)
    // first layers: pixels of a 16-byte chunk; a row in one or two arrays where the stride is as many chunks
    const int px = d.dtype == RRM_F32 ? 2 : 4;
    p.xarr = xcol && d.stride % px == 0 && d.stride / px <= 2 ? d.stride / px : 0;
    const int reach = p.xarr ? (2 * p.groups - 1) / p.xarr : 0;      // slots from a column's first chunk to its last
    p.Wq = xcol ? L.ow + reach : pitch(L.ow, d.w, fx_lo, fx_hi);
    p.Hq = pitch(L.oh, d.h, fy_lo, fy_hi);
    p.min_shift = fy_lo * p.Wq + fx_lo;
    const int max_shift = fy_hi * p.Wq + fx_hi;
    for (int i = 0; i < p.planes; ++i) {
        WinPlane& a = p.plane[i];
        a.ky0 = i / pxn; a.kx0 = i % pxn;
        const int fy = host_floor_div(a.ky0 - d.pad, d.stride), fx = xcol ? 0 : host_floor_div(a.kx0 - d.pad, d.stride);
        a.ny = ceil_div(d.kh - a.ky0, d.stride); a.nx = xcol ? 1 : ceil_div(d.kw - a.kx0, d.stride);
        a.ry = a.ky0 - d.pad - fy * d.stride; a.rx = xcol ? 0 : a.kx0 - d.pad - fx * d.stride;
        a.shift0 = fy * p.Wq + fx;
    }
    auto divisor = [](int v) {
        WinDiv r;
        unsigned s = 0;
        while ((1u << s) < (unsigned)v) ++s;
        r.sh = 31 + s;
        r.m = (unsigned)(((1ull << r.sh) + v - 1) / v);
        return r;
    };
    p.div_img = divisor(p.Hq * p.Wq); p.div_row = divisor(p.Wq);
    p.span = TC_M + max_shift - p.min_shift + reach;         // (one accumulator tile)
    if (p.span > WN_MAX_SPAN) return false;
    if (((long long)d.n + 1) * p.Hq * p.Wq + 2 * p.span > INT_MAX) return false;      // (positions are int)
    // (rows of the linear space without a projection pixel are work for nothing: with more than half of them a layer
    // such as a filter that covers the whole map is better off with its rows compacted)
    if ((long long)L.oh * L.ow * 2 < (long long)p.Hq * p.Wq) return false;
    const int plane_taps = ceil_div(d.kh, d.stride) * (xcol ? 1 : ceil_div(d.kw, d.stride));
    if (d.dtype == RRM_F32 && plane_taps * (xcol ? p.groups : 1) > WN_PROMOTE) return false;
    return true;
}

static bool win_xcol(const rrm_net* net, const Layer& L)
{
    return L.d.dtype == RRM_F32 ? L.d.c_in <= 4 : (L.d.dtype == RRM_I8 && net->tensors[L.d.src].cs == 4);
}

// Rows of the linear space that accumulator tiles cover, per frame.
static long long win_rows(const WinParams& p) { return ((long long)(p.n - 1) * p.Hq + p.oh - 1) * p.Wq + p.ow; }

static int slots(int span) { return round_up(span, 8) + 1; }    // (neighbouring chunks of a pixel fall into different banks)

// Wide tiles that leave half of the wave idle.
static bool win_few_tiles(const Layer& L, long long row_tiles, int wave) { return row_tiles * L.win_ntiles * 2 <= wave; }

// Shares of K form a cluster (at most 8 CTAs); integer delta passes add theirs onto the projection one by one.
static bool win_clustered(const Layer& L, bool dense, bool store) { return dense || store || L.d.dtype == RRM_F32 || (L.d.c_out & 3) != 0; }

// How a launch with column tiles of one width cuts the work: accumulator tiles and shares of K per CTA, window blocks, filter
// stages.  `wave`: CTAs that are to be kept busy.
static bool win_cut(const Layer& L, WinParams& p, bool xcol, bool dense, bool store, int frames, int wave, bool narrow)
{
    const bool f32 = L.d.dtype == RRM_F32;
    const int pieces = f32 ? 3 : 1;
    const long long rows = win_rows(p);
    const long long row_tiles = (rows + TC_M - 1) / TC_M * frames;
    // shares of K: whole blocks, or parts of one block's taps, until the tiles fill one wave
    const bool clustered = win_clustered(L, dense, store);
    p.narrow = narrow;
    p.bn = p.narrow ? WN_NARROW : L.win_bn;
    p.ntiles = p.narrow ? ceil_div(p.c_out, WN_NARROW) : L.win_ntiles;
    const long long tiles = row_tiles * p.ntiles;
    const int base_span = p.span, planes = p.planes;
    const int plane_taps = ceil_div(p.kh, p.stride) * (xcol ? 1 : ceil_div(p.kw, p.stride));
    const size_t unit = (size_t)p.bn * 32 * pieces, tail = sizeof(WinTail) + 128;
    const size_t room = f32 ? WN_SMEM_LIMIT - 1024 : WN_SMEM_LIMIT / 2 - 2048;   // (integer kernels: two CTAs per SM)
    // two accumulator tiles per CTA share every filter stage (what bounds a full machine is the filters' way from L2),
    // once that leaves a CTA per SM
    int mt = !f32 && tiles >= 2ll * 148 && rows > TC_M ? 2 : 1;
    // (a cluster of narrow tiles is worth it for shares of some 48 K steps; with several planes, whose blocks are small and cost
    // some 2.5 k clocks each for their windows, as soon as it leaves a block out: 256 -> 512 3x3 of stride 2 at 14 x 14, 4 images,
    // 27.9 -> 14.4 k clocks a CTA)
    const int steps = p.groups * p.kh * (xcol ? 1 : p.kw);
    const int most = !clustered ? 16 : (!p.narrow || planes > 1 ? 8 : (steps < 96 ? 1 : (steps / 48 < 8 ? steps / 48 : 8)));
    int want = 1;
    while (mt == 1 && want < most && tiles * (want + 1) <= wave) ++want;
    for (; mt >= 1; mt /= 2) {
        p.mt = mt;
        p.span = base_span + (mt - 1) * TC_M;
        if (p.span > WN_MAX_SPAN) continue;                  // (the tables hold no wider window: one tile, which win_geometry has checked)
        p.L = slots(p.span);
        p.all_tables = !xcol && planes * p.span <= 2 * WN_MAX_SPAN;
        // drained rows: a tile's (64 columns of it where there are two), or 32 rows x up to 64 columns per warp
        const size_t whole = (size_t)mt * TC_M * ((mt > 1 && p.bn > 64 ? 64 : p.bn) + 4) * 4;
        const size_t turned = (size_t)8 * 32 * ((p.bn < WN_TURN ? p.bn : WN_TURN) + 4) * 4;
        const size_t staging = whole > turned ? whole : turned;
        int gblk = xcol ? p.groups : (p.groups < 4 ? p.groups : 4);
        if (f32 && !xcol) while (gblk > 1 && gblk * plane_taps > 18) gblk = (gblk + 1) / 2;
        if (!xcol) while (gblk > 1 && planes * ceil_div(p.groups, gblk) < want) gblk = (gblk + 1) / 2;
        for (;; gblk = (gblk + 1) / 2) {
            p.gblk = gblk;
            p.nchb = ceil_div(p.groups, gblk);
            p.nblk = planes * p.nchb;
            p.tsplit = 1;
            p.ks = want < p.nblk ? want : p.nblk;
            p.per = ceil_div(p.nblk, p.ks);
            p.ks = ceil_div(p.nblk, p.per);                  // no empty share
            if (!f32 && p.ks == p.nblk && planes == 1 && want >= 2 * p.nblk && plane_taps >= 2) {
                p.tsplit = want / p.nblk < plane_taps ? want / p.nblk : plane_taps;
                p.ks = p.nblk * p.tsplit;
            }
            p.cluster = clustered && p.ks > 1;
            p.abytes = (unsigned)(((size_t)(p.xarr ? p.xarr : gblk * 2) * pieces * p.L * 16 + 127) & ~(size_t)127);
            p.a_lbo = p.xarr == 1 ? 1u : (unsigned)p.L;
            p.a_step = p.xarr ? 2u / (unsigned)p.xarr : 2u * (unsigned)p.L;
            p.tps = 1;
            while ((size_t)p.tps * 2 * gblk * unit <= (f32 ? 24u : 16u) * 1024 && p.tps < plane_taps) p.tps *= 2;
            p.stage_bytes = (unsigned)(p.tps * gblk * unit);
            for (p.abuf = p.per < WN_MAX_ABUF ? p.per : WN_MAX_ABUF; p.abuf >= 1; --p.abuf) {
                const size_t a = (size_t)p.abuf * p.abytes + tail;
                if (a + 3 * (size_t)p.stage_bytes > room) continue;
                const size_t fit = (room - a) / p.stage_bytes;
                p.stages = (int)(fit < WN_MAX_STAGES ? fit : WN_MAX_STAGES);
                const size_t used = (size_t)p.abuf * p.abytes + (size_t)p.stages * p.stage_bytes;
                p.tail_off = (unsigned)((used > staging ? used : staging) + 15) & ~15u;      // (the drained rows go where windows and stages were)
                if (p.tail_off + tail > room) continue;
                const unsigned cols = f32 ? 3 * p.bn + round_up(p.bn, 32) : (mt - 1) * p.bn + round_up(p.bn, 32);
                p.tmem_cols = 32;
                while (p.tmem_cols < cols) p.tmem_cols *= 2;
                return true;
            }
            if (gblk == 1 || xcol) break;
        }
    }
    return false;
}

// Clocks of a block of an integer launch: of its window's way into shared memory, and of its MMAs.
static long long win_fill_clocks(const WinParams& p) { return 1500 + 300ll * ceil_div(p.span * (p.xarr ? p.xarr : p.gblk * 2), WN_FILL); }
static long long win_mma_clocks(const WinParams& p, bool xcol)
{
    return (long long)p.groups * p.kh * (xcol ? 1 : p.kw) * (32 + p.bn) * p.mt / ((long long)p.nblk * p.tsplit);
}

// Dense int8 windows by asynchronous copies: with three buffers or more two blocks' copies are under way at a time, which pays
// where the MMAs are too short to hide a block's way through registers (9 x 36 short blocks, 409 -> 85 3x3 of stride 3 at
// 112 x 120, 12 images: 133.9 us through registers, 103.4 so; 31 of 340 timed launches fall under the rule, 5 % faster on
// average, at worst level but for one of 17.6 us, 4 % slower).  The others are up to 15 % slower so.
static bool win_async_windows(const WinParams& p, bool xcol) { return p.abuf >= 3 && win_mma_clocks(p, xcol) * 5 < win_fill_clocks(p) * 2; }

// What a CTA of an integer launch takes, in clocks, apart from what is the same for all cuts: its blocks one after the other
// (the window's way into shared memory, or the MMAs, whichever is longer; the shorter once more where nothing hides it) and the
// cluster's way out (meetings, rows read from the other shares; as far as the fullest tile's rows are projection pixels).  The
// figures are fitted to 1200 timed cuts of 132 layers: of both widths and all numbers of shares, 1x1 to 7x7, strides 1 to 4.
// Deltas update few of a tile's rows, so their clusters close early (59 -> 91 3x3 of stride 2 at 50 x 46, binary, 12 images, 1 % of
// the pixels changing: 18.7 us as clusters of 2, 20.7 as narrow tiles, which a dense pass is as fast with).
static long long win_clocks(const WinParams& p, bool xcol, bool dense)
{
    const long long rows = win_rows(p), full = rows < TC_M ? rows : TC_M;                     // (of the fullest tile)
    const long long pixels = (long long)p.n * p.oh * p.ow * full / rows;
    const long long fill = win_fill_clocks(p), mmas = win_mma_clocks(p, xcol);
    long long clocks = p.per * (fill > mmas ? fill : mmas) + (fill > mmas ? mmas : fill);
    if (p.cluster) clocks += 300ll * p.ks + (dense ? 4000 + 32ll * p.bn * pixels / TC_M : 2500);
    return clocks;
}

// Integers whose shares would form a cluster, and whose tiles leave half of the wave idle, may take tiles of 32 columns
// instead.  That saves the cluster's way out (8 to 10 k clocks with 128 columns) or most of it, and an MMA of 32 columns is
// shorter than one of 128; but every column tile lays out the windows of all its blocks, which shares of K divide.  Few blocks:
// narrow (us, wide / narrow: 28 -> 239 5x5 at 23 x 26 14.3 / 8.4; 96 -> 256 5x5 at 27 x 27 12.8 / 10.8).  Many blocks, of several
// planes or of 1x1 filters: wide (409 -> 85 3x3 of stride 3 at 112 x 120, 3 images, 36 blocks: 35.4 / 71.9; 1024 -> 256 1x1 at
// 14 x 14, 2 images: 12.0 / 16.9).  Over 109 such layers the estimate's choice is 11 % ahead of wide tiles alone, at worst
// 2 % behind; narrow tiles alone are 8 % ahead, at worst 103 % behind.
static bool win_plan(const Layer& L, WinParams& p, bool xcol, bool dense, bool store, int frames, int wave)
{
    if (win_clustered(L, dense, store) && L.win_narrow && win_few_tiles(L, (win_rows(p) + TC_M - 1) / TC_M * frames, wave)) {
        WinParams few = p;
        const bool narrow = win_cut(L, few, xcol, dense, store, frames, wave, true);
        if (!win_cut(L, p, xcol, dense, store, frames, wave, false)) return false;
        if (narrow && win_clocks(few, xcol, dense) <= win_clocks(p, xcol, dense)) p = few;
        return true;
    }
    return win_cut(L, p, xcol, dense, store, frames, wave, false);
}

// Shared memory of a launch: at least the CTA's share of tensor memory.
static size_t win_smem(const WinParams& p)
{
    const size_t need = p.tail_off + sizeof(WinTail) + 128, share = tmem_share(p.tmem_cols);
    return need > share ? need : share;
}

// Launches that overlap their predecessors (dense passes) are placed while those still hold some of the SMs: two CTAs of an
// integer launch then come to lie on one SM and leave others idle.  Launches of fewer CTAs than SMs, but of many, ask for more than
// half of an SM's shared memory, so that each has one to itself (411 -> 22 3x3 of stride 2, binary, 56 images of 27 x 37, 132
// CTAs: 37.3 us without overlap, 42.5 with, 36.3 so; dense chunks of 32 AlexNet-shaped frames 124.7 -> 119.2, of 2 x 8
// ResNet-18-shaped ones at 183 x 183 181 -> 172).  Below 90 CTAs they find room beside each other, and the next launch's wait beside
// them (24 AlexNet-shaped keyframes, two launches of 81 CTAs: 90.9, 92.0 with an SM each); short chains lose more by the wait for an
// SM than by sharing one (5 ResNet-18-shaped frames at 160 x 160, four launches of 132 CTAs of some 4 k clocks: 130.4, 133.4).
constexpr int WN_ALONE = 90;
constexpr long long WN_ALONE_CHAIN = 8200;                   // clocks of a CTA's blocks
constexpr size_t WN_ALONE_SMEM = 116 * 1024;

static bool win_alone(const WinParams& p, int dtype, bool xcol, long long ctas)
{
    return dtype != RRM_F32 && !p.cluster && ctas >= WN_ALONE && ctas <= 148 && win_clocks(p, xcol, true) >= WN_ALONE_CHAIN;
}

// Clusters cannot be placed so: their CTAs also have to lie in one part of the machine (one CTA an SM is up to 1.6 times as slow).
// Binary clusters of long chains, whose windows keep an SM's ALUs busy, are not launched early instead (457 -> 69 3x3 of stride 3 at
// 84 x 68, 11 images, 112 CTAs of 18 blocks each: 47.2 us without overlap, 53.9 with).
constexpr long long WN_LONG_CHAIN = 18000;                   // clocks of a CTA's blocks
static bool win_long_binary(const WinParams& p)
{
    const long long fill = win_fill_clocks(p), mmas = win_mma_clocks(p, false);
    return p.cluster && p.per * (fill > mmas ? fill : mmas) >= WN_LONG_CHAIN;
}

template <int DT, bool XCOL>
static int win_allow()
{
    constexpr bool COPIES = DT == T_I8 && !XCOL;             // (delta rows always, dense windows by win_async_windows)
    auto allow = [](auto kernel) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)WN_SMEM_LIMIT); };
    RRM_CUDA_TRY(allow(conv_win_kernel<DT, false, XCOL, false, COPIES>));
    RRM_CUDA_TRY(allow(conv_win_kernel<DT, true, XCOL, false, false>));
    RRM_CUDA_TRY(allow(conv_win_kernel<DT, true, XCOL, true, false>));
    if constexpr (COPIES) {
        RRM_CUDA_TRY(allow(conv_win_kernel<DT, true, XCOL, false, true>));
        RRM_CUDA_TRY(allow(conv_win_kernel<DT, true, XCOL, true, true>));
    }
    return RRM_OK;
}

// Whether the window kernel takes the layer, and the widths of its column tiles.  Every launch of a layer that is taken has
// to find a plan: whether a window and three filter stages fit shared memory depends on the width alone (a plan falls back to
// one accumulator tile, one K group per block and one window buffer, whatever it was first cut for), so one plan of each width
// decides.  The narrow tiles are no easier to fit than the wide ones: tiles of 96 columns have stages of 12 KB, narrow
// ones of 16 (first layers of wide windows fit only the former).
static bool win_choose(const rrm_net* net, Layer& L)
{
    const rrm_layer_desc& d = L.d;
    WinParams wide{}, narrow{};
    if (!win_geometry(net, L, wide)) return false;
    narrow = wide;                                           // (a plan widens the window it is given)
    const bool xcol = win_xcol(net, L), f32 = d.dtype == RRM_F32;
    L.win_ntiles = ceil_div(d.c_out, 128);
    // (integer layers: whole groups of 32 columns, so that a padded output row is covered by the column tiles)
    L.win_bn = round_up(ceil_div(d.c_out, L.win_ntiles), f32 ? 16 : 32);
    L.win_ntiles = ceil_div(d.c_out, L.win_bn);
    L.win_narrow = false;
    if (!win_plan(L, wide, xcol, true, false, 1, 148)) return false;
    // (more frames are only more tiles, and 148 is the larger wave: with too many tiles in one frame no launch takes narrow ones)
    L.win_narrow = !f32 && L.win_bn > WN_NARROW && win_few_tiles(L, (win_rows(wide) + TC_M - 1) / TC_M, 148);
    L.win_narrow = L.win_narrow && win_cut(L, narrow, xcol, true, false, 1, 148, true);
    return true;
}

// Packs the filters of a layer the window kernel takes; RRM_ERR_UNSUPPORTED: the layer keeps the other kernels.
int conv_win_create(rrm_net* net, Layer& L, const void* W_dev)
{
    const rrm_layer_desc& d = L.d;
    WinParams p{};
    if (!win_choose(net, L) || !win_geometry(net, L, p)) return RRM_ERR_UNSUPPORTED;
    const bool xcol = win_xcol(net, L), f32 = d.dtype == RRM_F32;
    const int taps = xcol ? d.kh : d.kh * d.kw;
    const size_t chunks = (size_t)L.win_ntiles * taps * p.groups * 2 * L.win_bn;
    const size_t bytes = chunks * 16 * (f32 ? 3 : 1);
    // the same filters once more, as tiles of 32 columns; where there is no room for both the layer goes without (one block
    // for both: an allocation costs some 60 us)
    const int few_ntiles = ceil_div(d.c_out, WN_NARROW);
    const size_t few_chunks = (size_t)few_ntiles * taps * p.groups * 2 * WN_NARROW;
    void *img = nullptr, *few = nullptr;
    if (L.win_narrow && cudaMalloc(&img, bytes + 16 + few_chunks * 16) != cudaSuccess) { cudaGetLastError(); img = nullptr; L.win_narrow = false; }
    if (!img && cudaMalloc(&img, bytes + 16) != cudaSuccess) { cudaGetLastError(); return RRM_ERR_ALLOC; }
    net->allocs.push_back(img);
    int* beyond = reinterpret_cast<int*>(reinterpret_cast<unsigned char*>(img) + bytes);
    if (L.win_narrow) few = beyond + 4;
    RRM_CUDA_TRY(cudaMemset(beyond, 0, 4));
    auto pack = [&](auto kernel) {
        auto go = [&](void* to, size_t n, int bn, int ntiles) {
            kernel<<<(unsigned)((n + 255) / 256), 256>>>(W_dev, reinterpret_cast<unsigned char*>(to), d.c_in, d.c_out, d.kh, d.kw, taps, p.groups, bn, ntiles, beyond);
        };
        go(img, chunks, L.win_bn, L.win_ntiles);
        if (few) go(few, few_chunks, WN_NARROW, few_ntiles);
    };
    if (f32) { if (xcol) pack(pack_weights_win_kernel<T_F32, true>); else pack(pack_weights_win_kernel<T_F32, false>); }
    else if (xcol) pack(pack_weights_win_kernel<T_I8, true>);
    else pack(pack_weights_win_kernel<T_I8, false>);
    RRM_CUDA_TRY(cudaGetLastError());
    if (f32) {
        int has = 0;
        RRM_CUDA_TRY(cudaMemcpy(&has, beyond, 4, cudaMemcpyDeviceToHost));
        if (has) {
            net->allocs.pop_back();
            cudaFree(img);
            return RRM_ERR_UNSUPPORTED;
        }
    }
    L.win_Wimg = img;
    L.win_Wnarrow = few;
    RRM_TRY((win_allow<T_F32, true>())); RRM_TRY((win_allow<T_F32, false>()));
    RRM_TRY((win_allow<T_I8, true>())); RRM_TRY((win_allow<T_I8, false>()));
    RRM_TRY((win_allow<T_BIN, false>()));
    L.win_tiles = ceil_div((int)win_rows(p), TC_M);
    L.win_ready = true;
    return RRM_OK;
}

// How a launch of the layer is cut (host arithmetic; the layer's sizes are set, nothing else).
int conv_win_query(const rrm_net& net, Layer& L, int form, int frames, rrm_conv_plan* out)
{
    *out = rrm_conv_plan{};
    WinParams p{};
    if (!win_choose(&net, L)) return RRM_OK;
    const bool xcol = win_xcol(&net, L), dense = form == RRM_PLAN_DENSE, seq = form == RRM_PLAN_SEQ;
    if (dense) L.d.n *= frames;                              // (a batch of dense frames is that many more images)
    if (!win_geometry(&net, L, p) || !win_plan(L, p, xcol, dense, seq, seq ? frames : 1, form == RRM_PLAN_PIPELINED ? 74 : 148))
        return RRM_ERR_UNSUPPORTED;                          // (never: win_choose takes no such layer)
    const long long rows = win_rows(p);
    out->columns = p.bn; out->tiles_per_cta = p.mt; out->shares = p.ks; out->clustered = p.cluster;
    out->ctas = (rows + p.mt * TC_M - 1) / (p.mt * TC_M) * p.ntiles * p.ks * (seq ? frames : 1);
    out->narrow_filters = L.win_narrow;
    out->async_windows = L.d.dtype == RRM_I8 && !xcol && (!dense || win_async_windows(p, xcol));
    return RRM_OK;
}

template <int DT, bool XCOL>
static cudaError_t win_launch(const WinParams& p, bool dense, bool act, dim3 grid, size_t smem, cudaStream_t st)
{
    auto go = [&](auto kernel) { return launch_seq_cluster(kernel, grid, dim3(WN_THREADS), smem, st, p.cluster ? p.ks : 1, p); };
    constexpr bool COPIES = DT == T_I8 && !XCOL;
    if (!dense) return go(conv_win_kernel<DT, false, XCOL, false, COPIES>);
    if constexpr (COPIES)
        if (win_async_windows(p, XCOL)) return act ? go(conv_win_kernel<DT, true, XCOL, true, true>) : go(conv_win_kernel<DT, true, XCOL, false, true>);
    return act ? go(conv_win_kernel<DT, true, XCOL, true, false>) : go(conv_win_kernel<DT, true, XCOL, false, false>);
}

// F*dI (dense: F*X + b); arguments as for launch_conv_tc.
int launch_conv_win(rrm_net* net, Layer& L, const Tensor& in, bool dense, bool stateless, cudaStream_t st,
                    const uint32_t* count_bitmap, void* P_dst, int frames, long long arena_stride, const WinOutput* out)
{
    const rrm_layer_desc& d = L.d;
    WinParams p{};
    if (!win_geometry(net, L, p)) return RRM_ERR_UNSUPPORTED;
    const bool xcol = win_xcol(net, L), bin = d.dtype == RRM_BIN;
    const bool batched = P_dst && frames >= 1 && arena_stride != 0;
    const int nf = batched ? frames : 1;
    if (!win_plan(L, p, xcol, dense, batched, nf, net->many_in_flight ? 74 : 148)) return RRM_ERR_UNSUPPORTED;
    if (p.span > WN_MAX_SPAN) return RRM_ERR_CAPACITY;       // (never: win_plan takes no such window)
    const void* X = stateless ? in.X2 : in.X;
    p.A = bin ? in.D : (dense ? X : in.D);
    p.Anew = (!dense && !stateless && in.Xn_cur) ? in.Xn_cur : X;    // (chunks of frames: this frame's copy of the new rows)
    p.in_act = in.act; p.oact = L.oact; p.ocount = L.ocount;
    p.Wimg = reinterpret_cast<const unsigned char*>(p.narrow ? L.win_Wnarrow : L.win_Wimg); p.bias = L.bias;
    p.P = P_dst && !dense ? P_dst : (stateless ? L.P2 : L.P);
    p.errw = net->errw;
    p.wait_limit = net->opt.wait_limit;
    p.count_bitmap = count_bitmap;
    p.frames = nf;
    p.row_stride = (long long)in.bytes(); p.arena_stride = arena_stride; p.p_stride = (long long)L.opixels() * d.c_out;
    p.store = batched ? 1 : 0;
    if (out) {
        p.X = out->X; p.res = out->res; p.cs = out->cs; p.bits = out->bits;
        p.bn_scale = L.bn_scale; p.bn_shift = L.bn_shift; p.shift = d.shift; p.act_fn = d.act; p.theta = d.theta;
        p.P = out->P; p.keep_from = out->P ? out->keep_from : INT_MAX;
    }
    const long long rows = win_rows(p);
    const dim3 grid((unsigned)((rows + p.mt * TC_M - 1) / (p.mt * TC_M)), (unsigned)p.ntiles, (unsigned)(nf * p.ks));
    size_t smem = win_smem(p);
    if (dense && pdl_enabled() && win_alone(p, d.dtype, xcol, (long long)grid.x * grid.y * grid.z) && smem < WN_ALONE_SMEM) smem = WN_ALONE_SMEM;
    const OverlapLaunches early(OverlapLaunches::on() && !(dense && bin && win_long_binary(p)));
    cudaError_t e;
    if (d.dtype == RRM_F32) e = xcol ? win_launch<T_F32, true>(p, dense, out, grid, smem, st) : win_launch<T_F32, false>(p, dense, out, grid, smem, st);
    else if (d.dtype == RRM_I8) e = xcol ? win_launch<T_I8, true>(p, dense, out, grid, smem, st) : win_launch<T_I8, false>(p, dense, out, grid, smem, st);
    else e = win_launch<T_BIN, false>(p, dense, out, grid, smem, st);
    RRM_CUDA_TRY(e);
    return RRM_OK;
}

}  // namespace rrm
