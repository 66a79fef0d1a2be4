// Dense tensor-core route of the sparse convolutions and large-batch FC layers (implicit GEMM on
// NHWC activations, float and int8).
//
// CADNN (arXiv 1905.00571), Section 1 ("computation pattern transformation"): a compressed layer is
// executed in the form the processor runs fastest.  A stored nonzero costs the sparse kernels one
// 32-bit shared-memory word per multiply-add, which bounds them at a quarter of the FMA rate; the tensor
// cores multiply the same layer with its pruned positions as zeros at a rate so much higher that they win
// from a few per cent of kept weights on (tcv_pays below has the rule).  Batch 32, 12.5 % kept, microseconds
// before / now: 64->64 3x3 56x56 118 / 60, 256->64 1x1 56x56 86 / 45, 256->256 3x3 14x14 122 / 48; int8 at 8 %,
// batch 8, 256->256 3x3 56x56 240 / 37.
//
// GEMM view: rows = output pixels (image, row, column flattened), columns = output channels, K = (kernel
// row, kernel column, input channel).  One block = a tile of pixels x channels (several shapes, see Cfg and
// choose); the K range can be split over a thread-block cluster whose partial sums meet in distributed
// shared memory (small maps would otherwise leave most multiprocessors idle).
//   * 8 loader warps gather the im2col rows from NHWC memory (out-of-image taps are zeros) into swizzled
//     K-major operand tiles, 128 source bytes per pixel and stage, in groups that fill alternate stages;
//     int8 layers of whole 64-channel rows leave that to the copy engine (engine_takes; not the split tiles of pooled layers);
//   * one thread copies the matching weight tiles (pre-swizzled by the packer) with bulk copies; the first
//     ones do not wait for the previous layer;
//   * one thread issues the tcgen05.mma's; accumulators live in tensor memory;
//   * the loader warps then finish the tile, with scale, bias and residual asked for at its start: float
//     tiles whose rows are channels as columns of 16 pixels straight from tensor memory, the others through
//     shared memory as [pixel][channel]; with a split reduction every block sends each other block its
//     pixels' sums, float from registers, int8 as bulk copies of the staged tile, counted on the receiver's barrier.
// What bounds it, from clock stamps in its warps.  At batch 1 a chain: 14x14, 256 -> 1024 1x1 with a residual, 32 x 128 tile split
// in four (clocks of 0.5 ns after the previous layer has ended): first stage in shared memory 1300, first products 2250, last 3330, complete
// 3610, sums read and sent 4370, received 5030, written 6050; 0.8 us from the end of one layer to the next.  Four to eight warps a
// scheduler share the issue slots, so what helps there is fewer instructions.  At large batch, float: the products (256 x 128 tiles
// run at 90 % of the tensor cores' rate while multiplying; their first loads and epilogue, 10 to 50 % of the time, are not
// overlapped).  Int8: epilogue instructions and the exchange.
//
// Float precision.  A float is the exact sum of three bf16 numbers (8 + 8 + 8 significand bits), a = a1 + a2 +
// a3 with |a2| <= 2^-9 |a|, |a3| <= 2^-18 |a|, from 2^-110 (8e-34) on (below, the third part loses bits under
// bf16's smallest number, 2^-133) and up to 3.39e38 (beyond, the first part rounds to infinity).  Loaders split activations, the packer splits weights, and the
// products a1 b1, a1 b2, a2 b1, a2 b2, a1 b3, a3 b1 are accumulated in fp32; what is left out is below 2^-25 of
// |a b|, less than the rounding of one fp32 multiply-add.  a1 b1 has an accumulator of its own: the small terms
// are summed apart and added once at the end, so they are not rounded away against the large sum.
// Int8 products accumulate in int32, exact in any order.
#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <cstdio>
#include <cuda.h>
#include <cuda_bf16.h>
#include "cadnn_internal.h"

namespace {

const int kSpin = 1 << 22;

struct TcvParams {
    const void *x;
    void *y;
    const unsigned char *wimg;
    const float *scale, *bias;
    const void *residual;
    float res_scale;
    int act, out_dtype;
    int h, w, c_in, h_out, w_out, c_out;
    int stride, pad, pad_w, kh, kw;
    int M, nkb, n_nt, S, npx;
    int stages, recv_off, bar_off;   // pipeline depth; byte offsets of the partial sums and of the barriers in shared memory
    int res_tile;                    // int8: the residual of the block's outputs is brought into shared memory, this many bytes at a time (0: no residual)
    int ldc, c_off, vec_ok;          // vec_ok: output and residual allow 4 channels per access
    int odd_half;                    // copy engine: 1 if the last stage's second 64 positions lie beyond K
    int kb_base, kb_rem;             // stages per block of a cluster: kb_base, and one more in the first kb_rem blocks
    int whole, tail;                 // int8 input: bytes of its whole 4-byte words, and bytes behind them
    int Rp;                          // K positions per kernel row: kw * c_in rounded up to 16 bytes
    FastDiv d_hw, d_wo, d_ci, d_Rp, d_S, d_nt, d_rows;
    signed char *pooled;             // int8: the 2 x 2 max pool of the output, written beside it; h_out, w_out, d_hw and d_wo are then the pool's
    int *gave_up;
    Prefetch ahead;
};

// One lane of a converged warp.  The compiler knows that a single lane runs what stands behind it and keeps the operands of copies and
// multiply-adds in uniform registers; behind `lane == 0` it emits a loop over the lanes around each of them.
__device__ __forceinline__ bool elected()
{
    unsigned r;
    asm volatile("{\n.reg .pred q;\nelect.sync _|q, 0xffffffff;\nselp.u32 %0, 1, 0, q;\n}\n" : "=r"(r));
    return r != 0;
}
__device__ __forceinline__ void mb_init(unsigned bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mb_expect_tx(unsigned bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mb_arrive(unsigned bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
// bounded wait; false = gave up (recorded)
__device__ __forceinline__ bool mb_wait(unsigned bar, unsigned parity, int *gave_up)
{
    for (int it = 0; it < kSpin; ++it) {
        unsigned ok;
        asm volatile("{\n.reg .pred q;\nmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\nselp.u32 %0, 1, 0, q;\n}\n"
                     : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (ok) return true;
    }
    atomicAdd(gave_up, 1);
    return false;
}
__device__ __forceinline__ void bulk_copy(unsigned dst, const void *src, unsigned bytes, unsigned bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
// Rows of the im2col matrix by the copy engine: `pixels` output pixels from the one whose window starts at (w, h) of image n on (both
// may lie in the padding), 64 channels from c on at window position (kx, ky), as 64-byte swizzled rows.
__device__ __forceinline__ void copy_pixels(unsigned dst, const CUtensorMap *map, int c, int w, int h, int n, int kx, int ky, unsigned bar)
{
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.im2col.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2], {%7, %8};\n"
                 ::"r"(dst), "l"(map), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n), "h"((unsigned short)kx), "h"((unsigned short)ky) : "memory");
}
// K-major operand tile, 64-byte rows, 64-byte swizzle (16-byte chunk index ^= (row / 2) % 4)
__device__ __forceinline__ unsigned long long smem_desc(unsigned addr)
{
    return (unsigned long long)((addr >> 4) & 0x3fffu) | (1ull << 16) | ((unsigned long long)(512u >> 4) << 32) | (1ull << 46) | (4ull << 61);
}
template <bool F32> __device__ __forceinline__ void mma(unsigned d, unsigned long long a, unsigned long long b, unsigned idesc, unsigned acc)
{
    if (F32)
        asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
                     ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
    else
        asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n}\n"
                     ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void tc_commit(unsigned bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}
// 16 accumulator columns of this warp's 32 rows (thread = row)
__device__ __forceinline__ void tmem_ld16(unsigned taddr, unsigned (&v)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 "
                 "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                 : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory"); }
// Keeps uses of the registers a tcgen05.ld fills behind the wait before this call: nothing else tells the compiler that they
// are not valid earlier.
__device__ __forceinline__ void tmem_arrived(unsigned (&v)[16])
{
    asm volatile("" : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]), "+r"(v[8]), "+r"(v[9]),
                      "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]));
}
__device__ __forceinline__ unsigned pack_bf16(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const unsigned *>(&v);
}
// two floats -> three packed bf16 pairs whose sum is the pair exactly
__device__ __forceinline__ void split2(float a, float b, unsigned &h, unsigned &m, unsigned &l)
{
    h = pack_bf16(a, b);
    a -= __uint_as_float(h << 16);
    b -= __uint_as_float(h & 0xffff0000u);
    m = pack_bf16(a, b);
    a -= __uint_as_float(m << 16);
    b -= __uint_as_float(m & 0xffff0000u);
    l = pack_bf16(a, b);
}
__device__ __forceinline__ void sts64(unsigned addr, unsigned a, unsigned b)
{
    asm volatile("st.shared.v2.b32 [%0], {%1, %2};\n" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ void sts128(unsigned addr, const uint4 &v)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ uint4 ld_vec(const void *p)
{
    uint4 v;
    asm volatile("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
// the same where `ok`, zeros elsewhere; a predicated load, so that several of a thread's are on their way at once
__device__ __forceinline__ uint4 ld_vec_if(const void *p, bool ok)
{
    uint4 v;
    asm volatile("{\n.reg .pred q;\nsetp.ne.b32 q, %5, 0;\nmov.b32 %0, 0;\nmov.b32 %1, 0;\nmov.b32 %2, 0;\nmov.b32 %3, 0;\n"
                 "@q ld.global.v4.b32 {%0, %1, %2, %3}, [%4];\n}\n"
                 : "=&r"(v.x), "=&r"(v.y), "=&r"(v.z), "=&r"(v.w) : "l"(p), "r"((int)ok));
    return v;
}
__device__ __forceinline__ unsigned ld_word_if(const void *p, bool ok)
{
    unsigned v;
    asm volatile("{\n.reg .pred q;\nsetp.ne.b32 q, %2, 0;\nmov.b32 %0, 0;\n@q ld.global.b32 %0, [%1];\n}\n" : "=&r"(v) : "l"(p), "r"((int)ok));
    return v;
}
__device__ __forceinline__ void st_word_if(float *p, float v, bool ok)
{
    asm volatile("{\n.reg .pred q;\nsetp.ne.b32 q, %2, 0;\n@q st.global.f32 [%0], %1;\n}\n" ::"l"(p), "f"(v), "r"((int)ok) : "memory");
}
__device__ __forceinline__ uint4 lds128(unsigned addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
// U values to address `addr` (as this block sees it) of block `owner` of the cluster; they count on that block's barrier
template <int U> __device__ __forceinline__ void send(unsigned addr, unsigned bar, int owner, const unsigned *v)
{
    unsigned a, b;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(a) : "r"(addr), "r"(owner));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(b) : "r"(bar), "r"(owner));
    if (U == 4)
        asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];\n"
                     ::"r"(a), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(b) : "memory");
    else if (U == 2)
        asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];\n" ::"r"(a), "r"(v[0]), "r"(v[1]), "r"(b) : "memory");
    else asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];\n" ::"r"(a), "r"(v[0]), "r"(b) : "memory");
}

// 4 or 16 bytes of global memory to shared memory, waited for with copies_landed by the thread that asked for them
__device__ __forceinline__ void copy4(unsigned dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy16(unsigned dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_landed() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
__device__ __forceinline__ float lds32(unsigned addr)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];\n" : "=f"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ float4 lds_float4(unsigned addr)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}

// copies `bytes` of this block's shared memory to address dst of block `owner`; counts on that block's barrier
__device__ __forceinline__ void send_bulk(unsigned dst, unsigned src, unsigned bytes, unsigned bar, int owner)
{
    asm volatile("{\n.reg .b32 a, b;\nmapa.shared::cluster.u32 a, %0, %4;\nmapa.shared::cluster.u32 b, %3, %4;\n"
                 "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [a], [%1], %2, [b];\n}\n"
                 ::"r"(dst), "r"(src), "r"(bytes), "r"(bar), "r"(owner) : "memory");
}

const int kTensorColumns = 512;   // of a multiprocessor
constexpr int accumulators(bool f32, int n) { return f32 && n <= 64 ? 3 : 2; }
constexpr int tensor_columns(bool f32, int n)
{
    return accumulators(f32, n) * n <= 128 ? 128 : accumulators(f32, n) * n <= 256 ? 256 : 512;
}

// How the activations come into shared memory: values one by one or as shifted words (pixels of any number of channels), 16 bytes at a
// time (whole 16-byte pieces of channels), or by the copy engine (int8, whole 64-channel rows).
enum class Gather { kValues, kPieces, kCopyEngine };

// Only the copy engine's kernels carry a tensor map among their parameters.
struct TcvEngineParams : TcvParams {
    CUtensorMap pixels;   // the input as im2col rows
};
// What a launch costs depends on the size of its parameters (driver 580): 24 or 32 bytes beyond a multiple of 64, an empty kernel takes
// 1.75 us as a programmatic dependent and 2.05 to 2.15 otherwise, with any other size 2.1 and 2.55 (every size from 8 to 608 bytes, alike
// in each 64).  The copy engine's kernels, 512 bytes, get a second parameter that nothing reads: small int8 layers called one by one (64 ->
// 64 1x1 7x7, 256 -> 64 1x1 56x56, 512 -> 1000 fc of 16 images) 3.6 to 3.8 us a call without it, 3.2 to 3.3 with it.
struct LaunchPad {
    unsigned char unused[32];
};
constexpr bool launches_fast(size_t parameters) { return parameters % 64 == 24 || parameters % 64 == 32; }
static_assert(launches_fast(sizeof(TcvParams)) && launches_fast(sizeof(TcvEngineParams) + sizeof(LaunchPad)), "launches take 0.4 us longer");
template <Gather GATHER> struct ParamsOf { typedef TcvParams type; };
template <> struct ParamsOf<Gather::kCopyEngine> { typedef TcvEngineParams type; };

// One kernel shape: PX pixels x CH channels per block.  SWAP: the channels are the 128 rows of the tensor-core tile and
// the pixels its columns (any multiple of 16 up to PX, so that small maps waste little); otherwise the 128 rows are pixels
// and the columns CH channels.
template <bool F32, int PX, int CH, bool SWAP, Gather GATHER> struct Cfg {
    static const int kParts = F32 ? 3 : 2;                 // operand tiles of 64-byte rows per stage
    static const int kKB = F32 ? 32 : 128;                 // K values per stage (128 source bytes per pixel)
    static const int kWBytes = kParts * CH * 64;
    static const int kN = SWAP ? PX : CH;
    // Accumulators, kN columns each (kN at most 64: three, by size of the terms; beyond: the large products and the small
    // ones; int8: two that take turns, so that no multiply-add waits for the one before it)
    static const int kAcc = accumulators(F32, kN);
    static const int kCols = tensor_columns(F32, kN);
    // Blocks per multiprocessor the registers are cut for (more than tensor memory holds would wait in tcgen05.alloc).  Int8 tiles
    // of 128 columns and layers with few stages are small enough for three (int8 ResNet-50, batch 32: 963 us with 62 to 78
    // registers, 923 us with 64).
    static const int kBlocks = PX > 128 ? 1 : F32 || GATHER == Gather::kValues || 3 * kCols > kTensorColumns ? 2 : 3;
    static_assert(kBlocks * kCols <= kTensorColumns, "a block would wait for tensor memory that its neighbours hold");
    static const int kRow = CH + 4;                        // words per pixel of the exchanged sums (conflict-free 16-byte access)
    static const int kLoadWarps = PX > 128 ? 16 : 8;
    static const int kThreads = (kLoadWarps + 2) * 32;     // + the weight-copy warp and the multiply-add warp
    // Loader warps work in groups that fill alternate stages, so that one's memory and fence latency hides behind the
    // others'; a thread then holds kRPT 16-byte pieces of its next stage in registers.
    // (At most as many groups as stages: a group waits for a stage by phase parity, which tells neighbouring phases apart only.)
    static const int kGroups = 2;
    static const int kGroupThreads = kLoadWarps * 32 / kGroups;
    static const int kRPT = PX * 8 / kGroupThreads;        // pixels per loader thread, kGroupThreads / 8 apart
};

// What a loader thread knows about a pixel: where its window starts.
struct Px {
    int off;   // element offset of (iy, ix, channel 0) from the tensor's start; negative where the window begins in the padding
    int yx;    // iy << 16 | ix (16 bits each); iy far outside for rows past the last pixel
};
const int kNoPixel = -30000;
__device__ __forceinline__ Px load_px(unsigned addr)
{
    Px r;
    asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];\n" : "=r"(r.off), "=r"(r.yx) : "r"(addr));
    return r;
}

// 16 source bytes of one im2col row: 4 floats or 16 int8 values from K position (ky, kx, ci)
template <bool F32>
__device__ __forceinline__ uint4 gather_vec(const TcvParams &p, const Px &r, int ky, int kx, int ci)
{
    const int iy = (r.yx >> 16) + ky, ix = (int)(short)r.yx + kx;
    const bool inside = (unsigned)iy < (unsigned)p.h && (unsigned)ix < (unsigned)p.w && ky < p.kh;
    const int o = r.off + (ky * p.w + kx) * p.c_in + ci;
    return ld_vec_if(reinterpret_cast<const char *>(p.x) + (long long)o * (F32 ? 4 : 1), inside);
}
// mask of the bytes n .. of a word, empty from n = 4 on (the instruction takes shifts beyond the width as the width)
__device__ __forceinline__ unsigned from_byte(int n)
{
    unsigned m;
    asm("shl.b32 %0, 0xffffffff, %1;\n" : "=r"(m) : "r"(8 * n));
    return m;
}
// The same when a pixel's channels are not a multiple of 16 bytes: positions r .. of row ky of the window, whose kw * c_in values
// lie behind each other in memory.  Values of the columns outside the image read as zero; positions past the row's end meet
// zero weights.  Floats come one by one; int8 values as the aligned words that hold any wanted one, shifted into place
// (TAIL: the tensor's last word is not whole, and its bytes are left to patch_tail).
template <bool F32, bool TAIL>
__device__ __forceinline__ uint4 gather_run(const TcvParams &p, const Px &px, int ky, int r)
{
    const int iy = (px.yx >> 16) + ky, ix = (int)(short)px.yx;
    const int a = max(0, -ix * p.c_in - r);
    int b = min(p.kw, p.w - ix) * p.c_in - r;
    if ((unsigned)iy >= (unsigned)p.h || ky >= p.kh) b = 0;
    const int o = px.off + ky * p.w * p.c_in + r;
    if (F32) {
        unsigned v[4];
        const float *x = reinterpret_cast<const float *>(p.x);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            v[j] = ld_word_if(x + o + j, j >= a && j < b);
        }
        return make_uint4(v[0], v[1], v[2], v[3]);
    }
    if (TAIL) b = min(b, p.whole - o);
    const int s = o & 3;
    const char *x = reinterpret_cast<const char *>(p.x) + (o - s);
    const int first = a + s, end = a < min(b, 16) ? min(b, 16) + s : 0;   // the wanted bytes of those words
    unsigned w[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        w[i] = ld_word_if(x + 4 * i, 4 * i + 4 > first && 4 * i < end);
    }
    unsigned v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        v[i] = __funnelshift_r(w[i], w[i + 1], 8 * s) & from_byte(max(a - 4 * i, 0)) & ~from_byte(max(b - 4 * i, 0));
    }
    return make_uint4(v[0], v[1], v[2], v[3]);
}
// The bytes behind the tensor's last whole word, written over the zeros that gather_run gave for them (addr: where its 16 bytes lie
// in shared memory).
__device__ __forceinline__ void patch_tail(const TcvParams &p, const Px &px, int ky, int r, unsigned addr)
{
    const int iy = (px.yx >> 16) + ky, ix = (int)(short)px.yx;
    if ((unsigned)iy >= (unsigned)p.h || ky >= p.kh) return;
    const int a = max(0, -ix * p.c_in - r), b = min(min(p.kw, p.w - ix) * p.c_in - r, 16);
    const int at = p.whole - (px.off + ky * p.w * p.c_in + r);   // position of the first of them
#pragma unroll 1
    for (int j = 0; j < p.tail; ++j)
        if (at + j >= a && at + j < b)
            asm volatile("st.shared.u8 [%0], %1;\n" ::"r"(addr + at + j), "r"((int)ld_act(reinterpret_cast<const signed char *>(p.x) + p.whole + j)) : "memory");
}

// With a pool the pixels of a tile are numbered by window: pixel m is number m % 4 of window m / 4 (maps of even size, so that the
// windows of all images form rows of w_out).  Its place among the output's pixels:
template <bool POOL> __device__ __forceinline__ int place_of(const TcvParams &p, int m)
{
    if (!POOL) return m;
    const int g = m >> 2, r = (int)fdiv((unsigned)g, p.d_wo);
    return (2 * r + ((m >> 1) & 1)) * (2 * p.w_out) + 2 * (g - r * p.w_out) + (m & 1);
}

// act_f32 without branches: with them in, a value took about 60 clocks wherever 16 stood in a row (the activation is
// a kernel argument, so each value jumped over what it did not need).  NaN and the sign of zero come out as they do there.
__device__ __forceinline__ float activate(float z, int act)
{
    const bool none = act == CADNN_ACT_NONE;
    const float top = act == CADNN_ACT_RELU6 ? 6.0f : __int_as_float(0x7f800000);
    z = (z > 0.0f) | none ? z : 0.0f;
    return z > top ? top : z;
}
__device__ __forceinline__ float finish_f(const TcvParams &p, unsigned sum, float sc, float bi, float r)
{
    return activate(__fmaf_rn(__uint_as_float(sum), sc, bi) + r, p.act);
}
__device__ __forceinline__ int byte_of(unsigned w, int j) { return (int)(signed char)((w >> (8 * j)) & 0xff); }
// that byte of a word whose bytes had their top bits turned, as a float: 2^23 + its value + 128 by placing it in a mantissa (a
// conversion takes four times as long)
__device__ __forceinline__ float turned_byte(unsigned w, int j) { return __uint_as_float(__byte_perm(w, 0x4b000000u, 0x7540u + j)) - 8388736.0f; }

// Four int8-layer output values, packed: requant_s8 with the activation's lower bound and the clamp's in one (NaN comes out as that
// bound there too), and rounded by an addition: a value of at most 127 plus 1.5 x 2^23 has it in the low byte, half to even.  The
// epilogue's instructions bound int8 layers of few stages: 18 a value before, 9 (6 without a residual).
__device__ __forceinline__ unsigned finish_q4(const TcvParams &p, const uint4 &t, unsigned r, const float4 &sc, const float4 &bi)
{
    float v[4] = {__fmaf_rn(__int2float_rn((int)t.x), sc.x, bi.x), __fmaf_rn(__int2float_rn((int)t.y), sc.y, bi.y),
                  __fmaf_rn(__int2float_rn((int)t.z), sc.z, bi.z), __fmaf_rn(__int2float_rn((int)t.w), sc.w, bi.w)};
    if (p.residual) {
        r ^= 0x80808080u;
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = __fmaf_rn(turned_byte(r, j), p.res_scale, v[j]);
    }
    const float least = p.act == CADNN_ACT_RELU ? 0.0f : -127.0f;
    unsigned q[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) q[j] = __float_as_uint(fminf(fmaxf(v[j], least), 127.0f) + 12582912.0f);
    return __byte_perm(__byte_perm(q[0], q[1], 0x0040), __byte_perm(q[2], q[3], 0x0040), 0x5410);
}

// Epilogue of 4 consecutive channels of one pixel: sums t, residual r (4 floats, or 4 int8 values in its first word), written
// to channel offset oi of the output; `left` channels exist.
template <bool F32>
__device__ __forceinline__ void finish4(const TcvParams &p, size_t oi, int left, const uint4 &t, const uint4 &r, const float4 &sc, const float4 &bi)
{
    if (F32) {
        float *dst = reinterpret_cast<float *>(p.y) + oi;
        const float4 o = make_float4(finish_f(p, t.x, sc.x, bi.x, __uint_as_float(r.x)), finish_f(p, t.y, sc.y, bi.y, __uint_as_float(r.y)),
                                     finish_f(p, t.z, sc.z, bi.z, __uint_as_float(r.z)), finish_f(p, t.w, sc.w, bi.w, __uint_as_float(r.w)));
        if (p.vec_ok) *reinterpret_cast<float4 *>(dst) = o;
        else {
            dst[0] = o.x;
            if (left > 1) dst[1] = o.y;
            if (left > 2) dst[2] = o.z;
            if (left > 3) dst[3] = o.w;
        }
    } else if (p.out_dtype == CADNN_S8) {
        const unsigned w4 = finish_q4(p, t, r.x, sc, bi);
        signed char *dst = reinterpret_cast<signed char *>(p.y) + oi;
        if (p.vec_ok) *reinterpret_cast<unsigned *>(dst) = w4;
        else
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j < left) dst[j] = (signed char)(w4 >> (8 * j));
    } else {   // int8 layer, 32-bit result: the raw sum, or the requantized value before rounding
        uint4 v = t;
        if (p.out_dtype == CADNN_F32) {
            v.x = __float_as_uint(requant_f32((int)t.x, sc.x, bi.x, p.act, p.residual != nullptr, byte_of(r.x, 0), p.res_scale));
            v.y = __float_as_uint(requant_f32((int)t.y, sc.y, bi.y, p.act, p.residual != nullptr, byte_of(r.x, 1), p.res_scale));
            v.z = __float_as_uint(requant_f32((int)t.z, sc.z, bi.z, p.act, p.residual != nullptr, byte_of(r.x, 2), p.res_scale));
            v.w = __float_as_uint(requant_f32((int)t.w, sc.w, bi.w, p.act, p.residual != nullptr, byte_of(r.x, 3), p.res_scale));
        }
        unsigned *dst = reinterpret_cast<unsigned *>(p.y) + oi;
        if (p.vec_ok) *reinterpret_cast<uint4 *>(dst) = v;
        else {
            dst[0] = v.x;
            if (left > 1) dst[1] = v.y;
            if (left > 2) dst[2] = v.z;
            if (left > 3) dst[3] = v.w;
        }
    }
}
// the residual of those 4 channels of a float layer
__device__ __forceinline__ uint4 load_residual(const TcvParams &p, int m, int co)
{
    const float *res = reinterpret_cast<const float *>(p.residual) + (size_t)m * p.c_out + co;
    if (p.vec_ok) return ld_vec(res);
    uint4 v = make_uint4(0, 0, 0, 0);
    const int left = p.c_out - co;
    v.x = __float_as_uint(ld_act(res));
    if (left > 1) v.y = __float_as_uint(ld_act(res + 1));
    if (left > 2) v.z = __float_as_uint(ld_act(res + 2));
    if (left > 3) v.w = __float_as_uint(ld_act(res + 3));
    return v;
}

// Epilogue of channel ch of a float layer for U consecutive pixels from m on: sums t, residuals r
template <int U>
__device__ __forceinline__ void finish_column(const TcvParams &p, int m, int ch, const unsigned (&t)[U], const unsigned (&r)[U], float sc, float bi)
{
    float *y = reinterpret_cast<float *>(p.y) + (size_t)m * p.ldc + p.c_off + ch;
#pragma unroll
    for (int i = 0; i < U; ++i) {
        st_word_if(y, finish_f(p, t[i], sc, bi, __uint_as_float(r[i])), m + i < p.M);
        y += p.ldc;
    }
}
template <int U> __device__ __forceinline__ void load_column_residual(const TcvParams &p, int m, int ch, unsigned (&r)[U])
{
    const float *res = reinterpret_cast<const float *>(p.residual) + (size_t)m * p.c_out + ch;
#pragma unroll
    for (int i = 0; i < U; ++i) {
        r[i] = ld_word_if(res, p.residual && m + i < p.M);
        res += p.c_out;
    }
}
// Split tile whose rows are channels: a thread takes channel ch (of the tile) and every second group of U pixels of this
// block's share, kBatch groups at a time.  Partial sums lie as [sender][group][channel][U], so that loads and stores of a warp are
// contiguous.  The first batch's residuals are asked for by the caller, ahead of the last multiply-adds: 64 pixels split in two
// (4 groups a thread) waited once per group for them, 2600 of the layer's 16000 clocks.
const int kBatch = 4;
template <int U>
__device__ __forceinline__ void load_split_residual(const TcvParams &p, int m0, int co, int first, int groups, unsigned (&r)[16])
{
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
        unsigned v[U];
#pragma unroll
        for (int i = 0; i < U; ++i) v[i] = 0;
        if (first + 2 * k < groups) load_column_residual<U>(p, m0 + (first + 2 * k) * U, co, v);
#pragma unroll
        for (int i = 0; i < U; ++i) r[k * U + i] = v[i];
    }
}
template <int U>
__device__ __forceinline__ void finish_split_columns(const TcvParams &p, unsigned at, int rows, int m0, int co, int ch, int first, float sc, float bi,
                                                     unsigned (&r)[16])
{
    const int groups = rows / U;
#pragma unroll 1
    for (int g0 = first; g0 < groups; g0 += 2 * kBatch) {
        if (g0 != first) load_split_residual<U>(p, m0, co, g0, groups, r);
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            const int g = g0 + 2 * k;
            if (g >= groups) break;
            unsigned t[U], res[U];
#pragma unroll
            for (int i = 0; i < U; ++i) {
                t[i] = 0;
                res[i] = r[k * U + i];
            }
            const unsigned from = at + (g * 128 + ch) * (U * 4);
#pragma unroll 4
            for (int q = 0; q < p.S; ++q) {
                unsigned v[4];
                const unsigned a = from + q * (rows * 128 * 4);
                if (U == 4) {
                    const uint4 w = lds128(a);
                    v[0] = w.x; v[1] = w.y; v[2] = w.z; v[3] = w.w;
                } else if (U == 2) asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];\n" : "=r"(v[0]), "=r"(v[1]) : "r"(a) : "memory");
                else asm volatile("ld.shared.b32 %0, [%1];\n" : "=r"(v[0]) : "r"(a) : "memory");
#pragma unroll
                for (int i = 0; i < U; ++i) t[i] = __float_as_uint(__uint_as_float(t[i]) + __uint_as_float(v[i]));
            }
            finish_column<U>(p, m0 + g * U, co, t, res, sc, bi);
        }
    }
}
// (What stays in this block is stored, not sent: the link between multiprocessors carries about 15 bytes a clock out of each, and its
// latency is the same for a block itself.  32 pixels x 128 channels split in 2 / 4 / 8, 224 blocks: 1830 / 1820 / 2240 clocks sent to
// all, 1270 / 1430 / 1930 to the others.)
template <int U>
__device__ __forceinline__ void send_columns(const TcvParams &p, unsigned at, unsigned bar, int rank, int rows, int j, int ch, const unsigned (&v)[16])
{
#pragma unroll
    for (int t = 0; t < 16; t += U) {
        const int owner = (int)fdiv((unsigned)(j + t), p.d_rows), row = (j + t) - owner * rows;
        const unsigned a = at + ((rank * (rows / U) + row / U) * 128 + ch) * (U * 4);
        if (owner == rank) {
            if (U == 4) sts128(a, make_uint4(v[t], v[t + 1], v[t + 2], v[t + 3]));
            else
#pragma unroll
                for (int i = 0; i < U; ++i) asm volatile("st.shared.b32 [%0], %1;\n" ::"r"(a + 4 * i), "r"(v[t + i]) : "memory");
        } else send<U>(a, bar, owner, v + t);
    }
}

// (POOL and TAIL are instantiations of their own: as branches at run time they cost the int8 ResNet-50, which has neither such a pool
// nor such a tensor, 0.7 and 0.4 %.)
template <bool F32, int PX, int CH, bool SWAP, Gather GATHER, bool POOL, bool TAIL, typename... Pad>
__global__ void __launch_bounds__(Cfg<F32, PX, CH, SWAP, GATHER>::kThreads, Cfg<F32, PX, CH, SWAP, GATHER>::kBlocks)
tcconv_kernel(const __grid_constant__ typename ParamsOf<GATHER>::type p, Pad...)
{
    const bool VEC = GATHER == Gather::kPieces, ENGINE = GATHER == Gather::kCopyEngine;
    typedef Cfg<F32, PX, CH, SWAP, GATHER> C;
    const int kLoadWarps = C::kLoadWarps;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const unsigned raw32 = (unsigned)__cvta_generic_to_shared(smem_raw);
    const unsigned base = (raw32 + 1023u) & ~1023u;
    const int S = p.stages;
    const unsigned bars = base + p.bar_off;             // full[S], empty[S], done, partial sums received, tensor-memory address
    const unsigned done = bars + 2 * S * 8, recv = done + 8, slot32 = recv + 8;
    volatile unsigned *slot = reinterpret_cast<volatile unsigned *>(smem_raw + (slot32 - raw32));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // (divisions here are multiplications by host-made constants: this is on the critical path of every small layer)
    const int tile = (int)fdiv(blockIdx.x, p.d_S), rank = (int)blockIdx.x - tile * p.S;
    const int mt = (int)fdiv((unsigned)tile, p.d_nt), nt = tile - mt * p.n_nt;
    const int kb0 = rank * p.kb_base + min(rank, p.kb_rem), kb1 = kb0 + p.kb_base + (rank < p.kb_rem ? 1 : 0);
    const int npx = SWAP ? p.npx : PX;                  // pixels of a tile
    const int m0 = mt * npx;
    const unsigned xpart = npx * 64;                    // bytes from one activation part of a stage to the next
    const unsigned xbytes = C::kParts * xpart, stage = xbytes + C::kWBytes;

    const unsigned pxs = slot32 + 16;                   // window starts of the tile's pixels, 8 bytes each
    const unsigned consts = pxs + PX * 8;               // scale and bias of the tile's channels
    const unsigned restile = consts + CH * 8;           // p.res_tile: the residual, CH bytes per pixel that this block finishes
    const int rows = npx / p.S, lo = rows * rank;       // those pixels: rows of them from number lo of the tile on

    // weights of stage kb: its CH x 64-byte tiles, 64 channels (4 KB) per bulk copy
    const int n64 = (p.c_out + 63) / 64;
    auto copy_weights = [&](int kb, int s) {
        const unsigned dst = base + s * stage + xbytes, full = bars + s * 8;
        int cnt = 0;
#pragma unroll
        for (int q = 0; q < CH / 64; ++q) cnt += nt * (CH / 64) + q < n64;
        unsigned bytes = cnt * C::kParts * 4096;
        if (ENGINE) bytes += 2 * kb + 1 < 2 * p.nkb - p.odd_half ? xbytes : xpart;
        mb_expect_tx(full, bytes);
#pragma unroll
        for (int q = 0; q < CH / 64; ++q) {
            const int nb = nt * (CH / 64) + q;
            if (nb >= n64) break;
            const unsigned char *src = p.wimg + ((size_t)nb * p.nkb + kb) * (C::kParts * 4096);
#pragma unroll
            for (int t = 0; t < C::kParts; ++t) bulk_copy(dst + t * (CH * 64) + q * 4096, src + t * 4096, 4096u, full);
        }
    };

    if (warp == kLoadWarps) {
        if (lane == 0) {
            for (int i = 0; i < S; ++i) {
                mb_init(bars + i * 8, ENGINE ? 1 : kLoadWarps / C::kGroups + 1);
                mb_init(bars + (S + i) * 8, 1);
            }
            mb_init(done, 1);
            mb_init(recv, 1);
            asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            // partial sums of this block's pixels from every other block of the cluster
            if (p.S > 1) mb_expect_tx(recv, (unsigned)((npx - rows) * (F32 ? CH : C::kRow) * 4));
        }
    } else if (warp == kLoadWarps + 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(slot32), "r"((unsigned)C::kCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    } else if (!ENGINE && tid < PX) {
        const int m = m0 + tid;
        const int at = POOL ? m >> 2 : m;
        const int img = (int)fdiv((unsigned)at, p.d_hw), q = at - img * p.h_out * p.w_out;
        int oy = (int)fdiv((unsigned)q, p.d_wo), ox = q - oy * p.w_out;
        if (POOL) {
            oy = 2 * oy + ((m >> 1) & 1);
            ox = 2 * ox + (m & 1);
        }
        const int iy = oy * p.stride - p.pad, ix = ox * p.stride - p.pad_w;
        const int yx = (m < p.M && tid < npx ? iy : kNoPixel) * 65536 | (ix & 0xffff), off = ((img * p.h + iy) * p.w + ix) * p.c_in;
        asm volatile("st.shared.v2.b32 [%0], {%1, %2};\n" ::"r"(pxs + tid * 8), "r"(off), "r"(yx) : "memory");
    }
    // loader threads: 16 source bytes (chunk c) of the pixels r0, r0 + kPS, ... in every kGroups-th stage
    const int kPS = C::kGroupThreads / 8;
    const int grp = tid / C::kGroupThreads, c = tid & 7, r0 = tid % C::kGroupThreads / 8;
    // K position of its next stage: kernel row ky, position ci in that row (VEC: channel ci of kernel column kx)
    const int k = (kb0 + grp) * C::kKB + c * (C::kKB / 8);
    int ky = (int)fdiv((unsigned)k, p.d_Rp), kx = 0, ci = k - ky * p.Rp;
    if (VEC) {
        kx = (int)fdiv((unsigned)ci, p.d_ci);
        ci -= kx * p.c_in;
    }
    __syncwarp();
    if (p.S > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;\n" ::: "memory");   // waited for before the first remote copy
    __syncthreads();

    // What the epilogue needs, asked for ahead so that it has arrived by then (loading it there cost a round trip to L2 for every four
    // channels or residual row: 64 -> 256 1x1 int8 with a residual, 128 x 128 tile, 9000 of 12500 clocks).
    auto request_epilogue = [&]() {
        if (tid < CH) {
            const int ch = nt * CH + tid;
            const unsigned a = consts + tid * 4;
            if (p.scale && ch < p.c_out) copy4(a, p.scale + ch);
            else asm volatile("st.shared.f32 [%0], %1;\n" ::"r"(a), "f"(1.0f) : "memory");
            if (p.bias && ch < p.c_out) copy4(a + CH * 4, p.bias + ch);
            else asm volatile("st.shared.f32 [%0], %1;\n" ::"r"(a + CH * 4), "f"(0.0f) : "memory");
        }
        if (!F32 && p.res_tile >= 4) {
            const int log = p.res_tile == 16 ? 4 : 2, per = CH >> log;
            for (int i = tid; i < rows * per; i += kLoadWarps * 32) {
                const int row = i / per, m = m0 + lo + row, at = (i - row * per) << log, ch = nt * CH + at;
                if (m >= p.M || ch >= p.c_out) continue;
                const char *src = reinterpret_cast<const char *>(p.residual) + (size_t)m * p.c_out + ch;
                if (log == 4) copy16(restile + row * CH + at, src);
                else copy4(restile + row * CH + at, src);
            }
        }
    };
    if (ENGINE && warp < kLoadWarps) {
        grid_dep_wait();
        request_epilogue();
        grid_dep_trigger();
    } else if (warp < kLoadWarps) {
        uint4 v[C::kRPT];
        // Window starts stay in registers, and the loads are predicated: with the starts read from shared memory for every stage and
        // the loads behind branches one piece was issued every 100 clocks, 430 of a stage's 1800 (64 pixels).
        // (Where registers are short because three blocks share a multiprocessor, they are read ahead of each stage's loads.)
        const bool kKeep = C::kBlocks < 3 || C::kRPT < 8;
        Px start[C::kRPT];
        auto read_starts = [&]() {
#pragma unroll
            for (int i = 0; i < C::kRPT; ++i) start[i] = load_px(pxs + (r0 + kPS * i) * 8);
        };
        if (kKeep) read_starts();
        auto request = [&]() {
            if (!kKeep) read_starts();
#pragma unroll
            for (int i = 0; i < C::kRPT; ++i) {
                const Px &px = start[i];
                v[i] = VEC ? gather_vec<F32>(p, px, ky, kx, ci) : gather_run<F32, TAIL>(p, px, ky, ci);
            }
            ci += C::kGroups * C::kKB;
            const int wrap = VEC ? p.c_in : p.Rp;
            while (ci >= wrap) {
                ci -= wrap;
                if (!VEC || ++kx == p.kw) { kx = 0; ++ky; }
            }
        };
        grid_dep_wait();
        if (kb0 + grp < kb1) request();
        request_epilogue();
        // swizzled place of the thread's chunk in pixel row r0 of an operand tile (rows kPS apart have the same pattern)
        const unsigned sw = (unsigned)((r0 >> 1) & 3);
        const unsigned at = F32 ? r0 * 64 + ((((unsigned)c >> 1) ^ sw) << 4) + (c & 1) * 8
                                : (c >> 2) * xpart + r0 * 64 + ((((unsigned)c & 3u) ^ sw) << 4);
        int s = grp;
        unsigned round = 0;
        bool alive = true;
        for (int kb = kb0 + grp; kb < kb1; kb += C::kGroups) {
            while (s >= S) { s -= S; ++round; }
            if (round > 0 && alive) alive = mb_wait(bars + (S + s) * 8, (round - 1) & 1u, p.gave_up);
            const unsigned a = base + s * stage + at;
#pragma unroll
            for (int i = 0; i < C::kRPT; ++i) {
                if (SWAP && r0 + kPS * i >= npx) continue;
                if (!F32) sts128(a + i * (kPS * 64), v[i]);
                else {
                    unsigned h0, h1, m0_, m1, l0, l1;
                    split2(__uint_as_float(v[i].x), __uint_as_float(v[i].y), h0, m0_, l0);
                    split2(__uint_as_float(v[i].z), __uint_as_float(v[i].w), h1, m1, l1);
                    sts64(a + i * (kPS * 64), h0, h1);
                    sts64(a + i * (kPS * 64) + xpart, m0_, m1);
                    sts64(a + i * (kPS * 64) + 2 * xpart, l0, l1);
                }
            }
            if (TAIL) {
                const int k = kb * C::kKB + c * (C::kKB / 8), row = (int)fdiv((unsigned)k, p.d_Rp);
#pragma unroll 1
                for (int i = 0; i < C::kRPT && (!SWAP || r0 + kPS * i < npx); ++i)
                    patch_tail(p, load_px(pxs + (r0 + kPS * i) * 8), row, k - row * p.Rp, a + i * (kPS * 64));
            }
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) mb_arrive(bars + s * 8);
            if (kb + C::kGroups < kb1) request();
            s += C::kGroups;
        }
        grid_dep_trigger();
    } else if (warp == kLoadWarps) {
        if (lane > 0 && lane <= Prefetch::kMax && p.ahead.bytes[lane - 1]) {
            // this block's share of the weights of layers to come
            const unsigned long long n = p.ahead.bytes[lane - 1], part = ((n + gridDim.x - 1) / gridDim.x + 127) & ~127ull, lo = part * blockIdx.x;
            if (lo < n)
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n"
                             ::"l"((const char *)p.ahead.at[lane - 1] + lo), "r"((unsigned)(min(part, n - lo) & ~15ull)) : "memory");
        }
        __syncwarp();
        if (elected()) {
            // where the window of the tile's first pixel starts, and the position of the next 64 values of K (copy engine)
            const int at = POOL ? m0 >> 2 : m0, img = (int)fdiv((unsigned)at, p.d_hw), q = at - img * p.h_out * p.w_out;
            const int oy = (int)fdiv((unsigned)q, p.d_wo), ox = q - oy * p.w_out, step = (POOL ? 2 : 1) * p.stride;
            const int iy = oy * step - p.pad, ix = ox * step - p.pad_w;
            int ky = (int)fdiv((unsigned)(kb0 * C::kKB), p.d_Rp), ci = kb0 * C::kKB - ky * p.Rp, kx = (int)fdiv((unsigned)ci, p.d_ci);
            ci -= kx * p.c_in;
            auto pixels = [&](int s) {
                if constexpr (GATHER == Gather::kCopyEngine) {
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    if (ky == p.kh) break;
                    const unsigned dst = base + s * stage + t * xpart;
                    if (!POOL) copy_pixels(dst, &p.pixels, ci, ix, iy, img, kx, ky, bars + s * 8);
                    else   // a quarter of the rows for each place in a window
#pragma unroll
                        for (int r = 0; r < 4; ++r)
                            copy_pixels(dst + r * (xpart / 4), &p.pixels, ci, ix, iy, img, kx + (r & 1) * p.stride, ky + (r >> 1) * p.stride, bars + s * 8);
                    ci += 64;
                    if (ci == p.c_in) {
                        ci = 0;
                        if (++kx == p.kw) { kx = 0; ++ky; }
                    }
                }
                }
            };
            const int ahead = ENGINE ? min(S, kb1 - kb0) : 0;
            if (ENGINE) {   // weights do not wait for the previous layer
                for (int i = 0; i < ahead; ++i) copy_weights(kb0 + i, i);
                grid_dep_wait();
                for (int i = 0; i < ahead; ++i) pixels(i);
            }
            int s = ahead == S ? 0 : ahead;
            unsigned round = ahead == S;
            for (int kb = kb0 + ahead; kb < kb1; ++kb) {
                if (round > 0 && !mb_wait(bars + (S + s) * 8, (round - 1) & 1u, p.gave_up)) break;
                copy_weights(kb, s);
                if (ENGINE) pixels(s);
                if (++s == S) { s = 0; ++round; }
            }
        }
    } else if (elected()) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const unsigned tmem = *slot;
        const int N = SWAP ? npx : CH;
        const unsigned fmt = (F32 ? 1u << 4 : 2u << 4) | (1u << 7) | (1u << 10) | (8u << 24);
        const unsigned id1 = fmt | ((unsigned)(N >> 3) << 17), id2 = fmt | ((unsigned)(2 * N >> 3) << 17);
        const unsigned ap = SWAP ? CH * 64 : xpart, bp = SWAP ? xpart : CH * 64;   // bytes from part to part of the two operands
        int s = 0;
        unsigned round = 0, acc = 0;
        for (int kb = kb0; kb < kb1; ++kb) {
            if (!mb_wait(bars + s * 8, round & 1u, p.gave_up)) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const unsigned xs = base + s * stage, ws = xs + xbytes;
            const unsigned a = SWAP ? ws : xs, w = SWAP ? xs : ws;
            if (F32) {
#pragma unroll
                for (int kk = 0; kk < 2; ++kk) {
                    const unsigned long long a1 = smem_desc(a + kk * 32), a2 = smem_desc(a + ap + kk * 32), a3 = smem_desc(a + 2 * ap + kk * 32);
                    const unsigned long long b1 = smem_desc(w + kk * 32), b2 = smem_desc(w + bp + kk * 32), b3 = smem_desc(w + 2 * bp + kk * 32);
                    // The parts of b lie behind each other, and so do the accumulators: one instruction can take several
                    // parts at once, which reads the a tile from shared memory less often.
                    if (C::kAcc == 3) {   // columns [large | 2^-9 terms | 2^-18 terms]
                        mma<true>(tmem, a1, b1, fmt | ((unsigned)(3 * N >> 3) << 17), acc);   // a1 b1 | a1 b2 | a1 b3
                        mma<true>(tmem + N, a2, b1, id2, 1);                                  // a2 b1 | a2 b2
                        mma<true>(tmem + 2 * N, a3, b1, id1, 1);                              // a3 b1
                    } else {              // columns [large | small terms]
                        if (2 * N <= 256) mma<true>(tmem, a1, b1, id2, acc);
                        else {
                            mma<true>(tmem, a1, b1, id1, acc);
                            mma<true>(tmem + N, a1, b2, id1, acc);
                        }
                        mma<true>(tmem + N, a2, b1, id1, 1);
                        mma<true>(tmem + N, a2, b2, id1, 1);
                        mma<true>(tmem + N, a1, b3, id1, 1);
                        mma<true>(tmem + N, a3, b1, id1, 1);
                    }
                    acc = 1;
                }
            } else {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    mma<false>(tmem + (kk & 1) * N, smem_desc(a + (kk >> 1) * ap + (kk & 1) * 32), smem_desc(w + (kk >> 1) * bp + (kk & 1) * 32), id1,
                               kk < 2 ? acc : 1);
                acc = 1;
            }
            tc_commit(bars + (S + s) * 8);
            if (++s == S) { s = 0; ++round; }
        }
        tc_commit(done);
    }
    __syncwarp();
    if (warp < kLoadWarps) {
        if (!F32 && p.res_tile == 1) {   // channels of no multiple of 4: byte by byte, 16 on their way at once
#pragma unroll 1
            for (int i = tid; i < rows * CH; i += kLoadWarps * 32 * 16) {
                int b[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    const int at = i + k * kLoadWarps * 32, m = m0 + lo + at / CH, ch = nt * CH + at % CH;
                    b[k] = 0;
                    if (at < rows * CH && m < p.M && ch < p.c_out) b[k] = ld_act(reinterpret_cast<const signed char *>(p.residual) + (size_t)m * p.c_out + ch);
                }
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    const int at = i + k * kLoadWarps * 32;
                    if (at < rows * CH) asm volatile("st.shared.u8 [%0], %1;\n" ::"r"(restile + at), "r"(b[k]) : "memory");
                }
            }
        }
        copies_landed();
        asm volatile("bar.sync 1, %0;\n" ::"n"(C::kLoadWarps * 32) : "memory");
    }

    // ---- epilogue (code that runs once per block costs its instruction fetches: loops stay rolled) ----
    const unsigned tmem = *slot;
    const int kVec = CH / 4, kStep = kLoadWarps * 32 / kVec;
    const int col = (tid % kVec) * 4, r1 = tid / kVec, co = nt * CH + col;
    const bool mine = warp < kLoadWarps && co < p.c_out;
    // (rows of the tile are channels:) this thread's channel in float tiles, and residuals of its next 16 pixels
    const int lch = (warp & 3) * 32 + lane, cch = nt * CH + lch;
    const bool column = F32 && SWAP && warp < kLoadWarps && cch < p.c_out;
    unsigned rc[16];
    // residuals of the next kAhead rows (four channels each)
    const int kAhead = 4;
    uint4 res[kAhead];
    auto load_rows = [&](int row) {
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            const int m = m0 + lo + row + i * kStep;
            res[i] = make_uint4(0, 0, 0, 0);
            if (p.residual && row + i * kStep < rows && m < p.M) res[i] = load_residual(p, m, co);
        }
    };
    // of the pixels this thread finishes first; on their way while the last multiply-adds run
    if (F32 && SWAP) {
#pragma unroll
        for (int i = 0; i < 16; ++i) rc[i] = 0;
        if (column && p.residual) {
            if (p.S == 1) load_column_residual<16>(p, m0 + (warp >> 2) * 16, cch, rc);
            else if (rows % 4 == 0) load_split_residual<4>(p, m0 + lo, cch, tid >> 7, rows / 4, rc);
            else if (rows % 2 == 0) load_split_residual<2>(p, m0 + lo, cch, tid >> 7, rows / 2, rc);
            else load_split_residual<1>(p, m0 + lo, cch, tid >> 7, rows, rc);
        }
    } else if (F32 && mine) load_rows(r1);
    __syncwarp();
    if (p.S > 1) asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");   // every block has initialised its barriers
    if (warp < kLoadWarps) {
        // a warp can read the 32 rows 32 q ..; the warps with the same q take turns on groups of 16 columns
        const int q = warp & 3, N = SWAP ? npx : CH;
        const unsigned from = tmem + ((unsigned)(q * 32) << 16);
        mb_wait(done, 0u, p.gave_up);
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
#pragma unroll 1
        for (int j = (warp >> 2) * 16; j < N; j += kLoadWarps * 4) {
            unsigned v[16], u[16];
            tmem_ld16(from + j, v);
            tmem_ld16(from + N + j, u);
            if (F32 && C::kAcc == 3) {
                unsigned t3[16];
                tmem_ld16(from + 2 * N + j, t3);
                tmem_wait();
                tmem_arrived(u);
                tmem_arrived(t3);
#pragma unroll
                for (int t = 0; t < 16; ++t) u[t] = __float_as_uint(__uint_as_float(u[t]) + __uint_as_float(t3[t]));
            } else {
                tmem_wait();
                tmem_arrived(u);
            }
            tmem_arrived(v);
#pragma unroll
            for (int t = 0; t < 16; ++t) v[t] = F32 ? __float_as_uint(__uint_as_float(v[t]) + __uint_as_float(u[t])) : v[t] + u[t];
            if (F32 && p.S > 1) {   // each pixel's sums to the block of the cluster that finishes it
                if (SWAP) {
                    if (rows % 4 == 0) send_columns<4>(p, base + p.recv_off, recv, rank, rows, j, lch, v);
                    else if (rows % 2 == 0) send_columns<2>(p, base + p.recv_off, recv, rank, rows, j, lch, v);
                    else send_columns<1>(p, base + p.recv_off, recv, rank, rows, j, lch, v);
                } else {
                    const int px = q * 32 + lane, owner = (int)fdiv((unsigned)px, p.d_rows), row = rank * rows + px - owner * rows;
#pragma unroll
                    for (int t = 0; t < 16; t += 4) {
                        const unsigned a = base + p.recv_off + (row * C::kRow + j + t) * 4;
                        if (owner == rank) sts128(a, make_uint4(v[t], v[t + 1], v[t + 2], v[t + 3]));
                        else send<4>(a, recv, owner, v + t);
                    }
                }
            } else if (F32 && SWAP) {   // 16 pixels of one channel, straight to memory: a warp writes 128 contiguous bytes of each pixel
                if (column) {
                    finish_column<16>(p, m0 + j, cch, v, rc, lds32(consts + lch * 4), lds32(consts + (CH + lch) * 4));
                    if (p.residual && j + kLoadWarps * 4 < N) load_column_residual<16>(p, m0 + j + kLoadWarps * 4, cch, rc);
                }
            } else if (SWAP) {   // to shared memory as [pixel][channel] (over the stages: all of them have been read)
                const unsigned at = base + (j * C::kRow + lch) * 4;
#pragma unroll
                for (int t = 0; t < 16; ++t) asm volatile("st.shared.b32 [%0], %1;\n" ::"r"(at + t * C::kRow * 4), "r"(v[t]) : "memory");
            } else {
                const unsigned at = base + ((q * 32 + lane) * C::kRow + j) * 4;
#pragma unroll
                for (int t = 0; t < 16; t += 4) sts128(at + t * 4, make_uint4(v[t], v[t + 1], v[t + 2], v[t + 3]));
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        if (!F32 && p.S > 1) asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    }
    __syncthreads();
    if (warp == kLoadWarps + 1) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"((unsigned)C::kCols) : "memory");
    }
    if (F32 && SWAP && p.S == 1) return;
    const unsigned slice = rows * C::kRow * 4;   // partial sums of one sender (as [pixel][channel])
    if (F32) {
        if (warp >= kLoadWarps) return;
        if (SWAP && p.S > 1) {
            mb_wait(recv, 0u, p.gave_up);
            if (!column) return;
            const unsigned at = base + p.recv_off;
            const float sc = lds32(consts + lch * 4), bi = lds32(consts + (CH + lch) * 4);
            if (rows % 4 == 0) finish_split_columns<4>(p, at, rows, m0 + lo, cch, lch, tid >> 7, sc, bi, rc);
            else if (rows % 2 == 0) finish_split_columns<2>(p, at, rows, m0 + lo, cch, lch, tid >> 7, sc, bi, rc);
            else finish_split_columns<1>(p, at, rows, m0 + lo, cch, lch, tid >> 7, sc, bi, rc);
            return;
        }
        if (p.S > 1) mb_wait(recv, 0u, p.gave_up);
    } else if (p.S > 1) {
        // Int8 layers exchange through staged tiles and bulk copies: packed stores need 4 channels in a thread, and the register
        // route's code costs them a third resident block per multiprocessor (int8 ResNet-50, batch 8: 421 against 451 us).
        if (tid < p.S && tid != rank) send_bulk(base + p.recv_off + rank * slice, base + tid * slice, slice, recv, tid);
        __syncwarp();
        if (warp < kLoadWarps) mb_wait(recv, 0u, p.gave_up);
        __syncwarp();
        // this block has received everything, so the others may go; it goes itself when they have received what it sent
        asm volatile("barrier.cluster.arrive.relaxed.aligned;\n" ::: "memory");
    }
    if (mine) {
        const float4 sc = lds_float4(consts + col * 4), bi = lds_float4(consts + (CH + col) * 4);
        if (POOL) {   // a thread takes the four pixels of a window
#pragma unroll 1
            for (int g = r1; 4 * g < rows && m0 + lo + 4 * g < p.M; g += kStep) {
                // (the copy engine leaves a window's pixels a quarter of the tile apart)
                const int next = ENGINE ? npx / 4 : 1;
                const unsigned in = ((ENGINE ? g : 4 * g) * C::kRow + col) * 4, at = base + p.recv_off + in, own = base + rank * slice + in;
                const int m = m0 + lo + 4 * g;
                unsigned best = 0x80808080u;
#pragma unroll 1
                for (int i = 0; i < 4; ++i) {
                    uint4 t = lds128(own + i * next * C::kRow * 4);
#pragma unroll 4
                    for (int q = 1; q < p.S; ++q) {
                        const uint4 u = lds128(at + i * next * C::kRow * 4 + (q <= rank ? q - 1 : q) * slice);
                        t.x += u.x; t.y += u.y; t.z += u.z; t.w += u.w;
                    }
                    const unsigned v = finish_q4(p, t, 0, sc, bi);
                    *reinterpret_cast<unsigned *>(reinterpret_cast<signed char *>(p.y) + (size_t)place_of<POOL>(p, m + i) * p.c_out + co) = v;
                    best = __vmaxs4(best, v);
                }
                *reinterpret_cast<unsigned *>(p.pooled + (size_t)(m >> 2) * p.c_out + co) = best;
            }
        } else {
            // (this block's own sums: int8 where they were staged, float among the received ones)
            unsigned at = base + p.recv_off + (r1 * C::kRow + col) * 4, own = at + rank * slice;
            if (!F32 || p.S == 1) own -= p.recv_off;
#pragma unroll 1
            for (int row = r1; row < rows; row += F32 ? kAhead * kStep : kStep) {
                uint4 r[kAhead];
                if (F32) {
#pragma unroll
                    for (int i = 0; i < kAhead; ++i) r[i] = res[i];
                    if (row + kAhead * kStep < rows) load_rows(row + kAhead * kStep);
                }
#pragma unroll
                for (int i = 0; i < (F32 ? kAhead : 1); ++i) {
                    const int m = m0 + lo + row + i * kStep;
                    if (row + i * kStep >= rows || m >= p.M) break;
                    uint4 t = lds128(own);
                    if (!F32) {
                        r[0] = make_uint4(0, 0, 0, 0);
                        if (p.res_tile) r[0].x = __float_as_uint(lds32(restile + row * CH + col));
                    }
#pragma unroll 4
                    for (int q = 1; q < p.S; ++q) {
                        const uint4 u = lds128(at + (q <= rank ? q - 1 : q) * slice);
                        if (F32) {
                            t.x = __float_as_uint(__uint_as_float(t.x) + __uint_as_float(u.x));
                            t.y = __float_as_uint(__uint_as_float(t.y) + __uint_as_float(u.y));
                            t.z = __float_as_uint(__uint_as_float(t.z) + __uint_as_float(u.z));
                            t.w = __float_as_uint(__uint_as_float(t.w) + __uint_as_float(u.w));
                        } else {
                            t.x += u.x; t.y += u.y; t.z += u.z; t.w += u.w;
                        }
                    }
                    at += kStep * C::kRow * 4;
                    own += kStep * C::kRow * 4;
                    finish4<F32>(p, (size_t)m * p.ldc + p.c_off + co, p.c_out - co, t, r[i], sc, bi);
                }
            }
        }
    }
    if (!F32 && p.S > 1) {
        __syncwarp();
        asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    }
}

constexpr int ceil_div(int a, int b) { return (a + b - 1) / b; }

struct Pick {
    int px, ch, split;   // pixels and channels per block, blocks per cluster
};

const int kSmemOfSm = 228 * 1024, kSmemReserved = 1024;   // shared memory of a multiprocessor, and what the system takes of it per block

// Shared memory of one block: its pipeline depth, where the exchanged sums and the barriers lie, and its size.
struct SmemPlan {
    int stages, recv_off, bar_off, bytes;
};
constexpr int tile_pixels(const Pick &k) { return k.ch == 64 ? 128 : k.px <= 64 ? 64 : k.px <= 128 ? 128 : 256; }   // PX of the kernel shape
constexpr SmemPlan plan_smem(bool f32, const Pick &k, int nkb, bool res_tile)
{
    const int PX = tile_pixels(k);
    const bool swap = k.ch == 128;
    const int stage = (f32 ? 3 : 2) * 64 * (k.px + k.ch), out = k.px * (k.ch + (f32 && swap ? 0 : 4)) * 4;
    const int res = res_tile ? k.px / k.split * k.ch : 0;
    const int budget = (PX > 128 ? 216 : 108) * 1024 - res;   // two blocks share a multiprocessor but for the largest shape
    SmemPlan s = {};
    s.stages = std::max(2, std::min(std::min(f32 ? 4 : 6, std::max(2, ceil_div(nkb, k.split))), (budget - (k.split > 1 ? out : 0)) / stage));
    // sums staged over the stages: int8 tiles, and unsplit float tiles whose rows are pixels
    s.recv_off = std::max(s.stages * stage, !f32 || (!swap && k.split == 1) ? out : 0);
    s.bar_off = (s.recv_off + (k.split > 1 ? out : 0) + 127) / 128 * 128;
    s.bytes = s.bar_off + 1024 + 128 + PX * 8 + k.ch * 8 + res;
    // Blocks of a cluster wait for each other while they hold tensor memory.  Were more of them resident than it has columns for,
    // two clusters could each hold what the other's last block waits for; so a block of c columns takes more than c / 640 of the
    // multiprocessor's shared memory, and five quarters of the columns never fit.  (Other blocks hold columns too, but finish by
    // themselves.)
    if (k.split > 1) s.bytes = std::max(s.bytes, (tensor_columns(f32, swap ? PX : k.ch) / 128 * kSmemOfSm / 5 - kSmemReserved + 128) & ~127);
    return s;
}
constexpr bool clusters_find_tensor_memory()
{
    for (int f32 = 0; f32 < 2; ++f32)
        for (int px = 16; px <= 128; px += 16)
            for (int ch = 64; ch <= 128; ch += 64)
                for (int split = 2; split <= 16; ++split)
                    for (int nkb = split; nkb <= 5 * split; ++nkb) {
                        const Pick k = {ch == 64 ? 128 : px, ch, split};
                        if (5 * (plan_smem(f32, k, nkb, false).bytes + kSmemReserved) <= tensor_columns(f32, ch == 64 ? 64 : tile_pixels(k)) / 128 * kSmemOfSm)
                            return false;
                    }
    return true;
}
static_assert(clusters_find_tensor_memory(), "clusters of split tiles could wait for each other's tensor memory");

// Block shape of a layer: the one a time model calls the fastest.  The model is linear in what a block does, with
// coefficients fitted to 37500 measured shapes (1950 layers: those of the workloads at batch 1 to 128, and random ones, launched back to
// back as programmatic dependents; least squares, then a search that lowers the excess of the chosen shapes over 4 of 5 layers):
//   time = start + P (b2 + n (c2 + d2 px / 64)) + Q (b1 + n (c1 + d1 px / 64))   [microseconds]
// n = stages per block, P = rounds in which every multiprocessor runs two blocks, Q = rounds with one.  How many clusters
// of a size run at once (a cluster has to fit one GPC) is the table cap1 / cap2 in choose, as cudaOccupancyMaxActiveClusters
// reported it on a B200.
// Mean excess of the chosen over the best measured shape, on the fifth that was left out: 0.8 to 1.7 % by gather (with the coefficients
// of the kernel before its epilogue and issue were mended 3.2 to 4.8 %).
struct Cost {
    float start, b2, c2, d2, b1, c1, d1;
};
const Cost kCost[5][9] = {   // by gather; 128 px x 64 ch, then up to 32, 64 and 128 px x 128 ch, each unsplit and split; 256 px x 128 ch
    // float, 16 bytes at a time
    {{0.871f, 2.86f, 0.0643f, 0.399f, 4.29f, 0.0f, 0.197f},
     {1.30f, 7.30f, 0.0f, 0.329f, 3.47f, 0.0405f, 0.185f},
     {0.0f, 2.12f, 0.617f, 0.297f, 1.93f, 0.267f, 0.191f},
     {0.588f, 2.95f, 0.221f, 0.392f, 1.79f, 0.263f, 0.232f},
     {0.0392f, 3.60f, 0.255f, 0.337f, 2.70f, 0.196f, 0.165f},
     {1.41f, 3.86f, 0.0385f, 0.488f, 2.11f, 0.155f, 0.312f},
     {2.47f, 3.83f, 0.208f, 0.457f, 1.43f, 0.342f, 0.307f},
     {0.638f, 0.0973f, 0.0747f, 0.0865f, 11.6f, 0.143f, 0.399f},
     {0.0f, 0.0219f, 0.0f, 0.0551f, 5.67f, 0.0278f, 0.255f}},
    // float, one value at a time
    {{2.07f, 1.89f, 0.0229f, 0.521f, 2.02f, 0.00927f, 0.336f},
     {0.00999f, 5.93f, 0.0f, 0.567f, 4.70f, 0.00640f, 0.290f},
     {0.0f, 1.54f, 0.503f, 0.640f, 1.56f, 0.292f, 0.309f},
     {0.158f, 3.60f, 0.327f, 0.375f, 2.03f, 0.430f, 0.0f},
     {0.153f, 2.78f, 0.143f, 0.786f, 2.40f, 0.177f, 0.298f},
     {0.905f, 3.28f, 0.0372f, 0.680f, 2.53f, 0.0833f, 0.381f},
     {3.42f, 1.99f, 0.195f, 0.692f, 2.18f, 0.232f, 0.213f},
     {0.0411f, 0.0227f, 0.0783f, 0.0140f, 5.94f, 0.338f, 0.134f},
     {0.0f, 0.0144f, 0.0142f, 0.0382f, 4.83f, 0.0834f, 0.280f}},
    // int8, copy engine
    {{0.0f, 0.504f, 0.427f, 0.333f, 1.99f, 0.0f, 0.200f},
     {0.0f, 2.41f, 0.0875f, 0.870f, 3.05f, 0.0f, 0.125f},
     {0.358f, 1.39f, 0.310f, 0.0f, 0.335f, 0.218f, 0.526f},
     {1.56f, 1.72f, 0.108f, 0.0430f, 0.0f, 0.161f, 0.417f},
     {0.0f, 2.71f, 0.115f, 0.457f, 17.7f, 1.94f, 2.14f},
     {2.47f, 1.76f, 0.0f, 0.128f, 0.279f, 0.379f, 0.762f},
     {0.0f, 1.55f, 0.300f, 0.505f, 5.85f, 0.446f, 0.0778f},
     {6.86f, 5.70f, 0.0f, 0.0412f, 10.9f, 0.122f, 0.452f},
     {0.0f, 12.4f, 0.0f, 0.613f, 7.77f, 0.0f, 0.186f}},
    // int8, 16 bytes at a time
    {{1.31f, 1.43f, 0.0624f, 0.430f, 0.0229f, 0.0677f, 0.341f},
     {1.12f, 16.0f, 0.0318f, 0.0422f, 1.94f, 0.122f, 0.262f},
     {0.0f, 1.35f, 0.282f, 0.567f, 0.456f, 0.156f, 0.732f},
     {0.906f, 1.29f, 0.774f, 0.588f, 0.0877f, 0.163f, 0.425f},
     {1.20f, 2.45f, 0.0359f, 0.617f, 1.33f, 0.212f, 0.209f},
     {2.55f, 2.11f, 0.0f, 0.533f, 0.340f, 0.0189f, 0.331f},
     {0.184f, 6.32f, 2.73f, 0.0299f, 6.04f, 0.126f, 0.203f},
     {0.186f, 46.7f, 0.242f, 1.48f, 5.14f, 0.0252f, 0.251f},
     {0.451f, 12.7f, 0.00654f, 2.34f, 4.30f, 0.0272f, 0.225f}},
    // int8, shifted words
    {{2.23f, 2.74f, 0.393f, 0.795f, 4.38f, 0.0928f, 0.328f},
     {3.30f, 1.99f, 0.0623f, 0.764f, 22.6f, 0.0870f, 0.382f},
     {0.313f, 2.48f, 0.560f, 1.03f, 1.65f, 0.0905f, 0.845f},
     {0.0f, 9.62f, 0.0393f, 6.15f, 0.0f, 0.552f, 0.632f},
     {1.15f, 3.60f, 0.297f, 0.651f, 2.52f, 0.114f, 0.598f},
     {1.29f, 3.16f, 0.0279f, 0.797f, 1.54f, 0.0f, 0.666f},
     {1.20f, 4.90f, 0.638f, 0.744f, 4.41f, 0.0f, 0.553f},
     {4.58f, 4.90f, 0.373f, 1.89f, 2.11f, 0.200f, 1.02f},
     {0.469f, 11.2f, 0.190f, 0.309f, 6.23f, 0.452f, 0.343f}}};

// kind: row of kCost
Pick choose(int kind, int c_out, long long M, int nkb, bool res_tile)
{
    const bool f32 = kind < 2;
    Pick best = {128, 64, 1};
    double best_t = 1e300;
    auto consider = [&](int px, int ch) {
        const long long tiles = (M + px - 1) / px * ceil_div(c_out, ch);
        for (int log = 0; log <= (px > 128 ? 0 : 4); ++log) {
            const int split = 1 << log;
            if (split > nkb || px % split) break;
            if (split > 1 && tiles * split > 330) break;      // the grid already fills the chip twice
            static const int cap1[5] = {148, 74, 33, 15, 7}, cap2[5] = {296, 148, 71, 33, 14};
            const Pick k = {px, ch, split};
            const bool two = plan_smem(f32, k, nkb, res_tile).bytes <= 113 * 1024;
            long long P = 0, Q = 0;
            if (two) {
                P = tiles / cap2[log];
                const long long rest = tiles - P * cap2[log];
                if (rest > cap1[log]) ++P;
                else if (rest > 0) Q = 1;
            } else Q = (tiles + cap1[log] - 1) / cap1[log];
            const Cost &c = kCost[kind][px > 128 ? 8 : (ch == 64 ? 0 : px <= 32 ? 2 : px <= 64 ? 4 : 6) + (split > 1)];
            const double n = ceil_div(nkb, split), u = px / 64.0;
            double t = c.start + P * (c.b2 + n * (c.c2 + c.d2 * u)) + Q * (c.b1 + n * (c.c1 + c.d1 * u));
            // In a network a layer's blocks stand in the way of the next one's, which start early where there is room: half a microsecond
            // for a chip full of them (ResNet-50, batch 1: 279.4 us without, 275.0 with 0.5, 275.9 with 1; int8, batch 8: 339.8, 339.8, 345.9).
            t += 0.5 * (double)std::min(tiles * split, 296ll) / 296;
            if (t < best_t) { best_t = t; best = k; }
        }
    };
    consider(128, 64);
    static const int fixed[] = {32, 64, 96, 112, 128, 192, 208, 224, 256};
    for (int px : fixed) consider(px, 128);
    for (int q = 1; q <= 16; ++q) {   // the pixels cut into q equal tiles
        const long long px = ((M + q - 1) / q + 15) / 16 * 16;
        if (px <= 256) consider((int)px, 128);
        if (px <= 16) break;
    }
    return best;
}

template <bool F32, int PX, int CH, bool SWAP, Gather GATHER, bool POOL, bool TAIL>
cadnn_status launch_one(typename ParamsOf<GATHER>::type p, int blocks, bool pdl, cudaStream_t st)
{
    const auto kern = []() {
        if constexpr (GATHER == Gather::kCopyEngine) return tcconv_kernel<F32, PX, CH, SWAP, GATHER, POOL, TAIL, LaunchPad>;
        else return tcconv_kernel<F32, PX, CH, SWAP, GATHER, POOL, TAIL>;
    }();
    typedef Cfg<F32, PX, CH, SWAP, GATHER> C;
    const SmemPlan sp = plan_smem(F32, {p.npx, CH, p.S}, p.nkb, p.res_tile != 0);
    if (sp.stages < C::kGroups || sp.stages * C::kParts * 64 * (p.npx + CH) > sp.recv_off || p.npx > PX) return CADNN_E_UNSUPPORTED;
    p.stages = sp.stages;
    p.recv_off = sp.recv_off;
    p.bar_off = sp.bar_off;
    const int smem = sp.bytes;
    static SmemLimit lim;
    cadnn_status rs = raise_smem_limit((const void *)kern, smem, &lim);
    if (rs != CADNN_OK) return rs;
    if (p.S > 8) CADNN_CUDA_TRY(cudaFuncSetAttribute((const void *)kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks, 1, 1);
    cfg.blockDim = dim3(C::kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (pdl) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (p.S > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = (unsigned)p.S;
        attr[n].val.clusterDim.y = 1;
        attr[n++].val.clusterDim.z = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    if constexpr (GATHER == Gather::kCopyEngine) CADNN_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, p, LaunchPad()));
    else CADNN_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, p));
    return CADNN_OK;
}

template <bool F32, Gather GATHER, bool POOL = false, bool TAIL = false> cadnn_status launch_shape(const typename ParamsOf<GATHER>::type &p, int ch, int blocks, bool pdl, cudaStream_t st)
{
    if (ch == 64) return launch_one<F32, 128, 64, false, GATHER, POOL, TAIL>(p, blocks, pdl, st);
    if (p.npx <= 64) return launch_one<F32, 64, 128, true, GATHER, POOL, TAIL>(p, blocks, pdl, st);
    if (TAIL || p.npx <= 128) return launch_one<F32, 128, 128, true, GATHER, POOL, TAIL>(p, blocks, pdl, st);   // (256 pixels would spill registers)
    return launch_one<F32, 256, 128, true, GATHER, POOL, false>(p, blocks, pdl, st);
}

}  // namespace

namespace {
// K positions per kernel row: kw * c_in values, padded to whole 16-byte pieces
int row_positions(const cadnn_layer_desc &d)
{
    const int per16 = d.dtype == CADNN_S8 ? 16 : 4;
    return ceil_div(d.kw * d.c_in, per16) * per16;
}
int stages_of(const cadnn_layer_desc &d) { return ceil_div(d.kh * row_positions(d), d.dtype == CADNN_S8 ? 128 : 32); }
}  // namespace

// When the dense route is taken.  Per multiply-add of the full layer the tensor cores cost the same whatever the mask; the
// sparse kernels cost per stored weight.  Measured on the 3x3 and 1x1 layers of the workloads at batch 1 to 32 (microseconds
// against density) the lines cross below 3 per cent, for float and for int8.  Float layers of at most 64 output channels keep the sparse
// kernels' 32-bit multiply-adds up to 6 per cent: the split products would be faster from 2 on (16 to 64 channels, batch 1 to 16, 6.5 to
// 8.2 against 8.2 to 14.4), but with so few terms a sum they are not everywhere as close to 64 bits (2-norm errors at 2.5 to 5.5 per cent, dense
// over sparse: 28 x 28 maps 0.55 to 1.00, 14 x 14 maps 0.70 to 1.09; activations of 1e-35, 4 per cent: 2.4e-6 against 6.3e-8).
bool tcv_pays(const cadnn_layer_desc &d, int64_t nnz)
{
    const double density = (double)nnz / ((double)d.c_out * d.kh * d.kw * d.c_in);
    return density >= (d.dtype == CADNN_F32 && d.c_out <= 64 ? 0.06 : 0.025);
}

namespace {

// Where weight (output channel co, kernel row ky, position i = kx * c_in + ci of that row) lies in the image
// [64-channel tile][stage][part][64 rows][64 bytes], rows swizzled like the operand tiles.  Parts: the three bf16 terms of a
// float, or the two 64-value halves of an int8 stage.
struct ImageDims {
    int nkb, Rp;
};
__host__ __device__ inline size_t image_at(const ImageDims &d, bool f32, int co, int ky, int i)
{
    const int k = ky * d.Rp + i, r = co & 63, sw = (r >> 1) & 3;
    const size_t tile = (size_t)(co >> 6) * d.nkb;
    if (f32) {
        const int c = k & 31;
        return (tile + (k >> 5)) * 3 * 4096 + r * 64 + (((c >> 3) ^ sw) << 4) + (c & 7) * 2;
    }
    const int c = k & 63;
    return ((tile + (k >> 7)) * 2 + ((k >> 6) & 1)) * 4096 + r * 64 + (((c >> 4) ^ sw) << 4) + (c & 15);
}
__host__ __device__ inline void image_put(unsigned char *image, const ImageDims &d, int co, int ky, int i, float v)
{
    __nv_bfloat16 *at = reinterpret_cast<__nv_bfloat16 *>(image + image_at(d, true, co, ky, i));
    for (int t = 0; t < 3; ++t) {
        const __nv_bfloat16 b = __float2bfloat16_rn(v);
        at[t * 2048] = b;
        v -= __bfloat162float(b);
    }
}

// The image written on the device from the sparse image that is there already (tiled CSR records: a header of row starts,
// then {value, tile offset} entries): one warp per (channel chunk, packed row).  Padding entries have the value 0, as the
// image has everywhere else.
struct ExpandParams {
    const uint32_t *ent;
    const int32_t *perm;
    unsigned char *image;
    ImageDims dims;
    int n_chunks, c_pad, n_groups, G, hdr_words, block_words, CIc, PPb, pitch, half, linear, s8, c_in;
};
__global__ void __launch_bounds__(256) expand_kernel(const ExpandParams p)
{
    const int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int c = blockIdx.y;
    if (row >= p.c_pad) return;
    const int co = p.perm[row];
    if (co < 0) return;
    const uint32_t *blk = p.ent + ((size_t)c * p.n_groups + row / p.G) * p.block_words, *ents = blk + p.hdr_words;
    const int first = (int)blk[row % p.G], last = (int)blk[row % p.G + 1];
    for (int e = first + lane; e < last; e += 32) {
        uint32_t off, bits;
        if (p.s8) {
            bits = ents[e] & 0xffu;
            off = ents[e] >> 8;
        } else {
            bits = ents[2 * (size_t)e];
            off = ents[2 * (size_t)e + 1];
        }
        if ((bits << 1) == 0) continue;   // +-0
        const int cl = (int)(off % (uint32_t)p.PPb) / (p.s8 ? 1 : 4), t = (int)(off / (uint32_t)p.PPb);
        int kx = 0, ky = 0;
        if (!p.linear) {
            const int pos = t % p.pitch;
            ky = t / p.pitch;
            kx = p.half ? (pos >= p.half ? 2 * (pos - p.half) + 1 : 2 * pos) : pos;
        }
        const int i = kx * p.c_in + c * p.CIc + cl;
        if (p.s8) p.image[image_at(p.dims, false, co, ky, i)] = (unsigned char)bits;
        else image_put(p.image, p.dims, co, ky, i, __uint_as_float(bits));
    }
}

// the same from the row CSR of a small-batch fc layer: one warp per packed row (padding entries have the value 0)
__global__ void __launch_bounds__(256) expand_fc_kernel(const void *vals, const uint16_t *idx, const int32_t *ptr, const int32_t *perm, int c_pad,
                                                        int s8, ImageDims dims, unsigned char *image)
{
    const int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int co = row < c_pad ? perm[row] : -1;
    if (co < 0) return;
    for (int e = ptr[row] + lane; e < ptr[row + 1]; e += 32) {
        if (s8) {
            const signed char v = reinterpret_cast<const signed char *>(vals)[e];
            if (v) image[image_at(dims, false, co, 0, idx[e])] = (unsigned char)v;
        } else {
            const float v = reinterpret_cast<const float *>(vals)[e];
            if (v != 0.0f) image_put(image, dims, co, 0, idx[e], v);
        }
    }
}

}  // namespace

// Fc layers packed for a batch of up to 8 run as a sparse matrix-vector product per image, or dense for the whole batch.
// Microseconds measured at 1 to 8 images, 300 to 25088 inputs, 3 to 30 % kept: sparse about 2.5 + 1.6 per image and million
// weights, dense 3.7 + the image's bytes at 7 (float) or 8 TB/s (int8) whatever the batch.  4096 -> 4096, 10 %, batch 8:
// 28.8 / 14.7 (float), 16.4 / 7.0 (int8).
bool tcv_fc_pays(const cadnn_weights *w, int n)
{
    const bool f32 = w->desc.dtype == CADNN_F32;
    const double dense_mb = (double)w->desc.c_out * w->desc.c_in * (f32 ? 6 : 1) * 1e-6;
    return n >= 3 && 3.7 + dense_mb / (f32 ? 7.0 : 8.0) < 2.5 + 1.6e-6 * n * (double)w->nnz;
}

// Builds the dense image of a handle whose sparse (or dense stem) image is on the device, where there is memory for it.
cadnn_status tcv_build(cadnn_weights *h)
{
    const cadnn_layer_desc &d = h->desc;
    int a = 0, b = 0, c = 0;   // for tests and tuning: the block shape, "pixels,channels,split"
    const char *e = getenv("CADNN_TCV");
    if (e && sscanf(e, "%d,%d,%d", &a, &b, &c) == 3 && a >= 16 && a <= 256 && a % 16 == 0 && (b == 128 || (b == 64 && a == 128)) && c >= 1) {
        h->tcv_force[0] = a; h->tcv_force[1] = b; h->tcv_force[2] = c;
    }
    if (d.flags & CADNN_PACK_HOST_ONLY) return CADNN_OK;
    const bool s8 = d.dtype == CADNN_S8;
    const ImageDims dims = {stages_of(d), row_positions(d)};
    const size_t bytes = (size_t)ceil_div(d.c_out, 64) * dims.nkb * (s8 ? 2 : 3) * 4096;
    const cudaError_t er = cudaMalloc(&h->d_tcv, bytes);
    if (er == cudaErrorMemoryAllocation) {   // the layer runs without it
        cudaGetLastError();
        h->d_tcv = nullptr;
        return CADNN_OK;
    }
    CADNN_CUDA_TRY(er);
    h->tcv_bytes = bytes;
    if (h->s.kind == KK_DENSE_SMALLC) {   // few weights, kept tap-major: written on the host
        std::vector<unsigned char> image(bytes, 0);
        for (int co = 0; co < d.c_out; ++co)
            for (int ky = 0; ky < d.kh; ++ky)
                for (int i = 0; i < d.kw * d.c_in; ++i)
                    image_put(image.data(), dims, co, ky, i, h->dense_f[((size_t)ky * d.kw * d.c_in + i) * d.c_out + co]);
        CADNN_CUDA_TRY(cudaMemcpy(h->d_tcv, image.data(), bytes, cudaMemcpyHostToDevice));
    } else if (h->s.kind == KK_FC_SPMV) {
        CADNN_CUDA_TRY(cudaMemsetAsync(h->d_tcv, 0, bytes, cudaStreamLegacy));
        expand_fc_kernel<<<(unsigned)ceil_div(h->c_pad, 8), 256, 0, cudaStreamLegacy>>>(h->d_vals, h->d_offs, h->d_ptr, h->d_perm, h->c_pad, s8, dims,
                                                                                      (unsigned char *)h->d_tcv);
        CADNN_CUDA_TRY(cudaGetLastError());
    } else {
        CADNN_CUDA_TRY(cudaMemsetAsync(h->d_tcv, 0, bytes, cudaStreamLegacy));
        const Schedule &s = h->s;
        ExpandParams p;
        p.ent = h->d_ent; p.perm = h->d_perm; p.image = (unsigned char *)h->d_tcv; p.dims = dims;
        p.n_chunks = s.n_chunks; p.c_pad = h->c_pad; p.n_groups = s.n_groups; p.G = s.G;
        p.hdr_words = (s.G + 1 + 3) / 4 * 4;
        p.block_words = p.hdr_words + s.max_entries * (s8 ? 1 : 2);
        p.CIc = s.CIc; p.PPb = s.PPb; p.pitch = std::max(1, s.pitch); p.half = s.half;
        p.linear = s.kind == KK_SCONV_LINEAR; p.s8 = s8; p.c_in = d.c_in;
        expand_kernel<<<dim3((unsigned)ceil_div(h->c_pad, 8), (unsigned)s.n_chunks), 256, 0, cudaStreamLegacy>>>(p);
        CADNN_CUDA_TRY(cudaGetLastError());
    }
    CADNN_CUDA_TRY(cudaStreamSynchronize(cudaStreamLegacy));
    return CADNN_OK;
}

void tcv_drop(cadnn_weights *h)
{
    cudaFree(h->d_tcv);
    h->d_tcv = nullptr;
    h->tcv_bytes = 0;
}

// the kernel's index ranges: 31-bit element offsets and pixel numbers, 16-bit image coordinates
bool tcv_fits(const cadnn_weights *w, int n)
{
    const cadnn_layer_desc &d = w->desc;
    const long long lim = (1ll << 31) - (1 << 20);
    return (long long)n * w->h_out * w->w_out < lim && ((long long)n * d.in_h + 2 * d.kh) * d.in_w * d.c_in < lim && d.in_h < 16000 && d.in_w < 16000;
}

// Whether the layer's launch can write the 2 x 2 max pool of its output too (int8 outputs without residual, whole channel pieces).
// The pool is then no launch of its own and reads nothing; int8 VGG-16 has five of them: batch 1 152.1 / 141.4 us, batch 4
// 318 / 313, batch 16 906 / 894.
bool tcv_pools(const cadnn_weights *w, int n)
{
    return w->d_tcv && w->desc.dtype == CADNN_S8 && w->s.kind != KK_FC_SPMV && w->h_out % 2 == 0 && w->w_out % 2 == 0 && w->desc.c_out % 16 == 0 &&
           tcv_fits(w, n);
}

namespace {

typedef CUresult (*EncodeIm2colFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *, const int *,
                                   const int *, cuuint32_t, cuuint32_t, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeIm2colFn encode_im2col_fn()
{
    static const EncodeIm2colFn fn = []() -> EncodeIm2colFn {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeIm2col", &ptr, cudaEnableDefault, &found) == cudaSuccess && found == cudaDriverEntryPointSuccess)
            return (EncodeIm2colFn)ptr;
        cudaGetLastError();
        return nullptr;
    }();
    return fn;
}

// Whether the copy engine can gather an int8 layer's im2col rows: each 64 values of K are 64 channels of one window position, and the
// geometry fits the tensor map's fields (corners of 8 bits, steps of up to 8 - twice the stride with a pool - and window offsets of 8).
// It takes the address arithmetic, the loads and the stores off the loader warps and keeps every stage of the ring in flight: a
// stage of the gather took 700 clocks whatever its pixels.
bool engine_takes(const cadnn_layer_desc &d)
{
    return d.dtype == CADNN_S8 && d.c_in % 64 == 0 && d.stride <= 4 && d.pad <= 127 && d.pad_w <= 127 && d.kh <= 128 && d.kw <= 128 && encode_im2col_fn();
}

// Whether a launch that does not overlap the one before it (pdl) gains by that: the engine's first fetch of the tensor map and of the pixels
// then stands alone, 0.3 to 0.4 us, which small layers do not make up for.  Launches one after the other in a captured graph, engine /
// gather, us each: 64 -> 64 1x1 7x7 3.46 / 3.18, 448 -> 384 3x3 8x8 5.26 / 4.71, 1024 -> 256 1x1 14x14 4.70 / 4.39, 2048 -> 1000 fc of 16 images
// 4.27 / 3.88, 4096 -> 4096 fc of 32 6.97 / 6.01; beyond the lines, 64 -> 256 1x1 56x56 (803 thousand outputs) 4.62 / 4.95, 25088 -> 4096 fc
// of 9 (925 million multiply-adds) 15.0 / 19.4.  (Of 45 layers within them one is faster by the engine, by 0.02 us.)
bool engine_pays_alone(long long M, int c_out, long long k)
{
    const double outputs = (double)M * ((c_out + 63) / 64 * 64);
    return outputs > 300e3 || outputs * k > 600e6;
}

// The input of n images as im2col rows of 64 channels, `rows` output pixels per copy (`pooled`: every second one of every second row).
bool encode_pixels(CUtensorMap *map, const cadnn_layer_desc &d, const void *x, int n, int rows, bool pooled)
{
    const cuuint64_t dims[4] = {(cuuint64_t)d.c_in, (cuuint64_t)d.in_w, (cuuint64_t)d.in_h, (cuuint64_t)n};
    const cuuint64_t strides[3] = {dims[0], dims[0] * dims[1], dims[0] * dims[1] * dims[2]};
    // the windows' first positions: from the padding to as far before the far padding's end as the window is wide
    const int lower[2] = {-d.pad_w, -d.pad}, upper[2] = {d.pad_w - (d.kw - 1), d.pad - (d.kh - 1)};
    const cuuint32_t step = (cuuint32_t)((pooled ? 2 : 1) * d.stride), steps[4] = {1, step, step, 1};
    return encode_im2col_fn()(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void *>(x), dims, strides, lower, upper, 64, (cuuint32_t)rows, steps,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

cadnn_status launch_tcv(const cadnn_weights *w, const void *x, int n, void *y, const LaunchEpilogue &ep, cudaStream_t st)
{
    const cadnn_layer_desc &d = w->desc;
    const bool f32 = d.dtype == CADNN_F32;
    const long long M = (long long)n * w->h_out * w->w_out;
    if (!w->d_tcv || !tcv_fits(w, n)) return CADNN_E_UNSUPPORTED;
    if (M == 0) return CADNN_OK;
    TcvParams p = {};
    p.x = x; p.y = y; p.wimg = (const unsigned char *)w->d_tcv;
    p.scale = ep.scale; p.bias = ep.bias; p.residual = ep.residual; p.res_scale = ep.res_scale;
    p.act = ep.act; p.out_dtype = ep.out_dtype;
    p.h = d.in_h; p.w = d.in_w; p.c_in = d.c_in; p.h_out = w->h_out; p.w_out = w->w_out; p.c_out = d.c_out;
    p.stride = d.stride; p.pad = d.pad; p.pad_w = d.pad_w; p.kh = d.kh; p.kw = d.kw;
    const long long in_bytes = (long long)n * d.in_h * d.in_w * d.c_in;   // (of int8)
    p.whole = (int)(in_bytes & ~3ll); p.tail = (int)(in_bytes & 3);
    p.M = (int)M; p.Rp = row_positions(d); p.nkb = stages_of(d);
    p.odd_half = (int)((long long)d.kh * p.Rp % 128 != 0);
    p.ldc = ep.out_c_total > 0 ? ep.out_c_total : d.c_out;
    p.c_off = ep.out_c_total > 0 ? ep.out_c_off : 0;
    p.vec_ok = d.c_out % 4 == 0 && p.ldc % 4 == 0 && p.c_off % 4 == 0;
    if (ep.pooled) {
        if (!tcv_pools(w, n) || ep.residual || ep.out_dtype != CADNN_S8 || ep.out_c_total > 0) return CADNN_E_UNSUPPORTED;
        p.pooled = (signed char *)ep.pooled;
        p.h_out /= 2;
        p.w_out /= 2;
    }
    p.res_tile = f32 || !ep.residual ? 0 : d.c_out % 16 == 0 ? 16 : d.c_out % 4 == 0 ? 4 : 1;
    p.d_hw = make_fastdiv(p.h_out * p.w_out); p.d_wo = make_fastdiv(p.w_out);
    p.d_ci = make_fastdiv(d.c_in); p.d_Rp = make_fastdiv(p.Rp);
    if (ep.prefetch) p.ahead = *ep.prefetch;
    cadnn_status rs = copy_timeout_word(&p.gave_up);
    if (rs != CADNN_OK) return rs;
    Pick pick = {w->tcv_force[0], w->tcv_force[1], w->tcv_force[2]};
    const bool engine = engine_takes(d) && (ep.pdl || p.pooled || pick.px > 0 || engine_pays_alone(M, d.c_out, (long long)d.kh * d.kw * d.c_in));
    // the last batch size's choice is kept in the handle, for each of what else it depends on: a residual tile, which takes shared memory, and
    // the gather (one word each, so that threads may race on it)
    std::atomic<uint64_t> &last = w->tcv_pick[2 * (p.res_tile != 0) + engine];
    const uint64_t kept = last.load(std::memory_order_relaxed);
    if (pick.px > 0) pick.split = std::max(1, pick.split);
    else if ((kept >> 32) == (uint64_t)n && kept != 0) pick = {(int)(kept & 0xfff), (int)(kept >> 12 & 0xfff), (int)(kept >> 24 & 0xff)};
    else {
        // (Pooled layers count as the copy engine's although their split tiles run on the gather: its shapes are within 0.6 us of the best of
        // 20 on each pooled layer of int8 VGG-16 at batch 1, 2, 4 and 8.  With the gather's coefficients for the split tiles, which know no
        // pooled epilogue, fewer blocks share the pooling: batch 1 / 2 / 4 / 8 104 / 141 / 207 / 332 us became 108 / 145 / 212 / 336.)
        pick = choose(f32 ? d.c_in % 4 != 0 : engine ? 2 : d.c_in % 16 == 0 ? 3 : 4, d.c_out, M, p.nkb, p.res_tile != 0);
        last.store((uint64_t)n << 32 | (uint64_t)pick.split << 24 | (uint64_t)pick.ch << 12 | (uint64_t)pick.px, std::memory_order_relaxed);
    }
    const bool vec = d.c_in % (f32 ? 4 : 16) == 0, run_tail = !f32 && !vec && p.tail;
    if (pick.ch == 64 || (run_tail && pick.px > 128)) pick.px = 128;
    p.npx = pick.px;
    p.n_nt = ceil_div(d.c_out, pick.ch);
    // every block of a cluster finishes the same number of pixels, and two stages and the partial sums have to fit
    p.S = pick.px > 128 ? 1 : std::min(pick.split, 16);
    // (with a pool: whole windows)
    while (p.S > 1 && (p.npx % p.S || p.S > p.nkb || (p.pooled && p.npx / p.S % 4))) --p.S;
    p.kb_base = p.nkb / p.S; p.kb_rem = p.nkb % p.S;
    p.d_S = make_fastdiv(p.S); p.d_nt = make_fastdiv(p.n_nt); p.d_rows = make_fastdiv(p.npx / p.S);
    const long long blocks = (M + p.npx - 1) / p.npx * p.n_nt * p.S;
    if (blocks > 2147483647ll) return CADNN_E_UNSUPPORTED;
    const int n_blocks = (int)blocks;
    if (f32) return vec ? launch_shape<true, Gather::kPieces>(p, pick.ch, n_blocks, ep.pdl, st) : launch_shape<true, Gather::kValues>(p, pick.ch, n_blocks, ep.pdl, st);
    if (run_tail)
        return p.pooled ? launch_shape<false, Gather::kValues, true, true>(p, pick.ch, n_blocks, ep.pdl, st)
                        : launch_shape<false, Gather::kValues, false, true>(p, pick.ch, n_blocks, ep.pdl, st);
    // (With a pool the copies of one stage are quarters of the tile, which have to be whole groups of 8 swizzled rows, and blocks of a
    // cluster would share out quarters of windows.)
    if (engine && !(p.pooled && (p.S > 1 || p.npx % 32))) {
        TcvEngineParams e;
        static_cast<TcvParams &>(e) = p;
        if (encode_pixels(&e.pixels, d, x, n, p.pooled ? p.npx / 4 : p.npx, p.pooled != nullptr))
            return p.pooled ? launch_shape<false, Gather::kCopyEngine, true>(e, pick.ch, n_blocks, ep.pdl, st)
                            : launch_shape<false, Gather::kCopyEngine>(e, pick.ch, n_blocks, ep.pdl, st);
    }
    if (p.pooled)
        return vec ? launch_shape<false, Gather::kPieces, true>(p, pick.ch, n_blocks, ep.pdl, st) : launch_shape<false, Gather::kValues, true>(p, pick.ch, n_blocks, ep.pdl, st);
    return vec ? launch_shape<false, Gather::kPieces>(p, pick.ch, n_blocks, ep.pdl, st) : launch_shape<false, Gather::kValues>(p, pick.ch, n_blocks, ep.pdl, st);
}
