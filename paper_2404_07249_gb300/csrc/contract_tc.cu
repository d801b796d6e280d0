// Tensor-core (tcgen05, sm_103a) triplet contraction with three-term split products.
//
// Computes sums M[(j, k)][i] = sum_x g_j(x) g_k(x) h_i(x) over the cells x (Sec. 4.3.1, eq. beta-def: the
// real-space sum of the separable bispectrum; with h = g the entry of pair (b, c) and single a is S_abc).  The work
// is a set of 128-row tiles: every row is one pair (j, k) and every tile has a window of W singles
// [s0, s0 + W), W in {16, 32}.  For the ideal bispectrum only the pairs and singles of closed triplets enter:
// the triplet a <= b <= c is read from pair (b, c) and single a, which prunes the 465 pairs x 30 singles of a
// 30-bin binning to 255 pairs in two tiles with windows of 16 and 32 singles.
//
// Arithmetic: the pair products A = g_j g_k (FP32) and the singles B are split into three BF16 parts of 8 bits each,
// v = v1 + v2 + v3 (v1 and v2 rounded to nearest, v3 what is left): all 24 bits, with FP32's exponent, so that a value
// keeps them however far it lies below the largest of its map.  (Two FP16 parts take fewer instructions and less storage,
// but their exponent ends 2^-40 below a scale that has to be taken from the maps' maxima: two maps with a peak of 2^12 in
// different cells left their products, and the sums, with an error of 3e-5.)  Per tile and K = 16 cells six MMAs of N = W run, smallest terms
// first: A1 B3, A3 B1, A2 B2, A1 B2, A2 B1, A1 B1; the three left out are below 2^-26 of the product.  The
// tensor core's internal accumulation is not round-to-nearest, so D restarts every 64 cells; the epilogue adds D into FP32
// registers (round-to-nearest) and those into FP64 shared memory every 2048 cells.  Cross-CTA sums are FP64 in a fixed
// order (deterministic).  Rows whose products' magnitude lies outside 2^-40 .. 2^40, and all singles, are scaled by powers of
// two from the maps' maxima (found by the z-pass that writes them, or by k_absmax), which the final sums undo: products of
// three maps of any magnitude then stay in FP32's range.
//
// Measured on this part (and shaping the design): an MMA issued from warp-uniform code with its operands in uniform
// registers costs ~16-20 cycles at N = 32 (the tensor pipe's rate), but ~200 cycles from a one-lane branch, so the
// issuing loop is warp-uniform (elect.sync inside the asm) and divide-free; tensor memory stores reach ~650 B/clk an
// SM.  What bounds the kernel is the producers: their gathers (two 16-byte loads for every four products; the shared-memory
// pipe is busy 76 % of the time, nearly half of it with bank conflicts) and ten instructions of split for two products (2.64
// of 4 instructions a clock); the tensor pipe is busy 27 % (half of the MMAs: 5 % less time).  So four producer groups,
// 16 cells at a time in few registers, and B warps that take every other stage; a stage is 64
// cells and the accumulators are double-buffered, so that no MMA waits for the epilogue.  Measured, ms, at 30 maps
// of 288^3 cells (two tiles) and at 20 maps of 192^3 (one tile): two TF32 parts in 32-cell stages 3.90 and 0.778, two
// FP16 parts 2.64 and 0.459, three BF16 parts with two producer groups and 32 cells at a time 3.39 and 0.549 (3.22 and
// 0.522 without a row scale of 1), with three groups and 16 cells 2.87 and 0.527, four groups 2.77 and 0.546, and B warps on
// alternate stages 2.71 and 0.498.  Tensor memory (512 columns) holds two accumulator buffers (W columns a tile each) and
// a ring of A stages (96 columns a tile a stage).
//
// One CTA per SM over a contiguous range of cells, in stages of 64 cells (two TMA ring slots).  Warp roles, by
// warpgroup (setmaxnreg moves registers from warpgroup 0 to the producers):
//   warp 0       TMEM allocation; lane 0 streams the maps with TMA (cp.async.bulk.tensor, 32 cells x all maps per
//                load, 128-byte swizzle) into an 8-slot shared-memory ring.
//   warp 1       MMA issue: waits for the stage (converged), issues every tile's MMAs and commits them to the A
//                stage's release barrier and the accumulator barrier.
//   warps 4-7    the B operand: scale and split the singles into BF16 rows of 64 cells (128-byte swizzle), one block of
//                rows a part; two warps a stage, one a slot.
//   producers    groups of four warps; group g makes the 32 cells of slots g, g + kProdGroups, ..  A thread owns one TMEM
//                lane, i.e. one row of every tile: it forms the pair products, splits them and writes the parts straight
//                into tensor memory (tcgen05.st: the A operand never touches shared memory).
//   epilogue     four warps: after every stage read D with tcgen05.ld (each warp its TMEM lane quarter), release it to
//                the issuer, accumulate.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <cstdlib>
#include <map>
#include <mutex>
#include <set>
#include <tuple>
#include <vector>

#include "polybin_internal.h"

namespace pb {
namespace tc {

constexpr int kSlotCells = 32;     // cells per TMA box row (128 bytes)
constexpr int kRingSlots = 8;
constexpr int kKC = 64;            // cells per A stage = two ring slots (four K = 16 MMA steps)
constexpr int kMaxAStages = 6;
constexpr int kSpill = 32;         // stages per FP32 register sum (2048 cells)
constexpr int kParts = 3;          // BF16 parts of a value
constexpr int kAccBufs = 2;        // accumulator buffers (the epilogue reads one while the MMAs fill the other)
constexpr int kDBuf = 1;           // blocks of d_cols accumulator columns: a tile's 2W columns there hold both its buffers
constexpr int kAcols = 32 * kParts;   // tensor memory columns of a tile's A stage: the parts of 64 cells, two a column
constexpr int kMaxTiles = 2;       // tiles per CTA (three leave no room for two A stages)
constexpr int kMaxUnits = 3;       // 16-column output units per CTA (16 FP32 sums each, in registers)
constexpr int kMaxGroups = 4;      // row groups (grid.y)
constexpr int kProdGroups = 4;     // producer warp groups; group g makes slots g, g + kProdGroups, .. (32 cells each)
constexpr int kProdWarps = 4 * kProdGroups;
constexpr int kEpiWarps = 4;
// Warpgroup 0: TMA (warp 0), MMA issue (warp 1), two idle warps; then the B operand (four warps), the producers and the
// epilogue, a warpgroup each (producers: kProdGroups).
constexpr int kBWarp0 = 4, kBWarps = 4;
constexpr int kProdWarp0 = kBWarp0 + kBWarps;
constexpr int kWarps = kProdWarp0 + kProdWarps + kEpiWarps;
// Register split (setmaxnreg, per warpgroup): the CTA is launched with kRegsLaunch registers a thread; warpgroup 0 and the B
// warps give registers back, the producers and the epilogue take them.
constexpr int kRegsLaunch = 72, kRegsCtl = 24, kRegsB = 64, kRegsProd = 80, kRegsEpi = 88;
static_assert((kRegsCtl + kRegsB) * 128 + kRegsProd * 32 * kProdWarps + kRegsEpi * 32 * kEpiWarps <= kRegsLaunch * 32 * kWarps,
              "register split exceeds the launch allocation");
constexpr int kThreads = 32 * kWarps;
constexpr int kMinSmem = 120 * 1024;   // one CTA per SM (the CTA allocates all 512 TMEM columns)
constexpr unsigned kSpinLimit = 1u << 22;
constexpr int kBloItems = 2;       // 16-byte chunks of a slot's singles region a thread of 256: <= 64 rows x 8 chunks

struct GroupDesc {
    int tile0;                 // first tile (row table index / 128)
    int ntiles, nunits, nA;    // tiles, 16-column units, A stages
    int unit_base;             // first unit of this group in the partial layout
    int d_cols;                // TMEM columns of the accumulators
    int a_col0;                // first TMEM column of the A ring
    int bstage_bytes;          // bytes of one part of a B stage: 128 for each row of the singles region
    int tile_w[kMaxTiles];
    int dm_col[kMaxTiles];     // TMEM column of tile t's accumulators: two buffers of W columns
    int tile_s0[kMaxTiles];    // first single of tile t's window
    int unit_tile[kMaxUnits], unit_c[kMaxUnits];
};

struct Params {
    long ncell, cells_cta;
    int ng, nh, hsep, h_row0;  // maps in the slot; singles; singles from the h part; first h row in a slot
    int slot_bytes, off_b, off_acc, off_bar;
    int s_off, s_chunks;       // singles region of a slot: byte offset and 16-byte chunks (B is made for all)
    const uint32_t *gmax, *hmax;   // max |map| bit patterns of the g rows and of the h rows (the scale factors)
    int total_units;
    const short2* rows;        // [tiles][128] pairs (j, k); (-1, -1) pads
    double* partial;           // [gridDim.x][total_units][16][128]
    int* err;
    GroupDesc grp[kMaxGroups];
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Non-blocking test of a phase (no suspension): the fast path of the waits below when the phase is already done.
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait of one thread; false (and the abort flag raised) on timeout or when another role aborted.
__device__ __forceinline__ bool thread_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* err) {
    if (mbar_test(bar, parity)) return true;
    for (unsigned it = 0; it < kSpinLimit; ++it) {
        if (mbar_try(bar, parity)) return true;
        if (*abort_flag) return false;
    }
    *abort_flag = 1;
    atomicExch(err, 1);
    return false;
}
// Bounded wait used while shutting down (no abort check): lets in-flight asynchronous work land.
__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity, int* err) {
    for (unsigned it = 0; it < kSpinLimit; ++it)
        if (mbar_try(bar, parity)) return;
    atomicExch(err, 1);
}
// Bounded wait of a whole warp with a warp-uniform outcome (the warp then runs .sync.aligned instructions).
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* err) {
    if (__all_sync(0xffffffffu, mbar_test(bar, parity))) return true;
    for (unsigned it = 0; it < kSpinLimit; ++it) {
        const bool done = mbar_try(bar, parity);
        if (__all_sync(0xffffffffu, done)) return true;
        if (__any_sync(0xffffffffu, *abort_flag != 0)) return false;
    }
    if ((threadIdx.x & 31) == 0) {
        *abort_flag = 1;
        atomicExch(err, 1);
    }
    __syncwarp();
    return false;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Packed FP32 pairs (two floats in one 64-bit register; sm_100+ f32x2 arithmetic).
__device__ __forceinline__ uint64_t f2pack(float a, float b) {
    return (uint64_t)__float_as_uint(a) | ((uint64_t)__float_as_uint(b) << 32);
}
__device__ __forceinline__ uint64_t mul_x2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t sub_x2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// Two values at once: v = hi + lo with hi = v rounded to TF32 (nearest, ties away from zero: add half a unit of the
// 10-bit mantissa, bit 12, and clear the 13 low bits; a carry moves into the exponent as it should) and lo = v - hi
// in FP32.  lo is symmetric about zero, so the tensor core's truncation of lo to TF32 is unbiased.  (Used by the Gram.)
__device__ __forceinline__ void split_x2(uint64_t v, uint64_t& hi, uint64_t& lo) {
    const uint32_t h0 = ((uint32_t)v + 0x1000u) & 0xFFFFE000u;
    const uint32_t h1 = ((uint32_t)(v >> 32) + 0x1000u) & 0xFFFFE000u;
    hi = (uint64_t)h0 | ((uint64_t)h1 << 32);
    lo = sub_x2(v, hi);
}
// Two values at once: v = p1 + p2 + p3 exactly (24 bits of a normal number), packed BF16 pairs (the first value in the low
// half): p1 and p2 rounded to nearest, each remainder exact in FP32; what is left then has at most 8 bits, so that p3 is its
// upper half.
__device__ __forceinline__ uint32_t bf16x2_rn(uint64_t v) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(__uint_as_float((uint32_t)(v >> 32))), "f"(__uint_as_float((uint32_t)v)));
    return r;
}
__device__ __forceinline__ uint64_t bf16x2_value(uint32_t p) { return (uint64_t)(p << 16) | ((uint64_t)(p & 0xFFFF0000u) << 32); }
__device__ __forceinline__ void split_b3(uint64_t v, uint32_t& p1, uint32_t& p2, uint32_t& p3) {
    p1 = bf16x2_rn(v);
    const uint64_t r = sub_x2(v, bf16x2_value(p1));
    p2 = bf16x2_rn(r);
    const uint64_t q = sub_x2(r, bf16x2_value(p2));
    p3 = __byte_perm((uint32_t)q, (uint32_t)(q >> 32), 0x7632);
}
// Scale exponents.  map_exp(m): the smallest e with m < 2^e for a map's largest magnitude m (bit pattern; 0 for a map
// with infinities or NaN, whose sums are not finite at any scale).  A row (j, k) is scaled by 2^row_exp: not at all (the
// producers then save a multiplication) where its products lie below 2^40 and not all below 2^-40, else to below 2^15; a
// single by 2^single_exp, to below 2^15.
__host__ __device__ inline int map_exp(uint32_t m) {
    const int e = (int)((m >> 23) & 255u);
    return e == 255 ? 0 : (e < 1 ? 1 : e) - 126;
}
// Largest magnitude of the map at slot row r (h rows start at h_row0).
__device__ __forceinline__ uint32_t row_max(const uint32_t* gmax, const uint32_t* hmax, int h_row0, int r) {
    return r < h_row0 ? gmax[r] : hmax[r - h_row0];
}
__host__ __device__ inline int clamp_exp(int e) { return e < -126 ? -126 : (e > 127 ? 127 : e); }
__host__ __device__ inline int row_exp(uint32_t mj, uint32_t mk) {
    const int e = map_exp(mj) + map_exp(mk);
    return e >= -40 && e <= 40 ? 0 : clamp_exp(15 - e);
}
__host__ __device__ inline int single_exp(uint32_t ma) { return clamp_exp(15 - map_exp(ma)); }
__device__ __forceinline__ float pow2f(int e) { return __uint_as_float((uint32_t)(e + 127) << 23); }   // -126 <= e <= 127

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* v) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]),
        "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]),
        "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31]));
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(v[0]),
                 "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]));
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* v) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
}
// tcgen05.wait::ld tied to a 16-register load, and to two.
__device__ __forceinline__ void tmem_wait_ld16(uint32_t* a) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]),
                   "+r"(a[8]), "+r"(a[9]), "+r"(a[10]), "+r"(a[11]), "+r"(a[12]), "+r"(a[13]), "+r"(a[14]), "+r"(a[15])
                 :
                 : "memory");
}
__device__ __forceinline__ void tmem_wait_ld32(uint32_t* a, uint32_t* b) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]),
                   "+r"(a[8]), "+r"(a[9]), "+r"(a[10]), "+r"(a[11]), "+r"(a[12]), "+r"(a[13]), "+r"(a[14]), "+r"(a[15]),
                   "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]), "+r"(b[4]), "+r"(b[5]), "+r"(b[6]), "+r"(b[7]),
                   "+r"(b[8]), "+r"(b[9]), "+r"(b[10]), "+r"(b[11]), "+r"(b[12]), "+r"(b[13]), "+r"(b[14]), "+r"(b[15])
                 :
                 : "memory");
}

// Shared-memory matrix descriptor for the 128-byte swizzle, K-major: 8-row x 128-byte atoms (1024-byte aligned,
// chunk c of row r at r * 128 + ((c ^ (r % 8)) << 4), the layout TMA writes), SBO = 1024 between 8-row groups; the
// K offset within the atom is added to the start address (32 bytes per K = 8 step of TF32).
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)1 << 16;                    // LBO: unused for a swizzled K-major operand
    d |= (uint64_t)(1024 >> 4) << 32;          // SBO
    d |= (uint64_t)1 << 46;                    // descriptor version for tcgen05
    d |= (uint64_t)2 << 61;                    // 128-byte swizzle
    return d;
}

// Instruction descriptor: kind::tf32, D = F32, A = B = TF32, both K-major.
__host__ __device__ constexpr uint32_t idesc_tf32(int M, int N) {
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// The same for kind::f16 with BF16 operands (D = F32, A = B = BF16, both K-major).
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// The MMA and its commit are executed by a whole converged warp and issued by the one lane that elect.sync picks
// (the same lane every time with all 32 active, so the commit tracks the MMAs of the issuing thread).  Keeping the
// issuing code warp-uniform, rather than inside a one-lane branch, lets the compiler hold the operands in uniform
// registers: measured on this part, one thread then issues an M = 128, N = 32 MMA every ~16 cycles (the tensor
// pipe's rate) instead of one every ~200 cycles from a divergent branch.
__device__ __forceinline__ void mma_tf32(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                         uint32_t accum) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\telect.sync _|q, 0xffffffff;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accum)
        : "memory");
}
__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                        uint32_t accum) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\telect.sync _|q, 0xffffffff;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accum)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
            "r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// 16-byte chunk `ch` (0..7) of map row `r` in a ring slot written by TMA with the 128-byte swizzle: within every
// 1024-byte block the chunk index is XORed with the row index modulo 8.
__device__ __forceinline__ const float4* ring_chunk(const unsigned char* slot, int r, int ch) {
    return reinterpret_cast<const float4*>(slot + r * 128 + ((ch ^ (r & 7)) << 4));
}

// Epilogue of NU output units (a compile-time count keeps the FP32 sums in registers): after every stage read this
// warp's TMEM lane quarter of the stage's accumulators with tcgen05.ld, release the D buffer, add into the FP32 sums;
// every kSpill stages add those into the FP64 sums in shared memory (FP64 is slow on this part, so only there);
// finally write this CTA's FP64 partials.
template <int NU>
__device__ __forceinline__ void epilogue(const GroupDesc& G, const Params& P, uint32_t tmem, double* acc64,
                                         uint64_t* d_full, uint64_t* d_empty, volatile int* abort_flag, int nstages,
                                         int warp, int lane) {
    const int q = warp & 3;
    const int row = 32 * q + lane;
    const uint32_t lane_base = (uint32_t)(32 * q) << 16;
    uint32_t cols[NU], bufw[NU];        // unit u: 16 columns of its tile's buffer (W columns from one buffer to the other)
#pragma unroll
    for (int u = 0; u < NU; ++u) {
        cols[u] = (uint32_t)(G.dm_col[G.unit_tile[u]] + G.unit_c[u]);
        bufw[u] = (uint32_t)G.tile_w[G.unit_tile[u]];
    }
    int* const err = P.err;
    double* const out = P.partial + ((size_t)blockIdx.x * P.total_units + G.unit_base) * 2048;

    float acc[NU][16];
#pragma unroll
    for (int u = 0; u < NU; ++u)
#pragma unroll
        for (int j = 0; j < 16; ++j) acc[u][j] = 0.f;
    for (int st = 0; st < nstages; ++st) {
        const int db = st & 1;
        if (!warp_wait(&d_full[db], (uint32_t)((st >> 1) & 1), abort_flag, err)) break;
        tc_fence_after();
        const uint32_t dbase = tmem + lane_base;
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            uint32_t v[16];
            tmem_ld16(dbase + cols[u] + (db ? bufw[u] : 0u), v);
            tmem_wait_ld16(v);
#pragma unroll
            for (int j = 0; j < 16; ++j) acc[u][j] += __uint_as_float(v[j]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&d_empty[db]);   // one arrival a warp (the warp's loads are done)
        if ((st + 1) % kSpill == 0) {
#pragma unroll
            for (int u = 0; u < NU; ++u)
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    acc64[(u * 16 + j) * 128 + row] += (double)acc[u][j];
                    acc[u][j] = 0.f;
                }
        }
    }
#pragma unroll
    for (int u = 0; u < NU; ++u)
#pragma unroll
        for (int j = 0; j < 16; ++j) acc64[(u * 16 + j) * 128 + row] += (double)acc[u][j];
    for (int i = 0; i < NU * 16; ++i) out[(size_t)i * 128 + row] = acc64[i * 128 + row];
}


// Producer warp of group gp: the 32 cells of slots gp, gp + kProdGroups, .. (two slots a 64-cell stage), for NT tiles (SC: some
// row of the warp is scaled).  A thread owns TMEM lane 32 (warp % 4) + lane, i.e. row `row` of every tile.  The 96
// columns of a tile's stage block are the parts [A1 8 | A2 8 | A3 8] (two cells a column) of each K step of 16 cells; a
// thread makes a step at a time and writes it with three 8-column TMEM stores (24 values in registers instead of 48).
template <int NT, bool SC>
__device__ __forceinline__ void produce(const GroupDesc& G, const Params& P, uint32_t tmem, const unsigned char* ring,
                                        uint64_t* slot_full, uint64_t* slot_empty, uint64_t* a_full, uint64_t* a_empty,
                                        volatile int* abort_flag, int nstages, int warp, int lane) {
    const int gp = (warp - kProdWarp0) >> 2;
    const int q = warp & 3;
    const int row = 32 * q + lane;
    const uint32_t lane_base = (uint32_t)(32 * q) << 16;
    const int nA = G.nA, a_col0 = G.a_col0, slot_bytes = P.slot_bytes;
    int* const err = P.err;
    int oj[NT], ok_[NT];          // byte offsets of the rows' maps in a slot, and their swizzle phases
    int xj[NT], xk[NT];
    bool pad[NT];
    uint64_t scale[NT];           // the row's power of two, twice
#pragma unroll
    for (int t = 0; t < NT; ++t) {
        const short2 jk = P.rows[(size_t)(G.tile0 + t) * 128 + row];
        pad[t] = jk.x < 0;
        const int j = max((int)jk.x, 0), k = max((int)jk.y, 0);
        oj[t] = j * 128; xj[t] = (j & 7) << 4;
        ok_[t] = k * 128; xk[t] = (k & 7) << 4;
        const float f = pad[t] ? 0.f : pow2f(row_exp(row_max(P.gmax, P.hmax, P.h_row0, j), row_max(P.gmax, P.hmax, P.h_row0, k)));
        scale[t] = f2pack(f, f);
    }
    // tensor-memory addresses from warp-uniform, divide-free values (the base is 0: the CTA holds all 512
    // columns; the issuing warp checks it), so that the compiler keeps the store addresses in uniform registers
    if (tmem != 0u) return;
    // slot sl: half sl % 2 of stage st = sl / 2, ring slot s = sl % kRingSlots, A stage as = st % nA
    int s = gp, st = gp >> 1, as = st;
    while (as >= nA) as -= nA;
    uint32_t sph = 0u, aph = st >= nA ? 0u : 1u;        // slot_full parity; a_empty parity of round st / nA - 1
    const uint32_t a_step = (uint32_t)kAcols * NT;
    uint32_t a_stage = (uint32_t)a_col0 + a_step * (uint32_t)as;
    const int nslots = 2 * nstages;
    for (int sl = gp; sl < nslots; sl += kProdGroups) {
        const uint32_t half = (uint32_t)(sl & 1);
        if (!warp_wait(&slot_full[s], sph, abort_flag, err)) break;
        const unsigned char* slot = ring + (size_t)s * slot_bytes;
        bool ok = true;
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            const unsigned char* rj = slot + oj[t];
            const unsigned char* rk = slot + ok_[t];
            const uint32_t dst = lane_base + a_stage + (uint32_t)(kAcols * t) + (uint32_t)(kAcols / 2) * half;
#pragma unroll
            for (int ks = 0; ks < 2; ++ks) {
                uint32_t v[kParts][8];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float4 x = *reinterpret_cast<const float4*>(rj + (((4 * ks + c) << 4) ^ xj[t]));
                    const float4 y = *reinterpret_cast<const float4*>(rk + (((4 * ks + c) << 4) ^ xk[t]));
                    uint64_t a = mul_x2(f2pack(x.x, x.y), f2pack(y.x, y.y)), b = mul_x2(f2pack(x.z, x.w), f2pack(y.z, y.w));
                    if (SC) {
                        a = mul_x2(a, scale[t]);
                        b = mul_x2(b, scale[t]);
                    }
                    split_b3(a, v[0][2 * c], v[1][2 * c], v[2][2 * c]);
                    split_b3(b, v[0][2 * c + 1], v[1][2 * c + 1], v[2][2 * c + 1]);
                }
                if (pad[t]) {
#pragma unroll
                    for (int p = 0; p < kParts; ++p)
#pragma unroll
                        for (int c = 0; c < 8; ++c) v[p][c] = 0u;
                }
                if (t == 0 && ks == 0) {
                    // tensor memory A stage `as` is free once the MMAs of stage st - nA completed
                    if (st >= nA) ok = warp_wait(&a_empty[as], aph, abort_flag, err);
                    tc_fence_after();
                }
                if (ok) {
#pragma unroll
                    for (int p = 0; p < kParts; ++p) tmem_st8(dst + (uint32_t)(8 * (kParts * ks + p)), v[p]);
                }
            }
        }
        if (!ok) break;
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        tc_fence_before();
        // one arrival a warp on each barrier: __syncwarp orders the other lanes' stores and reads before lane 0's
        // release
        __syncwarp();
        if (lane == 0) {
            mbar_arrive(&a_full[as]);
            mbar_arrive(&slot_empty[s]);
        }
        s += kProdGroups;
        if (s >= kRingSlots) { s -= kRingSlots; sph ^= 1u; }
        // kProdGroups slots on
        const int adv = ((int)half + kProdGroups) >> 1;
        st += adv;
        as += adv;
        a_stage += a_step * (uint32_t)adv;
        if (as >= nA) { as -= nA; aph ^= 1u; a_stage -= a_step * (uint32_t)nA; }
    }
}

// (the choice is the same for the 32 rows of a warp)
template <int NT>
__device__ __forceinline__ void producer(const GroupDesc& G, const Params& P, uint32_t tmem, const unsigned char* ring,
                                         uint64_t* slot_full, uint64_t* slot_empty, uint64_t* a_full, uint64_t* a_empty,
                                         volatile int* abort_flag, int nstages, int warp, int lane) {
    const int row = 32 * (warp & 3) + lane;
    bool sc = false;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
        const short2 jk = P.rows[(size_t)(G.tile0 + t) * 128 + row];
        if (jk.x >= 0) sc |= row_exp(row_max(P.gmax, P.hmax, P.h_row0, jk.x), row_max(P.gmax, P.hmax, P.h_row0, jk.y)) != 0;
    }
    if (__any_sync(0xffffffffu, sc))
        produce<NT, true>(G, P, tmem, ring, slot_full, slot_empty, a_full, a_empty, abort_flag, nstages, warp, lane);
    else
        produce<NT, false>(G, P, tmem, ring, slot_full, slot_empty, a_full, a_empty, abort_flag, nstages, warp, lane);
}

// B warp w (0 .. 3): the singles of ring slot b = w % 2 of stages w / 2, w / 2 + 2, .. -> BF16 rows of 64 cells (128
// bytes, 128-byte swizzle), cells 32 b .. 32 b + 31, one block of all rows a part (bstage_bytes), so
// that a window of W singles is W consecutive rows of a block.  A warp makes a group of eight rows at a time, lane (r, piece) = (lane / 4, lane % 4) eight cells
// of row r; the rows' scales wait in shared memory.  (Two warps with the scales read from global memory set the pace of the
// whole kernel.)
__device__ __forceinline__ void make_b(const GroupDesc& G, const Params& P, const unsigned char* ring,
                                       unsigned char* bst, const float* bscale, uint64_t* slot_full, uint64_t* slot_empty,
                                       uint64_t* a_full, uint64_t* a_empty, volatile int* abort_flag, int nstages, int w,
                                       int lane) {
    const int b = w & 1;
    const int nA = G.nA, slot_bytes = P.slot_bytes, part_bytes = G.bstage_bytes, stage_bytes = kParts * part_bytes;
    const int ngrp = P.s_chunks / 64;               // groups of eight rows (eight chunks a row)
    int* const err = P.err;
    const int r = lane >> 2, pc = lane & 3, x = r << 4;
    const int src0 = P.s_off + r * 128 + ((pc << 5) ^ x), src1 = P.s_off + r * 128 + (((pc << 5) + 16) ^ x);
    const int dst0 = r * 128 + (((4 * b + pc) << 4) ^ x);
    int s = w, as = w >> 1;
    uint32_t sph = 0u, aph = 1u;
    for (int st = w >> 1; st < nstages; st += 2) {
        if (!warp_wait(&slot_full[s], sph, abort_flag, err)) break;
        if (st >= nA && !warp_wait(&a_empty[as], aph, abort_flag, err)) break;
        const unsigned char* src = ring + (size_t)s * slot_bytes;
        unsigned char* dst = bst + (size_t)as * stage_bytes + dst0;
#pragma unroll 2
        for (int g = 0; g < ngrp; ++g) {
            const float f = bscale[8 * g + r];
            const uint64_t f2 = f2pack(f, f);
            const float4 u = *reinterpret_cast<const float4*>(src + src0 + g * 1024);
            const float4 v = *reinterpret_cast<const float4*>(src + src1 + g * 1024);
            uint4 p, q, o;
            split_b3(mul_x2(f2pack(u.x, u.y), f2), p.x, q.x, o.x);
            split_b3(mul_x2(f2pack(u.z, u.w), f2), p.y, q.y, o.y);
            split_b3(mul_x2(f2pack(v.x, v.y), f2), p.z, q.z, o.z);
            split_b3(mul_x2(f2pack(v.z, v.w), f2), p.w, q.w, o.w);
            *reinterpret_cast<uint4*>(dst + g * 1024) = p;
            *reinterpret_cast<uint4*>(dst + part_bytes + g * 1024) = q;
            *reinterpret_cast<uint4*>(dst + 2 * part_bytes + g * 1024) = o;
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // B stores -> tensor core
        __syncwarp();
        if (lane == 0) {
            mbar_arrive(&a_full[as]);
            mbar_arrive(&slot_empty[s]);
        }
        s += 4;
        if (s >= kRingSlots) { s -= kRingSlots; sph ^= 1u; }
        as += 2;
        if (as >= nA) { as -= nA; aph ^= 1u; }
    }
}

__global__ void __launch_bounds__(kThreads, 1)
    k_contract_tc(const __grid_constant__ CUtensorMap tmap_g, const __grid_constant__ CUtensorMap tmap_h,
                  const __grid_constant__ Params P) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const GroupDesc& G = P.grp[blockIdx.y];
    unsigned char* ring = smem;
    unsigned char* bst = smem + P.off_b;
    double* acc64 = reinterpret_cast<double*>(smem + P.off_acc);                 // [unit][16][128]
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + P.off_bar);
    uint64_t* slot_full = bars;                        // [kRingSlots]  TMA -> producers, B warps
    uint64_t* slot_empty = bars + kRingSlots;          // [kRingSlots]  producers, B warps -> TMA
    uint64_t* a_full = bars + 2 * kRingSlots;          // [kMaxAStages] producers, B warps -> issuer
    uint64_t* a_empty = a_full + kMaxAStages;          // [kMaxAStages] MMA commit -> producers, B warps
    uint64_t* d_full = a_empty + kMaxAStages;          // [kAccBufs]    MMA commit -> epilogue
    uint64_t* d_empty = d_full + kAccBufs;             // [kAccBufs]    epilogue -> issuer
    uint64_t* fin = d_empty + kAccBufs;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(fin + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    float* bscale = reinterpret_cast<float*>(tmem_slot + 2);                    // [64] scales of the singles region's rows

    // warp index through a shuffle from lane 0: the compiler then knows it is warp-uniform, so role branches and
    // the tensor-memory addresses derived from it stay in uniform registers
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const long c0 = (long)blockIdx.x * P.cells_cta;
    const long c1 = min(P.ncell, c0 + P.cells_cta);
    const int nstages = c0 < c1 ? (int)((c1 - c0 + kKC - 1) / kKC) : 0;
    const int nslots = 2 * nstages;             // cells beyond the maps read as zero (TMA out-of-bounds fill)
    // plan fields used in the loops, in registers
    const int nA = G.nA, ntiles = G.ntiles, a_col0 = G.a_col0;
    const int slot_bytes = P.slot_bytes;
    int* const err = P.err;

    for (int i = tid; i < G.nunits * 16 * 128; i += kThreads) acc64[i] = 0.0;
    if (tid < P.s_chunks / 8) bscale[tid] = pow2f(single_exp(row_max(P.gmax, P.hmax, P.h_row0, P.s_off / 128 + tid)));
    if (tid == 0) {
        for (int s = 0; s < kRingSlots; ++s) {
            mbar_init(&slot_full[s], 1);
            mbar_init(&slot_empty[s], 4 + 1);          // the slot's producer group and its B warp
        }
        for (int s = 0; s < kMaxAStages; ++s) {
            mbar_init(&a_full[s], 4 * 2 + 2);          // two slots a stage: four producer warps and a B warp each
            mbar_init(&a_empty[s], 1);
        }
        for (int i = 0; i < kAccBufs; ++i) {
            mbar_init(&d_full[i], 1);
            mbar_init(&d_empty[i], kEpiWarps);
        }
        mbar_init(fin, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp < kBWarp0) {
        // warpgroup 0 hands registers on (all four warps, one instruction)
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsCtl));
        if (warp == 0) {
            // ------------------------------------------------------------------ TMA producer
            if (lane == 0 && nslots > 0) {
                const uint32_t bytes = (uint32_t)(P.ng * 128 + (P.hsep ? P.nh * 128 : 0));
                const bool hsep = P.hsep != 0;
                const int hoff = P.h_row0 * 128;
                int issued = 0;
                for (int sl = 0; sl < nslots; ++sl) {
                    const int s = sl % kRingSlots;
                    if (sl >= kRingSlots &&
                        !thread_wait(&slot_empty[s], (uint32_t)((sl / kRingSlots - 1) & 1), abort_flag, err))
                        break;
                    unsigned char* dst = ring + (size_t)s * slot_bytes;
                    const int x = (int)(c0 + (long)sl * kSlotCells);
                    mbar_expect_tx(&slot_full[s], bytes);
                    tma_load_2d(dst, &tmap_g, x, 0, &slot_full[s]);
                    if (hsep) tma_load_2d(dst + hoff, &tmap_h, x, 0, &slot_full[s]);
                    ++issued;
                }
                // every load issued has landed before the CTA may exit
                for (int sl = max(0, issued - kRingSlots); sl < issued; ++sl)
                    drain_wait(&slot_full[sl % kRingSlots], (uint32_t)((sl / kRingSlots) & 1), err);
            }
            __syncwarp();
        } else if (warp == 1) {
            // ------------------------------------------------------------------ MMA issue
            // The whole warp runs the loop (converged; every lane polls the barriers); the elected lane issues and
            // commits inside mma_f16 / mma_commit.  Every operand is built from warp-uniform values (parameters,
            // constants, loop-carried counters; no division) so that the compiler keeps it in uniform registers: the
            // tensor memory base is the constant 0, which is what a CTA allocating all 512 columns receives.
            const bool tmem_ok = tmem == 0u;
            if (!tmem_ok && lane == 0) {
                *abort_flag = 1;
                atomicExch(err, 1);
            }
            // tile t's window of singles: W rows of each part of the B stage from row s0
            uint32_t idesc[kMaxTiles], dcol[kMaxTiles], dbuf[kMaxTiles];
            uint64_t bwin[kMaxTiles];
#pragma unroll
            for (int t = 0; t < kMaxTiles; ++t) {
                const int tt = t < ntiles ? t : 0;
                idesc[t] = idesc_bf16(128, G.tile_w[tt]);
                dcol[t] = (uint32_t)G.dm_col[tt];
                dbuf[t] = (uint32_t)G.tile_w[tt];
                bwin[t] = sdesc_sw128(smem_u32(bst) + (uint32_t)(128 * G.tile_s0[tt]));
            }
            const uint32_t a_step = (uint32_t)(kAcols * ntiles);
            // descriptor address steps (16-byte units; no carry out of the 14-bit field: shared memory < 2^18 bytes)
            const uint64_t b_part = (uint64_t)(G.bstage_bytes >> 4), b_step = kParts * b_part;
            int as = 0;
            uint32_t aph = 0, aa = (uint32_t)a_col0, db = 0, dph = 1;
            uint64_t bo = 0;
            for (int st = 0; st < nstages && tmem_ok; ++st) {
                // the epilogue has read this accumulator buffer's previous sums
                if (st >= kAccBufs && !warp_wait(&d_empty[db], dph, abort_flag, err)) break;
                if (!warp_wait(&a_full[as], aph, abort_flag, err)) break;
                tc_fence_after();
#pragma unroll
                for (int t = 0; t < kMaxTiles; ++t) {
                    if (t < ntiles) {
                        const uint32_t d = dcol[t] + (db ? dbuf[t] : 0u), a = aa + (uint32_t)(kAcols * t);
                        const uint64_t bd = bwin[t] + bo;
                        // K step ks: cells 16 ks .. 16 ks + 15, A part p at column 24 ks + 8 p.  B advances 32 bytes a
                        // step within the swizzle atom (2 in the descriptor)
                        auto products = [&](int pa, int pb) {
#pragma unroll
                            for (int ks = 0; ks < kKC / 16; ++ks)
                                mma_f16(d, a + (uint32_t)(8 * (kParts * ks + pa)),
                                        bd + pb * b_part + (uint64_t)(2 * ks), idesc[t], pa == 0 && pb == 2 && ks == 0 ? 0u : 1u);
                        };
                        products(0, 2);
                        products(2, 0);
                        products(1, 1);
                        products(0, 1);
                        products(1, 0);
                        products(0, 0);
                    }
                }
                mma_commit(&a_empty[as]);
                mma_commit(&d_full[db]);
                if (++as == nA) { as = 0; aph ^= 1u; aa = (uint32_t)a_col0; bo = 0; } else { aa += a_step; bo += b_step; }
                db ^= 1u;
                if (db == 0) dph ^= 1u;
            }
            // every MMA issued by the elected thread has completed before TMEM is released
            mma_commit(fin);
            drain_wait(fin, 0, err);
            __syncwarp();
        }
    } else if (warp < kProdWarp0) {
        // ------------------------------------------------------------------ the B operand
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsB));
        make_b(G, P, ring, bst, bscale, slot_full, slot_empty, a_full, a_empty, abort_flag, nstages, warp - kBWarp0, lane);
    } else if (warp < kProdWarp0 + kProdWarps) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsProd));
        // ------------------------------------------------------------------ producers
        switch (ntiles) {
            case 1: producer<1>(G, P, tmem, ring, slot_full, slot_empty, a_full, a_empty, abort_flag, nstages, warp, lane); break;
            default: producer<2>(G, P, tmem, ring, slot_full, slot_empty, a_full, a_empty, abort_flag, nstages, warp, lane); break;
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsEpi));
        // ------------------------------------------------------------------ epilogue
        switch (G.nunits) {
            case 1: epilogue<1>(G, P, tmem, acc64, d_full, d_empty, abort_flag, nstages, warp, lane); break;
            case 2: epilogue<2>(G, P, tmem, acc64, d_full, d_empty, abort_flag, nstages, warp, lane); break;
            default: epilogue<3>(G, P, tmem, acc64, d_full, d_empty, abort_flag, nstages, warp, lane); break;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

// absmax[row0 + r] = bit pattern of max |maps[r][x]| over the cells (blockIdx.y: map r; absmax zeroed before).  NaN and
// infinity order above every finite value as bit patterns.
__global__ void __launch_bounds__(256) k_absmax(const float4* __restrict__ maps, long n4, uint32_t* __restrict__ absmax) {
    const float4* m = maps + (size_t)blockIdx.y * n4;
    uint32_t a = 0;
    for (long i = (long)blockIdx.x * 256 + threadIdx.x; i < n4; i += (long)gridDim.x * 256) {
        const float4 v = m[i];
        a = max(max(a, max(__float_as_uint(v.x) & 0x7fffffffu, __float_as_uint(v.y) & 0x7fffffffu)),
                max(__float_as_uint(v.z) & 0x7fffffffu, __float_as_uint(v.w) & 0x7fffffffu));
    }
    a = __reduce_max_sync(0xffffffffu, a);
    if ((threadIdx.x & 31) == 0 && a) atomicMax(absmax + blockIdx.y, a);
}

// out[o] = 2^-(row and single exponents) sum over CTAs of partial[cta][gidx[o]], in CTA order (deterministic).  rows[o]
// holds the slot rows (j, k, single) of output o.
// 32 outputs x 16 slices of the CTAs a block (blockDim (32, 16)), as k_reduce_partials.
constexpr int kSlices = 16;
__global__ void __launch_bounds__(32 * kSlices) k_reduce_gather(const double* __restrict__ partial, int ncta, long stride,
                                                                const int* __restrict__ gidx,
                                                                const uchar4* __restrict__ rows,
                                                                const uint32_t* __restrict__ gmax,
                                                                const uint32_t* __restrict__ hmax, int h_row0, int n_out,
                                                                double* __restrict__ out) {
    __shared__ double red[kSlices][33];
    const int o = blockIdx.x * 32 + threadIdx.x;
    double s = 0.0;
    if (o < n_out) {
        const long g = gidx[o];
#pragma unroll 4
        for (int c = threadIdx.y; c < ncta; c += kSlices) s += partial[(long)c * stride + g];
    }
    red[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.y || o >= n_out) return;
    for (int q = 1; q < kSlices; ++q) s += red[q][threadIdx.x];
    const uchar4 r = rows[o];
    out[o] = ldexp(s, -row_exp(row_max(gmax, hmax, h_row0, r.x), row_max(gmax, hmax, h_row0, r.y)) -
                          single_exp(row_max(gmax, hmax, h_row0, r.z)));
}

// Self-test of the bounded waits: one thread waits on an mbarrier phase that nothing completes; the wait gives up
// after `limit` polls and raises the error flag, as a stalled pipeline would, and the kernel returns normally.
__global__ void k_wait_selftest(int* err, unsigned limit) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        unsigned it = 0;
        for (; it < limit; ++it)
            if (mbar_try(&bar, 0)) break;
        if (it == limit) atomicExch(err, 1);
    }
}

// ------------------------------------------------------------------------------------------------ self-check
// What the Gram matrix assumes of the tensor core, checked on known operands: an FP32 B operand is read as TF32
// by dropping its 13 low bits (B_hi = the raw row), and a TF32 value written to tensor memory as the A operand is
// used exactly.  A (tensor memory, M = 128, K = 8) has A[0][0] = 1 and A[1][0] = 1 + 2^-10; B (shared memory, N = 16,
// 128-byte swizzle) has B[0][0] = 1 + 3 2^-12, three quarters of a TF32 unit above 1.  Truncation gives D[0][0] = 1
// and D[1][0] = 1 + 2^-10; rounding to nearest would give 1 + 2^-10 and (1 + 2^-10)^2.  res: D[0][0], D[1][0] (FP32
// bit patterns) and a timeout flag.

__global__ void __launch_bounds__(128, 1) k_tf32_selfcheck(uint32_t* res) {
    __shared__ __align__(1024) unsigned char sB[16 * 128];
    __shared__ uint64_t bar;
    __shared__ uint32_t tslot;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    for (int i = tid; i < 16 * 128 / 4; i += 128) reinterpret_cast<uint32_t*>(sB)[i] = 0u;
    if (tid == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 32;" ::"r"(smem_u32(&tslot)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    __syncthreads();
    if (tid == 0) reinterpret_cast<float*>(sB)[0] = 1.0f + 3.0f * 0x1p-12f;   // row 0, chunk 0 (unswizzled position)
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tslot;
    {
        const int r = 32 * warp + lane;                  // TMEM lane of this thread
        uint32_t v[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
        if (r == 0) v[0] = __float_as_uint(1.0f);
        if (r == 1) v[0] = __float_as_uint(1.0f + 0x1p-10f);
        tmem_st8(tmem + ((uint32_t)(32 * warp) << 16), v);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) {
        mma_tf32(tmem + 8u, tmem, sdesc_sw128(smem_u32(sB)), idesc_tf32(128, 16), 0u);
        mma_commit(&bar);
        unsigned it = 0;
        for (; it < (1u << 20); ++it)
            if (mbar_try(&bar, 0)) break;
        if (lane == 0) res[2] = it == (1u << 20) ? 1u : 0u;
        tc_fence_after();
        uint32_t d[16];
        tmem_ld16(tmem + 8u, d);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (lane < 2) res[lane] = d[0];
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 32;" ::"r"(tmem));
}

// ------------------------------------------------------------------------------------------------ Gram
// Tensor-core Gram matrix of the bispectrum Fisher (Sec. 4.3.4, eq. bk-fish-def in Fourier space):
//   part[s][i][j] = sum_{k in split s} A[i][k] B[j][k],  A = Z (weighted), B = Y as float32 rows [n][K], K = 2 M
// (real and imaginary parts of the binned modes interleaved: re*re + im*im is the real part of conj(Z) Y).
// A CTA takes a 128 x 32 output tile and a contiguous range of K.  Arithmetic: A = A_hi + A_lo (A_hi rounded to TF32 by
// the producers, written to tensor memory), B_hi = the raw TMA tile (read as TF32 by truncation), B_lo = (B - trunc B) rounded to TF32; D_hh += A_hi B_hi, D_c += A_hi B_lo + A_lo B_hi; D restarts
// every 32 K (4 MMAs a column: the tensor core cuts each partial sum towards zero, and with 64 K the bispectrum Fisher term of
// 564 triplets came out 1.2e-7 too small instead of 4e-8; 10.72 -> 10.85 ms), FP32 register sums, FP64 register sums every
// 2048 K; FP64 partials per K split.
namespace gram {
constexpr int kBM = 128, kBN = 32, kKC = 32, kStages = 6, kPeriod = 1, kSpill = 64;
constexpr int kThreads = 384;   // warps 0 TMA/TMEM, 1 MMA, 2 B_lo, 3 idle, 4-7 A producers, 8-11 epilogue
constexpr int kAStage = kBM * 128, kBStage = kBN * 128;   // raw tiles: 32 floats (128 B) a row
constexpr int kSmem = kStages * (kAStage + 2 * kBStage) + 1024 + 256;

struct GP {
    long k_cta;       // K per CTA (multiple of kKC)
    long K;           // row length (floats)
    int nA, nB, nsplit;
    double* part;     // [nsplit][nI*128][nJ*32]
    long ldp;         // row stride of part (nJ * 32)
    long split_stride;
    int* err;
};

__global__ void __launch_bounds__(kThreads, 1)
    k_gram_tc(const __grid_constant__ CUtensorMap tA, const __grid_constant__ CUtensorMap tB, const __grid_constant__ GP P) {
    extern __shared__ __align__(1024) unsigned char gsm_raw[];
    unsigned char* sm = gsm_raw + ((1024u - (smem_u32(gsm_raw) & 1023u)) & 1023u);
    unsigned char* sA = sm;                                       // [kStages][kAStage]
    unsigned char* sB = sA + kStages * kAStage;                   // [kStages][kBStage]
    unsigned char* sBl = sB + kStages * kBStage;                  // [kStages][kBStage]
    uint64_t* bars = reinterpret_cast<uint64_t*>(sBl + kStages * kBStage);
    uint64_t* full = bars;                      // [kStages] TMA -> A producers, B_lo warp
    uint64_t* ready = full + kStages;           // [kStages] A producers + B_lo -> MMA
    uint64_t* empty = ready + kStages;          // [kStages] MMA commit -> TMA
    uint64_t* d_full = empty + kStages;         // MMA -> epilogue (period done)
    uint64_t* d_empty = d_full + 1;             // epilogue -> MMA
    uint64_t* fin = d_empty + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(fin + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int i0 = blockIdx.y * kBM, j0 = blockIdx.x * kBN;
    const long k0 = (long)blockIdx.z * P.k_cta;
    const long k1 = min(P.K, k0 + P.k_cta);
    const int nst = k0 < k1 ? (int)((k1 - k0 + kKC - 1) / kKC) : 0;
    int* const err = P.err;
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&ready[s], 5);
            mbar_init(&empty[s], 1);
        }
        mbar_init(d_full, 1);
        mbar_init(d_empty, 4);
        mbar_init(fin, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // TMEM columns: D_hh [0, 32), D_c [32, 64), A stage s: hi [64 + 64 s, +32), lo [+32, +64)
    if (warp == 0) {
        if (lane == 0 && nst > 0) {
            int issued = 0;
            for (int st = 0; st < nst; ++st) {
                const int s = st % kStages;
                if (st >= kStages && !thread_wait(&empty[s], (uint32_t)((st / kStages - 1) & 1), abort_flag, err)) break;
                const int x = (int)(k0 + (long)st * kKC);
                mbar_expect_tx(&full[s], (uint32_t)(kAStage + kBStage));
                tma_load_2d(sA + (size_t)s * kAStage, &tA, x, i0, &full[s]);
                tma_load_2d(sB + (size_t)s * kBStage, &tB, x, j0, &full[s]);
                ++issued;
            }
            for (int st = max(0, issued - kStages); st < issued; ++st)
                drain_wait(&full[st % kStages], (uint32_t)((st / kStages) & 1), err);
        }
        __syncwarp();
    } else if (warp == 1) {
        // MMA issue (whole warp converged; the elected lane issues)
        const bool tmem_ok = tmem == 0u;
        if (!tmem_ok && lane == 0) { *abort_flag = 1; atomicExch(err, 1); }
        const uint32_t idesc = idesc_tf32(kBM, kBN);
        const uint64_t bh0 = sdesc_sw128(smem_u32(sB)), bl0 = sdesc_sw128(smem_u32(sBl));
        const uint64_t bstep = (uint64_t)(kBStage >> 4);
        int s = 0, pos = 0, per = 0;
        uint32_t ph = 0;
        uint32_t aa = 64u;
        uint64_t bh = bh0, bl = bl0;
        for (int st = 0; st < nst && tmem_ok; ++st) {
            const bool pstart = pos == 0;
            if (pstart && per >= 1 && !warp_wait(d_empty, (uint32_t)((per - 1) & 1), abort_flag, err)) break;
            if (!warp_wait(&ready[s], ph, abort_flag, err)) break;
            tc_fence_after();
#pragma unroll
            for (int ks = 0; ks < kKC / 8; ++ks) {
                const uint32_t acc = (pstart && ks == 0) ? 0u : 1u;
                mma_tf32(0u, aa + 8u * ks, bh + (uint64_t)(2 * ks), idesc, acc);          // A_hi B_hi
                mma_tf32(32u, aa + 8u * ks, bl + (uint64_t)(2 * ks), idesc, acc);         // A_hi B_lo
                mma_tf32(32u, aa + 32u + 8u * ks, bh + (uint64_t)(2 * ks), idesc, 1u);    // + A_lo B_hi
            }
            mma_commit(&empty[s]);
            if (pos == kPeriod - 1 || st == nst - 1) mma_commit(d_full);
            if (++s == kStages) { s = 0; ph ^= 1u; aa = 64u; bh = bh0; bl = bl0; } else { aa += 64u; bh += bstep; bl += bstep; }
            if (++pos == kPeriod) { pos = 0; ++per; }
        }
        mma_commit(fin);
        drain_wait(fin, 0, err);
        __syncwarp();
    } else if (warp == 2) {
        // B_lo = (B - trunc B) rounded to TF32, same swizzled layout: 32 rows x 8 chunks, 8 chunks a lane
        int s = 0;
        uint32_t ph = 0;
        for (int st = 0; st < nst; ++st) {
            if (!warp_wait(&full[s], ph, abort_flag, err)) break;
            const unsigned char* src = sB + (size_t)s * kBStage;
            unsigned char* dst = sBl + (size_t)s * kBStage;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = lane + 32 * u;
                const uint4 g = *reinterpret_cast<const uint4*>(src + 16 * i);
                const uint64_t g01 = (uint64_t)g.x | ((uint64_t)g.y << 32);
                const uint64_t g23 = (uint64_t)g.z | ((uint64_t)g.w << 32);
                const uint64_t l01 = sub_x2(g01, g01 & 0xFFFFE000FFFFE000ull);
                const uint64_t l23 = sub_x2(g23, g23 & 0xFFFFE000FFFFE000ull);
                *reinterpret_cast<uint4*>(dst + 16 * i) =
                    make_uint4(((uint32_t)l01 + 0x1000u) & 0xFFFFE000u, ((uint32_t)(l01 >> 32) + 0x1000u) & 0xFFFFE000u,
                               ((uint32_t)l23 + 0x1000u) & 0xFFFFE000u, ((uint32_t)(l23 >> 32) + 0x1000u) & 0xFFFFE000u);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&ready[s]);
            if (++s == kStages) { s = 0; ph ^= 1u; }
        }
    } else if (warp >= 4 && warp < 8) {
        // A producers: thread = row r = 32 (warp % 4) + lane of the tile = TMEM lane r; hi / lo of the 32 K values
        const int q = warp & 3, r = 32 * q + lane;
        const uint32_t lane_base = (uint32_t)(32 * q) << 16;
        if (tmem == 0u) {
            int s = 0;
            uint32_t ph = 0;
            uint32_t ac = 64u;
            for (int st = 0; st < nst; ++st) {
                if (!warp_wait(&full[s], ph, abort_flag, err)) break;
                const unsigned char* row = sA + (size_t)s * kAStage;
                uint32_t v[32], w[32];
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float4 x = *ring_chunk(row, r, c);
                    uint64_t h0, l0, h1, l1;
                    split_x2(f2pack(x.x, x.y), h0, l0);
                    split_x2(f2pack(x.z, x.w), h1, l1);
                    v[4 * c + 0] = (uint32_t)h0; v[4 * c + 1] = (uint32_t)(h0 >> 32);
                    v[4 * c + 2] = (uint32_t)h1; v[4 * c + 3] = (uint32_t)(h1 >> 32);
                    w[4 * c + 0] = (uint32_t)l0; w[4 * c + 1] = (uint32_t)(l0 >> 32);
                    w[4 * c + 2] = (uint32_t)l1; w[4 * c + 3] = (uint32_t)(l1 >> 32);
                }
                tmem_st32(lane_base + ac, v);
                tmem_st32(lane_base + ac + 32u, w);
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&ready[s]);
                if (++s == kStages) { s = 0; ph ^= 1u; ac = 64u; } else { ac += 64u; }
            }
        }
    } else if (warp >= 8) {
        // epilogue: lane r of the tile; every period add D_hh + D_c into FP32 sums, every kSpill periods into FP64
        const int q = warp & 3, r = 32 * q + lane;
        const uint32_t lane_base = (uint32_t)(32 * q) << 16;
        const int nper = (nst + kPeriod - 1) / kPeriod;
        float acc[kBN];
        double acc64[kBN];
#pragma unroll
        for (int j = 0; j < kBN; ++j) { acc[j] = 0.f; acc64[j] = 0.0; }
        for (int per = 0; per < nper; ++per) {
            if (!warp_wait(d_full, (uint32_t)(per & 1), abort_flag, err)) break;
            tc_fence_after();
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t a[16], b[16];
                tmem_ld16(tmem + lane_base + 16u * h, a);
                tmem_ld16(tmem + lane_base + 32u + 16u * h, b);
                tmem_wait_ld32(a, b);
#pragma unroll
                for (int j = 0; j < 16; ++j) acc[16 * h + j] += __uint_as_float(a[j]) + __uint_as_float(b[j]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(d_empty);
            if ((per + 1) % kSpill == 0) {
#pragma unroll
                for (int j = 0; j < kBN; ++j) { acc64[j] += (double)acc[j]; acc[j] = 0.f; }
            }
        }
        double* out = P.part + (size_t)blockIdx.z * P.split_stride + (size_t)(i0 + r) * P.ldp + j0;
#pragma unroll
        for (int j = 0; j < kBN; ++j) out[j] = acc64[j] + (double)acc[j];
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

// out[i][j] += scale * sum_s part[s][i][j] (splits in order), i < nA, j < nB.
__global__ void k_gram_reduce(const double* __restrict__ part, int nsplit, long split_stride, long ldp, int nA, int nB,
                              double scale, double* __restrict__ out) {
    const long o = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= (long)nA * nB) return;
    const int i = (int)(o / nB), j = (int)(o - (long)i * nB);
    double s = 0.0;
    for (int q = 0; q < nsplit; ++q) s += part[(size_t)q * split_stride + (size_t)i * ldp + j];
    out[o] += scale * s;
}
}  // namespace gram

// ------------------------------------------------------------------------------------------------ host planner

// A pair row with the range of singles it needs and where each of its outputs goes.
struct NeedPair {
    int j, k;
    int lo, hi;                                   // singles needed: [lo, hi]
    std::vector<std::pair<int, int>> outs;        // (single, output index)
};

// Run-time choices of a plan that leave the kernel unchanged, tried by the autotuner: the per-tile cost of the
// tile-cutting DP (small: more, narrower tiles; large: fewer, wider ones), the number of tiles a row group (CTA)
// may take, and the cell split (0: one CTA per SM and row group, ngroups waves; 1: one wave of SMs / ngroups CTAs
// per group; 2: two CTAs per SM and row group, shorter cell ranges).
struct PlanOpts {
    int tile_cost = 8;
    int group_cap = kMaxTiles;
    int cta_mode = 0;
};

struct Plan {
    int ng = 0, nh = 0, hsep = 0, n_out = 0, ncta = 0, ngroups = 0, total_units = 0;
    PlanOpts opts{};
    bool tuned = false;
    float tuned_ms = 0.f;   // time of the chosen candidate (0 when not tuned)
    int tuned_of = 0;       // candidates timed
    // what the plan was built from (the autotuner rebuilds it with other options)
    std::vector<NeedPair> need;
    int sing_g = 0;
    long ncell = 0;
    long cells_cta = 0;
    Params base{};
    size_t smem = 0;
    short2* d_rows = nullptr;
    int* d_gidx = nullptr;
    uchar4* d_orows = nullptr;   // slot rows (j, k, single) of every output
    double* d_partial = nullptr;
    ~Plan() {
        if (d_orows) cudaFree(d_orows);
        if (d_rows) cudaFree(d_rows);
        if (d_gidx) cudaFree(d_gidx);
        if (d_partial) cudaFree(d_partial);
    }
};

static int round_w(int w) { return w <= 16 ? 16 : 32; }

// Tiles of <= 128 pairs, consecutive in the order of (hi, lo), cut by dynamic programming to minimise the summed
// window width (the tensor work) plus a per-tile cost.
static std::vector<std::pair<int, int>> cut_tiles(const std::vector<NeedPair>& P, int tile_cost) {
    const int n = (int)P.size();
    std::vector<long> f(n + 1, (long)1 << 40);
    std::vector<int> arg(n + 1, 0);
    f[0] = 0;
    for (int i = 1; i <= n; ++i) {
        int lo = 1 << 30, hi = -1;
        for (int j = i - 1; j >= 0 && j >= i - 128; --j) {
            lo = std::min(lo, P[j].lo);
            hi = std::max(hi, P[j].hi);
            const int s0 = lo / 8 * 8;
            if (hi + 1 - s0 > 32) break;
            const long c = f[j] + round_w(hi + 1 - s0) + tile_cost;
            if (c < f[i]) { f[i] = c; arg[i] = j; }
        }
    }
    std::vector<std::pair<int, int>> seg;
    for (int i = n; i > 0; i = arg[i]) seg.push_back({arg[i], i});
    std::reverse(seg.begin(), seg.end());
    return seg;
}

// A set of maps (slot rows, at most 128), and the largest number of them in one bank group (map % 8).
struct MapSet {
    uint64_t w[2] = {0, 0};
    void add(int m) { w[m >> 6] |= 1ull << (m & 63); }
    void drop(int m) { w[m >> 6] &= ~(1ull << (m & 63)); }
    bool has(int m) const { return (w[m >> 6] >> (m & 63)) & 1; }
    int size() const { return __builtin_popcountll(w[0]) + __builtin_popcountll(w[1]); }
    int clash() const {
        int most = 0;
        for (int g = 0; g < 8; ++g) {
            const uint64_t m = 0x0101010101010101ull << g;
            most = std::max(most, __builtin_popcountll(w[0] & m) + __builtin_popcountll(w[1] & m));
        }
        return most;
    }
};
static MapSet operator&(MapSet a, const MapSet& b) {
    a.w[0] &= b.w[0];
    a.w[1] &= b.w[1];
    return a;
}

// Orders the rows [first, last) of a tile, sorted by (j, k), for the producers' gathers, which bound the kernel by shared
// memory.  A 16-byte load of a warp is served for eight lanes at a time, or for sixteen where lanes i and i ^ 1, or i and
// i ^ 2, read the same address throughout (measured: 4 and 2 cycles a load); the slots' swizzle puts chunk c of map m into
// bank group c ^ (m % 8), so different maps of one group that are equal modulo 8 clash.
// Rows therefore come in quads (j1, k1) (j1, k2) (j2, k1) (j2, k2), whose lanes share j by i ^ 1 and k by i ^ 2, and four
// quads a half-warp are taken to clash least; rows that form no quad follow, eight at a time that clash least.
static void order_rows(std::vector<NeedPair>& need, int first, int last) {
    const std::vector<NeedPair> rest(need.begin() + first, need.begin() + last);
    const int n = (int)rest.size();
    std::vector<short> at(128 * 128, -1);                 // row of (j, k)
    MapSet ks[128];                                       // the k of the rows left of every j
    MapSet jset;
    bool plain = true;                                    // maps in range and no pair twice
    for (int i = 0; i < n; ++i) {
        const int j = rest[i].j, k = rest[i].k;
        if (j < 0 || k < 0 || j >= 128 || k >= 128) return;
        plain = plain && !ks[j].has(k);
        ks[j].add(k);
        jset.add(j);
        at[j * 128 + k] = (short)i;
    }
    std::vector<int> js, order;
    for (int j = 0; j < 128; ++j)
        if (jset.has(j)) js.push_back(j);
    if (plain) {
        // quads: of all pairs of j the one with the most k in common first, so that few rows are left over
        struct Quad { int r[4], j[2], k[2]; };
        std::vector<Quad> quads;
        for (;;) {
            int b1 = -1, b2 = -1, most = 0;
            for (size_t x = 0; x < js.size(); ++x)
                for (size_t y = x + 1; y < js.size(); ++y) {
                    const int c = (ks[js[x]] & ks[js[y]]).size() / 2;
                    if (c > most) { most = c; b1 = js[x]; b2 = js[y]; }
                }
            if (!most) break;
            const MapSet both = ks[b1] & ks[b2];
            for (int k = 0, k1 = -1, c = 0; c < 2 * most; ++k) {
                if (!both.has(k)) continue;
                ++c;
                if (k1 < 0) { k1 = k; continue; }
                quads.push_back({{at[b1 * 128 + k1], at[b1 * 128 + k], at[b2 * 128 + k1], at[b2 * 128 + k]}, {b1, b2}, {k1, k}});
                for (int q : {k1, k}) { ks[b1].drop(q); ks[b2].drop(q); }
                k1 = -1;
            }
        }
        std::vector<char> used(quads.size(), 0);
        for (size_t done = 0; done < quads.size();) {
            MapSet mj, mk;                                // of a half-warp
            for (int g = 0; g < 4 && done < quads.size(); ++g, ++done) {
                int best = -1, best_cost = 1 << 30;
                for (size_t i = 0; i < quads.size() && best_cost > 2; ++i) {
                    if (used[i]) continue;
                    MapSet a = mj, b = mk;
                    for (int q = 0; q < 2; ++q) { a.add(quads[i].j[q]); b.add(quads[i].k[q]); }
                    const int cost = a.clash() + b.clash();
                    if (cost < best_cost) { best_cost = cost; best = (int)i; }
                }
                used[best] = 1;
                for (int q = 0; q < 2; ++q) { mj.add(quads[best].j[q]); mk.add(quads[best].k[q]); }
                order.insert(order.end(), quads[best].r, quads[best].r + 4);
            }
        }
    }
    std::vector<char> used(n, 0);
    for (int i : order) used[i] = 1;
    MapSet mj, mk;                                        // of eight lanes
    while ((int)order.size() < n) {
        int best = -1, best_cost = 1 << 30;
        for (int i = 0; i < n && best_cost > 2; ++i) {
            if (used[i]) continue;
            MapSet a = mj, b = mk;
            a.add(rest[i].j);
            b.add(rest[i].k);
            const int cost = a.clash() + b.clash();
            if (cost < best_cost) { best_cost = cost; best = i; }
        }
        used[best] = 1;
        mj.add(rest[best].j);
        mk.add(rest[best].k);
        order.push_back(best);
        if (order.size() % 8 == 0) { mj = MapSet{}; mk = MapSet{}; }
    }
    for (int i = 0; i < n; ++i) need[first + i] = rest[order[i]];
}

// Pure host layout of a plan (no CUDA calls): tiles, row groups, TMEM / shared-memory layout, the row table and the
// gather index of every output.  Returns nullptr or an error message.
// sing_g = 1 with hsep = 1: the slot holds the g rows and the h rows (pairs may take one map from each, h rows at
// index h_row0 + i) and the singles are the g rows.
static const char* layout_plan(Plan& pl, long ncell, int nsm, int ng, int nh, int hsep, std::vector<NeedPair> need,
                               int n_out, std::vector<short2>& rows, std::vector<int>& gidx, int sing_g = 0,
                               const PlanOpts& opts = PlanOpts{}) {
    pl.ng = ng; pl.nh = nh; pl.hsep = hsep; pl.n_out = n_out;
    pl.opts = opts;
    if (opts.group_cap < 1 || opts.group_cap > kMaxTiles || opts.cta_mode < 0 || opts.cta_mode > 2)
        return "contract_tc: bad plan options";
    std::stable_sort(need.begin(), need.end(), [](const NeedPair& a, const NeedPair& b) {
        return std::tie(a.hi, a.lo) < std::tie(b.hi, b.lo);
    });
    for (const NeedPair& p : need)
        if (p.hi + 1 - p.lo / 8 * 8 > 32) return "contract_tc: a pair needs a window of more than 32 singles";
    auto seg = need.empty() ? std::vector<std::pair<int, int>>{} : cut_tiles(need, opts.tile_cost);
    struct TileH { int first, last, s0, W; };
    std::vector<TileH> tiles;
    for (auto& sg : seg) {
        int lo = 1 << 30, hi = -1;
        for (int i = sg.first; i < sg.second; ++i) { lo = std::min(lo, need[i].lo); hi = std::max(hi, need[i].hi); }
        const int s0 = lo / 8 * 8;
        std::stable_sort(need.begin() + sg.first, need.begin() + sg.second,
                         [](const NeedPair& a, const NeedPair& b) { return std::tie(a.j, a.k) < std::tie(b.j, b.k); });
        order_rows(need, sg.first, sg.second);
        tiles.push_back({sg.first, sg.second, s0, round_w(hi + 1 - s0)});
    }
    if (tiles.empty()) tiles.push_back({0, 0, 0, 16});
    // row groups: consecutive tiles while TMEM (the accumulators + two A stages) and the 3 output units allow
    std::vector<std::pair<int, int>> groups;
    for (int t = 0; t < (int)tiles.size();) {
        int e = t, dcols = 0, units = 0;
        while (e < (int)tiles.size() && e - t < opts.group_cap) {
            const int nd = dcols + 2 * tiles[e].W, nu = units + tiles[e].W / 16, nt = e - t + 1;
            if (nu > kMaxUnits || kDBuf * ((nd + 31) / 32 * 32) + 2 * kAcols * nt > 512) break;
            dcols = nd; units = nu; ++e;
        }
        if (e == t) return "contract_tc: tile does not fit tensor memory";
        groups.push_back({t, e});
        t = e;
    }
    if ((int)groups.size() > kMaxGroups) return "contract_tc: more than 4 row groups";
    pl.ngroups = (int)groups.size();

    Params& P = pl.base;
    P = Params{};
    P.ng = ng; P.nh = nh; P.hsep = hsep;
    const int grows = (ng + 7) / 8 * 8;
    P.h_row0 = grows;
    P.slot_bytes = (grows + (hsep ? (nh + 7) / 8 * 8 : 0)) * 128;
    const bool sh = hsep && !sing_g;                        // singles from the h rows
    const int srows = sh ? (nh + 7) / 8 * 8 : grows;       // rows of the singles region of a slot
    P.s_off = sh ? grows * 128 : 0;
    P.s_chunks = srows * 8;
    if (P.s_chunks > 256 * kBloItems) return "contract_tc: more than 64 rows of singles";
    int max_b = 0, max_units = 0;
    rows.assign(tiles.size() * 128, make_short2(-1, -1));
    gidx.assign(std::max(n_out, 1), 0);
    int unit_base = 0;
    for (int gi = 0; gi < pl.ngroups; ++gi) {
        GroupDesc& D = P.grp[gi];
        D = GroupDesc{};
        const int t0 = groups[gi].first, nt = groups[gi].second - t0;
        D.tile0 = t0; D.ntiles = nt; D.unit_base = unit_base;
        // accumulators (two buffers of W columns) of every tile, largest first, so each is aligned to its size
        std::vector<std::pair<int, int>> dl;   // (size, tile)
        for (int t = 0; t < nt; ++t) dl.push_back({2 * tiles[t0 + t].W, t});
        std::stable_sort(dl.begin(), dl.end(), [](auto& a, auto& b) { return a.first > b.first; });
        int col = 0;
        for (auto& x : dl) {
            D.dm_col[x.second] = col;
            col += x.first;
        }
        D.d_cols = (col + 31) / 32 * 32;
        D.a_col0 = kDBuf * D.d_cols;
        D.nA = std::min(kMaxAStages, (512 - D.a_col0) / (kAcols * nt));
        // windows of singles; B stages hold a slot's whole singles region, in parts
        for (int t = 0; t < nt; ++t) {
            const TileH& T = tiles[t0 + t];
            D.tile_w[t] = T.W;
            D.tile_s0[t] = T.s0;
        }
        D.bstage_bytes = srows * 128;
        max_b = std::max(max_b, D.nA * kParts * D.bstage_bytes);
        // output units
        int u = 0;
        for (int t = 0; t < nt; ++t)
            for (int c = 0; c < tiles[t0 + t].W; c += 16) { D.unit_tile[u] = t; D.unit_c[u] = c; ++u; }
        D.nunits = u;
        for (int x = u; x < kMaxUnits; ++x) { D.unit_tile[x] = kMaxTiles; D.unit_c[x] = 0; }
        max_units = std::max(max_units, u);
        // rows and the gather index of every output
        for (int t = 0; t < nt; ++t) {
            const TileH& T = tiles[t0 + t];
            int uf = 0;
            while (D.unit_tile[uf] != t) ++uf;
            for (int i = T.first; i < T.last; ++i) {
                const int r = i - T.first;
                rows[(size_t)(t0 + t) * 128 + r] = make_short2((short)need[i].j, (short)need[i].k);
                for (auto& so : need[i].outs) {
                    const int cc = so.first - T.s0;
                    const int gu = unit_base + uf + cc / 16;
                    gidx[so.second] = (gu * 16 + cc % 16) * 128 + r;
                }
            }
        }
        unit_base += u;
    }
    pl.total_units = unit_base;
    P.total_units = unit_base;
    P.off_b = kRingSlots * P.slot_bytes;
    P.off_acc = P.off_b + max_b;
    P.off_bar = P.off_acc + kMaxUnits * 16 * 128 * 8;
    // + 1024: the kernel aligns the start of its dynamic shared memory to 1024 bytes (128-byte swizzle atoms)
    pl.smem = std::max((size_t)kMinSmem, (size_t)P.off_bar + 64 * 8 + 64 * 4) + 1024;
    if (pl.smem > 227 * 1024) return "contract_tc: shared memory plan exceeds 227 KB";

    const long nsl = (ncell + kKC - 1) / kKC;
    const long want = opts.cta_mode == 1 ? std::max(1L, (long)nsm / pl.ngroups) : (opts.cta_mode == 2 ? 2L * nsm : (long)nsm);
    pl.ncta = (int)std::max(1L, std::min(want, nsl));
    pl.cells_cta = (nsl + pl.ncta - 1) / pl.ncta * kKC;
    pl.ncta = (int)((ncell + pl.cells_cta - 1) / pl.cells_cta);
    P.ncell = ncell;
    P.cells_cta = pl.cells_cta;
    return nullptr;
}

struct PlanCache {
    std::map<std::tuple<int, int, int, int, long>, Plan*> plans;   // (ng, nh, hsep, kind, ncell)
    double* gram_part = nullptr;                                   // Gram partials (K splits)
    size_t gram_cap = 0;
    uint32_t* d_absmax = nullptr;                                  // [2][64] maxima of g and h maps found here
    ~PlanCache() {
        if (d_absmax) cudaFree(d_absmax);
        for (auto& kv : plans) delete kv.second;
        if (gram_part) cudaFree(gram_part);
    }
};

static PlanCache* cache_of(polybin_ctx* ctx) {
    if (!ctx->tc) ctx->tc = new PlanCache();
    return static_cast<PlanCache*>(ctx->tc);
}

static int build_plan(polybin_ctx* ctx, Plan& pl, long ncell, int ng, int nh, int hsep, std::vector<NeedPair> need,
                      int n_out, int sing_g = 0, const PlanOpts& opts = PlanOpts{}, bool quiet = false) {
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return fail_cuda(ctx, e, "cudaDeviceGetAttribute", __FILE__, __LINE__);
    std::vector<short2> rows;
    std::vector<int> gidx;
    pl.need = need;
    pl.sing_g = sing_g;
    pl.ncell = ncell;
    std::vector<uchar4> orows(std::max(n_out, 1), make_uchar4(0, 0, 0, 0));
    const int srow0 = (hsep && !sing_g) ? (ng + 7) / 8 * 8 : 0;      // slot row of the first single
    for (const NeedPair& p : need)
        for (auto& so : p.outs)
            orows[so.second] = make_uchar4((unsigned char)p.j, (unsigned char)p.k, (unsigned char)(srow0 + so.first), 0);
    const char* msg = layout_plan(pl, ncell, nsm, ng, nh, hsep, std::move(need), n_out, rows, gidx, sing_g, opts);
    if (msg) return quiet ? POLYBIN_EINVAL : fail(ctx, POLYBIN_EINVAL, "%s", msg);
    PlanCache* pc = cache_of(ctx);
    if (!pc->d_absmax) PB_CUDA_OK(cudaMalloc(&pc->d_absmax, sizeof(uint32_t) * 2 * kMaxItems));
    PB_CUDA_OK(cudaMalloc(&pl.d_rows, sizeof(short2) * rows.size()));
    PB_CUDA_OK(cudaMemcpy(pl.d_rows, rows.data(), sizeof(short2) * rows.size(), cudaMemcpyHostToDevice));
    PB_CUDA_OK(cudaMalloc(&pl.d_gidx, sizeof(int) * gidx.size()));
    PB_CUDA_OK(cudaMemcpy(pl.d_gidx, gidx.data(), sizeof(int) * gidx.size(), cudaMemcpyHostToDevice));
    PB_CUDA_OK(cudaMalloc(&pl.d_orows, sizeof(uchar4) * orows.size()));
    PB_CUDA_OK(cudaMemcpy(pl.d_orows, orows.data(), sizeof(uchar4) * orows.size(), cudaMemcpyHostToDevice));
    PB_CUDA_OK(cudaMalloc(&pl.d_partial, sizeof(double) * (size_t)pl.ncta * pl.total_units * 2048));
    pl.base.rows = pl.d_rows;
    pl.base.partial = pl.d_partial;
    return POLYBIN_OK;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, []() {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

// 2D map over `rows` maps of ncell floats (map-major): box = 32 cells x all maps, 128-byte swizzle.
static int make_map(polybin_ctx* ctx, CUtensorMap* m, const float* base, int rows, long ncell) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return fail(ctx, POLYBIN_ECUDA, "contract_tc: cuTensorMapEncodeTiled is not available");
    if (reinterpret_cast<uintptr_t>(base) % 16) return fail(ctx, POLYBIN_EINVAL, "contract_tc: maps must be 16-byte aligned");
    const cuuint64_t dims[2] = {(cuuint64_t)ncell, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ncell * sizeof(float)};
    const cuuint32_t box[2] = {(cuuint32_t)kSlotCells, (cuuint32_t)rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(ctx, POLYBIN_ECUDA, "contract_tc: cuTensorMapEncodeTiled failed (%d)", (int)r);
    return POLYBIN_OK;
}

// 2D map over a row-major float32 matrix [height][width] (row stride width floats), box = box_w x box_h,
// 128-byte swizzle (box_w = 32 floats), out-of-range elements read as zero.
static int make_map2(polybin_ctx* ctx, CUtensorMap* m, const float* base, long width, long height, int box_w, int box_h) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return fail(ctx, POLYBIN_ECUDA, "gram: cuTensorMapEncodeTiled is not available");
    if (reinterpret_cast<uintptr_t>(base) % 16 || (width * (long)sizeof(float)) % 16)
        return fail(ctx, POLYBIN_EINVAL, "gram: rows must be 16-byte aligned");
    const cuuint64_t dims[2] = {(cuuint64_t)width, (cuuint64_t)height};
    const cuuint64_t strides[1] = {(cuuint64_t)width * sizeof(float)};
    const cuuint32_t box[2] = {(cuuint32_t)box_w, (cuuint32_t)box_h};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(ctx, POLYBIN_ECUDA, "gram: cuTensorMapEncodeTiled failed (%d)", (int)r);
    return POLYBIN_OK;
}

// gmax, hmax: the maps' maxima (kMaxItems entries each), or null: found here first.
static int launch(polybin_ctx* ctx, Plan& pl, const float* g, const float* h, double* d_out, const uint32_t* gmax,
                  const uint32_t* hmax) {
    CUtensorMap mg, mh;
    int rc = make_map(ctx, &mg, g, pl.ng, pl.base.ncell);
    if (rc) return rc;
    if (pl.hsep) {
        if ((rc = make_map(ctx, &mh, h, pl.nh, pl.base.ncell))) return rc;
    } else {
        mh = mg;
    }
    if ((rc = ensure_err_flag(ctx))) return rc;
    // (under capture the flag stays set for the rest of the graph, which clears it at its head and hands it out at its end)
    cudaError_t e = ctx->capturing ? cudaSuccess : cudaMemsetAsync(ctx->d_err, 0, sizeof(int), ctx->stream);
    if (e != cudaSuccess) return fail_cuda(ctx, e, "cudaMemsetAsync", __FILE__, __LINE__);
    e = cudaFuncSetAttribute((const void*)k_contract_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pl.smem);
    if (e != cudaSuccess) return fail_cuda(ctx, e, "cudaFuncSetAttribute(k_contract_tc)", __FILE__, __LINE__);
    {
        // the setmaxnreg split assumes exactly kRegsLaunch registers a thread at launch (a smaller allocation would
        // leave the producers' increase waiting for registers that do not exist)
        cudaFuncAttributes fa{};
        e = cudaFuncGetAttributes(&fa, (const void*)k_contract_tc);
        if (e != cudaSuccess) return fail_cuda(ctx, e, "cudaFuncGetAttributes(k_contract_tc)", __FILE__, __LINE__);
        if (fa.numRegs != kRegsLaunch)
            return fail(ctx, POLYBIN_ECUDA, "contract_tc: kernel built with %d registers a thread, %d expected", fa.numRegs,
                        kRegsLaunch);
    }
    PlanCache* pc = cache_of(ctx);
    Params P = pl.base;
    P.err = ctx->d_err;
    if (!gmax) {
        if ((rc = run_absmax(ctx, g, pl.ng, pl.base.ncell, pc->d_absmax))) return rc;
        gmax = pc->d_absmax;
    }
    if (pl.hsep && !hmax) {
        if ((rc = run_absmax(ctx, h, pl.nh, pl.base.ncell, pc->d_absmax + kMaxItems))) return rc;
        hmax = pc->d_absmax + kMaxItems;
    }
    P.gmax = gmax;
    P.hmax = pl.hsep ? hmax : gmax;
    {
        StageTimer timer(ctx, kStageContract);
        k_contract_tc<<<dim3(pl.ncta, pl.ngroups, 1), kThreads, pl.smem, ctx->stream>>>(mg, mh, P);
        ctx->launches += 1;
        e = cudaGetLastError();
        if (e != cudaSuccess) return fail_cuda(ctx, e, "k_contract_tc", __FILE__, __LINE__);
        k_reduce_gather<<<(pl.n_out + 31) / 32, dim3(32, kSlices), 0, ctx->stream>>>(
            pl.d_partial, pl.ncta, (long)pl.total_units * 2048, pl.d_gidx, pl.d_orows, P.gmax, P.hmax,
            pl.base.h_row0, pl.n_out, d_out);
        ctx->launches += 1;
        e = cudaGetLastError();
        if (e != cudaSuccess) return fail_cuda(ctx, e, "k_reduce_gather", __FILE__, __LINE__);
    }
    if (ctx->capturing) return POLYBIN_OK;   // the caller reads the error flags after the graph has run
    return read_err_flags(ctx, "contract_tc");
}

// Autotuner.  On the first launch of a plan outside stream capture (unless POLYBIN_AUTOTUNE=0), every distinct valid
// candidate of the option grid {tile cost 8, 24} x {2 or 1 tiles a group} x {cell splits 0, 1, 2} runs on the
// caller's own inputs, timed with CUDA events on the context stream (one launch to warm up, two timed); the fastest
// replaces the plan in the cache.  Candidates differ only in how cells and rows are split, so their results agree to
// FP32 rounding of the partial sums; after tuning every call takes the chosen plan.
static int tune_plan(polybin_ctx* ctx, Plan** pl_io, const float* g, const float* h, double* d_out, const uint32_t* gmax,
                     const uint32_t* hmax) {
    Plan* pl = *pl_io;
    if (pl->tuned) return POLYBIN_OK;
    if (ctx->capturing) {   // a captured graph keeps this plan's buffers: it must never be replaced
        pl->tuned = true;
        return POLYBIN_OK;
    }
    const char* env = std::getenv("POLYBIN_AUTOTUNE");
    if (env && env[0] == '0') { pl->tuned = true; return POLYBIN_OK; }
    PlanCache* pc = cache_of(ctx);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    PB_CUDA_OK(cudaEventCreate(&e0));
    PB_CUDA_OK(cudaEventCreate(&e1));
    auto time_plan = [&](Plan& c, float* ms) -> int {
        int rc;
        if ((rc = launch(ctx, c, g, h, d_out, gmax, hmax))) return rc;
        PB_CUDA_OK(cudaEventRecord(e0, ctx->stream));
        for (int i = 0; i < 2; ++i)
            if ((rc = launch(ctx, c, g, h, d_out, gmax, hmax))) return rc;
        PB_CUDA_OK(cudaEventRecord(e1, ctx->stream));
        PB_CUDA_OK(cudaEventSynchronize(e1));
        PB_CUDA_OK(cudaEventElapsedTime(ms, e0, e1));
        *ms *= 0.5f;
        return POLYBIN_OK;
    };
    float best_ms = 0.f;
    int rc = time_plan(*pl, &best_ms);
    Plan* best = pl;
    int tried = 1;
    std::vector<Plan*> others;
    auto sig = [](const Plan& c) {   // (tiles, groups, ncta, cells a CTA, units): equal signatures, equal launches
        int nt = 0;
        for (int i = 0; i < c.ngroups; ++i) nt += c.base.grp[i].ntiles;
        return std::make_tuple(nt, c.ngroups, c.ncta, c.cells_cta, c.total_units);
    };
    std::set<std::tuple<int, int, int, long, int>> seen;
    seen.insert(sig(*pl));
    const int costs[2] = {8, 24}, caps[2] = {kMaxTiles, 1};
    for (int ci = 0; ci < 2 && !rc; ++ci)
        for (int gi = 0; gi < 2 && !rc; ++gi)
            for (int mode = 0; mode < 3 && !rc; ++mode) {
                PlanOpts o;
                o.tile_cost = costs[ci];
                o.group_cap = caps[gi];
                o.cta_mode = mode;
                Plan* c = new Plan();
                if (build_plan(ctx, *c, pl->ncell, pl->ng, pl->nh, pl->hsep, pl->need, pl->n_out, pl->sing_g, o, true)) {
                    delete c;
                    continue;
                }
                if (!seen.insert(sig(*c)).second) { delete c; continue; }
                float ms = 0.f;
                rc = time_plan(*c, &ms);
                ++tried;
                others.push_back(c);
                if (!rc && ms < best_ms) { best_ms = ms; best = c; }
            }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    // keep the winner in the cache slot of the original plan
    for (auto& kv : pc->plans)
        if (kv.second == pl) kv.second = best;
    if (best != pl) delete pl;
    for (Plan* c : others)
        if (c != best) delete c;
    best->tuned = true;
    best->tuned_ms = best_ms;
    best->tuned_of = tried;
    *pl_io = best;
    return rc;
}

static int launch_tuned(polybin_ctx* ctx, Plan* pl, const float* g, const float* h, double* d_out, const uint32_t* gmax,
                        const uint32_t* hmax) {
    int rc;
    if ((rc = tune_plan(ctx, &pl, g, h, d_out, gmax, hmax))) return rc;
    return launch(ctx, *pl, g, h, d_out, gmax, hmax);
}

// Plan of all pairs (j <= k) of ng maps against the nh singles [0, nh), output M[(j, k)][i] pair-major.
static int full_plan(polybin_ctx* ctx, long ncell, int ng, int nh, int hsep, Plan** out) {
    PlanCache* pc = cache_of(ctx);
    auto key = std::make_tuple(ng, nh, hsep, 0, ncell);
    auto it = pc->plans.find(key);
    if (it != pc->plans.end()) { *out = it->second; return POLYBIN_OK; }
    std::vector<NeedPair> need;
    int p = 0;
    for (int j = 0; j < ng; ++j)
        for (int k = j; k < ng; ++k, ++p) {
            NeedPair np{j, k, 0, nh - 1, {}};
            for (int i = 0; i < nh; ++i) np.outs.push_back({i, p * nh + i});
            need.push_back(std::move(np));
        }
    Plan* pl = new Plan();
    int rc = build_plan(ctx, *pl, ncell, ng, nh, hsep, std::move(need), p * nh);
    if (rc) { delete pl; return rc; }
    pc->plans[key] = pl;
    *out = pl;
    return POLYBIN_OK;
}

// Plan of the closed triplets of the context on the contraction grid: triplet a <= b <= c from pair (b, c) and
// single a, output S' in triplet order.
static int triplet_plan(polybin_ctx* ctx, Plan** out) {
    PlanCache* pc = cache_of(ctx);
    const int nb = ctx->nb;
    auto key = std::make_tuple(nb, nb, 0, 1, ctx->cg.ncell);
    auto it = pc->plans.find(key);
    if (it != pc->plans.end()) { *out = it->second; return POLYBIN_OK; }
    std::map<std::pair<int, int>, NeedPair> m;
    const int nt = (int)ctx->Nabc.size();
    for (int t = 0; t < nt; ++t) {
        const int a = ctx->trip[3 * t], b = ctx->trip[3 * t + 1], c = ctx->trip[3 * t + 2];
        auto f = m.find({b, c});
        if (f == m.end()) f = m.emplace(std::make_pair(b, c), NeedPair{b, c, a, a, {}}).first;
        f->second.lo = std::min(f->second.lo, a);
        f->second.hi = std::max(f->second.hi, a);
        f->second.outs.push_back({a, t});
    }
    std::vector<NeedPair> need;
    for (auto& kv : m) need.push_back(std::move(kv.second));
    Plan* pl = new Plan();
    int rc = build_plan(ctx, *pl, ctx->cg.ncell, nb, nb, 0, std::move(need), nt);
    if (rc) { delete pl; return rc; }
    pc->plans[key] = pl;
    *out = pl;
    return POLYBIN_OK;
}

// Plan of the closed triplets for a multipole ell > 0 (Sec. 4.1, eq. ideal-bk: L_ell on the third bin): triplet
// a <= b <= c from the pair (g_b, g_{c,ell}) -- g_b a row of the g maps, g_{c,ell} a row of the h maps in the
// same slot -- and the single g_a, output S^ell' in triplet order.  Same pairs and windows as the ell = 0 plan.
static int ell_plan(polybin_ctx* ctx, Plan** out) {
    PlanCache* pc = cache_of(ctx);
    const int nb = ctx->nb;
    auto key = std::make_tuple(nb, nb, 1, 2, ctx->cg.ncell);
    auto it = pc->plans.find(key);
    if (it != pc->plans.end()) { *out = it->second; return POLYBIN_OK; }
    const int h0 = (nb + 7) / 8 * 8;
    std::map<std::pair<int, int>, NeedPair> m;
    const int nt = (int)ctx->Nabc.size();
    for (int t = 0; t < nt; ++t) {
        const int a = ctx->trip[3 * t], b = ctx->trip[3 * t + 1], c = ctx->trip[3 * t + 2];
        auto f = m.find({b, c});
        if (f == m.end()) f = m.emplace(std::make_pair(b, c), NeedPair{b, h0 + c, a, a, {}}).first;
        f->second.lo = std::min(f->second.lo, a);
        f->second.hi = std::max(f->second.hi, a);
        f->second.outs.push_back({a, t});
    }
    std::vector<NeedPair> need;
    for (auto& kv : m) need.push_back(std::move(kv.second));
    Plan* pl = new Plan();
    int rc = build_plan(ctx, *pl, ctx->cg.ncell, nb, nb, 1, std::move(need), nt, 1);
    if (rc) { delete pl; return rc; }
    pc->plans[key] = pl;
    *out = pl;
    return POLYBIN_OK;
}

}  // namespace tc

bool split_tc_available() { return true; }

// Runs k_tf32_selfcheck once per device (the first split-TF32 context on it); POLYBIN_ETOL if the tensor core does
// not read FP32 operands as the Gram matrix assumes.
int tf32_selfcheck(polybin_ctx* ctx) {
    static std::mutex mu;
    static int state[256] = {};   // 0 unchecked, 1 ok, -1 failed
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return fail_cuda(ctx, e, "cudaGetDevice", __FILE__, __LINE__);
    if (dev < 0 || dev >= 256) return POLYBIN_OK;
    std::lock_guard<std::mutex> lock(mu);
    if (state[dev] == 0) {
        uint32_t* d = nullptr;
        uint32_t h[3] = {0u, 0u, 1u};
        e = cudaMalloc(&d, sizeof(h));
        if (e == cudaSuccess) e = cudaMemsetAsync(d, 0, sizeof(h), ctx->stream);
        if (e == cudaSuccess) {
            tc::k_tf32_selfcheck<<<1, 128, 0, ctx->stream>>>(d);
            ctx->launches += 1;
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaMemcpyAsync(h, d, sizeof(h), cudaMemcpyDeviceToHost, ctx->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
        if (d) cudaFree(d);
        if (e != cudaSuccess) return fail_cuda(ctx, e, "tf32 self-check", __FILE__, __LINE__);
        float d00, d10;
        std::memcpy(&d00, &h[0], 4);
        std::memcpy(&d10, &h[1], 4);
        state[dev] = (h[2] == 0u && d00 == 1.0f && d10 == 1.0f + 0x1p-10f) ? 1 : -1;
        if (state[dev] < 0)
            return fail(ctx, POLYBIN_ETOL, "tf32 self-check: D00 = %.9g, D10 = %.9g (expected 1 and 1 + 2^-10): the tensor "
                        "core does not read FP32 operands as TF32 by truncation", (double)d00, (double)d10);
    }
    if (state[dev] < 0)
        return fail(ctx, POLYBIN_ETOL, "tf32 self-check failed on this device: split-TF32 mode unavailable");
    return POLYBIN_OK;
}

void destroy_tc(polybin_ctx* ctx) {
    delete static_cast<tc::PlanCache*>(ctx->tc);
    ctx->tc = nullptr;
}

int ensure_err_flag(polybin_ctx* ctx) {
    if (ctx->d_err) return POLYBIN_OK;
    cudaError_t e = cudaMalloc(&ctx->d_err, kErrFlags * sizeof(int));
    if (e != cudaSuccess) return fail_cuda(ctx, e, "cudaMalloc err flag", __FILE__, __LINE__);
    e = cudaMemset(ctx->d_err, 0, kErrFlags * sizeof(int));
    if (e != cudaSuccess) return fail_cuda(ctx, e, "cudaMemset err flag", __FILE__, __LINE__);
    return POLYBIN_OK;
}

// Reads the error flags after the work queued on the stream (synchronising it).
int read_err_flags(polybin_ctx* ctx, const char* what) {
    int herr[kErrFlags] = {};
    cudaError_t e = cudaMemcpyAsync(herr, ctx->d_err, sizeof(herr), cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    if (e != cudaSuccess) return fail_cuda(ctx, e, "error flags", __FILE__, __LINE__);
    if (herr[kErrPipeline]) return fail(ctx, POLYBIN_ETIMEOUT, "%s: a pipeline wait timed out", what);
    return POLYBIN_OK;
}

// Shapes the tensor-core kernel takes: <= 512 pairs, <= 32 singles, cells a multiple of 4, 16-byte aligned maps.
bool tc_shape_ok(long ncell, const float* g, int ng, const float* h, int nh) {
    if (ng < 1 || ng * (ng + 1) / 2 > 512 || nh < 1 || nh > 32) return false;
    if (ncell % 4 || ncell > 0x7fffffffL) return false;
    if (reinterpret_cast<uintptr_t>(g) % 16 || (h && reinterpret_cast<uintptr_t>(h) % 16)) return false;
    return true;
}

// M[(j <= k)][i] (pair-major, device) of ng maps g against nh singles h (h == nullptr: h = g), over ncell cells.
int run_contract_tc(polybin_ctx* ctx, const float* g, int ng, const float* h, int nh, double* d_out, long ncell,
                    const uint32_t* gmax, const uint32_t* hmax) {
    const int hsep = (h && h != g) ? 1 : 0;
    if (!hsep) nh = ng;
    tc::Plan* pl = nullptr;
    int rc = tc::full_plan(ctx, ncell, ng, nh, hsep, &pl);
    if (rc) return rc;
    return tc::launch_tuned(ctx, pl, g, hsep ? h : g, d_out, gmax, hmax);
}

int run_absmax(polybin_ctx* ctx, const float* maps, int nmaps, long ncell, uint32_t* absmax) {
    PB_CUDA_OK(cudaMemsetAsync(absmax, 0, sizeof(uint32_t) * kMaxItems, ctx->stream));
    const long n4 = ncell / 4;
    tc::k_absmax<<<dim3((unsigned)std::min((n4 + 1023) / 1024, 64L), nmaps, 1), 256, 0, ctx->stream>>>(
        reinterpret_cast<const float4*>(maps), n4, absmax);
    ctx->launches += 1;
    PB_CUDA_OK(cudaGetLastError());
    return POLYBIN_OK;
}

// Builds the closed-triplet plan ahead of time (before any stream capture).
int prepare_triplet_tc(polybin_ctx* ctx) {
    tc::Plan* pl = nullptr;
    return tc::triplet_plan(ctx, &pl);
}

// S^ell'_abc = sum g_a g_b g_{c,ell} of every closed triplet (device, triplet order) from the shell maps g and the
// Legendre-weighted maps gl on the contraction grid.
int run_triplet_sums_ell_tc(polybin_ctx* ctx, const float* g, const float* gl, double* d_S, const uint32_t* gmax,
                            const uint32_t* glmax) {
    tc::Plan* pl = nullptr;
    int rc = tc::ell_plan(ctx, &pl);
    if (rc) return rc;
    return tc::launch_tuned(ctx, pl, g, gl, d_S, gmax, glmax);
}

// out[i][j] += scale sum_k A[i][k] B[j][k] for float32 rows A [nA][K], B [nB][K] (K a multiple of 4, 16-byte aligned
// rows) on the tensor cores (3-term split TF32, FP64 sums across K splits in a fixed order).
int run_gram_tc(polybin_ctx* ctx, const float* A, int nA, const float* B, int nB, long K, double scale, double* d_out) {
    using namespace tc::gram;
    if (nA < 1 || nB < 1 || K < 1) return POLYBIN_OK;
    tc::PlanCache* pc = tc::cache_of(ctx);
    CUtensorMap mA, mB;
    int rc = tc::make_map2(ctx, &mA, A, K, nA, kKC, kBM);
    if (rc) return rc;
    if ((rc = tc::make_map2(ctx, &mB, B, K, nB, kKC, kBN))) return rc;
    const int nI = (nA + kBM - 1) / kBM, nJ = (nB + kBN - 1) / kBN;
    int dev = 0, nsm = 0;
    PB_CUDA_OK(cudaGetDevice(&dev));
    PB_CUDA_OK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    const long kst = (K + kKC - 1) / kKC;
    int nsplit = (int)std::max(1L, std::min(kst, (long)((2 * nsm + nI * nJ - 1) / (nI * nJ))));
    const long k_cta = (kst + nsplit - 1) / nsplit * kKC;
    nsplit = (int)((K + k_cta - 1) / k_cta);
    const long ldp = (long)nJ * kBN, split_stride = (long)nI * kBM * ldp;
    const size_t need = (size_t)nsplit * split_stride;
    if (need > pc->gram_cap) {
        if (pc->gram_part) cudaFree(pc->gram_part);
        pc->gram_part = nullptr;
        pc->gram_cap = 0;
        PB_CUDA_OK(cudaMalloc(&pc->gram_part, sizeof(double) * need));
        pc->gram_cap = need;
    }
    if ((rc = ensure_err_flag(ctx))) return rc;
    PB_CUDA_OK(cudaMemsetAsync(ctx->d_err, 0, sizeof(int), ctx->stream));
    PB_CUDA_OK(cudaFuncSetAttribute((const void*)k_gram_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem));
    {
        cudaFuncAttributes fa{};
        PB_CUDA_OK(cudaFuncGetAttributes(&fa, (const void*)k_gram_tc));
        if (fa.numRegs * kThreads > 65536)
            return fail(ctx, POLYBIN_ECUDA, "gram: kernel built with %d registers a thread", fa.numRegs);
    }
    GP P;
    P.k_cta = k_cta; P.K = K; P.nA = nA; P.nB = nB; P.nsplit = nsplit;
    P.part = pc->gram_part; P.ldp = ldp; P.split_stride = split_stride; P.err = ctx->d_err;
    k_gram_tc<<<dim3(nJ, nI, nsplit), kThreads, kSmem, ctx->stream>>>(mA, mB, P);
    ctx->launches += 1;
    PB_CUDA_OK(cudaGetLastError());
    const long nout = (long)nA * nB;
    k_gram_reduce<<<(unsigned)((nout + 255) / 256), 256, 0, ctx->stream>>>(pc->gram_part, nsplit, split_stride, ldp, nA, nB,
                                                                          scale, d_out);
    ctx->launches += 1;
    PB_CUDA_OK(cudaGetLastError());
    return read_err_flags(ctx, "gram");
}

// S'_abc of every closed triplet (device, triplet order) from the shell maps g on the contraction grid.
int run_triplet_sums_tc(polybin_ctx* ctx, const float* g, double* d_S, const uint32_t* gmax) {
    tc::Plan* pl = nullptr;
    int rc = tc::triplet_plan(ctx, &pl);
    if (rc) return rc;
    return tc::launch_tuned(ctx, pl, g, g, d_S, gmax, gmax);
}

}  // namespace pb

extern "C" int polybin_selftest_wait(polybin_ctx* ctx, int* timed_out) {
    if (!ctx || !timed_out) return pb::fail(ctx, POLYBIN_EINVAL, "polybin_selftest_wait: NULL argument");
    int rc = pb::ensure_err_flag(ctx);
    if (rc) return rc;
    PB_CUDA_OK(cudaMemsetAsync(ctx->d_err, 0, pb::kErrFlags * sizeof(int), ctx->stream));
    pb::tc::k_wait_selftest<<<1, 32, 0, ctx->stream>>>(ctx->d_err + pb::kErrPipeline, 1u << 14);
    ctx->launches++;
    PB_CUDA_OK(cudaGetLastError());
    int h[pb::kErrFlags] = {};
    PB_CUDA_OK(cudaMemcpyAsync(h, ctx->d_err, sizeof(h), cudaMemcpyDeviceToHost, ctx->stream));
    PB_CUDA_OK(cudaStreamSynchronize(ctx->stream));
    PB_CUDA_OK(cudaMemsetAsync(ctx->d_err, 0, pb::kErrFlags * sizeof(int), ctx->stream));
    *timed_out = h[pb::kErrPipeline] ? 1 : 0;
    return POLYBIN_OK;
}

// The closed-triplet plan of the context's tensor-core contraction (ell = 0) and what the autotuner chose.
extern "C" int polybin_contract_plan_info(polybin_ctx* ctx, int info[6], float* ms) {
    if (!ctx || !info) return pb::fail(ctx, POLYBIN_EINVAL, "polybin_contract_plan_info: NULL argument");
    for (int i = 0; i < 6; ++i) info[i] = -1;
    if (ms) *ms = 0.f;
    if (!ctx->tc) return POLYBIN_OK;
    pb::tc::PlanCache* pc = static_cast<pb::tc::PlanCache*>(ctx->tc);
    auto it = pc->plans.find(std::make_tuple(ctx->nb, ctx->nb, 0, 1, ctx->cg.ncell));
    if (it == pc->plans.end()) return POLYBIN_OK;
    const pb::tc::Plan& p = *it->second;
    info[0] = p.opts.tile_cost;
    info[1] = p.opts.group_cap;
    info[2] = p.opts.cta_mode;
    info[3] = p.ngroups;
    info[4] = p.ncta;
    info[5] = p.tuned ? p.tuned_of : 0;
    if (ms) *ms = p.tuned_ms;
    return POLYBIN_OK;
}
