// Surrogate network convolutions on the 5th-generation tensor cores
// (include/lbm_nn.h: lbm_nn_conv3x3, lbm_nn_conv3x3_wgrad).
//
// GEMM view of a periodic, dilated 3x3 convolution: M = pixels, N = cout,
// K = 9 taps x cin.  A tcgen05.mma (kind::f16: bfloat16 operands, FP32
// accumulation in tensor memory) multiplies 128 pixels of one image row by 16
// input channels.  Operands sit in shared memory in the 32-byte swizzled
// layout, one row (pixel, or weight row) of 16 channels per 32 bytes, so that
// the 128 pixels of a row shifted by a tap (dy, dx) are the same layout at
// another start address: a tap costs a descriptor, not a copy.  Activation
// rows arrive by TMA (cp.async.bulk.tensor) in that layout; the periodic halo
// columns by cp.async.
//
// Descriptor fields (measured on GB300 against host products): for swizzled K-major
// operands the stride-byte offset steps between 8-row groups; for swizzled MN-major
// operands the leading-byte offset steps between MN groups (of the swizzle's width)
// and the stride-byte offset between 8-row K groups.  The swizzle acts on absolute
// shared-memory address bits, so an operand may start at any pixel.  With M = 128 row
// m of the accumulator is TMEM lane m; with M = 64, rows 16q .. 16q + 15 are lanes
// 32q .. 32q + 15.
//
// Both kernels are persistent (one CTA per SM) and march down strips of image rows:
// 128 columns of the rows of one residue modulo the dilation d, so that each row of
// the input is loaded once per strip and used by the three output rows it touches.
// Warps have fixed roles (TMA issuer, halo loaders, MMA issuer, epilogue) and hand off
// through mbarriers; every wait is bounded: one that gives up sets bit 0 of *status and
// the CTA frees its tensor memory and returns.
#include "lbm.h"
#include "lbm_nn.h"
#include "nn_internal.h"

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

namespace {

constexpr int TC_COLS = 128;                    // pixels of one M tile (one image row)
constexpr long long TC_WAIT_LIMIT = 1LL << 24;  // polls of an mbarrier before giving up
constexpr size_t TC_MIN_SMEM = 120 * 1024;      // > half an SM: one CTA per SM (it owns all of TMEM it asks for)

// ------------------------------------------------------------------ PTX --
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Instruction descriptor of kind::f16: D FP32 (bits 4-5 = 1), A and B bfloat16
// (bits 7-9, 10-12 = 1), A / B MN-major (bits 15 / 16), N >> 3 (bits 17-22),
// M >> 4 (bits 24-28).
constexpr uint32_t idesc_bf16(int M, int N, int a_mn, int b_mn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity) {
    for (long long i = 0; i < TC_WAIT_LIMIT; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(ok)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

// Whole warp: allocate / free `cols` columns of tensor memory (power of 2 >= 32).
__device__ __forceinline__ void tmem_alloc(uint32_t slot, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(slot), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t taddr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(taddr), "r"(cols) : "memory");
}

// Whole warp: 16 consecutive 32-bit columns of this thread's lane.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

__host__ __device__ constexpr uint32_t pow2_cols(uint32_t n) {
    return n <= 32 ? 32 : (n <= 64 ? 64 : (n <= 128 ? 128 : (n <= 256 ? 256 : 512)));
}

// ------------------------------------------------------------ forward --
// Operand layout of the forward kernel: 32-byte swizzled, K-major.  A row
// (pixel, or weight row) is 16 channels = 32 bytes; groups of 8 rows are
// 256 bytes apart; the hardware exchanges the two 16-byte halves of rows 4..7
// of every 256-byte group by the absolute shared-memory address (byte-address
// bit 4 ^= bit 7; measured on GB300), so data written with that exchange can be
// read from any 32-byte-aligned start: the tap shift is still a start address.
// The tensor-memory-access unit (TMA) writes the same exchange (SWIZZLE_32B).
__device__ __forceinline__ uint32_t swz32(uint32_t a) { return a ^ (((a >> 7) & 1u) << 4); }

constexpr uint32_t LAYOUT_SW32 = 6;  // descriptor layout type, bits 61-63

// The same exchange for pixel slots of 32 or 128 bytes (128-byte swizzle: byte-address
// bits 4-6 ^= bits 7-9).
template <uint32_t PXB>
__device__ __forceinline__ uint32_t swz(uint32_t a) {
    return PXB == 128 ? a ^ (((a >> 7) & 7u) << 4) : swz32(a);
}
constexpr uint32_t LAYOUT_SW128 = 2;

// Shared-memory matrix descriptor in two words: the low one (start, leading-byte
// offset, in 16-byte units) moves with the operand, the high one (stride-byte offset,
// bit 46: the descriptor version of sm_100-class tensor cores, bits 61-63: the layout)
// stays.
__device__ __forceinline__ uint32_t sdesc_lo(uint32_t saddr, uint32_t lbo) {
    return ((saddr >> 4) & 0x3FFF) | (((lbo >> 4) & 0x3FFF) << 16);
}
__host__ __device__ constexpr uint32_t sdesc_hi(uint32_t sbo, uint32_t layout) {
    return ((sbo >> 4) & 0x3FFF) | (1u << 14) | (layout << 29);
}

// 1 on one lane of the (converged) warp.
__device__ __forceinline__ uint32_t elect_one() {
    uint32_t e;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(e));
    return e;
}
// D += A B on the lane with go != 0; descriptors as (low, high) words.
__device__ __forceinline__ void umma_if(uint32_t go, uint32_t d_tmem, uint32_t al, uint32_t ah, uint32_t bl, uint32_t bh,
                                        uint32_t idesc) {
    asm volatile(
        "{\n\t.reg .pred q, t;\n\t.reg .b64 a, b;\n\tsetp.ne.b32 q, %6, 0;\n\tsetp.eq.u32 t, 0, 0;\n\t"
        "mov.b64 a, {%1, %2};\n\tmov.b64 b, {%3, %4};\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, t;\n\t}\n" ::"r"(d_tmem),
        "r"(al), "r"(ah), "r"(bl), "r"(bh), "r"(idesc), "r"(go)
        : "memory");
}
__device__ __forceinline__ void commit_if(uint32_t go, uint32_t mbar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}\n" ::"r"(mbar),
        "r"(go)
        : "memory");
}

// Roles of the forward kernel (warp index): 0-11 epilogue (warp w reads TMEM lane
// quarter w % 4 of every third output row, w / 4), 12 the TMA issuer (lane 0), 13-16
// halo loaders (warp 13 + h the rows q = h mod 4), 17 the MMA issuer, which also owns
// the tensor memory.  Three groups of epilogue warps: with two, the mask epilogue's
// loads showed (58 us against 53).
constexpr int FW_GROUPS = 3, FW_EPI_WARPS = 4 * FW_GROUPS;
constexpr int FW_TMA_WARP = FW_EPI_WARPS, FW_HALO_WARP = FW_TMA_WARP + 1, FW_HALO_WARPS = 4;
constexpr int FW_MMA_WARP = FW_HALO_WARP + FW_HALO_WARPS, FW_THREADS = 32 * (FW_MMA_WARP + 1);
// Roles of the weight-gradient kernel: 0-3 epilogue, 4 TMA, 5-7 halo, 8-9 MMA.
constexpr int WG_TMA_WARP = 4, WG_HALO_WARP = 5, WG_HALO_WARPS = 3, WG_MMA_WARP = 8;
constexpr int WG_THREADS = 32 * 10;
// A row in shared memory: HALO halo slots, the 128 pixels of the strip, HALO halo slots
// (dilation <= HALO); the first pixel sits HALO slots into the row, on a 1024-byte (48
// channels) or 256-byte (16) boundary, where the swizzle's pattern starts.
constexpr int HALO = 8, PITCH = TC_COLS + 2 * HALO;

__device__ __forceinline__ void mbar_init_n(uint32_t mbar, uint32_t n) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(mbar), "r"(n) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}\n" ::"r"(mbar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_tx(uint32_t mbar, uint32_t bytes) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}\n" ::"r"(mbar),
                 "r"(bytes)
                 : "memory");
}

// One box of the activation tensor {channel, x, image row} -> shared memory,
// completing `bytes` on the mbarrier.
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int c, int xx, int row, uint32_t mbar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c), "r"(xx), "r"(row), "r"(mbar)
        : "memory");
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, int c, int xx, int row, int plane,
                                            uint32_t mbar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c), "r"(xx), "r"(row), "r"(plane), "r"(mbar)
        : "memory");
}

// Three 16-column loads of this thread's lane, one wait.
__device__ __forceinline__ void tmem_ld48(uint32_t taddr, float (&v)[48]) {
    uint32_t r[48];
#pragma unroll
    for (int q = 0; q < 3; ++q)
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
            : "=r"(r[16 * q + 0]), "=r"(r[16 * q + 1]), "=r"(r[16 * q + 2]), "=r"(r[16 * q + 3]), "=r"(r[16 * q + 4]),
              "=r"(r[16 * q + 5]), "=r"(r[16 * q + 6]), "=r"(r[16 * q + 7]), "=r"(r[16 * q + 8]),
              "=r"(r[16 * q + 9]), "=r"(r[16 * q + 10]), "=r"(r[16 * q + 11]), "=r"(r[16 * q + 12]),
              "=r"(r[16 * q + 13]), "=r"(r[16 * q + 14]), "=r"(r[16 * q + 15])
            : "r"(taddr + 16u * q));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int j = 0; j < 48; ++j) v[j] = __uint_as_float(r[j]);
}

// Whole warp: zero 16 consecutive 32-bit columns of this thread's lane.
__device__ __forceinline__ void tmem_zero16(uint32_t taddr) {
    const uint32_t z = 0;
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};\n" ::"r"(taddr),
        "r"(z)
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }

// The strips' rows in the order strip by strip; CTA b of G takes rows [T b / G, T (b + 1) / G)
// as runs of one strip each.
struct Run {
    long long left;  // rows of the CTA after this run
    int strip, r0, n;
};
__device__ __forceinline__ Run first_run(long long T, int rows) {
    const long long a = T * blockIdx.x / gridDim.x, b = T * (blockIdx.x + 1) / gridDim.x;
    Run R;
    R.strip = (int)(a / rows);
    R.r0 = (int)(a - (long long)R.strip * rows);
    R.n = (int)(b - a < rows - R.r0 ? b - a : rows - R.r0);
    R.left = b - a - R.n;
    return R;
}
__device__ __forceinline__ bool next_run(Run& R, int rows) {
    if (R.left <= 0) return false;
    ++R.strip;
    R.r0 = 0;
    R.n = (int)(R.left < rows ? R.left : rows);
    R.left -= R.n;
    return true;
}
// Strip: image n, residue rho, column block; image row (over all images) of its row r
// (periodic: r = -1 and r = rows wrap).
struct Strip {
    int n, rho, x0;
};
__device__ __forceinline__ Strip strip_of(int s, int d, int ncb) {
    Strip t;
    t.x0 = (s % ncb) * TC_COLS;
    s /= ncb;
    t.rho = s % d;
    t.n = s / d;
    return t;
}
__device__ __forceinline__ int strip_row(const Strip& t, int r, int rows, int d, int H) {
    return t.n * H + t.rho + (r < 0 ? r + rows : (r >= rows ? r - rows : r)) * d;
}
// A ring position: slot and the parity of its current round.
template <int S>
struct Ring {
    int s = 0;
    uint32_t round = 0;
    __device__ __forceinline__ void next() {
        if (++s == S) {
            s = 0;
            ++round;
        }
    }
};

// One output row (128 pixels x CO channels) is a slot of CO columns of a TMEM ring.
// Input row r of a strip meets the weights of its three row taps stacked along N (dy =
// +1, 0, -1), whose products go to output rows r - 1, r, r + 1 in adjacent slots: N =
// 3 CO, one MMA per 16 input channels and column tap (the shifted row is the same rows
// of shared memory from another start).  Every MMA accumulates: the epilogue zeroes a
// slot after reading it.
//
// Order of accumulation: an output takes its 16-channel groups one after another,
// within a group the input rows r - 1, r, r + 1, within a row the column taps (the
// order of a kernel that holds whole units of rows).  So group g of an input row is
// issued 2 g rows after its first group, when group g - 1 of the next row has been.
//
// What bounds it: the MMA warp, a serial chain.  48 -> 48 channels, 16 images of 256 x 256
// (clock64 in that warp; a CTA lasts 84,000 clocks and takes 54 rows): 14,400 clocks pass
// before its first MMA (the weights into shared memory, the slots zeroed), then each
// row takes 1,296: 190 waiting for a free output slot, 190 for an input row (384 and
// 271 with the mask epilogue) and 917 in the warp's own instructions, about half of them
// the issue of the nine MMAs, the rest the walk of the three staggered groups and the
// commits.  The tensor pipe is 42 % active, shared memory (l1tex) 44 % and DRAM 41 % of
// their peaks, so none of them bounds it.  A second issuer would have to share the
// accumulators, whose order of accumulation is kept.
// Units of 4 rows loaded with their 2 halo rows as 18 boxes of 4 KB took 54 us (76 at
// dilation 8, units of 2 rows) and 66 us (77) with the mask epilogue, bound by the TMA's time
// per box and pixel row; one box of 128-byte pixel slots per row, loaded once: 46 us at
// every dilation, 52 with the mask epilogue.
template <int CI, int CO>
struct Fw {
    static constexpr int KB = CI / 16;                         // 16-channel groups of the input
    static constexpr uint32_t XPB = CI == 48 ? 128 : 32;       // bytes of a pixel slot
    static constexpr uint32_t XROW = PITCH * XPB;
    static constexpr int S = CI == 48 ? 8 : 16;                // rows in the ring: 2 KB - 1 in use, the rest in flight
    static constexpr int NT = 10;                              // output slots: 2 KB + 1 open, the rest in the epilogue
    static constexpr uint32_t WBYTES = 9u * CI * CO * 2u;
    static constexpr uint32_t OUT = 32 * (CO == 48 ? 96 : 64); // a warp's 32 output pixels
    static constexpr uint32_t TCOLS = pow2_cols(NT * CO);
    static constexpr size_t smem() {
        return (size_t)S * XROW + FW_EPI_WARPS * OUT + WBYTES + CO * 4 + (2 * S + 2 * NT) * 8 + 16;
    }
};

template <int CI, int CO, int EPI>
__global__ void __launch_bounds__(FW_THREADS, 1)
    conv_tc_kernel(const __grid_constant__ CUtensorMap xmap, const uint8_t* __restrict__ x,
                   const __nv_bfloat16* __restrict__ w, const float* __restrict__ bias, uint8_t* __restrict__ y,
                   const float* res, const uint8_t* __restrict__ mask, int B, int H, int W, int d,
                   int* __restrict__ status) {
    using K = Fw<CI, CO>;
    constexpr int KB = K::KB, S = K::S, NT = K::NT;
    constexpr int NC = CI / 8;  // 16-byte chunks per input pixel
    static_assert(S % FW_HALO_WARPS == 0, "slots owned by one halo warp (a parity wait cannot tell two rounds apart)");
    static_assert(S > 2 * KB && NT > 2 * KB + 1, "rows and outputs open at a time");
    extern __shared__ __align__(1024) uint8_t smem[];
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    // [rows][output staging][weights][bias][barriers][tmem slot]
    const uint32_t sx0 = smem_u32(smem), sstg = sx0 + S * K::XROW, sw0 = sstg + FW_EPI_WARPS * K::OUT;
    float* s_bias = reinterpret_cast<float*>(smem + S * K::XROW + FW_EPI_WARPS * K::OUT + K::WBYTES);
    uint64_t* s_bar = reinterpret_cast<uint64_t*>(s_bias + CO);
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(s_bar + 2 * S + 2 * NT);
    const uint32_t bar0 = smem_u32(s_bar);
    auto full = [&](int s) { return bar0 + 8u * s; };
    auto empty = [&](int s) { return bar0 + 8u * (S + s); };
    auto tfull = [&](int s) { return bar0 + 8u * (2 * S + s); };
    auto tempty = [&](int s) { return bar0 + 8u * (2 * S + NT + s); };
    if (tid == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init_n(full(s), 1 + 32);  // the TMA issuer's expect_tx and the lanes of a halo warp
            mbar_init_n(empty(s), 1);
        }
        for (int s = 0; s < NT; ++s) {
            mbar_init_n(tfull(s), 1);
            mbar_init_n(tempty(s), 128);  // the four warps of an epilogue group
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == FW_MMA_WARP) tmem_alloc(smem_u32(s_tmem), K::TCOLS);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *s_tmem, 0);

    const int rows = H / d, ncb = W / TC_COLS;
    const long long T = (long long)B * d * ncb * rows;
    bool ok = true;

    if (warp < FW_EPI_WARPS || warp == FW_MMA_WARP) {
        // beside the first loads: weights [co][t][ci] -> blocks (dx, 16-channel group) of 3 CO rows
        // x 32 bytes, swizzled (row bi CO + o of a block holds tap dy = 1 - bi), the bias, and
        // zeroed output slots
        constexpr int NTH = 32 * (FW_EPI_WARPS + 1);
        const int t0 = warp == FW_MMA_WARP ? 32 * FW_EPI_WARPS + lane : tid;
        for (int i = t0; i < 9 * NC * CO; i += NTH) {
            const int o = i % CO, rest = i / CO, j = rest % NC, tap = rest / NC;  // tap = 3 bi + dxi
            const int bi = tap / 3, dxi = tap % 3, t = 3 * (2 - bi) + dxi;
            const uint4 v = *reinterpret_cast<const uint4*>(w + ((size_t)o * 9 + t) * CI + 8 * j);
            const uint32_t a = sw0 + (uint32_t)(((dxi * KB + (j >> 1)) * 3 + bi) * CO + o) * 32u + (uint32_t)(j & 1) * 16u;
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(swz32(a)), "r"(v.x), "r"(v.y), "r"(v.z),
                         "r"(v.w)
                         : "memory");
        }
        for (int i = t0; i < CO; i += NTH) s_bias[i] = (EPI != LBM_NN_MASK && bias) ? bias[i] : 0.0f;
        if (warp < FW_EPI_WARPS) {
            for (int k = warp >> 2; k < NT; k += FW_GROUPS)
#pragma unroll
                for (int c0 = 0; c0 < CO; c0 += 16)
                    tmem_zero16(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(k * CO + c0));
            tmem_wait_st();
        }
        fence_proxy_async();  // the weights (generic stores) before the tensor cores read them
        fence_before_sync();
        asm volatile("bar.sync 1, %0;\n" ::"n"(NTH) : "memory");
        fence_after_sync();
    }

    if (warp == FW_TMA_WARP) {
        if (lane == 0) {
            Ring<S> q;
            Run R = first_run(T, rows);
            do {
                const Strip t = strip_of(R.strip, d, ncb);
                for (int i = 0; i < R.n + 2; ++i, q.next()) {
                    if (q.round) ok = mbar_wait(empty(q.s), (q.round - 1) & 1);
                    if (!ok) break;
                    mbar_arrive_tx(full(q.s), TC_COLS * K::XPB);
                    tma_load_3d(sx0 + (uint32_t)q.s * K::XROW + HALO * K::XPB, &xmap, 0, t.x0,
                                strip_row(t, R.r0 - 1 + i, rows, d, H), full(q.s));
                }
            } while (ok && next_run(R, rows));
        }
        __syncwarp();
    } else if (warp >= FW_HALO_WARP && warp < FW_HALO_WARP + FW_HALO_WARPS) {
        // d columns on each side of every row, wrapped, 16 bytes per copy
        Ring<S> q;
        Run R = first_run(T, rows);
        do {
            const Strip t = strip_of(R.strip, d, ncb);
            for (int i = 0; i < R.n + 2; ++i, q.next()) {
                if (q.s % FW_HALO_WARPS != warp - FW_HALO_WARP) continue;
                if (q.round) ok = mbar_wait(empty(q.s), (q.round - 1) & 1);
                if (!ok) break;
                const long long row = strip_row(t, R.r0 - 1 + i, rows, d, H);
                for (int k = lane; k < 2 * d * NC; k += 32) {
                    const int jc = k % NC, e = k / NC;
                    int xx = e < d ? t.x0 - 1 - e : t.x0 + TC_COLS + (e - d);
                    const int slot = e < d ? HALO - 1 - e : HALO + TC_COLS + (e - d);
                    xx += xx < 0 ? W : (xx >= W ? -W : 0);
                    cp_async16(swz<K::XPB>(sx0 + (uint32_t)q.s * K::XROW + (uint32_t)slot * K::XPB + 16u * jc),
                               x + (row * W + xx) * (16LL * NC) + 16 * jc);
                }
                cp_async_commit();
                cp_async_wait_all();
                fence_proxy_async();
                mbar_arrive(full(q.s));
            }
        } while (ok && next_run(R, rows));
    } else if (warp == FW_MMA_WARP) {
        // The whole warp runs the loop with warp-uniform values (slots, descriptors), one
        // elected lane issues.
        const uint32_t leader = elect_one();
        const uint32_t xhi = sdesc_hi(K::XPB == 128 ? 1024 : 256, K::XPB == 128 ? LAYOUT_SW128 : LAYOUT_SW32);
        const uint32_t whi = sdesc_hi(256, LAYOUT_SW32);
        const uint32_t xl = sdesc_lo(sx0 + (uint32_t)(HALO - d) * K::XPB, 16), wl = sdesc_lo(sw0, 16);
        // where group kb of the input rows stands: run, row i of its n + 2, ring slot, and
        // the output slot of its first output row (row i - 2 of the run, or row 0)
        struct Walk {
            Run R;
            Ring<S> q;
            int i = 0, lo = 0;
            bool live = true;
        } at[KB];
#pragma unroll
        for (int kb = 0; kb < KB; ++kb) at[kb].R = first_run(T, rows);
        Ring<NT> fresh;  // the next output slot to open
        for (int step = 0; ok && at[KB - 1].live; ++step) {
#pragma unroll
            for (int kb = 0; kb < KB; ++kb) {
                Walk& a = at[kb];
                if (!ok || step < 2 * kb || !a.live) continue;
                if (kb == 0) {
                    if (a.i < a.R.n) {
                        if (fresh.round) ok = mbar_wait(tempty(fresh.s), (fresh.round - 1) & 1);
                        fresh.next();
                    }
                    ok = ok && mbar_wait(full(a.q.s), a.q.round & 1);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) continue;
                    fence_after_sync();
                }
                // output rows first .. first + c - 1 of the run from slot lo on, the first at
                // weight block bi (dy = 1 - bi)
                const int first = a.i < 2 ? 0 : a.i - 2, c = (a.i < a.R.n ? a.i : a.R.n - 1) - first + 1;
                const int bi = first - (a.i - 2), c1 = a.lo + c > NT ? NT - a.lo : c;
                const uint32_t row = xl + (uint32_t)a.q.s * (K::XROW / 16) + 2u * kb;
                auto taps = [&](int slot, int n, int b) {
                    const uint32_t idesc = idesc_bf16(128, 0, 0, 0) | ((uint32_t)(n * CO >> 3) << 17);
#pragma unroll
                    for (int dxi = 0; dxi < 3; ++dxi)
                        umma_if(leader, tmem + (uint32_t)(slot * CO), row + (uint32_t)(dxi * d) * (K::XPB / 16), xhi,
                                wl + (uint32_t)(((dxi * KB + kb) * 3 + b) * CO) * 2u, whi, idesc);
                };
                taps(a.lo, c1, bi);
                if (c1 < c) taps(0, c - c1, bi + c1);
                if (kb == KB - 1) {
                    commit_if(leader, empty(a.q.s));
                    if (a.i >= 2) commit_if(leader, tfull(a.lo));
                }
                a.q.next();
                if (a.i >= 2) a.lo = a.lo + 1 == NT ? 0 : a.lo + 1;
                if (++a.i == a.R.n + 2) {
                    a.i = 0;
                    a.live = next_run(a.R, rows);
                }
            }
        }
        __syncwarp();
    } else {
        // ---- epilogue: TMEM lane quarter, pixel x0 + 32 quarter + lane, the group's output rows
        // (a group meets a slot's rounds out of turn, but a row completes after all rows before
        // it, so a slot is never two rounds behind the one that a group waits for)
        const int quarter = warp & 3, group = warp >> 2;
        const uint32_t stg = sstg + (uint32_t)warp * K::OUT;  // this warp's output staging
        const uint32_t tq = tmem + ((uint32_t)(32 * quarter) << 16);
        Ring<NT> o;
        int turn = 0;
        Run R = first_run(T, rows);
        do {
            const Strip t = strip_of(R.strip, d, ncb);
            for (int j = 0; j < R.n; ++j, o.next(), turn = turn + 1 == FW_GROUPS ? 0 : turn + 1) {
                if (turn != group) continue;
                const long long px0 = (long long)strip_row(t, R.r0 + j, rows, d, H) * W + t.x0 + 32 * quarter;
                // the operands of the epilogue, requested before the wait
                uint4 mk[EPI == LBM_NN_MASK ? 6 : 1];
                float4 rs[EPI == LBM_NN_RESIDUAL ? 4 : 1];
                if constexpr (EPI == LBM_NN_MASK) {
#pragma unroll
                    for (int k = 0; k < 6; ++k) mk[k] = __ldg(reinterpret_cast<const uint4*>(mask + (px0 + lane) * 96) + k);
                }
                if constexpr (EPI == LBM_NN_RESIDUAL) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) rs[k] = reinterpret_cast<const float4*>(res + (px0 + lane) * 16)[k];
                }
                ok = mbar_wait(tfull(o.s), o.round & 1);
                if (!ok) break;
                fence_after_sync();
                const uint32_t tb = tq + (uint32_t)(o.s * CO);
                float v[CO];
                if constexpr (CO == 48) tmem_ld48(tb, v);
                else tmem_ld16(tb, v);
#pragma unroll
                for (int c0 = 0; c0 < CO; c0 += 16) tmem_zero16(tb + (uint32_t)c0);
                tmem_wait_st();
                fence_before_sync();
                mbar_arrive(tempty(o.s));
                uint4 out[K::OUT / 512];
                if constexpr (CO == 48) {
                    static_assert(EPI == LBM_NN_RELU || EPI == LBM_NN_MASK, "48-channel epilogues: ReLU or mask");
#pragma unroll
                    for (int q4 = 0; q4 < 6; ++q4) {
                        uint32_t u[4];
                        const uint32_t m[4] = {mk[EPI == LBM_NN_MASK ? q4 : 0].x, mk[EPI == LBM_NN_MASK ? q4 : 0].y,
                                               mk[EPI == LBM_NN_MASK ? q4 : 0].z, mk[EPI == LBM_NN_MASK ? q4 : 0].w};
                        float bq[8] = {};
                        if constexpr (EPI == LBM_NN_RELU) {
                            const float4 b0 = *reinterpret_cast<const float4*>(s_bias + 8 * q4);
                            const float4 b1 = *reinterpret_cast<const float4*>(s_bias + 8 * q4 + 4);
                            bq[0] = b0.x; bq[1] = b0.y; bq[2] = b0.z; bq[3] = b0.w;
                            bq[4] = b1.x; bq[5] = b1.y; bq[6] = b1.z; bq[7] = b1.w;
                        }
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int q = 4 * q4 + e;
                            if constexpr (EPI == LBM_NN_RELU)
                                u[e] = pack_bf16x2(fmaxf(v[2 * q] + bq[2 * e], 0.0f), fmaxf(v[2 * q + 1] + bq[2 * e + 1], 0.0f));
                            else
                                u[e] = pack_bf16x2(bf16_lo(m[e]) > 0.0f ? v[2 * q] : 0.0f,
                                                   bf16_hi(m[e]) > 0.0f ? v[2 * q + 1] : 0.0f);
                        }
                        out[q4] = make_uint4(u[0], u[1], u[2], u[3]);
                    }
                } else {
                    static_assert(EPI == LBM_NN_RESIDUAL && CO == 16, "16-channel epilogue: residual");
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float4 a = rs[EPI == LBM_NN_RESIDUAL ? k : 0];
                        out[k] = make_uint4(__float_as_uint(a.x + v[4 * k] + s_bias[4 * k]),
                                            __float_as_uint(a.y + v[4 * k + 1] + s_bias[4 * k + 1]),
                                            __float_as_uint(a.z + v[4 * k + 2] + s_bias[4 * k + 2]),
                                            __float_as_uint(a.w + v[4 * k + 3] + s_bias[4 * k + 3]));
                    }
                }
                // the warp's 32 pixels are one contiguous run of y: staged, then one bulk store
                // (after the previous one has read the staging)
                if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");
                __syncwarp();
#pragma unroll
                for (int k = 0; k < (int)(K::OUT / 512); ++k)
                    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(stg + (uint32_t)lane * (K::OUT / 32) + 16u * k),
                                 "r"(out[k].x), "r"(out[k].y), "r"(out[k].z), "r"(out[k].w)
                                 : "memory");
                fence_proxy_async();  // the staging (generic stores) before the bulk copy reads it
                __syncwarp();
                if (lane == 0) {
                    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(
                                     __cvta_generic_to_global(y + px0 * (K::OUT / 32))),
                                 "r"(stg), "r"(K::OUT)
                                 : "memory");
                    asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
                }
            }
        } while (ok && next_run(R, rows));
        // every store of this warp complete before the CTA (and its staging) goes away
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory");
    }
    if (!ok) atomicOr(status, 1);
    cp_async_wait_all();
    fence_before_sync();
    __syncthreads();
    if (warp == FW_MMA_WARP) {
        fence_after_sync();
        tmem_free(tmem, K::TCOLS);
    }
}

// Tensor maps of an NHWC bfloat16 activation.
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// {channel, x, image row}, one box per image row of 128 pixels: 48 channels as 128-byte pixel
// slots (box of 64 channels, the 16 beyond the tensor read as zeros; 128-byte
// swizzle), 16 channels as 32-byte ones.
bool row_map(CUtensorMap* map, const void* x, int C, int B, int H, int W) {
    const EncodeTiledFn fn = encode_tiled();
    if (!fn) return false;
    const bool wide = C == 48;
    const cuuint64_t dims[3] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)B * H};
    const cuuint64_t strides[2] = {(cuuint64_t)C * 2, (cuuint64_t)W * C * 2};
    const cuuint32_t box[3] = {wide ? 64u : 16u, (cuuint32_t)TC_COLS, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(x), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, wide ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_32B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// ... and one box per image row of 128 pixels as 16-channel planes (32-byte swizzle):
// {channel of the plane, x, image row, plane}.
bool plane_map(CUtensorMap* map, const void* x, int C, int B, int H, int W) {
    const EncodeTiledFn fn = encode_tiled();
    if (!fn) return false;
    const cuuint64_t dims[4] = {16, (cuuint64_t)W, (cuuint64_t)B * H, (cuuint64_t)C / 16};
    const cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)W * C * 2, 32};
    const cuuint32_t box[4] = {16, (cuuint32_t)TC_COLS, 1, (cuuint32_t)C / 16};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(x), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int CI, int CO, int EPI>
int conv_tc_launch(const void* x, const void* w, const float* bias, void* y, const float* res, const void* mask, int B,
                   int H, int W, int d, int* status, cudaStream_t s) {
    auto k = conv_tc_kernel<CI, CO, EPI>;
    static_assert(Fw<CI, CO>::smem() <= 227 * 1024, "shared memory");
    const size_t smem = std::max(Fw<CI, CO>::smem(), TC_MIN_SMEM);
    CUtensorMap map;
    if (!row_map(&map, x, CI, B, H, W)) return LBM_ERR_CUDA;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return LBM_ERR_CUDA;
    const int grid = (int)std::min<long long>((long long)B * H * (W / TC_COLS), (long long)nn_sm_count());
    k<<<grid, FW_THREADS, smem, s>>>(map, static_cast<const uint8_t*>(x), static_cast<const __nv_bfloat16*>(w), bias,
                                     static_cast<uint8_t*>(y), res, static_cast<const uint8_t*>(mask), B, H, W, d, status);
    return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}

// ------------------------------------------------------ weight gradient --
// dw[o][t][c] = sum_p dy[p][o] x[p + d off_t][c]: per tap a GEMM with K = pixels,
// 16 per MMA, both operands read MN-major (channels contiguous) from the rows as the
// TMA writes them.  A CTA marches down strips of image rows (columns 128 cb .., rows
// of one residue modulo d): each row of x and of dy is loaded once, and row k of x
// meets rows k - 1, k, k + 1 of dy while they are in the ring.
//
// What bounds it: the tensor cores' operand reads from shared memory and the rate of
// MMAs, so one MMA carries as many taps as the layouts allow:
// * N: the three dy rows stacked, 3 CO columns.  dy is stored as 16-channel planes
//   of 128 pixels (32-byte swizzle), the planes of a row and the rows of the ring
//   one after another, so that the 16-column groups of N are a constant 4 KB apart.
// * M: the column taps.  The groups of M step by the dilation, LBO = d pixels: with
//   48 input channels (64-channel rows of 128 bytes, 128-byte swizzle, the last 16
//   channels filled with zeros by the TMA) M = 128 covers dx = -1, 0 and M = 64 dx =
//   +1; with 16 (32-byte rows) M = 64 covers dx = -1, 0, 1 and an unused shift.
// One box per row of x and dy: the TMA's time goes per box and per pixel row of a
// box, and 4 KB boxes of 32-byte rows had been the floor (157 ns each).
// Measured, 48 -> 48 channels, 16 images of 256 x 256: 155 us with one M = 64, N = 48
// MMA per tap on units of two rows loaded with their halo rows; 48 us so (16 -> 48: 152
// and 33, 48 -> 16: 151 and 38).
// The accumulators (3 CO columns per M block) stay in tensor memory for the whole
// kernel; a CTA writes one partial per tap and a second kernel adds them in a fixed
// order: deterministic.

template <int CI, int CO>
struct Wg {
    static constexpr uint32_t XPB = CI == 48 ? 128 : 32;       // bytes of a pixel slot of x
    static constexpr uint32_t XROW = PITCH * XPB;           // a row of x with its halo slots
    static constexpr uint32_t DROW = (CO / 16) * TC_COLS * 32; // a row of dy: planes of 128 pixels
    // slots: the x rings a multiple of the halo warps, so that each owns its slots (a
    // parity wait cannot tell two rounds apart)
    static constexpr int SX = CI == 48 ? 6 : 9, SD = 9;
    // MMA issuers: one per M block, on accumulators of its own (a thread issues an MMA
    // only about every 100 cycles; two warps overlap: 52 -> 48 us)
    static constexpr int NI = CI == 48 ? 2 : 1;
    static constexpr uint32_t N3 = 3 * CO;
    static constexpr uint32_t TCOLS = pow2_cols(CI == 48 ? 2 * N3 : N3);
    static constexpr size_t smem() { return (size_t)SX * XROW + SD * DROW + (2 * SX + 2 * SD + 1) * 8 + 16; }
};

template <int CI, int CO>
__global__ void __launch_bounds__(WG_THREADS, 1)
    wgrad_tc_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap dmap,
                    const uint8_t* __restrict__ x, float* __restrict__ partials, float* __restrict__ bpart, int B, int H,
                    int W, int d, int* __restrict__ status) {
    using K = Wg<CI, CO>;
    constexpr int SX = K::SX, SD = K::SD;
    constexpr int NCX = CI / 8;  // 16-byte chunks of an x pixel
    static_assert(SX % WG_HALO_WARPS == 0, "x slots owned by one halo warp");
    static_assert(SD >= 4, "three rows of dy and one to load");
    extern __shared__ __align__(1024) uint8_t smem[];
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const uint32_t sx0 = smem_u32(smem), sd0 = sx0 + SX * K::XROW;
    uint64_t* s_bar = reinterpret_cast<uint64_t*>(smem + SX * K::XROW + SD * K::DROW);
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(s_bar + 2 * SX + 2 * SD + 1);
    const uint32_t bar0 = smem_u32(s_bar);
    auto xfull = [&](int s) { return bar0 + 8u * s; };
    auto xempty = [&](int s) { return bar0 + 8u * (SX + s); };
    auto dfull = [&](int s) { return bar0 + 8u * (2 * SX + s); };
    auto dempty = [&](int s) { return bar0 + 8u * (2 * SX + SD + s); };
    const uint32_t done = bar0 + 8u * (2 * SX + 2 * SD);
    if (tid == 0) {
        for (int s = 0; s < SX; ++s) {
            mbar_init_n(xfull(s), 1 + 32);  // the TMA issuer's expect_tx and the lanes of a halo warp
            mbar_init_n(xempty(s), K::NI);
        }
        for (int s = 0; s < SD; ++s) {
            mbar_init_n(dfull(s), 1);
            mbar_init_n(dempty(s), K::NI + (bpart ? 4 : 0));  // the issuers, and the warps that sum the bias gradient
        }
        mbar_init_n(done, K::NI);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == WG_MMA_WARP) tmem_alloc(smem_u32(s_tmem), K::TCOLS);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *s_tmem, 0);
    // every MMA accumulates: zero the accumulators
    if (warp < 4) {
        constexpr uint32_t USED = CI == 48 ? 2 * K::N3 : K::N3;
        for (uint32_t c = 0; c < USED; c += 16) tmem_zero16(tmem + ((uint32_t)(32 * warp) << 16) + c);
        tmem_wait_st();
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();

    const int rows = H / d, ncb = W / TC_COLS;
    const long long T = (long long)B * d * ncb * rows;
    bool ok = true;

    if (warp == WG_TMA_WARP) {
        // per run: dy rows r0 .. r0 + n - 1 and x rows r0 - 1 .. r0 + n, in the order the MMAs need them
        if (lane == 0) {
            Ring<SX> qx;
            Ring<SD> qd;
            Run R = first_run(T, rows);
            do {
                const Strip t = strip_of(R.strip, d, ncb);
                for (int i = 0; i < R.n + 2 && ok; ++i) {
                    if (i < R.n) {
                        if (qd.round) ok = mbar_wait(dempty(qd.s), (qd.round - 1) & 1);
                        if (!ok) break;
                        mbar_arrive_tx(dfull(qd.s), K::DROW);
                        tma_load_4d(sd0 + (uint32_t)qd.s * K::DROW, &dmap, 0, t.x0, strip_row(t, R.r0 + i, rows, d, H), 0,
                                    dfull(qd.s));
                        qd.next();
                    }
                    if (qx.round) ok = mbar_wait(xempty(qx.s), (qx.round - 1) & 1);
                    if (!ok) break;
                    mbar_arrive_tx(xfull(qx.s), TC_COLS * K::XPB);
                    tma_load_3d(sx0 + (uint32_t)qx.s * K::XROW + HALO * K::XPB, &xmap, 0, t.x0,
                                strip_row(t, R.r0 - 1 + i, rows, d, H), xfull(qx.s));
                    qx.next();
                }
            } while (ok && next_run(R, rows));
        }
        __syncwarp();
    } else if (warp >= WG_HALO_WARP && warp < WG_HALO_WARP + WG_HALO_WARPS) {
        // d columns on each side of every x row, wrapped, 16 bytes per copy
        Ring<SX> qx;
        int turn = 0;
        Run R = first_run(T, rows);
        do {
            const Strip t = strip_of(R.strip, d, ncb);
            for (int i = 0; i < R.n + 2 && ok; ++i, qx.next(), turn = turn == WG_HALO_WARPS - 1 ? 0 : turn + 1) {
                if (turn != warp - WG_HALO_WARP) continue;
                if (qx.round) ok = mbar_wait(xempty(qx.s), (qx.round - 1) & 1);
                if (!ok) break;
                const long long row = strip_row(t, R.r0 - 1 + i, rows, d, H);
                for (int k = lane; k < 2 * d * NCX; k += 32) {
                    const int jc = k % NCX, e = k / NCX;
                    int xx = e < d ? t.x0 - 1 - e : t.x0 + TC_COLS + (e - d);
                    const int slot = e < d ? HALO - 1 - e : HALO + TC_COLS + (e - d);
                    xx += xx < 0 ? W : (xx >= W ? -W : 0);
                    cp_async16(swz<K::XPB>(sx0 + (uint32_t)qx.s * K::XROW + (uint32_t)slot * K::XPB + 16u * jc),
                               x + (row * W + xx) * (16LL * NCX) + 16 * jc);
                }
                cp_async_commit();
                cp_async_wait_all();
                fence_proxy_async();
                mbar_arrive(xfull(qx.s));
            }
        } while (ok && next_run(R, rows));
    } else if (warp >= WG_MMA_WARP && warp < WG_MMA_WARP + K::NI) {
        // CI = 48: the first issuer dx = -1, 0 (M = 128), the second dx = +1 (M = 64);
        // CI = 16: one issuer, all dx (M = 64).  The whole warp runs the loop with
        // warp-uniform values (slots, descriptors), one elected lane issues.
        const int part = warp - WG_MMA_WARP;
        const uint32_t leader = elect_one();
        Ring<SX> qx;
        Ring<SD> qd;
        const uint32_t xhi = sdesc_hi(K::XPB == 128 ? 1024 : 256, K::XPB == 128 ? LAYOUT_SW128 : LAYOUT_SW32);
        const uint32_t dhi = sdesc_hi(256, LAYOUT_SW32);
        const uint32_t xl = sdesc_lo(sx0 + (uint32_t)(HALO + (part == 0 ? -d : d)) * K::XPB, (uint32_t)d * K::XPB);
        const uint32_t dl = sdesc_lo(sd0, TC_COLS * 32), block = tmem + (uint32_t)part * K::N3;
        const uint32_t shape = idesc_bf16(CI == 48 && part == 0 ? 128 : 64, 0, 1, 1);
        // n3 dy rows from slot s on, at stack position k
        auto stack = [&](int sx, int s, int n3, int k) {
            const uint32_t idesc = shape | ((uint32_t)(n3 * CO >> 3) << 17);
            uint32_t a = xl + (uint32_t)sx * (K::XROW / 16), b = dl + (uint32_t)s * (K::DROW / 16);
#pragma unroll
            for (int p0 = 0; p0 < TC_COLS; p0 += 16) {
                umma_if(leader, block + (uint32_t)(k * CO), a, xhi, b, dhi, idesc);
                a += K::XPB;  // 16 pixels, in 16-byte units
                b += 32;
            }
        };
        Run R = first_run(T, rows);
        do {
            int lo = qd.s;  // slot of the first dy row that the current x row meets
            for (int i = 0; i < R.n + 2 && ok; ++i) {
                if (i < R.n) {
                    ok = mbar_wait(dfull(qd.s), qd.round & 1);
                    qd.next();
                }
                ok = ok && mbar_wait(xfull(qx.s), qx.round & 1);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                fence_after_sync();
                // dy rows max(i - 2, 0) .. min(i, n - 1) of the run; stack position 0: row i - 2
                const int first = i < 2 ? 0 : i - 2, n3 = (i < R.n ? i : R.n - 1) - first + 1, k = first - (i - 2);
                const int n1 = lo + n3 > SD ? SD - lo : n3;
                stack(qx.s, lo, n1, k);
                if (n1 < n3) stack(qx.s, 0, n3 - n1, k + n1);
                commit_if(leader, xempty(qx.s));
                qx.next();
                if (i >= 2) {
                    commit_if(leader, dempty(lo));
                    lo = lo + 1 == SD ? 0 : lo + 1;
                }
            }
        } while (ok && next_run(R, rows));
        commit_if(leader, done);
        __syncwarp();
    } else if (warp < 4) {
        // ---- the bias gradient, while the issuers run: thread tid sums the channels of its pixel
        // of every dy row from the ring
        float a[CO] = {};
        if (bpart) {
            Ring<SD> qd;
            Run R = first_run(T, rows);
            do {
                for (int i = 0; i < R.n; ++i, qd.next()) {
                    ok = mbar_wait(dfull(qd.s), qd.round & 1);
                    if (!ok) break;
                    const uint32_t px = sd0 + (uint32_t)qd.s * K::DROW + 32u * tid;
#pragma unroll
                    for (int c = 0; c < CO / 8; ++c) {
                        uint32_t v[4];
                        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];\n"
                                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                                     : "r"(swz32(px + (uint32_t)(c >> 1) * (TC_COLS * 32) + 16u * (c & 1)))
                                     : "memory");
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            a[8 * c + 2 * e] += bf16_lo(v[e]);
                            a[8 * c + 2 * e + 1] += bf16_hi(v[e]);
                        }
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(dempty(qd.s));
                }
            } while (ok && next_run(R, rows));
#pragma unroll
            for (int c = 0; c < CO; ++c) {
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) a[c] += __shfl_down_sync(0xffffffffu, a[c], off);
            }
        }
        // ---- epilogue: stack position k of the columns is tap row dy = 1 - k
        ok = mbar_wait(done, 0) && ok;
        fence_after_sync();
        if (bpart) {
            // the warps' sums meet where the rows were (all of them have been used)
            float* s_sum = reinterpret_cast<float*>(smem);
            if (lane == 0)
#pragma unroll
                for (int c = 0; c < CO; ++c) s_sum[warp * CO + c] = a[c];
            asm volatile("bar.sync 1, 128;\n" ::: "memory");
            if (tid < CO)
                bpart[(size_t)blockIdx.x * CO + tid] =
                    (s_sum[tid] + s_sum[CO + tid]) + (s_sum[2 * CO + tid] + s_sum[3 * CO + tid]);
        }
        float* out = partials + (size_t)blockIdx.x * 9 * CI * CO;
        const uint32_t tq = tmem + ((uint32_t)(32 * warp) << 16);
        auto write = [&](uint32_t block, int dxi, int ci, bool mine) {
#pragma unroll 1
            for (int k = 0; k < 3; ++k) {
                const int t = (2 - k) * 3 + dxi;
#pragma unroll
                for (int c0 = 0; c0 < CO; c0 += 16) {
                    float v[16];
                    tmem_ld16(tq + block + (uint32_t)(k * CO + c0), v);
                    if (mine) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) out[((size_t)t * CO + c0 + e) * CI + ci] = ok ? v[e] : 0.0f;
                    }
                }
            }
        };
        if constexpr (CI == 48) {
            const int m = 32 * warp + lane;  // M = 128: row m is lane m, dx = -1 below 64, 0 above
            write(0, m / 64, m % 64, m % 64 < CI);
            write(K::N3, 2, 16 * warp + lane, lane < 16 && 16 * warp + lane < CI);  // M = 64
        } else {
            write(0, warp, lane, lane < 16 && warp < 3);  // M = 64: group g (dx = g - 1) in lanes 32 g ..
        }
    }
    if (!ok) atomicOr(status, 1);
    cp_async_wait_all();
    fence_before_sync();
    __syncthreads();
    if (warp == WG_MMA_WARP) {
        fence_after_sync();
        tmem_free(tmem, K::TCOLS);
    }
}

// dw[o][t][c] = sum_b partials[b][t][o][c], fixed order.  Latency-bound: a block
// takes 32 consecutive outputs (128 contiguous bytes of a partial) and deals the
// partials to 8 warps, whose sums it adds in order (44 us for 152 partials of 9 x 48
// x 48 when one thread added all of an output's partials; 6.2 us so).
// The blocks beyond those of dw add the bias gradient's partials alike.
constexpr int WR_OUT = 32, WR_SEG = 8;
__global__ void __launch_bounds__(WR_OUT * WR_SEG)
    wgrad_tc_reduce(const float* __restrict__ partials, int nb, int CO, int CI, float* __restrict__ dw,
                    const float* __restrict__ bpart, float* __restrict__ db) {
    const int wblocks = (9 * CO * CI + WR_OUT - 1) / WR_OUT;
    const bool bias = (int)blockIdx.x >= wblocks;
    const int n = bias ? CO : 9 * CO * CI;
    const float* __restrict__ src = bias ? bpart : partials;
    __shared__ float s[WR_SEG][WR_OUT];
    const int k = threadIdx.x % WR_OUT, seg = threadIdx.x / WR_OUT;
    const int i = ((int)blockIdx.x - (bias ? wblocks : 0)) * WR_OUT + k;
    float a = 0.0f;
    if (i < n) {
        const int per = (nb + WR_SEG - 1) / WR_SEG, b1 = min(nb, (seg + 1) * per);
#pragma unroll 8
        for (int b = seg * per; b < b1; ++b) a += __ldg(src + (size_t)b * n + i);
    }
    s[seg][k] = a;
    __syncthreads();
    if (seg == 0 && i < n) {
        float t = 0.0f;
#pragma unroll
        for (int j = 0; j < WR_SEG; ++j) t += s[j][k];
        const int c = i % CI, o = (i / CI) % CO, tap = i / (CI * CO);
        if (bias) db[i] = t;
        else dw[((size_t)o * 9 + tap) * CI + c] = t;
    }
}

// partials (and CTAs at most): one per two rows of a strip where they divide by two,
// else one per row
long long wgrad_parts(int B, int H, int W, int d) {
    return (long long)B * d * (H / d / ((H / d) % 2 == 0 ? 2 : 1)) * (W / TC_COLS);
}

template <int CI, int CO>
int wgrad_tc_launch(const void* x, const void* dy, float* dw, float* db, float* part, float* bpart, int B, int H, int W,
                    int d, int* status, cudaStream_t s) {
    auto k = wgrad_tc_kernel<CI, CO>;
    static_assert(Wg<CI, CO>::smem() <= 227 * 1024, "shared memory");
    const size_t smem = std::max(Wg<CI, CO>::smem(), TC_MIN_SMEM);
    CUtensorMap xmap, dmap;
    if (!row_map(&xmap, x, CI, B, H, W) || !plane_map(&dmap, dy, CO, B, H, W)) return LBM_ERR_CUDA;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return LBM_ERR_CUDA;
    const int grid = (int)std::min<long long>(wgrad_parts(B, H, W, d), (long long)nn_sm_count());
    k<<<grid, WG_THREADS, smem, s>>>(xmap, dmap, static_cast<const uint8_t*>(x), part, db ? bpart : nullptr, B, H, W, d, status);
    const int blocks = (9 * CO * CI + WR_OUT - 1) / WR_OUT + (db ? (CO + WR_OUT - 1) / WR_OUT : 0);
    wgrad_tc_reduce<<<blocks, WR_OUT * WR_SEG, 0, s>>>(part, grid, CO, CI, dw, bpart, db);
    return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}

bool conv_shape_ok(int B, int H, int W, int d) {
    return B >= 1 && d >= 1 && d <= 8 && H >= d && H % d == 0 && W >= TC_COLS && W % TC_COLS == 0 &&
           (long long)B * H * W < (1LL << 40);
}

}  // namespace

extern "C" {

int lbm_nn_conv3x3(const void* x, int32_t cin, const void* weights, const float* bias, int32_t cout, int32_t epilogue,
                   const float* residual, const void* mask, void* y, int32_t batch, int32_t h, int32_t w,
                   int32_t dilation, int32_t* status, void* stream) {
    if (!x || !weights || !y || !status || !conv_shape_ok(batch, h, w, dilation)) return LBM_ERR_ARG;
    if (((uintptr_t)x | (uintptr_t)weights | (uintptr_t)y | (uintptr_t)residual | (uintptr_t)mask) % 16 != 0)
        return LBM_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int d = dilation;
    if (epilogue == LBM_NN_RELU) {
        if (cin == 16 && cout == 48)
            return conv_tc_launch<16, 48, LBM_NN_RELU>(x, weights, bias, y, nullptr, nullptr, batch, h, w, d, status, s);
        if (cin == 48 && cout == 48)
            return conv_tc_launch<48, 48, LBM_NN_RELU>(x, weights, bias, y, nullptr, nullptr, batch, h, w, d, status, s);
    } else if (epilogue == LBM_NN_RESIDUAL) {
        if (!residual) return LBM_ERR_ARG;
        if (cin == 48 && cout == 16)
            return conv_tc_launch<48, 16, LBM_NN_RESIDUAL>(x, weights, bias, y, residual, nullptr, batch, h, w, d,
                                                             status, s);
    } else if (epilogue == LBM_NN_MASK) {
        if (!mask) return LBM_ERR_ARG;
        if (cin == 48 && cout == 48)
            return conv_tc_launch<48, 48, LBM_NN_MASK>(x, weights, nullptr, y, nullptr, mask, batch, h, w, d, status, s);
        if (cin == 16 && cout == 48)
            return conv_tc_launch<16, 48, LBM_NN_MASK>(x, weights, nullptr, y, nullptr, mask, batch, h, w, d, status, s);
    }
    return LBM_ERR_ARG;
}

size_t lbm_nn_wgrad_partial_bytes(int32_t cin, int32_t cout, int32_t batch, int32_t h, int32_t w, int32_t dilation) {
    if (!conv_shape_ok(batch, h, w, dilation) || cin < 1 || cout < 1) return 0;
    return (size_t)std::min<long long>(wgrad_parts(batch, h, w, dilation), (long long)nn_sm_count()) * 9 * cin * cout * sizeof(float);
}

int lbm_nn_conv3x3_wgrad_bias(const void* x, int32_t cin, const void* dy, int32_t cout, float* dw, float* db,
                              void* partials, size_t partial_bytes, float* bias_partials, int32_t batch, int32_t h,
                              int32_t w, int32_t dilation, int32_t* status, void* stream) {
    if (!x || !dy || !dw || !partials || !status || !conv_shape_ok(batch, h, w, dilation)) return LBM_ERR_ARG;
    if (db && !bias_partials) return LBM_ERR_ARG;
    if (((uintptr_t)x | (uintptr_t)dy) % 16 != 0) return LBM_ERR_ARG;
    if (partial_bytes < lbm_nn_wgrad_partial_bytes(cin, cout, batch, h, w, dilation)) return LBM_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    float* part = static_cast<float*>(partials);
    const int d = dilation;
    if (cin == 16 && cout == 48)
        return wgrad_tc_launch<16, 48>(x, dy, dw, db, part, bias_partials, batch, h, w, d, status, s);
    if (cin == 48 && cout == 48)
        return wgrad_tc_launch<48, 48>(x, dy, dw, db, part, bias_partials, batch, h, w, d, status, s);
    if (cin == 48 && cout == 16)
        return wgrad_tc_launch<48, 16>(x, dy, dw, db, part, bias_partials, batch, h, w, d, status, s);
    return LBM_ERR_ARG;
}

int lbm_nn_conv3x3_wgrad(const void* x, int32_t cin, const void* dy, int32_t cout, float* dw, void* partials,
                         size_t partial_bytes, int32_t batch, int32_t h, int32_t w, int32_t dilation, int32_t* status,
                         void* stream) {
    return lbm_nn_conv3x3_wgrad_bias(x, cin, dy, cout, dw, nullptr, partials, partial_bytes, nullptr, batch, h, w,
                                     dilation, status, stream);
}

}  // extern "C"
