// Blackwell (sm_100a) building blocks in inline PTX: mbarriers, TMA tile loads, tcgen05 MMA with
// TMEM accumulators.  Every wait is bounded: a wait that runs out returns false and the caller
// records GRAPHKV_ERR_TIMEOUT and drains instead of hanging the device.
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace graphkv {
namespace tc {

constexpr int kTileKeys = 128;                              // keys per MMA tile (UMMA M or N)
constexpr int kHalfBytes = kTileKeys * 64 * 2;              // 128 rows x 64 bf16 (one swizzle atom wide)
template <int kD> __host__ __device__ constexpr int tile_bytes() { return (kD / 64) * kHalfBytes; }
constexpr long long kWaitCycles = 4000000000LL;             // default limit of a wait: ~2 s at 2 GHz

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// ---- mbarrier ---------------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_inval(uint32_t bar)
{
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_fence_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait for the phase with the given parity to complete: false after `limit` clocks.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, long long limit)
{
    if (mbar_try(bar, parity)) return true;
    const long long t0 = clock64();
    while (true) {
#pragma unroll 1
        for (int i = 0; i < 64; ++i)
            if (mbar_try(bar, parity)) return true;
        if (clock64() - t0 > limit) return false;
    }
}

// ---- TMA --------------------------------------------------------------------------------------
__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap *tm)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(tm)) : "memory");
}
// 4-D tiled load global -> shared, completion counted in bytes on `bar`.
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *tm, uint32_t bar,
                                            int c0, int c1, int c2, int c3)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tm)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}
// The same over five dimensions.
__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap *tm, uint32_t bar,
                                            int c0, int c1, int c2, int c3, int c4)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tm)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
        : "memory");
}
// One key tile: keys key0 .. key0 + 127 of (h, b), all kD dimensions, announced on `bar`.
template <int kD>
__device__ __forceinline__ void tma_load_tile(uint32_t dst, const CUtensorMap *tm, uint32_t bar, int key0, int h, int b)
{
    mbar_expect_tx(bar, tile_bytes<kD>());
#pragma unroll
    for (int half = 0; half < kD / 64; ++half)
        tma_load_4d(dst + half * kHalfBytes, tm, bar, half * 64, key0, h, b);
}
// Generic-proxy writes to shared memory become visible to the async proxy (TMA, tensor core).
__device__ __forceinline__ void fence_proxy_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// ---- tcgen05 ----------------------------------------------------------------------------------
__device__ __forceinline__ void tmem_alloc(uint32_t smem_dst, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst),
                 "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory operand descriptor: K-major tile of 128-byte rows, 128-byte swizzle, 8-row
// groups 1024 bytes apart.  `addr` may be advanced by 32 bytes per 16-element K step.
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t addr)
{
    uint64_t d = 0;
    d |= static_cast<uint64_t>((addr & 0x3ffffu) >> 4);        // start address
    d |= static_cast<uint64_t>(1) << 16;                       // leading byte offset (unused here)
    d |= static_cast<uint64_t>(1024 >> 4) << 32;               // stride byte offset: 8 rows
    d |= static_cast<uint64_t>(1) << 46;                       // descriptor version (sm_100)
    d |= static_cast<uint64_t>(2) << 61;                       // SWIZZLE_128B
    return d;
}
// Instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, M x N tile.
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int m, int n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(n >> 3) << 17) |
           (static_cast<uint32_t>(m >> 4) << 24);
}
// D[tmem] (+)= A[smem] * B[smem]^T, issued by one thread.
__device__ __forceinline__ void umma_bf16(uint32_t taddr, uint64_t adesc, uint64_t bdesc,
                                          uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(taddr), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// One thread of a converged warp.
__device__ __forceinline__ bool elect_one()
{
    uint32_t is;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(is));
    return is != 0;
}
// This thread's warp, as a value the compiler knows to be the same in all its lanes.
__device__ __forceinline__ int warp_index() { return __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0); }

// Low word of an operand descriptor (umma_desc_sw128); the high word is the same for all.  16 elements along K are 2
// in it, 64 columns on half_bytes / 16.
__device__ __forceinline__ uint32_t umma_desc_lo(uint32_t addr) { return ((addr & 0x3ffffu) >> 4) | (1u << 16); }
constexpr uint32_t kUmmaDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
// D[tmem] = A B^T over kD columns: A and B by the low words of their descriptors.  Called by all lanes of a warp, with the
// same values: the operands then stay in uniform registers, where the instruction takes them from (issued from a branch
// that one lane takes, with descriptors put together there, eight products took 1100 to 1400 clocks to issue).
template <int kD>
__device__ __forceinline__ void umma_tile(uint32_t taddr, uint32_t a_lo, uint32_t a_half, uint32_t b_lo, uint32_t b_half, uint32_t idesc)
{
#pragma unroll
    for (int k = 0; k < kD / 16; ++k)
        asm volatile(
            "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\t"
            "mov.b64 a, {%1, %3};\n\t"
            "mov.b64 b, {%2, %3};\n\t"
            "setp.ne.u32 p, %5, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, p;\n\t}"
            ::"r"(taddr), "r"(a_lo + (k >> 2) * a_half + (k & 3) * 2), "r"(b_lo + (k >> 2) * b_half + (k & 3) * 2), "n"(kUmmaDescHi),
              "r"(idesc), "r"((uint32_t)(k > 0))
            : "memory");
}
// Arrive on `bar` once all MMAs issued so far by this thread have completed.
__device__ __forceinline__ void umma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}
// 16 consecutive fp32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
// Split form of the 32-column load: the registers hold the data only after tmem_ld_fence(r).
__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
          "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
          "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
// Split forms of the 16- and 8-column loads.
__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld8_issue(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}
// Waits for every TMEM load of this thread; the empty statements tie the registers to the wait so
// that no use of them can be scheduled above it.
template <int N> __device__ __forceinline__ void tmem_ld_fence(uint32_t (&r)[N])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int k = 0; k < N; ++k) asm volatile("" : "+r"(r[k]));
}

__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Packed pairs of floats in one 64-bit register: sm_100 issues an FMA or an add on both halves as
// one instruction, which halves the issue slots the exponent arithmetic of the score sweeps takes.
__device__ __forceinline__ uint64_t pack2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// ex2 of both halves on the MUFU unit
__device__ __forceinline__ uint64_t ex2_pair(uint64_t x)
{
    float lo, hi;
    unpack2(x, lo, hi);
    return pack2(ex2(lo), ex2(hi));
}

// 2^x of both halves for x <= 0, on the FMA and integer pipes (the MUFU unit is the ceiling of the score
// sweeps): x = n + f with n the nearest integer and f in [-1/2, 1/2], 2^f by a cubic fitted for relative error
// (max 1.03e-4), 2^n by adding n to the exponent field.  x is clamped at -125 (result ~0).
__device__ __forceinline__ uint64_t ex2_poly3_pair(uint64_t x)
{
    float lo, hi;
    unpack2(x, lo, hi);
    x = pack2(fmaxf(lo, -125.0f), fmaxf(hi, -125.0f));
    const uint64_t magic = pack2(12582912.0f, 12582912.0f);         // 1.5 * 2^23: the integer part lands in the low mantissa bits
    const uint64_t t = add2(x, magic);
    const uint64_t n = add2(t, pack2(-12582912.0f, -12582912.0f));
    const uint64_t f = fma2(n, pack2(-1.0f, -1.0f), x);
    uint64_t p = fma2(pack2(0.0549740307f, 0.0549740307f), f, pack2(0.242215246f, 0.242215246f));
    p = fma2(p, f, pack2(0.693289936f, 0.693289936f));
    p = fma2(p, f, pack2(1.0f, 1.0f));
    float plo, phi, tlo, thi;
    unpack2(p, plo, phi);
    unpack2(t, tlo, thi);
    return pack2(__int_as_float(__float_as_int(plo) + (__float_as_int(tlo) << 23)),
                 __int_as_float(__float_as_int(phi) + (__float_as_int(thi) << 23)));
}

// sum over i < 32 of 2^(v[i] * scale + c[i]) (times w[i]): nc(q), and with kWeighted nw(q), return
// elements 4q .. 4q+3 as two packed pairs.  kPoly of every four pairs take the polynomial.
template <int kPoly, bool kWeighted, class NegC, class Weight>
__device__ __forceinline__ float ex2_sum32(const float (&v)[32], uint64_t scale2, NegC nc, Weight nw)
{
    uint64_t acc0 = 0ull, acc1 = 0ull;             // (0.f, 0.f)
#pragma unroll
    for (int p = 0; p < 16; p += 2) {
        const ulonglong2 c = nc(p >> 1);
        const uint64_t x0 = fma2(pack2(v[2 * p], v[2 * p + 1]), scale2, c.x);
        const uint64_t x1 = fma2(pack2(v[2 * p + 2], v[2 * p + 3]), scale2, c.y);
        const uint64_t e0 = (p & 3) >= 4 - kPoly ? ex2_poly3_pair(x0) : ex2_pair(x0);
        const uint64_t e1 = ((p + 1) & 3) >= 4 - kPoly ? ex2_poly3_pair(x1) : ex2_pair(x1);
        if constexpr (kWeighted) {
            const ulonglong2 w = nw(p >> 1);
            acc0 = fma2(e0, w.x, acc0);
            acc1 = fma2(e1, w.y, acc1);
        } else {
            acc0 = add2(acc0, e0);
            acc1 = add2(acc1, e1);
        }
    }
    float lo, hi;
    unpack2(add2(acc0, acc1), lo, hi);
    return lo + hi;
}

// Byte offset of the 16-byte piece `c16` of row `r` inside a K-major, 128-byte-swizzled operand of
// `rows` rows x 128 (or 64) bf16: halves of 64 columns, rows 128 bytes apart.
__device__ __forceinline__ uint32_t sw128_offset(int rows, int r, int c16)
{
    return static_cast<uint32_t>((c16 >> 3) * rows * 128 + r * 128 + (((c16 & 7) ^ (r & 7)) << 4));
}

}  // namespace tc
}  // namespace graphkv
