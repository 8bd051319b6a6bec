// Device-side helpers shared by the salience kernels: PTX wrappers (mbarrier, TMA, tcgen05, cluster),
// the transposing warp reduction, and the key-tile geometry of a sample.
#pragma once

#include "common.cuh"

#include <math_constants.h>

namespace mvla {

// ------------------------------------------------------------------ small PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
// Programmatic dependent launch: a kernel launched with the programmatic-serialization attribute may
// start while its predecessor in the stream still runs.  pdl_trigger() lets the NEXT kernel start its
// prologue; pdl_wait() blocks until the PREVIOUS kernel has finished and its writes are visible.
// Both are no-ops for a kernel launched the ordinary way.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ uint32_t cluster_ctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_arrive_relaxed()
{
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_arrive_release()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait_acquire()
{
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Store into the shared memory of CTA `rank` of this cluster at the offset of `local_addr`.
__device__ __forceinline__ void st_peer_f32(uint32_t local_addr, uint32_t rank, float v)
{
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local_addr), "r"(rank));
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote), "f"(v) : "memory");
}
// One lane of a converged warp.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap* map)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}
__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Whether the phase of this parity is complete.  CLUSTER: with acquire at cluster scope (arrivals and data come from other
// CTAs).  (No suspend-time hint: with one it was measured to notice the completed phase about a microsecond late.)
template <bool CLUSTER>
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    if constexpr (CLUSTER)
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait: gives up after about one second and reports false.
template <bool CLUSTER = false>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity)
{
    const uint64_t t0 = global_ns();
    for (uint32_t it = 0; it < kSpinLimit; ++it) {
        if (mbar_try_wait<CLUSTER>(bar, parity)) return true;
        if ((it & 63u) == 63u && global_ns() - t0 > 1000000000ull) break;
    }
    return false;
}
// Asynchronous 8-byte store into the shared memory of CTA `rank` (same offset as `local_addr`); on
// landing it credits 8 bytes to that CTA's mbarrier at the offset of `local_bar`: the data and its
// "ready" signal travel together, one way.
__device__ __forceinline__ void st_async_pair(uint32_t local_addr, uint32_t local_bar, uint32_t rank, float2 v)
{
    uint32_t raddr, rbar;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(raddr) : "r"(local_addr), "r"(rank));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rbar) : "r"(local_bar), "r"(rank));
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];"
                 ::"r"(raddr), "f"(v.x), "f"(v.y), "r"(rbar) : "memory");
}
// 2^x in one instruction.
__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Exponents are taken against a reference that need not be the maximum; one (log2) above this moves the warp's reference.
constexpr float kRescaleAt = 64.f;
// One box of a 3-D tiled tensor map -> this CTA's shared memory; completion counted on `bar`.
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z,
                                            uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
                 " [%0], [%1, {%3, %4, %5}], [%2];"
                 ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y), "r"(z) : "memory");
}
// `bytes` (a multiple of 16) from a 16-byte boundary of global memory -> this CTA's shared memory; completion counted on `bar`.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D[tmem] (+)= A[smem] * B[smem]^T, bf16 inputs, fp32 accumulate; issued by one thread.
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "setp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// The same for 8-bit floating-point operands (both e4m3), fp32 accumulate; one instruction covers 32
// elements of the contraction.
__device__ __forceinline__ void umma_e4m3(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "setp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// Element size 2: bf16 operands; 1: e4m3 operands.  Either way one instruction consumes 32 bytes of every row.
__device__ __forceinline__ void umma_by_size(int esize, uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                             uint32_t idesc, uint32_t accumulate)
{
    if (esize == 2) umma_bf16(d_tmem, a_desc, b_desc, idesc, accumulate);
    else umma_e4m3(d_tmem, a_desc, b_desc, idesc, accumulate);
}
// A descriptor whose start address lies 16 x `units` bytes further on (below 256 KB: the low word does not carry).
__device__ __forceinline__ uint64_t desc_plus(uint64_t desc, uint32_t units)
{
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(static_cast<uint32_t>(desc) + units), "r"(static_cast<uint32_t>(desc >> 32)));
    return d;
}
// The MMAs over one box (128-byte swizzle rows) of both operands: `n` of them, 32 bytes of every row each, the first of them
// accumulating when asked and the others always.  Four in a row without a loop, in 32-bit descriptor arithmetic: issued
// one by one in a loop over run-time sizes the eight MMAs of a key tile of 128 bf16 elements took 750 cycles, like this 370 to 400,
// which is what they take to execute (N = 16 to 64).
__device__ __forceinline__ void umma_box(int esize, uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, int n, bool accumulate)
{
    const uint32_t first = accumulate ? 1u : 0u;
    if (n == 4 && esize == 2) {
#pragma unroll
        for (uint32_t kb = 0; kb < 4; ++kb) umma_bf16(d_tmem, desc_plus(a_desc, 2 * kb), desc_plus(b_desc, 2 * kb), idesc, kb ? 1u : first);
    } else if (n == 4) {
#pragma unroll
        for (uint32_t kb = 0; kb < 4; ++kb) umma_e4m3(d_tmem, desc_plus(a_desc, 2 * kb), desc_plus(b_desc, 2 * kb), idesc, kb ? 1u : first);
    } else {                                  // the last box of a head dim that is no multiple of 128 bytes
        for (int kb = 0; kb < n; ++kb) umma_by_size(esize, d_tmem, a_desc + 2 * kb, b_desc + 2 * kb, idesc, kb ? 1u : first);
    }
}
__device__ __forceinline__ void umma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// 16 consecutive fp32 columns of this thread's tensor-memory lane.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32"
                 "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Shared-memory matrix descriptor: K-major tile, 128-byte rows, 128-byte swizzle, groups of 8 rows
// 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr)
{
    uint64_t d = 0;
    d |= static_cast<uint64_t>((addr & 0x3FFFFu) >> 4);          // start address
    d |= static_cast<uint64_t>(1) << 16;                         // leading byte offset (unused here)
    d |= static_cast<uint64_t>(1024 >> 4) << 32;                 // stride byte offset
    d |= static_cast<uint64_t>(1) << 46;                         // descriptor version
    d |= static_cast<uint64_t>(2) << 61;                         // 128-byte swizzle
    return d;
}
// Instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, M = 128, N = n.
__device__ __forceinline__ uint32_t idesc_bf16_m128(int n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(n >> 3) << 17) | ((128u >> 4) << 24);
}
// Instruction descriptor: e4m3 x e4m3 -> fp32 (operand format code 0 for both), K-major, M = 128, N = n.
__device__ __forceinline__ uint32_t idesc_e4m3_m128(int n)
{
    return (1u << 4) | (static_cast<uint32_t>(n >> 3) << 17) | ((128u >> 4) << 24);
}
__device__ __forceinline__ uint32_t idesc_by_size(int esize, int n)
{
    return esize == 2 ? idesc_bf16_m128(n) : idesc_e4m3_m128(n);
}

// Reduce 16 per-thread values across the 32 lanes of a warp in 16 shuffles.  On return lane L
// holds the result of column col16(L); lanes L and L^1 hold the same column.
template <bool IS_MAX>
__device__ __forceinline__ float warp_reduce16(float (&v)[16], int lane)
{
#pragma unroll
    for (int w = 8; w >= 1; w >>= 1) {
        const int off = w * 2;
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < w; ++i) {
            const float send = up ? v[i] : v[i + w];
            const float keep = up ? v[i + w] : v[i];
            const float got = __shfl_xor_sync(0xffffffffu, send, off);
            v[i] = IS_MAX ? fmaxf(keep, got) : keep + got;
        }
    }
    const float got = __shfl_xor_sync(0xffffffffu, v[0], 1);
    return IS_MAX ? fmaxf(v[0], got) : v[0] + got;
}
__device__ __forceinline__ int col16(int lane)
{
    return ((lane >> 4) & 1) * 8 + ((lane >> 3) & 1) * 4 + ((lane >> 2) & 1) * 2 + ((lane >> 1) & 1);
}

struct TileInfo {
    int valid;   // keys of this tile that exist (0: tile past the end)
    int row0;    // first row in the packed tensors
    int vis0;    // visual index of the first key
};
__device__ __forceinline__ TileInfo tile_info(const SampleDev& s, int tt)
{
    const int t2 = (s.n_2d + kKeyTile - 1) / kKeyTile;
    const int t3 = (s.n_3d + kKeyTile - 1) / kKeyTile;
    TileInfo ti{0, 0, 0};
    if (tt < t2) {
        const int st = tt * kKeyTile;
        ti.valid = min(kKeyTile, s.n_2d - st);
        ti.row0 = s.seq_off + s.off_2d + st;
        ti.vis0 = st;
    } else if (tt < t2 + t3) {
        const int st = (tt - t2) * kKeyTile;
        ti.valid = min(kKeyTile, s.n_3d - st);
        ti.row0 = s.seq_off + s.off_3d + st;
        ti.vis0 = s.n_2d + st;
    }
    return ti;
}

__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }


}  // namespace mvla
