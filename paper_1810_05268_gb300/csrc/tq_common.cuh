// Pieces shared by the kernels fed by tensor copies with a register z queue
// (stencil_tq.cu: OT2, ot4_tq.cu: OT4): bounded mbarrier waits, the copy of a
// tile, the ring's layout.
#pragma once
#include <cuda.h>

#include "stencil_v3.cuh"

namespace ckfwi {
namespace {

__device__ __forceinline__ unsigned sa(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void bar_init(uint64_t* bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sa(bar)) : "memory");
}

__device__ __forceinline__ void bar_expect(uint64_t* bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(sa(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool bar_try(uint64_t* bar, unsigned parity)
{
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(sa(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// bounded wait with a short back-off; rounds < 0 gives up without looking
// (how a test makes a plane's wait run out); the drain before a CTA leaves
// always waits with the full bound, so no copy lands after it has gone
constexpr long long DRAIN_ROUNDS = 1LL << 22;
__device__ __forceinline__ bool bar_wait(uint64_t* bar, unsigned parity, long long rounds)
{
    if (rounds < 0) return false;
    for (int i = 0; i < 4; ++i)
        if (bar_try(bar, parity)) return true;
    for (long long i = 0; i < rounds; ++i) {
        __nanosleep(32);
        if (bar_try(bar, parity)) return true;
    }
    return false;
}

__device__ __forceinline__ void tile3(void* dst, const CUtensorMap* tm, int x, int y, int z, uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::
            "r"(sa(dst)),
        "l"(reinterpret_cast<unsigned long long>(tm)), "r"(x), "r"(y), "r"(z), "r"(sa(bar))
        : "memory");
}

// NP: point fields (one 32 x 16 tile a plane each)
template <int K, int PF, int NP = 2>
struct TQ {
    static constexpr int V = 4, TX = 8, TY = 16, D = PF;
    using G = G3<K, V, TX, TY>;
    // A tile of the staged field waits in the ring from when its column feeds
    // the queue (K planes ahead) until it is the centre plane.  At order 16
    // that is 67 KB a CTA, two or three CTAs an SM; there the queue loads its
    // column itself (the tile's copy finds it in L2) and the ring holds the
    // planes of the prefetch only: four CTAs an SM with one plane of it.  At
    // 300 x 600 x 600 a forward step takes 523 us (595 with the long ring, 554
    // the lean kernel), the split reverse step 985 us (1118).
    static constexpr bool COL = K > 4;
    static constexpr int LEAD = COL ? 0 : K;                   // planes from a group's u tile to its point tiles
    static constexpr int RU = LEAD + D + 1;                    // u tiles in the ring
    static constexpr int RP = D + 1;                           // point tiles of each point field
    static constexpr int UBYTES = G::TILE * 4;                 // one u box
    static constexpr int US = (UBYTES + 127) / 128 * 32;       // ring slot stride [floats], 128-byte multiple
    static constexpr int PT = G::BXP * TY;                     // floats of a point tile
    static constexpr int PBYTES = PT * 4;
    static constexpr size_t SMEM = (size_t)RU * US * 4 + NP * (size_t)RP * PBYTES + RU * 8 + 128;
};

// first 128-byte aligned address of the dynamic shared memory
__device__ __forceinline__ unsigned char* align128(unsigned char* p)
{
    const unsigned a = sa(p);
    return p + ((128u - (a & 127u)) & 127u);
}

}  // namespace
}  // namespace ckfwi
