// packets.cuh -- face values sent between the blocks of one cooperative launch:
// 16-byte packets {re, stamp, im, stamp} that the receiver polls (see
// sweep_resident.cu for why no packet is lost or taken twice), and the site flags
// of the kernels that cut a grid into blocks.
#pragma once
#include "lbmbt_internal.cuh"
#include "tma_common.cuh"

namespace lbmbt {
namespace {

__device__ __forceinline__ void send(uint4* to, float2 v, unsigned stamp)
{
    asm volatile("st.volatile.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(to), "r"(__float_as_uint(v.x)), "r"(stamp),
                 "r"(__float_as_uint(v.y)), "r"(stamp)
                 : "memory");
}

__device__ __forceinline__ uint4 peek(const uint4* from)
{
    uint4 p;
    asm volatile("ld.volatile.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(p.x), "=r"(p.y), "=r"(p.z), "=r"(p.w)
                 : "l"(from)
                 : "memory");
    return p;
}

// Polls a packet until both halves carry the stamp; `dead` once the limit has passed.
__device__ __noinline__ uint4 await(const uint4* from, unsigned stamp, bool& dead)
{
    uint4 p = peek(from);
    const unsigned long long t0 = globaltimer();
    for (unsigned n = 1; !dead && !(p.y == stamp && p.w == stamp); ++n) {
        if ((n & 63u) == 0 && globaltimer() - t0 > WAIT_NS) dead = true;
        p = peek(from);
    }
    return p;
}

// Site flags: bits 0..5 at a face of the grid, 6..9 on a face of the block (-y, +y,
// -z, +z), 10 a site at all, 11..14 in the layer behind a face of the block, 16..21
// the membrane links (of the half-link rule), 22..23 the phase.
enum : unsigned { S_GRID = 63u, S_SEND = 0x3c0u, S_SEND2 = 0x7800u, S_ON = 1024u };

}  // namespace
}  // namespace lbmbt
