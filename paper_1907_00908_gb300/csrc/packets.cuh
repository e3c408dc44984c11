// packets.cuh -- face values sent between the blocks of one cooperative launch:
// 16-byte packets {re, stamp, im, stamp} that the receiver polls (data and flag in one
// word, as the low-latency protocol of NCCL has them; see sweep_resident.cu for why
// no packet is lost or taken twice), and the site flags of the kernels that cut a grid
// into blocks.
#pragma once
#include "lbmbt_internal.cuh"
#include "tma_common.cuh"

namespace lbmbt {
namespace {

// Each half of a packet, a value and its stamp, is one 64-bit element of the access: a
// vector access is as many accesses as it has elements, in no stated order, so an
// element is what arrives as a whole.
__device__ __forceinline__ void send(uint4* to, float2 v, unsigned stamp)
{
    asm volatile("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%1, %3};\n\tmov.b64 b, {%2, %3};\n\t"
                 "st.volatile.global.v2.u64 [%0], {a, b};\n\t}" ::"l"(to), "r"(__float_as_uint(v.x)),
                 "r"(__float_as_uint(v.y)), "r"(stamp)
                 : "memory");
}

__device__ __forceinline__ uint4 peek(const uint4* from)
{
    uint4 p;
    asm volatile("{\n\t.reg .b64 a, b;\n\tld.volatile.global.v2.u64 {a, b}, [%4];\n\t"
                 "mov.b64 {%0, %1}, a;\n\tmov.b64 {%2, %3}, b;\n\t}"
                 : "=r"(p.x), "=r"(p.y), "=r"(p.z), "=r"(p.w)
                 : "l"(from)
                 : "memory");
    return p;
}

// A thread's waits: their bound, and whether it has passed (the thread then goes on
// without waiting).
struct Waits {
    unsigned long long limit_ns;
    bool dead;
};

// Polls a packet until both halves carry the stamp, or the bound has passed.
__device__ __noinline__ uint4 await(const uint4* from, unsigned stamp, Waits& w)
{
    uint4 p = peek(from);
    const unsigned long long t0 = globaltimer();
    for (unsigned n = 1; !w.dead && !(p.y == stamp && p.w == stamp); ++n) {
        if ((n & 63u) == 0 && globaltimer() - t0 > w.limit_ns) w.dead = true;
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
