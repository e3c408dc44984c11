// sweep_resident.cu -- many time steps in one launch for grids that fit on chip.
//
// A step of a small grid is latency, not work: one launch per step took 6.5 us
// at 32^3, of which the launch, the first copies and the drain are nearly all,
// on 32 of 152 SMs.  Here one cooperative launch runs every step.  The grid is
// cut into blocks of nx x hy x hz sites, one per CTA and SM, whose populations
// stay in shared memory (two time levels of populations 1-6; the rest population
// in registers).  Only the faces travel: per step a block sends one population
// of one layer of sites through each of its four faces.
//
// A face value is one 16-byte packet {re, stamp, im, stamp} in a buffer of the
// receiving block, and the receiver polls the packet itself: there is no grid
// barrier, no flag and no fence, so a step costs one store-to-load trip through
// L2.  Each 8-byte half carries its stamp, so a half that arrived alone is not
// taken.  Stamps count the steps of all launches on the context and never
// repeat, so what an earlier launch left in the buffers is never taken either.
// Four buffers take turns (step modulo 4).  A block overwrites the packet of
// step k at step k + 4, after it has received the neighbour's packet of step
// k + 3; the neighbour sent that after its block barrier of step k + 2, and all
// its threads had read step k before its barrier of step k + 1.
//
// Every poll is bounded (2 s); one that runs out sets the error word of the step
// control, and the block goes on without waiting.
//
// Arithmetic and order per site are those of the register sweep (same bits).
//
// Membranes at given positions (theta = 0 rule): where each of a link's six
// values lies and its six coefficients do not change over a run, so every launch
// lists the block's links once in shared memory and a step gathers and sums,
// one link a thread, before the sites take the results.  A face then carries
// three values a column: both populations of its axis in the outer layer and
// the outgoing one of the layer behind.
#include <algorithm>

#include "lbmbt_internal.cuh"
#include "sweep_common.cuh"
#include "links.cuh"
#include "packed.cuh"
#include "packets.cuh"

namespace lbmbt {
namespace {

constexpr int RES_NT = 512;           // threads of a block
constexpr int RES_MAX_SITES = 2048;   // sites of a block: 13 x 8 B each in shared memory

// A listed link: elements of a level of own g_ib, g_ib behind, own g_i, g_i(y),
// g_i behind y, g_ib(y); per value 4 bits, 1 + the boundary factor it takes and
// 8 if conjugated first; the coefficients.
struct LinkEntry {
    uint16_t at[6];
    uint32_t face;
    float A[3], B[3];
};
static_assert(sizeof(LinkEntry) == 40, "link entry");

// cmul() with its roundings written out: as the register sweep's reads beyond a
// face come out of the compiler, so that the fields are the same bits.
__device__ __forceinline__ float2 turn(float2 a, float2 b)
{
    return make_float2(__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)), __fmaf_rn(a.x, b.y, __fmul_rn(a.y, b.x)));
}

// Directions (bits 1..6) in which site s takes the position rule: a membrane
// behind it, none ahead, none behind the far node.
__device__ __forceinline__ unsigned rule_links(const MemberDesc* __restrict__ d, unsigned mk, int x, int y, int z, int np)
{
    unsigned rule = 0;
    const int c[3] = {x, y, z}, n[3] = {d->nx, d->ny, d->nz};
    for (int i = 1; i <= np; ++i) {
        const int ib = (i & 1) ? i + 1 : i - 1, a = (i - 1) >> 1;
        if (!(mk & (1u << (ib - 1))) || (mk & (1u << (i - 1)))) continue;
        int v[3] = {c[0], c[1], c[2]};
        v[a] = (v[a] + ((i & 1) ? n[a] - 1 : 1)) % n[a];   // a membrane never crosses a mirror face
        const unsigned mky = d->mask[((unsigned)v[2] * d->ny + v[1]) * d->nx + v[0]];
        if (!(mky & (1u << (ib - 1)))) rule |= 1u << i;
    }
    return rule;
}

// Largest number of listed links of a block.
__global__ void resident_links_kernel(const MemberDesc* __restrict__ members, const ResBlock* __restrict__ blocks, int np,
                                      int* out)
{
    __shared__ int n;
    if (threadIdx.x == 0) n = 0;
    __syncthreads();
    const ResBlock b = blocks[blockIdx.x];
    const MemberDesc* __restrict__ d = members + b.m;
    const int nx = d->nx, S = nx * b.hy * b.hz;
    if (d->dlt)
        for (int l = threadIdx.x; l < S; l += blockDim.x) {
            const int z = l / (nx * b.hy), row = l / nx - z * b.hy, x = l % nx, gy = b.y0 + row, gz = b.z0 + z;
            const unsigned rule = rule_links(d, d->mask[((unsigned)gz * d->ny + gy) * nx + x], x, gy, gz, np);
            if (rule) atomicAdd(&n, __popc(rule));
        }
    __syncthreads();
    if (threadIdx.x == 0) atomicMax(out, n);
}

// SPT sites a thread; D2: the D2Q5 lattice (no z populations, weights of a);
// GEN: the waveform may take values other than 0 and +-1; LK: a member has
// membrane positions.
template <int SPT, bool D2, bool GEN, bool LK>
__global__ void __launch_bounds__(RES_NT, 1) sweep_resident_kernel(const SweepArgs a, const ResArgs r)
{
    extern __shared__ __align__(16) unsigned char res_smem[];
    __shared__ float2 s_fac[2][6];   // boundary factors of this step and of the next
    __shared__ float s_f[2];
    __shared__ float2 s_phase[4];    // (omega, eps) per phase

    constexpr int NP = D2 ? 4 : 6;   // populations in shared memory: 1 .. NP
    const int t = threadIdx.x;
    const ResBlock b = r.blocks[blockIdx.x];
    const MemberDesc* __restrict__ d = a.members + b.m;
    const int nx = d->nx, ny = d->ny, nz = d->nz;
    const int S = nx * b.hy * b.hz, layer = nx * b.hy;
    // two time levels of [NP][S] and the received face values after each; the rotations
    const int lsz = NP * S + b.n_recv;
    float2* const lev = reinterpret_cast<float2*>(res_smem);
    float2* const rots = lev + 2 * lsz;
    float2* const lres = rots + S;                                       // results of the listed links
    LinkEntry* const lent = reinterpret_cast<LinkEntry*>(lres + r.max_links);
    __shared__ int s_links;
    if (LK) {
        if (threadIdx.x == 0) s_links = 0;
        __syncthreads();
    }
    const unsigned P = (unsigned)d->plane, sxy = (unsigned)nx * ny;
    const float2* __restrict__ src = d->state + (size_t)r.lsrc * 7 * P;
    const int bc[3] = {d->bc[0], d->bc[1], d->bc[2]};
    const u64 sh2 = pk(d->s_share, d->s_share);
    const int es = d->end_step;
    const int sig = es >= 0 ? es : r.sig_step, fstep = es >= 0 ? es : r.field_step;
    float2* const field = d->field;
    float2* const mout = d->mout;
    if (t < 4) s_phase[t] = make_float2(d->omega[t], d->eps[t]);

    // this thread's sites: element in the grid, flags, place in a z face (low
    // half) and in a y face, and where the y and z pulls come from (element of a
    // level, 16 bits each: -y, +y and -z, +z)
    unsigned gs[SPT], fl[SPT], pl[SPT], oy[SPT], oz[SPT];
    unsigned lk[SPT];   // LK: first result of the site's listed links, their directions << 16
    u64 p0[SPT];
    float thg[SPT];
#pragma unroll
    for (int j = 0; j < SPT; ++j) {
        const int l = t + j * RES_NT;
        gs[j] = fl[j] = pl[j] = oy[j] = oz[j] = lk[j] = 0u;
        p0[j] = 0ull;
        thg[j] = 0.f;
        if (l < S) {
            const int z = l / layer, in = l - z * layer, row = in / nx, x = in - row * nx;
            const int gy = b.y0 + row, gz = b.z0 + z;
            const unsigned s = (unsigned)gz * sxy + (unsigned)gy * nx + x;
            gs[j] = s;
            const unsigned mk = d->mask[s];
            const bool yl = row == 0, yh = row == b.hy - 1, zl = z == 0, zh = z == b.hz - 1;
            fl[j] = S_ON | (mk << 16) | (x == 0 ? 1u : 0u) | (x == nx - 1 ? 2u : 0u) | (gy == 0 ? 4u : 0u) |
                    (gy == ny - 1 ? 8u : 0u) | (gz == 0 ? 16u : 0u) | (gz == nz - 1 ? 32u : 0u) |
                    (yl && b.nbr[0] >= 0 ? 64u : 0u) | (yh && b.nbr[1] >= 0 ? 128u : 0u) |
                    (zl && b.nbr[2] >= 0 ? 256u : 0u) | (zh && b.nbr[3] >= 0 ? 512u : 0u);
            const int ez = z * nx + x;
            pl[j] = (unsigned)in | ((unsigned)ez << 16);
            // the neighbour's site, a received value, the far side of this block, or
            // (mirror) the own opposite population
            auto from = [&](bool face, int nb, int step, int wrap, int pop, int opp, int recv) -> unsigned {
                if (!face) return (unsigned)((pop - 1) * S + l + step);
                if (nb >= 0) return (unsigned)(NP * S + recv);
                return (unsigned)(nb == RES_SELF ? (pop - 1) * S + l + wrap : (opp - 1) * S + l);
            };
            const int wy = (b.hy - 1) * nx, wz = (b.hz - 1) * layer;
            oy[j] = from(yl, b.nbr[0], -nx, wy, 3, 4, b.recv[0] + ez) | (from(yh, b.nbr[1], nx, -wy, 4, 3, b.recv[1] + ez) << 16);
            if (!D2)
                oz[j] = from(zl, b.nbr[2], -layer, wz, 5, 6, b.recv[2] + in) |
                        (from(zh, b.nbr[3], layer, -wz, 6, 5, b.recv[3] + in) << 16);
            if (LK) {
                fl[j] |= (row == 1 && b.nbr[0] >= 0 ? 0x800u : 0u) | (row == b.hy - 2 && b.nbr[1] >= 0 ? 0x1000u : 0u) |
                         (z == 1 && b.nbr[2] >= 0 ? 0x2000u : 0u) | (z == b.hz - 2 && b.nbr[3] >= 0 ? 0x4000u : 0u);
                const unsigned rule = d->dlt ? rule_links(d, mk, x, gy, gz, NP) : 0u;
                if (rule) {
                    int e = atomicAdd(&s_links, __popc(rule));
                    lk[j] = (unsigned)e | rule << 16;
                    for (int i = 1; i <= NP; ++i) {
                        if (!(rule & (1u << i))) continue;
                        const int ib = (i & 1) ? i + 1 : i - 1, a3 = (i - 1) >> 1, dir = (i & 1) ? 1 : -1;
                        fl[j] &= ~(1u << (16 + ib - 1));   // not the half-link rule
                        LinkEntry L;
                        L.face = 0;
                        // element of population p at the node dd along axis a3, and its face
                        auto along = [&](int j6, int p, int dd) {
                            const int c = a3 == 0 ? x : a3 == 1 ? row : z, ext = a3 == 0 ? nx : a3 == 1 ? b.hy : b.hz;
                            const int stride = a3 == 0 ? 1 : a3 == 1 ? nx : layer, cp = c + dd;
                            int at = (p - 1) * S + l + dd * stride;
                            if (cp < 0 || cp >= ext) {
                                const bool lo = cp < 0;
                                const int side = lo ? 0 : 1;
                                const int nb = a3 == 0 ? (bc[0] == BC_PER ? RES_SELF : RES_MIRROR) : b.nbr[2 * (a3 - 1) + side];
                                const bool grid = a3 == 0 || (a3 == 1 ? (lo ? b.y0 == 0 : b.y0 + b.hy == ny)
                                                                      : (lo ? b.z0 == 0 : b.z0 + b.hz == nz));
                                const unsigned fc = 1u + 2 * a3 + side;
                                if (nb == RES_MIRROR) {
                                    const int m = lo ? -1 - cp : 2 * ext - 1 - cp, po = (p & 1) ? p + 1 : p - 1;
                                    at = (po - 1) * S + l + (m - c) * stride;
                                    if (bc[a3] != BC_MIR) L.face |= (8u | fc) << (4 * j6);
                                } else {
                                    if (grid) L.face |= fc << (4 * j6);
                                    if (nb == RES_SELF) {
                                        at += (lo ? ext : -ext) * stride;
                                    } else {
                                        const int far = lo ? -cp : cp - ext + 1;   // 1 or 2 layers beyond
                                        const int q = far == 2 ? 2 : p == 2 * a3 + 1 + side ? 0 : 1;
                                        at = NP * S + b.recv[2 * (a3 - 1) + side] + (a3 == 1 ? q * nx * b.hz + ez : q * layer + in);
                                    }
                                }
                            }
                            L.at[j6] = (uint16_t)at;
                        };
                        along(0, ib, 0);
                        along(1, ib, dir);
                        along(2, i, 0);
                        along(3, i, -dir);
                        along(4, i, -2 * dir);
                        along(5, ib, -dir);
                        link_coefficients(d->dlt[(size_t)(ib - 1) * P + s], d->lrho, L.A, L.B);
                        lent[e++] = L;
                    }
                }
            }
            rots[l] = rotation_m1(d, 1.f, x, gy, gz);
            if (GEN) thg[j] = __fmaf_rn(d->ctheta[2], (float)(gz + d->z0),
                                        __fmaf_rn(d->ctheta[1], (float)gy, __fmul_rn(d->ctheta[0], (float)x)));
            p0[j] = __ldcg(reinterpret_cast<const u64*>(src) + s);
#pragma unroll
            for (int i = 1; i <= NP; ++i) lev[(i - 1) * S + l] = __ldcg(src + (size_t)i * P + s);
        }
    }
    if (t < 6) s_fac[0][t] = __ldg(a.fac + ((size_t)r.k0 * a.n_members + b.m) * 6 + t);
    if (t == 6) s_f[0] = __ldg(d->fw + r.k0);

    // gradient segments: level n of the launch, n < n_steps, as it is at the start of step n
    auto put_level = [&](int n, int l, unsigned s, u64 v0, const u64* v) {
        u64* to = reinterpret_cast<u64*>(d->adj) + (size_t)(r.level0 + n) * 7 * P + s;
        __stcs(to, v0);
        for (int i = 1; i <= NP; ++i) __stcs(to + (size_t)i * P, v[(i - 1) * S + l]);
    };
    if (!D2 && r.levels)
#pragma unroll
        for (int j = 0; j < SPT; ++j)
            if (fl[j] & S_ON) put_level(0, t + j * RES_NT, gs[j], p0[j], reinterpret_cast<const u64*>(lev));

    Waits waits = {r.wait_ns, false};
    const uint4* const mine = r.inbox + (size_t)blockIdx.x * 4 * r.recv_max;
    // sends the populations that leave the block at a site on its faces, with the stamp of step n
    auto send_faces = [&](unsigned f, unsigned place, int n, float2 v3, float2 v4, float2 v5, float2 v6) {
        const unsigned stamp = r.stamp0 + (unsigned)n;
        const size_t turn = (size_t)(n & 3) * r.recv_max;
        const int in = (int)(place & 0xffffu), ez = (int)(place >> 16);
        auto to = [&](int face, int e) {
            return r.packets + ((size_t)b.nbr[face] * 4 * r.recv_max + turn + b.dest[face] + e);
        };
        if (f & 64u) send(to(0, ez), v4, stamp);
        if (f & 128u) send(to(1, ez), v3, stamp);
        if (f & 256u) send(to(2, in), v6, stamp);
        if (f & 512u) send(to(3, in), v5, stamp);
        if (LK) {
            const int ly = nx * b.hz;
            if (f & 64u) send(to(0, ly + ez), v3, stamp);
            if (f & 128u) send(to(1, ly + ez), v4, stamp);
            if (f & 0x800u) send(to(0, 2 * ly + ez), v4, stamp);
            if (f & 0x1000u) send(to(1, 2 * ly + ez), v3, stamp);
            if (f & 256u) send(to(2, layer + in), v5, stamp);
            if (f & 512u) send(to(3, layer + in), v6, stamp);
            if (f & 0x2000u) send(to(2, 2 * layer + in), v6, stamp);
            if (f & 0x4000u) send(to(3, 2 * layer + in), v5, stamp);
        }
    };
    constexpr unsigned SEND = S_SEND | (LK ? S_SEND2 : 0u);
#pragma unroll
    for (int j = 0; j < SPT; ++j)
        if (fl[j] & SEND) {   // the values that the first step pulls
            const float2* v = lev + t + j * RES_NT;
            send_faces(fl[j], pl[j], 0, v[2 * S], v[3 * S], D2 ? v[0] : v[4 * S], D2 ? v[0] : v[5 * S]);
        }

    for (int n = 0; n < r.n_steps; ++n) {
        const int k = r.k0 + n;
        float2* const cur = lev + (n & 1) * lsz;
        float2* const nxt = lev + ((n & 1) ^ 1) * lsz;
        // the next step's factors and waveform value
        float2 fnext = make_float2(0.f, 0.f);
        if (n + 1 < r.n_steps) {
            if (t < 6) fnext = __ldg(a.fac + ((size_t)(k + 1) * a.n_members + b.m) * 6 + t);
            if (t == 6) fnext.x = __ldg(d->fw + k + 1);
        }
        // the neighbours' face values, two polls in flight a thread
        {
            const unsigned stamp = r.stamp0 + (unsigned)n;
            const uint4* box = mine + (size_t)(n & 3) * r.recv_max;
            for (int e = t; e < b.n_recv; e += 2 * RES_NT) {
                const bool two = e + RES_NT < b.n_recv;
                uint4 p = peek(box + e), q = two ? peek(box + e + RES_NT) : p;
                if (!(p.y == stamp && p.w == stamp)) p = await(box + e, stamp, waits);
                cur[NP * S + e] = make_float2(__uint_as_float(p.x), __uint_as_float(p.z));
                if (two) {
                    if (!(q.y == stamp && q.w == stamp)) q = await(box + e + RES_NT, stamp, waits);
                    cur[NP * S + e + RES_NT] = make_float2(__uint_as_float(q.x), __uint_as_float(q.z));
                }
            }
        }
        __syncthreads();   // the level, its face values and the factors are complete
        const float2* fac = s_fac[n & 1];
        const float f = s_f[n & 1];
        if (LK) {   // the listed links, one a thread
            for (int e = t; e < s_links; e += RES_NT) {
                const LinkEntry L = lent[e];
                float2 v[6];
#pragma unroll
                for (int q = 0; q < 6; ++q) v[q] = cur[L.at[q]];
                if (L.face)
#pragma unroll
                    for (int q = 0; q < 6; ++q) {
                        const unsigned c = L.face >> (4 * q) & 15u;
                        if (c & 8u) v[q].y = -v[q].y;
                        if (c) v[q] = turn(v[q], fac[(c & 7u) - 1u]);
                    }
                lres[e] = link_sum(L.A, L.B, v[0], v[1], v[2], v[3], v[4], v[5]);
            }
            __syncthreads();
        }
        const bool do_sig = k == sig, do_fld = field != nullptr && k == fstep;
#pragma unroll
        for (int j = 0; j < SPT; ++j) {
            const int l = t + j * RES_NT;
            const unsigned F = fl[j];
            if (!(F & S_ON)) continue;
            const u64* const cur2 = reinterpret_cast<const u64*>(cur);
            const u64* c = cur2 + l;
            u64 g[NP + 1];
            g[0] = p0[j];
            // x: the block spans the axis
            g[1] = (F & 1u) ? (bc[0] == BC_PER ? c[nx - 1] : c[S]) : c[-1];
            g[2] = (F & 2u) ? (bc[0] == BC_PER ? c[S - (nx - 1)] : c[0]) : c[S + 1];
            g[3] = cur2[oy[j] & 0xffffu];
            g[4] = cur2[oy[j] >> 16];
            if (!D2) {
                g[NP - 1] = cur2[oz[j] & 0xffffu];
                g[NP] = cur2[oz[j] >> 16];
            }
            if (F & S_GRID) {
                if (F & 1u) g[1] = face2(g[1], bc[0], fac[0]);
                if (F & 2u) g[2] = face2(g[2], bc[0], fac[1]);
                if (F & 4u) g[3] = face2(g[3], bc[1], fac[2]);
                if (F & 8u) g[4] = face2(g[4], bc[1], fac[3]);
                if (!D2) {
                    if (F & 16u) g[NP - 1] = face2(g[NP - 1], bc[2], fac[4]);
                    if (F & 32u) g[NP] = face2(g[NP], bc[2], fac[5]);
                }
            }
            if (F & 0x3f0000u) {   // half-link membranes (Eq. B5)
                mix_if<0x20000u>(F, g[1], c[S], sh2);
                mix_if<0x10000u>(F, g[2], c[0], sh2);
                mix_if<0x80000u>(F, g[3], c[3 * S], sh2);
                mix_if<0x40000u>(F, g[4], c[2 * S], sh2);
                if (!D2) {
                    mix_if<0x200000u>(F, g[NP - 1], c[5 * S], sh2);
                    mix_if<0x100000u>(F, g[NP], c[4 * S], sh2);
                }
            }
            if (LK && lk[j]) {
                const u64* res = reinterpret_cast<const u64*>(lres) + (lk[j] & 0xffffu);
#pragma unroll
                for (int i = 1; i <= NP; ++i)
                    if (lk[j] & (0x10000u << i)) g[i] = *res++;
            }
            float2 q;
            if (GEN && f != 0.f && f != 1.f && f != -1.f) {   // rotation_m1's general form
                float sn, cs;
                sincosf(0.5f * __fmul_rn(f, thg[j]), &sn, &cs);
                q = make_float2(__fmul_rn(-2.f, __fmul_rn(sn, sn)), __fmul_rn(2.f, __fmul_rn(sn, cs)));
            } else {
                const float2 v = rots[l];
                q = make_float2(__fmul_rn(v.x, fabsf(f)), __fmul_rn(v.y, f));
            }
            const float2 pe = s_phase[F >> 22 & 3u];
            const u64 M = react_collide(g, reaction_q(q, pe.y), pe.x, a.w0, a.wxy);
            p0[j] = g[0];
            // the faces first: a neighbour waits for them (nobody after the last step)
            if ((F & SEND) && n + 1 < r.n_steps) 
                send_faces(F, pl[j], n + 1, unpk(g[3]), unpk(g[4]), unpk(g[NP - 1]), unpk(g[NP]));
#pragma unroll
            for (int i = 1; i <= NP; ++i) reinterpret_cast<u64*>(nxt)[(i - 1) * S + l] = g[i];
            if (!D2 && r.levels && n + 1 < r.n_steps) put_level(n + 1, l, gs[j], g[0], reinterpret_cast<const u64*>(nxt));
            if (do_sig || do_fld || r.mser) {
                const float2 v = unpk(M);
                if (do_sig) mout[gs[j]] = v;
                if (do_fld) field[gs[j]] = v;
                if (r.mser) r.mser[(size_t)n * r.mstride + d->moff + gs[j]] = v;
            }
        }
        if (t < 6) s_fac[(n & 1) ^ 1][t] = fnext;
        if (t == 6) s_f[(n & 1) ^ 1] = fnext.x;
    }

    // each site's values are this thread's own
    float2* __restrict__ dst = d->state + (size_t)r.ldst * 7 * P;
    const float2* __restrict__ end = lev + (r.n_steps & 1) * lsz;
#pragma unroll
    for (int j = 0; j < SPT; ++j) {
        const int l = t + j * RES_NT;
        if (!(fl[j] & S_ON)) continue;
        dst[gs[j]] = unpk(p0[j]);
#pragma unroll
        for (int i = 1; i <= NP; ++i) dst[(size_t)i * P + gs[j]] = end[(i - 1) * S + l];
        if (D2)
            for (int i = 5; i < Q; ++i) dst[(size_t)i * P + gs[j]] = make_float2(0.f, 0.f);
    }
    if (waits.dead) atomicOr(&a.ctl->err, 1);
}

// Parts of Z per member (out[m][parts]) from the magnetisation M of its sites,
// with the thread sums of the one-step sweep that the grid would otherwise take
// (FP32 over a thread's few sites, FP64 above), so that a signal does not
// depend on which sweep ran: the register sweep's thread has sites s, s + block,
// .. of a tile of block x spt, the bulk-copy sweep's l, l + block, .. of a unit of
// rpu rows.
__device__ __forceinline__ void signal_part(const MemberDesc& d, const float2* __restrict__ M, int rows, int block, int spt,
                                            int part, int parts, double2* out)
{
    __shared__ double2 sh[256];
    const long long N = d.N;
    // units of a plane (rows != 0) or tiles of the whole grid
    const long long span = rows ? (long long)d.nx * d.ny : N;
    const int unit = rows ? d.rpu * d.nx : block * spt;
    const long long per = (span + unit - 1) / unit, n_units = per * (N / span);
    double2 v = make_double2(0.0, 0.0);
    for (long long u = part; u < n_units; u += parts) {
        const long long s0 = (u / per) * span + (u % per) * unit, s1 = min(s0 + unit, (u / per + 1) * span);
        for (int t = threadIdx.x; t < block; t += 256) {
            float zr = 0.f, zi = 0.f;
            for (int j = 0; j < spt; ++j) {
                const long long s = s0 + t + (long long)j * block;
                if (s < s1) {
                    const float2 m = M[s];
                    zr += m.x;
                    zi += m.y;
                }
            }
            v.x += zr;
            v.y += zi;
        }
    }
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            sh[threadIdx.x].x += sh[threadIdx.x + o].x;
            sh[threadIdx.x].y += sh[threadIdx.x + o].y;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = sh[0];
}

__global__ void signal_kernel(const MemberDesc* __restrict__ members, int rows, int block, int spt,
                              double2* __restrict__ out)
{
    const MemberDesc& d = members[blockIdx.x];
    signal_part(d, d.mout, rows, block, spt, blockIdx.y, gridDim.y, out + (size_t)blockIdx.x * gridDim.y + blockIdx.y);
}

// The same of every step of a launch: blocks (member, part) x step.
__global__ void series_part_kernel(const MemberDesc* __restrict__ members, int rows, int block, int spt, int parts,
                                   const float2* __restrict__ mser, long long mstride, double2* __restrict__ zpart)
{
    const int m = blockIdx.x / parts, part = blockIdx.x - m * parts;
    const MemberDesc& d = members[m];
    signal_part(d, mser + (size_t)blockIdx.y * mstride + d.moff, rows, block, spt, part, parts,
                zpart + (size_t)blockIdx.y * gridDim.x + blockIdx.x);
}

// series[m][k0 + n] = sum of the member's parts of step n (one warp each).
__global__ void resident_series_kernel(const double2* __restrict__ zpart, const int* __restrict__ block_start,
                                       int n_members, int n_blocks, int n_steps, long long k0, long long stride,
                                       double2* __restrict__ series)
{
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w >= n_members * n_steps) return;
    const int m = w / n_steps, n = w - m * n_steps;
    double2 v = make_double2(0.0, 0.0);
    for (int b = block_start[m] + lane; b < block_start[m + 1]; b += 32) {
        const double2 p = zpart[(size_t)n * n_blocks + b];
        v.x += p.x;
        v.y += p.y;
    }
    for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_down_sync(0xffffffffu, v.x, o);
        v.y += __shfl_down_sync(0xffffffffu, v.y, o);
    }
    if (lane == 0) series[m * stride + k0 + n] = v;
}

using ResFn = void (*)(const SweepArgs, const ResArgs);

template <bool D2, bool GEN, bool LK>
ResFn res_spt(int spt)
{
    return spt <= 1 ? sweep_resident_kernel<1, D2, GEN, LK>
           : spt <= 2 ? sweep_resident_kernel<2, D2, GEN, LK> : sweep_resident_kernel<4, D2, GEN, LK>;
}
template <bool D2>
ResFn res_kernel(int spt, bool gen, bool links)
{
    if (links) return res_spt<D2, true, true>(spt);   // the general waveform form covers the others
    return gen ? res_spt<D2, true, false>(spt) : res_spt<D2, false, false>(spt);
}

}  // namespace

int resident_max_sites() { return RES_MAX_SITES; }
size_t resident_link_bytes() { return sizeof(LinkEntry) + sizeof(float2); }
cudaError_t launch_resident_links(const MemberDesc* members, const ResBlock* blocks, int n_blocks, bool d2, int* out,
                                  cudaStream_t st)
{
    resident_links_kernel<<<n_blocks, 256, 0, st>>>(members, blocks, d2 ? 4 : 6, out);
    return cudaGetLastError();
}

size_t resident_smem(int sites, int recv, bool d2) { return ((size_t)(d2 ? 9 : 13) * sites + 2 * recv) * sizeof(float2); }

cudaError_t launch_resident(const SweepArgs& a, const ResArgs& r, int n_blocks, int max_sites, size_t smem, bool d2,
                            bool general, cudaStream_t st)
{
    const int spt = (max_sites + RES_NT - 1) / RES_NT;
    const void* fn = (const void*)(d2 ? res_kernel<true>(spt, general, r.links) : res_kernel<false>(spt, general, r.links));
    const cudaError_t e = allow_smem(fn, smem);
    if (e != cudaSuccess) return e;
    SweepArgs aa = a;
    ResArgs rr = r;
    void* args[2] = {&aa, &rr};
    return cudaLaunchCooperativeKernel(fn, dim3(n_blocks), dim3(RES_NT), args, smem, st);
}

cudaError_t launch_signal(const MemberDesc* members, int n_members, bool rows, int block, int spt, int parts, double2* out,
                          cudaStream_t st)
{
    signal_kernel<<<dim3(n_members, parts), 256, 0, st>>>(members, rows ? 1 : 0, block, spt, out);
    return cudaGetLastError();
}

cudaError_t launch_series_parts(const MemberDesc* members, int n_members, bool rows, int block, int spt, int parts,
                                const float2* mser, long long mstride, int n_steps, double2* zpart, cudaStream_t st)
{
    series_part_kernel<<<dim3((unsigned)(n_members * parts), (unsigned)n_steps), 256, 0, st>>>(members, rows ? 1 : 0, block, spt,
                                                                                              parts, mser, mstride, zpart);
    return cudaGetLastError();
}

cudaError_t launch_resident_series(const double2* zpart, const int* block_start, int n_members, int n_blocks, int n_steps,
                                   long long k0, long long stride, double2* series, cudaStream_t st)
{
    const long long warps = (long long)n_members * n_steps;
    resident_series_kernel<<<(unsigned)((warps + 7) / 8), 256, 0, st>>>(zpart, block_start, n_members, n_blocks, n_steps,
                                                                        k0, stride, series);
    return cudaGetLastError();
}

}  // namespace lbmbt
