// adjoint_resident.cu -- the adjoint steps of a segment in one launch, for grids
// that fit on chip (blocks, packets and their protocol: sweep_resident.cu).
//
// A step nu^k -> nu^(k-1) of a small grid took 17 us at 48^3, nearly all of it
// launch and copy latency.  Here the adjoint state stays in shared memory and
// only its face values travel; the forward levels u^(k-1), which lie in memory,
// do not depend on it and are copied (cp.async) a step ahead.
//
// The transposed stream is the forward stream of the opposite populations: with
// A_i = nu_ibar (ibar the opposite of i), lambda_j(y), which is nu_j of the
// consumer at y + e_j, is what the forward sweep pulls as population jbar from A,
// with the same membrane mixing (own A_j = nu_jbar), the same mirror (the own
// opposite population) and the same boundary factors of step k (conj exp(i phi) of
// one face is exp(-i phi) of the other).  So one gather serves both: u^(k-1) with
// the factors of step k - 1, A with those of step k.  Derivation of the rest:
// adjoint.cu.
//
// The three sensitivities of every site and step go to memory (12 B), and a
// second kernel sums them in the groups and the order of the bulk-copy adjoint
// that the grid would otherwise take, so that a gradient does not depend on which
// adjoint ran.
//
// 48^3, 400 steps, checkpoint every 64: signal and gradient 5.8 ms against 15.0.
#include <algorithm>

#include "lbmbt_internal.cuh"
#include "sweep_common.cuh"
#include "packed.cuh"
#include "packets.cuh"

namespace lbmbt {
namespace {

constexpr int NT = 512;
constexpr int NP = 6;

__device__ __forceinline__ void copy8(u64* dst, const u64* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// Transform of a value pulled across a face (face_fix()), its roundings written
// out as they come out of the compiler in the bulk-copy adjoint, so that the
// gradients are the same numbers: `late` is the form of the transposed pulls
// across a periodic face.
__device__ __forceinline__ u64 face_turn(u64 p, int bc, float2 f, bool late)
{
    if (bc == BC_MIR) return p;
    float2 v = unpk(p);
    if (bc == BC_MIR_CONJ) {
        v.y = -v.y;
        late = false;
    }
    const float re = __fmaf_rn(v.x, f.x, -__fmul_rn(v.y, f.y));
    const float im = late ? __fmaf_rn(v.y, f.x, __fmul_rn(v.x, f.y)) : __fmaf_rn(v.x, f.y, __fmul_rn(v.y, f.x));
    return pk(re, im);
}

template <int SPT, bool GEN>
__global__ void __launch_bounds__(NT, 1) adjoint_resident_kernel(const AdjointArgs a, const ResArgs r)
{
    extern __shared__ __align__(16) unsigned char adj_smem[];
    __shared__ float2 s_fac[3][6];   // factors of steps k - 1, k and, next, k - 2 (index step % 3)
    __shared__ float2 s_phase[4];

    const int t = threadIdx.x;
    const ResBlock b = r.blocks[blockIdx.x];
    const MemberDesc* __restrict__ d = a.members + b.m;
    const int nx = d->nx, ny = d->ny, nz = d->nz;
    const int S = nx * b.hy * b.hz, layer = nx * b.hy;
    const int lsz = NP * S + b.n_recv;             // a level of A, and of u (then population 0)
    u64* const lev = reinterpret_cast<u64*>(adj_smem);          // [2][lsz] A_1 .. A_6, received values
    u64* const ulv = lev + 2 * lsz;                             // [2][lsz + S] u_1 .. u_6, face values, u_0
    float2* const rots = reinterpret_cast<float2*>(ulv + 2 * (lsz + S));
    const unsigned P = (unsigned)d->plane, sxy = (unsigned)nx * ny;
    const int bc[3] = {d->bc[0], d->bc[1], d->bc[2]};
    const float sh = d->s_share;
    const u64 sh2 = pk(sh, sh);
    float2 sL = make_float2(0.f, 0.f);
    if (a.first) {
        const double2 L = a.lam_init[b.m];
        sL = make_float2((float)L.x, (float)L.y);
    }
    if (t < 4) s_phase[t] = make_float2(d->omega[t], d->eps[t]);

    unsigned gs[SPT], fl[SPT], pl[SPT], oy[SPT], oz[SPT];
    u64 a0[SPT];
    float thg[SPT];
    const u64* __restrict__ nu_in = reinterpret_cast<const u64*>(d->adj + (size_t)r.lsrc * 7 * P);
#pragma unroll
    for (int j = 0; j < SPT; ++j) {
        const int l = t + j * NT;
        gs[j] = fl[j] = pl[j] = oy[j] = oz[j] = 0u;
        a0[j] = 0ull;
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
            auto from = [&](bool face, int nb, int step, int wrap, int pop, int opp, int recv) -> unsigned {
                if (!face) return (unsigned)((pop - 1) * S + l + step);
                if (nb >= 0) return (unsigned)(NP * S + recv);
                return (unsigned)(nb == RES_SELF ? (pop - 1) * S + l + wrap : (opp - 1) * S + l);
            };
            const int wy = (b.hy - 1) * nx, wz = (b.hz - 1) * layer;
            oy[j] = from(yl, b.nbr[0], -nx, wy, 3, 4, b.recv[0] + ez) | (from(yh, b.nbr[1], nx, -wy, 4, 3, b.recv[1] + ez) << 16);
            oz[j] = from(zl, b.nbr[2], -layer, wz, 5, 6, b.recv[2] + in) |
                    (from(zh, b.nbr[3], layer, -wz, 6, 5, b.recv[3] + in) << 16);
            rots[l] = rotation_m1(d, 1.f, x, gy, gz);
            if (GEN) thg[j] = __fmaf_rn(d->ctheta[2], (float)(gz + d->z0),
                                        __fmaf_rn(d->ctheta[1], (float)gy, __fmul_rn(d->ctheta[0], (float)x)));
            if (!a.first) {
                a0[j] = __ldcg(nu_in + s);
#pragma unroll
                for (int i = 1; i <= NP; ++i)
                    lev[(i - 1) * S + l] = __ldcg(nu_in + (size_t)((i & 1) ? i + 1 : i - 1) * P + s);
            }
        }
    }
    // copies the forward level in slot `slot` (own sites and the neighbours' face values)
    auto load_u = [&](int slot, u64* to) {
        const u64* from = reinterpret_cast<const u64*>(d->state + (size_t)slot * 7 * P);
#pragma unroll
        for (int j = 0; j < SPT; ++j) {
            const int l = t + j * NT;
            if (!(fl[j] & S_ON)) continue;
            copy8(to + lsz + l, from + gs[j]);
#pragma unroll
            for (int i = 1; i <= NP; ++i) copy8(to + (i - 1) * S + l, from + (size_t)i * P + gs[j]);
            // what this site pulls across the block's faces
            const int in = (int)(pl[j] & 0xffffu), ez = (int)(pl[j] >> 16);
            if (fl[j] & 64u) copy8(to + NP * S + b.recv[0] + ez, from + (size_t)3 * P + (fl[j] & 4u ? gs[j] + (sxy - nx) : gs[j] - nx));
            if (fl[j] & 128u) copy8(to + NP * S + b.recv[1] + ez, from + (size_t)4 * P + (fl[j] & 8u ? gs[j] - (sxy - nx) : gs[j] + nx));
            if (fl[j] & 256u)
                copy8(to + NP * S + b.recv[2] + in, from + (size_t)5 * P + (fl[j] & 16u ? gs[j] + (unsigned)(nz - 1) * sxy : gs[j] - sxy));
            if (fl[j] & 512u)
                copy8(to + NP * S + b.recv[3] + in, from + (size_t)6 * P + (fl[j] & 32u ? gs[j] - (unsigned)(nz - 1) * sxy : gs[j] + sxy));
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto factors = [&](int k) { return __ldg(a.ftab + ((size_t)k * a.n_members + b.m) * 6 + t); };

    Waits waits = {r.wait_ns, false};
    const uint4* const mine = r.inbox + (size_t)blockIdx.x * 4 * r.recv_max;
    auto send_faces = [&](unsigned f, unsigned place, int n, u64 v3, u64 v4, u64 v5, u64 v6) {
        const unsigned stamp = r.stamp0 + (unsigned)n;
        const size_t turn = (size_t)(n & 3) * r.recv_max;
        const int in = (int)(place & 0xffffu), ez = (int)(place >> 16);
        auto to = [&](int face, int e) {
            return r.packets + ((size_t)b.nbr[face] * 4 * r.recv_max + turn + b.dest[face] + e);
        };
        if (f & 64u) send(to(0, ez), unpk(v4), stamp);
        if (f & 128u) send(to(1, ez), unpk(v3), stamp);
        if (f & 256u) send(to(2, in), unpk(v6), stamp);
        if (f & 512u) send(to(3, in), unpk(v5), stamp);
    };
    // steps n = 0 .. n_steps - 1 are k = k0 - n (nu^k -> nu^(k-1)); u^(k-1) is in slot lsrc0 - n
    load_u(a.fwd_slot, ulv);
    if (t < 6) {
        s_fac[a.k % 3][t] = factors(a.k);
        s_fac[(a.k + 2) % 3][t] = factors(a.k - 1);
    }
    if (!a.first)
#pragma unroll
        for (int j = 0; j < SPT; ++j)
            if (fl[j] & S_SEND) {
                const u64* v = lev + t + j * NT;
                send_faces(fl[j], pl[j], 0, v[2 * S], v[3 * S], v[4 * S], v[5 * S]);
            }
    const size_t N = (size_t)d->N;
    float* const gsite = reinterpret_cast<float*>(d->field);   // [step][3][N]

    for (int n = 0; n < r.n_steps; ++n) {
        const int k = a.k - n;
        const bool first = a.first && n == 0;
        u64* const cur = lev + (n & 1) * lsz;
        u64* const nxt = lev + ((n & 1) ^ 1) * lsz;
        const u64* const u = ulv + (n & 1) * (lsz + S);
        float2 fnext = make_float2(0.f, 0.f);
        const bool more = n + 1 < r.n_steps;
        if (more && t < 6) fnext = factors(k - 2);
        const float f = __ldg(d->fw + k - 1);
        if (!first) {   // the neighbours' face values
            const unsigned stamp = r.stamp0 + (unsigned)n;
            const uint4* box = mine + (size_t)(n & 3) * r.recv_max;
            for (int e = t; e < b.n_recv; e += NT) {
                uint4 p = peek(box + e);
                if (!(p.y == stamp && p.w == stamp)) p = await(box + e, stamp, waits);
                cur[NP * S + e] = pk(__uint_as_float(p.x), __uint_as_float(p.z));
            }
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();   // both levels and the factors are complete
        if (more) load_u(a.fwd_slot - n - 1, ulv + ((n & 1) ^ 1) * (lsz + S));
        const float2* facK = s_fac[k % 3];
        const float2* facP = s_fac[(k + 2) % 3];
#pragma unroll
        for (int j = 0; j < SPT; ++j) {
            const int l = t + j * NT;
            const unsigned F = fl[j];
            if (!(F & S_ON)) continue;
            // pulls of populations 1..6 from a level, before (pre) and after the membranes
            auto gather = [&](const u64* v, const float2* fac, u64 (&g)[Q], bool mixed, bool late) {
                const u64* c = v + l;
                g[1] = (F & 1u) ? (bc[0] == BC_PER ? c[nx - 1] : c[S]) : c[-1];
                g[2] = (F & 2u) ? (bc[0] == BC_PER ? c[S - (nx - 1)] : c[0]) : c[S + 1];
                g[3] = v[oy[j] & 0xffffu];
                g[4] = v[oy[j] >> 16];
                g[5] = v[oz[j] & 0xffffu];
                g[6] = v[oz[j] >> 16];
                if (F & S_GRID) {
                    if (F & 1u) g[1] = face_turn(g[1], bc[0], fac[0], late);
                    if (F & 2u) g[2] = face_turn(g[2], bc[0], fac[1], late);
                    if (F & 4u) g[3] = face_turn(g[3], bc[1], fac[2], late);
                    if (F & 8u) g[4] = face_turn(g[4], bc[1], fac[3], late);
                    if (F & 16u) g[5] = face_turn(g[5], bc[2], fac[4], late);
                    if (F & 32u) g[6] = face_turn(g[6], bc[2], fac[5], late);
                }
                if (mixed && (F & 0x3f0000u)) {
                    mix_if<0x20000u>(F, g[1], c[S], sh2);
                    mix_if<0x10000u>(F, g[2], c[0], sh2);
                    mix_if<0x80000u>(F, g[3], c[3 * S], sh2);
                    mix_if<0x40000u>(F, g[4], c[2 * S], sh2);
                    mix_if<0x200000u>(F, g[5], c[5 * S], sh2);
                    mix_if<0x100000u>(F, g[6], c[4 * S], sh2);
                }
            };
            u64 gu[Q], lm[Q];   // g'^(k-1); lambda^k in the order of A (lm[i] = lambda_ibar)
            gu[0] = u[lsz + l];
            gather(u, facP, gu, true, false);
            if (first) {
#pragma unroll
                for (int i = 0; i < Q; ++i) lm[i] = pk(sL.x, sL.y);
            } else {
                lm[0] = a0[j];
                gather(cur, facK, lm, true, true);
            }
            float2 gp[Q], lam[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                gp[i] = unpk(gu[i]);
                lam[i] = unpk(lm[i == 0 ? 0 : (i & 1) ? i + 1 : i - 1]);
            }
            const float2 pe = s_phase[F >> 22 & 3u];
            const float om = pe.x, ep = pe.y;
            float2 rot;
            if (GEN && f != 0.f && f != 1.f && f != -1.f) {   // rotation_m1's general form
                float sn, cs;
                sincosf(0.5f * __fmul_rn(f, thg[j]), &sn, &cs);
                rot = make_float2(__fmul_rn(-2.f, __fmul_rn(sn, sn)), __fmul_rn(2.f, __fmul_rn(sn, cs)));
            } else {
                const float2 v = rots[l];
                rot = make_float2(__fmul_rn(v.x, fabsf(f)), __fmul_rn(v.y, f));
            }
            const float2 q = reaction_q(rot, ep);
            // as adjoint_tma_kernel, expression by expression and rounding by rounding
            float sgr = 0.f, sgi = 0.f, dr = 0.f, di = 0.f, lwr = 0.f, lwi = 0.f;
#pragma unroll
            for (int i2 = 0; i2 < Q; ++i2) {
                const float w = i2 == 0 ? W0 : WI;
                sgr += gp[i2].x;
                sgi += gp[i2].y;
                dr += lam[i2].x * gp[i2].x + lam[i2].y * gp[i2].y;
                di += lam[i2].x * gp[i2].y - lam[i2].y * gp[i2].x;
                lwr += w * lam[i2].x;
                lwi += w * lam[i2].y;
            }
            const float q1r = 1.f + q.x, q1i = q.y;
            const float Mr = q1r * sgr - q1i * sgi, Mi = q1r * sgi + q1i * sgr;
            const float dOm = (lwr * Mr + lwi * Mi) - (q1r * dr - q1i * di);
            const float om1 = 1.f - om;
            const float er = 1.f + rot.x, ei = rot.y;
            const float xr = __fmaf_rn(lwr, sgr, __fmul_rn(lwi, sgi)), xi = __fmaf_rn(lwr, sgi, -__fmul_rn(lwi, sgr));
            const float cr = __fmaf_rn(om, xr, __fmul_rn(om1, dr)), ci = __fmaf_rn(om, xi, __fmul_rn(om1, di));
            const float dEp = -__fmaf_rn(er, cr, -__fmul_rn(ei, ci));
            const float ar = q1r * om1, ai = -q1i * om1;
            const float br = om * (q1r * lwr + q1i * lwi), bi = om * (q1r * lwi - q1i * lwr);
#pragma unroll
            for (int i2 = 0; i2 < Q; ++i2) {
                const float2 l2 = lam[i2];
                lam[i2] = make_float2(ar * l2.x - ai * l2.y + br, ar * l2.y + ai * l2.x + bi);
                lm[i2 == 0 ? 0 : (i2 & 1) ? i2 + 1 : i2 - 1] = pk(lam[i2].x, lam[i2].y);   // order of A
            }
            a0[j] = lm[0];
            if ((F & S_SEND) && more) send_faces(F, pl[j], n + 1, lm[3], lm[4], lm[5], lm[6]);
#pragma unroll
            for (int i = 1; i <= NP; ++i) nxt[(i - 1) * S + l] = lm[i];
            float dS = 0.f;
            if (F & 0x3f0000u) {   // d/d s: <nu_i, v_i - o_i> on membrane links
                gather(u, facP, gu, false, false);
                const u64* c = u + l;
                const unsigned bitof[Q] = {0u, 0x20000u, 0x10000u, 0x80000u, 0x40000u, 0x200000u, 0x100000u};
#pragma unroll
                for (int i2 = 1; i2 < Q; ++i2)
                    if (F & bitof[i2]) {
                        const float2 vpre = unpk(gu[i2]), own = unpk(c[(((i2 & 1) ? i2 + 1 : i2 - 1) - 1) * S]);
                        dS += lam[i2].x * (vpre.x - own.x) + lam[i2].y * (vpre.y - own.y);
                    }
            }
            float* const to = gsite + (size_t)n * 3 * N + gs[j];
            __stcs(to, dOm);
            __stcs(to + N, dEp);
            __stcs(to + 2 * N, dS);
        }
        if (more && t < 6) s_fac[(k + 1) % 3][t] = fnext;   // step k - 2 takes the place of k + 1
    }

    u64* __restrict__ nu_out = reinterpret_cast<u64*>(d->adj + (size_t)r.ldst * 7 * P);
    const u64* __restrict__ end = lev + (r.n_steps & 1) * lsz;
#pragma unroll
    for (int j = 0; j < SPT; ++j) {
        const int l = t + j * NT;
        if (!(fl[j] & S_ON)) continue;
        nu_out[gs[j]] = a0[j];
#pragma unroll
        for (int i = 1; i <= NP; ++i) nu_out[(size_t)((i & 1) ? i + 1 : i - 1) * P + gs[j]] = end[(i - 1) * S + l];
    }
    if (waits.dead) atomicOr(a.ctl_err, 1);
}

// The gradient partials of n_steps adjoint steps from the sites' sensitivities, as
// the bulk-copy adjoint of this grid sums them: per thread in FP32 over the units
// of a member that a CTA walks, over the warp, and per step in FP64 into the slot
// of (the run's first unit, warp).
__global__ void adjoint_sum_kernel(const AdjointArgs a, long long n_units, int n_steps, int spt, int slots)
{
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    for (int n = 0; n < n_steps; ++n) {
        float acc[NGACC];
#pragma unroll
        for (int q = 0; q < NGACC; ++q) acc[q] = 0.f;
        int m_run = -1;
        long long u_run = -1;
        auto flush = [&]() {
#pragma unroll
            for (int q = 0; q < NGACC; ++q)
                for (int o = 16; o > 0; o >>= 1) acc[q] += __shfl_down_sync(0xffffffffu, acc[q], o);
            if (lane == 0) {
                double* g = a.gacc + ((size_t)u_run * slots + warp) * NGACC;
#pragma unroll
                for (int q = 0; q < NGACC; ++q) g[q] += (double)acc[q];
            }
#pragma unroll
            for (int q = 0; q < NGACC; ++q) acc[q] = 0.f;
        };
        for (long long u = blockIdx.x; u < n_units; u += gridDim.x) {
            const UnitGeo G = unit_geo(a.members, a.unit_start, a.n_members, u, true);
            if (G.m != m_run) {
                if (m_run >= 0) flush();
                m_run = G.m;
                u_run = u;
            }
            const MemberDesc* __restrict__ d = a.members + G.m;
            const size_t N = (size_t)d->N;
            const float* __restrict__ from = reinterpret_cast<const float*>(d->field) + (size_t)n * 3 * N;
            for (int j = 0; j < spt; ++j) {
                const int l = t + j * (int)blockDim.x;
                if (l >= G.L) break;
                const unsigned s = G.s0 + (unsigned)l;
                const int ph = d->mask[s] >> 6;
                const float dOm = from[s], dEp = from[N + s];
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    acc[p] += (ph == p) ? dOm : 0.f;
                    acc[4 + p] += (ph == p) ? dEp : 0.f;
                }
                acc[8] += from[2 * N + s];
            }
        }
        if (m_run >= 0) flush();
    }
}

}  // namespace

int adj_resident_max_sites() { return 2 * NT; }
size_t adj_resident_smem(int sites, int recv) { return ((size_t)27 * sites + 4 * recv) * sizeof(float2); }

cudaError_t launch_adjoint_sum(const AdjointArgs& a, long long n_units, int n_steps, int grid, int threads, int spt,
                               int slots, cudaStream_t st)
{
    adjoint_sum_kernel<<<grid, threads, 0, st>>>(a, n_units, n_steps, spt, slots);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_resident(const AdjointArgs& a, const ResArgs& r, int n_blocks, int max_sites, size_t smem,
                                    bool general, cudaStream_t st)
{
    using Fn = void (*)(const AdjointArgs, const ResArgs);
    const Fn k = max_sites <= NT ? (general ? adjoint_resident_kernel<1, true> : adjoint_resident_kernel<1, false>)
                                 : (general ? adjoint_resident_kernel<2, true> : adjoint_resident_kernel<2, false>);
    const void* fn = (const void*)k;
    const cudaError_t e = allow_smem(fn, smem);
    if (e != cudaSuccess) return e;
    AdjointArgs aa = a;
    ResArgs rr = r;
    void* args[2] = {&aa, &rr};
    return cudaLaunchCooperativeKernel(fn, dim3(n_blocks), dim3(NT), args, smem, st);
}

}  // namespace lbmbt
