// sweep_strip.cu -- the resident sweep of 2-D grids too large for sweep_resident.cu:
// all steps of a D2Q5 run in one cooperative launch, state on chip.
//
// A 1000 x 1000 slice took 31 us a step, launched twice a step, on a state of
// 80 MB that L2 just holds.  One time level is 40 MB, and the SMs' shared memory
// and registers together hold that: a block is a strip of at most eight whole
// rows, a thread has two or three columns of it, populations 1-4 lie in shared
// memory (32 B a site, one level, updated in place) and the rest population in
// registers.
//
// In place: the rows of a strip are done in order.  The population that arrives
// from the row before is kept in a register as that row is overwritten; the one
// from the row ahead is still the old one; the x neighbours' are read before a
// block barrier and overwritten after it.  Odd steps go down the strip and even
// steps up, so each face value is sent (stamped packets, packets.cuh) a whole
// pass before the neighbour needs it, and the trip through L2 costs nothing.
// A packet is polled by the thread of its column, and that thread sends the
// column's packets back, so the argument of sweep_resident.cu that a packet
// is read before it is overwritten holds column by column.
//
// Arithmetic and order per site are those of the register sweep (same bits).
// 1000 x 1000, 800 steps: 11.4 us a step against 31.
#include "lbmbt_internal.cuh"
#include "sweep_common.cuh"
#include "packed.cuh"
#include "packets.cuh"

namespace lbmbt {
namespace {

constexpr int NT = 512;

// Puts v in place of the front (up) or back value and turns the values by one.
template <int ROWS>
__device__ __forceinline__ void turn_rest(u64 (&p)[ROWS], u64 v, bool up)
{
    if (up) {
#pragma unroll
        for (int i = 0; i + 1 < ROWS; ++i) p[i] = p[i + 1];
        p[ROWS - 1] = v;
    } else {
#pragma unroll
        for (int i = ROWS - 1; i > 0; --i) p[i] = p[i - 1];
        p[0] = v;
    }
}

// Thread t has the columns t + c NT, c < CPT, of at most ROWS rows; GEN: the
// waveform may take values other than 0 and +-1.
template <int CPT, int ROWS, bool GEN>
__global__ void __launch_bounds__(NT, 1) sweep_strip_kernel(const SweepArgs a, const ResArgs r)
{
    extern __shared__ __align__(16) unsigned char strip_smem[];
    __shared__ float2 s_phase[4];            // (omega, eps) per phase
    __shared__ float2 s_ey[ROWS];      // rotation of a row
    __shared__ float2 s_fac[2][6];           // boundary factors of this step and of the next
    __shared__ float s_f[2];
    __shared__ double2 s_red[NT / 32];

    const int t = threadIdx.x;
    const ResBlock b = r.blocks[blockIdx.x];
    const MemberDesc* __restrict__ d = a.members + b.m;
    const int nx = d->nx, ny = d->ny, hy = b.hy;
    u64* const lev = reinterpret_cast<u64*>(strip_smem);   // [4][hy][nx]: populations 1..4
    const int R = hy * nx;
    const unsigned P = (unsigned)d->plane;
    const u64* __restrict__ src = reinterpret_cast<const u64*>(d->state + (size_t)r.lsrc * 7 * P + (size_t)b.y0 * nx);
    const int bcx = d->bc[0], bcy = d->bc[1];
    const u64 sh2 = pk(d->s_share, d->s_share);
    const int es = d->end_step;
    const int sig = es >= 0 ? es : r.sig_step, fstep = es >= 0 ? es : r.field_step;
    const int axes = d->axes;
    float2* const field = d->field;
    float2* const mout = d->mout;
    const bool ylo = b.y0 == 0, yhi = b.y0 + hy == ny;           // strip at a face of the grid
    const int below = b.nbr[0], above = b.nbr[1];
    if (t < 4) s_phase[t] = make_float2(d->omega[t], d->eps[t]);
    if (t < hy) s_ey[t] = (axes & 2) ? __ldg(d->etab + nx + b.y0 + t) : make_float2(0.f, 0.f);

    // this thread's columns
    u64 p0[CPT][ROWS];
    float2 ex[CPT];
    unsigned long long mk[CPT];              // mask bytes of the rows
    const float cx = GEN ? d->ctheta[0] : 0.f, cy = GEN ? d->ctheta[1] : 0.f;
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
        const int x = t + c * NT;
        mk[c] = 0;
        ex[c] = make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < ROWS; ++q) p0[c][q] = 0ull;
        if (x >= nx) continue;
        if (axes & 1) ex[c] = __ldg(d->etab + x);
#pragma unroll
        for (int q = 0; q < ROWS; ++q) {
            if (q >= hy) break;
            const unsigned s = (unsigned)q * nx + x;
            mk[c] |= (unsigned long long)d->mask[(size_t)b.y0 * nx + s] << (8 * q);
            p0[c][q] = __ldcg(src + s);
#pragma unroll
            for (int i = 1; i <= 4; ++i) lev[(i - 1) * R + s] = __ldcg(src + (size_t)i * P + s);
        }
    }

    if (t < 6) s_fac[0][t] = __ldg(a.fac + ((size_t)r.k0 * a.n_members + b.m) * 6 + t);
    if (t == 6) s_f[0] = __ldg(d->fw + r.k0);

    Waits waits = {r.wait_ns, false};
    const uint4* const mine = r.inbox + (size_t)blockIdx.x * 4 * r.recv_max;
    // own packets: [turn][0: from below, 1: from above][nx]
    auto receive = [&](int n, int face, int x) {
        const uint4* from = mine + (size_t)(n & 3) * r.recv_max + b.recv[face] + x;
        const unsigned stamp = r.stamp0 + (unsigned)n;
        uint4 p = peek(from);
        if (!(p.y == stamp && p.w == stamp)) p = await(from, stamp, waits);
        return pk(__uint_as_float(p.x), __uint_as_float(p.z));
    };
    auto post = [&](int n, int face, int x, u64 v) {
        send(r.packets + ((size_t)b.nbr[face] * 4 + (n & 3)) * r.recv_max + b.dest[face] + x, unpk(v), r.stamp0 + (unsigned)n);
    };
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
        const int x = t + c * NT;
        if (x >= nx) continue;
        if (below >= 0) post(0, 0, x, lev[3 * R + x]);
        if (above >= 0) post(0, 1, x, lev[2 * R + (hy - 1) * nx + x]);
    }
    __syncthreads();

    for (int n = 0; n < r.n_steps; ++n) {
        const int k = r.k0 + n;
        const float f = s_f[n & 1];
        const float2* fac = s_fac[n & 1];
        float2 fnext = make_float2(0.f, 0.f);   // the next step's
        if (n + 1 < r.n_steps) {
            if (t < 6) fnext = __ldg(a.fac + ((size_t)(k + 1) * a.n_members + b.m) * 6 + t);
            if (t == 6) fnext.x = __ldg(d->fw + k + 1);
        }
        const bool tab = !GEN || f == 0.f || f == 1.f || f == -1.f;
        const bool more = n + 1 < r.n_steps;
        const bool do_sig = k == sig, do_fld = field != nullptr && k == fstep;
        double zr = 0.0, zi = 0.0;
        // of the row done before: the old population that moves on; of the first
        // row done: the old one that a strip closed on itself needs at the end
        u64 carry[CPT], first[CPT];

        const bool UP = (n & 1) == 0;   // rows in rising order
        // The rest populations turn through their registers, so that the row loop
        // need not be unrolled (unrolled, its addresses spill): up from the front,
        // down from the back, past the rows that the strip does not have.
        auto skip = [&](bool upwards) {
#pragma unroll 1
            for (int q = hy; q < ROWS; ++q)
#pragma unroll
                for (int c = 0; c < CPT; ++c) turn_rest(p0[c], upwards ? p0[c][0] : p0[c][ROWS - 1], upwards);
        };
        if (!UP) skip(false);
#pragma unroll 1
        for (int j = 0; j < hy; ++j) {
            const int q = UP ? j : hy - 1 - j;
            const bool start = j == 0;
            u64 g1[CPT], g2[CPT], o1[CPT], o2[CPT];
#pragma unroll
            for (int c = 0; c < CPT; ++c) {
                const int x = t + c * NT;
                if (x >= nx) continue;
                const u64 *r1 = lev + q * nx, *r2 = lev + R + q * nx;
                o1[c] = r1[x];
                o2[c] = r2[x];
                if (x > 0) g1[c] = r1[x - 1];
                else g1[c] = face2(bcx == BC_PER ? r1[nx - 1] : o2[c], bcx, fac[0]);
                if (x < nx - 1) g2[c] = r2[x + 1];
                else g2[c] = face2(bcx == BC_PER ? r2[0] : o1[c], bcx, fac[1]);
            }
            __syncthreads();   // the row's x neighbours are read
#pragma unroll
            for (int c = 0; c < CPT; ++c) {
                const int x = t + c * NT;
                if (x >= nx) continue;
                u64* const r3 = lev + 2 * R + q * nx + x;
                u64* const r4 = lev + 3 * R + q * nx + x;
                const u64 o3 = *r3, o4 = *r4;
                u64 g[5];
                g[0] = UP ? p0[c][0] : p0[c][ROWS - 1];
                g[1] = g1[c];
                g[2] = g2[c];
                // the population along the pass comes from the row done before, the other
                // from the row ahead; at the ends of the strip from beyond it
                if (q == 0) {
                    g[3] = below >= 0 ? receive(n, 0, x) : below == RES_MIRROR ? o4 : UP ? lev[2 * R + (hy - 1) * nx + x] : first[c];
                    if (!UP && below == RES_SELF && hy == 1) g[3] = o3;
                    if (ylo) g[3] = face2(g[3], bcy, fac[2]);
                } else {
                    g[3] = UP ? carry[c] : *(r3 - nx);
                }
                if (q == hy - 1) {
                    g[4] = above >= 0 ? receive(n, 1, x) : above == RES_MIRROR ? o3 : !UP ? lev[3 * R + x] : first[c];
                    if (UP && above == RES_SELF && hy == 1) g[4] = o4;
                    if (yhi) g[4] = face2(g[4], bcy, fac[3]);
                } else {
                    g[4] = UP ? *(r4 + nx) : carry[c];
                }
                carry[c] = UP ? o3 : o4;
                if (start) first[c] = UP ? o4 : o3;
                const unsigned m = (unsigned)(mk[c] >> (8 * q)) & 0xffu;
                if (m & 15u) {   // half-link membranes (Eq. B5)
                    mix_if<2u>(m, g[1], o2[c], sh2);
                    mix_if<1u>(m, g[2], o1[c], sh2);
                    mix_if<8u>(m, g[3], o4, sh2);
                    mix_if<4u>(m, g[4], o3, sh2);
                }
                float2 rot;
                if (GEN && !tab) {   // rotation_m1's general form
                    const float th = __fmul_rn(f, __fmaf_rn(d->ctheta[2], (float)d->z0,
                                                            __fmaf_rn(cy, (float)(b.y0 + q), __fmul_rn(cx, (float)x))));
                    float sn, cs;
                    sincosf(0.5f * th, &sn, &cs);
                    rot = make_float2(__fmul_rn(-2.f, __fmul_rn(sn, sn)), __fmul_rn(2.f, __fmul_rn(sn, cs)));
                } else {
                    rot = (axes & 1) ? ((axes & 2) ? cadd_prod(ex[c], s_ey[q]) : ex[c]) : s_ey[q];
                    rot = make_float2(__fmul_rn(rot.x, fabsf(f)), __fmul_rn(rot.y, f));
                }
                const float2 pe = s_phase[m >> 6];
                const u64 M = react_collide(g, reaction_q(rot, pe.y), pe.x, a.w0, a.wxy);
                turn_rest(p0[c], g[0], UP);
                lev[q * nx + x] = g[1];
                lev[R + q * nx + x] = g[2];
                *r3 = g[3];
                *r4 = g[4];
                if (more) {
                    if (q == 0 && below >= 0) post(n + 1, 0, x, g[4]);
                    if (q == hy - 1 && above >= 0) post(n + 1, 1, x, g[3]);
                }
                if (do_sig || do_fld || r.series) {
                    const size_t s = (size_t)(b.y0 + q) * nx + x;
                    const float2 v = unpk(M);
                    if (do_sig) mout[s] = v;
                    if (do_fld) field[s] = v;
                    zr += v.x;
                    zi += v.y;
                }
            }
        }
        if (UP) skip(true);
        if (r.series) {   // this block's part of Z after the step
            for (int o = 16; o > 0; o >>= 1) {
                zr += __shfl_down_sync(0xffffffffu, zr, o);
                zi += __shfl_down_sync(0xffffffffu, zi, o);
            }
            if ((t & 31) == 0) s_red[t >> 5] = make_double2(zr, zi);
            __syncthreads();
            if (t == 0) {
                double2 v = make_double2(0.0, 0.0);
                for (int w = 0; w < NT / 32; ++w) {
                    v.x += s_red[w].x;
                    v.y += s_red[w].y;
                }
                r.zpart[(size_t)n * gridDim.x + blockIdx.x] = v;
            }
        }
        if (t < 6) s_fac[(n & 1) ^ 1][t] = fnext;
        if (t == 6) s_f[(n & 1) ^ 1] = fnext.x;
        __syncthreads();   // the last row done is the next step's first
    }

    u64* __restrict__ dst = reinterpret_cast<u64*>(d->state + (size_t)r.ldst * 7 * P + (size_t)b.y0 * nx);
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
        const int x = t + c * NT;
        if (x >= nx) continue;
#pragma unroll
        for (int q = 0; q < ROWS; ++q) {
            if (q >= hy) break;
            const unsigned s = (unsigned)q * nx + x;
            dst[s] = p0[c][q];
#pragma unroll
            for (int i = 1; i <= 4; ++i) dst[(size_t)i * P + s] = lev[(i - 1) * R + s];
            for (int i = 5; i < Q; ++i) dst[(size_t)i * P + s] = 0ull;
        }
    }
    if (waits.dead) atomicOr(&a.ctl->err, 1);
}

using StripFn = void (*)(const SweepArgs, const ResArgs);

}  // namespace

int strip_rows(int nx) { return nx <= 2 * NT ? 8 : nx <= 3 * NT ? 6 : 0; }
size_t strip_smem(int nx, int rows) { return (size_t)4 * nx * rows * sizeof(float2); }

cudaError_t launch_strip(const SweepArgs& a, const ResArgs& r, int n_blocks, int max_nx, size_t smem, bool general,
                         cudaStream_t st)
{
    const StripFn k = max_nx <= 2 * NT ? (general ? sweep_strip_kernel<2, 8, true> : sweep_strip_kernel<2, 8, false>)
                                       : (general ? sweep_strip_kernel<3, 6, true> : sweep_strip_kernel<3, 6, false>);
    const void* fn = (const void*)k;
    const cudaError_t e = allow_smem(fn, smem);
    if (e != cudaSuccess) return e;
    SweepArgs aa = a;
    ResArgs rr = r;
    void* args[2] = {&aa, &rr};
    return cudaLaunchCooperativeKernel(fn, dim3(n_blocks), dim3(NT), args, smem, st);
}

}  // namespace lbmbt
