// sweep_pair.cu -- two time steps per pass over the state.
//
// The one-step sweeps read and write the seven populations of every site once
// per step, 113 B, and run at 0.75-0.9 of the HBM copy rate on large grids:
// nothing is left but to touch the state less often.  This kernel advances
// hat g(t^k) to hat g(t^(k+2)) with one read and one write.
//
// Work item: a tile of w x h columns of one member over the planes [z0, z1).
// A thread has two neighbouring columns (x, x + 1); the block covers the tile
// grown by two columns in x and one in y on each side.  It marches along z.
// At plane z
//   step 1  every thread computes hat g(t^(k+1)) of its columns at z, the halo
//           columns included, from the plane's inputs in shared memory;
//   step 2  the threads of the tile compute hat g(t^(k+2)) at plane z - 1 from
//           the step-1 values around it and store it.
// Populations 0, 5 and 6 move along the thread's own columns: their step-1
// values of the last planes stay in registers.  Populations 1-4 cross columns
// and go through shared memory, double-buffered over planes, with one block
// barrier per plane.  A halo column beyond a periodic face is the wrapped
// site; its step 1 is that site's own.  Beyond a mirror face there is none.
// The cost is step 1 of the halo columns and of the two planes around
// [z0, z1); the item list balances it against idle SMs (api.cu).
//
// The inputs of a plane are seven TMA boxes, one per population, copied a
// plane ahead into shared memory by one thread; carried along the column, p5
// becomes the next plane's +z pull and p6 (copied from the plane above) its own
// value, so every row is read once per item.  For the boxes to need no special
// case at periodic faces the state of a run on this kernel has two ghost
// columns and rows on each side (row length nx + 4, rounded up to even for the
// 16-byte rule of TMA coordinates and strides; ny + 4 rows), which the store of
// the wrapped site fills.  Copies without tensor maps were slower: a bulk copy
// per row took 1.4 times the instructions, 16-byte cp.async by every thread
// twice the L2 sectors (it fetches 64-byte blocks): 276 and 268 ms against 230 on
// 512^3 tissue, three directions, 48 steps, with the same blocks.
//
// Two columns a thread because the kernel is issue-bound: with one column it
// took 382 thread instructions per site and step, most of them addresses,
// predicates and loop control that two columns share.  16-byte copies, shared
// accesses and stores (the state's rows are padded to an even length) and the packed f32x2
// operations of sm_100 and later halve what remains.  A packed operation
// rounds each half as the scalar one does and the order is that of the other
// sweeps, so the fields are the same bits.
#include <cuda.h>

#include <algorithm>

#include "lbmbt_internal.cuh"
#include "sweep_common.cuh"
#include "packed.cuh"
#include "tma_common.cuh"

namespace lbmbt {
namespace {

constexpr int PAIR_STAGES = 2;   // planes of input in shared memory: one in use, one in flight
constexpr int PAIR_MAX_EX = 40;  // pairs of columns in a row of a block
constexpr int PAIR_GHOST = 2;    // ghost columns and rows on each side
// A stage in 16-byte words: boxes of (rows of the grown tile) x ex pairs of
// p0 p1 p2 p5 p6, then of one row more of p3 (from one row below) and p4.
__host__ __device__ constexpr int stage_words(int nt) { return 7 * nt + 2 * PAIR_MAX_EX; }
__device__ __forceinline__ void tma_box(void* dst, const CUtensorMap* map, int x, int y, int z, int p, uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(
            smem_u32(dst)),
        "l"(map), "r"(x), "r"(y), "r"(z), "r"(p), "r"(smem_u32(bar))
        : "memory");
}

// The maps lie in global memory and are rewritten by a copy from the host at each
// set-up, at the same address.  They are read through a proxy of their own, which
// neither the copy nor the launch orders: the thread that issues boxes acquires
// each map it uses first.  Issued by thread 0 behind its ticket, the acquires cost 1 us a
// launch (117 x 90 x 75, 480 steps: 8.5 ms; beside the ticket 8.4; 128^3: 50.2 and 49.6).
__device__ __forceinline__ void acquire_map(const CUtensorMap* map)
{
    asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(map) : "memory");
}

// Exact running sum (two-sum) of one component.
__device__ __forceinline__ void two_sum(float& s, float& c, float v)
{
    const float t = __fadd_rn(s, v);
    const float b = __fsub_rn(t, s);
    c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(v, b)));
    s = t;
}

// Column flags.  Faces: a pull across them needs a transform.
enum : unsigned {
    A_XLO = 1u, A_XHI = 2u, B_XLO = 4u, B_XHI = 8u, F_YLO = 16u, F_YHI = 32u, F_FACE = 63u,
    A_ACT = 64u, B_ACT = 128u, A_IN = 256u, B_IN = 512u,
    F_S16 = 1024u,    // stores both columns as one word
    F_M16 = 2048u,    // reads both mask bytes as one word
    F_GHOST = 4096u   // stores ghost copies too
};

// GEN: the waveform may take values other than 0 and +-1.
template <int NT, int MINB, bool GEN, int STEPS>
__global__ void __launch_bounds__(NT, MINB) sweep_pair_kernel(const SweepArgs a, const PairItem* __restrict__ items,
                                                              const CUtensorMap* __restrict__ maps, int n_items)
{
    extern __shared__ __align__(128) unsigned char pair_smem[];
    constexpr int SW = stage_words(NT);
    ulonglong2* const sin = reinterpret_cast<ulonglong2*>(pair_smem);   // [PAIR_STAGES][SW] inputs of a plane
    ulonglong2* const smid = sin + PAIR_STAGES * SW;                    // [2][4][NT] step-1 populations 1..4
    float4* const ssum = reinterpret_cast<float4*>(smid + 2 * 4 * NT);  // [2][NT] running sums of M
    __shared__ float2 s_fac[12];     // boundary factors of step k, k + 1
    __shared__ float2 s_phase[4];    // (omega, eps) per phase
    __shared__ int s_ctl[6];
    __shared__ int s_bc[3];          // faces (read where a column is at one)
    // what a plane reads once: kept here rather than in registers
    __shared__ float2 *s_field, *s_mout, *s_dst;
    __shared__ const uint8_t* s_mask;
    __shared__ unsigned s_sxym;
    __shared__ int s_wrap[2];        // element shift of the ghost copies in x and y, 0 for a mirror
    __shared__ uint64_t full[PAIR_STAGES];   // the boxes of a stage have arrived
    __shared__ uint64_t never;               // nothing completes it (tests of the time-out)
    __shared__ int s_dead;                   // a wait ran out

    const int t = threadIdx.x;
    const PairItem it = items[blockIdx.x];
    const MemberDesc* __restrict__ d = a.members + it.m;
    if (t == 0) {
        s_ctl[0] = __ldcg(&a.ctl->k);
        s_ctl[1] = __ldcg(&a.ctl->slot_base);
        s_ctl[2] = __ldcg(&a.ctl->slot_mod);
        s_ctl[3] = __ldcg(&a.ctl->sig_step);
        s_ctl[4] = __ldcg(&a.ctl->field_step);
        s_ctl[5] = __ldcg(&a.ctl->series);
        for (int q = 0; q < PAIR_STAGES; ++q) mbar_init(&full[q], 1);
        mbar_init(&never, 1);
        fence_mbar_init();
        s_dead = 0;
    }
    __syncthreads();
    const int k = s_ctl[0];
    // this block has read the step word: its ticket (the last block advances it)
    if (t == 0) step_done(a.ctl, k, gridDim.x, true, STEPS, STEPS - 1);
    if (t < 6 * STEPS) s_fac[t] = __ldg(a.fac + ((size_t)(k + t / 6) * a.n_members + it.m) * 6 + t % 6);
    if (t < 4) s_phase[t] = make_float2(d->omega[t], d->eps[t]);
    if (t < 3) s_bc[t] = d->bc[t];
    if (t == 0) {
        s_field = d->field;
        s_mout = d->mout;
        s_mask = d->mask;
        s_sxym = (unsigned)d->nx * d->ny;
        s_wrap[0] = d->bc[0] == BC_PER ? d->nx : 0;
        s_wrap[1] = d->bc[1] == BC_PER ? d->ny * d->pitch : 0;
    }

    const int lsrc = (k - s_ctl[1]) % s_ctl[2];
    const int ldst = (lsrc + 1) % s_ctl[2];
    const bool series = s_ctl[5];
    const int es = d->end_step;
    const int sig = es >= 0 ? es : s_ctl[3], fstep = es >= 0 ? es : s_ctl[4];
    // A member past its own end, no series asked for: nothing of it is read any more (16
    // members of four edges, echoes at 0.4 to 1 of 160 steps: 20.8 ms against 27.5).
    if (es >= 0 && k > es && !series) return;
    // bits: M of step 1, 2 into the sums, the field, mout
    const bool fld = d->field != nullptr, out = d->mout != nullptr;
    const unsigned obs = (series || (k == sig && !out) ? 1u : 0u) | (series || (k + 1 == sig && !out) ? 2u : 0u) |
                         (k == fstep && fld ? 4u : 0u) | (k + 1 == fstep && fld ? 8u : 0u) |
                         (k == sig && out ? 16u : 0u) | (k + 1 == sig && out ? 32u : 0u);

    const int nx = d->nx, ny = d->ny, nz = d->nz;
    const unsigned P = (unsigned)d->plane, pitch = (unsigned)d->pitch, sxy = pitch * (ny + 2 * PAIR_GHOST);
    const bool mir = d->bc[2] != BC_PER;
    const float2* __restrict__ src = d->state + (size_t)lsrc * 7 * P;
    if (t == 0) s_dst = d->state + (size_t)ldst * 7 * P;
    const u64 sh2 = pk(d->s_share, d->s_share);
    const float f1 = __ldg(d->fw + k), f2 = STEPS == 2 ? __ldg(d->fw + k + 1) : 0.f;
    const int axes = d->axes;
    const bool tab1 = !GEN || f1 == 0.f || f1 == 1.f || f1 == -1.f;
    const bool tab2 = !GEN || f2 == 0.f || f2 == 1.f || f2 == -1.f;

    const bool mirx = d->bc[0] != BC_PER, miry = d->bc[1] != BC_PER;
    // this thread's columns A = (xa, y) and B = (xb, y), xb the next one
    const int exp_ = it.ex;   // pairs per row of the grown tile
    const int j = t / exp_, i = t - j * exp_;
    int xa = it.x0 - 2 + 2 * i, xb = xa + 1, y = it.y0 - 1 + j;
    unsigned fl = 0;
    const bool row_in = j >= 1 && j <= it.h;
    if (j < it.h + 2) {
        if (row_in && xa >= it.x0 && xa < it.x0 + it.w) fl |= A_IN;
        if (row_in && xb >= it.x0 && xb < it.x0 + it.w) fl |= B_IN;
        const bool oky = !miry || (y >= 0 && y < ny);
        if (oky && (!mirx || (xa >= 0 && xa < nx))) fl |= A_ACT;
        if (oky && (!mirx || (xb >= 0 && xb < nx))) fl |= B_ACT;
    }
    auto wrap = [](int v, int n) {
        while (v < 0) v += n;
        while (v >= n) v -= n;
        return v;
    };
    y = wrap(y, ny);
    xa = wrap(xa, nx);
    xb = wrap(xb, nx);
    if (xa == 0) fl |= A_XLO;
    if (xa == nx - 1) fl |= A_XHI;
    if (xb == 0) fl |= B_XLO;
    if (xb == nx - 1) fl |= B_XHI;
    if (y == 0) fl |= F_YLO;
    if (y == ny - 1) fl |= F_YHI;
    // the columns' element in a plane of the state, and in one of mask and field
    const unsigned sa = (unsigned)(y + PAIR_GHOST) * pitch + (xa + PAIR_GHOST), sam = (unsigned)y * nx + xa;
    const int ab = xb - xa;   // 1, or -(nx - 1) where the pair straddles the face (nx odd)
    if (ab == 1 && (fl & A_IN) && (fl & B_IN)) fl |= F_S16;
    if (ab == 1 && (sam & 1) == 0 && (nx & 1) == 0) fl |= F_M16;
    if ((!mirx && (xa < 2 || xa >= nx - 3)) || (!miry && (y < 2 || y >= ny - 2))) fl |= F_GHOST;

    // planes of step 1: one below and one above [z0, z1) unless a mirror face is there
    const int zb = STEPS == 2 && !(mir && it.z0 == 0) ? it.z0 - 1 : it.z0;
    const int zl = STEPS == 2 && !(mir && it.z1 == nz) ? it.z1 : it.z1 - 1;   // last plane of step 1
    const int ze = STEPS == 2 ? it.z1 : it.z1 - 1;                            // last iteration
    auto wrapz = [&](int z) { return z < 0 ? z + nz : z >= nz ? z - nz : z; };

    // Copies of a plane's inputs, issued by the first thread of the second warp: the
    // acquire of its maps runs beside the first warp's ticket
    const bool copier = t == 32;
    const CUtensorMap* map = maps + (2 * it.m + lsrc);
    auto issue = [&](int zi, int st) {
        const int z = wrapz(zi);
        ulonglong2* q = sin + st * SW;
        const int x = it.x0, y = it.y0 + 1;   // x0 - 2 and y0 - 1, and the ghosts before them
        mbar_arrive_expect_tx(&full[st], (uint32_t)(16 * it.ex * (7 * (it.hb + 2) + 2)));
        fence_proxy_async_smem();   // the stage was read last before the block barrier
        tma_box(q, map, x, y, z, 0, &full[st]);
        tma_box(q + NT, map, x, y, z, 1, &full[st]);
        tma_box(q + 2 * NT, map, x, y, z, 2, &full[st]);
        tma_box(q + 3 * NT, map, x, y, z, 5, &full[st]);
        // the plane above (beyond a mirror face: any, it is not used)
        tma_box(q + 4 * NT, map, x, y, z < nz - 1 ? z + 1 : mir ? z : 0, 6, &full[st]);
        tma_box(q + 5 * NT, map + 2 * a.n_members, x, y - 1, z, 3, &full[st]);
        tma_box(q + 6 * NT + PAIR_MAX_EX, map + 2 * a.n_members, x, y, z, 4, &full[st]);
    };
    auto load2 = [&](const float2* p) {   // both columns
        ulonglong2 r = make_ulonglong2(0ull, 0ull);
        if (fl & A_ACT) r.x = __ldg(reinterpret_cast<const u64*>(p));
        if (fl & B_ACT) r.y = __ldg(reinterpret_cast<const u64*>(p + ab));
        return r;
    };
    auto load_mask = [&](int z) -> unsigned {   // A in bits 0..7, B in bits 8..15
        const uint8_t* p = s_mask + ((size_t)z * s_sxym + sam);
        if (fl & F_M16) return (fl & A_ACT) ? __ldg(reinterpret_cast<const unsigned short*>(p)) : 0u;
        unsigned r = (fl & A_ACT) ? __ldg(p) : 0u;
        if (fl & B_ACT) r |= (unsigned)__ldg(p + ab) << 8;
        return r;
    };

    int issued = 0;   // the copier's: planes asked for
    if (copier) {
        acquire_map(map);
        acquire_map(map + 2 * a.n_members);
        for (int q = 0; q < PAIR_STAGES - 1; ++q)
            if (zb + q <= zl) { issue(zb + q, q); ++issued; }
    }
    __syncthreads();     // the shared constants are set
    ulonglong2 c5, o6;   // p5 of the plane below, own p6 of this plane
    // Mask bytes of the next plane and of the one after: a plane's are asked for two planes
    // ahead (one ahead they arrived late: 128^3 cylinders 50.4 against 49.3 ms)
    unsigned mkn, mkn2 = 0u;
    {
        const int z = wrapz(zb);
        c5 = make_ulonglong2(0ull, 0ull);
        if (z > 0 || !mir) c5 = load2(src + (size_t)(z > 0 ? z - 1 : nz - 1) * sxy + (5 * P + sa));
        o6 = load2(src + (size_t)z * sxy + (6 * P + sa));
        mkn = load_mask(z);
        if (zb < zl) mkn2 = load_mask(wrapz(zb + 1));
    }
    // reaction rotation: the x and y parts are the column's
    const float2* __restrict__ et = d->etab;
    const float2* __restrict__ etz = et + nx + ny;
    float2 ra = make_float2(0.f, 0.f), rb = ra, ezn = ra;
    float tha = 0.f, thb = 0.f;
    if (axes & 1) { ra = __ldg(et + xa); rb = __ldg(et + xb); }
    if (axes & 2) {
        const float2 v = __ldg(et + nx + y);
        ra = (axes & 1) ? cadd_prod(ra, v) : v;
        rb = (axes & 1) ? cadd_prod(rb, v) : v;
    }
    const bool tz = axes & 4, txy = axes & 3;
    if (tz) ezn = __ldg(etz + wrapz(zb));
    if (GEN) {
        tha = __fmaf_rn(d->ctheta[1], (float)y, __fmul_rn(d->ctheta[0], (float)xa));
        thb = __fmaf_rn(d->ctheta[1], (float)y, __fmul_rn(d->ctheta[0], (float)xb));
    }
    const float ctz = GEN ? d->ctheta[2] : 0.f;
    auto general = [&](float f, float thxy, int z) {   // rotation_m1's general form
        const float th = __fmul_rn(f, __fmaf_rn(ctz, (float)z, thxy));
        float sn, cs;
        sincosf(0.5f * th, &sn, &cs);
        return make_float2(__fmul_rn(-2.f, __fmul_rn(sn, sn)), __fmul_rn(2.f, __fmul_rn(sn, cs)));
    };
    // table form for f in {0, +-1}: (cos - 1, f sin), zero for f = 0
    auto signed_rot = [](float2 r, float f) { return make_float2(__fmul_rn(r.x, fabsf(f)), __fmul_rn(r.y, f)); };

    if (obs & 1u) ssum[t] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (STEPS == 2 && (obs & 2u)) ssum[NT + t] = make_float4(0.f, 0.f, 0.f, 0.f);
    // M of an observed step into the running sums and the field (rare)
    auto observe = [&](float4* acc, unsigned what, unsigned who, u64 ma, u64 mb, int z) {
        const float2 va = unpk(ma), vb = unpk(mb);
        if (what & 1u) {
            float4 v = *acc;
            if (who & A_IN) { two_sum(v.x, v.y, va.x); two_sum(v.z, v.w, va.y); }
            if (who & B_IN) { two_sum(v.x, v.y, vb.x); two_sum(v.z, v.w, vb.y); }
            *acc = v;
        }
        for (int q = 0; q < 2; ++q) {
            if (!(what & (q == 0 ? 4u : 16u))) continue;
            float2* fp = (q == 0 ? s_field : s_mout) + ((size_t)z * s_sxym + sam);
            if (who & A_IN) fp[0] = va;
            if (who & B_IN) fp[ab] = vb;
        }
    };
    // a tile's two columns are neighbours; xa even: on one word
    auto store = [&](int z, const u64 (&ga)[Q], const u64 (&gb)[Q]) {
        float2* o = s_dst + ((size_t)z * sxy + sa);
        auto put = [&](float2* to, bool qa, bool qb) {
            if ((fl & F_S16) && qa && qb) {
#pragma unroll
                for (int p = 0; p < Q; ++p) __stcs(reinterpret_cast<ulonglong2*>(to + (size_t)p * P), make_ulonglong2(ga[p], gb[p]));
            } else {
#pragma unroll
                for (int p = 0; p < Q; ++p) {
                    if (qa) __stcs(reinterpret_cast<u64*>(to + (size_t)p * P), ga[p]);
                    if (qb) __stcs(reinterpret_cast<u64*>(to + (size_t)p * P) + 1, gb[p]);
                }
            }
        };
        put(o, fl & A_IN, fl & B_IN);
        if (fl & F_GHOST) {   // copies beyond the opposite periodic faces
            const bool ina = fl & A_IN, inb = fl & B_IN;
            const int wx = xa < 2 ? s_wrap[0] : -s_wrap[0], wy = y < 2 ? s_wrap[1] : -s_wrap[1];
            const bool gx = wx != 0 && (xa < 2 || xa >= nx - 3), gy = wy != 0 && (y < 2 || y >= ny - 2);
            const bool qa = ina && (xa < 2 || xa >= nx - 2), qb = inb && (xa < 2 ? xa + 1 < 2 : xa + 1 >= nx - 2);
            if (gy) put(o + wy, ina, inb);
            if (gx) {
                // nx odd: the copies of a word are not on a word
                const unsigned keep = fl;
                if (wx & 1) fl &= ~F_S16;
                put(o + wx, qa, qb);
                if (gy) put(o + wx + wy, qa, qb);
                fl = keep;
            }
        }
    };

    // step-1 values of the plane below (populations 0, 5, 6 of these columns),
    // population 5 of the plane below that, its mask bytes and rotation
    const ulonglong2 zero2 = make_ulonglong2(0ull, 0ull);
    ulonglong2 m0 = zero2, m5 = zero2, m6 = zero2, j5 = zero2;
    unsigned mkp = 0;
    float2 qra = make_float2(0.f, 0.f), qrb = qra;

    int st = 0;           // stage of plane zi and the parity of its fill
    uint32_t ph = 0;
    // A copy did not arrive within the limit: the block finishes without waiting and
    // without asking for more (what it computes is lost), and reports.
    bool dead = false;
    if (a.test_wait_ns && !mbar_wait(&never, 0u, a.test_wait_ns)) s_dead = 1;
    for (int zi = zb; zi <= ze; ++zi) {
        if (zi <= zl && !dead && !mbar_wait(&full[st], ph)) s_dead = 1;
        __syncthreads();   // plane zi's inputs and plane zi - 1's step-1 values are visible
        dead = s_dead;     // of all threads
        if (copier && !dead && zi + PAIR_STAGES - 1 <= zl) {
            issue(zi + PAIR_STAGES - 1, st == 0 ? PAIR_STAGES - 1 : st - 1);
            ++issued;
        }
        const unsigned mk = mkn;
        ulonglong2 n0 = zero2, n5 = zero2, n6 = zero2;
        float2 nra = make_float2(0.f, 0.f), nrb = nra;
        if (zi <= zl) {   // step 1 at plane zi
            const int z = wrapz(zi);
            const ulonglong2* __restrict__ q = sin + st * SW + t;
            const float2 ez = ezn;
            mkn = mkn2;
            if (zi + 1 < zl) mkn2 = load_mask(wrapz(zi + 2));
            if (zi < zl) {
                if (tz) ezn = __ldg(etz + wrapz(zi + 1));
            }
            u64 ga[Q], gb[Q];
            const ulonglong2 *__restrict__ q3 = q + 5 * NT, *__restrict__ q4 = q + 6 * NT + PAIR_MAX_EX;
            const ulonglong2 p0 = q[0], p1 = q[NT], p2 = q[2 * NT], p3 = q3[0], p4 = q4[exp_], p5 = q[3 * NT],
                             p6 = q[4 * NT];
            ga[0] = p0.x; gb[0] = p0.y;
            ga[1] = q[NT - 1].y; gb[1] = p1.x;
            ga[2] = p2.y; gb[2] = q[2 * NT + 1].x;
            ga[3] = p3.x; gb[3] = p3.y;
            ga[4] = p4.x; gb[4] = p4.y;
            ga[5] = c5.x; gb[5] = c5.y;
            ga[6] = p6.x; gb[6] = p6.y;
            if (fl & F_FACE) {   // mirror: the own opposite population
                const int bcx = s_bc[0], bcy = s_bc[1];
                const bool mx = bcx != BC_PER;
                if (fl & A_XLO) ga[1] = face2(mx ? p2.x : ga[1], bcx, s_fac[0]);
                if (fl & A_XHI) ga[2] = face2(mx ? p1.x : ga[2], bcx, s_fac[1]);
                if (fl & B_XLO) gb[1] = face2(mx ? p2.y : gb[1], bcx, s_fac[0]);
                if (fl & B_XHI) gb[2] = face2(mx ? p1.y : gb[2], bcx, s_fac[1]);
                if (fl & F_YLO) {
                    const ulonglong2 v = bcy != BC_PER ? q4[0] : p3;
                    ga[3] = face2(v.x, bcy, s_fac[2]);
                    gb[3] = face2(v.y, bcy, s_fac[2]);
                }
                if (fl & F_YHI) {
                    const ulonglong2 v = bcy != BC_PER ? q3[exp_] : p4;
                    ga[4] = face2(v.x, bcy, s_fac[3]);
                    gb[4] = face2(v.y, bcy, s_fac[3]);
                }
            }
            if (z == 0) { ga[5] = face2(mir ? o6.x : ga[5], s_bc[2], s_fac[4]); gb[5] = face2(mir ? o6.y : gb[5], s_bc[2], s_fac[4]); }
            if (z == nz - 1) { ga[6] = face2(mir ? p5.x : ga[6], s_bc[2], s_fac[5]); gb[6] = face2(mir ? p5.y : gb[6], s_bc[2], s_fac[5]); }
            if (mk & 0x3f3fu) {
                const ulonglong2 v4 = q4[0], v3 = q3[exp_];
                mix_if<0x2u>(mk, ga[1], p2.x, sh2);
                mix_if<0x200u>(mk, gb[1], p2.y, sh2);
                mix_if<0x1u>(mk, ga[2], p1.x, sh2);
                mix_if<0x100u>(mk, gb[2], p1.y, sh2);
                mix_if<0x8u>(mk, ga[3], v4.x, sh2);
                mix_if<0x800u>(mk, gb[3], v4.y, sh2);
                mix_if<0x4u>(mk, ga[4], v3.x, sh2);
                mix_if<0x400u>(mk, gb[4], v3.y, sh2);
                mix_if<0x20u>(mk, ga[5], o6.x, sh2);
                mix_if<0x2000u>(mk, gb[5], o6.y, sh2);
                mix_if<0x10u>(mk, ga[6], p5.x, sh2);
                mix_if<0x1000u>(mk, gb[6], p5.y, sh2);
            }
            c5 = p5;
            o6 = p6;
            float2 rota, rotb;
            nra = ra;
            nrb = rb;
            if (tz) {
                nra = txy ? cadd_prod(ra, ez) : ez;
                nrb = txy ? cadd_prod(rb, ez) : ez;
            }
            if (GEN && !tab1) {
                rota = general(f1, tha, z);
                rotb = general(f1, thb, z);
            } else {
                rota = signed_rot(nra, f1);
                rotb = signed_rot(nrb, f1);
            }
            const float2 pa = s_phase[(mk >> 6) & 3u], pb = s_phase[mk >> 14];
            const u64 ma = react_collide<Q>(ga, reaction_q(rota, pa.y), pa.x);
            const u64 mb = react_collide<Q>(gb, reaction_q(rotb, pb.y), pb.x);
            if ((obs & 21u) && zi >= it.z0 && zi < it.z1) observe(ssum + t, obs, fl, ma, mb, z);
            if (STEPS == 1) {
                store(z, ga, gb);
            } else {
                ulonglong2* w = smid + (unsigned)(zi & 1) * (4 * NT) + t;
                w[0] = make_ulonglong2(ga[1], gb[1]);
                w[NT] = make_ulonglong2(ga[2], gb[2]);
                w[2 * NT] = make_ulonglong2(ga[3], gb[3]);
                w[3 * NT] = make_ulonglong2(ga[4], gb[4]);
                n0 = make_ulonglong2(ga[0], gb[0]);
                n5 = make_ulonglong2(ga[5], gb[5]);
                n6 = make_ulonglong2(ga[6], gb[6]);
            }
        }
        if (STEPS == 2) {
            const int z = zi - 1;   // step 2 at plane z
            if (z >= it.z0 && (fl & (A_IN | B_IN))) {
                const ulonglong2* __restrict__ w = smid + (unsigned)(z & 1) * (4 * NT) + t;
                u64 ga[Q], gb[Q];
                const ulonglong2 w1 = w[0], w2 = w[NT];
                const ulonglong2 v3 = w[2 * NT - exp_], v4 = w[3 * NT + exp_];
                ga[0] = m0.x; gb[0] = m0.y;
                ga[1] = w[-1].y; gb[1] = w1.x;
                ga[2] = w2.y; gb[2] = w[NT + 1].x;
                ga[3] = v3.x; gb[3] = v3.y;
                ga[4] = v4.x; gb[4] = v4.y;
                ga[5] = j5.x; gb[5] = j5.y;
                ga[6] = n6.x; gb[6] = n6.y;
                if (fl & F_FACE) {
                    const int bcx = s_bc[0], bcy = s_bc[1];
                    const bool mx = bcx != BC_PER, my = bcy != BC_PER;
                    if (fl & A_XLO) ga[1] = face2(mx ? w2.x : ga[1], bcx, s_fac[6]);
                    if (fl & A_XHI) ga[2] = face2(mx ? w1.x : ga[2], bcx, s_fac[7]);
                    if (fl & B_XLO) gb[1] = face2(mx ? w2.y : gb[1], bcx, s_fac[6]);
                    if (fl & B_XHI) gb[2] = face2(mx ? w1.y : gb[2], bcx, s_fac[7]);
                    if (fl & F_YLO) {
                        const ulonglong2 v = my ? w[3 * NT] : v3;
                        ga[3] = face2(v.x, bcy, s_fac[8]);
                        gb[3] = face2(v.y, bcy, s_fac[8]);
                    }
                    if (fl & F_YHI) {
                        const ulonglong2 v = my ? w[2 * NT] : v4;
                        ga[4] = face2(v.x, bcy, s_fac[9]);
                        gb[4] = face2(v.y, bcy, s_fac[9]);
                    }
                }
                if (z == 0) { ga[5] = face2(mir ? m6.x : ga[5], s_bc[2], s_fac[10]); gb[5] = face2(mir ? m6.y : gb[5], s_bc[2], s_fac[10]); }
                if (z == nz - 1) { ga[6] = face2(mir ? m5.x : ga[6], s_bc[2], s_fac[11]); gb[6] = face2(mir ? m5.y : gb[6], s_bc[2], s_fac[11]); }
                if (mkp & 0x3f3fu) {
                    const ulonglong2 u4 = w[3 * NT], u3 = w[2 * NT];
                    mix_if<0x2u>(mkp, ga[1], w2.x, sh2);
                    mix_if<0x200u>(mkp, gb[1], w2.y, sh2);
                    mix_if<0x1u>(mkp, ga[2], w1.x, sh2);
                    mix_if<0x100u>(mkp, gb[2], w1.y, sh2);
                    mix_if<0x8u>(mkp, ga[3], u4.x, sh2);
                    mix_if<0x800u>(mkp, gb[3], u4.y, sh2);
                    mix_if<0x4u>(mkp, ga[4], u3.x, sh2);
                    mix_if<0x400u>(mkp, gb[4], u3.y, sh2);
                    mix_if<0x20u>(mkp, ga[5], m6.x, sh2);
                    mix_if<0x2000u>(mkp, gb[5], m6.y, sh2);
                    mix_if<0x10u>(mkp, ga[6], m5.x, sh2);
                    mix_if<0x1000u>(mkp, gb[6], m5.y, sh2);
                }
                float2 rota, rotb;
                if (GEN && !tab2) {
                    rota = general(f2, tha, z);
                    rotb = general(f2, thb, z);
                } else {
                    rota = signed_rot(qra, f2);
                    rotb = signed_rot(qrb, f2);
                }
                const float2 pa = s_phase[(mkp >> 6) & 3u], pb = s_phase[mkp >> 14];
                const u64 ma = react_collide<Q>(ga, reaction_q(rota, pa.y), pa.x);
                const u64 mb = react_collide<Q>(gb, reaction_q(rotb, pb.y), pb.x);
                store(z, ga, gb);
                if (obs & 42u) observe(ssum + NT + t, obs >> 1, fl, ma, mb, z);
            }
            j5 = m5;
            m0 = n0;
            m5 = n5;
            m6 = n6;
            mkp = mk;
            qra = nra;
            qrb = nrb;
        }
        st = st == PAIR_STAGES - 1 ? 0 : st + 1;
        ph = st == 0 ? ph ^ 1u : ph;
    }
    if (dead && copier) {   // copies in flight end (wait bounded too) before their stages are used again or given back
        for (int q = max(0, issued - PAIR_STAGES); q < issued; ++q)
            mbar_wait(&full[q % PAIR_STAGES], (uint32_t)(q / PAIR_STAGES & 1));
        atomicOr(&a.ctl->err, 1);
    }

    if ((obs & 1u) || (STEPS == 2 && (obs & 2u))) {   // block-uniform
        __syncthreads();
        // a member's one signal goes to the first partial; the series keeps both steps apart
        double2* const red = reinterpret_cast<double2*>(pair_smem);
        for (int q = 0; q < STEPS; ++q) {
            if (!(obs & (1u << q))) continue;
            const float4 v = ssum[q * NT + t];
            double dr = (double)v.x + v.y, di = (double)v.z + v.w;
            for (int o = 16; o > 0; o >>= 1) {
                dr += __shfl_down_sync(0xffffffffu, dr, o);
                di += __shfl_down_sync(0xffffffffu, di, o);
            }
            if ((t & 31) == 0) red[t >> 5] = make_double2(dr, di);
            __syncthreads();
            if (t == 0) {
                double2 r = make_double2(0.0, 0.0);
                for (int b = 0; b < NT / 32; ++b) {
                    r.x += red[b].x;
                    r.y += red[b].y;
                }
                a.partial[blockIdx.x + (s_ctl[5] && q == 1 ? n_items : 0)] = r;
            }
            __syncthreads();
        }
    }
}

// State at M = 1: population i is its weight, in every element of the planes.
__global__ void pair_init_kernel(const MemberDesc* __restrict__ members, int n_members)
{
    for (int m = blockIdx.y; m < n_members; m += gridDim.y) {
        const MemberDesc& d = members[m];
        const long long n = 7 * d.plane / 2, per = d.plane / 2;
        float4* out = reinterpret_cast<float4*>(d.state);
        for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
            const float w = e < per ? W0 : WI;
            out[e] = make_float4(w, 0.f, w, 0.f);
        }
    }
}

// Copies level `src` of every member to the other one, from the one-step sweeps' layout to
// this one with its ghosts (to_pair) or back.
__global__ void pair_relayout_kernel(const MemberDesc* __restrict__ members, int n_members, int src, int to_pair)
{
    constexpr int G = PAIR_GHOST;
    for (int m = blockIdx.y; m < n_members; m += gridDim.y) {
        const MemberDesc& d = members[m];
        const int nx = d.nx, ny = d.ny, rows = ny + 2 * G;
        const long long n = to_pair ? (long long)d.pitch * rows * d.nz : d.N;
        const float2* from = d.state + (size_t)src * 7 * d.plane;
        float2* to = d.state + (size_t)(src ^ 1) * 7 * d.plane;
        for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
            long long o;
            if (to_pair) {   // ghosts are the wrapped sites; beyond a mirror face and nx + 4: any
                const long long row = e / d.pitch, z = row / rows;
                int x = (int)(e - row * d.pitch) - G, y = (int)(row - z * rows) - G;
                x = x < 0 ? x + nx : x >= nx ? x - nx : x;
                y = y < 0 ? y + ny : y >= ny ? y - ny : y;
                o = (z * ny + y) * nx + x;
            } else {
                const long long row = e / nx, z = row / ny;
                o = (z * rows + (row - z * ny) + G) * d.pitch + (e - row * nx) + G;
            }
            for (int i = 0; i < Q; ++i) to[(size_t)i * d.plane + e] = from[(size_t)i * d.plane + o];
        }
    }
}

// 256 threads x 2 columns, two blocks per SM (128 registers, 101 KB of shared
// memory each): one block's barrier and item start are hidden by the other.
// Measured before the masks were asked for two planes ahead (512^3 tissue / 128^3
// cylinders / 16 odd packs, ms a pass): 222 / 49.7 / 27.7; 512 threads x 1 block 223 /
// 50.2 / 32.5; 448 x 1 with a third stage 226 / 52.4 / 34.5; 224 x 2 with a third stage
// 230 / 55.7 / 31.2.  Since: 224 / 49.3 / 27.5 (20.8 with members past their echo
// skipped).
constexpr int PNT = 256, PMB = 2;
constexpr size_t PAIR_SMEM = (size_t)(PAIR_STAGES * stage_words(PNT) + 2 * 4 * PNT) * sizeof(ulonglong2) + 2 * PNT * sizeof(float4);

using PairFn = void (*)(SweepArgs, const PairItem*, const CUtensorMap*, int);

PairFn pair_kernel(bool general, int steps)
{
    if (general) return steps == 2 ? sweep_pair_kernel<PNT, PMB, true, 2> : sweep_pair_kernel<PNT, PMB, true, 1>;
    return steps == 2 ? sweep_pair_kernel<PNT, PMB, false, 2> : sweep_pair_kernel<PNT, PMB, false, 1>;
}

}  // namespace

int pair_threads() { return PNT; }
int pair_max_row() { return PAIR_MAX_EX; }
int pair_ghost() { return PAIR_GHOST; }
static_assert(sizeof(PairMap) == sizeof(CUtensorMap) && alignof(PairMap) >= alignof(CUtensorMap), "tensor map");

// Tensor map of one time level: [population][z][row][column] of 8-byte values,
// box of 2 ex columns x `rows` rows of one plane of one population.
cudaError_t pair_encode_map(PairMap* out, const void* level, const MemberDesc& d, int ex, int rows)
{
    using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static const Encode encode = [] {   // looked up once
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found) != cudaSuccess ||
            found != cudaDriverEntryPointSuccess)
            fn = nullptr;
        return reinterpret_cast<Encode>(fn);
    }();
    if (!encode) return cudaErrorNotSupported;
    const cuuint64_t row = (cuuint64_t)d.pitch, nrow = (cuuint64_t)d.ny + 2 * PAIR_GHOST;
    const cuuint64_t dims[4] = {row, nrow, (cuuint64_t)d.nz, 7};
    const cuuint64_t strides[3] = {row * 8, row * nrow * 8, (cuuint64_t)d.plane * 8};
    const cuuint32_t box[4] = {(cuuint32_t)(2 * ex), (cuuint32_t)rows, 1, 1}, one[4] = {1, 1, 1, 1};
    const CUresult r = encode(reinterpret_cast<CUtensorMap*>(out), CU_TENSOR_MAP_DATA_TYPE_INT64, 4, const_cast<void*>(level),
                              dims, strides, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                              CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t pair_prepare(bool general, int* ctas_per_sm)
{
    for (int steps = 1; steps <= 2; ++steps) {
        const void* f = (const void*)pair_kernel(general, steps);
        cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PAIR_SMEM);
        if (e == cudaSuccess && steps == 2)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, f, PNT, PAIR_SMEM);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_sweep_pair(const SweepArgs& a, const PairItem* items, const PairMap* maps, int n_items, bool general,
                              int steps, cudaStream_t st)
{
    pair_kernel(general, steps)<<<(unsigned)n_items, PNT, PAIR_SMEM, st>>>(a, items, reinterpret_cast<const CUtensorMap*>(maps),
                                                                         n_items);
    return cudaGetLastError();
}

cudaError_t launch_pair_relayout(const MemberDesc* members, int n_members, long long max_plane, int src, bool to_pair,
                                 cudaStream_t st)
{
    const long long bx = std::min<long long>((max_plane + 255) / 256, 152 * 16);
    pair_relayout_kernel<<<dim3((unsigned)bx, (unsigned)std::min(n_members, 65535)), 256, 0, st>>>(members, n_members, src,
                                                                                                to_pair ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_pair_init(const MemberDesc* members, int n_members, long long max_plane, cudaStream_t st)
{
    const long long bx = std::min<long long>((7 * max_plane / 2 + 1023) / 1024, 152 * 16);
    pair_init_kernel<<<dim3((unsigned)bx, (unsigned)std::min(n_members, 65535)), 256, 0, st>>>(members, n_members);
    return cudaGetLastError();
}

}  // namespace lbmbt
