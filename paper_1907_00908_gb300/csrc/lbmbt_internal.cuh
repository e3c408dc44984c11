// lbmbt_internal.cuh -- device-side descriptors shared by the kernels and the
// host side of liblbmbt (not part of the public C ABI).
//
// State layout in HBM (structure of arrays): for one member the post-collision
// populations hat g_i(x) of one time level are 7 planes of complex64
// (float2 = re, im), plane i at base + i*plane, site s = (z*ny + y)*nx + x.
// `plane` >= N is rounded up to a multiple of 64 sites so every plane starts
// 512-byte aligned.  A member owns `n_slots` such time levels back to back
// (stride 7*plane): 2 for the ping-pong of a run, c+1 for an adjoint segment.
#pragma once
#include <cstddef>
#include <cstdint>
#include <mutex>

#include <cuda_runtime.h>

namespace lbmbt {

// Lets launches of `fn` have `bytes` of dynamic shared memory.  The limit belongs to the
// kernel, not to a context: it is only ever raised, so that no context takes away what
// another one, prepared before or on another thread, launches with.
inline cudaError_t allow_smem(const void* fn, size_t bytes)
{
    static std::mutex mu;
    std::lock_guard<std::mutex> hold(mu);
    cudaFuncAttributes at;
    const cudaError_t e = cudaFuncGetAttributes(&at, fn);
    if (e != cudaSuccess || at.maxDynamicSharedSizeBytes >= (int)bytes) return e;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

constexpr int Q = 7;
// D3Q7 weights with eps_D = 1/4 (Sec. 2.3 pattern: w0 = eps_D, wi = eps_D/2).
constexpr float W0 = 0.25f;
constexpr float WI = 0.125f;
constexpr double EPS_D = 0.25;
// D2Q5 (Sec. 2.3, Eq. omega_i): eps_D = 1/3, w0 = 1/3, w1..4 = 1/6; run as
// the first five D3Q7 velocities on a grid of one z plane, z weights 0.
constexpr double EPS_D2 = 1.0 / 3.0;

// Outer-boundary handling of one axis for one member.
enum BcMode : int {
    BC_PER = 0,       // modified periodic (Sec. 2.4.3): wrap with exp(+-i phi)
    BC_MIR = 1,       // mirror, G parallel to the face: hat g_i(x_m) = hat g_ibar(x_n)
    BC_MIR_CONJ = 2,  // mirror, G normal to the face: conjugate + rewind (Sec. 2.4.4)
    // z faces of a slab cut out of a larger grid (the strips of Sec. 2.5):
    BC_HALO = 3,      // the neighbouring slab: value from the halo plane
    BC_HALO_PER = 4   // the neighbouring slab across the periodic global face:
                      // halo value times the wrap factor exp(+-i phi)
};

constexpr unsigned long long WAIT_NS = 2000000000ull;  // bound of every wait of a kernel: 2 s

struct MemberDesc {
    float2* state;        // n_slots time levels, each 7 planes
    float2* adj;          // adjoint sweep: 2 levels of 7 planes (or nullptr)
    float2* field;        // M(x) output (complex64 [N]) or nullptr
    const uint8_t* mask;  // per-site membrane bits 0..5 + phase bits 6..7
    long long N;          // sites
    long long plane;      // plane stride in sites
    long long tile0;      // first work-list tile of this member (site tiles)
    long long unit0;      // first row-unit of this member (bulk-copy sweep)
    long long cc0;        // first unit column of this member (bulk-copy sweep, z-marching form)
    int rpu;              // x-rows per unit of the bulk-copy sweep
    int rpu_adj;          // x-rows per unit of the bulk-copy adjoint sweep
    long long unit0_adj;  // first row-unit of this member (bulk-copy adjoint)
    // resident and two-step sweeps: where M goes at the signal step, for
    // launch_signal to sum (the field buffer, if it is written at that step
    // too); nullptr (two-step only): the sweep sums M itself
    float2* mout;
    int nx, ny, nz;
    int pitch;            // two-step sweep: length of the state's rows, with ghost columns
                          // (the other sweeps' rows are nx long)
    int bc[3];            // BcMode per axis
    double gG[3];         // gamma*G0, rad/(um ms)
    double dx;            // um
    float ctheta[3];      // -gG_a*dx*dt: reaction angle = f_k * sum_a ctheta_a * n_a
    float omega[4];       // 1/tau_p (Eq. tau_def)
    float eps[4];         // 1 - exp(-dt/T2_p), from expm1 in FP64; for the
                          // classical scheme dt/T2_p (its Euler source)
    float s_share;        // 1/(1+P): crossing share of a membrane link (Eq. B5)
    int axes;             // bit a set iff ctheta[a] != 0
    int memb;             // the geometry has at least one membrane link
    // exact division of site indices (< 2^28) by nx and ny: q = (n*m) >> s
    unsigned div_m[2];
    int div_s[2];
    // per-axis rotation tables (FP64-built): etab[off_a + n] =
    // (cos(ctheta_a n_a) - 1, sin(ctheta_a n_a)), offsets 0, nx, nx+ny, with
    // n_z = z0 + n (global plane index); or nullptr
    const float2* etab;
    // z extent within the whole grid: the member covers planes z0 .. z0+nz-1
    // of nzg (z0 = 0, nzg = nz unless the geometry is a slab)
    int z0, nzg;
    int zbc[2];           // BcMode of the low and high z face (bc[2] unless a slab)
    const float2* halo[2];  // slab halo planes (nx*ny complex64): hat g_5 of the
                          // plane below, hat g_6 of the plane above; or nullptr
    // membrane positions on the links (theta = 0 rule, Eqs. B4a-B4c):
    // dlt[(j-1)*plane + s] = distance in dx from s to the membrane on its
    // link to s + e_j; nullptr = half-link rule (Eq. B5) everywhere
    const float* dlt;
    float lrho;           // kappa dt / (eps_D dx): the coefficients depend on it only
    // membrane angles (one-plane D2Q5 grids, general-angle rule of Appendix
    // B): dth[(j-1)*plane + s] = signed angle between the membrane normal and
    // the link from s to s + e_j; nullptr = theta = 0 everywhere
    const float* dth;
    // the member's waveform: fw[k] = f_k as float (one entry past the end,
    // 0), Fw[k] = F_k = sum_{m<k} f_m dt (two entries past the end); the
    // run's shared tables unless the member has a waveform of its own
    const float* fw;
    const double* Fw;
    // step whose end signal partials (and field, if any) are this member's
    // own: its echo when it is shorter than the run; -1: the step control's
    int end_step;
    int moff;             // resident sweep, series: where its sites start among all members'
};
// Where the extents and faces lie decides how every thread of the register sweep loads
// them at its start: with nx .. pitch off a 16-byte word it took 0.4 us a step more (2-D,
// 1400 x 1100: 48.9 us for 48.4); with pitch and mout after the rest, where that sweep was
// as fast, the two-step sweep and the strips were 1 to 1.5 % slower.  That sweep is told
// the alignment; told to all kernels, it made the bulk-copy adjoint 1.5 % slower.
static_assert(offsetof(MemberDesc, nx) % 16 == 0 && offsetof(MemberDesc, pitch) == offsetof(MemberDesc, nx) + 12 &&
              offsetof(MemberDesc, bc) % 16 == 0 && sizeof(MemberDesc) % 16 == 0, "extents on one 16-byte word");

// Step control word in device memory.  Every block of a sweep reads k at its
// start.  The bulk-copy sweep's last CTA to be done with it (a two-level
// ticket, no waiting) advances k; after a register sweep a one-thread kernel
// does.  So a captured graph of steps replays from any step.  No kernel ever
// waits on it.
constexpr unsigned CTL_SHARDS = 32;   // first-level ticket counters (same-address atomics serialise)
struct StepCtl {
    int k;              // step index the next sweep performs
    unsigned done;      // shards of the current sweep whose blocks are all done (0 between sweeps)
    int sig_step;       // step whose end signal is reduced (-1: none)
    int field_step;     // step whose end field is written (-1: none)
    int slot_base;      // src slot = (k - slot_base) % slot_mod
    int slot_mod;       // dst slot = (k + 1 - slot_base) % slot_mod
    int series;         // 1: reduce the signal after every step
    int err;            // device-side error bits
    unsigned shard[CTL_SHARDS];   // blocks b % CTL_SHARDS == s of the current sweep that are done
};

struct SweepArgs {
    const MemberDesc* members;
    const long long* tile_start;  // n_members + 1 prefix of tiles
    int n_members;
    StepCtl* ctl;
    const float* f;               // waveform per step
    const double* F;              // F_k = sum_{m<k} f_m dt, per step
    double2* partial;             // per-tile (sum Re M, sum Im M)
    const float2* fac;            // [K+1][n_members][6] boundary factors of every step
    int links;                    // 1: a member has membrane positions (register sweep
                                  // variant with the Eqs. B4a-B4c rule); 2: and angles
    float w0, wxy, wz;            // equilibrium weights (register sweep, init):
                                  // D3Q7 1/4, 1/8, 1/8; D2Q5 1/3, 1/6, 0 (Sec. 2.3)
    unsigned long long test_wait_ns;  // tests of the timeout path only: > 0 makes each
                                  // consumer warp of the bulk-copy sweep and each thread of
                                  // the two-step sweep first wait, with this limit, on a
                                  // barrier nothing completes (0: off; resident sweeps: ResArgs)
    int zc;                       // bulk-copy sweep, z-marching form: units per column
                                  // (consecutive z-planes of the same rows; a power of two
                                  // that divides every member's nz), else 0
    int zc_log2;                  // log2(zc)
    long long n_cc;               // z-marching: columns of all members
    const long long* cc_start;    // z-marching: n_members + 1 prefix of columns
    int scheme;                   // 0 the hybrid scheme; 1 the classical LBM with the
                                  // reaction as a collision source (Appendix A, Eq. A12),
                                  // register sweep only: f and F are then read one step
                                  // ahead (f[k+1], F[k+1]), since the loop state hat g(t^k)
                                  // already holds step k's source
};

// ---- launchers (sweep.cu) ------------------------------------------------
cudaError_t launch_build_mask(const int32_t* labels, const uint8_t* phase_of_label, int n_labels,
                              int nx, int ny, int nz, const int bc[3], uint8_t* mask, int* err,
                              cudaStream_t st);
// Writes v to the control word (before a run of sweeps, which then advance
// it themselves); v.err < 0 leaves the error word as it is.
cudaError_t launch_ctl_set(StepCtl* ctl, const StepCtl& v, cudaStream_t st);
// Boundary factors of every step 0..K for every member, table[k][m][6], from
// each member's F table at k + F_shift (1 for the classical scheme, whose
// streamed populations already hold step k's source).
cudaError_t launch_factor_table(const MemberDesc* members, int n_members, int F_shift, long long K,
                                float2* table, cudaStream_t st);
cudaError_t launch_init(const SweepArgs& a, long long n_tiles, int block, int spt, int slot,
                        cudaStream_t st);
// Register sweep (one block per tile), then the one-thread step advance.
cudaError_t launch_sweep(const SweepArgs& a, long long n_tiles, int block, int spt, cudaStream_t st);
cudaError_t links_prepare();   // dynamic shared memory of the membrane-position sweeps
// Sums partial[tile_start[m]*per .. tile_start[m+1]*per) per member (tile_start NULL: [m*per ..
// (m+1)*per)).  steps =
// 2 (series after a two-step launch): the second step's partials follow at
// `stride`, and both steps enter the series.
cudaError_t launch_reduce(const double2* partial, const long long* tile_start, int per, int n_members,
                          double2* out, double2* series, long long series_stride,
                          const StepCtl* ctl, cudaStream_t st, int steps = 1, long long stride = 0);

// ---- bulk-copy sweep (sweep_tma.cu) --------------------------------------
// oz: the own rows of planes 5 and 6 go through the stage (wanted where
// planes are large, so those rows would otherwise come from DRAM a plane
// later); without it they are prefetched into registers with planes 3 and 4.
size_t tma_smem_bytes(int cap, int capx, int nst, int form);
int tma_partials_per_unit(int variant);
int tma_consumers(int variant);           // threads that have sites
int tma_sites_per_thread(int variant);
cudaError_t tma_prepare(int cap, int capx, int nst, int variant, int form, int* ctas_per_sm);
cudaError_t launch_sweep_tma(const SweepArgs& a, long long n_units, int cap, int capx, int nst, int variant, int form,
                             int grid, cudaStream_t st);

// ---- two-step sweep (sweep_pair.cu) --------------------------------------
// The state of a run on it has pair_ghost() ghost columns and rows on each side
// of every plane and rows of `pitch` columns, so all its steps are its own.
// One work item: columns [x0, x0 + w) x [y0, y0 + h), planes [z0, z1) of
// member m; x0 even.  The items of a member are consecutive, members in order;
// ex (pairs of columns in a row of a block, >= (w + 5) / 2) and hb (>= h) are the
// member's, those of its tensor maps' boxes.
struct PairItem {
    int m, x0, w, y0, h, z0, z1, ex, hb;
};
int pair_threads();            // threads of a block: ex (hb + 2) may not exceed them,
int pair_max_row();            // nor ex this
int pair_ghost();
struct alignas(128) PairMap {   // a tensor map (CUtensorMap)
    unsigned char b[128];
};
// Maps of a run: [2][n_members][2 levels], boxes of hb + 2 and of hb + 3 rows.
cudaError_t pair_encode_map(PairMap* out, const void* level, const MemberDesc& d, int ex, int rows);
// general: the waveform may take values other than 0 and +-1.
cudaError_t pair_prepare(bool general, int* ctas_per_sm);
// steps = 2: k -> k + 2, or 1: k -> k + 1 (the odd step of a run).  Signal
// partials (members without mout): one per item; in series mode always, and the
// second step's follow at n_items.
cudaError_t launch_sweep_pair(const SweepArgs& a, const PairItem* items, const PairMap* maps, int n_items, bool general,
                              int steps, cudaStream_t st);
cudaError_t launch_pair_init(const MemberDesc* members, int n_members, long long max_plane, cudaStream_t st);
// Level src of every member to level src ^ 1, from rows of nx to the layout with ghosts or back.
cudaError_t launch_pair_relayout(const MemberDesc* members, int n_members, long long max_plane, int src, bool to_pair,
                                 cudaStream_t st);

// ---- resident sweep (sweep_resident.cu) -----------------------------------
// One block of a small grid: all of x, rows [y0, y0 + hy), planes [z0, z0 + hz)
// of member m; nbr: the blocks across its -y, +y, -z, +z faces, or what is there
// instead; recv: where a face's values start among the n_recv it receives (one
// per site of the face; with membrane positions three);
// dest: where they start among the neighbour's.
constexpr int RES_SELF = -1, RES_MIRROR = -2;
struct ResBlock {
    int m, y0, hy, z0, hz, nbr[4], recv[4], dest[4], n_recv;
};
struct ResArgs {
    const ResBlock* blocks;
    uint4* packets;               // [n_blocks][4 turns][recv_max]
    const uint4* inbox;           // where they are waited for: packets (tests of the time-out:
                                  // a place that nobody sends to)
    unsigned long long wait_ns;   // bound of a wait
    int recv_max;
    int k0, n_steps;              // steps k0 .. k0 + n_steps - 1
    int lsrc, ldst;               // time levels read and written
    unsigned stamp0;              // stamp of step k0's packets
    int sig_step, field_step;     // as in StepCtl; a member's own end step goes before them
    int links;                    // 1: a member has membrane positions
    int max_links;                // listed links of a block at most (rounded up to even)
    int series;                   // strips: zpart[n][block] = the block's part of Z after each step
    double2* zpart;
    int levels;                   // 1: the levels of steps k0 .. k0 + n_steps - 1 go to the member's
                                  // adj, one after the other from slot level0 (gradient segments)
    int level0;
    float2* mser;                 // blocks, series: M after each step, [n_steps][mstride], a
    long long mstride;            // member's from moff on; else nullptr
};
int resident_max_sites();         // sites of a block
size_t resident_smem(int sites, int recv, bool d2);
// Membrane positions: shared memory per listed link, and the most a block lists
// (*out, zeroed before).
size_t resident_link_bytes();
cudaError_t launch_resident_links(const MemberDesc* members, const ResBlock* blocks, int n_blocks, bool d2, int* out,
                                  cudaStream_t st);
cudaError_t launch_resident(const SweepArgs& a, const ResArgs& r, int n_blocks, int max_sites, size_t smem, bool d2,
                            bool general, cudaStream_t st);
// 2-D grids (D2Q5) in strips of whole rows (sweep_strip.cu): rows of a block at
// most for this nx (0: too wide), its shared memory.
int strip_rows(int nx);
size_t strip_smem(int nx, int rows);
cudaError_t launch_strip(const SweepArgs& a, const ResArgs& r, int n_blocks, int max_nx, size_t smem, bool general,
                         cudaStream_t st);
// out[m][parts], to be summed; rows: the thread sums of the bulk-copy sweep
cudaError_t launch_signal(const MemberDesc* members, int n_members, bool rows, int block, int spt, int parts, double2* out,
                          cudaStream_t st);
// Parts of Z after each step from mser, with the same thread sums: [n_steps][n_members][parts].
cudaError_t launch_series_parts(const MemberDesc* members, int n_members, bool rows, int block, int spt, int parts,
                                const float2* mser, long long mstride, int n_steps, double2* zpart, cudaStream_t st);
// Their sums: zpart[n][n_blocks], a member's from block_start[m] to block_start[m + 1].
cudaError_t launch_resident_series(const double2* zpart, const int* block_start, int n_members, int n_blocks, int n_steps,
                                   long long k0, long long stride, double2* series, cudaStream_t st);

// ---- adjoint (adjoint.cu) -------------------------------------------------
// Per-tile gradient accumulators: [0..3] sum <lambda, w M - g> per phase
// (d/d omega_p), [4..7] sum <mu, -exp(i theta) g'> per phase (d/d eps_p),
// [8] sum over membrane links <nu, v - o> (d/d s).
constexpr int NGACC = 9;

struct AdjointArgs {
    const MemberDesc* members;    // state = the segment of forward levels
    const long long* tile_start;
    int n_members;
    int k;                        // adjoint step: nu^k -> nu^(k-1)
    int first;                    // 1: lambda^K is uniform, lam_init[member]
    int fwd_slot;                 // level of u^(k-1) in the member's state
    int lam_parity;               // nu^k is adj level lam_parity
    const double2* lam_init;      // per member Z / (N |Z|)
    float fprev;                  // f_(k-1)
    double* gacc;                 // per tile NGACC doubles, accumulated
    const float2* ftab;           // [K+1][n_members][6] boundary factors
    const long long* unit_start;  // bulk-copy adjoint: row-unit prefix
    int* ctl_err;                 // error word of the step control
    float w0, wxy, wz;            // equilibrium weights (register adjoint; the
                                  // bulk-copy adjoint has the D3Q7 ones built in)
};
// run: consecutive tiles per block (the block keeps its gradient partials over them)
cudaError_t launch_adjoint(const AdjointArgs& a, long long n_tiles, int block, int spt, int run, cudaStream_t st);
// Sums gacc slots [tile_start[m]*per, tile_start[m+1]*per) per member.
// resident adjoint (adjoint_resident.cu): steps a.k, a.k - 1, .. of r.n_steps; the
// forward level of step a.k - 1 is in slot a.fwd_slot of the member's state, that of
// the next in the slot before; nu^k is adj level r.lsrc, the result goes to
// r.ldst; the sites' sensitivities go to the member's field, floats [step][3][N],
// and launch_adjoint_sum adds them to gacc as the bulk-copy adjoint would (its
// grid, consumer threads, sites per thread and slots per unit).
int adj_resident_max_sites();
size_t adj_resident_smem(int sites, int recv);
cudaError_t launch_adjoint_sum(const AdjointArgs& a, long long n_units, int n_steps, int grid, int threads, int spt,
                               int slots, cudaStream_t st);
cudaError_t launch_adjoint_resident(const AdjointArgs& a, const ResArgs& r, int n_blocks, int max_sites, size_t smem,
                                    bool general, cudaStream_t st);
cudaError_t launch_reduce_grad(const double* gacc, const long long* tile_start, int per, int n_members, double* out,
                               cudaStream_t st);
// bulk-copy adjoint (adjoint_tma.cu)
int adj_tma_slots_per_unit();
int adj_tma_max_sites(int shape);
int adj_tma_consumers(int shape);          // threads that have sites; sites per thread: 2 for shape 0, else 1
cudaError_t adj_tma_prepare(int cap, int nst, int shape, int* ctas_per_sm);
cudaError_t launch_adjoint_tma(const AdjointArgs& a, long long n_units, int cap, int nst, int shape, int grid,
                               cudaStream_t st);

}  // namespace lbmbt
