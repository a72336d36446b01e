// qym_internal.cuh -- device helpers and launch declarations shared by the
// libqym translation units (sm_103a). Not part of the public ABI.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <utility>
#include <vector>

#include "../../include/qym.h"
#include "pair64.cuh"

namespace qym {

constexpr double kPi = 3.14159265358979323846;
constexpr int kHermMaxClusters = 160;  // entries of Dev::hcl (2 x 152 CTAs in clusters of 2 or more)

// ---------------------------------------------------------------- layout
// Units and partial slots of the pair-symmetric mixed kick (kick.cu): groups of G
// i-blocks of kSymBlock positions against ranges of rh half tiles (128
// positions); G = 0: not in use. A row's slots: one per range from its own block,
// then one per group of earlier i-blocks.
constexpr int kSymBlock = 512;
struct SymShape {
    int32_t G = 0, rh = 0, nc = 0, splits = 0;  // nc ranges; splits slots in all
};

// Device state of a context. Rows of all systems are concatenated; each
// system's star sits at its first row with Q = v = 0. Positions and
// velocities are float64 structure-of-arrays [3][rows].
struct Dev {
    int64_t rows = 0;
    int32_t nsys = 0;
    int64_t *offsets = nullptr;   // [nsys+1]
    int32_t *sys_of = nullptr;    // [rows] system of each row
    double *m = nullptr;          // [rows]
    double *q = nullptr, *v = nullptr;     // [3][rows] current state (DH)
    double *q1 = nullptr, *v1 = nullptr;   // [3][rows] Kepler output / step scratch
    double *rH = nullptr;         // [rows] Hill radius used by this step's encounter test
    double *rH_fixed = nullptr;   // [rows] Hill radii computed at init (hill_fixed)
    // kick operand packs, float32 (rebuilt from the FP64 state every step)
    float4 *pk_pos = nullptr;     // (x_hi, y_hi, z_hi, G m)
    float4 *pk_lo = nullptr;      // (x_lo, y_lo, z_lo, c = 2 rho^2, rho the crude reach)
    float *amag = nullptr;        // [rows] |a_int| of the last kick
    float *rH_bound = nullptr;    // [rows] Hill radius bound used by the crude test
    double *apart = nullptr;      // [splits][3][rows] kick partial accelerations
    int32_t splits = 1;
    SymShape sym;                 // pair-symmetric kick (one system in Morton order)
    int4 *sym_items = nullptr;    // its units: i-blocks [x, y), half tiles [z, w)
    int32_t sym_nitems = 0;
    int32_t *kick_cnt = nullptr;  // arrivals per i-block: with it the kick's last CTA of
                                  // each i-block adds the slots into slot 0 (kick.cu)
    int32_t *wh_flag = nullptr;   // [nsys] 1: this step of the system is integrated whole
                                  // by the Hermite (whole.cu); its sets are not
    double *vpre = nullptr;       // [3][rows] velocities entering the first kick
    // kick work items (one CTA each): (i0, i1, j0, j1) and the partial slot
    int4 *items = nullptr;
    int32_t *item_slot = nullptr;
    int32_t nitems = 0;
    int32_t item_chunk = 0;       // items == NULL (one system): j rows per split
    int32_t item_parts = 1;       // splits per chunk, of FOLD rows each (mixed kick; 1: whole)
    int32_t batch = 0;            // mixed kick of several systems: its sums keep their order
    // momentum reduction
    int4 *mchunks = nullptr;      // (row0, row1, sys, -) chunks of at most 1024 rows
    int32_t nmchunks = 0;
    double *mpart = nullptr;      // [nmchunks][3]
    int32_t *sys_chunk0 = nullptr;  // [nsys+1] first chunk of each system
    double *S = nullptr;          // [nsys][3] sum of m v over bodies
    // encounters
    int2 *cand = nullptr;         // crude candidate pairs (i < j)
    int64_t max_cand = 0;
    int4 *fchunk = nullptr;       // (i, j0, j1, -): j chunks [j0, j1) of row i whose crude
                                  // minimum fell below c_i, re-tested pair by pair
    int64_t max_fchunk = 0;
    int2 *enc = nullptr;          // rigorous encounter pairs
    int64_t max_enc = 0;
    int32_t *rescan = nullptr;    // rows whose crude bounds were exceeded
    int32_t *set_start = nullptr; // [max_sets+1]
    int32_t *set_mem = nullptr;   // [max_members]
    double *rcrit = nullptr;      // [max_sets]
    int32_t max_sets = 0, max_members = 0;
    // Hermite schedule: block steps of the set each row was in during the
    // last step (0 for rows in no set), the per-CTA queue of sets in order of
    // predicted cost, and the set each thread-block cluster takes (-1: none)
    int32_t *hcost = nullptr;     // [rows]
    int32_t *hsetcost = nullptr;  // [max_sets] largest hcost over each set's members
                                  // (raised by the set builder, cleared by the plan)
    int32_t *hq = nullptr;        // [max_sets]
    int32_t *hcl = nullptr;       // [kHermMaxClusters]
    int32_t *uf = nullptr;        // [rows] union-find parents, kept at -1 when idle
    int64_t *log = nullptr;       // [max_log][3] encounter records of one qym_step call
    int64_t max_log = 0;
    // heavy bodies of each system (mixed kick: their pull is summed in FP64)
    int32_t *heavy_rows = nullptr;   // ascending rows, system by system
    int32_t *heavy_start = nullptr;  // [nsys+1]
    double *heavy_thr = nullptr;     // [nsys] mass threshold (+inf: no split)
    double *kmu = nullptr;           // [nsys][3] mu = G m0, sqrt(mu), 1/mu (E_Kep)
    double *hfac = nullptr;          // [rows] (m / 3 m0)^(1/3): r_H = |Q| hfac (0 for stars)
    int32_t heavy_split = 0;         // 1 when the kick in use is the mixed one
    int32_t escape_reach = 0;        // 1: the crude reach is the escape-velocity one
    // counters (device): see Counters below
    unsigned long long *ctr = nullptr;
    int32_t *status = nullptr;    // QYM_ST_* bits
    // a system's step split over several GPUs: this context computes the
    // rows [own_lo, own_hi) (kick rows, finisher, Kepler drift, the
    // candidates of those rows, the Hermite of the sets whose lowest row is
    // among them); own_hi = 0: every row
    int64_t own_lo = 0, own_hi = 0;
    int32_t *set_root = nullptr;  // [max_sets] lowest row of each set (sets are numbered by it)
    int32_t log_refine = 1;       // the rigorous test logs its pairs (0: the split's import does)
    // order of the bodies in the kick's packs and partial sums (sort.cu):
    // position p holds row perm[p], row r sits at position inv[r]; NULL: row order
    int32_t *perm = nullptr, *inv = nullptr;
    int32_t *vmax = nullptr; // [nsys] largest |v| after the first kick (float bits), for the
                             // binned search; NULL: not kept
    float4 *far = nullptr;   // [rows] (offset from the tile's reference point, G m) in that order
    int32_t tiles_ready = 0; // 1: far and tile hold the present packs' tiles
    float4 *tile = nullptr;  // [3 x tiles] reference point and radius, box min, box max
};

// device counters, indices into Dev::ctr
enum Ctr : int {
    C_NCAND = 0,     // candidates this step (reset per step)
    C_NENC,          // encounter pairs this step (reset per step)
    C_NRESCAN,       // rows to re-search this step (reset per step)
    C_NSETS,         // sets this step (written by the set builder)
    C_NMEM,          // set members this step
    C_LOG,           // records in the encounter log (per qym_step call)
    C_SUM_CAND,      // running sums over the steps of one qym_step call
    C_SUM_ENC,
    C_SUM_SETS,
    C_MAX_SET,
    C_SUM_KITER,
    C_SUM_HSTEPS,
    C_SUM_RESCAN,
    C_STEP,          // step index within the current qym_step call
    C_MAX_HSET,      // most Hermite steps taken by one set in one step
    C_HSMALL,        // next set for the Hermite kernel's per-CTA queue (reset per step)
    C_NFCHUNK,       // flagged (row, j chunk) entries of the last search kick
    C_FCDONE,        // CTAs of the chunk re-test done (its last CTA resets both)
    C_HNQ,           // sets in the Hermite kernel's per-CTA queue this step
    C_NACTIVE,       // overlapping tile pairs of the binned search (reset per step)
    C_COUNT
};

// a step's counters join the call's; the next step's start from zero
__device__ __forceinline__ void step_counters_end(unsigned long long *ctr) {
    ctr[C_SUM_CAND] += ctr[C_NCAND];
    ctr[C_SUM_ENC] += ctr[C_NENC];
    ctr[C_SUM_RESCAN] += ctr[C_NRESCAN];
    ctr[C_STEP] += 1;
}
__device__ __forceinline__ void step_counters_begin(unsigned long long *ctr) {
    ctr[C_NCAND] = 0;
    ctr[C_NACTIVE] = 0;
    ctr[C_NENC] = 0;
    ctr[C_NRESCAN] = 0;
    ctr[C_NSETS] = 0;
    ctr[C_HSMALL] = 0;
    ctr[C_NFCHUNK] = 0;
    ctr[C_FCDONE] = 0;
}

// ---------------------------------------------------------------- helpers
// one MUFU instruction; inputs here are squared separations, never denormal
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

struct alignas(32) D4 {
    double x, y, z, w;
};

__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = a + b;
    float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

__device__ __forceinline__ float warp_min(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = fminf(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}

// split a double into a float pair with hi + lo == x to ~2^-48 relative
__device__ __forceinline__ void split_ds(double x, float &hi, float &lo) {
    hi = __double2float_rn(x);
    lo = __double2float_rn(x - (double)hi);
}

// pull of the heavy bodies hs[k0], hs[k0 + step], ... below nh (ascending rows,
// i excluded) on the body at (x, y, z): sum -G m_h (r_i - r_h) / |r_i - r_h|^3,
// each pair to FP64 accuracy on the FP32 pipes (pair64.cuh), seven FP64
// instructions instead of 25; lengths scaled by the body's own largest
// coordinate, weights each by itself
__device__ __forceinline__ void heavy_pull(const int32_t *hs, int k0, int step, int nh, int64_t i,
                                           double x, double y, double z, const double *q,
                                           const double *m, int64_t R, double G, double &ax,
                                           double &ay, double &az) {
    if (k0 >= nh) return;
    const int hm = max(p64::hi_abs(x), max(p64::hi_abs(y), p64::hi_abs(z)));
    const int kb = (hm >> 20) - 1023;
    const bool kb_ok = kb >= -200 && kb <= 200;
    const int kbs = kb_ok ? kb : 0;
    const p64::F3 X = p64::split3(p64::scale2(x, kbs)), Y = p64::split3(p64::scale2(y, kbs));
    const p64::F3 Z = p64::split3(p64::scale2(z, kbs));
    for (int k = k0; k < nh; k += step) {
        const int64_t h = hs[k];
        if (h == i) continue;
        const double qx = q[h], qy = q[R + h], qz = q[2 * R + h], gm = G * m[h];
        const int ka = (p64::hi_abs(gm) >> 20) - 1023;
        const p64::F3 r2 = p64::norm2(p64::diff(X, p64::split3(p64::scale2(qx, kbs))),
                                      p64::diff(Y, p64::split3(p64::scale2(qy, kbs))),
                                      p64::diff(Z, p64::split3(p64::scale2(qz, kbs))));
        const double dx = x - qx, dy = y - qy, dz = z - qz;
        double s;
        const bool ka_ok = ka >= -200 && ka <= 200;
        const int kas = ka_ok ? ka : 0;
        const bool ok = p64::g_over_r3(p64::split3(p64::scale2(gm, kas)), r2, rsqrt_ftz(r2.h),
                                       (uint64_t)(int64_t)(kas - 3 * kbs) << 52, s);
        if (!(ok && kb_ok && ka_ok && p64::r2_fits(r2.h))) {
            const double d2 = dx * dx + dy * dy + dz * dz;
            const double ri = rsqrt(d2);
            s = gm * (ri * ri) * ri;
        }
        ax -= s * dx;
        ay -= s * dy;
        az -= s * dz;
    }
}

// The same in FP64 by one thread, body after body: what a batch's finisher adds. Its
// encounters amplify a last place by up to 1e9 within a few steps, so its pulls keep
// their roundings (512 systems of 2 planets, 1.06e6 rows: the finisher 101 us, 71 with heavy_pull).
__device__ __forceinline__ void heavy_pull_fp64(const int32_t *hs, int nh, int64_t i, double x,
                                                double y, double z, const double *q, const double *m,
                                                int64_t R, double G, double &ax, double &ay, double &az) {
    for (int k = 0; k < nh; ++k) {
        const int64_t h = hs[k];
        if (h == i) continue;
        const double dx = x - q[h], dy = y - q[R + h], dz = z - q[2 * R + h];
        const double r2 = dx * dx + dy * dy + dz * dz;
        const double ri = rsqrt(r2);
        const double s = G * m[h] * (ri * ri) * ri;
        ax -= s * dx;
        ay -= s * dy;
        az -= s * dz;
    }
}

// whether mass m reaches the threshold thr > 0 (their bits compared: FP64
// comparisons hold the FP64 pipe; negative masses and NaN do not reach it)
__device__ __forceinline__ bool mass_reaches(double m, double thr) {
    const unsigned long long t = (unsigned long long)__double_as_longlong(thr);
    return (unsigned long long)__double_as_longlong(m) - t <= 0x7ff0000000000000ull - t;
}

// Heavy list of one system by one CTA of 1024 threads: the first QYM_HEAVY_CAP
// bodies (ascending rows) with m >= heavy_mass * m[0]; hl[QYM_HEAVY_CAP]
// receives their count. A thread takes up to 32 consecutive rows with all loads
// in flight (one row per thread and round, with three barriers each, took 21 us
// for 16384 rows). s: 33 ints of shared memory.
__device__ __forceinline__ void heavy_list(int64_t rows, const double *m, double heavy_mass,
                                           int32_t *hl, int *s) {
    const double thr = heavy_mass * m[0];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int per = (int)min((int64_t)32, (rows + 1022) >> 10);  // rows per thread
    int base = 0;
    for (int64_t c = 1; c < rows; c += per * 1024) {
        const int64_t r0 = c + per * (int64_t)threadIdx.x;
        unsigned hv = 0;
#pragma unroll 32
        for (int k = 0; k < 32; ++k)
            if (k < per && r0 + k < rows && mass_reaches(m[r0 + k], thr)) hv |= 1u << k;
        const int cnt = __popc(hv);
        int inc = cnt;
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        __syncthreads();
        if (lane == 31) s[w] = inc;
        __syncthreads();
        const int ws = s[lane];
        const int before = __reduce_add_sync(0xffffffffu, lane < w ? ws : 0);
        int pos = base + before + inc - cnt;
        base += __reduce_add_sync(0xffffffffu, ws);
        for (; hv; hv &= hv - 1, ++pos)
            if (pos < QYM_HEAVY_CAP) hl[pos] = (int32_t)(r0 + __ffs(hv) - 1);
    }
    if (threadIdx.x == 0) hl[QYM_HEAVY_CAP] = base < QYM_HEAVY_CAP ? base : QYM_HEAVY_CAP;
}

// the calling thread's context-free error message (qym_last_error(NULL))
void set_thread_error(const std::string &msg);

// The valid slots of position pr under the pair-symmetric kick, k = 0 .. n - 1:
// the ranges that reach its own i-block b or lie past it, then the groups that
// start before b
struct SymSlots {
    int c0, n1, n;
    __device__ __forceinline__ SymSlots(const SymShape &y, int64_t pr) {
        const int b = pr > 0 ? (int)((pr - 1) / kSymBlock) : 0;
        c0 = 4 * b / y.rh;
        n1 = y.nc - c0;
        n = n1 + (b + y.G - 1) / y.G;
    }
    __device__ __forceinline__ int slot(int k, int nc) const { return k < n1 ? c0 + k : nc + k - n1; }
};

// ---------------------------------------------------------------- launches
// Launches in a chain: each kernel may be set up while the one before it in
// the stream still runs (programmatic dependent launch) and waits for it, and
// for the visibility of all it wrote, in chain_wait(), its first statement. The
// kernels of a small step are a few microseconds each, so the ~1 us a launch
// otherwise takes between them counts. Only then does it let the next kernel be
// set up: allowed before the wait, the kernels of a chain pile up on the SMs, and
// a later one finds room on a few of them only (a drift of 16384 bodies took 65
// us instead of 41).
__device__ __forceinline__ void chain_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <class... P, class... A>
cudaError_t launch_chain(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                         A &&...args) {
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

// Each returns cudaSuccess or the launch error. All work goes on `st`.

// kepler.cu
struct KeplerArgs {
    int64_t n;            // bodies
    const double *q0, *v0; // [3][ld] inputs
    double *q1, *v1;       // [3][ld] outputs
    int64_t ld;            // leading dimension (stride between x, y, z blocks)
    const int64_t *rows;   // optional row map: body k is row rows[k]; NULL: row row0 + k
    int64_t row0;
    double mu, sqmu, imu, dt;   // mu with sqrt(mu) and 1/mu (all rows, when kmu is NULL)
    int32_t solver, guess, max_iter;
    const float *mlp_w;    // guess network weights (QYM_GUESS_MLP) or NULL
    double *x_out;         // [n] or NULL
    double *x0_out;        // [n] starting guesses, or NULL
    // training rows (u1..u4, t) [log_cap][5], or NULL; row of body k:
    // (*log_base + *log_step) * n + k, or k when log_step is NULL
    float *log;
    int64_t log_cap;
    const unsigned long long *log_base, *log_step;
    int32_t *iters;        // [n] or NULL
    int32_t *status;       // or NULL
    unsigned long long *iter_sum;  // or NULL
    // per-row mu, sqrt(mu), 1/mu: kmu[3 sys_of[row] + 0..2] when kmu != NULL
    const int32_t *sys_of;
    const double *kmu;
};
cudaError_t launch_kepler(const KeplerArgs &a, cudaStream_t st);

// mlp.cu: learned Kepler guess, inference and training
size_t mlp_workspace_bytes();
cudaError_t launch_mlp_forward(int64_t n, const float *w, const float *u, float *y, cudaStream_t st);
cudaError_t launch_mlp_grad(int64_t n, const float *w, const float *rows, float *grad, float *loss,
                            void *work, cudaStream_t st);
cudaError_t launch_mlp_adam(float *w, float *m, float *v, const float *grad, int64_t t, float lr,
                            float beta1, float beta2, float eps, cudaStream_t st);
cudaError_t launch_mlp_train(float *w, float *m, float *v, int64_t t0, const float *rows, int64_t n,
                             int64_t batch, int32_t epochs, float lr, float lr_final, float *losses,
                             void *work, cudaStream_t st);

// step kernels (step.cu)
// sum m v per system into d.S; for_drift: only for the drift that follows, which
// adds a small system's chunks itself (one launch less)
cudaError_t launch_momentum(const Dev &d, cudaStream_t st, bool for_drift = false);
int momentum_launches(const Dev &d, bool for_drift);
// kick_span: the time of the kick(s) between this pack and the Kepler drift
// (tau/2, or tau when two half kicks are merged); it sizes the crude reach.
// ctr_end, ctr_begin: also count the step that ends with this drift, and clear
// the counters of the step that begins after it
cudaError_t launch_drift_pack_from(const Dev &d, const double *qs, const double *vs,
                                   double h_close, double h_open, double tau, double a_E,
                                   double G, int flag_next, int hill_fixed, cudaStream_t st,
                                   double kick_span, double a_allow = 1.01, int ctr_end = 0,
                                   int ctr_begin = 0);
// a_allow: the bound on |a| / |a of the last kick| that the crude reach of the
// preceding pack assumed (checked when check != 0)
// skip_whole: leave v of the systems flagged in d.wh_flag (their step was
// integrated whole: no second kick)
cudaError_t launch_kick_finish_v(const Dev &d, double *v, const double *q, double dt, double G,
                                 int check, int hill_fixed, cudaStream_t st,
                                 double a_allow = 1.01, int skip_whole = 0);
cudaError_t launch_hill_init(const Dev &d, double G, cudaStream_t st);
cudaError_t launch_to_dh_impl(const Dev &d, int inverse, double *vout, double *mt_scratch,
                              cudaStream_t st);

// kick.cu
struct KickTune {
    int32_t threads = 128;  // threads per CTA
    int32_t ipt = 2;        // i rows per thread
    int32_t splits = 1;     // j splits per system
};
// flag: what a pass over the tiles does
enum KickMode {
    KICK_FORCE = 0,        // the interaction sums only
    KICK_SEARCH = 1,       // the sums and the crude encounter search
    KICK_SEARCH_ONLY = 2,  // the crude encounter search alone (no sums written)
};
cudaError_t launch_kick_tiles(const Dev &d, int prec, int flag, double G, int threads, int ipt,
                              cudaStream_t st);
cudaError_t launch_accel_single(int64_t rows, const double *m, const double *q, double *a,
                                double G, int prec, double heavy_mass, void *work,
                                size_t work_bytes, cudaStream_t st);
size_t accel_single_workspace(int64_t rows, int prec);
// items of the i rows in [i_lo, i_hi) (default: all rows) against all j
void kick_items_host(const int64_t *offsets, int32_t nsys, const KickTune &t,
                     int4 *items, int32_t *slots, int32_t *nitems, int32_t *splits_used,
                     int32_t max_items, int64_t i_lo = 0, int64_t i_hi = INT64_MAX,
                     int32_t align = 1);
KickTune default_kick_tune(int64_t iblocks_nb, int64_t nbmax, int prec, int64_t max_splits);
SymShape sym_shape(int64_t nb, int64_t max_slots);
void sym_items_host(int64_t nb, const SymShape &y, std::vector<int4> &items);
constexpr int kKickTile = 256;  // j rows per shared-memory tile of the kick
int32_t kick_items_count(const int64_t *offsets, int32_t nsys, const KickTune &t,
                         int64_t i_lo = 0, int64_t i_hi = INT64_MAX);

// sort.cu: Morton order of a system's bodies for the kick
struct SortScratch {
    int *box;              // [6]
    uint32_t *k0, *k1;     // [rows] keys
    int32_t *v0, *v1;      // [rows] rows
    uint32_t *hist;        // [256 * sort_blocks(rows)]
};
int64_t sort_blocks(int64_t n);
// with hl, also the heavy list (heavy_list below) of the same rows
cudaError_t launch_sort_rows(int64_t rows, const double *q, const SortScratch &s, int32_t *perm,
                             int32_t *inv, cudaStream_t st, const double *m = nullptr,
                             double heavy_mass = 0.0, int32_t *hl = nullptr);
int sort_launches(int64_t rows);  // kernels launch_sort_rows enqueues (without hl)
cudaError_t launch_heavy_list(int64_t rows, const double *m, double heavy_mass, int32_t *hl,
                              cudaStream_t st);

// search.cu: candidates by spatial binning after the Kepler drift
struct SearchArgs {
    double tau, a_E;
    float4 *box_lo, *box_hi; // [rows] widened boxes by position
    float4 *x0h, *x0l, *x1h, *x1l, *v0f, *v1f;  // [rows] by position (x0h.w: a_E r_H)
    int *tbox_bits;          // [6 x tiles] tile boxes: min x, y, z, -max x, y, z as ordered
                             // integer images (reset to INT_MAX every step)
    const int32_t *tile0;    // [nsys] first tile of each system
    const int4 *tiles;       // (system, p0, p1, -)
    int32_t ntiles;
    const int2 *tpairs;      // (tile I, tile J), I <= J, same system
    int64_t ntpairs;
    int2 *active;            // [ntpairs] tile pairs whose boxes overlap (count: C_NACTIVE)
};
cudaError_t launch_binned_search(const Dev &d, const SearchArgs &s, double tau, double a_E,
                                 cudaStream_t st);
void search_tiles_host(const int64_t *offsets, int32_t nsys, std::vector<int4> &tiles,
                       std::vector<int2> &tpairs);

// encounter.cu
struct SetScratch {
    int32_t *blk, *sid, *size, *fill;
    unsigned long long *rc_bits;
};
cudaError_t launch_refine(const Dev &d, double tau, double a_E, cudaStream_t st);
cudaError_t launch_sets_impl(const Dev &d, const qym_params &p, const SetScratch &s, cudaStream_t st);
bool sets_one(const Dev &d);      // whether one CTA builds the sets and plans the Hermite
int sets_launches(const Dev &d);  // kernels from the sets to the Hermite's plan
int hermite_clusters(const Dev &d, const qym_params &p);
cudaError_t launch_pair_test(int64_t rows, const double *q0, const double *v0, const double *q1,
                             const double *v1, const double *rH, double tau, double a_E,
                             int64_t npairs, const int32_t *pairs, double *d2, int32_t *flag,
                             cudaStream_t st);

// hermite.cu
cudaError_t hermite_prepare();
cudaError_t launch_transition(int64_t n, const double *s, double rc, double *K, double *Kp,
                              double *Kpp, cudaStream_t st);
cudaError_t launch_hermite(const Dev &d, const qym_params &p, double tau, cudaStream_t st);

// whole.cu: the whole-system Hermite (Sec. 2.3, last paragraph)
enum WholeCtl { WC_NA = 0, WC_DONE, WC_NCH, WC_COUNT };
struct WholeArgs {
    int64_t R;           // rows of the context's [3][R] arrays
    int64_t r0;          // the system's star row; its bodies are rows r0+1 .. r0+nb
    int64_t ld;          // stride of the scratch arrays' coordinates
    int32_t nb;          // bodies
    int32_t grid;        // CTAs of the force kernel
    const double *m;
    double G, m0, eps2, eta, eta_s, T, sg, tick;
    int64_t max_steps;   // block steps
    double *x, *u, *xp, *up, *a0, *j0;  // [3][ld]
    // the prediction split into float hi + lo parts for the light partners'
    // FP32 pair terms: (x, y, z, G m) and (x, y, z, -) of the position, the
    // velocity's the same; heavy bodies (m >= heavy_thr) enter at G m = 0 and
    // are summed in FP64 over `heavy` instead
    float4 *pf_hi, *pf_lo, *vf_hi, *vf_lo;  // [ld]
    double heavy_thr;
    const int32_t *heavy;  // the system's heavy bodies (indices of its bodies, ascending)
    int32_t nheavy;
    double *part;        // [max(grid, nb)][6] partner-range sums
    long long *ti;       // [nb] time of each body (ticks of |tau| 2^-48)
    int32_t *lev;        // [nb] step level
    int32_t *act;        // [nb] bodies of the block step
    int32_t *ctl;        // [WC_COUNT]
    long long *tn, *steps;
    int32_t *status;
};
cudaError_t launch_wh_trigger(const Dev &d, double planet_mass, int32_t *flag, cudaStream_t st);
cudaError_t launch_wh_start(const WholeArgs &w, const double *q, const double *vpre, cudaStream_t st);
cudaError_t launch_wh_blocks(const WholeArgs &w, int nblocks, cudaStream_t st);
cudaError_t launch_wh_store(const WholeArgs &w, double *q1, double *v1, cudaStream_t st);

// energy.cu
// One system: nranges items (CTAs) per i-block, no tables. A batch: tables (device) of
// the i-blocks (first row, last row + 1, end of the system, its star row), of the items
// (i-block, range), and of each system's first i-block and item.
struct EnergyPlan {
    const int4 *blocks = nullptr;
    const int2 *items = nullptr;
    const int32_t *block0 = nullptr, *item0 = nullptr;  // [nsys+1]
    int32_t nblocks = 0, nitems = 0;
    int32_t range = 0, nranges = 0;  // j rows per item; items per i-block (one system)
};
struct EnergyTables {
    std::vector<int4> blocks;
    std::vector<int2> items;
    std::vector<int32_t> block0, item0;
};
EnergyPlan energy_plan(const int64_t *offsets, int32_t nsys, EnergyTables *t);  // t: for a batch
int64_t energy_partials(const EnergyPlan &pl);  // doubles of `part`
cudaError_t launch_energy(const EnergyPlan &pl, int32_t nsys, const int64_t *offsets, int64_t R,
                          const double *m, const double *q, const double *v, double G, double *part,
                          double *E, cudaStream_t st);

}  // namespace qym
