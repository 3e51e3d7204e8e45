// pp_propagate.cu -- per-mode Dirac propagation, projection and momentum sum
// (Sec. II.A of arXiv 1704.08919: Eqs. (kin_mom), (free_spin1), (wf_init),
// (dirac_eq_mom), (pair_prod_homo); Eq. (opt_prob)).
//
// Reduction used on the GPU.  For a field in the x-y plane the Hermitian
// operator O = p_z gamma^5 + sigma_z (x) sigma_z (gamma^5 = sigma_x (x) 1 in the
// Dirac representation) commutes with H(t) = alpha.(p - A(t)) + beta at every
// t, and O^2 = (1 + p_z^2) 1.  Each eigenspace of O (eigenvalue s eps_perp,
// eps_perp = sqrt(1 + p_z^2), s = +-1) is invariant and holds one positive- and
// one negative-energy state; in a fixed orthonormal basis of that eigenspace H
// acts as the 2x2 matrix h_s . sigma with
//     h_s(t) = (P_x(t), s P_y(t), eps_perp),   P = p - A(t).
// So the 4-spinor equation for both spins is two 2-level equations.  RK4 is a
// polynomial in dt H, so it commutes with the constant change of basis: RK4 on
// the two 2-level systems produces exactly the RK4 iterates of the 4-spinor
// equation.  The negative-energy subspace at t_0 is spanned by the two
// negative eigenvectors |-, h_s(t_0)>, and the full spin trace of Eq.
// (pair_prod_homo) is
//     f(p) = sum_s |<+, h_s(t_end) | U_s |-, h_s(t_0)>|^2.
//
// The step of each scheme acts on a 2-level state as alpha - i g.sigma with real alpha and g
// (pp_policies.cuh).  In the compensated FP32 path the state is a two-float (hi, lo) pair and the increment is
// added with Fast2Sum, so the O(1) state does not lose the small increments' low bits; the initial state,
// the projection and the momentum sum are FP64 in every path.
#include <map>
#include <mutex>

#include "pp_policies.cuh"

namespace {

// One CTA per block of modes and candidate (grid (blocks, candidates)), and per segment where seg_out is given
// (grid (blocks, candidates, layers)): room for seg_rows segments per block and candidate, seg_done a count for each.  A CTA of a candidate that another launch takes returns at
// once.  ROLE: MAIN or SERIES.
template <class P, int THREADS, int TILE_BYTES, Role ROLE>
__global__ void __launch_bounds__(THREADS, kResidentThreads<RolePolicy<P, ROLE>> / THREADS)
    propagate_kernel(const double *__restrict__ A, int ld, int ns_uniform,
                     const int *__restrict__ ns_array, const typename P::Entry *__restrict__ table,
                     int padded, double dt, pp_grid g, double *__restrict__ n_p,
                     double *__restrict__ partial, long long wait_limit, int skip_copies,
                     unsigned int *__restrict__ status, const int *__restrict__ plans,
                     const double *__restrict__ nodes, void *__restrict__ seg_out, int *__restrict__ seg_done,
                     int seg_rows)
{
    using Q = RolePolicy<P, ROLE>;
    __shared__ ItemSmem<Q, THREADS, TILE_BYTES> sm;
    const int c = blockIdx.y;
    if (!takes_candidate<P, ROLE>(plans, c, 0))
        return;
    const int nmodes = g.nx * g.ny * g.nz;
    const int ngroups = (nmodes + kGroup - 1) / kGroup;
    const int ns = ns_array ? ns_array[c] : ns_uniform;
    const double *Ax = A + (size_t)c * 2 * ld;
    if (threadIdx.x == 0) {
        mbar_init(&sm.bar[0], 1);
        mbar_init(&sm.bar[1], 1);
        mbar_fence_init();
    }
    __syncthreads();
    int tiles = 0;
    const int plan = HasPlan<P>::value ? plans[c] : 0;
    const auto *row = reinterpret_cast<const typename Q::Entry *>(table + (size_t)c * padded);
    double *n_out = n_p ? n_p + (size_t)c * nmodes : nullptr, *part = partial + (size_t)c * ngroups;
    SegmentWork work{-1, nullptr, nullptr};
    if constexpr (Segments<Q>::kCuts) {
        // one CTA per segment (blockIdx.z)
        if (seg_out) {
            const int nent = item_entries<Q>(ns, plan), most = Segments<Q>::most(nmodes, ns);
            const int len = (nent + most - 1) / most;
            const size_t item = (size_t)c * gridDim.x + blockIdx.x;
            using Real = typename std::remove_reference<decltype(Q::State::hi[0][0])>::type;
            work = SegmentWork{(int)blockIdx.z, (Real *)seg_out + item * seg_rows * (Q::kComp ? 16 : 8) * THREADS,
                               seg_done + item};
            if (work.seg * len >= nent)
                return;
        }
    }
    process_item<Q, THREADS, TILE_BYTES, ROLE>(sm, blockIdx.x, g, ns, plan, row, Ax, Ax + ld, dt, n_out, part, wait_limit,
                                               skip_copies, status, tiles, nodes, work);
}

// The candidates that the other launches leave: a grid that fills the GPU at most once walks over all items, so that it costs
// microseconds where there are none (a CTA per item took 0.2 ms for 32768 items).
template <class P, int THREADS, int TILE_BYTES>
__global__ void __launch_bounds__(THREADS)
    propagate_rest_kernel(const double *__restrict__ A, int ld, int ns_uniform,
                          const int *__restrict__ ns_array, const typename P::Entry *__restrict__ table,
                          int padded, double dt, pp_grid g, int ncand, double *__restrict__ n_p,
                          double *__restrict__ partial, long long wait_limit, int skip_copies,
                          unsigned int *__restrict__ status, const int *__restrict__ plans,
                          const double *__restrict__ nodes, int first_rest)
{
    __shared__ ItemSmem<P, THREADS, TILE_BYTES> sm;
    const int nmodes = g.nx * g.ny * g.nz;
    const int ngroups = (nmodes + kGroup - 1) / kGroup;
    const int nblk = (nmodes + THREADS - 1) / THREADS;
    int tiles = 0;
    bool ready = false;
    for (int c = 0; c < ncand; ++c) {
        if (!takes_candidate<P, REST>(plans, c, first_rest))
            continue;
        if (!ready) {
            if (threadIdx.x == 0) {
                mbar_init(&sm.bar[0], 1);
                mbar_init(&sm.bar[1], 1);
                mbar_fence_init();
            }
            __syncthreads();
            ready = true;
        }
        const int ns = ns_array ? ns_array[c] : ns_uniform;
        const double *Ax = A + (size_t)c * 2 * ld;
        // consecutive candidates' blocks go to consecutive CTAs
        const int first = (int)(((long long)blockIdx.x - (long long)c * nblk % gridDim.x + gridDim.x) % gridDim.x);
        for (int blk = first; blk < nblk; blk += gridDim.x)
            if (!process_item<P, THREADS, TILE_BYTES, REST>(
                    sm, blk, g, ns, plans[c], table + (size_t)c * padded, Ax, Ax + ld, dt,
                    n_p ? n_p + (size_t)c * nmodes : nullptr, partial + (size_t)c * ngroups, wait_limit, skip_copies,
                    status, tiles, nodes))
                return;  // barrier phases are unknown after a wait gave up: this CTA stops
    }
}

// N[c] = sum of the per-block partials of candidate c, in a fixed order.
__global__ void finalize_kernel(const double *__restrict__ partial, int nblk, double *__restrict__ N,
                                unsigned int *__restrict__ status)
{
    __shared__ double red[256];
    int c = blockIdx.x;
    double acc = 0.0;
    for (int i = threadIdx.x; i < nblk; i += blockDim.x)
        acc += partial[(size_t)c * nblk + i];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s)
            red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double v = red[0];
        if (!isfinite(v))
            pp_flag(status, PP_FLAG_NONFINITE);
        N[c] = v;
    }
}

// A call's device buffers: the step table, the partial sums, the plans (one int per candidate), for uneven step
// counts room for a copy of n_steps, and the nodes of the grid up to kMaxNodes of them.
constexpr int kMaxNodes = 8192;
struct CallBuffers {
    void *table;
    double *partial;
    int *plans;
    int *ns;
    double *nodes;  // room for the grid's nodes (fill_nodes), or nullptr
    bool segments;  // whether segments of the time axis may have CTAs of their own, with scratch for their propagators
};

// Step counts of a call: the largest, and whether all are equal.
struct StepCounts {
    int max = 0, first = 0;
    bool uniform = true;
    StepCounts(int ncand, int ld, const int32_t *ns_host)
    {
        first = ns_host ? ns_host[0] : (ld - 1) / 2;
        for (int c = 0; c < ncand; ++c) {
            const int ns = ns_host ? ns_host[c] : first;
            max = ns > max ? ns : max;
            uniform &= (ns == first);
        }
    }
};

// The least that a step's angle can be bounded by, whatever the potential (step_size, MagnusPolicy::make_entry6), and the angle of a step
// from which on the main kernel takes none.
double least_angle(const pp_grid &g, double dt)
{
    const double px = fmax(fabs(g.x0), fabs(g.x1)), py = fmax(fabs(g.y0), fabs(g.y1)), pz = fmax(fabs(g.z0), fabs(g.z1));
    return dt * sqrt(px * px + py * py + 1.0 + pz * pz);
}
template <class P>
constexpr double kMainAngle = 1.00001 * (IsBlock<typename MainPolicy<P>::type>::value ? (P::kComp ? kBlockAngleComp : kBlockAngle) / 2
                                                                                        : kSeriesLimit);

// Scratch of the segments' propagators.  Segments get CTAs of their own while a launch has less than kSegmentCtas CTAs without them
// (16 per SM).  The scratch has one size, whatever the call's, so that it never moves while a captured graph holds its address:
// room for the propagators of kSegmentBytes and a count per CTA.  A candidate needs at most 64 bytes for each of kSegTarget
// modes times segments and a partly filled block per segment, 23 MB; calls of more candidates than fit take several launches of
// thousands of CTAs each, so that the size costs nothing.
constexpr int kSegmentCtas = 152 * 16;
constexpr size_t kSegmentBytes = (size_t)64 << 20, kSegmentScratch = kSegmentBytes + kSegmentCtas * sizeof(int);

template <class P, int THREADS, int TILE_BYTES>
int launch(const CallBuffers &buf, const StepCounts &sc, int padded, const double *A, int ncand, int ld,
           const int32_t *ns_host, double dt, const pp_grid *grid, double *N, double *n_p, cudaStream_t stream)
{
    using V = typename P::Entry;
    unsigned int *status = pp::status_word();
    if (!status)
        return pp::fail(PP_ERR_CUDA, "status word unavailable");
    const int nmodes = grid->nx * grid->ny * grid->nz;
    const int nblk = (nmodes + THREADS - 1) / THREADS;
    const int ngroups = (nmodes + kGroup - 1) / kGroup;
    V *table = (V *)buf.table;
    using Q = typename MainPolicy<P>::type;
    int layers = buf.segments && (long long)nblk * ncand < kSegmentCtas ? Segments<Q>::most(nmodes, sc.max) : 1;
    void *seg_out = nullptr;
    int *seg_done = nullptr;
    int seg_rows = 0, ndone = 0, per_launch = ncand;
    if (layers > 1) {
        using Real = typename std::remove_reference<decltype(Q::State::hi[0][0])>::type;
        const size_t per = (size_t)nblk * layers * (Q::kComp ? 16 : 8) * THREADS * sizeof(Real);  // of one candidate
        // without the memory, or with a stream in capture that must not allocate it, each CTA walks all segments, to the
        // same result
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        cudaStreamIsCapturing(stream, &cap);
        if (per <= kSegmentBytes &&
            (cap == cudaStreamCaptureStatusNone || pp::scratch_holds(pp::SCR_SEGMENTS, kSegmentScratch)) &&
            pp::scratch(pp::SCR_SEGMENTS, kSegmentScratch, &seg_out) == PP_OK) {
            seg_rows = layers;
            ndone = nblk * ncand;
            per_launch = (int)(kSegmentBytes / per < (size_t)ncand ? kSegmentBytes / per : (size_t)ncand);
            seg_done = (int *)((char *)seg_out + kSegmentBytes);
        } else {
            cudaGetLastError();
            pp::clear_error();
            seg_out = nullptr;
            layers = 1;
        }
    }
    const int *ns_array = nullptr;
    if (!sc.uniform) {
        cudaError_t e = cudaMemcpyAsync(buf.ns, ns_host, sizeof(int) * ncand, cudaMemcpyHostToDevice, stream);
        if (e != cudaSuccess)
            return pp::cuda_fail(e, "copy of n_steps");
        ns_array = buf.ns;
    }
    if constexpr (IsBlock<typename MainPolicy<P>::type>::value) {
        plan_kernel<P::kComp><<<ncand * kPlanCtas, kPlanThreads, 0, stream>>>(A, ld, sc.first, ns_array, padded, dt, *grid, table,
                                                                  buf.plans, n_p != nullptr, seg_done, ndone, buf.nodes);
    } else {
        if constexpr (HasPlan<P>::value) {
            cudaError_t e = cudaMemsetAsync(buf.plans, 0, sizeof(int) * ncand, stream);
            if (e != cudaSuccess)
                return pp::cuda_fail(e, "plan reset");
        }
        dim3 tg((padded + 255) / 256, ncand);
        build_table_kernel<P><<<tg, 256, 0, stream>>>(A, ld, sc.first, ns_array, padded, dt, *grid, table, buf.plans, seg_done,
                                                     ndone, buf.nodes);
    }
    pp::profile_mark_start(stream);
    // Steps that leave the main kernel's range by the grid's momenta alone leave it nothing to do.
    const bool main_empty = HasPlan<P>::value && least_angle(*grid, dt) > kMainAngle<P>;
    // as many candidates at a time as the segments' scratch holds (one launch without segments)
    for (int c0 = 0; c0 < ncand && !main_empty; c0 += per_launch) {
        const int nc = ncand - c0 < per_launch ? ncand - c0 : per_launch;
        propagate_kernel<P, THREADS, TILE_BYTES, MAIN><<<dim3(nblk, nc, layers), THREADS, 0, stream>>>(
            A + (size_t)c0 * 2 * ld, ld, sc.first, ns_array ? ns_array + c0 : nullptr, table + (size_t)c0 * padded, padded,
            dt, *grid, n_p ? n_p + (size_t)c0 * nmodes : nullptr, buf.partial + (size_t)c0 * ngroups,
            (long long)pp::wait_limit(), pp::skip_copies(), status, buf.plans + c0, buf.nodes, seg_out,
            seg_done ? seg_done + (size_t)c0 * nblk : nullptr, seg_rows);
    }
    if constexpr (HasPlan<P>::value) {
        // single steps are rare (rough potentials) except for the densities of long runs, which get a kernel of their own
        int first_rest = kKindSeries;
        if constexpr (IsBlock<typename MainPolicy<P>::type>::value && !P::kComp) {
            if (n_p && single_steps(sc.max, dt)) {
                // (CTAs of 256 threads: 131 ms where 128-thread CTAs take 140, 4 pulses on 128 x 128 x 64 modes, 20000 steps)
                propagate_kernel<P, 256, 8192, SERIES><<<dim3((nmodes + 255) / 256, ncand), 256, 0, stream>>>(
                    A, ld, sc.first, ns_array, table, padded, dt, *grid, n_p, buf.partial,
                    (long long)pp::wait_limit(), pp::skip_copies(), status, buf.plans, buf.nodes, nullptr, nullptr,
                    0);
                first_rest = kKindWide;
            }
        }
        // Where the kernel finds nothing to do it should cost little, so it fills the GPU once; where it has everything to do, CTAs that
        // come and go overlap one item's FP64 ends with another's steps (16 pulses on 64 x 64 x 32 modes, 400 steps of 0.3: 3.26 ms
        // with the empty main kernel and 8 CTAs per SM, 2.99 with 64 and without it; one launch for each kind of step took 3.05).
        const int most = 152 * ((main_empty ? 8192 : 1024) / THREADS);
        const long long items = (long long)nblk * ncand;
        propagate_rest_kernel<P, THREADS, TILE_BYTES>
            <<<(int)(items < most ? items : most), THREADS, 0, stream>>>(
                A, ld, sc.first, ns_array, table, padded, dt, *grid, ncand, n_p, buf.partial,
                (long long)pp::wait_limit(), pp::skip_copies(), status, buf.plans, buf.nodes, first_rest);
    }
    pp::profile_mark_stop(stream);
    finalize_kernel<<<ncand, 256, 0, stream>>>(buf.partial, ngroups, N, status);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return pp::cuda_fail(e, "pair-number kernel launch");
    return PP_OK;
}

template <class P, int THREADS, int TILE_BYTES>
int run(const double *A, int ncand, int ld, const int32_t *ns_host, double dt, const pp_grid *grid,
        double *N, double *n_p, cudaStream_t stream)
{
    using V = typename P::Entry;
    constexpr int TILE = TILE_BYTES / (int)sizeof(V);
    const StepCounts sc(ncand, ld, ns_host);
    const int padded = ((sc.max + TILE - 1) / TILE) * TILE;
    const int ngroups = (grid->nx * grid->ny * grid->nz + kGroup - 1) / kGroup;
    CallBuffers buf;
    void *partial = nullptr;
    int rc = pp::scratch(pp::SCR_TABLE, (size_t)ncand * padded * sizeof(V), &buf.table);
    if (rc)
        return rc;
    rc = pp::scratch(pp::SCR_PARTIAL, (size_t)ncand * ngroups * sizeof(double) + 1024 * sizeof(int) +
                                          2 * (size_t)ncand * sizeof(int) + kMaxNodes * sizeof(double),
                     &partial);
    if (rc)
        return rc;
    buf.partial = (double *)partial;
    buf.plans = (int *)(((uintptr_t)(buf.partial + (size_t)ncand * ngroups) + 255) & ~(uintptr_t)255);
    buf.ns = (int *)(((uintptr_t)(buf.plans + ncand) + 255) & ~(uintptr_t)255);
    buf.nodes = node_count(*grid) <= kMaxNodes
                    ? (double *)(((uintptr_t)(buf.ns + ncand) + 255) & ~(uintptr_t)255)
                    : nullptr;
    buf.segments = true;
    return launch<P, THREADS, TILE_BYTES>(buf, sc, padded, A, ncand, ld, ns_host, dt, grid, N, n_p, stream);
}

// ---------------------------------------------------------------- no-allocation variant
// Scratch of pp_pair_number_static: a fixed device array in this file, held by
// every GPU that loads the library until the process exits.  It holds, in
// order, the step table, the per-block partial sums, the per-candidate
// plans, (for uneven step
// counts) a copy of n_steps and the grid's nodes; each call writes every byte it later reads, and
// calls that overlap on the GPU race on it.
constexpr size_t kStaticScratchBytes = (size_t)16 << 20;
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Device address of g_static_scratch on the current device, looked up once per
// device (host code must not use the symbol itself as a device address).
unsigned char *static_scratch_address()
{
    constexpr int kMaxDev = 64;
    static unsigned char *addr[kMaxDev] = {};
    static std::mutex mu;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev)
        return nullptr;
    std::lock_guard<std::mutex> lk(mu);
    if (!addr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess)
            return nullptr;
        addr[dev] = (unsigned char *)p;
    }
    return addr[dev];
}

template <class P, int THREADS, int TILE_BYTES>
int run_static(const double *A, int ncand, int ld, const int32_t *ns_host, double dt,
               const pp_grid *grid, double *N, double *n_p, cudaStream_t stream)
{
    using V = typename P::Entry;
    constexpr int TILE = TILE_BYTES / (int)sizeof(V);
    const StepCounts sc(ncand, ld, ns_host);
    const int padded = ((sc.max + TILE - 1) / TILE) * TILE;
    const int ngroups = (grid->nx * grid->ny * grid->nz + kGroup - 1) / kGroup;
    const size_t table_bytes = align256((size_t)ncand * padded * sizeof(V));
    const size_t part_bytes = align256((size_t)ncand * ngroups * sizeof(double));
    const size_t plan_bytes = align256((size_t)ncand * sizeof(int));
    const size_t ns_bytes = sc.uniform ? 0 : align256((size_t)ncand * sizeof(int));
    const size_t need = table_bytes + part_bytes + plan_bytes + ns_bytes;
    if (need > kStaticScratchBytes)
        return pp::fail(PP_ERR_INVALID_ARG,
                        "this call needs %zu bytes of scratch; the static scratch holds %zu "
                        "(use fewer candidates, steps or modes, or pp_pair_number)",
                        need, kStaticScratchBytes);
    unsigned char *base = static_scratch_address();
    if (!base)
        return pp::fail(PP_ERR_CUDA, "cudaGetSymbolAddress of the static scratch failed");
    // the nodes where there is room for them: without, they are computed by each mode, to the same values
    const bool room = node_count(*grid) <= kMaxNodes && need + node_count(*grid) * sizeof(double) <= kStaticScratchBytes;
    const CallBuffers buf{base, (double *)(base + table_bytes), (int *)(base + table_bytes + part_bytes),
                          (int *)(base + table_bytes + part_bytes + plan_bytes), room ? (double *)(base + need) : nullptr,
                          false};
    return launch<P, THREADS, TILE_BYTES>(buf, sc, padded, A, ncand, ld, ns_host, dt, grid, N, n_p, stream);
}

// ---------------------------------------------------------------- launch configurations
// (threads per CTA, bytes per shared-memory tile buffer).  FP32 paths may use
// any of them (chosen by pp_tune_pair_number, else kDefault*); FP64 paths use
// configuration 0.  The arithmetic does not depend on the configuration.
constexpr int kNumConfigs = 6;
constexpr int kCfgThreads[kNumConfigs] = {256, 128, 512, 256, 128, 512};
constexpr int kCfgTileBytes[kNumConfigs] = {8192, 8192, 8192, 32768, 32768, 32768};

using LaunchFn = int (*)(const double *, int, int, const int32_t *, double, const pp_grid *, double *,
                         double *, cudaStream_t);

template <class P, bool ALL>
struct ConfigTable {
    LaunchFn run_fn[kNumConfigs];
    LaunchFn static_fn[kNumConfigs];
    ConfigTable()
    {
        if constexpr (ALL) {
            run_fn[0] = &run<P, 256, 8192>;
            run_fn[1] = &run<P, 128, 8192>;
            run_fn[2] = &run<P, 512, 8192>;
            run_fn[3] = &run<P, 256, 32768>;
            run_fn[4] = &run<P, 128, 32768>;
            run_fn[5] = &run<P, 512, 32768>;
            static_fn[0] = &run_static<P, 256, 8192>;
            static_fn[1] = &run_static<P, 128, 8192>;
            static_fn[2] = &run_static<P, 512, 8192>;
            static_fn[3] = &run_static<P, 256, 32768>;
            static_fn[4] = &run_static<P, 128, 32768>;
            static_fn[5] = &run_static<P, 512, 32768>;
        } else {
            for (int k = 0; k < kNumConfigs; ++k) {
                run_fn[k] = &run<P, 256, 8192>;
                static_fn[k] = &run_static<P, 256, 8192>;
            }
        }
    }
};

// Policy by (precision, scheme).  FP32 RK4 is compensated in either FP32 precision: without, its step multiplies the state by
// alpha = 1 - |u|^2 / 2 + ... rounded to FP32, an error of the norm that all components and modes share and that does not average
// out (14 pulses of 10000 steps: N off by 2.3e-6 rms and -1.6e-6 in the mean, where the four stages applied to the state were at
// 1.2e-6 and -0.3e-6; compensated 1e-7), and a mode's density is no better than 1e-5.  94 instead of 61 instructions a step: 8 pulses on
// 64 x 64 x 32 modes, 4000 steps 11.9 instead of 8.5 ms; the four stages took 19.8.
struct PolicySlot {
    const LaunchFn *run_fn;
    const LaunchFn *static_fn;
    bool tunable;
    int default_cfg;
};

const PolicySlot &policy_slot(int precision, int scheme)
{
    static const ConfigTable<Rk4Policy<double, false>, true> d_rk4;  // tunable: small FP64 grids
    static const ConfigTable<MagnusPolicy<double, false>, false> d_mag;
    static const ConfigTable<SplitPolicy<double, false>, false> d_spl;
    static const ConfigTable<Rk4Policy<float, true>, true> f_rk4;
    static const ConfigTable<MagnusPolicy<float, true>, true> f_mag;
    static const ConfigTable<SplitPolicy<float, true>, true> f_spl;
    static const ConfigTable<MagnusPolicy<float, false>, true> x_mag;
    static const ConfigTable<SplitPolicy<float, false>, true> x_spl;
    // Defaults from timing all configurations (pp_tune_pair_number) on 64 x 64 x 32 modes: CTAs of 128 threads leave less of
    // the last wave idle and overlap one CTA's FP64 projection with another's steps (FP64 RK4 30.2 ms
    // instead of 34.5 ms at 256 threads; on 32 x 32 x 16 modes 8.5 instead of 16.9 ms, 128 CTAs instead of 64 for 152
    // SMs; FP32 Magnus 12.6 instead of 13.0 ms, RK4 12.3 instead of 12.9 ms).
    static const PolicySlot slots[3][3] = {
        {{d_rk4.run_fn, d_rk4.static_fn, true, 1}, {d_mag.run_fn, d_mag.static_fn, false, 0},
         {d_spl.run_fn, d_spl.static_fn, false, 0}},
        {{f_rk4.run_fn, f_rk4.static_fn, true, 1}, {f_mag.run_fn, f_mag.static_fn, true, 1},
         {f_spl.run_fn, f_spl.static_fn, true, 0}},
        {{f_rk4.run_fn, f_rk4.static_fn, true, 1}, {x_mag.run_fn, x_mag.static_fn, true, 1},
         {x_spl.run_fn, x_spl.static_fn, true, 0}},
    };
    return slots[precision][scheme];
}

// Tuned configurations, keyed by the workload shape.
struct TuneKey {
    int precision, scheme, ncand, nmodes, max_ns;
    bool operator<(const TuneKey &o) const
    {
        if (precision != o.precision) return precision < o.precision;
        if (scheme != o.scheme) return scheme < o.scheme;
        if (ncand != o.ncand) return ncand < o.ncand;
        if (nmodes != o.nmodes) return nmodes < o.nmodes;
        return max_ns < o.max_ns;
    }
};
std::mutex g_tune_mu;
std::map<TuneKey, int> g_tuned;

TuneKey make_key(int precision, int scheme, int ncand, int ld, const int32_t *ns, const pp_grid *g)
{
    int max_ns = 0;
    for (int c = 0; c < ncand; ++c) {
        const int v = ns ? ns[c] : (ld - 1) / 2;
        max_ns = v > max_ns ? v : max_ns;
    }
    return TuneKey{precision, scheme, ncand, g->nx * g->ny * g->nz, max_ns};
}

int chosen_config(int precision, int scheme, int ncand, int ld, const int32_t *ns, const pp_grid *g)
{
    const PolicySlot &slot = policy_slot(precision, scheme);
    if (!slot.tunable)
        return 0;
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto it = g_tuned.find(make_key(precision, scheme, ncand, ld, ns, g));
    if (it != g_tuned.end())
        return it->second;
    // FP32 RK4 on few modes is bound by each warp's chain, which a tile's end holds up: tiles of 1024 steps
    // instead of 256 (8 pulses on 600 modes, 800 steps: 80 us instead of 92), where CTAs would not share an SM's memory
    if (precision != PP_FP64 && scheme == PP_RK4 && (long long)ncand * g->nx * g->ny * g->nz <= 152 * 3 * 128)
        return 4;
    return slot.default_cfg;
}

}  // namespace

namespace pp {

int launch_pair_number(const double *A, int ncand, int ld, const int32_t *n_steps_host, double dt,
                       const pp_grid *grid, int precision, int scheme, double *N, double *n_p,
                       cudaStream_t stream)
{
    const int cfg = chosen_config(precision, scheme, ncand, ld, n_steps_host, grid);
    return policy_slot(precision, scheme)
        .run_fn[cfg](A, ncand, ld, n_steps_host, dt, grid, N, n_p, stream);
}

int launch_pair_number_static(const double *A, int ncand, int ld, const int32_t *n_steps_host,
                              double dt, const pp_grid *grid, int precision, int scheme, double *N,
                              double *n_p, cudaStream_t stream)
{
    const int cfg = chosen_config(precision, scheme, ncand, ld, n_steps_host, grid);
    return policy_slot(precision, scheme)
        .static_fn[cfg](A, ncand, ld, n_steps_host, dt, grid, N, n_p, stream);
}

size_t static_scratch_bytes() { return kStaticScratchBytes; }

int num_launch_configs() { return kNumConfigs; }

int tune_pair_number(const double *A, int ncand, int ld, const int32_t *n_steps_host, double dt,
                     const pp_grid *grid, int precision, int scheme, double *N, int32_t *chosen,
                     float *config_ms, cudaStream_t stream)
{
    const PolicySlot &slot = policy_slot(precision, scheme);
    const int ncfg = slot.tunable ? kNumConfigs : 1;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t e = cudaEventCreate(&e0);
    if (e == cudaSuccess)
        e = cudaEventCreate(&e1);
    if (e != cudaSuccess)
        return cuda_fail(e, "tuner event");
    int best = slot.default_cfg;
    float best_ms = 3.0e38f;
    int rc = PP_OK;
    for (int k = 0; k < ncfg && rc == PP_OK; ++k) {
        // one untimed launch (table build, caches), then one timed launch
        rc = slot.run_fn[k](A, ncand, ld, n_steps_host, dt, grid, N, nullptr, stream);
        if (rc)
            break;
        cudaEventRecord(e0, stream);
        rc = slot.run_fn[k](A, ncand, ld, n_steps_host, dt, grid, N, nullptr, stream);
        cudaEventRecord(e1, stream);
        if (rc)
            break;
        float ms = 0.0f;
        e = cudaEventSynchronize(e1);
        if (e == cudaSuccess)
            e = cudaEventElapsedTime(&ms, e0, e1);
        if (e != cudaSuccess) {
            rc = cuda_fail(e, "tuner timing");
            break;
        }
        if (config_ms)
            config_ms[k] = ms;
        if (ms < best_ms) {
            best_ms = ms;
            best = k;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (rc)
        return rc;
    if (slot.tunable) {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        g_tuned[make_key(precision, scheme, ncand, ld, n_steps_host, grid)] = best;
    }
    if (chosen)
        *chosen = best;
    return PP_OK;
}

void clear_tuning()
{
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tuned.clear();
}

void launch_config(int k, int *threads, int *tile_bytes)
{
    *threads = kCfgThreads[k];
    *tile_bytes = kCfgTileBytes[k];
}

}  // namespace pp
