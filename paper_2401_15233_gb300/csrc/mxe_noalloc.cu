// mxe_noalloc.cu -- a 1D solve that allocates no device memory.
//
// Some callers cannot allocate device memory: a host program whose device
// memory is wholly owned by its own pool allocator (an outside cudaMalloc
// either fails under the pool's cap or breaks its accounting), or a
// time-critical loop that cannot pay for cudaMalloc/cudaFree, which
// synchronise the device.  mxe_tube_run_noalloc serves them: the caller
// passes the state, and every other buffer the persistent tube kernel needs
// (the RK stage buffer, the tube descriptor, the clock and the ghost states)
// lives in file-scope __device__ arrays of fixed size below.  Every GPU that
// loads the library holds these arrays until the process exits.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <mutex>

#include "../../include/maxent.h"
#include "mxe_internal.h"

namespace mxe {
const void* tubes_f64_kernel(int system, bool planar, int chunk);
cudaError_t launch_tubes_f64(const void* kern, int ctas, bool coop, const TubeArgs& a,
                             cudaStream_t st);
int tubes_threads();

constexpr int NOALLOC_MAX_CELLS = 16384;    // 14 x 16384 doubles = 1.75 MiB of stage buffer

static __device__ __align__(256) double g_stage[14 * NOALLOC_MAX_CELLS];
static __device__ __align__(256) TubeDesc g_tube[1];
static __device__ __align__(256) TubeClock g_clock[1];
static __device__ __align__(256) double g_ghost[2 * 14];
static __device__ __align__(256) TubeSync g_sync[1];
static __device__ __align__(256) unsigned g_nonplanar[1];

struct NoallocPtrs {
    bool ready = false;
    double* stage = nullptr;
    TubeDesc* tube = nullptr;
    TubeClock* clock = nullptr;
    double* ghost = nullptr;
    TubeSync* sync = nullptr;
    unsigned* nonplanar = nullptr;
    int slots = 0;                  // CTAs that are resident at once
};
constexpr int MAX_DEVICES = 64;
static NoallocPtrs g_ptrs[MAX_DEVICES];
static std::mutex g_mutex;

// Device addresses of the file-scope arrays for the current device.  In host
// code the array names are host-side stand-ins, not device addresses, so
// they are looked up once per device, with that device current.
static cudaError_t noalloc_ptrs(NoallocPtrs& out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_mutex);
    NoallocPtrs& p = g_ptrs[dev];
    if (!p.ready) {
        if ((e = cudaGetSymbolAddress((void**)&p.stage, g_stage)) != cudaSuccess) return e;
        if ((e = cudaGetSymbolAddress((void**)&p.tube, g_tube)) != cudaSuccess) return e;
        if ((e = cudaGetSymbolAddress((void**)&p.clock, g_clock)) != cudaSuccess) return e;
        if ((e = cudaGetSymbolAddress((void**)&p.ghost, g_ghost)) != cudaSuccess) return e;
        if ((e = cudaGetSymbolAddress((void**)&p.sync, g_sync)) != cudaSuccess) return e;
        if ((e = cudaGetSymbolAddress((void**)&p.nonplanar, g_nonplanar)) != cudaSuccess)
            return e;
        int nsm = 0, per = 2;
        if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) !=
            cudaSuccess)
            return e;
        for (int system : {5, 14})
            for (int chunk : {31, 63}) {
                int v = 0;
                if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                         &v, tubes_f64_kernel(system, false, chunk), tubes_threads(), 0)) !=
                    cudaSuccess)
                    return e;
                per = v < per ? v : per;
            }
        p.slots = per * nsm;
        p.ready = true;
    }
    out = p;
    return cudaSuccess;
}

// Writes the tube descriptor, a fresh clock and zeroed barrier slots into the
// fixed arrays, and finds out whether the 14-moment state in U is planar (its
// z-odd moments 3, 6, 8, 12 zero): the march then carries the other ten, as a
// context's does.  Everything arrives by value as kernel arguments, so no host
// buffer has to outlive the call (a cudaMemcpyAsync from a stack variable would).
__global__ void __launch_bounds__(1024)
mxe_noalloc_init(const TubeDesc td, const TubeClock ck, const double* U, int system) {
    bool np = system != 14;
    for (int i = threadIdx.x; i < td.n && !np; i += blockDim.x)
        np = U[3LL * td.n + i] != 0.0 || U[6LL * td.n + i] != 0.0 || U[8LL * td.n + i] != 0.0 ||
             U[12LL * td.n + i] != 0.0;
    np = __syncthreads_or(np);
    if (threadIdx.x == 0) {
        g_tube[0] = td;
        g_clock[0] = ck;
        g_sync[0] = TubeSync{};
        g_nonplanar[0] = np ? 1u : 0u;
    }
}

}  // namespace mxe

using namespace mxe;

extern "C" mxe_status mxe_tube_run_noalloc(const mxe_config* cfg, int bc_lo, int bc_hi,
                                           int tau_model, double tau_ref, double rho_ref,
                                           double T_ref, double* U, double t0, double t_end,
                                           int max_steps, double* t_out, int* steps_out,
                                           void* stream) {
    if (!cfg || !U) return MXE_EINVAL;
    if (cfg->system != 5 && cfg->system != 14) return MXE_EINVAL;
    if (cfg->ny != 1 || cfg->nx < 4 || !(cfg->x1 > cfg->x0)) return MXE_EINVAL;
    if (cfg->nx > NOALLOC_MAX_CELLS) return MXE_EINVAL;          // beyond the fixed scratch
    if (cfg->precision != MXE_FP64) return MXE_EINVAL;
    if (cfg->order != 1 && cfg->order != 2) return MXE_EINVAL;
    if (cfg->integrator != MXE_FE && cfg->integrator != MXE_RK2) return MXE_EINVAL;
    if (cfg->flux != MXE_FLUX_HLL && cfg->flux != MXE_FLUX_RUSANOV) return MXE_EINVAL;
    if (cfg->limiter != MXE_LIM_MINMOD && cfg->limiter != MXE_LIM_VANALBADA) return MXE_EINVAL;
    if (!(cfg->cfl > 0.0) || !(cfg->sigma_lim > 0.0 && cfg->sigma_lim < 1.0) ||
        !(cfg->k_ws >= 1.0))
        return MXE_EINVAL;
    if ((bc_lo != MXE_BC_TRANSMISSIVE && bc_lo != MXE_BC_PERIODIC) ||
        (bc_hi != MXE_BC_TRANSMISSIVE && bc_hi != MXE_BC_PERIODIC) ||
        ((bc_lo == MXE_BC_PERIODIC) != (bc_hi == MXE_BC_PERIODIC)))
        return MXE_EINVAL;
    if (tau_model < 0 || tau_model > 2 || (tau_model != 0 && !(tau_ref > 0.0))) return MXE_EINVAL;
    if (max_steps < 0) return MXE_EINVAL;

    NoallocPtrs p;
    if (noalloc_ptrs(p) != cudaSuccess) return MXE_ECUDA;
    cudaStream_t st = (cudaStream_t)stream;

    TubeDesc td{};
    td.off = 0;
    td.n = cfg->nx;
    td.dx = (cfg->x1 - cfg->x0) / cfg->nx;
    td.rp = RelaxParams{tau_model, tau_ref, rho_ref, T_ref};
    TubeClock ck{};               // the clock must start from t0 with no steps and no status
    ck.t = t0;
    mxe_noalloc_init<<<1, 1024, 0, st>>>(td, ck, U, cfg->system);
    if (cudaGetLastError() != cudaSuccess) return MXE_ECUDA;

    TubeArgs a{};
    a.U = U;
    a.Us = p.stage;
    a.tubes = p.tube;
    a.clk = p.clock;
    a.bc_type[0] = bc_lo;
    a.bc_type[1] = bc_hi;
    a.ghost = p.ghost;            // read only for Dirichlet sides, which are not offered here
    a.ntubes = 1;
    a.system = cfg->system;
    a.integrator = cfg->integrator;
    a.sp.sigma_lim = cfg->sigma_lim;
    a.sp.k_ws = cfg->k_ws;
    a.sp.flux = cfg->flux;
    a.sp.limiter = cfg->limiter;
    a.sp.order = cfg->order;
    a.cfl = cfg->cfl;
    a.t_end = t_end;
    a.max_steps = max_steps;
    a.teams = nullptr;            // every CTA of the launch works on the one tube
    a.sync = p.sync;
    a.spin = TEAM_SPIN_LIMIT;
    a.nonplanar = p.nonplanar;
    // one CTA per 31 cells while they are all resident, else chunks of 63 in
    // equal passes (the rule of a context's team plan)
    int chunk = 31, ctas = (cfg->nx + 30) / 31;
    if (ctas > p.slots) {
        chunk = 63;
        const int ch = (cfg->nx + 62) / 63, pass = (ch + p.slots - 1) / p.slots;
        ctas = (ch + pass - 1) / pass;
    }
    cudaError_t e =
        launch_tubes_f64(tubes_f64_kernel(cfg->system, false, chunk), ctas, ctas > 1, a, st);
    if (e == cudaErrorCooperativeLaunchTooLarge) {       // a stream of fewer SMs: one CTA alone
        cudaGetLastError();
        e = launch_tubes_f64(tubes_f64_kernel(cfg->system, false, 63), 1, false, a, st);
    }
    if (e != cudaSuccess) return MXE_ECUDA;
    if (t_out || steps_out) {
        if (cudaMemcpyAsync(&ck, p.clock, sizeof ck, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            return MXE_ECUDA;
        if (t_out) *t_out = ck.t;
        if (steps_out) *steps_out = (int)ck.steps;
        if (ck.status & ST_TIMEOUT) return MXE_ETIMEOUT;
        if (ck.status & ST_NONFINITE) return MXE_ENONFINITE;
    }
    return MXE_OK;
}
