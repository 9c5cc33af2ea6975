// mxe_tubes.cu -- persistent solver for 1D problems (the 5-moment system of
// Sec. 2.3 and the 14-moment system of Sec. 2.4 in one space dimension),
// single or batched, FP64 path.
//
// A team of CTAs owns one tube for the whole launch and marches it on the
// tube's own clock (dt from the team's CFL reduction), so tubes of different
// lengths and Knudsen numbers never wait for one another.  Within a stage the
// team's CTAs take the tube's chunks of C cells in turn: stage the primitives
// of the chunk plus a 2-cell halo in shared memory, one shared limiter per
// cell, one thread per face STATE (the two states of a face in adjacent lanes,
// which exchange them by shuffle and form half of the face's fluxes each), then
// flux differences, BGK source and the RK update.
//
// Why teams: FP64 is bound per SM (2 operations a clock) and, below four
// warps, per sub-partition (64 clocks a warp instruction whatever its active
// lanes), so a tube on one CTA runs on 1/152 of the chip.  A stage's chain of
// FP64 instructions costs the same for 31 cells on an SM (62 of 64 lanes of two
// warps on two sub-partitions) as for one, so a tube is spread until a CTA has
// 31 cells (C = 31) and only then gets C = 63 (four warps, 76 clocks an
// instruction) and several chunks a CTA.  The teams' barrier costs 1.0-1.1 us
// (measured, 8 to 152 CTAs) against 10-20 us for a stage.
// The step times are beside team_plan() in mxe_capi.cu.
//
// The CTAs of a team wait for one another, so a launch with a team of more
// than one CTA is cooperative (all CTAs resident); the wait is bounded, and
// a team that gives up sets ST_TIMEOUT and returns.
#include "mxe_internal.h"
#include "mxe_policy.cuh"
#include "mxe_team.cuh"

namespace mxe {

constexpr int NTT = 128;

// primitive state of tube cell gi (boundary ghosts included); other CTAs of
// the team wrote it in the previous stage: read from L2
template <class PH>
__device__ __forceinline__ void load_prim_1d(const TubeArgs& a, const double* U,
                                             const TubeDesc& td, int gi, double* Q) {
    if (gi < 0 || gi >= td.n) {
        int s = gi < 0 ? 0 : 1;
        int ty = a.bc_type[s];
        if (ty == 2) {
#pragma unroll
            for (int k = 0; k < PH::NF; ++k) Q[k] = a.ghost[s * 14 + PH::ufield(k)];
            return;
        }
        if (ty == 1) gi = ((gi % td.n) + td.n) % td.n;
        else gi = gi < 0 ? 0 : td.n - 1;
    }
    double Uc[PH::NF];
#pragma unroll
    for (int k = 0; k < PH::NF; ++k) Uc[k] = __ldcg(U + (long long)PH::ufield(k) * td.n + gi);
    PH::cons2prim_rn(Uc, Q);
}

template <class PH, int C>
struct TubeShared {
    double W[PH::NF * (C + 4)];          // primitives of the chunk and its halo
    double F[PH::NF * (C + 1)];          // face fluxes
    double ph[C + 2];                    // limiters
    double red[NTT / 32];
    unsigned st;
};

// One stage over the chunks of this CTA: out = base + coef dt L(in).
// Returns the thread's max CFL rate of `out` if `final`.
template <class PH, int C>
__device__ __forceinline__ double tube_stage(const TubeArgs& a, const ParamsT<double>& p,
                                             const TubeDesc& td, double itau, unsigned rank,
                                             unsigned nb, const double* in, const double* base,
                                             double* out, double coef, double dt, bool final,
                                             TubeShared<PH, C>& sh, unsigned& status) {
    constexpr int NF = PH::NF, BOX = C + 4, H = (NF + 1) / 2;
    const int tid = threadIdx.x, n = td.n;
    const double idx = 1.0 / td.dx;
    double rmax = 0.0;
    for (int c0 = (int)rank * C; c0 < n; c0 += (int)nb * C) {
        const int m = min(C, n - c0);                      // cells of this chunk
        for (int i = tid; i < m + 4; i += NTT) {
            double Q[NF];
            load_prim_1d<PH>(a, in, td, c0 - 2 + i, Q);
#pragma unroll
            for (int k = 0; k < NF; ++k) sh.W[k * BOX + i] = Q[k];
        }
        __syncthreads();
        for (int i = tid; i < m + 2; i += NTT)             // box cells 1 .. m+2
            sh.ph[i] = p.order == 2 ? f64::limiter<NF>(sh.W, i + 1, 1, BOX, p.limiter) : 0.0;
        __syncthreads();
        if (tid < ((2 * (m + 1) + 31) & ~31)) {            // whole warps: the lanes exchange
            const int f = min(tid >> 1, m);                // face between box cells f+1 | f+2
            const bool right = tid & 1;
            const int c = f + 1 + (right ? 1 : 0);
            const double h = (right ? -0.25 : 0.25) * sh.ph[c - 1];
            double Q[NF], U[NF], F[NF], Fo[H], lo, hi;
#pragma unroll
            for (int k = 0; k < NF; ++k) {
                const double* w = sh.W + k * BOX + c;
                Q[k] = f64::face_value(w[-1], w[0], w[1], h);
            }
            PH::template face<double, 0>(Q, p.sigma_lim, p.k_ws, U, F, lo, hi);
            f64::pair_flux<NF>(U, F, lo, hi, right, p.flux, Fo);
            if ((tid >> 1) <= m) {
#pragma unroll
                for (int k = 0; k < H; ++k)
                    if (!right) sh.F[k * (C + 1) + f] = Fo[k];
                    else if (H + k < NF) sh.F[(H + k) * (C + 1) + f] = Fo[k];
            }
        }
        __syncthreads();
        if (tid < m) {
            const int i = c0 + tid;
            double Qc[NF], L[NF], Un[NF];
#pragma unroll
            for (int k = 0; k < NF; ++k) Qc[k] = sh.W[k * BOX + tid + 2];
            const bool implicit = td.rp.model != 0 && td.rp.implicit;
            if (td.rp.model != 0 && !implicit) {
                const double pr = PH::pressure64(Qc);
                PH::source64(Qc, pr, f64::inv_tau(td.rp.model, itau, Qc[0], pr), L);
            } else {
#pragma unroll
                for (int k = 0; k < NF; ++k) L[k] = 0.0;
            }
            const double cdt = mul_rn(coef, dt);
            bool bad = false;
#pragma unroll
            for (int k = 0; k < NF; ++k) {
                L[k] -= (sh.F[k * (C + 1) + tid + 1] - sh.F[k * (C + 1) + tid]) * idx;
                Un[k] = add_rn(__ldcg(base + (long long)PH::ufield(k) * n + i), mul_rn(cdt, L[k]));
            }
            double Qn[NF];
            if (implicit) {                                // point-implicit source over cdt
                PH::cons2prim_rn(Un, Qn);
                PH::relax_cons(Un, Qn, PH::tau(p, Qn), cdt);
            }
#pragma unroll
            for (int k = 0; k < NF; ++k) {
                out[(long long)PH::ufield(k) * n + i] = Un[k];
                bad |= !f64::is_finite(Un[k]);
            }
            if (final) {
                PH::cons2prim_rn(Un, Qn);
                if (bad) status |= ST_NONFINITE;
                if (PH::nonpositive_x(Qn)) status |= ST_NONPOSITIVE;
                double r = PH::template rate_x<double>(Qn, p.sigma_lim, p.k_ws) * idx;
                if (!f64::ge0(r)) r = __longlong_as_double(0x7ff0000000000000ll);
                rmax = f64::max_(rmax, r);
            }
        }
        __syncthreads();
    }
    return rmax;
}

// Team-wide max of the CFL rate and OR of the status bits, in one of three
// slots (slot = epoch mod 3).  After the barrier of epoch e the first CTA
// clears slot (e+2) mod 3: every CTA read it (epoch e-1) before arriving at
// barrier e, and none writes it (epoch e+2) before barrier e+1, which the
// first CTA reaches only after the clear.
__device__ __forceinline__ bool team_reduce(TubeSync* s, int spin, unsigned rank, unsigned nb,
                                            unsigned& target, unsigned& epoch, double r,
                                            unsigned st, double* red, unsigned* sst, double& m,
                                            unsigned& st_out) {
    const int tid = threadIdx.x;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r = f64::max_(r, __shfl_xor_sync(0xffffffffu, r, o));
    st = __reduce_or_sync(0xffffffffu, st);
    if (tid == 0) *sst = 0u;
    __syncthreads();
    if ((tid & 31) == 0) {
        red[tid >> 5] = r;
        if (st) atomicOr(sst, st);
    }
    __syncthreads();
    const unsigned slot = epoch++ % 3u;
    if (nb == 1u) {
        m = red[0];
#pragma unroll
        for (int w = 1; w < NTT / 32; ++w) m = f64::max_(m, red[w]);
        st_out = *sst;
        return true;
    }
    if (tid == 0) {
        double v = red[0];
#pragma unroll
        for (int w = 1; w < NTT / 32; ++w) v = f64::max_(v, red[w]);
        atomicMax(&s->rate[slot], (unsigned long long)__double_as_longlong(v));
        if (*sst) atomicOr(&s->stat[slot], *sst);
    }
    if (!team_barrier(s, nb, target, spin)) return false;
    m = __longlong_as_double((long long)__ldcg(&s->rate[slot]));
    st_out = __ldcg(&s->stat[slot]);
    if (rank == 0 && tid == 0) {
        const unsigned old = (slot + 2u) % 3u;
        __stcg(&s->rate[old], 0ull);
        __stcg(&s->stat[old], 0u);
    }
    return true;
}

template <class PH, int C>
__device__ __forceinline__ void tubes_body(const TubeArgs& a) {
    __shared__ TubeShared<PH, C> sh;
    constexpr int NF = PH::NF;
    const TubeTeam tm = a.teams ? a.teams[blockIdx.x]
                                : TubeTeam{0, (int)blockIdx.x, (int)gridDim.x, 0};
    const unsigned rank = (unsigned)tm.rank, nb = (unsigned)tm.size;
    const TubeDesc td = a.tubes[tm.tube];
    TubeClock* ck = a.clk + tm.tube;
    TubeSync* sy = a.sync + tm.tube;
    const ParamsT<double> p = make_params<double>(a.sp, td.rp);
    const double itau = f64::tau_factor(td.rp.model, td.rp.tau_ref, td.rp.rho_ref, td.rp.T_ref);
    double* cur = a.U + td.off;
    double* nxt = a.Us + td.off;
    const int tid = threadIdx.x, n = td.n;
    unsigned target = 0, epoch = 0, status = 0, st = 0;
    bool ok = true;

    // CFL rate of the current state
    double r = 0.0, m = 0.0;
    for (int c0 = (int)rank * C; c0 < n; c0 += (int)nb * C)
        if (tid < min(C, n - c0)) {
            double Uc[NF], Q[NF];
#pragma unroll
            for (int k = 0; k < NF; ++k)
                Uc[k] = __ldcg(cur + (long long)PH::ufield(k) * n + c0 + tid);
            PH::cons2prim_rn(Uc, Q);
            double ri = PH::template rate_x<double>(Q, p.sigma_lim, p.k_ws) * (1.0 / td.dx);
            if (!f64::ge0(ri)) ri = __longlong_as_double(0x7ff0000000000000ll);
            r = f64::max_(r, ri);
        }
    ok = team_reduce(sy, a.spin, rank, nb, target, epoch, r, 0u, sh.red, &sh.st, m, st);
    double t = ck->t;
    long long steps = ck->steps;
    double last_dt = ck->last_dt;
    st = 0u;
    for (int s = 0; ok && s < a.max_steps; ++s) {
        double dt;
        if (a.dt_fixed) {
            if (s >= a.n_fixed) break;
            dt = a.dt_fixed[s];
        } else {
            if (!(t < a.t_end)) break;
            dt = a.cfl / m;
            if (t + dt > a.t_end) dt = a.t_end - t;
        }
        if (!(dt > 0.0)) break;
        double rr;
        status = 0u;
        if (a.integrator == 1) {
            tube_stage<PH, C>(a, p, td, itau, rank, nb, cur, cur, nxt, 0.5, dt, false, sh, status);
            if (!(ok = team_barrier(sy, nb, target, a.spin))) break;
            rr = tube_stage<PH, C>(a, p, td, itau, rank, nb, nxt, cur, cur, 1.0, dt, true, sh,
                                   status);
        } else {
            rr = tube_stage<PH, C>(a, p, td, itau, rank, nb, cur, cur, nxt, 1.0, dt, true, sh,
                                   status);
            double* tmp = cur;
            cur = nxt;
            nxt = tmp;
        }
        if (!(ok = team_reduce(sy, a.spin, rank, nb, target, epoch, rr, status, sh.red, &sh.st, m,
                               st)))
            break;
        t += dt;
        last_dt = dt;
        ++steps;
        if (st) break;                       // team-uniform
    }
    // forward Euler after an odd number of steps: the state sits in the stage
    // buffer; every CTA brings its own cells back
    if (ok && cur != a.U + td.off)
        for (int c0 = (int)rank * C; c0 < n; c0 += (int)nb * C)
            if (tid < min(C, n - c0)) {
#pragma unroll
                for (int k = 0; k < NF; ++k) {
                    const long long o = (long long)PH::ufield(k) * n + c0 + tid;
                    nxt[o] = cur[o];
                }
            }
    if (tid == 0 && !ok) atomicOr(&ck->status, ST_TIMEOUT);
    if (tid == 0 && rank == 0 && ok) {
        ck->t = t;
        ck->steps = steps;
        ck->last_dt = last_dt;
        ck->rate = m;
        if (st) atomicOr(&ck->status, st);
    }
}

#define MXE_TUBES(NAME, PH, C)                                                       \
    extern "C" __global__ void __launch_bounds__(NTT) NAME(const TubeArgs a) {       \
        tubes_body<PH, C>(a);                                                        \
    }
// 14 moments with the state's planarity found on the device (a caller's array)
#define MXE_TUBES14(NAME, C)                                                         \
    extern "C" __global__ void __launch_bounds__(NTT) NAME(const TubeArgs a) {       \
        if (a.nonplanar && __ldcg(a.nonplanar) == 0u) tubes_body<PhysPlanar, C>(a);  \
        else tubes_body<PhysGeneral, C>(a);                                          \
    }
MXE_TUBES(mxe_tubes5_f64, Phys5, 63)
MXE_TUBES14(mxe_tubes14_f64, 63)
MXE_TUBES(mxe_tubes14_f64_planar, PhysPlanar, 63)
MXE_TUBES(mxe_tubes5_f64_c31, Phys5, 31)
MXE_TUBES14(mxe_tubes14_f64_c31, 31)
MXE_TUBES(mxe_tubes14_f64_planar_c31, PhysPlanar, 31)
#undef MXE_TUBES14
#undef MXE_TUBES

// A launch whose teams wait inside is cooperative: all of its CTAs are resident.
cudaError_t launch_tubes_f64(const void* kern, int ctas, bool coop, const TubeArgs& a,
                             cudaStream_t st) {
    void* args[] = {(void*)&a};
    if (coop) return cudaLaunchCooperativeKernel(kern, dim3(ctas), dim3(NTT), args, 0, st);
    return cudaLaunchKernel(kern, dim3(ctas), dim3(NTT), args, 0, st);
}

int tubes_threads() { return NTT; }
// chunk: 31 or 63 cells a CTA pass
const void* tubes_f64_kernel(int system, bool planar, int chunk) {
    if (chunk == 31)
        return system == 5 ? (const void*)mxe_tubes5_f64_c31
                           : planar ? (const void*)mxe_tubes14_f64_planar_c31
                                    : (const void*)mxe_tubes14_f64_c31;
    return system == 5 ? (const void*)mxe_tubes5_f64
                       : planar ? (const void*)mxe_tubes14_f64_planar
                                : (const void*)mxe_tubes14_f64;
}

}  // namespace mxe
