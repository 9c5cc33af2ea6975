// mxe_grid2d.cu -- fused finite-volume stage for the 14-moment system on a
// 2D Cartesian grid (Sec. 3 of Boccelli et al., JCP 2024), FP64 path.
//
// One thread block owns a tile of TX x TY = 15 x 16 cells.  It stages the
// primitive moments of the tile plus a 2-cell halo in shared memory (BCs are
// applied while loading: transmissive, periodic, Dirichlet slots), computes
// one shared limiter per cell and direction, evaluates every x- and y-face
// once (two face states, closure, flux, wave speeds, HLL/Rusanov) with one
// thread per face, differences the face fluxes, adds the BGK source and
// writes the RK stage.  The final stage of a step also reduces the CFL rate
// of the new state (warp shuffle, block, one atomicMax per block) so that
// the next step's dt is formed on the device.
//
// Tile shape: 16 x 16 x-faces and 15 x 17 y-faces map onto 256 threads with
// at most one idle thread.  The kernel is instantiated for the general
// 14-moment state and for planar states (ten active moments).  Grids of few
// such tiles take one of two smaller tiles with one thread per face state
// (stage_f64_lanes below).
#include "mxe_internal.h"
#include "mxe_policy.cuh"

namespace mxe {

constexpr int TX = 15, TY = 16, NT2 = 256;
constexpr int BX = TX + 4, BY = TY + 4;          // 19 x 20 staged box
constexpr int NBOX = BX * BY;
constexpr int NPHX = (TX + 2) * TY;              // 272 x-limiters (box cols 1..17)
constexpr int NPHY = TX * (TY + 2);              // 270 y-limiters (box rows 1..18)

// time step of this step (identical in every thread of every block)
__device__ __forceinline__ double step_dt(const DevClock* clk, int slot, double cfl,
                                          double t_end, double dt_fixed, double& t) {
    t = clk->t[slot];
    if (dt_fixed > 0.0) return dt_fixed;
    double m = __longlong_as_double((long long)clk->rate[slot]);
    double dt = cfl / m;
    if (t + dt > t_end) dt = t_end - t;
    return dt;
}

// Boundary logic: returns the ghost state of a Dirichlet ghost cell
// (nullptr otherwise) and maps (gi, gj) into the grid (periodic wrap,
// transmissive clamp).
__device__ __forceinline__ const double* map_cell(const Grid2D& g, int& gi, int& gj) {
    bool xin = (gi >= 0 && gi < g.nx), yin = (gj >= 0 && gj < g.ny);
    if (!xin && yin) {
        int s = gi < 0 ? 0 : 1;
        const SideDesc& sd = g.side[s];
        if (sd.type == 1) {
            gi = ((gi % g.nx) + g.nx) % g.nx;
            return nullptr;
        }
        for (int n = 0; n < sd.nspans; ++n)
            if (gj >= sd.lo[n] && gj <= sd.hi[n]) return g.ghost + (s * GHOST_SLOTS + 1 + n) * 14;
        if (sd.type == 2) return g.ghost + (s * GHOST_SLOTS) * 14;
        gi = gi < 0 ? 0 : g.nx - 1;
    } else if (xin && !yin) {
        int s = gj < 0 ? 2 : 3;
        const SideDesc& sd = g.side[s];
        if (sd.type == 1) {
            gj = ((gj % g.ny) + g.ny) % g.ny;
            return nullptr;
        }
        for (int n = 0; n < sd.nspans; ++n)
            if (gi >= sd.lo[n] && gi <= sd.hi[n]) return g.ghost + (s * GHOST_SLOTS + 1 + n) * 14;
        if (sd.type == 2) return g.ghost + (s * GHOST_SLOTS) * 14;
        gj = gj < 0 ? 0 : g.ny - 1;
    } else if (!xin && !yin) {          // corner: never used by the stencil
        gi = gi < 0 ? 0 : g.nx - 1;
        gj = gj < 0 ? 0 : g.ny - 1;
    }
    return nullptr;
}

template <class PH>
__device__ __forceinline__ void load_prim_f64(const Stage2DArgs& a, int gi, int gj, double* Q) {
    const Grid2D& g = a.g;
    const double* gs = map_cell(g, gi, gj);
    if (gs) {
#pragma unroll
        for (int k = 0; k < PH::NF; ++k) Q[k] = gs[PH::ufield(k)];
        return;
    }
    const double* p = a.Uin + (long long)gj * g.pitch + gi;
    double U[PH::NF];
#pragma unroll
    for (int k = 0; k < PH::NF; ++k) U[k] = __ldg(p + PH::ufield(k) * g.fstride);
    PH::cons2prim_rn(U, Q);
}

// Numerical face flux of the face between box cells c and c + stride.
template <class PH, int K>
__device__ __forceinline__ void face_flux_f64(const double* W, int c, int stride, double phl,
                                              double phr, const ParamsT<double>& p, double* F) {
    constexpr int NF = PH::NF;
    double Q[NF], UL[NF], FL[NF], UR[NF], FR[NF], l0, l1, r0, r1;
    const double hl = 0.25 * phl, hr = -0.25 * phr;
#pragma unroll
    for (int k = 0; k < NF; ++k) {
        const double* w = W + k * NBOX + c;
        Q[k] = f64::face_value(w[-stride], w[0], w[stride], hl);
    }
    PH::template face<double, K>(Q, p.sigma_lim, p.k_ws, UL, FL, l0, l1);
#pragma unroll
    for (int k = 0; k < NF; ++k) {
        const double* w = W + k * NBOX + c + stride;
        Q[k] = f64::face_value(w[-stride], w[0], w[stride], hr);
    }
    PH::template face<double, K>(Q, p.sigma_lim, p.k_ws, UR, FR, r0, r1);
    f64::riemann<NF>(UL, FL, l0, l1, UR, FR, r0, r1, p.flux, F);
}

template <int NT = NT2>
__device__ __forceinline__ void block_max_atomic(double r, unsigned long long* dst, double* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        r = f64::max_(r, __shfl_xor_sync(0xffffffffu, r, o));
    }
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) red[wid] = r;
    __syncthreads();
    if (wid == 0) {
        r = lane < (NT / 32) ? red[lane] : 0.0;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            r = f64::max_(r, __shfl_xor_sync(0xffffffffu, r, o));
        }
        if (lane == 0) atomicMax(dst, (unsigned long long)__double_as_longlong(r));
    }
}

// Clock bookkeeping of the final stage (block (0,0), thread 0).
__device__ __forceinline__ void advance_clock(const Stage2DArgs& a, double dt, double t) {
    int s1 = (a.slot + 1) % 3, s2 = (a.slot + 2) % 3;
    a.clk->rate[s2] = 0ull;
    if (!(dt > 0.0)) {
        a.clk->t[s1] = t;
        a.clk->rate[s1] = a.clk->rate[a.slot];
    } else {
        a.clk->t[s1] = t + dt;
        a.clk->last_dt = dt;
        if (a.dt_hist && a.clk->steps < a.dt_hist_cap) a.dt_hist[a.clk->steps] = dt;
        a.clk->steps += 1;
    }
}

// The owned cell (gi, gj) from its residual L: the stage's state, written out,
// and in the final stage its status bits and CFL rate (returned).
template <class PH>
__device__ __forceinline__ double update_cell(const Stage2DArgs& a, const ParamsT<double>& p,
                                              double dt, int gi, int gj, const double* L) {
    constexpr int NF = PH::NF;
    const Grid2D& g = a.g;
    const long long o = (long long)gj * g.pitch + gi;
    double Un[NF];
    bool bad = false;
    const double cdt = mul_rn(a.coef, dt);
#pragma unroll
    for (int k = 0; k < NF; ++k)
        Un[k] = add_rn(a.Ubase[o + PH::ufield(k) * g.fstride], mul_rn(cdt, L[k]));
    if (p.tau_model != 0 && p.src_implicit) {   // point-implicit source over cdt
        double Qv[NF];
        PH::cons2prim_rn(Un, Qv);
        PH::relax_cons(Un, Qv, PH::tau(p, Qv), cdt);
    }
#pragma unroll
    for (int k = 0; k < NF; ++k) {
        a.Uout[o + PH::ufield(k) * g.fstride] = Un[k];
        bad |= !f64::is_finite(Un[k]);
    }
    if (!a.final_stage) return 0.0;
    double Qn[NF];
    PH::cons2prim_rn(Un, Qn);
    if (PH::nonpositive64(Qn)) atomicOr(&a.clk->status, ST_NONPOSITIVE);
    if (bad) atomicOr(&a.clk->status, ST_NONFINITE);
    if (a.skip_rate) return 0.0;
    double ax, ay;
    PH::rates(Qn, p.sigma_lim, p.k_ws, ax, ay);
    double r = ax * g.idx;
    r = r + ay * g.idy;
    if (!f64::ge0(r)) r = __longlong_as_double(0x7ff0000000000000ll);  // NaN -> inf
    return r;
}

// The explicit source of a cell (zero otherwise)
template <class PH>
__device__ __forceinline__ void cell_source(const ParamsT<double>& p, double tau_factor,
                                            const double* Qc, double* L) {
    if (p.tau_model != 0 && !p.src_implicit) {
        const double pr = PH::pressure64(Qc);
        PH::source64(Qc, pr, f64::inv_tau(p.tau_model, tau_factor, Qc[0], pr), L);
    } else {
#pragma unroll
        for (int k = 0; k < PH::NF; ++k) L[k] = 0.0;
    }
}

template <int NF>
constexpr size_t smem_f64() {
    return sizeof(double) * (NF * NBOX + NF * NT2 + NPHX + NPHY + 8);
}

// ---------------------------------------------------------------------------
// FP64 stage kernel.  Stage 1 of RK2: Uout = Ubase + dt/2 L(Uin);
// final stage (RK2 stage 2 or FE): Uout = Ubase + dt L(Uin), plus the CFL
// rate of Uout, clock advance and status.
// ---------------------------------------------------------------------------
template <class PH>
__device__ __forceinline__ void stage_f64(const Stage2DArgs& a) {
    constexpr int NF = PH::NF;
    extern __shared__ __align__(16) double smem[];
    double* W = smem;                                // [NF][BY][BX]
    double* Fb = W + NF * NBOX;                      // [NF][256]
    double* phx = Fb + NF * NT2;                     // [TY][TX+2]
    double* phy = phx + NPHX;                        // [TY+2][TX]
    double* red = phy + NPHY;                        // [8]
    __shared__ double sdt[3];

    const int tid = threadIdx.x;
    if (tid == 0) {
        double tt;
        sdt[0] = step_dt(a.clk, a.slot, a.cfl, a.t_end, a.dt_fixed, tt);
        sdt[1] = tt;
    }
    if (tid == 32) sdt[2] = f64::tau_factor(a.rp.model, a.rp.tau_ref, a.rp.rho_ref, a.rp.T_ref);
    __syncthreads();
    const double dt = sdt[0], t = sdt[1];
    if (a.final_stage && blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) advance_clock(a, dt, t);
    if (!(dt > 0.0)) return;

    const ParamsT<double> p = make_params<double>(a.sp, a.rp);
    const Grid2D& g = a.g;
    const int i0 = blockIdx.x * TX, j0 = blockIdx.y * TY;
    for (int c = tid; c < NBOX; c += NT2) {
        int bx = c % BX, by = c / BX;
        double Q[NF];
        load_prim_f64<PH>(a, i0 + bx - 2, j0 + by - 2, Q);
#pragma unroll
        for (int k = 0; k < NF; ++k) W[k * NBOX + c] = Q[k];
    }
    __syncthreads();
    for (int n = tid; n < NPHX; n += NT2) {
        int bx = 1 + n % (TX + 2), by = 2 + n / (TX + 2);
        phx[n] = p.order == 2 ? f64::limiter<NF>(W, by * BX + bx, 1, NBOX, p.limiter) : 0.0;
    }
    for (int n = tid; n < NPHY; n += NT2) {
        int bx = 2 + n % TX, by = 1 + n / TX;
        phy[n] = p.order == 2 ? f64::limiter<NF>(W, by * BX + bx, BX, NBOX, p.limiter) : 0.0;
    }
    __syncthreads();
    {   // x faces: face fx in [0,16) of row cy, between box cells fx+1 | fx+2
        int fx = tid & 15, cy = tid >> 4, by = cy + 2;
        double F[NF];
        face_flux_f64<PH, 0>(W, by * BX + fx + 1, 1, phx[cy * (TX + 2) + fx],
                             phx[cy * (TX + 2) + fx + 1], p, F);
#pragma unroll
        for (int k = 0; k < NF; ++k) Fb[k * NT2 + tid] = F[k];
    }
    __syncthreads();
    const int cx = tid % TX, cy = tid / TX;          // owned cell (tid < 240)
    const bool owner = tid < TX * TY;
    double L[NF];
    if (owner) {
        double Qc[NF];
#pragma unroll
        for (int k = 0; k < NF; ++k) Qc[k] = W[k * NBOX + (cy + 2) * BX + cx + 2];
        cell_source<PH>(p, sdt[2], Qc, L);
#pragma unroll
        for (int k = 0; k < NF; ++k)
            L[k] -= (Fb[k * NT2 + cy * 16 + cx + 1] - Fb[k * NT2 + cy * 16 + cx]) * g.idx;
    }
    __syncthreads();
    if (tid < TX * (TY + 1)) {   // y faces: face fy in [0,17) of column cx
        int fcx = tid % TX, fy = tid / TX, bx = fcx + 2;
        double F[NF];
        face_flux_f64<PH, 1>(W, (fy + 1) * BX + bx, BX, phy[fy * TX + fcx],
                             phy[(fy + 1) * TX + fcx], p, F);
#pragma unroll
        for (int k = 0; k < NF; ++k) Fb[k * NT2 + tid] = F[k];
    }
    __syncthreads();

    double r = 0.0;
    if (owner) {
#pragma unroll
        for (int k = 0; k < NF; ++k)
            L[k] -= (Fb[k * NT2 + (cy + 1) * TX + cx] - Fb[k * NT2 + cy * TX + cx]) * g.idy;
        const int gi = i0 + cx, gj = j0 + cy;
        if (gi < g.nx && gj < g.ny) r = update_cell<PH>(a, p, dt, gi, gj, L);
    }
    if (a.final_stage) block_max_atomic(r, &a.clk->rate[(a.slot + 1) % 3], red);
}

extern "C" __global__ void __launch_bounds__(NT2, 1) mxe_stage14_2d_f64(const Stage2DArgs a) {
    stage_f64<PhysGeneral>(a);
}
extern "C" __global__ void __launch_bounds__(NT2, 1)
mxe_stage14_2d_f64_planar(const Stage2DArgs a) {
    stage_f64<PhysPlanar>(a);
}

// ---------------------------------------------------------------------------
// The same stage on a smaller tile, one thread per face STATE (the two states
// of a face in adjacent lanes, which exchange them by shuffle and form half
// of the face's fluxes each), x and y faces side by side on different warps.
//
// FP64 is bound per SM (2 operations a clock), and below one warp on each of
// the four sub-partitions by the chain of a single warp, whatever its active
// lanes: the 15 x 16 tile has 8 warps walk through 4 face states each, and a
// grid of a few such tiles leaves the other SMs idle meanwhile.  The 5 x 5
// tile (30 + 30 faces: two warps of x and two of y states) is the least work
// an SM can do in one pass; the 7 x 8 tile (64 + 63 faces, 8 warps) computes 5 % fewer
// faces per cell.  f64_tile() in mxe_capi.cu chooses and has the times.
// ---------------------------------------------------------------------------
template <int TX_, int TY_, int NT_>
struct LaneGeo {
    static constexpr int TX = TX_, TY = TY_, NT = NT_;
    static constexpr int BX = TX + 4, NBOX = BX * (TY + 4);
    static constexpr int NPX = (TX + 2) * TY, NPY = TX * (TY + 2);
    static constexpr int NFX = (TX + 1) * TY, NFY = TX * (TY + 1);
    static constexpr int NSX = (2 * NFX + 31) / 32 * 32;          // x states, whole warps
    static_assert(NSX + 2 * NFY <= NT && TX * TY <= NT && NT % 32 == 0, "one pass of the threads");
};
template <class PH, class G>
struct LaneShared {
    double W[PH::NF * G::NBOX];                 // primitives of the tile and its halo
    double F[PH::NF * (G::NFX + G::NFY)];       // face fluxes
    double ph[G::NPX + G::NPY];                 // limiters
    double red[8], sdt[3];
};

// The pair of lanes evaluates the face between box cells c and c + stride;
// phl points to the left cell's limiter, the right one's is dph further on.
template <class PH, class G, int K>
__device__ __forceinline__ void lane_face(LaneShared<PH, G>& sh, int c, const double* phl, int dph,
                                          const ParamsT<double>& p, int face, bool valid) {
    constexpr int NF = PH::NF, H = (NF + 1) / 2, S = K == 0 ? 1 : G::BX;
    const bool right = threadIdx.x & 1;
    const int b = right ? c + S : c;
    const double h = right ? -0.25 * phl[dph] : 0.25 * phl[0];
    double Q[NF], U[NF], F[NF], Fo[H], lo, hi;
#pragma unroll
    for (int k = 0; k < NF; ++k) {
        const double* w = sh.W + k * G::NBOX + b;
        Q[k] = f64::face_value(w[-S], w[0], w[S], h);
    }
    PH::template face<double, K>(Q, p.sigma_lim, p.k_ws, U, F, lo, hi);
    f64::pair_flux<NF>(U, F, lo, hi, right, p.flux, Fo);
    if (!valid) return;
#pragma unroll
    for (int k = 0; k < H; ++k)
        if (!right) sh.F[k * (G::NFX + G::NFY) + face] = Fo[k];
        else if (H + k < NF) sh.F[(H + k) * (G::NFX + G::NFY) + face] = Fo[k];
}

template <class PH, class G>
__device__ __forceinline__ void stage_f64_lanes(const Stage2DArgs& a) {
    constexpr int NF = PH::NF, NFACE = G::NFX + G::NFY;
    __shared__ LaneShared<PH, G> sh;
    const int tid = threadIdx.x;
    if (tid == 0) {
        double tt;
        sh.sdt[0] = step_dt(a.clk, a.slot, a.cfl, a.t_end, a.dt_fixed, tt);
        sh.sdt[1] = tt;
    }
    if (tid == 32)
        sh.sdt[2] = f64::tau_factor(a.rp.model, a.rp.tau_ref, a.rp.rho_ref, a.rp.T_ref);
    const ParamsT<double> p = make_params<double>(a.sp, a.rp);
    const Grid2D& g = a.g;
    const int i0 = blockIdx.x * G::TX, j0 = blockIdx.y * G::TY;
    for (int c = tid; c < G::NBOX; c += G::NT) {
        double Q[NF];
        load_prim_f64<PH>(a, i0 + c % G::BX - 2, j0 + c / G::BX - 2, Q);
#pragma unroll
        for (int k = 0; k < NF; ++k) sh.W[k * G::NBOX + c] = Q[k];
    }
    __syncthreads();
    const double dt = sh.sdt[0], t = sh.sdt[1];
    if (a.final_stage && blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) advance_clock(a, dt, t);
    if (!(dt > 0.0)) return;
    for (int n = tid; n < G::NPX + G::NPY; n += G::NT) {
        const bool x = n < G::NPX;                   // x limiters, then y limiters
        const int m = x ? n : n - G::NPX, wd = x ? G::TX + 2 : G::TX;
        const int c = (m / wd + (x ? 2 : 1)) * G::BX + m % wd + (x ? 1 : 2);
        sh.ph[n] = p.order == 2
            ? f64::limiter<NF>(sh.W, c, x ? 1 : G::BX, G::NBOX, p.limiter) : 0.0;
    }
    __syncthreads();
    if (tid < G::NSX) {                              // x faces: TY rows of TX + 1
        const int f = min(tid >> 1, G::NFX - 1), fx = f % (G::TX + 1), fy = f / (G::TX + 1);
        lane_face<PH, G, 0>(sh, (fy + 2) * G::BX + fx + 1, sh.ph + fy * (G::TX + 2) + fx, 1, p, f,
                            tid < 2 * G::NFX);
    } else if (tid < G::NSX + (2 * G::NFY + 31) / 32 * 32) {     // y faces: TY + 1 rows of TX
        const int f = min((tid - G::NSX) >> 1, G::NFY - 1), fx = f % G::TX, fy = f / G::TX;
        lane_face<PH, G, 1>(sh, (fy + 1) * G::BX + fx + 2, sh.ph + G::NPX + f, G::TX, p,
                            G::NFX + f, tid - G::NSX < 2 * G::NFY);
    }
    __syncthreads();
    double r = 0.0;
    if (tid < G::TX * G::TY) {
        const int cx = tid % G::TX, cy = tid / G::TX, gi = i0 + cx, gj = j0 + cy;
        double Qc[NF], L[NF];
#pragma unroll
        for (int k = 0; k < NF; ++k) Qc[k] = sh.W[k * G::NBOX + (cy + 2) * G::BX + cx + 2];
        cell_source<PH>(p, sh.sdt[2], Qc, L);
        const double* fx = sh.F + cy * (G::TX + 1) + cx;
        const double* fy = sh.F + G::NFX + cy * G::TX + cx;
#pragma unroll
        for (int k = 0; k < NF; ++k) {
            L[k] -= (fx[k * NFACE + 1] - fx[k * NFACE]) * g.idx;
            L[k] -= (fy[k * NFACE + G::TX] - fy[k * NFACE]) * g.idy;
        }
        if (gi < g.nx && gj < g.ny) r = update_cell<PH>(a, p, dt, gi, gj, L);
    }
    if (a.final_stage) block_max_atomic<G::NT>(r, &a.clk->rate[(a.slot + 1) % 3], sh.red);
}

using Lane5 = LaneGeo<5, 5, 128>;
using Lane7 = LaneGeo<7, 8, 256>;
#define MXE_LANES(NAME, PH, G)                                                           \
    extern "C" __global__ void __launch_bounds__(G::NT) NAME(const Stage2DArgs a) {      \
        stage_f64_lanes<PH, G>(a);                                                       \
    }
MXE_LANES(mxe_stage14_2d_f64_t5, PhysGeneral, Lane5)
MXE_LANES(mxe_stage14_2d_f64_planar_t5, PhysPlanar, Lane5)
MXE_LANES(mxe_stage14_2d_f64_t7, PhysGeneral, Lane7)
MXE_LANES(mxe_stage14_2d_f64_planar_t7, PhysPlanar, Lane7)
#undef MXE_LANES

F64Tile f64_tile_kernel(bool planar, int tx) {
    if (tx == Lane5::TX)
        return {planar ? mxe_stage14_2d_f64_planar_t5 : mxe_stage14_2d_f64_t5, Lane5::TX,
                Lane5::TY, Lane5::NT, 0};
    if (tx == Lane7::TX)
        return {planar ? mxe_stage14_2d_f64_planar_t7 : mxe_stage14_2d_f64_t7, Lane7::TX,
                Lane7::TY, Lane7::NT, 0};
    return {planar ? mxe_stage14_2d_f64_planar : mxe_stage14_2d_f64, TX, TY, NT2,
            planar ? smem_f64<NP>() : smem_f64<14>()};
}

// Initial CFL rate of the current state into slot `slot` of the clock.
template <class PH>
__device__ __forceinline__ void rate_f64(const double* U, const Grid2D& g, const SchemeParams& sp,
                                         DevClock* clk, int slot) {
    __shared__ double red[8];
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int j = blockIdx.y;
    double r = 0.0;
    if (i < g.nx) {
        long long o = (long long)j * g.pitch + i;
        double Un[PH::NF], Qn[PH::NF];
#pragma unroll
        for (int k = 0; k < PH::NF; ++k) Un[k] = U[o + PH::ufield(k) * g.fstride];
        PH::cons2prim_rn(Un, Qn);
        double ax, ay;
        PH::rates(Qn, sp.sigma_lim, sp.k_ws, ax, ay);
        r = ax * g.idx;
        r = r + ay * g.idy;
        if (!(r >= 0.0)) r = __longlong_as_double(0x7ff0000000000000ll);
    }
    block_max_atomic(r, &clk->rate[slot], red);
}
extern "C" __global__ void mxe_rate14_2d(const double* U, Grid2D g, SchemeParams sp,
                                         DevClock* clk, int slot) {
    rate_f64<PhysGeneral>(U, g, sp, clk, slot);
}
extern "C" __global__ void mxe_rate14_2d_planar(const double* U, Grid2D g, SchemeParams sp,
                                                DevClock* clk, int slot) {
    rate_f64<PhysPlanar>(U, g, sp, clk, slot);
}

int tile_x() { return TX; }
int tile_y() { return TY; }

}  // namespace mxe
