// mxe_grid2d_mixed.cu -- mixed-precision fused stage for the 14-moment
// system on a 2D grid (GB300: FP64 issues at 1/64 of the FP32 rate).
//
// State: the conserved moments U^n stay in FP64 (the conservation
// accumulator).  Every stage runs in FP32 on primitive moments:
//   W   FP32 primitives of U^n        (stencil input of stage 1)
//   Ws  FP32 primitives of U*         (stage-1 output, stencil of stage 2)
// Stage 1:  L = L(W);    W*      = prim(U^n + dt/2 L)
// Stage 2:  L = L(W*);   U^{n+1} = U^n + dt L (FP64 add of the FP32
//           increment);  W^{n+1} = prim(U^{n+1})
// The primitives of U + dU are formed from the FP32 increment dU with
// formulas whose terms all scale with dU (prim_increment14 / _p), so the
// bulk-motion cancellation of a conserved-to-primitive conversion never
// happens in FP32.  W is re-derived from U in FP64 every few steps (inside
// the final stage of that step, or by mxe_resync14_2d when the state is set)
// so that its FP32 rounding does not accumulate.
// Face states whose closure is ill-conditioned (sigma in [sigma_lim,
// sig_lo) near the Junk subspace, sigma > sig_hi near the realizability
// boundary, or det P* < det_min) are re-evaluated in FP64.
//
// Same tiling as the FP64 kernel: 15 x 16 cells per block, 2-cell halo in
// shared memory, one thread per face; instantiated for the general and the
// planar (ten-moment) state.
#include "mxe_internal.h"
#include "mxe_mixed_x2.cuh"

namespace mxe {

constexpr int TXm = 15, TYm = 16, NTm = 256;
constexpr int BXm = TXm + 4, BYm = TYm + 4;
constexpr int NBOXm = BXm * BYm;
constexpr int NPHXm = (TXm + 2) * TYm;
constexpr int NPHYm = TXm * (TYm + 2);



__device__ __forceinline__ const double* map_cell_m(const Grid2D& g, int& gi, int& gj) {
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
    } else if (!xin && !yin) {
        gi = gi < 0 ? 0 : g.nx - 1;
        gj = gj < 0 ? 0 : g.ny - 1;
    }
    return nullptr;
}

template <class PH>
__device__ __forceinline__ void load_prim_f32(const Stage2DArgs& a, int gi, int gj, float* Q) {
    const Grid2D& g = a.g;
    const double* gs = map_cell_m(g, gi, gj);
    if (gs) {
#pragma unroll
        for (int k = 0; k < PH::NF; ++k) Q[k] = (float)gs[PH::ufield(k)];
        return;
    }
    const float* p = a.Win + (long long)gj * g.pitch + gi;
#pragma unroll
    for (int k = 0; k < PH::NF; ++k) Q[k] = __ldg(p + k * g.fstride);
}

template <int NF>
__device__ __forceinline__ float phi_box_m(const float* W, int c, int stride, int lim) {
    float phi = 1.0f;
    const FlatRef<float> fr = flat_ref<NF>(W + c, NBOXm);
#pragma unroll
    for (int k = 0; k < NF; ++k) {
        const float* w = W + k * NBOXm + c;
        float dm = w[0] - w[-stride], dp = w[stride] - w[0];
        float pk;
        if (dm * dp > 0.0f) {
            if (lim == 1) {      // approximate quotient (2 ulp): the limiter is a ratio
                pk = __fdividef(2.0f * dm * dp, dm * dm + dp * dp);
            } else {
                float am = fabsf(dm), ap = fabsf(dp);
                pk = __fdividef(2.0f * fminf(am, ap), am + ap);
            }
        } else {
            pk = (dm == 0.0f && dp == 0.0f) ? 1.0f : 0.0f;
        }
        if (pk < phi) {          // a flat field (phi_k = 1) never lowers phi
            const float m = abs_max(dm, dp);
            if (!(m <= FLAT_REL_F32 * fabsf(w[0]) || field_flat<NF>(fr, k, m))) phi = pk;
        }
    }
    return phi;
}

template <int NF>
__device__ __forceinline__ void face_prims_m(const float* W, int c, int stride, float phi,
                                             float hs, float* Qf) {
    float hp = hs * phi;
#pragma unroll
    for (int k = 0; k < NF; ++k) {
        const float* w = W + k * NBOXm + c;
        float cen = 0.5f * (w[stride] - w[-stride]);
        Qf[k] = w[0] + hp * cen;
    }
}

// Face flux of face `tid` in direction K; the left face state is staged in
// this thread's column of Ls to keep register pressure low.
template <class PH, int K>
__device__ __forceinline__ void face_flux_m(const float* W, int cl, int cr, int stride, float phl,
                                            float phr, const ParamsT<float>& p,
                                            const MixedPolicy& mp, double sl64, double kw64,
                                            float* Ls, float* F, unsigned& nflag) {
    constexpr int NF = PH::NF;
    constexpr int FS = 2 * NF + 2;
    float Qf[NF], R[FS], Lv[FS];
    face_prims_m<NF>(W, cl, stride, phl, 0.5f, Qf);
    nflag += face_state_m<PH, K>(Qf, p, mp, sl64, kw64, Lv) ? 1u : 0u;
#pragma unroll
    for (int n = 0; n < FS; ++n) Ls[n * NTm] = Lv[n];
    face_prims_m<NF>(W, cr, stride, phr, -0.5f, Qf);
    nflag += face_state_m<PH, K>(Qf, p, mp, sl64, kw64, R) ? 1u : 0u;
    float lminL = Ls[(2 * NF) * NTm], lmaxL = Ls[(2 * NF + 1) * NTm];
    float lminR = R[2 * NF], lmaxR = R[2 * NF + 1];
    if (p.flux == 1) {
        float s = fmaxf(fmaxf(fabsf(lminL), fabsf(lmaxL)), fmaxf(fabsf(lminR), fabsf(lmaxR)));
#pragma unroll
        for (int k = 0; k < NF; ++k)
            F[k] = 0.5f * (Ls[(NF + k) * NTm] + R[NF + k]) - 0.5f * s * (R[k] - Ls[k * NTm]);
        return;
    }
    float SL = fminf(lminL, lminR), SR = fmaxf(lmaxL, lmaxR);
    if (SL >= 0.0f) {
#pragma unroll
        for (int k = 0; k < NF; ++k) F[k] = Ls[(NF + k) * NTm];
    } else if (SR <= 0.0f) {
#pragma unroll
        for (int k = 0; k < NF; ++k) F[k] = R[NF + k];
    } else {
        float inv = 1.0f / (SR - SL);
        float cl_ = SR * inv, cr_ = -SL * inv, cu = SL * SR * inv;
#pragma unroll
        for (int k = 0; k < NF; ++k)
            F[k] = cl_ * Ls[(NF + k) * NTm] + cr_ * R[NF + k] + cu * (R[k] - Ls[k * NTm]);
    }
}

__device__ __forceinline__ void block_max_atomic_m(float r, unsigned long long* dst, float* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r = fmaxf(r, __shfl_xor_sync(0xffffffffu, r, o));
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) red[wid] = r;
    __syncthreads();
    if (wid == 0) {
        r = lane < (int)(blockDim.x >> 5) ? red[lane] : 0.0f;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) r = fmaxf(r, __shfl_xor_sync(0xffffffffu, r, o));
        if (lane == 0)
            atomicMax(dst, (unsigned long long)__double_as_longlong((double)r));
    }
}

__device__ __forceinline__ double step_dt_m(const DevClock* clk, int slot, double cfl,
                                            double t_end, double dt_fixed, double& t) {
    t = clk->t[slot];
    if (dt_fixed > 0.0) return dt_fixed;
    double m = __longlong_as_double((long long)clk->rate[slot]);
    double dt = cfl / m;
    if (t + dt > t_end) dt = t_end - t;
    return dt;
}

// Own-cell prefetch of the final stage (U^n FP64 and W^n FP32 into shared
// memory at kernel start): an option of the ten-field planar state at two
// blocks per SM (at three blocks per SM its shared memory does not fit, and
// the same cells are prefetched into L2 instead).
template <int NF, bool PFON>
constexpr int prefetch_cells() { return (PFON && NF == NP) ? TXm * TYm : 0; }

// shared memory: own-cell prefetch, stencil box, x face fluxes, staged
// left face states (whose first NF rows then hold the y face fluxes),
// limiters, reduction scratch
template <int NF, bool PFON>
constexpr size_t smem_mixed() {
    return sizeof(double) * (NF * prefetch_cells<NF, PFON>()) +
           sizeof(float) * (NF * prefetch_cells<NF, PFON>() + NF * NBOXm + NF * NTm +
                            (2 * NF + 2) * NTm + NPHXm + NPHYm + 8);
}

__device__ __forceinline__ void cp_async8(void* sdst, const void* gsrc) {
    unsigned s = (unsigned)__cvta_generic_to_shared(sdst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gsrc));
}
__device__ __forceinline__ void cp_async4(void* sdst, const void* gsrc) {
    unsigned s = (unsigned)__cvta_generic_to_shared(sdst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gsrc));
}


template <class PH, bool PFON>
__device__ __forceinline__ void stage_mixed(const Stage2DArgs& a, const ParamsT<float>& p,
                                            const MixedPolicy& mp) {
    constexpr int NF = PH::NF;
    constexpr int NC = TXm * TYm;
    constexpr int PF = prefetch_cells<NF, PFON>();
    extern __shared__ __align__(16) double smd[];
    double* Upf = smd;                               // [NF][PF] own-cell U^n (final stage)
    float* Wpf = (float*)(Upf + NF * PF);            // [NF][PF] own-cell W^n (final stage)
    float* W = Wpf + NF * PF;                        // [NF][BY][BX]
    float* Fx = W + NF * NBOXm;                      // [NF][256] x-face fluxes
    float* Ls = Fx + NF * NTm;                       // [2NF+2][256] left face states
    // y-face fluxes: column tid of Ls, written by thread tid once its y face
    // is done with the staged left state (no other thread uses that column)
    float* Fy = Ls;
    float* phx = Ls + (2 * NF + 2) * NTm;            // [TY][TX+2]
    float* phy = phx + NPHXm;                        // [TY+2][TX]
    float* red = phy + NPHYm;                        // [8]
    __shared__ double sdt[2];
    __shared__ unsigned cnt;

    const int tid = threadIdx.x;
    if (tid == 0) {
        double tt;
        sdt[0] = step_dt_m(a.clk, a.slot, a.cfl, a.t_end, a.dt_fixed, tt);
        sdt[1] = tt;
        cnt = 0u;
    }
    __syncthreads();
    const double dt = sdt[0], t = sdt[1];
    if (a.final_stage && blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) {
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
    if (!(dt > 0.0)) return;

    const Grid2D& g = a.g;
    const int i0 = blockIdx.x * TXm, j0 = blockIdx.y * TYm;
    const int cx = tid % TXm, cy = tid / TXm;
    const bool owner = tid < NC;
    const int gi = i0 + cx, gj = j0 + cy;
    const bool inside = owner && gi < g.nx && gj < g.ny;
    const long long o = (long long)gj * g.pitch + gi;
    // final stage: start fetching this cell's U^n and W^n now; they are
    // needed only after all face fluxes are done (into shared memory, or
    // into L2 where there is no room)
    if (PF && a.final_stage && inside) {
#pragma unroll
        for (int k = 0; k < NF; ++k) {
            cp_async8(Upf + k * PF + tid, a.Ubase + o + PH::ufield(k) * g.fstride);
            cp_async4(Wpf + k * PF + tid, a.Wbase + o + k * g.fstride);
        }
    } else if (a.final_stage && inside) {
#pragma unroll
        for (int k = 0; k < NF; ++k) {
            asm volatile("prefetch.global.L2 [%0];" ::"l"(a.Ubase + o + PH::ufield(k) * g.fstride));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(a.Wbase + o + k * g.fstride));
        }
    }
    asm volatile("cp.async.commit_group;\n" ::);
    for (int c = tid; c < NBOXm; c += NTm) {
        int bx = c % BXm, by = c / BXm;
        float Q[NF];
        load_prim_f32<PH>(a, i0 + bx - 2, j0 + by - 2, Q);
#pragma unroll
        for (int k = 0; k < NF; ++k) W[k * NBOXm + c] = Q[k];
    }
    __syncthreads();
    for (int n = tid; n < NPHXm + NPHYm; n += NTm) {
        float v = 0.0f;
        if (n < NPHXm) {
            int bx = 1 + n % (TXm + 2), by = 2 + n / (TXm + 2);
            if (p.order == 2) v = phi_box_m<NF>(W, by * BXm + bx, 1, p.limiter);
            phx[n] = v;
        } else {
            int m = n - NPHXm;
            int bx = 2 + m % TXm, by = 1 + m / TXm;
            if (p.order == 2) v = phi_box_m<NF>(W, by * BXm + bx, BXm, p.limiter);
            phy[m] = v;
        }
    }
    __syncthreads();

    const double sl64 = a.sp.sigma_lim, kw64 = a.sp.k_ws;
    unsigned nflag = 0;
    {   // x face tid, then y face tid (no barrier in between)
        int fx = tid & 15, fcy = tid >> 4, by = fcy + 2;
        float F[NF];
        face_flux_m<PH, 0>(W, by * BXm + fx + 1, by * BXm + fx + 2, 1, phx[fcy * (TXm + 2) + fx],
                           phx[fcy * (TXm + 2) + fx + 1], p, mp, sl64, kw64, Ls + tid, F, nflag);
#pragma unroll
        for (int k = 0; k < NF; ++k) Fx[k * NTm + tid] = F[k];
        if (tid < TXm * (TYm + 1)) {
            int fcx = tid % TXm, fy = tid / TXm, bx = fcx + 2;
            face_flux_m<PH, 1>(W, (fy + 1) * BXm + bx, (fy + 2) * BXm + bx, BXm,
                               phy[fy * TXm + fcx], phy[(fy + 1) * TXm + fcx], p, mp, sl64, kw64,
                               Ls + tid, F, nflag);
#pragma unroll
            for (int k = 0; k < NF; ++k) Fy[k * NTm + tid] = F[k];
        }
    }
    // final stage without the shared-memory prefetch: load this cell's U^n
    // and W^n now, so that their latency overlaps the barrier and the
    // source and flux-difference arithmetic below
    double Ureg[PF ? 1 : NF];
    float Wreg[PF ? 1 : NF];
    if (!PF && a.final_stage && inside) {
#pragma unroll
        for (int k = 0; k < NF; ++k) {
            Ureg[k] = a.Ubase[o + PH::ufield(k) * g.fstride];
            Wreg[k] = a.Wbase[o + k * g.fstride];
        }
    }
    asm volatile("cp.async.wait_group 0;\n" ::);
    __syncthreads();

    float r = 0.0f;
    if (owner) {
        float L[NF];
        float Qc[NF];
#pragma unroll
        for (int k = 0; k < NF; ++k) Qc[k] = W[k * NBOXm + (cy + 2) * BXm + cx + 2];
        if (p.tau_model != 0 && !p.src_implicit) {
            PH::source(Qc, PH::tau(p, Qc), L);
        } else {
#pragma unroll
            for (int k = 0; k < NF; ++k) L[k] = 0.0f;
        }
#pragma unroll
        for (int k = 0; k < NF; ++k) {
            L[k] -= (Fx[k * NTm + cy * 16 + cx + 1] - Fx[k * NTm + cy * 16 + cx]) * a.idxf;
            L[k] -= (Fy[k * NTm + (cy + 1) * TXm + cx] - Fy[k * NTm + cy * TXm + cx]) * a.idyf;
        }
        if (inside) {
            float cdt = (float)(a.coef * dt);
            float dU[NF], Wc[NF], Wn[NF];
#pragma unroll
            for (int k = 0; k < NF; ++k) dU[k] = cdt * L[k];
            const bool implicit = p.tau_model != 0 && p.src_implicit;
            if (!a.final_stage) {
                // W* = prim(U^n + dt/2 L): base primitives are this cell's W^n (= stencil)
#pragma unroll
                for (int k = 0; k < NF; ++k) Wc[k] = W[k * NBOXm + (cy + 2) * BXm + cx + 2];
                PH::increment(Wc, dU, Wn);
                if (implicit) {      // point-implicit source over cdt
                    float N[NF];
                    PH::relax_prim(Wn, 1.0f / (1.0f + cdt / PH::tau(p, Wn)), N);
                }
#pragma unroll
                for (int k = 0; k < NF; ++k) a.Wout[o + k * g.fstride] = Wn[k];
            } else {
                bool bad = false;
#pragma unroll
                for (int k = 0; k < NF; ++k) Wc[k] = PF ? Wpf[k * PF + tid] : Wreg[k];
                PH::increment(Wc, dU, Wn);
                if (implicit) {      // relax W, and U by (g - 1)(U - U_M)
                    float N[NF];
                    float gm = 1.0f / (1.0f + cdt / PH::tau(p, Wn));
                    PH::relax_prim(Wn, gm, N);
#pragma unroll
                    for (int k = 0; k < NF; ++k) dU[k] += (gm - 1.0f) * N[k];
                }
#pragma unroll
                for (int k = 0; k < NF; ++k) {
                    double ub = PF ? Upf[k * PF + tid] : Ureg[k];
                    double un = ub + (double)dU[k];
                    a.Uout[o + PH::ufield(k) * g.fstride] = un;
                    bad |= !isfinite(un);
                }
                if (a.resync) {      // the periodic re-sync: W^{n+1} = prim(U^{n+1}) in FP64
                    double Un[NF], Q64[NF];
#pragma unroll
                    for (int k = 0; k < NF; ++k) Un[k] = a.Uout[o + PH::ufield(k) * g.fstride];
                    PH::cons2prim_fast(Un, Q64);
#pragma unroll
                    for (int k = 0; k < NF; ++k) Wn[k] = (float)Q64[k];
                }
#pragma unroll
                for (int k = 0; k < NF; ++k) a.Wout[o + k * g.fstride] = Wn[k];
                if (PH::nonpositive(Wn)) atomicOr(&a.clk->status, ST_NONPOSITIVE);
                if (bad) atomicOr(&a.clk->status, ST_NONFINITE);
                float ax, ay;
                PH::rates(Wn, p.sigma_lim, p.k_ws, ax, ay);
                r = ax * a.idxf + ay * a.idyf;
                if (!(r >= 0.0f)) r = __int_as_float(0x7f800000);     // NaN -> inf
            }
        }
    }
    unsigned wf = __reduce_add_sync(0xffffffffu, nflag);
    if ((tid & 31) == 0 && wf) atomicAdd(&cnt, wf);
    if (a.final_stage) block_max_atomic_m(r, &a.clk->rate[(a.slot + 1) % 3], red);
    __syncthreads();
    if (tid == 0) {
        atomicAdd(&a.clk->n_face, (unsigned long long)(2 * (16 * 16 + TXm * (TYm + 1))));
        if (cnt) atomicAdd(&a.clk->n_face64, (unsigned long long)cnt);
    }
}

extern "C" __global__ void __launch_bounds__(NTm, 2)
mxe_stage14_2d_mixed(const Stage2DArgs a, const ParamsT<float> p, const MixedPolicy mp) {
    stage_mixed<PhysGeneral, false>(a, p, mp);
}
// general state at three blocks per SM (at most 80 registers)
extern "C" __global__ void __launch_bounds__(NTm, 3)
mxe_stage14_2d_mixed_b3(const Stage2DArgs a, const ParamsT<float> p, const MixedPolicy mp) {
    stage_mixed<PhysGeneral, false>(a, p, mp);
}
extern "C" __global__ void __launch_bounds__(NTm, 2)
mxe_stage14_2d_mixed_planar(const Stage2DArgs a, const ParamsT<float> p, const MixedPolicy mp) {
    stage_mixed<PhysPlanar, true>(a, p, mp);
}
// planar state at three blocks per SM (at most 80 registers, L2 prefetch)
extern "C" __global__ void __launch_bounds__(NTm, 3)
mxe_stage14_2d_mixed_planar_b3(const Stage2DArgs a, const ParamsT<float> p,
                               const MixedPolicy mp) {
    stage_mixed<PhysPlanar, false>(a, p, mp);
}

// ---------------------------------------------------------------------------
// Packed stage (the default).  Planar states: a block of 320
// threads owns a TX x TY tile; every thread evaluates up to two x faces and
// two y faces as packed pairs of face states, the limiters of about two
// cells (both directions of an interior cell in one evaluation), and
// updates up to two cells.  The tile is 31 x 18: a row of 32 x faces is one
// warp (no shared-memory bank conflicts in the face phase), the owned cells
// of a warp sit in one or two rows (124-byte segments of each field in
// global memory), and few halo cells are loaded and limited.
//
// What bounds it is instruction issue, so registers go before occupancy: two
// blocks of ten warps an SM leave 96 registers a thread, at which the face
// evaluation hardly spills.  4096 x 4096 RK2 step:
//   31 x 15, 256 threads, 3 blocks, 80 registers  3.91 ms (3.79 with the wave
//                                                 speeds last)
//   31 x 15, 256 threads, 2 blocks, 128           3.50
//   31 x 23, 256 threads, 2 blocks, 128           3.50
//   31 x 11, 192 threads, 3 blocks, 96            3.42
//   31 x 19, 320 threads, 2 blocks, 96            3.36
//   31 x  7, 128 threads, 4 blocks, 128           3.81
//   31 x  9, 160 threads, 4 blocks, 96            3.84
//   31 x 11, 192 threads, 4 blocks, 80            4.21
// (taken before the box was asked for ahead of the step size and the items came in
// rows of a warp; with both, 31 x 18: 3.21 ms, and 228 us at 1024 x 1024, which it fits
// in whole waves; 31 x 17: 3.26 and 233, 31 x 19: 3.29 and 243, TileO: 3.62 and 253).
template <int TX_, int TY_, int NT_>
struct TileGeo {
    static constexpr int TX = TX_, TY = TY_, NT = NT_;
    static constexpr int BX = TX + 4, BY = TY + 4, NBOX = BX * BY;
    static constexpr int NC = TX * TY;             // owned cells
    static constexpr int NFX = (TX + 1) * TY;      // x faces
    static constexpr int NFY = TX * (TY + 1);      // y faces
    static constexpr int NPX = (TX + 2) * TY;      // x limiters
    static constexpr int NPY = TX * (TY + 2);      // y limiters
    // work items of cells and y faces come in rows of RW, of which the last has
    // none: a warp then reads whole rows of the box (or half-rows), without the
    // bank conflicts and the divisions of rows of TX.  The items of TX + 1 x
    // faces fill such rows.
    static constexpr unsigned RW = TX + 1;
    static_assert((RW & (RW - 1)) == 0 && RW <= 32, "a row is a part of a warp");
    // limiter work items: the owned cells (both directions), then the halo
    // columns (x only) and the halo rows (y only)
    static constexpr int NLC = TY * (TX + 1), NLIM = NLC + 2 * TY + 2 * TX;
    static constexpr int NYI = (TY + 1) * (TX + 1);      // items of the y faces
    // y faces start on the warp after the last x face where all fit in one pass
    static constexpr int NFXW = (NFX + 31) / 32 * 32;
    static constexpr int YOFF = NFXW + NYI <= NT ? NFXW : 0;
};
using TileP = TileGeo<31, 18, 320>;
// General states: 14 fields of the box and of the fluxes fill 96 KB, and the
// face evaluation wants 128 registers.
using TileG = TileGeo<31, 15, 256>;
// Smaller tiles for grids of few TileP tiles, which would leave SMs idle; x
// and y faces of the smallest one are evaluated side by side by different
// warps.  mixed_tile() in mxe_capi.cu chooses and has the times.
// TileO, three blocks an SM of 80 registers, is slower on large grids and faster on those
// in between whose TileP tiles begin another wave (450 x 450: 56 against 64 us).
using TileO = TileGeo<31, 15, 256>;
using TileM = TileGeo<31, 7, 256>;
using TileS = TileGeo<15, 7, 256>;

// shared memory of the packed stage: stencil box, x and y face fluxes,
// limiters, reduction scratch
template <class G, int NF>
constexpr size_t smem_mixed_x2() {
    return sizeof(float) * (NF * (G::NBOX + G::NFX + G::NFY) + G::NPX + G::NPY + G::NT / 32);
}

template <class PH, class G, bool RUS>
__device__ __forceinline__ void stage_mixed_x2(const Stage2DArgs& a, const ParamsT<float>& p,
                                               const MixedPolicy& mp) {
    constexpr int NF = PH::NF;
    extern __shared__ __align__(16) double smd[];
    float* W = (float*)smd;                          // [NF][BY][BX]
    float* Fx = W + NF * G::NBOX;                    // [NF][TY][TX+1]
    float* Fy = Fx + NF * G::NFX;                    // [NF][TY+1][TX]
    float* phx = Fy + NF * G::NFY;                   // [TY][TX+2]
    float* phy = phx + G::NPX;                       // [TY+2][TX]
    float* red = phy + G::NPY;                       // [NT / 32]
    __shared__ double sdt[2];
    __shared__ float scdt;
    __shared__ unsigned cnt;

    const int tid = threadIdx.x;
    if (tid == 0) {
        double tt;
        sdt[0] = step_dt_m(a.clk, a.slot, a.cfl, a.t_end, a.dt_fixed, tt);
        sdt[1] = tt;
        scdt = (float)(a.coef * sdt[0]);
        cnt = 0u;
    }
    // the box is on its way before the step size is known
    const Grid2D& g = a.g;
    const int i0 = blockIdx.x * G::TX, j0 = blockIdx.y * G::TY;
    // final stage: the owned cells' U^n and W^n are needed only after the
    // face fluxes; start moving them into L2 now
    if (a.final_stage) {
        for (int c = tid; c < G::NLC; c += G::NT) {
            const int cx = c % G::RW, gi = i0 + cx, gj = j0 + c / G::RW;
            if (cx < G::TX && gi < g.nx && gj < g.ny) {
                const long long o = (long long)gj * g.pitch + gi;
#pragma unroll
                for (int k = 0; k < NF; ++k) {
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(a.Ubase + o + PH::ufield(k) * g.fstride));
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(a.Wbase + o + k * g.fstride));
                }
            }
        }
    }
    const bool interior = i0 >= 2 && j0 >= 2 && i0 + G::TX + 2 <= g.nx && j0 + G::TY + 2 <= g.ny;
    if (interior) {      // the whole box inside the grid: asynchronous copies, no ghost cells
        const float* src = a.Win + (long long)(j0 - 2) * g.pitch + (i0 - 2);
        for (int c = tid; c < G::NBOX; c += G::NT) {
            const float* s0 = src + (long long)(c / G::BX) * g.pitch + c % G::BX;
#pragma unroll
            for (int k = 0; k < NF; ++k) cp_async4(W + k * G::NBOX + c, s0 + k * g.fstride);
        }
        asm volatile("cp.async.commit_group;\n" ::);
    } else {
        for (int c = tid; c < G::NBOX; c += G::NT) {
            const int bx = c % G::BX, by = c / G::BX;
            float Q[NF];
            load_prim_f32<PH>(a, i0 + bx - 2, j0 + by - 2, Q);
#pragma unroll
            for (int k = 0; k < NF; ++k) W[k * G::NBOX + c] = Q[k];
        }
    }
    asm volatile("cp.async.wait_group 0;\n" ::);
    __syncthreads();
    const double dt = sdt[0], t = sdt[1];
    if (a.final_stage && blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) {
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
    if (!(dt > 0.0)) return;
    for (int n = tid; n < G::NLIM; n += G::NT) {
        if (n < G::NLC) {                  // owned cell: both directions
            const int bx = 2 + n % G::RW, by = 2 + n / G::RW;
            if (bx >= 2 + G::TX) continue;
            float2 v = make_float2(0.0f, 0.0f);
            if (p.order == 2) v = phi_pair_m<NF, G::NBOX, G::BX>(W, by * G::BX + bx, p.limiter);
            phx[(by - 2) * (G::TX + 2) + bx - 1] = v.x;
            phy[(by - 1) * G::TX + bx - 2] = v.y;
        } else if (n < G::NLC + 2 * G::TY) {    // halo column: x only
            const int m = n - G::NLC;
            const int bx = (m < G::TY) ? 1 : G::TX + 2, by = 2 + m % G::TY;
            float v = 0.0f;
            if (p.order == 2) v = phi_one_m<NF, G::NBOX>(W, by * G::BX + bx, 1, p.limiter);
            phx[(by - 2) * (G::TX + 2) + bx - 1] = v;
        } else {                                // halo row: y only
            const int m = n - G::NLC - 2 * G::TY;
            const int by = (m < G::TX) ? 1 : G::TY + 2, bx = 2 + m % G::TX;
            float v = 0.0f;
            if (p.order == 2) v = phi_one_m<NF, G::NBOX>(W, by * G::BX + bx, G::BX, p.limiter);
            phy[(by - 1) * G::TX + bx - 2] = v;
        }
    }
    __syncthreads();

    const double sl64 = a.sp.sigma_lim, kw64 = a.sp.k_ws;
    unsigned nflag = 0;
#pragma unroll 1
    for (int f = tid; f < G::NFX; f += G::NT) {       // x faces: TY rows of TX + 1
        const int fx = f % (G::TX + 1), fy = f / (G::TX + 1);
        float F[NF];
        face_flux_x2<PH, 0, G::NBOX, RUS>(W, (fy + 2) * G::BX + fx + 1, 1, phx[fy * (G::TX + 2) + fx],
                                 phx[fy * (G::TX + 2) + fx + 1], p, mp, sl64, kw64, F, nflag);
#pragma unroll
        for (int k = 0; k < NF; ++k) Fx[k * G::NFX + f] = F[k];
    }
#pragma unroll 1
    for (int n = tid - G::YOFF; n < G::NYI; n += G::NT) {       // y faces: TY + 1 rows of TX
        const int fx = n % G::RW, fy = n / G::RW;
        if (n < 0 || fx >= G::TX) continue;
        const int f = fy * G::TX + fx;
        float F[NF];
        face_flux_x2<PH, 1, G::NBOX, RUS>(W, (fy + 1) * G::BX + fx + 2, G::BX, phy[fy * G::TX + fx],
                                 phy[(fy + 1) * G::TX + fx], p, mp, sl64, kw64, F, nflag);
#pragma unroll
        for (int k = 0; k < NF; ++k) Fy[k * G::NFY + f] = F[k];
    }
    __syncthreads();

    float r = 0.0f;
    const float cdt = scdt;
    const bool implicit = p.tau_model != 0 && p.src_implicit;
#pragma unroll 1
    for (int c = tid; c < G::NLC; c += G::NT) {
        const int cx = c % G::RW, cy = c / G::RW;
        const int gi = i0 + cx, gj = j0 + cy;
        if (cx >= G::TX || gi >= g.nx || gj >= g.ny) continue;
        const long long o = (long long)gj * g.pitch + gi;
        const int cb = (cy + 2) * G::BX + cx + 2;
        // final stage: this cell's W^n and U^n, loaded first so that their
        // latency overlaps the source and flux-difference arithmetic
        float Wc[NF];
        double Ub[NF];
        if (a.final_stage) {
#pragma unroll
            for (int k = 0; k < NF; ++k) {
                Wc[k] = a.Wbase[o + k * g.fstride];
                Ub[k] = a.Ubase[o + PH::ufield(k) * g.fstride];
            }
        }
        float L[NF], Qc[NF];
#pragma unroll
        for (int k = 0; k < NF; ++k) Qc[k] = W[k * G::NBOX + cb];
        if (p.tau_model != 0 && !p.src_implicit) {
            PH::source(Qc, PH::tau(p, Qc), L);
        } else {
#pragma unroll
            for (int k = 0; k < NF; ++k) L[k] = 0.0f;
        }
        const int ex = cy * (G::TX + 1) + cx, ey = cy * G::TX + cx;
#pragma unroll
        for (int k = 0; k < NF; ++k) {
            L[k] -= (Fx[k * G::NFX + ex + 1] - Fx[k * G::NFX + ex]) * a.idxf;
            L[k] -= (Fy[k * G::NFY + ey + G::TX] - Fy[k * G::NFY + ey]) * a.idyf;
        }
        float dU[NF], Wn[NF];
#pragma unroll
        for (int k = 0; k < NF; ++k) dU[k] = cdt * L[k];
        if (!a.final_stage) {
            // W* = prim(U^n + dt/2 L): the base primitives are this cell's W^n (= stencil)
            PH::increment(Qc, dU, Wn);
            if (implicit) {      // point-implicit source over cdt
                float N[NF];
                PH::relax_prim(Wn, 1.0f / (1.0f + cdt / PH::tau(p, Wn)), N);
            }
#pragma unroll
            for (int k = 0; k < NF; ++k) a.Wout[o + k * g.fstride] = Wn[k];
        } else {
            PH::increment(Wc, dU, Wn);
            if (implicit) {      // relax W, and U by (g - 1)(U - U_M)
                float N[NF];
                float gm = 1.0f / (1.0f + cdt / PH::tau(p, Wn));
                PH::relax_prim(Wn, gm, N);
#pragma unroll
                for (int k = 0; k < NF; ++k) dU[k] += (gm - 1.0f) * N[k];
            }
            // U^{n+1} = U^n + dU in FP64 (the conservation accumulator);
            // a non-finite increment marks the state non-finite
            bool bad = false;
#pragma unroll
            for (int k = 0; k < NF; ++k) {
                a.Uout[o + PH::ufield(k) * g.fstride] = Ub[k] + f32_to_f64_bits(dU[k]);
                bad |= !(fabsf(dU[k]) < __int_as_float(0x7f800000));
            }
            if (a.resync) {      // the periodic re-sync: W^{n+1} = prim(U^{n+1}) in FP64
                double Un[NF], Q64[NF];
#pragma unroll
                for (int k = 0; k < NF; ++k) Un[k] = a.Uout[o + PH::ufield(k) * g.fstride];
                PH::cons2prim_fast(Un, Q64);
#pragma unroll
                for (int k = 0; k < NF; ++k) Wn[k] = (float)Q64[k];
            }
#pragma unroll
            for (int k = 0; k < NF; ++k) a.Wout[o + k * g.fstride] = Wn[k];
            if (PH::nonpositive(Wn)) atomicOr(&a.clk->status, ST_NONPOSITIVE);
            if (bad) atomicOr(&a.clk->status, ST_NONFINITE);
            float ax, ay;
            if constexpr (NF == NP) x2::rates_x2(Wn, p.sigma_lim, p.k_ws, ax, ay);
            else PH::rates(Wn, p.sigma_lim, p.k_ws, ax, ay);
            float rc = ax * a.idxf + ay * a.idyf;
            if (!(rc >= 0.0f)) rc = __int_as_float(0x7f800000);     // NaN -> inf
            r = fmaxf(r, rc);
        }
    }
    unsigned wf = __reduce_add_sync(0xffffffffu, nflag);
    if ((tid & 31) == 0 && wf) atomicAdd(&cnt, wf);
    if (a.final_stage) block_max_atomic_m(r, &a.clk->rate[(a.slot + 1) % 3], red);
    else __syncthreads();
    if (tid == 0) {
        atomicAdd(&a.clk->n_face, (unsigned long long)(2 * (G::NFX + G::NFY)));
        if (cnt) atomicAdd(&a.clk->n_face64, (unsigned long long)cnt);
    }
}

// packed face-state pairs, BLK blocks per SM
#define MXE_X2(NAME, PH, G, RUS, BLK)                                                        \
    extern "C" __global__ void __launch_bounds__(G::NT, BLK)                              \
    NAME(const Stage2DArgs a, const ParamsT<float> p, const MixedPolicy mp) {             \
        stage_mixed_x2<PH, G, RUS>(a, p, mp);                                                  \
    }
MXE_X2(mxe_stage14_2d_mixed_planar_x2, PhysPlanar, TileP, false, 2)
MXE_X2(mxe_stage14_2d_mixed_planar_x2_rus, PhysPlanar, TileP, true, 2)
MXE_X2(mxe_stage14_2d_mixed_planar_x2_o, PhysPlanar, TileO, false, 3)
MXE_X2(mxe_stage14_2d_mixed_planar_x2_o_rus, PhysPlanar, TileO, true, 3)
MXE_X2(mxe_stage14_2d_mixed_planar_x2_m, PhysPlanar, TileM, false, 2)
MXE_X2(mxe_stage14_2d_mixed_planar_x2_m_rus, PhysPlanar, TileM, true, 2)
MXE_X2(mxe_stage14_2d_mixed_planar_x2_s, PhysPlanar, TileS, false, 2)
MXE_X2(mxe_stage14_2d_mixed_planar_x2_s_rus, PhysPlanar, TileS, true, 2)
MXE_X2(mxe_stage14_2d_mixed_x2, PhysGeneral, TileG, false, 2)
MXE_X2(mxe_stage14_2d_mixed_x2_rus, PhysGeneral, TileG, true, 2)
MXE_X2(mxe_stage14_2d_mixed_x2_m, PhysGeneral, TileM, false, 2)
MXE_X2(mxe_stage14_2d_mixed_x2_m_rus, PhysGeneral, TileM, true, 2)
MXE_X2(mxe_stage14_2d_mixed_x2_s, PhysGeneral, TileS, false, 2)
MXE_X2(mxe_stage14_2d_mixed_x2_s_rus, PhysGeneral, TileS, true, 2)
#undef MXE_X2

template <class PH, class G>
static MixedTile tile_of(void (*kern)(const Stage2DArgs, const ParamsT<float>, const MixedPolicy)) {
    return {(const void*)kern, G::TX, G::TY, G::NT, smem_mixed_x2<G, PH::NF>()};
}
// n = 0: TileP or TileG, 1: TileM, 2: TileS, 3: TileO (planar)
MixedTile mixed_tile_kernel(bool planar, bool rus, int n) {
#define MXE_TILE(NAME, PH, G) tile_of<PH, G>(rus ? NAME##_rus : NAME)
    if (planar)
        return n == 3   ? MXE_TILE(mxe_stage14_2d_mixed_planar_x2_o, PhysPlanar, TileO)
               : n == 2 ? MXE_TILE(mxe_stage14_2d_mixed_planar_x2_s, PhysPlanar, TileS)
               : n == 1 ? MXE_TILE(mxe_stage14_2d_mixed_planar_x2_m, PhysPlanar, TileM)
                        : MXE_TILE(mxe_stage14_2d_mixed_planar_x2, PhysPlanar, TileP);
    return n == 2   ? MXE_TILE(mxe_stage14_2d_mixed_x2_s, PhysGeneral, TileS)
           : n == 1 ? MXE_TILE(mxe_stage14_2d_mixed_x2_m, PhysGeneral, TileM)
                    : MXE_TILE(mxe_stage14_2d_mixed_x2, PhysGeneral, TileG);
#undef MXE_TILE
}

size_t stage14_2d_mixed_smem(bool planar, int blocks_per_sm) {
    if (!planar) return smem_mixed<14, false>();      // both general variants
    return blocks_per_sm >= 3 ? smem_mixed<NP, false>() : smem_mixed<NP, true>();
}

// W = FP32 primitives of U, converted in FP64 (set-up and periodic re-sync).
template <class PH>
__device__ __forceinline__ void resync(const double* U, float* W, const Grid2D& g) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int j = blockIdx.y;
    if (i >= g.nx) return;
    long long o = (long long)j * g.pitch + i;
    double Uc[PH::NF], Q[PH::NF];
#pragma unroll
    for (int k = 0; k < PH::NF; ++k) Uc[k] = U[o + PH::ufield(k) * g.fstride];
    PH::cons2prim_fast(Uc, Q);
#pragma unroll
    for (int k = 0; k < PH::NF; ++k) W[o + k * g.fstride] = f64::to_f32(Q[k]);
}
extern "C" __global__ void mxe_resync14_2d(const double* U, float* W, Grid2D g) {
    resync<PhysGeneral>(U, W, g);
}
extern "C" __global__ void mxe_resync14_2d_planar(const double* U, float* W, Grid2D g) {
    resync<PhysPlanar>(U, W, g);
}

// Initial CFL rate from the FP32 primitives.
template <class PH>
__device__ __forceinline__ void rate_mixed(const float* W, const Grid2D& g, const ParamsT<float>& p,
                                           float idxf, float idyf, DevClock* clk, int slot) {
    __shared__ float red[8];
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int j = blockIdx.y;
    float r = 0.0f;
    if (i < g.nx) {
        long long o = (long long)j * g.pitch + i;
        float Q[PH::NF];
#pragma unroll
        for (int k = 0; k < PH::NF; ++k) Q[k] = W[o + k * g.fstride];
        float ax, ay;
        PH::rates(Q, p.sigma_lim, p.k_ws, ax, ay);
        r = ax * idxf + ay * idyf;
        if (!(r >= 0.0f)) r = __int_as_float(0x7f800000);
    }
    block_max_atomic_m(r, &clk->rate[slot], red);
}
extern "C" __global__ void mxe_rate14_2d_mixed(const float* W, Grid2D g, ParamsT<float> p,
                                               float idxf, float idyf, DevClock* clk, int slot) {
    rate_mixed<PhysGeneral>(W, g, p, idxf, idyf, clk, slot);
}
extern "C" __global__ void mxe_rate14_2d_mixed_planar(const float* W, Grid2D g, ParamsT<float> p,
                                                      float idxf, float idyf, DevClock* clk,
                                                      int slot) {
    rate_mixed<PhysPlanar>(W, g, p, idxf, idyf, clk, slot);
}

}  // namespace mxe
