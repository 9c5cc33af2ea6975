// mxe_util.cu -- set-up and read-back kernels: primitive <-> conserved
// conversion, state validation, ghost-state round trip, diagnostics.
// Nothing here is on the time-stepping path.
#include "mxe_fast64.cuh"
#include "mxe_internal.h"
#include "mxe_planar.cuh"

namespace mxe {

// Returns false if the thread has no cell.  dense: offset of field 0 in the
// API's dense array; dev: offset in the device array; fs/dfs: field strides.
__device__ __forceinline__ bool cell_of(const CellMap& m, long long& dense, long long& dfs,
                                        long long& dev, long long& fs, long long& idx) {
    if (m.mode == 0) {
        int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
        if (i >= m.nx || j >= m.ny) return false;
        idx = (long long)j * m.nx + i;
        dense = idx;
        dfs = (long long)m.nx * m.ny;
        dev = (long long)j * m.pitch + i;
        fs = m.fstride;
        return true;
    }
    int b = blockIdx.y;
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= m.ntubes || i >= m.tubes[b].n) return false;
    dense = dev = m.tubes[b].off + i;
    dfs = fs = m.tubes[b].n;
    idx = m.tubes[b].off / m.nf + i;     // cell number in the concatenation
    return true;
}

__device__ __forceinline__ double raw_sigma(const double* Q, int nf) {
    if (nf == 5) {
        double th = Q[2] / Q[0];
        double qs = Q[3] / (Q[0] * th * sqrt(th));
        double rs = Q[4] / (Q[0] * th * th);
        return sigma5(qs, rs);
    }
    Dimless14<double> d;
    dimless14(Q, d);
    return d.sig;
}

// A state that is realizable by a clear margin, decided without the FP64 pipe
// (2 operations a clock and SM here, against 128 in FP32): every |Q| 0 or
// in [1e-30, 1e30], and in FP32 sigma <= 0.99 and, of P* = 3 P / tr P, the
// diagonal > 0, the leading minor > 1e-4 and det >= 1e-3 (a positive definite P* of
// that determinant has a leading minor of at least det / 3).  A positive diagonal
// of trace 3 bounds each of its elements by 3, the minor then P*_xy, and the last
// condition P*_xz and P*_yz: the FP32 errors of the minor (2e-6) and of det (3e-5)
// are far below their margins.  Without those bounds both could be cancellation
// noise of large elements, of any sign.
__device__ __forceinline__ bool clearly_realizable(const double* Q, int nf) {
    bool screen = true;
    float Qf[14];
    for (int k = 0; k < nf; ++k) {
        const unsigned e = (f64::hi32(Q[k]) >> 20) & 0x7ffu;
        const bool zero = ((f64::hi32(Q[k]) & 0x7fffffffu) | f64::lo32(Q[k])) == 0u;
        screen &= zero || (e >= 924u && e <= 1122u);         // 2^-99 .. 2^99
        Qf[k] = f64::narrow(Q[k]);
    }
    if (!screen) return false;
    if (nf == 5) {
        const float th = Qf[2] / Qf[0];
        return sigma5(Qf[3] / (Qf[0] * th * sqrtf(th)), Qf[4] / (Qf[0] * th * th)) <= 0.99f;
    }
    Dimless14<float> d;
    dimless14(Qf, d);
    const float* P = d.Ps;                                    // every test false for NaN
    return d.th > 0.0f && P[0] > 0.0f && P[3] > 0.0f && P[5] > 0.0f && fabsf(P[2]) <= 3.0f &&
           fabsf(P[4]) <= 3.0f && P[0] * P[3] - P[1] * P[1] > 1e-4f && d.det >= 1e-3f &&
           d.sig <= 0.99f;
}

// 0 ok; 1 non-finite; 2 rho <= 0 or P not positive definite; 3 sigma > 1
// (with 1e-9 of slack)
__device__ __forceinline__ int check_prim(const double* Q, int nf) {
    for (int k = 0; k < nf; ++k)
        if (!f64::is_finite(Q[k])) return 1;
    if (f64::le0(Q[0])) return 2;
    if (nf == 5 && f64::le0(Q[2])) return 2;
    if (clearly_realizable(Q, nf)) return 0;
    if (nf == 14) {
        double a = Q[4], b = Q[5], c = Q[6], d = Q[7], e = Q[8], f = Q[9];
        double m2 = a * d - b * b;
        double det = a * (d * f - e * e) - b * (b * f - e * c) + c * (b * e - d * c);
        if (!(a > 0.0) || !(m2 > 0.0) || !(det > 0.0)) return 2;
    }
    return raw_sigma(Q, nf) <= 1.0 + 1e-9 ? 0 : 3;
}

__device__ __forceinline__ void to_prim(const double* U, double* Q, int nf) {
    if (nf == 5) cons2prim5(U, Q); else cons2prim14(U, Q);
}
__device__ __forceinline__ void to_cons(const double* Q, double* U, int nf) {
    if (nf == 5) prim2cons5(Q, U); else prim2cons14(Q, U);
}

// Validate a dense input array; the smallest failing cell number and its
// code go to bad[0], bad[1] (64-bit: code in the top bits).
// (the field count is a template parameter so that the per-cell arrays stay
// in registers)
template <int NF>
__device__ __forceinline__ void validate_body(const CellMap& m, int kind, const double* src,
                                              unsigned long long* bad, unsigned* nonplanar,
                                              double* copy) {
    long long dense, dfs, dev, fs, idx;
    const bool has = cell_of(m, dense, dfs, dev, fs, idx);
    bool np = false;
    if (has) {
        double V[NF], Q[NF];
#pragma unroll
        for (int k = 0; k < NF; ++k) V[k] = src[dense + k * dfs];
        if (copy) {
#pragma unroll
            for (int k = 0; k < NF; ++k) copy[dense + k * dfs] = V[k];
        }
        if (kind == 0) {
#pragma unroll
            for (int k = 0; k < NF; ++k) Q[k] = V[k];
        } else {
            to_prim(V, Q, NF);
        }
        int code = check_prim(Q, NF);
        if (code) atomicMin(bad, ((unsigned long long)idx << 2) | (unsigned long long)code);
        // planar iff the z-odd moments (u_z, P_xz, P_yz, q_z) vanish; on the
        // conserved side they are rho u_z, E_xz, E_yz, H_z (same positions)
        if (NF == 14) {
            auto zero = [](double x) {
                return ((f64::hi32(x) & 0x7fffffffu) | f64::lo32(x)) == 0u;
            };
            np = !(zero(V[3]) && zero(V[6]) && zero(V[8]) && zero(V[12]));
        }
    }
    // one atomic per warp that saw a non-planar cell (blocks are whole warps)
    if (__any_sync(0xffffffffu, np) && (threadIdx.x & 31) == 0) atomicOr(nonplanar, 1u);
}

// copy (may be null): receives src, same layout (a host-resident src is then
// read once, over the host link, by this kernel)
extern "C" __global__ void mxe_k_validate(CellMap m, int nf, int kind, const double* src,
                                          unsigned long long* bad, unsigned* nonplanar,
                                          double* copy) {
    if (nf == 5) validate_body<5>(m, kind, src, bad, nonplanar, copy);
    else validate_body<14>(m, kind, src, bad, nonplanar, copy);
}

// planar: the state has no z-odd moments (ten fields are converted).  W (may
// be null): FP32 primitives of a mixed grid, NF fields or (planar) ten.
// FP64-pipe bound: 4096 x 4096 cells of 14 moments, primitive in: 1.37 ms + 1.75 ms
// for W from the conserved state; in one pass with ten fields and W from the
// given primitives the two and the check fit the memory traffic
// better: 4096 x 4096 set-up 6.0 -> 3.0 ms in all.
template <int NF>
__device__ __forceinline__ void setstate_body(const CellMap& m, int kind, const double* src,
                                              double* U, float* Wp, bool planar) {
    long long dense, dfs, dev, fs, idx;
    if (!cell_of(m, dense, dfs, dev, fs, idx)) return;
    if constexpr (NF == 14) {
        if (kind == 0 && planar) {
            double Q[NP], C[NP];
#pragma unroll
            for (int k = 0; k < NP; ++k) Q[k] = src[dense + planar_field(k) * dfs];
            prim2cons_p(Q, C);
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                U[dev + planar_field(k) * fs] = C[k];
                if (Wp) Wp[dev + k * fs] = f64::to_f32(Q[k]);
            }
            const int odd[4] = {3, 6, 8, 12};
#pragma unroll
            for (int k = 0; k < 4; ++k) U[dev + odd[k] * fs] = 0.0;
            return;
        }
    }
    double V[NF], C[NF];
#pragma unroll
    for (int k = 0; k < NF; ++k) V[k] = src[dense + k * dfs];
    if (kind == 0) {
        to_cons(V, C, NF);
#pragma unroll
        for (int k = 0; k < NF; ++k)
            if (Wp) Wp[dev + k * fs] = f64::to_f32(V[k]);
    } else {
#pragma unroll
        for (int k = 0; k < NF; ++k) C[k] = V[k];
    }
#pragma unroll
    for (int k = 0; k < NF; ++k) U[dev + k * fs] = C[k];
}

extern "C" __global__ void mxe_k_setstate(CellMap m, int nf, int kind, const double* src,
                                          double* U, float* W, int planar) {
    if (nf == 5) setstate_body<5>(m, kind, src, U, nullptr, false);
    else setstate_body<14>(m, kind, src, U, W, planar != 0);
}

// kind 0 primitive, 1 conserved, 2 raw sigma (one field)
template <int NF>
__device__ __forceinline__ void getstate_body(const CellMap& m, int kind, const double* U,
                                              double* dst) {
    long long dense, dfs, dev, fs, idx;
    if (!cell_of(m, dense, dfs, dev, fs, idx)) return;
    double V[NF], Q[NF];
#pragma unroll
    for (int k = 0; k < NF; ++k) V[k] = U[dev + k * fs];
    if (kind == 1) {
#pragma unroll
        for (int k = 0; k < NF; ++k) dst[dense + k * dfs] = V[k];
        return;
    }
    to_prim(V, Q, NF);
    if (kind == 0) {
#pragma unroll
        for (int k = 0; k < NF; ++k) dst[dense + k * dfs] = Q[k];
        return;
    }
    dst[idx] = raw_sigma(Q, NF);
}

extern "C" __global__ void mxe_k_getstate(CellMap m, int nf, int kind, const double* U,
                                          double* dst) {
    if (nf == 5) getstate_body<5>(m, kind, U, dst);
    else getstate_body<14>(m, kind, U, dst);
}

// Boundary ghost states as the stencil sees them: prim -> conserved -> prim.
extern "C" __global__ void mxe_k_ghost(int nf, int n, const double* in, double* out) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    double Q[14], U[14];
    for (int k = 0; k < 14; ++k) Q[k] = in[s * 14 + k];
    to_cons(Q, U, nf);
    to_prim(U, Q, nf);
    for (int k = 0; k < 14; ++k) out[s * 14 + k] = k < nf ? Q[k] : 0.0;
}

// Diagnostics in two passes with a fixed summation order (the result does
// not depend on the scheduling of blocks).  Pass 1: each block writes
// DIAG_W partials: [0, nf) field sums over its cells, [16] min raw sigma,
// [17] sigma < sigma_lim, [18] sigma > 1, [19] non-positive, [20]
// non-finite cell counts (counts held exactly as doubles).
constexpr int DIAG_W = 24;

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_min_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

template <int NF>
__device__ __forceinline__ void diag_body(const CellMap& m, const double* U, double sigma_lim,
                                          double* part) {
    constexpr int nf = NF;
    __shared__ double sh[4][DIAG_W];
    double v[DIAG_W];
#pragma unroll
    for (int k = 0; k < DIAG_W; ++k) v[k] = 0.0;
    v[16] = INFINITY;
    long long dense, dfs, dev, fs, idx;
    if (cell_of(m, dense, dfs, dev, fs, idx)) {
        double V[NF], Q[NF];
#pragma unroll
        for (int k = 0; k < nf; ++k) V[k] = U[dev + k * fs];
        bool fin = true;
#pragma unroll
        for (int k = 0; k < nf; ++k) {
            fin &= isfinite(V[k]);
            v[k] = V[k];
        }
        if (!fin) {
            v[20] = 1.0;
        } else {
            to_prim(V, Q, nf);
            bool pos = Q[0] > 0.0 &&
                       (nf == 5 ? Q[2] > 0.0 : (Q[4] > 0.0 && Q[7] > 0.0 && Q[9] > 0.0));
            if (!pos) {
                v[19] = 1.0;
            } else {
                double sg = raw_sigma(Q, nf);
                v[17] = sg < sigma_lim ? 1.0 : 0.0;
                v[18] = sg > 1.0 ? 1.0 : 0.0;
                v[16] = sg;
            }
        }
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < DIAG_W; ++k) {
        double r = k == 16 ? warp_min_d(v[k]) : warp_sum_d(v[k]);
        if (lane == 0) sh[w][k] = r;
    }
    __syncthreads();
    if (threadIdx.x < DIAG_W) {
        int k = threadIdx.x;
        double r = sh[0][k];
        for (int q = 1; q < 4; ++q) r = k == 16 ? fmin(r, sh[q][k]) : r + sh[q][k];
        part[((long long)blockIdx.y * gridDim.x + blockIdx.x) * DIAG_W + k] = r;
    }
}

extern "C" __global__ void __launch_bounds__(128)
mxe_k_diag(CellMap m, int nf, const double* U, double sigma_lim, double* part) {
    if (nf == 5) diag_body<5>(m, U, sigma_lim, part);
    else diag_body<14>(m, U, sigma_lim, part);
}

// Pass 2 (one block of 256 threads): acc[k] = the partials combined, each
// thread over a fixed stride of blocks, then a fixed tree.
extern "C" __global__ void __launch_bounds__(256)
mxe_k_diag_reduce(const double* part, long long nblocks, double* acc) {
    __shared__ double sh[256];
    for (int k = 0; k < 21; ++k) {
        double r = k == 16 ? INFINITY : 0.0;
        for (long long b = threadIdx.x; b < nblocks; b += 256) {
            double x = part[b * DIAG_W + k];
            r = k == 16 ? fmin(r, x) : r + x;
        }
        sh[threadIdx.x] = r;
        __syncthreads();
        for (int h = 128; h > 0; h >>= 1) {
            if (threadIdx.x < h)
                sh[threadIdx.x] = k == 16 ? fmin(sh[threadIdx.x], sh[threadIdx.x + h])
                                          : sh[threadIdx.x] + sh[threadIdx.x + h];
            __syncthreads();
        }
        if (threadIdx.x == 0) acc[k] = sh[0];
        __syncthreads();
    }
}

}  // namespace mxe
