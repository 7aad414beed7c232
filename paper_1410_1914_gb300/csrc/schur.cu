// Steady state of the D3Q7 scheme as a fixed point in C alone.
//
// At steady state every population obeys, along the line of its own axis,
//     g_i(x + c_i) = g*_i(x) = (1 - omega_x) g_i(x) + omega_x w C(x) + w S(x)
// (Eq. 21 with the equilibrium w C of Eq. 23 and the a_i S source), and a
// closed face returns the population along the opposite direction (wall:
// times 1 or the catalytic factor r; fixed value: -g* + 2 w C_bc; zero flux:
// g*).  Given C, each run of open faces along an axis is therefore a linear
// two-stream problem with two unknowns (the populations entering its two
// ends), solved exactly by sweeps along the run; a closed loop of y or z
// (no closed face) is a geometric series.  The rest population is
// g_0 = w_0 (C + S / omega).  Summing the incoming populations,
//     C = F(C) = (sum_{i>0} g_i[C] + w_0 S / omega) / (1 - w_0),
// an affine map whose fixed point is exactly the steady state the time
// march approaches; the populations are eliminated without approximation.
//
// (I - M) C = f (M: the linear part of F, f = F(0)) is solved by flexible
// GMRES in FP64, preconditioned by the cell-centred finite-volume operator
// of the same relaxation times: link conductance 2 D_a D_b / (D_a + D_b)
// with D = (1/omega - 1/2) / 4 (the steady one-dimensional flux of the
// scheme, exact in 1D), 2 D on a fixed-value face, 2 k D / (2 D + k) on a
// catalytic face; its systems are solved by diagonal-preconditioned
// conjugate gradients in FP64.  This reaches the steady state where the
// pore / ionomer contrast of dissolved O2 (relaxation times within 1e-5 of
// 1/2 in the ionomer, Eq. 10-15) makes the march and the population-space
// Krylov solves stall: relaxation times near 1/2 leave the non-equilibrium
// populations almost undamped, which the line sweeps resolve exactly.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <chrono>
#include <vector>

#include "device_util.cuh"
#include "dsa.cuh"
#include "handle.cuh"

using namespace cl;

namespace {

constexpr int kSB = 256;          // threads per block
constexpr double kWa = 0.125;     // D3Q7 axis weight
constexpr double kWr = 0.25;      // D3Q7 rest weight

// A run of open faces along one axis: len cells, or -len for a closed loop
// (y, z) of len cells, listed in order from entry pos of the axis on.  p = kL g*_-(first) + hL enters at the
// first cell, m = kR g*_+(last) + hR at the last; al is the product of the
// cells' decays 1 - omega, inv = 1 / (1 - kL al kR al) (a loop: 1 / (1 - al)).
struct Run {
    int pos, len;
    double al, inv, kL, kR, hL, hR;
};

struct SchurArgs {
    int nx, ny, nz, n;
    const int* __restrict__ list;
    const int* __restrict__ nb;         // [6][n], DsaLink below 0
    const double* __restrict__ D;       // per-cell diffusivity [m^2/s] (box)
    double dt_cs2dx2;                   // dt / (cs^2 dx^2): tau = 1/2 + D dt / (cs^2 dx^2) (Eq. 24)
    double rfac;                        // uniform catalytic factor
    const double* __restrict__ kscale;  // per-cell factor on k_lu (box, nullable)
    double k_lu;
    const double* __restrict__ src;     // per-cell source per step (box, nullable)
    double c_in, c_out;
    // formed once per call
    double* om64;   // [n] omega in FP64
    double* G;      // [6][n] conductance of each link (0 where closed)
    double* dinv;   // [n] 1 / diagonal of the finite-volume operator
    Run* runs;      // by axis, from run_base on
    long long run_base[3];
    int* ord;       // [3][n] the cells of each axis run by run, and
    double2* dso;   // [3][n] their 1 - omega and omega w
    int* n_runs;    // [3] runs, then [3] cells listed, then [3] cells that may start one
};

__device__ __forceinline__ double cat_factor(const SchurArgs& a, int c) {
    return a.kscale ? cell_rfac(a.k_lu, a.kscale[c]) : a.rfac;
}

// lattice diffusivity cs^2 (tau - 1/2) = D dt / dx^2
__device__ __forceinline__ double cell_D(const SchurArgs& a, int c) { return 0.25 * a.D[c] * a.dt_cs2dx2; }

// omega (FP64, from the cell's D as the FP64 oracle forms it) and the finite-volume operator L_D (link conductance
// 2 D_a D_b / (D_a + D_b); 2 D on a fixed-value face; 2 k D / (2 D + k) on a catalytic face)
__global__ void __launch_bounds__(kSB) k_schur_setup(SchurArgs a) {
    for (int i = blockIdx.x * kSB + threadIdx.x; i < a.n; i += gridDim.x * kSB) {
        const int c = a.list[i];
        const double Dc = cell_D(a, c);
        double diag = 0.0;
        for (int d = 0; d < 6; ++d) {
            const int to = a.nb[(long long)d * a.n + i];
            double g = 0.0;
            if (to >= 0) {
                const double Dn = cell_D(a, a.list[to]);
                g = 2.0 * Dc * Dn / (Dc + Dn);
                diag += g;
            } else if (to == DSA_FIXED) {
                diag += 2.0 * Dc;
            } else if (to == DSA_SINK) {
                const double k = a.k_lu * (a.kscale ? a.kscale[c] : 1.0);
                diag += 2.0 * k * Dc / (2.0 * Dc + k);
            }
            a.G[(long long)d * a.n + i] = g;
        }
        a.om64[i] = 1.0 / (0.5 + a.D[c] * a.dt_cs2dx2);
        a.dinv[i] = diag > 0.0 ? 1.0 / diag : 0.0;
    }
}

// Returning factor and added amount of closed link `to` of box cell c
__device__ __forceinline__ void end_rule(const SchurArgs& a, int to, bool minus, int c, double& k, double& h) {
    h = 0.0;
    if (to == DSA_FIXED) {  // only the x faces of the box have one
        k = -1.0;
        h = 2.0 * kWa * (minus ? a.c_in : a.c_out);
    } else {
        k = to == DSA_SINK ? cat_factor(a, c) : 1.0;
    }
}

// whether cell i may start a run of axis ax: its - face is closed, or it is the cell of coordinate 0 of a y or z line
__device__ __forceinline__ bool may_start(const SchurArgs& a, int ax, int i) {
    if (a.nb[(long long)(2 * ax + 1) * a.n + i] < 0) return true;
    if (ax == 0) return false;
    const int c = a.list[i];
    return (ax == 1 ? (c / a.nx) % a.ny : c / (a.nx * a.ny)) == 0;
}

// how many runs there can be, which the allocation follows (a run record is 56 bytes; one for every cell and axis was
// more than the operator)
__global__ void __launch_bounds__(kSB) k_schur_count(SchurArgs a) {
    int cnt[3] = {0, 0, 0};
    for (int i = blockIdx.x * kSB + threadIdx.x; i < a.n; i += gridDim.x * kSB)
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) cnt[ax] += may_start(a, ax, i);
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const int t = __reduce_add_sync(0xffffffffu, cnt[ax]);
        if ((threadIdx.x & 31) == 0 && t) atomicAdd(a.n_runs + 6 + ax, t);
    }
}

// The runs of axis blockIdx.y, in any order (runs do not share cells): each cell whose - face is closed starts one;
// a y or z line without a closed face is a loop, recorded by its cell of coordinate 0.
__global__ void __launch_bounds__(kSB) k_schur_runs(SchurArgs a) {
    const int ax = blockIdx.y;
    const int* __restrict__ fwd = a.nb + (long long)(2 * ax) * a.n;
    const int* __restrict__ bwd = a.nb + (long long)(2 * ax + 1) * a.n;
    for (int i = blockIdx.x * kSB + threadIdx.x; i < a.n; i += gridDim.x * kSB) {
        if (!may_start(a, ax, i)) continue;
        Run r;
        const bool start = bwd[i] < 0;
        int len = 1, last = i, t = fwd[i];
        r.al = 1.0 - a.om64[i];
        for (; t >= 0 && t != i; t = fwd[t]) {
            r.al *= 1.0 - a.om64[t];
            last = t;
            ++len;
        }
        if (start) {
            r.len = len;
            end_rule(a, bwd[i], true, a.list[i], r.kL, r.hL);
            end_rule(a, fwd[last], false, a.list[last], r.kR, r.hR);
            r.inv = 1.0 / (1.0 - r.kL * r.al * r.kR * r.al);
        } else {
            if (t != i) continue;  // the line has a closed face
            r.len = -len;
            r.inv = 1.0 / (1.0 - r.al);
            r.kL = r.kR = r.hL = r.hR = 0.0;
        }
        r.pos = atomicAdd(a.n_runs + 3 + ax, len);
        const long long at = (long long)ax * a.n + r.pos;
        for (int k = 0, u = i; k < len; ++k, u = fwd[u]) {
            a.ord[at + k] = u;
            a.dso[at + k] = make_double2(1.0 - a.om64[u], a.om64[u] * kWa);
        }
        a.runs[a.run_base[ax] + atomicAdd(a.n_runs + ax, 1)] = r;
    }
}

// A warp's time is its longest run's FP64 instructions, at 16 cycles each on
// an SM: blocks of one warp spread the runs over the SMs (16^3: 23 us with 256
// threads a block).
constexpr int kWalkT = 32;

// One thread per run: the incoming populations of the two directions of its
// axis from C into T[axis] (their sum).  OUT: also the post-collision
// populations (f32 state layout, N cells a plane) and, per run, the amounts
// consumed on its catalytic ends (flux[axis]), entering at x = 0 (flux[3]) and
// leaving at x = L (flux[4]), lattice units per step, FP64.
template <bool OUT>
__global__ void __launch_bounds__(kWalkT) k_walk(SchurArgs a, const double* __restrict__ C, double* __restrict__ T,
                                              int homog, float* __restrict__ pop, long long N,
                                              double* __restrict__ flux) {
    const int ax = blockIdx.y, n = a.n;
    double* __restrict__ Ta = T + (long long)ax * n;
    const int nr = a.n_runs[ax];
    const bool src = !homog && a.src;
    for (int q = blockIdx.x * kWalkT + threadIdx.x; q < nr; q += gridDim.x * kWalkT) {
        const Run r = a.runs[a.run_base[ax] + q];
        const bool loop = r.len < 0;
        const int len = loop ? -r.len : r.len;
        const int* __restrict__ ord = a.ord + (long long)ax * n + r.pos;
        const double2* __restrict__ dso = a.dso + (long long)ax * n + r.pos;
        auto coef = [&](int t, double& dec, double& s) {
            const double2 ds = dso[t];
            const int i = ord[t];
            dec = ds.x;
            s = ds.y * C[i];
            if (src) s += kWa * a.src[a.list[i]];
        };
        // forward: g*_+(last) = al p + beB; backward: g*_-(first) = al m + beA
        double beA = 0.0, beB = 0.0, pre = 1.0;
#pragma unroll 4
        for (int t = 0; t < len; ++t) {
            double dec, s;
            coef(t, dec, s);
            beB = fma(dec, beB, s);
            beA = fma(pre, s, beA);
            pre *= dec;
        }
        double p, m;
        if (loop) {
            // populations arriving at the first cell from behind, and at the last cell from ahead
            p = beB * r.inv;
            m = beA * r.inv;
        } else {
            const double hL = homog ? 0.0 : r.hL, hR = homog ? 0.0 : r.hR;
            p = (r.kL * r.al * (r.kR * beB + hR) + r.kL * beA + hL) * r.inv;
            m = r.kR * (r.al * p + beB) + hR;
            if (OUT) {
                // what leaves through the run's end faces: g*_-(first) and g*_+(last)
                const double gA = r.al * m + beA, gB = r.al * p + beB;
                const int first = ord[0];
                const int tA = a.nb[(long long)(2 * ax + 1) * n + first], tB = a.nb[(long long)(2 * ax) * n + ord[len - 1]];
                double R = 0.0, jin = 0.0, jout = 0.0;
                if (tA == DSA_FIXED) jin = 2.0 * kWa * a.c_in - 2.0 * gA;
                else if (tA == DSA_SINK) R += (1.0 - r.kL) * gA;
                if (tB == DSA_FIXED) jout = 2.0 * gB - 2.0 * kWa * a.c_out;
                else if (tB == DSA_SINK) R += (1.0 - r.kR) * gB;
                flux[(long long)ax * n + first] = R;
                if (ax == 0) {
                    flux[3LL * n + first] = jin;
                    flux[4LL * n + first] = jout;
                }
            }
        }
        double g = p;
#pragma unroll 4
        for (int t = 0; t < len; ++t) {
            double dec, s;
            coef(t, dec, s);
            const int i = ord[t];
            Ta[i] = g;
            g = fma(dec, g, s);
            if (OUT) pop[(1 + 2 * ax) * N + a.list[i]] = (float)g;
        }
        g = m;
#pragma unroll 4
        for (int t = len - 1; t >= 0; --t) {
            double dec, s;
            coef(t, dec, s);
            const int i = ord[t];
            Ta[i] += g;
            g = fma(dec, g, s);
            if (OUT) pop[(2 + 2 * ax) * N + a.list[i]] = (float)g;
        }
    }
}

// F = (T + w0 S / omega) / (1 - w0), T the sum over the axes; out = F, or z - F (minus); OUT: the rest population
// g_0 = w0 (C + S / omega)
template <bool OUT>
__global__ void __launch_bounds__(kSB) k_walk_fin(SchurArgs a, const double* __restrict__ C,
                                                  const double* __restrict__ T, int homog, int minus,
                                                  double* __restrict__ out, float* __restrict__ pop) {
    const int n = a.n;
    for (int i = blockIdx.x * kSB + threadIdx.x; i < n; i += gridDim.x * kSB) {
        const double S = (!homog && a.src) ? a.src[a.list[i]] / a.om64[i] : 0.0;
        const double F = ((T[i] + T[n + i]) + T[2LL * n + i] + kWr * S) / (1.0 - kWr);
        out[i] = minus ? C[i] - F : F;
        if (OUT) pop[a.list[i]] = (float)(kWr * (C[i] + S));
    }
}

// The finite-volume operator for the resident conjugate gradients (pcg.cuh): z = L_D^{-1} v
struct FvOp {
    int n;
    const int* __restrict__ nb;
    const double* __restrict__ G;
    const double* __restrict__ dinv_;
    const double* __restrict__ v;
    double* __restrict__ z;
    struct Row {
        int j[6];
        double g[6];
    };
    __device__ __forceinline__ Row load(int i) const {
        Row r;
#pragma unroll
        for (int d = 0; d < 6; ++d) {
            r.j[d] = nb[(long long)d * n + i];
            r.g[d] = G[(long long)d * n + i];
        }
        return r;
    }
    template <class S>
    __device__ __forceinline__ double off(const Row& r, const double* u) const {
        double t = 0.0;
#pragma unroll
        for (int d = 0; d < 6; ++d)
            if (r.j[d] >= 0) t = fma(r.g[d], S::ld(u + r.j[d]), t);
        return t;
    }
    __device__ __forceinline__ double rhs(int i) const { return v[i]; }
    __device__ __forceinline__ double dinv(int i) const { return dinv_[i]; }
    __device__ __forceinline__ void done(int i, double x) const { z[i] = x; }
};

constexpr int kCgT64 = 256;
constexpr int kCgStreamT64 = 512;

bool prec_streams64(int n) { return (n + kCgT64 - 1) / kCgT64 > 8 * device_sms(); }

// Few cells go to one cluster: its barrier costs a third of the grid's meetings.  FP64 runs at 2 lanes per cycle and
// SM, so past a few hundred cells per SM the arithmetic outweighs that and the whole grid takes over.
cudaError_t prec64(const FvOp& op, const PcgArgs<double>& a, cudaStream_t s) {
    const int sms = device_sms(), n = op.n;
    const auto blocks = [&](int k) { return (n + k * kCgT64 - 1) / (k * kCgT64); };
    if (blocks(2) <= kPcgMaxCluster) {
        // the whole cluster, however few the cells
        const cudaError_t e =
            blocks(1) <= kPcgMaxCluster
                ? pcg_launch_cluster<double, FvOp, 1, kCgT64>(op, a, std::min(kPcgMaxCluster, (n + 31) / 32), s)
                : pcg_launch_cluster<double, FvOp, 2, kCgT64>(op, a, kPcgMaxCluster, s);
        if (e != cudaErrorLaunchOutOfResources) return e;
    }
    if (blocks(1) <= sms) return pcg_launch_grid<double, FvOp, 1, kCgT64>(op, a, std::min(sms, (n + 63) / 64), s);
    switch (blocks(1) <= 8 * sms ? (blocks(1) + sms - 1) / sms : 0) {
        case 2: return pcg_launch_grid<double, FvOp, 2, kCgT64>(op, a, sms, s);
        case 3:
        case 4: return pcg_launch_grid<double, FvOp, 4, kCgT64>(op, a, sms, s);
        case 5:
        case 6:
        case 7:
        case 8: return pcg_launch_grid<double, FvOp, 8, kCgT64>(op, a, sms, s);
    }
    return pcg_launch_grid<double, FvOp, 0, kCgStreamT64>(op, a, sms, s);
}

// h[j] = V_j . w (one block per vector and chunk of kDotCells cells; part[chunk][j])
constexpr int kDotCells = 8192;
__global__ void __launch_bounds__(kSB) k_mdot(const double* __restrict__ V, int n, const double* __restrict__ w,
                                              double* __restrict__ part) {
    const int c0 = blockIdx.y * kDotCells, c1 = min(n, c0 + kDotCells);
    const double* __restrict__ v = V + (long long)blockIdx.x * n;
    double acc[1] = {0.0};
    for (int c = c0 + threadIdx.x; c < c1; c += kSB) acc[0] = fma(v[c], w[c], acc[0]);
    block_sum_store<1>(acc, part + (long long)blockIdx.y * gridDim.x + blockIdx.x);
}

// part[0][j] += the other chunks' parts, in order: one thread per vector, its loads in flight together
__global__ void __launch_bounds__(32) k_mdot_sum(double* __restrict__ part, int m, int chunks) {
    const int j = blockIdx.x * 32 + threadIdx.x;
    if (j >= m) return;
    double h = part[j];
#pragma unroll 8
    for (int k = 1; k < chunks; ++k) h += part[(long long)k * m + j];
    part[j] = h;
}

// Up to this many chunks every block of k_msub adds them up itself, which saves a launch; beyond, blocks times chunks
// grows as the square of the cells.  Added up once, 60 iterations from the start (Pt layers, ms an iteration): 29 k
// cells 0.395 (four chunks, by every block), 50 k 0.581 to 0.551, 118 k 1.10 to 0.90, 943 k 19.4 to 6.9, 1.84 M 61.3
// to 13.8.
constexpr int kFoldChunks = 4;

// w -= sum_j h[j] V_j with h[j] = sum over chunks of part[chunk][j]: blocks of 32 cells, the vectors shared out over
// 8 warps.  hout gets h (block 0); nrm (nullable): this block's part of |w|^2.
__global__ void __launch_bounds__(kSB) k_msub(const double* __restrict__ V, int n, int m, int chunks,
                                              const double* __restrict__ part, double* __restrict__ w,
                                              double* __restrict__ hout, double* __restrict__ nrm) {
    __shared__ double sh[kSB / 32][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.x * 32 + lane;
    double acc = 0.0;
    for (int j = warp; j < m; j += kSB / 32) {
        double h = part[j];
        for (int k = 1; k < chunks; ++k) h += part[(long long)k * m + j];
        if (c < n) acc = fma(h, V[(long long)j * n + c], acc);
        if (blockIdx.x == 0 && lane == 0) hout[j] = h;
    }
    sh[warp][lane] = acc;
    __syncthreads();
    if (warp == 0) {
        double t = 0.0;
        for (int k = 0; k < kSB / 32; ++k) t += sh[k][lane];
        double v = 0.0;
        if (c < n) {
            v = w[c] - t;
            w[c] = v;
        }
        if (nrm) {
            v *= v;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) nrm[blockIdx.x] = v;
        }
    }
}

// parts of |v|^2, 32 cells each
__global__ void __launch_bounds__(kSB) k_norm_part(const double* __restrict__ v, int n, double* __restrict__ nrm) {
    const int c = blockIdx.x * kSB + threadIdx.x;
    double t = c < n ? v[c] * v[c] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0 && (c >> 5) < (n + 31) / 32) nrm[c >> 5] = t;
}

// *out = sqrt(sum of the parts), one block
__global__ void __launch_bounds__(kSB) k_norm_fin(const double* __restrict__ nrm, int parts, double* __restrict__ out) {
    double acc[1] = {0.0};
    for (int k = threadIdx.x; k < parts; k += kSB) acc[0] += nrm[k];
    __shared__ double tot[1];
    block_sum_store<1>(acc, tot);
    if (threadIdx.x == 0) *out = sqrt(tot[0]);
}

// y = x / *norm (not touched where the norm is 0)
__global__ void __launch_bounds__(kSB) k_scale64(int n, const double* __restrict__ norm, const double* __restrict__ x,
                                                 double* __restrict__ y) {
    __shared__ double f;
    if (threadIdx.x == 0) f = *norm > 0.0 ? 1.0 / *norm : 0.0;
    __syncthreads();
    if (f == 0.0) return;
    for (int c = blockIdx.x * kSB + threadIdx.x; c < n; c += gridDim.x * kSB) y[c] = f * x[c];
}

// x += sum_k y[k] Z_k
__global__ void __launch_bounds__(kSB) k_comb64(const double* __restrict__ Z, int n, int m,
                                                const double* __restrict__ y, double* __restrict__ x) {
    for (int c = blockIdx.x * kSB + threadIdx.x; c < n; c += gridDim.x * kSB) {
        double t = x[c];
        for (int k = 0; k < m; ++k) t = fma(y[k], Z[(long long)k * n + c], t);
        x[c] = t;
    }
}

// sums over the cells of the three axes' consumption, the inflow and the outflow
__global__ void __launch_bounds__(1024) k_flux_sum(const double* __restrict__ flux, int n, double* __restrict__ out) {
    double acc[3] = {0.0, 0.0, 0.0};
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        acc[0] += (flux[i] + flux[n + i]) + flux[2LL * n + i];
        acc[1] += flux[3LL * n + i];
        acc[2] += flux[4LL * n + i];
    }
    block_sum_store<3>(acc, out);
}

// C of the stored state, less the last collision's source
__global__ void __launch_bounds__(kSB) k_field64(SchurArgs a, long long N, const float* __restrict__ pop,
                                                 double* __restrict__ C) {
    for (int i = blockIdx.x * kSB + threadIdx.x; i < a.n; i += gridDim.x * kSB) {
        const int c = a.list[i];
        double v = 0.0;
        for (int q = 0; q < 7; ++q) v += (double)pop[q * N + c];
        C[i] = a.src ? v - a.src[c] : v;
    }
}

struct Mem {
    cudaStream_t s;
    std::vector<void*> p;
    explicit Mem(cudaStream_t st) : s(st) {}
    template <class T>
    cudaError_t get(T** out, long long n) {
        void* v = nullptr;
        cudaError_t e = cudaMallocAsync(&v, sizeof(T) * (size_t)(n > 0 ? n : 1), s);
        if (e == cudaSuccess) p.push_back(v);
        *out = (T*)v;
        return e;
    }
    ~Mem() {
        cudaStreamSynchronize(s);
        for (void* v : p) cudaFreeAsync(v, s);
        cudaStreamSynchronize(s);
    }
};

}  // namespace

extern "C" cl_status cl_lbm_solve_steady_lines(cl_handle h, double tol, int max_iter, int restart, double cg_tol,
                                               cl_steady_info* info) {
    if (!h) { set_msg_txt("NULL handle"); return CL_ERR_ARG; }
    if (!h->have_structure) { set_msg_txt("no structure loaded"); return CL_ERR_STATE; }
    if (h->march || h->q != 7) {
        set_msg_txt("the line-eliminated steady solve needs D3Q7 with the plain f32 population storage");
        return CL_ERR_STATE;
    }
    if (!(tol > 0.0) || max_iter < 1 || restart < 1 || !(cg_tol > 0.0 && cg_tol < 1.0)) {
        set_msg_txt("tol > 0, max_iter >= 1, restart >= 1 and 0 < cg_tol < 1 required");
        return CL_ERR_ARG;
    }
    auto t0 = std::chrono::steady_clock::now();
    cudaStream_t s = h->s;
    const long long N = h->N;
    const int m = restart < max_iter ? restart : max_iter;
    cl_steady_info inf;
    memset(&inf, 0, sizeof(inf));
    cl_status result = CL_ERR_NOT_CONVERGED;
    {
        Mem mem(s);
        // the active cells and their links (dsa.cuh)
        DsaCells d;
        d.q = 7;
        int* scan = nullptr;
        const int nscan = dsa_scan_blocks(N);
        CK(mem.get(&scan, nscan + 1));
        CK(mem.get(&d.inv, N));
        CK(launch_dsa_count(h->mask, nullptr, N, scan, scan + nscan, s));
        CK(cudaMemcpyAsync(&d.n, scan + nscan, sizeof(int), cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
        const int n = d.n;
        d.np = n;
        CK(mem.get(&d.list, n));
        CK(mem.get(&d.nb, 6LL * n));
        CK(mem.get(&d.sink, n));
        CK(mem.get(&d.dinv, n));
        CK(mem.get(&d.omega, n));
        CK(launch_dsa_number(h->mask, nullptr, N, scan, d.inv, d.list, s));
        StepArgs sa;
        memset(&sa, 0, sizeof(sa));
        sa.nx = h->nx; sa.ny = h->ny; sa.nz = h->nz; sa.N = N;
        sa.mask = h->mask;
        sa.omega = h->omega;
        sa.rsink = (float)reactive_sink_d(h);
        sa.kscale = h->kscale;
        sa.k_lu = h->k_lu;
        sa.bc_in = h->p.bc_in; sa.bc_out = h->p.bc_out;
        CK(launch_dsa_links7(d, sa, s));
        SchurArgs a;
        a.nx = h->nx; a.ny = h->ny; a.nz = h->nz; a.n = n;
        a.list = d.list;
        a.nb = d.nb;
        a.D = h->D;
        a.dt_cs2dx2 = h->dt / (0.25 * h->p.dx_m * h->p.dx_m);
        a.rfac = reactive_factor_d(h);
        a.kscale = h->kscale;
        a.k_lu = h->k_lu;
        a.src = h->src;
        a.c_in = h->p.c_in; a.c_out = h->p.c_out;
        CK(mem.get(&a.om64, n));
        CK(mem.get(&a.G, 6LL * n));
        CK(mem.get(&a.dinv, n));
        CK(mem.get(&a.ord, 3LL * n));
        CK(mem.get(&a.dso, 3LL * n));
        CK(mem.get(&a.n_runs, 9));
        CK(cudaMemsetAsync(a.n_runs, 0, 9 * sizeof(int), s));
        const int nb = std::min((n + kSB - 1) / kSB, 152 * 8);
        k_schur_count<<<nb, kSB, 0, s>>>(a);
        k_schur_setup<<<nb, kSB, 0, s>>>(a);
        CK(cudaGetLastError());
        int n_runs[3];  // at most
        CK(cudaMemcpyAsync(n_runs, a.n_runs + 6, sizeof(n_runs), cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
        a.run_base[0] = 0;
        a.run_base[1] = n_runs[0];
        a.run_base[2] = (long long)n_runs[0] + n_runs[1];
        CK(mem.get(&a.runs, (long long)n_runs[0] + n_runs[1] + n_runs[2]));
        k_schur_runs<<<dim3(nb, 3), kSB, 0, s>>>(a);
        CK(cudaGetLastError());
        const int most_runs = std::max(1, std::max(n_runs[0], std::max(n_runs[1], n_runs[2])));
        const dim3 walk_grid(std::min((most_runs + kWalkT - 1) / kWalkT, 152 * 64), 3);
        double *V = nullptr, *Z = nullptr, *x = nullptr, *w = nullptr, *T = nullptr, *part = nullptr, *nrm = nullptr;
        double *hv = nullptr, *dy = nullptr;
        const int chunks = (n + kDotCells - 1) / kDotCells, parts = (n + 31) / 32;
        CK(mem.get(&V, (long long)(m + 1) * n));
        CK(mem.get(&Z, (long long)m * n));
        CK(mem.get(&x, n));
        CK(mem.get(&w, n));
        CK(mem.get(&T, 3LL * n));
        CK(mem.get(&part, (long long)chunks * (m + 1)));
        CK(mem.get(&nrm, parts));
        CK(mem.get(&hv, 2LL * (m + 1) + 3));  // the two passes' coefficients, a norm, spare
        CK(mem.get(&dy, m));
        double* dnorm = hv + 2 * (size_t)(m + 1);
        // z = L_D^{-1} v to cg_tol (diagonal-preconditioned CG, FP64)
        PcgArgs<double> cg = {};
        cg.n = n;
        cg.tol2 = cg_tol * cg_tol;
        cg.max_iters = 100000;
        CK(mem.get(&cg.u, n));
        if (prec_streams64(n)) {
            CK(mem.get(&cg.x, n));
            CK(mem.get(&cg.r, n));
            CK(mem.get(&cg.p, n));
            CK(mem.get(&cg.s, n));
            CK(mem.get(&cg.w, n));
        }
        cg.meet_blocks = device_sms();
        char* meet_mem = nullptr;
        CK(mem.get(&meet_mem, (long long)pcg_meet_bytes(cg.meet_blocks)));
        cg.meet_mem = meet_mem;
        CK(mem.get(&cg.out, 1));
        CK(cudaMemsetAsync(cg.out, 0, sizeof(PcgOut), s));
        cg.waits = PcgWaits(h->wait_limit, h->never_arrive);
        cg.no_cluster = h->no_cluster;
        FvOp op;
        op.n = n;
        op.nb = d.nb;
        op.G = a.G;
        op.dinv_ = a.dinv;
        // F(C) (affine: homog = 0; linear part: homog = 1) or C - F(C) (minus) into out
        auto apply_F = [&](const double* C, int homog, int minus, double* out) -> cl_status {
            k_walk<false><<<walk_grid, kWalkT, 0, s>>>(a, C, T, homog, nullptr, N, nullptr);
            k_walk_fin<false><<<nb, kSB, 0, s>>>(a, C, T, homog, minus, out, nullptr);
            CK(cudaGetLastError());
            return CL_OK;
        };
        auto norm = [&](const double* v, double* out) -> cl_status {
            k_norm_part<<<(n + kSB - 1) / kSB, kSB, 0, s>>>(v, n, nrm);
            k_norm_fin<<<1, kSB, 0, s>>>(nrm, parts, dnorm);
            CK(cudaGetLastError());
            CK(cudaMemcpyAsync(out, dnorm, sizeof(double), cudaMemcpyDeviceToHost, s));
            CK(cudaStreamSynchronize(s));
            return CL_OK;
        };
        // start from the current state's concentration
        k_field64<<<nb, kSB, 0, s>>>(a, N, h->pop[h->cur], x);
        CK(cudaGetLastError());
        // the scale of the residual: |b| = |F(0)|, the right-hand side of (I - M) C = b; a warm
        // start that is already close needs no iteration
        double r0 = 0.0;
        CK(cudaMemsetAsync(w, 0, sizeof(double) * (size_t)n, s));
        CKS(apply_F(w, 0, 0, V));
        CKS(norm(V, &r0));
        if (!(r0 > 0.0)) r0 = 1.0;
        std::vector<double> H((size_t)(m + 1) * m), cs_(m), sn_(m), g(m + 1), hcol(m + 1), hh(2 * (size_t)(m + 1) + 1);
        while (inf.iterations < max_iter) {
            // r = F(x) - x  into V[0] (its negative; the sign enters below)
            CKS(apply_F(x, 0, 1, w));
            double beta;
            CKS(norm(w, &beta));
            inf.residual = beta / r0;
            if (!isfinite(beta)) { set_msg_txt("non-finite residual"); result = CL_ERR_DIVERGED; break; }
            if (beta <= tol * r0 || beta == 0.0) { result = CL_OK; break; }
            k_scale64<<<nb, kSB, 0, s>>>(n, dnorm, w, V);
            std::fill(g.begin(), g.end(), 0.0);
            g[0] = -beta;
            int j = 0;
            for (; j < m && inf.iterations < max_iter; ++j) {
                op.v = V + (long long)j * n;
                op.z = Z + (long long)j * n;
                CK(prec64(op, cg, s));
                // w = (I - M) z = z - F_lin(z)
                CKS(apply_F(op.z, 1, 1, w));
                // classical Gram-Schmidt, twice; |w| and the next vector
                for (int pass = 0; pass < 2; ++pass) {
                    k_mdot<<<dim3(j + 1, chunks), kSB, 0, s>>>(V, n, w, part);
                    if (chunks > kFoldChunks) k_mdot_sum<<<(j + 32) / 32, 32, 0, s>>>(part, j + 1, chunks);
                    k_msub<<<parts, kSB, 0, s>>>(V, n, j + 1, chunks > kFoldChunks ? 1 : chunks, part, w,
                                                 hv + (size_t)pass * (j + 1), pass ? nrm : nullptr);
                }
                double* hn_dev = hv + 2 * (size_t)(j + 1);
                k_norm_fin<<<1, kSB, 0, s>>>(nrm, parts, hn_dev);
                k_scale64<<<nb, kSB, 0, s>>>(n, hn_dev, w, V + (long long)(j + 1) * n);
                CK(cudaGetLastError());
                PcgOut po;
                CK(cudaMemcpyAsync(&po, cg.out, sizeof(po), cudaMemcpyDeviceToHost, s));
                CK(cudaMemcpyAsync(hh.data(), hv, sizeof(double) * (2 * (size_t)(j + 1) + 1), cudaMemcpyDeviceToHost, s));
                CK(cudaStreamSynchronize(s));
                if (po.gave_up) {
                    set_msg_txt("a wait of the steady solve's blocks for one another ran out");
                    return CL_ERR_TIMEOUT;
                }
                if (po.bad == 1) { set_msg_txt("inner conjugate gradients broke down"); return CL_ERR_DIVERGED; }
                inf.inner_iterations += po.iters;
                for (int k = 0; k <= j; ++k) hcol[k] = hh[k] + hh[j + 1 + k];
                const double hn = hh[2 * (size_t)(j + 1)];
                hcol[j + 1] = hn;
                ++inf.iterations;
                // Givens rotations of the new column
                for (int k = 0; k < j; ++k) {
                    const double t = cs_[k] * hcol[k] + sn_[k] * hcol[k + 1];
                    hcol[k + 1] = -sn_[k] * hcol[k] + cs_[k] * hcol[k + 1];
                    hcol[k] = t;
                }
                const double den = hypot(hcol[j], hcol[j + 1]);
                cs_[j] = den > 0 ? hcol[j] / den : 1.0;
                sn_[j] = den > 0 ? hcol[j + 1] / den : 0.0;
                hcol[j] = den;
                hcol[j + 1] = 0.0;
                g[j + 1] = -sn_[j] * g[j];
                g[j] = cs_[j] * g[j];
                for (int k = 0; k <= j; ++k) H[(size_t)k * m + j] = hcol[k];
                if (fabs(g[j + 1]) <= 0.5 * tol * r0 || hn == 0.0) { ++j; break; }
            }
            // x += Z y, y from the triangular system H y = g
            std::vector<double> y(j, 0.0);
            for (int k = j - 1; k >= 0; --k) {
                double t = g[k];
                for (int l = k + 1; l < j; ++l) t -= H[(size_t)k * m + l] * y[l];
                y[k] = t / H[(size_t)k * m + k];
            }
            if (j > 0) {
                CK(cudaMemcpyAsync(dy, y.data(), sizeof(double) * j, cudaMemcpyHostToDevice, s));
                k_comb64<<<nb, kSB, 0, s>>>(Z, n, j, dy, x);
                CK(cudaGetLastError());
                CK(cudaStreamSynchronize(s));  // y is the host's
            }
            ++inf.cycles;
        }
        if (result == CL_ERR_NOT_CONVERGED) {
            // the residual of the last iterate
            CKS(apply_F(x, 0, 1, w));
            double rn;
            CKS(norm(w, &rn));
            inf.residual = r0 > 0 ? rn / r0 : 0.0;
            if (rn <= tol * r0) result = CL_OK;
        }
        // the state: post-collision populations of the steady field, and its fluxes in FP64
        double* flux = V;  // the basis is done with
        if (m < 4) CK(mem.get(&flux, 5LL * n));
        CK(cudaMemsetAsync(flux, 0, sizeof(double) * 5 * (size_t)n, s));
        k_walk<true><<<walk_grid, kWalkT, 0, s>>>(a, x, T, 0, h->pop[h->cur], N, flux);
        k_walk_fin<true><<<nb, kSB, 0, s>>>(a, x, T, 0, 0, w, h->pop[h->cur]);
        k_flux_sum<<<1, 1024, 0, s>>>(flux, n, hv);
        CK(cudaGetLastError());
        double fl[3];
        CK(cudaMemcpyAsync(fl, hv, sizeof(fl), cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
        inf.R = fl[0];
        inf.J_in = fl[1];
        inf.J_out = fl[2];
    }
    inf.seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    if (info) *info = inf;
    return result;
}
