// Diagonal-preconditioned conjugate gradients in one resident kernel, shared
// by the preconditioners of the steady solves (dsa.cu: f32, schur.cu: FP64).
//
// A solve is a few dozen to a few hundred iterations on a vector that fits
// the chip, so its time is the cost of the steps between iterations, not of
// memory: as five kernels per iteration it took about 46 us an iteration at
// 96^3 (400 k active cells), of which the kernels' own work was a fraction.
// Here every thread keeps the x, r, p, s = L p and w = L u of its cells in
// registers; only u = M^-1 r goes through memory, because the neighbours
// read it.  The recurrences are those of Chronopoulos and Gear (J. Comput.
// Appl. Math. 25 (1989) 153): r.u, u.L u and r.r come from one reduction, so
// an iteration has two meetings of all blocks (u visible; the sums known)
// instead of three.  L u itself is r - sum_links g u_nb, since u = r / diag.
//
// The blocks meet in one of two ways: a cluster of up to 16 blocks through
// the hardware's cluster barrier, the partial sums pushed into each other's
// shared memory (3.1 us an iteration at 6 k cells); or the whole grid,
// launched cooperatively so that every block is resident, through a counter in
// global memory that one thread of each block polls, with a bounded wait (5.4
// us an iteration at 50 k cells, 7.6 us at 400 k on 152 blocks).  Partial sums
// tagged with their meeting's number, polled where they lie, save a trip to
// memory but have every block read every other's word while it is awaited:
// 8.9 and 14.1 us.
// The sums are formed in a fixed order, so that every block sees the same
// scalars, takes the same branches, and a solve repeats bit by bit.  The
// scalars are FP64, also where the vectors are f32: the threads' f32 sums are
// added without rounding errors (F3) and converted by the three warps that add
// up the block.  One thread of each block turns the sums into alpha and beta:
// FP64 runs at 1/64 of the FP32 rate here, and the two divisions done by every
// thread cost more than the rest of the iteration (9.4 us an iteration with 512
// threads a block, 14.7 us with 1024).  Against f32 scalars and f32 sums of a
// warp, a solve at 96^3 (4003 iterations) takes 51.1 ms instead of 49.5.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include <type_traits>

#include "device_util.cuh"

namespace cl {

struct PcgOut {
    double rr, rr0;  // r.r at the end and at the start
    int iters;
    int bad;  // 0 converged or out of iterations; 1 breakdown or non-finite; 2 nothing to solve
    // Set by a block whose wait ran out, of any kernel of the call (the Gram-Schmidt too), and never cleared: a block
    // may give up a meeting that the others still make, and then only this word says that its share is missing.
    unsigned gave_up;
};

// Words the blocks of a grid meet through.
struct PcgMeet {
    double* part;       // [2][3][blocks] partial sums
    unsigned* counter;  // arrivals (zeroed before the launch)
    unsigned* gave_up;  // PcgOut::gave_up
    long long limit;    // SM clocks a block waits
    int never_arrive;   // test hook (cl_lbm_set_wait_test): 1: no meeting comes about; 2: the last block waits for one
                        // arrival too many at its last meeting of a Gram-Schmidt
};
inline size_t pcg_meet_bytes(int blocks) { return sizeof(double) * 6 * (size_t)blocks + sizeof(unsigned); }

constexpr long long kPcgWaitClocks = 1LL << 32;  // about 2 s of SM clock

// How long the blocks of a call wait, from the handle's test settings (0: the default).
struct PcgWaits {
    long long limit = kPcgWaitClocks;
    int never_arrive = 0;
    PcgWaits() = default;
    PcgWaits(long long limit_clocks, int never) : limit(limit_clocks > 0 ? limit_clocks : kPcgWaitClocks), never_arrive(never) {}
};

inline PcgMeet pcg_meet(void* p, int blocks, PcgOut* out, const PcgWaits& w) {
    PcgMeet m;
    m.part = (double*)p;
    m.counter = (unsigned*)(m.part + 6 * (size_t)blocks);
    m.gave_up = &out->gave_up;
    m.limit = w.limit;
    m.never_arrive = w.never_arrive;
    return m;
}

// Scratch of a solve (device).  x, r, p, s, w: n values each, only for the
// variant whose vectors do not fit the registers.
template <class T>
struct PcgArgs {
    int n;
    int chunk;  // cells per block
    double tol2;
    int max_iters;
    T* u;
    T *x, *r, *p, *s, *w;
    PcgMeet meet;
    void* meet_mem;     // pcg_meet_bytes(meet_blocks)
    int meet_blocks;
    PcgWaits waits;
    int no_cluster;  // take the grid whatever the size
    PcgOut* out;  // zeroed once per call
};

constexpr int kPcgMaxCluster = 16;

// All blocks of a cooperative launch.
struct PcgGrid {
    unsigned target = 0;
    // everything the blocks wrote is visible to all; false when the wait ran out (last: of a Gram-Schmidt, for the hook)
    __device__ __forceinline__ bool meet(const PcgMeet& m, bool last = false) {
        bool ok = true;
        __syncthreads();
        if (gridDim.x == 1) return true;
        if (threadIdx.x == 0) {
            target += gridDim.x;
            const unsigned extra = m.never_arrive == 1 || (m.never_arrive == 2 && last && blockIdx.x == gridDim.x - 1);
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(m.counter) : "memory");
            const long long t0 = clock64();
            for (int polls = 1;; ++polls) {
                unsigned v;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(m.counter) : "memory");
                if (v >= target + extra) break;
                if ((polls & 1023) == 0) {  // another block's giving up, or this wait's own bound
                    if (clock64() - t0 > m.limit) atomicExch(m.gave_up, 1u);
                    if (*(volatile unsigned*)m.gave_up) { ok = false; break; }
                }
            }
        }
        return __syncthreads_and(ok);
    }
    // Slot v's partial of this block, and after a meeting the sum over all blocks (on every lane).
    __device__ __forceinline__ void put(const PcgMeet& m, double (*)[kPcgMaxCluster], int v, double val, int lane) {
        if (lane == 0) m.part[v * gridDim.x + blockIdx.x] = val;
    }
    __device__ __forceinline__ double get(const PcgMeet& m, double (*)[kPcgMaxCluster], int v, int lane) {
        double t = 0.0;
        for (unsigned b = lane; b < gridDim.x; b += 32) t += __ldcg(m.part + v * gridDim.x + b);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        return t;
    }
    template <class T>
    static __device__ __forceinline__ T ld(const T* u) { return *u; }  // the acquire above drops stale L1 lines
};

// One thread block cluster.
struct PcgCluster {
    __device__ __forceinline__ bool meet(const PcgMeet&) {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        return true;
    }
    __device__ __forceinline__ void put(const PcgMeet&, double (*box)[kPcgMaxCluster], int v, double val, int lane) {
        if (lane < (int)gridDim.x) {
            const unsigned local = (unsigned)__cvta_generic_to_shared(&box[v][blockIdx.x]);
            unsigned remote;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(lane));
            asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote), "d"(val) : "memory");
        }
    }
    __device__ __forceinline__ double get(const PcgMeet&, double (*box)[kPcgMaxCluster], int v, int lane) {
        double t = lane < (int)gridDim.x ? box[v][lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        return t;
    }
    template <class T>
    static __device__ __forceinline__ T ld(const T* u) { return __ldcg(u); }  // written by other SMs
};

// The operator of a solve:
//   Row        what one row of L needs (neighbour indices, conductances)
//   load(i)    the row of cell i
//   off(row)   sum over open links of g u[neighbour], u read through S::ld
//   rhs(i), dinv(i), done(i, x)
// K cells per thread in registers; K = 0 keeps the vectors in memory.
template <class T, class Op, int K, int NT, class S>
__global__ void __launch_bounds__(NT, 1) k_pcg(Op op, PcgArgs<T> a) {
    constexpr int KR = K > 0 ? K : 1;
    constexpr int NW = NT / 32;
    constexpr bool kKeep = K > 0 && K * sizeof(typename Op::Row) <= 192;  // rows stay in registers too
    static_assert(NW % 2 == 0 && NW >= 4, "an even number of warps");
    using Part = std::conditional_t<sizeof(T) == 8, double, F3>;
    __shared__ Part sh[3][sizeof(T) == 8 ? NT : NW];
    __shared__ double box[3][kPcgMaxCluster];
    __shared__ double tot[3];
    __shared__ T s_al, s_be;  // alpha, beta of the next iteration
    __shared__ int s_go;      // 1 iterate, 0 stop
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int i0 = blockIdx.x * a.chunk;
    const int i1 = min(a.n, i0 + a.chunk);
    T xr[KR] = {}, rr_[KR] = {}, pr[KR] = {}, sr[KR] = {}, wr[KR] = {}, dv[KR] = {};
    typename Op::Row rows[kKeep ? KR : 1];
    S sync;
    auto each = [&](auto&& f) {
        if constexpr (K > 0) {
#pragma unroll
            for (int k = 0; k < KR; ++k) {
                const int i = i0 + k * NT + tid;
                if (i < i1) f(k, i);
            }
        } else {
            for (int i = i0 + tid; i < i1; i += NT) f(0, i);
        }
    };
    auto X = [&](int k, int i) -> T& { if constexpr (K > 0) return xr[k]; else return a.x[i]; };
    auto R = [&](int k, int i) -> T& { if constexpr (K > 0) return rr_[k]; else return a.r[i]; };
    auto P = [&](int k, int i) -> T& { if constexpr (K > 0) return pr[k]; else return a.p[i]; };
    auto Sv = [&](int k, int i) -> T& { if constexpr (K > 0) return sr[k]; else return a.s[i]; };
    auto W = [&](int k, int i) -> T& { if constexpr (K > 0) return wr[k]; else return a.w[i]; };
    auto D = [&](int k, int i) -> T { if constexpr (K > 0) return dv[k]; else return op.dinv(i); };

    // w = L u and the three sums; false when a wait ran out
    auto apply = [&]() -> bool {
        if (!sync.meet(a.meet)) return false;  // u is visible
        T g0 = T(0), g1 = T(0), g2 = T(0);
        each([&](int k, int i) {
            const T d = D(k, i), r = R(k, i);
            T off;
            if constexpr (kKeep) off = op.template off<S>(rows[k], a.u);
            else off = op.template off<S>(op.load(i), a.u);
            const T u = d * r;
            const T w = (d != T(0) ? r : T(0)) - off;
            W(k, i) = w;
            g0 = fma(r, u, g0);
            g1 = fma(w, u, g1);
            g2 = fma(r, r, g2);
        });
        if constexpr (sizeof(T) == 8) {
            // three warps add up the threads' sums: a shuffle tree in every warp would issue an FP64 addition for
            // idle lanes too, and those are what the SM has least of
            sh[0][tid] = g0;
            sh[1][tid] = g1;
            sh[2][tid] = g2;
        } else {
            // the threads' f32 sums are added without a rounding error (F3) and turned into FP64 by the three warps that
            // add up the block: half of the lanes go on with g2, a quarter each with g0 and g1
            const bool hi16 = lane & 16, hi8 = lane & 8;
            const float x0 = __shfl_xor_sync(0xffffffffu, hi16 ? g0 : g2, 16), x1 = __shfl_xor_sync(0xffffffffu, g1, 16);
            float s0, e0, s1, e1;
            two_sum(hi16 ? g2 : g0, x0, s0, e0);
            two_sum(hi16 ? T(0) : g1, hi16 ? T(0) : x1, s1, e1);
            F3 v = {hi8 ? s1 : s0, hi8 ? e1 : e0, 0.f};
            f3_add(v, F3{__shfl_xor_sync(0xffffffffu, hi8 ? s0 : s1, 8), __shfl_xor_sync(0xffffffffu, hi8 ? e0 : e1, 8), 0.f});
#pragma unroll
            for (int o = 4; o > 0; o >>= 1)
                f3_add(v, F3{__shfl_xor_sync(0xffffffffu, v.a, o), __shfl_xor_sync(0xffffffffu, v.b, o),
                             __shfl_xor_sync(0xffffffffu, v.c, o)});
            if ((lane & 7) == 0 && lane < 24) sh[lane >> 3][warp] = v;
        }
        __syncthreads();
        if (warp < 3) {
            double v = 0.0;
            if constexpr (sizeof(T) == 8) {
                double v2 = 0.0;
#pragma unroll
                for (int k = 0; k < NW; k += 2) {
                    v += sh[warp][k * 32 + lane];
                    v2 += sh[warp][k * 32 + 32 + lane];
                }
                v += v2;
            } else {
                v = lane < NW ? f3_get(sh[warp][lane]) : 0.0;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            sync.put(a.meet, box, warp, v, lane);  // every lane holds the sum
        }
        if (!sync.meet(a.meet)) return false;
        if (warp < 3) {
            const double v = sync.get(a.meet, box, warp, lane);
            if (lane == 0) tot[warp] = v;
        }
        __syncthreads();
        return true;
    };

    each([&](int k, int i) {
        if constexpr (kKeep) rows[k] = op.load(i);
        const T b = op.rhs(i), d = op.dinv(i);
        if constexpr (K > 0) dv[k] = d;
        X(k, i) = T(0);
        P(k, i) = T(0);
        Sv(k, i) = T(0);
        R(k, i) = b;
        a.u[i] = d * b;
    });
    // the scalars are the last warp's: with few cells a block it has none
    constexpr int kLead = NT - 32;
    PcgOut o = {};
    // Scalars in FP64 for either type.  What lies between a meeting and the next update is a chain of FP64 latencies: with
    // f32 vectors, whose iterations are short, the two divisions go through f32 reciprocals (recip) side by side.
    double inv_gamma = 0.0, inv_alpha = 0.0, stop = 0.0;
    bool met = true;
    for (bool start = true;; start = false) {
        met = apply();
        if (!met) break;
        double gamma = 0.0, alpha = 0.0;
        bool formed = false;  // the reciprocals of this iteration
        if (tid == kLead) {
            const double gn = tot[0], delta = tot[1], rr = tot[2];
            int go = 1;
            double be = 0.0;
            gamma = gn;
            o.rr = rr;
            if (start) {
                o.rr0 = rr;
                stop = a.tol2 * rr;
            } else {
                ++o.iters;
            }
            if (!isfinite(gn) || !isfinite(rr) || !isfinite(delta)) { o.bad = 1; go = 0; }
            else if (rr == 0.0 || gn == 0.0) { o.bad = start ? 2 : 0; go = 0; }
            else if ((!start && rr <= stop) || o.iters >= a.max_iters) go = 0;
            else {
                be = gn * inv_gamma;
                double den = delta - be * gn * inv_alpha;
                const auto clear = [](float v) { return v > 1e-30f && v < 1e30f; };  // recip's range
                if (sizeof(T) == 4 && clear((float)den) && clear((float)gn)) {
                    inv_gamma = recip(gn);
                    alpha = gn * recip(den);
                    inv_alpha = den * inv_gamma;
                    formed = true;
                } else {
                    if (!(den > 0.0)) {  // rounding has spoilt the recurrence: start it again from this residual
                        den = delta;
                        be = 0.0;
                    }
                    if (!(den > 0.0) || !(gn > 0.0)) { o.bad = 1; go = 0; }
                    else alpha = gn / den;
                }
            }
            s_al = (T)alpha;
            s_be = (T)be;
            s_go = go;
        }
        __syncthreads();
        if (!s_go) break;
        const T al = s_al, be = s_be;
        if (tid == kLead && !formed) {  // while the others update
            inv_gamma = 1.0 / gamma;
            inv_alpha = 1.0 / alpha;
        }
        each([&](int k, int i) {
            const T d = D(k, i), r = R(k, i);
            const T p = fma(be, P(k, i), d * r);
            const T s = fma(be, Sv(k, i), W(k, i));
            P(k, i) = p;
            Sv(k, i) = s;
            X(k, i) = fma(al, p, X(k, i));
            const T rn = fma(-al, s, r);
            R(k, i) = rn;
            a.u[i] = d * rn;
        });
    }
    each([&](int k, int i) { op.done(i, X(k, i)); });
    if (blockIdx.x == 0 && tid == kLead) {  // gave_up is the waits'
        a.out->rr = o.rr;
        a.out->rr0 = o.rr0;
        a.out->iters = o.iters;
        a.out->bad = o.bad;
    }
}

// SMs of the current device
inline int device_sms() {
    int dev = 0, nsm = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    return nsm;
}

// cudaErrorLaunchOutOfResources, with no error left behind: the device (or the part of it that this context may use)
// cannot place such a cluster, and the caller takes the grid.
template <class T, class Op, int K, int NT>
cudaError_t pcg_launch_cluster(const Op& op, PcgArgs<T> a, int blocks, cudaStream_t s) {
    a.chunk = (a.n + blocks - 1) / blocks;
    if (a.chunk > K * NT) return cudaErrorInvalidValue;
    if (a.no_cluster) return cudaErrorLaunchOutOfResources;
    auto kern = k_pcg<T, Op, K, NT, PcgCluster>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(NT);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = blocks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int fit = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&fit, kern, &cfg);
    if (e != cudaSuccess || fit < 1) {
        cudaGetLastError();
        return cudaErrorLaunchOutOfResources;
    }
    return cudaLaunchKernelEx(&cfg, kern, op, a);
}

template <class T, class Op, int K, int NT>
cudaError_t pcg_launch_grid(const Op& op, PcgArgs<T> a, int blocks, cudaStream_t s) {
    a.chunk = (a.n + blocks - 1) / blocks;  // the same share for every block
    if ((K > 0 && a.chunk > K * NT) || blocks > a.meet_blocks) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(a.meet_mem, 0, pcg_meet_bytes(blocks), s);
    if (e != cudaSuccess) return e;
    a.meet = pcg_meet(a.meet_mem, blocks, a.out, a.waits);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(NT);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;  // every block resident: they wait on one another
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_pcg<T, Op, K, NT, PcgGrid>, op, a);
}

}  // namespace cl
