// Diffusion preconditioner and flexible-GMRES vector kernels of the
// preconditioned Krylov steady solve (plain f32 populations, either lattice).
//
// The slow modes of the step map S are diffusive: a correction of
// equilibrium shape, w_i eps, changes the cell sums by L eps in one step,
// where L is the graph Laplacian of the active cells with the lattice weight
// w_i on each link (the one-step exchange of equilibrium populations), 2 w_i
// on a fixed-concentration face (anti-bounce-back returns -w_i eps),
// (1 - r) w_i on a catalytic face (the sink keeps 1 - r of what meets it) and
// nothing on a bounce-back face.  The preconditioner P v = v + w_i eps with
// L eps = sum_i v_i puts those modes near 1, so that a Krylov method on
// (I - A) x = b (A: the step with zero boundary values) needs a number of
// step applications that does not grow with the box.  L is symmetric
// positive definite (with a fixed-concentration face or a sink) and is
// solved by conjugate gradients with its diagonal as preconditioner, in one
// resident kernel per solve (pcg.cuh).
//
// All vectors hold the active cells only (dsa.cuh): less than half of the
// box's memory, traffic and arithmetic on the layers of the paper.
#include "device_util.cuh"
#include "dsa.cuh"

namespace cl {

namespace {

constexpr int kDT = 256;
constexpr int kScanCells = 2048;  // cells per block of the numbering

__host__ __device__ constexpr int d19_cx(int i) {
    constexpr int t[19] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0};
    return t[i];
}
__host__ __device__ constexpr int d19_cy(int i) {
    constexpr int t[19] = {0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1};
    return t[i];
}
__host__ __device__ constexpr int d19_cz(int i) {
    constexpr int t[19] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1};
    return t[i];
}
// link weight of population i; opposite link (pairs 1-2, 3-4, ...)
template <int Q>
__host__ __device__ constexpr float link_w(int i) {
    return Q == 7 ? (i == 0 ? kW0 : kW1) : (i == 0 ? 1.f / 3.f : (i <= 6 ? 1.f / 18.f : 1.f / 36.f));
}
__host__ __device__ constexpr int link_opp(int i) { return i == 0 ? 0 : ((i & 1) ? i + 1 : i - 1); }

__device__ __forceinline__ bool cell_active(const uint16_t* m7, const uint32_t* m19, long long c) {
    return m7 ? (m7[c] & kActiveBit) != 0 : (m19[c] & kQ19Active) != 0;
}

// ------------------------------------------------------------- numbering
// active cells per block of kScanCells cells
__global__ void __launch_bounds__(kDT) k_dsa_count(const uint16_t* __restrict__ m7, const uint32_t* __restrict__ m19,
                                                   long long cells, int* __restrict__ part) {
    const long long c0 = (long long)blockIdx.x * kScanCells;
    int cnt = 0;
    for (int k = threadIdx.x; k < kScanCells; k += kDT) {
        const long long c = c0 + k;
        cnt += c < cells && cell_active(m7, m19, c);
    }
    __shared__ int sh[kDT / 32];
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < kDT / 32; ++w) t += sh[w];
        part[blockIdx.x] = t;
    }
}

// exclusive scan of the block counts, in place; the total to *count
__global__ void __launch_bounds__(1024) k_dsa_scan(int* __restrict__ part, int nblk, int* __restrict__ count) {
    __shared__ int sh[32];
    __shared__ int carry;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int b0 = 0; b0 < nblk; b0 += 1024) {
        const int b = b0 + threadIdx.x;
        const int v = b < nblk ? part[b] : 0;
        int s = v;
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += t;
        }
        if (lane == 31) sh[warp] = s;
        __syncthreads();
        if (warp == 0) {
            int t = sh[lane];
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, t, o);
                if (lane >= o) t += u;
            }
            sh[lane] = t;
        }
        __syncthreads();
        const int before = carry + (warp ? sh[warp - 1] : 0) + s - v;
        if (b < nblk) part[b] = before;
        __syncthreads();
        if (threadIdx.x == 0) carry += sh[31];
        __syncthreads();
    }
    if (threadIdx.x == 0) *count = carry;
}

// inv and list: warps take 32 cells at a time, in order within the block's range
__global__ void __launch_bounds__(kDT) k_dsa_number(const uint16_t* __restrict__ m7, const uint32_t* __restrict__ m19,
                                                    long long cells, const int* __restrict__ part,
                                                    int* __restrict__ inv, int* __restrict__ list) {
    constexpr int NW = kDT / 32;
    constexpr int per = kScanCells / NW;  // cells per warp
    __shared__ int cnt[NW];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long c0 = (long long)blockIdx.x * kScanCells + (long long)warp * per;
    int t = 0;
    for (int k = 0; k < per; k += 32) {
        const long long c = c0 + k + lane;
        t += __popc(__ballot_sync(0xffffffffu, c < cells && cell_active(m7, m19, c)));
    }
    if (lane == 0) cnt[warp] = t;
    __syncthreads();
    int at = part[blockIdx.x];
    for (int w = 0; w < warp; ++w) at += cnt[w];
    for (int k = 0; k < per; k += 32) {
        const long long c = c0 + k + lane;
        const bool act = c < cells && cell_active(m7, m19, c);
        const unsigned b = __ballot_sync(0xffffffffu, act);
        const int i = at + __popc(b & ((1u << lane) - 1u));
        if (c < cells) inv[c] = act ? i : -1;
        if (act) list[i] = (int)c;
        at += __popc(b);
    }
}

// ------------------------------------------------------------------ links
__device__ __forceinline__ int wrap(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

__global__ void __launch_bounds__(kDT) k_dsa_links7(DsaCells d, StepArgs a) {
    for (int i = blockIdx.x * kDT + threadIdx.x; i < d.n; i += gridDim.x * kDT) {
        const int c = d.list[i];
        const unsigned nx = (unsigned)a.nx, ny = (unsigned)a.ny;
        const unsigned row = (unsigned)c / nx;
        const int x = (int)((unsigned)c - row * nx), y = (int)(row % ny), z = (int)(row / ny);
        const uint16_t m = a.mask[c];
        const float sink = a.kscale ? (float)cell_sink(a.k_lu, a.kscale[c]) : a.rsink;
        float diag = 0.f;
#pragma unroll
        for (int k = 1; k <= 6; ++k) {
            int to;
            if ((m >> (k - 1)) & 1u) {
                if (k == 2 && x == 0) to = a.bc_in == CL_BC_DIRICHLET ? DSA_FIXED : DSA_NOFLUX;
                else if (k == 1 && x == a.nx - 1) to = a.bc_out == CL_BC_DIRICHLET ? DSA_FIXED : DSA_NOFLUX;
                else to = ((m >> (kReactShift + k - 1)) & 1u) ? DSA_SINK : DSA_WALL;
                diag += to == DSA_FIXED ? 2.f * kW1 : (to == DSA_SINK ? sink * kW1 : 0.f);
            } else {
                const int yy = wrap(y + d19_cy(k), a.ny), zz = wrap(z + d19_cz(k), a.nz);
                to = d.inv[x + d19_cx(k) + (long long)a.nx * (yy + (long long)a.ny * zz)];
                diag += kW1;
            }
            d.nb[(long long)(k - 1) * d.n + i] = to;
        }
        d.sink[i] = sink;
        d.dinv[i] = diag > 0.f ? 1.f / diag : 0.f;
        d.omega[i] = a.omega[c];
    }
}

// a closed link takes precedence over the face of the box, as in the step kernel
__global__ void __launch_bounds__(kDT) k_dsa_links19(DsaCells d, Q19Args a) {
    for (int i = blockIdx.x * kDT + threadIdx.x; i < d.n; i += gridDim.x * kDT) {
        const int c = d.list[i];
        const int row = c / a.px;
        const int x = c - row * a.px, y = row % a.ny, z = row / a.ny;
        const uint32_t m = a.mask[c];
        const uint32_t rb = (m & kQ19HasReact) ? a.react[c] : 0u;
        float diag = 0.f;
#pragma unroll
        for (int k = 1; k < 19; ++k) {
            const float w = link_w<19>(k);
            const int cx = d19_cx(k);
            int to;
            if ((m >> (k - 1)) & 1u) {
                to = ((rb >> (k - 1)) & 1u) ? DSA_SINK : DSA_WALL;
                if (to == DSA_SINK) diag += a.rsink * w;
            } else if ((cx < 0 && x == 0) || (cx > 0 && x == a.nx - 1)) {
                to = (cx < 0 ? a.bc_in : a.bc_out) == CL_BC_DIRICHLET ? DSA_FIXED : DSA_NOFLUX;
                if (to == DSA_FIXED) diag += 2.f * w;
            } else {
                const int yy = wrap(y + d19_cy(k), a.ny), zz = wrap(z + d19_cz(k), a.nz);
                to = d.inv[(long long)(x + cx) + (long long)a.px * (yy + (long long)a.ny * zz)];
                diag += w;
            }
            d.nb[(long long)(k - 1) * d.n + i] = to;
        }
        d.sink[i] = a.rsink;
        d.dinv[i] = diag > 0.f ? 1.f / diag : 0.f;
        d.omega[i] = a.omega[c];
    }
}

// -------------------------------------------------------------- operators
// w = z - A z: the step kernels' arithmetic on the active cells (pull-stream,
// closed links from the cell's own opposite population, BGK collision), with
// boundary values 0.
template <int Q>
__global__ void __launch_bounds__(kDT) k_dsa_apply(DsaCells d, const float* __restrict__ z, float* __restrict__ w) {
    const int n = d.n;
    const long long np = d.np;
    for (int i = blockIdx.x * kDT + threadIdx.x; i < n; i += gridDim.x * kDT) {
        float own[Q], g[Q];
        int to[Q];
#pragma unroll
        for (int k = 1; k < Q; ++k) to[k] = d.nb[(long long)(k - 1) * n + i];
#pragma unroll
        for (int k = 0; k < Q; ++k) own[k] = z[k * np + i];
        const float sink = d.sink[i], om = d.omega[i];
        g[0] = own[0];
#pragma unroll
        for (int k = 1; k < Q; ++k) {
            const int o = link_opp(k), t = to[o];  // population k arrives through link o
            const float back = own[o];
            float v = t >= 0 ? z[k * np + t] : back;
            if (t == DSA_FIXED) v = 0.f - back;
            else if (t == DSA_SINK) v = back - sink * back;
            g[k] = v;
        }
        float C;
        if constexpr (Q == 7) {
            C = ((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + g[6]);
        } else {
            C = (((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7]))) +
                (((g[8] + g[9]) + (g[10] + g[11])) + ((g[12] + g[13]) + (g[14] + g[15]))) + ((g[16] + g[17]) + g[18]);
        }
#pragma unroll
        for (int k = 0; k < Q; ++k) w[k * np + i] = own[k] - (g[k] - om * (g[k] - link_w<Q>(k) * C));
    }
}

// The Laplacian for pcg.cuh: u_nb summed per weight class, then weighted.
template <int Q>
struct LapOp {
    int n;
    long long np;
    const int* __restrict__ nb;
    const float* __restrict__ dinv_;
    const float* __restrict__ v;
    float* __restrict__ z;
    struct Row {
        int j[Q - 1];
    };
    __device__ __forceinline__ Row load(int i) const {
        Row r;
#pragma unroll
        for (int k = 0; k < Q - 1; ++k) r.j[k] = nb[(long long)k * n + i];
        return r;
    }
    template <class S>
    __device__ __forceinline__ float off(const Row& r, const float* u) const {
        float s = 0.f, t = 0.f;
#pragma unroll
        for (int k = 0; k < 6; ++k) s += r.j[k] >= 0 ? S::ld(u + r.j[k]) : 0.f;
        if constexpr (Q == 19) {
#pragma unroll
            for (int k = 6; k < 18; ++k) t += r.j[k] >= 0 ? S::ld(u + r.j[k]) : 0.f;
            return fmaf(link_w<19>(1), s, link_w<19>(7) * t);
        } else {
            return link_w<7>(1) * s;
        }
    }
    __device__ __forceinline__ float rhs(int i) const {
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < Q; ++k) s += v[k * np + i];
        return s;
    }
    __device__ __forceinline__ float dinv(int i) const { return dinv_[i]; }
    __device__ __forceinline__ void done(int i, float x) const {
#pragma unroll
        for (int k = 0; k < Q; ++k) z[k * np + i] = fmaf(link_w<Q>(k), x, v[k * np + i]);
    }
};

// ----------------------------------------------------------- Gram-Schmidt
// s + e += a b with the rounding errors of the product and of the sum kept
// (Dot2 of Ogita, Rump and Oishi, SIAM J. Sci. Comput. 26 (2005) 1955): the
// result is as if formed in twice the working precision.  V is normalised, so
// the products stay inside the f32 range.  FP64 runs at 1/64
// of the FP32 rate on this GPU, and a product of two f32 in FP64 takes three
// FP64 instructions (two conversions and the FMA).
__device__ __forceinline__ void dot2(float a, float b, float& s, float& e) {
    // rounded as written: a contraction to FMA would break the error terms
    const float p = __fmul_rn(a, b);
    const float pe = __fmaf_rn(a, b, -p);
    float se;
    two_sum(s, p, s, se);
    e = __fadd_rn(e, __fadd_rn(pe, se));
}

// the warp's sum of s + e on every lane, the errors of the additions kept
__device__ __forceinline__ void warp_dot2(float& s, float& e) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float a = __shfl_xor_sync(0xffffffffu, s, o), b = __shfl_xor_sync(0xffffffffu, e, o);
        float se;
        two_sum(s, a, s, se);
        e = __fadd_rn(__fadd_rn(e, b), se);
    }
}

constexpr int kMgsT = 512;

// One launch orthogonalises w against V[0..j]: w stays in registers (K4
// float4 per thread; 0: in memory), each V_k is read once from memory and a
// second time, for the subtraction, from the SM's own cache, and the blocks
// meet once per vector.  As a dot product, its finish and a subtraction per
// vector the same took 38 + 3 + 10 us per vector at 96^3.  A block whose wait
// runs out leaves its share of V[j + 1] unwritten; it says so in PcgOut::gave_up,
// not in col: at the last meeting the others may not miss it.
template <int K4>
__global__ void __launch_bounds__(kMgsT, 2) k_dsa_mgs(const float* __restrict__ V, long long stride, int j, float* w,
                                                      long long L4, float* vnext, double* __restrict__ col,
                                                      PcgMeet meet) {
    constexpr int KR = K4 > 0 ? K4 : 1;
    constexpr int NW = kMgsT / 32;
    __shared__ double sh[NW];
    __shared__ double tot;
    __shared__ float s_f;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long t0 = (long long)blockIdx.x * kMgsT + threadIdx.x, step = (long long)gridDim.x * kMgsT;
    float4 wr[KR];
    float4* w4 = reinterpret_cast<float4*>(w);
    auto each = [&](auto&& f) {
        if constexpr (K4 > 0) {
#pragma unroll
            for (int k = 0; k < KR; ++k) {
                const long long i = t0 + k * step;
                if (i < L4) f(wr[k], i);
            }
        } else {
            for (long long i = t0; i < L4; i += step) {
                float4 v = w4[i];
                f(v, i);
                w4[i] = v;  // this thread's own elements
            }
        }
    };
    // the sum over the grid of each thread's s + e, in a fixed order; false when a wait ran out.  Two
    // sets of partials in turn: a block still reading one is not overwritten.
    PcgGrid sync;
    int set = 0;
    auto total = [&](float s, float e, bool last = false) -> bool {
        warp_dot2(s, e);
        if (lane == 0) sh[warp] = (double)s + (double)e;
        __syncthreads();
        if (warp == 0) {
            double t = lane < NW ? sh[lane] : 0.0;
#pragma unroll
            for (int o = NW / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            sync.put(meet, nullptr, set, t, lane);
        }
        if (!sync.meet(meet, last)) return false;
        if (warp == 0) {
            const double t = sync.get(meet, nullptr, set, lane);
            if (lane == 0) { tot = t; s_f = (float)t; }
        }
        set ^= 1;
        __syncthreads();
        return true;
    };
    if constexpr (K4 > 0) each([&](float4& v, long long i) { v = w4[i]; });
    float h = 0.f;
    for (int k = 0; k <= j; ++k) {
        const float4* vk = reinterpret_cast<const float4*>(V + k * stride);
        const float4* vp = reinterpret_cast<const float4*>(V + (k > 0 ? k - 1 : 0) * stride);
        float s = 0.f, e = 0.f;
        each([&](float4& v, long long i) {
            const float4 b = __ldg(vk + i);
            if (k > 0) {
                const float4 q = __ldg(vp + i);
                v.x = fmaf(-h, q.x, v.x);
                v.y = fmaf(-h, q.y, v.y);
                v.z = fmaf(-h, q.z, v.z);
                v.w = fmaf(-h, q.w, v.w);
            }
            dot2(b.x, v.x, s, e);
            dot2(b.y, v.y, s, e);
            dot2(b.z, v.z, s, e);
            dot2(b.w, v.w, s, e);
        });
        if (k < j) {  // the next vector comes in while the blocks meet
            const float4* vx = reinterpret_cast<const float4*>(V + (k + 1) * stride);
            if ((lane & 7) == 0)
                for (long long i = t0; i < L4; i += step) asm volatile("prefetch.global.L2 [%0];" ::"l"(vx + i));
        }
        if (!total(s, e)) return;
        if (blockIdx.x == 0 && threadIdx.x == 0) col[k] = tot;
        h = s_f;
    }
    {
        const float4* vp = reinterpret_cast<const float4*>(V + (long long)j * stride);
        float s = 0.f, e = 0.f;
        each([&](float4& v, long long i) {
            const float4 q = __ldg(vp + i);
            v.x = fmaf(-h, q.x, v.x);
            v.y = fmaf(-h, q.y, v.y);
            v.z = fmaf(-h, q.z, v.z);
            v.w = fmaf(-h, q.w, v.w);
            dot2(v.x, v.x, s, e);
            dot2(v.y, v.y, s, e);
            dot2(v.z, v.z, s, e);
            dot2(v.w, v.w, s, e);
        });
        if (!total(s, e, true)) return;
    }
    if (threadIdx.x == 0) {
        const double nrm = sqrt(tot);
        if (blockIdx.x == 0) col[j + 1] = nrm;
        s_f = nrm > 0.0 ? (float)(1.0 / nrm) : 0.f;
    }
    __syncthreads();
    const float f = s_f;
    float4* vn = reinterpret_cast<float4*>(vnext);
    each([&](float4& v, long long i) { vn[i] = make_float4(f * v.x, f * v.y, f * v.z, f * v.w); });
}

constexpr int kMaxUpdate = 32;
__global__ void __launch_bounds__(kDT) k_dsa_update(float* __restrict__ e, const float* __restrict__ Z,
                                                    long long stride, int m, const double* __restrict__ y,
                                                    long long L) {
    __shared__ float f[kMaxUpdate];
    if (threadIdx.x < m) f[threadIdx.x] = (float)y[threadIdx.x];
    __syncthreads();
    for (long long i = blockIdx.x * (long long)kDT + threadIdx.x; i < L; i += (long long)gridDim.x * kDT) {
        float v = e[i];
        for (int k = 0; k < m; ++k) v = fmaf(f[k], Z[k * stride + i], v);
        e[i] = v;
    }
}

__global__ void __launch_bounds__(kDT) k_dsa_gather(DsaCells d, const float* __restrict__ c, long long cells,
                                                    float* __restrict__ out) {
    for (int i = blockIdx.x * kDT + threadIdx.x; i < d.n; i += gridDim.x * kDT) {
        const int at = d.list[i];
        for (int k = 0; k < d.q; ++k) out[(long long)k * d.np + i] = c[k * cells + at];
    }
}

__global__ void __launch_bounds__(kDT) k_dsa_add64(DsaCells d, const float* __restrict__ e, double sign,
                                                   long long cells, double* __restrict__ x) {
    for (int i = blockIdx.x * kDT + threadIdx.x; i < d.n; i += gridDim.x * kDT) {
        const int at = d.list[i];
        for (int k = 0; k < d.q; ++k) x[k * cells + at] += sign * (double)e[(long long)k * d.np + i];
    }
}

int cell_blocks(int n) {
    const int b = (n + kDT - 1) / kDT;
    return b < 1 ? 1 : (b < 152 * 16 ? b : 152 * 16);
}

// ------------------------------------------------------ dispatch of the CG
constexpr int kCgT = 512;       // threads per block
constexpr int kCgStreamT = 1024;

template <int Q>
LapOp<Q> lap_op(const DsaCells& d, const float* v, float* z) {
    LapOp<Q> op;
    op.n = d.n;
    op.np = d.np;
    op.nb = d.nb;
    op.dinv_ = d.dinv;
    op.v = v;
    op.z = z;
    return op;
}

template <int Q>
cudaError_t prec_q(const DsaCells& d, const float* v, float* z, const PcgArgs<float>& a, cudaStream_t s) {
    const LapOp<Q> op = lap_op<Q>(d, v, z);
    const int sms = device_sms();
    const auto blocks = [&](int k) { return (d.n + k * kCgT - 1) / (k * kCgT); };
    if (blocks(2) <= kPcgMaxCluster) {
        const cudaError_t e = pcg_launch_cluster<float, LapOp<Q>, 2, kCgT>(op, a, blocks(2), s);
        if (e != cudaErrorLaunchOutOfResources) return e;
    }
    if (blocks(2) <= sms) return pcg_launch_grid<float, LapOp<Q>, 2, kCgT>(op, a, blocks(2), s);
    switch (blocks(1) <= 8 * sms ? (blocks(1) + sms - 1) / sms : 0) {  // every SM, the fewest cells per thread
        case 3: return pcg_launch_grid<float, LapOp<Q>, 3, kCgT>(op, a, sms, s);
        case 4: return pcg_launch_grid<float, LapOp<Q>, 4, kCgT>(op, a, sms, s);
        case 5: return pcg_launch_grid<float, LapOp<Q>, 5, kCgT>(op, a, sms, s);
        case 6: return pcg_launch_grid<float, LapOp<Q>, 6, kCgT>(op, a, sms, s);
        case 7:
        case 8: return pcg_launch_grid<float, LapOp<Q>, 8, kCgT>(op, a, sms, s);
    }
    return pcg_launch_grid<float, LapOp<Q>, 0, kCgStreamT>(op, a, sms, s);
}

}  // namespace

int dsa_scan_blocks(long long cells) { return (int)((cells + kScanCells - 1) / kScanCells); }

cudaError_t launch_dsa_count(const uint16_t* mask7, const uint32_t* mask19, long long cells, int* part, int* count,
                             cudaStream_t s) {
    const int nb = dsa_scan_blocks(cells);
    k_dsa_count<<<nb, kDT, 0, s>>>(mask7, mask19, cells, part);
    k_dsa_scan<<<1, 1024, 0, s>>>(part, nb, count);
    return cudaGetLastError();
}

cudaError_t launch_dsa_number(const uint16_t* mask7, const uint32_t* mask19, long long cells, const int* part,
                              int* inv, int* list, cudaStream_t s) {
    k_dsa_number<<<dsa_scan_blocks(cells), kDT, 0, s>>>(mask7, mask19, cells, part, inv, list);
    return cudaGetLastError();
}

cudaError_t launch_dsa_links7(const DsaCells& d, const StepArgs& a, cudaStream_t s) {
    k_dsa_links7<<<cell_blocks(d.n), kDT, 0, s>>>(d, a);
    return cudaGetLastError();
}

cudaError_t launch_dsa_links19(const DsaCells& d, const Q19Args& a, cudaStream_t s) {
    k_dsa_links19<<<cell_blocks(d.n), kDT, 0, s>>>(d, a);
    return cudaGetLastError();
}

cudaError_t launch_dsa_apply(const DsaCells& d, const float* z, float* w, cudaStream_t s) {
    if (d.q == 19) k_dsa_apply<19><<<cell_blocks(d.n), kDT, 0, s>>>(d, z, w);
    else k_dsa_apply<7><<<cell_blocks(d.n), kDT, 0, s>>>(d, z, w);
    return cudaGetLastError();
}

bool dsa_prec_streams(int n) { return (n + kCgT - 1) / kCgT > 8 * device_sms(); }

cudaError_t launch_dsa_prec(const DsaCells& d, const float* v, float* z, PcgArgs<float> a, cudaStream_t s) {
    a.n = d.n;
    return d.q == 19 ? prec_q<19>(d, v, z, a, s) : prec_q<7>(d, v, z, a, s);
}

int dsa_mgs_blocks() { return 2 * device_sms(); }

template <int K4>
static cudaError_t mgs_k(int blocks, const float* V, long long stride, int j, float* w, long long L4, float* vnext,
                         double* col, void* meet_mem, PcgOut* out, const PcgWaits& waits, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(meet_mem, 0, pcg_meet_bytes(blocks), s);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(kMgsT);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_dsa_mgs<K4>, V, stride, j, w, L4, vnext, col, pcg_meet(meet_mem, blocks, out, waits));
}

cudaError_t launch_dsa_mgs(float* V, long long stride, int j, float* w, long long L, double* col, void* meet_mem,
                           PcgOut* out, const PcgWaits& waits, cudaStream_t s) {
    const long long L4 = L / 4;
    const int most = dsa_mgs_blocks();
    const auto blocks = [&](int k4) { return (L4 + (long long)k4 * kMgsT - 1) / ((long long)k4 * kMgsT); };
    float* vn = V + (long long)(j + 1) * stride;
    // small vectors: few blocks, whose meetings cost less; then every SM with the fewest elements per thread
    if (blocks(1) <= most) return mgs_k<1>((int)blocks(1), V, stride, j, w, L4, vn, col, meet_mem, out, waits, s);
    switch (blocks(1) <= 8LL * most ? (int)((blocks(1) + most - 1) / most) : 0) {
        case 2: return mgs_k<2>(most, V, stride, j, w, L4, vn, col, meet_mem, out, waits, s);
        case 3: return mgs_k<3>(most, V, stride, j, w, L4, vn, col, meet_mem, out, waits, s);
        case 4: return mgs_k<4>(most, V, stride, j, w, L4, vn, col, meet_mem, out, waits, s);
        case 5:
        case 6: return mgs_k<6>(most, V, stride, j, w, L4, vn, col, meet_mem, out, waits, s);
        case 7:
        case 8: return mgs_k<8>(most, V, stride, j, w, L4, vn, col, meet_mem, out, waits, s);
    }
    return mgs_k<0>(most, V, stride, j, w, L4, vn, col, meet_mem, out, waits, s);
}

cudaError_t launch_dsa_update(float* e, const float* Z, long long stride, int m, const double* y, long long L,
                              cudaStream_t s) {
    if (m > kMaxUpdate) return cudaErrorInvalidValue;
    const long long b = (L + kDT - 1) / kDT;
    k_dsa_update<<<(int)(b < 152 * 8 ? b : 152 * 8), kDT, 0, s>>>(e, Z, stride, m, y, L);
    return cudaGetLastError();
}

cudaError_t launch_dsa_gather(const DsaCells& d, const float* c, long long cells, float* out, cudaStream_t s) {
    k_dsa_gather<<<cell_blocks(d.n), kDT, 0, s>>>(d, c, cells, out);
    return cudaGetLastError();
}

cudaError_t launch_dsa_add64(const DsaCells& d, const float* e, double sign, long long cells, double* x,
                             cudaStream_t s) {
    k_dsa_add64<<<cell_blocks(d.n), kDT, 0, s>>>(d, e, sign, cells, x);
    return cudaGetLastError();
}

// ------------------------------------------------- vectors of one cycle's start
namespace {

// Products in FP64: these vectors are residuals in the caller's unit of concentration (any magnitude below 1e30), whose
// squares leave the f32 range.  A few calls per correction, 14 us at 2.8 M elements.
__global__ void __launch_bounds__(kDT) k_dot(const float* __restrict__ x, const float* __restrict__ y, long long L,
                                             double* __restrict__ part) {
    double acc[1] = {0.0};
    for (long long i = blockIdx.x * (long long)kDT + threadIdx.x; i < L; i += (long long)gridDim.x * kDT)
        acc[0] = fma((double)x[i], (double)y[i], acc[0]);
    block_sum_store<1>(acc, part + 2 * blockIdx.x);
}

// *out = sum of the partials (take_sqrt: its square root)
__global__ void __launch_bounds__(kDT) k_dot_fin(const double* __restrict__ part, int nblk, double* __restrict__ out,
                                                 int take_sqrt) {
    double acc[1] = {0.0};
    for (int b = threadIdx.x; b < nblk; b += blockDim.x) acc[0] += part[2 * b];
    __shared__ double tot[1];
    block_sum_store<1>(acc, tot);
    if (threadIdx.x == 0) *out = take_sqrt ? sqrt(tot[0]) : tot[0];
}

// y = x / nrm[0] (0 if the norm is 0)
__global__ void __launch_bounds__(kDT) k_scale_dev(float* __restrict__ y, const float* __restrict__ x,
                                                   const double* __restrict__ nrm, long long L) {
    const double n = nrm[0];
    const float s = n > 0.0 ? (float)(1.0 / n) : 0.f;
    for (long long i = blockIdx.x * (long long)kDT + threadIdx.x; i < L; i += (long long)gridDim.x * kDT)
        y[i] = s * x[i];
}

// out = a - b
__global__ void __launch_bounds__(kDT) k_sub(const float* __restrict__ a, const float* __restrict__ b,
                                             float* __restrict__ out, long long L) {
    for (long long i = blockIdx.x * (long long)kDT + threadIdx.x; i < L; i += (long long)gridDim.x * kDT)
        out[i] = a[i] - b[i];
}

}  // namespace

cudaError_t launch_dot_dev(const float* x, const float* y, long long L, int nblk, double* part, double* out,
                           int take_sqrt, cudaStream_t s) {
    k_dot<<<nblk, kDT, 0, s>>>(x, y, L, part);
    k_dot_fin<<<1, kDT, 0, s>>>(part, nblk, out, take_sqrt);
    return cudaGetLastError();
}

cudaError_t launch_scale_dev(float* y, const float* x, const double* nrm, long long L, int nblk, cudaStream_t s) {
    k_scale_dev<<<nblk, kDT, 0, s>>>(y, x, nrm, L);
    return cudaGetLastError();
}

cudaError_t launch_sub(const float* a, const float* b, float* out, long long L, int nblk, cudaStream_t s) {
    k_sub<<<nblk, kDT, 0, s>>>(a, b, out, L);
    return cudaGetLastError();
}

}  // namespace cl
