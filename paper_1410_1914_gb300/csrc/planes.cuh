// Per-plane sums along x, shared by the readouts of every storage.
//
// out[5 x + k] over the cells of plane x: sum of C, active cells, consumption
// on catalytic faces, inflow part (x = 0), outflow part (x = L).  With one
// block per plane every load took one cell from its own sector: 1.2 ms for a
// 256^3 layer, 4.5 ms for 400^3.  Here lanes are neighbouring planes, so rows are
// read as they lie, a block sums a share of the rows, and a second kernel
// adds the shares in order (the sums repeat bit by bit).
//
// FP64 issues at 1/64 of the FP32 rate, so the sums over a share's rows run in triples
// of floats (F3) that are added in FP64 once per kPlaneFlush rows.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include "device_util.cuh"

namespace cl {

constexpr int kPlaneFlush = 16;

struct PlaneAcc {
    double v[5];
    F3 c;  // running sum of C
    F3 r;  // of the consumption, before the sink's factor
    unsigned n;
};

// Op: load(x, row) reads what a cell needs, without a condition, so that kRows rows are in flight; use(item, acc)
// adds it.  inflow(row), outflow(row): the parts of the planes x = 0 and x = L, summed with one row per thread: as a
// condition among the rows their FP64 instructions were predicated off but issued in every one, and were the time of
// the kernel.  sink(): the factor of the consumption gathered in PlaneAcc::r.
template <class Op>
__global__ void __launch_bounds__(256) k_plane_part(Op op, int nx, int rows, int share, double* __restrict__ part) {
    __shared__ double sh[8][5][32];
    __shared__ double edge[2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int x = blockIdx.x * 32 + lane;
    const int r0 = blockIdx.y * share, r1 = min(rows, r0 + share);
    PlaneAcc a;
#pragma unroll
    for (int k = 0; k < 5; ++k) a.v[k] = 0.0;
    a.n = 0;
    const double sink = op.sink();
    constexpr int U = Op::kRows;
    static_assert(kPlaneFlush % U == 0, "whole groups of rows between flushes");
    for (int b = r0 + warp; b < r1; b += 8 * kPlaneFlush) {
        a.c = a.r = F3{0.f, 0.f, 0.f};
        if (x < nx)
            for (int g = 0; g < kPlaneFlush && b + 8 * g < r1; g += U) {
                typename Op::Item it[U];
#pragma unroll
                for (int u = 0; u < U; ++u) it[u] = op.load(x, min(b + 8 * (g + u), r1 - 1));
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (b + 8 * (g + u) < r1) op.use(it[u], a);
            }
        a.v[0] += f3_get(a.c);
        if (__any_sync(0xffffffffu, a.r.a != 0.f || a.r.b != 0.f)) a.v[2] += sink * f3_get(a.r);
    }
    a.v[1] += (double)a.n;
    if (threadIdx.x < 2) edge[threadIdx.x] = 0.0;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        if (blockIdx.x != (e == 0 ? 0 : gridDim.x - 1)) continue;
        double t = 0.0;
        for (int r = r0 + threadIdx.x; r < r1; r += 256) t += e == 0 ? op.inflow(r) : op.outflow(r);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) sh[warp][0][0] = t;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int w = 0; w < 8; ++w) s += sh[w][0][0];
            edge[e] = s;
        }
        __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) sh[warp][k][lane] = a.v[k];
    __syncthreads();
    if (warp < 5 && x < nx) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += sh[w][warp][lane];
        if (warp == 3 && x == 0) t += edge[0];
        if (warp == 4 && x == nx - 1) t += edge[1];
        part[((long long)blockIdx.y * nx + x) * 5 + warp] = t;
    }
}

static __global__ void __launch_bounds__(256) k_plane_sum(const double* __restrict__ part, int n5, int shares,
                                                          double* __restrict__ out) {
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= n5) return;
    double t = 0.0;
    for (int s = 0; s < shares; ++s) t += part[(long long)s * n5 + i];
    out[i] = t;
}

// shares of the rows: one wave of blocks, at least 64 rows each
inline int plane_shares(int nx, long long rows) {
    const int xb = (nx + 31) / 32;
    const long long want = (152 * 4) / xb, most = (rows + 63) / 64;
    const long long k = want < most ? want : most;
    return (int)(k < 1 ? 1 : k);
}
// doubles of `out` and the shares' partials behind it
inline long long plane_doubles(int nx, long long rows) { return 5LL * nx * (1 + plane_shares(nx, rows)); }

template <class Op>
cudaError_t launch_planes(const Op& op, int nx, long long rows, double* out, cudaStream_t s) {
    const int most = plane_shares(nx, rows);
    const int share = (int)((rows + most - 1) / most);
    const int shares = (int)((rows + share - 1) / share);
    double* part = out + 5LL * nx;
    k_plane_part<Op><<<dim3((nx + 31) / 32, shares), 256, 0, s>>>(op, nx, (int)rows, share, part);
    k_plane_sum<<<(5 * nx + 255) / 256, 256, 0, s>>>(part, 5 * nx, shares, out);
    return cudaGetLastError();
}

}  // namespace cl
