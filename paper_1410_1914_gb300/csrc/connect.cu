// Connected-phase labelling of Sec. 2.1.3 and its statistics on the GPU.
//
// The paper scans the box with a 13-neighbour label pass (the already
// scanned half of the 26-neighbourhood of Fig. 4a) and repeats scans in
// several directions until labels settle.  Here ccl.cu labels each portion by
// its smallest cell index; then atomics record per portion whether it reaches
// the end planes x = 0 and x = L and how many cells it has, and one more pass
// counts the statistics (whole numbers, summed in any order).
#include "cl_lbm.h"
#include "device_util.cuh"
#include "handle.cuh"
#include "internal.cuh"
#include "ccl.cuh"

namespace cl {

namespace {

__device__ __forceinline__ bool in_set(uint8_t p, unsigned set) { return p < 4 && ((set >> p) & 1u); }

// end planes reached by each portion: one thread per row
__global__ void k_cc_ends(int nx, long long rows, const int* __restrict__ L, unsigned* ends) {
    for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < rows;
         r += (long long)gridDim.x * blockDim.x)
        for (unsigned e = 1; e <= 2; ++e) {
            const int root = L[r * nx + (e == 1 ? 0 : nx - 1)];
            // most rows find the bit set by another of the same portion
            if (root >= 0 && !(*(volatile unsigned*)(ends + root) & e)) atomicOr(ends + root, e);
        }
}

// Cells per portion.  Most cells belong to one portion, whose counter every
// cell would add to (2 ms at 200^3): a warp walks consecutive cells and keeps
// the count of the portion it is in, adding it when another one takes over.
__global__ void __launch_bounds__(256) k_cc_tally(long long N, const int* __restrict__ L, int* size) {
    const int lane = threadIdx.x & 31;
    const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
    const long long per = ((N + warps - 1) / warps + 31) / 32 * 32;
    const long long w = blockIdx.x * (long long)(blockDim.x >> 5) + (threadIdx.x >> 5);
    const long long c0 = w * per, c1 = N < c0 + per ? N : c0 + per;
    int cur = -1, cnt = 0;
    for (long long b = c0; b < c1; b += 32) {
        const int r = b + lane < c1 ? L[b + lane] : -1;
        const unsigned all = __ballot_sync(0xffffffffu, r >= 0);
        if (all == 0) continue;
        const unsigned same = cur >= 0 ? __ballot_sync(0xffffffffu, r == cur) : 0u;
        unsigned rest = all & ~same;
        if (same == 0) {
            if (cur >= 0 && lane == 0) atomicAdd(size + cur, cnt);
            cur = __shfl_sync(0xffffffffu, r, __ffs(all) - 1);
            const unsigned g = __ballot_sync(0xffffffffu, r == cur);
            cnt = __popc(g);
            rest = all & ~g;
        } else {
            cnt += __popc(same);
        }
        while (rest) {
            const int o = __shfl_sync(0xffffffffu, r, __ffs(rest) - 1);
            const unsigned g = __ballot_sync(0xffffffffu, r == o);
            if (lane == 0) atomicAdd(size + o, __popc(g));
            rest &= ~g;
        }
    }
    if (cur >= 0 && lane == 0) atomicAdd(size + cur, cnt);
}

// v: cells, portions, transport portions, transport cells, surface faces, transport surface faces.  One warp per
// row of 32 cells, counted from bit masks.
__global__ void __launch_bounds__(256) k_cc_stats(const uint8_t* __restrict__ phase, int nx, int ny, int nz,
                                                  unsigned set, int periodic, const int* __restrict__ L,
                                                  const unsigned* __restrict__ ends, const int* __restrict__ size,
                                                  unsigned long long* total, int* largest) {
    const int lane = threadIdx.x & 31;
    const int nw = (nx + 31) >> 5;
    const long long words = (long long)nw * ny * nz;
    unsigned v[6] = {0, 0, 0, 0, 0, 0};  // lane 0's
    int big = 0;
    for (long long w = blockIdx.x * 8LL + (threadIdx.x >> 5); w < words; w += gridDim.x * 8LL) {
        const int row = (int)(w / nw), wx = (int)(w - (long long)row * nw);
        const int y = row % ny, z = row / ny;
        const int x = wx * 32 + lane, c = x + nx * row;
        const bool in = x < nx;
        const int r = in ? L[c] : -1;
        const unsigned m = __ballot_sync(0xffffffffu, r >= 0);
        if (m == 0) continue;
        const bool tr = r >= 0 && ends[r] == 3u;
        const unsigned t = __ballot_sync(0xffffffffu, tr);
        const unsigned root = __ballot_sync(0xffffffffu, r == c && r >= 0);
        if (r == c && r >= 0) big = max(big, size[c]);
        v[0] += __popc(m);
        v[1] += __popc(root);
        v[2] += __popc(root & t);
        v[3] += __popc(t);
        // faces toward in-box cells outside the set
        const uint8_t* pr = phase + (long long)nx * row;
        unsigned off = __ballot_sync(0xffffffffu, x + 1 < nx && !in_set(pr[x + 1 < nx ? x + 1 : 0], set));
        v[4] += __popc(m & off);
        v[5] += __popc(t & off);
        off = __ballot_sync(0xffffffffu, x > 0 && in && !in_set(pr[in && x > 0 ? x - 1 : 0], set));
        v[4] += __popc(m & off);
        v[5] += __popc(t & off);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            int yy = y + (k == 0) - (k == 1), zz = z + (k == 2) - (k == 3);
            if (periodic) {
                yy = yy < 0 ? yy + ny : (yy >= ny ? yy - ny : yy);
                zz = zz < 0 ? zz + nz : (zz >= nz ? zz - nz : zz);
            } else if (yy < 0 || yy >= ny || zz < 0 || zz >= nz) {
                continue;
            }
            off = __ballot_sync(0xffffffffu, in && !in_set(phase[(in ? x : 0) + (long long)nx * (yy + ny * zz)], set));
            v[4] += __popc(m & off);
            v[5] += __popc(t & off);
        }
    }
    for (int o = 16; o > 0; o >>= 1) big = max(big, __shfl_xor_sync(0xffffffffu, big, o));
    __shared__ unsigned long long sh[6];
    if (threadIdx.x < 6) sh[threadIdx.x] = 0;
    __syncthreads();
    if (lane == 0) {
        if (big > 0) atomicMax(largest, big);
#pragma unroll
        for (int k = 0; k < 6; ++k) atomicAdd(sh + k, (unsigned long long)v[k]);
    }
    __syncthreads();
    if (threadIdx.x < 6 && sh[threadIdx.x]) atomicAdd(total + threadIdx.x, sh[threadIdx.x]);
}

}  // namespace

}  // namespace cl

using namespace cl;

extern "C" cl_status cl_phase_connectivity(const uint8_t* phase, int nx, int ny, int nz, unsigned phase_set,
                                           int neighbours, int periodic_yz, int32_t* labels, cl_phase_stats* out,
                                           int ptr_is_device, void* cuda_stream) {
    if (!phase || !out) { set_msg_txt("NULL argument"); return CL_ERR_ARG; }
    const long long N = (long long)nx * ny * nz;
    if (nx < 1 || ny < 1 || nz < 1 || N >= (1LL << 31)) { set_msg_txt("box size out of range"); return CL_ERR_ARG; }
    if (neighbours != 6 && neighbours != 26) { set_msg_txt("neighbours must be 6 or 26"); return CL_ERR_ARG; }
    if (phase_set == 0 || phase_set > 15) { set_msg_txt("phase_set must name codes 0..3"); return CL_ERR_ARG; }
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const int grid = 152 * 8, block = 256;
    // scratch: labels, ends, sizes (4 B each per cell), results [phase copy]
    const size_t cells4 = (sizeof(int) * (size_t)N + 255) / 256 * 256;  // keeps every region 256-byte aligned
    const size_t scratch = 3 * cells4 + 256 + (ptr_is_device ? 0 : (size_t)N);
    unsigned char* base = nullptr;
    CK(cudaMallocAsync((void**)&base, scratch, s));
    int* L = (int*)base;
    unsigned* ends = (unsigned*)(base + cells4);
    int* size = (int*)(base + 2 * cells4);
    unsigned long long* tot = (unsigned long long*)(base + 3 * cells4);
    int* ints = (int*)(tot + 8);  // [0] largest, [1] error bits
    const uint8_t* ph = phase;
    if (!ptr_is_device) {
        uint8_t* pcopy = base + 3 * cells4 + 256;
        cudaError_t e = cudaMemcpyAsync(pcopy, phase, (size_t)N, cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) { cudaFreeAsync(base, s); set_msg("phase upload", e); return from_cuda(e); }
        ph = pcopy;
    }
    const long long rows = (long long)ny * nz;
    const int rgrid = (int)(rows < (long long)grid * block ? (rows + block - 1) / block : grid);
    // ends and sizes are next to each other, the results behind them
    cudaError_t e = cudaMemsetAsync(base + cells4, 0, 2 * cells4 + 256, s);
    if (e == cudaSuccess) e = launch_validate(ph, N, ints + 1, s);
    if (e == cudaSuccess)
        e = launch_ccl(ph, nx, ny, nz, phase_set, neighbours == 6, periodic_yz != 0, L, ints + 1, s);
    if (e == cudaSuccess) {
        k_cc_ends<<<rgrid, block, 0, s>>>(nx, rows, L, ends);
        k_cc_tally<<<grid, block, 0, s>>>(N, L, size);
        k_cc_stats<<<grid, block, 0, s>>>(ph, nx, ny, nz, phase_set, periodic_yz != 0, L, ends, size, tot, ints);
        e = cudaGetLastError();
    }
    unsigned long long res[6];
    int hi[2] = {0, 0};
    if (e == cudaSuccess) e = cudaMemcpyAsync(res, tot, sizeof(res), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(hi, ints, sizeof(hi), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && labels)
        e = cudaMemcpyAsync(labels, L, sizeof(int) * (size_t)N,
                            ptr_is_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(base, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) { set_msg("cl_phase_connectivity", e); return from_cuda(e); }
    if (hi[1] & 1) { set_msg_txt("phase code outside 0..3"); return CL_ERR_ARG; }
    if (hi[1] & 2) { set_msg_txt("connectivity labelling exceeded its iteration bound"); return CL_ERR_TIMEOUT; }
    out->n_cells = (long long)res[0];
    out->n_portions = (long long)res[1];
    out->n_transport_portions = (long long)res[2];
    out->n_transport_cells = (long long)res[3];
    out->surface_faces = (long long)res[4];
    out->transport_surface_faces = (long long)res[5];
    out->largest_portion = hi[0];
    return CL_OK;
}
