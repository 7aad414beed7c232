// Connected-component labelling by tiles.
//
// One union per neighbouring pair of cells through global memory was the
// whole time of the labelling (a 200^3 layer: 7 ms for 26 neighbours; 256^3:
// 3.6 ms for 6): millions of finds through long parent chains, most of them
// for pairs already united.  Instead
//   1. a block labels a tile of 32 x 8 x 8 cells in shared memory.  A warp
//      reads a row of 32 cells as one bit mask; the nodes are the runs of set
//      cells, and two rows unite only where their runs first touch;
//   2. the pairs that cross a tile's faces are united in global memory, again
//      only where two runs first touch;
//   3. every cell takes its root.
// Measured: 26 neighbours at 200^3 0.19 + 0.24 + 0.10 ms for the three steps
// (from 7.1 ms), 6 neighbours at 256^3 0.18 + 0.27 + 0.19 ms (from 3.8 ms).
// Roots are only ever linked to smaller indices (uf.cuh), and a tile's local
// order is the order of the cell indices, so the final root of a component is
// its smallest cell index.
#include "ccl.cuh"
#include "uf.cuh"

namespace cl {

namespace {

constexpr int kTY = 8, kTZ = 8, kRows = kTY * kTZ;
constexpr int kCT = 256;

__device__ __forceinline__ bool in_set(uint8_t p, unsigned set) { return p < 4 && ((set >> p) & 1u); }

// first cell of lane's run in the row mask m (bit lane set)
__device__ __forceinline__ int run_start(unsigned m, int lane) {
    const unsigned below = ~m & ((1u << lane) - 1u);
    return 32 - __clz(below);
}

// Where the runs of row r first touch those of row q: the lanes of r to unite
// with q's cell at the lane itself, at lane - 1 and at lane + 1.  rp, qp: the
// rows' bits at lane - 1 (bit l of rp = cell l - 1 of r), rn, qn at lane + 1.
__device__ __forceinline__ void touch(unsigned r, unsigned rp, unsigned rn, unsigned q, unsigned qp, unsigned qn,
                                      bool diagonal, unsigned& same, unsigned& left, unsigned& right) {
    same = r & q & ~(rp & qp);
    left = diagonal ? r & ~q & qp & ~rp : 0u;
    right = diagonal ? r & ~q & qn & ~rn : 0u;
}

// (dy, dz) of the rows of the earlier half of the neighbourhood: faces (-1, 0), (0, -1); then edges (-1, -1), (1, -1)
__device__ __forceinline__ int row_dy(int k) { return k == 0 ? -1 : (k == 1 ? 0 : (k == 2 ? -1 : 1)); }
__device__ __forceinline__ int row_dz(int k) { return k == 0 ? 0 : -1; }

__global__ void __launch_bounds__(kCT) k_ccl_tiles(const uint8_t* __restrict__ phase, int nx, int ny, int nz,
                                                   unsigned set, int faces_only, int nw, int ty,
                                                   int* __restrict__ L, int* err) {
    __shared__ unsigned mask[kRows];
    __shared__ int lab[kRows * 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int wx = (int)(blockIdx.x % (unsigned)nw), t = (int)(blockIdx.x / (unsigned)nw);
    const int x = wx * 32 + lane;
    const int y0 = (t % ty) * kTY, z0 = (t / ty) * kTZ;
    for (int r = warp; r < kRows; r += kCT / 32) {
        const int y = y0 + r % kTY, z = z0 + r / kTY;
        bool on = false;
        if (x < nx && y < ny && z < nz) on = in_set(phase[x + (long long)nx * (y + (long long)ny * z)], set);
        const unsigned m = __ballot_sync(0xffffffffu, on);
        if (lane == 0) mask[r] = m;
        lab[r * 32 + lane] = on ? r * 32 + run_start(m, lane) : -1;
    }
    __syncthreads();
    const int nrow = faces_only ? 2 : 4;
    for (int r = warp; r < kRows; r += kCT / 32) {
        const unsigned m = mask[r];
        if (m == 0) continue;
        for (int k = 0; k < nrow; ++k) {
            const int yy = r % kTY + row_dy(k), zz = r / kTY + row_dz(k);
            if (yy < 0 || yy >= kTY || zz < 0) continue;
            const int qr = yy + kTY * zz;
            const unsigned q = mask[qr];
            unsigned same, left, right;
            touch(m, m << 1, m >> 1, q, q << 1, q >> 1, !faces_only, same, left, right);
            const unsigned bit = 1u << lane;
            // the nodes are the first cells of the runs
            if (same & bit) uf_union(lab, r * 32 + run_start(m, lane), qr * 32 + run_start(q, lane), err);
            if (left & bit) uf_union(lab, r * 32 + run_start(m, lane), qr * 32 + run_start(q, lane - 1), err);
            if (right & bit) uf_union(lab, r * 32 + run_start(m, lane), qr * 32 + lane + 1, err);
        }
    }
    __syncthreads();
    for (int r = warp; r < kRows; r += kCT / 32) {
        const int y = y0 + r % kTY, z = z0 + r / kTY;
        if (x >= nx || y >= ny || z >= nz) continue;
        int out = -1;
        if ((mask[r] >> lane) & 1u) {
            const int root = uf_find(lab, r * 32 + run_start(mask[r], lane), err);
            const int rr = root >> 5;
            out = wx * 32 + (root & 31) + nx * ((y0 + rr % kTY) + ny * (z0 + rr / kTY));
        }
        L[x + (long long)nx * (y + (long long)ny * z)] = out;
    }
}

// One warp per row of 32 cells: the pairs with cells of other tiles.
__global__ void __launch_bounds__(kCT) k_ccl_seams(const uint8_t* __restrict__ phase, int nx, int ny, int nz,
                                                   unsigned set, int faces_only, int periodic, int* L, int* err) {
    const int lane = threadIdx.x & 31;
    const int nw = (nx + 31) >> 5;
    const long long total = (long long)nw * ny * nz;
    const int nrow = faces_only ? 2 : 4;
    for (long long w = blockIdx.x * (long long)(kCT / 32) + (threadIdx.x >> 5); w < total;
         w += (long long)gridDim.x * (kCT / 32)) {
        const int row = (int)(w / nw), wx = (int)(w - (long long)row * nw);
        const int y = row % ny, z = row / ny;
        const int x = wx * 32 + lane;
        const uint8_t* pr = phase + (long long)nx * row;
        const unsigned m = __ballot_sync(0xffffffffu, x < nx && in_set(pr[x], set));
        if (m == 0) continue;
        // the cells just left and right of these 32 (every lane reads both)
        const bool ml = wx > 0 && in_set(pr[wx * 32 - 1], set);
        const bool mr = wx * 32 + 32 < nx && in_set(pr[wx * 32 + 32], set);
        const unsigned bit = 1u << lane;
        const int c = x + nx * row;
        if (lane == 0 && (m & 1u) && ml) uf_union(L, c, c - 1, err);
        for (int k = 0; k < nrow; ++k) {
            const int dy = row_dy(k), dz = row_dz(k);
            int yy = y + dy, zz = z + dz;
            // inside the tile: only what crosses its x faces is left
            const bool inside = (unsigned)(y % kTY + dy) < (unsigned)kTY && z % kTZ + dz >= 0 && yy < ny;
            if (periodic) {
                yy = yy < 0 ? yy + ny : (yy >= ny ? yy - ny : yy);
                zz = zz < 0 ? zz + nz : zz;
            } else if (yy < 0 || yy >= ny || zz < 0) {
                continue;
            }
            const int qrow = yy + ny * zz;
            const uint8_t* pq = phase + (long long)nx * qrow;
            if (inside) {
                if (faces_only) continue;
                // lane 0 with q's cell at -1, lane 31 with q's cell at 32
                const int cq = wx * 32 + nx * qrow;
                if (lane == 0 && (m & 1u) && wx > 0 && !ml && in_set(pq[wx * 32 - 1], set) &&
                    !in_set(pq[wx * 32], set))
                    uf_union(L, c, cq - 1, err);
                if (lane == 31 && (m >> 31) && wx * 32 + 32 < nx && !mr && in_set(pq[wx * 32 + 32], set) &&
                    !in_set(pq[wx * 32 + 31], set))
                    uf_union(L, c, cq + 32, err);
                continue;
            }
            const unsigned q = __ballot_sync(0xffffffffu, x < nx && in_set(pq[x], set));
            const bool ql = wx > 0 && in_set(pq[wx * 32 - 1], set);
            const bool qh = wx * 32 + 32 < nx && in_set(pq[wx * 32 + 32], set);
            unsigned same, left, right;
            touch(m, (m << 1) | (ml ? 1u : 0u), (m >> 1) | (mr ? 0x80000000u : 0u), q, (q << 1) | (ql ? 1u : 0u),
                  (q >> 1) | (qh ? 0x80000000u : 0u), !faces_only, same, left, right);
            const int cq = x + nx * qrow;
            if (same & bit) uf_union(L, c, cq, err);
            if (left & bit) uf_union(L, c, cq - 1, err);
            if (right & bit) uf_union(L, c, cq + 1, err);
        }
    }
}

__global__ void __launch_bounds__(kCT) k_ccl_roots(long long N, int* L, int* err) {
    for (long long c = blockIdx.x * (long long)kCT + threadIdx.x; c < N; c += (long long)gridDim.x * kCT)
        if (L[c] >= 0) L[c] = uf_find(L, (int)c, err);
}

}  // namespace

cudaError_t launch_ccl(const uint8_t* phase, int nx, int ny, int nz, unsigned set, bool faces_only, bool periodic,
                       int* L, int* err, cudaStream_t s) {
    const long long N = (long long)nx * ny * nz;
    const int ty = (ny + kTY - 1) / kTY, tz = (nz + kTZ - 1) / kTZ, nw = (nx + 31) / 32;
    const int g = 152 * 16;
    const long long tiles = (long long)nw * ty * tz;  // at most N
    k_ccl_tiles<<<(unsigned)tiles, kCT, 0, s>>>(phase, nx, ny, nz, set, faces_only, nw, ty, L, err);
    k_ccl_seams<<<g, kCT, 0, s>>>(phase, nx, ny, nz, set, faces_only, periodic, L, err);
    k_ccl_roots<<<g, kCT, 0, s>>>(N, L, err);
    return cudaGetLastError();
}

}  // namespace cl
