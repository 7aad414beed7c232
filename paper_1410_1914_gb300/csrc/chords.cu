// Pore lengths of Sec. 2.1.3 and diffusivities (Eq. 7-9) from bit masks.
//
// The length of a pore cell in a direction is the run of pore cells through
// it.  Read line by line (k_chord_xlines_warp, k_chord_loops_warp), every
// direction gathers one byte and updates one double per cell at addresses a
// row or a plane apart: 0.23 ms a direction at 256^3, 3.0 ms for the 13.
// Here the pore cells are bits, 32 cells of a row to a word (2 MB at 256^3),
// and a thread counts the runs of 32 cells at once: it walks away from its
// word one cell at a time, forward and backward, and ANDs the word found
// there (two neighbouring words funnel-shifted, for directions with an x
// component) into the cells still `alive`.  All alive cells have the same
// count, the step number, so the counts are kept as bit planes and a step
// flips, for the alive cells, the planes in which the step number changes:
// two on average.  The sums over the axis, face-diagonal and body-diagonal
// directions are bit planes too; whole numbers, so their order is free.
//
// Long runs (a reservoir plane, an open box) are crossed 16 cells at a time
// where the words of a second set, the AND of 16 cells along the direction,
// say that every alive cell of the warp goes on that far.
//
// Runs stay below 2^11 by the caller's rule (the line kernels' own bound), so
// that 14 planes hold the sum of six of them.
//
// Every row of words ends with an empty word, and one stands before the
// first: a cell still alive was a pore inside the row one step ago, so it and
// the word beside it lie between those.  A thread with no cell alive reads
// whatever lies there (kPad words stand on either side of the sets) and
// ANDs it into nothing, so that no load waits for the one before it.
//
// Measured at 256^3 (porosity 0.45): 0.04 + 0.10 + 1.5 ms for the three
// kernels, D included (its FP64 arithmetic took 0.8 ms by itself).  What is
// left is instruction issue: a warp walks on until the last of its 1024 cells
// has met a wall, 27 steps a way on average where a run is 8.
#include "chords.cuh"
#include "device_util.cuh"

#include <math.h>

namespace cl {

namespace {

constexpr int kPl = 14;    // planes of a sum
constexpr int kCPl = 12;   // planes of a run
constexpr int kBT = 128;   // threads per block of the counting kernel
constexpr int kPad = 80;   // words before and after the sets: 2^11 cells and a word or two

__constant__ int c_dir[13][3] = {{1, 0, 0},  {0, 1, 0},  {0, 0, 1},  {1, 1, 0},  {1, -1, 0},
                                 {1, 0, 1},  {1, 0, -1}, {0, 1, 1},  {0, 1, -1}, {1, 1, 1},
                                 {1, 1, -1}, {1, -1, 1}, {1, -1, -1}};

struct Box {
    int nx, ny, nz, nw, pitch;  // nw: words per row; pitch: nw + 1
    unsigned words, span;       // words: nw per row; span: elements of a set
};

// word index -> row and word of the row; element of a set
struct Word {
    unsigned row;
    int wx;
    __device__ __forceinline__ Word(const Box& b, unsigned w) : row(w / b.nw), wx((int)(w - row * b.nw)) {}
    __device__ __forceinline__ unsigned at(const Box& b) const { return 1u + row * b.pitch + wx; }
};

__global__ void __launch_bounds__(256) k_pore_bits(const uint8_t* __restrict__ phase, Box b, uint32_t* __restrict__ B) {
    const int lane = threadIdx.x & 31;
    for (unsigned w = blockIdx.x * 8u + (threadIdx.x >> 5); w < b.words; w += gridDim.x * 8u) {
        const Word q(b, w);
        const int x = q.wx * 32 + lane;
        uint8_t p = 1;
        if (x < b.nx) p = phase[x + (long long)b.nx * q.row];
        const uint32_t m = __ballot_sync(0xffffffffu, p == 0 || p == 3);
        if (lane == 0) {
            B[q.at(b)] = m;
            if (q.wx == b.nw - 1) B[q.at(b) + 1] = 0;
            if (w == 0) B[0] = 0;
        }
    }
}

__device__ __forceinline__ int far_wrap(int a, int by, int n) {
    const int t = (a + by) % n;
    return t < 0 ? t + n : t;
}

// A walk from a word along (sx, sy, sz): EX, EY, EZ say which of them are not 0.  Every step adds one offset to the
// row; where y or z leaves the box (a countdown) the row jumps back.
template <int EX, int EY, int EZ>
struct Walk {
    int sx, sy, sz;
    int at;        // steps from the word
    unsigned row;  // element of the word at shift 0 of the row now reached
    int delta, cy, cz;
    __device__ __forceinline__ void place(const Box& b, int wx, int y, int z) {
        row = 1u + (unsigned)(y + b.ny * z) * b.pitch + wx;
        cy = sy > 0 ? b.ny - y : y + 1;
        cz = sz > 0 ? b.nz - z : z + 1;
    }
    __device__ __forceinline__ Walk(const Box& b, int sx_, int sy_, int sz_, int wx, int y, int z)
        : sx(sx_), sy(sy_), sz(sz_), at(0) {
        delta = b.pitch * ((EY ? sy : 0) + (EZ ? sz * b.ny : 0));
        place(b, wx, y, z);
    }
    __device__ __forceinline__ int y(const Box& b) const { return sy > 0 ? b.ny - cy : cy - 1; }
    __device__ __forceinline__ int z(const Box& b) const { return sz > 0 ? b.nz - cz : cz - 1; }
    __device__ __forceinline__ void step(const Box& b) {
        row += delta;
        ++at;
        if (EY && --cy == 0) {
            row -= sy * b.ny * b.pitch;
            cy = b.ny;
        }
        if (EZ && --cz == 0) {
            row -= sz * b.nz * b.ny * b.pitch;
            cz = b.nz;
        }
    }
    // the 32 cells `at` steps from the word's
    __device__ __forceinline__ uint32_t bits(const uint32_t* __restrict__ S, unsigned r, int s) const {
        if (!EX) return S[r];
        const uint32_t* p = S + (int)(r + (s >> 5));
        return __funnelshift_r(p[0], p[1], s & 31);
    }
    __device__ __forceinline__ uint32_t here(const uint32_t* __restrict__ S) const {
        return bits(S, row, EX ? sx * at : 0);
    }
};

// A[d]: cells from which 16 cells on end along direction d are pores
__global__ void __launch_bounds__(256) k_pore_ahead(const uint32_t* __restrict__ B, Box b, uint32_t* __restrict__ A) {
    const int d = blockIdx.y;
    uint32_t* __restrict__ Ad = A + (size_t)d * b.span;
    for (unsigned w = blockIdx.x * 256u + threadIdx.x; w < b.words; w += gridDim.x * 256u) {
        const Word q(b, w);
        const int y = (int)(q.row % b.ny), z = (int)(q.row / b.ny);
        uint32_t acc = B[q.at(b)];
        Walk<1, 1, 1> k(b, c_dir[d][0], c_dir[d][1], c_dir[d][2], q.wx, y, z);
        // a component of 0 never reaches its end
        if (c_dir[d][1] == 0) k.cy = 1 << 30;
        if (c_dir[d][2] == 0) k.cz = 1 << 30;
        for (int n = 1; n < 16 && acc; ++n) {
            k.step(b);
            acc &= k.here(B);
        }
        Ad[q.at(b)] = acc;
        if (q.wx == b.nw - 1) Ad[q.at(b) + 1] = 0;
        if (w == 0) Ad[0] = 0;
    }
}

// S += C, as numbers held in bit planes
__device__ __forceinline__ void add_planes(uint32_t (&S)[kPl], const uint32_t (&C)[kCPl]) {
    uint32_t carry = 0;
#pragma unroll
    for (int p = 0; p < kCPl; ++p) {
        const uint32_t t = S[p] ^ C[p];
        const uint32_t c = (S[p] & C[p]) | (carry & t);
        S[p] = t ^ carry;
        carry = c;
    }
#pragma unroll
    for (int p = kCPl; p < kPl; ++p) {
        const uint32_t c = S[p] & carry;
        S[p] ^= carry;
        carry = c;
    }
}

// Counts of consecutive pore cells away from the word's cells: `alive` in, and out those that reached `limit`
// (AHEAD; a loop's length).  AHEAD: the cell itself counts (step 0 is its own); else only the cells behind it.
template <int EX, int EY, int EZ, bool AHEAD>
__device__ __forceinline__ uint32_t count_runs(const uint32_t* __restrict__ B, const uint32_t* __restrict__ A,
                                               const Box& b, int ey, int ez, int wx, int y, int z, uint32_t alive,
                                               int limit, uint32_t (&C)[kCPl]) {
    constexpr int sgn = AHEAD ? 1 : -1;
    constexpr bool kLimit = AHEAD && !EX;  // runs along x end by themselves
#pragma unroll
    for (int p = 0; p < kCPl; ++p) C[p] = 0;
    Walk<EX, EY, EZ> w(b, sgn * EX, sgn * ey, sgn * ez, wx, y, z);
    int k = 0;  // cells counted so far
    if (!AHEAD) {
        w.step(b);
        alive &= w.here(B);
    }
    while ((!kLimit || k < limit) && __any_sync(0xffffffffu, alive != 0)) {
        if (k >= 16 && (k & 15) == 0 && (!kLimit || k + 16 <= limit)) {
            // cells at .. at + 15 steps away, seen from the end the set was built from
            constexpr int from = AHEAD ? 0 : 15;
            const int yy = EY ? far_wrap(w.y(b), from * w.sy, b.ny) : y, zz = EZ ? far_wrap(w.z(b), from * w.sz, b.nz) : z;
            const uint32_t a16 = w.bits(A, 1u + (unsigned)(yy + b.ny * zz) * b.pitch + wx, EX * sgn * (w.at + from));
            if (__all_sync(0xffffffffu, (alive & ~a16) == 0)) {
                const int t = k ^ (k + 16);
#pragma unroll
                for (int p = 4; p < kCPl; ++p)
                    if ((t >> p) & 1) C[p] ^= alive;
                k += 16;
                w.at += 16;
                w.place(b, wx, EY ? far_wrap(w.y(b), 16 * w.sy, b.ny) : y, EZ ? far_wrap(w.z(b), 16 * w.sz, b.nz) : z);
                alive &= w.here(B);
                continue;
            }
        }
        // eight steps from a multiple of eight: the low three planes flip in a fixed pattern
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (kLimit && k + u >= limit) break;
            C[0] ^= alive;
            if (u & 1) C[1] ^= alive;
            if ((u & 3) == 3) C[2] ^= alive;
            if (u == 7) {
                const int t = (k >> 3) ^ ((k >> 3) + 1);
#pragma unroll
                for (int p = 3; p < kCPl; ++p)
                    if ((t >> (p - 3)) & 1) C[p] ^= alive;
            }
            w.step(b);
            alive &= w.here(B);
        }
        k += 8;
    }
    return alive;
}

// adds both ways of one direction to S; loop: the length of the direction's loops (no x component)
template <int EX, int EY, int EZ>
__device__ __forceinline__ void add_dir(const uint32_t* __restrict__ B, const uint32_t* __restrict__ A, const Box& b,
                                        int d, int loop, int wx, int y, int z, uint32_t pore, uint32_t (&S)[kPl]) {
    const int ey = EY ? c_dir[d][1] : 0, ez = EZ ? c_dir[d][2] : 0;
    const uint32_t* Ad = A + (size_t)d * b.span;
    uint32_t C[kCPl];
    // a loop of pores counts its cells once
    const uint32_t full = count_runs<EX, EY, EZ, true>(B, Ad, b, ey, ez, wx, y, z, pore, loop, C) & (EX ? 0u : ~0u);
    add_planes(S, C);
    count_runs<EX, EY, EZ, false>(B, Ad, b, ey, ez, wx, y, z, pore & ~full, 0, C);
    add_planes(S, C);
}

// D of every cell, and the whole-number sums over the pore cells: tot[0..2] axis, face- and body-diagonal runs,
// tot[3] pore cells
// The FP64 arithmetic of D is done for 32 active pore cells at a time, gathered over the warp's words: FP64 issues at
// 1/64 of the FP32 rate, for idle lanes too.
__global__ void __launch_bounds__(kBT) k_chord_bits(const uint32_t* __restrict__ B, const uint32_t* __restrict__ A,
                                                    const uint8_t* __restrict__ phase,
                                                    const uint8_t* __restrict__ active, Box b, int3 loops, double len1,
                                                    double len2, double len3, double D_b, double D_ion, int knudsen,
                                                    double* __restrict__ D, unsigned long long* __restrict__ tot) {
    __shared__ uint32_t pl[kBT / 32][3 * kPl][32];
    __shared__ unsigned short qs[kBT / 32][3][64];  // gathered cells: run sums
    __shared__ int qc[kBT / 32][64];                // and indices
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long sum[4] = {0, 0, 0, 0};
    const unsigned w0 = blockIdx.x * kBT + warp * 32;
    if (w0 < b.words) {
        const Word wd(b, w0 + lane < b.words ? w0 + lane : b.words - 1);
        const unsigned row = wd.row;
        const int wx = wd.wx, y = (int)(row % b.ny), z = (int)(row / b.ny);
        const uint32_t pore = w0 + lane < b.words ? B[wd.at(b)] : 0u;
        unsigned any[3];
#pragma unroll
        for (int g = 0; g < 3; ++g) {
            uint32_t S[kPl];
#pragma unroll
            for (int p = 0; p < kPl; ++p) S[p] = 0;
            if (g == 0) {
                add_dir<1, 0, 0>(B, A, b, 0, 0, wx, y, z, pore, S);
                add_dir<0, 1, 0>(B, A, b, 1, loops.x, wx, y, z, pore, S);
                add_dir<0, 0, 1>(B, A, b, 2, loops.y, wx, y, z, pore, S);
            } else if (g == 1) {
                for (int d = 3; d < 5; ++d) add_dir<1, 1, 0>(B, A, b, d, 0, wx, y, z, pore, S);
                for (int d = 5; d < 7; ++d) add_dir<1, 0, 1>(B, A, b, d, 0, wx, y, z, pore, S);
                for (int d = 7; d < 9; ++d) add_dir<0, 1, 1>(B, A, b, d, loops.z, wx, y, z, pore, S);
            } else {
                for (int d = 9; d < 13; ++d) add_dir<1, 1, 1>(B, A, b, d, 0, wx, y, z, pore, S);
            }
            unsigned top = 0;
#pragma unroll
            for (int p = 0; p < kPl; ++p) {
                pl[warp][g * kPl + p][lane] = S[p];
                if (S[p]) top = p + 1;
            }
            any[g] = __reduce_max_sync(0xffffffffu, top);
        }
        __syncwarp();
        int queued = 0;
        auto flush = [&](int n) {  // D of the first n gathered cells
            __syncwarp();
            if (lane < n) {
                // s = d_p (Sec. 2.1.3) times vkn / 3 / D_b is D_kn / D_b (Eq. 8); Eq. 9 as D_b s / (1 + s)
                const double s = fma(len3, (double)qs[warp][2][lane],
                                     fma(len2, (double)qs[warp][1][lane], len1 * (double)qs[warp][0][lane]));
                D[qc[warp][lane]] = s * D_b * recip(1.0 + s);
            }
            __syncwarp();
        };
        // lane = cell, one word after the other
        for (int j = 0; j < 32 && w0 + j < b.words; ++j) {
            const unsigned rj = __shfl_sync(0xffffffffu, row, j);
            const int x = __shfl_sync(0xffffffffu, wx, j) * 32 + lane;
            const uint32_t pj = __shfl_sync(0xffffffffu, pore, j);
            unsigned s[3] = {0, 0, 0};
            if (pj) {
#pragma unroll
                for (int g = 0; g < 3; ++g)
                    for (unsigned p = 0; p < any[g]; ++p) s[g] |= ((pl[warp][g * kPl + p][j] >> lane) & 1u) << p;
            }
            const bool in = x < b.nx;
            const int c = x + (int)((long long)b.nx * rj);  // N < 2^31
            const bool is_pore = (pj >> lane) & 1u;
            const bool act = in && active[c];
            const bool work = act && is_pore && knudsen;
            if (in && !work) D[c] = act ? (is_pore ? D_b : D_ion) : 0.0;
            if (is_pore) {
                sum[0] += s[0];
                sum[1] += s[1];
                sum[2] += s[2];
                sum[3] += 1;
            }
            const unsigned m = __ballot_sync(0xffffffffu, work);
            if (work) {
                const int at = queued + __popc(m & ((1u << lane) - 1u));
#pragma unroll
                for (int g = 0; g < 3; ++g) qs[warp][g][at] = (unsigned short)s[g];
                qc[warp][at] = c;
            }
            queued += __popc(m);
            if (queued >= 32) {
                flush(32);
                queued -= 32;
                if (lane < queued) {  // the rest moves to the front
#pragma unroll
                    for (int g = 0; g < 3; ++g) qs[warp][g][lane] = qs[warp][g][32 + lane];
                    qc[warp][lane] = qc[warp][32 + lane];
                }
                __syncwarp();
            }
        }
        flush(queued);
    }
    __shared__ unsigned long long sh[4];
    if (threadIdx.x < 4) sh[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        for (int o = 16; o > 0; o >>= 1) sum[k] += __shfl_xor_sync(0xffffffffu, sum[k], o);
        if (lane == 0 && sum[k]) atomicAdd(sh + k, sum[k]);
    }
    __syncthreads();
    if (threadIdx.x < 4 && sh[threadIdx.x]) atomicAdd(tot + threadIdx.x, sh[threadIdx.x]);
}

long long gcd_ll(long long a, long long b) {
    while (b) { const long long t = a % b; a = b; b = t; }
    return a;
}

}  // namespace

bool chord_bits_fit(int nx, int ny, int nz, int most, double dx, double vkn, double D_b) {
    // D_kn / D_b of a run of one cell; it is divided through its f32 reciprocal
    const double unit = dx / 39.0 * vkn / D_b;
    if (!(unit > 1e-25 && unit < 1e25)) return false;
    const int nw = (nx + 31) / 32;
    const long long lcm = (long long)ny / gcd_ll(ny, nz) * nz;
    // the bit set and 13 sets of 16 cells ahead, an empty word before each, in one double per cell of scratch
    const long long span = (nw + 1LL) * ny * nz + 1, N = (long long)nx * ny * nz;
    return 14 * span + 2 * kPad <= 2 * N && nx <= most && lcm <= most;
}

cudaError_t launch_chord_bits(const uint8_t* phase, const uint8_t* active, int nx, int ny, int nz, double dx,
                              double vkn, double D_b, double D_ion, int knudsen, double* scratch, double* D,
                              unsigned long long* tot, cudaStream_t s) {
    Box b;
    b.nx = nx; b.ny = ny; b.nz = nz;
    b.nw = (nx + 31) / 32;
    b.pitch = b.nw + 1;
    b.words = (unsigned)((long long)b.nw * ny * nz);
    b.span = 1u + (unsigned)((long long)b.pitch * ny * nz);
    uint32_t* B = (uint32_t*)scratch + kPad;
    uint32_t* A = B + b.span;
    cudaError_t e = cudaMemsetAsync(tot, 0, 4 * sizeof(*tot), s);
    if (e != cudaSuccess) return e;
    const auto blocks = [](long long n, int per, int most) {
        const long long k = (n + per - 1) / per;
        return (unsigned)(k < most ? k : most);
    };
    k_pore_bits<<<blocks(b.words, 8, 152 * 16), 256, 0, s>>>(phase, b, B);
    k_pore_ahead<<<dim3(blocks(b.words, 256, 152 * 8), 13), 256, 0, s>>>(B, b, A);
    const int3 loops = make_int3(ny, nz, (int)((long long)ny / gcd_ll(ny, nz) * nz));
    // D_kn / D_b = (s1 + sqrt2 s2 + sqrt3 s3) dx / 13 / 3 vkn / D_b
    const double unit = dx / 13.0 / 3.0 * vkn / D_b;
    k_chord_bits<<<blocks(b.words, kBT, 1 << 30), kBT, 0, s>>>(B, A, phase, active, b, loops, unit, sqrt(2.0) * unit,
                                                               sqrt(3.0) * unit, D_b, D_ion, knudsen, D, tot);
    return cudaGetLastError();
}

}  // namespace cl
