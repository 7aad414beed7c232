// Structure generation on the GPU: the quartet structure generation set
// (QSGS) growth of Sec. 2.1.2, the solid-not-touching-ionomer region of the
// micropore step (Sec. 5.3) and the reactive-face sampling of the Pt layer.
// Input generation only (none of the solver's arithmetic); the results are
// bit-identical to the host generator of the inputs module, so that either
// can feed the solver and the oracle.
//
// Random numbers: SplitMix64 (Steele, Lea and Flood, OOPSLA 2014) folded over
// (seed, stream, a, b); a uniform double in [0, 1) is the top 53 bits times
// 2^-53.  Growth (Sec. 2.1.2.1): seeds placed once with probability c_d, then
// synchronous sweeps over the state at the start of the sweep.  A cell that
// may convert and has grown 6-neighbours (x, y and z wrap) is accepted with
// two or more of them (rule 2a), else with probability p_alpha (rule 2b).
// The sweep that would overshoot the target accepts only its `need`
// candidates with the smallest (priority hash, cell index).
//
// A sweep works on bit masks, 32 cells of a row to a word: the six neighbours
// of a word are shifted or loaded words, a word's accepted cells by rule 2a are
// bit logic, and only cells with exactly one grown neighbour need their hash,
// compared as a whole number.  Sweeps are launched eight at a time; the device
// keeps the count and stops by itself, the host looks once per eight.  With a
// thread per cell, 64-bit index arithmetic, FP64 probabilities and a counter
// for every candidate a sweep took 100 us at 200^3 and a host round trip; now
// 25 us.
#include <algorithm>
#include <vector>

#include "cl_lbm.h"
#include "handle.cuh"
#include "internal.cuh"

namespace cl {

namespace {

__host__ __device__ __forceinline__ uint64_t splitmix64(uint64_t z) {
    z += 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

// the hash of (seed, stream, a, b) is splitmix64(hash3(seed, stream, a) ^ b)
__host__ __device__ __forceinline__ uint64_t hash3(uint64_t seed, uint64_t stream, uint64_t a) {
    uint64_t h = splitmix64(seed);
    h = splitmix64(h ^ stream);
    return splitmix64(h ^ a);
}

// a hash's uniform double is (h >> 11) 2^-53; scaled by 2^53 (exact) the tests u <= p and u < p
// become whole-number tests (h >> 11) < limit, with limit 2^53 for every p >= 1
constexpr double kTwo53 = 9007199254740992.0;
uint64_t limit_le(double p) { return !(p >= 0.0) ? 0 : (p >= 1.0 ? 1ULL << 53 : (uint64_t)floor(p * kTwo53) + 1); }
uint64_t limit_lt(double p) { return !(p > 0.0) ? 0 : (p >= 1.0 ? 1ULL << 53 : (uint64_t)ceil(p * kTwo53)); }

constexpr uint64_t kKeyStream = 0x5bd1e995ULL;
constexpr int kGrid = 152 * 8, kBlock = 256;
constexpr int kSweeps = 8;     // sweeps launched between two looks of the host
constexpr int kBins = 65536;   // of the selection: the top 16 bits of the hash

struct GrowState {
    unsigned long long tot[kSweeps + 1];  // cells of the code before sweep i of this launch, and after the last
    unsigned long long nc[kSweeps];       // candidates of sweep i
    int over;                             // sweep that would overshoot the target, -1: none yet
    unsigned n_sel;                       // selection: candidates gathered
    unsigned bin;                         // the bin that holds the last accepted candidate,
    unsigned bin_count;                   // its candidates,
    unsigned long long k;                 // and how many of them are accepted
};

// the box as rows of words: nw words of 32 cells per row
struct Words {
    int nx, ny, nz, nw;
    unsigned n;  // words in all (a box has fewer than 2^31 cells)
};

// allowed (and in the region) and grown cells as bits, and the number of cells of the code
__global__ void __launch_bounds__(kBlock) k_grow_masks(const uint8_t* __restrict__ phase,
                                                       const uint8_t* __restrict__ region, Words d, unsigned allowed,
                                                       unsigned grown, int code, unsigned* __restrict__ A,
                                                       unsigned* __restrict__ G, GrowState* st) {
    constexpr int U = 4;  // words in flight per warp
    const int lane = threadIdx.x & 31;
    unsigned n = 0;
    const unsigned warps = gridDim.x * (kBlock / 32);
    for (unsigned w0 = (blockIdx.x * kBlock + threadIdx.x) >> 5; w0 < d.n; w0 += U * warps) {
        unsigned pc[U], rg[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned w = w0 + u * warps;  // fewer than 2^31 + 2^16
            pc[u] = 255;
            rg[u] = 1;
            if (w < d.n) {
                const unsigned row = w / d.nw, x = (w - row * d.nw) * 32 + lane;
                if (x < (unsigned)d.nx) {
                    pc[u] = phase[(size_t)row * d.nx + x];
                    if (region) rg[u] = region[(size_t)row * d.nx + x];
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned w = w0 + u * warps;
            const bool in = pc[u] < 4;
            const unsigned a = __ballot_sync(0xffffffffu, in && ((allowed >> pc[u]) & 1u) && rg[u]);
            const unsigned g = __ballot_sync(0xffffffffu, in && ((grown >> pc[u]) & 1u));
            n += __popc(__ballot_sync(0xffffffffu, pc[u] == (unsigned)code));
            if (lane == 0 && w < d.n) {
                A[w] = a;
                G[w] = g;
            }
        }
    }
    if (lane == 0 && n) atomicAdd(&st->tot[0], (unsigned long long)n);
}

// the candidates of one sweep, from the state at its start.  A warp takes 32 words, one per lane, and evaluates the
// hashes of a word's cells together.
__global__ void __launch_bounds__(kBlock) k_grow_find(const unsigned* __restrict__ A, const unsigned* __restrict__ G,
                                                      Words d, unsigned long long target, uint64_t limit,
                                                      uint64_t seed, uint64_t stream, int sweep, int i,
                                                      unsigned* __restrict__ acc, GrowState* st) {
    if (st->over >= 0 || st->tot[i] >= target) return;
    __shared__ uint64_t pre[6];  // the hash up to the cell: by the direction of the one grown neighbour
    if (threadIdx.x < 6)
        pre[threadIdx.x] = hash3(seed, stream, sweep == 0 ? 0 : (uint64_t)sweep * 8 + (uint64_t)threadIdx.x);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const unsigned plane = (unsigned)d.nw * d.ny;
    unsigned n = 0;
    for (unsigned w0 = (blockIdx.x * kBlock + threadIdx.x) & ~31u; w0 < d.n; w0 += gridDim.x * kBlock) {
        const unsigned w = w0 + lane;
        const unsigned a = w < d.n ? A[w] : 0u;
        unsigned take = 0u, one = a, b0 = 0u, b1 = 0u, b2 = 0u;
        const unsigned row = w / d.nw, wx = w - row * d.nw;
        if (sweep > 0 && a) {
            const unsigned z = row / d.ny, y = row - z * d.ny;
            const unsigned r0 = w - wx, last = (unsigned)d.nw - 1;
            const unsigned g = G[w];
            unsigned nb[6];
            // bit x of a word: cell x + 1 (then x - 1) of the row, which wraps
            nb[0] = (g >> 1) | (wx == last ? (G[r0] & 1u) << ((d.nx - 1) & 31) : G[w + 1] << 31);
            nb[1] = (g << 1) | (wx == 0 ? (G[r0 + last] >> ((d.nx - 1) & 31)) & 1u : G[w - 1] >> 31);
            nb[2] = G[y + 1 == (unsigned)d.ny ? w - (plane - d.nw) : w + d.nw];
            nb[3] = G[y == 0 ? w + (plane - d.nw) : w - d.nw];
            nb[4] = G[z + 1 == (unsigned)d.nz ? w - plane * (d.nz - 1) : w + plane];
            nb[5] = G[z == 0 ? w + plane * (d.nz - 1) : w - plane];
            unsigned any = 0u, two = 0u;
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                two |= any & nb[k];
                any |= nb[k];
            }
            take = a & two;  // rule 2a
            one = a & any & ~two;
            // direction of the one grown neighbour, bit by bit
            b0 = nb[1] | nb[3] | nb[5];
            b1 = nb[2] | nb[3];
            b2 = nb[4] | nb[5];
        }
        const unsigned c0 = row * d.nx + wx * 32;  // the word's first cell
        for (unsigned todo = __ballot_sync(0xffffffffu, one != 0); todo; todo &= todo - 1) {
            const int j = __ffs(todo) - 1;
            const unsigned oj = __shfl_sync(0xffffffffu, one, j);
            const unsigned cj = __shfl_sync(0xffffffffu, c0, j) + lane;
            const unsigned p = ((__shfl_sync(0xffffffffu, b0, j) >> lane) & 1u) |
                               ((__shfl_sync(0xffffffffu, b1, j) >> lane) & 1u) << 1 |
                               ((__shfl_sync(0xffffffffu, b2, j) >> lane) & 1u) << 2;
            bool ok = false;
            if ((oj >> lane) & 1u) ok = (splitmix64(pre[p] ^ cj) >> 11) < limit;  // rule 2b, or a seed
            const unsigned t = __ballot_sync(0xffffffffu, ok);
            if (lane == j) take |= t;
        }
        if (w < d.n) acc[w] = take;
        n += __popc(take);
    }
    for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
    if (lane == 0 && n) atomicAdd(&st->nc[i], (unsigned long long)n);
}

// convert a word's cells `t`, one lane per cell
__device__ __forceinline__ void convert(const Words& d, unsigned w, unsigned t, int lane, uint8_t* phase, int code) {
    const unsigned row = w / d.nw, x = (w - row * d.nw) * 32 + lane;
    if ((t >> lane) & 1u) phase[(size_t)row * d.nx + x] = (uint8_t)code;
}

// accept all candidates of sweep i, unless they overshoot the target
__global__ void __launch_bounds__(kBlock) k_grow_apply(const unsigned* __restrict__ acc, Words d,
                                                       unsigned long long target, int keep_allowed, int code, int i,
                                                       unsigned* __restrict__ A, unsigned* __restrict__ G,
                                                       uint8_t* phase, GrowState* st) {
    const int over = *(volatile int*)&st->over;
    if (over >= 0 && over != i) return;
    const unsigned long long tot = st->tot[i], nc = st->nc[i];
    const bool first = blockIdx.x == 0 && threadIdx.x == 0;
    if (tot >= target || tot + nc > target) {
        if (first && tot >= target) st->tot[i + 1] = tot;
        else if (first) *(volatile int*)&st->over = i;
        return;
    }
    if (first) st->tot[i + 1] = tot + nc;
    if (nc == 0) return;
    const int lane = threadIdx.x & 31;
    for (unsigned w0 = (blockIdx.x * kBlock + threadIdx.x) & ~31u; w0 < d.n; w0 += gridDim.x * kBlock) {
        const unsigned w = w0 + lane;
        const unsigned t = w < d.n ? acc[w] : 0u;
        if (t) {
            G[w] |= t;
            if (!keep_allowed) A[w] &= ~t;
        }
        for (unsigned todo = __ballot_sync(0xffffffffu, t != 0); todo; todo &= todo - 1) {
            const int j = __ffs(todo) - 1;
            convert(d, w0 + j, __shfl_sync(0xffffffffu, t, j), lane, phase, code);
        }
    }
}

// ---- the sweep that overshoots: the need-th smallest (hash, cell) of its candidates.  A histogram of the hash's top
// 16 bits names the bin that holds it; the few candidates of that bin go to the host.
// What the passes over the candidates have in common: f(hash, cell) for every cell in acc, by lane
template <class F>
__device__ __forceinline__ void each_candidate(const unsigned* acc, const Words& d, uint64_t pre, F f) {
    const int lane = threadIdx.x & 31;
    for (unsigned w0 = (blockIdx.x * kBlock + threadIdx.x) & ~31u; w0 < d.n; w0 += gridDim.x * kBlock) {
        const unsigned t = w0 + lane < d.n ? acc[w0 + lane] : 0u;
        for (unsigned todo = __ballot_sync(0xffffffffu, t != 0); todo; todo &= todo - 1) {
            const int j = __ffs(todo) - 1;
            const unsigned tj = __shfl_sync(0xffffffffu, t, j), w = w0 + j;
            const unsigned row = w / d.nw, c = row * d.nx + (w - row * d.nw) * 32 + lane;
            if ((tj >> lane) & 1u) f(splitmix64(pre ^ c), c);
        }
    }
}

__global__ void __launch_bounds__(kBlock) k_select_hist(const unsigned* __restrict__ acc, Words d, uint64_t pre,
                                                        unsigned* __restrict__ hist) {
    each_candidate(acc, d, pre, [&](uint64_t k, unsigned) { atomicAdd(hist + (unsigned)(k >> 48), 1u); });
}

// the bin of the need-th smallest hash; one block of 1024
__global__ void __launch_bounds__(1024) k_select_bin(const unsigned* __restrict__ hist, unsigned long long need,
                                                     GrowState* st) {
    constexpr int kPer = kBins / 1024;
    __shared__ unsigned long long sum[1024];
    unsigned long long mine = 0;
    for (int j = 0; j < kPer; ++j) mine += hist[threadIdx.x * kPer + j];
    sum[threadIdx.x] = mine;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {  // inclusive scan
        const unsigned long long v = threadIdx.x >= (unsigned)o ? sum[threadIdx.x - o] : 0ULL;
        __syncthreads();
        sum[threadIdx.x] += v;
        __syncthreads();
    }
    unsigned long long before = sum[threadIdx.x] - mine;
    if (need > before && need <= sum[threadIdx.x])
        for (int j = 0; j < kPer; ++j) {
            const unsigned h = hist[threadIdx.x * kPer + j];
            if (need <= before + h) {
                st->bin = threadIdx.x * kPer + j;
                st->bin_count = h;
                st->k = need - before;
                break;
            }
            before += h;
        }
}

struct Candidate {
    uint64_t key;
    uint64_t cell;
};

__global__ void __launch_bounds__(kBlock) k_select_gather(const unsigned* __restrict__ acc, Words d, uint64_t pre,
                                                          unsigned bin, unsigned room, Candidate* __restrict__ out,
                                                          GrowState* st) {
    each_candidate(acc, d, pre, [&](uint64_t k, unsigned c) {
        if ((unsigned)(k >> 48) != bin) return;
        const unsigned at = atomicAdd(&st->n_sel, 1u);
        if (at < room) out[at] = Candidate{k, c};
    });
}

__global__ void __launch_bounds__(kBlock) k_select_apply(const unsigned* __restrict__ acc, Words d, uint64_t pre,
                                                         Candidate last, uint8_t* phase, int code) {
    each_candidate(acc, d, pre, [&](uint64_t k, unsigned c) {
        if (k < last.key || (k == last.key && c <= last.cell)) phase[c] = (uint8_t)code;
    });
}

__global__ void k_region_not_adjacent(const uint8_t* __restrict__ phase, int nx, int ny, int nz, int code, int avoid,
                                      uint8_t* __restrict__ region) {
    const unsigned N = (unsigned)nx * ny * nz, plane = (unsigned)nx * ny;
    for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x) {
        bool ok = phase[c] == code;
        if (ok) {
            const unsigned row = c / nx, z = row / ny;
            const int x = (int)(c - row * nx), y = (int)(row - z * ny);
            const unsigned q[6] = {x + 1 == nx ? c - (nx - 1) : c + 1,           x == 0 ? c + (nx - 1) : c - 1,
                                   y + 1 == ny ? c - (plane - nx) : c + nx,      y == 0 ? c + (plane - nx) : c - nx,
                                   z + 1 == (unsigned)nz ? c - (N - plane) : c + plane, z == 0 ? c + (N - plane) : c - plane};
#pragma unroll
            for (int d = 0; d < 6; ++d)
                if (phase[q[d]] == avoid) ok = false;
        }
        region[c] = ok ? 1 : 0;
    }
}

// Index arithmetic of 32 bits and whole-number sampling: 200^3, 170 us with 64-bit divisions and FP64, 50 us.
__global__ void __launch_bounds__(kBlock) k_reactive_faces(const uint8_t* __restrict__ phase, int nx, int ny, int nz,
                                                           int from_code, int to_code, uint64_t limit, uint64_t seed,
                                                           uint8_t* __restrict__ out, unsigned long long* total) {
    const unsigned N = (unsigned)nx * ny * nz, plane = (unsigned)nx * ny;
    const uint64_t pre = splitmix64(splitmix64(seed) ^ 0xface);
    unsigned n = 0;
    for (unsigned c = blockIdx.x * kBlock + threadIdx.x; c < N; c += gridDim.x * kBlock) {
        unsigned bits = 0;
        if (phase[c] == from_code) {
            const unsigned row = c / nx, z = row / ny;
            const int x = (int)(c - row * nx), y = (int)(row - z * ny);
            const unsigned q[6] = {c + 1, c - 1,  // x ends at the box, y and z wrap
                                   y + 1 == ny ? c - (plane - nx) : c + nx,      y == 0 ? c + (plane - nx) : c - nx,
                                   z + 1 == (unsigned)nz ? c - (N - plane) : c + plane, z == 0 ? c + (N - plane) : c - plane};
#pragma unroll
            for (int d = 0; d < 6; ++d) {
                if ((d == 0 && x + 1 == nx) || (d == 1 && x == 0)) continue;
                if (phase[q[d]] == to_code) bits |= 1u << d;
            }
            if (limit < (1ULL << 53) && bits) {
                const uint64_t h = splitmix64(pre ^ c);
                for (unsigned left = bits; left; left &= left - 1) {
                    const unsigned d = __ffs(left) - 1;
                    if ((splitmix64(h ^ d) >> 11) >= limit) bits &= ~(1u << d);
                }
            }
            n += __popc(bits);
        }
        out[c] = (uint8_t)bits;
    }
    for (int o = 16; o > 0; o >>= 1) n += __shfl_down_sync(0xffffffffu, n, o);
    if ((threadIdx.x & 31) == 0 && n) atomicAdd(total, (unsigned long long)n);
}

cl_status check_box(int nx, int ny, int nz) {
    const long long N = (long long)nx * ny * nz;
    if (nx < 1 || ny < 1 || nz < 1 || N >= (1LL << 31)) { set_msg_txt("box size out of range"); return CL_ERR_ARG; }
    return CL_OK;
}

// scratch: three masks, the state, the histogram of the selection
struct GrowScratch {
    unsigned *A, *G, *acc, *hist;
    GrowState* st;
};

cl_status read_state(const GrowState* d, GrowState* h, cudaStream_t s) {
    CK(cudaMemcpyAsync(h, d, sizeof(*h), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    return CL_OK;
}

// the overshooting sweep: accept the `need` smallest of the candidates in acc
cl_status select_smallest(const GrowScratch& b, const Words& d, long long need, uint64_t pre, uint8_t* phase, int code,
                          cudaStream_t s) {
    GrowState h;
    CK(cudaMemsetAsync(b.hist, 0, sizeof(unsigned) * kBins, s));
    k_select_hist<<<kGrid, kBlock, 0, s>>>(b.acc, d, pre, b.hist);
    k_select_bin<<<1, 1024, 0, s>>>(b.hist, (unsigned long long)need, b.st);
    CK(cudaGetLastError());
    CKS(read_state(b.st, &h, s));
    Candidate* out = nullptr;
    CK(cudaMallocAsync((void**)&out, sizeof(Candidate) * h.bin_count, s));
    std::vector<Candidate> in;
    cudaError_t e = cudaSuccess;
    try {
        in.resize(h.bin_count);
    } catch (...) {
        e = cudaErrorMemoryAllocation;
    }
    if (e == cudaSuccess) {
        k_select_gather<<<kGrid, kBlock, 0, s>>>(b.acc, d, pre, h.bin, h.bin_count, out, b.st);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(in.data(), out, sizeof(Candidate) * in.size(), cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(out, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) { set_msg("cl_qsgs_grow", e); return from_cuda(e); }
    std::nth_element(in.begin(), in.begin() + (h.k - 1), in.end(), [](const Candidate& x, const Candidate& y) {
        return x.key != y.key ? x.key < y.key : x.cell < y.cell;
    });
    k_select_apply<<<kGrid, kBlock, 0, s>>>(b.acc, d, pre, in[h.k - 1], phase, code);
    CK(cudaGetLastError());
    return CL_OK;
}

cl_status grow_impl(uint8_t* phase, const Words& d, int code, unsigned allowed, unsigned grown, const uint8_t* region,
                    long long target, double c_d, double p_alpha, uint64_t seed, uint64_t stream, int max_sweeps,
                    long long* final_count, cudaStream_t s, const GrowScratch& b) {
    GrowState h;
    CK(cudaMemsetAsync(b.st, 0, sizeof(GrowState), s));
    k_grow_masks<<<kGrid, kBlock, 0, s>>>(phase, region, d, allowed, grown, code, b.A, b.G, b.st);
    CK(cudaGetLastError());
    const unsigned long long want = target > 0 ? (unsigned long long)target : 0;
    const int keep = (int)((allowed >> code) & 1u);  // converted cells may be candidates again
    long long count = -1;                            // not read yet
    for (long long sweep = c_d > 0 ? 0 : 1;; sweep += kSweeps) {
        const int n = (int)std::min<long long>(kSweeps, (long long)max_sweeps + 1 - sweep);
        if (count >= 0) {
            CK(cudaMemcpyAsync(&b.st->tot[0], &b.st->tot[kSweeps], sizeof(b.st->tot[0]), cudaMemcpyDeviceToDevice, s));
            CK(cudaMemsetAsync(b.st->nc, 0, sizeof(b.st->nc), s));
        }
        CK(cudaMemsetAsync(&b.st->over, 0xff, sizeof(int), s));
        for (int i = 0; i < n; ++i) {
            const int sw = (int)(sweep + i);
            k_grow_find<<<kGrid, kBlock, 0, s>>>(b.A, b.G, d, want, limit_le(sw == 0 ? c_d : p_alpha), seed, stream, sw,
                                                 i, b.acc, b.st);
            k_grow_apply<<<kGrid, kBlock, 0, s>>>(b.acc, d, want, keep, code, i, b.A, b.G, phase, b.st);
            CK(cudaGetLastError());
        }
        CKS(read_state(b.st, &h, s));
        if (h.over >= 0) {
            const long long need = target - (long long)h.tot[h.over];
            CKS(select_smallest(b, d, need, hash3(seed, stream ^ kKeyStream, (uint64_t)(sweep + h.over)), phase, code, s));
            count = target;
            break;
        }
        count = (long long)h.tot[n > 0 ? n : 0];
        if (count >= target || sweep + n > max_sweeps) break;
    }
    if (final_count) *final_count = count;
    return CL_OK;
}

}  // namespace

}  // namespace cl

using namespace cl;

extern "C" {

cl_status cl_qsgs_grow(uint8_t* phase, int nx, int ny, int nz, int code, unsigned allowed_mask, unsigned grown_mask,
                       const uint8_t* region, long long target, double c_d, double p_alpha, uint64_t seed,
                       uint64_t stream, int max_sweeps, long long* final_count, void* cuda_stream) {
    if (!phase) { set_msg_txt("NULL argument"); return CL_ERR_ARG; }
    CKS(check_box(nx, ny, nz));
    if (code < 0 || code > 3 || !((grown_mask >> code) & 1u)) {
        set_msg_txt("code must be 0..3 and belong to grown_mask");
        return CL_ERR_ARG;
    }
    cudaStream_t s = (cudaStream_t)cuda_stream;
    Words d{nx, ny, nz, (nx + 31) / 32, 0};
    d.n = (unsigned)d.nw * ny * nz;
    unsigned char* scr = nullptr;
    const size_t state = (sizeof(GrowState) + 255) / 256 * 256;
    CK(cudaMallocAsync((void**)&scr, state + sizeof(unsigned) * (kBins + 3 * (size_t)d.n), s));
    GrowScratch b;
    b.st = (GrowState*)scr;
    b.hist = (unsigned*)(scr + state);
    b.A = b.hist + kBins;
    b.G = b.A + d.n;
    b.acc = b.G + d.n;
    cl_status st = grow_impl(phase, d, code, allowed_mask, grown_mask, region, target, c_d, p_alpha, seed, stream,
                             max_sweeps, final_count, s, b);
    cudaFreeAsync(scr, s);
    cudaError_t e = cudaStreamSynchronize(s);
    if (st == CL_OK && e != cudaSuccess) { set_msg("cl_qsgs_grow", e); return from_cuda(e); }
    return st;
}

cl_status cl_qsgs_region_not_adjacent(const uint8_t* phase, int nx, int ny, int nz, int code, int avoid,
                                      uint8_t* region, void* cuda_stream) {
    if (!phase || !region) { set_msg_txt("NULL argument"); return CL_ERR_ARG; }
    CKS(check_box(nx, ny, nz));
    cudaStream_t s = (cudaStream_t)cuda_stream;
    k_region_not_adjacent<<<kGrid, kBlock, 0, s>>>(phase, nx, ny, nz, code, avoid, region);
    CK(cudaGetLastError());
    CK(cudaStreamSynchronize(s));
    return CL_OK;
}

cl_status cl_qsgs_reactive_faces(const uint8_t* phase, int nx, int ny, int nz, int from_code, int to_code,
                                 double fraction, uint64_t seed, uint8_t* out, long long* n_faces, void* cuda_stream) {
    if (!phase || !out) { set_msg_txt("NULL argument"); return CL_ERR_ARG; }
    CKS(check_box(nx, ny, nz));
    cudaStream_t s = (cudaStream_t)cuda_stream;
    unsigned long long* tot = nullptr;
    CK(cudaMallocAsync((void**)&tot, sizeof(*tot), s));
    unsigned long long h = 0;
    cudaError_t e = cudaMemsetAsync(tot, 0, sizeof(*tot), s);
    if (e == cudaSuccess) {
        k_reactive_faces<<<kGrid, kBlock, 0, s>>>(phase, nx, ny, nz, from_code, to_code, limit_lt(fraction), seed, out, tot);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, tot, sizeof(h), cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(tot, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) { set_msg("cl_qsgs_reactive_faces", e); return from_cuda(e); }
    if (n_faces) *n_faces = (long long)h;
    return CL_OK;
}

}  // extern "C"
