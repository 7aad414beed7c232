// The preconditioned Krylov steady solve on the active cells alone.
//
// Its vectors hold the active cells only (45 % of a Pt layer's box), plane
// by plane: population q of active cell i is element q * np + i, np being
// the cell count rounded up to 32 (the pad stays zero).  nb[(k - 1) * n + i]
// is the active index of the cell that link k of cell i leads to, or what
// the link meets instead.
#pragma once

#include "internal.cuh"
#include "pcg.cuh"

namespace cl {

enum DsaLink { DSA_WALL = -1, DSA_SINK = -2, DSA_FIXED = -3, DSA_NOFLUX = -4 };

struct DsaCells {
    int q;         // 7 or 19
    int n, np;     // active cells; plane stride
    int* list;     // [n] cell index in the population layout (D3Q19: padded rows)
    int* inv;      // [cells] active index
    int* nb;       // [(q - 1) * n]
    float* sink;   // [n] 1 - r of the cell's catalytic links
    float* dinv;   // [n] 1 / diag(L), 0 where the row is empty
    float* omega;  // [n]
};

// Numbers the active cells in index order: inv, and *count (device).  part:
// dsa_scan_blocks(cells) ints.
int dsa_scan_blocks(long long cells);
cudaError_t launch_dsa_count(const uint16_t* mask7, const uint32_t* mask19, long long cells, int* part, int* count,
                             cudaStream_t s);
cudaError_t launch_dsa_number(const uint16_t* mask7, const uint32_t* mask19, long long cells, const int* part,
                              int* inv, int* list, cudaStream_t s);
// Links, diagonals, sinks and relaxation rates of the listed cells
cudaError_t launch_dsa_links7(const DsaCells& d, const StepArgs& a, cudaStream_t s);
cudaError_t launch_dsa_links19(const DsaCells& d, const Q19Args& a, cudaStream_t s);

// w = (I - A) z, A the step with zero boundary values and no source
cudaError_t launch_dsa_apply(const DsaCells& d, const float* z, float* w, cudaStream_t s);
// z = v + w_i eps, L eps = sum_i v_i (conjugate gradients until r.r is tol2 of its start).  The caller asks
// for 1e-1: bulk, Knudsen and reactive layers of 24^3 to 160^3 (D3Q7) and 24^3 to 110^3 (D3Q19) take 16 to 139 outer
// iterations against 15 to 135 at 1e-2, with 40 to 80 % of the inner ones (4003 against 10323 at 96^3, 9261 against
// 12406 at 128^3).  What a correction leaves behind then has more of the slow modes, whose error is the largest for a
// residual: at the same residual the field was off by 4.5e-9 of itself (40 layers of 24^3 to 96^3, solved to 1e-8,
// geometric mean) against 2.7e-9 at 1e-2.  So the last correction goes on to 4e-4 instead of 1e-3: 2.4e-9, for 6 % of
// the time (the looser inner solves save 35 %).
cudaError_t launch_dsa_prec(const DsaCells& d, const float* v, float* z, PcgArgs<float> a, cudaStream_t s);
// whether the CG of n cells keeps its vectors in memory (PcgArgs x .. w)
bool dsa_prec_streams(int n);

// Modified Gram-Schmidt of w against V[0..j] (vectors of L floats, `stride`
// apart), in one launch: col[k] = V_k.w, w -= col[k] V_k, col[j + 1] = |w|,
// V[j + 1] = w / |w|.  meet_mem: pcg_meet_bytes(dsa_mgs_blocks()); out->gave_up
// says that a wait ran out.
cudaError_t launch_dsa_mgs(float* V, long long stride, int j, float* w, long long L, double* col, void* meet_mem,
                           PcgOut* out, const PcgWaits& waits, cudaStream_t s);
int dsa_mgs_blocks();
// e += sum_k y[k] Z_k, k < m
cudaError_t launch_dsa_update(float* e, const float* Z, long long stride, int m, const double* y, long long L,
                              cudaStream_t s);
// c (population layout) -> active cells, and x64 += sign * e (active cells -> population layout)
cudaError_t launch_dsa_gather(const DsaCells& d, const float* c, long long cells, float* out, cudaStream_t s);
cudaError_t launch_dsa_add64(const DsaCells& d, const float* e, double sign, long long cells, double* x,
                             cudaStream_t s);

}  // namespace cl
