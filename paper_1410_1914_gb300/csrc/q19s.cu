// D3Q19 (Eq. 22-24) on the (C, delta) state: the same pull-stream + BGK step
// as q19.cu, written on small quantities so that FP32 (or FP16) storage
// keeps the steady state to the FP64 answer.
//
// State per active cell after a step (post-collision, Eq. 21 with the
// equilibrium a_i C of Eq. 23):
//     g*_i = a_i C + delta_i,   i = 1..18,   delta_0 = -(delta_1 + ... + delta_18)
// C is an unevaluated sum hi + lo of two floats, stored side by side (one
// 8-byte load per source cell); the deviations are f32 (or f16 scaled by
// s_d).  With e_i
// the arriving population minus a_i C(x):
//     open link:   e_i = a_i (C(x - c_i) - C(x)) + delta_i(x - c_i)
//     wall:        e_i = r delta_opp(x) - (1 - r) a_i C(x)   (r = 1 unless reactive)
//     Dirichlet:   e_i = 2 a_i (C_bc - C(x)) - delta_opp(x)   (anti-bounce-back)
//     zero flux:   e_i = delta_opp(x)
//     dC = sum_i e_i + delta_0(x),  C' = C + dC (double-float),
//     delta'_i = (1 - omega) (e_i - a_i dC)
// which is the BGK step rewritten exactly; delta_0 is implied, so the mass
// of a cell is exact by construction.  Link classes as in q19.cu.
#include <cuda_fp16.h>
#include <math.h>

#include "device_util.cuh"
#include "internal.cuh"
#include "planes.cuh"

namespace cl {

namespace {

__host__ __device__ constexpr int s19_cx(int i) {
    constexpr int t[19] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0};
    return t[i];
}
__host__ __device__ constexpr int s19_cy(int i) {
    constexpr int t[19] = {0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1};
    return t[i];
}
__host__ __device__ constexpr int s19_cz(int i) {
    constexpr int t[19] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1};
    return t[i];
}
__host__ __device__ constexpr int s19_opp(int i) { return i == 0 ? 0 : ((i & 1) ? i + 1 : i - 1); }
// the link with direction (cx, cy, cz)
__host__ __device__ constexpr int s19_link(int cx, int cy, int cz) {
    for (int i = 0; i < 19; ++i)
        if (s19_cx(i) == cx && s19_cy(i) == cy && s19_cz(i) == cz) return i;
    return 0;
}
// bits i - 1 of the links whose x component is cx
__host__ __device__ constexpr uint32_t s19_links(int cx) {
    uint32_t m = 0;
    for (int i = 1; i < 19; ++i)
        if (s19_cx(i) == cx) m |= 1u << (i - 1);
    return m;
}
__host__ __device__ constexpr float s19_w(int i) {
    return i == 0 ? 1.f / 3.f : (i <= 6 ? 1.f / 18.f : 1.f / 36.f);
}

struct SF32 {
    using T = float;
    static __device__ __forceinline__ float ld(T v) { return v; }
    static __device__ __forceinline__ T st(float v) { return v; }
};
struct SF16 {
    using T = __half;
    static __device__ __forceinline__ float ld(T v) { return __half2float(v); }
    static __device__ __forceinline__ T st(float v) { return __float2half_rn(v); }
};

// Deviations are stored in groups of 32 cells of a row, [group][18][32], so that
// the 18 of a cell lie at fixed distances from one address.  Index of the first
// one (i = 1) of padded cell c; the others follow 32 apart.
template <class I>
__device__ __forceinline__ I dev_at(I c) {
    return (c >> 5) * (I)(18 * 32) + (c & (I)31);
}

// (hi, lo) + d, renormalised
__device__ __forceinline__ void df_add19(float hi, float lo, float d, float& ho, float& lo_out) {
    float s, e;
    two_sum(hi, d, s, e);
    e += lo;
    ho = s + e;
    lo_out = e - (ho - s);
}

}  // namespace

// ------------------------------------------------------------------- step
// A lane updates two neighbouring cells: own and y/z-shifted values come in
// pairs (one load for two cells), x-shifted ones as the pair's inner value and
// one more load, so a cell costs half the loads and index arithmetic of a
// lane per cell; the 18 deviations of a cell lie at fixed distances from one
// address, and sums and updates of the two cells are one instruction.  A block holds 256 cells of one plane, rows of 64 (of 32 where
// the padded row is not a multiple of 64: no idle lanes), so that y-neighbour
// rows are mostly its own, already in L1.  Every load is issued whatever the
// link's class -- in bounds, see below -- and the classes select afterwards;
// the end planes and catalytic links, which few cells have, are then set in
// branches.  Deviations stay in storage units inside the update (scaled by s_d,
// 1 for FP32), so nothing is rescaled on its way in or out.
// Bound by issue and by the latency of the loads: 128^3 Pt layer, FP16 state,
// 78 us a step with a cell per lane and plane-by-plane deviations, 49 us;
// FP32 state 72, 56 us.
// The reducing step keeps its sums in triples of floats (F3) down to the warp
// and in FP64 from there: one FP64 lane per cell took 515 us at 128^3 (FP16
// state), 87 us now; the same sums in pairs of floats and f32 took 75 us, with
// the residual off by 1e-9.  Four blocks on an SM: its 139 registers left three
// (100 us).
constexpr int kS19T = 128;

template <class S>
__device__ __forceinline__ float2 ld_pair(const typename S::T* p);
template <>
__device__ __forceinline__ float2 ld_pair<SF32>(const float* p) {
    return *reinterpret_cast<const float2*>(p);
}
template <>
__device__ __forceinline__ float2 ld_pair<SF16>(const __half* p) {
    return __half22float2(*reinterpret_cast<const __half2*>(p));
}
__device__ __forceinline__ void st_pair(float* p, float a, float b) { *reinterpret_cast<float2*>(p) = make_float2(a, b); }
__device__ __forceinline__ void st_pair(__half* p, float a, float b) {
    *reinterpret_cast<__half2*>(p) = __floats2half2_rn(a, b);
}

// w (hi + lo) + d, rounded once, where the first two floats of the sum settle it, whatever their rounding errors hide
// (all but a few in a million); else *clear = false
__device__ __forceinline__ float population(float w, float hi, float lo, float d, bool* clear) {
    const float p = __fmul_rn(w, hi), pe = __fmaf_rn(w, hi, -p), q = __fmul_rn(w, lo);
    float t, e;
    two_sum(p, d, t, e);
    const float low = (e + pe) + q, hidden = 0x1p-22f * ((fabsf(e) + fabsf(pe)) + fabsf(q));
    const float up = t + (low + hidden);
    *clear = *clear && up == t + (low - hidden);
    return up;
}

// The same whatever it takes: the sum is exact in three floats (but for 2^-70 of it), and the second is rounded to odd
// where the third is not 0, so that the last addition sees on which side of a tie it lies.
__device__ __noinline__ float population_at_tie(float w, float hi, float lo, float d) {
    const float p = __fmul_rn(w, hi), pe = __fmaf_rn(w, hi, -p), q = __fmul_rn(w, lo), qe = __fmaf_rn(w, lo, -q);
    float t, e, l, m, n, r;
    two_sum(p, d, t, e);
    two_sum(e, pe, l, m);
    two_sum(l, q, l, n);
    two_sum(t, l, t, l);
    two_sum(l, __fadd_rn(__fadd_rn(m, n), qe), l, r);
    const int bits = __float_as_int(l);
    if (r != 0.f && !(bits & 1)) l = __int_as_float(bits + ((r > 0.f) == (l > 0.f) ? 1 : -1));
    return isfinite(t) ? t + l : t;
}

template <class S, bool REDUCE, int LX, class I>  // LX lanes to a row
__global__ void __launch_bounds__(kS19T, REDUCE ? 4 : 0) k_step19s(Q19State src, Q19State dst, Q19Args a) {
    using T = typename S::T;
    constexpr bool HALF = sizeof(T) == 2;
    const int x = (blockIdx.x * LX + threadIdx.x % LX) * 2;
    const int y = blockIdx.y * (kS19T / LX) + threadIdx.x / LX, z = blockIdx.z;
    const int nx = a.nx, ny = a.ny, nz = a.nz, px = a.px;
    const I c = (I)x + (I)px * ((I)y + (I)ny * (I)z);  // even: px is a multiple of 32
    const bool in_row = x < px && y < ny;
    const uint2 mm = in_row ? *reinterpret_cast<const uint2*>(a.mask + c) : make_uint2(0u, 0u);
    const uint32_t m[2] = {mm.x, mm.y};
    // Whole 32-byte sectors are written -- 8 cells of FP32 or of C, 16 of FP16 (rows start on 32-cell boundaries) --
    // so every lane of a sector with an active cell goes through the update; inactive cells come out as zeros.
    const unsigned lane = threadIdx.x & 31u;
    const unsigned vote = __ballot_sync(0xffffffffu, ((m[0] | m[1]) & kQ19Active) != 0);
    const bool st_hl = ((vote >> (lane & ~3u)) & 0xFu) != 0;
    const bool st_d = in_row && (HALF ? ((vote >> (lane & ~7u)) & 0xFFu) != 0 : st_hl);
    const float s_d = HALF ? a.s_d : 1.f, inv_d = HALF ? a.inv_d : 1.f;
    const float2* __restrict__ shl = src.hl;
    const T* __restrict__ sd = reinterpret_cast<const T*>(src.d);
    constexpr F3 kNone = {0.f, 0.f, 0.f};
    F3 jin = kNone, jout = kNone, r = kNone;                 // through the end planes; R before the sink's factor
    F3 sum_c = kNone, sum_dc = kNone, sum_abs = kNone;       // C, |dC|, |C|
    bool bad[2] = {false, false};                            // not finite
    if (st_d) {
        float hn[2], ln[2];
        const I plane = (I)px * (I)ny;
        const I oym = y == 0 ? (I)(ny - 1) * (I)px : (I)0 - (I)px;
        const I oyp = y == ny - 1 ? (I)0 - (I)(ny - 1) * (I)px : (I)px;
        const I ozm = z == 0 ? (I)(nz - 1) * plane : (I)0 - plane;
        const I ozp = z == nz - 1 ? (I)0 - (I)(nz - 1) * plane : plane;
        // the cells left and right of the pair; at the row's ends the pair's own (the value is not used there)
        const int xl = x > 0 ? -1 : 0, xr = x + 2 < px ? 2 : 1;
        // the same steps in deviations, whatever the row (rows start on groups)
        const int dl = x > 0 && x % 32 == 0 ? -(18 * 32 - 31) : xl, dr2 = x % 32 == 30 && xr == 2 ? 18 * 32 - 30 : xr;
        const float4 own4 = *reinterpret_cast<const float4*>(shl + c);
        const float hx[2] = {own4.x, own4.z}, lx[2] = {own4.y, own4.w};
        const F2 own_a = f2(own4.x, own4.y), own_b = f2(own4.z, own4.w);
        const float rs_ = a.rsink;  // 1 - r
        const I cd = dev_at(c);
        const T* dc = sd + cd;
        float own[18][2];
        F2 sdd2 = f2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < 18; ++i) {
            const float2 v = ld_pair<S>(dc + i * 32);
            own[i][0] = v.x;
            own[i][1] = v.y;
            sdd2 = f2_add(sdd2, f2(v.x, v.y));  // the sum of the own deviations is -delta_0
        }
        const float2 sdd = f2_get(sdd2);
        // e_i of open and inert links, row by row of sources: (dy, dz) of the row, its links that come from the
        // cell at the same x, from x - 1 and from x + 1 (0: none)
        float ev[18][2];
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            constexpr int row_dy[9] = {0, -1, 1, 0, 0, -1, 1, -1, 1}, row_dz[9] = {0, 0, 0, -1, 1, -1, 1, 1, -1};
            const int dy = row_dy[q], dz = row_dz[q];
            const I r = c + (dy < 0 ? oym : (dy > 0 ? oyp : (I)0)) + (dz < 0 ? ozm : (dz > 0 ? ozp : (I)0));
            const T* dr = q == 0 ? dc : sd + dev_at(r);
            const float2* hr = shl + r;
            const float4 n4 = q == 0 ? own4 : *reinterpret_cast<const float4*>(hr);
            const F2 na = f2(n4.x, n4.y), nb = f2(n4.z, n4.w);
#pragma unroll
            for (int cx = -1; cx <= 1; ++cx) {
                if ((dy != 0 && dz != 0 && cx != 0) || (q == 0 && cx == 0)) continue;
                const int i = s19_link(cx, -dy, -dz), j = s19_opp(i);
                F2 sa = na, sb = nb;  // C of the cells that the pair's populations come from, and their deviations
                float2 nd;
                if (cx == 0) {
                    nd = ld_pair<S>(dr + (i - 1) * 32);
                } else {
                    const float2 o = hr[cx > 0 ? xl : xr];
                    const float od = S::ld(dr[(cx > 0 ? dl : dr2) + (i - 1) * 32]);
                    const float2 v = q == 0 ? make_float2(own[i - 1][0], own[i - 1][1]) : ld_pair<S>(dr + (i - 1) * 32);
                    if (cx > 0) {
                        sa = f2(o.x, o.y);
                        sb = na;
                        nd = make_float2(od, v.x);
                    } else {
                        sa = nb;
                        sb = f2(o.x, o.y);
                        nd = make_float2(v.y, od);
                    }
                }
                const float2 da = f2_get(f2_sub(sa, own_a)), db = f2_get(f2_sub(sb, own_b));
                const float ws = s19_w(i) * s_d;
                const float2 open = f2_get(f2_fma(f2(ws, ws), f2(da.x + da.y, db.x + db.y), f2(nd.x, nd.y)));
                ev[i - 1][0] = (m[0] >> (j - 1)) & 1u ? own[j - 1][0] : open.x;
                ev[i - 1][1] = (m[1] >> (j - 1)) & 1u ? own[j - 1][1] : open.y;
            }
        }
        const float2 om = *reinterpret_cast<const float2*>(a.omega + c);
        uint32_t rbits[2];
        float2 snap = make_float2(0.f, 0.f);
        if (REDUCE) snap = *reinterpret_cast<const float2*>(a.Csnap + c);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const bool inlet = x + k == 0, outlet = x + k == nx - 1;
            uint32_t rb = 0u;
            if (inlet || outlet || (m[k] & kQ19HasReact)) {
                if (m[k] & kQ19HasReact) rb = a.react[c + k];
#pragma unroll
                for (int i = 1; i < 19; ++i) {
                    const int j = s19_opp(i);
                    const float ws = s19_w(i) * s_d, nd = own[j - 1][k];
                    const bool wall = (m[k] >> (j - 1)) & 1u;
                    if (wall) {
                        if ((rb >> (j - 1)) & 1u) ev[i - 1][k] = fmaf(-rs_, nd + ws * (hx[k] + lx[k]), nd);
                    } else if (s19_cx(i) > 0 && inlet) {
                        ev[i - 1][k] = a.bc_in == CL_BC_DIRICHLET ? 2.0f * ws * ((a.c_in - hx[k]) - lx[k]) - nd : nd;
                    } else if (s19_cx(i) < 0 && outlet) {
                        ev[i - 1][k] = a.bc_out == CL_BC_DIRICHLET ? 2.0f * ws * ((a.c_out - hx[k]) - lx[k]) - nd : nd;
                    }
                }
            }
            rbits[k] = rb;
        }
        F2 se = f2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < 18; ++i) se = f2_add(se, f2(ev[i][0], ev[i][1]));
        const F2 dC2 = f2_sub(se, sdd2);  // sum e_i + delta_0, storage units
        const float2 dCs = f2_get(dC2);
        df_add19(hx[0], lx[0], dCs.x * inv_d, hn[0], ln[0]);
        df_add19(hx[1], lx[1], dCs.y * inv_d, hn[1], ln[1]);
        // an inactive cell's result (finite: it read zeros and state values) becomes zero
        const bool on[2] = {(m[0] & kQ19Active) != 0, (m[1] & kQ19Active) != 0};
        const F2 om1 = f2(on[0] ? 1.0f - om.x : 0.f, on[1] ? 1.0f - om.y : 0.f);
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (!on[k]) hn[k] = ln[k] = 0.f;
        T* dd = reinterpret_cast<T*>(dst.d) + cd;
        float2 dn[18];
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            const float w = s19_w(i);
            dn[i - 1] = f2_get(f2_mul(om1, f2_fma(f2(-w, -w), dC2, f2(ev[i - 1][0], ev[i - 1][1]))));
            st_pair(dd + (i - 1) * 32, dn[i - 1].x, dn[i - 1].y);
        }
        if (st_hl) *reinterpret_cast<float4*>(dst.hl + c) = make_float4(hn[0], ln[0], hn[1], ln[1]);
        if (REDUCE) {
            float Cf[2], dc[2], de[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                Cf[k] = on[k] ? hn[k] + ln[k] : 0.f;
                two_sum(Cf[k], on[k] ? (k == 0 ? -snap.x : -snap.y) : 0.f, dc[k], de[k]);
                if (dc[k] < 0.f) {
                    dc[k] = -dc[k];
                    de[k] = -de[k];
                }
                bad[k] = !isfinite(hn[k]);
            }
            // sum += n / 36 (c - C) of cell k, c being three floats: the equilibrium parts of its links, axis links
            // counted twice
            auto equilibrium = [&](F3& sum, float n, float c, const float2& rest, float hi, float lo) {
                const float w = n * s19_w(7), we = fmaf(n, s19_w(7), -w);
                float s, e;
                two_sum(c, -hi, s, e);
                f3_add_product(sum, w, s);
                f3_add_product_low(sum, we, s);
                f3_add_product_low(sum, w, e);
                f3_add_product_low(sum, w, rest.x);
                f3_add_product_low(sum, w, -lo);
                sum.c = fmaf(we, (e + rest.x) - lo, fmaf(w, rest.y, sum.c));
            };
            auto count = [](uint32_t links) { return (float)(__popc(links) + __popc(links & 0x3fu)); };
            // the inlet is cell 0 of a pair, the outlet either; 2 (w c - g*_i) and 2 (g*_i - w c) over their open links
            if (x == 0 && on[0] && a.bc_in == CL_BC_DIRICHLET) {
                const uint32_t open = ~m[0] & s19_links(-1);
                equilibrium(jin, 2.0f * count(open), a.c_in, a.c_in_rest, hn[0], ln[0]);
#pragma unroll
                for (int i = 1; i < 19; ++i)
                    if (s19_cx(i) < 0 && ((open >> (i - 1)) & 1u)) f3_add(jin, -2.0f * (dn[i - 1].x * inv_d));
            }
            const int ko = (nx - 1) & 1;
            if (x == nx - 1 - ko && (ko ? on[1] : on[0]) && a.bc_out == CL_BC_DIRICHLET) {
                const uint32_t open = ~(ko ? m[1] : m[0]) & s19_links(1);
                equilibrium(jout, -2.0f * count(open), a.c_out, a.c_out_rest, ko ? hn[1] : hn[0], ko ? ln[1] : ln[0]);
#pragma unroll
                for (int i = 1; i < 19; ++i)
                    if (s19_cx(i) > 0 && ((open >> (i - 1)) & 1u))
                        f3_add(jout, 2.0f * ((ko ? dn[i - 1].y : dn[i - 1].x) * inv_d));
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const uint32_t rb = on[k] ? rbits[k] & ((1u << 18) - 1u) : 0u;  // g*_i = w C + d of the catalytic links
                if (rb == 0u) continue;
                equilibrium(r, -count(rb), 0.f, make_float2(0.f, 0.f), hn[k], ln[k]);
#pragma unroll
                for (int i = 1; i < 19; ++i)
                    if ((rb >> (i - 1)) & 1u) f3_add(r, (k == 0 ? dn[i - 1].x : dn[i - 1].y) * inv_d);
            }
            two_sum(Cf[0], Cf[1], sum_c.a, sum_c.b);
            two_sum(fabsf(Cf[0]), fabsf(Cf[1]), sum_abs.a, sum_abs.b);
            two_sum(dc[0], dc[1], sum_dc.a, sum_dc.b);
            f3_add_low(sum_dc, de[0]);
            f3_add_low(sum_dc, de[1]);
        }
        if (REDUCE) {
            if (on[0]) snap.x = hn[0] + ln[0];
            if (on[1]) snap.y = hn[1] + ln[1];
            *reinterpret_cast<float2*>(a.Csnap + c) = snap;
        }
    }
    if (REDUCE) {
        // Four sums over the warp in six additions: half of the lanes go on with two of them, then a quarter with one.
        auto other = [](const F3& v, int o) {
            return F3{__shfl_xor_sync(0xffffffffu, v.a, o), __shfl_xor_sync(0xffffffffu, v.b, o),
                      __shfl_xor_sync(0xffffffffu, v.c, o)};
        };
        const bool hi16 = lane & 16u, hi8 = lane & 8u;
        F3 v0 = hi16 ? sum_abs : sum_c, v1 = hi16 ? r : sum_dc;
        f3_add(v0, other(hi16 ? sum_c : sum_abs, 16));
        f3_add(v1, other(hi16 ? sum_dc : r, 16));
        F3 v = hi8 ? v1 : v0;
        f3_add(v, other(hi8 ? v0 : v1, 8));
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) f3_add(v, other(v, o));
        const unsigned nbad = __popc(__ballot_sync(0xffffffffu, bad[0])) + __popc(__ballot_sync(0xffffffffu, bad[1]));
        __shared__ F3 part[kS19T / 32][4];           // sum C, sum |dC|, sum |C|, R
        __shared__ F3 ends[2][kS19T / LX];           // the rows' cells of the end planes: one lane each
        __shared__ unsigned part_bad[kS19T / 32];
        if ((lane & 7u) == 0) part[threadIdx.x >> 5][lane >> 3] = v;
        if (lane == 0) part_bad[threadIdx.x >> 5] = nbad;
        const int row = threadIdx.x / LX, out_lane = (nx - 1) / 2 - blockIdx.x * LX;
        if (threadIdx.x % LX == 0) ends[0][row] = jin;
        if (threadIdx.x % LX == (out_lane >= 0 && out_lane < LX ? out_lane : 0)) ends[1][row] = jout;
        __syncthreads();
        if (threadIdx.x < RED_N) {
            double v = 0.0;
            if (threadIdx.x == RED_JIN || threadIdx.x == RED_JOUT) {
                for (int q = 0; q < kS19T / LX; ++q) v += f3_get(ends[threadIdx.x == RED_JOUT][q]);
            } else if (threadIdx.x == RED_NONFINITE) {
                for (int w = 0; w < kS19T / 32; ++w) v += (double)part_bad[w];
            } else {
                const int k = threadIdx.x == RED_SUMC ? 0 : (threadIdx.x == RED_DC ? 1 : (threadIdx.x == RED_ABSC ? 2 : 3));
                for (int w = 0; w < kS19T / 32; ++w) v += f3_get(part[w][k]);
            }
            if (threadIdx.x == RED_R) v *= a.rsink_d;
            const long long blk = blockIdx.x + (long long)gridDim.x * (blockIdx.y + (long long)gridDim.y * blockIdx.z);
            a.partials[blk * RED_N + threadIdx.x] = v;
        }
    }
}

// ----------------------------------------------------------- init / readout
// C0 (unpadded, nullable: the linear ramp) into (hi, lo), deviations 0.
template <class S>
__global__ void k_init19s(Q19State st, Q19Args a, const float* __restrict__ C0, const float2* __restrict__ ramp) {
    using T = typename S::T;
    const long long NP = a.NP;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < NP;
         p += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(p % a.px);
        float hi = 0.f, lo = 0.f;
        if (a.mask[p] & kQ19Active) {
            if (C0) {
                hi = C0[x + (long long)a.nx * (p / a.px)];
            } else {
                hi = ramp[x].x;
                lo = ramp[x].y;
            }
        }
        st.hl[p] = make_float2(hi, lo);
        for (int i = 0; i < 18; ++i) reinterpret_cast<T*>(st.d)[dev_at((unsigned long long)p) + i * 32] = S::st(0.f);
        a.Csnap[p] = hi + lo;
    }
}

// per x-plane (planes.cuh): the deviations are read only where a catalytic or boundary link needs them
template <class S>
struct State19PlaneOp {
    using T = typename S::T;
    static constexpr int kRows = 4;
    Q19State st;
    Q19Args a;
    struct Item {
        long long p;
        uint32_t m;
        float2 hl;
    };
    __device__ __forceinline__ double sink() const { return a.rsink_d; }
    __device__ __forceinline__ float d(int i, long long p) const {
        return S::ld(reinterpret_cast<const T*>(st.d)[dev_at((unsigned long long)p) + (i - 1) * 32]) *
               (sizeof(T) == 2 ? a.inv_d : 1.f);
    }
    __device__ __forceinline__ Item load(int x, int row) const {
        Item t;
        t.p = x + (long long)a.px * row;
        t.m = a.mask[t.p];
        t.hl = st.hl[t.p];
        return t;
    }
    __device__ __forceinline__ void use(const Item& t, PlaneAcc& acc) const {
        if (!(t.m & kQ19Active)) return;
        f3_add(acc.c, t.hl.x);
        f3_add_low(acc.c, t.hl.y);
        acc.n += 1;
        if (!(t.m & kQ19HasReact)) return;
        for (unsigned left = a.react[t.p]; left; left &= left - 1) {  // g*_i = a_i C + d_i of the catalytic links
            const int i = __ffs(left);
            const float w = s19_w(i);
            f3_add_product(acc.r, w, t.hl.x);
            f3_add_product_low(acc.r, w, t.hl.y);
            f3_add(acc.r, d(i, t.p));
        }
    }
    // 2 (a_i C_bc - g*_i) over the open links through the plane (sgn -1: x = 0, which take in; +1: x = L)
    __device__ __forceinline__ double through(int x, int row, int sgn, double c_bc) const {
        const Item t = load(x, row);
        double s = 0.0;
        if (!(t.m & kQ19Active)) return s;
        const double C = (double)t.hl.x + (double)t.hl.y;
        for (int i = 1; i < 19; ++i)
            if (s19_cx(i) == sgn && !((t.m >> (i - 1)) & 1u))
                s += 2.0 * ((double)s19_w(i) * c_bc - ((double)s19_w(i) * C + (double)d(i, t.p)));
        return s;
    }
    __device__ __forceinline__ double inflow(int row) const {
        return a.bc_in == CL_BC_DIRICHLET ? through(0, row, -1, a.c_in_d) : 0.0;
    }
    __device__ __forceinline__ double outflow(int row) const {
        return a.bc_out == CL_BC_DIRICHLET ? -through(a.nx - 1, row, 1, a.c_out_d) : 0.0;
    }
};

// Unpadded C and/or g* as [19][nz][ny][nx]; g*_i = a_i C + delta_i of the pair (hi, lo), rounded once.  A call at 128^3,
// FP32 and FP16 state: 246 and 245 us with FP64 per population; 111 and 71 us in pairs of floats, which may round to the
// other side near a tie; 72 and 69 us, all 18 deviations in flight and the ties apart.
template <class S>
__global__ void __launch_bounds__(256) k_out19s(Q19State st, Q19Args a, float* __restrict__ C, float* __restrict__ gout) {
    using T = typename S::T;
    constexpr bool HALF = sizeof(T) == 2;
    const long long N = (long long)a.nx * a.ny * a.nz;
    for (long long c = blockIdx.x * 256LL + threadIdx.x; c < N; c += gridDim.x * 256LL) {
        const long long row = N < (1LL << 32) ? (long long)((uint32_t)c / (uint32_t)a.nx) : c / a.nx;
        const long long p = (c - row * a.nx) + (long long)a.px * row;
        const bool act = (a.mask[p] & kQ19Active) != 0;
        const float2 hl = act ? st.hl[p] : make_float2(0.f, 0.f);
        if (C) C[c] = hl.x + hl.y;
        if (!gout) continue;
        const T* dp = reinterpret_cast<const T*>(st.d) + dev_at((unsigned long long)p);
        float d[19], g[19];
        d[0] = 0.f;
#pragma unroll
        for (int i = 1; i < 19; ++i) d[i] = act ? S::ld(dp[(i - 1) * 32]) * (HALF ? a.inv_d : 1.f) : 0.f;
#pragma unroll
        for (int i = 1; i < 19; ++i) d[0] -= d[i];
        bool clear = true;
#pragma unroll
        for (int i = 0; i < 19; ++i) g[i] = population(s19_w(i), hl.x, hl.y, d[i], &clear);
        if (!clear)
#pragma unroll
            for (int i = 0; i < 19; ++i) g[i] = population_at_tie(s19_w(i), hl.x, hl.y, d[i]);
#pragma unroll
        for (int i = 0; i < 19; ++i) gout[i * N + c] = g[i];
    }
}

// -------------------------------------------------------------- launchers
// lanes of a row: 64-cell rows read the widest, 32-cell ones leave no lane idle (px is a multiple of 32)
static int step19s_lanes(int px) { return px % 64 == 0 ? 32 : 16; }

static dim3 step19s_grid(int px, int ny, int nz) {
    const int lx = step19s_lanes(px), rows = kS19T / lx;
    return dim3((unsigned)(px / (2 * lx)), (unsigned)((ny + rows - 1) / rows), (unsigned)nz);
}

cudaError_t launch_step19s(int storage, const Q19State& src, const Q19State& dst, const Q19Args& a, bool reduce,
                           cudaStream_t s) {
    const dim3 g = step19s_grid(a.px, a.ny, a.nz);
    const bool narrow = !a.wide && 19LL * a.NP < (1LL << 32), wide_row = step19s_lanes(a.px) == 32;
#define CL_Q19S(SS, R, LX, II) k_step19s<SS, R, LX, II><<<g, kS19T, 0, s>>>(src, dst, a)
#define CL_Q19L(SS, R, II) do { if (wide_row) CL_Q19S(SS, R, 32, II); else CL_Q19S(SS, R, 16, II); } while (0)
    if (storage == CL_STORE_FP16DEV) {
        if (narrow) { if (reduce) CL_Q19L(SF16, true, uint32_t); else CL_Q19L(SF16, false, uint32_t); }
        else { if (reduce) CL_Q19L(SF16, true, unsigned long long); else CL_Q19L(SF16, false, unsigned long long); }
    } else {
        if (narrow) { if (reduce) CL_Q19L(SF32, true, uint32_t); else CL_Q19L(SF32, false, uint32_t); }
        else { if (reduce) CL_Q19L(SF32, true, unsigned long long); else CL_Q19L(SF32, false, unsigned long long); }
    }
#undef CL_Q19L
#undef CL_Q19S
    return cudaGetLastError();
}

int step19s_blocks(int px, int ny, int nz) {
    const dim3 g = step19s_grid(px, ny, nz);
    return (int)(g.x * g.y * g.z);
}

cudaError_t launch_init19s(int storage, const Q19State& st, const Q19Args& a, const float* C0, const float2* ramp,
                           cudaStream_t s) {
    if (storage == CL_STORE_FP16DEV) k_init19s<SF16><<<152 * 8, 256, 0, s>>>(st, a, C0, ramp);
    else k_init19s<SF32><<<152 * 8, 256, 0, s>>>(st, a, C0, ramp);
    return cudaGetLastError();
}

cudaError_t launch_readout19s(int storage, const Q19State& st, const Q19Args& a, double* out, cudaStream_t s) {
    const long long rows = (long long)a.ny * a.nz;
    if (storage == CL_STORE_FP16DEV) return launch_planes(State19PlaneOp<SF16>{st, a}, a.nx, rows, out, s);
    return launch_planes(State19PlaneOp<SF32>{st, a}, a.nx, rows, out, s);
}

cudaError_t launch_out19s(int storage, const Q19State& st, const Q19Args& a, float* C, float* g, cudaStream_t s) {
    if (storage == CL_STORE_FP16DEV) k_out19s<SF16><<<152 * 8, 256, 0, s>>>(st, a, C, g);
    else k_out19s<SF32><<<152 * 8, 256, 0, s>>>(st, a, C, g);
    return cudaGetLastError();
}

}  // namespace cl
