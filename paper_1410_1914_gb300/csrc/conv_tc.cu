// 3x3x3 convolutions of the warm-start network on the 5th-generation tensor
// cores (tcgen05.mma kind::f16, BF16 operands, FP32 accumulators in tensor
// memory).  Implicit GEMMs: out[v][n] = sum over taps t and input channels c
// of in[shift(v, t)][c] * w[t][n][c]; the weight gradient is the GEMM over
// voxels.  Three kernels:
//
//   k_conv3d_march       forward / data gradient of up to 64 input channels: a
//                        CTA marches an 8 x 16 column of output voxels along z
//                        with the weights resident in shared memory; each input
//                        plane is staged once and serves three output planes.
//   k_conv3d_halo        the same where the weights do not fit: one CTA per
//                        8 x 16 block of output voxels; the 10 x 18 x 3 input
//                        halo is staged once per channel chunk and every tap
//                        is a shifted descriptor into it; weights stream.
//   k_conv3d_tc          forward with one gather per tap and voxel; taken
//                        where batch x planes is above 65535, the other two's
//                        grid limit.
//   k_conv3d_wgrad_tc    weight gradient: per voxel block the input tile and
//                        the halo of 16 output-gradient channels are staged
//                        once and serve all 27 taps, whose accumulators stay in
//                        tensor memory over a slice of blocks.
//
// Roles of k_conv3d_halo and k_conv3d_tc (160 threads): warps 0-3 stage operands with cp.async (zero fill
// outside the box; y and z wrap by index), make them visible to the tensor
// core (fence.proxy.async) and arrive on the stage's `full` barrier, then
// run the epilogue (tcgen05.ld of their 32 TMEM lanes: warp w owns lanes
// 32w..32w+31); warp 4 allocates and frees the tensor memory and its lane 0
// issues the MMAs of each stage and commits them to the stage's `empty`
// barrier and, after the last stage, to `done`.
//
// Shared-memory operands use the no-swizzle core-matrix layouts: 8 rows of
// 16 bytes, contiguous.  K-major (forward): a row is 8 input channels of one
// voxel; LBO steps to the next 8 channels, SBO to the next 8 rows.  MN-major
// (weight gradient): a row is 8 channels of one voxel read along K = voxels;
// LBO steps to the next 8 voxels, SBO to the next 8 channels.
//
// Every wait is bounded; on expiry the CTA records an error bit, stops
// issuing work, waits (bounded) for the MMAs it issued, frees its tensor
// memory and returns.
#include <cuda_bf16.h>
#include <stdint.h>

#include "internal.cuh"
#include "nn.cuh"

namespace cl {

namespace {

constexpr int kTcM = 128;       // output voxels per CTA (TMEM lanes)
constexpr int kFwStages = 6;    // shared-memory stages of the forward kernel
constexpr int kLag = kFwStages - 2;  // its stages whose copies are in flight per thread
constexpr int kTcThreads = 160; // 4 producer/epilogue warps + 1 MMA warp

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void bar_init(uint64_t* b, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(b)), "r"(count) : "memory");
}

__device__ __forceinline__ bool bar_try_wait(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(b)), "r"(parity)
        : "memory");
    return ok != 0;
}

// bounded wait (~1 s of SM clock); false on expiry
__device__ __forceinline__ bool bar_wait(uint64_t* b, uint32_t parity) {
    if (bar_try_wait(b, parity)) return true;
    const long long t0 = clock64();
    while (!bar_try_wait(b, parity))
        if (clock64() - t0 > (1LL << 31)) return false;
    return true;
}

__device__ __forceinline__ void bar_arrive(uint64_t* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(b)) : "memory");
}

// 16-byte asynchronous copy global -> shared; zero fill when !valid.  The
// .ca form keeps the line in L1: the taps of neighbouring voxels read the
// same activation rows again within the CTA.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async16_ca(uint32_t dst, const void* src, bool valid) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// generic-proxy writes to shared memory become visible to the tensor core
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// shared-memory matrix descriptor: K-major, no swizzle
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;  // descriptor version of this architecture
    return d;                // base offset 0, swizzle none
}

// instruction descriptor, kind::f16: D f32, A and B bf16, both K-major
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16_ss(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* b) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(b))
                 : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// The MMA warp runs its loop as a whole, so that descriptors and addresses stay in
// uniform registers, and one elected lane issues.
__device__ __forceinline__ bool elect_one() {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r));
    return r != 0;
}

// warp index as a warp-uniform value
__device__ __forceinline__ int warp_index() { return __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0); }

// bias, ReLU and rounding of 16 accumulators into 16 channels of a voxel
__device__ __forceinline__ void store16(const uint32_t (&acc)[16], const float* bias, int relu, __nv_bfloat16* out) {
    uint32_t pk[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        float a = __uint_as_float(acc[2 * j]) + (bias ? bias[2 * j] : 0.f);
        float b = __uint_as_float(acc[2 * j + 1]) + (bias ? bias[2 * j + 1] : 0.f);
        if (relu) { a = fmaxf(a, 0.f); b = fmaxf(b, 0.f); }
        __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
        pk[j] = *reinterpret_cast<uint32_t*>(&h);
    }
    uint4* dst = reinterpret_cast<uint4*>(out);
    dst[0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
    dst[1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
}

struct TcShape {
    int CK;        // channels per k-step (16..64, divides ci)
    int N;         // output channels (co)
    int ncols;     // TMEM columns (power of two >= max(32, N))
    int a_bytes;   // 128 x CK x 2
    int b_bytes;   // N x CK x 2
    int stage;     // a_bytes + b_bytes
    int smem;      // dynamic shared memory
};

}  // namespace

__host__ __device__ inline TcShape tc_shape(int ci, int co) {
    TcShape s;
    // widest channel chunk that divides ci and keeps the stages within ~200 KB
    const int cands[4] = {64, 48, 32, 16};
    s.CK = 16;
    for (int i = 0; i < 4; ++i) {
        const int ck = cands[i];
        if (ck > ci || ci % ck) continue;
        if (1024 + kFwStages * (kTcM + co) * ck * 2 <= 200 * 1024) { s.CK = ck; break; }
    }
    s.N = co;
    int c = 32;
    while (c < co) c <<= 1;
    s.ncols = c;
    s.a_bytes = kTcM * s.CK * 2;
    s.b_bytes = co * s.CK * 2;
    s.stage = s.a_bytes + s.b_bytes;
    s.smem = 1024 + kFwStages * s.stage;
    return s;
}

__global__ void __launch_bounds__(kTcThreads) k_conv3d_tc(const __nv_bfloat16* __restrict__ in,
                                                          const __nv_bfloat16* __restrict__ w,
                                                          const float* __restrict__ bias,
                                                          __nv_bfloat16* __restrict__ out, ConvGeom g, int relu,
                                                          int* err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    const TcShape sh = tc_shape(g.ci, g.co);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);
    uint64_t* empty = full + kFwStages;
    uint64_t* done = empty + kFwStages;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);
    unsigned char* stages = smem + 1024;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long long M = (long long)g.N * g.D * g.H * g.W;
    const long long v0 = (long long)blockIdx.x * kTcM;
    const int CK = sh.CK, kgroups = CK / 8;
    const int ksteps = 27 * (g.ci / CK);
    const uint32_t sbo_a = (uint32_t)kgroups * 128u, sbo_b = sbo_a;

    if (tid == 0) {
        for (int s = 0; s < kFwStages; ++s) {
            bar_init(&full[s], 128);
            bar_init(&empty[s], 1);
        }
        bar_init(done, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 4) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                     "r"(sh.ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp < 4) {
        // ------------------------------------------------------ producers
        const int r = tid;  // output row of this thread
        const long long v = v0 + r;
        const bool row_ok = v < M;
        int x = 0, y = 0, z = 0;
        long long nb = 0;
        if (row_ok) {
            x = (int)(v % g.W);
            long long q = v / g.W;
            y = (int)(q % g.H);
            q /= g.H;
            z = (int)(q % g.D);
            nb = q / g.D;
        }
        const uint32_t a_row = (uint32_t)(r >> 3) * sbo_a + (uint32_t)(r & 7) * 16u;
        bool ok = true;
        int issued = 0;  // stages whose copies were issued
        for (int ks = 0; ks < ksteps; ++ks) {
            const int s = ks % kFwStages;
            if (ks >= kFwStages) {
                if (!bar_wait(&empty[s], ((ks / kFwStages) - 1) & 1)) { ok = false; }
            }
            if (!ok || *(volatile int*)abort_flag) { ok = false; break; }
            const int t = ks / (g.ci / CK);
            const int c0 = (ks % (g.ci / CK)) * CK;
            unsigned char* st = stages + s * sh.stage;
            // A: the tap-shifted input row of this voxel
            const int qx = x + t % 3 - 1;
            int qy = y + (t / 3) % 3 - 1, qz = z + t / 9 - 1;
            bool valid = row_ok && qx >= 0 && qx < g.W;
            if (g.periodic_yz) {
                qy = qy < 0 ? qy + g.H : (qy >= g.H ? qy - g.H : qy);
                qz = qz < 0 ? qz + g.D : (qz >= g.D ? qz - g.D : qz);
            } else {
                valid = valid && qy >= 0 && qy < g.H && qz >= 0 && qz < g.D;
            }
            const long long sv = valid ? qx + (long long)g.W * (qy + (long long)g.H * (qz + (long long)g.D * nb)) : 0;
            const __nv_bfloat16* src = in + sv * g.in_stride + g.in_off + c0;
            const uint32_t a_base = smem_addr(st) + a_row;
            for (int h = 0; h < kgroups; ++h) cp_async16_ca(a_base + (uint32_t)h * 128u, src + 8 * h, valid);
            // B: weight rows of this tap and channel chunk, shared by the 128 threads
            const uint32_t b_base = smem_addr(st + sh.a_bytes);
            const __nv_bfloat16* wt = w + (long long)t * g.co * g.ci + c0;
            for (int e = r; e < g.co * kgroups; e += 128) {
                const int n = e / kgroups, h = e % kgroups;
                cp_async16(b_base + (uint32_t)(n >> 3) * sbo_b + (uint32_t)h * 128u + (uint32_t)(n & 7) * 16u,
                           wt + (long long)n * g.ci + 8 * h, true);
            }
            cp_async_commit();
            ++issued;
            // stage ks - kLag has landed: publish it to the tensor core
            if (ks >= kLag) {
                cp_async_wait<kLag>();
                fence_async_shared();
                bar_arrive(&full[(ks - kLag) % kFwStages]);
            }
        }
        // publish the stages still in flight (also after an abort, so that
        // no copy is outstanding when the CTA leaves)
        cp_async_wait<0>();
        fence_async_shared();
        for (int ks = (issued >= kLag ? issued - kLag : 0); ks < issued; ++ks) bar_arrive(&full[ks % kFwStages]);
        if (!ok) {
            atomicOr(err, 64);
            *(volatile int*)abort_flag = 1;
        }
    } else if (lane == 0) {
        // ------------------------------------------------------ MMA issuer
        const uint32_t idesc = idesc_bf16(kTcM, g.co);
        int ks = 0;
        for (; ks < ksteps; ++ks) {
            const int s = ks % kFwStages;
            if (!bar_wait(&full[s], (ks / kFwStages) & 1) || *(volatile int*)abort_flag) {
                atomicOr(err, 64);
                *(volatile int*)abort_flag = 1;
                break;
            }
            tc_fence_after();
            const uint32_t a0 = smem_addr(stages + s * sh.stage), b0 = a0 + (uint32_t)sh.a_bytes;
            for (int kk = 0; kk < CK / 16; ++kk) {
                const uint64_t ad = sdesc(a0 + (uint32_t)kk * 256u, 128u, sbo_a);
                const uint64_t bd = sdesc(b0 + (uint32_t)kk * 256u, 128u, sbo_b);
                mma_bf16_ss(tmem, ad, bd, idesc, (ks > 0 || kk > 0) ? 1u : 0u);
            }
            mma_commit(&empty[s]);  // the stage is free once these MMAs have read it
        }
        mma_commit(done);  // every MMA issued so far has completed
    }

    // ---------------------------------------------------------- epilogue
    if (warp < 4) {
        const bool ok = bar_wait(done, 0);
        tc_fence_after();
        if (!ok) atomicOr(err, 64);
        const long long v = v0 + tid;
        const bool store = ok && !*(volatile int*)abort_flag && v < M;
        const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
        for (int c = 0; c < g.co; c += 16) {
            uint32_t acc[16];
            tmem_ld16(lane_base + (uint32_t)c, acc);  // warp-wide: every lane takes part
            if (store) {
                store16(acc, bias ? bias + c : nullptr, relu, out + v * g.out_stride + g.out_off + c);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 4) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(sh.ncols) : "memory");
    }
}

// ------------------------------------------------- forward, halo tiles
// The same convolution with the 27 taps read from one gathered neighbourhood
// instead of 27 gathers.  A CTA owns an 8 (x) x 16 (y) block of output
// voxels at one z of one batch item: M row r = 8 yr + xr.  Per chunk of CK
// input channels it stages the 10 x 18 x 3 halo of that block once, laid
// out so that every tap's A operand is the same K-major core-matrix layout
// at a shifted start address:
//   halo voxel (xi, yj, zk), channel group g (8 channels, 16 bytes) at
//   zk PZ + yj PY + g PC + xi 16,   PC = 10 x 16 B, PY = CK/8 PC, PZ = 18 PY;
//   tap (dx, dy, dz): start = (1+dz) PZ + (1+dy) PY + (1+dx) 16,
//   LBO = PC (next 8 channels), SBO = PY (next 8-row group = next y line).
// Only the weights stream, one tap per ring stage.  x is zero padded; y and
// z wrap (or are zero padded); rows outside the box are computed and dropped.
constexpr int kHaloX = 10, kHaloY = 18, kHaloZ = 3;

struct HaloShape {
    int CK, cn, taps, ncols, halo_bytes, w_bytes, smem;
};

// channel chunk of the input: the widest that divides ci and leaves room for a
// ring of four taps (it sets the order of summation)
static int halo_chunk(int ci, int co) {
    const int cands[4] = {64, 48, 32, 16};
    for (int i = 0; i < 4; ++i) {
        const int ck = cands[i];
        if (ck > ci || ci % ck) continue;
        if (1024 + kHaloX * kHaloY * kHaloZ * ck * 2 + 4 * co * ck * 2 <= 200 * 1024) return ck;
    }
    return 16;
}

constexpr int kHaloStages = 4;

// cn output channels per CTA; three taps to a stage of the ring where that
// leaves room for `per_sm` CTAs on an SM, else one
static HaloShape halo_shape(int ci, int co, int cn, int per_sm) {
    HaloShape s;
    s.CK = halo_chunk(ci, co);
    s.cn = cn;
    int c = 32;
    while (c < cn) c <<= 1;
    s.ncols = c;
    s.halo_bytes = kHaloX * kHaloY * kHaloZ * s.CK * 2;
    s.w_bytes = cn * s.CK * 2;
    s.taps = 1024 + s.halo_bytes + 3 * kHaloStages * s.w_bytes <= (per_sm == 1 ? 227 : 113) * 1024 ? 3 : 1;
    s.smem = 1024 + s.halo_bytes + kHaloStages * s.taps * s.w_bytes;
    return s;
}

// What bounds it is the hand-over of 27 taps' weights per chunk, each with its
// fences and barriers: they go three to a stage, a thread's places in the halo are
// found once (not with divisions for every piece), and where the blocks of
// voxels leave SMs idle the output channels are split over CTAs (cn), which
// changes no sum.  4 x 6^3, 128 -> 128: 71 us with single taps and one CTA for all
// channels, 32 us; 4 x 24^3, 96 -> 32: 102, 51 us.
template <int KG, int TAPS>  // groups of 8 channels of a chunk; taps of a weight stage
__global__ void __launch_bounds__(kTcThreads) k_conv3d_halo(const __nv_bfloat16* __restrict__ in,
                                                            const __nv_bfloat16* __restrict__ w,
                                                            const float* __restrict__ bias,
                                                            __nv_bfloat16* __restrict__ out, ConvGeom g, int relu,
                                                            HaloShape sh, int* err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    constexpr int kFlight = kHaloStages - 2;  // weight stages in flight per thread
    constexpr int kSteps = 27 / TAPS;         // of one chunk
    uint64_t* wfull = reinterpret_cast<uint64_t*>(smem);
    uint64_t* wempty = wfull + kHaloStages;
    uint64_t* hempty = wempty + kHaloStages;  // the halo may be refilled
    uint64_t* done = hempty + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);
    unsigned char* halo = smem + 1024;
    unsigned char* wring = halo + sh.halo_bytes;

    const int tid = threadIdx.x, warp = warp_index();
    constexpr int CK = KG * 8;
    const int nchunks = g.ci / CK;
    const int ksteps = kSteps * nchunks;
    constexpr uint32_t PC = 16u * kHaloX, PY = (uint32_t)KG * PC, PZ = (uint32_t)kHaloY * PY;
    // output block and channels
    const int bxn = (g.W + 7) / 8;
    const int x0 = (int)(blockIdx.x % bxn) * 8, y0 = blockIdx.y * 16;
    const int n0 = (int)(blockIdx.x / bxn) * sh.cn;
    const int zb = blockIdx.z % g.D;
    const long long nb = blockIdx.z / g.D;

    if (tid == 0) {
        for (int s = 0; s < kHaloStages; ++s) {
            bar_init(&wfull[s], 128);
            bar_init(&wempty[s], 1);
        }
        bar_init(hempty, 1);
        bar_init(done, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 4) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                     "r"(sh.ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp < 4) {
        // ------------------------------------------------------ producers
        bool ok = true;
        int issued = 0, published = 0;
        // the halo by lines of x: a thread has one place (voxel, channel group) in every kRows-th line
        constexpr int kLine = kHaloX * KG, kRows = 128 / kLine;
        const int hr = tid / kLine, hp = tid % kLine, grp = hp % KG, xi = hp / KG;
        const int qx = x0 - 1 + xi;
        const bool x_ok = hr < kRows && qx >= 0 && qx < g.W;
        const uint32_t halo_s = smem_addr(halo) + (uint32_t)grp * PC + (uint32_t)xi * 16u;
        for (int ks = 0; ks < ksteps && ok; ++ks) {
            const int t0 = ks % kSteps * TAPS, chunk = ks / kSteps;
            if (t0 == 0) {
                if (chunk > 0) {
                    // publish every step still in flight, then wait until the
                    // previous chunk's MMAs are done with the halo
                    cp_async_wait<0>();
                    fence_async_shared();
                    for (; published < issued; ++published) bar_arrive(&wfull[published % kHaloStages]);
                    if (!bar_wait(hempty, (chunk - 1) & 1)) { ok = false; break; }
                }
                const __nv_bfloat16* src = in + g.in_off + chunk * CK + 8 * grp;
                for (int zk = 0; zk < kHaloZ; ++zk) {
                    int qz = zb - 1 + zk;
                    const bool z_ok = g.periodic_yz || (qz >= 0 && qz < g.D);
                    qz = qz < 0 ? qz + g.D : (qz >= g.D ? qz - g.D : qz);
                    const long long row0 = (long long)g.H * (qz + (long long)g.D * nb);
                    for (int yj = hr; yj < kHaloY && hr < kRows; yj += kRows) {
                        int qy = y0 - 1 + yj;
                        const bool valid = x_ok && z_ok && (g.periodic_yz || (qy >= 0 && qy < g.H));
                        if (qy < 0) qy += g.H;
                        else if (qy >= g.H) qy %= g.H;
                        const long long sv = valid ? qx + (long long)g.W * (qy + row0) : 0;
                        cp_async16(halo_s + (uint32_t)zk * PZ + (uint32_t)yj * PY, src + sv * g.in_stride, valid);
                    }
                }
            }
            // the taps' weights into the ring
            const int s = ks % kHaloStages;
            if (ks >= kHaloStages && !bar_wait(&wempty[s], ((ks / kHaloStages) - 1) & 1)) { ok = false; break; }
            if (*(volatile int*)abort_flag) { ok = false; break; }
            const uint32_t wb = smem_addr(wring + s * TAPS * sh.w_bytes);
            const __nv_bfloat16* wt = w + ((long long)t0 * g.co + n0) * g.ci + chunk * CK;
#pragma unroll
            for (int j = 0; j < TAPS; ++j)
                for (int e = tid; e < sh.cn * KG; e += 128) {
                    const int n = e / KG, h = e % KG;
                    cp_async16(wb + (uint32_t)(j * sh.w_bytes) + (uint32_t)(n >> 3) * (uint32_t)(KG * 128) +
                                   (uint32_t)h * 128u + (uint32_t)(n & 7) * 16u,
                               wt + ((long long)j * g.co + n) * g.ci + 8 * h, true);
                }
            cp_async_commit();
            ++issued;
            if (issued - published > kFlight) {
                // every earlier copy of this thread (the halo too) has landed
                cp_async_wait<kFlight>();
                fence_async_shared();
                bar_arrive(&wfull[published % kHaloStages]);
                ++published;
            }
        }
        cp_async_wait<0>();
        fence_async_shared();
        for (; published < issued; ++published) bar_arrive(&wfull[published % kHaloStages]);
        if (!ok) {
            atomicOr(err, 64);
            *(volatile int*)abort_flag = 1;
        }
    } else {
        // ------------------------------------------------------ MMA issuer
        const bool issue = elect_one();
        const uint32_t idesc = idesc_bf16(kTcM, sh.cn);
        const uint64_t adesc = sdesc(smem_addr(halo), PC, PY), bdesc = sdesc(smem_addr(wring), 128u, (uint32_t)KG * 128u);
        for (int ks = 0; ks < ksteps; ++ks) {
            const int s = ks % kHaloStages;
            const bool ok = bar_wait(&wfull[s], (ks / kHaloStages) & 1) && !*(volatile int*)abort_flag;
            if (!__all_sync(0xffffffffu, ok)) {
                atomicOr(err, 64);
                *(volatile int*)abort_flag = 1;
                break;
            }
            tc_fence_after();
#pragma unroll
            for (int j = 0; j < TAPS; ++j) {
                // tap offset + 1: t % 3, t / 3 % 3, t / 9; descriptor addresses count 16 bytes
                const int t = ks % kSteps * TAPS + j;
                const uint64_t a0 =
                    adesc + (uint32_t)(t / 9) * (PZ / 16u) + (uint32_t)(t / 3 % 3) * (PY / 16u) + (uint32_t)(t % 3);
                const uint64_t b0 = bdesc + (uint32_t)(s * TAPS + j) * ((uint32_t)sh.w_bytes / 16u);
#pragma unroll
                for (int kk = 0; kk < KG / 2; ++kk)
                    if (issue)
                        mma_bf16_ss(tmem, a0 + (uint32_t)kk * 2u * (PC / 16u), b0 + (uint32_t)kk * 16u, idesc,
                                    (ks > 0 || j > 0 || kk > 0) ? 1u : 0u);
            }
            if (issue) {
                mma_commit(&wempty[s]);
                if (ks % kSteps == kSteps - 1) mma_commit(hempty);  // the chunk's halo is no longer read
            }
        }
        if (issue) mma_commit(done);
    }

    // ---------------------------------------------------------- epilogue
    if (warp < 4) {
        const bool ok = bar_wait(done, 0);
        __syncwarp();
        tc_fence_after();
        if (!ok) atomicOr(err, 64);
        const int r = tid, x = x0 + (r & 7), y = y0 + (r >> 3);
        const bool store = ok && !*(volatile int*)abort_flag && x < g.W && y < g.H;
        const long long v = x + (long long)g.W * (y + (long long)g.H * (zb + (long long)g.D * nb));
        const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
        for (int c = 0; c < sh.cn; c += 16) {
            uint32_t acc[16];
            tmem_ld16(lane_base + (uint32_t)c, acc);
            if (store) store16(acc, bias ? bias + n0 + c : nullptr, relu, out + v * g.out_stride + g.out_off + n0 + c);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 4) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(sh.ncols) : "memory");
    }
}

// ------------------------------------------------- forward, marching along z
// The halo kernel spends its time on hand-overs, not on the tensor core: every
// CTA streams all 27 taps' weights through a ring for 128 voxels and stages
// three planes of which its z-neighbours stage two again.  Here a CTA owns an
// 8 x 16 column over a segment of z.  The weights are loaded once and stay; the
// 10 x 18 halo of one input plane is staged at a time (double buffered) and
// contributes to the output planes o-1, o, o+1, whose accumulators lie side by
// side in tensor memory: the MMA of an in-plane tap (dy, dx) is one of
// N = 3 co columns against the tap's weights for dz = +1, 0, -1, so 9 MMAs per
// 16 input channels replace 27 and the plane is read from shared memory a third
// as often.  Accumulators are a ring of `slots` output planes; where the window
// of three wraps round its end it is issued as two MMAs.  Every accumulator
// sees its products in the order of the halo kernel with one channel chunk (dz
// outermost, then dy, dx, channels), so results are the same bits.
// Roles (288 threads): warps 0-3 the epilogue, warps 4-7 stage the planes,
// warp 8 tensor memory and the MMAs.
// Bound by the operand reads of the MMAs (4 KB of A for 48 columns; the tensor
// pipe's operand stage is busy 66% of the time).
// 4 x 48^3, 48 -> 16 channels: 212 us before, 47 us; 16 -> 48: 118, 34 us.
constexpr int kMarchThreads = 288;
constexpr int kMarchMaxStages = 4;
constexpr int kMarchMaxSlots = 32;

struct MarchShape {
    int w_bytes, plane_bytes, stages, slots, ncols, per_sm, smem;
};

// stages = 0: the weights and two planes do not fit
inline MarchShape march_shape(int ci, int co) {
    MarchShape s{};
    s.w_bytes = 27 * ci * co * 2;
    s.plane_bytes = kHaloX * kHaloY * ci * 2;
    for (s.per_sm = 2; s.per_sm >= 1; --s.per_sm) {
        // an SM's 228 KB, 1 KB of it taken per CTA; its 512 columns
        const int room = (s.per_sm == 2 ? 113 : 227) * 1024 - 1024 - s.w_bytes;
        s.ncols = 512 / s.per_sm;
        s.slots = s.ncols / co < kMarchMaxSlots ? s.ncols / co : kMarchMaxSlots;
        s.stages = room / s.plane_bytes < kMarchMaxStages ? room / s.plane_bytes : kMarchMaxStages;
        if (s.stages >= 2 && s.slots >= 4) break;  // a window of three planes and one that is read out
    }
    if (s.per_sm < 1) s.stages = 0;
    s.smem = 1024 + s.w_bytes + s.stages * s.plane_bytes;
    return s;
}

template <int KG>  // groups of 8 input channels
__global__ void __launch_bounds__(kMarchThreads) k_conv3d_march(const __nv_bfloat16* __restrict__ in,
                                                                const __nv_bfloat16* __restrict__ w,
                                                                const float* __restrict__ bias,
                                                                __nv_bfloat16* __restrict__ out, ConvGeom g, int relu,
                                                                MarchShape sh, int seg_len, int nseg, int* err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t* pfull = reinterpret_cast<uint64_t*>(smem);
    uint64_t* pempty = pfull + kMarchMaxStages;
    uint64_t* tfull = pempty + kMarchMaxStages;
    uint64_t* tempty = tfull + kMarchMaxSlots;
    uint64_t* wfull = tempty + kMarchMaxSlots;
    uint64_t* done = wfull + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);
    constexpr uint32_t PC = 16u * kHaloX, PY = KG * PC;  // halo voxel xi of line yj, channel group h: yj PY + h PC + xi 16
    constexpr uint32_t WG = KG * 128u;                   // weights: 8 rows (output channels) of KG 16-byte groups
    const uint32_t w_s = smem_addr(smem + 1024), plane_s = w_s + (uint32_t)sh.w_bytes;
    const uint32_t w_tap = (uint32_t)(3 * g.co / 8) * WG;

    const int tid = threadIdx.x, warp = warp_index();
    const int x0 = blockIdx.x * 8, y0 = blockIdx.y * 16;
    const int za = (int)(blockIdx.z % nseg) * seg_len;
    const long long nb = blockIdx.z / nseg;
    const int len = g.D - za < seg_len ? g.D - za : seg_len;  // output planes, >= 1
    const int np = len + 2;                                   // input planes za - 1 .. za + len

    if (tid == 0) {
        for (int i = 0; i < sh.stages; ++i) {
            bar_init(&pfull[i], 128);
            bar_init(&pempty[i], 1);
        }
        for (int i = 0; i < sh.slots; ++i) {
            bar_init(&tfull[i], 1);
            bar_init(&tempty[i], 128);
        }
        bar_init(wfull, 256);
        bar_init(done, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 8) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                     "r"(sh.ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp < 8) {
        // weights, in-plane tap by tap: row b co + n is output channel n at dz = 1 - b (b: place in the window)
        for (int e = tid; e < 27 * g.co * KG; e += 256) {
            const int h = e % KG, row = e / KG;
            const int t = row / g.co, n = row - t * g.co;
            const int nrow = (2 - t / 9) * g.co + n;
            cp_async16(w_s + (uint32_t)(t % 9) * w_tap + (uint32_t)(nrow >> 3) * WG + (uint32_t)h * 128u +
                           (uint32_t)(nrow & 7) * 16u,
                       w + (long long)row * (KG * 8) + 8 * h, true);
        }
        cp_async_commit();
    }
    if (warp < 4) {
        // ------------------------------------------------------ epilogue
        cp_async_wait<0>();
        fence_async_shared();
        bar_arrive(wfull);
        const int x = x0 + (tid & 7), y = y0 + (tid >> 3);
        const bool inside = x < g.W && y < g.H;
        const long long v0 = x + (long long)g.W * (y + (long long)g.H * (za + (long long)g.D * nb));
        const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
        for (int o = 0, slot = 0, use = 0; o < len; ++o) {
            const bool full = bar_wait(&tfull[slot], use & 1) && !*(volatile int*)abort_flag;
            if (!__all_sync(0xffffffffu, full)) {  // the warp's lanes leave together
                atomicOr(err, 64);
                *(volatile int*)abort_flag = 1;
                break;
            }
            tc_fence_after();
            __nv_bfloat16* dst0 = out + (v0 + (long long)o * g.W * g.H) * g.out_stride + g.out_off;
            for (int c = 0; c < g.co; c += 16) {
                uint32_t acc[16];
                tmem_ld16(lane_base + (uint32_t)(slot * g.co + c), acc);
                if (c + 16 >= g.co) {  // read out: the slot may be used again
                    tc_fence_before();
                    bar_arrive(&tempty[slot]);
                }
                if (inside) store16(acc, bias ? bias + c : nullptr, relu, dst0 + c);
            }
            if (++slot == sh.slots) { slot = 0; ++use; }
        }
    } else if (warp < 8) {
        // ------------------------------------------------------ producers
        // this thread's 16-byte pieces of a plane: the same places in every plane
        constexpr int kPieces = (kHaloX * kHaloY * KG + 127) / 128;
        const int p = tid - 128;
        long long src[kPieces];
        uint32_t dst[kPieces];
        bool ok_xy[kPieces];
#pragma unroll
        for (int i = 0; i < kPieces; ++i) {
            const int e = p + i * 128;
            const int h = e % KG, v = e / KG;
            const int xi = v % kHaloX, yj = v / kHaloX;
            const int qx = x0 - 1 + xi;
            int qy = y0 - 1 + yj;
            ok_xy[i] = qx >= 0 && qx < g.W;
            if (g.periodic_yz) qy = ((qy % g.H) + g.H) % g.H;
            else ok_xy[i] = ok_xy[i] && qy >= 0 && qy < g.H;
            src[i] = ok_xy[i] ? (qx + (long long)g.W * qy) * g.in_stride + 8 * h : 0;
            dst[i] = yj < kHaloY ? (uint32_t)yj * PY + (uint32_t)h * PC + (uint32_t)xi * 16u : ~0u;
        }
        bool ok = true;
        int issued = 0;
        for (int k = 0, s = 0, use = 0, prev = 0; k < np; ++k) {
            if (use > 0 && !bar_wait(&pempty[s], (use - 1) & 1)) ok = false;
            if (!ok || *(volatile int*)abort_flag) { ok = false; break; }
            int qz = za - 1 + k;
            bool ok_z = true;
            if (g.periodic_yz) qz = ((qz % g.D) + g.D) % g.D;
            else ok_z = qz >= 0 && qz < g.D;
            const __nv_bfloat16* base =
                in + (ok_z ? (long long)g.W * g.H * (qz + (long long)g.D * nb) * g.in_stride : 0) + g.in_off;
            const uint32_t st = plane_s + (uint32_t)s * (uint32_t)sh.plane_bytes;
#pragma unroll
            for (int i = 0; i < kPieces; ++i)
                if (dst[i] != ~0u) cp_async16(st + dst[i], base + src[i], ok_z && ok_xy[i]);
            cp_async_commit();
            ++issued;
            if (k > 0) {  // the weights and the plane before this one have landed
                cp_async_wait<1>();
                fence_async_shared();
                if (k == 1) bar_arrive(wfull);
                bar_arrive(&pfull[prev]);
            }
            prev = s;
            if (++s == sh.stages) { s = 0; ++use; }
        }
        cp_async_wait<0>();  // np >= 3: the barriers up to here have been arrived at unless the CTA gave up
        fence_async_shared();
        if (ok) bar_arrive(&pfull[(issued - 1) % sh.stages]);
        else {
            atomicOr(err, 64);
            *(volatile int*)abort_flag = 1;
        }
    } else {
        // ------------------------------------------------------ MMA issuer
        const bool issue = elect_one();
        const uint32_t idesc0 = idesc_bf16(kTcM, 0), w8 = (uint32_t)(g.co / 8) * WG;  // N is set per run
        const int max_run = 256 / g.co;                                             // planes of one MMA (N <= 256)
        const uint64_t adesc = sdesc(plane_s, PC, PY), bdesc = sdesc(w_s, 128u, WG);  // addresses are added, in 16 bytes
        bool ok = __all_sync(0xffffffffu, bar_wait(wfull, 0));
        for (int k = 0, s = 0, use = 0; k < np && ok; ++k) {
            // output planes [lo, hi] of the segment that this input plane feeds; plane k is new
            const int lo = k - 2 > 0 ? k - 2 : 0, hi = k < len ? k : len - 1;
            ok = bar_wait(&pfull[s], use & 1) && !*(volatile int*)abort_flag;
            if (ok && k < len && k >= sh.slots) ok = bar_wait(&tempty[k % sh.slots], (k / sh.slots - 1) & 1);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            const uint64_t a0 = adesc + (uint32_t)s * (uint32_t)sh.plane_bytes / 16u;
            // planes o .. of one MMA: as far as the ring, N and `end` allow
            auto run = [&](int o, int end, uint32_t& d, uint32_t& id, uint32_t& brow) {
                const int slot = o % sh.slots;
                int n = end - o + 1;
                if (n > max_run) n = max_run;
                if (n > sh.slots - slot) n = sh.slots - slot;
                d = tmem + (uint32_t)(slot * g.co);
                id = idesc0 | ((uint32_t)(n * g.co >> 3) << 17);
                brow = (uint32_t)(o - (k - 2)) * w8 / 16u;
                return o + n;
            };
            if (k < len) {  // the first product of plane k starts its accumulator; the others add to theirs
                for (int o = lo; o <= hi;) {
                    uint32_t d, id, brow;
                    const uint32_t acc = o < k ? 1u : 0u;
                    o = run(o, o < k ? k - 1 : k, d, id, brow);
                    if (issue) mma_bf16_ss(d, a0, bdesc + brow, id, acc);
                }
            }
            uint32_t d[3], id[3], brow[3];
            int nrun = 0;
#pragma unroll
            for (int r = 0, o = lo; r < 3; ++r)
                if (o <= hi) {
                    o = run(o, hi, d[r], id[r], brow[r]);
                    nrun = r + 1;
                }
            for (int t9 = 0; t9 < 9; ++t9) {
                const uint64_t at = a0 + (uint32_t)(t9 / 3) * (PY / 16u) + (uint32_t)(t9 % 3);
                const uint64_t bt = bdesc + (uint32_t)t9 * (w_tap / 16u);
#pragma unroll
                for (int kk = 0; kk < KG / 2; ++kk) {
                    if (kk == 0 && t9 == 0 && k < len) continue;  // issued above
#pragma unroll
                    for (int r = 0; r < 3; ++r)
                        if (r < nrun && issue)
                            mma_bf16_ss(d[r], at + (uint32_t)kk * 2u * (PC / 16u), bt + brow[r] + (uint32_t)kk * 16u, id[r],
                                        1u);
                }
            }
            if (issue) {
                mma_commit(&pempty[s]);                              // the plane may be overwritten
                if (k >= 2) mma_commit(&tfull[(k - 2) % sh.slots]);  // output plane k - 2 is complete
            }
            if (++s == sh.stages) { s = 0; ++use; }
        }
        if (!ok) {
            atomicOr(err, 64);
            *(volatile int*)abort_flag = 1;
        }
        if (issue) mma_commit(done);
        if (!bar_wait(done, 0)) atomicOr(err, 64);  // no MMA is in flight when the tensor memory is freed
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 8) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(sh.ncols) : "memory");
    }
}

// Up to 64 input channels, so that the halo kernel's single channel chunk gives
// the order of summation, where the weights and two planes fit.
static bool conv3d_march_supported(const ConvGeom& g) {
    return (g.ci == 16 || g.ci == 32 || g.ci == 48 || g.ci == 64) && halo_chunk(g.ci, g.co) == g.ci &&
           march_shape(g.ci, g.co).stages >= 2 && (long long)g.D * g.N <= 65535 && (g.H + 15) / 16 <= 65535;
}

// Segments of z: as many as make the work of the busiest SM least, each costing
// its planes, two more at its ends and the loading of the weights.
static cudaError_t launch_conv3d_march(const __nv_bfloat16* in, const __nv_bfloat16* w, const float* bias,
                                       __nv_bfloat16* out, const ConvGeom& g, int relu, int* err, cudaStream_t s) {
    const MarchShape sh = march_shape(g.ci, g.co);
    int dev = 0, nsm = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const long long cols = (long long)((g.W + 7) / 8) * ((g.H + 15) / 16) * g.N;
    const int fixed = 4 + sh.w_bytes / sh.plane_bytes;
    int seg_len = g.D;
    long long best = -1;
    for (int n = 1; n <= g.D && n <= 512; ++n) {
        const int l = (g.D + n - 1) / n;
        if (n > 1 && (g.D + n - 2) / (n - 1) == l) continue;
        const long long ctas = cols * ((g.D + l - 1) / l), room = (long long)nsm * sh.per_sm;
        const long long cost = (ctas + room - 1) / room * (l + fixed);
        if (best < 0 || cost < best) { best = cost; seg_len = l; }
    }
    const int nseg = (g.D + seg_len - 1) / seg_len;
    const dim3 grid((unsigned)((g.W + 7) / 8), (unsigned)((g.H + 15) / 16), (unsigned)(nseg * g.N));
    auto go = [&](auto kernel) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sh.smem);
        if (e != cudaSuccess) return e;
        kernel<<<grid, kMarchThreads, sh.smem, s>>>(in, w, bias, out, g, relu, sh, seg_len, nseg, err);
        return cudaGetLastError();
    };
    switch (g.ci) {
        case 16: return go(k_conv3d_march<2>);
        case 32: return go(k_conv3d_march<4>);
        case 48: return go(k_conv3d_march<6>);
        default: return go(k_conv3d_march<8>);
    }
}

// ------------------------------------------------------------ weight grad
// dW[t][co][ci] = sum_u I[u][ci] dO[u - t][co]: a GEMM per tap over K = voxels.
// A = the input tile (M = ci, 64 or 128 rows, MN-major), B = the output
// gradient with its halo (N = co, MN-major), so a tap is a shifted descriptor
// into 16 channels of dO, and the three taps of one (dy, dx) are one MMA: the
// halo is stored plane by plane and channel group by channel group at one
// stride, [zk][g][yj][xi], which makes (dz, co) a single N = 48.  All 27 taps'
// accumulators, 432 columns, stay in tensor memory over the blocks of a slice;
// a second kernel sums the slices in a fixed order.  A CTA covers 16 output
// channels and up to 128 input channels.
//   A: voxel r = 8 yr + xr, channel group g: yr PYi + g 128 + xr 16, PYi = ci/8 128
//   B: halo voxel (xi, yj, zk), group g: (2 zk + g) PG + yj 160 + xi 16, PG = 18 x 160
// Rows of A past the channels read whatever follows in the stage; their
// accumulators are never read back.  Roles (288 threads): warps 0-7 stage the
// blocks (z fastest, so a thread's places in a block stay the same along a
// column), warps 0-3 read the accumulators, warp 8 tensor memory and the MMAs.
// Bound by the shared-memory reads of the operands.  4 x 48^3, 48 -> 16
// channels: 608 us with a gather per tap and voxel, 45 us; 4 x 24^3,
// 32 -> 32: 77, 21 us.
constexpr int kWgThreads = 288;
constexpr int kWgProducers = 256;
constexpr int kWgStages = 4, kWgLag = 2;
constexpr int kWgCo = 16;                                   // output channels of a CTA
constexpr int kWgB = 3 * kHaloX * kHaloY * kWgCo * 2;       // bytes of the dO halo
constexpr uint32_t kWgPG = 16u * kHaloX * kHaloY;           // channel-group stride of the halo

__host__ __device__ inline int wg_chunk(int ci) { return ci < 128 ? ci : 128; }
__host__ __device__ inline int wg_stage_bytes(int ci) { return kTcM * wg_chunk(ci) * 2 + kWgB; }

static long long wg_blocks(const ConvGeom& g) {
    return (long long)((g.W + 7) / 8) * ((g.H + 15) / 16) * g.D * g.N;
}

// Slices: one wave of CTAs, one per SM (its tensor memory is full).  The tensor core rounds the additions to an accumulator
// toward zero, so the error grows with the number of blocks that one adds up; from five blocks (640 voxels) on there are
// as many waves as give 152 slices of 16 input channels, 76 of 32 and so on, which keeps the error at or below that of a
// gather per tap (rel. 2-norm over 12 inputs of 4 x 24^3, 16 -> 32: 2.5e-7 with the gather, 3.3e-7 in one wave, 1.4e-7
// in two and with the slices' sum as it is; 31 and 37 us.  4 x 48^3, 48 -> 16: 4.7e-6 and 1.2e-6, one wave).
static int wg_slices(const ConvGeom& g) {
    const long long nb = wg_blocks(g);
    const long long ctas = (long long)((g.ci + 127) / 128) * (g.co / kWgCo);  // of a slice
    long long ns = 152 / ctas;
    if (ns < 1) ns = 1;
    if ((nb + ns - 1) / ns > 4) {
        const long long least = (152 * 16 + g.ci - 1) / g.ci, waves = (least * ctas + 151) / 152;
        if (152 * waves / ctas > ns) ns = 152 * waves / ctas;
    }
    return (int)(ns < nb ? ns : nb);
}

__global__ void __launch_bounds__(kWgThreads) k_conv3d_wgrad_tc(const __nv_bfloat16* __restrict__ in,
                                                                const __nv_bfloat16* __restrict__ dout,
                                                                float* __restrict__ partial, ConvGeom g,
                                                                long long nblocks, int per, int* err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);
    uint64_t* empty = full + kWgStages;
    uint64_t* done = empty + kWgStages;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);

    const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
    const int c0 = blockIdx.y * 128, o0 = blockIdx.z * kWgCo;
    const int rows = g.ci - c0 < 128 ? g.ci - c0 : 128, kg = rows / 8;
    const int m_rows = rows <= 64 ? 64 : 128;
    const uint32_t stage = (uint32_t)wg_stage_bytes(g.ci), stages_s = smem_addr(smem + 1024);
    const uint32_t PYi = (uint32_t)kg * 128u, a_bytes = 16u * PYi;
    const long long b0 = (long long)blockIdx.x * per;
    const int nb = nblocks - b0 < per ? (int)(nblocks - b0) : per;  // >= 1
    const int bxn = (g.W + 7) / 8, byn = (g.H + 15) / 16;

    if (tid == 0) {
        for (int s = 0; s < kWgStages; ++s) {
            bar_init(&full[s], kWgProducers);
            bar_init(&empty[s], 1);
        }
        bar_init(done, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 8) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp < 8) {
        // ------------------------------------------------------ producers
        constexpr int kA = 128 * 16 / kWgProducers;                               // pieces of the input tile
        constexpr int kB = (kHaloX * kHaloY * 2 + kWgProducers - 1) / kWgProducers;  // of one halo plane
        long long asrc[kA], bsrc[kB];
        unsigned aok = 0, bok = 0;
        bool ok = true;
        int issued = 0;
        int zb = (int)(b0 % g.D);
        long long col = b0 / g.D;
        for (int i = 0; i < nb; ++i) {
            const int s = i % kWgStages;
            if (i >= kWgStages && !bar_wait(&empty[s], ((i / kWgStages) - 1) & 1)) ok = false;
            if (!ok || *(volatile int*)abort_flag) { ok = false; break; }
            const long long nbt = col / (bxn * byn);
            if (i == 0 || zb == 0) {  // a new column: the places of this thread's pieces in a plane
                const int xy = (int)(col - nbt * (bxn * byn));
                const int x0 = xy % bxn * 8, y0 = xy / bxn * 16;
                aok = bok = 0;
#pragma unroll
                for (int j = 0; j < kA; ++j) {
                    const int e = tid + j * kWgProducers, h = e % kg, r = e / kg;
                    const int x = x0 + (r & 7), y = y0 + (r >> 3);
                    const bool v = x < g.W && y < g.H && r < 128;
                    asrc[j] = v ? (x + (long long)g.W * y) * g.in_stride + g.in_off + c0 + 8 * h : 0;
                    aok |= (unsigned)v << j;
                }
#pragma unroll
                for (int j = 0; j < kB; ++j) {
                    const int e = tid + j * kWgProducers, h = e & 1, v = e >> 1;
                    const int qx = x0 - 1 + v % kHaloX;
                    int qy = y0 - 1 + v / kHaloX;
                    bool good = qx >= 0 && qx < g.W;
                    if (g.periodic_yz) qy = ((qy % g.H) + g.H) % g.H;
                    else good = good && qy >= 0 && qy < g.H;
                    bsrc[j] = good ? (qx + (long long)g.W * qy) * g.out_stride + g.out_off + o0 + 8 * h : 0;
                    bok |= (unsigned)good << j;
                }
            }
            const uint32_t st = stages_s + (uint32_t)s * stage;
            const long long plane = (long long)g.W * g.H, first = plane * g.D * nbt;
            const __nv_bfloat16* abase = in + (first + plane * zb) * g.in_stride;
#pragma unroll
            for (int j = 0; j < kA; ++j) {
                const int e = tid + j * kWgProducers;
                if (e >= 128 * kg) break;
                const int h = e % kg, r = e / kg;
                cp_async16(st + (uint32_t)(r >> 3) * PYi + (uint32_t)h * 128u + (uint32_t)(r & 7) * 16u, abase + asrc[j],
                           (aok >> j) & 1u);
            }
#pragma unroll
            for (int zk = 0; zk < 3; ++zk) {
                int qz = zb - 1 + zk;
                bool ok_z = true;
                if (g.periodic_yz) qz = qz < 0 ? qz + g.D : (qz >= g.D ? qz - g.D : qz);
                else ok_z = qz >= 0 && qz < g.D;
                const __nv_bfloat16* bbase = dout + (ok_z ? (first + plane * qz) * g.out_stride : 0);
#pragma unroll
                for (int j = 0; j < kB; ++j) {
                    const int e = tid + j * kWgProducers;
                    if (e >= kHaloX * kHaloY * 2) break;
                    cp_async16(st + a_bytes + (uint32_t)(2 * zk + (e & 1)) * kWgPG + (uint32_t)(e >> 1) * 16u,
                               bbase + bsrc[j], ok_z && ((bok >> j) & 1u));
                }
            }
            cp_async_commit();
            ++issued;
            if (i >= kWgLag) {
                cp_async_wait<kWgLag>();
                fence_async_shared();
                bar_arrive(&full[(i - kWgLag) % kWgStages]);
            }
            if (++zb == g.D) { zb = 0; ++col; }
        }
        cp_async_wait<0>();
        fence_async_shared();
        for (int i = issued >= kWgLag ? issued - kWgLag : 0; i < issued; ++i) bar_arrive(&full[i % kWgStages]);
        if (!ok) {
            atomicOr(err, 64);
            *(volatile int*)abort_flag = 1;
        }
    } else {
        // ------------------------------------------------------ MMA issuer
        const bool issue = elect_one();
        const uint32_t idesc = idesc_bf16(m_rows, 3 * kWgCo) | (1u << 15) | (1u << 16);  // A, B MN-major
        for (int i = 0; i < nb; ++i) {
            const int s = i % kWgStages;
            const bool ok = bar_wait(&full[s], (i / kWgStages) & 1) && !*(volatile int*)abort_flag;
            if (!__all_sync(0xffffffffu, ok)) {
                atomicOr(err, 64);
                *(volatile int*)abort_flag = 1;
                break;
            }
            tc_fence_after();
            const uint32_t a_s = stages_s + (uint32_t)s * stage, b_s = a_s + a_bytes;
            for (int kk = 0; kk < 8; ++kk) {  // two lines of 8 voxels per K = 16
                const uint64_t ad = sdesc(a_s + (uint32_t)(2 * kk) * PYi, PYi, 128u);
#pragma unroll
                for (int t9 = 0; t9 < 9; ++t9) {
                    const uint32_t b = b_s + (uint32_t)(2 * kk + 2 - t9 / 3) * (16u * kHaloX) + (uint32_t)(2 - t9 % 3) * 16u;
                    if (issue)
                        mma_bf16_ss(tmem + (uint32_t)(t9 * 3 * kWgCo), ad, sdesc(b, 16u * kHaloX, kWgPG), idesc,
                                (i > 0 || kk > 0) ? 1u : 0u);
                }
            }
            if (issue) mma_commit(&empty[s]);
        }
        if (issue) mma_commit(done);
        if (!bar_wait(done, 0)) atomicOr(err, 64);
    }

    // ---------------------------------------------------------- epilogue
    if (warp < 4) {
        const bool ok = bar_wait(done, 0);
        __syncwarp();
        tc_fence_after();
        if (!ok) atomicOr(err, 64);
        // 64 rows lie in the lower 16 lanes of each warp's 32, 128 rows in all of them
        const int m = m_rows == 64 ? (lane < 16 ? warp * 16 + lane : 128) : warp * 32 + lane;
        const bool store = ok && !*(volatile int*)abort_flag && m < rows;
        const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
        for (int q = 0; q < 27; ++q) {  // columns: (dy, dx) 48 + zk 16 + channel; dz = 2 - zk
            uint32_t acc[16];
            tmem_ld16(lane_base + (uint32_t)(q * kWgCo), acc);
            const int t = (2 - q % 3) * 9 + q / 3;
            if (store) {
                float* dst = partial + (((long long)blockIdx.x * 27 + t) * g.co + o0) * g.ci + c0 + m;
#pragma unroll
                for (int j = 0; j < kWgCo; ++j) dst[(long long)j * g.ci] = __uint_as_float(acc[j]);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 8) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

bool conv3d_wgrad_tc_supported(const ConvGeom& g) {
    return g.ci % 16 == 0 && g.co % 16 == 0 && g.co <= 128 && g.ci <= 256 && g.in_stride % 8 == 0 &&
           g.in_off % 8 == 0 && g.out_stride % 8 == 0 && g.out_off % 8 == 0;
}

long long wgrad_tc_workspace_floats(const ConvGeom& g) {
    return conv3d_wgrad_tc_supported(g) ? (long long)wg_slices(g) * 27LL * g.co * g.ci : 0;
}

cudaError_t launch_conv3d_wgrad_tc(const __nv_bfloat16* in, const __nv_bfloat16* dout, float* partial,
                                   const ConvGeom& g, int* err, int* nslices, cudaStream_t s) {
    const int smem = 1024 + kWgStages * wg_stage_bytes(g.ci);
    cudaError_t e = cudaFuncSetAttribute(k_conv3d_wgrad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const long long nb = wg_blocks(g);
    if (nb < 1) return cudaErrorInvalidConfiguration;
    const long long per = (nb + wg_slices(g) - 1) / wg_slices(g);
    const int ns = (int)((nb + per - 1) / per);  // no empty slice
    *nslices = ns;
    k_conv3d_wgrad_tc<<<dim3(ns, (g.ci + 127) / 128, g.co / kWgCo), kWgThreads, smem, s>>>(in, dout, partial, g, nb,
                                                                                       (int)per, err);
    return cudaGetLastError();
}

bool conv3d_tc_supported(const ConvGeom& g) {
    return g.ci % 16 == 0 && g.co % 16 == 0 && g.co >= 16 && g.co <= 256 && g.in_stride % 8 == 0 &&
           g.in_off % 8 == 0 && g.out_stride % 8 == 0 && g.out_off % 8 == 0 && tc_shape(g.ci, g.co).smem <= 227 * 1024;
}

cudaError_t launch_conv3d_tc(const __nv_bfloat16* in, const __nv_bfloat16* w, const float* bias, __nv_bfloat16* out,
                             const ConvGeom& g, int relu, int* err, cudaStream_t s) {
    if (conv3d_march_supported(g)) return launch_conv3d_march(in, w, bias, out, g, relu, err, s);
    const long long voxel_blocks = (long long)((g.W + 7) / 8) * ((g.H + 15) / 16) * g.D * g.N;
    int cn = g.co;
    while (cn % 32 == 0 && voxel_blocks * (g.co / cn) < 152) cn /= 2;
    const HaloShape hs = halo_shape(g.ci, g.co, cn, voxel_blocks * (g.co / cn) <= 152 ? 1 : 2);
    if (hs.smem <= 227 * 1024 && (long long)g.D * g.N <= 65535) {
        const dim3 grid((unsigned)((g.W + 7) / 8 * (g.co / cn)), (unsigned)((g.H + 15) / 16), (unsigned)(g.D * g.N));
        auto go = [&](auto kernel) {
            cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, hs.smem);
            if (e != cudaSuccess) return e;
            kernel<<<grid, kTcThreads, hs.smem, s>>>(in, w, bias, out, g, relu, hs, err);
            return cudaGetLastError();
        };
        const bool three = hs.taps == 3;
        switch (hs.CK) {
            case 64: return three ? go(k_conv3d_halo<8, 3>) : go(k_conv3d_halo<8, 1>);
            case 48: return three ? go(k_conv3d_halo<6, 3>) : go(k_conv3d_halo<6, 1>);
            case 32: return three ? go(k_conv3d_halo<4, 3>) : go(k_conv3d_halo<4, 1>);
            default: return three ? go(k_conv3d_halo<2, 3>) : go(k_conv3d_halo<2, 1>);
        }
    }
    const TcShape sh = tc_shape(g.ci, g.co);
    cudaError_t e = cudaFuncSetAttribute(k_conv3d_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, sh.smem);
    if (e != cudaSuccess) return e;
    const long long M = (long long)g.N * g.D * g.H * g.W;
    const unsigned grid = (unsigned)((M + kTcM - 1) / kTcM);
    k_conv3d_tc<<<grid, kTcThreads, sh.smem, s>>>(in, w, bias, out, g, relu, err);
    return cudaGetLastError();
}

}  // namespace cl
