// mlp.cu -- learned warm start for the ILVES Newton solve.
//
// The paper starts Newton from lambda_0 = 0 (supplement Sec. 2.3).  This file adds a
// small network that predicts lambda_0 from local geometry, trained on multipliers of
// the plain solver; the Newton loop is unchanged and still decides convergence.
//
//   features  16 per constraint (own violation / alignment / masses, 4 line-graph
//             neighbour slots with their violation, coupling cosine and shared mass)
//   network   16 -> 128 -> ReLU -> 128 -> ReLU -> 1, bfloat16 weights and inputs,
//             float32 accumulation, on the 5th-generation tensor cores (tcgen05.mma,
//             operands in shared memory, accumulators in tensor memory): per 128-row tile
//             one MMA for layer 1, its epilogue writes the bfloat16 A tile of layer 2
//             (eight MMAs), whose epilogue does the third layer as a per-row dot product
//   target    y = lambda * scale, scale = 4 (w_i + w_j) s.rho / d^2  -> lambda_0 = y / scale
//   training  forward on the tensor cores storing activations, backward on the float32
//             pipes (register-tiled products per CTA, partial gradients summed in a fixed
//             order), Adam on float32 master weights, bfloat16 copies refreshed.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <random>
#include <vector>

#include "devmath.cuh"
#include "ilves.h"
#include "internal.h"
#include "topology_impl.h"

namespace ilves {

constexpr int NF = ILVES_MLP_FEATURES, NH = ILVES_MLP_HIDDEN;
constexpr int P_W1 = 0, P_B1 = P_W1 + NH * NF, P_W2 = P_B1 + NH, P_B2 = P_W2 + NH * NH, P_W3 = P_B2 + NH,
              P_B3 = P_W3 + NH, P_N = P_B3 + 1;
static_assert(P_N == ILVES_MLP_PARAMS, "parameter count");
constexpr int TILE = 128;  // rows per tensor-core tile (M of the MMA)
constexpr int kFwdThreads = 2 * TILE;  // two threads to a row

// ------------------------------------------------------------------------------------
// features
// ------------------------------------------------------------------------------------
struct FeatArgs {
    const double* x_old;
    const double* x_unc;
    const double* inv_mass;
    const double* d;
    const int32_t* con_i;
    const int32_t* con_j;
    const int4* nbr;  // four neighbour slots: neighbour << 1 | (sign product < 0), or -1
    float4* ws_con;   // per constraint: (s.xyz, sigma0 / d^2), (rho.xyz, d)
    float* ws_atom;   // per atom: inverse mass
    int32_t n_c;
    int32_t n_atoms;
};

__device__ __forceinline__ float3 ld3(const double* x, int64_t a) {
    return make_float3(narrow(x[3 * a]), narrow(x[3 * a + 1]), narrow(x[3 * a + 2]));
}
__device__ __forceinline__ float3 sub3(float3 a, float3 b) { return make_float3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ float dot3(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }

// Prep pass: per-constraint float32 geometry and per-atom weights into the topology's
// warm-start workspace, so the feature stage gathers 20 bytes per neighbour instead of four
// float64 atom positions.
__device__ __forceinline__ void let_next_start();
__global__ void k_ws_prep(FeatArgs F) {
    let_next_start();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < F.n_c) {
        const int i = F.con_i[k], j = F.con_j[k];
        const float3 s = sub3(ld3(F.x_unc, i), ld3(F.x_unc, j));
        const float3 r = sub3(ld3(F.x_old, i), ld3(F.x_old, j));
        const float dk = narrow(F.d[k]), d2 = dk * dk;
        F.ws_con[2 * k] = make_float4(s.x, s.y, s.z, (dot3(s, s) - d2) / d2);
        F.ws_con[2 * k + 1] = make_float4(r.x, r.y, r.z, dk);
    }
    if (k < F.n_atoms) F.ws_atom[k] = narrow(F.inv_mass[k]);
}

// Features of constraint k from the workspace; `half` selects which of the 16 features this
// thread writes (two threads per row): half 0 = own terms + slots 0-1 (neighbours at atom i),
// half 1 = slots 2-3 (at atom j; the scale is produced by half 0).  The shared atom of a slot
// is the half's own atom and its sign comes with the neighbour, so a neighbour costs two loads
// in the second of two rounds.
template <int half>
__device__ __forceinline__ void ws_features(const FeatArgs& F, int k, float* f, float& scale) {
    const int2 nb = __ldg(reinterpret_cast<const int2*>(F.nbr + k) + half);
    const float4 s4 = F.ws_con[2 * k], r4 = F.ws_con[2 * k + 1];
    const float wi = F.ws_atom[F.con_i[k]], wj = F.ws_atom[F.con_j[k]], W = wi + wj;
    const float inv_w = W > 0.f ? 1.0f / W : 0.f;
    const float dk = r4.w;
    const float3 s = make_float3(s4.x, s4.y, s4.z);
    if (half == 0) {
        const float3 r = make_float3(r4.x, r4.y, r4.z);
        const float inv_d2 = 1.0f / (dk * dk), sr = dot3(s, r);
        const float3 sm = sub3(s, r);
        f[0] = s4.w;
        f[1] = sr * inv_d2 - 1.0f;
        f[2] = (wi - wj) * inv_w;
        f[3] = dot3(sm, sm) * inv_d2;
        scale = 4.0f * W * sr * inv_d2;
    }
#pragma unroll
    for (int qq = 0; qq < 2; ++qq) {
        const int q = 2 * half + qq, e = qq == 0 ? nb.x : nb.y;
        float g0 = 0.f, g1 = 0.f, g2 = 0.f;
        if (e >= 0) {
            const int l = e >> 1;
            const float4 rl4 = F.ws_con[2 * l + 1];
            g0 = F.ws_con[2 * l].w;
            const float sgn = (e & 1) ? -1.f : 1.f;
            g1 = sgn * dot3(s, make_float3(rl4.x, rl4.y, rl4.z)) / (dk * rl4.w);
            g2 = (half == 0 ? wi : wj) * inv_w;
        }
        f[4 + 3 * q] = g0;
        f[5 + 3 * q] = g1;
        f[6 + 3 * q] = g2;
    }
}

__global__ void k_features(FeatArgs F, float* __restrict__ feat, float* __restrict__ scale) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= F.n_c) return;
    float f[NF], sc = 0.f;
    ws_features<0>(F, k, f, sc);
    ws_features<1>(F, k, f, sc);
#pragma unroll
    for (int q = 0; q < NF; ++q) feat[(int64_t)k * NF + q] = f[q];
    if (scale) scale[k] = sc;
}

// Jacobi guess lambda_0 = sigma_0 / A_kk at x_unc (no network): y = f0, own terms only.
__global__ void k_diag_guess(FeatArgs F, float* __restrict__ lambda0) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= F.n_c) return;
    const int i = F.con_i[k], j = F.con_j[k];
    const float3 s = sub3(ld3(F.x_unc, i), ld3(F.x_unc, j));
    const float3 r = sub3(ld3(F.x_old, i), ld3(F.x_old, j));
    const float dk = narrow(F.d[k]), d2 = dk * dk;
    const float W = narrow(F.inv_mass[i]) + narrow(F.inv_mass[j]);
    const float a = 4.0f * W * dot3(s, r);
    const float l0 = (dot3(s, s) - d2) / a;
    lambda0[k] = (a != 0.f && isfinite(l0)) ? l0 : 0.f;
}

// ------------------------------------------------------------------------------------
// tensor-core forward (tcgen05: operands in shared memory, accumulators in tensor memory)
// ------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

__device__ __forceinline__ void copy16(void* smem, const void* gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void copy_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Dependent launches: a kernel launched with launch_after may start while the kernel before it in
// the stream still runs, once every CTA of that one has passed let_next_start (or ended); what
// it reads of that kernel's results comes after wait_for_previous, which returns when that
// kernel has completed.  The set-up of the next kernel (its launch, weights, tensor memory) then
// overlaps the end of the previous one.  A dependent kernel is resident while those results are
// written, so they are not constant for its life: it takes them by plain pointers (no const
// __restrict__, no __ldg), whose loads stay behind the wait and go through the coherent path.
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <class... P, class... A>
static cudaError_t launch_after(void (*kernel)(P...), int grid, int block, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

struct MlpWeights {
    const __nv_bfloat16* w1;  // [NH][NF]  (out x in) bfloat16
    const __nv_bfloat16* w2;  // [NH][NH]
    const float* params;      // float32 master parameters (biases, w3, b3 read from here)
};

// Operand tiles use the tensor cores' canonical K-major layout without swizzling: the
// tile is cut into core matrices of 8 rows x 16 bytes (8 bfloat16 of K), each stored as
// 128 contiguous bytes; core (row group g, K chunk c) sits at g * SBO + c * 128.
__device__ __forceinline__ uint32_t core_offset(int row, int kchunk, int kchunks) {
    return (uint32_t)((row >> 3) * (kchunks * 128) + kchunk * 128 + (row & 7) * 16);
}
// shared-memory matrix descriptor: start >> 4, leading (K) byte offset >> 4, stride (row
// group) byte offset >> 4, descriptor version 1 (bits 46-47), no swizzle
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}
// instruction descriptor, kind::f16: f32 accumulator (bits 4-5 = 1), bf16 A and B (bits
// 7-9, 10-12 = 1), both K-major, N >> 3 at bits 17-22, M >> 4 at bits 24-28
constexpr uint32_t kIdescBf16 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NH >> 3) << 17) |
                                ((uint32_t)(TILE >> 4) << 24);
// one 128-column accumulator: layer 2 reuses the columns once layer 1's epilogue has
// moved them to shared memory
constexpr uint32_t kTmemCols = NH;

__device__ __forceinline__ uint32_t saddr_of(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void async_proxy_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(kIdescBf16), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
                 : "memory");
}
// bounded wait for the mbarrier phase of the given parity; false if it gave up
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity) {
    for (int it = 0; it < (1 << 22); ++it) {
        uint32_t done;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (done) return true;
        if (it > 64) __nanosleep(64);
    }
    return false;
}
// 32 consecutive accumulator columns of this thread's row (warp w reads lanes 32w..32w+31)
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

// shared-memory plan of the forward kernel (bytes from a 128-byte aligned base); about
// 74 KB, so at most three CTAs share an SM and their tensor memory (3 x 128 of 512
// columns) always fits
constexpr uint32_t SM_W1 = 0, SM_W2 = SM_W1 + NH * NF * 2, SM_A1 = SM_W2 + NH * NH * 2,
                   SM_A2 = SM_A1 + TILE * NF * 2, SM_B = SM_A2 + TILE * NH * 2, SM_Y = SM_B + 3 * NH * 4,
                   SM_BAR = SM_Y + TILE * 4, SM_USED = SM_BAR + 16;
constexpr uint32_t SM_REQUEST = SM_USED + 128;
static_assert(4 * (SM_REQUEST + 1024) > 228 * 1024 && kTmemCols * 3 <= 512, "at most three CTAs per SM");

// Persistent forward over 128-row tiles.  Per tile: rows -> bfloat16 A tile; one MMA
// (K = 16) into the 128 tensor-memory columns; epilogue (+b1, ReLU, bfloat16) writes the
// second A tile; eight MMAs (K = 128) into the same columns; epilogue (+b2, ReLU, dot
// with w3, +b3) gives y.  Two threads per row: thread t of warp w owns row 32 (w & 3) + t, which
// is that tensor-memory lane, and half w / 4 of its features and of the 128 columns.  Input
// rows come from a feature matrix or, fused, are built from the topology (output lambda_0 = y
// / scale); in training mode the hidden activations are stored for the backward pass.  A wait
// that gives up counts in *err and ends the kernel after freeing its tensor memory.
//
// What bounds it: the MMAs take a few per cent of a tile's time; the rest is the features'
// gathers (two dependent rounds, about 3,700 cycles with three CTAs to an SM) and the two
// epilogues' 128 columns a row (about 2,200 each).  Two threads to a row halve both chains and
// double the warps an SM overlaps them with (24 on three CTAs): a warm start of 258,048
// constraints, with its prep pass, 50.6 -> 43.7 us, and 37.7 as a dependent launch.
template <bool kFused, bool kTrain>
__global__ void __launch_bounds__(kFwdThreads, 3)
k_mlp_forward(MlpWeights Wt, const float* __restrict__ X, int n, FeatArgs F, float* __restrict__ out,
              __nv_bfloat16* __restrict__ h1_out, float* __restrict__ h2_out, int* __restrict__ err,
              int wait_test) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    float* b1s = reinterpret_cast<float*>(sm + SM_B);
    float* b2s = b1s + NH;
    float* w3s = b2s + NH;
    float* ys = reinterpret_cast<float*>(sm + SM_Y);  // the second half's part of each row's y
    uint64_t* bar = reinterpret_cast<uint64_t*>(sm + SM_BAR);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + SM_BAR + 8);
    const int tid = threadIdx.x, warp = tid >> 5, lrow = tid & (TILE - 1), half = tid / TILE;
    const uint32_t mbar = saddr_of(bar);
    if (warp == 0) {  // 128 tensor-memory columns for this CTA
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr_of(tmem_slot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar), "r"(1) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // weights into the canonical layout: 16-byte chunks of 8 K values, taken in the layout's
    // order (row within the core matrix fastest), so the shared-memory writes are linear; the
    // copies run while the first tile's rows are built
    for (int e = tid; e < NH * NF / 8; e += kFwdThreads) {
        const int r8 = e & 7, kc = (e >> 3) % (NF / 8), row = 8 * (e / NF) + r8;
        copy16(sm + SM_W1 + 16 * e, reinterpret_cast<const uint4*>(Wt.w1) + row * (NF / 8) + kc);
    }
    for (int e = tid; e < NH * NH / 8; e += kFwdThreads) {
        const int r8 = e & 7, kc = (e >> 3) % (NH / 8), row = 8 * (e / NH) + r8;
        copy16(sm + SM_W2 + 16 * e, reinterpret_cast<const uint4*>(Wt.w2) + row * (NH / 8) + kc);
    }
    for (int e = tid; e < NH; e += kFwdThreads) {
        b1s[e] = Wt.params[P_B1 + e];
        b2s[e] = Wt.params[P_B2 + e];
        w3s[e] = Wt.params[P_W3 + e];
    }
    const float b3 = Wt.params[P_B3];
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t t_half = ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(NH / 2 * half);  // this thread's columns
    const uint64_t dA1 = smem_desc(saddr_of(sm + SM_A1), 128, (NF / 8) * 128);
    const uint64_t dW1 = smem_desc(saddr_of(sm + SM_W1), 128, (NF / 8) * 128);
    const uint64_t dA2 = smem_desc(saddr_of(sm + SM_A2), 128, (NH / 8) * 128);
    const uint64_t dW2 = smem_desc(saddr_of(sm + SM_W2), 128, (NH / 8) * 128);
    if constexpr (kFused) wait_for_previous();  // the records of k_ws_prep
    if constexpr (kTrain) let_next_start();
    uint32_t parity = 0;
    bool ok = true;
    const int n_tiles = (n + TILE - 1) / TILE;
    if (wait_test) {  // testing: wait on a phase nothing completes (no MMA in flight), so the wait runs out
        ok = __syncthreads_and(mbar_wait(mbar, parity)) != 0;
    }
    for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
        const int row = tile * TILE + lrow;
        // ---- input row -> bfloat16 A tile
        float sc = 0.f;
        if constexpr (kFused) {  // half 0: features 0-9 and the scale, half 1: features 10-15
            float f[NF];
#pragma unroll
            for (int c = 0; c < NF; ++c) f[c] = 0.f;
            uint32_t* k1 = reinterpret_cast<uint32_t*>(sm + SM_A1 + core_offset(lrow, 1, NF / 8));
            if (half == 0) {
                if (row < n) ws_features<0>(F, row, f, sc);
                *reinterpret_cast<uint4*>(sm + SM_A1 + core_offset(lrow, 0, NF / 8)) =
                    make_uint4(pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]), pack_bf16(f[4], f[5]), pack_bf16(f[6], f[7]));
                k1[0] = pack_bf16(f[8], f[9]);
            } else {
                if (row < n) ws_features<1>(F, row, f, sc);
                k1[1] = pack_bf16(f[10], f[11]);
                k1[2] = pack_bf16(f[12], f[13]);
                k1[3] = pack_bf16(f[14], f[15]);
            }
        } else {  // eight features each
            float4 v[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
            if (row < n) {
                const float4* xr = reinterpret_cast<const float4*>(X + (int64_t)row * NF) + 2 * half;
                v[0] = __ldg(xr);
                v[1] = __ldg(xr + 1);
            }
            *reinterpret_cast<uint4*>(sm + SM_A1 + core_offset(lrow, half, NF / 8)) =
                make_uint4(pack_bf16(v[0].x, v[0].y), pack_bf16(v[0].z, v[0].w), pack_bf16(v[1].x, v[1].y),
                           pack_bf16(v[1].z, v[1].w));
        }
        copy_wait_all();  // (the weights; nothing is in flight after the first tile)
        async_proxy_fence();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        // ---- layer 1: one MMA, K = 16
        if (tid == 0) {
            tc_mma(tmem, dA1, dW1, 0u);
            tc_commit(mbar);
        }
        ok = __syncthreads_and(mbar_wait(mbar, parity)) != 0;  // one decision for the whole CTA
        parity ^= 1u;
        tc_fence_after();
        if (!ok) break;
#pragma unroll 1
        for (int ch = 0; ch < 2; ++ch) {
            float v[32];
            tmem_ld32(tmem + t_half + 32 * ch, v);
            const int c0 = NH / 2 * half + 32 * ch;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 ba = *reinterpret_cast<const float4*>(b1s + c0 + 8 * q);
                const float4 bb = *reinterpret_cast<const float4*>(b1s + c0 + 8 * q + 4);
                const float* w = v + 8 * q;
                const uint4 u = make_uint4(pack_bf16(fmaxf(w[0] + ba.x, 0.f), fmaxf(w[1] + ba.y, 0.f)),
                                           pack_bf16(fmaxf(w[2] + ba.z, 0.f), fmaxf(w[3] + ba.w, 0.f)),
                                           pack_bf16(fmaxf(w[4] + bb.x, 0.f), fmaxf(w[5] + bb.y, 0.f)),
                                           pack_bf16(fmaxf(w[6] + bb.z, 0.f), fmaxf(w[7] + bb.w, 0.f)));
                *reinterpret_cast<uint4*>(sm + SM_A2 + core_offset(lrow, c0 / 8 + q, NH / 8)) = u;
                if constexpr (kTrain) {
                    if (row < n) reinterpret_cast<uint4*>(h1_out + (int64_t)row * NH + c0)[q] = u;
                }
            }
        }
        async_proxy_fence();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        // ---- layer 2: eight MMAs along K = 128 (16 per step: two core matrices, 256 bytes)
        if (tid == 0) {
#pragma unroll
            for (int k = 0; k < NH / 16; ++k) tc_mma(tmem, dA2 + (uint64_t)(k * 16), dW2 + (uint64_t)(k * 16), k > 0);
            tc_commit(mbar);
        }
        ok = __syncthreads_and(mbar_wait(mbar, parity)) != 0;
        parity ^= 1u;
        tc_fence_after();
        if (!ok) break;
        float y = 0.f;
#pragma unroll 1
        for (int ch = 0; ch < 2; ++ch) {
            float v[32];
            tmem_ld32(tmem + t_half + 32 * ch, v);
            const int c0 = NH / 2 * half + 32 * ch;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float4 b = *reinterpret_cast<const float4*>(b2s + c0 + 4 * q);
                const float4 w = *reinterpret_cast<const float4*>(w3s + c0 + 4 * q);
                float* u = v + 4 * q;
                u[0] = fmaxf(u[0] + b.x, 0.f);
                u[1] = fmaxf(u[1] + b.y, 0.f);
                u[2] = fmaxf(u[2] + b.z, 0.f);
                u[3] = fmaxf(u[3] + b.w, 0.f);
                y = fmaf(u[0], w.x, y);
                y = fmaf(u[1], w.y, y);
                y = fmaf(u[2], w.z, y);
                y = fmaf(u[3], w.w, y);
                if constexpr (kTrain) {
                    if (row < n)
                        reinterpret_cast<float4*>(h2_out + (int64_t)row * NH + c0)[q] = make_float4(u[0], u[1], u[2], u[3]);
                }
            }
        }
        tc_fence_before();
        if (half == 1) ys[lrow] = y;
        __syncthreads();
        if (half == 0 && row < n) {
            y = (y + ys[lrow]) + b3;
            if constexpr (kFused) {
                const float l0 = y / sc;
                out[row] = (sc != 0.f && isfinite(l0)) ? l0 : 0.f;
            } else {
                out[row] = y;
            }
        }
    }
    copy_wait_all();  // (a wait given up before the first tile)
    if (!ok && tid == 0) atomicAdd(err, 1);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols)
                                : "memory");
}

// ------------------------------------------------------------------------------------
// float32 backward: three register-tiled products per chunk of rows
// ------------------------------------------------------------------------------------
// A CTA takes rows_per_cta rows, up to kBwdRows at a time, held in shared memory with W2:
//   dz2 = (dy w3) masked by h2 > 0,   gW2 += dz2^T h1,   dh1 = dz2 W2,   dz1 = dh1 masked by
//   h1 > 0,   gW1 += dz1^T X,   and the column sums.
// What bounds it: the float32 pipes (70 kFLOP a row; 0.57 GFLOP for 8192 rows).  Each thread
// holds an 8 x 8 tile of gW2 across the whole range (and 4 x 8 of dh1), so an operand read
// from shared memory feeds eight FMAs; two FMAs go in one instruction (fma.rn.f32x2, the same
// roundings), which leaves issue slots for the loads.  Every CTA writes its own partial
// gradient (and loss); k_grad_reduce adds them in a fixed order of eight interleaved chains, so
// the gradient is the same on every run and its rounding error does not grow with the number
// of CTAs, as it did with float32 atomics.  Rows are spread over the SMs, but at least kBwdMinRows
// to a CTA, below which the 75 KB of W2 in and gradient out cost more than they save.
// A whole gradient of 8192 rows takes 32.8 us (38.9 before its kernels were dependent launches:
// forward 12, this kernel 20, reduction 5); with one thread per hidden unit, rows streamed one
// by one with three barriers each and float32 atomics it took 227 us.
constexpr int kBwdRows = 64, kBwdMinRows = 16, kBwdThreads = 256;
constexpr int kPartStride = (P_N + 1 + 3) & ~3;  // a CTA's partial gradient, then its loss
constexpr int kBwdSmem = (NH * NH + 2 * kBwdRows * NH + kBwdRows * NF + kBwdRows) * (int)sizeof(float);

__device__ __forceinline__ float2 fma2(float a, float2 b, float2 c) {
    float2 d;
    asm("{\n.reg .b64 ra, rb, rc;\nmov.b64 ra, {%2, %2};\nmov.b64 rb, {%3, %4};\nmov.b64 rc, {%5, %6};\n"
        "fma.rn.f32x2 rc, ra, rb, rc;\nmov.b64 {%0, %1}, rc;\n}\n"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
__global__ void __launch_bounds__(kBwdThreads, 1)
k_mlp_backward(const float* __restrict__ X, const float* __restrict__ t, int n, int rows_per_cta, const float* y,
               const __nv_bfloat16* h1, const float* h2, const __nv_bfloat16* __restrict__ w2b,
               const float* __restrict__ params, float* __restrict__ partial) {
    extern __shared__ __align__(16) float bsm[];
    float* w2s = bsm;                       // [c][k], the bfloat16 weights the forward used
    float* dzs = w2s + NH * NH;             // dz2 [r][c], then dz1 [r][k]
    float* h1s = dzs + kBwdRows * NH;       // [r][k]
    float* xs = h1s + kBwdRows * NH;        // [r][f]
    float* dys = xs + kBwdRows * NF;        // [r]
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
#pragma unroll
    for (int q0 = 0; q0 < NH * NH / 8 / kBwdThreads; ++q0) {
        const int e = tid + kBwdThreads * q0;
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(w2b) + e);
        const __nv_bfloat162* b = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
        for (int q = 0; q < 4; ++q) *reinterpret_cast<float2*>(w2s + 8 * e + 2 * q) = __bfloat1622float2(b[q]);
    }
    const int c = tid & (NH - 1), half = tid >> 7;
    const int c4 = 4 * (tid & 31), r8 = tid >> 5;  // dz2 and its column sums: columns c4 .. c4 + 3, every 8th row
    const float4 w3v = make_float4(params[P_W3 + c4], params[P_W3 + c4 + 1], params[P_W3 + c4 + 2], params[P_W3 + c4 + 3]);
    const float inv_n = 1.0f / (float)n;
    // rows (columns) of a tile: ty * 4 .. + 3 and 64 + ty * 4 .. + 3 (tx alike), so the lanes of a warp
    // read consecutive 16-byte words
    float2 gw2[8][4], gw1[4];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) gw2[a][b] = make_float2(0.f, 0.f);
#pragma unroll
    for (int b = 0; b < 4; ++b) gw1[b] = make_float2(0.f, 0.f);
    float4 gb2 = make_float4(0.f, 0.f, 0.f, 0.f), gw3 = gb2;
    float gb1 = 0.f, gb3 = 0.f, lsum = 0.f;
    const int rb = blockIdx.x * rows_per_cta, re = min(n, rb + rows_per_cta);
    let_next_start();
    wait_for_previous();  // the forward's activations
    for (int r0 = rb; r0 < re; r0 += kBwdRows) {
        const int rows = min(kBwdRows, re - r0), rows4 = (rows + 3) & ~3;  // completed with zero rows
        __syncthreads();
        if (tid < rows4) {
            float dy = 0.f;
            if (tid < rows) {
                const float res = y[r0 + tid] - t[r0 + tid];
                dy = 2.0f * res * inv_n;
                lsum += res * res * inv_n;
                gb3 += dy;
            }
            dys[tid] = dy;
        }
        for (int e = tid; e < rows4 * (NF / 4); e += kBwdThreads)
            reinterpret_cast<float4*>(xs)[e] = e < rows * (NF / 4)
                                                   ? __ldg(reinterpret_cast<const float4*>(X + (int64_t)r0 * NF) + e)
                                                   : make_float4(0.f, 0.f, 0.f, 0.f);
        for (int e = tid; e < rows4 * (NH / 8); e += kBwdThreads) {
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (e < rows * (NH / 8)) v = reinterpret_cast<const uint4*>(h1 + (int64_t)r0 * NH)[e];
            const __nv_bfloat162* b = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
            for (int q = 0; q < 4; ++q) *reinterpret_cast<float2*>(h1s + 8 * e + 2 * q) = __bfloat1622float2(b[q]);
        }
        __syncthreads();
        {
            float4 h[kBwdRows / 8];
#pragma unroll
            for (int q = 0; q < kBwdRows / 8; ++q) {
                const int r = r8 + 8 * q;
                h[q] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (r < rows) h[q] = *reinterpret_cast<const float4*>(h2 + (int64_t)(r0 + r) * NH + c4);
            }
#pragma unroll
            for (int q = 0; q < kBwdRows / 8; ++q) {
                const int r = r8 + 8 * q;
                if (r >= rows4) break;
                const float dy = dys[r];
                const float4 z = make_float4(h[q].x > 0.f ? dy * w3v.x : 0.f, h[q].y > 0.f ? dy * w3v.y : 0.f,
                                             h[q].z > 0.f ? dy * w3v.z : 0.f, h[q].w > 0.f ? dy * w3v.w : 0.f);
                gw3.x += dy * h[q].x;
                gw3.y += dy * h[q].y;
                gw3.z += dy * h[q].z;
                gw3.w += dy * h[q].w;
                gb2.x += z.x;
                gb2.y += z.y;
                gb2.z += z.z;
                gb2.w += z.w;
                *reinterpret_cast<float4*>(dzs + r * NH + c4) = z;
            }
        }
        __syncthreads();
        // gW2[c][k] += sum_r dz2[r][c] h1[r][k]
#pragma unroll 2
        for (int r = 0; r < rows4; ++r) {
            const float4 a0 = *reinterpret_cast<const float4*>(dzs + r * NH + 4 * ty);
            const float4 a1 = *reinterpret_cast<const float4*>(dzs + r * NH + 64 + 4 * ty);
            const float4 b0 = *reinterpret_cast<const float4*>(h1s + r * NH + 4 * tx);
            const float4 b1 = *reinterpret_cast<const float4*>(h1s + r * NH + 64 + 4 * tx);
            const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float2 bv[4] = {{b0.x, b0.y}, {b0.z, b0.w}, {b1.x, b1.y}, {b1.z, b1.w}};
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) gw2[a][b] = fma2(av[a], bv[b], gw2[a][b]);
        }
        // dh1[r][k] = sum_c dz2[r][c] W2[c][k], rows ty, ty + 16, ty + 32, ty + 48
        float2 dh[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) dh[a][b] = make_float2(0.f, 0.f);
        if (ty < rows4) {  // rows past rows4 repeat the last one: computed, not stored
#pragma unroll 1
            for (int cc = 0; cc < NH; cc += 4) {
                float av[4][4];
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    const float4 v = *reinterpret_cast<const float4*>(dzs + min(ty + 16 * a, rows4 - 1) * NH + cc);
                    av[a][0] = v.x;
                    av[a][1] = v.y;
                    av[a][2] = v.z;
                    av[a][3] = v.w;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float4 b0 = *reinterpret_cast<const float4*>(w2s + (cc + q) * NH + 4 * tx);
                    const float4 b1 = *reinterpret_cast<const float4*>(w2s + (cc + q) * NH + 64 + 4 * tx);
                    const float2 bv[4] = {{b0.x, b0.y}, {b0.z, b0.w}, {b1.x, b1.y}, {b1.z, b1.w}};
#pragma unroll
                    for (int a = 0; a < 4; ++a)
#pragma unroll
                        for (int b = 0; b < 4; ++b) dh[a][b] = fma2(av[a][q], bv[b], dh[a][b]);
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int r = ty + 16 * a;
            if (r < rows4) {
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const int k = (b < 2 ? 0 : 64) + 4 * tx + 2 * (b & 1);
                    const float2 h = *reinterpret_cast<const float2*>(h1s + r * NH + k);
                    *reinterpret_cast<float2*>(dzs + r * NH + k) =
                        make_float2(h.x > 0.f ? dh[a][b].x : 0.f, h.y > 0.f ? dh[a][b].y : 0.f);
                }
            }
        }
        __syncthreads();
        // gW1[k][f] += sum_r dz1[r][k] X[r][f]: unit k = c, features 8 half .. + 7
#pragma unroll 4
        for (int r = 0; r < rows4; ++r) {
            const float dz1 = dzs[r * NH + c];
            const float4 x0 = *reinterpret_cast<const float4*>(xs + r * NF + 8 * half);
            const float4 x1 = *reinterpret_cast<const float4*>(xs + r * NF + 8 * half + 4);
            gw1[0] = fma2(dz1, make_float2(x0.x, x0.y), gw1[0]);
            gw1[1] = fma2(dz1, make_float2(x0.z, x0.w), gw1[1]);
            gw1[2] = fma2(dz1, make_float2(x1.x, x1.y), gw1[2]);
            gw1[3] = fma2(dz1, make_float2(x1.z, x1.w), gw1[3]);
            if (half == 0) gb1 += dz1;
        }
    }
    float* grad = partial + (int64_t)blockIdx.x * kPartStride;
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        float4* g = reinterpret_cast<float4*>(grad + P_W2 + ((a < 4 ? 0 : 64) + 4 * ty + (a & 3)) * NH + 4 * tx);
        g[0] = make_float4(gw2[a][0].x, gw2[a][0].y, gw2[a][1].x, gw2[a][1].y);
        g[16] = make_float4(gw2[a][2].x, gw2[a][2].y, gw2[a][3].x, gw2[a][3].y);
    }
    float4* g1 = reinterpret_cast<float4*>(grad + P_W1 + c * NF + 8 * half);
    g1[0] = make_float4(gw1[0].x, gw1[0].y, gw1[1].x, gw1[1].y);
    g1[1] = make_float4(gw1[2].x, gw1[2].y, gw1[3].x, gw1[3].y);
    // the column sums of the eight row groups, the sums over rows
    __syncthreads();
    *reinterpret_cast<float4*>(dzs + r8 * NH + c4) = gb2;
    *reinterpret_cast<float4*>(dzs + (8 + r8) * NH + c4) = gw3;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        gb3 += __shfl_xor_sync(0xFFFFFFFFu, gb3, o);
        lsum += __shfl_xor_sync(0xFFFFFFFFu, lsum, o);
    }
    if (tid == 32) {
        dys[0] = gb3;
        dys[1] = lsum;
    }
    __syncthreads();
    if (half == 0) grad[P_B1 + c] = gb1;
    float sum = 0.f;  // half 0: gb2[c], half 1: gw3[c]
#pragma unroll
    for (int q = 0; q < 8; ++q) sum += dzs[(8 * half + q) * NH + c];
    grad[(half == 0 ? P_B2 : P_W3) + c] = sum;
    if (tid == 0) {
        grad[P_B3] = gb3 + dys[0];
        grad[P_N] = lsum + dys[1];
    }
}

// The partial gradients' sum: 32 columns of four values to a CTA, eight threads to a column that
// each add every eighth partial, then one adds the eight.
constexpr int kRedThreads = 256;
__global__ void __launch_bounds__(kRedThreads)
k_grad_reduce(const float* partial, int n_part, float* __restrict__ grad, float* __restrict__ loss) {
    __shared__ float4 acc[kRedThreads];
    wait_for_previous();  // the partial gradients
    const int col = blockIdx.x * 32 + (threadIdx.x & 31), row = threadIdx.x >> 5;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (col < kPartStride / 4)
#pragma unroll 8
        for (int p = row; p < n_part; p += kRedThreads / 32) {
            const float4 v = reinterpret_cast<const float4*>(partial + (int64_t)p * kPartStride)[col];
            s.x += v.x;
            s.y += v.y;
            s.z += v.z;
            s.w += v.w;
        }
    acc[threadIdx.x] = s;
    __syncthreads();
    if (row != 0) return;
#pragma unroll
    for (int q = 1; q < kRedThreads / 32; ++q) {
        const float4 v = acc[32 * q + threadIdx.x];
        s.x += v.x;
        s.y += v.y;
        s.z += v.z;
        s.w += v.w;
    }
    const float out[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int i = 4 * col + q;
        if (i < P_N) grad[i] = out[q];
        else if (i == P_N) *loss = out[q];
    }
}

// Adam on the float32 master parameters; refreshes the bfloat16 weight copies.
__global__ void k_adam(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ g, float lr, float b1c, float b2c, __nv_bfloat16* __restrict__ w1b,
                       __nv_bfloat16* __restrict__ w2b) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P_N) return;
    const float beta1 = 0.9f, beta2 = 0.999f, eps = 1e-8f;
    const float gi = g[i];
    const float mi = beta1 * m[i] + (1.f - beta1) * gi;
    const float vi = beta2 * v[i] + (1.f - beta2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / b1c) / (sqrtf(vi / b2c) + eps);
    p[i] = pi;
    if (i < P_B1) w1b[i - P_W1] = __float2bfloat16_rn(pi);
    else if (i >= P_W2 && i < P_B2) w2b[i - P_W2] = __float2bfloat16_rn(pi);
}

__global__ void k_refresh_bf16(const float* __restrict__ p, __nv_bfloat16* __restrict__ w1b,
                               __nv_bfloat16* __restrict__ w2b) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < NH * NF) w1b[i] = __float2bfloat16_rn(p[P_W1 + i]);
    if (i < NH * NH) w2b[i] = __float2bfloat16_rn(p[P_W2 + i]);
}

}  // namespace ilves

using namespace ilves;

struct ilves_mlp {
    int32_t device = -1;
    int32_t max_batch = 0;
    int64_t step = 0;
    float* params = nullptr;
    float* m = nullptr;
    float* v = nullptr;
    float* grad = nullptr;
    float* partial = nullptr;  // one partial gradient and loss per CTA of the backward kernel
    int32_t n_part = 0;        // at most this many
    float* loss = nullptr;
    float* y = nullptr;
    __nv_bfloat16* w1b = nullptr;
    __nv_bfloat16* w2b = nullptr;
    __nv_bfloat16* h1 = nullptr;
    float* h2 = nullptr;
    int* err = nullptr;  // tensor-core waits that gave up (see ilves_mlp_check)
    int32_t wait_test = 0;  // testing: forward kernels wait on a phase nothing completes
};

static ilves_status mlp_status(cudaError_t e) {
    if (e == cudaSuccess) return ILVES_OK;
    return e == cudaErrorMemoryAllocation ? ILVES_ERR_OOM : ILVES_ERR_CUDA;
}

static FeatArgs feat_args(const ilves_topology* T, const double* x_old, const double* x_unc, const double* inv_mass,
                          const double* d) {
    FeatArgs F;
    F.x_old = x_old;
    F.x_unc = x_unc;
    F.inv_mass = inv_mass;
    F.d = d;
    F.con_i = T->d_con_i;
    F.con_j = T->d_con_j;
    F.nbr = reinterpret_cast<const int4*>(T->d_nbr);
    F.ws_con = reinterpret_cast<float4*>(T->d_ws_con);
    F.ws_atom = T->d_ws_atom;
    F.n_c = T->n_c;
    F.n_atoms = T->n_atoms;
    return F;
}

// Launches the tensor-core forward: persistent CTAs, at most three per SM (the shared
// memory request guarantees it), one 128-row tile at a time.
template <bool kFused, bool kTrain>
static cudaError_t launch_forward(const MlpWeights& Wt, const float* X, int n, const FeatArgs& F, float* out,
                                  __nv_bfloat16* h1, float* h2, int* err, int wait_test, cudaStream_t s) {
    static bool attr_set[64] = {};
    int dev = 0, sms = 152;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        e = cudaFuncSetAttribute(k_mlp_forward<kFused, kTrain>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)SM_REQUEST);
        if (e != cudaSuccess) return e;
        attr_set[dev] = true;
    }
    const int tiles = (n + TILE - 1) / TILE;
    const int grid = std::max(1, std::min(tiles, 3 * sms));
    if constexpr (kFused)  // follows k_ws_prep
        return launch_after(k_mlp_forward<kFused, kTrain>, grid, kFwdThreads, SM_REQUEST, s, Wt, X, n, F, out, h1, h2, err,
                            wait_test);
    k_mlp_forward<kFused, kTrain><<<grid, kFwdThreads, SM_REQUEST, s>>>(Wt, X, n, F, out, h1, h2, err, wait_test);
    return cudaGetLastError();
}

extern "C" int64_t ilves_mlp_param_count(void) { return P_N; }

extern "C" ilves_status ilves_mlp_check(const ilves_mlp* M, int32_t* waits_given_up) {
    if (!M || !waits_given_up) return ILVES_ERR_INVALID_ARG;
    int v = 0;
    const cudaError_t e = cudaMemcpy(&v, M->err, sizeof(int), cudaMemcpyDeviceToHost);
    *waits_given_up = v;
    if (e != cudaSuccess) return mlp_status(e);
    return v ? ILVES_ERR_TIMEOUT : ILVES_OK;
}

extern "C" ilves_status ilves_mlp_set_wait_test(ilves_mlp* M, int32_t on) {
    if (!M) return ILVES_ERR_INVALID_ARG;
    M->wait_test = on ? 1 : 0;
    return ILVES_OK;
}

extern "C" ilves_status ilves_mlp_create(int32_t max_batch, uint64_t seed, ilves_mlp** out) {
    if (!out || max_batch <= 0) return ILVES_ERR_INVALID_ARG;
    *out = nullptr;
    ilves_mlp* M = new ilves_mlp();
    cudaGetDevice(&M->device);
    M->max_batch = max_batch;
    cudaError_t e = cudaSuccess;
    auto alloc = [&](void** p, size_t bytes) {
        if (e == cudaSuccess) e = cudaMalloc(p, bytes);
    };
    alloc((void**)&M->params, P_N * sizeof(float));
    alloc((void**)&M->m, P_N * sizeof(float));
    alloc((void**)&M->v, P_N * sizeof(float));
    alloc((void**)&M->grad, P_N * sizeof(float));
    M->n_part = 152;
    if (cudaDeviceGetAttribute(&M->n_part, cudaDevAttrMultiProcessorCount, M->device) != cudaSuccess) M->n_part = 152;
    M->n_part = std::min(M->n_part, std::max(1, (max_batch + kBwdMinRows - 1) / kBwdMinRows));
    alloc((void**)&M->partial, (size_t)M->n_part * kPartStride * sizeof(float));
    alloc((void**)&M->loss, sizeof(float));
    alloc((void**)&M->y, (size_t)max_batch * sizeof(float));
    alloc((void**)&M->w1b, NH * NF * sizeof(__nv_bfloat16));
    alloc((void**)&M->w2b, NH * NH * sizeof(__nv_bfloat16));
    alloc((void**)&M->h1, (size_t)max_batch * NH * sizeof(__nv_bfloat16));
    alloc((void**)&M->h2, (size_t)max_batch * NH * sizeof(float));
    alloc((void**)&M->err, sizeof(int));
    if (e == cudaSuccess) e = cudaMemset(M->err, 0, sizeof(int));
    if (e != cudaSuccess) {
        ilves_mlp_destroy(M);
        return mlp_status(e);
    }
    // He-uniform weights, zero biases
    std::vector<float> h(P_N, 0.f);
    std::mt19937_64 rng(seed);
    std::uniform_real_distribution<float> u(-1.f, 1.f);
    for (int i = 0; i < NH * NF; ++i) h[P_W1 + i] = u(rng) * std::sqrt(6.f / NF);
    for (int i = 0; i < NH * NH; ++i) h[P_W2 + i] = u(rng) * std::sqrt(6.f / NH);
    for (int i = 0; i < NH; ++i) h[P_W3 + i] = u(rng) * std::sqrt(3.f / NH);
    ilves_status s = ilves_mlp_set_params(M, h.data());
    if (s != ILVES_OK) {
        ilves_mlp_destroy(M);
        return s;
    }
    *out = M;
    return ILVES_OK;
}

extern "C" void ilves_mlp_destroy(ilves_mlp* M) {
    if (!M) return;
    for (void* p : {(void*)M->params, (void*)M->m, (void*)M->v, (void*)M->grad, (void*)M->partial, (void*)M->loss,
                    (void*)M->y, (void*)M->w1b, (void*)M->w2b, (void*)M->h1, (void*)M->h2, (void*)M->err})
        if (p) cudaFree(p);
    delete M;
}

extern "C" ilves_status ilves_mlp_set_params(ilves_mlp* M, const float* host_params) {
    if (!M || !host_params) return ILVES_ERR_INVALID_ARG;
    cudaError_t e = cudaMemcpy(M->params, host_params, P_N * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(M->m, 0, P_N * sizeof(float));
    if (e == cudaSuccess) e = cudaMemset(M->v, 0, P_N * sizeof(float));
    if (e != cudaSuccess) return mlp_status(e);
    M->step = 0;
    k_refresh_bf16<<<(NH * NH + 255) / 256, 256>>>(M->params, M->w1b, M->w2b);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    return mlp_status(e);
}

extern "C" ilves_status ilves_mlp_get_params(const ilves_mlp* M, float* host_params) {
    if (!M || !host_params) return ILVES_ERR_INVALID_ARG;
    return mlp_status(cudaMemcpy(host_params, M->params, P_N * sizeof(float), cudaMemcpyDeviceToHost));
}

extern "C" ilves_status ilves_mlp_features(const ilves_topology* T, const double* x_old, const double* x_unc,
                                           const double* inv_mass, const double* d, float* features, float* scale,
                                           void* stream) {
    if (!T || !T->on_device || !features) return ILVES_ERR_INVALID_ARG;
    if (T->n_c == 0) return ILVES_OK;
    if (!x_old || !x_unc || !inv_mass || !d) return ILVES_ERR_INVALID_ARG;
    const FeatArgs F = feat_args(T, x_old, x_unc, inv_mass, d);
    const int np = std::max(T->n_c, T->n_atoms);
    k_ws_prep<<<(np + 255) / 256, 256, 0, (cudaStream_t)stream>>>(F);
    k_features<<<(T->n_c + 127) / 128, 128, 0, (cudaStream_t)stream>>>(F, features, scale);
    return mlp_status(cudaGetLastError());
}

extern "C" ilves_status ilves_mlp_forward(const ilves_mlp* M, const float* features, int32_t n, float* y,
                                          void* stream) {
    if (!M || n < 0 || (n > 0 && (!features || !y))) return ILVES_ERR_INVALID_ARG;
    if (n == 0) return ILVES_OK;
    if (reinterpret_cast<uintptr_t>(features) & 15u) return ILVES_ERR_INVALID_ARG;
    const MlpWeights Wt{M->w1b, M->w2b, M->params};
    FeatArgs F{};
    return mlp_status(
        launch_forward<false, false>(Wt, features, n, F, y, nullptr, nullptr, M->err, M->wait_test, (cudaStream_t)stream));
}

extern "C" ilves_status ilves_warm_start(const ilves_mlp* M, const ilves_topology* T, const double* x_old,
                                         const double* x_unc, const double* inv_mass, const double* d,
                                         float* lambda0, void* stream) {
    if (!T || !T->on_device || (T->n_c > 0 && !lambda0)) return ILVES_ERR_INVALID_ARG;
    if (T->n_c == 0) return ILVES_OK;
    if (!x_old || !x_unc || !inv_mass || !d) return ILVES_ERR_INVALID_ARG;
    const FeatArgs F = feat_args(T, x_old, x_unc, inv_mass, d);
    if (!M) {
        k_diag_guess<<<(T->n_c + 127) / 128, 128, 0, (cudaStream_t)stream>>>(F, lambda0);
    } else {
        const MlpWeights Wt{M->w1b, M->w2b, M->params};
        const int np = std::max(T->n_c, T->n_atoms);
        k_ws_prep<<<(np + 255) / 256, 256, 0, (cudaStream_t)stream>>>(F);
        const cudaError_t e =
            launch_forward<true, false>(Wt, nullptr, T->n_c, F, lambda0, nullptr, nullptr, M->err, M->wait_test,
                                        (cudaStream_t)stream);
        if (e != cudaSuccess) return mlp_status(e);
    }
    return mlp_status(cudaGetLastError());
}

// forward with stored activations + backward into grad and loss
static ilves_status mlp_gradient(ilves_mlp* M, const float* X, const float* t, int32_t n, float* grad, float* loss,
                                 cudaStream_t s) {
    const MlpWeights Wt{M->w1b, M->w2b, M->params};
    FeatArgs F{};
    if (reinterpret_cast<uintptr_t>(X) & 15u) return ILVES_ERR_INVALID_ARG;
    cudaError_t e = launch_forward<false, true>(Wt, X, n, F, M->y, M->h1, M->h2, M->err, M->wait_test, s);
    if (e != cudaSuccess) return mlp_status(e);
    static bool attr_set[64] = {};
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return mlp_status(e);
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(k_mlp_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, kBwdSmem);
        if (e != cudaSuccess) return mlp_status(e);
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    const int rows = std::max(kBwdMinRows, (n + M->n_part - 1) / M->n_part), parts = (n + rows - 1) / rows;
    e = launch_after(k_mlp_backward, parts, kBwdThreads, kBwdSmem, s, X, t, n, rows, M->y, M->h1, M->h2, M->w2b, M->params,
                     M->partial);
    if (e != cudaSuccess) return mlp_status(e);
    return mlp_status(launch_after(k_grad_reduce, (kPartStride / 4 + 31) / 32, kRedThreads, 0, s, M->partial, parts, grad, loss));
}

extern "C" ilves_status ilves_mlp_gradient(ilves_mlp* M, const float* features, const float* target, int32_t n,
                                           float* grad_out, float* loss_out, void* stream) {
    if (!M || n <= 0 || n > M->max_batch || !features || !target) return ILVES_ERR_INVALID_ARG;
    const cudaStream_t s = (cudaStream_t)stream;
    return mlp_gradient(M, features, target, n, grad_out ? grad_out : M->grad, loss_out ? loss_out : M->loss, s);
}

extern "C" ilves_status ilves_mlp_train_step(ilves_mlp* M, const float* features, const float* target, int32_t n,
                                             float lr, float* loss_out, void* stream) {
    if (!M || n <= 0 || n > M->max_batch || !features || !target || !(lr >= 0.f)) return ILVES_ERR_INVALID_ARG;
    const cudaStream_t s = (cudaStream_t)stream;
    ilves_status st = mlp_gradient(M, features, target, n, M->grad, loss_out ? loss_out : M->loss, s);
    if (st != ILVES_OK) return st;
    M->step += 1;
    const float b1c = 1.f - std::pow(0.9f, (float)M->step), b2c = 1.f - std::pow(0.999f, (float)M->step);
    k_adam<<<(P_N + 255) / 256, 256, 0, s>>>(M->params, M->m, M->v, M->grad, lr, b1c, b2c, M->w1b, M->w2b);
    return mlp_status(cudaGetLastError());
}
