// Learned warm start for GMRES: a per-element multilayer perceptron that maps local
// geometry and source-term features to the element's (phi, dphi/dn), trained on solutions
// the solver itself produces. GMRES started from its prediction still converges to the same
// residual, so the network only changes the number of iterations, never the answer.
//
// Arithmetic: BF16 weights and activations, FP32 accumulation, on the fifth-generation tensor
// cores (tcgen05.mma with tensor-memory accumulators): the fused inference and gradient of the
// default shape (width 128) and a generic tiled GEMM for the passes of other shapes; FP32 master
// weights and Adam moments. Hidden layers use ReLU, the output layer is linear, the loss is the
// mean squared error.
#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <vector>

#include "pb_internal.cuh"

#define MLP_MAXL 8
#define MLP_STAGE (1 << 20)

struct pb_mlp {
    int nin = 0, width = 0, depth = 0, nout = 0;  // depth = number of hidden layers
    int nl = 0;                                   // weight layers = depth + 1
    int din[MLP_MAXL] = {}, dout[MLP_MAXL] = {};  // padded dimensions (multiples of 16)
    long long woff[MLP_MAXL + 1] = {}, boff[MLP_MAXL + 1] = {};
    cudaStream_t st = nullptr;
    float *W = nullptr, *Wm = nullptr, *Wv = nullptr, *G = nullptr;  // all weights then biases
    __nv_bfloat16* Wb = nullptr;                                      // BF16 copy of the weights
    // training buffers (grown on demand): the outputs, per layer BF16 activations, dZ of two
    // consecutive layers, and the slices of the gradient
    int cap = 0;
    float* Z = nullptr;
    __nv_bfloat16* Ab[MLP_MAXL + 1] = {};
    __nv_bfloat16* dZb[2] = {};
    float* part = nullptr;
    int part_n = 0;
    float* lossbuf = nullptr;  // the loss, after the gradient in G
    int* derr = nullptr;  // after the loss: [0] set when a bounded wait on the tensor cores gives up, [1] the
                          // Adam steps left out since
    float* hbuf = nullptr;  // pinned copy of G, the loss and the flag (MLP_STAGE parameters at most, else null)
    long long nparam = 0;
    int adam_t = 0;
    std::string err;
};

static int mlp_fail(pb_mlp* m, int code, const char* msg)
{
    if (m) m->err = msg;
    return code;
}
static int mlp_check_err(pb_mlp* m, float* loss = nullptr);

// ---------- tcgen05 helpers ----------
#define TC_ROWS 128
__device__ __forceinline__ unsigned tc_su32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
// shared-memory matrix descriptor: start address, leading (K) and stride (8-row) byte offsets,
// descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t tc_desc(unsigned addr, unsigned lbo, unsigned sbo)
{
    return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
           (1ull << 46);
}
// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major, N, M = 128
__device__ __forceinline__ unsigned tc_idesc(int nn)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(nn >> 3) << 17) | ((unsigned)(TC_ROWS >> 4) << 24);
}
__device__ __forceinline__ bool tc_wait(unsigned bar, unsigned ph)
{
    for (unsigned it = 0; it < (1u << 24); ++it) {
        unsigned ok;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(ok) : "r"(bar), "r"(ph) : "memory");
        if (ok) return true;
    }
    return false;
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// byte offset of element (r, k) in the no-swizzle K-major layout of a matrix with K columns
__device__ __forceinline__ unsigned tc_off(int r, int k, int K) { return (r >> 3) * (K / 8) * 128 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2; }
// 32 consecutive FP32 accumulator columns of this warp's 32 lanes (rows)
__device__ __forceinline__ void tc_ld32(unsigned taddr, float* v)
{
    unsigned r[32];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                   "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
                   "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
                   "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}


// ---------- BF16 GEMMs of the training passes on the fifth-generation tensor cores ----------
// C[M x N] = sum_k A(i, k) B(k, j) in FP32, one block of four warps per 128 x 128 tile of C and per
// slice of K (blockIdx.z; slice z writes its own FP32 array, added up afterwards in slice order).
// Every operand is stored with 8 or more consecutive elements along one index (all padded layer
// widths are multiples of 16): along k (AK / BK: element (i, k) at [i * ld + k]) or along the
// other index ((i, k) at [k * ld + i], the transposed operands of the gradients). A thread moves
// 8-element (16-byte) vectors: along k straight into shared memory, otherwise eight of them
// transposed in registers. Chunks of 64 along K go to two shared-memory stages in the no-swizzle
// K-major layout, whose core matrices (8 rows x 16 bytes) lie GT_LBO = 144 bytes apart along k:
// at 128 bytes the eight vectors a transposed block writes per row would all hit one bank group.
// tcgen05.mma (M = 128, N = the tile's width rounded up to 16, K = 16) accumulates in tensor
// memory while the next chunk is loaded; a stage is reused when the commit of its last MMAs has
// arrived. Every wait is bounded (a wait that gives up sets *err, waits once more and stops).
// The epilogue (one row per thread) does what used to be passes of their own:
//   EPI_PART: FP32 tile into the slice's array; EPI_ACT: bias, ReLU, BF16 for the next layer;
//   EPI_OUT: bias, FP32 (the output layer); EPI_MASK: the ReLU derivative, BF16 dZ.
// What bounds these launches (4096 x 128 x 128 and smaller) is latency: one block's chain of
// load, MMA and epilogue. Element-by-element staging through 2-byte loads and K slices of 2048
// took 128 us per launch: a mini-batch's gradient (4096 rows, 18-128-128-128-2, to the host) took
// 1469 us then and takes 215 us through these launches.
#define GT_K 64
#define GT_LBO 144
#define GT_SBO ((GT_K / 8) * GT_LBO)
#define GT_STAGE (16 * GT_SBO)  // bytes of one operand's stage: 128 rows
#define GT_SMEM (4 * GT_STAGE)
enum { EPI_PART, EPI_ACT, EPI_OUT, EPI_MASK };
__device__ __forceinline__ unsigned gt_off(int r, int k8) { return (r >> 3) * GT_SBO + k8 * GT_LBO + (r & 7) * 16; }

// rows [r0, r0 + 128) (fewer than R: zeros), k in [k0, ke) of an operand stored along k
__device__ __forceinline__ void gt_stage_k(unsigned char* sm, const __nv_bfloat16* __restrict__ X, long long ld, int r0,
                                           int R, int k0, int ke, int rows)
{
#pragma unroll
    for (int v = 0; v < 8; ++v) {
        const int e = threadIdx.x + 128 * v;  // 8 rows x 8 vectors per 64 threads: rows fastest
        const int r = (e >> 6) * 8 + (e & 7), k8 = (e >> 3) & 7;
        const int k = k0 + 8 * k8;
        if (r >= rows) continue;
        uint4 w = make_uint4(0, 0, 0, 0);
        if (r0 + r < R && k < ke) w = *reinterpret_cast<const uint4*>(X + (long long)(r0 + r) * ld + k);
        *reinterpret_cast<uint4*>(sm + gt_off(r, k8)) = w;
    }
}
// the same of an operand stored along its rows: 8 x 8 blocks, transposed; R is a multiple of 8.
// SUM: adds the block's eight k into cs[8] (the column sums that are the bias gradient)
template <bool SUM>
__device__ __forceinline__ void gt_stage_r(unsigned char* sm, const __nv_bfloat16* __restrict__ X, long long ld, int r0,
                                           int R, int k0, int ke, int rows, float* cs)
{
    const int rb = threadIdx.x & 15, k8 = threadIdx.x >> 4;  // rows fastest: coalesced loads
    if (8 * rb >= rows) return;
    uint4 v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int k = k0 + 8 * k8 + q;
        v[q] = make_uint4(0, 0, 0, 0);
        if (r0 + 8 * rb < R && k < ke) v[q] = *reinterpret_cast<const uint4*>(X + (long long)k * ld + r0 + 8 * rb);
    }
    if (SUM) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const unsigned w[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                cs[2 * c] += __uint_as_float(w[c] << 16);
                cs[2 * c + 1] += __uint_as_float(w[c] & 0xffff0000u);
            }
        }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        unsigned w[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) w[q] = c == 0 ? v[q].x : c == 1 ? v[q].y : c == 2 ? v[q].z : v[q].w;
        *reinterpret_cast<uint4*>(sm + gt_off(8 * rb + 2 * c, k8)) =
            make_uint4(__byte_perm(w[0], w[1], 0x5410), __byte_perm(w[2], w[3], 0x5410),
                       __byte_perm(w[4], w[5], 0x5410), __byte_perm(w[6], w[7], 0x5410));
        *reinterpret_cast<uint4*>(sm + gt_off(8 * rb + 2 * c + 1, k8)) =
            make_uint4(__byte_perm(w[0], w[1], 0x7632), __byte_perm(w[2], w[3], 0x7632),
                       __byte_perm(w[4], w[5], 0x7632), __byte_perm(w[6], w[7], 0x7632));
    }
}

struct GemmArgs {
    int M, N, K;
    const __nv_bfloat16 *A, *B;
    long long lda, ldb;
    float* C;                   // EPI_PART, EPI_OUT: FP32 result (row stride N; slice z at + z * cstr)
    long long cstr;
    __nv_bfloat16* Cb;          // EPI_ACT, EPI_MASK: BF16 result (row stride N)
    const float* bias;          // EPI_ACT, EPI_OUT
    const __nv_bfloat16* mask;  // EPI_MASK: the activations whose positive entries pass
    float* csum;                // EPI_PART: column sums of A over k (the bias gradient), slice z at + z * cstr
    int kslice;                 // multiple of GT_K
};

template <bool AK, bool BK, int EPI>
__global__ void __launch_bounds__(128) k_gemm_tc(GemmArgs g, int* __restrict__ err)
{
    extern __shared__ __align__(128) unsigned char gsm[];
    __shared__ __align__(8) unsigned long long bar[2];
    __shared__ unsigned tslot;
    __shared__ float csh[EPI == EPI_PART ? 8 : 1][EPI == EPI_PART ? 128 : 1];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int i0 = blockIdx.x * 128, j0 = blockIdx.y * 128;
    const int kb = blockIdx.z * g.kslice, ke = min(g.K, kb + g.kslice);
    const int nn = min(128, ((g.N - j0) + 15) & ~15);  // columns of this tile (a multiple of 16)
    if (tid == 0) {
        for (int b = 0; b < 2; ++b)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_su32(&bar[b])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_su32(&tslot)),
                     "r"(128)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned taddr = tslot, idesc = tc_idesc(nn);
    float cs[8] = {};
    unsigned ph[2] = {0u, 0u};
    bool alive = true;
    int c = 0;
    for (int k0 = kb; k0 < ke; k0 += GT_K, ++c) {
        const int b = c & 1;
        unsigned char *As = gsm + b * 2 * GT_STAGE, *Bs = As + GT_STAGE;
        if (c >= 2) {  // the MMAs that read this stage two chunks ago are done
            if (!__syncthreads_and(tc_wait(tc_su32(&bar[b]), ph[b]))) {
                if (tid == 0) atomicExch(err, 1);
                tc_wait(tc_su32(&bar[b]), ph[b]);  // let the MMAs in flight finish before the memory goes
                tc_wait(tc_su32(&bar[b ^ 1]), ph[b ^ 1]);
                alive = false;
                break;
            }
            ph[b] ^= 1u;
        }
        if (AK) gt_stage_k(As, g.A, g.lda, i0, g.M, k0, ke, 128);
        else gt_stage_r<EPI == EPI_PART>(As, g.A, g.lda, i0, g.M, k0, ke, 128, cs);
        if (BK) gt_stage_k(Bs, g.B, g.ldb, j0, g.N, k0, ke, nn);
        else gt_stage_r<false>(Bs, g.B, g.ldb, j0, g.N, k0, ke, nn, cs);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (tid == 0) {
            const int steps = (min(GT_K, ke - k0) + 15) / 16;
            for (int ks = 0; ks < steps; ++ks) {
                const uint64_t ad = tc_desc(tc_su32(As) + ks * 2 * GT_LBO, GT_LBO, GT_SBO);
                const uint64_t bd = tc_desc(tc_su32(Bs) + ks * 2 * GT_LBO, GT_LBO, GT_SBO);
                asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                             " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
                             ::"r"(taddr), "l"(ad), "l"(bd), "r"(idesc), "r"((unsigned)(c > 0 || ks > 0)) : "memory");
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                         ::"r"(tc_su32(&bar[b])) : "memory");
        }
    }
    // the outstanding commits (the last two chunks')
    for (int d = max(0, c - 2); d < c && alive; ++d) {
        const int b = d & 1;
        if (!__syncthreads_and(tc_wait(tc_su32(&bar[b]), ph[b]))) {
            if (tid == 0) atomicExch(err, 1);
            tc_wait(tc_su32(&bar[b]), ph[b]);
            alive = false;
        }
        ph[b] ^= 1u;
    }
    tc_fence_after();
    const int i = i0 + 32 * warp + lane;
    for (int c0 = 0; c0 < nn && alive; c0 += 32) {
        float v[32];
        __syncwarp();
        if (c > 0) tc_ld32(taddr + ((unsigned)(32 * warp) << 16) + c0, v);  // (columns past nn are not used)
        else
            for (int q = 0; q < 32; ++q) v[q] = 0.f;
        if (i >= g.M) continue;
        const int w = min(32, nn - c0);  // 16 or 32
#pragma unroll
        for (int q = 0; q < 32; q += 8) {
            if (q >= w) break;
            const int j = j0 + c0 + q;
            const long long o = (long long)i * g.N + j;
            if (EPI == EPI_PART || EPI == EPI_OUT) {
                float* dst = g.C + (EPI == EPI_PART ? blockIdx.z * g.cstr : 0) + o;
#pragma unroll
                for (int h = 0; h < 8; h += 4) {
                    float4 f = make_float4(v[q + h], v[q + h + 1], v[q + h + 2], v[q + h + 3]);
                    if (EPI == EPI_OUT) {
                        const float* bi = g.bias + j + h;
                        f = make_float4(f.x + bi[0], f.y + bi[1], f.z + bi[2], f.w + bi[3]);
                    }
                    *reinterpret_cast<float4*>(dst + h) = f;
                }
            } else {
                __align__(16) __nv_bfloat16 r[8];
                if (EPI == EPI_ACT) {
#pragma unroll
                    for (int h = 0; h < 8; ++h) r[h] = __float2bfloat16(fmaxf(v[q + h] + g.bias[j + h], 0.f));
                } else {
                    const uint4 mk = *reinterpret_cast<const uint4*>(g.mask + o);
                    const unsigned mw[4] = {mk.x, mk.y, mk.z, mk.w};
#pragma unroll
                    for (int h = 0; h < 8; ++h) {
                        const float a = __uint_as_float(h & 1 ? mw[h >> 1] & 0xffff0000u : mw[h >> 1] << 16);
                        r[h] = __float2bfloat16(a > 0.f ? v[q + h] : 0.f);
                    }
                }
                *reinterpret_cast<uint4*>(g.Cb + o) = *reinterpret_cast<const uint4*>(r);
            }
        }
    }
    if (EPI == EPI_PART && alive && blockIdx.y == 0) {  // column sums: the threads' k groups in order
#pragma unroll
        for (int q = 0; q < 8; ++q) csh[tid >> 4][(tid & 15) * 8 + q] = cs[q];
        __syncthreads();
        float s = 0.f;
        for (int q = 0; q < 8; ++q) s += csh[q][tid];
        if (i0 + tid < g.M) g.csum[blockIdx.z * g.cstr + i0 + tid] = s;
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(128) : "memory");
}

template <bool AK, bool BK, int EPI>
static bool gemm(cudaStream_t st, GemmArgs g, int slices, int* err)
{
    if (cudaFuncSetAttribute(k_gemm_tc<AK, BK, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, GT_SMEM) !=
        cudaSuccess)
        return false;
    const int per = (g.K + slices - 1) / slices;
    g.kslice = (per + GT_K - 1) / GT_K * GT_K;
    const dim3 grid((g.M + 127) / 128, (g.N + 127) / 128, slices);
    k_gemm_tc<AK, BK, EPI><<<grid, 128, GT_SMEM, st>>>(g, err);
    return true;
}

// ---------- elementwise pieces ----------
// Before a training pass: the weights as BF16, the input rows (n x nin, FP32) as a zero-padded
// BF16 matrix (n x dpad), and a zero loss
__global__ void k_prepare(long long nw, const float* __restrict__ w, __nv_bfloat16* __restrict__ wb, int n, int nin,
                          int dpad, const float* __restrict__ X, __nv_bfloat16* __restrict__ Y, float* __restrict__ loss)
{
    const long long tot = (long long)n * dpad, stride = (long long)gridDim.x * blockDim.x;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0) *loss = 0.f;
    for (long long i = t; i < nw; i += stride) wb[i] = __float2bfloat16(w[i]);
    for (long long i = t; i < tot; i += stride) {
        int r = (int)(i / dpad), c = (int)(i % dpad);
        Y[i] = __float2bfloat16(c < nin ? X[(long long)r * nin + c] : 0.f);
    }
}

// output layer: dZ = 2 (Y - T) / (n nout) on the real outputs (BF16), loss partial sums
__global__ void k_mse(int n, int nout, int dpad, const float* __restrict__ Y, const float* __restrict__ T,
                      __nv_bfloat16* __restrict__ dZ, float* __restrict__ loss)
{
    __shared__ float red[256];
    float s = 0.f;
    long long tot = (long long)n * dpad;
    const float sc = 2.f / ((float)n * (float)nout);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < tot; i += (long long)gridDim.x * blockDim.x) {
        int r = (int)(i / dpad), c = (int)(i % dpad);
        float g = 0.f;
        if (c < nout) {
            float e = Y[i] - T[(long long)r * nout + c];
            s += e * e;
            g = sc * e;
        }
        dZ[i] = __float2bfloat16(g);
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(loss, red[0] / ((float)n * (float)nout));
}

// the gradient (and, with lpart, the loss): the slices' parts added in slice order (results do not
// depend on scheduling)
__global__ void k_sum_slices(long long n, int slices, const float* __restrict__ part, float* __restrict__ out,
                             const float* __restrict__ lpart, float* __restrict__ loss)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        float s = 0.f;
#pragma unroll 16
        for (int z = 0; z < slices; ++z) s += part[z * n + i];
        out[i] = s;
    }
    if (lpart && blockIdx.x == 0 && threadIdx.x == 0) {
        float s = 0.f;
        for (int z = 0; z < slices; ++z) s += lpart[z];
        *loss = s;
    }
}

// (err[0] set: the gradient is not whole; the step is left out and counted)
__global__ void k_adam(long long n, float* __restrict__ w, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ g, float lr, float b1, float b2, float c1, float c2, float eps,
                       int* __restrict__ err)
{
    if (err[0]) {
        if (blockIdx.x == 0 && threadIdx.x == 0) ++err[1];
        return;
    }
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        float gi = g[i];
        float mi = b1 * m[i] + (1.f - b1) * gi;
        float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

// deterministic initialisation: uniform(-s, s) with s = sqrt(6 / (fan_in + fan_out)) (SplitMix64)
__global__ void k_init(long long n, float* __restrict__ w, float s, unsigned long long seed)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        unsigned long long z = seed + 0x9E3779B97F4A7C15ULL * (unsigned long long)(i + 1);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
        z = z ^ (z >> 31);
        double u = (double)(z >> 11) * (1.0 / 9007199254740992.0);
        w[i] = (float)((2.0 * u - 1.0) * s);
    }
}

static int grid1(long long n) { return (int)std::min<long long>((n + 255) / 256, 152 * 8); }

// slices of the rows that a weight gradient sums over: of 128 rows or more (at 4096 rows 32 blocks
// per gradient; 2 slices of 2048 rows took 128 us each), at most 64, and at most 64 MB of parts
// (a wide network's gradients have tiles enough)
static int grad_slices(const pb_mlp* m, int n)
{
    const long long most = std::max(1LL, std::min(64LL, (16LL << 20) / m->nparam));
    return (int)std::max(1LL, std::min(most, (long long)n / 128));
}

static int ensure_cap(pb_mlp* m, int n)
{
    if (n <= m->cap) return PB_OK;
    cudaStreamSynchronize(m->st);
    cudaFree(m->Z);
    m->Z = nullptr;
    for (int l = 0; l <= m->nl; ++l) {
        cudaFree(m->Ab[l]);
        m->Ab[l] = nullptr;
    }
    int dmax = 16;
    for (int l = 0; l < m->nl; ++l) dmax = std::max(dmax, std::max(m->din[l], m->dout[l]));
    for (auto& d : m->dZb) {
        cudaFree(d);
        d = nullptr;
    }
    bool ok = cudaMalloc(&m->Z, sizeof(float) * (size_t)n * m->dout[m->nl - 1]) == cudaSuccess;
    for (int l = 0; l < m->nl; ++l)
        ok &= cudaMalloc(&m->Ab[l], sizeof(__nv_bfloat16) * (size_t)n * m->din[l]) == cudaSuccess;
    for (auto& d : m->dZb) ok &= cudaMalloc(&d, sizeof(__nv_bfloat16) * (size_t)n * dmax) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        m->cap = 0;
        return mlp_fail(m, PB_ERR_NOMEM, "mlp: out of memory");
    }
    m->cap = n;
    return PB_OK;
}

// the gradient's slices, and a loss per slice after them (only a backward pass needs them)
static int ensure_part(pb_mlp* m, int slices)
{
    if (slices <= m->part_n) return PB_OK;
    cudaStreamSynchronize(m->st);
    cudaFree(m->part);
    m->part = nullptr;
    m->part_n = 0;
    if (cudaMalloc(&m->part, sizeof(float) * ((size_t)m->nparam + 1) * slices) != cudaSuccess) {
        cudaGetLastError();
        return mlp_fail(m, PB_ERR_NOMEM, "mlp: out of memory");
    }
    m->part_n = slices;
    return PB_OK;
}

// forward pass over n rows; keeps the outputs and the BF16 activations for a backward pass
static int mlp_forward(pb_mlp* m, const float* X, int n)
{
    int rc = ensure_cap(m, n);
    if (rc) return rc;
    const long long most = std::max(m->nparam, (long long)n * m->din[0]);
    k_prepare<<<grid1(most), 256, 0, m->st>>>(m->nparam, m->W, m->Wb, n, m->nin, m->din[0], X, m->Ab[0], m->lossbuf);
    bool ok = true;
    for (int l = 0; l < m->nl; ++l) {
        // Z = A W^T: B(kk, j) = W[j][kk]
        GemmArgs g = {n, m->dout[l], m->din[l], m->Ab[l], m->Wb + m->woff[l], m->din[l], m->din[l]};
        g.bias = m->W + m->boff[l];
        if (l + 1 < m->nl) {
            g.Cb = m->Ab[l + 1];
            ok &= gemm<true, true, EPI_ACT>(m->st, g, 1, m->derr);
        } else {
            g.C = m->Z;
            ok &= gemm<true, true, EPI_OUT>(m->st, g, 1, m->derr);
        }
    }
    return ok && cudaGetLastError() == cudaSuccess ? PB_OK : mlp_fail(m, PB_ERR_CUDA, "mlp forward launch failed");
}

// backward pass after mlp_forward: gradients into m->G, loss into m->lossbuf
static int mlp_backward(pb_mlp* m, const float* T, int n)
{
    const int L = m->nl, slices = grad_slices(m, n);
    int rc = ensure_part(m, slices);
    if (rc) return rc;
    const int dl = m->dout[L - 1];
    k_mse<<<grid1((long long)n * dl), 256, 0, m->st>>>(n, m->nout, dl, m->Z, T, m->dZb[0], m->lossbuf);
    bool ok = true;
    int cur = 0;
    for (int l = L - 1; l >= 0; --l, cur ^= 1) {
        const int k = m->din[l], d = m->dout[l];
        // dW = dZ^T A: A-operand (i = out unit, kk = row) = dZ[kk][i]; B(kk = row, j = in) = A[kk][j];
        // db = the column sums of dZ
        GemmArgs w = {d, k, n, m->dZb[cur], m->Ab[l], d, k};
        w.C = m->part + m->woff[l];
        w.csum = m->part + m->boff[l];
        w.cstr = m->nparam;
        ok &= gemm<false, false, EPI_PART>(m->st, w, slices, m->derr);
        if (l > 0) {
            // dZ_prev = relu'(Z_prev) (dZ W): A(i = row, kk = out) = dZ[i][kk]; B(kk = out, j = in) = W[kk][j]
            GemmArgs g = {n, k, d, m->dZb[cur], m->Wb + m->woff[l], d, k};
            g.Cb = m->dZb[cur ^ 1];
            g.mask = m->Ab[l];
            ok &= gemm<true, false, EPI_MASK>(m->st, g, 1, m->derr);
        }
    }
    k_sum_slices<<<grid1(m->nparam), 256, 0, m->st>>>(m->nparam, slices, m->part, m->G, nullptr, nullptr);
    return ok && cudaGetLastError() == cudaSuccess ? PB_OK : mlp_fail(m, PB_ERR_CUDA, "mlp backward launch failed");
}

extern "C" int pb_mlp_create(int nin, int width, int depth, int nout, unsigned long long seed, void* stream,
                             pb_mlp** out)
{
    if (!out || nin < 1 || width < 16 || width % 16 || depth < 1 || depth + 1 > MLP_MAXL || nout < 1 || nout > 64)
        return PB_ERR_ARG;
    pb_mlp* m = new pb_mlp();
    m->nin = nin;
    m->width = width;
    m->depth = depth;
    m->nout = nout;
    m->nl = depth + 1;
    m->st = (cudaStream_t)stream;
    auto pad = [](int x) { return (x + 15) / 16 * 16; };
    long long o = 0;
    for (int l = 0; l < m->nl; ++l) {
        m->din[l] = l == 0 ? pad(nin) : width;
        m->dout[l] = l + 1 < m->nl ? width : pad(nout);
        m->woff[l] = o;
        o += (long long)m->din[l] * m->dout[l];
    }
    m->woff[m->nl] = o;
    for (int l = 0; l < m->nl; ++l) {
        m->boff[l] = o;
        o += m->dout[l];
    }
    m->boff[m->nl] = o;
    m->nparam = o;
    bool ok = cudaMalloc(&m->W, sizeof(float) * o) == cudaSuccess;
    ok &= cudaMalloc(&m->Wm, sizeof(float) * o) == cudaSuccess;
    ok &= cudaMalloc(&m->Wv, sizeof(float) * o) == cudaSuccess;
    ok &= cudaMalloc(&m->G, sizeof(float) * (o + 3)) == cudaSuccess;
    ok &= cudaMalloc(&m->Wb, sizeof(__nv_bfloat16) * o) == cudaSuccess;
    m->lossbuf = m->G + o;
    m->derr = (int*)(m->G + o + 1);
    ok = ok && cudaMemset(m->derr, 0, 2 * sizeof(int)) == cudaSuccess;
    // (without it, should the host have no pinned memory left, the copies go one by one)
    if (ok && o <= MLP_STAGE && cudaMallocHost(&m->hbuf, sizeof(float) * (o + 2)) != cudaSuccess) {
        cudaGetLastError();
        m->hbuf = nullptr;
    }
    if (!ok) {
        cudaGetLastError();
        delete m;
        return PB_ERR_NOMEM;
    }
    cudaMemsetAsync(m->W, 0, sizeof(float) * o, m->st);
    cudaMemsetAsync(m->Wm, 0, sizeof(float) * o, m->st);
    cudaMemsetAsync(m->Wv, 0, sizeof(float) * o, m->st);
    for (int l = 0; l < m->nl; ++l) {
        long long n = (long long)m->din[l] * m->dout[l];
        float s = sqrtf(6.f / (float)((l == 0 ? nin : width) + (l + 1 < m->nl ? width : nout)));
        k_init<<<grid1(n), 256, 0, m->st>>>(n, m->W + m->woff[l], s, seed + 7919ULL * l);
    }
    // padded input columns and output rows carry zero weights
    std::vector<float> h(o);
    cudaMemcpyAsync(h.data(), m->W, sizeof(float) * o, cudaMemcpyDeviceToHost, m->st);
    cudaStreamSynchronize(m->st);
    for (int l = 0; l < m->nl; ++l) {
        int realin = l == 0 ? nin : width, realout = l + 1 < m->nl ? width : nout;
        for (int j = 0; j < m->dout[l]; ++j)
            for (int kk = 0; kk < m->din[l]; ++kk)
                if (j >= realout || kk >= realin) h[m->woff[l] + (long long)j * m->din[l] + kk] = 0.f;
    }
    cudaMemcpyAsync(m->W, h.data(), sizeof(float) * o, cudaMemcpyHostToDevice, m->st);
    if (cudaStreamSynchronize(m->st) != cudaSuccess) {
        cudaGetLastError();
        delete m;
        return PB_ERR_CUDA;
    }
    *out = m;
    return PB_OK;
}

extern "C" int pb_mlp_destroy(pb_mlp* m)
{
    if (!m) return PB_OK;
    cudaStreamSynchronize(m->st);
    cudaFree(m->W);
    cudaFree(m->Wm);
    cudaFree(m->Wv);
    cudaFree(m->G);
    cudaFree(m->Wb);
    cudaFreeHost(m->hbuf);
    cudaFree(m->Z);
    for (int l = 0; l <= MLP_MAXL; ++l) cudaFree(m->Ab[l]);
    for (auto& d : m->dZb) cudaFree(d);
    cudaFree(m->part);
    delete m;
    return PB_OK;
}

extern "C" const char* pb_mlp_last_error(const pb_mlp* m) { return m ? m->err.c_str() : "null network"; }

extern "C" int pb_mlp_param_count(pb_mlp* m, long long* n)
{
    if (!m || !n) return PB_ERR_ARG;
    *n = m->nparam;
    return PB_OK;
}

extern "C" int pb_mlp_get_params(pb_mlp* m, float* host)
{
    if (!m || !host) return PB_ERR_ARG;
    if (cudaMemcpyAsync(host, m->W, sizeof(float) * m->nparam, cudaMemcpyDeviceToHost, m->st) != cudaSuccess ||
        cudaStreamSynchronize(m->st) != cudaSuccess)
        return mlp_fail(m, PB_ERR_CUDA, "mlp: copy failed");
    return PB_OK;
}

extern "C" int pb_mlp_set_params(pb_mlp* m, const float* host)
{
    if (!m || !host) return PB_ERR_ARG;
    if (cudaMemcpyAsync(m->W, host, sizeof(float) * m->nparam, cudaMemcpyHostToDevice, m->st) != cudaSuccess ||
        cudaStreamSynchronize(m->st) != cudaSuccess)
        return mlp_fail(m, PB_ERR_CUDA, "mlp: copy failed");
    return PB_OK;
}

// ---------- fused inference: every layer in one kernel ----------
// For width 128, a first layer of at most 32 padded inputs and at most 16 padded outputs: all
// weights are converted to BF16 once per block and every tile of rows runs through all layers
// inside the kernel, so the features are read once and two outputs written per row.
#define FUSED_W 128
struct MlpDesc {
    long long woff[MLP_MAXL], boff[MLP_MAXL];
    int nin, din0, nl, nout;  // inputs, padded inputs (row length of W_0), layers, outputs
};

// ---------- fused inference on the fifth-generation tensor cores (tcgen05) ----------
// The layers and rounding points of the layer-by-layer path, one tile of 128 rows at a time: the
// tile's BF16 activations sit in shared memory in the K-major layout without swizzle that the
// MMA reads through matrix descriptors (8 x 16-byte core matrices: the next core matrix along K
// 128 bytes on, the next group of 8 rows K / 8 x 128 bytes on); one thread issues the layer's
// tcgen05.mma instructions (M = 128, N = 128 or 16, K = 16 each, BF16 in, FP32 accumulate) into a
// 128-column tensor-memory accumulator and commits them to an mbarrier; each warp then reads its
// 32 rows back with tcgen05.ld, adds the bias, applies ReLU, rounds to BF16 and writes the next
// layer's operand in place. Every wait is bounded: a wait that gives up sets *err, lets the MMAs
// in flight finish (bounded again), frees the tensor memory and leaves.
static size_t tc_smem(int nl, int din0)
{
    return sizeof(__nv_bfloat16) * ((size_t)FUSED_W * din0 + (size_t)(nl - 2) * FUSED_W * FUSED_W + 16 * FUSED_W +
                                    (size_t)TC_ROWS * FUSED_W) +
           sizeof(float) * ((size_t)(nl - 1) * FUSED_W + 16) + 128;
}

__global__ void __launch_bounds__(128, 1) k_mlp_tc(int n, const float* __restrict__ X, const float* __restrict__ W,
                                                   MlpDesc md, float* __restrict__ Y, int* __restrict__ err)
{
    extern __shared__ __align__(128) unsigned char tsm[];
    __shared__ __align__(8) unsigned long long bar;
    __shared__ unsigned tslot;
    const int nl = md.nl, din0 = md.din0;
    __nv_bfloat16* w0 = (__nv_bfloat16*)tsm;                           // [128 x din0]
    __nv_bfloat16* wh = w0 + FUSED_W * din0;                           // [nl-2][128 x 128]
    __nv_bfloat16* wl = wh + (size_t)(nl - 2) * FUSED_W * FUSED_W;     // [16 x 128]
    __nv_bfloat16* as = wl + 16 * FUSED_W;                             // [128 x 128] activations
    float* bs = (float*)(as + TC_ROWS * FUSED_W);                      // [nl-1][128] then [16]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // weights (row o of layer l is output o: the B operand, K-major) and biases
    for (int i = tid; i < FUSED_W * din0; i += 128)
        *(__nv_bfloat16*)((char*)w0 + tc_off(i / din0, i % din0, din0)) = __float2bfloat16(W[md.woff[0] + i]);
    for (int l = 1; l < nl - 1; ++l)
        for (int i = tid; i < FUSED_W * FUSED_W; i += 128)
            *(__nv_bfloat16*)((char*)(wh + (size_t)(l - 1) * FUSED_W * FUSED_W) + tc_off(i / FUSED_W, i % FUSED_W, FUSED_W)) =
                __float2bfloat16(W[md.woff[l] + i]);
    for (int i = tid; i < 16 * FUSED_W; i += 128)
        *(__nv_bfloat16*)((char*)wl + tc_off(i / FUSED_W, i % FUSED_W, FUSED_W)) = __float2bfloat16(W[md.woff[nl - 1] + i]);
    for (int l = 0; l < nl - 1; ++l)
        for (int i = tid; i < FUSED_W; i += 128) bs[l * FUSED_W + i] = W[md.boff[l] + i];
    for (int i = tid; i < 16; i += 128) bs[(nl - 1) * FUSED_W + i] = W[md.boff[nl - 1] + i];
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_su32(&bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_su32(&tslot)),
                     "r"(FUSED_W)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned taddr = tslot, tw = taddr + ((unsigned)(32 * warp) << 16);
    unsigned ph = 0u;
    bool alive = true;
    const int ntiles = (n + TC_ROWS - 1) / TC_ROWS;
    for (int tile = blockIdx.x; tile < ntiles && alive; tile += gridDim.x) {
        // the tile's features, BF16, zero beyond nin and beyond n, in the layer-0 layout
        {
            const int r = tid, row = tile * TC_ROWS + r;
            for (int k0 = 0; k0 < din0; k0 += 8) {
                __align__(16) __nv_bfloat16 v[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int c = k0 + q;
                    v[q] = __float2bfloat16(row < n && c < md.nin ? X[(size_t)row * md.nin + c] : 0.f);
                }
                *(uint4*)((char*)as + tc_off(r, k0, din0)) = *(const uint4*)v;
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        for (int l = 0; l < nl && alive; ++l) {
            const bool last = l == nl - 1;
            const int K = l == 0 ? din0 : FUSED_W, nn = last ? 16 : FUSED_W;
            const __nv_bfloat16* wb = l == 0 ? w0 : last ? wl : wh + (size_t)(l - 1) * FUSED_W * FUSED_W;
            if (tid == 0) {
                const unsigned sbo = (K / 8) * 128, id = tc_idesc(nn);
                for (int ks = 0; ks < K / 16; ++ks) {
                    const uint64_t ad = tc_desc(tc_su32(as) + ks * 256, 128, sbo);
                    const uint64_t bd = tc_desc(tc_su32(wb) + ks * 256, 128, sbo);
                    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                                 " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
                                 ::"r"(taddr), "l"(ad), "l"(bd), "r"(id), "r"((unsigned)(ks > 0)) : "memory");
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                             ::"r"(tc_su32(&bar)) : "memory");
            }
            if (!__syncthreads_and(tc_wait(tc_su32(&bar), ph))) {
                if (tid == 0) atomicExch(err, 1);
                tc_wait(tc_su32(&bar), ph);  // let the MMAs in flight finish before the memory goes
                alive = false;
                break;
            }
            ph ^= 1u;
            tc_fence_after();
            const float* bias = bs + l * FUSED_W;
            const int r = 32 * warp + lane, row = tile * TC_ROWS + r;
            if (last) {
                float v[32];
                tc_ld32(tw, v);  // (columns 16..31 are not part of this layer's result)
                for (int c = 0; c < md.nout; ++c)
                    if (row < n) Y[(size_t)row * md.nout + c] = v[c] + bias[c];
            } else {
                for (int c0 = 0; c0 < FUSED_W; c0 += 32) {
                    float v[32];
                    tc_ld32(tw + c0, v);
#pragma unroll
                    for (int q0 = 0; q0 < 32; q0 += 8) {
                        __align__(16) __nv_bfloat16 o[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) o[q] = __float2bfloat16(fmaxf(v[q0 + q] + bias[c0 + q0 + q], 0.f));
                        *(uint4*)((char*)as + tc_off(r, c0 + q0, FUSED_W)) = *(const uint4*)o;
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            tc_fence_before();
            __syncthreads();
            tc_fence_after();
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(FUSED_W) : "memory");
}

static bool fused_ok(const pb_mlp* m)
{
    return m->width == FUSED_W && m->din[0] <= 32 && m->dout[m->nl - 1] == 16 && m->nl >= 2 &&
           tc_smem(m->nl, m->din[0]) <= 200 * 1024;
}

static MlpDesc mlp_desc(const pb_mlp* m)
{
    MlpDesc md;
    for (int l = 0; l < MLP_MAXL; ++l) {
        md.woff[l] = l < m->nl ? m->woff[l] : 0;
        md.boff[l] = l < m->nl ? m->boff[l] : 0;
    }
    md.nin = m->nin;
    md.din0 = m->din[0];
    md.nl = m->nl;
    md.nout = m->nout;
    return md;
}

static int mlp_forward_fused(pb_mlp* m, const float* X, int n, float* Y)
{
    const size_t smem = tc_smem(m->nl, m->din[0]);
    if (cudaFuncSetAttribute(k_mlp_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return mlp_fail(m, PB_ERR_CUDA, "mlp: shared memory attribute failed");
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int tiles = (n + TC_ROWS - 1) / TC_ROWS;
    const int grid = std::max(1, std::min(tiles, nsm));  // one block per SM (its tensor memory and shared memory)
    k_mlp_tc<<<grid, 128, smem, m->st>>>(n, X, m->W, mlp_desc(m), Y, m->derr);
    if (cudaGetLastError() != cudaSuccess) return mlp_fail(m, PB_ERR_CUDA, "mlp fused forward launch failed");
    return mlp_check_err(m);
}

extern "C" int pb_mlp_forward(pb_mlp* m, const float* X, int n, float* Y)
{
    if (!m || !X || !Y || n < 1) return PB_ERR_ARG;
    if (fused_ok(m)) return mlp_forward_fused(m, X, n, Y);
    int rc = mlp_forward(m, X, n);
    if (rc) return rc;
    // real outputs of the last layer, row-major n x nout
    const int L = m->nl, dl = m->dout[L - 1];
    if (cudaMemcpy2DAsync(Y, sizeof(float) * m->nout, m->Z, sizeof(float) * dl, sizeof(float) * m->nout, n,
                          cudaMemcpyDeviceToDevice, m->st) != cudaSuccess)
        return mlp_fail(m, PB_ERR_CUDA, "mlp: output copy failed");
    return mlp_check_err(m);
}

// ---------- fused gradient: forward and backward of a tile of rows in one kernel ----------
// For the networks of the fused inference: one block per 128 rows runs the tile through all layers
// and back, every weight gradient included, with the rounding points of the layer-by-layer passes
// (BF16 activations and dZ, FP32 accumulation and bias, one FP32 part per slice of rows, parts added
// in slice order). Those are a chain of a dozen launches whose blocks mostly wait for their own
// loads; here only the weights and the rows come from memory. All operands sit in shared memory in
// the row-major K-major layout without swizzle, once: the backward products read the same core
// matrices (8 rows x 16 bytes) as MN-major operands through the transpose bits of the instruction
// descriptor, the core matrices along the outer index then being the descriptor's stride and those
// along K its leading offset. dZ of a layer replaces the activations it was masked with. A weight
// gradient is computed as its transpose (lanes = inputs), so that a column leaves tensor memory as
// 128 contiguous bytes per warp (by rows, each lane's stores would go to a line of their own),
// and is stored while the next layer's products run (two accumulators, 128 columns each).
// What bounds it: the chain of 2 nl - 1 dependent steps of a tile (MMA, tensor memory to
// registers, shared memory). A gradient of 4096 rows (18-128-128-128-2, to the host) takes 63 us,
// and 215 us in twelve launches.
#define FG_T 256
static size_t fg_smem(int nl, int din0)
{
    return sizeof(__nv_bfloat16) * ((size_t)2 * FUSED_W * din0 + (size_t)(2 * nl - 3) * FUSED_W * FUSED_W + 32 * FUSED_W) +
           sizeof(float) * ((size_t)(nl - 1) * FUSED_W + 16) + 128;
}

// D = A B over `steps` K steps of 16; a, b: start, leading offset, stride, bytes per K step
struct TcOp {
    unsigned at, lbo, sbo, step;
};
__device__ __forceinline__ TcOp tc_kmaj(const void* p, int cols) { return {tc_su32(p), 128u, (unsigned)cols * 16u, 256u}; }
__device__ __forceinline__ TcOp tc_mnmaj(const void* p, int cols)
{
    return {tc_su32(p), (unsigned)cols * 16u, 128u, (unsigned)cols * 32u};
}
__device__ __forceinline__ void tc_gemm(unsigned d, TcOp a, TcOp b, int steps, unsigned idesc)
{
    for (int ks = 0; ks < steps; ++ks) {
        const uint64_t ad = tc_desc(a.at + ks * a.step, a.lbo, a.sbo), bd = tc_desc(b.at + ks * b.step, b.lbo, b.sbo);
        asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                     " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
                     ::"r"(d), "l"(ad), "l"(bd), "r"(idesc), "r"((unsigned)(ks > 0)) : "memory");
    }
}
#define TC_TRA (1u << 15)  // A, B stored along M, N
#define TC_TRB (1u << 16)

// rows x cols FP32 weights (cols a multiple of 16) as BF16 in the K-major layout
__device__ __forceinline__ void fg_weights(unsigned char* sm, const float* __restrict__ w, int rows, int cols)
{
    const int k8n = cols >> 3, tot = rows * k8n;
#pragma unroll 8
    for (int e = threadIdx.x; e < tot; e += FG_T) {  // 8 rows fastest: full sectors, no bank conflicts
        const int r = (e & 7) + 8 * ((e >> 3) / k8n), k8 = (e >> 3) % k8n;
        const float4* src = reinterpret_cast<const float4*>(w + (size_t)r * cols + 8 * k8);
        const float4 a = src[0], b = src[1];
        __nv_bfloat162 o[4] = {__floats2bfloat162_rn(a.x, a.y), __floats2bfloat162_rn(a.z, a.w),
                               __floats2bfloat162_rn(b.x, b.y), __floats2bfloat162_rn(b.z, b.w)};
        *reinterpret_cast<uint4*>(sm + tc_off(r, 8 * k8, cols)) = *reinterpret_cast<const uint4*>(o);
    }
}

__global__ void __launch_bounds__(FG_T, 1) k_mlp_grad_tc(int n, const float* __restrict__ X, const float* __restrict__ T,
                                                         const float* __restrict__ W, MlpDesc md, float* __restrict__ part,
                                                         long long pstr, float* __restrict__ lpart, int* __restrict__ err)
{
    extern __shared__ __align__(128) unsigned char tsm[];
    __shared__ __align__(8) unsigned long long bar;
    __shared__ unsigned tslot;
    __shared__ float red[4];
    constexpr int HB = FUSED_W * FUSED_W * 2;  // bytes of a 128 x 128 operand
    const int nl = md.nl, din0 = md.din0;
    unsigned char* w0 = tsm;                          // [128 x din0]
    unsigned char* wh = w0 + FUSED_W * din0 * 2;      // [nl-2][128 x 128]
    unsigned char* wl = wh + (size_t)(nl - 2) * HB;   // [16 x 128]
    unsigned char* xs = wl + 16 * FUSED_W * 2;        // [128 x din0] the input rows
    unsigned char* as = xs + TC_ROWS * din0 * 2;      // [nl-1][128 x 128] activations, later dZ
    unsigned char* dz = as + (size_t)(nl - 1) * HB;   // [128 x 16] dZ of the output layer
    float* bs = (float*)(dz + TC_ROWS * 16 * 2);      // [nl-1][128] then [16]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int half = warp >> 2;                       // columns [64 half, 64 half + 64)
    const int r = 32 * (warp & 3) + lane;             // tensor-memory lane
    part += blockIdx.x * pstr;
    fg_weights(w0, W + md.woff[0], FUSED_W, din0);
    for (int l = 1; l < nl - 1; ++l) fg_weights(wh + (size_t)(l - 1) * HB, W + md.woff[l], FUSED_W, FUSED_W);
    fg_weights(wl, W + md.woff[nl - 1], 16, FUSED_W);
    for (int l = 0; l < nl - 1; ++l)
        for (int i = tid; i < FUSED_W; i += FG_T) bs[l * FUSED_W + i] = W[md.boff[l] + i];
    if (tid < 16) bs[(nl - 1) * FUSED_W + tid] = W[md.boff[nl - 1] + tid];
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_su32(&bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_su32(&tslot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned taddr = tslot, tlane = (unsigned)(32 * (warp & 3)) << 16;
    const float sc = 2.f / ((float)n * (float)md.nout);
    unsigned ph = 0u;
    bool alive = true, first = true;
    const int ntiles = (n + TC_ROWS - 1) / TC_ROWS;

    // end of a step: this thread's shared-memory writes and tensor-memory reads before the next MMAs
    auto step = [&]() {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
    };
    auto commit = [&]() {
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                     ::"r"(tc_su32(&bar)) : "memory");
    };
    auto wait = [&]() {
        if (!__syncthreads_and(tc_wait(tc_su32(&bar), ph))) {
            if (tid == 0) atomicExch(err, 1);
            tc_wait(tc_su32(&bar), ph);  // let the MMAs in flight finish before the memory goes
            alive = false;
        }
        ph ^= 1u;
        tc_fence_after();
    };
    auto put = [&](long long o, float v) { part[o] = first ? v : part[o] + v; };
    // the weight gradient of layer l, out of its accumulator
    auto store_dw = [&](int l) {
        const unsigned t = taddr + 128u + 128u * (l & 1) + tlane;
        float v[32];
        if (l == 0) {  // lanes = outputs, columns = inputs
            if (half) return;
            tc_ld32(t, v);
#pragma unroll
            for (int c = 0; c < 32; ++c)
                if (c < din0) put(md.woff[0] + (long long)r * din0 + c, v[c]);
        } else if (l == nl - 1) {  // lanes = inputs, columns = outputs
            if (half) return;
            tc_ld32(t, v);
#pragma unroll
            for (int c = 0; c < 16; ++c) put(md.woff[l] + c * FUSED_W + r, v[c]);
        } else {
            for (int c0 = 64 * half; c0 < 64 * half + 64; c0 += 32) {
                tc_ld32(t + c0, v);
#pragma unroll
                for (int c = 0; c < 32; ++c) put(md.woff[l] + (long long)(c0 + c) * FUSED_W + r, v[c]);
            }
        }
    };
    // the bias gradient: column sums of dZ, 8 columns x 8 rows at a time per warp
    auto store_db = [&](int l, const unsigned char* z, int cols) {
        for (int g = warp; g < cols / 8; g += FG_T / 32) {
            float a = 0.f, b = 0.f;
#pragma unroll
            for (int q = 0; q < TC_ROWS / 8; ++q) {
                const unsigned u = *reinterpret_cast<const unsigned*>(z + (size_t)q * cols * 16 + g * 128 + lane * 4);
                a += __uint_as_float(u << 16);
                b += __uint_as_float(u & 0xffff0000u);
            }
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) {
                a += __shfl_xor_sync(0xffffffffu, a, o);
                b += __shfl_xor_sync(0xffffffffu, b, o);
            }
            if (lane < 4) {
                put(md.boff[l] + 8 * g + 2 * lane, a);
                put(md.boff[l] + 8 * g + 2 * lane + 1, b);
            }
        }
    };

    for (int tile = blockIdx.x; tile < ntiles && alive; tile += gridDim.x) {
        const int row = tile * TC_ROWS + r;
        for (int k0 = 8 * half; k0 < din0; k0 += 16) {
            __align__(16) __nv_bfloat16 v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int c = k0 + q;
                v[q] = __float2bfloat16(row < n && c < md.nin ? X[(size_t)row * md.nin + c] : 0.f);
            }
            *(uint4*)(xs + tc_off(r, k0, din0)) = *(const uint4*)v;
        }
        step();
        // forward
        for (int l = 0; l < nl && alive; ++l) {
            const bool last = l == nl - 1;
            const int K = l == 0 ? din0 : FUSED_W;
            if (tid == 0) {
                const unsigned char* a = l == 0 ? xs : as + (size_t)(l - 1) * HB;
                const unsigned char* w = l == 0 ? w0 : last ? wl : wh + (size_t)(l - 1) * HB;
                tc_gemm(taddr, tc_kmaj(a, K), tc_kmaj(w, K), K / 16, tc_idesc(last ? 16 : FUSED_W));
                commit();
            }
            wait();
            if (!alive) break;
            const float* bias = bs + l * FUSED_W;
            if (last) {  // dZ = 2 (Y - T) / (n nout) on the real outputs and rows; the loss
                if (half == 0) {
                    float v[32], s = 0.f;
                    tc_ld32(taddr + tlane, v);
                    __align__(16) __nv_bfloat16 o[16];
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        float g = 0.f;
                        if (c < md.nout && row < n) {
                            const float e = v[c] + bias[c] - T[(size_t)row * md.nout + c];
                            s += e * e;
                            g = sc * e;
                        }
                        o[c] = __float2bfloat16(g);
                    }
                    *(uint4*)(dz + tc_off(r, 0, 16)) = *(const uint4*)o;
                    *(uint4*)(dz + tc_off(r, 8, 16)) = *(const uint4*)(o + 8);
#pragma unroll
                    for (int o2 = 16; o2 > 0; o2 >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o2);
                    if (lane == 0) red[warp] = s;
                }
            } else {
                for (int c0 = 64 * half; c0 < 64 * half + 64; c0 += 32) {
                    float v[32];
                    tc_ld32(taddr + tlane + c0, v);
#pragma unroll
                    for (int q0 = 0; q0 < 32; q0 += 8) {
                        __align__(16) __nv_bfloat16 o[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            o[q] = __float2bfloat16(row < n ? fmaxf(v[q0 + q] + bias[c0 + q0 + q], 0.f) : 0.f);
                        *(uint4*)(as + (size_t)l * HB + tc_off(r, c0 + q0, FUSED_W)) = *(const uint4*)o;
                    }
                }
            }
            step();
        }
        if (!alive) break;
        if (tid == 0) {
            const float s = (red[0] + red[1] + red[2] + red[3]) / ((float)n * (float)md.nout);
            lpart[blockIdx.x] = first ? s : lpart[blockIdx.x] + s;
        }
        // backward: dZ of layer l in dz (the output layer) or in place of the activations l + 1
        for (int l = nl - 1; l >= 0 && alive; --l) {
            const bool last = l == nl - 1;
            const int N = last ? 16 : FUSED_W;
            unsigned char* z = last ? dz : as + (size_t)l * HB;
            unsigned char* a = l == 0 ? xs : as + (size_t)(l - 1) * HB;
            if (tid == 0) {
                const unsigned acc = taddr + 128u + 128u * (l & 1);
                if (l > 0) {
                    const unsigned char* w = last ? wl : wh + (size_t)(l - 1) * HB;
                    tc_gemm(taddr, tc_kmaj(z, N), tc_mnmaj(w, FUSED_W), N / 16, tc_idesc(FUSED_W) | TC_TRB);
                    tc_gemm(acc, tc_mnmaj(a, FUSED_W), tc_mnmaj(z, N), TC_ROWS / 16, tc_idesc(N) | TC_TRA | TC_TRB);
                } else {
                    tc_gemm(acc, tc_mnmaj(z, FUSED_W), tc_mnmaj(a, din0), TC_ROWS / 16, tc_idesc(din0) | TC_TRA | TC_TRB);
                }
                commit();
            }
            __syncwarp();
            if (!last) store_dw(l + 1);
            store_db(l, z, N);
            wait();
            if (!alive) break;
            if (l > 0) {  // dZ of layer l - 1 = relu'(Z) dA
                for (int c0 = 64 * half; c0 < 64 * half + 64; c0 += 32) {
                    float v[32];
                    tc_ld32(taddr + tlane + c0, v);
#pragma unroll
                    for (int q0 = 0; q0 < 32; q0 += 8) {
                        uint4* at = (uint4*)(a + tc_off(r, c0 + q0, FUSED_W));
                        const uint4 mk = *at;
                        const unsigned mw[4] = {mk.x, mk.y, mk.z, mk.w};
                        __align__(16) __nv_bfloat16 o[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const float m = __uint_as_float(q & 1 ? mw[q >> 1] & 0xffff0000u : mw[q >> 1] << 16);
                            o[q] = __float2bfloat16(m > 0.f ? v[q0 + q] : 0.f);
                        }
                        *at = *(const uint4*)o;
                    }
                }
            }
            step();
        }
        if (alive) store_dw(0);
        tc_fence_before();
        first = false;
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(512) : "memory");
}

// the loss and the gradient of a batch into m->lossbuf and m->G: fused where a tile's operands of
// all layers fit in shared memory (width 128, up to 32 inputs, 16 outputs and 3 hidden layers),
// else layer by layer (4096 rows, 18-128-128-128-2, to the host: 63 us fused, 215 us layer by layer)
static int mlp_loss_grad(pb_mlp* m, const float* X, const float* T, int n)
{
    const size_t need = fg_smem(m->nl, m->din[0]), smem = 225 * 1024;  // one block per SM: it takes all tensor memory
    if (!fused_ok(m) || need > smem) {
        const int rc = mlp_forward(m, X, n);
        return rc ? rc : mlp_backward(m, T, n);
    }
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int slices = std::max(1, std::min((n + TC_ROWS - 1) / TC_ROWS, nsm));
    const int rc = ensure_part(m, slices);
    if (rc) return rc;
    if (cudaFuncSetAttribute(k_mlp_grad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return mlp_fail(m, PB_ERR_CUDA, "mlp: shared memory attribute failed");
    k_mlp_grad_tc<<<slices, FG_T, smem, m->st>>>(n, X, T, m->W, mlp_desc(m), m->part, m->nparam,
                                                 m->part + (size_t)m->nparam * m->part_n, m->derr);
    k_sum_slices<<<grid1(m->nparam), 256, 0, m->st>>>(m->nparam, slices, m->part, m->G,
                                                      m->part + (size_t)m->nparam * m->part_n, m->lossbuf);
    return cudaGetLastError() == cudaSuccess ? PB_OK : mlp_fail(m, PB_ERR_CUDA, "mlp gradient launch failed");
}

// Synchronises; PB_ERR_TIMEOUT (the flag cleared, Adam's count of steps without those left out) if a bounded
// wait of a tensor-core kernel gave up. loss: the loss of the last gradient, or nullptr
static int mlp_check_err(pb_mlp* m, float* loss)
{
    struct {
        float loss;
        int err, skipped;
    } h = {};
    if (cudaMemcpyAsync(&h, m->lossbuf, sizeof(h), cudaMemcpyDeviceToHost, m->st) != cudaSuccess ||
        cudaStreamSynchronize(m->st) != cudaSuccess)
        return mlp_fail(m, PB_ERR_CUDA, "mlp: sync failed");
    if (loss) *loss = h.loss;
    if (!h.err) return PB_OK;
    m->adam_t -= h.skipped;
    cudaMemsetAsync(m->derr, 0, 2 * sizeof(int), m->st);
    return mlp_fail(m, PB_ERR_TIMEOUT, "mlp: a bounded wait on the tensor cores gave up");
}

extern "C" int pb_mlp_set_wait_flag(pb_mlp* m)
{
    if (!m) return PB_ERR_ARG;
    const int one = 1;
    if (cudaMemcpyAsync(m->derr, &one, sizeof(int), cudaMemcpyHostToDevice, m->st) != cudaSuccess ||
        cudaStreamSynchronize(m->st) != cudaSuccess)
        return mlp_fail(m, PB_ERR_CUDA, "mlp: copy failed");
    return PB_OK;
}

extern "C" int pb_mlp_gradient(pb_mlp* m, const float* X, const float* T, int n, float* loss, float* grad_host)
{
    if (!m || !X || !T || n < 1) return PB_ERR_ARG;
    int rc = mlp_loss_grad(m, X, T, n);
    if (rc) return rc;
    if (m->hbuf && grad_host) {  // gradient, loss and flag in one copy
        if (cudaMemcpyAsync(m->hbuf, m->G, sizeof(float) * (m->nparam + 2), cudaMemcpyDeviceToHost, m->st) != cudaSuccess)
            return mlp_fail(m, PB_ERR_CUDA, "mlp: copy failed");
        if (cudaStreamSynchronize(m->st) != cudaSuccess) return mlp_fail(m, PB_ERR_CUDA, "mlp: sync failed");
        if (loss) *loss = m->hbuf[m->nparam];
        memcpy(grad_host, m->hbuf, sizeof(float) * m->nparam);
        int herr;
        memcpy(&herr, m->hbuf + m->nparam + 1, sizeof(int));
        return herr ? mlp_check_err(m) : PB_OK;
    }
    if (loss && cudaMemcpyAsync(loss, m->lossbuf, sizeof(float), cudaMemcpyDeviceToHost, m->st) != cudaSuccess)
        return mlp_fail(m, PB_ERR_CUDA, "mlp: copy failed");
    if (grad_host &&
        cudaMemcpyAsync(grad_host, m->G, sizeof(float) * m->nparam, cudaMemcpyDeviceToHost, m->st) != cudaSuccess)
        return mlp_fail(m, PB_ERR_CUDA, "mlp: copy failed");
    if (cudaStreamSynchronize(m->st) != cudaSuccess) return mlp_fail(m, PB_ERR_CUDA, "mlp: sync failed");
    return mlp_check_err(m);
}

extern "C" int pb_mlp_train_step(pb_mlp* m, const float* X, const float* T, int n, float lr, float* loss)
{
    if (!m || !X || !T || n < 1 || !(lr > 0)) return PB_ERR_ARG;
    int rc = mlp_loss_grad(m, X, T, n);
    if (rc) return rc;
    m->adam_t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    float c1 = 1.f - powf(b1, (float)m->adam_t), c2 = 1.f - powf(b2, (float)m->adam_t);
    k_adam<<<grid1(m->nparam), 256, 0, m->st>>>(m->nparam, m->W, m->Wm, m->Wv, m->G, lr, b1, b2, c1, c2, 1e-8f, m->derr);
    if (cudaGetLastError() != cudaSuccess) return mlp_fail(m, PB_ERR_CUDA, "mlp: launch failed");
    return loss ? mlp_check_err(m, loss) : PB_OK;
}

// ---------- features of the learned warm start ----------
// Per element, in element order (16 columns; r = distance from the centroid c to charge k):
//   0-2   c minus the mean charge position, over the radius of gyration of the centroids
//   3-5   unit normal
//   6     log(A / mean A)
//   7     curvature: 1 - mean n_i . n_j over the other triangles sharing a vertex with i
//   8, 9  S1 and S2 at the centroid (the source terms of eqbim_3/eqbim_4)
//   10    U = sum_k |q_k| / (4 pi r)
//   11    distance to the nearest charge / 3 Angstrom
//   12    screened source sum_k q_k exp(-kappa r) / (4 pi eps_in r)
//   13,14 smoothed sources sum_k q_k / (4 pi eps_in sqrt(r^2 + a^2)), a = 4 and 8 Angstrom
//   15    charge density around c: sum_k exp(-r^2 / 50) / 10
//   16,17 smoothed normal fields -sum_k q_k n.(c - x_k) / (4 pi eps_in (r^2 + a^2)^(3/2)),
//         a = 4 and 8 Angstrom
// Columns 8, 9, 10, 12, 13, 14, 16 and 17 are divided by their root mean square over the
// molecule.
// Targets: phi / (rms S1 * 2 eps_in / (eps_in + eps_out)) and
// dphi / (rms S2 * 2 eps_out / (eps_in + eps_out)) -- the image-charge values at a flat
// dielectric interface, so that targets are O(1) for molecules of any size and charge.
#define NFEAT 18
#define NSTAT 20  // column normalisers [0, 18) and the two target scales [18], [19]

struct PoolTmp {
    pb_ctx* c;
    void* p = nullptr;
    PoolTmp(pb_ctx* cc, size_t bytes) : c(cc)
    {
        if (cudaMallocFromPoolAsync(&p, bytes, c->pool, c->st) != cudaSuccess) {
            cudaGetLastError();
            p = nullptr;
        }
    }
    ~PoolTmp()
    {
        if (p) cudaFreeAsync(p, c->st);
    }
};

// raw columns in sorted order. The charge sums run in FP32 (coordinates relative to the charge
// centre, charges staged through shared memory 256 at a time), each tile's partial sums added
// into FP64: the features only feed the network, and FP32 keeps this pass to a few ms even for
// 200k elements x 2000 charges.
#define FT 256
__global__ void __launch_bounds__(FT) k_feat_pass(int nt, int nc, const double4_32a* __restrict__ ep,
                                                  const double4_32a* __restrict__ en,
                                                  const double* __restrict__ qpos, const double* __restrict__ q,
                                                  const int* __restrict__ toff, const int* __restrict__ tj, double cx,
                                                  double cy, double cz, double eps_in, double kappa,
                                                  float* __restrict__ raw)
{
    __shared__ float4 sq[FT];
    const int k = blockIdx.x * FT + threadIdx.x;
    const bool act = k < nt;
    double4_32a p = {0, 0, 0, 0}, n = {0, 0, 0, 0};
    if (act) {
        p = ep[k];
        n = en[k];
    }
    const float px = (float)(p.x - cx), py = (float)(p.y - cy), pz = (float)(p.z - cz);
    const float nx = (float)n.x, ny = (float)n.y, nz = (float)n.z, kap = (float)kappa;
    double s1 = 0, s2 = 0, u = 0, sk = 0, sa4 = 0, sa8 = 0, dens = 0, e4 = 0, e8 = 0;
    float dmin2 = 3.0e38f;
    for (int t0 = 0; t0 < nc; t0 += FT) {
        __syncthreads();
        if (t0 + threadIdx.x < nc) {
            const int t = t0 + threadIdx.x;
            sq[threadIdx.x] = make_float4((float)(qpos[3 * t] - cx), (float)(qpos[3 * t + 1] - cy),
                                          (float)(qpos[3 * t + 2] - cz), (float)q[t]);
        }
        __syncthreads();
        const int m = min(FT, nc - t0);
        float f1 = 0, f2 = 0, fu = 0, fk = 0, f4 = 0, f8 = 0, fd = 0, g4 = 0, g8 = 0;
        for (int j = 0; j < m; ++j) {
            const float4 c = sq[j];
            const float dx = px - c.x, dy = py - c.y, dz = pz - c.z;
            const float r2 = dx * dx + dy * dy + dz * dz, ri = rsqrtf(r2);
            const float nd = nx * dx + ny * dy + nz * dz;
            const float w4 = rsqrtf(r2 + 16.f), w8 = rsqrtf(r2 + 64.f);
            f1 += c.w * ri;
            f2 -= c.w * nd * ri * ri * ri;
            fu += fabsf(c.w) * ri;
            fk += c.w * __expf(-kap * r2 * ri) * ri;
            f4 += c.w * w4;
            f8 += c.w * w8;
            g4 -= c.w * nd * w4 * w4 * w4;
            g8 -= c.w * nd * w8 * w8 * w8;
            fd += __expf(-r2 * 0.02f);
            dmin2 = fminf(dmin2, r2);
        }
        s1 += f1;
        s2 += f2;
        u += fu;
        sk += fk;
        sa4 += f4;
        sa8 += f8;
        e4 += g4;
        e8 += g8;
        dens += fd;
    }
    if (!act) return;
    double curv = 0;
    int cnt = 0;
    for (int t = toff[k]; t < toff[k + 1]; ++t) {
        int j = tj[t];
        if (j == k) continue;
        double4_32a m2 = en[j];
        curv += n.x * m2.x + n.y * m2.y + n.z * m2.z;
        ++cnt;
    }
    curv = cnt ? 1.0 - curv / cnt : 0.0;
    const double i4pi = 0.07957747154594767;
    float* r = raw + (size_t)k * NFEAT;
    r[0] = (float)(p.x - cx);
    r[1] = (float)(p.y - cy);
    r[2] = (float)(p.z - cz);
    r[3] = (float)n.x;
    r[4] = (float)n.y;
    r[5] = (float)n.z;
    r[6] = (float)p.w;
    r[7] = (float)curv;
    r[8] = (float)(s1 * i4pi / eps_in);
    r[9] = (float)(s2 * i4pi / eps_in);
    r[10] = (float)(u * i4pi);
    r[11] = sqrtf(dmin2) / 3.f;
    r[12] = (float)(sk * i4pi / eps_in);
    r[13] = (float)(sa4 * i4pi / eps_in);
    r[14] = (float)(sa8 * i4pi / eps_in);
    r[15] = (float)(dens / 10.0);
    r[16] = (float)(e4 * i4pi / eps_in);
    r[17] = (float)(e8 * i4pi / eps_in);
}

// the normalisers, one block: sums of squares (means for column 6) over the molecule
#define NRED 10
__global__ void k_feat_stats(int nt, const float* __restrict__ raw, double eps_in, double eps_out,
                             double* __restrict__ stats)
{
    const int cols[NRED] = {0, 6, 8, 9, 10, 12, 13, 14, 16, 17};
    __shared__ double red[NRED][256];
    double s[NRED];
    for (int c = 0; c < NRED; ++c) s[c] = 0;
    for (int k = threadIdx.x; k < nt; k += 256) {
        const float* r = raw + (size_t)k * NFEAT;
        s[0] += (double)r[0] * r[0] + (double)r[1] * r[1] + (double)r[2] * r[2];
        s[1] += r[6];
        for (int c = 2; c < NRED; ++c) s[c] += (double)r[cols[c]] * r[cols[c]];
    }
    for (int c = 0; c < NRED; ++c) red[c][threadIdx.x] = s[c];
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (threadIdx.x < h)
            for (int c = 0; c < NRED; ++c) red[c][threadIdx.x] += red[c][threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        for (int c = 0; c < NSTAT; ++c) stats[c] = 1.0;
        stats[0] = sqrt(red[0][0] / nt) + 1e-30;
        stats[6] = red[1][0] / nt;
        for (int c = 2; c < NRED; ++c) stats[cols[c]] = sqrt(red[c][0] / nt) + 1e-30;
        stats[18] = stats[8] * 2.0 * eps_in / (eps_in + eps_out);
        stats[19] = stats[9] * 2.0 * eps_out / (eps_in + eps_out);
    }
}

// normalise and scatter from sorted to element order; optionally the scaled targets
__global__ void k_feat_finish(int nt, const int* __restrict__ order, const float* __restrict__ raw,
                              const double* __restrict__ stats, float* __restrict__ F, const double* __restrict__ x,
                              float* __restrict__ T)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nt) return;
    const float* r = raw + (size_t)k * NFEAT;
    const int e = order[k];
    float* f = F + (size_t)e * NFEAT;
#pragma unroll
    for (int c = 0; c < NFEAT; ++c) {
        const float s = (float)stats[c < 3 ? 0 : c];
        f[c] = c == 6 ? logf(r[6] / s) : r[c] / s;
    }
    if (T) {
        T[2 * (size_t)e] = (float)(x[e] / stats[18]);
        T[2 * (size_t)e + 1] = (float)(x[nt + e] / stats[19]);
    }
}

static int features(pb_ctx* c, float* F, const double* x, float* T, double* stats)
{
    const int nt = c->nt;
    std::vector<double> qp(3 * (size_t)std::max(c->nc, 1));
    double cx = 0, cy = 0, cz = 0;
    if (c->nc > 0) {
        PB_CUDA(c, cudaMemcpyAsync(qp.data(), c->qpos, sizeof(double) * 3 * c->nc, cudaMemcpyDeviceToHost, c->st));
        PB_CUDA(c, cudaStreamSynchronize(c->st));
        for (int k = 0; k < c->nc; ++k) {
            cx += qp[3 * k];
            cy += qp[3 * k + 1];
            cz += qp[3 * k + 2];
        }
        cx /= c->nc;
        cy /= c->nc;
        cz /= c->nc;
    }
    PoolTmp raw(c, sizeof(float) * (size_t)nt * NFEAT);
    if (!raw.p) return pb_fail(c, PB_ERR_NOMEM, "features: out of memory");
    k_feat_pass<<<(nt + FT - 1) / FT, FT, 0, c->st>>>(nt, c->nc, c->e64p, c->e64n, c->qpos, c->q, c->touch_off,
                                                     c->touch_j, cx, cy, cz, c->prm.eps_in, c->prm.kappa,
                                                     (float*)raw.p);
    PB_LAUNCH(c);
    k_feat_stats<<<1, 256, 0, c->st>>>(nt, (const float*)raw.p, c->prm.eps_in, c->prm.eps_out, stats);
    PB_LAUNCH(c);
    k_feat_finish<<<(nt + 255) / 256, 256, 0, c->st>>>(nt, c->order, (const float*)raw.p, stats, F, x, T);
    PB_LAUNCH(c);
    return PB_OK;
}

extern "C" int pb_features(pb_ctx* c, float* F, const double* x, float* T, double* scales)
{
    if (!c) return PB_ERR_ARG;
    if (c->dead) return PB_ERR_CUDA;
    if (!c->built) return pb_fail(c, PB_ERR_STATE, "features before build_tree");
    if (c->prm.basis != PB_BASIS_CONSTANT) return pb_fail(c, PB_ERR_ARG, "features: piecewise-constant basis only");
    if (!F || (!x) != (!T)) return pb_fail(c, PB_ERR_ARG, "features: F is required, x and T go together");
    PoolTmp stats(c, sizeof(double) * NSTAT);
    if (!stats.p) return pb_fail(c, PB_ERR_NOMEM, "features: out of memory");
    int rc = features(c, F, x, T, (double*)stats.p);
    if (rc) return rc;
    if (scales) {
        PB_CUDA(c, cudaMemcpyAsync(scales, stats.p, sizeof(double) * NSTAT, cudaMemcpyDeviceToHost, c->st));
        PB_CUDA(c, cudaStreamSynchronize(c->st));
    }
    return PB_OK;
}

// x0 from the network output Y (element order, nt x 2) times the two target scales
__global__ void k_unscale(int nt, const float* __restrict__ Y, const double* __restrict__ stats,
                          double* __restrict__ x)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nt) return;
    x[k] = (double)Y[2 * (size_t)k] * stats[18];
    x[nt + k] = (double)Y[2 * (size_t)k + 1] * stats[19];
}

extern "C" int pb_learned_guess(pb_ctx* c, pb_mlp* m, double* x)
{
    if (!c || !m || !x) return PB_ERR_ARG;
    if (c->dead) return PB_ERR_CUDA;
    if (!c->built) return pb_fail(c, PB_ERR_STATE, "learned guess before build_tree");
    if (c->prm.basis != PB_BASIS_CONSTANT) return pb_fail(c, PB_ERR_ARG, "learned guess: piecewise-constant basis only");
    if (m->nin != NFEAT || m->nout != 2) return pb_fail(c, PB_ERR_ARG, "learned guess: network must map 18 -> 2");
    const int nt = c->nt;
    PoolTmp F(c, sizeof(float) * (size_t)nt * NFEAT), Y(c, sizeof(float) * (size_t)nt * 2),
        stats(c, sizeof(double) * NSTAT);
    if (!F.p || !Y.p || !stats.p) return pb_fail(c, PB_ERR_NOMEM, "learned guess: out of memory");
    int rc = features(c, (float*)F.p, nullptr, nullptr, (double*)stats.p);
    if (rc) return rc;
    if (m->st != c->st) PB_CUDA(c, cudaStreamSynchronize(c->st));
    rc = pb_mlp_forward(m, (const float*)F.p, nt, (float*)Y.p);
    if (rc) return pb_fail(c, rc, "%s", m->err.c_str());
    if (m->st != c->st) PB_CUDA(c, cudaStreamSynchronize(m->st));
    k_unscale<<<(nt + 255) / 256, 256, 0, c->st>>>(nt, (const float*)Y.p, (const double*)stats.p, x);
    PB_LAUNCH(c);
    return PB_OK;
}
