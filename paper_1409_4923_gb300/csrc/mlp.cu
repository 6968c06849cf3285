// mlp.cu -- surrogate network: the C ABI of include/sde_mlp.h, the
// layer-by-layer forward pass on BF16 tensor-core GEMMs with fused epilogues,
// and the guided scan's selection.  Training runs in mlp_train.cu, the default
// forward pass in mlp_tc.cu.
//
// Every GEMM here is one templated kernel: a 64 x 64 output tile per
// 128-thread block, 32-deep K slices staged in shared memory, 2 x 2 warps of
// 32 x 32, mma.m16n8k16 BF16 x BF16 -> FP32 with fragments loaded by ldmatrix
// (transposed where the operand is stored the other way round).  Epilogues
// fuse the bias and SiLU.
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "sde.h"
#include "sde_mlp.h"
#include "mlp_train.h"

cudaError_t sde_tc_prepare();
cudaError_t sde_tc_h2_maps(__nv_bfloat16* h2, uint64_t rows, CUtensorMap* store, CUtensorMap* load);
cudaError_t sde_tc_forward(int M, const float* x, const float* maps, uint32_t log_mask,
                           const __nv_bfloat16* W1, const float* b1, const CUtensorMap& w2, const float* b2,
                           const CUtensorMap& w3, const float* b3, const __nv_bfloat16* W4, const float* b4,
                           const CUtensorMap& h2_store, const CUtensorMap& h2_load, float* y, int* error,
                           int sm_count, cudaStream_t st);

namespace {

using sde_train::kH;
using sde_train::kIn;
using sde_train::kInPad;
using sde_train::kNParams;
using sde_train::kOut;
using sde_train::kOutPad;
using sde_train::oB1;
using sde_train::oB2;
using sde_train::oB3;
using sde_train::oB4;
using sde_train::oW1;
using sde_train::oW2;
using sde_train::oW3;
using sde_train::oW4;
constexpr uint64_t kMaxBatch = 65536;
constexpr uint64_t kMaxForwardChunk = 1u << 20;

enum { EPI_F32 = 0, EPI_FWD_SILU = 1, EPI_FWD_LINEAR = 2 };

struct GemmArgs {
    int M, N, K;
    const __nv_bfloat16* A; int lda;
    const __nv_bfloat16* B; int ldb;
    float* C; int ldc;                  // EPI_F32 / EPI_FWD_LINEAR output
    __nv_bfloat16* O; int ldo;          // EPI_FWD_SILU: BF16 activation
    const float* bias;                  // EPI_FWD_*
};

__device__ __forceinline__ float silu(float x) { return x / (1.0f + __expf(-x)); }
__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}

__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}

__device__ __forceinline__ void mma_bf16(float* d, const uint32_t* a, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
                 "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

constexpr int BM = 64, BN = 64, BK = 32;

// C tile (BM x BN) = op(A) op(B).  A_KM: A stored [K][M] (else [M][K]); B_KN:
// B stored [K][N] (else [N][K]).  Operands are loaded 8 BF16 at a time; rows
// or columns outside the matrix are zero-filled.
template <bool A_KM, bool B_KN, int EPI>
__global__ void __launch_bounds__(128) gemm_bf16_kernel(const GemmArgs g)
{
    __shared__ __align__(16) __nv_bfloat16 sA[A_KM ? BK : BM][(A_KM ? BM : BK) + 8];
    __shared__ __align__(16) __nv_bfloat16 sB[B_KN ? BK : BN][(B_KN ? BN : BK) + 8];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int ke = g.K;
    const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
    float acc[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.0f;

    // ---- staging of A and B (2 x 16-byte chunks per thread each): the next
    // K tile is fetched into registers while the current one is multiplied
    uint4 va[2], ub[2];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int c = tid + 128 * j;
            va[j] = make_uint4(0u, 0u, 0u, 0u);
            ub[j] = make_uint4(0u, 0u, 0u, 0u);
            if (!A_KM) {
                const int r = c >> 2, col = (c & 3) * 8;
                const int gm = m0 + r, gk = k0 + col;
                if (gm < g.M && gk < ke) va[j] = *(const uint4*)(g.A + (size_t)gm * g.lda + gk);
            } else {
                const int r = c >> 3, col = (c & 7) * 8;
                const int gk = k0 + r, gm = m0 + col;
                if (gk < ke && gm < g.M) va[j] = *(const uint4*)(g.A + (size_t)gk * g.lda + gm);
            }
            if (!B_KN) {
                const int r = c >> 2, col = (c & 3) * 8;
                const int gn = n0 + r, gk = k0 + col;
                if (gn < g.N && gk < ke) ub[j] = *(const uint4*)(g.B + (size_t)gn * g.ldb + gk);
            } else {
                const int r = c >> 3, col = (c & 7) * 8;
                const int gk = k0 + r, gn = n0 + col;
                if (gk < ke && gn < g.N) ub[j] = *(const uint4*)(g.B + (size_t)gk * g.ldb + gn);
            }
        }
    };
    auto stash = [&]() {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int c = tid + 128 * j;
            if (!A_KM) *(uint4*)&sA[c >> 2][(c & 3) * 8] = va[j];
            else *(uint4*)&sA[c >> 3][(c & 7) * 8] = va[j];
            if (!B_KN) *(uint4*)&sB[c >> 2][(c & 3) * 8] = ub[j];
            else *(uint4*)&sB[c >> 3][(c & 7) * 8] = ub[j];
        }
    };
    fetch(0);
    for (int k0 = 0; k0 < ke; k0 += BK) {
        stash();
        __syncthreads();
        if (k0 + BK < ke) fetch(k0 + BK);
#pragma unroll
        for (int kk = 0; kk < BK; kk += 16) {
            uint32_t af[2][4];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                const int mb = wm + mt * 16;
                if (!A_KM) {
                    const int r = mb + (lane & 15), col = kk + (lane >> 4) * 8;
                    ldsm_x4(smem_u32(&sA[r][col]), af[mt][0], af[mt][1], af[mt][2], af[mt][3]);
                } else {
                    const int r = kk + (lane >> 4) * 8 + (lane & 7), col = mb + ((lane >> 3) & 1) * 8;
                    ldsm_x4_t(smem_u32(&sA[r][col]), af[mt][0], af[mt][1], af[mt][2], af[mt][3]);
                }
            }
            uint32_t bf[4][2];
#pragma unroll
            for (int np = 0; np < 2; ++np) {
                const int nb = wn + np * 16;
                uint32_t r0, r1, r2, r3;
                if (!B_KN) {
                    const int r = nb + (lane >> 4) * 8 + (lane & 7), col = kk + ((lane >> 3) & 1) * 8;
                    ldsm_x4(smem_u32(&sB[r][col]), r0, r1, r2, r3);
                } else {
                    const int r = kk + ((lane >> 3) & 1) * 8 + (lane & 7), col = nb + (lane >> 4) * 8;
                    ldsm_x4_t(smem_u32(&sB[r][col]), r0, r1, r2, r3);
                }
                bf[np * 2][0] = r0; bf[np * 2][1] = r1;
                bf[np * 2 + 1][0] = r2; bf[np * 2 + 1][1] = r3;
            }
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) mma_bf16(acc[mt][nt], af[mt], bf[nt][0], bf[nt][1]);
        }
        __syncthreads();
    }

    // ---- epilogue: thread holds rows g, g+8 and columns 2t, 2t+1 of each 16 x 8 tile
    const int gi = lane >> 2, ti = lane & 3;
    float* C = g.C;
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int m = m0 + wm + mt * 16 + gi + h * 8;
                if (m >= g.M) continue;
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int n = n0 + wn + nt * 8 + ti * 2 + e;
                    if (n >= g.N) continue;
                    float v = acc[mt][nt][h * 2 + e];
                    if (EPI == EPI_F32) {
                        C[(size_t)m * g.ldc + n] = v;
                    } else if (EPI == EPI_FWD_LINEAR) {
                        C[(size_t)m * g.ldc + n] = v + g.bias[n];
                    } else {
                        v += g.bias[n];
                        g.O[(size_t)m * g.ldo + n] = __float2bfloat16_rn(silu(v));
                    }
                }
            }
}

template <bool A_KM, bool B_KN, int EPI>
cudaError_t gemm(const GemmArgs& a, cudaStream_t st)
{
    dim3 grid((a.N + BN - 1) / BN, (a.M + BM - 1) / BM);
    gemm_bf16_kernel<A_KM, B_KN, EPI><<<grid, 128, 0, st>>>(a);
    return cudaGetLastError();
}

// Raw inputs -> mapped BF16 inputs [Mp][16] (rows >= M and columns >= 7 zero).
__global__ void input_map_kernel(const float* __restrict__ x, uint64_t M, uint64_t Mp,
                                 const float* __restrict__ maps, uint32_t log_mask,
                                 __nv_bfloat16* __restrict__ X)
{
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= Mp * kInPad) return;
    const uint64_t m = i / kInPad;
    const int c = (int)(i % kInPad);
    float v = 0.0f;
    if (m < M && c < kIn) {
        float r = x[m * kIn + c];
        if (log_mask & (1u << c)) r = log10f(r);
        v = (r - maps[c]) * maps[kIn + c];
    }
    X[i] = __float2bfloat16_rn(v);
}

// Standardised outputs y' [Mp][8] -> y [M][2] in raw units.
__global__ void output_map_kernel(const float* __restrict__ yp, uint64_t M,
                                  const float* __restrict__ maps, float* __restrict__ y)
{
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M * kOut) return;
    const uint64_t m = i / kOut;
    const int o = (int)(i % kOut);
    y[i] = yp[m * kOutPad + o] * maps[2 * kIn + kOut + o] + maps[2 * kIn + o];
}

__global__ void to_bf16_kernel(const float* __restrict__ w, __nv_bfloat16* __restrict__ wb, size_t n)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) wb[i] = __float2bfloat16_rn(w[i]);
}

unsigned nblk(size_t n, unsigned t = 256) { return (unsigned)((n + t - 1) / t); }

// Flags of the surrogate-guided scan: predicted model error above tol,
// predicted Monte Carlo stderr above se_tol, or a sign change of the
// predicted <v> against a 4-neighbour.
__global__ void guided_flags_kernel(const float* __restrict__ v1, const float* __restrict__ v2,
                                    const float* __restrict__ lse, uint32_t nx, uint32_t ny, float kappa,
                                    float r0, float se_scale, float tol, float se_tol,
                                    uint8_t* __restrict__ flags, uint32_t* __restrict__ count)
{
    const uint64_t p = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= (uint64_t)nx * ny) return;
    const uint32_t i = (uint32_t)(p / ny), j = (uint32_t)(p % ny);
    const float v = 0.5f * (v1[p] + v2[p]);
    const float model_err = kappa * fabsf(v1[p] - v2[p]) + r0;
    const float se = se_scale * exp10f(lse[p]);
    bool f = !(model_err <= tol) || !(se <= se_tol);
    const bool neg = v < 0.0f;
    auto differs = [&](uint64_t q) { return ((0.5f * (v1[q] + v2[q])) < 0.0f) != neg; };
    if (i > 0 && differs(p - ny)) f = true;
    if (i + 1 < nx && differs(p + ny)) f = true;
    if (j > 0 && differs(p - 1)) f = true;
    if (j + 1 < ny && differs(p + 1)) f = true;
    flags[p] = f ? 1 : 0;
    const unsigned ballot = __ballot_sync(__activemask(), f);
    if (f && (threadIdx.x & 31u) == (uint32_t)(__ffs(ballot) - 1)) atomicAdd(count, (uint32_t)__popc(ballot));
}

}  // namespace

struct sde_mlp {
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    sde_train::Net train{};          // what does not change between training calls
    cudaStream_t fit_stream = nullptr;     // sde_mlp_fit's steps run here, in order after `stream`
    cudaEvent_t fit_ev = nullptr;
    std::string err;
    float* w = nullptr;              // FP32 master parameters
    __nv_bfloat16* wb = nullptr;     // BF16 copies
    float* grad = nullptr;
    float* m1 = nullptr;
    float* m2 = nullptr;
    float* maps = nullptr;           // shift[7], scale[7], out_shift[2], out_scale[2]
    uint32_t log_mask = 0;
    uint64_t step = 0;
    // activation workspace for up to cap rows
    uint64_t cap = 0;
    __nv_bfloat16* X = nullptr;      // [cap][16]
    __nv_bfloat16* A[3] = {nullptr, nullptr, nullptr};         // [cap][256] activations
    float* Yp = nullptr;             // [cap][8]
    __nv_bfloat16* dY = nullptr;     // [cap][8]
    __nv_bfloat16* dH[3] = {nullptr, nullptr, nullptr};        // [cap][256]
    float* res = nullptr;            // [cap][2] residuals
    double* loss64 = nullptr;
    double* host_loss = nullptr;     // pinned: the FP64 loss, then the training kernels' report word
    int use_tc = 1;                  // forward pass on the fused tcgen05 kernels
    __nv_bfloat16* h2 = nullptr;     // their [h2_rows][256] intermediate, and its tensor maps
    uint64_t h2_rows = 0;
    CUtensorMap h2_store{}, h2_load{};
    int sm_count = 0;
    int* tc_error = nullptr;         // device words set when a wait ran out: [0] forward, [1] training
};

static std::string g_mlp_error;

static int mfail(sde_mlp* n, int code, const std::string& msg)
{
    if (n) n->err = msg; else g_mlp_error = msg;
    return code;
}

#define MLP_CUDA(n, call) do { cudaError_t e_ = (call); if (e_ != cudaSuccess) \
    return mfail((n), e_ == cudaErrorMemoryAllocation ? SDE_ENOMEM : SDE_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); } while (0)

static void free_acts(sde_mlp* n)
{
    cudaFree(n->X); n->X = nullptr;
    for (int i = 0; i < 3; ++i) {
        cudaFree(n->A[i]); cudaFree(n->dH[i]);
        n->A[i] = nullptr; n->dH[i] = nullptr;
    }
    cudaFree(n->Yp); cudaFree(n->dY); cudaFree(n->res);
    n->Yp = nullptr; n->dY = nullptr; n->res = nullptr;
    n->cap = 0;
}

static uint64_t pad64(uint64_t m) { return (m + 63u) & ~(uint64_t)63u; }

static int ensure_acts(sde_mlp* n, uint64_t Mp, bool train)
{
    if (Mp <= n->cap && (!train || n->dY)) return SDE_OK;
    cudaStreamSynchronize(n->stream);
    free_acts(n);
    const uint64_t c = Mp;
    MLP_CUDA(n, cudaMalloc(&n->X, c * kInPad * sizeof(__nv_bfloat16)));
    for (int i = 0; i < 3; ++i) {
        MLP_CUDA(n, cudaMalloc(&n->A[i], c * kH * sizeof(__nv_bfloat16)));
        if (train) MLP_CUDA(n, cudaMalloc(&n->dH[i], c * kH * sizeof(__nv_bfloat16)));
    }
    MLP_CUDA(n, cudaMalloc(&n->Yp, c * kOutPad * sizeof(float)));
    if (train) {
        MLP_CUDA(n, cudaMalloc(&n->dY, c * kOutPad * sizeof(__nv_bfloat16)));
        MLP_CUDA(n, cudaMalloc(&n->res, c * kOut * sizeof(float)));
    }
    n->cap = c;
    return SDE_OK;
}

// The tcgen05 forward's intermediate for M rows (whole 128-row tiles).
static int ensure_h2(sde_mlp* n, uint64_t M)
{
    const uint64_t rows = (M + 127u) & ~(uint64_t)127u;
    if (rows <= n->h2_rows) return SDE_OK;
    if (n->h2) {
        cudaStreamSynchronize(n->stream);
        cudaFree(n->h2);
        n->h2 = nullptr;
        n->h2_rows = 0;
    }
    MLP_CUDA(n, cudaMalloc(&n->h2, rows * kH * sizeof(__nv_bfloat16)));
    MLP_CUDA(n, sde_tc_h2_maps(n->h2, rows, &n->h2_store, &n->h2_load));
    n->h2_rows = rows;
    return SDE_OK;
}

// Forward pass on Mp (padded) rows already mapped into n->X; standardised
// outputs into n->Yp.
static cudaError_t forward_rows(sde_mlp* n, uint64_t Mp)
{
    const int M = (int)Mp;
    GemmArgs a{};
    a.M = M; a.N = kH; a.K = kInPad; a.A = n->X; a.lda = kInPad; a.B = n->wb + oW1; a.ldb = kInPad;
    a.O = n->A[0]; a.ldo = kH; a.bias = n->w + oB1;
    cudaError_t e = gemm<false, false, EPI_FWD_SILU>(a, n->stream);
    for (int l = 1; l < 3 && e == cudaSuccess; ++l) {
        GemmArgs b{};
        b.M = M; b.N = kH; b.K = kH; b.A = n->A[l - 1]; b.lda = kH;
        b.B = n->wb + (l == 1 ? oW2 : oW3); b.ldb = kH;
        b.O = n->A[l]; b.ldo = kH;
        b.bias = n->w + (l == 1 ? oB2 : oB3);
        e = gemm<false, false, EPI_FWD_SILU>(b, n->stream);
    }
    if (e == cudaSuccess) {
        GemmArgs c{};
        c.M = M; c.N = kOutPad; c.K = kH; c.A = n->A[2]; c.lda = kH; c.B = n->wb + oW4; c.ldb = kH;
        c.C = n->Yp; c.ldc = kOutPad; c.bias = n->w + oB4;
        e = gemm<false, false, EPI_FWD_LINEAR>(c, n->stream);
    }
    return e;
}

// The network and its training workspace as the training kernels take them.
static sde_train::Net train_net(const sde_mlp* n)
{
    sde_train::Net t = n->train;
    t.w = n->w; t.wb = n->wb; t.m1 = n->m1; t.m2 = n->m2; t.maps = n->maps; t.log_mask = n->log_mask;
    t.X = n->X; t.dY = n->dY; t.res = n->res;
    for (int i = 0; i < 3; ++i) { t.A[i] = n->A[i]; t.dH[i] = n->dH[i]; }
    return t;
}

// Adam's update of step t (1, 2, ...) with learning rate lr.
static sde_train::Update adam_update(float lr, float beta1, float beta2, float eps, uint64_t t, float* loss)
{
    sde_train::Update u{};
    u.lr = lr; u.b1 = beta1; u.b2 = beta2; u.eps = eps; u.loss = loss;
    u.c1 = (float)(1.0 / (1.0 - std::pow((double)beta1, (double)t)));
    u.c2 = (float)(1.0 / (1.0 - std::pow((double)beta2, (double)t)));
    return u;
}

// After a synchronisation: whether a training step gave up.
static int train_status(sde_mlp* n)
{
    if (*n->train.report == 0) return SDE_OK;
    return mfail(n, SDE_ETIMEDOUT, "a training step's wait for its weights ran out; the parameters are those before that "
                                   "step and stay so until sde_mlp_set_params");
}

extern "C" {

const char* sde_mlp_last_error(const sde_mlp* n) { return n ? n->err.c_str() : g_mlp_error.c_str(); }

int sde_mlp_create(sde_mlp** out, uint64_t seed, void* cuda_stream)
{
    if (!out) return mfail(nullptr, SDE_EINVAL, "out is NULL");
    *out = nullptr;
    sde_mlp* n = new (std::nothrow) sde_mlp();
    if (!n) return mfail(nullptr, SDE_ENOMEM, "host allocation failed");
    cudaError_t e = cudaSuccess;
    if (cuda_stream == nullptr) {
        e = cudaStreamCreate(&n->stream);
        n->own_stream = e == cudaSuccess;
    } else {
        n->stream = (cudaStream_t)cuda_stream;
    }
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&n->fit_stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&n->fit_ev, cudaEventDisableTiming);
    const size_t P = kNParams;
    if (e == cudaSuccess) e = cudaMalloc(&n->w, P * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&n->wb, P * sizeof(__nv_bfloat16));
    if (e == cudaSuccess) e = cudaMalloc(&n->grad, P * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&n->m1, P * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&n->m2, P * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&n->maps, 32 * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&n->loss64, sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&n->tc_error, 2 * sizeof(int));
    if (e == cudaSuccess) e = cudaMemset(n->tc_error, 0, 2 * sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&n->train.loss_part, sde_train::kLossBlocks * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&n->train.loss_done, sizeof(uint32_t));
    if (e == cudaSuccess) e = cudaMemset(n->train.loss_done, 0, sizeof(uint32_t));
    if (e == cudaSuccess) e = sde_train::prepare();
    if (e == cudaSuccess) e = sde_tc_prepare();
    if (e == cudaSuccess) e = sde_train::weight_maps(n->wb, &n->train.w2, &n->train.w3);
    n->train.error = n->tc_error + 1;
    n->train.polls = sde_train::kDefaultPolls;
    if (e == cudaSuccess) {
        int dev = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n->sm_count, cudaDevAttrMultiProcessorCount, dev);
        n->train.sm_count = (uint32_t)n->sm_count;
    }
    if (e == cudaSuccess) e = cudaMallocHost(&n->host_loss, 2 * sizeof(double));
    n->train.report = (volatile int*)(n->host_loss + 1);
    if (e != cudaSuccess) {
        mfail(nullptr, SDE_ECUDA, std::string("sde_mlp_create: ") + cudaGetErrorString(e));
        sde_mlp_destroy(n);
        return SDE_ECUDA;
    }
    // Glorot-uniform weights from a splitmix64 stream, zero biases and padding
    std::vector<float> h(P, 0.0f);
    uint64_t s = seed ^ 0x5DEECE66DULL;
    auto next_u = [&s]() {
        s += 0x9E3779B97F4A7C15ULL;
        uint64_t z = s;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
        z ^= z >> 31;
        return (double)(z >> 11) * (1.0 / 9007199254740992.0);
    };
    auto fill = [&](size_t off, int rows, int cols, int live_rows, int live_cols) {
        const double lim = std::sqrt(6.0 / (double)(live_rows + live_cols));
        for (int r = 0; r < rows; ++r)
            for (int c = 0; c < cols; ++c)
                h[off + (size_t)r * cols + c] =
                    (r < live_rows && c < live_cols) ? (float)((2.0 * next_u() - 1.0) * lim) : 0.0f;
    };
    fill(oW1, kH, kInPad, kH, kIn);
    fill(oW2, kH, kH, kH, kH);
    fill(oW3, kH, kH, kH, kH);
    fill(oW4, kOutPad, kH, kOut, kH);
    float maps[32] = {0};
    for (int i = 0; i < kIn; ++i) maps[kIn + i] = 1.0f;
    maps[2 * kIn + kOut] = maps[2 * kIn + kOut + 1] = 1.0f;
    e = cudaMemcpyAsync(n->maps, maps, sizeof(maps), cudaMemcpyHostToDevice, n->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(n->stream);
    *out = n;
    if (e != cudaSuccess) return mfail(n, SDE_ECUDA, cudaGetErrorString(e));
    return sde_mlp_set_params(n, h.data());
}

int sde_mlp_set_maps(sde_mlp* n, const float* shift, const float* scale, uint32_t log_mask,
                     const float* out_shift, const float* out_scale)
{
    if (!n || !shift || !scale || !out_shift || !out_scale) return SDE_EINVAL;
    float maps[32] = {0};
    for (int i = 0; i < kIn; ++i) {
        if (!std::isfinite(shift[i]) || !std::isfinite(scale[i])) return mfail(n, SDE_EINVAL, "non-finite input map");
        maps[i] = shift[i];
        maps[kIn + i] = scale[i];
    }
    for (int o = 0; o < kOut; ++o) {
        if (!std::isfinite(out_shift[o]) || !(out_scale[o] != 0.0f) || !std::isfinite(out_scale[o]))
            return mfail(n, SDE_EINVAL, "bad output map");
        maps[2 * kIn + o] = out_shift[o];
        maps[2 * kIn + kOut + o] = out_scale[o];
    }
    if (log_mask >> kIn) return mfail(n, SDE_EINVAL, "log mask has bits beyond the 7 inputs");
    n->log_mask = log_mask;
    MLP_CUDA(n, cudaMemcpyAsync(n->maps, maps, sizeof(maps), cudaMemcpyHostToDevice, n->stream));
    MLP_CUDA(n, cudaStreamSynchronize(n->stream));
    return SDE_OK;
}

int sde_mlp_set_params(sde_mlp* n, const float* host)
{
    if (!n || !host) return SDE_EINVAL;
    const size_t P = kNParams;
    MLP_CUDA(n, cudaMemcpyAsync(n->w, host, P * sizeof(float), cudaMemcpyHostToDevice, n->stream));
    to_bf16_kernel<<<nblk(P), 256, 0, n->stream>>>(n->w, n->wb, P);
    MLP_CUDA(n, cudaGetLastError());
    MLP_CUDA(n, cudaMemsetAsync(n->m1, 0, P * sizeof(float), n->stream));
    MLP_CUDA(n, cudaMemsetAsync(n->m2, 0, P * sizeof(float), n->stream));
    MLP_CUDA(n, cudaMemsetAsync(n->train.error, 0, sizeof(int), n->stream));
    MLP_CUDA(n, cudaStreamSynchronize(n->stream));
    *n->train.report = 0;
    n->step = 0;
    return SDE_OK;
}

int sde_mlp_get_params(sde_mlp* n, float* host)
{
    if (!n || !host) return SDE_EINVAL;
    MLP_CUDA(n, cudaMemcpyAsync(host, n->w, kNParams * sizeof(float), cudaMemcpyDeviceToHost, n->stream));
    MLP_CUDA(n, cudaStreamSynchronize(n->stream));
    return train_status(n);
}

int sde_mlp_forward(sde_mlp* n, const float* x, uint64_t M, float* y)
{
    if (!n || !x || !y || M == 0) return n ? mfail(n, SDE_EINVAL, "bad forward arguments") : SDE_EINVAL;
    // the tensor-core layers keep their weights resident per CTA: large chunks
    // amortise the weight loads
    const uint64_t chunk = n->use_tc ? kMaxForwardChunk : kMaxBatch;
    const uint64_t rows = M < chunk ? M : chunk;
    int rc = n->use_tc ? ensure_h2(n, rows) : ensure_acts(n, pad64(rows), false);
    if (rc) return rc;
    for (uint64_t r0 = 0; r0 < M; r0 += chunk) {
        const uint64_t m = (M - r0) < chunk ? (M - r0) : chunk;
        const uint64_t Mp = pad64(m);
        if (n->use_tc) {
            // two fused tcgen05 kernels: maps and layers 1-2, layers 3-4 and the output map
            MLP_CUDA(n, sde_tc_forward((int)m, x + r0 * kIn, n->maps, n->log_mask, n->wb + oW1, n->w + oB1,
                                       n->train.w2, n->w + oB2, n->train.w3, n->w + oB3, n->wb + oW4, n->w + oB4,
                                       n->h2_store, n->h2_load, y + r0 * kOut, n->tc_error, n->sm_count, n->stream));
            continue;
        }
        input_map_kernel<<<nblk(Mp * kInPad), 256, 0, n->stream>>>(x + r0 * kIn, m, Mp, n->maps, n->log_mask, n->X);
        MLP_CUDA(n, cudaGetLastError());
        MLP_CUDA(n, forward_rows(n, Mp));
        output_map_kernel<<<nblk(m * kOut), 256, 0, n->stream>>>(n->Yp, m, n->maps, y + r0 * kOut);
        MLP_CUDA(n, cudaGetLastError());
    }
    return SDE_OK;
}

int sde_mlp_gradients(sde_mlp* n, const float* x, const float* t, uint64_t M, float* host_grad,
                      double* host_loss)
{
    if (!n || !x || !t || !host_grad || M == 0 || M > kMaxBatch)
        return n ? mfail(n, SDE_EINVAL, "bad gradient arguments (1 <= M <= 65536)") : SDE_EINVAL;
    const uint64_t Mp = pad64(M);
    int rc = ensure_acts(n, Mp, true);
    if (rc) return rc;
    sde_train::Batch b{};
    b.x = x; b.t = t; b.M = (uint32_t)M;
    sde_train::Update u{};
    u.grad = n->grad; u.loss64 = n->loss64;
    MLP_CUDA(n, sde_train::step(train_net(n), b, u, n->stream));
    MLP_CUDA(n, cudaMemcpyAsync(host_grad, n->grad, kNParams * sizeof(float), cudaMemcpyDeviceToHost, n->stream));
    MLP_CUDA(n, cudaMemcpyAsync(n->host_loss, n->loss64, sizeof(double), cudaMemcpyDeviceToHost, n->stream));
    MLP_CUDA(n, cudaStreamSynchronize(n->stream));
    if ((rc = train_status(n))) return rc;
    if (host_loss) *host_loss = *n->host_loss;
    return SDE_OK;
}

int sde_mlp_train_step(sde_mlp* n, const float* x, const float* t, uint64_t M, float lr, float beta1,
                       float beta2, float eps, float* loss_dev)
{
    if (!n || !x || !t || M == 0 || M > kMaxBatch)
        return n ? mfail(n, SDE_EINVAL, "bad train arguments (1 <= M <= 65536)") : SDE_EINVAL;
    if (!(lr > 0.0f) || !(beta1 >= 0.0f && beta1 < 1.0f) || !(beta2 >= 0.0f && beta2 < 1.0f) || !(eps > 0.0f))
        return mfail(n, SDE_EINVAL, "bad Adam hyper-parameters");
    int rc = ensure_acts(n, pad64(M), true);
    if (rc) return rc;
    sde_train::Batch b{};
    b.x = x; b.t = t; b.M = (uint32_t)M;
    MLP_CUDA(n, sde_train::step(train_net(n), b, adam_update(lr, beta1, beta2, eps, n->step + 1, loss_dev), n->stream));
    n->step += 1;
    return SDE_OK;
}

int sde_mlp_fit(sde_mlp* n, const float* X, const float* T, uint64_t N, uint64_t steps, uint32_t batch,
                float lr, float lr_final, float beta1, float beta2, float eps, uint64_t seed, float* losses)
{
    if (!n) return SDE_EINVAL;
    if (!X || !T || N == 0 || N > (1ull << 30) || steps == 0 || steps > (1ull << 22) || batch == 0 ||
        batch > kMaxBatch || batch > N)
        return mfail(n, SDE_EINVAL,
                     "bad fit arguments (1 <= batch <= min(N, 65536), N <= 2^30, 1 <= steps <= 2^22)");
    if (!(lr > 0.0f) || !(lr_final > 0.0f) || !(beta1 >= 0.0f && beta1 < 1.0f) || !(beta2 >= 0.0f && beta2 < 1.0f) ||
        !(eps > 0.0f))
        return mfail(n, SDE_EINVAL, "bad Adam hyper-parameters");
    int rc = ensure_acts(n, pad64(batch), true);
    if (rc) return rc;
    sde_train::Batch b{};
    b.x = X; b.t = T; b.M = batch; b.N = (uint32_t)N; b.seed = seed;
    b.bits = 2;
    while ((1ull << b.bits) < N) b.bits += 2;
    const uint64_t per_epoch = N / batch;
    const sde_train::Net net = train_net(n);
    const double pi = 3.14159265358979323846;
    cudaError_t e = cudaEventRecord(n->fit_ev, n->stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(n->fit_stream, n->fit_ev, 0);
    // half-cosine decay of the learning rate, Adam's corrections as in sde_mlp_train_step
    for (uint64_t k = 0; k < steps && e == cudaSuccess; ++k) {
        const double frac = steps > 1 ? (double)k / (double)(steps - 1) : 0.0;
        const float lr_k = (float)((double)lr_final + 0.5 * ((double)lr - (double)lr_final) * (1.0 + std::cos(pi * frac)));
        b.pos0 = (uint32_t)(k % per_epoch) * batch;
        b.epoch = k / per_epoch;
        b.settled = k > 0;
        e = sde_train::step(net, b, adam_update(lr_k, beta1, beta2, eps, n->step + k + 1, losses ? losses + k : nullptr),
                            n->fit_stream);
    }
    if (e == cudaSuccess) e = cudaEventRecord(n->fit_ev, n->fit_stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(n->stream, n->fit_ev, 0);
    const cudaError_t es = cudaStreamSynchronize(n->fit_stream);
    if (e == cudaSuccess) e = es;
    MLP_CUDA(n, e);
    if ((rc = train_status(n))) return rc;
    n->step += steps;
    return SDE_OK;
}

int sde_mlp_gemm_bf16(sde_mlp* n, int a_layout, int b_layout, uint32_t M, uint32_t N, uint32_t K,
                      const void* A, uint32_t lda, const void* B, uint32_t ldb, float* C, uint32_t ldc)
{
    if (!n || !A || !B || !C || M == 0 || N == 0 || K == 0) return SDE_EINVAL;
    if ((lda | ldb) & 7u || ((uintptr_t)A | (uintptr_t)B) & 15u)
        return mfail(n, SDE_EINVAL, "operands need 16-byte aligned rows (leading dimensions % 8 == 0)");
    if ((a_layout == 0 && K % 8) || (a_layout == 1 && M % 8) || (b_layout == 0 && K % 8) || (b_layout == 1 && N % 8))
        return mfail(n, SDE_EINVAL, "the contiguous dimension of each operand must be a multiple of 8");
    GemmArgs g{};
    g.M = (int)M; g.N = (int)N; g.K = (int)K;
    g.A = (const __nv_bfloat16*)A; g.lda = (int)lda; g.B = (const __nv_bfloat16*)B; g.ldb = (int)ldb;
    g.C = C; g.ldc = (int)ldc;
    cudaError_t e;
    if (a_layout == 0 && b_layout == 0) e = gemm<false, false, EPI_F32>(g, n->stream);
    else if (a_layout == 0 && b_layout == 1) e = gemm<false, true, EPI_F32>(g, n->stream);
    else if (a_layout == 1 && b_layout == 1) e = gemm<true, true, EPI_F32>(g, n->stream);
    else if (a_layout == 1 && b_layout == 0) e = gemm<true, false, EPI_F32>(g, n->stream);
    else return mfail(n, SDE_EINVAL, "layout must be 0 or 1");
    MLP_CUDA(n, e);
    MLP_CUDA(n, cudaStreamSynchronize(n->stream));
    return SDE_OK;
}

int sde_mlp_set_tensor_path(sde_mlp* n, int use_tcgen05)
{
    if (!n || (use_tcgen05 != 0 && use_tcgen05 != 1)) return SDE_EINVAL;
    n->use_tc = use_tcgen05;
    return SDE_OK;
}

int sde_mlp_sync(sde_mlp* n)
{
    if (!n) return SDE_EINVAL;
    MLP_CUDA(n, cudaStreamSynchronize(n->stream));
    int err = 0;
    MLP_CUDA(n, cudaMemcpy(&err, n->tc_error, sizeof(int), cudaMemcpyDeviceToHost));
    if (err) return mfail(n, SDE_ETIMEDOUT, "a tensor-core completion wait ran out (mbarrier not signalled)");
    return train_status(n);
}

int sde_mlp_set_wait_polls(sde_mlp* n, uint32_t polls)
{
    if (!n) return SDE_EINVAL;
    n->train.polls = polls;
    return SDE_OK;
}

int sde_guided_flags(sde_mlp* n, const float* v1, const float* v2, const float* lse, uint32_t nx,
                     uint32_t ny, float kappa, float r0, float se_scale, float tol, float se_tol, uint8_t* flags,
                     uint32_t* count)
{
    if (!n || !v1 || !v2 || !lse || !flags || !count || nx == 0 || ny == 0) return SDE_EINVAL;
    const uint64_t total = (uint64_t)nx * ny;
    guided_flags_kernel<<<nblk(total), 256, 0, n->stream>>>(v1, v2, lse, nx, ny, kappa, r0, se_scale, tol,
                                                            se_tol, flags, count);
    MLP_CUDA(n, cudaGetLastError());
    return SDE_OK;
}

void sde_mlp_destroy(sde_mlp* n)
{
    if (!n) return;
    if (n->stream || n->own_stream) cudaStreamSynchronize(n->stream);
    free_acts(n);
    cudaFree(n->h2);
    cudaFree(n->w); cudaFree(n->wb); cudaFree(n->grad); cudaFree(n->m1); cudaFree(n->m2);
    cudaFree(n->maps); cudaFree(n->loss64); cudaFree(n->tc_error);
    cudaFree(n->train.loss_part); cudaFree(n->train.loss_done);
    if (n->host_loss) cudaFreeHost(n->host_loss);
    if (n->fit_stream) cudaStreamDestroy(n->fit_stream);
    if (n->fit_ev) cudaEventDestroy(n->fit_ev);
    if (n->own_stream) cudaStreamDestroy(n->stream);
    delete n;
}

}  // extern "C"
