// Learned warm start: a small MLP that maps a problem description to initial
// ansatz angles, trained and run on the GPU by the kernels below (FP32).
//
//   h1 = GELU(W1 x + b1), h2 = GELU(W2 h1 + b2), y = W3 h2 + b3,
//   GELU(z) = z (1 + erf(z / sqrt 2)) / 2,
//   loss = sum M (y - t)^2 / sum M  (masked mean squared error),
//
// with back-propagation and Adam.  A training step is seven launches: three
// forward products (the last one forms the loss and its derivative), two
// backward products, one launch for all the weight gradients (split over the
// batch) and one that adds the splits and updates.  Every sum runs in a fixed
// order, so gradients are deterministic.  Parameters are one flat FP32 vector:
// W1 [H x I], b1 [H], W2 [H x H], b2 [H], W3 [O x H], b3 [O] (row-major).
#include <algorithm>
#include <cmath>
#include <cstdio>

#include "internal.cuh"

struct dvqls_ws {
    dvqls_ctx* ctx;
    int I, H, O;
    long long np;
    float* params;  // np
    float* grad;    // np
    float* m;       // np
    float* v;       // np
    long long step;
    int cap;        // batch capacity of the activations
    float* act;     // X, z1, h1, z2, h2, y, dy, dz2, dz1, T, M (batch-major), loss parts, gradient parts
    float* lossbuf; // 2 floats: sum M (y-t)^2, sum M
    char* pin;      // small pinned buffer for the loss
};

namespace dvqls {
namespace {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// FP32 products on 64 x 64 tiles, 4 x 4 outputs per thread, the operands of 16
// steps of k staged in shared memory by asynchronous copies, three tiles ahead.
// One row of threads per k needs two 16-byte shared loads for 16 FMAs, which the
// FMA pipe bounds; but a CTA has its SM to itself here, so a tile's 512 cycles of
// FMAs do not cover a load from L2 one tile ahead (in registers: 123 us for the step
// below; with copies three ahead 110).  64 x 64 (not larger) so that the batch of 2,000
// with 256 hidden units still gives 128 CTAs.  A training step of that batch took 605 us
// with 16 x 16 tiles, no split over the batch (16 CTAs for the 256 x 256 gradient) and
// bias gradients of one thread per column.  Two groups of 256 threads per CTA, each with
// every other tile of k, gave 114.
constexpr int GT = 64, GK = 16, GTH = 256;

constexpr int GSTG = 4;  // tiles of k in shared memory: three on the way while one is multiplied

struct GemmSmem {
    float A[GSTG][GK][GT + 4], B[GSTG][GK][GT + 4];
};

// Operand tile (rows row0 .., k0 .. k0 + GK - 1) into S[k][row], zero outside, by
// asynchronous copies: row-major with k contiguous (KMAJOR) or with the row
// contiguous.  Single floats: a matrix of the flat parameter vector starts at any
// multiple of four bytes.
template <bool KMAJOR, int TR = GT>
__device__ __forceinline__ void gemm_fetch(float (*S)[GT + 4], const float* __restrict__ P, long long ld, int row0, int rows,
                                           int k0, int kend) {
#pragma unroll
    for (int q = 0; q < TR * GK / GTH; ++q) {
        const int e = threadIdx.x + q * GTH;
        const int r = KMAJOR ? e / GK : e % TR, k = KMAJOR ? e % GK : e / TR;
        const bool in = row0 + r < rows && k0 + k < kend;
        const float* src = in ? (KMAJOR ? P + (row0 + r) * ld + k0 + k : P + (k0 + k) * ld + row0 + r) : P;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(&S[k][r])),
                     "l"(__cvta_generic_to_global(src)), "r"(in ? 4 : 0)
                     : "memory");
    }
}

// acc[i][j] = sum over k in [k0, kend) of A(m0 + R ty + i, k) B(k, n0 + 4 tx + j), R = 4
// rows per thread or 1 (tiles of 16 R x 64);
// rsum (threads below 64, when wanted): the sum over k of A(m0 + t, k).
template <bool AK, bool BK, int R = 4>
__device__ __forceinline__ void gemm_tile(GemmSmem& sm, const float* __restrict__ A, long long lda, int m0, int M,
                                          const float* __restrict__ B, long long ldb, int n0, int N, int k0, int kend,
                                          float (&acc)[R][4], bool want_rsum, float& rsum) {
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    const int tiles = (kend - k0 + GK - 1) / GK;
    auto issue = [&](int u) {  // one group of copies per tile, empty past the last
        if (u < tiles) {
            gemm_fetch<AK, 16 * R>(sm.A[u % GSTG], A, lda, m0, M, k0 + u * GK, kend);
            gemm_fetch<BK>(sm.B[u % GSTG], B, ldb, n0, N, k0 + u * GK, kend);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int u = 0; u < GSTG - 1; ++u) issue(u);
    for (int u = 0; u < tiles; ++u) {
        asm volatile("cp.async.wait_group %0;" ::"n"(GSTG - 2) : "memory");
        __syncthreads();  // tile u is there for all threads, and all have read tile u - 1
        issue(u + GSTG - 1);
        const int buf = u % GSTG;
#pragma unroll
        for (int q = 0; q < GK; ++q) {
            alignas(16) float av[R];
            if constexpr (R == 4) *reinterpret_cast<float4*>(av) = *reinterpret_cast<const float4*>(&sm.A[buf][q][4 * ty]);
            else av[0] = sm.A[buf][q][ty];
            const float4 b = *reinterpret_cast<const float4*>(&sm.B[buf][q][4 * tx]);
            const float bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
        if (want_rsum && threadIdx.x < GT) {
#pragma unroll
            for (int q = 0; q < GK; ++q) rsum += sm.A[buf][q][threadIdx.x];
        }
    }
}

__device__ __forceinline__ float gelu_grad(float x) {
    return 0.5f * (1.f + erff(x * 0.70710678118654752f)) + x * expf(-0.5f * x * x) * 0.3989422804014327f;
}

enum Epilogue {
    EPI_GELU,  // C = GELU(Z), Z = product + bias
    EPI_BIAS,  // C = product + bias
    EPI_LOSS,  // C = scale mask (product + bias - target), and the CTA's parts of the loss
    EPI_BACK,  // C = product GELU'(Z)
};

// C[m, n] = epilogue of sum_k A[m, k] B(k, n), A row-major with k contiguous; BK:
// B(k, n) = B[n ldb + k], else B[k ldb + n].  EPI_LOSS writes (sum M e^2, sum M)
// of the CTA's outputs to part[2 * CTA].
template <int EPI, bool BK, int R = 4>
__global__ void __launch_bounds__(GTH) k_gemm(int M, int N, int K, const float* __restrict__ A, const float* __restrict__ B,
                                              int ldb, const float* __restrict__ bias, float* Z, float* C,
                                              const float* __restrict__ target, const float* __restrict__ mask,
                                              float* part, float scale) {
    pdl_wait();
    __shared__ GemmSmem sm;
    const int m0 = blockIdx.y * (16 * R), n0 = blockIdx.x * GT, tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float acc[R][4], none = 0.f;
    gemm_tile<true, BK, R>(sm, A, K, m0, M, B, ldb, n0, N, 0, K, acc, false, none);
    float s1 = 0.f, s2 = 0.f;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int m = m0 + R * ty + i;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = n0 + 4 * tx + j;
            if (m >= M || n >= N) continue;
            const long long at = (long long)m * N + n;
            float v = acc[i][j];
            if (EPI == EPI_BACK) {
                C[at] = v * gelu_grad(Z[at]);
                continue;
            }
            v += bias[n];
            if (EPI == EPI_GELU) {
                Z[at] = v;
                v = 0.5f * v * (1.f + erff(v * 0.70710678118654752f));
            }
            if (EPI == EPI_LOSS) {
                const float mk = mask[at], e = v - target[at];
                s1 += mk * e * e;
                s2 += mk;
                v = mk * e * scale;
            }
            C[at] = v;
        }
    }
    if (EPI == EPI_LOSS) {
        for (int o = 16; o; o >>= 1) {
            s1 += __shfl_xor_sync(0xffffffffu, s1, o);
            s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        }
        __syncthreads();
        float* red = &sm.A[0][0][0];
        if ((threadIdx.x & 31) == 0) {
            red[threadIdx.x >> 5] = s1;
            red[8 + (threadIdx.x >> 5)] = s2;
        }
        __syncthreads();
        if (threadIdx.x < 2) {
            float s = 0.f;
            for (int k = 0; k < GTH / 32; ++k) s += red[8 * threadIdx.x + k];
            part[2 * (blockIdx.y * gridDim.x + blockIdx.x) + threadIdx.x] = s;
        }
    }
}

// The gradients of the three weight matrices and biases, before the factor
// 2 / (scale sum M): job q is gW[m, n] = sum_b D[b, m] Hq[b, n] (rows of D: the layer's
// derivative; rows of Hq: its input) and gb[m] = sum_b D[b, m].  Grid: (tiles of
// all three jobs, splits of the batch); split s writes its sums to part[s np ..].
struct GradJob {
    const float* D;
    const float* In;
    int M, N, tiles_n, first;  // first: the job's first tile
    long long w_off, b_off;
};
struct GradJobs {
    GradJob j[3];
};
__global__ void __launch_bounds__(GTH) k_wgrad(GradJobs jobs, int batch, int per, long long np, float* part) {
    pdl_wait();
    __shared__ GemmSmem sm;
    const int tile = blockIdx.x;
    const GradJob J = tile >= jobs.j[2].first ? jobs.j[2] : tile >= jobs.j[1].first ? jobs.j[1] : jobs.j[0];
    const int u = tile - J.first, m0 = (u / J.tiles_n) * GT, n0 = (u % J.tiles_n) * GT;
    const int k0 = blockIdx.y * per, kend = min(batch, k0 + per);
    const bool bias = u % J.tiles_n == 0;
    float acc[4][4], rsum = 0.f;
    gemm_tile<false, false>(sm, J.D, J.M, m0, J.M, J.In, J.N, n0, J.N, k0, kend, acc, bias, rsum);
    float* out = part + blockIdx.y * np;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int m = m0 + 4 * ty + i, n = n0 + 4 * tx + j;
            if (m < J.M && n < J.N) out[J.w_off + (long long)m * J.N + n] = acc[i][j];
        }
    if (bias && threadIdx.x < GT && m0 + int(threadIdx.x) < J.M) out[J.b_off + m0 + threadIdx.x] = rsum;
}

struct AdamArgs {
    float lr, b1, b2, eps, c1, c2;
};
// The gradient from its splits (added in order) and the loss parts, written to
// grad (when not null), or used at once for the Adam update.  The first CTA
// leaves the loss sums in lossbuf.
__global__ void __launch_bounds__(256) k_grad_update(long long np, int splits, const float* __restrict__ part,
                                                     int nloss, const float* __restrict__ lpart, float* lossbuf,
                                                     float* grad, float* p, float* m, float* v, AdamArgs a, float unscale) {
    pdl_wait();
    __shared__ float red[2];
    if (threadIdx.x < 32) {  // the same sums in the same order in every CTA
        float s1 = 0.f, s2 = 0.f;
        for (int k = threadIdx.x; k < nloss; k += 32) {
            s1 += lpart[2 * k];
            s2 += lpart[2 * k + 1];
        }
        for (int o = 16; o; o >>= 1) {
            s1 += __shfl_xor_sync(0xffffffffu, s1, o);
            s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        }
        if (threadIdx.x == 0) {
            red[0] = s1;
            red[1] = s2;
            if (blockIdx.x == 0) {
                lossbuf[0] = s1;
                lossbuf[1] = s2;
            }
        }
    }
    const long long i = blockIdx.x * 256LL + threadIdx.x;
    float g = 0.f;
    if (i < np) {
#pragma unroll 4
        for (int s = 0; s < splits; ++s) g += part[s * np + i];
    }
    __syncthreads();
    if (i >= np) return;
    g *= red[1] > 0.f ? 2.f * unscale / red[1] : 0.f;
    if (grad) {
        grad[i] = g;
        return;
    }
    const float mi = a.b1 * m[i] + (1.f - a.b1) * g;
    const float vi = a.b2 * v[i] + (1.f - a.b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    p[i] -= a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + a.eps);
}

// Splits of the batch for the weight gradients: enough CTAs for two per SM, 64
// rows per split at least.
int grad_tiles(const dvqls_ws* w) {
    const int h = ceil_div(w->H, GT);
    return h * ceil_div(w->I, GT) + h * h + ceil_div(w->O, GT) * h;
}
int max_splits(const dvqls_ws* w) { return std::max(1, std::min(32, 2 * w->ctx->num_sms / grad_tiles(w))); }

struct Views {
    const float *X, *T, *M;  // the batch: the caller's device arrays, or the copies below
    float *Xc, *Tc, *Mc, *z1, *h1, *z2, *h2, *y, *dy, *d2, *d1, *lpart, *gpart;
};

// Carves the activations of `cap` rows out of `base` (nullptr: counts only);
// returns the number of floats.
long long carve(const dvqls_ws* w, long long cap, float* base, Views& a) {
    long long at = 0;
    auto take = [&](long long n) {
        float* r = base ? base + at : nullptr;
        at += n;
        return r;
    };
    a.Xc = take(cap * w->I);
    a.z1 = take(cap * w->H);
    a.h1 = take(cap * w->H);
    a.z2 = take(cap * w->H);
    a.h2 = take(cap * w->H);
    a.y = take(cap * w->O);
    a.dy = take(cap * w->O);
    a.d2 = take(cap * w->H);
    a.d1 = take(cap * w->H);
    a.Tc = take(cap * w->O);
    a.Mc = take(cap * w->O);
    a.lpart = take(2LL * ceil_div(cap, GT) * ceil_div(w->O, GT));
    a.gpart = take(max_splits(w) * w->np);
    a.X = a.Xc;
    a.T = a.Tc;
    a.M = a.Mc;
    return at;
}

Views views(dvqls_ws* w) {
    Views a;
    carve(w, w->cap, w->act, a);
    return a;
}

int ensure_batch(dvqls_ws* w, int batch) {
    if (batch <= w->cap) return DVQLS_OK;
    dvqls_ctx* ctx = w->ctx;
    DVQLS_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    if (w->act) cudaFree(w->act);
    w->act = nullptr;
    int cap = std::max(batch, 64);
    Views none;
    if (cudaMalloc(&w->act, carve(w, cap, nullptr, none) * sizeof(float)) != cudaSuccess) {
        cudaGetLastError();
        w->cap = 0;
        return set_error(ctx, DVQLS_ERR_ALLOC, "warm-start activations for batch %d", cap);
    }
    w->cap = cap;
    return DVQLS_OK;
}

// Each kernel starts with griddepcontrol.wait, so its launch need not wait for its
// predecessor's end.  None triggers its dependent early: the dependent's CTAs would be
// placed on the SMs that have room at that moment, two on one and none on another (batch of
// 2,000, 512 hidden units: a step 253 us with early triggers, 185 without).
template <typename... KArgs, typename... Args>
int launch(dvqls_ctx* ctx, void (*kern)(KArgs...), dim3 grid, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(256);
    cfg.stream = ctx->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    DVQLS_CUDA_TRY(ctx, cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...));
    return DVQLS_OK;
}

struct Params {
    const float *W1, *b1, *W2, *b2, *W3, *b3;
};
Params params_of(const dvqls_ws* w) {
    Params p;
    p.W1 = w->params;
    p.b1 = p.W1 + (long long)w->H * w->I;
    p.W2 = p.b1 + w->H;
    p.b2 = p.W2 + (long long)w->H * w->H;
    p.W3 = p.b2 + w->H;
    p.b3 = p.W3 + (long long)w->O * w->H;
    return p;
}

dim3 gemm_grid(int M, int N) { return dim3(ceil_div(N, GT), ceil_div(M, GT)); }

// The power of two that takes the place of 1 / sum M in back-propagation, where sum M is not known
// yet: a derivative summed over the batch stays in the range of its mean.
float loss_scale(const dvqls_ws* w, int B) { return ldexpf(1.f, -int(std::ceil(std::log2(double(B) * w->O)))); }

// Hidden layers, then y (loss = false) or the loss parts and dy = M (y - t).
int forward(dvqls_ws* w, const Views& a, int B, bool loss) {
    dvqls_ctx* ctx = w->ctx;
    const int I = w->I, H = w->H, O = w->O;
    const Params p = params_of(w);
    // Tiles of 16 rows where those of 64 would leave half of the SMs idle: a quarter of the FMAs
    // per tile of k, four times the CTAs, the same sums (inference of 16 rows with 512 hidden units:
    // 62 us with 64-row tiles, 51 with these; of 100 rows 68 and 52).
    auto low = [&](int N) { return 2 * ceil_div(B, GT) * ceil_div(N, GT) < ctx->num_sms; };
    auto layer = [&](auto tall, auto flat, int N, int K, const float* in, const float* W, const float* b, float* z, float* out) {
        if (low(N))
            return launch(ctx, flat, dim3(ceil_div(N, GT), ceil_div(B, 16)), B, N, K, in, W, K, b, z, out, nullptr, nullptr,
                          nullptr, 1.f);
        return launch(ctx, tall, gemm_grid(B, N), B, N, K, in, W, K, b, z, out, nullptr, nullptr, nullptr, 1.f);
    };
    int rc = layer(k_gemm<EPI_GELU, true>, k_gemm<EPI_GELU, true, 1>, H, I, a.X, p.W1, p.b1, a.z1, a.h1);
    if (!rc) rc = layer(k_gemm<EPI_GELU, true>, k_gemm<EPI_GELU, true, 1>, H, H, a.h1, p.W2, p.b2, a.z2, a.h2);
    if (rc) return rc;
    if (loss)
        return launch(ctx, k_gemm<EPI_LOSS, true>, gemm_grid(B, O), B, O, H, a.h2, p.W3, H, p.b3, nullptr, a.dy, a.T, a.M,
                      a.lpart, loss_scale(w, B));
    return layer(k_gemm<EPI_BIAS, true>, k_gemm<EPI_BIAS, true, 1>, O, H, a.h2, p.W3, p.b3, nullptr, a.y);
}

// Gradient of the masked loss, into w->grad (adam = nullptr) or straight into
// the update.
int backward(dvqls_ws* w, const Views& a, int B, const AdamArgs* adam) {
    dvqls_ctx* ctx = w->ctx;
    const int I = w->I, H = w->H, O = w->O;
    const Params p = params_of(w);
    // d2[b, h] = sum_o dy[b, o] W3[o, h] GELU'(z2), d1[b, k] = sum_h d2[b, h] W2[h, k] GELU'(z1)
    int rc = launch(ctx, k_gemm<EPI_BACK, false>, gemm_grid(B, H), B, H, O, a.dy, p.W3, H, nullptr, a.z2, a.d2, nullptr,
                    nullptr, nullptr, 1.f);
    if (!rc)
        rc = launch(ctx, k_gemm<EPI_BACK, false>, gemm_grid(B, H), B, H, H, a.d2, p.W2, H, nullptr, a.z1, a.d1, nullptr,
                    nullptr, nullptr, 1.f);
    if (rc) return rc;
    GradJobs jobs;
    int tiles = 0;
    auto job = [&](int q, const float* D, const float* in, int M, int N, const float* W, const float* b) {
        const int tn = ceil_div(N, GT);
        jobs.j[q] = {D, in, M, N, tn, tiles, W - w->params, b - w->params};
        tiles += ceil_div(M, GT) * tn;
    };
    job(0, a.d2, a.h1, H, H, p.W2, p.b2);
    job(1, a.dy, a.h2, O, H, p.W3, p.b3);
    job(2, a.d1, a.X, H, I, p.W1, p.b1);
    const int splits = std::min(max_splits(w), ceil_div(B, GT));
    const int per = ceil_div(B, splits);
    rc = launch(ctx, k_wgrad, dim3(tiles, ceil_div(B, per)), jobs, B, per, w->np, a.gpart);
    if (rc) return rc;
    const dim3 lg = gemm_grid(B, O);
    return launch(ctx, k_grad_update, dim3(ceil_div(w->np, 256)), w->np, ceil_div(B, per), a.gpart, int(lg.x * lg.y), a.lpart,
                  w->lossbuf, adam ? nullptr : w->grad, w->params, w->m, w->v, adam ? *adam : AdamArgs{}, 1.f / loss_scale(w, B));
}

int copy_in(dvqls_ws* w, float* dst, const float* src, long long n) {
    if (!src) return set_error(w->ctx, DVQLS_ERR_INVALID_ARG, "NULL input");
    DVQLS_CUDA_TRY(w->ctx, cudaMemcpyAsync(dst, src, size_t(n) * 4, cudaMemcpyDefault, w->ctx->stream));
    return DVQLS_OK;
}

// A batch array for the kernels: the caller's own when it is (aligned) device
// memory, else a copy.
int batch_in(dvqls_ws* w, const float*& use, float* copy, const float* src, long long n) {
    if (is_device_ptr(w->ctx, src) && reinterpret_cast<uintptr_t>(src) % alignof(float) == 0) {
        use = src;
        return DVQLS_OK;
    }
    use = copy;
    return copy_in(w, copy, src, n);
}

int read_loss(dvqls_ws* w, float* loss) {
    if (!loss) return DVQLS_OK;
    float* hb = reinterpret_cast<float*>(w->pin);
    DVQLS_CUDA_TRY(w->ctx, cudaMemcpyAsync(hb, w->lossbuf, 8, cudaMemcpyDeviceToHost, w->ctx->stream));
    DVQLS_CUDA_TRY(w->ctx, cudaStreamSynchronize(w->ctx->stream));
    *loss = hb[1] > 0.f ? hb[0] / hb[1] : 0.f;
    return DVQLS_OK;
}

}  // namespace
}  // namespace dvqls

using namespace dvqls;

extern "C" long long dvqls_ws_param_count(int I, int H, int O) {
    if (I < 1 || H < 1 || O < 1) return -1;
    return (long long)H * I + H + (long long)H * H + H + (long long)O * H + O;
}

extern "C" void dvqls_ws_destroy(dvqls_ws* w) {
    if (!w) return;
    cudaSetDevice(w->ctx->device);
    cudaStreamSynchronize(w->ctx->stream);
    if (w->params) cudaFree(w->params);
    if (w->act) cudaFree(w->act);
    if (w->pin) cudaFreeHost(w->pin);
    cudaGetLastError();
    delete w;
}

extern "C" int dvqls_ws_create(dvqls_ctx* ctx, int I, int H, int O, const float* params, dvqls_ws** out) {
    if (!ctx) return DVQLS_ERR_INVALID_ARG;
    ctx->err.clear();
    if (!out || !params) return set_error(ctx, DVQLS_ERR_INVALID_ARG, "NULL argument");
    *out = nullptr;
    const long long np = dvqls_ws_param_count(I, H, O);
    if (np < 1 || I > 4096 || H > 4096 || O > 4096) return set_error(ctx, DVQLS_ERR_INVALID_ARG, "bad dimensions");
    cudaSetDevice(ctx->device);
    dvqls_ws* w = new dvqls_ws();
    w->ctx = ctx;
    w->I = I;
    w->H = H;
    w->O = O;
    w->np = np;
    // params, grad, m, v in one allocation, then the loss buffer.
    if (cudaMalloc(&w->params, size_t(4 * np + 64) * sizeof(float)) != cudaSuccess ||
        cudaMallocHost(&w->pin, 64) != cudaSuccess) {
        cudaGetLastError();
        dvqls_ws_destroy(w);
        return set_error(ctx, DVQLS_ERR_ALLOC, "warm-start parameters");
    }
    w->grad = w->params + np;
    w->m = w->grad + np;
    w->v = w->m + np;
    w->lossbuf = w->v + np;
    int rc = copy_in(w, w->params, params, np);
    if (!rc && cudaMemsetAsync(w->m, 0, size_t(2 * np) * 4, ctx->stream) != cudaSuccess) rc = DVQLS_ERR_CUDA;
    if (!rc && cudaStreamSynchronize(ctx->stream) != cudaSuccess) rc = DVQLS_ERR_CUDA;
    if (rc) {
        cudaGetLastError();
        dvqls_ws_destroy(w);
        return set_error(ctx, rc, "warm-start initialisation");
    }
    *out = w;
    return DVQLS_OK;
}

extern "C" int dvqls_ws_infer(dvqls_ws* w, int batch, const float* feats, float* out) {
    DVQLS_NVTX("dvqls_ws_infer");
    if (!w) return DVQLS_ERR_INVALID_ARG;
    dvqls_ctx* ctx = w->ctx;
    ctx->err.clear();
    if (batch < 1 || !feats || !out) return set_error(ctx, DVQLS_ERR_INVALID_ARG, "batch < 1 or NULL");
    cudaSetDevice(ctx->device);
    int rc = ensure_batch(w, batch);
    if (rc) return rc;
    Views a = views(w);
    rc = batch_in(w, a.X, a.Xc, feats, (long long)batch * w->I);
    if (!rc) rc = forward(w, a, batch, false);
    if (rc) return rc;
    DVQLS_CUDA_TRY(ctx, cudaMemcpyAsync(out, a.y, size_t(batch) * w->O * 4, cudaMemcpyDefault, ctx->stream));
    DVQLS_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    return DVQLS_OK;
}

static int grad_common(dvqls_ws* w, int batch, const float* feats, const float* target, const float* mask,
                       const AdamArgs* adam) {
    dvqls_ctx* ctx = w->ctx;
    if (batch < 1 || !feats || !target || !mask) return set_error(ctx, DVQLS_ERR_INVALID_ARG, "batch < 1 or NULL");
    cudaSetDevice(ctx->device);
    int rc = ensure_batch(w, batch);
    if (rc) return rc;
    Views a = views(w);
    rc = batch_in(w, a.X, a.Xc, feats, (long long)batch * w->I);
    if (!rc) rc = batch_in(w, a.T, a.Tc, target, (long long)batch * w->O);
    if (!rc) rc = batch_in(w, a.M, a.Mc, mask, (long long)batch * w->O);
    if (!rc) rc = forward(w, a, batch, true);
    if (!rc) rc = backward(w, a, batch, adam);
    return rc;
}

extern "C" int dvqls_ws_grad(dvqls_ws* w, int batch, const float* feats, const float* target, const float* mask,
                             float* loss, float* grad) {
    if (!w) return DVQLS_ERR_INVALID_ARG;
    w->ctx->err.clear();
    if (!grad) return set_error(w->ctx, DVQLS_ERR_INVALID_ARG, "grad is NULL");
    int rc = grad_common(w, batch, feats, target, mask, nullptr);
    if (rc) return rc;
    DVQLS_CUDA_TRY(w->ctx, cudaMemcpyAsync(grad, w->grad, size_t(w->np) * 4, cudaMemcpyDefault, w->ctx->stream));
    rc = read_loss(w, loss);
    if (rc) return rc;
    DVQLS_CUDA_TRY(w->ctx, cudaStreamSynchronize(w->ctx->stream));
    return DVQLS_OK;
}

extern "C" int dvqls_ws_train_step(dvqls_ws* w, int batch, const float* feats, const float* target, const float* mask,
                                   float lr, float* loss) {
    DVQLS_NVTX("dvqls_ws_train_step");
    if (!w) return DVQLS_ERR_INVALID_ARG;
    w->ctx->err.clear();
    if (!(lr > 0.f)) return set_error(w->ctx, DVQLS_ERR_INVALID_ARG, "lr must be > 0");
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f, t = float(w->step + 1);
    const AdamArgs adam{lr, b1, b2, eps, 1.f - powf(b1, t), 1.f - powf(b2, t)};
    int rc = grad_common(w, batch, feats, target, mask, &adam);
    if (rc) return rc;
    w->step += 1;
    return read_loss(w, loss);
}

extern "C" int dvqls_ws_get_params(dvqls_ws* w, float* params) {
    if (!w) return DVQLS_ERR_INVALID_ARG;
    if (!params) return set_error(w->ctx, DVQLS_ERR_INVALID_ARG, "NULL params");
    cudaSetDevice(w->ctx->device);
    DVQLS_CUDA_TRY(w->ctx, cudaMemcpyAsync(params, w->params, size_t(w->np) * 4, cudaMemcpyDefault, w->ctx->stream));
    DVQLS_CUDA_TRY(w->ctx, cudaStreamSynchronize(w->ctx->stream));
    return DVQLS_OK;
}

// File: "DVQLSWS1", int32 I, H, O, int64 Adam step, then params, m, v (FP32).
extern "C" int dvqls_ws_save(dvqls_ws* w, const char* path) {
    if (!w) return DVQLS_ERR_INVALID_ARG;
    if (!path) return set_error(w->ctx, DVQLS_ERR_INVALID_ARG, "NULL path");
    cudaSetDevice(w->ctx->device);
    std::vector<float> buf(size_t(3 * w->np));
    DVQLS_CUDA_TRY(w->ctx, cudaStreamSynchronize(w->ctx->stream));
    DVQLS_CUDA_TRY(w->ctx, cudaMemcpy(buf.data(), w->params, size_t(w->np) * 4, cudaMemcpyDeviceToHost));
    DVQLS_CUDA_TRY(w->ctx, cudaMemcpy(buf.data() + w->np, w->m, size_t(2 * w->np) * 4, cudaMemcpyDeviceToHost));
    FILE* f = fopen(path, "wb");
    if (!f) return set_error(w->ctx, DVQLS_ERR_INVALID_ARG, "cannot open %s", path);
    const int dims[3] = {w->I, w->H, w->O};
    bool ok = fwrite("DVQLSWS1", 1, 8, f) == 8 && fwrite(dims, 4, 3, f) == 3 && fwrite(&w->step, 8, 1, f) == 1 &&
              fwrite(buf.data(), 4, buf.size(), f) == buf.size();
    ok = (fclose(f) == 0) && ok;
    return ok ? DVQLS_OK : set_error(w->ctx, DVQLS_ERR_INVALID_ARG, "write failed: %s", path);
}

extern "C" int dvqls_ws_load(dvqls_ctx* ctx, const char* path, dvqls_ws** out) {
    if (!ctx) return DVQLS_ERR_INVALID_ARG;
    ctx->err.clear();
    if (!path || !out) return set_error(ctx, DVQLS_ERR_INVALID_ARG, "NULL argument");
    FILE* f = fopen(path, "rb");
    if (!f) return set_error(ctx, DVQLS_ERR_INVALID_ARG, "cannot open %s", path);
    char magic[8];
    int dims[3];
    long long step = 0;
    bool ok = fread(magic, 1, 8, f) == 8 && memcmp(magic, "DVQLSWS1", 8) == 0 && fread(dims, 4, 3, f) == 3 &&
              fread(&step, 8, 1, f) == 1;
    const long long np = ok ? dvqls_ws_param_count(dims[0], dims[1], dims[2]) : -1;
    std::vector<float> buf(np > 0 ? size_t(3 * np) : 0);
    ok = ok && np > 0 && fread(buf.data(), 4, buf.size(), f) == buf.size();
    fclose(f);
    if (!ok) return set_error(ctx, DVQLS_ERR_INVALID_ARG, "not a warm-start file: %s", path);
    int rc = dvqls_ws_create(ctx, dims[0], dims[1], dims[2], buf.data(), out);
    if (rc) return rc;
    (*out)->step = step;
    DVQLS_CUDA_TRY(ctx, cudaMemcpy((*out)->m, buf.data() + np, size_t(2 * np) * 4, cudaMemcpyHostToDevice));
    return DVQLS_OK;
}
