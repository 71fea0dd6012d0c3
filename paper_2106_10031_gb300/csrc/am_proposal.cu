// am_proposal.cu -- the learned constraint proposal: a small MLP, trained on the GPU, that
// scores every hidden neuron of the meshed net by how likely its plane carries an edge of a
// cell's face.  The march clips with its 32 best-scored rows first; the all-row check that
// follows keeps the mesh exact whatever the scores are.
//
//   x (7 + L) -> h1 = relu(W1 x + b1) (H) -> h2 = relu(W2 h1 + b2) (H) -> z = W3 h2 + b3 (n_out)
//   training loss: mean binary cross-entropy of sigmoid(z) against the 0/1 boundary labels.
//
// Training is mixed precision: FP32 master weights, BF16 operands for every matrix product,
// FP32 accumulation, Adam.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cuda_bf16.h>
#include <vector>

#include "am_kernels.h"

namespace am {

// ---- products of BF16 operands on the FP32 pipes
//
// Every element of a product is one chain of fused multiply-adds over k in ascending order from zero, so it
// does not depend on the tile, the launch or the device's load (a split of k, or the tensor cores' own order,
// would move the BF16 roundings between the layers).  The loss and the bias gradients are sums of partial sums
// whose number follows the tile, so with another batch their last bits may differ; runs repeat bit for bit.
// What bounds a training step of this MLP (batch 1024, 15 -> 256 -> 256 -> 2048: 1.8 G multiply-adds, 46 us at
// the FP32 peak) is keeping the FP32 pipes fed along chains of up to 2048 k: slices of 32 k are staged in
// shared memory as FP32, the next two slices' loads in flight while one is multiplied, the operands of the
// next k read while those of one are multiplied, each thread keeps a TM x TN block of sums, and the products
// that wait for the same input share one launch, with their bias, activation, loss or backward step as the
// epilogue.  A step takes 291 us; 933 with a 64 x 64 kernel per product (4 loads per 8 multiply-adds, strided
// global reads), its element-wise kernels and a copy of the loss to the host per step.

constexpr int kGK = 32;     // K slice
constexpr int kLossSteps = 4096;     // losses kept on the device between copies

enum { kEpiStore = 0, kEpiBias = 1, kEpiBiasRelu = 2, kEpiBce = 3, kEpiReluBack = 4, kEpiColsum = 5 };

// C[M x N] = op(A)[M x K] op(B)[K x N] and an epilogue.  A is row-major M x K (lda = K) or, with ta, stored
// K x M (lda = M); B is row-major K x N (ldb = N) or, with tb, stored N x K.
struct GemmJob {
    int M, N, K, lda, ldb, ta, tb, epi;
    int ldc, ldy;                 // row strides of C and H, and of Y
    int va, vb;                   // A, B: rows of 16-byte pieces (8 | ld, 16-byte aligned)
    const __nv_bfloat16 *A, *B;
    float *C;
    const float *bias;            // kEpiBias, kEpiBiasRelu, kEpiBce: per column
    __nv_bfloat16 *H;             // BF16 result: activations (kEpiBiasRelu), dz (kEpiBce), da (kEpiReluBack)
    const float *Y;               // kEpiBce: labels, kEpiReluBack: the layer's pre-activations
    float scale;                  // kEpiBce: 1 / (rows cols)
    float *loss_parts;            // kEpiBce: one sum of softplus(z) - y z per tile
};
constexpr int kMaxJobs = 3;
struct GemmJobs {
    GemmJob j[kMaxJobs];
    int first[kMaxJobs + 1];      // first tile of each job (kEpiColsum: blocks of 32 columns)
    int n;
};

// db[c] = sum over rows of C[r, c]: 32 columns per block, the rows in T / 32 groups (8 or 4, with the launch's
// tile) combined in shared memory
template <int T>
__device__ __forceinline__ void colsum_block(const GemmJob &g, int tile, float *sh)
{
    constexpr int G = T / 32;
    const int c = tile * 32 + (threadIdx.x & 31), q = threadIdx.x >> 5;
    float s = 0.0f;
    if (c < g.N) {
#pragma unroll 8
        for (int r = q; r < g.M; r += G) s += g.C[(size_t)r * g.ldc + c];
    }
    sh[threadIdx.x] = s;
    __syncthreads();
    if (q == 0 && c < g.N) {
        for (int w = 1; w < G; ++w) s += sh[threadIdx.x + 32 * w];
        const_cast<float *>(g.bias)[c] = s;          // the job's output vector
    }
}

// 8 consecutive BF16 elements at p (n of them inside the matrix, none if n <= 0).  The 16-byte form is one
// predicated load and nothing looks at its value: the elements past n, which the row's stride covers, are
// zeroed by tail8 when the slice is stored.  (With the mask here every load was waited for where it was
// issued, and a slice of 32 k took two trips to L2 longer: 332 us per step of 1024 samples.)
__device__ __forceinline__ void load8(uint4 &v, const __nv_bfloat16 *p, int n, bool vec)
{
    v = make_uint4(0u, 0u, 0u, 0u);
    if (vec) {
        asm volatile("{\n\t.reg .pred q;\n\tsetp.gt.s32 q, %5, 0;\n\t@q ld.global.v4.u32 {%0, %1, %2, %3}, [%4];\n\t}"
                     : "+r"(v.x), "+r"(v.y), "+r"(v.z), "+r"(v.w) : "l"(p), "r"(n) : "memory");
        return;
    }
    unsigned w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const unsigned lo = 2 * j < n ? __bfloat16_as_ushort(p[2 * j]) : 0u;
        const unsigned hi = 2 * j + 1 < n ? __bfloat16_as_ushort(p[2 * j + 1]) : 0u;
        w[j] = lo | (hi << 16);
    }
    v = make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ uint4 tail8(uint4 v, int n)
{
    if (n < 8) {
        unsigned *w = &v.x;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (2 * j >= n) w[j] = 0u;
            else if (2 * j + 1 >= n) w[j] &= 0xffffu;
        }
    }
    return v;
}

template <int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN)) gemm_jobs_kernel(const __grid_constant__ GemmJobs jobs)
{
    constexpr int T = (BM / TM) * (BN / TN), CX = BN / TN;
    constexpr int LA = BM + 4, LB = BN + 4;          // row strides: 16-byte rows
    static_assert(BM == BN && BM * kGK / 8 == T && BM % 32 == 0, "one 16-byte piece of A and of B per thread and slice");
    __shared__ __align__(16) float As[2][kGK][LA];
    __shared__ __align__(16) float Bs[2][kGK][LB];
    int ji = 0;
    while (ji + 1 < jobs.n && (int)blockIdx.x >= jobs.first[ji + 1]) ++ji;
    const GemmJob &g = jobs.j[ji];
    const int tile = (int)blockIdx.x - jobs.first[ji];
    if (g.epi == kEpiColsum) {
        colsum_block<T>(g, tile, &As[0][0][0]);
        return;
    }
    const int tiles_n = (g.N + BN - 1) / BN;
    const int row0 = tile / tiles_n * BM, col0 = tile % tiles_n * BN;
    const int tid = threadIdx.x, tx = tid % CX, ty = tid / CX, lane = tid & 31, warp = tid >> 5;
    // a thread's piece of a slice.  Stored k-contiguous: 8 k of row km, the rows along the lanes (the
    // stores of one k then fall in 32 banks); stored m-contiguous: 8 rows from mm of k = mk
    const int km = tid % BM, kq = 8 * (tid / BM), mm = 8 * (tid % (BM / 8)), mk = tid / (BM / 8);
    const int M = g.M, N = g.N, K = g.K;
    // elements of a thread's piece inside the matrix, and its place
    auto inside = [&](bool mfirst, int m0, int m_end, int k0) {
        if (mfirst) return k0 + mk < K ? m_end - (m0 + mm) : 0;
        return m0 + km < m_end ? K - (k0 + kq) : 0;
    };
    auto place = [&](const __nv_bfloat16 *X, int ld, bool mfirst, int m0, int k0) {
        return mfirst ? X + (size_t)(k0 + mk) * ld + m0 + mm : X + (size_t)(m0 + km) * ld + k0 + kq;
    };
    auto put = [&](float *S, int ls, bool mfirst, const uint4 v) {
        const unsigned w[4] = {v.x, v.y, v.z, v.w};
        float f[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            f[2 * j] = __uint_as_float(w[j] << 16);
            f[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
        }
        if (mfirst) {
            float4 *o = reinterpret_cast<float4 *>(S + mk * ls + mm);
            o[0] = make_float4(f[0], f[1], f[2], f[3]);
            o[1] = make_float4(f[4], f[5], f[6], f[7]);
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) S[(kq + j) * ls + km] = f[j];
        }
    };
    uint4 ra[2], rb[2];              // the slices of k0 + 32 and k0 + 64
    auto load = [&](uint4 &a, uint4 &b, int k0) {
        if (k0 >= K) return;
        load8(a, place(g.A, g.lda, g.ta, row0, k0), inside(g.ta, row0, M, k0), g.va);
        load8(b, place(g.B, g.ldb, !g.tb, col0, k0), inside(!g.tb, col0, N, k0), g.vb);
    };
    auto store = [&](int buf, const uint4 &a, const uint4 &b, int k0) {
        if (k0 >= K) return;
        put(&As[buf][0][0], LA, g.ta, tail8(a, inside(g.ta, row0, M, k0)));
        put(&Bs[buf][0][0], LB, !g.tb, tail8(b, inside(!g.tb, col0, N, k0)));
    };
    float acc[TM][TN] = {};
    auto multiply = [&](const int buf) {
        // operands of k + D in flight while those of k are multiplied: shared memory answers after 34
        // cycles, and few warps share a scheduler
        constexpr int D = TM == 4 ? 2 : 4;
        float av[D][TM], bv[D][TN];
        auto operands = [&](int kk) {
            if constexpr (TM == 4) *reinterpret_cast<float4 *>(av[kk % D]) = *reinterpret_cast<const float4 *>(&As[buf][kk][ty * TM]);
            else *reinterpret_cast<float2 *>(av[kk % D]) = *reinterpret_cast<const float2 *>(&As[buf][kk][ty * TM]);
            *reinterpret_cast<float4 *>(bv[kk % D]) = *reinterpret_cast<const float4 *>(&Bs[buf][kk][tx * TN]);
        };
#pragma unroll
        for (int kk = 0; kk < D; ++kk) operands(kk);
#pragma unroll
        for (int kk = 0; kk < kGK; ++kk) {
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(av[kk % D][i], bv[kk % D][j], acc[i][j]);
            if (kk + D < kGK) operands(kk + D);
        }
    };
    load(ra[0], rb[0], 0);
    load(ra[1], rb[1], kGK);
    store(0, ra[0], rb[0], 0);
    __syncthreads();
    for (int k0 = 0; k0 < K; k0 += 2 * kGK) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = k0 + h * kGK;
            if (k >= K) break;
            load(ra[h], rb[h], k + 2 * kGK);
            multiply(h);
            store(h ^ 1, ra[h ^ 1], rb[h ^ 1], k + kGK);
            __syncthreads();
        }
    }
    float part = 0.0f;
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const int r = row0 + ty * TM + i, c = col0 + tx * TN + j;
            if (r >= g.M || c >= g.N) continue;
            const size_t o = (size_t)r * g.ldc + c;
            const float v = acc[i][j] + 0.0f;
            if (g.epi == kEpiStore) {
                g.C[o] = v;
            } else if (g.epi == kEpiBias) {
                g.C[o] = v + g.bias[c];
            } else if (g.epi == kEpiBiasRelu) {
                const float z = v + g.bias[c];
                g.C[o] = z;
                g.H[o] = __float2bfloat16_rn(fmaxf(z, 0.0f));
            } else if (g.epi == kEpiBce) {
                // dz = (sigmoid(z) - y) / (rows cols), and this element of the loss
                const float z = v + g.bias[c], y = g.Y[(size_t)r * g.ldy + c];
                part += (z > 0.0f ? z + log1pf(expf(-z)) : log1pf(expf(z))) - y * z;
                const float d = (1.0f / (1.0f + expf(-z)) - y) * g.scale;
                g.H[o] = __float2bfloat16_rn(d);
                g.C[o] = d;
            } else {
                // da = dh (a > 0)
                const float d = g.Y[(size_t)r * g.ldy + c] > 0.0f ? v : 0.0f;
                g.H[o] = __float2bfloat16_rn(d);
                g.C[o] = d;
            }
        }
    if (g.epi == kEpiBce) {
        float *red = &As[0][0][0];
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        if (lane == 0) red[warp] = part;
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < T / 32; ++w) part += red[w];
            g.loss_parts[tile] = part;
        }
    }
}

// the products of one launch
struct JobList {
    GemmJobs q{};
    void add(const GemmJob &g) { q.j[q.n++] = g; }
    // launches them; returns the number of tiles (of a product with the loss: its partial sums)
    int run(cudaStream_t st)
    {
        // 64 x 64 tiles (3 shared-memory wavefronts per 16 multiply-adds of a warp) when they fill the
        // chip twice, else 32 x 32 (four times as many, of half the threads): the logits of 1024 samples
        // take 50 us in 512 large tiles, dW3 and dh2 124 us in 832 small ones where 192 large ones leave
        // most schedulers one warp.  One 64 x 32 tile for both took 3.12 ms for 8 steps against 2.66.
        auto tiles = [&](int B) {
            int t = 0;
            for (int i = 0; i < q.n; ++i) {
                const GemmJob &g = q.j[i];
                q.first[i] = t;
                t += g.epi == kEpiColsum ? (g.N + 31) / 32 : ((g.M + B - 1) / B) * ((g.N + B - 1) / B);
            }
            q.first[q.n] = t;
            return t;
        };
        int t = tiles(64);
        if (t >= 2 * 152) {
            gemm_jobs_kernel<64, 64, 4, 4><<<t, 256, 0, st>>>(q);
        } else {
            t = tiles(32);
            gemm_jobs_kernel<32, 32, 2, 4><<<t, 128, 0, st>>>(q);
        }
        q = GemmJobs{};
        return t;
    }
};

static GemmJob product(int M, int N, int K, const __nv_bfloat16 *A, int lda, bool ta, const __nv_bfloat16 *B, int ldb,
                       bool tb, float *C, int epi)
{
    GemmJob g{};
    g.M = M; g.N = N; g.K = K;
    g.A = A; g.lda = lda; g.ta = ta;
    g.B = B; g.ldb = ldb; g.tb = tb;
    g.C = C;
    g.ldc = g.ldy = N;
    g.epi = epi;
    g.va = lda % 8 == 0 && (uintptr_t)A % 16 == 0;
    g.vb = ldb % 8 == 0 && (uintptr_t)B % 16 == 0;
    return g;
}

static GemmJob column_sum(const float *G, int rows, int cols, int ld, float *db)
{
    GemmJob g{};
    g.M = rows; g.N = cols;
    g.ldc = ld;
    g.C = const_cast<float *>(G);
    g.bias = db;
    g.epi = kEpiColsum;
    return g;
}

static int blocks_for(int64_t n) { return (int)std::min<int64_t>((n + 255) / 256, 152 * 16); }

// BF16 copy of a rows x cols matrix with row stride ld >= cols (the padding is zero)
__global__ void pad_bf16_kernel(const float *x, int rows, int cols, int ld, __nv_bfloat16 *y)
{
    const int64_t n = (int64_t)rows * ld;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(i % ld);
        y[i] = __float2bfloat16_rn(c < cols ? x[i / ld * cols + c] : 0.0f);
    }
}

static int up8(int n) { return (n + 7) & ~7; }      // row stride of the activations: 16-byte pieces

__global__ void to_bf16_kernel(const float *x, __nv_bfloat16 *y, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = __float2bfloat16_rn(x[i]);
}

// losses[it] = the sum of n partial sums (FP64) over count, for a training step; one block
__global__ void loss_kernel(const float *parts, int n, double count, float *loss)
{
    __shared__ double red[8];
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) s += (double)parts[i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)blockDim.x / 32; ++w) s += red[w];
        *loss = (float)(s / count);
    }
}

// Adam (Kingma & Ba 2015) on the FP32 master weights, then the BF16 copy
__global__ void adam_kernel(float *w, const float *g, float *m, float *v, __nv_bfloat16 *wb, int64_t n, float lr,
                            float b1, float b2, float eps, float c1, float c2)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        w[i] = wi;
        if (wb) wb[i] = __float2bfloat16_rn(wi);
    }
}

// transposed BF16 copy of a rows x cols FP32 matrix with row stride ld >= rows (the padding is
// zero), for coalesced BF16-pair reads in the march
__global__ void transpose_bf16_kernel(const float *W, int rows, int cols, int ld, __nv_bfloat16 *WT)
{
    const int64_t n = (int64_t)ld * cols;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(i / ld), r = (int)(i % ld);
        WT[i] = __float2bfloat16_rn(r < rows ? W[(size_t)r * cols + c] : 0.0f);
    }
}

// One warp per face.  The face plane comes from the vertices (Newell's normal, which points
// along +grad F because faces are stored CCW about it); the march computes the same plane from
// a_F, so both give one feature vector up to rounding.
__global__ void __launch_bounds__(256) proposal_samples_kernel(SampleArgs a)
{
    __shared__ float feat[8][7 + kMaxLayers];
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t i = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); i < a.nf; i += warps) {
        const int64_t f = a.f0 + i;
        const int64_t cb = a.coff[f] - a.c0;
        if (cb >= a.max_samples) continue;
        const int m = (int)(a.coff[f + 1] - a.coff[f]);
        const int64_t cell = a.perm[f];
        const double *V = a.ar.verts + cell * a.ar.maxv * 3;
        const int32_t *E = a.ar.edges + cell * a.ar.maxv;
        double nx = 0.0, ny = 0.0, nz = 0.0, cx = 0.0, cy = 0.0, cz = 0.0;
        for (int j = 0; j < m; ++j) {
            const double *p = V + 3 * j, *q = V + 3 * ((j + 1) % m);
            nx += p[1] * q[2] - p[2] * q[1];
            ny += p[2] * q[0] - p[0] * q[2];
            nz += p[0] * q[1] - p[1] * q[0];
            cx += p[0]; cy += p[1]; cz += p[2];
        }
        const double inv = 1.0 / sqrt(nx * nx + ny * ny + nz * nz);
        nx *= inv; ny *= inv; nz *= inv;
        const double off = -(nx * cx + ny * cy + nz * cz) / m;
        float *x = feat[threadIdx.x >> 5];
        if (lane < a.L) {
            const unsigned long long *key = a.ar.keys + cell * a.ar.kw;
            const int r0 = a.row0[lane + 1], n = a.width[lane + 1];
            int cnt = 0;
            for (int b = r0; b < r0 + n; ++b) cnt += (int)((key[b >> 6] >> (b & 63)) & 1ull);
            x[7 + lane] = (float)cnt / (float)n;
        }
        if (lane == 0) { x[3] = (float)nx; x[4] = (float)ny; x[5] = (float)nz; x[6] = (float)off; }
        for (int j = 0; j < m && cb + j < a.max_samples; ++j) {
            const int64_t smp = cb + j;
            const double *p = V + 3 * j, *q = V + 3 * ((j + 1) % m);
            if (lane < 3) x[lane] = (float)(0.5 * (p[lane] + q[lane]));
            __syncwarp();
            for (int c = lane; c < a.n_in; c += 32) a.X[smp * a.n_in + c] = x[c];
            __syncwarp();
            float *y = a.Y + smp * a.N;
            for (int k = lane; k < a.N; k += 32) y[k] = 0.0f;
            __syncwarp();
            for (int t = lane; t < m; t += 32)
                if (E[t] < a.N) y[E[t]] = 1.0f;
            __syncwarp();
        }
    }
}

void launch_proposal_samples(const SampleArgs &a, cudaStream_t st)
{
    const int64_t blocks = std::min<int64_t>((a.nf + 7) / 8, 152 * 8);
    if (blocks > 0) proposal_samples_kernel<<<(int)blocks, 256, 0, st>>>(a);
}


// ------------------------------------------------------------------------------------------

cudaError_t proposal_alloc(ProposalDev &p, int n_in, int hidden, int n_out, int max_batch)
{
    p.n_in = n_in;
    p.hidden = hidden;
    p.n_out = n_out;
    p.max_batch = max_batch;
    const int64_t sizes[6] = {(int64_t)hidden * n_in, hidden, (int64_t)hidden * hidden, hidden, (int64_t)n_out * hidden,
                              n_out};
    int64_t tot = 0;
    for (int i = 0; i < 6; ++i) { p.off[i] = tot; tot += sizes[i]; }
    p.off[6] = tot;
    p.n_params = tot;
    cudaError_t e;
    if ((e = cudaMalloc(&p.w, sizeof(float) * tot))) return e;
    if ((e = cudaMalloc(&p.g, sizeof(float) * tot))) return e;
    if ((e = cudaMalloc(&p.m, sizeof(float) * tot))) return e;
    if ((e = cudaMalloc(&p.v, sizeof(float) * tot))) return e;
    if ((e = cudaMalloc(&p.wb, sizeof(__nv_bfloat16) * tot))) return e;
    if ((e = cudaMalloc(&p.w2t, sizeof(__nv_bfloat16) * hidden * hidden))) return e;
    if ((e = cudaMalloc(&p.w3t, sizeof(__nv_bfloat16) * hidden * (n_out + 1)))) return e;
    const int64_t act = (int64_t)max_batch * up8(std::max(std::max(hidden, n_out), n_in));
    for (int i = 0; i < 8; ++i)
        if ((e = cudaMalloc(&p.buf[i], sizeof(float) * act))) return e;
    for (int i = 0; i < 6; ++i)
        if ((e = cudaMalloc(&p.bbuf[i], sizeof(__nv_bfloat16) * act))) return e;
    const int64_t tiles = (int64_t)((max_batch + 31) / 32) * ((n_out + 31) / 32);
    if ((e = cudaMalloc(&p.loss_parts, sizeof(float) * tiles))) return e;
    if ((e = cudaMalloc(&p.losses, sizeof(float) * kLossSteps))) return e;
    // the forward pass of whole batches on the tensor cores (inference: am_proposal_forward and
    // the level march), when the shape allows it; W2 and W3 are read in place from the BF16 copy
    return prop_tc_alloc(p.tc, n_in, hidden, n_out, std::max(max_batch, 4096), p.wb + p.off[2], p.wb + p.off[4]);
}

void proposal_free(ProposalDev &p)
{
    void *b[] = {p.w, p.g, p.m, p.v, p.wb, p.w2t, p.w3t, p.loss_parts, p.losses};
    for (void *x : b)
        if (x) cudaFree(x);
    for (int i = 0; i < 8; ++i)
        if (p.buf[i]) cudaFree(p.buf[i]);
    for (int i = 0; i < 6; ++i)
        if (p.bbuf[i]) cudaFree(p.bbuf[i]);
    prop_tc_free(p.tc);
    p = ProposalDev{};
}

void proposal_sync_copies(ProposalDev &p, cudaStream_t st)
{
    to_bf16_kernel<<<blocks_for(p.n_params), 256, 0, st>>>(p.w, p.wb, p.n_params);
    const int ld3 = (p.n_out + 1) & ~1;
    transpose_bf16_kernel<<<blocks_for((int64_t)p.hidden * p.hidden), 256, 0, st>>>(p.w + p.off[2], p.hidden, p.hidden,
                                                                                   p.hidden, p.w2t);
    transpose_bf16_kernel<<<blocks_for((int64_t)ld3 * p.hidden), 256, 0, st>>>(p.w + p.off[4], p.n_out, p.hidden, ld3,
                                                                              p.w3t);
    prop_tc_sync_weights(p.tc, p.w + p.off[0], st);
}

// Forward pass over B samples (B <= max_batch).  Activations: buf0 a1, buf1 a2 (FP32, for the backward
// pass); bbuf0 x, bbuf1 h1, bbuf2 h2 (BF16).  Without labels the logits go to buf2; with labels Y the loss's
// partial sums to loss_parts and dz to buf3 (FP32) and bbuf3 (BF16).  Returns the number of partial sums.
static int forward(ProposalDev &p, const float *X, const float *Y, int B, cudaStream_t st)
{
    const int H = p.hidden, I = p.n_in, O = p.n_out;
    const __nv_bfloat16 *W1 = p.wb + p.off[0], *W2 = p.wb + p.off[2], *W3 = p.wb + p.off[4];
    JobList q;
    pad_bf16_kernel<<<blocks_for((int64_t)B * up8(I)), 256, 0, st>>>(X, B, I, up8(I), p.bbuf[0]);
    GemmJob g = product(B, H, I, p.bbuf[0], up8(I), false, W1, I, true, p.buf[0], kEpiBiasRelu);          // a1 = X W1^T + b1
    g.bias = p.w + p.off[1];
    g.H = p.bbuf[1];
    q.add(g);
    q.run(st);
    g = product(B, H, H, p.bbuf[1], H, false, W2, H, true, p.buf[1], kEpiBiasRelu);                  // a2 = h1 W2^T + b2
    g.bias = p.w + p.off[3];
    g.H = p.bbuf[2];
    q.add(g);
    q.run(st);
    g = product(B, O, H, p.bbuf[2], H, false, W3, H, true, Y ? p.buf[3] : p.buf[2], Y ? kEpiBce : kEpiBias);   // z = h2 W3^T + b3
    g.bias = p.w + p.off[5];
    g.H = p.bbuf[3];
    g.Y = Y;
    if (Y) g.ldc = up8(O);
    g.scale = 1.0f / (float)((int64_t)B * O);
    g.loss_parts = p.loss_parts;
    q.add(g);
    return q.run(st);
}

// Gradients (into p.g) over B samples, after forward with labels.  da2: buf5, bbuf4; da1: buf6, bbuf5.
static void backward(ProposalDev &p, int B, cudaStream_t st)
{
    const int H = p.hidden, I = p.n_in, O = p.n_out;
    JobList q;
    q.add(product(O, H, B, p.bbuf[3], up8(O), true, p.bbuf[2], H, false, p.g + p.off[4], kEpiStore));             // dW3 = dz^T h2
    GemmJob g = product(B, H, O, p.bbuf[3], up8(O), false, p.wb + p.off[4], H, false, p.buf[5], kEpiReluBack);    // dh2 = dz W3
    g.Y = p.buf[1];
    g.H = p.bbuf[4];
    q.add(g);
    q.add(column_sum(p.buf[3], B, O, up8(O), p.g + p.off[5]));
    q.run(st);
    q.add(product(H, H, B, p.bbuf[4], H, true, p.bbuf[1], H, false, p.g + p.off[2], kEpiStore));             // dW2 = da2^T h1
    g = product(B, H, H, p.bbuf[4], H, false, p.wb + p.off[2], H, false, p.buf[6], kEpiReluBack);            // dh1 = da2 W2
    g.Y = p.buf[0];
    g.H = p.bbuf[5];
    q.add(g);
    q.add(column_sum(p.buf[5], B, H, H, p.g + p.off[3]));
    q.run(st);
    q.add(product(H, I, B, p.bbuf[5], H, true, p.bbuf[0], up8(I), false, p.g + p.off[0], kEpiStore));             // dW1 = da1^T x
    q.add(column_sum(p.buf[6], B, H, H, p.g + p.off[1]));
    q.run(st);
}

cudaError_t proposal_forward(ProposalDev &p, const float *X, int n, float *Z, cudaStream_t st)
{
    if (p.tc.ok) {
        // tensor cores: BF16 operands (features, h1, h2 rounded to BF16 as in training), FP32
        // accumulation, FP32 logits
        for (int s = 0; s < n; s += p.tc.max_rows) {
            const int B = std::min(p.tc.max_rows, n - s);
            cudaError_t e = prop_tc_pack(p.tc, X + (size_t)s * p.n_in, B, st);
            if (e) return e;
            e = prop_tc_forward(p.tc, p.w + p.off[1], p.w + p.off[3], p.w + p.off[5], B, Z + (size_t)s * p.n_out, true,
                                p.n_out, p.tc.err, st);
            if (e) return e;
        }
        return cudaGetLastError();
    }
    for (int s = 0; s < n; s += p.max_batch) {
        const int B = std::min(p.max_batch, n - s);
        forward(p, X + (size_t)s * p.n_in, nullptr, B, st);
        cudaError_t e = cudaMemcpyAsync(Z + (size_t)s * p.n_out, p.buf[2], sizeof(float) * B * p.n_out,
                                        cudaMemcpyDeviceToDevice, st);
        if (e) return e;
    }
    return cudaGetLastError();
}

cudaError_t proposal_grad(ProposalDev &p, const float *X, const float *Y, int n, float *loss, cudaStream_t st)
{
    if (n > p.max_batch) return cudaErrorInvalidValue;
    const int parts = forward(p, X, Y, n, st);
    backward(p, n, st);
    loss_kernel<<<1, 256, 0, st>>>(p.loss_parts, parts, (double)n * p.n_out, p.losses);
    cudaError_t e = cudaMemcpyAsync(loss, p.losses, sizeof(float), cudaMemcpyDeviceToHost, st);
    if (e) return e;
    return cudaStreamSynchronize(st);
}

cudaError_t proposal_train(ProposalDev &p, const float *X, const float *Y, int64_t n, int batch, int steps, float lr,
                           float *losses, cudaStream_t st)
{
    if (batch > p.max_batch || batch < 1 || n < batch) return cudaErrorInvalidValue;
    int64_t cursor = 0;
    int done = 0;                                // losses copied out; the device keeps up to kLossSteps
    for (int it = 0; it < steps; ++it) {
        if (cursor + batch > n) cursor = 0;
        const int parts = forward(p, X + cursor * p.n_in, Y + cursor * p.n_out, batch, st);
        backward(p, batch, st);
        cursor += batch;
        p.step += 1;
        const float b1 = 0.9f, b2 = 0.999f;
        const float c1 = 1.0f - powf(b1, (float)p.step), c2 = 1.0f - powf(b2, (float)p.step);
        adam_kernel<<<blocks_for(p.n_params), 256, 0, st>>>(p.w, p.g, p.m, p.v, p.wb, p.n_params, lr, b1, b2, 1e-8f, c1, c2);
        cudaError_t e = cudaGetLastError();
        if (e) return e;
        if (!losses) continue;
        loss_kernel<<<1, 256, 0, st>>>(p.loss_parts, parts, (double)batch * p.n_out, p.losses + (it - done));
        if (it + 1 - done == kLossSteps || it + 1 == steps) {
            e = cudaMemcpyAsync(losses + done, p.losses, sizeof(float) * (it + 1 - done), cudaMemcpyDeviceToHost, st);
            if (e) return e;
            if ((e = cudaStreamSynchronize(st))) return e;
            done = it + 1;
        }
    }
    proposal_sync_copies(p, st);
    return cudaGetLastError();
}

}  // namespace am
