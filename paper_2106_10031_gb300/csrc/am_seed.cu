// am_seed.cu -- trigger cells by dichotomy along rays (Alg. 1 step 2; Sec. 4.3.2), with the
// sphere-tracing walk (Sec. 4.3.1) and the random-pair sampling (Sec. 4.3.2) in front of it.
//
// One thread block per ray.  F and the state pattern (Def. 2) come from a block-parallel
// FP64 forward pass (Eq. 1).  The bracket [t_lo, t_hi] keeps F of opposite signs at its
// ends and is halved until both ends share one activation pattern; inside that cell F is
// affine along the ray, so the root is t* = t_lo + F_lo / (F_lo - F_hi) (t_hi - t_lo).
// A second kernel pushes each new seed cell into the active set (hash table + arena).
#include <algorithm>

#include "am_block.cuh"
#include "am_kernels.h"

namespace am {

constexpr int kSeedThreads = 256;

__host__ __device__ inline int seed_smem_bytes(int max_n, int max_w)
{
    (void)max_w;
    const int words = (max_n + 31) / 32;
    return max_n * (int)sizeof(double) + 3 * words * (int)sizeof(unsigned) + 16 + 64 * (int)sizeof(double);
}

// Forward pass at x: F (returned to every thread) and the pattern bits in `bits`.  H holds every
// hidden layer's output (N values, layer l at row0[l]), which the residual shortcuts read.
__device__ double seed_forward(const NetDev &net, const double *x, double *H, unsigned *bits, double *red)
{
    const int tid = threadIdx.x, T = blockDim.x;
    for (int w = tid; w < (net.N + 31) / 32; w += T) bits[w] = 0u;
    __syncthreads();
    for (int l = 1; l <= net.L; ++l) {
        const int nl = net.width[l], np = l > 1 ? net.width[l - 1] : 0, rl = net.row0[l];
        const double *Cl = net.Cl[l], *AT = net.AT[l];
        const double *hp = l > 1 ? H + net.row0[l - 1] : nullptr;
        const int src = net.sc_src[l];
        const double *hs = src > 0 ? H + net.row0[src] : nullptr, *S = net.sc_S[l];
        const int ns = src > 0 ? net.width[src] : 0;
        for (int k = tid; k < nl; k += T) {
            double a = Cl[k * 4 + 0] * x[0] + Cl[k * 4 + 1] * x[1] + Cl[k * 4 + 2] * x[2] + Cl[k * 4 + 3];
            for (int j = 0; j < np; ++j) {
                const double hj = hp[j];
                if (hj != 0.0) a += AT[(size_t)j * nl + k] * hj;
            }
            if (hs) {                                          // the residual shortcut S_l h_src
                if (S) for (int j = 0; j < ns; ++j) a += S[(size_t)k * ns + j] * hs[j];
                else a += hs[k];
            }
            H[rl + k] = a > 0.0 ? a : net.slope * a;         // ReLU, or leaky with slope != 0
            if (a > 0.0) atomicOr(bits + ((rl + k) >> 5), 1u << ((rl + k) & 31));
        }
        __syncthreads();
    }
    const double *hL = H + net.row0[net.L];
    const int nL = net.width[net.L];
    if (net.M >= 2) {
        // final max pooling (Sec. 5.2): F = max_i F_i, the pooled index j = the first maximum,
        // as its one-hot key bit n_units + j
        double F = 0.0;
        int j = 0;
        for (int i = 0; i < net.M; ++i) {
            const double *wh = net.w_heads + (size_t)i * nL;
            double f = 0.0;
            for (int k = tid; k < nL; k += T) f += wh[k] * hL[k];
            f = warp_sum(f);
            if ((tid & 31) == 0) red[tid >> 5] = f;
            __syncthreads();
            double Fi = net.b_heads[i];
            for (int w = 0; w < T / 32; ++w) Fi += red[w];
            __syncthreads();
            if (i == 0 || Fi > F) { F = Fi; j = i; }
        }
        if (tid == 0) atomicOr(bits + ((net.n_units + j) >> 5), 1u << ((net.n_units + j) & 31));
        __syncthreads();
        return F;
    }
    double f = 0.0;
    for (int k = tid; k < nL; k += T) f += net.w_out[k] * hL[k];
    f = warp_sum(f);
    if ((tid & 31) == 0) red[tid >> 5] = f;
    __syncthreads();
    double F = net.b_out;
    for (int w = 0; w < T / 32; ++w) F += red[w];
    __syncthreads();
    return F;
}

__global__ void __launch_bounds__(kSeedThreads) seed_kernel(SeedArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const NetDev &net = a.nets[a.net];
    const int words = (net.N + 31) / 32;
    double *H = (double *)smem;
    unsigned *blo = (unsigned *)(H + a.max_n), *bhi = blo + (a.max_n + 31) / 32, *bm = bhi + (a.max_n + 31) / 32;
    double *red = (double *)(((uintptr_t)(bm + (a.max_n + 31) / 32) + 15) & ~(uintptr_t)15);
    const int ray = blockIdx.x, tid = threadIdx.x;
    const double o[3] = {a.origins[ray * 3], a.origins[ray * 3 + 1], a.origins[ray * 3 + 2]};
    const double d[3] = {a.dirs[ray * 3], a.dirs[ray * 3 + 1], a.dirs[ray * 3 + 2]};
    double x[3];

    double tlo = 0.0, thi = a.R;
    for (int c = 0; c < 3; ++c) x[c] = o[c];
    double flo = seed_forward(net, x, H, blo, red);
    for (int c = 0; c < 3; ++c) x[c] = o[c] + a.R * d[c];
    double fhi = seed_forward(net, x, H, bhi, red);
    int rc = 1;
    if (!((flo < 0.0 && fhi > 0.0) || (flo > 0.0 && fhi < 0.0))) rc = -4;
    int it = 0;
    while (rc == 1) {
        int diff = 0;
        for (int w = tid; w < words; w += blockDim.x) diff |= (blo[w] != bhi[w]);
        diff = __syncthreads_or(diff);
        if (!diff) break;
        if (it >= a.max_halvings) { rc = -5; break; }
        const double tm = 0.5 * (tlo + thi);
        for (int c = 0; c < 3; ++c) x[c] = o[c] + tm * d[c];
        const double fm = seed_forward(net, x, H, bm, red);
        if ((fm < 0.0) == (flo < 0.0) && fm != 0.0) {
            tlo = tm; flo = fm;
            for (int w = tid; w < words; w += blockDim.x) blo[w] = bm[w];
        } else {
            thi = tm; fhi = fm;
            for (int w = tid; w < words; w += blockDim.x) bhi[w] = bm[w];
        }
        __syncthreads();
        ++it;
    }
    if (tid == 0) a.seed_ok[ray] = rc;
    if (rc == 1) {
        const double ts = tlo + flo / (flo - fhi) * (thi - tlo);
        if (tid < 3) a.seed_x[ray * 3 + tid] = o[tid] + ts * d[tid];
        for (int w = tid; w < a.ar.kw; w += blockDim.x) {
            const unsigned lo = 2 * w < words ? blo[2 * w] : 0u;
            const unsigned hi = 2 * w + 1 < words ? blo[2 * w + 1] : 0u;
            a.seed_keys[(size_t)ray * a.ar.kw + w] = (unsigned long long)lo | ((unsigned long long)hi << 32);
        }
    } else if (tid == 0) {
        atomicOr(a.ar.counters + kStatus, rc == -4 ? kStSeedNoSign : kStSeedNoCell);
    }
}

// Push the seed cells: allocate an id, write the key, then claim the hash slot with the
// ref (id, no flip).  A ray landing in an already known cell marks its id dead (-2).  One warp per ray: the
// hash is an exclusive or over the key's bits, a word per lane, and lane 0 does the rest (1024 seeds of a
// 3-[256]x8-1 net take 23 us, with a thread per ray 172).
__global__ void seed_insert_kernel(SeedArgs a)
{
    const int ray = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (ray >= a.n_rays || a.seed_ok[ray] != 1) return;
    const Arena &ar = a.ar;
    const NetDev &net = a.nets[a.net];
    const unsigned long long *k = a.seed_keys + (size_t)ray * ar.kw;
    unsigned long long h = 0ull;
    for (int w = lane; w < ar.kw; w += 32) {
        unsigned long long x = k[w];
        while (x) {
            const int b = __ffsll((long long)x) - 1;
            h ^= ar.zob[w * 64 + b];
            x &= x - 1;
        }
    }
    for (int o = 16; o > 0; o >>= 1) h ^= __shfl_xor_sync(0xffffffffu, h, o);
    h ^= net.salt;
    long long id = 0;
    if (lane == 0) id = (long long)atomicAdd(ar.counters + kNCells, 1ull);
    id = __shfl_sync(0xffffffffu, id, 0);
    if (id >= ar.cap) {
        if (lane == 0) atomicOr(ar.counters + kStatus, kStCellCap);
        return;
    }
    for (int w = lane; w < ar.kw; w += 32) ar.keys[id * ar.kw + w] = k[w];
    __threadfence();
    __syncwarp();
    if (lane != 0) return;
    ar.net[id] = a.net;
    ar.hash[id] = h;
    ar.nverts[id] = -1;
    ar.entry_plane[id] = -1;
    ar.parent[id] = -1;
    for (int c = 0; c < 3; ++c) ar.entry_pt[id * 3 + c] = (float)a.seed_x[ray * 3 + c];
    __threadfence();
    const unsigned long long mine = slot_make(h, (unsigned long long)id, kNoFlip);
    unsigned long long pos = h & ar.slot_mask;
    for (int probe = 0; probe < kMaxProbe; ++probe) {
        unsigned long long cur = atomicCAS(ar.slots + pos, 0ull, mine);
        if (cur == 0ull) {
            atomicAdd(a.n_new, 1ull);
            atomicExch(ar.ready + id, 1u);
            return;
        }
        if (slot_tag(cur) == hash_tag(h) && __ldcg(ar.net + slot_parent(cur)) == a.net &&
            ref_keys_equal(ar, id, kNoFlip, slot_parent(cur), slot_flip(cur))) {
            ar.nverts[id] = -2;
            atomicExch(ar.ready + id, 1u);
            return;
        }
        pos = (pos + 1) & ar.slot_mask;
    }
    ar.nverts[id] = -2;
    atomicExch(ar.ready + id, 1u);
    atomicOr(ar.counters + kStatus, kStHashFull);
}

// ---- customised triggers (Sec. 4.3)

// grad F at the point whose pattern the last seed_forward left in `bits`, by backpropagation
// through the units: E[r] = dF/dh_r accumulates from every layer that reads unit r (the next
// layer through W_{l+1}^T, and a residual shortcut through S_q^T), then D_r = g'(a_r) E[r] = dF/da_r
// with g' = 1 on active units and the slope (0 for a ReLU) on the others, and
// grad F = sum_l Cl_l[:, 0:3]^T D_l (the layers fed by x, shortcuts from x included).
// E: N doubles (overwrites the forward pass's H); red: 64 doubles.  Every thread returns g.
__device__ void seed_grad(const NetDev &net, const unsigned *bits, double *E, double *red, double g[3])
{
    const int tid = threadIdx.x, T = blockDim.x;
    double gx = 0.0, gy = 0.0, gz = 0.0;
    const int rL = net.row0[net.L], nU = net.M >= 2 ? net.n_units : net.N;
    const double *wo = net.w_out;                   // a pooled net: the head of the pooled index
    if (net.M >= 2)
        for (int i = 0; i < net.M; ++i)
            if ((bits[(nU + i) >> 5] >> ((nU + i) & 31)) & 1u) { wo = net.w_heads + (size_t)i * net.width[net.L]; break; }
    for (int r = tid; r < nU; r += T) E[r] = r >= rL ? wo[r - rL] : 0.0;
    __syncthreads();
    for (int l = net.L; l >= 1; --l) {
        const int nl = net.width[l], rl = net.row0[l];
        const double *Cl = net.Cl[l];
        for (int k = tid; k < nl; k += T) {
            const double gp = (bits[(rl + k) >> 5] >> ((rl + k) & 31)) & 1u ? 1.0 : net.slope;
            const double dk = gp * E[rl + k];
            E[rl + k] = dk;
            gx += Cl[k * 4 + 0] * dk;
            gy += Cl[k * 4 + 1] * dk;
            gz += Cl[k * 4 + 2] * dk;
        }
        __syncthreads();
        if (l > 1) {
            const int np = net.width[l - 1], rp = net.row0[l - 1];
            const double *AT = net.AT[l];
            for (int j = tid; j < np; j += T) {
                double acc = 0.0;
                for (int k = 0; k < nl; ++k) acc += AT[(size_t)j * nl + k] * E[rl + k];
                E[rp + j] += acc;
            }
            __syncthreads();
        }
        const int src = net.sc_src[l];
        if (src > 0) {
            const int ns = net.width[src], rs = net.row0[src];
            const double *S = net.sc_S[l];
            for (int j = tid; j < ns; j += T) {
                double acc = 0.0;
                if (S) for (int k = 0; k < nl; ++k) acc += S[(size_t)k * ns + j] * E[rl + k];
                else acc = E[rl + j];
                E[rs + j] += acc;
            }
            __syncthreads();
        }
    }
    gx = warp_sum(gx); gy = warp_sum(gy); gz = warp_sum(gz);
    if ((tid & 31) == 0) { red[(tid >> 5) * 3 + 0] = gx; red[(tid >> 5) * 3 + 1] = gy; red[(tid >> 5) * 3 + 2] = gz; }
    __syncthreads();
    g[0] = g[1] = g[2] = 0.0;
    for (int w = 0; w < T / 32; ++w) { g[0] += red[w * 3]; g[1] += red[w * 3 + 1]; g[2] += red[w * 3 + 2]; }
    __syncthreads();
}

// Sphere tracing (Sec. 4.3.1), one block per start point: x <- x - eta F(x) grad F(x) until
// |F| <= eps or max_steps steps, then the bracket along the unit gradient n through the last
// point: o = x - h n, d = 2h n with h = 2|F|/|grad F| + pad, bisected over t in [0, 1] by
// seed_kernel.  A cell with grad F = 0 leaves d = 0, which seed_kernel reports as a ray
// without a sign change.
__global__ void __launch_bounds__(kSeedThreads) trace_kernel(TraceArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const NetDev &net = a.nets[a.net];
    double *H = (double *)smem;
    unsigned *bits = (unsigned *)(H + a.max_n);
    double *red = (double *)(((uintptr_t)(bits + 3 * ((a.max_n + 31) / 32)) + 15) & ~(uintptr_t)15);
    const int i = blockIdx.x, tid = threadIdx.x;
    double x[3] = {a.starts[i * 3], a.starts[i * 3 + 1], a.starts[i * 3 + 2]};
    double F = 0.0, g[3] = {0.0, 0.0, 0.0};
    bool flat = false;
    for (int t = 0;; ++t) {
        F = seed_forward(net, x, H, bits, red);
        seed_grad(net, bits, H, red, g);
        if (fabs(F) <= a.eps || t >= a.max_steps) break;
        if (g[0] == 0.0 && g[1] == 0.0 && g[2] == 0.0) { flat = true; break; }
        for (int c = 0; c < 3; ++c) x[c] = x[c] - a.eta * F * g[c];
    }
    if (tid == 0) {
        if (flat) {
            for (int c = 0; c < 3; ++c) { a.origins[i * 3 + c] = x[c]; a.dirs[i * 3 + c] = 0.0; }
        } else {
            const double gn = sqrt(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
            const double h = 2.0 * fabs(F) / gn + a.pad;
            for (int c = 0; c < 3; ++c) {
                const double n = g[c] / gn;
                a.origins[i * 3 + c] = x[c] - h * n;
                a.dirs[i * 3 + c] = (2.0 * h) * n;
            }
        }
    }
}

// ------------------------------------------------------------------------------------------
// The same forward pass in double-float arithmetic, up to kDfPts points per block, for nets without
// hidden shortcuts, pooling or leaky units: the pairs (hi, lo) of FP32 words carry about 44 bits
// (the product of two pairs split exactly by an FMA, sums by TwoSum), so F and the pattern bits
// agree with an FP64 evaluation wherever they are not within ~1e-12 of zero.  The arithmetic runs on the
// FP32 pipes (this part's FP64 pipe is 1/64 of them), 12 instructions per product, which bound it.
//
// A warp takes one point and 32 units, and only that point's active inputs (about half of them: the
// others are zero, and a product with zero changes no bit of the sum), from a list of (hi, lo, offset of
// the weights) in shared memory; warps of the block's other points run beside it on the same 32 units and
// find the weights in the L1.  With eight points per thread, all inputs and 8 warps per SM, the 16384
// samples of a 3-[256]x8-1 net took 3.99 ms and the dichotomy of its 1024 segments 8.64; 3.09 and 3.48 now.

constexpr int kDfPts = 4;                  // points per block, at most
constexpr int kDfThreads = 512;            // threads per block, at most
constexpr int kDfSums = kSeedThreads / 32; // partial sums of F: units 32 v + lane + kSeedThreads i in sum v

__host__ __device__ inline int df_seed_smem_bytes(int max_n, int max_w)
{
    const int words = (max_n + 31) / 32, chunks = (max_w + 31) / 32;
    return kDfPts * (max_w + 8) * (int)sizeof(float4)            // active inputs
           + kDfPts * max_w * (int)sizeof(float2)                // a layer's outputs
           + kDfPts * (chunks + 1) * (int)sizeof(unsigned)       // its active units, and the list's length
           + 3 * kDfPts * words * (int)sizeof(unsigned)          // patterns: the bracket's ends, the midpoint
           + kDfPts * 8 * (int)sizeof(float)                     // the points as pairs
           + kDfPts * kDfSums * (int)sizeof(float2)              // partial sums of F
           + kDfPts * (int)sizeof(double) + 64;
}

struct DfSm {
    float4 *list;               // point p at [p (max_w + 8)]: active inputs (hi, lo, offset of their weights)
    float2 *z;                  // point p at [p max_w]: the last layer's outputs, zero where inactive
    float2 *red;
    unsigned *on;               // point p at [p chunks]: the layer's active units
    int *cnt;                   // entries of p's list, a multiple of eight
    unsigned *blo, *bhi, *bm;   // patterns, point p at [p words]
    float *xp;                  // point p: [xh, yh, zh, xl, yl, zl] at [8 p]
    double *F;
    int max_w, chunks;
};

__device__ inline DfSm df_carve(unsigned char *base, int max_n, int max_w)
{
    const int words = (max_n + 31) / 32;
    DfSm s;
    s.max_w = max_w;
    s.chunks = (max_w + 31) / 32;
    s.list = reinterpret_cast<float4 *>(base);
    s.z = reinterpret_cast<float2 *>(s.list + kDfPts * (max_w + 8));
    s.red = s.z + kDfPts * max_w;
    unsigned *u = reinterpret_cast<unsigned *>(s.red + kDfPts * kDfSums);
    s.on = u;
    s.cnt = reinterpret_cast<int *>(u + kDfPts * s.chunks);
    u += kDfPts * (s.chunks + 1);
    s.blo = u;
    s.bhi = u + kDfPts * words;
    s.bm = u + 2 * kDfPts * words;
    s.xp = reinterpret_cast<float *>(u + 3 * kDfPts * words);
    s.F = reinterpret_cast<double *>(((uintptr_t)(s.xp + 8 * kDfPts) + 15) & ~(uintptr_t)15);
    return s;
}

// (sh, sl) += (ah + al)(zh + zl): TwoProd of the hi words by FMA, the cross terms into the
// error, TwoSum into the sum
__device__ __forceinline__ void dfs_fma(float &sh, float &sl, float ah, float al, float zh, float zl)
{
    const float p = __fmul_rn(ah, zh);
    float pe = __fmaf_rn(ah, zh, -p);
    pe = __fmaf_rn(ah, zl, pe);
    pe = __fmaf_rn(al, zh, pe);
    const float t = __fadd_rn(sh, p);
    const float bp = __fsub_rn(t, sh);
    const float te = __fadd_rn(__fsub_rn(sh, __fsub_rn(t, bp)), __fsub_rn(p, bp));
    sh = t;
    sl = __fadd_rn(sl, __fadd_rn(te, pe));
}

__device__ __forceinline__ void dfs_add(float &sh, float &sl, float bh, float bl)
{
    const float t = __fadd_rn(sh, bh);
    const float bp = __fsub_rn(t, sh);
    const float te = __fadd_rn(__fsub_rn(sh, __fsub_rn(t, bp)), __fsub_rn(bh, bp));
    sh = t;
    sl = __fadd_rn(sl, __fadd_rn(te, bl));
}

// point p of the block at x (thread p): its coordinates as pairs
__device__ __forceinline__ void df_set_point(const DfSm &s, int p, const double *x)
{
    for (int c = 0; c < 3; ++c) {
        const float h = (float)x[c];
        s.xp[8 * p + c] = h;
        s.xp[8 * p + 3 + c] = (float)(x[c] - (double)h);
    }
}

// Layer l of the block's first n points, U units a lane: 32 U units and one point per warp at a time.
template <int U>
__device__ __forceinline__ void df_layer(const NetDev &net, const DfSm &s, unsigned *bits, int n, int l)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int words = (net.N + 31) / 32, nl = net.width[l], rl = net.row0[l], chunks = (nl + 32 * U - 1) / (32 * U);
    const float *Ch = net.Clhi[l], *Cc = net.Cllo[l];
#pragma unroll 1
    for (int item = wid; item < n * chunks; item += warps) {
        const int p = item % n, k0 = item / n * (32 * U);
        float sh[U], sl[U];
        const float *Ah[U], *Al[U];
#pragma unroll
        for (int e = 0; e < U; ++e) {
            const int k = min(k0 + 32 * e + lane, nl - 1);
            Ah[e] = l > 1 ? net.AThi[l] + k : nullptr;
            Al[e] = l > 1 ? net.ATlo[l] + k : nullptr;
            sh[e] = Ch[4 * k + 3];
            sl[e] = Cc[4 * k + 3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {                // the input columns (layer 1, and skip layers)
                const float wh = Ch[4 * k + c], wl = Cc[4 * k + c];
                if (wh == 0.0f && wl == 0.0f) continue;
                dfs_fma(sh[e], sl[e], wh, wl, s.xp[8 * p + c], s.xp[8 * p + 3 + c]);
            }
        }
        const int m = l > 1 ? s.cnt[p] : 0;
        if (m > 0) {
            // B inputs at a time, the next B's weights on their way (the lists end on a multiple of 8)
            constexpr int B = 4 / U;
            const float4 *in = s.list + p * (s.max_w + 8);
            struct Ahead { float2 z[B]; float h[B][U], lo[B][U]; } a, b;
            auto fetch = [&](Ahead &q, int t) {
#pragma unroll
                for (int u = 0; u < B; ++u) {
                    const float4 v = in[t + u];
                    q.z[u] = make_float2(v.x, v.y);
#pragma unroll
                    for (int e = 0; e < U; ++e) {
                        q.h[u][e] = __ldg(Ah[e] + __float_as_int(v.z));
                        q.lo[u][e] = __ldg(Al[e] + __float_as_int(v.z));
                    }
                }
            };
            auto multiply = [&](const Ahead &q) {
#pragma unroll
                for (int u = 0; u < B; ++u)
#pragma unroll
                    for (int e = 0; e < U; ++e) dfs_fma(sh[e], sl[e], q.h[u][e], q.lo[u][e], q.z[u].x, q.z[u].y);
            };
            fetch(a, 0);
#pragma unroll 1
            for (int t = 0; t < m; t += 2 * B) {
                fetch(b, t + B);
                multiply(a);
                if (t + 2 * B < m) fetch(a, t + 2 * B);
                multiply(b);
            }
        }
#pragma unroll
        for (int e = 0; e < U; ++e) {
            const int k = k0 + 32 * e + lane;
            const float t = __fadd_rn(sh[e], sl[e]);       // renormalise: sign(pair) = sign(hi)
            const float lo = __fsub_rn(sl[e], __fsub_rn(t, sh[e]));
            const bool act = k < nl && t > 0.0f;
            if (k < nl) s.z[p * s.max_w + k] = act ? make_float2(t, lo) : make_float2(0.0f, 0.0f);
            const unsigned b = __ballot_sync(0xffffffffu, act);
            if (lane == 0 && k < nl) {
                s.on[p * s.chunks + (k >> 5)] = b;
                const int bit = rl + k, sft = bit & 31;
                unsigned *o = bits + p * words + (bit >> 5);
                if (b << sft) atomicOr(o, b << sft);
                if (sft && (b >> (32 - sft))) atomicOr(o + 1, b >> (32 - sft));
            }
        }
    }
}

// F at the block's first n (1 to kDfPts) points (s.xp, set by the caller) into s.F, and their patterns
// (Def. 2) into bits[p words].  Every thread calls it.
__device__ void df_forward(const NetDev &net, const DfSm &s, unsigned *bits, int n)
{
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, wid = tid >> 5, warps = T >> 5;
    const int words = (net.N + 31) / 32, L = net.L;
    const bool all = !net.df_finite;               // a product of a zero with a weight out of range is no zero
    for (int w = tid; w < n * words; w += T) bits[w] = 0u;
    __syncthreads();
#pragma unroll 1
    for (int l = 1; l <= L; ++l) {
        // two units a lane share the point's input and most of the address arithmetic (16 instructions per
        // product against 20: 3.27 ms for the samples above with one unit), when that leaves three quarters of the warps one item at least
        const int nl = net.width[l], chunks = (nl + 31) >> 5;
        if (nl > 32 && n * ((nl + 63) >> 6) >= 3 * (warps >> 2)) df_layer<2>(net, s, bits, n, l);
        else df_layer<1>(net, s, bits, n, l);
        __syncthreads();
        if (l == L) break;
        // the active outputs, in order, as the next layer's inputs
        const int n2 = net.width[l + 1];
        for (int item = wid; item < n * 4; item += warps) {
            const int p = item >> 2, q = item & 3;
            float4 *out = s.list + p * (s.max_w + 8);
            int at = 0;
            for (int c = 0; c < chunks; ++c) {
                unsigned b = s.on[p * s.chunks + c];
                if (all) b = 32 * c + 32 <= nl ? full : (1u << (nl - 32 * c)) - 1u;
                if ((c & 3) == q && ((b >> lane) & 1u)) {
                    const int k = 32 * c + lane;
                    const float2 z = s.z[p * s.max_w + k];
                    out[at + __popc(b & ((1u << lane) - 1u))] = make_float4(z.x, z.y, __int_as_float(k * n2), 0.0f);
                }
                at += __popc(b);
            }
            if (q == 0) {                                  // zeros to a multiple of eight (weights of unit 0)
                const int m = (at + 7) & ~7;
                if (lane < m - at) out[at + lane] = make_float4(0.0f, 0.0f, __int_as_float(0), 0.0f);
                if (lane == 0) s.cnt[p] = m;
            }
        }
        __syncthreads();
    }
    const int nL = net.width[L];
    for (int item = wid; item < n * kDfSums; item += warps) {
        const int p = item / kDfSums, v = item % kDfSums;
        float fh = 0.0f, fl = 0.0f;
        for (int k = 32 * v + lane; k < nL; k += kSeedThreads) {
            const float2 z = s.z[p * s.max_w + k];
            dfs_fma(fh, fl, net.w_out_hi[k], net.w_out_lo[k], z.x, z.y);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float oh = __shfl_xor_sync(full, fh, o), ol = __shfl_xor_sync(full, fl, o);
            dfs_add(fh, fl, oh, ol);
        }
        if (lane == 0) s.red[item] = make_float2(fh, fl);
    }
    __syncthreads();
    if (tid < n) {
        double F = net.b_out;
        for (int v = 0; v < kDfSums; ++v) {
            const float2 f = s.red[tid * kDfSums + v];
            F += (double)f.x + (double)f.y;
        }
        s.F[tid] = F;
    }
    __syncthreads();
}

// Points per block for n of them: one per SM before they share weights.  Threads: a warp for every 32 units
// and point, up to kDfThreads (1024 pairs of a 3-[24]x3-1 net: 334 us, 397 with 512 threads).
static int df_points(int n) { return std::min(kDfPts, std::max(1, (n + 151) / 152)); }
static int df_threads(int width) { return std::min(kDfThreads, 32 * kDfPts * ((width + 31) / 32)); }

// F at every sample point (random-pair trigger, Sec. 4.3.2), a.per_block points per block
__global__ void __launch_bounds__(kDfThreads, 2) sample_eval_df_kernel(PairArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const NetDev &net = a.nets[a.net];
    const DfSm s = df_carve(smem, a.max_n, a.max_w);
    const int i0 = blockIdx.x * a.per_block, P = min(a.per_block, a.n_points - i0);
    if (threadIdx.x < kDfPts) {
        const int i = i0 + (threadIdx.x < P ? threadIdx.x : 0);
        const double x[3] = {a.points[3 * i], a.points[3 * i + 1], a.points[3 * i + 2]};
        df_set_point(s, threadIdx.x, x);
    }
    __syncthreads();
    df_forward(net, s, s.bm, P);
    if (threadIdx.x < P) a.F[i0 + threadIdx.x] = s.F[threadIdx.x];
}

// The dichotomy of seed_kernel for a.per_block rays per block, in double-float: one batched forward
// pass per halving step of the block's rays that still bracket more than one cell, packed into
// the first slots so that a step with fewer rays left evaluates fewer points.
__global__ void __launch_bounds__(kDfThreads, 2) seed_df_kernel(SeedArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double tlo[kDfPts], thi[kDfPts], flo[kDfPts], fhi[kDfPts], tm[kDfPts];
    __shared__ int rc[kDfPts], act[kDfPts], side[kDfPts], slot_ray[kDfPts], n_act;
    const NetDev &net = a.nets[a.net];
    const DfSm s = df_carve(smem, a.max_n, a.max_w);
    const int tid = threadIdx.x, words = (net.N + 31) / 32;
    const int r0 = blockIdx.x * a.per_block, P = min(a.per_block, a.n_rays - r0);
    auto point = [&](int q, int p, double t) {          // slot q: ray p's point at t (rays past P: ray 0)
        const int r = r0 + (p < P ? p : 0);
        const double x[3] = {a.origins[3 * r] + t * a.dirs[3 * r], a.origins[3 * r + 1] + t * a.dirs[3 * r + 1],
                             a.origins[3 * r + 2] + t * a.dirs[3 * r + 2]};
        df_set_point(s, q, x);
    };
    if (tid < kDfPts) { tlo[tid] = 0.0; thi[tid] = a.R; point(tid, tid, 0.0); }
    __syncthreads();
    df_forward(net, s, s.blo, P);
    if (tid < kDfPts) { flo[tid] = s.F[tid]; point(tid, tid, a.R); }
    __syncthreads();
    df_forward(net, s, s.bhi, P);
    if (tid < kDfPts) {
        fhi[tid] = s.F[tid];
        const double f0 = flo[tid], f1 = fhi[tid];
        rc[tid] = tid >= P ? 0 : ((f0 < 0.0 && f1 > 0.0) || (f0 > 0.0 && f1 < 0.0)) ? 1 : -4;
    }
    __syncthreads();
    for (int it = 0;; ++it) {
        if (tid < kDfPts) {
            int diff = 0;
            if (rc[tid] == 1)
                for (int w = 0; w < words; ++w) diff |= s.blo[tid * words + w] != s.bhi[tid * words + w];
            act[tid] = diff;
            side[tid] = 0;
        }
        __syncthreads();
        if (tid == 0) {
            int q = 0;
            for (int p = 0; p < kDfPts; ++p)
                if (act[p]) slot_ray[q++] = p;
            n_act = q;
        }
        __syncthreads();
        const int nact = n_act;
        if (nact == 0) break;
        if (it >= a.max_halvings) {
            if (tid < kDfPts && act[tid]) rc[tid] = -5;
            break;
        }
        if (tid < nact) {
            const int p = slot_ray[tid];
            tm[p] = 0.5 * (tlo[p] + thi[p]);
            point(tid, p, tm[p]);
        }
        __syncthreads();
        df_forward(net, s, s.bm, nact);
        if (tid < nact) {
            const int p = slot_ray[tid];
            const double fm = s.F[tid];
            if ((fm < 0.0) == (flo[p] < 0.0) && fm != 0.0) { tlo[p] = tm[p]; flo[p] = fm; side[p] = 1; }
            else { thi[p] = tm[p]; fhi[p] = fm; side[p] = 2; }
        }
        __syncthreads();
        for (int q = tid; q < nact * words; q += blockDim.x) {
            const int slot = q / words, w = q - slot * words, p = slot_ray[slot];
            if (side[p] == 1) s.blo[p * words + w] = s.bm[q];
            else if (side[p] == 2) s.bhi[p * words + w] = s.bm[q];
        }
        __syncthreads();
    }
    __syncthreads();
    for (int p = 0; p < P; ++p) {
        const int ray = r0 + p;
        if (rc[p] == 1) {
            const double ts = tlo[p] + flo[p] / (flo[p] - fhi[p]) * (thi[p] - tlo[p]);
            if (tid < 3) a.seed_x[ray * 3 + tid] = a.origins[ray * 3 + tid] + ts * a.dirs[ray * 3 + tid];
            for (int w = tid; w < a.ar.kw; w += blockDim.x) {
                const unsigned lo = 2 * w < words ? s.blo[p * words + 2 * w] : 0u;
                const unsigned hi = 2 * w + 1 < words ? s.blo[p * words + 2 * w + 1] : 0u;
                a.seed_keys[(size_t)ray * a.ar.kw + w] = (unsigned long long)lo | ((unsigned long long)hi << 32);
            }
        } else if (tid == 0) {
            atomicOr(a.ar.counters + kStatus, rc[p] == -4 ? kStSeedNoSign : kStSeedNoCell);
        }
        if (tid == 0) a.seed_ok[ray] = rc[p];
    }
}

// F at every sample point (random-pair trigger, Sec. 4.3.2), one block per point.
__global__ void __launch_bounds__(kSeedThreads) sample_eval_kernel(PairArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const NetDev &net = a.nets[a.net];
    double *H = (double *)smem;
    unsigned *bits = (unsigned *)(H + a.max_n);
    double *red = (double *)(((uintptr_t)(bits + 3 * ((a.max_n + 31) / 32)) + 15) & ~(uintptr_t)15);
    const int i = blockIdx.x;
    const double x[3] = {a.points[i * 3], a.points[i * 3 + 1], a.points[i * 3 + 2]};
    const double F = seed_forward(net, x, H, bits, red);
    if (threadIdx.x == 0) a.F[i] = F;
}

// Pair the r-th sample with F < 0 and the r-th sample with F > 0 (sample order) for r below
// min(#neg, #pos, max_pairs) and write segment r: origin x-, direction x+ - x- (t in [0, 1]).
// One block of kPairThreads threads walks the samples in chunks; ranks come from a block
// scan of ballot counts.
constexpr int kPairThreads = 1024;
__global__ void __launch_bounds__(kPairThreads) pair_build_kernel(PairArgs a)
{
    __shared__ int wneg[kPairThreads / 32], wpos[kPairThreads / 32];
    __shared__ int base[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) base[0] = base[1] = 0;
    __syncthreads();
    for (int c0 = 0; c0 < a.n_points; c0 += kPairThreads) {
        if (base[0] >= a.max_pairs && base[1] >= a.max_pairs) break;   // block-uniform
        const int i = c0 + tid;
        const double f = i < a.n_points ? a.F[i] : 0.0;
        const bool neg = i < a.n_points && f < 0.0, pos = i < a.n_points && f > 0.0;
        const unsigned bn = __ballot_sync(0xffffffffu, neg), bp = __ballot_sync(0xffffffffu, pos);
        if (lane == 0) { wneg[warp] = __popc(bn); wpos[warp] = __popc(bp); }
        __syncthreads();
        int rn = base[0] + __popc(bn & ((1u << lane) - 1u)), rp = base[1] + __popc(bp & ((1u << lane) - 1u));
        for (int w = 0; w < warp; ++w) { rn += wneg[w]; rp += wpos[w]; }
        if (neg && rn < a.max_pairs) a.neg_idx[rn] = i;
        if (pos && rp < a.max_pairs) a.pos_idx[rp] = i;
        __syncthreads();
        if (tid == 0) {
            int tn = 0, tp = 0;
            for (int w = 0; w < kPairThreads / 32; ++w) { tn += wneg[w]; tp += wpos[w]; }
            base[0] += tn; base[1] += tp;
        }
        __syncthreads();
    }
    const int n_pairs = min(min(base[0], base[1]), a.max_pairs);
    __syncthreads();   // every neg_idx / pos_idx write of the loop is visible below
    for (int r = tid; r < n_pairs; r += kPairThreads) {
        const int in = a.neg_idx[r], ip = a.pos_idx[r];
        for (int c = 0; c < 3; ++c) {
            const double xm = a.points[in * 3 + c];
            a.origins[r * 3 + c] = xm;
            a.dirs[r * 3 + c] = a.points[ip * 3 + c] - xm;
        }
    }
    if (tid == 0) *a.n_pairs = n_pairs;
}

cudaError_t prepare_seed_kernels(int max_n, int max_w)
{
    const int bytes = seed_smem_bytes(max_n, max_w), dbytes = df_seed_smem_bytes(max_n, max_w);
    const void *plain[3] = {(const void *)seed_kernel, (const void *)trace_kernel, (const void *)sample_eval_kernel};
    const void *df[2] = {(const void *)sample_eval_df_kernel, (const void *)seed_df_kernel};
    cudaError_t e = cudaSuccess;
    for (const void *k : plain)
        if (e == cudaSuccess) e = allow_smem(k, bytes);
    for (const void *k : df)
        if (e == cudaSuccess) e = allow_smem(k, dbytes);
    return e;
}

void launch_trace(const TraceArgs &a, cudaStream_t st)
{
    trace_kernel<<<a.n, kSeedThreads, seed_smem_bytes(a.max_n, a.max_w), st>>>(a);
}

void launch_pairs(const PairArgs &args, cudaStream_t st)
{
    PairArgs a = args;
    a.per_block = df_points(a.n_points);
    if (a.df)
        sample_eval_df_kernel<<<(a.n_points + a.per_block - 1) / a.per_block, df_threads(a.width),
                                df_seed_smem_bytes(a.max_n, a.max_w), st>>>(a);
    else
        sample_eval_kernel<<<a.n_points, kSeedThreads, seed_smem_bytes(a.max_n, a.max_w), st>>>(a);
    pair_build_kernel<<<1, kPairThreads, 0, st>>>(a);
}

void launch_seed(const SeedArgs &args, cudaStream_t st)
{
    SeedArgs a = args;
    a.per_block = df_points(a.n_rays);
    if (a.df)
        seed_df_kernel<<<(a.n_rays + a.per_block - 1) / a.per_block, df_threads(a.width),
                         df_seed_smem_bytes(a.max_n, a.max_w), st>>>(a);
    else
        seed_kernel<<<a.n_rays, kSeedThreads, seed_smem_bytes(a.max_n, a.max_w), st>>>(a);
    seed_insert_kernel<<<(a.n_rays + 3) / 4, 128, 0, st>>>(a);
}

}  // namespace am
