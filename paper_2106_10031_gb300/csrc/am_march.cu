// am_march.cu -- the march: one thread block solves one analytic cell at a time.
//
// Per cell (Alg. 1 steps 4-11):
//   a2 compose : Z_l = W_l diag(s_{l-1}) Z_{l-1} + C_l (Lemma 1, Cor. 1) over the active
//                neurons of the previous layer, then a_F (Eq. 8);
//   a3 rows    : c_k = (1 - 2 s_k) Z_k (Eq. 10) plus the box rows;
//   a4 clip    : the lines in which the rows nearest to a point known to lie on the face (the
//                midpoint of the edge the cell was entered through, or the seed point) and the
//                box's rows meet the face plane a_F [x;1] = 0 (Eq. 12) are cut against each other
//                all at once, and what is left of them closes into the polygon (fast_face); a
//                face this does not settle is cut out of a square around the box section by its
//                32 candidate rows one by one (slow_clip).  Vertices from their planes (Eq. 11);
//   a5 check   : every thread then tests every row at every vertex of that polygon (Alg. 1
//                step 8 for the output); a violated row is cut in and the check repeated, so
//                the result is the clip by all rows whatever the candidates were;
//   a6 emit    : corners and edge planes to the face arena;
//   a7 march   : each edge on a neuron plane flips that neuron (Alg. 1 step 10) and pushes
//                the neighbour through the hash table (step 11).
//
// Two arithmetic modes.  kFP64: everything in FP64, a plane within delta of a vertex counts as
// satisfied (and as a degenerate event), as in the oracle.  kDF (mixed): the compose runs in
// double-float arithmetic on the FP32 pipes (TwoProd/TwoSum, the error-free transformations of
// Ogita, Rump & Oishi, "Accurate sum and dot product", 2005) and carries a rigorous bound on
// each row's error; polygon vertices are solved in FP64; every sign decision of the check is
// certified against the bounds (FP32 first, FP64 for the close calls) and a cell with an
// undecidable test is solved again in kFP64.
//
// Two schedules.  Persistent: a grid of resident blocks takes tickets (cell ids, in order)
// from a counter and waits, with a time limit, for the ticket's cell to be published; it stops
// when every handed-out cell is finished.  Levels: one launch per breadth-first level.
#include <algorithm>
#include <cuda_bf16.h>

#include "am_block.cuh"
#include "am_kernels.h"

namespace am {

// The minimum resident blocks per SM the compiler must allow for (register budget); can be set at
// build time for launch-shape sweeps.
#ifndef AM_MIN_BLOCKS
#define AM_MIN_BLOCKS 2
#endif
constexpr int kT = 256;           // threads per block
constexpr int kNW = kT / 32;      // warps per block
constexpr int kMaxPoly = 64;      // polygon vertices in flight
constexpr int kNear = 32;         // rows clipped by warp 0 before the full check
constexpr int kPicks = kNear / kNW;   // candidates each warp contributes
constexpr int kLines = 64;        // candidate lines of the one-pass polygon: the box's and the nearest rows'
constexpr int kParts = kT / kLines;   // threads that share a line's interval
constexpr int kPartBytes = 40 * kT;   // scratch: the one-pass polygon, the proposal's layers
constexpr int kLinePicks = 10;    // nearest rows a warp contributes at most (all of them when N <= 32)
constexpr int kFastFix = 4;       // rounds of the one-pass polygon before the sequential clip takes the cell
// What a cell's compose reads of its net, kept in shared memory while the block stays on the net: every
// field of the global record costs an L2 round trip per cell (taking a cell from the queue empties
// the L1).  The weights lie at offsets of one FP64 block and of its copy as double-float pairs.
struct NetHot {
    int id;                       // the net (-1: none)
    int L, N, units, M, fp64_only, df_ok, ws;   // ws: weights (FP64 words from C_1 to the end of the hidden layers)
    float b_out_hi, b_out_lo;
    double b_out;
    const double *d;              // C_1, FP64
    const float *h, *l;           // the same as hi and lo words
    int offA[kMaxLayers + 1], offC[kMaxLayers + 1], offw;
    short width[kMaxLayers + 2], row0[kMaxLayers + 2];
};
constexpr int kOHot = 9 * kT * 4;   // its place in the scratch region: past the proposal's layers

static_assert(2 * ((kMaxNeurons + 63) / 64) <= kT, "one thread per 32-bit word of a key");
static_assert(kT % 32 == 0 && kNW <= 32 && kNear % kNW == 0 && kT >= kLines, "block shape");
static_assert(kParts == 4 && 256 + 16 * kLines * 2 + 16 * kLines <= 3328 && 3328 + 32 * 8 <= kOHot && kOHot + sizeof(NetHot) <= kPartBytes,
              "the scratch region");
constexpr int kMaxFix = 8;        // check / fix-up rounds
constexpr int kThreadPushWords = 8;   // keys up to this many 64-bit words are pushed by one thread per edge
constexpr float kU = 5.9604645e-8f;            // 2^-24
constexpr float kTiny = 1e-30f, kHuge = 1e30f;   // |normal|^2 outside of which FP32 does not judge a row
constexpr float kDfLoose = 1e-6f;              // certified row error (as a distance) beyond which kDF gives up
constexpr double kVertexTol = 1e-5;            // largest vertex error bound (relative) kept from kDF

enum { kFP64 = 0, kDF = 1 };

// Optional per-phase cycle counters (build with -DAM_PHASE_TIMERS): thread 0 of each block adds
// the clock64() cycles of each phase of each cell to counters[kPhase0 + phase * kCtrStride].  Every
// thread reads the clock: a read by one thread splits its warp, and what it then costs to run the code
// after it twice was most of what the timers showed.
#ifdef AM_PHASE_TIMERS
#define AM_TICK(t) do { (t) = clock64(); } while (0)
#define AM_PHASE(a, i, t0, t1) do { if (threadIdx.x == 0) atomicAdd((a).ar.counters + kPhase0 + (i) * kCtrStride, \
    (unsigned long long)((t1) - (t0))); } while (0)
#else
#define AM_TICK(t) do { } while (0)
#define AM_PHASE(a, i, t0, t1) do { } while (0)
#endif

// ------------------------------------------------------------------------------------------
// shared-memory layout

// The regions of fixed size come first, at constant offsets; then the key and the rows' arrays,
// sized by the largest loadable net.
constexpr int al16(int x) { return (x + 15) & ~15; }
constexpr int kOSc = 0;                                     // scalars
constexpr int kONear = kOSc + 512;
constexpr int kOPe = kONear + 4 * 4 * kNear;
constexpr int kODvb = kOPe + 2 * kMaxPoly * 4;
constexpr int kOVf = kODvb + kMaxPoly * 4;
constexpr int kOPf = kOVf + kMaxPoly * 4 * 4;
constexpr int kOPv = kOPf + 2 * kMaxPoly * 3 * 4;
constexpr int kOPart = kOPv + 2 * kMaxPoly * 3 * 8;
constexpr int kOMask = kOPart + kPartBytes;
static_assert(kONear % 16 == 0 && kOVf % 16 == 0 && kOPv % 16 == 0 && kOPart % 16 == 0 && kOMask % 16 == 0, "alignment");

__host__ __device__ inline int lay_rows(int max_n) { return kOMask + al16(((max_n + 63) / 64) * 8); }   // whole key words
__host__ __device__ inline int lay_nr(int max_n) { return max_n + kBoxPlanes + kSquarePlanes; }
// rows (32 B each: FP64, or the FP32 hi words, then the lo words), then err, rinv and viol
__host__ __device__ inline int lay_total(int max_n)
{
    return lay_rows(max_n) + lay_nr(max_n) * 32 + 3 * al16(lay_nr(max_n) * 4);
}

int march_smem_bytes(int max_n, int max_w)
{
    (void)max_w;
    return lay_total(max_n);
}

// The proposal's scores use the scratch region below the net's record: 64 features + 2 hidden layers + 2 kT
// partial sums.
int proposal_max_hidden() { return (kOHot / 4 - 64 - 2 * kT) / 2; }

// The tensor-core compose keeps one layer's B fragments (16 bytes per lane per 16 input rows)
// in the low-part row array (16 bytes per row): 32 ceil(n_{l-1} / 16) <= max_n + 10 rows.
bool tc_fits(const int *width, int L, int max_n)
{
    for (int l = 2; l <= L; ++l)
        if (32 * ((width[l - 1] + 15) / 16) > max_n + kBoxPlanes + kSquarePlanes) return false;
    return true;
}

struct Sh {
    NetHot *hot;
    unsigned long long *zb;       // hash words of the ring's planes
    unsigned *mask;
    double *r64;            // FP64 rows [nr][4]
    float *rhi, *rlo;       // DF rows [nr][4] each
    float *err, *rinv;
    int *lst;               // the active units, ascending (the violator array, free during the compose)
    int *lst0;              // lst0[l]: first entry of lst of a unit of layer l (1 .. L), lst0[L + 1] = all
    float *carry;           // kDF compose: e_j + g |row_j|_1 of every row (the rinv array, free until the compose ends)
    float4 *line;           // the face's candidate lines (a, b, c, row id) in the face plane's coordinates
    float4 *seg;            // each line's interval (t0, t1, j0, j1)
    int *ring;              // 4 x kLines ints of the ring's assembly
    float *partf;
    double *partd;
    double (*pv)[kMaxPoly][3];
    int (*pe)[kMaxPoly];
    float (*pf)[kMaxPoly][3];   // kDF: the FP32 polygon of the candidate pass
    float (*vf)[4];             // final vertices in FP32 and max(1, |v|_inf)
    float *dvb;
    int *near_k, *near_w;
    float *near_d, *near_dw;
    int *viol;
    // scalars
    double *aF;             // 4 (FP64 value, or hi+lo of the DF value)
    float *aFhi, *aFlo;     // 4 + 4
    float *eF;              // 1
    int *si;                // 32 ints: 0 m, 1 buf, 2 status, 3 nviol, 4 amb, 5 ndeg, 6 emit, 7 ticket,
                            //          8 near count, 9 fix rounds, 10 a vertex too uncertain
    int *wsum;              // 32 ints
    float *ent;             // the point the cell was entered through
    unsigned long long *hsh;   // the cell's hash
    int *nid;               // and its net
    unsigned long long *blk;   // per-block statistics, flushed once when the block exits:
                               // 0 solved, 1 empty, 2 degenerate, 3 fixups, 4 refined, 5 close calls,
                               // 6 cuts of the sequential clip
};

extern __shared__ __align__(16) unsigned char march_smem[];

// Every function that is not inlined makes its own view: the pointers are then known to lie in shared
// memory, most of them at constant offsets (a view passed by reference lives in local memory, and each
// access through it loads its pointer from there first).
__device__ __forceinline__ Sh make_sh(int max_n)
{
    unsigned char *const base = march_smem;
    const int nr = lay_nr(max_n), o = lay_rows(max_n), n4 = al16(nr * 4);
    Sh s;
    s.mask = (unsigned *)(base + kOMask);
    s.hot = (NetHot *)(base + kOPart + kOHot);
    s.zb = (unsigned long long *)(base + kOPart + 3328);
    s.r64 = (double *)(base + o);
    s.rhi = (float *)(base + o);
    s.rlo = s.rhi + 4 * nr;
    s.err = (float *)(base + o + 32 * nr);
    s.rinv = (float *)(base + o + 32 * nr + n4);
    s.carry = s.rinv;
    s.viol = (int *)(base + o + 32 * nr + 2 * n4);
    s.lst = s.viol;
    s.lst0 = (int *)(base + kOPart);                    // 256 B, then the fast face's scratch
    s.line = (float4 *)(base + kOPart + 256);
    s.seg = s.line + kLines;
    s.ring = (int *)(s.seg + kLines);
    s.partf = (float *)(base + kOPart);
    s.partd = (double *)(base + kOPart);
    s.pv = (double(*)[kMaxPoly][3])(base + kOPv);
    s.pe = (int(*)[kMaxPoly])(base + kOPe);
    s.pf = (float(*)[kMaxPoly][3])(base + kOPf);
    s.vf = (float(*)[4])(base + kOVf);
    s.dvb = (float *)(base + kODvb);
    s.near_k = (int *)(base + kONear);
    s.near_d = (float *)(s.near_k + kNear);
    s.near_w = (int *)(s.near_d + kNear);
    s.near_dw = (float *)(s.near_w + kNear);
    double *sc = (double *)(base + kOSc);
    s.aF = sc;                                   // 4 doubles
    s.aFhi = (float *)(sc + 4);                  // 4 floats
    s.aFlo = s.aFhi + 4;                         // 4 floats
    s.eF = s.aFlo + 4;                           // 1 float (+3 pad)
    s.si = (int *)(s.eF + 4);                    // 32 ints
    s.wsum = s.si + 32;                          // 32 ints
    s.blk = (unsigned long long *)(s.wsum + 32); // 8 x u64
    s.hsh = s.blk + 8;
    s.ent = (float *)(s.hsh + 1);                // 3 floats
    s.nid = (int *)(s.ent + 3);
    return s;
}

// ------------------------------------------------------------------------------------------
// arithmetic helpers

__device__ __forceinline__ bool bit_of(const unsigned *mask, int k) { return (mask[k >> 5] >> (k & 31)) & 1u; }

// s += a * z in double-float: (sh, sl) accumulates, a = ah + al, z = zh + zl.  The product
// ah*zh is split exactly (TwoProd with an FMA), the sum with TwoSum; the small cross terms and
// every error term go to sl.  Explicit _rn intrinsics keep the compiler from fusing them.
__device__ __forceinline__ void df_fma(float &sh, float &sl, float ah, float al, float zh, float zl)
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

// (sh, sl) += (bh, bl) (TwoSum on the high parts)
__device__ __forceinline__ void df_add(float &sh, float &sl, float bh, float bl)
{
    const float t = __fadd_rn(sh, bh);
    const float bp = __fsub_rn(t, sh);
    const float te = __fadd_rn(__fsub_rn(sh, __fsub_rn(t, bp)), __fsub_rn(bh, bp));
    sh = t;
    sl = __fadd_rn(sl, __fadd_rn(te, bl));
}

// renormalise so that |lo| <= ulp(hi) / 2 (Fast2Sum)
__device__ __forceinline__ void df_norm(float &h, float &l)
{
    const float s = __fadd_rn(h, l);
    l = __fsub_rn(l, __fsub_rn(s, h));
    h = s;
}

// gamma-style coefficient of the double-float dot product bound: 2 (m + 4)^2 u^2
__device__ __forceinline__ float df_gamma(int m) { return 2.0f * (float)(m + 4) * (float)(m + 4) * kU * kU; }

// row k as FP64 (both modes; in kDF hi + lo is exact in FP64)
template <int M>
__device__ __forceinline__ void row64(const Sh &s, int k, double *r)
{
    if (M == kFP64) {
        r[0] = s.r64[4 * k]; r[1] = s.r64[4 * k + 1]; r[2] = s.r64[4 * k + 2]; r[3] = s.r64[4 * k + 3];
    } else {
        for (int c = 0; c < 4; ++c) r[c] = (double)s.rhi[4 * k + c] + (double)s.rlo[4 * k + c];
    }
}

// ------------------------------------------------------------------------------------------
// a2 on the tensor cores: hidden layers 2..L of the compose as split-BF16 products

// D (16 x 8, FP32) += A (16 x 16, BF16, row) * B (16 x 8, BF16, col); fragments as in the PTX
// ISA's mma.m16n8k16 layouts (a: 4 x b32, b: 2 x b32, lower element in the lower half)
__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint4 &a, const uint2 &b)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};\n"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y));
}

__device__ __forceinline__ unsigned bf16_bits(float x)
{
    return (unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(x));
}

constexpr int kTcTiles = 4;         // 16-row output tiles a warp accumulates at once

// Z_l = W_l diag(s_{l-1}) Z_{l-1} + C_l for l = 2..L on the tensor cores.  Z_{l-1} (FP32 rows,
// sign-adjusted, in s.rhi; inactive rows zero) is split into three BF16 parts and laid out as
// B1 = [Z_hi | Z_mid] and B2 = [Z_lo | 0] (16 x 8 fragments); W_l comes as three BF16 parts.
// Four MMAs per tile: (W_hi + W_mid + W_lo) B1 + W_hi B2, whose two column halves sum to
// W (Z_hi + Z_mid) + W_hi Z_lo: the dropped products and split residuals are below 2^-26 |W||Z|,
// so the FP32 accumulation dominates.  The B fragments live in s.rlo, unused by this path
// (it is zeroed before return: tensor-core rows have no low part).
// Error estimate per row m (l1 over its 4 coefficients), not a bound:
//   8 (2.8 2^-24 sqrt(T) + 2^-25) max_j |W_mj| sum_c |z_c|_2  +  |W_m|_2 rms(e_{l-1}),  T = 4 Kt
// (random-sign model of the accumulation over T MMAs, each product's share bounded through
// max|W_mj| and the column norm; the previous rows' estimates propagate by root mean square,
// without a new factor, so the safety does not compound with depth).
// Inlined: 4000 patterns of a 3-[512]x8-1 decoder take 4.32 ms, 5.18 with it out of line (the march kernels, which
// never take it, drop it).
__device__ __forceinline__ void compose_tc_layers(const NetDev &net, int max_n, int nr)
{
    const Sh s = make_sh(max_n);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, g = lane >> 2, t4 = lane & 3;
    uint4 *Bf = reinterpret_cast<uint4 *>(s.rlo);   // per (kt, lane): B1 (x, y), B2 (z, w)
    float *red = reinterpret_cast<float *>(s.wsum);   // 0..3: sum z_c^2, 4: sum e^2 (no scans here)
    for (int l = 2; l <= net.L; ++l) {
        const int np = net.width[l - 1], nl = net.width[l], rp = net.row0[l - 1], rl = net.row0[l];
        const int Kt = (np + 15) >> 4, Mt = (nl + 15) >> 4;
        if (tid < 8) red[tid] = 0.0f;
        __syncthreads();
        // B fragments: item (kt, lane') holds rows kt*16 + 2t' + {0, 1, 8, 9} of column g'
        for (int it = tid; it < Kt * 32; it += kT) {
            const int kt = it >> 5, gg = (it & 31) >> 2, tt = it & 3;
            const int c = gg & 3;
            const bool second = gg >= 4;              // columns 4..7: Z_mid in B1, zero in B2
            unsigned v1[4], v2[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int k = kt * 16 + 2 * tt + (q & 1) + (q >> 1) * 8;
                float z = 0.0f;
                if (k < np && bit_of(s.mask, rp + k)) z = -s.rhi[4 * (rp + k) + c];   // active: z = -row
                const float zh = __bfloat162float(__float2bfloat16_rn(z));
                const float zm = __bfloat162float(__float2bfloat16_rn(z - zh));
                v1[q] = bf16_bits(second ? zm : zh);
                v2[q] = second ? 0u : bf16_bits((z - zh) - zm);
            }
            Bf[it] = make_uint4(v1[0] | (v1[1] << 16), v1[2] | (v1[3] << 16), v2[0] | (v2[1] << 16),
                                v2[2] | (v2[3] << 16));
        }
        {
            float z2[4] = {0.0f, 0.0f, 0.0f, 0.0f}, e2 = 0.0f;
            for (int k = tid; k < np; k += kT)
                if (bit_of(s.mask, rp + k)) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) z2[c] = fmaf(s.rhi[4 * (rp + k) + c], s.rhi[4 * (rp + k) + c], z2[c]);
                    e2 = fmaf(s.err[rp + k], s.err[rp + k], e2);
                }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
                for (int c = 0; c < 4; ++c) z2[c] += __shfl_xor_sync(0xffffffffu, z2[c], o);
                e2 += __shfl_xor_sync(0xffffffffu, e2, o);
            }
            if (lane == 0) {
#pragma unroll
                for (int c = 0; c < 4; ++c) atomicAdd(red + c, z2[c]);
                atomicAdd(red + 4, e2);
            }
        }
        __syncthreads();
        const float zn = sqrtf(red[0]) + sqrtf(red[1]) + sqrtf(red[2]) + sqrtf(red[3]);
        const float erms = sqrtf(red[4] / (float)np);
        const float kloc = 8.0f * (2.8f * 5.9604644775390625e-8f * sqrtf((float)(4 * Kt)) + 2.98023223876953125e-8f);
        const uint4 *Wf = net.Wf[l];
        const float *wn = net.wn[l];
        for (int mt0 = wid; mt0 < Mt; mt0 += kNW * kTcTiles) {
            float acc[kTcTiles][4];
#pragma unroll
            for (int i = 0; i < kTcTiles; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.0f;
            for (int kt = 0; kt < Kt; ++kt) {
                const uint4 bb = Bf[kt * 32 + lane];
                const uint2 b1 = make_uint2(bb.x, bb.y), b2 = make_uint2(bb.z, bb.w);
#pragma unroll
                for (int i = 0; i < kTcTiles; ++i) {
                    const int mt = mt0 + i * kNW;
                    if (mt < Mt) {
                        const uint4 *tp = Wf + ((size_t)mt * Kt + kt) * 96;
                        const uint4 ah = __ldg(tp + lane), am = __ldg(tp + 32 + lane), al = __ldg(tp + 64 + lane);
                        mma_bf16_16816(acc[i], ah, b1);
                        mma_bf16_16816(acc[i], am, b1);
                        mma_bf16_16816(acc[i], al, b1);
                        mma_bf16_16816(acc[i], ah, b2);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < kTcTiles; ++i) {
                const int mt = mt0 + i * kNW;
                if (mt >= Mt) continue;                  // warp-uniform
                float o[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) o[q] = acc[i][q] + __shfl_xor_sync(0xffffffffu, acc[i][q], 2);
                if (t4 < 2) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {        // rows g and g + 8
                        const int m = mt * 16 + g + 8 * h;
                        if (m >= nl) continue;
                        const int r = rl + m;
                        const float sg = bit_of(s.mask, r) ? -1.0f : 1.0f;
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            const int c = 2 * t4 + j;
                            const float v = o[2 * h + j] + (net.Clhi[l][4 * m + c] + net.Cllo[l][4 * m + c]);
                            s.rhi[4 * r + c] = sg * v;
                        }
                        if (t4 == 0) s.err[r] = fmaf(kloc * wn[2 * m + 1], zn, wn[2 * m] * erms);
                    }
                }
            }
        }
        __syncthreads();
    }
    for (int i = tid; i < 4 * nr; i += kT) s.rlo[i] = 0.0f;
    __syncthreads();
}

// ------------------------------------------------------------------------------------------
// a2/a3: compose the rows of every neuron of the cell, and a_F

// The block's copy of a net's record; the caller has a barrier on both sides.
__device__ __noinline__ void fill_hot(const NetDev *netp, int id, int max_n)
{
    const Sh s = make_sh(max_n);
    NetHot &h = *s.hot;
    const NetDev &net = *netp;
    const int l = threadIdx.x, L = net.L;
    if (l >= 1 && l <= L) {
        h.width[l] = (short)net.width[l];
        h.row0[l] = (short)net.row0[l];
        h.offA[l] = l > 1 ? (int)(net.AT[l] - net.Cl[1]) : 0;
        h.offC[l] = (int)(net.Cl[l] - net.Cl[1]);
    }
    if (l == 0) {
        h.id = id;
        h.L = L;
        h.N = net.N;
        h.M = net.M;
        h.units = net.M >= 2 ? net.n_units : net.N;
        h.fp64_only = net.fp64_only;
        h.df_ok = net.df_ok;
        h.b_out = net.b_out;
        h.b_out_hi = net.b_out_hi;
        h.b_out_lo = net.b_out_lo;
        h.d = net.Cl[1];
        h.h = net.Clhi[1];
        h.l = net.Cllo[1];
        h.offw = (int)(net.w_out - net.Cl[1]);
        h.ws = h.offw + net.width[L];
    }
}

// Start the net's weights on their way into the L1 (emptied when the cell was taken), one line per thread,
// while the cell's record is read; nets too large for the L1 load theirs as they go.
template <int M>
__device__ __forceinline__ void touch_weights(const NetHot &h)
{
    constexpr int kLine = 128, kMost = 96 * 1024;
    const int bytes = h.ws * (M == kFP64 ? 8 : 4);
    if (bytes > (M == kFP64 ? kMost : kMost / 2)) return;
    unsigned v;
#pragma unroll 1
    for (int i = threadIdx.x * kLine; i < bytes; i += kT * kLine) {
        if (M == kFP64) {
            asm volatile("ld.global.ca.u32 %0, [%1];" : "=r"(v) : "l"(reinterpret_cast<const char *>(h.d) + i));
        } else {
            asm volatile("ld.global.ca.u32 %0, [%1];" : "=r"(v) : "l"(reinterpret_cast<const char *>(h.h) + i));
            asm volatile("ld.global.ca.u32 %0, [%1];" : "=r"(v) : "l"(reinterpret_cast<const char *>(h.l) + i));
        }
    }
}

// -x by the sign bit: this part's FP64 pipe issues a warp instruction in about 64 cycles
__device__ __forceinline__ double flip(double x, bool f)
{
    return __longlong_as_double(__double_as_longlong(x) ^ (f ? (long long)0x8000000000000000ull : 0ll));
}

// The residual shortcut of layer l (Sec. 5.1) for column c of its row k, FP64: sum_j S_kj H_src[j] with
// H_src = diag(g) Z_src (g = 1 on active units, the slope on the others) and the stored row
// (1 - 2 s) Z, so H_src[j] = -row_j when unit j is active and slope * row_j otherwise; S = null
// is the identity (H_src[k]).
__device__ __forceinline__ double add_shortcut(const NetDev &net, const Sh &s, int l, int k, int c, double a)
{
    const int src = net.sc_src[l];
    if (src <= 0) return a;
    const int rs = net.row0[src], ns = net.width[src];
    const double *S = net.sc_S[l];
    const int j0 = S ? 0 : k, j1 = S ? ns : k + 1;
#pragma unroll 1
    for (int j = j0; j < j1; ++j) {
        const double w = S ? __ldg(S + (size_t)k * ns + j) : 1.0;
        const int r = rs + j;
        const double f = w * (bit_of(s.mask, r) ? -1.0 : net.slope);
        if (f == 0.0) continue;
        a += f * s.r64[4 * r + c];
    }
    return a;
}

// The cell's active units in one ascending list (diag(s_l) selects these rows of every layer), with
// the first entry of each layer: every warp scans the mask's words itself (a popcount scan over
// its lanes) and writes the entries of the words it owns, so the whole list takes one barrier,
// the caller's.
__device__ __forceinline__ void active_list(const NetHot &net, const Sh &s)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned full = 0xffffffffu, below = (1u << lane) - 1u;
    const int units = net.units, nw = (units + 31) >> 5, L = net.L;
    int base = 0;
#pragma unroll 1
    for (int c = 0; c < nw; c += 32) {
        unsigned word = c + lane < nw ? s.mask[c + lane] : 0u;
        if (c + lane == units >> 5) word &= (1u << (units & 31)) - 1u;
        const int n = __popc(word);
        int inc = n;
#pragma unroll 1
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(full, inc, o);
            if (lane >= o) inc += y;
        }
        const int exc = base + inc - n;
#pragma unroll 1
        for (int q = wid; q < 32 && c + q < nw; q += kNW) {
            const unsigned wq = __shfl_sync(full, word, q);
            const int eq = __shfl_sync(full, exc, q);
            if ((wq >> lane) & 1u) s.lst[eq + __popc(wq & below)] = 32 * (c + q) + lane;
        }
        if (wid == 0) {
            const int r0 = lane < L ? net.row0[lane + 1] : 0, w = r0 >> 5;      // L <= 32
            const int e = __shfl_sync(full, exc, w & 31);
            const unsigned ww = __shfl_sync(full, word, w & 31);
            if (lane < L && w >= c && w < c + 32) s.lst0[lane + 1] = e + __popc(ww & ((1u << (r0 & 31)) - 1u));
        }
        base += __shfl_sync(full, inc, 31);
    }
    if (threadIdx.x == 0) s.lst0[L + 1] = base;
}

// After the last layer of a max-pooled net
__device__ __noinline__ void pool_rows(const NetDev &net, int max_n)
{
    const Sh s = make_sh(max_n);
    const int tid = threadIdx.x;
    // final max pooling (Sec. 5.2): a_F(i) of every head into row n_units + i, then the face
    // plane a_F(j) of the cell's pooled index j and the pooling rows a_F(i) - a_F(j)
    const int nL = net.width[net.L], rL = net.row0[net.L];
    for (int i = 0; i < net.M; ++i) {
        const double *wh = net.w_heads + (size_t)i * nL;
        double f[4] = {0.0, 0.0, 0.0, 0.0};
        for (int k = tid; k < nL; k += kT) {
            const double w = bit_of(s.mask, rL + k) ? wh[k] : -net.slope * wh[k];
            if (w != 0.0)
                for (int c = 0; c < 4; ++c) f[c] -= w * s.r64[4 * (rL + k) + c];
        }
        for (int c = 0; c < 4; ++c) f[c] = warp_sum(f[c]);
        if ((tid & 31) == 0)
            for (int c = 0; c < 4; ++c) s.partd[4 * (tid >> 5) + c] = f[c];
        __syncthreads();
        if (tid == 0) {
            double F[4] = {0.0, 0.0, 0.0, net.b_heads[i]};
            for (int w = 0; w < kNW; ++w)
                for (int c = 0; c < 4; ++c) F[c] += s.partd[4 * w + c];
            for (int c = 0; c < 4; ++c) s.r64[4 * (net.n_units + i) + c] = F[c];
        }
        __syncthreads();
    }
    if (tid == 0) {
        int j = 0;
        for (int i = 0; i < net.M; ++i)
            if (bit_of(s.mask, net.n_units + i)) { j = i; break; }
        for (int c = 0; c < 4; ++c) {
            s.aF[c] = s.r64[4 * (net.n_units + j) + c];
            s.aFhi[c] = (float)s.aF[c];
        }
        s.eF[0] = 0.0f;
    }
    __syncthreads();
    if (tid < net.M)
        for (int c = 0; c < 4; ++c) s.r64[4 * (net.n_units + tid) + c] -= s.aF[c];
    __syncthreads();
}

// sum over the active units t0 .. t1 of the list of -W_kr row_rc (active: z = -row), FP64: one column c of
// row k.  The next four weights are on their way while four products issue (a warp's four take about
// 300 cycles, an L2 round trip 300 to 600); the bounds are the same for every thread, so products
// past the end are skipped, not issued.
__device__ __forceinline__ double dot_active(const Sh &s, const double *AT, int nl, int rp, int k, int c, int t0, int t1)
{
    double acc = 0.0, w[4] = {0.0, 0.0, 0.0, 0.0};
    AT += k;
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (t0 + u < t1) w[u] = __ldg(AT + (s.lst[t0 + u] - rp) * nl);
#pragma unroll 1
    for (int t = t0; t < t1; t += 4) {
        double wn[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (t + 4 + u < t1) wn[u] = __ldg(AT + (s.lst[t + 4 + u] - rp) * nl);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (t + u < t1) acc -= w[u] * s.r64[4 * s.lst[t + u] + c];
#pragma unroll
        for (int u = 0; u < 4; ++u) w[u] = wn[u];
    }
    return acc;
}

// Rows of every layer in FP64, the nets that compose in FP64 only (leaky units, hidden shortcuts, max
// pooling): one thread per row and column, as compose<kFP64>.  Returns without a barrier after a_F.
__device__ __noinline__ void compose_general(const NetDev &net, int max_n)
{
    const Sh s = make_sh(max_n);
    const int tid = threadIdx.x;
    const bool leaky = net.slope != 0.0;
    active_list(*s.hot, s);
    for (int i = tid; i < 4 * net.width[1]; i += kT) s.r64[i] = flip(net.Cl[1][i], bit_of(s.mask, i >> 2));
    __syncthreads();
    for (int l = 2; l <= net.L; ++l) {
        const int nl = net.width[l], rp = net.row0[l - 1], rl = net.row0[l], np = net.width[l - 1];
        const int t0 = s.lst0[l - 1], t1 = s.lst0[l];
        const double *AT = net.AT[l], *C = net.Cl[l];
        const double sl = net.slope;
        for (int item = tid; item < 4 * nl; item += kT) {
            const int k = item >> 2, c = item & 3;
            double acc = 0.0;
            if (leaky) {
                // every row takes part (diag(s + slope (1 - s))): active: z = -row (weight 1);
                // inactive: z = +row, weight slope
#pragma unroll 4
                for (int j = 0; j < np; ++j) {
                    double w = __ldg(AT + (size_t)j * nl + k);
                    if (!bit_of(s.mask, rp + j)) w *= -sl;
                    acc -= w * s.r64[4 * (rp + j) + c];
                }
            } else {
                acc = dot_active(s, AT, nl, rp, k, c, t0, t1);
            }
            acc = add_shortcut(net, s, l, k, c, acc);
            s.r64[4 * rl + item] = flip(acc + C[item], bit_of(s.mask, rl + k));
        }
        __syncthreads();
    }
    if (net.M >= 2) {
        pool_rows(net, max_n);
        return;
    }
    // a_F = w_out^T diag(s_L) Z_L + [0 | b_out] (Cor. 1, Eq. 8): active: row = -Z (weight 1); inactive:
    // row = +Z, weight slope; warp 0, lane 4 p + c: column c over every 8th unit
    if (tid < 32) {
        const int nL = net.width[net.L], rL = net.row0[net.L], c = tid & 3;
        double f = 0.0;
        for (int k = tid >> 2; k < nL; k += 8) {
            const double w = bit_of(s.mask, rL + k) ? net.w_out[k] : -net.slope * net.w_out[k];
            if (w != 0.0) f -= w * s.r64[4 * (rL + k) + c];
        }
        for (int o = 4; o < 32; o <<= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
        if (c == 3) f += net.b_out;
        if (tid < 4) {
            s.aF[c] = f;
            s.aFhi[c] = (float)f;
        }
        if (tid == 0) s.eF[0] = 0.0f;
    }
}

// kDF: the lanes that share a row's sum, log2.  Layers of at most kNarrow units take one lane per row and
// column (4 n_l S <= kT), wider ones a lane per row (n_l S <= kT, or S = 1 in several passes).
constexpr int kNarrow = kT / 8;
__device__ __forceinline__ int df_split(int nl)
{
    return nl <= 8 ? 3 : nl <= 16 ? 2 : nl <= kNarrow ? 1 : nl <= kT / 4 ? 2 : nl <= kT / 2 ? 1 : 0;
}

// The partial sums of a row that its error bound allows for: a block's threads shared out, whatever
// df_split (never more) takes, so that a bound depends on the net alone.
__device__ __forceinline__ int df_parts(int nl) { return nl >= kT ? 1 : kT / nl; }

// Rows of every layer.  FP64: one thread per row and column (k, c), the four columns of a row in
// neighbouring lanes, so a layer of n rows issues 4 n / 32 chains of its active units and nothing
// else on the FP64 pipe, whose warp instructions take about 64 cycles each whatever the lanes do
// (splitting a narrow layer's sums over the block's warps issued the partial sums' additions on top: a
// 3-12-6-3-2-1 net's compose took 91,700 cycles so, 7,100 now; 1000 patterns of a 3-[44]x5-1 net
// 136 us, 98 now).  Double-float: df_split.  One barrier per layer.  Returns without a barrier after
// a_F, which warp 0 computes.  Two blocks of a 3-[64]x4-1 net keep the FP64 pipe busy through it:
// 24,600 products per cell at the 1.7 the pipe takes per cycle are 14,500 cycles.
template <int M>
__device__ __forceinline__ void compose(const NetDev &netg, const Sh &s, bool tc, int max_n)
{
    const NetHot &net = *s.hot;
    const int nrows = lay_nr(max_n);
    const int tid = threadIdx.x;
    const unsigned full = 0xffffffffu;
    if (M == kFP64 && net.fp64_only) {
        compose_general(netg, max_n);
        return;
    }
    active_list(net, s);
    // layer 1: Z_1 = C_1 (cell independent)
    {
        const int n1 = net.width[1];
        if (M == kFP64) {
#pragma unroll 1
            for (int i = tid; i < 4 * n1; i += kT) s.r64[i] = flip(net.d[i], bit_of(s.mask, i >> 2));
        } else {
            int nact = 0;
#pragma unroll 1
            for (int w = 0; w < n1; w += 32) nact += __popc(s.mask[w >> 5] & (n1 - w < 32 ? (1u << (n1 - w)) - 1u : ~0u));
            const float g = df_gamma(nact + (net.L > 1 ? df_parts(net.width[2]) : 1) + 2);
#pragma unroll 1
            for (int i0 = 0; i0 < 4 * n1; i0 += kT) {
                const int i = i0 + tid, k = i >> 2;
                const bool on = i < 4 * n1;
                const float h = on ? net.h[i] : 0.0f, lo = on ? net.l[i] : 0.0f;
                float l1 = fabsf(h);
                l1 += __shfl_xor_sync(full, l1, 1);
                l1 += __shfl_xor_sync(full, l1, 2);
                if (on) {
                    const float sg = bit_of(s.mask, k) ? -1.0f : 1.0f;
                    s.rhi[i] = sg * h;
                    s.rlo[i] = sg * lo;
                    // representation of C: double-float, or FP32 alone on the tensor-core path
                    const float e = (tc ? kU : 2.0f * kU * kU) * l1 * 1.01f;
                    s.err[k] = e;
                    s.carry[k] = __fmaf_ru(g, l1 * 1.001f, e);
                }
            }
        }
    }
    __syncthreads();
    if (M == kDF && tc) compose_tc_layers(netg, max_n, nrows);
#pragma unroll 1
    for (int l = (M == kDF && tc) ? net.L + 1 : 2; l <= net.L; ++l) {
        const int nl = net.width[l], rp = net.row0[l - 1], rl = net.row0[l];
        const int t0 = s.lst0[l - 1], t1 = s.lst0[l];
        if (M == kFP64) {
            const double *AT = net.d + net.offA[l], *C = net.d + net.offC[l];
            if (nl > kT / 2) {
                // wide layers: a row per thread, whose weight feeds four products (a column per thread would
                // read every weight four times from the L2: 1.16 ms against 1.02 ms for 1000 patterns of a
                // 3-[250]x5-1 net, 1.59 ms against 1.22 ms for 400 of a 3-[500]x4-1 net)
#pragma unroll 1
                for (int k = tid; k < nl; k += kT) {
                    double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
#pragma unroll 4
                    for (int t = t0; t < t1; ++t) {
                        const int r = s.lst[t];
                        const double w = __ldg(AT + (r - rp) * nl + k);
                        const double *z = s.r64 + 4 * r;
                        a0 -= w * z[0]; a1 -= w * z[1]; a2 -= w * z[2]; a3 -= w * z[3];
                    }
                    const bool act = bit_of(s.mask, rl + k);
                    double *r = s.r64 + 4 * (rl + k);
                    r[0] = flip(a0 + C[4 * k], act); r[1] = flip(a1 + C[4 * k + 1], act);
                    r[2] = flip(a2 + C[4 * k + 2], act); r[3] = flip(a3 + C[4 * k + 3], act);
                }
            } else if (tid < 4 * nl) {
                // one column of row k, and of row k + kT / 4 where the warp has one: 4 n_l <= 2 kT
                const int k = tid >> 2, c = tid & 3, k2 = min(k + kT / 4, nl - 1);
                double acc, acc2 = 0.0;
                const double Ci = C[tid];
                if ((tid & ~31) + kT < 4 * nl) {
                    acc = 0.0;
#pragma unroll 4
                    for (int t = t0; t < t1; ++t) {
                        const int r = s.lst[t];
                        const double *w = AT + (r - rp) * nl;
                        const double z = s.r64[4 * r + c];          // active: z = -row
                        acc -= __ldg(w + k) * z;
                        acc2 -= __ldg(w + k2) * z;
                    }
                    if (k + kT / 4 < nl) s.r64[4 * (rl + k2) + c] = flip(acc2 + C[4 * k2 + c], bit_of(s.mask, rl + k2));
                } else {
                    acc = dot_active(s, AT, nl, rp, k, c, t0, t1);
                }
                s.r64[4 * rl + tid] = flip(acc + Ci, bit_of(s.mask, rl + k));
            }
        } else {
            const float *Ah = net.h + net.offA[l], *Al = net.l + net.offA[l];
            const int sh = df_split(nl), S = 1 << sh;
            const float g = df_gamma(t1 - t0 + df_parts(nl) + 2);
            const float gn = l < net.L ? df_gamma(s.lst0[l + 1] - t1 + df_parts(net.width[l + 1]) + 2) : 0.0f;
            if (nl <= kNarrow) {
                // one lane per row, column and part of the sum, in one pass of the block
                const int sp = tid & (S - 1), c = (tid >> sh) & 3, k = tid >> (sh + 2);
                const bool on = k < nl;
                const float ch = on ? net.h[net.offC[l] + 4 * k + c] : 0.0f, cl = on ? net.l[net.offC[l] + 4 * k + c] : 0.0f;
                float h = 0.0f, lo = 0.0f, eb = 0.0f;
                if (on) {
#pragma unroll 2
                    for (int t = t0 + sp; t < t1; t += S) {
                        const int r = s.lst[t];
                        const float ah = __ldg(Ah + (r - rp) * nl + k), al = __ldg(Al + (r - rp) * nl + k);
                        df_fma(h, lo, ah, al, -s.rhi[4 * r + c], -s.rlo[4 * r + c]);      // z = -row
                        eb = __fmaf_ru(fabsf(ah), s.carry[r], eb);
                    }
                }
#pragma unroll 1
                for (int o = 1; o < S; o <<= 1) {
                    const float oh = __shfl_xor_sync(full, h, o), ol = __shfl_xor_sync(full, lo, o);
                    df_add(h, lo, oh, ol);
                    eb = __fadd_ru(eb, __shfl_xor_sync(full, eb, o));
                }
                df_add(h, lo, ch, cl);
                df_norm(h, lo);
                float l1 = fabsf(h), cl1 = fabsf(ch);
#pragma unroll 1
                for (int o = S; o < 4 * S; o <<= 1) {
                    l1 += __shfl_xor_sync(full, l1, o);
                    cl1 += __shfl_xor_sync(full, cl1, o);
                }
                if (on && sp == 0) {
                    const float sg = bit_of(s.mask, rl + k) ? -1.0f : 1.0f;
                    s.rhi[4 * (rl + k) + c] = sg * h;
                    s.rlo[4 * (rl + k) + c] = sg * lo;
                    const float e = __fmaf_ru(g, cl1, eb) * 1.01f;
                    s.err[rl + k] = e;
                    s.carry[rl + k] = __fmaf_ru(gn, l1 * 1.001f, e);
                }
            } else {
                // S lanes per row
#pragma unroll 1
                for (int i0 = 0; i0 < nl * S; i0 += kT) {
                    const int item = i0 + tid, k = item >> sh, sp = item & (S - 1);
                    float h0 = 0.f, h1 = 0.f, h2 = 0.f, h3 = 0.f, l0 = 0.f, l1 = 0.f, l2 = 0.f, l3 = 0.f, eb = 0.f;
                    if (k < nl) {
#pragma unroll 4
                        for (int t = t0 + sp; t < t1; t += S) {
                            const int r = s.lst[t];
                            const float ah = __ldg(Ah + (r - rp) * nl + k), al = __ldg(Al + (r - rp) * nl + k);
                            const float4 zh = *reinterpret_cast<const float4 *>(s.rhi + 4 * r);      // z = -row
                            const float4 zl = *reinterpret_cast<const float4 *>(s.rlo + 4 * r);
                            df_fma(h0, l0, ah, al, -zh.x, -zl.x);
                            df_fma(h1, l1, ah, al, -zh.y, -zl.y);
                            df_fma(h2, l2, ah, al, -zh.z, -zl.z);
                            df_fma(h3, l3, ah, al, -zh.w, -zl.w);
                            eb = __fmaf_ru(fabsf(ah), s.carry[r], eb);
                        }
                    }
#pragma unroll 1
                    for (int o = 1; o < S; o <<= 1) {
                        df_add(h0, l0, __shfl_xor_sync(full, h0, o), __shfl_xor_sync(full, l0, o));
                        df_add(h1, l1, __shfl_xor_sync(full, h1, o), __shfl_xor_sync(full, l1, o));
                        df_add(h2, l2, __shfl_xor_sync(full, h2, o), __shfl_xor_sync(full, l2, o));
                        df_add(h3, l3, __shfl_xor_sync(full, h3, o), __shfl_xor_sync(full, l3, o));
                        eb = __fadd_ru(eb, __shfl_xor_sync(full, eb, o));
                    }
                    if (k < nl && sp == 0) {
                        const float *Ch = net.h + net.offC[l] + 4 * k, *Cc = net.l + net.offC[l] + 4 * k;
                        df_add(h0, l0, Ch[0], Cc[0]); df_add(h1, l1, Ch[1], Cc[1]);
                        df_add(h2, l2, Ch[2], Cc[2]); df_add(h3, l3, Ch[3], Cc[3]);
                        df_norm(h0, l0); df_norm(h1, l1); df_norm(h2, l2); df_norm(h3, l3);
                        const float sg = bit_of(s.mask, rl + k) ? -1.0f : 1.0f;
                        *reinterpret_cast<float4 *>(s.rhi + 4 * (rl + k)) = make_float4(sg * h0, sg * h1, sg * h2, sg * h3);
                        *reinterpret_cast<float4 *>(s.rlo + 4 * (rl + k)) = make_float4(sg * l0, sg * l1, sg * l2, sg * l3);
                        const float cl1 = fabsf(Ch[0]) + fabsf(Ch[1]) + fabsf(Ch[2]) + fabsf(Ch[3]);
                        const float e = __fmaf_ru(g, cl1, eb) * 1.01f;
                        s.err[rl + k] = e;
                        s.carry[rl + k] = __fmaf_ru(gn, (fabsf(h0) + fabsf(h1) + fabsf(h2) + fabsf(h3)) * 1.001f, e);
                    }
                }
            }
        }
        __syncthreads();
    }
    // a_F = w_out^T diag(s_L) Z_L + [0 | b_out]  (Cor. 1, Eq. 8), warp 0: lane 4 p + c takes column c of
    // every 8th active unit
    if (tid < 32) {
        const int rL = net.row0[net.L], t0 = s.lst0[net.L], t1 = s.lst0[net.L + 1], c = tid & 3;
        if (M == kFP64) {
            double f = 0.0;
#pragma unroll 4
            for (int t = t0 + (tid >> 2); t < t1; t += 8) {
                const int r = s.lst[t];
                f -= net.d[net.offw + r - rL] * s.r64[4 * r + c];
            }
#pragma unroll 1
            for (int o = 4; o < 32; o <<= 1) f += __shfl_xor_sync(full, f, o);
            if (c == 3) f += net.b_out;
            if (tid < 4) {
                s.aF[c] = f;
                s.aFhi[c] = (float)f;
            }
            if (tid == 0) s.eF[0] = 0.0f;
        } else {
            // double-float with a bound on the l1 error of the four columns
            const float g = df_gamma(t1 - t0 + 40);
            float h = 0.0f, lo = 0.0f, eb = 0.0f, e2 = 0.0f;
#pragma unroll 2
            for (int t = t0 + (tid >> 2); t < t1; t += 8) {
                const int r = s.lst[t];
                const float wh = net.h[net.offw + r - rL], wl = net.l[net.offw + r - rL], zh = s.rhi[4 * r + c];
                df_fma(h, lo, wh, wl, -zh, -s.rlo[4 * r + c]);
                // this column's rounding, and (once) the row's error
                eb = __fmaf_ru(fabsf(wh), g * fabsf(zh) * 1.001f, eb);
                if (tc) e2 = fmaf(wh * s.err[r], wh * s.err[r], e2);        // estimates, by root sum of squares
                else if (c == 0) eb = __fmaf_ru(fabsf(wh), s.err[r], eb);
            }
#pragma unroll 1
            for (int o = 4; o < 32; o <<= 1) {
                const float oh = __shfl_xor_sync(full, h, o), ol = __shfl_xor_sync(full, lo, o);
                df_add(h, lo, oh, ol);
                eb = __fadd_ru(eb, __shfl_xor_sync(full, eb, o));
                e2 += __shfl_xor_sync(full, e2, o);
            }
            eb = __fadd_ru(eb, __shfl_xor_sync(full, eb, 1));
            eb = __fadd_ru(eb, __shfl_xor_sync(full, eb, 2));
            if (tc) eb += 2.0f * sqrtf(e2);
            if (c == 3) df_add(h, lo, net.b_out_hi, net.b_out_lo);
            df_norm(h, lo);
            if (tid < 4) {
                s.aFhi[c] = h;
                s.aFlo[c] = lo;
                s.aF[c] = (double)h + (double)lo;
            }
            if (tid == 0) s.eF[0] = __fmaf_ru(g, fabsf(net.b_out_hi), eb) * 1.01f;
        }
    }
}

// ------------------------------------------------------------------------------------------
// polygon helpers (warp 0)

template <class R>
__device__ __forceinline__ R pdist(const R *r, R ri, const R *v)
{
    return (r[0] * v[0] + r[1] * v[1] + r[2] * v[2] + r[3]) * ri;
}

// One cut of the polygon P[buf] (edge planes E[buf], m vertices) by row k, warp-parallel.  A
// vertex is cut off when its distance from row k's plane exceeds tol.  The two new vertices are
// re-solved from their planes and the face plane aF.  Returns the new vertex count (0 = empty,
// -1 = inconsistent or overflow); *swapped tells whether the result went to buffer buf ^ 1.
// row q in the vertex type R: FP64 rows (any mode) or the FP32 high parts (kDF heuristic pass)
template <class R, int M>
__device__ __forceinline__ void fetch_row(const Sh &s, int q, R *r)
{
    if constexpr (sizeof(R) == 8) {
        row64<M>(s, q, (double *)r);
    } else {
        r[0] = s.rhi[4 * q]; r[1] = s.rhi[4 * q + 1]; r[2] = s.rhi[4 * q + 2]; r[3] = s.rhi[4 * q + 3];
    }
}

template <class R, int M>
__device__ __forceinline__ int warp_cut(const Sh &s, R (*P)[kMaxPoly][3], int m, int buf, int k, R tol, const R *aF,
                                        bool *swapped)
{
    int (*E)[kMaxPoly] = s.pe;
    const int lane = threadIdx.x & 31;
    *swapped = false;
    R rk[4];
    fetch_row<R, M>(s, k, rk);
    const R rn = sqrt(rk[0] * rk[0] + rk[1] * rk[1] + rk[2] * rk[2]);
    if (rn == R(0)) return m;
    const R ri = R(1) / rn;
    const bool o0 = lane < m && pdist(rk, ri, P[buf][lane]) > tol;
    const bool o1 = lane + 32 < m && pdist(rk, ri, P[buf][lane + 32]) > tol;
    const unsigned long long out = (unsigned long long)__ballot_sync(0xffffffffu, o0) |
                                   ((unsigned long long)__ballot_sync(0xffffffffu, o1) << 32);
    const int nout = __popcll(out);
    if (nout == 0) return m;
    if (nout == m) return 0;
    int ia = -1, ib = -1;
    for (int i = lane; i < m; i += 32) {
        const bool oi = (out >> i) & 1ull;
        if (oi && !((out >> ((i + m - 1) % m)) & 1ull)) ia = i;
        if (oi && !((out >> ((i + 1) % m)) & 1ull)) ib = i;
    }
    for (int o = 16; o > 0; o >>= 1) {
        ia = max(ia, __shfl_xor_sync(0xffffffffu, ia, o));
        ib = max(ib, __shfl_xor_sync(0xffffffffu, ib, o));
    }
    if (ia < 0 || ib < 0 || ((ib - ia + m) % m) + 1 != nout) return -1;
    const int nin = m - nout;
    if (nin + 2 > kMaxPoly) return -1;
    const int nb = buf ^ 1;
    const int ea = E[buf][(ia + m - 1) % m], eb = E[buf][ib];
    for (int i = lane; i < m; i += 32) {                 // the kept run b+1 .. a-1, in order
        if ((out >> i) & 1ull) continue;
        const int ni = (i - (ib + 1) + m) % m;
        P[nb][ni][0] = P[buf][i][0]; P[nb][ni][1] = P[buf][i][1]; P[nb][ni][2] = P[buf][i][2];
        E[nb][ni] = E[buf][i];
    }
    bool ok = true;
    if (lane < 2) {
        R pa[4], pb[4], v[3];
        fetch_row<R, M>(s, lane == 0 ? ea : k, pa);
        fetch_row<R, M>(s, lane == 0 ? k : eb, pb);
        ok = solve3<R>(pa, pb, aF, v, nullptr);
        P[nb][nin + lane][0] = v[0]; P[nb][nin + lane][1] = v[1]; P[nb][nin + lane][2] = v[2];
        E[nb][nin + lane] = lane == 0 ? k : eb;
    }
    ok = __all_sync(0xffffffffu, ok);
    __syncwarp();
    *swapped = true;
    return ok ? nin + 2 : -1;
}

// kDF: the final vertices in FP64 from the double-float rows, with the bound dv on how far the
// exact vertex (exact rows) can be, |v* - v|_inf <= |M^-1|_inf max(e_a, e_b, e_F) max(1,|v|) (1.1).
__device__ __forceinline__ void df_final_vertices(const Sh &s, int m, int buf, double vtol)
{
    const int lane = threadIdx.x & 31;
    for (int i = lane; i < m; i += 32) {
        const int ea = s.pe[buf][(i + m - 1) % m], eb = s.pe[buf][i];
        double ra[4], rb[4], v[3], inorm = 0.0;
        row64<kDF>(s, ea, ra);
        row64<kDF>(s, eb, rb);
        const bool ok = solve3<double>(ra, rb, s.aF, v, &inorm);
        const double X = fmax(1.0, fmax(fabs(v[0]), fmax(fabs(v[1]), fabs(v[2]))));
        const double e = fmax((double)s.err[ea], fmax((double)s.err[eb], (double)s.eF[0]));
        s.pv[buf][i][0] = v[0]; s.pv[buf][i][1] = v[1]; s.pv[buf][i][2] = v[2];
        s.dvb[i] = ok ? (float)(inorm * e * X * 1.1 + 4e-16 * X) * 1.01f : 3.0e38f;
        if (s.dvb[i] > vtol * X) s.si[10] = 1;           // this vertex is not known well enough
    }
    __syncwarp();
}

// ------------------------------------------------------------------------------------------
// learned proposal: scores of every neuron row for this cell (block-wide forward pass)

// Features: entry point (3), unit face-plane normal (3), plane offset (1), active fraction of
// each hidden layer (L).  Scores go to z[0..N) (logits; larger = more likely an edge plane).
// y = W x for one cell, W^T stored as n_in rows of n_pairs BF16 pairs (row stride 2 n_pairs).
// Threads take output pairs; when there are fewer pairs than threads the j range is split G
// ways and the partial sums go to part (G x 2 n_pairs floats).  G == 1: y = act(W x + b).
__device__ __forceinline__ void gemv_bf16x2(const __nv_bfloat16 *wt, int n_pairs, int n_in, int n_out,
                                            const float *x, const float *b, bool relu, float *y, float *part, int G)
{
    const __nv_bfloat162 *w = reinterpret_cast<const __nv_bfloat162 *>(wt);
    for (int q = threadIdx.x; q < n_pairs * G; q += kT) {
        const int pr = q % n_pairs, g = q / n_pairs;
        const int j0 = g * n_in / G, j1 = (g + 1) * n_in / G;
        float a0 = 0.0f, a1 = 0.0f;
        const __nv_bfloat162 *wp = w + pr;
#pragma unroll 32
        for (int j = j0; j < j1; ++j) {         // 32 weight loads in flight: the weights stream from L2
            const float2 wf = __bfloat1622float2(wp[(size_t)j * n_pairs]);
            const float xj = x[j];
            a0 = fmaf(wf.x, xj, a0);
            a1 = fmaf(wf.y, xj, a1);
        }
        const int o = 2 * pr;
        if (G == 1) {
            a0 += b[o];
            y[o] = relu ? fmaxf(a0, 0.0f) : a0;
            if (o + 1 < n_out) {
                a1 += b[o + 1];
                y[o + 1] = relu ? fmaxf(a1, 0.0f) : a1;
            }
        } else {
            part[g * 2 * n_pairs + o] = a0;
            part[g * 2 * n_pairs + o + 1] = a1;
        }
    }
    if (G > 1) {
        __syncthreads();
        for (int o = threadIdx.x; o < n_out; o += kT) {
            float a = b[o];
            for (int g = 0; g < G; ++g) a += part[g * 2 * n_pairs + o];
            y[o] = relu ? fmaxf(a, 0.0f) : a;
        }
    }
}

// Learned proposal (no counterpart in the paper): sigmoid-free scores z[0:N] of every neuron for
// this cell, from its entry point, the unit normal and offset of a_F and the per-layer active
// fractions of its pattern.  Hidden widths are even (BF16 pairs); W3^T rows are padded to even.
__device__ void proposal_scores(const MarchArgs &a, const NetDev &net, int64_t cell, const Sh &s, float *z)
{
    const ProposalView &P = a.prop;
    const int tid = threadIdx.x, H = P.hidden, O = P.n_out, I = P.n_in;
    // the start of the scratch region, up to the net's record at kOHot, which stays (proposal_max_hidden)
    float *x = s.partf;
    float *h1 = x + 64, *h2 = h1 + H, *part = h2 + H;
    if (tid == 0) {
        x[0] = __ldcg(a.ar.entry_pt + cell * 3);
        x[1] = __ldcg(a.ar.entry_pt + cell * 3 + 1);
        x[2] = __ldcg(a.ar.entry_pt + cell * 3 + 2);
        const double *F = s.aF;
        const double inv = 1.0 / sqrt(F[0] * F[0] + F[1] * F[1] + F[2] * F[2]);
        x[3] = (float)(F[0] * inv); x[4] = (float)(F[1] * inv); x[5] = (float)(F[2] * inv); x[6] = (float)(F[3] * inv);
        for (int l = 1; l <= net.L; ++l) {
            const int r0 = net.row0[l], n = net.width[l];
            int cnt = 0;
            for (int w = r0 >> 5; w <= (r0 + n - 1) >> 5; ++w) {
                unsigned bits = s.mask[w];
                const int lo = max(r0 - 32 * w, 0), hi = min(r0 + n - 32 * w, 32);
                bits &= (hi >= 32 ? 0xffffffffu : ((1u << hi) - 1u)) & ~((1u << lo) - 1u);
                cnt += __popc(bits);
            }
            x[6 + l] = (float)cnt / (float)n;
        }
    }
    __syncthreads();
    for (int t = tid; t < H; t += kT) {
        float acc = P.b1[t];
        for (int i = 0; i < I; ++i) acc = fmaf(__bfloat162float(P.w1[(size_t)t * I + i]), x[i], acc);
        h1[t] = fmaxf(acc, 0.0f);
    }
    __syncthreads();
    const int H2 = H >> 1, O2 = (O + 1) >> 1;
    gemv_bf16x2(P.w2t, H2, H, H, h1, P.b2, true, h2, part, H2 >= kT ? 1 : kT / H2);
    __syncthreads();
    gemv_bf16x2(P.w3t, O2, H, O, h2, P.b3, false, z, part, O2 >= kT ? 1 : kT / O2);
    __syncthreads();
}

// ------------------------------------------------------------------------------------------
// the face in one pass

// FP64 to FP32 towards zero with integer operations (a conversion instruction goes through the FP64
// pipe): within 2^-23 of x relative; 0 below FP32's normal range, about 3.4e38 above it
__device__ __forceinline__ float f32_toward_zero(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned m = min(hi & 0x7fffffffu, 0x47efffffu);
    unsigned f = (__funnelshift_l(lo, m, 3) - 0x40000000u) & 0x7fffffffu;   // exponent 11 bits -> 8: minus 896
    if (m < 0x38100000u) f = 0u;
    return __uint_as_float(f | (hi & 0x80000000u));
}

// FP64 row k in FP32, towards zero (one copy of the code: it runs three times per cell)
__device__ __noinline__ float4 row32_fp64(const double *r64, int k)
{
    const double2 a = reinterpret_cast<const double2 *>(r64)[2 * k], b = reinterpret_cast<const double2 *>(r64)[2 * k + 1];
    return make_float4(f32_toward_zero(a.x), f32_toward_zero(a.y), f32_toward_zero(b.x), f32_toward_zero(b.y));
}

// row k in FP32: its hi words (kDF), or its FP64 words towards zero
template <int M>
__device__ __forceinline__ float4 row32(const Sh &s, int k)
{
    if (M == kDF) return *reinterpret_cast<const float4 *>(s.rhi + 4 * k);
    return row32_fp64(s.r64, k);
}

// Warp 0: the ring of the lines' intervals (s.seg).  A line carries an edge when the part of it
// inside all others is not empty; the line that ends an edge carries the next one.  Writes the
// edge planes s.pe[0][0 .. m) counter-clockwise; returns m, or 0 when the edges do not close into one
// ring.
__device__ __forceinline__ int ring_of_lines(const Sh &s, int n)
{
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    int *cl = s.ring, *cn = cl + kLines, *cp = cn + kLines, *rk = cp + kLines;
    int m = 0;
#pragma unroll 1
    for (int i = lane; i < kLines; i += 32) {
        const float4 p = s.seg[i];
        const bool alive = i < n && p.y > p.x;
        const unsigned b = __ballot_sync(full, alive);
        const int r = m + __popc(b & ((1u << lane) - 1u));
        rk[i] = alive ? r : -1;
        if (alive) {
            cl[r] = i; cn[r] = __float_as_int(p.w); cp[r] = __float_as_int(p.z);
        }
        m += __popc(b);
    }
    __syncwarp();
    bool ok = m >= 3 && m <= 32;
    int nxt = -1, prv = -1, k = -1;
    if (ok && lane < m) {
        const int jn = cn[lane], jp = cp[lane];
        nxt = jn >= 0 ? rk[jn] : -1;
        prv = jp >= 0 ? rk[jp] : -1;
        k = __float_as_int(s.line[cl[lane]].w);
    }
    const int back = __shfl_sync(full, prv, nxt & 31);
    ok = ok && (lane >= m || (nxt >= 0 && prv >= 0 && back == lane));
    if (!__all_sync(full, ok)) return 0;
    int cur = 0, pos = 0, left = m;
#pragma unroll 1
    do {
        if (lane == cur) pos = m - left;
        cur = __shfl_sync(full, nxt, cur);
        --left;
    } while (cur != 0 && left > 0);
    if (cur != 0 || left != 0) return 0;             // no cycle, or a shorter one
    if (lane < m) s.pe[0][pos] = k;
    __syncwarp();
    return m;
}

// Warp 0: the ring's vertices in FP64, each from the rows of its two edges and the face plane
// (Eq. 11, solve3's Cramer's rule), one lane per vertex and coordinate: the warp issues the
// instructions of one coordinate instead of three, and an FP64 warp instruction takes about 64
// cycles for one lane as for 32.  Also the vertices in FP32 with the vertex term of the check's
// bound (vf[i][3]) and kDF's vertex error bounds.  False when a vertex is not known well enough.
template <int M>
__device__ __forceinline__ bool ring_vertices(const Arena &ar, const Sh &s, int m, int N)
{
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    // the planes' hash words, for the pushes
    const int ze = lane < m ? s.pe[0][lane] : N;
    const unsigned long long zv = ze < N ? __ldg(ar.zob + ze) : 0ull;
    const double *R = s.r64;
    if (M == kDF) {
        // the edges' rows as FP64, one lane per coefficient, into the spare polygon buffer
        double *e = &s.pv[1][0][0];
        for (int i = lane; i < 4 * m; i += 32) {
            const int q = 4 * s.pe[0][i >> 2] + (i & 3);
            e[i] = (double)s.rhi[q] + (double)s.rlo[q];
        }
        __syncwarp();
        R = e;
    }
    const int v = lane / 3, d = lane - 3 * v, d1 = d == 2 ? 0 : d + 1, d2 = d == 0 ? 2 : d - 1;
    const int l0 = 3 * v, l1 = l0 + 1, l2 = l0 + 2 > 31 ? 31 : l0 + 2;
    bool good = true;
#pragma unroll 1
    for (int b = 0; b < m; b += 10) {
        const int i = b + v;
        const bool on = v < 10 && i < m;
        const int iq = on ? i : 0, ip = iq == 0 ? m - 1 : iq - 1;
        const int ka = s.pe[0][ip], kb = s.pe[0][iq];
        const double *p = R + 4 * (M == kDF ? ip : ka), *q = R + 4 * (M == kDF ? iq : kb), *f = s.aF;
        const double c0 = q[d1] * f[d2] - q[d2] * f[d1], c1 = f[d1] * p[d2] - f[d2] * p[d1],
                     c2 = p[d1] * q[d2] - p[d2] * q[d1];
        const double det = p[0] * __shfl_sync(full, c0, l0) + p[1] * __shfl_sync(full, c0, l1) + p[2] * __shfl_sync(full, c0, l2);
        const double inv = -1.0 / det;
        const double x = (p[3] * c0 + q[3] * c1 + f[3] * c2) * inv;
        const float xf = (float)x;
        float X = fmaxf(1.0f, fabsf(xf));
        X = fmaxf(X, fmaxf(__shfl_sync(full, X, l0), fmaxf(__shfl_sync(full, X, l1), __shfl_sync(full, X, l2)))) * 1.0001f;
        float w = 10.5f * kU * X;
        bool fine = isfinite(xf);
        if (M == kDF) {
            // |M^-1|_inf max(e_a, e_b, e_F) max(1, |v|) (1.1): as df_final_vertices
            float rs = (float)(fabs(c0) + fabs(c1) + fabs(c2)) * 1.0001f;
            rs = fmaxf(__shfl_sync(full, rs, l0), fmaxf(__shfl_sync(full, rs, l1), __shfl_sync(full, rs, l2)));
            const float in = rs * fabsf((float)inv) * 1.0001f;
            const float e = fmaxf(s.err[ka], fmaxf(s.err[kb], s.eF[0]));
            const float dv = fmaf(in * e, X * 1.1f, 4e-16f * X) * 1.01f;
            fine = fine && dv <= (float)kVertexTol * X;
            w = fmaf(8.5f * kU, X, dv) * 1.0001f;
            if (on && d == 0) s.dvb[i] = dv;
        }
        if (on) {
            s.pv[0][i][d] = x;
            s.vf[i][d] = xf;
            if (d == 0) s.vf[i][3] = w;
            good = good && fine;
        }
        if (on && d == 0) s.pf[0][i][0] = X;
    }
    s.zb[lane] = zv;
    return __all_sync(full, good);
}

// A close call of the FP32 test (or one that is not finite): row k at vertex i in FP64, as the
// sequential clip tests it.  1: violated, 2: within the tolerance or undecidable, 0: it holds.  Out
// of line: FP32 decides nearly every pair.
template <int M>
__device__ __noinline__ int close_call(int max_n, double delta, int k, int i, float ri, float rl1, float band, float Xm)
{
    const Sh s = make_sh(max_n);
    const double *v6 = s.pv[0][i];
    if (M == kFP64) {
        const double dd = pdist((const double *)(s.r64 + 4 * k), (double)ri, v6);
        if (dd > delta) return 1;
        return dd < -delta ? 0 : 2;
    }
    atomicAdd(s.blk + 5, 1ull);
    double r6[4];
    row64<kDF>(s, k, r6);
    const double s6 = r6[0] * v6[0] + r6[1] * v6[1] + r6[2] * v6[2] + r6[3];
    const double m6 = fabs(r6[0] * v6[0]) + fabs(r6[1] * v6[1]) + fabs(r6[2] * v6[2]) + fabs(r6[3]);
    const double B6 = (double)s.err[k] * (double)Xm + (double)rl1 * 1.0001 * (double)s.dvb[i] + (double)band + 1e-15 * m6;
    if (s6 > B6) return 1;
    return s6 < -B6 ? 0 : 2;
}

// The face of the cell without the sequential cuts: every warp contributes its rows nearest to the
// entry point, the lines in which these rows (and the box) meet the face plane are cut against
// each other all at once (each line's interval inside all the others, in FP32 coordinates of the
// plane about the entry point), and the intervals that remain close into the polygon's ring.  Its
// vertices are solved in FP64 from their planes; then every row is tested at every vertex in FP32
// with a certified bound, a close call in FP64.  Rows found violated join the edges as the lines
// of another round.  The ring is kept only when every row that is not an edge at a vertex is
// beyond the tolerance there, which makes it the cell's face whatever FP32 did before: the vertices
// are then the system's own, in order.  Anything else (a row within the tolerance, an open
// ring, a vertex not known well enough, too many rounds) returns false, and the sequential clip
// (kFP64) or FP64 (kDF) decides the cell from the start.
//
// What bounds it is the serial chain of a cell, so the chain is short: about five barriers and a
// dozen FP64 instructions, where the cuts one by one issued some 400 FP64 instructions in one warp
// (about 64 cycles each, for one lane as for 32).  From the rows to the checked face a cell of a
// 3-[64]x4-1 net in FP64 took 69,700 cycles of its block with the cuts one by one and takes 12,800; a
// 3-[32]x4-1 net in mixed precision 68,000 and 11,200.  The march of the first (44,304 cells from one
// ray) went from 12.3 to 4.6 ms, of the second (10,472 cells) from 3.6 to 1.5 ms.
template <int M>
__device__ __forceinline__ bool fast_face(const MarchArgs &a, int N, const Sh &s, int *rounds)
{
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const unsigned full = 0xffffffffu;
    const int NC = N + kBoxPlanes;
    long long tq0 = 0, tq1 = 0;
    AM_TICK(tq0);
    int n;                                           // lines
    {
        const float px = s.ent[0], py = s.ent[1], pz = s.ent[2];
        const int nwr = min(kNW, (N + 31) >> 5), P = nwr == 1 ? 32 : min(kLinePicks, (kLines - kBoxPlanes) / nwr);
        float b1 = 3.0e38f, b2 = 3.0e38f;
        int k1 = -1, k2 = -1;
        bool loose = false;
#pragma unroll 1
        for (int k = tid; k < N; k += kT) {
            const float4 r = row32<M>(s, k);
            const float n2 = r.x * r.x + r.y * r.y + r.z * r.z;
            if (!(n2 > kTiny && n2 < kHuge)) continue;
            const float ri = rsqrtf(n2);
            if (M == kDF) loose |= s.err[k] * ri > kDfLoose;
            const float d = fabsf(fmaf(r.x, px, fmaf(r.y, py, fmaf(r.z, pz, r.w)))) * ri;
            if (d < b1) { b2 = b1; k2 = k1; b1 = d; k1 = k; }
            else if (d < b2) { b2 = d; k2 = k; }
        }
        // kDF: as in the sequential clip, a row error that no useful number of tests survives
        if (M == kDF && tid == 0)
            loose |= s.eF[0] * rsqrtf(s.aFhi[0] * s.aFhi[0] + s.aFhi[1] * s.aFhi[1] + s.aFhi[2] * s.aFhi[2]) > kDfLoose;
        if (loose) s.si[4] = 1;
        if (wid < nwr) {
            int *near = s.near_k + kBoxPlanes + wid * P;
            if (nwr == 1) {
                near[lane] = k1;
            } else {
#pragma unroll 1
                for (int q = 0; q < P; ++q) {
                    // the distance's bits, the lane in the lowest five: one reduction picks the row
                    const unsigned key = k1 >= 0 ? (__float_as_uint(b1) & ~31u) | (unsigned)lane : 0xffffffffu;
                    const unsigned best = __reduce_min_sync(full, key);
                    if (best == 0xffffffffu) {
                        if (lane == 0)
                            for (int z = q; z < P; ++z) near[z] = -1;
                        break;
                    }
                    if (key == best) { near[q] = k1; b1 = b2; k1 = k2; k2 = -1; }
                }
            }
        }
        if (tid < kBoxPlanes) s.near_k[tid] = N + tid;
        n = kBoxPlanes + nwr * P;
    }
    __syncthreads();
    AM_TICK(tq1);
    AM_PHASE(a, 2, tq0, tq1);
    if (M == kDF && s.si[4]) return false;
    for (int round = 0;; ++round) {
        AM_TICK(tq0);
        if (tid < kLines) {
            // the lines in the plane's coordinates (u, w) about the entry point
            float A = 0.0f, B = 0.0f, C = -1.0f;
            const int k = tid < n ? s.near_k[tid] : -1;
            if (k >= 0) {
                const float f0 = s.aFhi[0], f1 = s.aFhi[1], f2 = s.aFhi[2];
                const float inv = rsqrtf(f0 * f0 + f1 * f1 + f2 * f2);
                const float n0 = f0 * inv, n1 = f1 * inv, n2 = f2 * inv;
                const float ax = fabsf(n0), ay = fabsf(n1), az = fabsf(n2);
                const int ei = (ax <= ay && ax <= az) ? 0 : (ay <= az ? 1 : 2);
                // u = n x e_i, w = n x u
                float u0 = ei == 0 ? 0.0f : (ei == 1 ? -n2 : n1), u1 = ei == 0 ? n2 : (ei == 1 ? 0.0f : -n0),
                      u2 = ei == 0 ? -n1 : (ei == 1 ? n0 : 0.0f);
                const float un = rsqrtf(u0 * u0 + u1 * u1 + u2 * u2);
                u0 *= un; u1 *= un; u2 *= un;
                const float w0 = n1 * u2 - n2 * u1, w1 = n2 * u0 - n0 * u2, w2 = n0 * u1 - n1 * u0;
                const float4 r = row32<M>(s, k);
                A = r.x * u0 + r.y * u1 + r.z * u2;
                B = r.x * w0 + r.y * w1 + r.z * w2;
                const float q2 = A * A + B * B;
                if (q2 > 1e-10f * (r.x * r.x + r.y * r.y + r.z * r.z)) {
                    const float q = rsqrtf(q2);
                    C = fmaf(r.x, s.ent[0], fmaf(r.y, s.ent[1], fmaf(r.z, s.ent[2], r.w))) * q;
                    A *= q; B *= q;
                } else {
                    A = B = 0.0f;                     // (nearly) parallel to the face plane: no line in it
                }
            }
            s.line[tid] = make_float4(A, B, C, __int_as_float(k));
        }
        __syncthreads();
        AM_TICK(tq1);
        AM_PHASE(a, 1, tq0, tq1);
        {
            // line i's interval inside a quarter of the others: at -c n + t (-b, a), line j holds for
            // t D <= c_i (n_i . n_j) - c_j, D = n_i x n_j
            const int i = tid / kParts;
            float t0 = -3.0e38f, t1 = 3.0e38f;
            int j0 = -1, j1 = -1;
            const float4 L = s.line[i];
#pragma unroll 2
            for (int j = tid & (kParts - 1); j < n; j += kParts) {
                const float4 o = s.line[j];
                const float D = L.x * o.y - L.y * o.x, num = L.z * (L.x * o.x + L.y * o.y) - o.z;
                const float t = __fdividef(num, D);
                if (D > 1e-7f && t < t1) { t1 = t; j1 = j; }
                if (D < -1e-7f && t > t0) { t0 = t; j0 = j; }
                // beside a parallel line that cuts it off
                if (fabsf(D) <= 1e-7f && j != i && num < 0.0f) t1 = -3.0e38f;
            }
            if (L.x == 0.0f && L.y == 0.0f) t1 = -3.0e38f;
#pragma unroll 1
            for (int o = 1; o < kParts; o <<= 1) {
                const float u0 = __shfl_xor_sync(full, t0, o), u1 = __shfl_xor_sync(full, t1, o);
                const int i0 = __shfl_xor_sync(full, j0, o), i1 = __shfl_xor_sync(full, j1, o);
                if (u0 > t0) { t0 = u0; j0 = i0; }
                if (u1 < t1) { t1 = u1; j1 = i1; }
            }
            if ((tid & (kParts - 1)) == 0) s.seg[i] = make_float4(t0, t1, __int_as_float(j0), __int_as_float(j1));
        }
        if (tid == 0) { s.si[3] = 0; s.si[4] = 0; }
        __syncthreads();
        AM_TICK(tq0);
        AM_PHASE(a, 3, tq1, tq0);
        if (wid == 0) {
            const int m = ring_of_lines(s, n);
            const bool ok = m > 0 && ring_vertices<M>(a.ar, s, m, N);
            if (lane == 0) s.si[0] = ok ? m : 0;
        }
        __syncthreads();
        AM_TICK(tq1);
        AM_PHASE(a, 4, tq0, tq1);
        const int m = s.si[0];
        if (m == 0) return false;
        // ---- a5: every row at every vertex; the area flag s.si[6] (1: clear of the smallest kept area, 2:
        //      FP64 decides) by the last warp, which has the fewest rows
        if (wid == kNW - 1) {
            const float4 *v = reinterpret_cast<const float4 *>(s.vf);
            const bool clear = area_clear(v[0], v[m / 3], v[2 * m / 3], area_min(a.box_hi));
            if (lane == 0) s.si[6] = clear ? 1 : 2;
        }
        float Xm = 1.0f;
        if (M == kDF)
#pragma unroll 1
            for (int i = 0; i < m; ++i) Xm = fmaxf(Xm, s.pf[0][i][0]);
#pragma unroll 1
        for (int k = tid; k < NC; k += kT) {
            const float4 r = row32<M>(s, k);
            const float n2 = r.x * r.x + r.y * r.y + r.z * r.z;
            if (!(n2 > kTiny && n2 < kHuge)) {
                // a zero normal (a constant row) holds in its own cell; FP32 does not judge a tiny one
                const bool zero = M == kDF ? n2 == 0.0f && s.rlo[4 * k] == 0.0f && s.rlo[4 * k + 1] == 0.0f && s.rlo[4 * k + 2] == 0.0f
                                           : s.r64[4 * k] == 0.0 && s.r64[4 * k + 1] == 0.0 && s.r64[4 * k + 2] == 0.0;
                if (!zero) s.si[4] = 1;
                continue;
            }
            const float ri = rsqrtf(n2), rl1 = fabsf(r.x) + fabsf(r.y) + fabsf(r.z);
            const float band = (float)a.delta * (n2 * ri) * 1.01f;     // delta |r|: the tolerance band
            // the bound |r|_1 w_v + c_r: FP32 evaluation (4 terms), the row and the vertex rounded to FP32
            // (8.5 u; 10.5 u with the row rounded towards zero), the vertex's and the row's own error
            const float cr = M == kDF ? __fmaf_ru(s.err[k], Xm, __fmaf_ru(8.5f * kU, fabsf(r.w), band))
                                      : __fmaf_ru(10.5f * kU, fabsf(r.w), band);
            bool viol = false, edge = false;
            int ea = s.pe[0][m - 1];
#pragma unroll 2
            for (int i = 0; i < m; ++i) {
                const int eb = s.pe[0][i];
                const bool own = k == ea || k == eb;
                edge |= k == eb;
                ea = eb;
                if (own) continue;
                const float4 V = *reinterpret_cast<const float4 *>(s.vf[i]);
                const float sl = fmaf(r.x, V.x, fmaf(r.y, V.y, fmaf(r.z, V.z, r.w)));
                const float B = __fmaf_ru(rl1, V.w, cr);
                if (sl < -B) continue;
                if (sl > B) { viol = true; continue; }
                const int c = close_call<M>(a.max_n, a.delta, k, i, ri, rl1, band, Xm);
                viol |= c == 1;
                if (c == 2) s.si[4] = 1;
            }
            if (viol) {
                if (edge) {
                    s.si[4] = 1;                      // FP32 kept an edge that the vertices deny
                } else {
                    const int p = atomicAdd(s.si + 3, 1);
                    s.viol[p] = k;
                }
            }
        }
        __syncthreads();
        AM_TICK(tq0);
        AM_PHASE(a, 5, tq1, tq0);
        if (s.si[4]) return false;
        const int nv = s.si[3];
        if (nv == 0) {
            *rounds = round;
            return true;
        }
        if (round + 1 >= kFastFix || m + nv > kLines) return false;
        // another round: the edges and the violated rows
        if (tid < m) s.near_k[tid] = s.pe[0][tid];
        else if (tid < m + nv) s.near_k[tid] = s.viol[tid - m];
        n = m + nv;
        __syncthreads();
    }
}

// ------------------------------------------------------------------------------------------
// one cell

template <int M>
__device__ __noinline__ void load_rows(const MarchArgs &a, int N, int64_t cell)
{
    const Sh s = make_sh(a.max_n);
    const int tid = threadIdx.x;
    // rows composed beforehand on the tensor cores, as FP32 pairs (the hi words [hi x 4] of
    // rows 0..N, then their lo words [lo x 4])
    // (signs as compose<M>, a_F last).  The pairs are the rows: the double-float tests are
    // certified against them with no further row error, as FP64 tests take FP64 rows.
    const float4 *src = reinterpret_cast<const float4 *>(a.rows_in) + (cell - a.begin) * (int64_t)(N + 1) * 2;
    for (int k = tid; k < N; k += kT) {
        const float4 h = __ldcs(src + k), l = __ldcs(src + (N + 1) + k);
        if (M == kFP64) {
            double *r = s.r64 + 4 * k;
            r[0] = (double)h.x + (double)l.x; r[1] = (double)h.y + (double)l.y;
            r[2] = (double)h.z + (double)l.z; r[3] = (double)h.w + (double)l.w;
        } else {
            *reinterpret_cast<float4 *>(s.rhi + 4 * k) = h;
            *reinterpret_cast<float4 *>(s.rlo + 4 * k) = l;
            s.err[k] = 0.0f;
        }
    }
    if (tid < 4) {
        const float h = reinterpret_cast<const float *>(src + N)[tid];
        const float l = reinterpret_cast<const float *>(src + 2 * N + 1)[tid];
        s.aF[tid] = (double)h + (double)l;
        if (M == kDF) { s.aFhi[tid] = h; s.aFlo[tid] = l; }
    }
    if (tid == 0) s.eF[0] = 0.0f;
    __syncthreads();
}

// The sequential clip: the square about the box section cut by the candidate rows one by one, then
// every row checked at every vertex; leaves the polygon in shared memory (s.si[0] vertices in buffer
// s.si[1], status s.si[2]).  Returns the fix-up rounds, or -1 (kDF) when FP64 must decide the cell.
// Out of line: the one-pass polygon (fast_face) takes nearly every cell.
template <int M>
__device__ __noinline__ int slow_clip(const MarchArgs &a, const NetDev &net, int64_t cell)
{
    const Sh s = make_sh(a.max_n);
    const Arena &ar = a.ar;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int N = net.N, NC = N + kBoxPlanes;          // checked rows: neurons + box
    int rounds = 0;
    __syncthreads();
    // the frame and the initial square (thread 0)
    if (tid == 0) {
        // an FP32 frame is enough: the square only has to contain the box section, and its
        // planes never bound a face (the box planes always cut them away)
        const float F[4] = {(float)s.aF[0], (float)s.aF[1], (float)s.aF[2], (float)s.aF[3]};
        const float nn = F[0] * F[0] + F[1] * F[1] + F[2] * F[2];
        int m = 0;
        if (nn > 0.0f && isfinite(nn)) {
            const float inn = 1.0f / nn;
            const float p0[3] = {-F[3] * F[0] * inn, -F[3] * F[1] * inn, -F[3] * F[2] * inn};
            const float inv = rsqrtf(nn);
            const float n[3] = {F[0] * inv, F[1] * inv, F[2] * inv};
            const float ax = fabsf(n[0]), ay = fabsf(n[1]), az = fabsf(n[2]);
            const int ei = (ax <= ay && ax <= az) ? 0 : (ay <= az ? 1 : 2);
            const float e0 = ei == 0 ? 1.0f : 0.0f, e1 = ei == 1 ? 1.0f : 0.0f, e2 = ei == 2 ? 1.0f : 0.0f;
            float u[3] = {n[1] * e2 - n[2] * e1, n[2] * e0 - n[0] * e2, n[0] * e1 - n[1] * e0};
            const float un = rsqrtf(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
            u[0] *= un; u[1] *= un; u[2] *= un;
            const float w[3] = {n[1] * u[2] - n[2] * u[1], n[2] * u[0] - n[0] * u[2], n[0] * u[1] - n[1] * u[0]};
            const float sz = 1.05f * 1.7320508f * (float)a.box;
            // square edges -w, +u, +w, -u (ids N+6..N+9), counter-clockwise about n
            const float d[4][3] = {{-w[0], -w[1], -w[2]}, {u[0], u[1], u[2]}, {w[0], w[1], w[2]}, {-u[0], -u[1], -u[2]}};
            const float cu[4] = {-1.0f, 1.0f, 1.0f, -1.0f}, cw[4] = {-1.0f, -1.0f, 1.0f, 1.0f};
            for (int i = 0; i < 4; ++i) {
                const int k = N + kBoxPlanes + i;
                const float r[4] = {d[i][0], d[i][1], d[i][2], -(d[i][0] * p0[0] + d[i][1] * p0[1] + d[i][2] * p0[2]) - sz};
                for (int c = 0; c < 4; ++c) {
                    if (M == kFP64) s.r64[4 * k + c] = (double)r[c];
                    else { s.rhi[4 * k + c] = r[c]; s.rlo[4 * k + c] = 0.0f; }
                }
                if (M == kDF) s.err[k] = 0.0f;
                for (int c = 0; c < 3; ++c) {
                    const float x = p0[c] + sz * (cu[i] * u[c] + cw[i] * w[c]);
                    s.pv[0][i][c] = (double)x;
                    s.pf[0][i][c] = x;
                }
                s.pe[0][i] = k;
            }
            m = 4;
        }
        s.si[0] = m; s.si[1] = 0; s.si[2] = 0; s.si[3] = 0; s.si[4] = 0; s.si[5] = 0; s.si[9] = 0; s.si[10] = 0;
    }
    __syncthreads();
    // inverse norms, FP32 (they only scale distances used for ordering and the FP64 tolerance
    // test, never a sign)
    for (int k = tid; k < NC + kSquarePlanes; k += kT) {
        float n2;
        if (M == kFP64) {
            const double *r = s.r64 + 4 * k;
            n2 = (float)(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]);
        } else {
            const float *r = s.rhi + 4 * k;
            n2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2];
        }
        s.rinv[k] = n2 > 0.0f ? rsqrtf(n2) : 0.0f;
    }
    if (M == kDF) {
        // When a row's certified error, as a distance, exceeds kDfLoose the sign tests of this
        // cell cannot be certified in any useful number: the rigorous bound grows by the row
        // sums of |W_l| per layer (deep, wide nets).  Go to FP64 at once instead of clipping
        // twice.
        int loose = 0;
        for (int k = tid; k < N; k += kT) loose |= s.err[k] * s.rinv[k] > kDfLoose;
        if (tid == 0) loose |= s.eF[0] * rsqrtf((float)(s.aF[0] * s.aF[0] + s.aF[1] * s.aF[1] + s.aF[2] * s.aF[2])) > kDfLoose;
        if (__syncthreads_or(loose)) return -1;
    } else {
        __syncthreads();
    }

    // ---- candidate rows, each thread keeps its best two, each warp contributes its four best:
    //      the rows nearest to the entry point, or the rows the learned proposal scores highest
    //      (the entry plane first), or none at all (the all-row check then clips alone)
    const bool learned = a.candidates == kCandLearned && a.prop.n_out == N && a.prop.n_in == 7 + net.L;
    float *score = (float *)s.viol;
    // the scores of a level batch come from the tensor cores; else this block computes them
    const __nv_bfloat16 *gscore = learned && a.scores_in ? a.scores_in + (cell - a.begin) * (int64_t)a.scores_ld : nullptr;
    if (learned && !gscore) proposal_scores(a, net, cell, s, score);
    {
        const float px = __ldcg(ar.entry_pt + cell * 3), py = __ldcg(ar.entry_pt + cell * 3 + 1),
                    pz = __ldcg(ar.entry_pt + cell * 3 + 2);
        const int entry = __ldcg(ar.entry_plane + cell);
        float b1 = 3.0e38f, b2 = 3.0e38f;
        int k1 = -1, k2 = -1;
        for (int k = (a.candidates == kCandNone ? NC : tid); k < NC; k += kT) {
            if (s.rinv[k] == 0.0f) continue;
            float d;
            if (learned) {
                if (k >= N) continue;
                d = k == entry ? -3.0e37f : -(gscore ? __bfloat162float(gscore[k]) : score[k]);
            } else if (M == kFP64) {
                const double *r = s.r64 + 4 * k;
                d = (float)fabs(r[0] * px + r[1] * py + r[2] * pz + r[3]) * s.rinv[k];
            } else {
                const float *r = s.rhi + 4 * k;
                d = fabsf(r[0] * px + r[1] * py + r[2] * pz + r[3]) * s.rinv[k];
            }
            if (d < b1) { b2 = b1; k2 = k1; b1 = d; k1 = k; }
            else if (d < b2) { b2 = d; k2 = k; }
        }
#pragma unroll 1
        for (int pick = 0; pick < kPicks; ++pick) {
            float bd = b1;
            int bk = k1;
            for (int o = 16; o > 0; o >>= 1) {
                const float od = __shfl_xor_sync(0xffffffffu, bd, o);
                const int ok = __shfl_xor_sync(0xffffffffu, bk, o);
                if (ok >= 0 && (bk < 0 || od < bd || (od == bd && ok < bk))) { bd = od; bk = ok; }
            }
            if (lane == 0) { s.near_w[wid * kPicks + pick] = bk; s.near_dw[wid * kPicks + pick] = bd; }
            if (bk >= 0 && bk == k1) { b1 = b2; k1 = k2; b2 = 3.0e38f; k2 = -1; }
        }
    }
    __syncthreads();

    // ---- a4: warp 0 cuts the square with the candidates, nearest cutting row first.  A row
    // that holds on the polygon holds on every later (smaller) one, so it retires at once.
    if (wid == 0) {
        float d = s.near_dw[lane];
        const int k = s.near_w[lane];
        bool live = k >= 0 && d < 3.0e38f;
        if (learned && live) {
            // the proposal chose the rows; they are cut nearest first, as the geometric rule's
            // (the entry plane passes through the entry point, so it still comes first)
            const float px = __ldcg(ar.entry_pt + cell * 3), py = __ldcg(ar.entry_pt + cell * 3 + 1),
                        pz = __ldcg(ar.entry_pt + cell * 3 + 2);
            float r[4];
            if (M == kFP64) {
                double r64[4];
                fetch_row<double, M>(s, k, r64);
                r[0] = (float)r64[0]; r[1] = (float)r64[1]; r[2] = (float)r64[2]; r[3] = (float)r64[3];
            } else {
                fetch_row<float, M>(s, k, r);
            }
            d = fabsf(r[0] * px + r[1] * py + r[2] * pz + r[3]) * s.rinv[k];
        }
        // order-preserving unsigned image of the distance (scores may be negative)
        const unsigned du = __float_as_uint(d);
        const unsigned key = (du & 0x80000000u) ? ~du : (du | 0x80000000u);
            int m = s.si[0], buf = 0, status = 0, ncut = 0;
        const float aFf[4] = {s.aFhi[0], s.aFhi[1], s.aFhi[2], s.aFhi[3]};
        while (m > 0) {
            bool cut = false;
            if (live) {
                if (M == kFP64) {
                    double r[4];
                    fetch_row<double, M>(s, k, r);
                    const double ri = (double)s.rinv[k];
                    for (int i = 0; i < m && !cut; ++i) cut = pdist(r, ri, s.pv[buf][i]) > a.delta;
                } else {
                    float r[4];
                    fetch_row<float, M>(s, k, r);
                    const float ri = s.rinv[k];
                    for (int i = 0; i < m && !cut; ++i) cut = pdist(r, ri, s.pf[buf][i]) > 1e-7f;
                }
            }
            live = cut;
            if (!__any_sync(0xffffffffu, cut)) break;
            const unsigned kmin = __reduce_min_sync(0xffffffffu, cut ? key : 0xffffffffu);
            const int kc = (int)__reduce_min_sync(0xffffffffu, (cut && key == kmin) ? (unsigned)k : 0xffffffffu);
            if (k == kc) live = false;
            bool sw;
            int nm;
            if (M == kFP64) nm = warp_cut<double, M>(s, s.pv, m, buf, kc, a.delta, s.aF, &sw);
            else nm = warp_cut<float, M>(s, s.pf, m, buf, kc, 1e-7f, aFf, &sw);
            if (nm < 0) { status = 1; m = 0; break; }
            if (sw) buf ^= 1;
            m = nm;
            ++ncut;
        }
            if (M == kDF && m > 0) df_final_vertices(s, m, buf, kVertexTol);
        if (lane == 0) { s.si[0] = m; s.si[1] = buf; s.si[2] = status; s.blk[6] += (unsigned long long)ncut; }
    }
    __syncthreads();

    // ---- a5: every row at every vertex; violators are cut in by warp 0 and the check repeats
    for (rounds = 0;; ++rounds) {
        const int m = s.si[0], buf = s.si[1];
        if (M == kDF && s.si[10]) return -1;     // a vertex too uncertain: FP64
        // kDF: a polygon emptied (or a clip that failed) in the uncertified FP32 candidate pass
        // proves nothing: FP64 decides
        if (M == kDF && (m == 0 || s.si[2])) return -1;
        if (m == 0 || s.si[2]) break;
        for (int i = tid; i < m; i += kT) {
            const double *v = s.pv[buf][i];
            s.vf[i][0] = (float)v[0]; s.vf[i][1] = (float)v[1]; s.vf[i][2] = (float)v[2];
            s.vf[i][3] = (float)fmax(1.0, fmax(fabs(v[0]), fmax(fabs(v[1]), fabs(v[2])))) * 1.0001f;
        }
        if (tid == 0) { s.si[3] = 0; s.si[4] = 0; }
        __syncthreads();
        int ndeg = 0, close = 0;
        for (int k = tid; k < NC; k += kT) {
            if (s.rinv[k] == 0.0f) continue;        // zero normal: constant row, holds in its own cell
            bool viol = false, amb = false;
            if (M == kFP64) {
                const double *r = s.r64 + 4 * k;
                const double ri = (double)s.rinv[k];
                for (int i = 0; i < m; ++i) {
                    const int ea = s.pe[buf][(i + m - 1) % m], eb = s.pe[buf][i];
                    if (k == ea || k == eb) continue;
                    const double dd = pdist(r, ri, s.pv[buf][i]);
                    if (dd > a.delta) viol = true;
                    else if (dd >= -a.delta) ++ndeg;
                }
            } else {
                const float *r = s.rhi + 4 * k;
                const float rl1 = fabsf(r[0]) + fabsf(r[1]) + fabsf(r[2]);
                const float band = (float)a.delta / s.rinv[k] * 1.01f;   // delta |r|: the oracle's tolerance band
                const float ek = s.err[k];
                for (int i = 0; i < m; ++i) {
                    const int ea = s.pe[buf][(i + m - 1) % m], eb = s.pe[buf][i];
                    if (k == ea || k == eb) continue;
                    const float *v = s.vf[i];
                    const float sl = r[0] * v[0] + r[1] * v[1] + r[2] * v[2] + r[3];
                    const float mag = fabsf(r[0] * v[0]) + fabsf(r[1] * v[1]) + fabsf(r[2] * v[2]) + fabsf(r[3]);
                    // FP32 evaluation (4 terms) + dropping lo + rounding v to FP32: (4 + 4) u |r||v|
                    const float B = __fmaf_ru(8.5f * kU, mag, __fmaf_ru(ek, v[3], __fmaf_ru(rl1, s.dvb[i], band)));
                    if (sl > B) { viol = true; continue; }
                    if (sl >= -B) {                    // close call: FP64 re-evaluation
                        ++close;
                        double r6[4];
                        row64<kDF>(s, k, r6);
                        const double *v6 = s.pv[buf][i];
                        const double s6 = r6[0] * v6[0] + r6[1] * v6[1] + r6[2] * v6[2] + r6[3];
                        const double m6 = fabs(r6[0] * v6[0]) + fabs(r6[1] * v6[1]) + fabs(r6[2] * v6[2]) + fabs(r6[3]);
                        const double B6 = (double)ek * (double)v[3] + (double)rl1 * 1.0001 * (double)s.dvb[i] +
                                          (double)band + 1e-15 * m6;
                        if (s6 > B6) viol = true;
                        else if (s6 >= -B6) amb = true;
                    }
                }
                // A violated row that already carries an edge of the polygon: the FP32 candidate
                // pass cut by a row that does not really cut the face (its exact vertices then lie
                // outside the neighbouring edges' rows).  Cutting again would repeat that plane
                // with a zero-length edge, so the cell goes to FP64, which decides every cut.
                if (viol)
                    for (int i = 0; i < m; ++i) amb |= s.pe[buf][i] == k;
            }
            if (viol) {
                const int p = atomicAdd(s.si + 3, 1);
                s.viol[p] = k;
            }
            if (amb) s.si[4] = 1;
        }
        {
            int tot;
            block_scan_excl(ndeg, s.wsum, &tot);
            ndeg = tot;
            block_scan_excl(close, s.wsum, &tot);
            if (tid == 0) s.blk[5] += (unsigned long long)tot;
        }
        if (tid == 0) s.si[5] = ndeg;
        __syncthreads();
        if (s.si[4]) return -1;
        const int nviol = s.si[3];
        if (nviol == 0) break;
        if (rounds + 1 >= kMaxFix) {
            if (tid == 0) s.si[2] = 2;
            __syncthreads();
            break;
        }
        if (wid == 0) {
            int mm = m, bb = buf, status = 0, t = 0;
            const double tol = M == kFP64 ? a.delta : 0.0;
            bool changed = false;
            for (; t < nviol && mm > 0; ++t) {
                bool sw;
                const int nm = warp_cut<double, M>(s, s.pv, mm, bb, s.viol[t], tol, s.aF, &sw);
                if (nm < 0) { status = 1; mm = 0; break; }
                if (sw) bb ^= 1;
                changed |= sw || nm != mm;
                mm = nm;
            }
            if (M == kDF && mm > 0) df_final_vertices(s, mm, bb, kVertexTol);
            if (lane == 0) {
                s.si[0] = mm; s.si[1] = bb; s.si[2] = status; s.si[9] += 1; s.blk[6] += (unsigned long long)t;
                // kDF: rows the certified FP32 test calls violated that the cut on the pairs in FP64
                // does not move: the two views of the rows disagree, so FP64 decides the cell
                if (M == kDF && !changed && status == 0) s.si[10] = 1;
            }
        }
        __syncthreads();
    }
    if (tid == 0) s.si[6] = 2;
    __syncthreads();
    return rounds;
}

// Warp 0: whether the polygon's area exceeds the smallest kept one, as a fan about vertex 0
__device__ __noinline__ void area_test(int max_n, int buf, int m, double box)
{
    const Sh s = make_sh(max_n);
    const int lane = threadIdx.x & 31;
    const double *p0 = s.pv[buf][0];
    double nx = 0.0, ny = 0.0, nz = 0.0;
    for (int i = lane + 1; i < m - 1; i += 32) {
        const double *p = s.pv[buf][i], *q = s.pv[buf][i + 1];
        const double ax = p[0] - p0[0], ay = p[1] - p0[1], az = p[2] - p0[2];
        const double bx = q[0] - p0[0], by = q[1] - p0[1], bz = q[2] - p0[2];
        nx += ay * bz - az * by; ny += az * bx - ax * bz; nz += ax * by - ay * bx;
    }
    nx = warp_sum(nx); ny = warp_sum(ny); nz = warp_sum(nz);
    const double amin = 2e-24 * box * box;          // twice the smallest kept area
    if (lane == 0) s.si[6] = nx * nx + ny * ny + nz * nz > amin * amin;
}

// Pushes of keys wider than kThreadPushWords: one warp per edge, the key words split over the lanes
__device__ __noinline__ void push_wide(const MarchArgs &a, int64_t cell, int buf, int m, int N, int pool0, int pool1, int pj)
{
    const Sh s = make_sh(a.max_n);
    const Arena &ar = a.ar;
    const unsigned long long h = *s.hsh;
    for (int i = threadIdx.x >> 5; i < m; i += kNW) {
        const int e = s.pe[buf][i];
        if (e >= N) continue;
        const double *p = s.pv[buf][i], *q = s.pv[buf][i + 1 == m ? 0 : i + 1];
        const bool pool = e >= pool0 && e < pool1;
        insert_neighbor_warp(ar, s.mask, cell, *s.nid, (unsigned)e, h ^ ar.zob[e] ^ (pool ? ar.zob[pool0 + pj] : 0ull),
                             0.5f * (f32_toward_zero(p[0]) + f32_toward_zero(q[0])),
                             0.5f * (f32_toward_zero(p[1]) + f32_toward_zero(q[1])),
                             0.5f * (f32_toward_zero(p[2]) + f32_toward_zero(q[2])), true, pool0, pool1,
                             pool ? pool0 + pj : -1);
    }
}

struct CellOut {
    int emit;        // corners written (0 = empty)
    int ambiguous;   // kDF: an undecidable sign test; nothing written
};

template <int M>
__device__ __forceinline__ CellOut solve_cell(const MarchArgs &a, const NetDev &net, int64_t cell)
{
    const Sh s = make_sh(a.max_n);
    const Arena &ar = a.ar;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int N = s.hot->N;
    long long tp0 = 0, tp1 = 0, tp2 = 0, tp3 = 0;
    AM_TICK(tp0);
    // box rows (exact)
    // (kDF: the pairs are stored as they are, exact FP32 words: the normal's components are
    // 0 and +-1 and the offset is the host's split of the box, so no conversion runs here)
    if (tid < 4 * kBoxPlanes) {
        const int i = tid >> 2, c = tid & 3;
        const bool ax = c == (i >> 1);
        if (M == kFP64) {
            s.r64[4 * N + tid] = c == 3 ? -a.box : (ax ? ((i & 1) ? -1.0 : 1.0) : 0.0);
        } else {
            s.rhi[4 * N + tid] = c == 3 ? -a.box_hi : (ax ? ((i & 1) ? -1.0f : 1.0f) : 0.0f);
            s.rlo[4 * N + tid] = c == 3 ? -a.box_lo : 0.0f;
            s.err[N + i] = 0.0f;
        }
    }
    if (tid < 11) s.si[tid] = 0;
    int rounds = 0;
    bool fast = false;
    if (a.rows_in) {
        load_rows<M>(a, N, cell);
    } else {
        compose<M>(net, s, false, a.max_n);
        __syncthreads();
        AM_TICK(tp1);
        AM_PHASE(a, 0, tp0, tp1);
        if (a.candidates == kCandNearest) {
            fast = fast_face<M>(a, N, s, &rounds);
            if (M == kDF && !fast) return CellOut{0, 1};
        }
    }
    if (!fast) {
        AM_TICK(tp2);
        rounds = slow_clip<M>(a, net, cell);
        AM_TICK(tp3);
        AM_PHASE(a, 9, tp2, tp3);
        if (rounds < 0) return CellOut{0, 1};
    }

    AM_TICK(tp2);
    // ---- a6 emit, a7 march
    const int m = s.si[0], buf = s.si[1];
    int status = s.si[2];
    if (!fast)
#pragma unroll 1
        for (int i = 0; i < m; ++i)
            if (s.pe[buf][i] >= N + kBoxPlanes) status = 3;   // a square edge: the plane misses the box
    int emit = (m >= 3 && status == 0) ? m : 0;
    if (emit && s.si[6] == 2) {
        __syncthreads();
        if (wid == 0) area_test(a.max_n, buf, m, a.box);
        __syncthreads();
    }
    if (emit && !s.si[6]) emit = 0;
    if (emit > ar.maxv) {
        if (tid == 0) atomicOr(ar.counters + kStatus, kStFaceVerts);
        emit = 0;
    }
    if (tid == 0) {
        ar.nverts[cell] = emit;
        s.blk[0] += 1;
        if (!emit) s.blk[1] += 1;
        if (emit) s.blk[2] += (unsigned long long)s.si[5];
        if (rounds) s.blk[3] += 1;
        if (status == 1 || status == 2) atomicOr(ar.counters + kStatus, kStClip);
    }
    AM_TICK(tp3);
    AM_PHASE(a, 6, tp2, tp3);
    if (emit) {
        // the face record (warps 1..; warp 0 pushes); m <= kMaxPoly
        static_assert(3 * kMaxPoly + 32 <= kT && kMaxPoly + 32 <= kT, "one thread per word of a face");
        if ((unsigned)(tid - 32) < 3u * (unsigned)m) ar.verts[cell * ar.maxv * 3 + (tid - 32)] = (&s.pv[buf][0][0])[tid - 32];
        if ((unsigned)(tid - 32) < (unsigned)m) ar.edges[cell * ar.maxv + (tid - 32)] = s.pe[buf][tid - 32];
        // a max-pooled net (Sec. 5.2): crossing pooling plane n_units + i moves the pooled index j
        // to i (two key bits change), and the new cell enters through its pooling row of j
        int pj = 0, pool0 = kNoPool, pool1 = kNoPool;
        if (s.hot->M >= 2) {
            pool0 = s.hot->units;
            pool1 = N;
#pragma unroll 1
            while (pj < s.hot->M - 1 && !bit_of(s.mask, pool0 + pj)) ++pj;
        }
        if (ar.kw <= kThreadPushWords) {
            // narrow keys: one lane of warp 0 per edge
            if (wid == 0) {
                const unsigned long long h = *s.hsh;
                const int nid = *s.nid;
#pragma unroll 1
                for (int i0 = 0; i0 < m; i0 += 32) {
                    const int i = i0 + lane, e = i < m ? s.pe[buf][i] : N;
                    const bool on = e < N;
                    unsigned long long hc = 0;
                    int entry = -1;
                    float mid[3] = {0.0f, 0.0f, 0.0f};
                    if (on) {
                        hc = h ^ (fast ? s.zb[i] : ar.zob[e]);
                        if (e >= pool0 && e < pool1) {
                            entry = pool0 + pj;
                            hc ^= ar.zob[entry];
                        }
                        // the shared edge's midpoint: it only orders the neighbour's candidates
                        const double *p = s.pv[buf][i], *q = s.pv[buf][i + 1 == m ? 0 : i + 1];
#pragma unroll
                        for (int c = 0; c < 3; ++c) mid[c] = 0.5f * (f32_toward_zero(p[c]) + f32_toward_zero(q[c]));
                    }
                    insert_neighbors(ar, s.mask, cell, nid, on, (unsigned)e, hc, mid[0], mid[1], mid[2], pool0, pool1, entry);
                }
            }
        } else {
            push_wide(a, cell, buf, m, N, pool0, pool1, pj);
        }
    }
    if (ar.kw > kThreadPushWords) __syncthreads();     // every warp has pushed
    AM_TICK(tp2);
    AM_PHASE(a, 7, tp3, tp2);
    return CellOut{emit, 0};
}

// FP64 for the cells (and nets) the double-float kernel does not decide
__device__ __noinline__ void solve_cell_fp64(const MarchArgs &a, const NetDev &net, int64_t cell)
{
    solve_cell<kFP64>(a, net, cell);
}

template <int MODE>
__device__ __forceinline__ void process_cell(const MarchArgs &a, int64_t cell, const Sh &s)
{
    const Arena &ar = a.ar;
    // the cell's record was written by another block of this launch: read it through L2, every
    // word in flight at once
    const unsigned long long *key = ar.keys + cell * ar.kw;
    const int dead = __ldcg(ar.nverts + cell), nid = __ldcg(ar.net + cell);
    if ((int)threadIdx.x < 2 * ar.kw)                      // all key words (at most 256): pushes copy them
        s.mask[threadIdx.x] = __ldcg(reinterpret_cast<const unsigned *>(key) + threadIdx.x);
    if (threadIdx.x >= kT - 3) s.ent[kT - 1 - threadIdx.x] = __ldcg(ar.entry_pt + cell * 3 + (kT - 1 - threadIdx.x));
    if (threadIdx.x == kT - 4) *s.hsh = __ldcg(ar.hash + cell);
    if (threadIdx.x == kT - 5) *s.nid = nid;
    const NetDev &net = a.nets[nid];
    const bool other = s.hot->id != nid;
    if (!other) {
        if (MODE == kDF && s.hot->df_ok) touch_weights<kDF>(*s.hot);
        else touch_weights<kFP64>(*s.hot);
    }
    __syncthreads();
    if (dead == -2) return;                              // a duplicate seed id: never solved
    if (other) {
        fill_hot(&net, nid, a.max_n);
        __syncthreads();
    }
    if (MODE == kDF && !s.hot->df_ok && !a.rows_in) {
        if (threadIdx.x == 0) s.blk[4] += 1;             // solved in FP64 (the net's bound is too loose)
        solve_cell_fp64(a, net, cell);
    } else if (MODE == kDF) {
        const CellOut o = solve_cell<kDF>(a, net, cell);
        if (o.ambiguous) {
            if (threadIdx.x == 0) s.blk[4] += 1;
            __syncthreads();
            solve_cell_fp64(a, net, cell);
        }
    } else {
        solve_cell<kFP64>(a, net, cell);
    }
}

// ------------------------------------------------------------------------------------------
// schedules

__device__ __forceinline__ long long global_ns()
{
    long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned ld_relaxed(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Ticket of the next cell to solve, or -1 when the march is over (every handed-out cell is
// finished), the ticket is beyond the limit, or a wait ran out of time (status flag set).
// Waiting polls the ticket's own flag with plain loads and an exponential back-off, so that idle
// blocks do not flood the counters' cache lines with atomics.  An acquire empties the SM's L1, and with
// it the weights of the block beside this one: the flag is read relaxed, with one fence once it is
// set, and the counters (acquired: only they end the march) are read every 8th time.
__device__ long long next_ticket(const MarchArgs &a)
{
    unsigned long long *C = a.ar.counters;
    const long long t = (long long)atomicAdd(C + kHead, 1ull);
    if (t >= a.limit) return -1;
    const long long t0 = global_ns();
    unsigned ns = 16, poll = 0;
    for (;;) {
        if (ld_relaxed(a.ar.ready + t) != 0u) {
            // acquire: the cell's record, written before its flag was released
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
            return t;
        }
        if ((poll++ & 7) == 7) {
            // every handed-out cell finished (done read before the count: no cell can still push)
            const unsigned long long done = ld_acquire(C + kDone);
            const unsigned long long n = ld_acquire(C + kNCells);
            if (done >= n && (unsigned long long)t >= n) return -1;
            if (global_ns() - t0 > a.wait_ns) { atomicOr(C + kStatus, kStTimeout); return -1; }
        }
        __nanosleep(ns);
        ns = min(2 * ns, 128u);
    }
}

// per-block statistics: zero at entry, one atomic flush at exit
__device__ __forceinline__ void blk_init(const Sh &s)
{
    if (threadIdx.x < 8) s.blk[threadIdx.x] = 0ull;
    if (threadIdx.x == 8) s.hot->id = -1;
    __syncthreads();
}

__device__ __forceinline__ void blk_flush(const MarchArgs &a, const Sh &s)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long *C = a.ar.counters;
        if (s.blk[0]) atomicAdd(C + kSolved, s.blk[0]);
        if (s.blk[1]) atomicAdd(C + kEmpty, s.blk[1]);
        if (s.blk[2]) atomicAdd(C + kDegenerate, s.blk[2]);
        if (s.blk[3]) atomicAdd(C + kFixups, s.blk[3]);
        if (s.blk[4]) atomicAdd(C + kRefined, s.blk[4]);
        if (s.blk[5]) atomicAdd(C + kCloseCalls, s.blk[5]);
        if (s.blk[6]) atomicAdd(C + kCuts, s.blk[6]);
    }
}

template <int MODE>
__global__ void __launch_bounds__(kT, AM_MIN_BLOCKS) march_persistent_kernel(const __grid_constant__ MarchArgs a)
{
    const Sh s = make_sh(a.max_n);
    __shared__ long long ticket;
    blk_init(s);
    for (;;) {
        long long tw0 = 0, tw1 = 0;
        AM_TICK(tw0);
        // the last warp draws the next ticket while warp 0 may still be pushing the last cell's
        // neighbours
        if (threadIdx.x == kT - 1) ticket = next_ticket(a);
        __syncthreads();
        AM_TICK(tw1);
        AM_PHASE(a, 8, tw0, tw1);
        const long long t = ticket;
        if (t < 0) break;
        process_cell<MODE>(a, t, s);
        if (threadIdx.x < 32) {
            // the pushes of warp 0's lanes (kw > kThreadPushWords: of every warp, after a barrier) are
            // counted before the cell is
            __syncwarp();
            if (threadIdx.x == 0) {
                asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(a.ar.counters + kDone), "l"(1ull) : "memory");
            }
        }
    }
    blk_flush(a, s);
}

template <int MODE>
__global__ void __launch_bounds__(kT, AM_MIN_BLOCKS) march_range_kernel(const __grid_constant__ MarchArgs a)
{
    const Sh s = make_sh(a.max_n);
    blk_init(s);
    if (a.list) {
        const int64_t n = (int64_t)__ldcg(a.list_count);
        for (int64_t i = blockIdx.x; i < n; i += gridDim.x) {
            process_cell<MODE>(a, a.list[i], s);
            __syncthreads();
        }
    } else {
        for (int64_t cell = a.begin + blockIdx.x; cell < a.end; cell += gridDim.x) {
            process_cell<MODE>(a, cell, s);
            __syncthreads();
        }
    }
    blk_flush(a, s);
}

template <int MODE>
__global__ void __launch_bounds__(kT, AM_MIN_BLOCKS)
    compose_kernel(const __grid_constant__ MarchArgs a, const NetDev *netp, const unsigned long long *keys, int kw_in, int64_t n,
                   double *rows, float *err)
{
    const Sh s = make_sh(a.max_n);
    const NetDev &net = *netp;
    const int N = net.N, mw = 2 * ((a.max_n + 63) / 64);
    fill_hot(netp, 0, a.max_n);
    for (int64_t c = blockIdx.x; c < n; c += gridDim.x) {
        for (int w = threadIdx.x; w < mw; w += kT)
            s.mask[w] = (w >> 1) < kw_in ? (unsigned)(keys[c * kw_in + (w >> 1)] >> ((w & 1) * 32)) : 0u;
        __syncthreads();
        compose<MODE>(net, s, a.tc != 0, a.max_n);
        __syncthreads();
        double *out = rows + c * (int64_t)(N + 1) * 4;
        for (int k = threadIdx.x; k < N; k += kT) {
            double r[4];
            row64<MODE>(s, k, r);
            out[4 * k] = r[0]; out[4 * k + 1] = r[1]; out[4 * k + 2] = r[2]; out[4 * k + 3] = r[3];
            if (err) err[c * (N + 1) + k] = MODE == kFP64 ? 0.0f : s.err[k];
        }
        if (threadIdx.x == 0) {
            for (int q = 0; q < 4; ++q) out[4 * N + q] = s.aF[q];
            if (err) err[c * (N + 1) + N] = MODE == kFP64 ? 0.0f : s.eF[0];
        }
        __syncthreads();
    }
}

void launch_compose(const MarchArgs &a, int mode, const NetDev *net, const unsigned long long *keys, int key_words,
                    int64_t n, double *rows, float *err, cudaStream_t st)
{
    const int smem = march_smem_bytes(a.max_n, a.max_w);
    const int grid = (int)std::min<int64_t>(n, 152 * 8);
    if (mode == kDF) compose_kernel<kDF><<<grid, kT, smem, st>>>(a, net, keys, key_words, n, rows, err);
    else compose_kernel<kFP64><<<grid, kT, smem, st>>>(a, net, keys, key_words, n, rows, err);
}

cudaError_t prepare_march_kernels(int max_n, int max_w, int *blocks_per_sm)
{
    const int smem = march_smem_bytes(max_n, max_w);
    const void *ks[6] = {(const void *)march_persistent_kernel<kFP64>, (const void *)march_persistent_kernel<kDF>,
                         (const void *)march_range_kernel<kFP64>, (const void *)march_range_kernel<kDF>,
                         (const void *)compose_kernel<kFP64>, (const void *)compose_kernel<kDF>};
    cudaError_t e;
    for (const void *k : ks)
        if ((e = allow_smem(k, smem))) return e;
    int b0 = 0, b1 = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b0, march_persistent_kernel<kFP64>, kT, smem))) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b1, march_persistent_kernel<kDF>, kT, smem))) return e;
    *blocks_per_sm = b0 < b1 ? b0 : b1;
    return cudaSuccess;
}

void launch_march(const MarchArgs &a, int mode, bool persistent, int grid, cudaStream_t st)
{
    const int smem = march_smem_bytes(a.max_n, a.max_w);
    // shared memory for two resident blocks, the rest of the unified L1 for the weights and the stack (the
    // driver rounds the carveout to a supported split); said per launch, as it depends on the context
    cudaLaunchAttribute carve{};
    carve.id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    carve.val.sharedMemCarveout = (unsigned)std::min(100, (int)((2.0 * (smem + 1024) * 100.0) / (228.0 * 1024.0)) + 3);
    cudaLaunchConfig_t c{};
    c.gridDim = dim3((unsigned)grid);
    c.blockDim = dim3(kT);
    c.dynamicSmemBytes = (size_t)smem;
    c.stream = st;
    c.attrs = &carve;
    c.numAttrs = 1;
    if (persistent) {
        if (mode == kDF) cudaLaunchKernelEx(&c, march_persistent_kernel<kDF>, a);
        else cudaLaunchKernelEx(&c, march_persistent_kernel<kFP64>, a);
    } else {
        if (mode == kDF) cudaLaunchKernelEx(&c, march_range_kernel<kDF>, a);
        else cudaLaunchKernelEx(&c, march_range_kernel<kFP64>, a);
    }
}

}  // namespace am
