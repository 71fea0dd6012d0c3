// am_clip_warp.cu -- the clip of the sliced level march with one warp per cell (Alg. 1 steps 6-11
// on rows composed beforehand on the tensor cores).
//
// A block holds kWW warps and each warp solves its own cell start to finish, so the serial
// parts of a cell (the cuts of its polygon) occupy one warp instead of idling a whole block,
// and many cells are in flight per SM.  The rows are read from memory where the block version
// stages them in shared memory: FP32 pairs, a_F last, the cell's N + 1 hi words [hi x 4] and then
// its N + 1 lo words [lo x 4], so a pass that reads only hi words reads half the bytes.  Per cell:
//   candidates : each lane keeps the two rows nearest to the point the cell was entered through
//                among the rows it scans, and with learned candidates also the row the proposal
//                scores highest among them (the proposal extends the nearest set);
//   clip       : a square about that point, in FP32 coordinates of the face plane, is cut by the lines of
//                those 64 (96) candidates, nearest cutting line first, then every vertex is solved
//                in FP64 from its two planes (Eq. 11).  The square need not contain the box's
//                section (a seed may lie outside the box): a cell with an edge of it left goes to
//                the block kernel;
//   check      : every row at every vertex with a certified FP32 bound; the rows it does not clear
//                (the edges' own among them) one by one, close calls in FP64; violated rows join
//                the edges as the lines of another round;
//   emit, push : the face record, then each neuron edge pushes its neighbour (Alg. 1 step 10).
// A cell that needs more than this (a test the FP64 close call cannot decide, a row within the
// tolerance band of a vertex, a polygon beyond the warp's capacity, too many violators) is
// handed, untouched, to a list that the block kernel then solves with its FP64 fallback, so the
// result is the block kernel's in every case.
#include <algorithm>
#include <cuda_bf16.h>

#include "am_block.cuh"
#include "am_kernels.h"

namespace am {

namespace {

constexpr int kWW = 8;            // warps (cells) per block
constexpr int kWPoly = 48;        // polygon vertices a warp holds
constexpr int kWViol = 32;        // violated rows cut in per check round
constexpr int kWMaxKw = 128;      // key words (N <= 8190)
constexpr int kWMaxFix = 8;       // check / fix-up rounds
constexpr float kWU = 5.9604645e-8f;   // 2^-24

// a warp of the finish pass (after the dense check on the tensor cores)
struct WarpSh {
    double pv[2][kWPoly][3];      // FP64 polygon
    float mid[kWPoly][3];         // the edges' midpoints, for the pushes
    int pe[2][kWPoly];            // edge planes (edge i: vertex i -> i + 1)
    float4 vf[kWPoly];            // FP32 vertices (x, y, z) and the vertex term of the check's bound (w)
    int2 ve[kWPoly];              // the planes of the two edges at each vertex
    float dvb[kWPoly];            // bound on each FP64 vertex's error
    int viol[kWViol];
    double aF[4];
    int nviol;
    unsigned key[2 * kWMaxKw];    // the cell's key as 32-bit words (pushes copy it)
};

int warp_smem_bytes() { return kWW * (int)sizeof(WarpSh); }

// the rows of one cell: N rows in memory, the 6 box rows analytic
struct WRows {
    const float4 *p;              // [hi, lo] per row
    int N;
    float box, box_lo;            // the box as an FP32 pair: box rows' offsets -box (hi), -box_lo (lo)
    __device__ __forceinline__ float4 hi(int k) const
    {
        if (k < N) return __ldg(p + k);
        const int i = k - N;
        const float sg = (i & 1) ? -1.0f : 1.0f;
        return make_float4((i >> 1) == 0 ? sg : 0.0f, (i >> 1) == 1 ? sg : 0.0f, (i >> 1) == 2 ? sg : 0.0f, -box);
    }
    __device__ __forceinline__ void f64(int k, double *r) const
    {
        const float4 h = hi(k);
        if (k < N) {
            const float4 l = __ldg(p + (N + 1) + k);
            r[0] = (double)h.x + (double)l.x; r[1] = (double)h.y + (double)l.y;
            r[2] = (double)h.z + (double)l.z; r[3] = (double)h.w + (double)l.w;
        } else {
            r[0] = h.x; r[1] = h.y; r[2] = h.z;
            r[3] = (double)h.w - (double)box_lo;
        }
    }
};

__device__ __forceinline__ double wpdist(const double *r, double ri, const double *v)
{
    return (r[0] * v[0] + r[1] * v[1] + r[2] * v[2] + r[3]) * ri;
}

// One cut of the polygon P[buf] (m vertices) by row k, the warp's lanes over the vertices: a
// vertex is cut off when its distance from row k's plane exceeds tol; the two new vertices are
// solved from their planes and the face plane aF.  Returns the new count (0 = empty, -1 =
// inconsistent or beyond kWPoly); *swapped: the result went to buffer buf ^ 1.
__device__ int wcut(WarpSh &S, double (*P)[kWPoly][3], int m, int buf, int k, double tol, const double *aF, const WRows &rv,
                    bool *swapped)
{
    const int lane = threadIdx.x & 31;
    *swapped = false;
    double rk[4];
    rv.f64(k, rk);
    const double rn = sqrt(rk[0] * rk[0] + rk[1] * rk[1] + rk[2] * rk[2]);
    if (rn == 0.0) return m;
    const double ri = 1.0 / rn;
    const bool o0 = lane < m && wpdist(rk, ri, P[buf][lane]) > tol;
    const bool o1 = lane + 32 < m && wpdist(rk, ri, P[buf][lane + 32]) > tol;
    const unsigned long long out = (unsigned long long)__ballot_sync(0xffffffffu, o0) |
                                   ((unsigned long long)__ballot_sync(0xffffffffu, o1) << 32);
    const int nout = __popcll(out);
    if (nout == 0) return m;
    if (nout == m) return 0;
    int ia = -1, ib = -1;
    for (int i = lane; i < m; i += 32) {
        const bool oi = (out >> i) & 1ull;
        const int ip = i == 0 ? m - 1 : i - 1, in = i + 1 == m ? 0 : i + 1;
        if (oi && !((out >> ip) & 1ull)) ia = i;
        if (oi && !((out >> in) & 1ull)) ib = i;
    }
    for (int o = 16; o > 0; o >>= 1) {
        ia = max(ia, __shfl_xor_sync(0xffffffffu, ia, o));
        ib = max(ib, __shfl_xor_sync(0xffffffffu, ib, o));
    }
    if (ia < 0 || ib < 0 || ((ib - ia + m) % m) + 1 != nout) return -1;
    const int nin = m - nout;
    if (nin + 2 > kWPoly) return -1;
    const int nb = buf ^ 1;
    const int ea = S.pe[buf][ia == 0 ? m - 1 : ia - 1], eb = S.pe[buf][ib];
    for (int i = lane; i < m; i += 32) {                 // the kept run b+1 .. a-1, in order
        if ((out >> i) & 1ull) continue;
        int ni = i - (ib + 1);
        if (ni < 0) ni += m;
        P[nb][ni][0] = P[buf][i][0]; P[nb][ni][1] = P[buf][i][1]; P[nb][ni][2] = P[buf][i][2];
        S.pe[nb][ni] = S.pe[buf][i];
    }
    bool ok = true;
    if (lane < 2) {
        double pa[4], pb[4], v[3];
        rv.f64(lane == 0 ? ea : k, pa);
        rv.f64(lane == 0 ? k : eb, pb);
        ok = solve3<double>(pa, pb, aF, v, nullptr);
        P[nb][nin + lane][0] = v[0]; P[nb][nin + lane][1] = v[1]; P[nb][nin + lane][2] = v[2];
        S.pe[nb][nin + lane] = lane == 0 ? k : eb;
    }
    ok = __all_sync(0xffffffffu, ok);
    __syncwarp();
    *swapped = true;
    return ok ? nin + 2 : -1;
}

// the polygon's vertices in FP64 from its planes' rows (exact pairs: no row error term), with
// the bound on their rounding; false when a vertex cannot be solved
__device__ bool wfinal(WarpSh &S, int m, int buf, const WRows &rv)
{
    const int lane = threadIdx.x & 31;
    bool ok = true;
    for (int i = lane; i < m; i += 32) {
        const int ea = S.pe[buf][i == 0 ? m - 1 : i - 1], eb = S.pe[buf][i];
        double ra[4], rb[4], v[3];
        rv.f64(ea, ra);
        rv.f64(eb, rb);
        const bool good = solve3<double>(ra, rb, S.aF, v, nullptr);
        const double X = fmax(1.0, fmax(fabs(v[0]), fmax(fabs(v[1]), fabs(v[2]))));
        S.pv[buf][i][0] = v[0]; S.pv[buf][i][1] = v[1]; S.pv[buf][i][2] = v[2];
        S.dvb[i] = (float)(4e-16 * X) * 1.01f;
        ok = ok && good;
    }
    ok = __all_sync(0xffffffffu, ok);
    __syncwarp();
    return ok;
}

// the cell's key as 32-bit words in the warp's shared memory (pushes copy it)
__device__ __forceinline__ void wload_key(WarpSh &S, const Arena &ar, int64_t cell)
{
    const int lane = threadIdx.x & 31;
    for (int w = lane; w < ar.kw; w += 32) {
        const unsigned long long x = __ldcg(ar.keys + cell * ar.kw + w);
        S.key[2 * w] = (unsigned)x;
        S.key[2 * w + 1] = (unsigned)(x >> 32);
    }
}

// The cell's rows view, and its key and face plane a_F in the warp's shared memory
__device__ void wcell_setup(const MarchArgs &a, WarpSh &S, int64_t cell, int N, WRows &rv)
{
    const int lane = threadIdx.x & 31;
    rv.p = reinterpret_cast<const float4 *>(a.rows_in) + (cell - a.begin) * 2 * (int64_t)(N + 1);
    rv.N = N;
    rv.box = a.box_hi;
    rv.box_lo = a.box_lo;
    wload_key(S, a.ar, cell);
    if (lane < 4) {
        const float h = reinterpret_cast<const float *>(rv.p + N)[lane];
        const float l = reinterpret_cast<const float *>(rv.p + 2 * N + 1)[lane];   // lo block: N + 1 + N
        S.aF[lane] = (double)h + (double)l;
    }
    __syncwarp();
}

// A close call of the FP32 test: row k at the FP64 vertex v6 from the exact pair, against the
// vertex's own error (|r|_1 dvb), the tolerance band and the FP64 evaluation's rounding.
// Returns 1 when the row is violated, 2 when the vertex is within the band (the FP64 path
// decides), 0 when it holds.  Out of line: the FP32 test decides nearly every pair.
__device__ __noinline__ int wclose(const WRows &rv, int k, const double *v6, float rl1, float dvb, float delta)
{
    double r6[4];
    rv.f64(k, r6);
    const float4 h = rv.hi(k);
    const float band = delta * sqrtf(h.x * h.x + h.y * h.y + h.z * h.z);   // delta |r|: the tolerance band
    const double s6 = r6[0] * v6[0] + r6[1] * v6[1] + r6[2] * v6[2] + r6[3];
    const double m6 = fabs(r6[0] * v6[0]) + fabs(r6[1] * v6[1]) + fabs(r6[2] * v6[2]) + fabs(r6[3]);
    const double B6 = (double)rl1 * 1.0001 * (double)dvb + (double)band + 1e-15 * m6;
    if (s6 > B6) return 1;
    return s6 >= -B6 ? 2 : 0;
}

// The certified all-row check of the polygon in buffer buf (FP64 vertices): every row at every
// vertex in FP32 with a bound, close calls in FP64 from the exact pair; violated rows are cut in
// (FP64) and the check repeats, at most kWMaxFix rounds.  Returns true when the cell must go to
// the block kernel (a row within the band, a violated row that is already an edge, too many
// violators or rounds, a cut that fails).
__device__ bool wcheck(const MarchArgs &a, WarpSh &S, const WRows &rv, int N, int &m, int &buf, int &rounds,
                       int &ncut, int &cell_close)
{
    const int lane = threadIdx.x & 31;
    const unsigned FULL = 0xffffffffu;
    const int NC = N + kBoxPlanes;
    const float delta = (float)a.delta * 1.01f;
    bool fallback = false;
    while (true) {
        for (int i = lane; i < m; i += 32) {
            const double *v = S.pv[buf][i];
            const float x = (float)v[0], y = (float)v[1], z = (float)v[2];
            // the bound on the FP32 test of row r at this vertex (evaluation, the dropped lo words,
            // the vertex rounded to FP32: 8.5 u (|r|_1 |v|_inf + |r_3|); the FP64 vertex's own error:
            // |r|_1 dvb) is |r|_1 w + c_r with w = 8.5 u max(1, |v|_inf) + dvb and c_r = 8.5 u |r_3|
            // + delta |r| (|r . v| <= |r|_1 |v|_inf; each coordinate within half an ulp of v's)
            const float X = fmaxf(1.0f, fmaxf(fabsf(x), fmaxf(fabsf(y), fabsf(z)))) * 1.0001f;
            S.vf[i] = make_float4(x, y, z, __fmaf_ru(8.5f * kWU, X, S.dvb[i]));
            S.ve[i] = make_int2(S.pe[buf][i == 0 ? m - 1 : i - 1], S.pe[buf][i]);
        }
        if (lane == 0) S.nviol = 0;
        __syncwarp();
        bool amb = false;
        int close = 0;
        for (int k0 = lane; k0 < NC; k0 += 32 * 4) {
            float4 rr[4];
            float rl1[4], cr[4];
            bool viol[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = k0 + 32 * u;
                rr[u] = k < N ? __ldg(rv.p + k) : (k < NC ? rv.hi(k) : make_float4(0.0f, 0.0f, 0.0f, 0.0f));
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float4 r = rr[u];
                const float n2 = r.x * r.x + r.y * r.y + r.z * r.z;
                // a zero normal (a constant row, which holds in its own cell) or no row: skipped
                rl1[u] = n2 == 0.0f ? -1.0f : fabsf(r.x) + fabsf(r.y) + fabsf(r.z);
                cr[u] = __fmaf_ru(8.5f * kWU, fabsf(r.w), delta * sqrtf(n2));   // + delta |r|: the tolerance band
                viol[u] = false;
            }
            for (int i = 0; i < m; ++i) {
                const float4 V = S.vf[i];
                const int2 E = S.ve[i];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int k = k0 + 32 * u;
                    if (rl1[u] < 0.0f || k == E.x || k == E.y) continue;
                    const float4 r = rr[u];
                    const float sl = fmaf(r.x, V.x, fmaf(r.y, V.y, fmaf(r.z, V.z, r.w)));
                    const float B = __fmaf_ru(rl1[u], V.w, cr[u]);
                    if (sl > B) { viol[u] = true; continue; }
                    if (sl >= -B) {                        // close call: FP64 from the exact pair
                        ++close;
                        const int c = wclose(rv, k, S.pv[buf][i], rl1[u], S.dvb[i], delta);
                        viol[u] |= c == 1;
                        amb |= c == 2;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (!viol[u]) continue;
                const int k = k0 + 32 * u;
                for (int i = 0; i < m; ++i) amb |= S.pe[buf][i] == k;   // a spurious FP32 cut
                const int p = atomicAdd(&S.nviol, 1);
                if (p < kWViol) S.viol[p] = k;
                else amb = true;
            }
        }
        for (int o = 16; o > 0; o >>= 1) close += __shfl_xor_sync(FULL, close, o);
        cell_close += close;
        if (__any_sync(FULL, amb)) { fallback = true; break; }
        __syncwarp();
        const int nviol = S.nviol;
        if (nviol == 0) break;
        if (rounds + 1 >= kWMaxFix) { fallback = true; break; }
        for (int t = 0; t < nviol && m > 0; ++t) {
            bool sw;
            const int nm = wcut(S, S.pv, m, buf, S.viol[t], 0.0, S.aF, rv, &sw);
            if (nm < 0) { fallback = true; break; }
            if (sw) buf ^= 1;
            m = nm;
        }
        ncut += nviol;
        if (fallback || m == 0) { fallback = true; break; }
        if (!wfinal(S, m, buf, rv)) { fallback = true; break; }
        ++rounds;
    }
    return fallback;
}

// a6 emit, a7 march for a solved cell: the face record (empty when it has fewer than 3 vertices or no
// area), then one push per neuron edge; returns whether a face was written
__device__ bool wemit(const MarchArgs &a, WarpSh &S, int64_t cell, int net_id, int N, int m, int buf)
{
    const int lane = threadIdx.x & 31;
    const Arena &ar = a.ar;
    int emit = m >= 3 ? m : 0;
    if (emit) {
        const double *p0 = S.pv[buf][0];
        double nx = 0.0, ny = 0.0, nz = 0.0;
        for (int i = lane + 1; i < m - 1; i += 32) {
            const double *p = S.pv[buf][i], *q = S.pv[buf][i + 1];
            const double ax = p[0] - p0[0], ay = p[1] - p0[1], az = p[2] - p0[2];
            const double bx = q[0] - p0[0], by = q[1] - p0[1], bz = q[2] - p0[2];
            nx += ay * bz - az * by; ny += az * bx - ax * bz; nz += ax * by - ay * bx;
        }
        nx = warp_sum(nx); ny = warp_sum(ny); nz = warp_sum(nz);
        const double amin = 2e-24 * a.box * a.box;    // twice the smallest kept area
        if (!(nx * nx + ny * ny + nz * nz > amin * amin)) emit = 0;
    }
    if (emit > ar.maxv) {
        if (lane == 0) atomicOr(ar.counters + kStatus, kStFaceVerts);
        emit = 0;
    }
    if (lane == 0) ar.nverts[cell] = emit;
    if (emit) {
        for (int i = lane; i < m; i += 32) {
            ar.edges[cell * ar.maxv + i] = S.pe[buf][i];
            double *v = ar.verts + (cell * ar.maxv + i) * 3;
            v[0] = S.pv[buf][i][0]; v[1] = S.pv[buf][i][1]; v[2] = S.pv[buf][i][2];
        }
        const unsigned long long h = __ldcg(ar.hash + cell);
        // the entry point of each neighbour (the midpoint of the shared edge), one edge per lane
        float (*mid)[3] = S.mid;
        for (int i = lane; i < m; i += 32) {
            const double *p = S.pv[buf][i], *q = S.pv[buf][i + 1 == m ? 0 : i + 1];
            mid[i][0] = (float)(0.5 * (p[0] + q[0]));
            mid[i][1] = (float)(0.5 * (p[1] + q[1]));
            mid[i][2] = (float)(0.5 * (p[2] + q[2]));
        }
        __syncwarp();
        for (int i = 0; i < m; ++i) {
            const int e = S.pe[buf][i];
            if (e >= N) continue;
            insert_neighbor_warp(ar, S.key, cell, net_id, (unsigned)e, h ^ ar.zob[e], mid[i][0], mid[i][1], mid[i][2],
                                 false);
        }
    }
    return emit != 0;
}

}  // namespace

#ifndef AM_CLIP_MIN_BLOCKS
#define AM_CLIP_MIN_BLOCKS 3
#endif
// ---- the clip of a level
//
// What bounds it is instruction issue and fetch: 24 warps per SM run different cells through different parts
// of the code, and above 32 KB of it an SM sub-partition fetches one instruction every two cycles (above
// 128 KB, one every six).  So the code is short (40 KB, 141 before), its loops rolled, and the work per
// (row, vertex) pair is four FMAs and a maximum.  The polygon lives in the warp's registers, one vertex
// per lane, and the pushes of all edges probe the hash table at once.  Per mesh: 3-[256]x8-1 (1.63 M
// faces, learned candidates) 71.5 -> 33.3 ms, a decoder (3+256)-[128]x8-1 (884,000 faces) 29.2 -> 12.3 ms,
// 3-[60]x6-1 (72,000 faces) 2.6 -> 1.3 ms.  The rows read twice are 32.8 KB of hi words per cell at N = 2048:
// 107 GB of the first mesh, 16 ms at the measured copy bandwidth.

constexpr int kRing = 32;         // polygon vertices: one per lane
constexpr int kFlag = 64;         // rows per check that the maximum test may hand to the exact one

struct ClipSh {
    double pv[kRing][3];          // FP64 vertices
    double e64[kRing][4];         // the edges' rows in FP64
    float4 vf[kRing];             // FP32 vertices and the vertex term of the check's bound
    int pe[kRing];                // edge planes (edge i: vertex i -> i + 1)
    int flag[kFlag];              // rows of the exact test
    int viol[32];                 // violated rows
    int nflag, nviol;
    double aF[4];
    unsigned key[2 * kWMaxKw];    // the cell's key as 32-bit words (pushes copy it)
};

__device__ __forceinline__ float rsqrt_approx(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// hi words of row k: memory, or a box row
__device__ __forceinline__ float4 clip_row(const float4 *p, int N, float box, int k)
{
    if (k < N) return __ldg(p + k);
    const int i = k - N;
    const float sg = (i & 1) ? -1.0f : 1.0f;
    return make_float4((i >> 1) == 0 ? sg : 0.0f, (i >> 1) == 1 ? sg : 0.0f, (i >> 1) == 2 ? sg : 0.0f, -box);
}

// The face plane's frame about the entry point e: coordinates (u . (x - e), w . (x - e)).  line: row r there
// as a unit normal and an offset, (0, 0, -1) when it is (nearly) parallel to the plane.
struct PlaneFrame {
    float u0, u1, u2, w0, w1, w2, ex, ey, ez;
    __device__ __forceinline__ void set(float f0, float f1, float f2)
    {
        const float inv = rsqrtf(f0 * f0 + f1 * f1 + f2 * f2);
        const float n0 = f0 * inv, n1 = f1 * inv, n2 = f2 * inv;
        const float ax = fabsf(n0), ay = fabsf(n1), az = fabsf(n2);
        const int ei = (ax <= ay && ax <= az) ? 0 : (ay <= az ? 1 : 2);
        u0 = ei == 0 ? 0.0f : (ei == 1 ? -n2 : n1);       // u = n x e_i, w = n x u
        u1 = ei == 0 ? n2 : (ei == 1 ? 0.0f : -n0);
        u2 = ei == 0 ? -n1 : (ei == 1 ? n0 : 0.0f);
        const float un = rsqrtf(u0 * u0 + u1 * u1 + u2 * u2);
        u0 *= un; u1 *= un; u2 *= un;
        w0 = n1 * u2 - n2 * u1; w1 = n2 * u0 - n0 * u2; w2 = n0 * u1 - n1 * u0;
    }
    __device__ __forceinline__ float3 line(const float4 r) const
    {
        const float A = r.x * u0 + r.y * u1 + r.z * u2, B = r.x * w0 + r.y * w1 + r.z * w2, q2 = A * A + B * B;
        const bool on = q2 > 1e-10f * (r.x * r.x + r.y * r.y + r.z * r.z);
        const float q = on ? rsqrt_approx(q2) : 0.0f;
        return make_float3(A * q, B * q, on ? fmaf(r.x, ex, fmaf(r.y, ey, fmaf(r.z, ez, r.w))) * q : -1.0f);
    }
};

// One row of the exact test: its FP32 value against the bound at every vertex that is not its own, close
// calls in FP64 from the exact pair.  Returns 1 when violated, 2 when FP64 cannot decide or it is an
// edge that is violated elsewhere, 0 when it holds; *close counts the FP64 evaluations.  Out of line:
// a cell has it for its edges' rows and one row in a few cells.
__device__ __noinline__ int clip_exact_row(ClipSh &S, const float4 *p, int N, float box, float box_lo, int k, int m,
                                           float delta, int *close)
{
    const float4 r = clip_row(p, N, box, k);
    const float rl1 = fabsf(r.x) + fabsf(r.y) + fabsf(r.z);
    const float band = delta * sqrtf(r.x * r.x + r.y * r.y + r.z * r.z);      // delta |r|: the tolerance band
    const float cr = __fmaf_ru(8.5f * kWU, fabsf(r.w), band);
    bool viol = false, amb = false, edge = false;
    int ea = S.pe[m - 1];
#pragma unroll 1
    for (int i = 0; i < m; ++i) {
        const int eb = S.pe[i];
        const bool own = k == ea || k == eb;
        edge |= k == eb;
        ea = eb;
        if (own) continue;
        const float4 V = S.vf[i];
        const float sl = fmaf(r.x, V.x, fmaf(r.y, V.y, fmaf(r.z, V.z, r.w)));
        const float B = __fmaf_ru(rl1, V.w, cr);
        if (sl < -B) continue;
        if (sl > B) { viol = true; continue; }
        ++*close;
        const float4 l = k < N ? __ldg(p + (N + 1) + k) : make_float4(0.0f, 0.0f, 0.0f, -box_lo);
        const double r0 = (double)r.x + (double)l.x, r1 = (double)r.y + (double)l.y, r2 = (double)r.z + (double)l.z,
                     r3 = (double)r.w + (double)l.w;
        const double *v6 = S.pv[i];
        const double s6 = r0 * v6[0] + r1 * v6[1] + r2 * v6[2] + r3;
        const double m6 = fabs(r0 * v6[0]) + fabs(r1 * v6[1]) + fabs(r2 * v6[2]) + fabs(r3);
        const float X = fmaxf(1.0f, fmaxf(fabsf(V.x), fmaxf(fabsf(V.y), fabsf(V.z)))) * 1.0001f;
        const double B6 = (double)rl1 * 1.0001 * (double)(4e-16f * X * 1.01f) + (double)band + 1e-15 * m6;
        if (s6 > B6) viol = true;
        else if (!(s6 < -B6)) amb = true;
    }
    return amb || (viol && edge) ? 2 : (viol ? 1 : 0);
}

// whether the FP64 polygon's area exceeds the smallest kept one (a fan about vertex 0 summed over the
// lanes); out of line: FP32 decides all but degenerate faces
__device__ __noinline__ bool clip_area(const ClipSh &S, int m, double box)
{
    const int lane = threadIdx.x & 31;
    const double *p0 = S.pv[0];
    double nx = 0.0, ny = 0.0, nz = 0.0;
    if (lane >= 1 && lane < m - 1) {
        const double *p = S.pv[lane], *q = S.pv[lane + 1];
        const double ax = p[0] - p0[0], ay = p[1] - p0[1], az = p[2] - p0[2];
        const double bx = q[0] - p0[0], by = q[1] - p0[1], bz = q[2] - p0[2];
        nx = ay * bz - az * by; ny = az * bx - ax * bz; nz = ax * by - ay * bx;
    }
    nx = warp_sum(nx); ny = warp_sum(ny); nz = warp_sum(nz);
    const double amin = 2e-24 * box * box;            // twice the smallest kept area
    return nx * nx + ny * ny + nz * nz > amin * amin;
}

// The ring's vertices in FP64 from its planes' exact pairs (Eq. 11, solve3's Cramer's rule): the rows as
// FP64 one lane per coefficient, the vertices one lane per coordinate (an FP64 warp instruction takes
// about 64 cycles for one lane as for 32: 25 of them per face instead of 110).  Also the FP32 vertices and
// the vertex term w = 8.5 u X + the vertex's own error of the check's bound.  False: a vertex is not finite.
__device__ __forceinline__ bool clip_vertices(ClipSh &S, const float4 *p, int N, float box, float box_lo, int m)
{
    const int lane = threadIdx.x & 31;
    const unsigned FULL = 0xffffffffu;
    const float *pf = reinterpret_cast<const float *>(p);
#pragma unroll 1
    for (int q = lane; q < 4 * m; q += 32) {
        const int k = S.pe[q >> 2], c = q & 3, i = k - N;
        float h, l;
        if (k < N) {
            h = __ldg(pf + 4 * k + c);
            l = __ldg(pf + 4 * (N + 1 + k) + c);
        } else {
            h = c == 3 ? -box : (c == (i >> 1) ? ((i & 1) ? -1.0f : 1.0f) : 0.0f);
            l = c == 3 ? -box_lo : 0.0f;
        }
        S.e64[q >> 2][c] = (double)h + (double)l;
    }
    __syncwarp();
    const int v = lane / 3, d = lane - 3 * v, d1 = d == 2 ? 0 : d + 1, d2 = d == 0 ? 2 : d - 1;
    const int l0 = 3 * v, l1 = l0 + 1, l2 = min(l0 + 2, 31);
    bool good = true;
#pragma unroll 1
    for (int b = 0; b < m; b += 10) {
        const int i = b + v;
        const bool on = v < 10 && i < m;
        const int iq = on ? i : 0, ip = iq == 0 ? m - 1 : iq - 1;
        const double *pa = S.e64[ip], *q = S.e64[iq], *f = S.aF;
        const double c0 = q[d1] * f[d2] - q[d2] * f[d1], c1 = f[d1] * pa[d2] - f[d2] * pa[d1],
                     c2 = pa[d1] * q[d2] - pa[d2] * q[d1];
        const double det = pa[0] * __shfl_sync(FULL, c0, l0) + pa[1] * __shfl_sync(FULL, c0, l1) + pa[2] * __shfl_sync(FULL, c0, l2);
        const double inv = -1.0 / det;
        const double x = (pa[3] * c0 + q[3] * c1 + f[3] * c2) * inv;
        const float xf = (float)x;
        float X = fmaxf(1.0f, fabsf(xf));
        X = fmaxf(X, fmaxf(__shfl_sync(FULL, X, l0), fmaxf(__shfl_sync(FULL, X, l1), __shfl_sync(FULL, X, l2)))) * 1.0001f;
        if (on) {
            S.pv[i][d] = x;
            reinterpret_cast<float *>(S.vf + i)[d] = xf;
            if (d == 0) S.vf[i].w = __fmaf_ru(8.5f * kWU, X, 4e-16f * X * 1.01f);
            good = good && isfinite(xf);
        }
    }
    return __all_sync(FULL, good);
}

__global__ void __launch_bounds__(kWW * 32, AM_CLIP_MIN_BLOCKS) clip_warp_kernel(const __grid_constant__ MarchArgs a)
{
    extern __shared__ __align__(16) unsigned char wsm[];
    ClipSh &S = reinterpret_cast<ClipSh *>(wsm)[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const unsigned FULL = 0xffffffffu;
    const Arena &ar = a.ar;
    unsigned n_solved = 0, n_empty = 0, n_fix = 0, n_cuts = 0, n_close = 0, n_fb = 0;
    const int64_t stride = (int64_t)gridDim.x * kWW;
    const float box = a.box_hi, delta = (float)a.delta * 1.01f;
    // with a.work the warps take cells one at a time from a shared counter (cells differ in
    // their cost: the cuts, the fix-up rounds), else in a fixed stride
    auto next = [&](int64_t cur) -> int64_t {
        if (!a.work) return cur + stride;
        unsigned long long t = 0;
        if (lane == 0) t = atomicAdd(a.work, 1ull);
        return a.begin + (int64_t)__shfl_sync(FULL, t, 0);
    };
    for (int64_t cell = a.work ? next(0) : a.begin + (int64_t)blockIdx.x * kWW + (threadIdx.x >> 5); cell < a.end;
         cell = next(cell)) {
        if (__ldcg(ar.nverts + cell) == -2) continue;          // a duplicate seed id: never solved
        const int net_id = __ldcg(ar.net + cell);
        const int N = a.nets[net_id].N;
        const float4 *p = reinterpret_cast<const float4 *>(a.rows_in) + (cell - a.begin) * 2 * (int64_t)(N + 1);
        PlaneFrame fr;
        fr.ex = __ldcg(ar.entry_pt + cell * 3); fr.ey = __ldcg(ar.entry_pt + cell * 3 + 1);
        fr.ez = __ldcg(ar.entry_pt + cell * 3 + 2);
        __syncwarp();                                    // the last cell's readers of S are done
#pragma unroll 1
        for (int w = lane; w < 2 * ar.kw; w += 32) S.key[w] = __ldcg(reinterpret_cast<const unsigned *>(ar.keys + cell * ar.kw) + w);
        if (lane < 4) S.aF[lane] = (double)reinterpret_cast<const float *>(p + N)[lane] + (double)reinterpret_cast<const float *>(p + 2 * N + 1)[lane];
        const float4 F = __ldg(p + N);
        const bool learned = a.candidates == kCandLearned && a.scores_in && a.prop.n_out == N;
        const __nv_bfloat16 *sc = learned ? a.scores_in + (cell - a.begin) * (int64_t)a.scores_ld : nullptr;
        // ---- candidates: per lane the two rows nearest to the entry point of those it scans, by the
        //      distance's bits with the scan's index (N <= 8192: below 256) in the lowest eight
        unsigned b1 = 0xffffffffu, b2 = 0xffffffffu;
        float s3 = 3.0e38f;
        int k3 = -1;
#pragma unroll 1
        for (int u0 = 0; 32 * u0 < N; u0 += 8) {
            float4 r[8];
            float q[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int k = lane + 32 * (u0 + u);
                r[u] = k < N ? __ldg(p + k) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
            if (learned) {
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int k = lane + 32 * (u0 + u);
                    q[u] = k < N ? -__bfloat162float(sc[k]) : 3.0e38f;
                }
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (q[u] < s3) { s3 = q[u]; k3 = lane + 32 * (u0 + u); }
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const float n2 = r[u].x * r[u].x + r[u].y * r[u].y + r[u].z * r[u].z;
                const float d = fabsf(fmaf(r[u].x, fr.ex, fmaf(r[u].y, fr.ey, fmaf(r[u].z, fr.ez, r[u].w)))) * rsqrt_approx(n2);
                // no normal (or no row): infinity or not a number, above every distance
                const unsigned c = n2 > 0.0f ? (__float_as_uint(d) & ~255u) | (unsigned)(u0 + u) : 0xffffffffu;
                b2 = min(b2, max(b1, c));
                b1 = min(b1, c);
            }
        }
        // slots: the nearest two (a box row in the place of the second where it is nearer) and the
        // proposal's best row
        int kk[3] = {b1 == 0xffffffffu ? -1 : lane + 32 * (int)(b1 & 255u), b2 == 0xffffffffu ? -1 : lane + 32 * (int)(b2 & 255u),
                     learned ? k3 : -1};
        if (lane < kBoxPlanes) {
            const float4 r = clip_row(p, N, box, N + lane);
            const float d = fabsf(fmaf(r.x, fr.ex, fmaf(r.y, fr.ey, fmaf(r.z, fr.ez, r.w))));
            if (kk[1] < 0 || __float_as_uint(d) < b2) kk[1] = N + lane;
        }
        if (kk[2] == kk[0] || kk[2] == kk[1]) kk[2] = -1;      // already a candidate
        fr.set(F.x, F.y, F.z);
        const float nn = F.x * F.x + F.y * F.y + F.z * F.z;
        bool fallback = !(nn > 0.0f && isfinite(nn));
        int m = 0, rounds = 0, close = 0;
        unsigned ncut = 0;
        float vx = 0.0f, vy = 0.0f;
        while (!fallback) {
            // ---- the candidate clip (FP32, in the plane): a square about the entry point, then the nearest
            //      cutting line first; a line that holds on the polygon holds on every smaller one and retires
            float cA[3], cB[3], cC[3];
            bool live[3];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                float3 L = make_float3(0.0f, 0.0f, -1.0f);
                if (kk[j] >= 0) L = fr.line(clip_row(p, N, box, kk[j]));
                cA[j] = L.x; cB[j] = L.y; cC[j] = L.z;
                live[j] = kk[j] >= 0;
            }
            // reaches past the box from any point in it; from a point outside, an edge of the square may
            // remain, which the block kernel takes
            const float sz = 2.1f * 1.7320508f * box;
            vx = (lane == 1 || lane == 2) ? sz : -sz;
            vy = lane >= 2 ? sz : -sz;
            float eA = lane == 1 ? 1.0f : (lane == 3 ? -1.0f : 0.0f), eB = lane == 0 ? -1.0f : (lane == 2 ? 1.0f : 0.0f), eC = -sz;
            int id = -1 - lane;                          // the square's edges: never the face's
            m = 4;
#pragma unroll 1
            while (true) {
                float mx[3] = {-3.0e38f, -3.0e38f, -3.0e38f};
#pragma unroll 1
                for (int i = 0; i < m; ++i) {
                    const float x = __shfl_sync(FULL, vx, i), y = __shfl_sync(FULL, vy, i);
#pragma unroll
                    for (int j = 0; j < 3; ++j) mx[j] = fmaxf(mx[j], fmaf(cA[j], x, fmaf(cB[j], y, cC[j])));
                }
                unsigned mine = 0xffffffffu;
                int slot = 0;
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    live[j] = live[j] && mx[j] > 1e-7f;
                    const unsigned c = live[j] ? __float_as_uint(fabsf(cC[j])) : 0xffffffffu;
                    if (c < mine) { mine = c; slot = j; }
                }
                const unsigned best = __reduce_min_sync(FULL, mine);
                if (best == 0xffffffffu) break;
                const int src = __ffs(__ballot_sync(FULL, mine == best)) - 1;
                const float A = __shfl_sync(FULL, slot == 0 ? cA[0] : (slot == 1 ? cA[1] : cA[2]), src);
                const float B = __shfl_sync(FULL, slot == 0 ? cB[0] : (slot == 1 ? cB[1] : cB[2]), src);
                const float C = __shfl_sync(FULL, slot == 0 ? cC[0] : (slot == 1 ? cC[1] : cC[2]), src);
                const int kc = __shfl_sync(FULL, slot == 0 ? kk[0] : (slot == 1 ? kk[1] : kk[2]), src);
#pragma unroll
                for (int j = 0; j < 3; ++j)
                    if (lane == src && slot == j) live[j] = false;
                // the cut: the vertices beyond the line leave, two on it take their place
                const unsigned full = m == 32 ? FULL : (1u << m) - 1u;
                const unsigned out = __ballot_sync(FULL, lane < m && fmaf(A, vx, fmaf(B, vy, C)) > 1e-7f);
                const int nout = __popc(out);
                const unsigned first = out & ~((out << 1) | (out >> (m - 1))) & full;
                const int nin = m - nout;
                // nothing cut (rounding), or everything, or more than one run, or no lane left
                if (nout == 0) continue;
                if (nin == 0 || __popc(first) != 1 || nin + 2 > kRing) { fallback = true; break; }
                const int ia = __ffs(first) - 1;
                int ib = ia + nout - 1;
                if (ib >= m) ib -= m;
                // lane q takes the q-th kept vertex after the run; then the run's two ends with their edges
                int from = ib + 1 + lane;
                if (from >= m) from -= m;
                if (lane == nin) from = ia == 0 ? m - 1 : ia - 1;
                if (lane == nin + 1) from = ib;
                from &= 31;
                vx = __shfl_sync(FULL, vx, from); vy = __shfl_sync(FULL, vy, from);
                eA = __shfl_sync(FULL, eA, from); eB = __shfl_sync(FULL, eB, from); eC = __shfl_sync(FULL, eC, from);
                id = __shfl_sync(FULL, id, from);
                if (lane == nin || lane == nin + 1) {
                    const float D = __fdividef(1.0f, eA * B - eB * A);
                    vx = (eB * C - B * eC) * D;
                    vy = (A * eC - eA * C) * D;
                    if (lane == nin) { eA = A; eB = B; eC = C; id = kc; }
                }
                m = nin + 2;
                ++ncut;
            }
            if (fallback) break;
            // a square's edge left (an open polygon), or one that FP32 emptied, proves nothing
            if (__any_sync(FULL, lane < m && (id < 0 || !isfinite(vx) || !isfinite(vy)))) { fallback = true; break; }
            if (lane < m) S.pe[lane] = id;
            if (lane == 0) S.nflag = S.nviol = 0;
            __syncwarp();
            if (!clip_vertices(S, p, N, box, a.box_lo, m)) { fallback = true; break; }
            __syncwarp();
            if (a.chk && m <= kChkMaxV) break;           // the dense check runs on the tensor cores (check_tc)
            // ---- the all-row check: per row the largest of its value plus its bound over the vertices (the
            //      bound |r|_1 w + c_r with c_r = 11 u |r_3| + delta |r|_1: rounding of the sum included);
            //      below zero the row holds everywhere, else the exact test takes it
#pragma unroll 1
            for (int k0 = lane; k0 < N; k0 += 32 * 4) {
                float4 r[4];
                float l1[4], c0[4], mx[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int k = k0 + 32 * u;
                    r[u] = k < N ? __ldg(p + k) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    l1[u] = (fabsf(r[u].x) + fabsf(r[u].y) + fabsf(r[u].z)) * 1.3f;
                    // a zero normal (a constant row, which holds in its own cell) or no row
                    c0[u] = l1[u] > 0.0f ? r[u].w + fmaf(11.0f * kWU, fabsf(r[u].w), delta * l1[u]) : -3.0e38f;
                    mx[u] = -3.0e38f;
                }
#pragma unroll 1
                for (int i = 0; i < m; ++i) {
                    const float4 V = S.vf[i];
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        mx[u] = fmaxf(mx[u], fmaf(r[u].x, V.x, fmaf(r[u].y, V.y, fmaf(r[u].z, V.z, fmaf(l1[u], V.w, c0[u])))));
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (!(mx[u] < 0.0f)) {
                        const int q = atomicAdd(&S.nflag, 1);
                        if (q < kFlag) S.flag[q] = k0 + 32 * u;
                    }
            }
            if (lane < kBoxPlanes) {                     // the box's rows: coordinate +-x, y, z against the box
                float mx = -3.0e38f;
#pragma unroll 1
                for (int i = 0; i < m; ++i) {
                    const float x = reinterpret_cast<const float *>(S.vf + i)[lane >> 1], w = S.vf[i].w;
                    mx = fmaxf(mx, ((lane & 1) ? -x : x) - box + fmaf(1.3f, w, 11.0f * kWU * box + delta));
                }
                if (!(mx < 0.0f)) {
                    const int q = atomicAdd(&S.nflag, 1);
                    if (q < kFlag) S.flag[q] = N + lane;
                }
            }
            __syncwarp();
            const int nf = S.nflag;
            bool amb = nf > kFlag;
#pragma unroll 1
            for (int t = lane; t < min(nf, kFlag); t += 32) {
                const int k = S.flag[t];
                const int c = clip_exact_row(S, p, N, box, a.box_lo, k, m, delta, &close);
                amb |= c == 2;
                if (c == 1) {
                    const int q = atomicAdd(&S.nviol, 1);
                    if (q < 32) S.viol[q] = k;
                    else amb = true;
                }
            }
            if (__any_sync(FULL, amb)) { fallback = true; break; }
            __syncwarp();
            const int nv = S.nviol;
            if (nv == 0) break;
            if (++rounds >= kWMaxFix) { fallback = true; break; }
            // another round: the edges and the violated rows
            kk[0] = lane < m ? id : -1;
            kk[1] = lane < nv ? S.viol[lane] : -1;
            kk[2] = -1;
            __syncwarp();
        }
        if (!fallback && a.chk && m <= kChkMaxV) {
            // the dense check runs on the tensor cores (check_tc); the finish pass emits the cell
            n_cuts += ncut;
            unsigned long long q = 0;
            if (lane == 0) q = atomicAdd(a.chk_count, 1ull);
            q = __shfl_sync(FULL, q, 0);
            CheckRec &R = a.chk[q];
            if (lane == 0) { R.cell = (int32_t)cell; R.m = m; }
            if (lane < m) {
                R.pe[lane] = S.pe[lane];
                R.v[lane][0] = S.pv[lane][0]; R.v[lane][1] = S.pv[lane][1]; R.v[lane][2] = S.pv[lane][2];
            }
            continue;
        }
        if (fallback) {
            // the block kernel solves this cell (double-float, then FP64 where needed)
            if (lane == 0) {
                const unsigned long long q = atomicAdd(a.fb_count, 1ull);
                a.fb_list[q] = (int32_t)cell;
            }
            n_fb += 1;
            continue;
        }
        // ---- a6 emit: the face's area in FP32 where that is clear of every rounding, else in FP64
        int emit = area_clear(S.vf[0], S.vf[m / 3], S.vf[2 * m / 3], area_min(a.box_hi)) || clip_area(S, m, a.box) ? m : 0;
        if (emit > ar.maxv) {
            if (lane == 0) atomicOr(ar.counters + kStatus, kStFaceVerts);
            emit = 0;
        }
        if (lane == 0) ar.nverts[cell] = emit;
        n_solved += 1;
        if (!emit) n_empty += 1;
        if (rounds) n_fix += 1;
        n_cuts += ncut;
        n_close += (unsigned)close;                      // per lane, summed at the end
        if (!emit) continue;
#pragma unroll 1
        for (int i = lane; i < 3 * m; i += 32) ar.verts[cell * ar.maxv * 3 + i] = (&S.pv[0][0])[i];
        const int e = lane < m ? S.pe[lane] : N;
        if (lane < m) ar.edges[cell * ar.maxv + lane] = e;
        // ---- a7 march: each neuron edge pushes its neighbour, entered at the shared edge's midpoint
        const float4 v0 = S.vf[lane < m ? lane : 0], v1 = S.vf[lane + 1 < m ? lane + 1 : 0];
        insert_neighbors_level(ar, S.key, cell, net_id, e < N, (unsigned)e, __ldcg(ar.hash + cell) ^ (e < N ? __ldg(ar.zob + e) : 0ull),
                               0.5f * (v0.x + v1.x), 0.5f * (v0.y + v1.y), 0.5f * (v0.z + v1.z));
    }
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1) n_close += __shfl_xor_sync(FULL, n_close, o);
    if (lane == 0) {
        unsigned long long *C = ar.counters;
        if (n_solved) atomicAdd(C + kSolved, (unsigned long long)n_solved);
        if (n_empty) atomicAdd(C + kEmpty, (unsigned long long)n_empty);
        if (n_fix) atomicAdd(C + kFixups, (unsigned long long)n_fix);
        if (n_cuts) atomicAdd(C + kCuts, (unsigned long long)n_cuts);
        if (n_close) atomicAdd(C + kCloseCalls, (unsigned long long)n_close);
        if (n_fb) atomicAdd(C + kWarpFallback, (unsigned long long)n_fb);
    }
}

// After check_tc: one warp per record.  A cell whose rows all hold is emitted and pushes its
// neighbours; a cell with a violated or undecided row gets the warp's own check (violators cut in,
// FP64 close calls), and what that cannot decide goes to the block kernel's list.
__global__ void __launch_bounds__(kWW * 32) clip_warp_finish_kernel(MarchArgs a)
{
    extern __shared__ __align__(16) unsigned char wsm[];
    WarpSh &S = reinterpret_cast<WarpSh *>(wsm)[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const Arena &ar = a.ar;
    unsigned long long n_solved = 0, n_empty = 0, n_fix = 0, n_cuts = 0, n_close = 0, n_fb = 0;
    const int64_t n = (int64_t)__ldcg(a.chk_count);
    const int64_t stride = (int64_t)gridDim.x * kWW;
    for (int64_t idx = (int64_t)blockIdx.x * kWW + (threadIdx.x >> 5); idx < n; idx += stride) {
        const CheckRec &R = a.chk[idx];
        const int64_t cell = R.cell;
        int m = R.m, buf = 0, rounds = 0, ncut = 0, cell_close = 0;
        const int net_id = __ldcg(ar.net + cell);
        const int N = a.nets[net_id].N;
        bool fallback = false;
        if (a.chk_status[idx] == 0) {
            wload_key(S, ar, cell);
        } else {
            WRows rv;
            wcell_setup(a, S, cell, N, rv);
            for (int i = lane; i < m; i += 32) {
                S.pe[0][i] = R.pe[i];
            }
            __syncwarp();
            fallback = !wfinal(S, m, 0, rv);                    // the same FP64 vertices and their bounds
            if (!fallback) fallback = wcheck(a, S, rv, N, m, buf, rounds, ncut, cell_close);
        }
        if (fallback) {
            if (lane == 0) {
                const unsigned long long p = atomicAdd(a.fb_count, 1ull);
                a.fb_list[p] = (int32_t)cell;
            }
            n_fb += 1;
            continue;
        }
        if (a.chk_status[idx] == 0) {
            for (int i = lane; i < m; i += 32) {
                S.pe[0][i] = R.pe[i];
                S.pv[0][i][0] = R.v[i][0]; S.pv[0][i][1] = R.v[i][1]; S.pv[0][i][2] = R.v[i][2];
            }
        }
        __syncwarp();
        const bool emitted = wemit(a, S, cell, net_id, N, m, buf);
        n_solved += 1;
        if (!emitted) n_empty += 1;
        if (rounds) n_fix += 1;
        n_cuts += (unsigned long long)ncut;
        n_close += (unsigned long long)cell_close;
        __syncwarp();
    }
    if (lane == 0) {
        unsigned long long *C = ar.counters;
        if (n_solved) atomicAdd(C + kSolved, n_solved);
        if (n_empty) atomicAdd(C + kEmpty, n_empty);
        if (n_fix) atomicAdd(C + kFixups, n_fix);
        if (n_cuts) atomicAdd(C + kCuts, n_cuts);
        if (n_close) atomicAdd(C + kCloseCalls, n_close);
        if (n_fb) atomicAdd(C + kWarpFallback, n_fb);
    }
}

static int clip_smem_bytes() { return kWW * (int)sizeof(ClipSh); }

static int g_clip_resident = 0;       // clip_warp_kernel blocks resident on the whole GPU at once

cudaError_t prepare_clip_warp()
{
    cudaError_t e = cudaFuncSetAttribute(clip_warp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, clip_smem_bytes());
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(clip_warp_finish_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, warp_smem_bytes());
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0, per_sm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, clip_warp_kernel, kWW * 32, clip_smem_bytes());
    if (e != cudaSuccess) return e;
    g_clip_resident = std::max(1, sms * per_sm);
    return cudaSuccess;
}

void launch_clip_warp(const MarchArgs &a, cudaStream_t st)
{
    const int64_t n = a.end - a.begin;
    // with a work counter: one resident wave that drains the cells; else one warp per cell
    const int64_t cap = a.work && g_clip_resident > 0 ? g_clip_resident : 152 * 64;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((n + kWW - 1) / kWW, cap));
    clip_warp_kernel<<<grid, kWW * 32, clip_smem_bytes(), st>>>(a);
}

void launch_clip_warp_finish(const MarchArgs &a, cudaStream_t st)
{
    const int64_t n = a.end - a.begin;                 // the records are at most the cells
    const int grid = (int)std::min<int64_t>((n + kWW - 1) / kWW, 152 * 16);
    clip_warp_finish_kernel<<<grid, kWW * 32, warp_smem_bytes(), st>>>(a);
}

}  // namespace am
