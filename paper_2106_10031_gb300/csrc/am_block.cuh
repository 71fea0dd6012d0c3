// am_block.cuh -- block-wide primitives (scan, compaction, reductions) and the cell
// hash-table insert used by the marching kernels.
#pragma once

#include "am_common.cuh"

namespace am {

constexpr int kMaxProbe = 1 << 16;   // hash probe limit per insert (a bounded loop)

// Exclusive block scan of one int per thread.  wsum: shared scratch of 32 ints.  Every
// thread of the block must call it.  *total receives the block sum.
__device__ __forceinline__ int block_scan_excl(int v, int *wsum, int *total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int s = lane < nw ? wsum[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < nw) wsum[lane] = s;
    }
    __syncthreads();
    const int base = wid ? wsum[wid - 1] : 0;
    *total = wsum[nw - 1];
    __syncthreads();
    return base + x - v;
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Block argmax of (value, index): the larger value wins, ties go to the smaller index.
// idx < 0 marks "no candidate".  red_v/red_i: shared scratch of 32 entries each.
__device__ __forceinline__ void block_argmax(double v, int idx, double *red_v, int *red_i, double *out_v,
                                             int *out_i)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        double v2 = __shfl_xor_sync(0xffffffffu, v, o);
        int i2 = __shfl_xor_sync(0xffffffffu, idx, o);
        bool take = (i2 >= 0) && (idx < 0 || v2 > v || (v2 == v && i2 < idx));
        if (take) { v = v2; idx = i2; }
    }
    if (lane == 0) { red_v[wid] = v; red_i[wid] = idx; }
    __syncthreads();
    if (wid == 0) {
        v = lane < nw ? red_v[lane] : 0.0;
        idx = lane < nw ? red_i[lane] : -1;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            double v2 = __shfl_xor_sync(0xffffffffu, v, o);
            int i2 = __shfl_xor_sync(0xffffffffu, idx, o);
            bool take = (i2 >= 0) && (idx < 0 || v2 > v || (v2 == v && i2 < idx));
            if (take) { v = v2; idx = i2; }
        }
        if (lane == 0) { red_v[0] = v; red_i[0] = idx; }
    }
    __syncthreads();
    *out_v = red_v[0];
    *out_i = red_i[0];
    __syncthreads();
}

constexpr int kNoPool = 1 << 30;       // pooling bit range of a net without pooling

// Word w of the key reached from key word x by crossing plane `flip` (kNoFlip: none).  A unit's
// plane flips its bit (Alg. 1 step 10); a pooling plane of a max-pooled net (pool0 <= flip < pool1,
// Sec. 5.2) moves the one-hot pooled index, bits pool0 .. pool1 - 1, to flip.
__device__ __forceinline__ unsigned long long child_word(unsigned long long x, int w, unsigned flip, int pool0,
                                                         int pool1)
{
    if (flip == kNoFlip) return x;
    if ((int)flip >= pool0 && (int)flip < pool1) {
        const int lo = max(pool0 - 64 * w, 0), hi = min(pool1 - 64 * w, 64);
        if (lo < hi) x &= ~((hi >= 64 ? ~0ull : ((1ull << hi) - 1ull)) & ~((1ull << lo) - 1ull));
        if ((int)(flip >> 6) == w) x |= 1ull << (flip & 63);
        return x;
    }
    if ((int)(flip >> 6) == w) x ^= 1ull << (flip & 63);
    return x;
}

// Twice the smallest kept area (1e-24 box^2) from above, for area_clear (in FP32: the FP64 pipe is a scarce one)
__device__ __forceinline__ float area_min(float box) { return fmaxf(2e-24f * box * box * 1.0001f, 1e-30f); }

// Whether a face is larger than the smallest kept one beyond every rounding: the triangle of three of its
// vertices lies in it.  p, q, r are the vertices in FP32, each coordinate within u |v|_inf (u = 2^-24, X the
// largest coordinate) of the FP64 one that the area rule reads, so a side's coordinate is off by
// d <= 4.1 u X, a component of the cross product by d (|a|_1 + |b|_1) + 2 d^2 and its own rounding, at most
// 3 u X (|a|_1 + |b|_1): below 12 u X (|a|_1 + |b|_1) wherever the component exceeds that (2 d^2 = 34 u^2 X^2
// matters only for sides of that size, whose product is smaller).  False: FP64 decides, from the FP64 vertices.
// Nothing here is a length of its own, so it holds in a box of any size; three vertices cost less than the
// sum over all edges (no reduction over the lanes).
__device__ __forceinline__ bool area_clear(const float4 p, const float4 q, const float4 r, float amin)
{
    const float ax = q.x - p.x, ay = q.y - p.y, az = q.z - p.z, bx = r.x - p.x, by = r.y - p.y, bz = r.z - p.z;
    const float c = fmaxf(fabsf(ay * bz - az * by), fmaxf(fabsf(az * bx - ax * bz), fabsf(ax * by - ay * bx)));
    const float s = fabsf(ax) + fabsf(ay) + fabsf(az) + fabsf(bx) + fabsf(by) + fabsf(bz);
    const float X = fmaxf(fmaxf(fmaxf(fabsf(p.x), fabsf(p.y)), fmaxf(fabsf(p.z), fabsf(q.x))),
                          fmaxf(fmaxf(fabsf(q.y), fabsf(q.z)), fmaxf(fmaxf(fabsf(r.x), fabsf(r.y)), fabsf(r.z))));
    return c > fmaf(12.0f * 5.9604645e-8f * X, s, amin);
}

// the words of two keys a and b crossed at fa and fb, compared (max-pooled nets; out of line)
static __device__ __noinline__ unsigned long long pooled_diff(unsigned long long a, unsigned long long b, int w, unsigned fa,
                                                       unsigned fb, int pool0, int pool1)
{
    return child_word(a, w, fa, pool0, pool1) ^ child_word(b, w, fb, pool0, pool1);
}

// key(pa) crossed at fa == key(pb) crossed at fb ?  (kNoFlip = nothing crossed)
// Keys written by other blocks of a running kernel are read through L2 (ld.global.cg): the
// SM's L1 is not coherent with other SMs' writes and may hold a stale copy of the line.
__device__ __forceinline__ bool ref_keys_equal(const Arena &ar, int64_t pa, unsigned fa, int64_t pb, unsigned fb,
                                               int pool0 = kNoPool, int pool1 = kNoPool)
{
    const unsigned long long *ka = ar.keys + pa * ar.kw, *kb = ar.keys + pb * ar.kw;
    for (int w = 0; w < ar.kw; ++w) {
        const unsigned long long x = child_word(__ldcg(ka + w), w, fa, pool0, pool1) ^
                                     child_word(__ldcg(kb + w), w, fb, pool0, pool1);
        if (x) return false;
    }
    return true;
}

// Alg. 1 steps 10-11: the neighbour across plane `flip` (hash h) is pushed unless it was seen
// before; a whole warp calls this, one neighbour per lane with `on` set.  The slot records
// (parent, flip), from which any later probe rebuilds the key, so a claim never waits for a key
// to be written.  The lanes that claimed a slot take their cell ids from one atomic, write the
// new cells' records there (key, net, hash, the crossed plane as the new cell names it, entry,
// or flip when entry < 0, and a point of the shared edge), then publish them through ready[id].
// pool0, pool1: the pooling bits of a max-pooled net (child_word).  Four words of a compared key
// are in flight at once.
__device__ __forceinline__ void insert_neighbors(const Arena &ar, const unsigned *mask, int64_t parent, int net,
                                                 bool on, unsigned flip, unsigned long long h, float px, float py,
                                                 float pz, int pool0, int pool1, int entry)
{
    const int lane = threadIdx.x & 31;
    const unsigned long long mine = slot_make(h, (unsigned long long)parent, flip);
    bool claimed = false;
    if (on) {
        unsigned long long pos = h & ar.slot_mask;
        int probe = 0;
        for (; probe < kMaxProbe; ++probe) {
            const unsigned long long cur = atomicCAS(ar.slots + pos, 0ull, mine);
            if (cur == 0ull) { claimed = true; break; }
            if (slot_tag(cur) == hash_tag(h)) {
                // Keys written by other blocks of a running kernel are read through L2 (ld.global.cg):
                // the SM's L1 is not coherent with other SMs' writes
                const int64_t pb = slot_parent(cur);
                const unsigned fb = slot_flip(cur);
                const int nb = __ldcg(ar.net + pb);
                unsigned long long diff = 0ull;
#pragma unroll 1
                for (int w0 = 0; w0 < ar.kw; w0 += 4) {
                    unsigned long long kb[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) kb[q] = w0 + q < ar.kw ? __ldcg(ar.keys + pb * ar.kw + w0 + q) : 0ull;
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (w0 + q < ar.kw) {
                            // the parent's key is its state, held by the block in shared memory
                            const int w = w0 + q;
                            unsigned long long d = kb[q] ^ ((unsigned long long)mask[2 * w] | ((unsigned long long)mask[2 * w + 1] << 32));
                            if (pool0 == kNoPool) {      // two unit planes: two bits flip (fb may be kNoFlip: no word)
                                if ((int)(flip >> 6) == w) d ^= 1ull << (flip & 63);
                                if ((int)(fb >> 6) == w && fb != kNoFlip) d ^= 1ull << (fb & 63);
                                diff |= d;
                            } else {
                                diff |= pooled_diff(d ^ kb[q], kb[q], w, flip, fb, pool0, pool1);
                            }
                        }
                }
                if (nb == net && diff == 0ull) break;
            }
            pos = (pos + 1) & ar.slot_mask;
        }
        if (probe == kMaxProbe) atomicOr(ar.counters + kStatus, kStHashFull);
    }
    __syncwarp();
    const unsigned who = __ballot_sync(0xffffffffu, claimed);
    if (who == 0u) return;
    const int lead = __ffs(who) - 1;
    unsigned long long base = 0ull;
    if (lane == lead) base = atomicAdd(ar.counters + kNCells, (unsigned long long)__popc(who));
    base = __shfl_sync(0xffffffffu, base, lead);
    if (!claimed) return;
    const long long id = (long long)base + __popc(who & ((1u << lane) - 1u));
    if (id >= ar.cap) {
        atomicOr(ar.counters + kStatus, kStCellCap);
        return;
    }
    unsigned long long *kn = ar.keys + id * ar.kw;
#pragma unroll 1
    for (int w = 0; w < ar.kw; ++w) {
        const unsigned long long x = (unsigned long long)mask[2 * w] | ((unsigned long long)mask[2 * w + 1] << 32);
        kn[w] = child_word(x, w, flip, pool0, pool1);
    }
    ar.net[id] = net;
    ar.hash[id] = h;
    ar.nverts[id] = -1;
    ar.entry_plane[id] = entry >= 0 ? entry : (int32_t)flip;
    ar.parent[id] = (int32_t)parent;
    ar.entry_pt[id * 3 + 0] = px;
    ar.entry_pt[id * 3 + 1] = py;
    ar.entry_pt[id * 3 + 2] = pz;
    // publish: every write above is visible to whoever acquires the flag
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(ar.ready + id), "r"(1u) : "memory");
}

// The same pushes for the level schedule, any key width, plain nets: one neighbour per lane with `on` set.  The
// lanes probe at once (the atomics of all edges are in flight together); a key to compare is read by the
// whole warp, its words over the lanes, edge by edge.  The new cells are read only by later launches,
// after this kernel has ended, so nothing is fenced.
__device__ __forceinline__ void insert_neighbors_level(const Arena &ar, const unsigned *mask, int64_t parent, int net,
                                                       bool on, unsigned flip, unsigned long long h, float px, float py,
                                                       float pz)
{
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    const unsigned long long mine = slot_make(h, (unsigned long long)parent, flip);
    unsigned long long pos = h & ar.slot_mask;
    bool claimed = false, pending = on;
    int probe = 0;
#pragma unroll 1
    while (__any_sync(full, pending) && probe < kMaxProbe) {
        ++probe;
        unsigned long long cur = 0ull;
        if (pending) cur = atomicCAS(ar.slots + pos, 0ull, mine);
        if (pending && cur == 0ull) { claimed = true; pending = false; }
        unsigned cmp = __ballot_sync(full, pending && slot_tag(cur) == hash_tag(h));
#pragma unroll 1
        while (cmp) {
            const int src = __ffs(cmp) - 1;
            cmp &= cmp - 1;
            const unsigned long long c = __shfl_sync(full, cur, src);
            const unsigned fl = __shfl_sync(full, flip, src), fb = slot_flip(c);
            const int64_t pb = slot_parent(c);
            bool diff = lane == 0 && __ldcg(ar.net + pb) != net;
#pragma unroll 1
            for (int w = lane; w < 2 * ar.kw; w += 32) {
                unsigned d = mask[w] ^ __ldcg(reinterpret_cast<const unsigned *>(ar.keys + pb * ar.kw) + w);
                if ((int)(fl >> 5) == w) d ^= 1u << (fl & 31);
                if (fb != kNoFlip && (int)(fb >> 5) == w) d ^= 1u << (fb & 31);
                diff |= d != 0u;
            }
            diff = __any_sync(full, diff);
            if (lane == src && !diff) pending = false;        // seen before
        }
        pos = (pos + 1) & ar.slot_mask;
    }
    if (pending) atomicOr(ar.counters + kStatus, kStHashFull);
    unsigned who = __ballot_sync(full, claimed);
    if (who == 0u) return;
    const int lead = __ffs(who) - 1;
    unsigned long long base = 0ull;
    if (lane == lead) base = atomicAdd(ar.counters + kNCells, (unsigned long long)__popc(who));
    base = __shfl_sync(full, base, lead);
    const long long id = (long long)base + __popc(who & ((1u << lane) - 1u));
    if (claimed) {
        if (id >= ar.cap) {
            atomicOr(ar.counters + kStatus, kStCellCap);
        } else {
            ar.net[id] = net;
            ar.hash[id] = h;
            ar.nverts[id] = -1;
            ar.entry_plane[id] = (int32_t)flip;
            ar.parent[id] = (int32_t)parent;
            ar.entry_pt[id * 3 + 0] = px;
            ar.entry_pt[id * 3 + 1] = py;
            ar.entry_pt[id * 3 + 2] = pz;
            ar.ready[id] = 1u;
        }
    }
#pragma unroll 1
    while (who) {
        const int src = __ffs(who) - 1;
        who &= who - 1;
        const long long nid = __shfl_sync(full, id, src);
        const unsigned fl = __shfl_sync(full, flip, src);
        if (nid >= ar.cap) continue;
        unsigned *kn = reinterpret_cast<unsigned *>(ar.keys + nid * ar.kw);
#pragma unroll 1
        for (int w = lane; w < 2 * ar.kw; w += 32) kn[w] = mask[w] ^ ((int)(fl >> 5) == w ? 1u << (fl & 31) : 0u);
    }
}

// The same push by a whole warp (every lane calls it with the same arguments): lane 0 claims
// the slot and the id, the lanes copy and compare the key words in parallel.  For wide keys
// (N = 4096: 64 words) this turns 2 kw serial L2 round trips per tag hit into 2 kw / 32.
// publish = false (the level schedule: the new cell is read only by later launches, after this
// kernel has ended) skips the fence and the release store that a persistent consumer needs.
__device__ __forceinline__ void insert_neighbor_warp(const Arena &ar, const unsigned *mask, int64_t parent, int net,
                                                     unsigned flip, unsigned long long h, float px, float py,
                                                     float pz, bool publish = true, int pool0 = kNoPool,
                                                     int pool1 = kNoPool, int entry = -1)
{
    const int lane = threadIdx.x & 31;
    const unsigned long long mine = slot_make(h, (unsigned long long)parent, flip);
    unsigned long long pos = h & ar.slot_mask;
    for (int probe = 0; probe < kMaxProbe; ++probe) {
        unsigned long long cur = 0ull;
        if (lane == 0) cur = atomicCAS(ar.slots + pos, 0ull, mine);
        cur = __shfl_sync(0xffffffffu, cur, 0);
        if (cur == 0ull) {
            long long id = 0;
            if (lane == 0) id = (long long)atomicAdd(ar.counters + kNCells, 1ull);
            id = __shfl_sync(0xffffffffu, id, 0);
            if (id >= ar.cap) {
                if (lane == 0) atomicOr(ar.counters + kStatus, kStCellCap);
                return;
            }
            // the parent's key is its state, held by the block in shared memory
            unsigned long long *kn = ar.keys + id * ar.kw;
            for (int w = lane; w < ar.kw; w += 32) {
                const unsigned long long x = (unsigned long long)mask[2 * w] | ((unsigned long long)mask[2 * w + 1] << 32);
                kn[w] = child_word(x, w, flip, pool0, pool1);
            }
            if (lane == 0) {
                ar.net[id] = net;
                ar.hash[id] = h;
                ar.nverts[id] = -1;
                ar.entry_plane[id] = entry >= 0 ? entry : (int32_t)flip;
                ar.parent[id] = (int32_t)parent;
                ar.entry_pt[id * 3 + 0] = px;
                ar.entry_pt[id * 3 + 1] = py;
                ar.entry_pt[id * 3 + 2] = pz;
            }
            if (publish) {
                __threadfence();      // every lane's key words are visible device-wide ...
                __syncwarp();
                // ... before the flag that publishes them
                if (lane == 0) asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(ar.ready + id), "r"(1u) : "memory");
            } else if (lane == 0) {
                ar.ready[id] = 1u;    // visible to later launches at the kernel boundary
            }
            return;
        }
        if (slot_tag(cur) == hash_tag(h)) {
            const int64_t pb = slot_parent(cur);
            const unsigned fb = slot_flip(cur);
            if (__ldcg(ar.net + pb) == net) {
                const unsigned long long *ka = ar.keys + parent * ar.kw, *kb = ar.keys + pb * ar.kw;
                bool diff = false;
                for (int w = lane; w < ar.kw; w += 32) {
                    const unsigned long long x = child_word(__ldcg(ka + w), w, flip, pool0, pool1) ^
                                                 child_word(__ldcg(kb + w), w, fb, pool0, pool1);
                    diff |= x != 0ull;
                }
                if (!__any_sync(0xffffffffu, diff)) return;
            }
        }
        pos = (pos + 1) & ar.slot_mask;
    }
    if (lane == 0) atomicOr(ar.counters + kStatus, kStHashFull);
}

// Vertex of planes p, q and the face plane f (Eq. 11 with biases) by Cramer's rule with cross
// products; optionally the infinity norm of the inverse system matrix.
template <class R>
__device__ __forceinline__ bool solve3(const R *p, const R *q, const R *f, R *v, R *inv_norm)
{
    const R c0x = q[1] * f[2] - q[2] * f[1], c0y = q[2] * f[0] - q[0] * f[2], c0z = q[0] * f[1] - q[1] * f[0];
    const R c1x = f[1] * p[2] - f[2] * p[1], c1y = f[2] * p[0] - f[0] * p[2], c1z = f[0] * p[1] - f[1] * p[0];
    const R c2x = p[1] * q[2] - p[2] * q[1], c2y = p[2] * q[0] - p[0] * q[2], c2z = p[0] * q[1] - p[1] * q[0];
    const R det = p[0] * c0x + p[1] * c0y + p[2] * c0z;
    if (det == R(0)) return false;
    const R inv = R(-1) / det;
    v[0] = (p[3] * c0x + q[3] * c1x + f[3] * c2x) * inv;
    v[1] = (p[3] * c0y + q[3] * c1y + f[3] * c2y) * inv;
    v[2] = (p[3] * c0z + q[3] * c1z + f[3] * c2z) * inv;
    if (inv_norm) {
        const R ax = fabs(c0x) + fabs(c1x) + fabs(c2x), ay = fabs(c0y) + fabs(c1y) + fabs(c2y),
                az = fabs(c0z) + fabs(c1z) + fabs(c2z);
        *inv_norm = fmax(ax, fmax(ay, az)) * fabs(inv);
    }
    return isfinite(v[0]) && isfinite(v[1]) && isfinite(v[2]);
}

}  // namespace am
