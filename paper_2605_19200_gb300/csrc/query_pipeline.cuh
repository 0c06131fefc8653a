// query_pipeline.cuh -- the batched query as a sequence of kernels on one stream.
//
//  1. Spatial binning: each point gets the Morton code of its cell in a grid over
//     the chunk's box; a counting sort by cell yields a copy of the points in
//     which the points of a warp are neighbours, and which all later stages read.
//  2. Traversal (Algorithm 1), one packet of 64 points per warp (k_trav3; in 2D k_trav2 in
//     trav2d.cuh): the points walk the tree together; far nodes (and, in 3D, far
//     leaves) add their Taylor term (Eq. 3) to each point's accumulator.  2D leaves
//     are evaluated in place (their chord's angle) unless the point is inside the
//     leaf's box.  3D leaves that need the exact evaluation are not evaluated in the
//     traversal: the (point, leaf) pairs are appended to a work list through a
//     shared-memory buffer, one atomic per 128 pairs.  With few packets the tree is
//     split into subtrees, and the smallest queries take one warp per point (k_wide3),
//     as do points whose pairs did not fit the list.
//  3. 3D only: far pairs whose panels stop at level 0 or 1 (nearly all) read the
//     curves' query-independent node tables (k_pair_fast, k_pair_fast2: a warp's
//     pairs come in runs of one leaf); the rest take the full evaluation
//     (k_pair_eval: foot-point search, adaptive panels).  Pairs FP32 cannot resolve
//     go to the FP64 near band (one warp per pair).
//  4. Finish: value, label and status per point; points whose value lies within
//     the repair band of a half-integer, or that were flagged, are appended to
//     the FP64 repair list (warp traversal + FP64 pairs, one warp per pair).
#pragma once

#include "gwn_internal.h"
#include "kernels2d.cuh"
#include "kernels3d.cuh"
#include "far3d.cuh"
#include "pairs3d.cuh"
#include "trav2d.cuh"

namespace gwn {

// Sums that do not depend on the order of their additions (direct sum, no-alloc query): in units of
// 2^-44 (rounding 2.8e-14, where an FP32 leaf's is 1e-9 and more; a total of up to 5e5),
// what is not finite in `rest`
constexpr float kSumUnit = 17592186044416.f;  // 2^44
__device__ __forceinline__ void add_fixed(long long* sum, float* rest, int i, double v) {
    if (isfinite(v)) atomicAdd(reinterpret_cast<unsigned long long*>(&sum[i]), (unsigned long long)__double2ll_rn(v * (double)kSumUnit));
    else atomicAdd(&rest[i], (float)v);
}

constexpr int kBinBits2 = 9;   // 512 x 512 cells in 2D
constexpr int kBinBits3 = 5;   // 32^3 cells in 3D (default; the autotuner picks 4, 5 or 6 per model)
constexpr int kMaxBinCells = 1 << 18;  // 2^(2 x 9) = 2^(3 x 6)

__device__ __forceinline__ uint32_t spread_bits2(uint32_t x) {
    x &= 0x0000ffffu;
    x = (x | (x << 8)) & 0x00ff00ffu;
    x = (x | (x << 4)) & 0x0f0f0f0fu;
    x = (x | (x << 2)) & 0x33333333u;
    x = (x | (x << 1)) & 0x55555555u;
    return x;
}
__device__ __forceinline__ uint32_t spread_bits3(uint32_t x) {
    x &= 0x000003ffu;
    x = (x | (x << 16)) & 0xff0000ffu;
    x = (x | (x << 8)) & 0x0300f00fu;
    x = (x | (x << 4)) & 0x030c30c3u;
    x = (x | (x << 2)) & 0x09249249u;
    return x;
}

__device__ __forceinline__ void flush_work(const WorkLocal& wl, unsigned long long* work) {
    for (int k = 0; k < kWorkCount; ++k)
        if (wl.v[k]) atomicAdd(&work[k], wl.v[k]);
}

__device__ __forceinline__ void load_point_f(const void* pts, int dtype, int dim, long long i, float* q) {
    if (dtype == GWN_F32) {
        const float* p = reinterpret_cast<const float*>(pts) + i * dim;
        for (int k = 0; k < dim; ++k) q[k] = p[k];
    } else {
        const double* p = reinterpret_cast<const double*>(pts) + i * dim;
        for (int k = 0; k < dim; ++k) q[k] = (float)p[k];
    }
}

// order-preserving integer key of a float (larger float, larger key) and back
__device__ __forceinline__ unsigned float_key(float f) {
    const unsigned u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_float(unsigned k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// bounding box of the n points: box[0..2] receive the complemented keys of the
// minima and box[3..5] the keys of the maxima (box zeroed beforehand, so that
// atomicMax serves both), one atomic per block and coordinate
template <int DIM>
__global__ void __launch_bounds__(128) k_bbox(const void* pts, int dtype, int n, unsigned* box) {
    __shared__ unsigned sk[4][6];
    const unsigned full = 0xffffffffu;
    unsigned kmin[3] = {0u, 0u, 0u}, kmax[3] = {0u, 0u, 0u};  // complemented minima, maxima
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        float q[3] = {0, 0, 0};
        load_point_f(pts, dtype, DIM, i, q);
        for (int k = 0; k < DIM; ++k) {
            if (q[k] != q[k]) continue;  // NaN: no cell of its own
            const unsigned key = float_key(q[k]);
            kmin[k] = max(kmin[k], ~key);
            kmax[k] = max(kmax[k], key);
        }
    }
    for (int k = 0; k < 3; ++k)
        for (int off = 16; off > 0; off >>= 1) {
            kmin[k] = max(kmin[k], __shfl_xor_sync(full, kmin[k], off));
            kmax[k] = max(kmax[k], __shfl_xor_sync(full, kmax[k], off));
        }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0)
        for (int k = 0; k < 3; ++k) {
            sk[warp][k] = kmin[k];
            sk[warp][3 + k] = kmax[k];
        }
    __syncthreads();
    if (threadIdx.x < 6) {
        unsigned v = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v = max(v, sk[w][threadIdx.x]);
        if (v) atomicMax(&box[threadIdx.x], v);
    }
}

template <int DIM>
__global__ void k_bin(const void* pts, int dtype, int n, const unsigned* box, int bits, int* key, int* hist) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float q[3] = {0, 0, 0};
    load_point_f(pts, dtype, DIM, i, q);
    const float cells = (float)(1 << bits);
    // the grid spans the chunk's own box (k_bbox), so that points gathered in a
    // small part of the model's box still fall into many cells
    float l[3] = {0.f, 0.f, 0.f}, s[3] = {0.f, 0.f, 0.f};
    for (int k = 0; k < DIM; ++k) {
        l[k] = key_float(~box[k]);
        const float e = key_float(box[3 + k]) - l[k];
        s[k] = e > 0.f ? 1.f / e : 0.f;
    }
    uint32_t c[3];
    for (int k = 0; k < DIM; ++k) {
        float t = (q[k] - l[k]) * s[k] * cells;
        t = fminf(fmaxf(t, 0.f), cells - 1.f);
        c[k] = (uint32_t)t;
    }
    int code = DIM == 2 ? (int)(spread_bits2(c[0]) | (spread_bits2(c[1]) << 1))
                        : (int)(spread_bits3(c[0]) | (spread_bits3(c[1]) << 1) | (spread_bits3(c[2]) << 2));
    key[i] = code;
    atomicAdd(&hist[code], 1);
}

// Exclusive scan of hist[0..K) in place, kScanTile values per block: the blocks' sums,
// then every block scans its own tile onto the sum of the tiles before it (at most
// 64 for 2^18 cells).  One block for all of it took 340 us for the 2^18 cells of a 2D
// grid and 45 us in 3D.
constexpr int kScanTile = 4096;
__device__ __forceinline__ int warp_incl_scan(int v) {
    for (int off = 1; off < 32; off <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, off);
        if ((threadIdx.x & 31) >= off) v += u;
    }
    return v;
}
__global__ void __launch_bounds__(1024) k_scan_sums(const int* hist, int K, int* sums) {
    __shared__ int part[32];
    int v = 0;
    for (int j = 0; j < 4; ++j) {
        const int i = blockIdx.x * kScanTile + j * 1024 + threadIdx.x;
        if (i < K) v += hist[i];
    }
    v = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        v = __reduce_add_sync(0xffffffffu, part[threadIdx.x]);
        if (threadIdx.x == 0) sums[blockIdx.x] = v;
    }
}
__global__ void __launch_bounds__(1024) k_scan(int* hist, int K, const int* sums) {
    __shared__ int part[32];
    __shared__ int base;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int i = blockIdx.x * kScanTile + 4 * threadIdx.x;
    int v[4], t = 0;
    for (int j = 0; j < 4; ++j) {
        v[j] = i + j < K ? hist[i + j] : 0;
        t += v[j];
    }
    const int incl = warp_incl_scan(t);
    if (lane == 31) part[wid] = incl;
    if (wid == 0) {
        int b = 0;
        for (int j = lane; j < (int)blockIdx.x; j += 32) b += sums[j];
        b = __reduce_add_sync(0xffffffffu, b);
        if (lane == 0) base = b;
    }
    __syncthreads();
    if (wid == 0) {
        const int p = part[lane];
        part[lane] = warp_incl_scan(p) - p;
    }
    __syncthreads();
    int at = base + part[wid] + incl - t;
    for (int j = 0; j < 4; ++j) {
        if (i + j < K) hist[i + j] = at;
        at += v[j];
    }
}

// The pipeline's own copy of a chunk's points, in binned order: (x, y, z, index of
// the point in the chunk).  Every later stage -- traversal, pairs, near band -- names
// a point by its place in this copy, so that the points of a warp and of
// neighbouring pairs are neighbours in memory (one 16-byte load per point instead
// of three gathers at a permuted index, atomics into shared sectors), and only
// k_finish goes back to the caller's order.
template <int DIM>
__global__ void k_scatter_points(const void* pts, int dtype, int n, const int* key, int* cursor, float4* spos,
                                 float* wacc, uint32_t* st, long long* near) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float q[3] = {0, 0, 0};
    load_point_f(pts, dtype, DIM, i, q);
    const int pos = key ? atomicAdd(&cursor[key[i]], 1) : i;  // no key: the caller's order (few points)
    spos[pos] = make_float4(q[0], q[1], q[2], __int_as_float(i));
    if (near) near[i] = 0;
    if (DIM == 3) wacc[i] = 0.f;  // the warps of a split packet add to these
    st[i] = 0u;
}

// the first of n slots of a list of cap entries; a full list is not counted further, so
// that the count stays within 32 bits however many pairs a query has
__device__ __forceinline__ long long list_slots(int* count, int n, long long cap) {
    if (*(volatile int*)count >= cap) return cap;
    return (long long)atomicAdd(count, n);
}

constexpr int kPairBuf = 128;  // (point, leaf) pairs buffered per warp in shared memory

// write a warp's buffered pairs (n of them, warp-uniform) to the pair list with
// one atomic and coalesced stores.  If the list is full, the lanes that own the
// entries which did not fit are added to `ovf` (every lane gets the same mask);
// their points skip the pair pass and are evaluated again without the list (k_wide3).
__device__ __forceinline__ void flush_warp_pairs(const int2* buf, const unsigned char* own, int n, const Workspace& ws,
                                                 unsigned& ovf) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    long long base = 0;
    if (lane == 0 && n > 0) base = list_slots(&ws.counters[0], n, ws.pair_cap);
    base = __shfl_sync(full, base, 0);
    unsigned lost = 0;
    for (int j = lane; j < n; j += 32) {
        const long long pos = base + j;
        if (pos < ws.pair_cap) ws.pairs[pos] = buf[j];
        else lost |= 1u << own[j];
    }
    for (int off = 16; off > 0; off >>= 1) lost |= __shfl_xor_sync(full, lost, off);
    ovf |= lost;
}

// flush_warp_pairs for a packet of 64 queries: own = lane + 32 x half
__device__ __forceinline__ void flush_packet_pairs(const int2* buf, const unsigned char* own, int n, const Workspace& ws,
                                                   unsigned& ovf0, unsigned& ovf1) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    long long base = 0;
    if (lane == 0 && n > 0) base = list_slots(&ws.counters[0], n, ws.pair_cap);
    base = __shfl_sync(full, base, 0);
    unsigned lost0 = 0, lost1 = 0;
    for (int j = lane; j < n; j += 32) {
        const long long pos = base + j;
        if (pos < ws.pair_cap) ws.pairs[pos] = buf[j];
        else if (own[j] < 32) lost0 |= 1u << own[j];
        else if (own[j] < 64) lost1 |= 1u << (own[j] - 32);
    }
    if (__any_sync(full, lost0 | lost1)) {
        ovf0 |= __reduce_or_sync(full, lost0);
        ovf1 |= __reduce_or_sync(full, lost1);
    }
}

__device__ __forceinline__ bool is_dense(Dense d) { return d.found && *d.found > d.limit; }

// before a dense chunk's second walk: what the first one left
__global__ void k_dense_reset(Workspace ws, int n, Dense d) {
    if (!is_dense(d)) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        ws.wacc[i] = 0.f;
        ws.st[i] = 0u;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) ws.counters[0] = ws.counters[3] = 0;
}

// bytes of dynamic shared memory of k_trav3 (one warp) with a stack of `depth` entries
inline size_t trav3_smem(int depth) { return (size_t)depth * 12 + kPairBuf * (sizeof(int2) + 1); }

// traversal with deferred 3D leaves, one packet of 64 queries per warp, two to a
// lane: the queries (neighbours in the binned order) walk the tree together.
// The warp holds one internal node and the masks of the queries for which that
// node was near; an iteration tests both children of the node for those queries:
// far ones add the child's Taylor term, and for a leaf the ones that need it
// exactly write their pairs, for an internal child the ones for which it is near
// need its subtree.  The walk goes on into a near child and keeps the other (if
// it is near too) on a warp stack in shared memory.  A block is one warp: packets
// differ in length, and in blocks of four a long one held the others' registers
// (5.94 -> 5.37 ms on 1.3M points, 4.7k leaves).  Node and moment loads are the
// same address for the whole warp, and lanes never wait on each other's
// different branches; testing the children inline makes one loop iteration and
// at most one stack entry per near node, not one per node tested.
// What bounds it is instruction issue, and of that the part that does not depend
// on the query (loads, masks, stack, loop) is paid per packet: 64 instead of 32
// queries halve it, and the two queries of a lane share packed fp32x2 far tests and
// terms (far3_harm2), which take half the issue slots of scalar ones.
// Exact 3D leaves go to the pair list: at a leaf, the queries that need
// it exactly write their (point, leaf) pairs next to each other into the
// warp's shared-memory buffer, which is flushed to the list with one atomic
// when full, so the list comes out in runs of one leaf, each padded to an even
// length (point -1; k_pair_fast2 takes two pairs of a leaf per lane).  Every thread of the grid
// reaches the flushes (lanes past the end of the points take part with an empty
// mask).  Points whose pairs did not fit go to `olist_out` (k_wide3).
// A packet's walk is a chain of dependent loads (1 to 2 ms, however few the
// queries), so with too few packets to fill the GPU the tree is cut into gridDim.y
// subtrees, one warp per packet and subtree (cut: TreeCut): the warp first tests
// the subtree's ancestors, where the queries for which one is far drop out (its
// term is added by the first subtree below it), and the warps of a packet add up
// their sums.
// depth: entries of the warp stack (pending near siblings along the packet's
// path), chosen per model from its tree depth.  O3: the model evaluates the
// order-3 terms; COUNT: work counters (instances of their own, for the registers).
// again: the second walk of a dense chunk (d), nothing where the chunk is not dense
template <bool O3, bool COUNT>
__global__ void __launch_bounds__(32, 28) k_trav3(DevTree t, const float4* spos, int n, float beta2, float beta2l,
                                                  int depth, TreeCut cut, Workspace ws, unsigned long long* work,
                                                  int* olist_out, Dense d, bool again) {
    extern __shared__ int2 sdyn[];
    if (again && !is_dense(d)) return;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x;
    const unsigned lbit = 1u << lane;
    int2* buf = sdyn;
    int* stk_node = reinterpret_cast<int*>(sdyn + kPairBuf);
    unsigned* stk0 = reinterpret_cast<unsigned*>(stk_node + depth);
    unsigned* stk1 = stk0 + depth;
    unsigned char* own = reinterpret_cast<unsigned char*>(sdyn + kPairBuf) + (size_t)12 * depth;
    WorkLocal wl = {};
    const int q0 = blockIdx.x * 64 + lane, q1 = q0 + 32;
    const bool act0 = q0 < n, act1 = q1 < n;
    f32x2 nq[3];  // minus the two points
    {
        float4 a = make_float4(0, 0, 0, 0), b = a;
        if (act0) a = spos[q0];
        if (act1) b = spos[q1];
        nq[0] = pack2(-a.x, -b.x); nq[1] = pack2(-a.y, -b.y); nq[2] = pack2(-a.z, -b.z);
    }
    float w0 = 0.f, w1 = 0.f;
    uint32_t st0 = 0, st1 = 0;
    int bcnt = 0;                      // warp-uniform: entries in buf
    unsigned nfound = 0;               // warp-uniform: exact pairs
    unsigned ovf0 = 0, ovf1 = 0;       // queries with pairs that did not fit the list
    int sp = 0;                        // warp-uniform
    const float b2l = t.leaf_far ? beta2l : INFINITY;

    // Test node or leaf c for the queries of the masks (c and masks warp-uniform):
    // Taylor terms for the far ones, pairs for those that need a leaf
    // exactly; the masks return the queries for which an internal c is near.
    auto test = [&](int c, const float4& h, unsigned& m0, unsigned& m1, bool add) {
        const f32x2 rx = add2(pack2(h.x, h.x), nq[0]), ry = add2(pack2(h.y, h.y), nq[1]),
                    rz = add2(pack2(h.z, h.z), nq[2]);
        float ra, rb;
        unpack2(fma2(rz, rz, fma2(ry, ry, mul2(rx, rx))), ra, rb);
        const float thr = (c < 0 ? b2l : beta2) * h.w;
        const bool in0 = m0 & lbit, in1 = m1 & lbit;
        const bool f0 = in0 && ra > thr, f1 = in1 && rb > thr;
        if (COUNT && add) {
            wl.v[c < 0 ? kWorkLeafTests : kWorkNodes] += (int)in0 + (int)in1;
            wl.v[kWorkFar] += (int)f0 + (int)f1;
        }
        if (add && (f0 || f1)) {
            const int idx = c < 0 ? t.n_internal + ~c : c;
            float a, b;
            unpack2(far3_harm2<O3>(t.hmom + (size_t)idx * t.hstride, rx, ry, rz, pack2(rsqrt_hw(ra), rsqrt_hw(rb))), a, b);
            if (f0) w0 += a;
            if (f1) w1 += b;
        }
        m0 = __ballot_sync(full, in0 && !f0);
        m1 = __ballot_sync(full, in1 && !f1);
        if (c < 0) {
            const int nn = __popc(m0) + __popc(m1), even = nn + (nn & 1);
            if (nn) {
                if (bcnt + even > kPairBuf) {
                    __syncwarp();
                    flush_packet_pairs(buf, own, bcnt, ws, ovf0, ovf1);
                    bcnt = 0;
                    __syncwarp();
                }
                if (m0 & lbit) {
                    const int pos = bcnt + __popc(m0 & (lbit - 1u));
                    buf[pos] = make_int2(q0, ~c);
                    own[pos] = (unsigned char)lane;
                }
                if (m1 & lbit) {
                    const int pos = bcnt + __popc(m0) + __popc(m1 & (lbit - 1u));
                    buf[pos] = make_int2(q1, ~c);
                    own[pos] = (unsigned char)(lane + 32);
                }
                if (lane == 0 && even > nn) {
                    buf[bcnt + nn] = make_int2(-1, ~c);
                    own[bcnt + nn] = 64;
                }
                nfound += nn;
                bcnt += even;
            }
            m0 = m1 = 0u;
        }
    };

    unsigned m0 = __ballot_sync(full, act0), m1 = __ballot_sync(full, act1);
    // the subtree's ancestors, then its root
    const int4 sub = __ldg(cut.sub + blockIdx.y);  // root, first path entry, path entries
    int node = sub.x;  // warp-uniform
#pragma unroll 1
    for (int k = 0; k <= sub.z && (m0 | m1); ++k) {
        const int e = k < sub.z ? __ldg(cut.path + sub.y + k) : 0;  // 2 node + (1: this subtree adds its term)
        const int c = k < sub.z ? e >> 1 : node;
        test(c, c < 0 ? GWN_LDG(t.lhdr + ~c) : GWN_LDG(t.hdr + c), m0, m1, k == sub.z || (e & 1));
    }
    while (m0 | m1) {
        // the child indices and both children's headers, loaded together
        const int2 ch = GWN_LDG(t.child + node);
        const float4 ha = GWN_LDG(t.chdr + 2 * node), hb = GWN_LDG(t.chdr + 2 * node + 1);
        unsigned b0 = m0, b1 = m1;
        test(ch.x, ha, m0, m1, true);
        test(ch.y, hb, b0, b1, true);
        if (m0 | m1) {
            if (b0 | b1) {
                if (sp < depth) {
                    if (lane == 0) {
                        stk_node[sp] = ch.y;
                        stk0[sp] = b0;
                        stk1[sp] = b1;
                    }
                    ++sp;
                } else {  // the second subtree is dropped for these queries
                    if (b0 & lbit) st0 |= GWN_QS_STACK_OVERFLOW;
                    if (b1 & lbit) st1 |= GWN_QS_STACK_OVERFLOW;
                }
                __syncwarp();
            }
            node = ch.x;
        } else if (b0 | b1) {
            node = ch.y;
            m0 = b0;
            m1 = b1;
        } else {
            if (sp == 0) break;
            --sp;
            node = stk_node[sp];
            m0 = stk0[sp];
            m1 = stk1[sp];
            __syncwarp();
        }
    }
    __syncwarp();
    flush_packet_pairs(buf, own, bcnt, ws, ovf0, ovf1);
    if (lane == 0 && nfound) atomicAdd(ws.found + again, (unsigned long long)nfound);
    if (ovf0 & lbit) st0 |= kPairOverflow;
    if (ovf1 & lbit) st1 |= kPairOverflow;
    auto put = [&](int q, float w, uint32_t st) {
        bool listed = false;
        if (gridDim.y == 1) {
            ws.wacc[q] = w;
            ws.st[q] = st;
        } else {
            atomicAdd(&ws.wacc[q], w);
            if (st) listed = atomicOr(&ws.st[q], st) & kPairOverflow;
        }
        if ((st & kPairOverflow) && !listed) olist_out[atomicAdd(&ws.counters[3], 1)] = q;
    };
    if (act0) put(q0, w0, st0);
    if (act1) put(q1, w1, st1);
    if (COUNT) flush_work(wl, work);
}

// k_trav3 with the packet local expansion (order-2 models, query option
// local_ratio; a local-expansion far field beyond the paper): the same walk,
// and a node or leaf that every active lane of the packet needs, that passes
// the far test for every point of the packet's box (|x0 - p| > beta r + rho,
// p and rho the box's centre and half diagonal) and lies beyond kappa rho
// (kappa2 = kappa^2) is not evaluated per lane: it goes to a per-warp list,
// and 32 of them at a time each lane forms one node's second-order local
// expansion about p (far3_local2), summed over the warp; every lane evaluates
// the summed expansion at its own point at the end.  A kernel of its own:
// sharing k_trav3's body cost the plain traversal 4 % (9.16 -> 9.51 ms on a
// 2M-query model) at the same register count.
template <int STACK>
__global__ void __launch_bounds__(128) k_trav3_local(DevTree t, const float4* spos, int n, float beta2, float beta2l,
                                                     Workspace ws, unsigned long long* work, int* olist_out,
                                                     float kappa2) {
    __shared__ int2 sstk[4][STACK];
    __shared__ int2 sbuf[4][kPairBuf];
    __shared__ unsigned char sown[4][kPairBuf];
    __shared__ int slocal[4][32];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    int2* stk = sstk[threadIdx.x >> 5];
    int2* buf = sbuf[threadIdx.x >> 5];
    unsigned char* own = sown[threadIdx.x >> 5];
    int* lst = slocal[threadIdx.x >> 5];
    WorkLocal wl = {};
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const bool active = i < n;
    const int qi = active ? i : 0;
    float q[3] = {0, 0, 0};
    if (active) {
        const float4 p = spos[qi];
        q[0] = p.x; q[1] = p.y; q[2] = p.z;
    }
    float w = 0.f;
    uint32_t st = 0;
    int bcnt = 0;                      // warp-uniform: entries in buf
    unsigned nfound = 0;               // warp-uniform: exact pairs
    unsigned ovf = 0;                  // lanes with pairs that did not fit the list
    int sp = 0;                        // warp-uniform
    const unsigned amask = __ballot_sync(full, active);

    // packet box of the active lanes (centre p, half diagonal rho) and the
    // local expansion's coefficients (F, grad F, Hessian), the same in all lanes
    float pc[3] = {0.f, 0.f, 0.f}, rho = 0.f, lc[10];
    int lcnt = 0;  // warp-uniform: entries in lst
    {
        float d2 = 0.f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            float lo = active ? q[k] : 3.0e38f, hi = active ? q[k] : -3.0e38f;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                lo = fminf(lo, __shfl_xor_sync(full, lo, off));
                hi = fmaxf(hi, __shfl_xor_sync(full, hi, off));
            }
            pc[k] = 0.5f * (lo + hi);
            d2 += (hi - lo) * (hi - lo);
        }
        rho = 0.5f * sqrtf(d2);
#pragma unroll
        for (int k = 0; k < 10; ++k) lc[k] = 0.f;
    }
    // every lane takes one listed node's expansion, and the warp sums them
    auto flush_local = [&]() {
        float v[10];
#pragma unroll
        for (int k = 0; k < 10; ++k) v[k] = 0.f;
        __syncwarp();
        if (lane < lcnt) {
            const int c = lst[lane];
            const float4 h = c < 0 ? GWN_LDG(t.lhdr + ~c) : GWN_LDG(t.hdr + c);
            const float4* M = c < 0 ? t.lmom + (size_t)(~c) * kMom3Vec : t.mom + (size_t)c * kMom3Vec;
            far3_local2(M, h.x - pc[0], h.y - pc[1], h.z - pc[2], v);
        }
#pragma unroll
        for (int k = 0; k < 10; ++k) {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) v[k] += __shfl_xor_sync(full, v[k], off);
            lc[k] += v[k];
        }
        lcnt = 0;
        __syncwarp();
    };
    // c is far for the whole packet box and beyond kappa rho: list it (true)
    auto packet_far = [&](int c, unsigned msk, const float4& h, float b2) -> bool {
        if (msk != amask) return false;
        const float dx = h.x - pc[0], dy = h.y - pc[1], dz = h.z - pc[2];
        const float dd = dx * dx + dy * dy + dz * dz;
        const float lim = sqrtf(b2 * h.w) + rho;
        if (!(dd > kappa2 * rho * rho && dd > lim * lim)) return false;
        if (lane == 0) lst[lcnt] = c;
        if (work && ((amask >> lane) & 1u)) wl.v[kWorkLocal] += 1;
        if (++lcnt == 32) flush_local();
        return true;
    };

    // Test node or leaf c for the lanes of `msk` (warp-uniform c and msk):
    // Taylor terms for the far lanes, pairs for the lanes that need a leaf
    // exactly; returns the lanes for which an internal c is near.
    auto test = [&](int c, unsigned msk) -> unsigned {
        const bool mine = (msk >> lane) & 1u;
        if (c < 0) {
            const int li = ~c;
            const float4 h = GWN_LDG(t.lhdr + li);
            if (work && mine) wl.v[kWorkLeafTests] += 1;
            if (t.leaf_far && packet_far(c, msk, h, beta2l)) return 0u;
            const float rx = h.x - q[0], ry = h.y - q[1], rz = h.z - q[2];
            const bool far = mine && t.leaf_far && rx * rx + ry * ry + rz * rz > beta2l * h.w;
            if (far) {
                if (work) wl.v[kWorkFar] += 1;
                w += far3_node32(t.lmom + (size_t)li * kMom3Vec, rx, ry, rz, false);
            }
            const unsigned need = __ballot_sync(full, mine && !far);
            if (need) {
                const int nn = __popc(need);
                if (bcnt + nn > kPairBuf) {
                    __syncwarp();
                    flush_warp_pairs(buf, own, bcnt, ws, ovf);
                    bcnt = 0;
                    __syncwarp();
                }
                if ((need >> lane) & 1u) {
                    const int pos = bcnt + __popc(need & ((1u << lane) - 1u));
                    buf[pos] = make_int2(qi, li);
                    own[pos] = (unsigned char)lane;
                }
                nfound += nn;
                bcnt += nn;
            }
            return 0u;
        }
        const float4 h = GWN_LDG(t.hdr + c);
        if (work && mine) wl.v[kWorkNodes] += 1;
        if (packet_far(c, msk, h, beta2)) return 0u;
        const float rx = h.x - q[0], ry = h.y - q[1], rz = h.z - q[2];
        const bool far = mine && rx * rx + ry * ry + rz * rz > beta2 * h.w;
        if (far) {
            if (work) wl.v[kWorkFar] += 1;
            w += far3_node32(t.mom + (size_t)c * kMom3Vec, rx, ry, rz, false);
        }
        return __ballot_sync(full, mine && !far);
    };

    int node = t.root;  // warp-uniform
    unsigned mask = __ballot_sync(full, active);
    if (mask) mask = test(node, mask);  // the root itself (a leaf when the model has one)
    while (mask) {
        const int2 ch = GWN_LDG(t.child + node);
        const unsigned na = test(ch.x, mask);
        const unsigned nb = test(ch.y, mask);
        if (na) {
            if (nb) {
                if (sp < STACK) {
                    if (lane == 0) stk[sp] = make_int2(ch.y, (int)nb);
                    ++sp;
                } else if ((nb >> lane) & 1u) {
                    st |= GWN_QS_STACK_OVERFLOW;  // the second subtree is dropped for these lanes
                }
                __syncwarp();
            }
            node = ch.x;
            mask = na;
        } else if (nb) {
            node = ch.y;
            mask = nb;
        } else {
            if (sp == 0) break;
            --sp;
            const int2 e = stk[sp];
            node = e.x;
            mask = (unsigned)e.y;
            __syncwarp();
        }
    }
    {
        if (lcnt > 0) flush_local();
        // F(D - s) ~ F - grad F . s + s^T H s / 2, s = q - p
        const float sx = q[0] - pc[0], sy = q[1] - pc[1], sz = q[2] - pc[2];
        w += lc[0] - (lc[1] * sx + lc[2] * sy + lc[3] * sz) +
             0.5f * (lc[4] * sx * sx + lc[5] * sy * sy + lc[6] * sz * sz) + lc[7] * sx * sy + lc[8] * sx * sz +
             lc[9] * sy * sz;
    }
    __syncwarp();
    flush_warp_pairs(buf, own, bcnt, ws, ovf);
    if ((ovf >> lane) & 1u) st |= kPairOverflow;
    if (active) {
        ws.wacc[qi] = w;
        ws.st[qi] = st;
        if (st & kPairOverflow) olist_out[atomicAdd(&ws.counters[3], 1)] = qi;
    }
    if (lane == 0 && nfound) atomicAdd(ws.found, (unsigned long long)nfound);
    if (work) flush_work(wl, work);
}

}  // namespace gwn
#include "few3d.cuh"  // the packet walk and pair kernels of a handful of points
namespace gwn {

// One warp per query: the traversal and the far exact leaves of a query spread over
// the lanes.  Used for few points, where a packet's walk (one node at a time) and
// the later stages are all latency, and for the points whose pairs did not fit
// the pair list.  A warp step takes up to 32 near nodes from the warp's stack and
// tests their 64 children; far children go to a queue that is evaluated 32 terms at a
// time, leaves that are needed exactly to another one, which the warp works
// through leaf by leaf from the (n, w n x x') tables with two lanes per curve (two
// nodes each; on level 1 one half of the curve each).  Leaves near the point or with
// deeper panels go to `slow` for k_pair_eval; points whose slow pairs do not fit
// are listed in olist_out (k_overflow3).  LIST: the exact leaves all go to the pair
// list instead (k_pair_fast, one thread per pair): for few points the leaves of a
// query one after the other are the longest chain.
// A query costs about twice the instructions of its share of a packet, with 64
// times the warps.
// list: the points to take (null: all n), n_dev: their number on the device; again: as in
// k_trav3, without it a dense chunk's leaves take beta2
constexpr int kWideStack = 768;  // stack_take
template <bool O3, bool COUNT, bool LIST>
__global__ void __launch_bounds__(128) k_wide3(DevTree t, const float4* spos, int n, const int* list, const int* n_dev,
                                               float beta2, float beta2l, Workspace ws, int2* slow, long long slow_cap,
                                               int* olist_out, unsigned long long* work, Dense d,
                                               bool again) {
    if (again && !is_dense(d)) return;
    __shared__ int sstk[4][kWideStack];
    __shared__ int sfar[4][96], sleaf[4][128];
    __shared__ float4 slfar[LIST ? 1 : 4][LIST ? 1 : 128];
    __shared__ int2 slrange[LIST ? 1 : 4][LIST ? 1 : 128];
    const unsigned full = 0xffffffffu;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    int *stk = sstk[wid], *fq = sfar[wid], *lq = sleaf[wid];
    WorkLocal wl = {};
    if (n_dev) n = *n_dev;
    const float b2l = t.leaf_far ? (is_dense(d) ? beta2 : beta2l) : INFINITY;
    const float ratio2 = kRatio32 * kRatio32, inv4pi = 0.07957747154594767f;
    unsigned long long npair = 0;
    // few points: a block (an SM) each first
    for (int k = wid * gridDim.x + blockIdx.x; k < n; k += gridDim.x * 4) {
        const int qi = list ? list[k] : k;
        const float4 p = spos[qi];
        float acc = 0.f;
        int sp = 0, nf = 0, nl = 0;  // warp-uniform
        uint32_t st = 0;
        // the terms of the last m queued nodes or leaves, one per lane
        auto far_terms = [&](int m) {
            if (lane < m) {
                const int idx = fq[nf - m + lane];
                const float4 h = idx < t.n_internal ? __ldg(t.hdr + idx) : __ldg(t.lhdr + (idx - t.n_internal));
                const float4* M = t.hmom + (size_t)idx * t.hstride;
                float f[O3 ? 24 : 16];
#pragma unroll
                for (int v = 0; v < (O3 ? 6 : 4); ++v) {
                    const float4 a = __ldg(M + v);
                    f[4 * v] = a.x; f[4 * v + 1] = a.y; f[4 * v + 2] = a.z; f[4 * v + 3] = a.w;
                }
                const float rx = h.x - p.x, ry = h.y - p.y, rz = h.z - p.z;
                acc += far3_harm<float>(f, rx, ry, rz, rsqrt_hw(rx * rx + ry * ry + rz * rz), O3);
            }
            if (COUNT && lane < m) wl.v[kWorkFar] += 1;
            nf -= m;
            __syncwarp();
        };
        auto exact_leaves = [&]() {
            npair += nl;
            if (LIST) {
                long long base = 0;
                if (lane == 0 && nl) base = list_slots(&ws.counters[0], nl, ws.pair_cap);
                base = __shfl_sync(full, base, 0);
                for (int j = lane; j < nl; j += 32)
                    if (base + j < ws.pair_cap) ws.pairs[base + j] = make_int2(qi, lq[j]);
                if (base + nl > ws.pair_cap) st |= kPairOverflow;
                nl = 0;
                __syncwarp();
                return;
            }
            // the leaves' records together, then one leaf after the other
            float4* lf = slfar[LIST ? 0 : wid];
            int2* lr = slrange[LIST ? 0 : wid];
            for (int j = lane; j < nl; j += 32) {
                lf[j] = __ldg(t.lfar + lq[j]);
                lr[j] = __ldg(t.lrange + lq[j]);
            }
            __syncwarp();
            for (int j = 0; j < nl; ++j) {
                const int li = lq[j];
                const float4 L = lf[j];
                const int2 range = lr[j];
                const float qx = p.x - L.x, qy = p.y - L.y, qz = p.z - L.z;
                const float d2 = qx * qx + qy * qy + qz * qz;
                bool bad = !(d2 > L.w);
                float val = 0.f;
                int nodes = 0;
                if (!bad) {
                    const float l = rsqrtf(d2);
                    const f32x2 qn[3] = {pack2(-qx, -qx), pack2(-qy, -qy), pack2(-qz, -qz)};
                    const f32x2 s[3] = {pack2(-qx * l, -qx * l), pack2(-qy * l, -qy * l), pack2(-qz * l, -qz * l)};
                    const int half = lane & 1;
                    for (int c0 = 0; c0 < range.y; c0 += 16) {
                        const int c = c0 + (lane >> 1);
                        const bool on = c < range.y;
                        const float4* H = t.c3m + (size_t)(range.x + (on ? c : 0)) * kC3NodeVec;
                        const float4 hd = __ldg(H);
                        const bool first = on && hd.x < kInfF;  // starts at level 0
                        float sum = 0.f, dm = 1e30f;
                        if (on) far_pair(reinterpret_cast<const ulonglong2*>(H + 1 + 3 * half), qn, s, sum, dm);
                        dm = fminf(dm, __shfl_xor_sync(full, dm, 1));
                        if (first && hd.x * hd.x <= ratio2 * dm) {
                            val += sum;
                            nodes += 2;
                        } else if (on) {
                            far_panel(H + 7 + 6 * half, qn, s, sum, dm);
                            const float len = half ? hd.z : hd.y;
                            if (!(len * len <= ratio2 * dm)) bad = true;
                            val += sum;
                            nodes += first ? 6 : 4;
                        }
                    }
                }
                if (!__any_sync(full, bad)) {
                    acc += val * inv4pi;
                    if (COUNT) wl.v[kWorkFastNodes] += nodes;
                } else {
                    long long slot = 0;
                    if (lane == 0) {
                        slot = list_slots(&ws.counters[8], 1, slow_cap);
                        if (slot < slow_cap) slow[slot] = make_int2(qi, li);
                    }
                    if (__shfl_sync(full, slot, 0) >= slow_cap) st |= kPairOverflow;
                }
            }
            nl = 0;
            __syncwarp();
        };
        // the lanes whose child c (header h) is tested: queued far, queued leaf, or stacked
        auto test = [&](bool on, int c, const float4& h) {
            const float rx = h.x - p.x, ry = h.y - p.y, rz = h.z - p.z;
            const bool far = on && rx * rx + ry * ry + rz * rz > (c < 0 ? b2l : beta2) * h.w;
            if (COUNT && on) wl.v[c < 0 ? kWorkLeafTests : kWorkNodes] += 1;
            const unsigned F = __ballot_sync(full, far), S = __ballot_sync(full, on && !far && c >= 0),
                           E = __ballot_sync(full, on && !far && c < 0);
            if (far) fq[nf + __popc(F & below)] = c < 0 ? t.n_internal + ~c : c;
            else if (on && c >= 0) stk[sp + __popc(S & below)] = c;
            else if (on) lq[nl + __popc(E & below)] = ~c;
            nf += __popc(F);
            sp += __popc(S);
            nl += __popc(E);
        };
        test(lane == 0, t.root, t.root < 0 ? __ldg(t.lhdr + ~t.root) : __ldg(t.hdr + t.root));
        __syncwarp();
        while (sp > 0) {
            const int take = stack_take(sp, 32, kWideStack);
            if (take <= 0) {
                st |= GWN_QS_STACK_OVERFLOW;  // the rest is dropped, the point repaired
                break;
            }
            const bool on = lane < take;
            const int node = on ? stk[sp - 1 - lane] : 0;
            sp -= take;
            const int2 ch = __ldg(t.child + node);
            const float4 ha = __ldg(t.chdr + 2 * node), hb = __ldg(t.chdr + 2 * node + 1);
            __syncwarp();
            test(on, ch.x, ha);
            test(on, ch.y, hb);
            __syncwarp();
            while (nf >= 32) far_terms(32);
            if (nl >= 64) exact_leaves();
        }
        far_terms(nf);
        exact_leaves();
        for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(full, acc, off);
        if (lane == 0) {
            ws.wacc[qi] = acc;
            ws.st[qi] = st;
            if (st & kPairOverflow) olist_out[atomicAdd(&ws.counters[3], 1)] = qi;
        }
        __syncwarp();
    }
    if (lane == 0 && npair) atomicAdd(ws.found + (!LIST || again), npair);
    if (COUNT) flush_work(wl, work);
}

// points with a pair that did not fit a list in the last pass: whole traversal again, leaves in
// place (at beta2: tighter than the far test of the other points' leaves)
__global__ void __launch_bounds__(128) k_overflow3(DevTree t, const float4* spos, float beta2, Workspace ws,
                                                   const int* list, long long* near = nullptr) {
    int cnt = ws.counters[3];
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < cnt; k += gridDim.x * blockDim.x) {
        int qi = list[k];
        const float4 p = spos[qi];
        uint32_t st = 0;
        ws.wacc[qi] = query3_32(t, p.x, p.y, p.z, beta2, st);
        if (near) near[qi] = 0;
        ws.st[qi] = st;
    }
}

// exact 3D leaves from the node tables, one thread per (point, leaf) pair in the
// order of the list: a packet of 64 neighbouring queries writes its pairs in runs of
// one leaf, so the pairs of a warp share one or two leaves' tables.  (Sorting the list
// by leaf first made this kernel 10 to 15 % faster -- rings, 84M pairs: 2.54 against
// 2.96 ms -- but the two sorting passes cost 1.2 ms.)  Pairs whose point lies outside the leaf's
// 1.1-radius sphere and whose panels stop at level 0 or 1 add their value
// here (leaf3_far32).  The others -- points near the leaf, whose string needs
// the foot-point search, and curves that need deeper panels -- are appended in
// order to `slow` (counter [8]) for k_pair_eval.  Every thread of a block runs
// the same iterations, so a warp appends with a single atomic.
__global__ void __launch_bounds__(128) k_pair_fast(DevTree t, const float4* spos, long long npair_cap,
                                                   int* counters, const int2* pairs, float* wacc, uint32_t* st,
                                                   int2* slow, long long slow_cap, int* olist,
                                                   unsigned long long* work) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    WorkLocal wl = {};
    const long long np = min((long long)counters[0], npair_cap);
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long base = (long long)blockIdx.x * blockDim.x; base < np; base += stride) {
        const long long k = base + threadIdx.x;
        bool to_slow = false;
        int2 pr = make_int2(0, 0);
        if (k < np) {
            pr = pairs[k];
            if (pr.x >= 0 && !(st[pr.x] & kPairOverflow)) {  // not padding, nor a point that is evaluated again
                const float4 q = spos[pr.x];
                const float4 L = __ldg(t.lfar + pr.y);
                const float qx = q.x - L.x, qy = q.y - L.y, qz = q.z - L.z;
                const float d2 = qx * qx + qy * qy + qz * qz;
                float v;
                int nodes;
                if (d2 > L.w && leaf3_far32(t.c3m, __ldg(t.lrange + pr.y), qx, qy, qz, d2, &v, &nodes)) {
                    atomicAdd(&wacc[pr.x], v);
                    if (work) wl.v[kWorkFastNodes] += (unsigned long long)nodes;
                }
                else
                    to_slow = true;
            }
        }
        const unsigned m = __ballot_sync(full, to_slow);
        if (m) {
            const int leader = __ffs(m) - 1;
            int slot0 = 0;
            if (lane == leader) slot0 = atomicAdd(&counters[8], __popc(m));
            slot0 = __shfl_sync(full, slot0, leader);
            if (to_slow) {
                const int slot = slot0 + __popc(m & ((1u << lane) - 1u));
                if (slot < slow_cap) slow[slot] = pr;
                else if (!(atomicOr(&st[pr.x], kPairOverflow) & kPairOverflow)) olist[atomicAdd(&counters[3], 1)] = pr.x;
            }
        }
    }
    if (work) flush_work(wl, work);
}

// k_pair_fast for the padded list of k_trav3: two pairs of one leaf per lane, which
// share every table load.  One pair per lane ran at 42 % of the FMA pipe and 60 % of
// the load pipe's wavefronts (a broadcast 16-byte load holds it for two cycles),
// and neither more warps, nor the tables in shared memory, nor the atomics left out moved it.
__global__ void __launch_bounds__(128) k_pair_fast2(DevTree t, const float4* spos, long long npair_cap,
                                                    int* counters, const int4* pairs, float* wacc, uint32_t* st,
                                                    int2* slow, long long slow_cap, int* olist,
                                                    unsigned long long* work) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const float ratio2 = kRatio32 * kRatio32;
    WorkLocal wl = {};
    const long long np = min((long long)counters[0], npair_cap) / 2;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long base = (long long)blockIdx.x * blockDim.x; base < np; base += stride) {
        const long long k = base + threadIdx.x;
        int4 pr = make_int4(-1, 0, -1, 0);
        bool on0 = false, on1 = false, slow0 = false, slow1 = false;
        if (k < np) {
            pr = pairs[k];
            on0 = pr.x >= 0 && !(st[pr.x] & kPairOverflow);
            on1 = pr.z >= 0 && !(st[pr.z] & kPairOverflow);
        }
        if (on0 || on1) {
            const float4 L = __ldg(t.lfar + pr.y), p0 = spos[on0 ? pr.x : pr.z], p1 = spos[on1 ? pr.z : pr.x];
            const int2 range = __ldg(t.lrange + pr.y);
            const float x0 = p0.x - L.x, y0 = p0.y - L.y, z0 = p0.z - L.z, x1 = p1.x - L.x, y1 = p1.y - L.y, z1 = p1.z - L.z;
            const float d0 = x0 * x0 + y0 * y0 + z0 * z0, d1 = x1 * x1 + y1 * y1 + z1 * z1;
            slow0 = !(d0 > L.w);
            slow1 = !(d1 > L.w);
            const float l0 = rsqrtf(d0), l1 = rsqrtf(d1);
            const f32x2 qa[3] = {pack2(-x0, -x0), pack2(-y0, -y0), pack2(-z0, -z0)};
            const f32x2 qb[3] = {pack2(-x1, -x1), pack2(-y1, -y1), pack2(-z1, -z1)};
            const f32x2 sa[3] = {mul2(qa[0], pack2(l0, l0)), mul2(qa[1], pack2(l0, l0)), mul2(qa[2], pack2(l0, l0))};
            const f32x2 sb[3] = {mul2(qb[0], pack2(l1, l1)), mul2(qb[1], pack2(l1, l1)), mul2(qb[2], pack2(l1, l1))};
            float acc0 = 0.f, acc1 = 0.f;
            int n0 = 0, n1 = 0;
            // the panel's four nodes for both pairs
            auto panel = [&](const float4* P, float& fa, float& da, float& fb, float& db) {
                const ulonglong2* V = reinterpret_cast<const ulonglong2*>(P);
                f32x2 ua = 0, ub = 0;
                da = db = 1e30f;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const ulonglong2 a = __ldg(V + 3 * h), b = __ldg(V + 3 * h + 1), c = __ldg(V + 3 * h + 2);
                    far_nodes2(a, b, c, qa, sa, ua, da);
                    far_nodes2(a, b, c, qb, sb, ub, db);
                }
                fa = sum2(ua);
                fb = sum2(ub);
            };
            const float4* H = t.c3m + (size_t)range.x * kC3NodeVec;
            for (int c = 0; c < range.y && !(slow0 && slow1); ++c, H += kC3NodeVec) {
                const float4 hd = __ldg(H);
                float fa, da, fb, db;
                panel(H + 1, fa, da, fb, db);
                n0 += 4;
                n1 += 4;
                // an infinite length (a curve that starts below level 0) never passes
                const bool ok0 = hd.x * hd.x <= ratio2 * da, ok1 = hd.x * hd.x <= ratio2 * db;
                if (ok0) acc0 += fa;
                if (ok1) acc1 += fb;
                if (!(ok0 && ok1)) {
                    float ga, ea, gb, eb;
                    panel(H + 7, fa, da, fb, db);
                    panel(H + 13, ga, ea, gb, eb);
                    if (!ok0) {
                        acc0 += fa + ga;
                        n0 += 8;
                        if (!(hd.y * hd.y <= ratio2 * da && hd.z * hd.z <= ratio2 * ea)) slow0 = true;
                    }
                    if (!ok1) {
                        acc1 += fb + gb;
                        n1 += 8;
                        if (!(hd.y * hd.y <= ratio2 * db && hd.z * hd.z <= ratio2 * eb)) slow1 = true;
                    }
                }
            }
            if (on0 && !slow0) {
                atomicAdd(&wacc[pr.x], acc0 * 0.07957747154594767f);  // 1 / (4 pi)
                if (work) wl.v[kWorkFastNodes] += (unsigned long long)n0;
            }
            if (on1 && !slow1) {
                atomicAdd(&wacc[pr.z], acc1 * 0.07957747154594767f);
                if (work) wl.v[kWorkFastNodes] += (unsigned long long)n1;
            }
        }
        const unsigned ma = __ballot_sync(full, on0 && slow0), mb = __ballot_sync(full, on1 && slow1);
        if (ma | mb) {
            int slot0 = 0;
            if (lane == 0) slot0 = atomicAdd(&counters[8], __popc(ma) + __popc(mb));
            slot0 = __shfl_sync(full, slot0, 0) + __popc(ma & ((1u << lane) - 1u)) + __popc(mb & ((1u << lane) - 1u));
            auto put = [&](int q, int slot) {
                if (slot < slow_cap) slow[slot] = make_int2(q, pr.y);
                else if (!(atomicOr(&st[q], kPairOverflow) & kPairOverflow)) olist[atomicAdd(&counters[3], 1)] = q;
            };
            if (on0 && slow0) put(pr.x, slot0);
            if (on1 && slow1) put(pr.z, slot0 + (on0 && slow0 ? 1 : 0));
        }
    }
    if (work) flush_work(wl, work);
}

// The direct sum's far pairs (every leaf for every point, summed in FP64 so that the
// thousands of additions do not round): a block holds 128 points and walks one of
// gridDim.y slices of the leaves, whose tables it reads at the same address in
// all lanes; the slices' sums add up in fixed point (add_fixed).  Near and deeper pairs go to
// `slow` (k_pair_eval), points whose slow pairs do not fit to olist (k_direct_overflow3).  acc,
// rest and st zeroed beforehand.
__global__ void __launch_bounds__(128) k_direct3(DevTree t, const float4* spos, int n, long long* acc, float* rest, uint32_t* st,
                                                 int* counters, int2* slow, long long slow_cap, int* olist) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * 128 + threadIdx.x;
    const bool act = i < n;
    const float4 p = act ? spos[i] : make_float4(0, 0, 0, 0);
    const int l0 = (int)((long long)t.n_leaves * blockIdx.y / gridDim.y),
              l1 = (int)((long long)t.n_leaves * (blockIdx.y + 1) / gridDim.y);
    double sum = 0.0;
    for (int l = l0; l < l1; ++l) {
        const float4 L = __ldg(t.lfar + l);
        const float qx = p.x - L.x, qy = p.y - L.y, qz = p.z - L.z;
        const float d2 = qx * qx + qy * qy + qz * qz;
        float v = 0.f;
        int nodes;
        const bool ok = d2 > L.w && leaf3_far32(t.c3m, __ldg(t.lrange + l), qx, qy, qz, d2, &v, &nodes);
        if (ok) sum += (double)v;
        const unsigned m = __ballot_sync(full, act && !ok);
        if (m) {
            long long slot = 0;
            if (lane == 0) slot = list_slots(&counters[8], __popc(m), slow_cap);
            slot = __shfl_sync(full, slot, 0) + __popc(m & ((1u << lane) - 1u));
            if (act && !ok) {
                if (slot < slow_cap) slow[slot] = make_int2(i, l);
                else if (!(atomicOr(&st[i], kPairOverflow) & kPairOverflow)) olist[atomicAdd(&counters[3], 1)] = i;
            }
        }
    }
    if (act) add_fixed(acc, rest, i, sum);
}

// direct sums whose near pairs did not fit the list: one thread per point
__global__ void __launch_bounds__(128) k_direct_overflow3(DevTree t, const float4* spos, long long* acc, float* rest, uint32_t* stv,
                                                          const int* counters, const int* olist) {
    const int cnt = counters[3];
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < cnt; k += gridDim.x * blockDim.x) {
        const int i = olist[k];
        const float4 p = spos[i];
        double w = 0.0;
        uint32_t st = 0;
        for (int l = 0; l < t.n_leaves; ++l) w += (double)leaf3_eval32(t, l, p.x, p.y, p.z, st);
        acc[i] = 0;
        rest[i] = 0.f;
        add_fixed(acc, rest, i, w);
        stv[i] = st;
    }
}

// The pairs that k_pair_fast left (count *count): points near their leaf, and
// curves that need panels below level 1.  A block takes 128 pairs at a time through
// phases, so that what only some pairs or curves need is done by full warps:
//   1. one thread per pair: the string direction; a pair near its leaf whose
//      point projects into the leaf's control-net box (lhit) is listed for the
//      foot-point search;
//   2. one thread per listed search (leaf_hit_solve), and one thread per pair for
//      the level-0 panels of its curves from the FP32 node tables; the halves of the
//      curves that need shorter panels are listed (a thread that finds the list full
//      goes on from that curve once the listed halves are done);
//   3. one thread per listed half: its level-1 panel from the table; those that need
//      shorter ones push their two panels of level 2;
//   4. steps of up to kNearTake panels from the top of that stack, four lanes to a panel (one
//      Gauss-Legendre node each, from the curve's Bernstein form): the integral, or two
//      panels of the next level onto the stack.
// Pairs FP32 cannot resolve go to the FP64 near band; where its list is full their point goes
// to olist (the points evaluated again in place), or, without one, is flagged for the repair.
// One thread doing all of this for its pair from the Bernstein form alone (28 D + 70 flops per node, the
// tables 34) took 5.8 ms on 1.3M points of a 4.7k-leaf model, whole curves below level 1 per
// thread 1.8 ms with 10 to 12 active lanes per instruction.
// Acc: float (the traversal, onto wacc), or long long, whose sums -- a pair's panels and a
// point's pairs -- add up in fixed point, so that two runs give the same bits whatever
// the order of the list (the direct sum and the no-alloc query).
constexpr int kNearHalves = 2048, kNearPanels = 2048, kNearStep = 512, kNearTake = 256;
template <typename Acc>
__global__ void __launch_bounds__(128, 5) k_pair_eval(DevTree t, const float4* spos, long long npair_cap,
                                                   const int* count, int* counters, const int2* pairs, Acc* wacc,
                                                   uint32_t* st, int2* pairs64, int npair64_cap, int* olist,
                                                   unsigned long long* work) {
    constexpr bool kFixed = sizeof(Acc) == 8;
    __shared__ Acc sacc[128];
    __shared__ float sq[3][128], ss[3][128];
    __shared__ int sleaf[128], sfail[128], shit[128];
    // pair | panel index | level | curve, 7 + 10 + 4 + 10 bits
    __shared__ unsigned stask[kNearHalves], spanel[kNearPanels], schild[2 * kNearTake];
    __shared__ int nhit, nhalf, npanel, nchild;
    constexpr int kMaxCurve = 1 << 10;
    WorkLocal wl = {};
    const int tid = threadIdx.x, lane = tid & 31;
    const float inv4pi = 0.07957747154594767f;
    const float ratio2 = kRatio32 * kRatio32;
    const long long np = min((long long)*count, npair_cap);
    auto entry = [](int o, int c, int level, unsigned idx) {
        return (unsigned)o | idx << 7 | (unsigned)level << 17 | (unsigned)c << 21;
    };
    auto add = [&](int o, float v) {
        if constexpr (kFixed) {
            if (isfinite(v)) atomicAdd(reinterpret_cast<unsigned long long*>(&sacc[o]), (unsigned long long)__float2ll_rn(v * kSumUnit));
            else sfail[o] = 1;
        } else {
            atomicAdd(&sacc[o], v);
        }
    };
    // panel idx of `level` of curve c of the leaf of pair o and what is below it, by one thread
    auto whole_panel = [&](int o, int c, int level, unsigned idx) {
        const int k = t.lrange[sleaf[o]].x + c;
        const Curve3Info ci = t.c3[k];
        const Geo32 g{nullptr, t.c3pts + ci.ctrl_off};
        const float q[3] = {sq[0][o], sq[1][o], sq[2][o]}, s[3] = {ss[0][o], ss[1][o], ss[2][o]};
        const int l0 = max(level, ci.min_level), sub = l0 - level;
        float a = 0.f;
        bool deep = false;
        for (unsigned j = idx << sub; j < ((idx + 1) << sub); ++j)
            a += panel_subtree<float>(g, ci.deg, q, s, l0, j, kLevel32, kRatio32, deep, work ? &wl : nullptr);
        add(o, ci.mult * a * inv4pi);
        if (deep) sfail[o] = 1;
    };
    for (long long base = (long long)blockIdx.x * 128; base < np; base += (long long)gridDim.x * 128) {
        if (tid == 0) nhit = nhalf = npanel = nchild = 0;
        sacc[tid] = 0;
        sfail[tid] = 0;
        __syncthreads();
        bool act = base + tid < np;
        int2 pr = make_int2(0, 0);
        float q[3] = {0, 0, 0}, s[3] = {0, 0, 0};
        if (act) {
            pr = pairs[base + tid];
            if (st[pr.x] & kPairOverflow) act = false;  // the next pass evaluates the whole point again
        }
        if (act) {
            const float4 p = spos[pr.x], L = __ldg(t.lfar + pr.y);
            q[0] = p.x - L.x; q[1] = p.y - L.y; q[2] = p.z - L.z;
            const float d2 = q[0] * q[0] + q[1] * q[1] + q[2] * q[2];
            if (work) wl.v[kWorkLeaves] += 1;
            if (d2 > L.w) {
                const float l = rsqrtf(d2);
                s[0] = -q[0] * l; s[1] = -q[1] * l; s[2] = -q[2] * l;
            } else {
                const Leaf3Info& I = t.leaf3[pr.y];
                const float n0 = I.nrm[0], n1 = I.nrm[1], n2 = I.nrm[2];
                const float h = q[0] * n0 + q[1] * n1 + q[2] * n2;
                const float sig = h >= 0.f ? 1.f : -1.f;
                s[0] = -sig * n0; s[1] = -sig * n1; s[2] = -sig * n2;
                if (work) wl.v[kWorkHits] += 1;
                const float4 A = __ldg(t.lhit + 3 * pr.y), B = __ldg(t.lhit + 3 * pr.y + 1), C = __ldg(t.lhit + 3 * pr.y + 2);
                const float p1 = q[0] * A.x + q[1] * A.y + q[2] * A.z, p2 = q[0] * B.x + q[1] * B.y + q[2] * B.z;
                const float top = sig > 0.f ? C.w - h : h - C.z;  // the net's highest point along the half line
                // negated, so that a NaN coordinate goes on to the search and is flagged there
                if (!(p1 < A.w || p1 > B.w || p2 < C.x || p2 > C.y || top < -hit_tau_eps<float>(I.diag)))
                    shit[atomicAdd(&nhit, 1)] = tid;
            }
            sq[0][tid] = q[0]; sq[1][tid] = q[1]; sq[2][tid] = q[2];
            ss[0][tid] = s[0]; ss[1][tid] = s[1]; ss[2][tid] = s[2];
            sleaf[tid] = pr.y;
        }
        __syncthreads();
        if (tid < nhit) {
            const int o = shit[tid], li = sleaf[o];
            const Leaf3Info I = t.leaf3[li];
            const Geo32 g{t.net3 + (size_t)li * kNet3Vec, nullptr};
            const float4 A = __ldg(t.lhit + 3 * li), B = __ldg(t.lhit + 3 * li + 1);
            const float e1[3] = {A.x, A.y, A.z}, e2[3] = {B.x, B.y, B.z};
            const float qo[3] = {sq[0][o], sq[1][o], sq[2][o]};
            const float sig = qo[0] * I.nrm[0] + qo[1] * I.nrm[1] + qo[2] * I.nrm[2] >= 0.f ? 1.f : -1.f;
            float hits = 0.f;
            const int hr = leaf_hit_solve<float>(t, I, g, qo, I.nrm, e1, e2, sig, hit_tau_eps<float>(I.diag), &hits, kNear32);
            if (hr == kHitUnsure) sfail[o] = 1;
            else if (hr == kHitOk) add(o, -hits);
        }
        const int2 range = act ? __ldg(t.lrange + pr.y) : make_int2(0, 0);
        int c = 0;  // next curve
        bool more;
        do {
            float acc = 0.f;
            for (; c < range.y; ++c) {
                const float4* H = t.c3n + (size_t)(range.x + c) * kC3NodeVec;
                const float4 hd = __ldg(H);
                if (hd.x < kInfF) {
                    float pa, da;
                    fast_panel(H + 1, q, s, pa, da);
                    if (work) wl.v[kWorkFastNodes] += 4;
                    if (hd.x * hd.x <= ratio2 * da) {
                        if constexpr (kFixed) add(tid, hd.w * pa * inv4pi);
                        else acc += hd.w * pa;
                        continue;
                    }
                }
                if (c >= kMaxCurve) {
                    for (int j = 0; j < 2; ++j) whole_panel(tid, c, 1, j);
                    continue;
                }
                const int slot = atomicAdd(&nhalf, 2);
                if (slot >= kNearHalves) break;  // full: this curve in the next turn
                for (int j = 0; j < 2; ++j) stask[slot + j] = entry(tid, c, 1, j);
            }
            if constexpr (!kFixed) {
                if (act) atomicAdd(&sacc[tid], acc * inv4pi);
            }
            __syncthreads();
            const int nh = min(nhalf, kNearHalves);
            for (int h0 = 0; h0 < nh; h0 += kNearStep) {
                // level 1, one thread per half curve; the stack is empty
                for (int j = h0 + tid; j < min(nh, h0 + kNearStep); j += 128) {
                    const unsigned e = stask[j];
                    const int o = e & 127, half = e >> 7 & 1, cj = e >> 21;
                    const int k = t.lrange[sleaf[o]].x + cj;
                    const float4* H = t.c3n + (size_t)k * kC3NodeVec;
                    const float4 hd = __ldg(H);
                    const float len = half ? hd.z : hd.y;
                    if (len < kInfF) {
                        const float qo[3] = {sq[0][o], sq[1][o], sq[2][o]}, so[3] = {ss[0][o], ss[1][o], ss[2][o]};
                        float pa, da;
                        fast_panel(H + 7 + 6 * half, qo, so, pa, da);
                        if (work) wl.v[kWorkFastNodes] += 4;
                        if (len * len <= ratio2 * da) {
                            add(o, 0.5f * hd.w * pa * inv4pi);
                            continue;
                        }
                    }
                    // level 2; by this thread where the curve's own first level is lower
                    if (t.c3[k].min_level <= 2) {
                        const int slot = atomicAdd(&npanel, 2);
                        for (int i = 0; i < 2; ++i) spanel[slot + i] = entry(o, cj, 2, 2 * half + i);
                    } else {
                        for (int i = 0; i < 2; ++i) whole_panel(o, cj, 2, 2 * half + i);
                    }
                }
                __syncthreads();
                int sp = npanel;  // block-uniform
                while (sp > 0) {
                    const int take = stack_take(sp, kNearTake, kNearPanels);
                    for (int j0 = 0; j0 < take; j0 += 32) {
                        const int j = j0 + (tid >> 2), node = tid & 3;
                        const bool on = j < take;
                        float f = 0.f, dm = 1e30f, x[3] = {0, 0, 0};
                        unsigned e = 0;
                        Curve3Info ci{0, 1, 0.f, 0};
                        float h = 1.f;
                        if (on) {
                            e = spanel[sp - take + j];
                            const int o = e & 127;
                            ci = t.c3[t.lrange[sleaf[o]].x + (int)(e >> 21)];
                            const Geo32 g{nullptr, t.c3pts + ci.ctrl_off};
                            const float qo[3] = {sq[0][o], sq[1][o], sq[2][o]}, so[3] = {ss[0][o], ss[1][o], ss[2][o]};
                            h = 1.f / (float)(1u << (e >> 17 & 15));
                            f = Gl8<float>::w(node) * gl_node_any<float>(g, ci.deg, (float)(e >> 7 & 1023) * h + h * Gl8<float>::x(node),
                                                                         qo, so, x, &dm);
                            if (work) {
                                wl.v[kWorkGlNodes] += 1;
                                wl.v[kWorkGlDeg] += ci.deg;
                            }
                        }
                        const unsigned full = 0xffffffffu;
                        const float e0 = x[0] - __shfl_up_sync(full, x[0], 1), e1 = x[1] - __shfl_up_sync(full, x[1], 1),
                                    e2 = x[2] - __shfl_up_sync(full, x[2], 1);
                        float len = node ? Num<float>::sqrt_fast(e0 * e0 + e1 * e1 + e2 * e2) : 0.f;
                        for (int off = 1; off < 4; off <<= 1) {
                            f += __shfl_xor_sync(full, f, off);
                            len += __shfl_xor_sync(full, len, off);
                            dm = fminf(dm, __shfl_xor_sync(full, dm, off));
                        }
                        len *= Gl8<float>::span_inv;
                        if (on && node == 0) {
                            const int o = e & 127, level = e >> 17 & 15;
                            const unsigned idx = e >> 7 & 1023;
                            const bool refine = len * len > ratio2 * dm;
                            if (!refine || level >= kLevel32) {
                                add(o, ci.mult * f * h * inv4pi);
                                if (refine) sfail[o] = 1;
                            } else {
                                const int slot = atomicAdd(&nchild, 2);
                                for (int i = 0; i < 2; ++i) schild[slot + i] = entry(o, e >> 21, level + 1, 2 * idx + i);
                            }
                        }
                    }
                    __syncthreads();
                    const int k = nchild;
                    sp -= take;
                    for (int j = tid; j < k; j += 128) spanel[sp + j] = schild[j];
                    sp += k;
                    __syncthreads();
                    if (tid == 0) nchild = npanel = 0;
                    __syncthreads();
                }
            }
            if (tid == 0) nhalf = 0;
            more = __syncthreads_or(c < range.y);
        } while (more);
        if (act) {
            if (!sfail[tid]) {
                if constexpr (kFixed) atomicAdd(reinterpret_cast<unsigned long long*>(&wacc[pr.x]), (unsigned long long)sacc[tid]);
                else atomicAdd(&wacc[pr.x], sacc[tid]);
            } else {
                const int slot = atomicAdd(&counters[2], 1);
                if (slot < npair64_cap) {
                    pairs64[slot] = pr;
                    atomicOr(&st[pr.x], GWN_QS_NEAR);
                } else if (!olist) {
                    atomicOr(&st[pr.x], GWN_QS_STACK_OVERFLOW);
                } else if (!(atomicOr(&st[pr.x], kPairOverflow) & kPairOverflow)) {
                    olist[atomicAdd(&counters[3], 1)] = pr.x;
                }
            }
        }
        __syncthreads();  // the lists are reset next
    }
    if (work) flush_work(wl, work);
}

// 4-point FP64 panels are used for leaves whose boundary curves all have degree
// <= 6 (pieces of degree 1 composed with the bicubic net); curves of higher
// degree (rational trims) take 8-point panels, whose error does not depend on
// how close the rational parametrisation's poles come to the panel
__device__ __forceinline__ bool leaf_fits_w4(const DevTree& t, int li) {
    const Leaf3Info I = t.leaf3[li];
    int dmax = 0;
    for (int c = threadIdx.x & 31; c < I.c3_cnt; c += 32) dmax = max(dmax, t.c3[I.c3_off + c].deg);
    for (int off = 16; off > 0; off >>= 1) dmax = max(dmax, __shfl_xor_sync(0xffffffffu, dmax, off));
    return dmax <= 6;
}

// the near band with one warp per pair (leaf3_warp64), onto near in fixed point where given, else
// onto wacc
__global__ void __launch_bounds__(128) k_pair_eval64_warp(DevTree t, const float4* spos, int npair64_cap,
                                                          const int* counters, const int2* pairs64, float* wacc,
                                                          uint32_t* st, long long* near = nullptr) {
    __shared__ int2 sstk[4][kQuadStack];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int np = min(counters[2], npair64_cap);
    // few pairs: an SM each first, since the warps of an SM share its two FP64 lanes
    for (int k = wid * gridDim.x + blockIdx.x; k < np; k += gridDim.x * 4) {
        const int2 pr = pairs64[k];
        if (st[pr.x] & kPairOverflow) continue;  // evaluated again in place
        const float4 p = spos[pr.x];
        const double q[3] = {(double)p.x, (double)p.y, (double)p.z};
        double v = 0;
        const bool ok = leaf_fits_w4(t, pr.y) ? leaf3_warp64<4>(t, pr.y, q, kRatio64BandW4, kLevel64, sstk[wid], &v)
                                              : leaf3_warp64<8>(t, pr.y, q, kRatio64Band, kLevel64, sstk[wid], &v);
        if (lane == 0) {
            if (ok && near) add_fixed(near, wacc, pr.x, (double)(float)v);
            else if (ok) atomicAdd(&wacc[pr.x], (float)v);
            if (!ok) atomicOr(&st[pr.x], GWN_QS_UNRESOLVED);
        }
        __syncwarp();
    }
}

// outputs of one chunk (points off .. off + n - 1 of the query); points to
// repair go to the query's list (index off + i) while it has room, else to the
// chunk's own list (index i), repaired right after the chunk
// parts > 0 (2D): wacc holds the subtrees' sums (value2); near: sums in fixed point
template <typename Acc>
__global__ void k_finish(int n, const float4* spos, const Acc* wacc, const uint32_t* stv, int precision, float band, double* out_w,
                         int* out_label, uint32_t* out_status, int* rlist, int* rcount, int off, int* rlist_g,
                         int* gcount, int gcap, int parts = 0, const long long* near = nullptr) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int i = __float_as_int(spos[k].w);  // place in the binned copy -> the caller's order
    double w = sizeof(Acc) == 4 && parts ? (double)value2(reinterpret_cast<const float*>(wacc), near, n, parts, k)
               : near                    ? (double)wacc[k] + (double)near[k] * (1.0 / (double)kSumUnit)
                                         : (double)wacc[k];
    uint32_t st = stv[k];
    if (precision == GWN_PREC_FP32_REPAIR) {
        double fr = w - floor(w);
        if (fabs(fr - 0.5) < (double)band || (st & (GWN_QS_STACK_OVERFLOW | GWN_QS_UNRESOLVED))) {
            int slot = atomicAdd(gcount, 1);
            if (slot < gcap) {
                rlist_g[slot] = off + i;
            } else {
                slot = atomicAdd(rcount, 1);
                rlist[slot] = i;
            }
        }
    }
    out_w[i] = w;
    if (out_label) out_label[i] = (int)round(w);
    if (out_status) out_status[i] = st;
}

}  // namespace gwn

namespace gwn {

__device__ __forceinline__ void load_point_d(const void* pts, int dtype, long long i, double q[3]) {
    if (dtype == GWN_F32) {
        const float* p = reinterpret_cast<const float*>(pts) + (size_t)i * 3;
        q[0] = p[0]; q[1] = p[1]; q[2] = p[2];
    } else {
        const double* p = reinterpret_cast<const double*>(pts) + (size_t)i * 3;
        q[0] = p[0]; q[1] = p[1]; q[2] = p[2];
    }
}

// How an FP64 pass integrates its leaves: panel length / distance bound of the 8-point
// rule, and whether leaves of low degree may take 4-point panels at half of it.
// The repair: kRatio64Repair, yes; GWN_PREC_FP64: kRatio64Exact, no.
struct Rule64 {
    double ratio;
    bool w4;
};

// FP64 pairs from the FP64 node tables, one warp per pair
// (leaf3_fast64_warp: far pairs whose 8-point panels stop at level 0 or 1); the
// others go to the second list for k_rpairs3_warp
__global__ void __launch_bounds__(128) k_rpairs3_fast(DevTree t, const void* pts, int dtype, RepairList R, Rule64 rule) {
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long np = min((long long)*R.npairs, kRepairPairCap);
    for (long long j = (long long)wid * gridDim.x + blockIdx.x; j < np; j += (long long)gridDim.x * 4) {
        const int2 pr = R.pairs[j];
        double q[3];
        load_point_d(pts, dtype, R.idx[R.val ? pr.x / R.per : pr.x], q);
        double v = 0;
        const bool ok = leaf3_fast64_warp(t, pr.y, q, rule.ratio, &v);
        if (lane == 0) {
            if (ok && R.val) R.val[pr.x] = v;
            else if (ok) atomicAdd(&R.rw[pr.x], v);
            else R.pairs2[atomicAdd(R.npairs2, 1)] = pr;
        }
        __syncwarp();
    }
}

// the full FP64 evaluation of leaf li by a warp (stk: kQuadStack entries)
__device__ __forceinline__ bool leaf64_warp(const DevTree& t, int li, const double q[3], Rule64 rule, int2* stk, double* v) {
    return rule.w4 && leaf_fits_w4(t, li) ? leaf3_warp64<4>(t, li, q, 0.5 * rule.ratio, kLevel64, stk, v)
                                          : leaf3_warp64<8>(t, li, q, rule.ratio, kLevel64, stk, v);
}

// FP64 pairs with one warp per pair (leaf3_warp64): those the tables left
__global__ void __launch_bounds__(128) k_rpairs3_warp(DevTree t, const void* pts, int dtype, RepairList R, Rule64 rule) {
    __shared__ int2 sstk[4][kQuadStack];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long np = min((long long)*R.npairs2, kRepairPairCap);
    for (long long j = (long long)wid * gridDim.x + blockIdx.x; j < np; j += (long long)gridDim.x * 4) {
        const int2 pr = R.pairs2[j];
        const int k = R.val ? pr.x / R.per : pr.x;
        double q[3];
        load_point_d(pts, dtype, R.idx[k], q);
        double v = 0;
        const bool ok = leaf64_warp(t, pr.y, q, rule, sstk[wid], &v);
        if (lane == 0) {
            if (R.val) R.val[pr.x] = ok ? v : 0.0;
            else if (ok) atomicAdd(&R.rw[k], v);
            if (!ok) atomicOr(&R.rst[k], GWN_QS_UNRESOLVED);
        }
        __syncwarp();
    }
}

// every leaf of every listed point as an FP64 pair (the direct sum); the host
// bounds the points so that the pairs fit
__global__ void k_rpairs_all(RepairList R, int n, int n_leaves) {
    const long long np = (long long)n * n_leaves, stride = (long long)gridDim.x * blockDim.x;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < np; j += stride) {
        R.pairs[j] = make_int2((int)j, (int)(j % n_leaves));  // per == n_leaves
        if (j < n) {
            R.rw[j] = 0.0;
            R.rst[j] = 0u;
            R.cnt[j] = n_leaves;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *R.npairs = (int)np;
}

// the pairs' values of each listed point (RepairList::val), in order, onto rw: one
// warp per point, lanes strided
__global__ void k_rsum(RepairList R, int n) {
    const int lane = threadIdx.x & 31;
    const int k = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (k >= n) return;
    const double* v = R.val + (size_t)k * R.per;
    const int cnt = R.cnt[k];
    double a = 0.0;
    for (int j = lane; j < cnt; j += 32) a += v[j];
    for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
    if (lane == 0) R.rw[k] += a;
}

// between the passes: the overflow list just written becomes the second pass's
// input list, and the pair list is emptied
__global__ void k_next_round(Workspace ws) {
    if (threadIdx.x == 0) {
        ws.counters[5] = ws.counters[3];
        ws.counters[6] += ws.counters[3];
        ws.counters[9] += ws.counters[8];  // pairs the full evaluator took
        ws.counters[3] = 0;
        ws.counters[0] = 0;  // the near-band list (counters[2]) spans both passes
        ws.counters[8] = 0;
    }
}

// a chunk's counters into the query's totals; last: the query-wide repair pass too
// (repaired points and FP64 pairs)
__global__ void k_accum(Workspace ws, bool last) {
    const int k = threadIdx.x;
    if (k < kCounterCount) ws.acc[k] += k == 0 ? ws.found[0] + ws.found[1] : (unsigned long long)ws.counters[k];
    if (!last) return;
    __syncwarp();
    if (k == 0) ws.acc[1] += (unsigned long long)min(ws.gcount[0], ws.rcap);
    if (k == 1) ws.acc[4] += (unsigned long long)ws.gcount[1];
}

// FP64 values, labels and status; keep (the repair): the FP32 status bits k_finish
// wrote stay; add: bits every listed point gets
__global__ void k_rfinish(RepairList R, double* out_w, int* out_label, uint32_t* out_status, bool keep, uint32_t add) {
    const int cnt = min(*R.count, R.cap);
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < cnt; k += gridDim.x * blockDim.x) {
        int qi = R.idx[k];
        double w = R.rw[k];
        out_w[qi] = w;
        if (out_label) out_label[qi] = (int)round(w);
        if (out_status) out_status[qi] = (keep ? out_status[qi] : 0u) | R.rst[k] | add;
    }
}

}  // namespace gwn

namespace gwn {

// ---- Warp-cooperative FP64 traversal (3D).  One warp per repaired point:
// the warp keeps a node stack in shared memory and each step the lanes take up
// to 32 nodes from its top, apply the far test in FP64 and push the children
// of the nodes that fail it (positions by a warp prefix sum).  This spreads one
// point's traversal over 32 lanes, which matters because FP64 issue is slow
// and latency-bound when a single thread walks the tree.  Exact leaves are
// appended to the FP64 pair list (k_rpairs3_fast).  Points whose
// pairs did not fit the list are marked and taken by the INPLACE instance (marked:
// these points only), where the warp evaluates the leaves itself.
constexpr int kWarpStack = 2048;
constexpr int kRepairWarps = 4;  // warps per block

template <bool INPLACE>
__global__ void __launch_bounds__(32 * kRepairWarps) k_rtrav_warp(DevTree t, const void* pts, int dtype, double beta2r,
                                                                  RepairList R, double beta2rl, Rule64 rule, bool marked) {
    __shared__ int sstack[kRepairWarps][kWarpStack];
    __shared__ int2 squad[INPLACE ? kRepairWarps : 1][INPLACE ? kQuadStack : 1];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gw = wid * gridDim.x + blockIdx.x;  // few points: an SM each first
    const int nw = gridDim.x * kRepairWarps;
    const int cnt = min(*R.count, R.cap);
    int* stk = sstack[wid];
    for (int k = gw; k < cnt; k += nw) {
        if (marked && !(R.rst[k] & kPairOverflow)) continue;
        const int qi = R.idx[k];
        double q[3];
        load_point_d(pts, dtype, qi, q);
        double acc = 0.0;
        uint32_t st = 0;
        int npair = 0;  // warp-uniform
        if (lane == 0) stk[0] = t.root;
        int sp = 1;
        __syncwarp();
        while (sp > 0) {
            const int take = stack_take(sp, 32, kWarpStack);
            if (take <= 0) {
                st |= GWN_QS_UNRESOLVED;  // stack full: the rest is dropped (flagged)
                break;
            }
            const int node = lane < take ? stk[sp - 1 - lane] : 0;
            sp -= take;
            __syncwarp();
            int c0 = 0, c1 = 0, npush = 0;
            bool exact = false;  // a 3D leaf the pair list or the warp takes
            if (lane < take) {
                if (node < 0) {
                    const int li = ~node;
                    const double* h = t.lhdr64 + (size_t)li * 4;
                    double rx = h[0] - q[0], ry = h[1] - q[1], rz = h[2] - q[2];
                    if (beta2rl > 0 && t.leaf_far && rx * rx + ry * ry + rz * rz > beta2rl * h[3]) {
                        acc += far3_harm<double>(t.hmom64 + (size_t)(t.n_internal + li) * kHarm, rx, ry, rz,
                                                 rsqrt(rx * rx + ry * ry + rz * rz), t.order3_64);
                    } else {
                        exact = true;
                    }
                } else {
                    const double* h = t.hdr64 + (size_t)node * 4;
                    double rx = h[0] - q[0], ry = h[1] - q[1], rz = h[2] - q[2];
                    double d2 = rx * rx + ry * ry + rz * rz;
                    if (beta2r > 0 && d2 > beta2r * h[3]) {
                        acc += far3_harm<double>(t.hmom64 + (size_t)node * kHarm, rx, ry, rz, rsqrt(d2), t.order3_64);
                    } else {
                        int2 ch = t.child[node];
                        c0 = ch.x;
                        c1 = ch.y;
                        npush = 2;
                    }
                }
            }
            unsigned need = __ballot_sync(0xffffffffu, exact);
            if (INPLACE) {
                for (; need; need &= need - 1) {
                    const int li = ~__shfl_sync(0xffffffffu, node, __ffs(need) - 1);
                    double v = 0;
                    const bool ok = leaf3_fast64_warp(t, li, q, rule.ratio, &v) ||
                                    leaf64_warp(t, li, q, rule, squad[INPLACE ? wid : 0], &v);
                    if (lane == 0) {
                        if (ok) acc += v;
                        else st |= GWN_QS_UNRESOLVED;
                    }
                }
            } else if (need && R.val) {
                // this point's pairs number in order; those past its share mark it
                const int j = npair + __popc(need & ((1u << lane) - 1u));
                const unsigned fit = __ballot_sync(0xffffffffu, exact && j < R.per);
                int slot = 0;
                if (lane == 0 && fit) slot = atomicAdd(R.npairs, __popc(fit));
                slot = __shfl_sync(0xffffffffu, slot, 0) + __popc(fit & ((1u << lane) - 1u));
                if (exact && j < R.per) R.pairs[slot] = make_int2(k * R.per + j, ~node);
                npair += __popc(need);
                if (npair > R.per) st |= kPairOverflow;
            } else if (need) {
                long long slot = 0;
                if (lane == 0) slot = list_slots(R.npairs, __popc(need), kRepairPairCap);
                slot = __shfl_sync(0xffffffffu, slot, 0) + __popc(need & ((1u << lane) - 1u));
                if (exact) {
                    if (slot < kRepairPairCap) R.pairs[slot] = make_int2(k, ~node);
                    else st |= kPairOverflow;
                }
            }
            // warp prefix sum of the pushes
            int incl = npush;
            for (int off = 1; off < 32; off <<= 1) {
                int v = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += v;
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            if (npush) {
                stk[sp + incl - 2] = c1;
                stk[sp + incl - 1] = c0;
            }
            sp += total;
            __syncwarp();
        }
        for (int off = 16; off > 0; off >>= 1) {
            acc += __shfl_xor_sync(0xffffffffu, acc, off);
            st |= __shfl_xor_sync(0xffffffffu, st, off);
        }
        if (lane == 0) {
            R.rw[k] = acc;
            R.rst[k] = st;
            if (R.val) R.cnt[k] = INPLACE ? 0 : min(npair, R.per);
        }
        __syncwarp();
    }
}

}  // namespace gwn
