// few3d.cuh -- 3D FP32 queries of a handful of points.
//
// Where every point of a query lies outside a closed shape, its values are what the rounding
// and the truncation of terms that cancel leave, 1e-5 and less, and any other order of
// the sums or form of the terms changes their leading digits.  Such queries are small ones (a
// box filled to a tenth leaves 16 points all outside one time in five), so queries of
// at most kFewPoints points keep one order and one arithmetic: one packet walks the tree
// child by child, far terms in the folded form (far3_node32), and the exact pairs are
// sorted by leaf and evaluated by one thread each from the tables of x and x' (leaf3_fast32) or
// the curves' Bernstein form (leaf3_try32), which add to their points as they come (a warp's
// in one order, warps almost always in theirs); the direct sum adds its leaves in their order.
// The walk and the near pairs are chains of latencies: on 1.4k leaves 1 point takes 0.3 to 0.5 ms,
// 16 points 0.98 ms (17 points, by k_wide3: 0.15 ms); the direct sum of 16 points 0.52 ms (17:
// 0.12 ms).
#pragma once

#include "gwn_internal.h"
#include "kernels3d.cuh"

namespace gwn {

constexpr int kFewPoints = 16;
constexpr int kFewStack = 128;

// The walk, one warp: the points go through the tree together (masks as in k_trav3), the
// exact leaves' pairs to the list
template <bool O3>
__global__ void __launch_bounds__(32) k_few_walk(DevTree t, const float4* spos, int n, float beta2, float beta2l,
                                                 Workspace ws, unsigned long long* work, int* olist_out) {
    __shared__ int2 stk[kFewStack];
    __shared__ int2 buf[kPairBuf];
    __shared__ unsigned char own[kPairBuf];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    WorkLocal wl = {};
    const int qi = lane;
    const bool active = qi < n;
    float q[3] = {0, 0, 0};
    if (active) {
        const float4 p = spos[qi];
        q[0] = p.x; q[1] = p.y; q[2] = p.z;
    }
    float w = 0.f;
    uint32_t st = 0;
    int bcnt = 0;      // warp-uniform: entries in buf
    unsigned nfound = 0;
    unsigned ovf = 0;  // lanes with pairs that did not fit the list
    int sp = 0;        // warp-uniform

    // node or leaf c (header h) for the lanes of msk; returns those for which an internal c is near
    auto test = [&](int c, unsigned msk, const float4& h) -> unsigned {
        const bool mine = (msk >> lane) & 1u;
        if (c < 0) {
            const int li = ~c;
            const float rx = h.x - q[0], ry = h.y - q[1], rz = h.z - q[2];
            const bool far = mine && t.leaf_far && rx * rx + ry * ry + rz * rz > beta2l * h.w;
            if (work && mine) wl.v[kWorkLeafTests] += 1;
            if (far) {
                if (work) wl.v[kWorkFar] += 1;
                w += far3_node32(t.lmom + (size_t)li * kMom3Vec, rx, ry, rz, O3);
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
        const float rx = h.x - q[0], ry = h.y - q[1], rz = h.z - q[2];
        const bool far = mine && rx * rx + ry * ry + rz * rz > beta2 * h.w;
        if (work && mine) wl.v[kWorkNodes] += 1;
        if (far) {
            if (work) wl.v[kWorkFar] += 1;
            w += far3_node32(t.mom + (size_t)c * kMom3Vec, rx, ry, rz, O3);
        }
        return __ballot_sync(full, mine && !far);
    };

    int node = t.root;  // warp-uniform
    unsigned mask = __ballot_sync(full, active);
    if (mask) mask = test(node, mask, node < 0 ? GWN_LDG(t.lhdr + ~node) : GWN_LDG(t.hdr + node));  // the root
    while (mask) {
        const int2 ch = GWN_LDG(t.child + node);
        const float4 ha = GWN_LDG(t.chdr + 2 * node), hb = GWN_LDG(t.chdr + 2 * node + 1);
        const unsigned na = test(ch.x, mask, ha);
        const unsigned nb = test(ch.y, mask, hb);
        if (na) {
            if (nb) {
                if (sp < kFewStack) {
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

// Counting sort of the few points' pairs by leaf, one block.  A leaf's pairs stand next to
// each other in the list (one warp wrote it, a leaf at a time), and keep their order.
__global__ void __launch_bounds__(1024) k_few_sort(int n_leaves, long long cap, const int* counters, const int2* pairs,
                                                   int* first, int2* out) {
    __shared__ int part[32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int np = (int)min((long long)counters[0], cap);
    for (int l = tid; l < n_leaves; l += 1024) first[l] = 0;
    __syncthreads();
    for (int k = tid; k < np; k += 1024) atomicAdd(&first[pairs[k].y], 1);
    __syncthreads();
    // exclusive scan, a range of leaves per thread
    const int per = (n_leaves + 1023) / 1024, l0 = min(tid * per, n_leaves), l1 = min(l0 + per, n_leaves);
    int sum = 0;
    for (int l = l0; l < l1; ++l) sum += first[l];
    const int incl = warp_incl_scan(sum);
    if (lane == 31) part[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        const int p = part[lane];
        part[lane] = warp_incl_scan(p) - p;
    }
    __syncthreads();
    int at = part[wid] + incl - sum;
    for (int l = l0; l < l1; ++l) {
        const int c = first[l];
        first[l] = at;
        at += c;
    }
    __syncthreads();
    for (int k = tid; k < np; k += 1024) {
        const int2 pr = pairs[k];
        int j = k;
        while (j > 0 && pairs[j - 1].y == pr.y) --j;
        out[first[pr.y] + k - j] = pr;
    }
}

// the sorted pairs whose point lies outside the leaf's 1.1-radius sphere and whose panels stop at
// level 0 or 1, from the tables; the others, in order, to `slow`
__global__ void __launch_bounds__(128) k_few_fast(DevTree t, const float4* spos, long long npair_cap, int* counters,
                                                  const int2* pairs, float* wacc, const uint32_t* st, int2* slow,
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
            if (!(st[pr.x] & kPairOverflow)) {  // k_overflow3 evaluates the point
                const float4 p = spos[pr.x];
                const float q[3] = {p.x, p.y, p.z};
                const Leaf3Info I = t.leaf3[pr.y];
                const float qr[3] = {q[0] - I.cen[0], q[1] - I.cen[1], q[2] - I.cen[2]};
                const float d2 = qr[0] * qr[0] + qr[1] * qr[1] + qr[2] * qr[2];
                const float rfar = 1.1f * I.rad;
                float v;
                if (d2 > rfar * rfar && leaf3_fast32(t, I, qr, d2, &v, work ? &wl : nullptr))
                    atomicAdd(&wacc[pr.x], v);
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
            if (to_slow) slow[slot0 + __popc(m & ((1u << lane) - 1u))] = pr;
        }
    }
    if (work) flush_work(wl, work);
}

// those, one thread each; what FP32 cannot resolve to the near band
__global__ void __launch_bounds__(128, 5) k_few_eval(DevTree t, const float4* spos, int* counters, const int2* pairs,
                                                     float* wacc, uint32_t* st, int2* pairs64, int npair64_cap,
                                                     unsigned long long* work) {
    WorkLocal wl = {};
    const int np = counters[8];
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < np; k += gridDim.x * blockDim.x) {
        const int2 pr = pairs[k];
        const float4 p = spos[pr.x];
        float v;
        if (leaf3_try32(t, pr.y, p.x, p.y, p.z, &v, work ? &wl : nullptr, false)) {
            atomicAdd(&wacc[pr.x], v);
        } else {
            const int slot = atomicAdd(&counters[2], 1);
            if (slot < npair64_cap) pairs64[slot] = pr;
            atomicOr(&st[pr.x], slot < npair64_cap ? GWN_QS_NEAR : GWN_QS_STACK_OVERFLOW);
        }
    }
    if (work) flush_work(wl, work);
}

// The direct sum: every leaf of every point, one thread each, and the sums in leaf order
__global__ void __launch_bounds__(128) k_few_direct(DevTree t, const float4* spos, int n, float* val, uint32_t* st) {
    const long long np = (long long)n * t.n_leaves;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < np; k += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(k / t.n_leaves);
        const float4 p = spos[i];
        uint32_t s = 0;
        val[k] = leaf3_eval32(t, (int)(k % t.n_leaves), p.x, p.y, p.z, s);
        if (s) atomicOr(&st[i], s);
    }
}
__global__ void __launch_bounds__(32 * kFewPoints) k_few_direct_sum(int n, int n_leaves, const float* val, double* acc) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, i = threadIdx.x >> 5;
    if (i >= n) return;
    double w = 0.0;
    for (int l0 = 0; l0 < n_leaves; l0 += 32) {
        const float v = l0 + lane < n_leaves ? val[(size_t)i * n_leaves + l0 + lane] : 0.f;
        const int c = min(32, n_leaves - l0);
        for (int j = 0; j < c; ++j) w += (double)__shfl_sync(full, v, j);
    }
    if (lane == 0) acc[i] = w;
}

}  // namespace gwn
