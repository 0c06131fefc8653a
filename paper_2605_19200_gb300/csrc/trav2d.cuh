// trav2d.cuh -- the 2D query on the device: packets of 64 queries in packed fp32x2,
// the far field as a complex polynomial, far leaves in place, near ones through a list.
//
// Far field: away from a cluster its winding number is harmonic, so the folded
// Taylor form (gwn_internal.h) is the real part of a polynomial without constant
// term in zeta = (x + i y) / |r|^2, r = x0 - q:
//     w = Re(zeta (c1 + zeta (c2 + zeta c3))),
// three complex coefficients (6 numbers instead of 12) and 13 operations instead of 35.
// Far leaves (q outside the box of the control points) subtend the angle of their
// chord; most are seen under a small one, where a polynomial of the tangent takes the
// place of atan2.
#pragma once

#include <cstring>

#include "gwn_internal.h"
#include "kernels2d.cuh"
#include "pairs3d.cuh"

namespace gwn {

constexpr int kHarm2 = 6;       // (c1.re c1.im c2.re c2.im c3.re c3.im)
constexpr int kLeaf2Far = 3;    // float4 per leaf: (centre, -max x, -min x) (-max y, -min y, first point) (last point, 0, 0),
                                // box and points relative to the centre
constexpr int kLeaf2Far64 = 8;  // doubles per leaf: min x, max x, min y, max y, first point, last point

// complex coefficients h[6] of a folded block f (fold_moments_2d's layout)
inline void harmonic2_from_folded(const double* f, double* h) {
    const double xx = f[3] + f[2], yy = f[5] + f[2];  // degree 2: quadratic + f2 r^2
    h[0] = f[0];
    h[1] = -f[1];
    h[2] = 0.5 * (xx - yy);
    h[3] = -0.5 * f[4];
    h[4] = f[8] + f[6];                               // degree 3: cubic + r^2 (f6 x + f7 y)
    h[5] = f[11] + f[7];
}

template <typename T>
GWN_HD inline T far2_harm(const T* h, T rx, T ry, T i2) {
    const T x = rx * i2, y = ry * i2;
    const T ur = h[2] + x * h[4] - y * h[5], ui = h[3] + x * h[5] + y * h[4];
    const T vr = h[0] + x * ur - y * ui, vi = h[1] + x * ui + y * ur;
    return x * vr - y * vi;
}

// exact FP64 value of leaf li for a q outside its box, as the complex number whose
// argument is its angle; false inside the box
GWN_HD inline bool leaf2_chord64(const double* L, double qx, double qy, double& dot, double& cross) {
    if (!(L[0] > qx || L[1] < qx || L[2] > qy || L[3] < qy)) return false;
    const double ax = L[4] - qx, ay = L[5] - qy, bx = L[6] - qx, by = L[7] - qy;
    cross = ax * by - ay * bx;
    dot = ax * bx + ay * by;
    return true;
}

// The FP64 sum of leaf angles with one arc tangent for four leaves: an angle of at most
// atan(0.9376) = 43.2 degrees multiplies the running complex number (the product's argument stays
// below 173 degrees, far from the cut at 180, where rounding would decide the sign: leaves of
// exactly 45 degrees are what halved sides of a square show its centre), larger ones and those
// whose product could leave the range of a double take their own.  An FP64 atan2 is about a
// hundred instructions on a pipe that runs at 1/64 of the FP32 rate, a product four; the
// conditions look at the upper words of the two numbers, off that pipe (16384 points on the
// star: 244 us, with FP64 comparisons 3 to 4 % more).
struct Angle64 {
    double re = 1.0, im = 0.0, sum = 0.0;
    double w = 0.0;  // values that are not angles
    int n = 0;
    GWN_HD inline void add(double dot, double cross) {
        unsigned long long bd, bc;
        memcpy(&bd, &dot, sizeof(bd));
        memcpy(&bc, &cross, sizeof(bc));
        const unsigned d = (unsigned)(bd >> 32), c = (unsigned)(bc >> 32) & 0x7fffffffu;
        // dot between 2^-199 and 2^199 (four factors stay within a double); an eighth of a binade above
        // |cross|: at least 1/16 of dot
        if ((d >> 20) - (1023u - 199u) < 398u && c + 0x20000u <= d) {
            const double r = re * dot - im * cross;
            im = re * cross + im * dot;
            re = r;
            if (++n == 4) flush();
        } else {
            sum += atan2(cross, dot);
        }
    }
    GWN_HD inline void flush() {
        if (n) sum += atan2(im, re);
        re = 1.0;
        im = 0.0;
        n = 0;
    }
    GWN_HD inline double value() {  // GWN of the leaves added
        flush();
        return w + sum * Num<double>::inv2pi;
    }
};

#if defined(__CUDACC__)
__device__ __forceinline__ f32x2 dup2(float a) { return pack2(a, a); }

// angle of (dot, cross) for two queries; the halves with |cross| <= dot / 4 (an
// angle below 14 degrees) from the odd series of the arc tangent to t^11 (next term below
// 5e-9 of the angle), the others from atan2f
__device__ __forceinline__ void angle2(f32x2 cross, f32x2 dot, bool on0, bool on1, float& a0, float& a1) {
    float c0, c1, d0, d1;
    unpack2(cross, c0, c1);
    unpack2(dot, d0, d1);
    const f32x2 t = mul2(cross, pack2(rcp_hw(d0), rcp_hw(d1))), t2 = mul2(t, t);
    f32x2 p = fma2(t2, dup2((float)(-1.0 / 11)), dup2((float)(1.0 / 9)));
    p = fma2(t2, p, dup2((float)(-1.0 / 7)));
    p = fma2(t2, p, dup2((float)(1.0 / 5)));
    p = fma2(t2, p, dup2((float)(-1.0 / 3)));
    unpack2(fma2(mul2(t, t2), p, t), a0, a1);
    if (on0 && !(fabsf(c0) <= 0.25f * d0)) a0 = atan2f(c0, d0);
    if (on1 && !(fabsf(c1) <= 0.25f * d1)) a1 = atan2f(c1, d1);
}

// 2D traversal, one packet of 64 binned queries per warp as k_trav3 (masks, warp stack
// of `depth` entries, split over subtrees).  chdr2: per internal node its children's
// (x0, y0, r^2, index).  A leaf whose box holds the query goes to the near list
// (k_near2), a point whose list entry does not fit to olist (k_overflow2).  Two
// runs of a 2D query give the same bits: subtree j's sum of point q goes to
// part[j n + q], summed in order by k_finish, and the near leaves add up in fixed point.
template <bool COUNT>
__global__ void __launch_bounds__(128) k_trav2(DevTree t, const float4* spos, int n, float beta2, int depth, TreeCut cut,
                                               Workspace ws, unsigned long long* work) {
    extern __shared__ int sdyn2[];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned lbit = 1u << lane;
    int* stk_node = sdyn2 + wid * 3 * depth;
    unsigned* stk0 = reinterpret_cast<unsigned*>(stk_node + depth);
    unsigned* stk1 = stk0 + depth;
    WorkLocal wl = {};
    const int q0 = blockIdx.x * 256 + wid * 64 + lane, q1 = q0 + 32;
    const bool act0 = q0 < n, act1 = q1 < n;
    f32x2 nx, ny;  // minus the two points
    {
        float4 a = make_float4(0, 0, 0, 0), b = a;
        if (act0) a = spos[q0];
        if (act1) b = spos[q1];
        nx = pack2(-a.x, -b.x);
        ny = pack2(-a.y, -b.y);
    }
    float w0 = 0.f, w1 = 0.f;
    uint32_t st0 = 0, st1 = 0;
    int sp = 0;  // warp-uniform

    // the queries of m (half h) whose leaf li is not far: to the list
    auto list_near = [&](unsigned m, int q, int li, uint32_t& st) {
        long long slot = 0;  // a full list is not counted further (32-bit count)
        if (lane == 0)
            slot = *(volatile int*)&ws.counters[8] >= ws.slow_cap ? ws.slow_cap
                                                                  : (long long)atomicAdd(&ws.counters[8], __popc(m));
        slot = __shfl_sync(full, slot, 0) + __popc(m & (lbit - 1u));
        if (m & lbit) {
            if (slot < ws.slow_cap) ws.pairs2[slot] = make_int2(q, li);
            else st |= kPairOverflow;
        }
    };
    // node or leaf c (node header h) for the queries of the masks, which return those
    // for which an internal c is near
    auto test = [&](int c, const float4& h, unsigned& m0, unsigned& m1, bool add) {
        const bool in0 = m0 & lbit, in1 = m1 & lbit;
        if (c < 0) {
            const float4* L = t.l2far + (size_t)(~c) * kLeaf2Far;
            const float4 A = __ldg(L), B = __ldg(L + 1);
            const float2 C = __ldg(reinterpret_cast<const float2*>(L + 2));
            const f32x2 rx = add2(dup2(A.x), nx), ry = add2(dup2(A.y), ny);  // centre - q
            float x0, x1, y0, y1;
            unpack2(rx, x0, x1);
            unpack2(ry, y0, y1);
            if (COUNT) wl.v[kWorkLeaves] += (int)in0 + (int)in1;
            // outside the box: min x - (q - centre) > 0 and so on (NaN: inside)
            const bool f0 = in0 && (x0 < A.z || x0 > A.w || y0 < B.x || y0 > B.y);
            const bool f1 = in1 && (x1 < A.z || x1 > A.w || y1 < B.x || y1 > B.y);
            if (f0 || f1) {
                const f32x2 ax = add2(dup2(B.z), rx), ay = add2(dup2(B.w), ry), bx = add2(dup2(C.x), rx),
                            by = add2(dup2(C.y), ry);
                const f32x2 cross = fma2(mul2(ay, bx), dup2(-1.f), mul2(ax, by));
                const f32x2 dot = fma2(ay, by, mul2(ax, bx));
                float a0, a1;
                angle2(cross, dot, f0, f1, a0, a1);
                if (f0) w0 += a0 * Num<float>::inv2pi;
                if (f1) w1 += a1 * Num<float>::inv2pi;
            }
            m0 = __ballot_sync(full, in0 && !f0);
            m1 = __ballot_sync(full, in1 && !f1);
            if (m0) list_near(m0, q0, ~c, st0);
            if (m1) list_near(m1, q1, ~c, st1);
            m0 = m1 = 0u;
            return;
        }
        const f32x2 rx = add2(dup2(h.x), nx), ry = add2(dup2(h.y), ny);
        float ra, rb;
        unpack2(fma2(ry, ry, mul2(rx, rx)), ra, rb);
        const float thr = beta2 * h.z;
        const bool f0 = in0 && ra > thr, f1 = in1 && rb > thr;
        if (COUNT && add) {
            wl.v[kWorkNodes] += (int)in0 + (int)in1;
            wl.v[kWorkFar] += (int)f0 + (int)f1;
        }
        if (add && (f0 || f1)) {
            const float4 A = __ldg(t.hmom2 + 2 * (size_t)c);
            const float2 B = __ldg(reinterpret_cast<const float2*>(t.hmom2 + 2 * (size_t)c + 1));
            const f32x2 i2 = pack2(rcp_hw(ra), rcp_hw(rb));
            const f32x2 x = mul2(rx, i2), y = mul2(ry, i2), my = mul2(y, dup2(-1.f));
            const f32x2 ur = fma2(my, dup2(B.y), fma2(x, dup2(B.x), dup2(A.z)));
            const f32x2 ui = fma2(y, dup2(B.x), fma2(x, dup2(B.y), dup2(A.w)));
            const f32x2 vr = fma2(my, ui, fma2(x, ur, dup2(A.x)));
            const f32x2 vi = fma2(y, ur, fma2(x, ui, dup2(A.y)));
            float a, b;
            unpack2(fma2(my, vi, mul2(x, vr)), a, b);
            if (f0) w0 += a;
            if (f1) w1 += b;
        }
        m0 = __ballot_sync(full, in0 && !f0);
        m1 = __ballot_sync(full, in1 && !f1);
    };

    unsigned m0 = __ballot_sync(full, act0), m1 = __ballot_sync(full, act1);
    // the subtree's ancestors, then its root
    const int4 sub = __ldg(cut.sub + blockIdx.y);
    int node = sub.x;  // warp-uniform
#pragma unroll 1
    for (int k = 0; k <= sub.z && (m0 | m1); ++k) {
        const int e = k < sub.z ? __ldg(cut.path + sub.y + k) : 0;
        const int c = k < sub.z ? e >> 1 : node;
        float4 h = make_float4(0, 0, 0, 0);
        if (c >= 0) {
            h = __ldg(t.hdr + c);
            h.z = h.w;  // (x0, y0, r^2)
        }
        test(c, h, m0, m1, k == sub.z || (e & 1));
    }
    while (m0 | m1) {
        const float4 ha = __ldg(t.chdr2 + 2 * node), hb = __ldg(t.chdr2 + 2 * node + 1);
        const int ca = __float_as_int(ha.w), cb = __float_as_int(hb.w);
        unsigned b0 = m0, b1 = m1;
        test(ca, ha, m0, m1, true);
        test(cb, hb, b0, b1, true);
        if (m0 | m1) {
            if (b0 | b1) {
                if (sp < depth) {
                    if (lane == 0) {
                        stk_node[sp] = cb;
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
            node = ca;
        } else if (b0 | b1) {
            node = cb;
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
    auto put = [&](int q, float w, uint32_t st) {
        ws.part[(size_t)blockIdx.y * n + q] = w;
        if (st && !(atomicOr(&ws.st[q], st) & kPairOverflow) && (st & kPairOverflow))
            ws.olist[atomicAdd(&ws.counters[3], 1)] = q;
    };
    if (act0) put(q0, w0, st0);
    if (act1) put(q1, w1, st1);
    if (COUNT) {
        for (int k = 0; k < kWorkCount; ++k)
            if (wl.v[k]) atomicAdd(&work[k], wl.v[k]);
    }
}

// The listed (query, leaf) pairs whose query lies in the leaf's box, one thread each
// (bisection, FP64 near band in place).  The values add up in units of 2^-40, so that
// their order does not matter (rounding 5e-13, far below an FP32 leaf's).
constexpr float kNearUnit = 1099511627776.f;  // 2^40
__global__ void __launch_bounds__(128) k_near2(DevTree t, const float4* spos, const int* counters, const int2* pairs,
                                               long long cap, float* part, long long* near, uint32_t* st) {
    const long long np = min((long long)counters[8], cap);
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < np; k += (long long)gridDim.x * blockDim.x) {
        const int2 pr = pairs[k];
        const float4 p = spos[pr.x];
        uint32_t s = 0;
        const float v = leaf2_eval32(t, pr.y, p.x, p.y, s);
        if (isfinite(v))
            atomicAdd(reinterpret_cast<unsigned long long*>(&near[pr.x]), (unsigned long long)__float2ll_rn(v * kNearUnit));
        else
            atomicAdd(&part[pr.x], v);
        if (s) atomicOr(&st[pr.x], s);
    }
}

// points whose near pairs did not fit the list: whole traversal, leaves in place
__global__ void __launch_bounds__(128) k_overflow2(DevTree t, const float4* spos, int n, int parts, float beta2,
                                                   Workspace ws) {
    const int cnt = ws.counters[3];
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < cnt; k += gridDim.x * blockDim.x) {
        const int q = ws.olist[k];
        const float4 p = spos[q];
        uint32_t st = 0;
        const float w = query2_32(t, p.x, p.y, beta2, st);
        for (int j = 0; j < parts; ++j) ws.part[(size_t)j * n + q] = j ? 0.f : w;
        ws.near[q] = 0;
        ws.st[q] = st;
    }
}

// the FP32 value of point q of a 2D chunk: its subtrees' sums in order, then the near leaves
__device__ __forceinline__ float value2(const float* part, const long long* near, int n, int parts, int q) {
    float w = part[q];
    for (int j = 1; j < parts; ++j) w += part[(size_t)j * n + q];
    const long long v = near[q];
    return v ? w + (float)((double)v * (1.0 / (double)kNearUnit)) : w;
}

// FP64 value of one leaf into the sums
__device__ __forceinline__ void leaf2_add64(const DevTree& t, int li, double qx, double qy, Angle64& a, uint32_t& st) {
    double dot, cross;
    if (leaf2_chord64(t.l2far64 + (size_t)li * kLeaf2Far64, qx, qy, dot, cross)) a.add(dot, cross);
    else a.w += leaf2_eval64(t, li, qx, qy, st);
}

// 2D FP64 traversal of one query (GWN_PREC_FP64); beta2 <= 0: every leaf.  Leaves
// whose box holds the query wait in `box` (kBoxLeaves entries, `stride` apart) until the
// walk is done: their bisection is long, and in place a warp would go through
// it at every leaf that holds any one of its queries.
constexpr int kBoxLeaves = 8;
__device__ __forceinline__ double query2_harm64(const DevTree& t, double qx, double qy, double beta2, uint32_t& st,
                                                int* box, int stride) {
    int nbox = 0;
    double w = 0.0;
    Angle64 a;
    int stack[kStack64];
    int sp = 0;
    int node = t.root;
    while (true) {
        if (node < 0) {
            double dot, cross;
            if (leaf2_chord64(t.l2far64 + (size_t)(~node) * kLeaf2Far64, qx, qy, dot, cross)) a.add(dot, cross);
            else if (nbox < kBoxLeaves) box[nbox++ * stride] = ~node;
            else a.w += leaf2_eval64(t, ~node, qx, qy, st);
        } else {
            const double* h = t.hdr64 + (size_t)node * 4;
            const double rx = h[0] - qx, ry = h[1] - qy, r2 = rx * rx + ry * ry;
            if (r2 > beta2 * h[3]) {
                w += far2_harm<double>(t.hmom2_64 + (size_t)node * kHarm2, rx, ry, 1.0 / r2);
            } else {
                const int2 ch = t.child[node];
                if (sp < kStack64) stack[sp++] = ch.y; else st |= GWN_QS_UNRESOLVED;
                node = ch.x;
                continue;
            }
        }
        if (sp == 0) break;
        node = stack[--sp];
    }
    for (int j = 0; j < nbox; ++j) a.w += leaf2_eval64(t, box[j * stride], qx, qy, st);
    return w + a.value();
}

// FP64 repair of the listed points, one block per point (the walk of one point is a chain
// of FP64 latencies, and a query lists few): each step the threads take up to
// 256 nodes from the top of the block's stack, add the terms of the far ones and the
// angles of the leaves, and push the children of the others in thread order.
constexpr int kBlockStack2 = 4096;
__global__ void __launch_bounds__(256) k_rtrav2(DevTree t, const void* pts, int dtype, double beta2r, RepairList R,
                                                double* out_w, int* out_label, uint32_t* out_status) {
    __shared__ int stk[kBlockStack2];
    __shared__ int wcnt[8];
    __shared__ double wsum[8];
    __shared__ uint32_t wst[8];
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int cnt = min(*R.count, R.cap);
    for (int k = blockIdx.x; k < cnt; k += gridDim.x) {
        const int qi = R.idx[k];
        double qx, qy;
        if (dtype == GWN_F32) {
            const float* p = reinterpret_cast<const float*>(pts) + (size_t)qi * 2;
            qx = p[0]; qy = p[1];
        } else {
            const double* p = reinterpret_cast<const double*>(pts) + (size_t)qi * 2;
            qx = p[0]; qy = p[1];
        }
        double acc = 0.0;
        Angle64 a;
        uint32_t st = 0;
        if (tid == 0) stk[0] = t.root;
        int sp = 1;  // block-uniform
        __syncthreads();
        while (sp > 0) {
            const int take = stack_take(sp, 256, kBlockStack2);
            if (take <= 0) {
                st |= GWN_QS_UNRESOLVED;  // stack full: the rest is dropped (flagged)
                break;
            }
            const int node = tid < take ? stk[sp - 1 - tid] : 0;
            sp -= take;
            int2 ch = make_int2(0, 0);
            bool push = false;
            if (tid < take) {
                if (node < 0) {
                    leaf2_add64(t, ~node, qx, qy, a, st);
                } else {
                    const double* h = t.hdr64 + (size_t)node * 4;
                    const double rx = h[0] - qx, ry = h[1] - qy, r2 = rx * rx + ry * ry;
                    if (beta2r > 0 && r2 > beta2r * h[3]) {
                        acc += far2_harm<double>(t.hmom2_64 + (size_t)node * kHarm2, rx, ry, 1.0 / r2);
                    } else {
                        ch = t.child[node];
                        push = true;
                    }
                }
            }
            const unsigned m = __ballot_sync(full, push);
            if (lane == 0) wcnt[wid] = __popc(m);
            __syncthreads();
            int at = 0, total = 0;
            for (int w = 0; w < 8; ++w) {
                at += w < wid ? wcnt[w] : 0;
                total += wcnt[w];
            }
            if (push) {
                const int j = sp + 2 * (at + __popc(m & ((1u << lane) - 1u)));
                stk[j] = ch.y;
                stk[j + 1] = ch.x;
            }
            sp += 2 * total;
            __syncthreads();
        }
        acc += a.value();
        for (int off = 16; off > 0; off >>= 1) {
            acc += __shfl_xor_sync(full, acc, off);
            st |= __shfl_xor_sync(full, st, off);
        }
        if (lane == 0) {
            wsum[wid] = acc;
            wst[wid] = st;
        }
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < 8; ++w) {
                acc += wsum[w];
                st |= wst[w];
            }
            out_w[qi] = acc;
            if (out_label) out_label[qi] = (int)round(acc);
            if (out_status) out_status[qi] |= st | GWN_QS_REPAIRED;
        }
        __syncthreads();
    }
}
#endif

}  // namespace gwn
