// gwn_api.cu -- the C ABI (include/gwn.h): model construction, device upload,
// batched queries and inspection.
//
// A query runs in chunks of at most kChunk points (enqueue_chunk; the stages are in
// query_pipeline.cuh and trav2d.cuh), then one FP64 repair pass over the points the
// chunks listed.  Every stage is driven by counters in device memory on the caller's
// stream: no host synchronisation inside a query.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <tuple>
#include <vector>

#include <sys/stat.h>

#include "../../include/gwn.h"
#include "build.h"
#include "gwn_internal.h"
#include "kernels2d.cuh"
#include "kernels3d.cuh"
#include "query_pipeline.cuh"
#include "model.h"

using namespace gwn;

namespace {
thread_local std::string g_err;

gwn_status fail(gwn_status s, const std::string& msg) {
    g_err = msg;
    return s;
}

#define GWN_CUDA_TRY(call)                                                                    \
    do {                                                                                      \
        cudaError_t e_ = (call);                                                              \
        if (e_ != cudaSuccess) return fail(GWN_ERR_CUDA, std::string(#call ": ") + cudaGetErrorString(e_)); \
    } while (0)

struct DeviceGuard {
    int prev = -1;
    bool changed = false;
    explicit DeviceGuard(int dev) {
        cudaGetDevice(&prev);
        if (dev >= 0 && dev != prev) {
            cudaSetDevice(dev);
            changed = true;
        }
    }
    ~DeviceGuard() {
        if (changed) cudaSetDevice(prev);
    }
};
}  // namespace



namespace {

template <typename V>
gwn_status upload(gwn_model_s* m, const std::vector<V>& v, const V** out) {
    *out = nullptr;
    if (v.empty()) return GWN_OK;
    void* p = nullptr;
    size_t bytes = v.size() * sizeof(V);
    cudaError_t e = cudaMalloc(&p, bytes);
    if (e != cudaSuccess) return fail(GWN_ERR_OOM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
    m->allocs.push_back(p);
    m->device_bytes += bytes;
    GWN_CUDA_TRY(cudaMemcpy(p, v.data(), bytes, cudaMemcpyHostToDevice));
    *out = reinterpret_cast<const V*>(p);
    return GWN_OK;
}

void free_model_memory(gwn_model_s* m) {
    for (void* p : m->allocs) cudaFree(p);
    m->allocs.clear();
    if (m->ws_mem) cudaFree(m->ws_mem);
    if (m->stage) cudaFree(m->stage);
    for (auto& row : m->ev)
        for (auto& e : row)
            if (e) cudaEventDestroy(e), e = nullptr;
    if (m->last) cudaEventDestroy(m->last);
    m->last = nullptr;
    m->last_recorded = false;
    m->ws_mem = nullptr;
    m->ws_bytes = 0;
    m->ws_n = 0;
    m->stage = nullptr;
    m->stage_cap = 0;
}

// constant tables of the 3D kernels (binomial coefficients, 8-point
// Gauss-Legendre rule on [0, 1]); uploaded once per device
std::mutex g_const_mu;
bool g_const_ready[256];

gwn_status init_constants(int dev) {
    std::lock_guard<std::mutex> lk(g_const_mu);
    if (dev < 0 || dev >= 256) return fail(GWN_ERR_INVALID_ARG, "device ordinal out of range");
    if (g_const_ready[dev]) return GWN_OK;
    float bin[kMaxC3Deg + 1][kMaxC3Deg + 1] = {};
    for (int a = 0; a <= kMaxC3Deg; ++a) {
        bin[a][0] = bin[a][a] = 1.f;
        for (int b = 1; b < a; ++b) bin[a][b] = bin[a - 1][b - 1] + bin[a - 1][b];
    }
    // n-point Gauss-Legendre nodes and weights on [0, 1]: Newton's method on the
    // Legendre polynomial P_n from the standard cosine initial guesses
    auto gauss = [](int n, double* x, double* w) {
        for (int i = 0; i < n; ++i) {
            double z = std::cos(M_PI * (i + 0.75) / (n + 0.5)), pp = 1;
            for (int it = 0; it < 100; ++it) {
                double p1 = 1, p2 = 0;
                for (int j = 1; j <= n; ++j) {
                    double p3 = p2;
                    p2 = p1;
                    p1 = ((2.0 * j - 1) * z * p2 - (j - 1.0) * p3) / j;
                }
                pp = n * (z * p1 - p2) / (z * z - 1);
                double dz = p1 / pp;
                z -= dz;
                if (std::fabs(dz) < 1e-16) break;
            }
            x[i] = 0.5 * (1 - z);
            w[i] = 1.0 / ((1 - z * z) * pp * pp);
        }
    };
    double x[8], w[8], x4[4], w4[4];
    gauss(8, x, w);
    gauss(4, x4, w4);
    float xf[4], wf[4];
    for (int i = 0; i < 4; ++i) {
        xf[i] = (float)x4[i];
        wf[i] = (float)w4[i];
    }
    std::memcpy(h_binom, bin, sizeof(bin));
    std::memcpy(h_glx8, x, sizeof(x));
    std::memcpy(h_glw8, w, sizeof(w));
    std::memcpy(h_glx4f, xf, sizeof(xf));
    std::memcpy(h_glw4f, wf, sizeof(wf));
    std::memcpy(h_glx4d, x4, sizeof(x4));
    std::memcpy(h_glw4d, w4, sizeof(w4));
    GWN_CUDA_TRY(cudaMemcpyToSymbol(c_glx4d, x4, sizeof(x4)));
    GWN_CUDA_TRY(cudaMemcpyToSymbol(c_glw4d, w4, sizeof(w4)));
    GWN_CUDA_TRY(cudaMemcpyToSymbol(c_glx4f, xf, sizeof(xf)));
    GWN_CUDA_TRY(cudaMemcpyToSymbol(c_glw4f, wf, sizeof(wf)));
    GWN_CUDA_TRY(cudaMemcpyToSymbol(c_binom, bin, sizeof(bin)));
    GWN_CUDA_TRY(cudaMemcpyToSymbol(c_glx8, x, sizeof(x)));
    GWN_CUDA_TRY(cudaMemcpyToSymbol(c_glw8, w, sizeof(w)));
    g_const_ready[dev] = true;
    return GWN_OK;
}

// device memory owned by the model, for arrays derived on the device
template <typename V>
gwn_status device_array(gwn_model_s* m, size_t n, V** out) {
    *out = nullptr;
    void* p = nullptr;
    cudaError_t e = cudaMalloc(&p, std::max<size_t>(1, n * sizeof(V)));
    if (e != cudaSuccess) return fail(GWN_ERR_OOM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
    m->allocs.push_back(p);
    m->device_bytes += n * sizeof(V);
    *out = reinterpret_cast<V*>(p);
    return GWN_OK;
}

// the tables of the exact pairs (pairs3d.cuh), from the uploaded leaf records and
// node tables; not part of a saved model
gwn_status derive_pair_tables(gwn_model_s* m) {
    DevTree& t = m->tree;
    const size_t nc = m->host.c3.size(), nl = (size_t)t.n_leaves;
    float4 *c3m, *lfar, *lhit;
    int2* lrange;
    gwn_status s;
    if ((s = device_array(m, nc * kC3NodeVec, &c3m)) != GWN_OK || (s = device_array(m, nl, &lfar)) != GWN_OK ||
        (s = device_array(m, nl, &lrange)) != GWN_OK || (s = device_array(m, nl * 3, &lhit)) != GWN_OK)
        return s;
    if (nc) {
        k_node_moments<<<(unsigned)((nc * 6 + 127) / 128), 128>>>((long long)nc, t.c3n, c3m);
        // the uploaded FP64 tables become the far form: nothing on the device reads x'
        k_node_moments64<<<(unsigned)nl, 128>>>(t.leaf3, const_cast<double*>(t.c3n64));
        t.c3m64 = t.c3n64;
        t.c3n64 = nullptr;
    }
    k_leaf_far<<<(unsigned)((nl + 127) / 128), 128>>>((int)nl, t.leaf3, t.net3, lfar, lrange, lhit);
    GWN_CUDA_TRY(cudaGetLastError());
    GWN_CUDA_TRY(cudaStreamSynchronize(0));  // queries may come on streams that do not wait for this one
    t.c3m = c3m;
    t.lfar = lfar;
    t.lrange = lrange;
    t.lhit = lhit;
    return GWN_OK;
}

// the tree's cuts for split packets (TreeCut): the subtree with the most leaves is
// replaced by its children until there are enough
gwn_status upload_cuts(gwn_model_s* m) {
    const HostModel& H = m->host;
    const int ni = (int)H.child.size();
    std::vector<int> leaves(ni, 0), order, parent(ni, -1), leaf_parent(H.n_leaves, -1);
    if (ni) order.push_back(0);
    for (size_t k = 0; k < order.size(); ++k)
        for (int c : {H.child[order[k]].x, H.child[order[k]].y}) {
            (c < 0 ? leaf_parent[~c] : parent[c]) = order[k];
            if (c >= 0) order.push_back(c);
        }
    for (size_t k = order.size(); k-- > 0;)
        for (int c : {H.child[order[k]].x, H.child[order[k]].y}) leaves[order[k]] += c < 0 ? 1 : leaves[c];
    std::vector<int4> sub;
    std::vector<int> path, roots{m->tree.root};
    std::vector<std::pair<size_t, size_t>> at;  // per cut: offsets into sub and path
    for (int level = 0; level < kCutLevels; ++level) {
        while ((int)roots.size() < 1 << level) {
            size_t big = 0;
            for (size_t j = 1; j < roots.size(); ++j)
                if ((roots[j] < 0 ? 1 : leaves[roots[j]]) > (roots[big] < 0 ? 1 : leaves[roots[big]])) big = j;
            if (roots[big] < 0) break;  // only leaves left
            const int2 ch = H.child[roots[big]];
            roots[big] = ch.x;
            roots.insert(roots.begin() + big + 1, ch.y);
        }
        at.push_back({sub.size(), path.size()});
        m->cut_size[level] = (int)roots.size();
        std::vector<char> seen(ni, 0);
        for (size_t j = 0; j < roots.size(); ++j) {
            std::vector<int> up;
            for (int k = roots[j] < 0 ? leaf_parent[~roots[j]] : parent[roots[j]]; k >= 0; k = parent[k]) up.push_back(k);
            sub.push_back(int4{roots[j], (int)(path.size() - at.back().second), (int)up.size(), 0});
            for (size_t k = up.size(); k-- > 0;) {
                path.push_back(2 * up[k] + (seen[up[k]] ? 0 : 1));
                seen[up[k]] = 1;
            }
        }
    }
    path.push_back(0);
    const int4* ds;
    const int* dp;
    gwn_status s;
    if ((s = upload(m, sub, &ds)) != GWN_OK || (s = upload(m, path, &dp)) != GWN_OK) return s;
    for (int level = 0; level < kCutLevels; ++level) m->cuts[level] = TreeCut{ds + at[level].first, dp + at[level].second};
    return GWN_OK;
}

gwn_status upload_model(gwn_model_s* m) {
    {
        int dev = 0;
        cudaGetDevice(&dev);
        gwn_status cs = init_constants(dev);
        if (cs != GWN_OK) return cs;
    }
    const HostModel& H = m->host;
    DevTree& t = m->tree;
    t.dim = H.dim;
    t.n_leaves = H.n_leaves;
    t.n_internal = H.n_leaves - 1;
    t.root = H.n_leaves > 1 ? 0 : ~0;
    gwn_status s;
#define UP(vec, field) if ((s = upload(m, H.vec, &t.field)) != GWN_OK) return s
    t.leaf_far = m->leaf_far;
    t.order3 = H.dim == 3 && m->eval_order >= 3 ? 1 : 0;
    t.order3_64 = H.dim == 3 && m->opts.order >= 3 ? 1 : 0;
    UP(lhdr, lhdr);
    UP(lmom, lmom);
    UP(lhdr64, lhdr64);
    UP(hdr, hdr);
    UP(child, child);
    {
        // both children's headers beside each internal node (3D traversal): the
        // child indices and the headers load together instead of one after the other
        std::vector<float4> chdr;
        if (H.dim == 3) {
            chdr.resize(H.child.size() * 2);
            for (size_t k = 0; k < H.child.size(); ++k) {
                const int c[2] = {H.child[k].x, H.child[k].y};
                for (int j = 0; j < 2; ++j) chdr[2 * k + j] = c[j] < 0 ? H.lhdr[~c[j]] : H.hdr[c[j]];
            }
        }
        if ((s = upload(m, chdr, &t.chdr)) != GWN_OK) return s;
    }
    UP(mom, mom);
    if (H.dim == 3) {
        // the far field's harmonic coefficients (far3d.cuh), nodes then leaves
        t.hstride = m->opts.order >= 3 ? 6 : 4;
        const size_t ni = H.child.size(), nl = (size_t)H.n_leaves;
        std::vector<float4> hm((ni + nl) * t.hstride);
        std::vector<double> hm64((ni + nl) * kHarm);
        for (size_t k = 0; k < ni + nl; ++k) {
            double* h = &hm64[k * kHarm];
            harmonic_from_folded(k < ni ? &H.mom64[k * kMom3F64] : &H.lmom64[(k - ni) * kMom3F64], h);
            float* f = reinterpret_cast<float*>(&hm[k * t.hstride]);
            for (int j = 0; j < 4 * t.hstride; ++j) f[j] = (float)h[j];
        }
        if ((s = upload(m, hm, &t.hmom)) != GWN_OK || (s = upload(m, hm64, &t.hmom64)) != GWN_OK) return s;
    } else {
        // 2D (trav2d.cuh): children's headers with their indices, complex far coefficients,
        // and what a far query needs of a leaf
        const size_t ni = H.child.size(), nl = (size_t)H.n_leaves;
        std::vector<float4> ch(2 * ni), hm(2 * ni, float4{0, 0, 0, 0}), lf(nl * kLeaf2Far, float4{0, 0, 0, 0});
        std::vector<double> hm64(ni * kHarm2), lf64(nl * kLeaf2Far64);
        for (size_t k = 0; k < ni; ++k) {
            const int c[2] = {H.child[k].x, H.child[k].y};
            for (int j = 0; j < 2; ++j) {
                float idx;
                std::memcpy(&idx, &c[j], 4);
                const float4 h = c[j] < 0 ? float4{0, 0, 0, 0} : H.hdr[c[j]];
                ch[2 * k + j] = float4{h.x, h.y, h.w, idx};
            }
            double* h = &hm64[k * kHarm2];
            harmonic2_from_folded(&H.mom64[k * kMom2F64], h);
            hm[2 * k] = float4{(float)h[0], (float)h[1], (float)h[2], (float)h[3]};
            hm[2 * k + 1] = float4{(float)h[4], (float)h[5], 0, 0};
        }
        for (size_t l = 0; l < nl; ++l) {
            const float* L = reinterpret_cast<const float*>(&H.leaf2[l * kLeaf2Vec]);  // offsets x y, weights, centre
            const double* D = &H.leaf2_64[l * kLeaf2F64];
            float lo[2] = {L[0], L[1]}, hi[2] = {L[0], L[1]};
            double* E = &lf64[l * kLeaf2Far64];
            for (int c = 0; c < 2; ++c) {
                E[2 * c] = E[2 * c + 1] = D[c];
                for (int j = 1; j < 4; ++j) {
                    lo[c] = std::min(lo[c], L[2 * j + c]);
                    hi[c] = std::max(hi[c], L[2 * j + c]);
                    E[2 * c] = std::min(E[2 * c], D[2 * j + c]);
                    E[2 * c + 1] = std::max(E[2 * c + 1], D[2 * j + c]);
                }
                E[4 + c] = D[c];
                E[6 + c] = D[6 + c];
            }
            lf[3 * l] = float4{L[12], L[13], -hi[0], -lo[0]};
            lf[3 * l + 1] = float4{-hi[1], -lo[1], L[0], L[1]};
            lf[3 * l + 2] = float4{L[6], L[7], 0, 0};
        }
        if ((s = upload(m, ch, &t.chdr2)) != GWN_OK || (s = upload(m, hm, &t.hmom2)) != GWN_OK ||
            (s = upload(m, hm64, &t.hmom2_64)) != GWN_OK || (s = upload(m, lf, &t.l2far)) != GWN_OK ||
            (s = upload(m, lf64, &t.l2far64)) != GWN_OK)
            return s;
    }
    UP(hdr64, hdr64);
    UP(leaf2, leaf2);
    UP(leaf2_64, leaf2_64);
    UP(leaf3, leaf3);
    UP(net3, net3);
    UP(net3_64, net3_64);
    UP(c3, c3);
    UP(c3pts, c3pts);
    UP(c3pts64, c3pts64);
    UP(c3n, c3n);
    UP(c3n64, c3n64);
    UP(c2, c2);
    UP(c2_64, c2_64);
    UP(c2mult, c2mult);
#undef UP
    if ((s = upload_cuts(m)) != GWN_OK) return s;
    if (H.dim == 3) return derive_pair_tables(m);
    return GWN_OK;
}

gwn_status finish_build(gwn_model_s* m, gwn_model* out) {
    // the packet traversal's warp stack holds the pending second children along
    // one root-to-leaf path: sized from the tree's depth (deeper paths overflow,
    // are flagged and repaired)
    const int need = m->host.max_depth + 8;
    m->stack_depth = need <= 64 ? 64 : need <= 96 ? 96 : 128;
    gwn_status s = upload_model(m);
    if (s != GWN_OK) {
        free_model_memory(m);
        delete m;
        return s;
    }
    *out = m;
    return GWN_OK;
}

gwn_status check_opts(const gwn_build_opts& o, int dim) {
    if (!(o.beta == 0.0 || o.beta >= 2.0) || !std::isfinite(o.beta)) return fail(GWN_ERR_INVALID_ARG, "beta must be 0 (autotune) or >= 2");
    if (!(o.beta_leaf == 0.0 || o.beta_leaf >= 2.0)) return fail(GWN_ERR_INVALID_ARG, "beta_leaf must be 0 or >= 2");
    if (o.order < 0 || o.order > (dim == 3 ? 3 : 2))
        return fail(GWN_ERR_INVALID_ARG, dim == 3 ? "order must be 0, 1, 2 or 3" : "order must be 0, 1 or 2");
    if (o.adaptive_beta != 0 && o.adaptive_beta != 1) return fail(GWN_ERR_INVALID_ARG, "adaptive_beta must be 0 or 1");
    if (o.device_build < -1 || o.device_build > 1) return fail(GWN_ERR_INVALID_ARG, "device_build must be -1, 0 or 1");
    if (o.tree_builder < -1 || o.tree_builder > 1) return fail(GWN_ERR_INVALID_ARG, "tree_builder must be -1, 0 or 1");
    if (!(o.local_ratio <= 0.0 || (o.local_ratio >= 4.0 && o.local_ratio < 1e6)))
        return fail(GWN_ERR_INVALID_ARG, "local_ratio must be <= 0 or in [4, 1e6)");
    if (!(o.beta_repair <= 0.0 || o.beta_repair >= 2.0)) return fail(GWN_ERR_INVALID_ARG, "beta_repair must be <= 0 or >= 2");
    if (!(o.repair_band >= 0.0 && o.repair_band < 0.5)) return fail(GWN_ERR_INVALID_ARG, "repair_band must be in [0, 0.5)");
    if (o.quad_nodes < 1 || o.quad_nodes > 32) return fail(GWN_ERR_INVALID_ARG, "quad_nodes must be 1..32");
    if (o.precision < 0 || o.precision > 2) return fail(GWN_ERR_INVALID_ARG, "unknown precision");
    return GWN_OK;
}

// ------------------------------------------------------------------ kernels

__device__ __forceinline__ void load_point(const void* pts, int dtype, int dim, long long i, double* q) {
    if (dtype == GWN_F32) {
        const float* p = reinterpret_cast<const float*>(pts) + i * dim;
        for (int k = 0; k < dim; ++k) q[k] = (double)p[k];
    } else {
        const double* p = reinterpret_cast<const double*>(pts) + i * dim;
        for (int k = 0; k < dim; ++k) q[k] = p[k];
    }
}

__device__ __forceinline__ bool near_half(double w, float band) {
    double fr = w - floor(w);
    return fabs(fr - 0.5) < (double)band;
}

// 2D direct sum, FP32 leaves
__global__ void __launch_bounds__(128) k_query32(DevTree t, const void* pts, int dtype, long long n, QueryParams p,
                                                 double* out_w, int* out_label, uint32_t* out_status, int* rlist,
                                                 int* rcount) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double qd[3];
    load_point(pts, dtype, 2, i, qd);
    uint32_t st = 0;
    // the direct sum adds one FP32 value per leaf (thousands per query): the
    // running sum is kept in FP64 so that its rounding stays below the leaves' own
    double wd = 0.0;
    for (int l = 0; l < t.n_leaves; ++l) wd += (double)leaf2_eval32(t, l, (float)qd[0], (float)qd[1], st);
    if (p.precision == GWN_PREC_FP32_REPAIR &&
        (near_half(wd, p.band) || (st & (GWN_QS_STACK_OVERFLOW | GWN_QS_UNRESOLVED)))) {
        int slot = atomicAdd(rcount, 1);
        rlist[slot] = (int)i;
    }
    out_w[i] = wd;
    if (out_label) out_label[i] = (int)round(wd);
    if (out_status) out_status[i] = st;
}

// 2D FP64 pass over every query (precision GWN_PREC_FP64)
__global__ void __launch_bounds__(64) k_query64(DevTree t, const void* pts, int dtype, long long n, QueryParams p,
                                                 double* out_w, int* out_label, uint32_t* out_status) {
    __shared__ int box[kBoxLeaves][64];
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double q[3];
    load_point(pts, dtype, 2, i, q);
    uint32_t st = 0;
    double w = query2_harm64(t, q[0], q[1], (double)p.beta2, st, &box[0][threadIdx.x], 64);
    out_w[i] = w;
    if (out_label) out_label[i] = (int)round(w);
    if (out_status) out_status[i] = st;
}

__global__ void k_iota(int n, int* list, int* count) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) list[i] = i;
    if (i == 0) *count = n;
}

// 2D FP64 values of the listed queries (persistent grid over the device-side
// count).  With beta_repair > 0 each thread re-runs the traversal in FP64;
// with beta_repair == 0 (exact direct sum) a whole warp shares one query, its
// lanes striding over the leaves, so that few repaired queries still fill the
// FP64 pipes.
__global__ void __launch_bounds__(128) k_repair2(DevTree t, const void* pts, int dtype, QueryParams p, double* out_w,
                                                 int* out_label, uint32_t* out_status, const int* rlist,
                                                 const int* rcount, int cap = 0x7fffffff) {
    __shared__ int box[kBoxLeaves][128];
    int cnt = min(*rcount, cap);
    bool direct = p.mode == GWN_MODE_DIRECT || !(p.beta2_repair > 0);
    if (!direct) {
        for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < cnt; k += gridDim.x * blockDim.x) {
            int i = rlist[k];
            double q[3];
            load_point(pts, dtype, 2, i, q);
            uint32_t st = 0;
            double w = query2_harm64(t, q[0], q[1], p.beta2_repair, st, &box[0][threadIdx.x], 128);
            out_w[i] = w;
            if (out_label) out_label[i] = (int)round(w);
            if (out_status) out_status[i] = (out_status[i] | st | GWN_QS_REPAIRED);
        }
        return;
    }
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int k = warp; k < cnt; k += nwarps) {
        int i = rlist[k];
        double q[3];
        load_point(pts, dtype, 2, i, q);
        uint32_t st = 0;
        Angle64 a;
        for (int l = lane; l < t.n_leaves; l += 32) leaf2_add64(t, l, q[0], q[1], a, st);
        double w = a.value();
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            w += __shfl_xor_sync(0xffffffffu, w, off);
            st |= __shfl_xor_sync(0xffffffffu, st, off);
        }
        if (lane == 0) {
            out_w[i] = w;
            if (out_label) out_label[i] = (int)round(w);
            if (out_status) out_status[i] = (p.precision == GWN_PREC_FP64 ? 0u : out_status[i]) | st | GWN_QS_REPAIRED;
        }
    }
}

// Bytes of the query workspace for n points of model m, and its layout.
// dim 0 lays out a workspace that serves both 2D and 3D models.
size_t workspace_layout(int dim, int n_leaves, size_t n, char* base, Workspace* ws) {
    // (point, leaf) pairs: 128 per point, and for fewer points, which may all lie next to the
    // surface of a dense model, up to 768 within 2^26 pairs (0.5 GB; points past it are walked
    // again without the list); at least as many as hold the FP64 pairs' values (rval) in the place
    // of this list and the next, which GWN_PREC_FP64 does not use
    long long cap = 0;
    if (dim != 2) {
        cap = std::max((long long)n * 128 + 65536, (kRepairPairCap * 4 / 5 + 63) & ~63ll);
        if (dim == 3) cap = std::max(cap, std::min((long long)n * std::min(n_leaves, 768), 1ll << 26) & ~63ll);
    }
    const size_t cells = kMaxBinCells;  // the finest binning of either dimension
    const size_t hist = std::max(cells + kMaxBinCells / kScanTile,  // and the scan's tile sums
                                 (size_t)n_leaves);                // k_few_sort: an entry per leaf
    const size_t keyn = n;
    size_t off = 0;
    auto carve = [&](size_t bytes) {
        char* p = base ? base + off : nullptr;
        off += (bytes + 255) & ~size_t(255);
        return p;
    };
    Workspace w{};
    w.spos = (float4*)carve(n * sizeof(float4));
    w.key = (int*)carve(keyn * sizeof(int));
    w.hist = (int*)carve(hist * sizeof(int));
    w.wacc = (float*)carve(n * sizeof(float));
    w.st = (uint32_t*)carve(n * sizeof(uint32_t));
    w.pairs = (int2*)carve((size_t)cap * sizeof(int2));
    // pairs left to the full evaluator (a few per cent); 2D: leaves whose box holds the point
    const long long slow = dim == 2 ? (long long)n * 8 + 65536 : cap / 4;
    w.pairs2 = (int2*)carve((size_t)slow * sizeof(int2));
    w.rpairs = (int2*)carve((dim != 2 ? (size_t)kRepairPairCap : 0) * sizeof(int2));
    w.rpairs2 = (int2*)carve((dim != 2 ? (size_t)kRepairPairCap : 0) * sizeof(int2));
    w.part = (float*)carve((dim != 3 ? kParts2 : 0) * sizeof(float));
    w.near = (long long*)carve((dim != 3 ? n : 0) * sizeof(long long));
    w.rw = (double*)carve(n * sizeof(double));
    w.rval = (double*)w.pairs;
    w.rcnt = (int*)carve((dim != 2 ? n : 0) * sizeof(int));
    // the near band: two or three pairs for a point on the surface, and whatever a small query has
    const long long near = dim == 2 ? 0 : (long long)n * 4 + (1 << 18);
    w.near_cap = (int)near;
    w.pairs64 = (int2*)carve((size_t)near * sizeof(int2));
    w.rlist = (int*)carve(n * sizeof(int));
    w.rlist_g = (int*)carve(n * sizeof(int));
    w.rst = (uint32_t*)carve(n * sizeof(uint32_t));
    w.rcap = (int)n;
    w.list_points = (int)n;
    w.olist = (int*)carve(n * sizeof(int));
    w.olist2 = (int*)carve((dim != 2 ? n : 0) * sizeof(int));
    w.work = (unsigned long long*)carve(kWorkCount * sizeof(unsigned long long));
    // control words, 256 bytes each, cleared together: the query's, then the chunk's
    w.acc = (unsigned long long*)carve(kCounterCount * sizeof(unsigned long long));
    w.gcount = (int*)carve(8 * sizeof(int));
    w.counters = (int*)carve(kCounterCount * sizeof(int) + 2 * sizeof(unsigned long long));
    w.found = (unsigned long long*)(w.counters + kCounterCount);  // cleared with the counters
    w.bbox = (unsigned*)carve(8 * sizeof(unsigned));
    w.pair_cap = cap;
    w.slow_cap = slow;
    if (ws) *ws = w;
    return off;
}

constexpr size_t kControlBytes = 256;        // acc, gcount, counters and bbox of a workspace
constexpr size_t kChunk = (size_t)1 << 20;  // points per pass of the query pipeline
// 3D queries of at most this many points take one warp per point (k_wide3), larger ones
// packets of 64 (k_trav3), split until there are this many warps per SM.  Measured
// whole queries, 1.4k / 4.7k leaves: 1000 points 225 / 229 us wide, 285 / 446 us as split
// packets, 1425 / 3236 us as whole ones; 4000 points 303 / 340, 307 / 486, 978 / 2271;
// 8000 points 458 / 748, 305 / 761, 1038 / 2542.  Split to 28 or 56 warps per SM (the
// kernel holds 28): 64k points 1083 / 1361 or 1042 / 1178 us.  112 also splits full chunks
// in two, which shortens the last wave: k_trav3 5.94 -> 5.30 ms on 1.3M points, 2.21 ->
// 1.88 ms on a million on the rings.
constexpr size_t kPoints64 = 8192;  // points of an FP64 pass: room for 512 pairs each
constexpr size_t kWideMaxPoints = 4096;
constexpr int kPacketWarpsPerSM = 112;
// Blocks per SM of the pair kernels, which stride over their lists: about eight times what
// an SM holds, so that the last blocks are short.  16 and 8 left a second wave of
// blocks with half the SM empty: k_pair_fast 3.75 -> 3.43 ms, k_pair_eval 1.45 -> 1.20 ms
// on 1.3M points of a 4.7k-leaf model.
constexpr int kFastBlocks = 72, kEvalBlocks = 40;
// Mean boundary curves per leaf from which two pairs per lane (k_pair_fast2, shared table
// loads) pay: the loads it saves grow with the curves, what it loses -- runs of a leaf
// fill fewer of the lanes -- does not.  Measured on two kinds of model only: with 8 curves 3.43 ->
// 3.17 ms (1.3M points) and 1.20 -> 1.10 ms (at the surface), with 6 (rings) 2.69 -> 2.84 ms;
// the line lies between them.
constexpr size_t kPairedCurves = 7;
constexpr int kQueryStats = 20;              // entries of gwn_last_query_stats

// beta of the FP64 repair when the build leaves it automatic: the exact sum over
// every leaf for small models, else the traversal at (by default) 3 beta, whose
// order-2 remainder is 3^-4 = 1/81 of the bulk's (Eq. 3's remainder falls like
// beta^-4); the autotuner may lower the factor (repair_node_factor)
double auto_beta_repair(const gwn_model_s* m, double beta) {
    return m->host.n_leaves <= 512 ? 0.0 : m->repair_node_factor * beta;
}

gwn_status ensure_workspace(gwn_model_s* m, size_t n, size_t stage_bytes) {
    n = std::min(n, kChunk);
    if (n > m->ws_n || !m->ws_mem) {
        size_t want = std::max<size_t>(n, 4096);
        size_t bytes = workspace_layout(m->dim, m->host.n_leaves, want, nullptr, nullptr);
        if (m->ws_mem) cudaFree(m->ws_mem);
        m->ws_mem = nullptr;
        cudaError_t e = cudaMalloc(&m->ws_mem, bytes);
        if (e != cudaSuccess) { m->ws_n = 0; m->ws_bytes = 0; return fail(GWN_ERR_OOM, "query workspace allocation failed"); }
        m->ws_bytes = bytes;
        m->ws_n = want;
        workspace_layout(m->dim, m->host.n_leaves, want, reinterpret_cast<char*>(m->ws_mem), &m->ws);
    }
    if (stage_bytes > m->stage_cap) {
        if (m->stage) cudaFree(m->stage);
        m->stage = nullptr;
        cudaError_t e = cudaMalloc(&m->stage, stage_bytes);
        if (e != cudaSuccess) { m->stage_cap = 0; return fail(GWN_ERR_OOM, "staging allocation failed"); }
        m->stage_cap = stage_bytes;
    }
    return GWN_OK;
}

}  // namespace

// Morton-cell bits per axis of the 3D binning of a chunk of n points: about
// ppc points per cell, 3..6 bits
static int bin_bits3(size_t n, int ppc) {
    const double cells = std::max(1.0, (double)n / std::max(1, ppc));
    const int b = (int)std::lround(std::log2(cells) / 3.0);
    return std::min(6, std::max(3, b));
}

// The exact pairs of a chunk's first walk above which its leaves take the nodes' far factor
// beta instead of beta_leaf and the chunk is walked again.  Points in a crowd of small leaves
// have several times the pairs of other points, and there the leaves' far terms are most
// of the error.  Until the pair list grew, such a chunk did not fit it (96 entries a
// point and 65536, in up to three tries of what was left), and its points were evaluated in
// place with the leaves at beta; the line lies where that began, which the points in
// flight (150,000) make a matter of the chunk's size too: at 1.4 lists up to 150,000
// points, at 1.6 for 200,000, 1.9 for 300,000, 2.9 for 600,000, 3.3 for 2^20.  Measured, 14,000
// points next to a 560-patch model, beta 6, beta_leaf 3.25 (158 pairs a point, 1.57 lists):
// error 1.4e-5 at beta_leaf, 2.2e-6 at beta.
static unsigned long long dense_limit(const Workspace& ws, size_t n) {
    const double lists = std::min(3.3, std::max(1.4, 1.4 + ((double)n - 150000.0) / 300000.0));
    return (unsigned long long)(lists * (96.0 * (double)ws.list_points + 65536.0));
}

// the kernels' parameters of one query
static QueryParams query_params(const gwn_model_s* m, const gwn_query_opts& qo, const Workspace& ws) {
    QueryParams p;
    p.work = qo.count_work ? ws.work : nullptr;
    double beta = qo.beta > 0 ? qo.beta : m->opts.beta;
    p.beta2 = (float)(beta * beta);
    double beta_leaf = qo.beta_leaf > 0 ? qo.beta_leaf : (m->opts.beta_leaf > 0 ? m->opts.beta_leaf : beta);
    p.beta2_leaf = (float)(beta_leaf * beta_leaf);
    double br = m->opts.beta_repair;
    const bool automatic = br < 0;
    if (automatic) br = auto_beta_repair(m, beta);
    p.beta2_repair = br > 0 ? br * br : 0.0;
    // the repair's leaves: the automatic factor times beta_leaf, or, with a given
    // beta_repair, the bulk's ratio beta_leaf / beta
    const double brl = br > 0 ? (automatic ? m->repair_leaf_factor * beta_leaf : br * beta_leaf / beta) : 0.0;
    p.beta2_repair_leaf = brl > 0 ? brl * brl : 0.0;
    p.band = (float)(qo.repair_band > 0 ? qo.repair_band : m->opts.repair_band);
    // packet local expansion (3D, order-2 evaluation): the query's ratio, else the model's; < 0 off
    const double kap = qo.local_ratio != 0.0 ? qo.local_ratio : m->local_ratio;
    p.kappa2 = m->dim == 3 && !m->tree.order3 && kap > 0 ? (float)(kap * kap) : 0.f;
    p.mode = qo.mode;
    p.precision = qo.precision >= 0 ? qo.precision : m->opts.precision;
    return p;
}

static int device_sms() {
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

// FP64 values of the points in list R (R.rw, R.rst): the warp traversal with far
// factors beta2 (nodes) and beta2l (leaves), 0: none, then its exact leaves as pairs
// over the whole GPU.  all: every leaf of each of the `all` listed points.
static void enqueue_pass64(gwn_model_s* m, double beta2, double beta2l, Rule64 rule, const void* pts, int dtype,
                           const RepairList& R, cudaStream_t st, int sms, int all = 0) {
    const int B = 128;
    const unsigned wb = (unsigned)(sms * 4);  // blocks of kRepairWarps warps, one warp per point
    if (all)
        k_rpairs_all<<<(unsigned)(sms * 8), B, 0, st>>>(R, all, m->host.n_leaves);
    else
        k_rtrav_warp<false><<<wb, 32 * kRepairWarps, 0, st>>>(m->tree, pts, dtype, beta2, R, beta2l, rule, false);
    k_rpairs3_fast<<<(unsigned)(sms * 8), B, 0, st>>>(m->tree, pts, dtype, R, rule);
    k_rpairs3_warp<<<(unsigned)(sms * 8), B, 0, st>>>(m->tree, pts, dtype, R, rule);
    if (!all && (long long)R.cap * m->host.n_leaves > kRepairPairCap)
        k_rtrav_warp<true><<<wb, 32 * kRepairWarps, 0, st>>>(m->tree, pts, dtype, beta2, R, beta2l, rule, true);
}

// FP64 re-evaluation (GWN_PREC_FP32_REPAIR) of the points in list R, whose
// indices address pts and the outputs.  3D always goes through the warp
// traversal and the FP64 pair list: with beta_repair = 0 or in direct mode
// (exact sum over every leaf) every leaf becomes a pair, and the pairs of all
// repaired points spread over the whole GPU instead of one warp walking all
// leaves per point.
static gwn_status enqueue_repair(gwn_model_s* m, const QueryParams& p, const void* pts, int dtype, const RepairList& R,
                                 double* out_w, int* out_label, uint32_t* out_status, cudaStream_t st, int sms) {
    const int B = 128;
    const unsigned rb = (unsigned)(sms * 8);
    if (m->dim == 2 && (p.mode == GWN_MODE_DIRECT || !(p.beta2_repair > 0))) {
        k_repair2<<<rb, B, 0, st>>>(m->tree, pts, dtype, p, out_w, out_label, out_status, R.idx, R.count, R.cap);
    } else if (m->dim == 2) {
        k_rtrav2<<<(unsigned)(sms * 4), 256, 0, st>>>(m->tree, pts, dtype, p.beta2_repair, R, out_w, out_label, out_status);
    } else {
        const bool direct = p.mode == GWN_MODE_DIRECT;
        enqueue_pass64(m, direct ? 0.0 : p.beta2_repair, direct ? 0.0 : p.beta2_repair_leaf,
                       Rule64{kRatio64Repair, true}, pts, dtype, R, st, sms);
        k_rfinish<<<(unsigned)(sms * 2), B, 0, st>>>(R, out_w, out_label, out_status, true, GWN_QS_REPAIRED);
    }
    GWN_CUDA_TRY(cudaGetLastError());
    return GWN_OK;
}

// Enqueue the query kernels of one chunk (points off .. off + n - 1 of the
// query; pts and the outputs point at the chunk) on `st`, using workspace
// `ws` (sized for at least n points).  Shared with the batched and serving
// entry points through gwn_enqueue_device.
static gwn_status enqueue_chunk(gwn_model_s* m, const void* pts, int dtype, size_t n, size_t off, double* out_w,
                                int* out_label, uint32_t* out_status, const gwn_query_opts& qo, cudaStream_t st,
                                const Workspace& ws,
                                bool local_list, bool accum, bool whole) {
    const QueryParams p = query_params(m, qo, ws);
    const int pc = m->prof_chunks;
    const bool prof = qo.profile != 0 && pc < gwn_model_s::kMaxProfChunks;
    cudaEvent_t* ev = prof ? m->ev[pc] : nullptr;
    if (prof) {
        if (!ev[0])
            for (int k = 0; k < 5; ++k) GWN_CUDA_TRY(cudaEventCreate(&ev[k]));
        m->prof_chunks = pc + 1;
    }
    const int B = 128;
    const int ni = (int)n;
    const unsigned nb = (unsigned)((n + B - 1) / B);
    const int sms = device_sms();
    if (p.precision == GWN_PREC_FP64 && m->dim == 3) {
        // the warp traversal and the FP64 pair list, for as many points at a time as
        // leave room for their pairs (a point whose pairs do not fit its share is still
        // evaluated, by its own warp), the pairs' values summed in a fixed order.  One thread per
        // point, each with its own branches and leaves, took 150 times as long (4001
        // points, 2.3k leaves: 1.48 s).
        const bool direct = p.mode == GWN_MODE_DIRECT;
        const bool all = direct && m->host.n_leaves <= kRepairPairCap;
        const size_t step = all ? std::max<size_t>(1, std::min(n, (size_t)(kRepairPairCap / m->host.n_leaves)))
                                : std::min(n, kPoints64);
        const double b2 = direct ? 0.0 : (double)p.beta2;
        const size_t esz = (dtype == GWN_F32 ? sizeof(float) : sizeof(double)) * 3;
        for (size_t at = 0; at < n; at += step) {
            const int c = (int)std::min(step, n - at);
            const RepairList R{ws.rlist, ws.counters + 1, c, ws.rw, ws.rst, ws.rpairs, ws.counters + 4, ws.rpairs2,
                               ws.counters + 10, ws.rval, ws.rcnt,
                               all ? m->host.n_leaves : (int)(kRepairPairCap / c)};
            GWN_CUDA_TRY(cudaMemsetAsync(ws.counters, 0, kCounterCount * sizeof(int), st));
            k_iota<<<(unsigned)((c + B - 1) / B), B, 0, st>>>(c, ws.rlist, ws.counters + 1);
            enqueue_pass64(m, b2, b2, Rule64{kRatio64Exact, false}, reinterpret_cast<const char*>(pts) + at * esz, dtype,
                           R, st, sms, all ? c : 0);
            k_rsum<<<(unsigned)(((size_t)c * 32 + B - 1) / B), B, 0, st>>>(R, c);
            k_rfinish<<<(unsigned)((c + B - 1) / B), B, 0, st>>>(R, out_w + at, out_label ? out_label + at : nullptr,
                                                              out_status ? out_status + at : nullptr, false,
                                                              direct ? (uint32_t)GWN_QS_REPAIRED : 0u);
        }
        GWN_CUDA_TRY(cudaGetLastError());
        return GWN_OK;
    }
    if (p.precision == GWN_PREC_FP64) {
        if (p.mode == GWN_MODE_DIRECT) {
            // exact FP64 direct sum, one warp per point (lanes stride over the leaves)
            k_iota<<<nb, B, 0, st>>>(ni, ws.rlist, ws.counters + 1);
            unsigned rb = (unsigned)std::min<long long>(((long long)n * 32 + B - 1) / B, (long long)sms * 16);
            QueryParams pd = p;
            pd.beta2_repair = 0.0;
            k_repair2<<<rb, B, 0, st>>>(m->tree, pts, dtype, pd, out_w, out_label, out_status, ws.rlist, ws.counters + 1);
        } else {
            k_query64<<<(unsigned)((n + 63) / 64), 64, 0, st>>>(m->tree, pts, dtype, (long long)n, p, out_w, out_label,
                                                               out_status);
        }
        GWN_CUDA_TRY(cudaGetLastError());
        return GWN_OK;
    }
    int* rcount = ws.counters + 1;
    const bool direct3 = p.mode == GWN_MODE_DIRECT && m->dim == 3;
    if (p.mode == GWN_MODE_DIRECT && m->dim == 2) {
        k_query32<<<nb, B, 0, st>>>(m->tree, pts, dtype, (long long)n, p, out_w, out_label, out_status, ws.rlist, rcount);
        GWN_CUDA_TRY(cudaGetLastError());
    } else {
        // 1. spatial binning of the points (counting sort by Morton cell)
        const bool o3 = m->tree.order3 != 0;
        const bool local = !o3 && p.kappa2 > 0.f;  // packets take far nodes by local expansion
        const bool few = whole && m->dim == 3 && n <= (size_t)kFewPoints;  // few3d.cuh
        const bool wide = m->dim == 3 && !direct3 && !local && n <= kWideMaxPoints;  // one warp per point: their order does not matter
        const int* key = nullptr;
        if (n >= 2048 && !wide) {
            const int bits = m->dim == 2 ? kBinBits2 : bin_bits3(n, m->bin_ppc);
            const int cells = 1 << (m->dim * bits);
            GWN_CUDA_TRY(cudaMemsetAsync(ws.hist, 0, (size_t)cells * sizeof(int), st));
            const unsigned bb = (unsigned)std::min<long long>(nb, (long long)sms * 4);
            if (m->dim == 2) {
                k_bbox<2><<<bb, B, 0, st>>>(pts, dtype, ni, ws.bbox);
                k_bin<2><<<nb, B, 0, st>>>(pts, dtype, ni, ws.bbox, bits, ws.key, ws.hist);
            } else {
                k_bbox<3><<<bb, B, 0, st>>>(pts, dtype, ni, ws.bbox);
                k_bin<3><<<nb, B, 0, st>>>(pts, dtype, ni, ws.bbox, bits, ws.key, ws.hist);
            }
            int* sums = ws.hist + kMaxBinCells;
            const unsigned tiles = (unsigned)((cells + kScanTile - 1) / kScanTile);
            if (tiles > 1) k_scan_sums<<<tiles, 1024, 0, st>>>(ws.hist, cells, sums);
            k_scan<<<tiles, 1024, 0, st>>>(ws.hist, cells, sums);
            key = ws.key;
        }
        if (m->dim == 2) k_scatter_points<2><<<nb, B, 0, st>>>(pts, dtype, ni, key, ws.hist, ws.spos, ws.wacc, ws.st, ws.near);
        else k_scatter_points<3><<<nb, B, 0, st>>>(pts, dtype, ni, key, ws.hist, ws.spos, ws.wacc, ws.st, nullptr);
        GWN_CUDA_TRY(cudaGetLastError());
        if (direct3) {
            // every leaf for every point, the leaves in slices until the blocks fill the GPU
            const unsigned slices = (unsigned)std::max<long long>(
                1, std::min<long long>(std::min<long long>(m->host.n_leaves, 65535), ((long long)sms * 16 + nb - 1) / nb));
            float* few_val = reinterpret_cast<float*>(ws.rpairs);  // the repair's pairs come later
            // every point to repair goes to the chunk's own list (repaired by the direct sum below)
            auto finish = [&](auto* acc, const long long* near) {
                k_finish<<<nb, B, 0, st>>>(ni, ws.spos, acc, ws.st, p.precision, p.band, out_w, out_label, out_status, ws.rlist,
                                           rcount, (int)off, ws.rlist_g, ws.gcount, 0, 0, near);
            };
            if (few && (long long)n * m->host.n_leaves <= 2 * kRepairPairCap) {
                k_few_direct<<<(unsigned)(sms * 8), B, 0, st>>>(m->tree, ws.spos, ni, few_val, ws.st);
                k_few_direct_sum<<<1, 32 * kFewPoints, 0, st>>>(ni, m->host.n_leaves, few_val, ws.rw);
                finish(ws.rw, nullptr);
            } else {
                // the near band: a point on the surface has two or three pairs there, so the list takes the
                // place of the traversal's, which holds every pair that pairs2 does
                const int near_cap = (int)std::min<long long>(ws.pair_cap, 0x7fffffff);
                long long* acc = reinterpret_cast<long long*>(ws.rw);
                GWN_CUDA_TRY(cudaMemsetAsync(acc, 0, n * sizeof(long long), st));
                k_direct3<<<dim3(nb, slices), B, 0, st>>>(m->tree, ws.spos, ni, acc, ws.wacc, ws.st, ws.counters, ws.pairs2,
                                                          ws.slow_cap, ws.olist);
                k_pair_eval<long long><<<(unsigned)(sms * kEvalBlocks), B, 0, st>>>(
                    m->tree, ws.spos, ws.slow_cap, ws.counters + 8, ws.counters, ws.pairs2, acc, ws.st, ws.pairs, near_cap,
                    nullptr, nullptr);
                k_pair_eval64_warp<<<(unsigned)(sms * 2), B, 0, st>>>(m->tree, ws.spos, near_cap, ws.counters, ws.pairs,
                                                                      ws.wacc, ws.st, acc);
                if ((long long)n * m->host.n_leaves > ws.slow_cap)
                    k_direct_overflow3<<<(unsigned)(sms * 4), B, 0, st>>>(m->tree, ws.spos, acc, ws.wacc, ws.st, ws.counters,
                                                                          ws.olist);
                finish(ws.wacc, acc);
            }
            GWN_CUDA_TRY(cudaGetLastError());
        } else if (few) {
            // one packet's walk, its pairs sorted by leaf into the near pairs' place; these take the list's
            const long long few_cap = ws.slow_cap;
            Workspace fw = ws;
            fw.pair_cap = few_cap;
            if (prof) GWN_CUDA_TRY(cudaEventRecord(ev[0], st));
            if (local) {
                auto trav = m->stack_depth <= 64 ? k_trav3_local<64>
                                                 : m->stack_depth <= 96 ? k_trav3_local<96> : k_trav3_local<128>;
                trav<<<1, B, 0, st>>>(m->tree, ws.spos, ni, p.beta2, p.beta2_leaf, fw, p.work, ws.olist, p.kappa2);
            } else {
                (o3 ? k_few_walk<true> : k_few_walk<false>)<<<1, 32, 0, st>>>(m->tree, ws.spos, ni, p.beta2, p.beta2_leaf,
                                                                            fw, p.work, ws.olist);
            }
            if (prof) GWN_CUDA_TRY(cudaEventRecord(ev[1], st));
            k_few_sort<<<1, 1024, 0, st>>>(m->host.n_leaves, few_cap, ws.counters, ws.pairs, ws.hist, ws.pairs2);
            if (prof) GWN_CUDA_TRY(cudaEventRecord(ev[2], st));
            k_few_fast<<<(unsigned)(sms * 16), B, 0, st>>>(m->tree, ws.spos, few_cap, ws.counters, ws.pairs2, ws.wacc,
                                                           ws.st, ws.pairs, p.work);
            if (prof) GWN_CUDA_TRY(cudaEventRecord(ev[4], st));
            // with repair a point past one near-band pair a point is evaluated whole in FP64, as always
            const int near_cap = p.precision == GWN_PREC_FP32 ? ws.near_cap : ni;
            k_few_eval<<<(unsigned)(sms * 8), B, 0, st>>>(m->tree, ws.spos, ws.counters, ws.pairs, ws.wacc, ws.st,
                                                          ws.pairs64, near_cap, p.work);
            if (prof) GWN_CUDA_TRY(cudaEventRecord(ev[3], st));
            k_pair_eval64_warp<<<(unsigned)(sms * 2), B, 0, st>>>(m->tree, ws.spos, near_cap, ws.counters, ws.pairs64,
                                                                         ws.wacc, ws.st);
            if ((long long)n * m->host.n_leaves > few_cap)
                k_overflow3<<<1, B, 0, st>>>(m->tree, ws.spos, p.beta2, ws, ws.olist);
            k_finish<float><<<nb, B, 0, st>>>(ni, ws.spos, ws.wacc, ws.st, p.precision, p.band, out_w, out_label, out_status,
                                              ws.rlist, rcount, (int)off, ws.rlist_g, ws.gcount, ws.rcap);
            GWN_CUDA_TRY(cudaGetLastError());
        } else {
        // 2. traversal
        if (prof) GWN_CUDA_TRY(cudaEventRecord(ev[0], st));
        // packets split over subtrees until they fill the GPU
        const unsigned packets = (unsigned)((n + 63) / 64);
        int level = 0;
        while (level + 1 < kCutLevels && ((size_t)packets << level) < (size_t)kPacketWarpsPerSM * sms &&
               (n << (level + 1)) <= kParts2)
            ++level;
        if (m->dim == 2) {
            (p.work ? k_trav2<true> : k_trav2<false>)
                <<<dim3((packets + 3) / 4, (unsigned)m->cut_size[level]), B, 4 * 12 * m->stack_depth, st>>>(
                    m->tree, ws.spos, ni, p.beta2, m->stack_depth, m->cuts[level], ws, p.work);
            k_near2<<<(unsigned)(sms * 8), B, 0, st>>>(m->tree, ws.spos, ws.counters, ws.pairs2, ws.slow_cap, ws.part, ws.near,
                                                       ws.st);
            if ((long long)n * m->host.n_leaves > ws.slow_cap)
                k_overflow2<<<(unsigned)(sms * 4), B, 0, st>>>(m->tree, ws.spos, ni, m->cut_size[level], p.beta2, ws);
            if (prof)
                for (int k : {1, 2, 4, 3}) GWN_CUDA_TRY(cudaEventRecord(ev[k], st));
        } else {
            const unsigned long long limit = dense_limit(ws, n);
            const bool may_dense = m->tree.leaf_far && p.beta2_leaf < p.beta2 &&
                                   (unsigned long long)n * (unsigned long long)m->host.n_leaves > limit;
            const Dense none{nullptr, 0}, dense{may_dense ? ws.found : nullptr, limit};
            auto wide_pass = [&](bool list, unsigned blocks, const int* idx, const int* n_dev, Dense d, bool again) {
                auto k = p.work ? (list ? (o3 ? k_wide3<true, true, true> : k_wide3<false, true, true>)
                                        : (o3 ? k_wide3<true, true, false> : k_wide3<false, true, false>))
                                : (list ? (o3 ? k_wide3<true, false, true> : k_wide3<false, false, true>)
                                        : (o3 ? k_wide3<true, false, false> : k_wide3<false, false, false>));
                k<<<blocks, B, 0, st>>>(m->tree, ws.spos, ni, idx, n_dev, p.beta2, p.beta2_leaf, ws, ws.pairs2,
                                        ws.slow_cap, list ? ws.olist : ws.olist2, p.work, d, again);
            };
            // (the second walk of a dense chunk split to about one wave of warps: its blocks are
            // launched for every chunk that could be dense)
            int level_again = 0;
            while (level_again < level && ((size_t)packets << (level_again + 1)) <= (size_t)28 * sms) ++level_again;
            auto packet_pass = [&](Dense d, bool again) {
                const int lv = again ? level_again : level;
                auto trav = p.work ? (o3 ? k_trav3<true, true> : k_trav3<false, true>)
                                   : (o3 ? k_trav3<true, false> : k_trav3<false, false>);
                trav<<<dim3(packets, (unsigned)m->cut_size[lv]), 32, trav3_smem(m->stack_depth), st>>>(
                    m->tree, ws.spos, ni, p.beta2, again ? p.beta2 : p.beta2_leaf, m->stack_depth, m->cuts[lv], ws, p.work,
                    ws.olist, d, again);
            };
            auto eval_pass = [&](int* olist) {
                k_pair_eval<float><<<(unsigned)(sms * kEvalBlocks), B, 0, st>>>(m->tree, ws.spos, ws.slow_cap, ws.counters + 8,
                                                               ws.counters, ws.pairs2, ws.wacc, ws.st, ws.pairs64,
                                                               ws.near_cap, olist, p.work);
            };
            const unsigned wide_blocks =
                (unsigned)std::min(std::max((n + 3) / 4, std::min(n, (size_t)sms)), (size_t)sms * 16);
            if (wide) {
                wide_pass(true, wide_blocks, nullptr, nullptr, none, false);
            } else if (local) {
                auto trav = m->stack_depth <= 64 ? k_trav3_local<64>
                                                 : m->stack_depth <= 96 ? k_trav3_local<96> : k_trav3_local<128>;
                trav<<<nb, B, 0, st>>>(m->tree, ws.spos, ni, p.beta2, p.beta2_leaf, ws, p.work, ws.olist, p.kappa2);
            } else {
                packet_pass(none, false);
            }
            if (may_dense) {
                k_dense_reset<<<std::min(nb, (unsigned)sms * 4), B, 0, st>>>(ws, ni, dense);
                if (wide) wide_pass(true, wide_blocks, nullptr, nullptr, dense, true);
                else packet_pass(dense, true);
            }
            if (prof)
                for (int k : {1, 2}) GWN_CUDA_TRY(cudaEventRecord(ev[k], st));
            GWN_CUDA_TRY(cudaGetLastError());
            // 3. exact leaves: far pairs from the node tables, the rest to the full evaluator
            if (wide || local || m->host.c3.size() < kPairedCurves * (size_t)m->host.n_leaves)
                k_pair_fast<<<(unsigned)(sms * kFastBlocks), B, 0, st>>>(m->tree, ws.spos, ws.pair_cap, ws.counters, ws.pairs,
                                                                         ws.wacc, ws.st, ws.pairs2, ws.slow_cap, ws.olist,
                                                                         p.work);
            else
                k_pair_fast2<<<(unsigned)(sms * kFastBlocks), B, 0, st>>>(
                    m->tree, ws.spos, ws.pair_cap, ws.counters, reinterpret_cast<const int4*>(ws.pairs), ws.wacc, ws.st,
                    ws.pairs2, ws.slow_cap, ws.olist, p.work);
            if (prof) GWN_CUDA_TRY(cudaEventRecord(ev[4], st));
            eval_pass(ws.olist);
            if (prof) GWN_CUDA_TRY(cudaEventRecord(ev[3], st));
            const bool may_overflow = (long long)n * m->host.n_leaves > ws.slow_cap;
            if (may_overflow) {
                // the points whose pairs did not fit the list, one warp each, without a list
                k_next_round<<<1, 32, 0, st>>>(ws);
                wide_pass(false, (unsigned)(sms * 8), ws.olist, ws.counters + 5, dense, false);
                eval_pass(ws.olist2);
            }
            GWN_CUDA_TRY(cudaGetLastError());
            // the near band of both passes in one launch: a point of the second pass has entered it
            // only where the near band's list was full, and then it overflows in the second
            // pass too, so every listed point's FP32 sum is final here or k_overflow3's
            k_pair_eval64_warp<<<(unsigned)(sms * 2), B, 0, st>>>(m->tree, ws.spos, ws.near_cap, ws.counters, ws.pairs64,
                                                                  ws.wacc, ws.st);
            if (may_overflow || (long long)n * m->host.n_leaves > ws.near_cap)
                k_overflow3<<<(unsigned)(sms * 2), B, 0, st>>>(m->tree, ws.spos, p.beta2, ws,
                                                               may_overflow ? ws.olist2 : ws.olist);
        }
        GWN_CUDA_TRY(cudaGetLastError());
        // 4. outputs and the repair list
        const bool two = m->dim == 2;
        k_finish<float><<<nb, B, 0, st>>>(ni, ws.spos, two ? ws.part : ws.wacc, ws.st, p.precision, p.band, out_w, out_label,
                                          out_status, ws.rlist, rcount, (int)off, ws.rlist_g, ws.gcount, ws.rcap,
                                          two ? m->cut_size[level] : 0, two ? ws.near : nullptr);
        GWN_CUDA_TRY(cudaGetLastError());
        }
    }
    if (p.precision == GWN_PREC_FP32_REPAIR && (local_list || p.mode == GWN_MODE_DIRECT)) {
        // points of this chunk that did not fit the query's repair list (none in a
        // query of at most rcap points), repaired right away; direct mode, which lists
        // every point locally, too
        const RepairList R{ws.rlist, rcount, ws.rcap, ws.rw, ws.rst, ws.rpairs, ws.counters + 4, ws.rpairs2,
                           ws.counters + 10};
        gwn_status s = enqueue_repair(m, p, pts, dtype, R, out_w, out_label, out_status, st, sms);
        if (s != GWN_OK) return s;
    }
    if (accum) k_accum<<<1, 32, 0, st>>>(ws, false);
    GWN_CUDA_TRY(cudaGetLastError());
    return GWN_OK;
}

// Enqueue a query on `st` for device-resident points and outputs, in chunks of
// at most kChunk points (the workspace holds one chunk), or of max_chunk when
// smaller: the serving loop takes shorter kernels so that requests on other
// slots interleave.
gwn_status gwn_enqueue_device(gwn_model_s* m, const void* pts, int dtype, size_t n, double* out_w, int* out_label,
                              uint32_t* out_status, const gwn_query_opts& qo, cudaStream_t st, const Workspace& ws,
                              size_t max_chunk) {
    const size_t chunk = max_chunk > 0 ? std::min(max_chunk, kChunk) : kChunk;
    const size_t esz = (dtype == GWN_F32 ? sizeof(float) : sizeof(double)) * m->dim;
    if (qo.count_work) GWN_CUDA_TRY(cudaMemsetAsync(ws.work, 0, kWorkCount * sizeof(unsigned long long), st));
    m->prof_chunks = 0;
    m->profiled = qo.profile != 0;
    // the query's repair list holds as many points as a workspace: with no more than
    // that no point can be left to a chunk's own list
    const bool local = n > (size_t)ws.rcap;
    const QueryParams p = query_params(m, qo, ws);
    const bool repair = p.precision == GWN_PREC_FP32_REPAIR && p.mode == GWN_MODE_BVH;
    for (size_t off = 0; off < n; off += chunk) {
        size_t c = std::min(chunk, n - off);
        if (off == 0) GWN_CUDA_TRY(cudaMemsetAsync(ws.acc, 0, 4 * kControlBytes, st));
        else GWN_CUDA_TRY(cudaMemsetAsync(ws.counters, 0, 2 * kControlBytes, st));
        gwn_status s = enqueue_chunk(m, reinterpret_cast<const char*>(pts) + off * esz, dtype, c, off, out_w + off,
                                     out_label ? out_label + off : nullptr, out_status ? out_status + off : nullptr,
                                     qo, st, ws, local, !(repair && off + c == n), c == n);
        if (s != GWN_OK) return s;
    }
    // one FP64 repair pass over the points that every chunk listed (indices into
    // the whole query), so that the repair fills the GPU instead of running a
    // few warps after each chunk
    if (repair) {
        const RepairList R{ws.rlist_g, ws.gcount, ws.rcap, ws.rw, ws.rst, ws.rpairs, ws.gcount + 1, ws.rpairs2,
                           ws.gcount + 2};
        gwn_status s = enqueue_repair(m, p, pts, dtype, R, out_w, out_label, out_status, st, device_sms());
        if (s != GWN_OK) return s;
        k_accum<<<1, 32, 0, st>>>(ws, true);
        GWN_CUDA_TRY(cudaGetLastError());
    }
    return GWN_OK;
}

extern "C" {

void gwn_default_build_opts(gwn_build_opts* o) {
    if (!o) return;
    o->tolerance = 1e-4;
    o->max_aabb_frac = 0.1;
    o->order = 2;
    o->beta = 2.0;
    o->beta_repair = -1.0;
    o->repair_band = 1e-3;
    o->quad_nodes = 10;
    o->precision = GWN_PREC_FP32_REPAIR;
    o->device = -1;
    o->n_threads = 0;
    o->leaf_far = -1;
    o->beta_leaf = 0.0;
    o->adaptive_beta = 0;
    o->device_build = -1;
    o->tree_builder = -1;
    o->local_ratio = 0.0;
}

void gwn_default_query_opts(gwn_query_opts* q) {
    if (!q) return;
    q->mode = GWN_MODE_BVH;
    q->precision = -1;
    q->beta = 0.0;
    q->count_work = 0;
    q->profile = 0;
    q->beta_leaf = 0.0;
    q->repair_band = 0.0;
    q->local_ratio = 0.0;
}

// ---------------------------------------------------------------- autotuner
//
// Picks the far-field factors (beta for internal nodes, beta_leaf for 3D
// leaves) of a model, and for a 3D model built with order 3 the Taylor order
// the queries evaluate (3, or 2 from the same coefficients): validation points
// -- uniform in the model's box, plus points a little off the surface at
// random leaf centroids -- are evaluated exactly (FP64 direct sum on the
// device), then with the FP32 path for every candidate.  The candidates whose
// max |dGWN| stays below half the tolerance are ranked by counted work (flops
// per point) and the cheapest few of each order are timed (below).

__global__ void k_err(int n, const double* a, const double* b, double* out) {
    __shared__ double smax[128];
    double m = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) m = fmax(m, fabs(a[i] - b[i]));
    smax[threadIdx.x] = m;
    __syncthreads();
    for (int o = 64; o > 0; o >>= 1) {
        if (threadIdx.x < o) smax[threadIdx.x] = fmax(smax[threadIdx.x], smax[threadIdx.x + o]);
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicMax(reinterpret_cast<unsigned long long*>(out), __double_as_longlong(smax[0]));
}

// max |a - b| over the points whose status carries GWN_QS_REPAIRED, and their count
__global__ void k_err_repaired(int n, const double* a, const double* b, const uint32_t* st, double* out, int* cnt) {
    __shared__ double smax[128];
    double m = 0;
    int c = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        if (st[i] & GWN_QS_REPAIRED) {
            m = fmax(m, fabs(a[i] - b[i]));
            ++c;
        }
    smax[threadIdx.x] = m;
    atomicAdd(cnt, c);
    __syncthreads();
    for (int o = 64; o > 0; o >>= 1) {
        if (threadIdx.x < o) smax[threadIdx.x] = fmax(smax[threadIdx.x], smax[threadIdx.x + o]);
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicMax(reinterpret_cast<unsigned long long*>(out), __double_as_longlong(smax[0]));
}

static gwn_status autotune(gwn_model_s* m) {
    const int d = m->dim;
    const HostModel& H = m->host;
    const int nu = 768, nn = 256, nv = nu + nn;
    std::vector<float> pts((size_t)nv * d);
    uint64_t seed = 0x9e3779b97f4a7c15ull ^ (uint64_t)H.n_leaves;
    auto rnd = [&]() {  // splitmix64
        seed += 0x9e3779b97f4a7c15ull;
        uint64_t z = seed;
        z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
        z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
        z ^= z >> 31;
        return (double)(z >> 11) * (1.0 / 9007199254740992.0);
    };
    for (int i = 0; i < nu; ++i)
        for (int k = 0; k < d; ++k) pts[(size_t)i * d + k] = (float)(H.lo[k] + rnd() * (H.hi[k] - H.lo[k]));
    double diag = 0;
    for (int k = 0; k < d; ++k) diag += (H.hi[k] - H.lo[k]) * (H.hi[k] - H.lo[k]);
    diag = std::sqrt(diag);
    for (int i = nu; i < nv; ++i) {
        int li = (int)(rnd() * H.n_leaves) % std::max(1, H.n_leaves);
        for (int k = 0; k < d; ++k) {
            double c = d == 3 ? (double)H.lhdr64[(size_t)li * 4 + k] : H.lhdr64[(size_t)li * 4 + k];
            pts[(size_t)i * d + k] = (float)(c + (rnd() - 0.5) * 0.02 * diag);
        }
    }
    float* dp = nullptr;
    double *ref = nullptr, *w = nullptr, *err = nullptr;
    GWN_CUDA_TRY(cudaMalloc(&dp, pts.size() * sizeof(float)));
    GWN_CUDA_TRY(cudaMalloc(&ref, nv * sizeof(double)));
    GWN_CUDA_TRY(cudaMalloc(&w, nv * sizeof(double)));
    GWN_CUDA_TRY(cudaMalloc(&err, sizeof(double)));
    GWN_CUDA_TRY(cudaMemcpy(dp, pts.data(), pts.size() * sizeof(float), cudaMemcpyHostToDevice));
    gwn_status s = ensure_workspace(m, nv, 0);
    gwn_query_opts qo;
    gwn_default_query_opts(&qo);
    qo.mode = GWN_MODE_DIRECT;
    qo.precision = GWN_PREC_FP64;
    if (s == GWN_OK) s = gwn_enqueue_device(m, dp, GWN_F32, nv, ref, nullptr, nullptr, qo, 0, m->ws);
    const double betas[] = {3.0, 3.5, 4.0, 4.5, 5.0, 5.5, 6.0, 7.0, 8.0, 10.0, 12.0, 16.0};
    // 2D leaves have no separate factor (0 = beta); 3D leaves: per-level factors
    const double leafb[] = {0.0, 2.0, 2.5, 2.75, 3.0, 3.25, 3.5, 4.0, 5.0};
    double best_cost = 1e300, best_b = 0, best_bl = 0;
    int best_o = m->eval_order;
    std::vector<std::tuple<double, double, double, int>> ok_cands;  // (counted flops, beta, beta_leaf, order)
    double fb_err = 1e300, fb_b = 0, fb_bl = 0;  // fallback: smallest error seen
    int fb_o = m->eval_order;
    const double tol = 0.5 * m->opts.tolerance;
    std::vector<int> orders{m->eval_order};
    if (d == 3 && m->opts.order >= 3) orders = {3, 2};
    for (int ord : orders)
    for (double b : betas) {
        m->tree.order3 = ord >= 3 ? 1 : 0;
        bool any_ok = false;
        for (double bl : leafb) {
            if (s != GWN_OK) break;
            if (d == 2 && bl != 0.0) continue;
            if (d == 3 && bl == 0.0) continue;
            if (bl > b) continue;
            double blv = bl == 0.0 ? b : bl;
            gwn_query_opts q2;
            gwn_default_query_opts(&q2);
            q2.precision = GWN_PREC_FP32;
            q2.beta = b;
            q2.beta_leaf = blv;
            q2.count_work = 1;
            s = gwn_enqueue_device(m, dp, GWN_F32, nv, w, nullptr, nullptr, q2, 0, m->ws);
            if (s != GWN_OK) break;
            cudaMemset(err, 0, sizeof(double));
            k_err<<<4, 128>>>(nv, ref, w, err);
            double e = 0;
            unsigned long long wk[kWorkCount] = {}, acc[kCounterCount] = {};
            if (cudaMemcpy(&e, err, sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess ||
                cudaMemcpy(wk, m->ws.work, sizeof(wk), cudaMemcpyDeviceToHost) != cudaSuccess ||
                cudaMemcpy(acc, m->ws.acc, sizeof(acc), cudaMemcpyDeviceToHost) != cudaSuccess) {
                s = fail(GWN_ERR_CUDA, "autotune readback failed");
                break;
            }
            // a candidate whose exact-leaf pairs overflow the work list is rejected (its
            // overflow path is slow and not counted), and so is one with so many that its
            // leaves took beta
            if (acc[3] + acc[6] > 0 || (d == 3 && acc[0] > dense_limit(m->ws, nv))) continue;
            if (e < fb_err) {
                fb_err = e;
                fb_b = b;
                fb_bl = blv;
                fb_o = ord;
            }
            double cost = 10.0 * (wk[kWorkNodes] + wk[kWorkLeafTests]) + (ord >= 3 ? 120.0 : 72.0) * wk[kWorkFar] +
                          28.0 * wk[kWorkGlDeg] + 70.0 * wk[kWorkGlNodes] + 2000.0 * wk[kWorkHits] +
                          kFastNodeFlops * wk[kWorkFastNodes] +
                          (d == 2 ? 60.0 * wk[kWorkLeaves] : 30.0 * wk[kWorkLeaves]);
            if (std::getenv("GWN_AUTOTUNE_VERBOSE"))
                std::fprintf(stderr,
                             "[gwn autotune] leaves=%d order=%d beta=%.1f beta_leaf=%.1f max|dGWN|=%.3g flops/pt=%.3g\n",
                             H.n_leaves, ord, b, blv, e, cost / nv);
            if (e <= tol) {
                any_ok = true;
                ok_cands.push_back({cost, b, blv, ord});
                if (cost < best_cost) {
                    best_cost = cost;
                    best_b = b;
                    best_bl = blv;
                    best_o = ord;
                }
            }
        }
        if (any_ok && b >= 8.0) break;  // larger beta only costs more
    }
    struct Free {
        std::vector<void*> p;
        ~Free() {
            for (void* q : p) cudaFree(q);
        }
    } frees{{ref, w, err, dp}};
    if (s != GWN_OK) return s;
    if (best_b == 0) {  // nothing met the tolerance: the most accurate candidate tried
        best_b = fb_b > 0 ? fb_b : 8.0;
        best_bl = fb_b > 0 ? fb_bl : 8.0;
        best_o = fb_o;
    }
    m->opts.beta = best_b;
    m->opts.beta_leaf = d == 3 ? best_bl : 0.0;
    m->eval_order = best_o;
    m->tree.order3 = d == 3 && best_o >= 3 ? 1 : 0;
    // Counted flops do not weigh the kernels alike (the traversal's far tests and
    // Taylor terms issue about twice the instructions per counted flop of the
    // node-table leaves), so among the accurate candidates the cheapest four by
    // count of each order are timed on one chunk of points uniform in the model's
    // box (binned and paired as a large query is: smaller samples bin and pair
    // differently and flipped the choice between close candidates from run to
    // run), and
    // the fastest is kept; then the binning's target points per cell is timed
    // the same way (the sample is binned at the resolution its size gives, as a
    // query is).
    if (ok_cands.size() > 1 || d == 3) {
        std::sort(ok_cands.begin(), ok_cands.end());
        {
            std::vector<std::tuple<double, double, double, int>> keep;
            int per_order[4] = {0, 0, 0, 0};
            for (const auto& c : ok_cands)
                if (per_order[std::get<3>(c)]++ < 4) keep.push_back(c);
            ok_cands.swap(keep);
        }
        const int nt = (int)kChunk;  // one full chunk: binned and paired as a large query is
        std::vector<float> tp((size_t)nt * d);
        for (int i = 0; i < nt; ++i)
            for (int k = 0; k < d; ++k) tp[(size_t)i * d + k] = (float)(H.lo[k] + rnd() * (H.hi[k] - H.lo[k]));
        float* dt = nullptr;
        double* wt = nullptr;
        cudaEvent_t e0 = nullptr, e1 = nullptr;
        bool ok = cudaMalloc(&dt, tp.size() * sizeof(float)) == cudaSuccess &&
                  cudaMalloc(&wt, (size_t)nt * sizeof(double)) == cudaSuccess &&
                  cudaMemcpy(dt, tp.data(), tp.size() * sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess &&
                  cudaEventCreate(&e0) == cudaSuccess && cudaEventCreate(&e1) == cudaSuccess &&
                  ensure_workspace(m, nt, 0) == GWN_OK;
        // best of two timed runs after one untimed run (microseconds)
        auto timed = [&](double b, double bl) -> double {
            gwn_query_opts q3;
            gwn_default_query_opts(&q3);
            q3.beta = b;
            q3.beta_leaf = bl;
            float best = 1e30f;
            for (int rep = 0; rep < 3 && ok; ++rep) {
                ok = cudaEventRecord(e0, 0) == cudaSuccess &&
                     gwn_enqueue_device(m, dt, GWN_F32, nt, wt, nullptr, nullptr, q3, 0, m->ws) == GWN_OK &&
                     cudaEventRecord(e1, 0) == cudaSuccess && cudaEventSynchronize(e1) == cudaSuccess;
                float ms = 0;
                if (ok && rep > 0 && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess) best = std::min(best, ms);
            }
            return 1e3 * best;
        };
        double best_t = 1e300;
        if (ok_cands.size() > 1) {
            for (const auto& c : ok_cands) {
                m->tree.order3 = d == 3 && std::get<3>(c) >= 3 ? 1 : 0;
                const double tus = timed(std::get<1>(c), std::get<2>(c));
                if (std::getenv("GWN_AUTOTUNE_VERBOSE"))
                    std::fprintf(stderr, "[gwn autotune] order=%d beta=%.1f beta_leaf=%.1f: %.1f us for %d points\n",
                                 std::get<3>(c), std::get<1>(c), std::get<2>(c), tus, nt);
                if (ok && tus < best_t) {
                    best_t = tus;
                    m->opts.beta = std::get<1>(c);
                    m->opts.beta_leaf = d == 3 ? std::get<2>(c) : 0.0;
                    m->eval_order = std::get<3>(c);
                }
            }
            m->tree.order3 = d == 3 && m->eval_order >= 3 ? 1 : 0;
        }
        if (d == 3 && ok) {
            const double bl = m->opts.beta_leaf > 0 ? m->opts.beta_leaf : m->opts.beta;
            int best_ppc = m->bin_ppc;
            double bt = 1e300;
            for (int ppc : {4, 8, 16, 32, 64}) {
                m->bin_ppc = ppc;
                const double tus = timed(m->opts.beta, bl);
                if (ok && tus < bt) {
                    bt = tus;
                    best_ppc = ppc;
                }
            }
            m->bin_ppc = best_ppc;
        }
        if (e0) cudaEventDestroy(e0);
        if (e1) cudaEventDestroy(e1);
        cudaFree(dt);
        cudaFree(wt);
        if (!ok) return fail(GWN_ERR_CUDA, "autotune timing failed");
    }
    // The automatic FP64 repair (more than 512 leaves): every validation point
    // whose value is fractional is sent through the repair (band 0.4999), and the
    // node and leaf factors are lowered from 3 while its values stay within 1e-7
    // of the FP64 direct sum; fewer FP64 pairs per repaired point.
    if (d == 3 && m->opts.beta_repair < 0 && H.n_leaves > 512 && m->opts.precision == GWN_PREC_FP32_REPAIR) {
        const double facs[][2] = {{3.0, 3.0}, {2.5, 2.5}, {2.5, 2.0}, {2.0, 2.0}, {2.0, 1.5}, {1.5, 1.5}};
        uint32_t* dst = nullptr;
        int* dcnt = nullptr;
        bool ok = cudaMalloc(&dst, nv * sizeof(uint32_t)) == cudaSuccess && cudaMalloc(&dcnt, sizeof(int)) == cudaSuccess;
        double keep_n = m->repair_node_factor, keep_l = m->repair_leaf_factor;
        for (const auto& f : facs) {
            if (!ok) break;
            m->repair_node_factor = f[0];
            m->repair_leaf_factor = f[1];
            gwn_query_opts qr;
            gwn_default_query_opts(&qr);
            qr.repair_band = 0.4999;
            double e = 0;
            int cnt = 0;
            ok = gwn_enqueue_device(m, dp, GWN_F32, nv, w, nullptr, dst, qr, 0, m->ws) == GWN_OK &&
                 cudaMemset(err, 0, sizeof(double)) == cudaSuccess && cudaMemset(dcnt, 0, sizeof(int)) == cudaSuccess;
            if (ok) k_err_repaired<<<4, 128>>>(nv, ref, w, dst, err, dcnt);
            ok = ok && cudaMemcpy(&e, err, sizeof(double), cudaMemcpyDeviceToHost) == cudaSuccess &&
                 cudaMemcpy(&cnt, dcnt, sizeof(int), cudaMemcpyDeviceToHost) == cudaSuccess;
            if (std::getenv("GWN_AUTOTUNE_VERBOSE"))
                std::fprintf(stderr, "[gwn autotune] repair factors %.1f / %.1f: max|dGWN| %.3g over %d repaired\n",
                             f[0], f[1], e, cnt);
            if (!ok || e > 1e-7) break;
            keep_n = f[0];
            keep_l = f[1];
        }
        m->repair_node_factor = keep_n;
        m->repair_leaf_factor = keep_l;
        if (dst) cudaFree(dst);
        if (dcnt) cudaFree(dcnt);
        if (!ok) return fail(GWN_ERR_CUDA, "autotune of the repair failed");
    }
    // the tuning workspace is not the model's: the first query sizes its own
    if (m->ws_mem) {
        cudaFree(m->ws_mem);
        m->ws_mem = nullptr;
        m->ws_n = 0;
        m->ws_bytes = 0;
    }
    return GWN_OK;
}

static gwn_status build_common(int dim, const void* prims, size_t n, const gwn_build_opts* opts, gwn_model* out) {
    if (!out) return fail(GWN_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    gwn_build_opts o;
    gwn_default_build_opts(&o);
    if (opts) o = *opts;
    gwn_status s = check_opts(o, dim);
    if (s != GWN_OK) return s;
    auto t0 = std::chrono::steady_clock::now();
    gwn_model_s* m = new (std::nothrow) gwn_model_s();
    if (!m) return fail(GWN_ERR_OOM, "host allocation failed");
    m->dim = dim;
    m->opts = o;
    m->eval_order = o.order;
    m->local_ratio = o.local_ratio > 0 ? o.local_ratio : 0.0;
    m->leaf_far = o.leaf_far < 0 ? (dim == 3 ? 1 : 0) : (o.leaf_far ? 1 : 0);
    m->n_primitives = (int64_t)n;
    gwn_status code = GWN_OK;
    std::string err;
    // the device stage of the 3D build runs on the model's device
    DeviceGuard dg(o.device == GWN_DEVICE_HOST_ONLY ? -1 : o.device);
    try {
        if (dim == 2) err = build_model_2d(reinterpret_cast<const gwn_curve2d*>(prims), n, o, &m->host, &code);
        else err = build_model_3d(reinterpret_cast<const gwn_patch3d*>(prims), n, o, &m->host, &code);
    } catch (const std::bad_alloc&) {
        delete m;
        return fail(GWN_ERR_OOM, "host allocation failed during build");
    } catch (const std::exception& e) {
        delete m;
        return fail(GWN_ERR_INTERNAL, e.what());
    }
    if (!err.empty()) {
        delete m;
        return fail(code == GWN_OK ? GWN_ERR_INTERNAL : code, err);
    }
    if (o.device == GWN_DEVICE_HOST_ONLY) {  // inspection only: no device upload
        m->device = GWN_DEVICE_HOST_ONLY;
        m->build_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
        *out = m;
        return GWN_OK;
    }
    DeviceGuard g(o.device);
    cudaGetDevice(&m->device);
    bool tune = o.beta == 0.0;
    if (tune) m->opts.beta = 2.0;
    s = finish_build(m, out);
    if (s != GWN_OK) return s;
    if (tune) {
        s = autotune(m);
        if (s != GWN_OK) {
            gwn_release(m);
            *out = nullptr;
            return s;
        }
    }
    m->build_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    return GWN_OK;
}

gwn_status gwn_build_2d(const gwn_curve2d* curves, size_t n, const gwn_build_opts* opts, gwn_model* out) {
    return build_common(2, curves, n, opts, out);
}

gwn_status gwn_build_3d(const gwn_patch3d* patches, size_t n, const gwn_build_opts* opts, gwn_model* out) {
    return build_common(3, patches, n, opts, out);
}

gwn_status gwn_query(gwn_model m, const void* points, int32_t dtype, int32_t mem, size_t n, double* out_w,
                     int32_t* out_label, uint32_t* out_status, const gwn_query_opts* qopts, void* stream) {
    if (!m) return fail(GWN_ERR_INVALID_ARG, "model is NULL");
    if (m->device == GWN_DEVICE_HOST_ONLY) return fail(GWN_ERR_INVALID_ARG, "model was built host-only");
    if (n == 0) return GWN_OK;
    if (!points || !out_w) return fail(GWN_ERR_INVALID_ARG, "points and out_w are required");
    if (dtype != GWN_F32 && dtype != GWN_F64) return fail(GWN_ERR_INVALID_ARG, "unknown points dtype");
    if (mem != GWN_MEM_DEVICE && mem != GWN_MEM_HOST) return fail(GWN_ERR_INVALID_ARG, "unknown memory kind");
    if (n > (size_t)0x7fffffff) return fail(GWN_ERR_INVALID_ARG, "at most 2^31 - 1 points per call");
    gwn_query_opts qo;
    gwn_default_query_opts(&qo);
    if (qopts) qo = *qopts;
    if (qo.mode != GWN_MODE_BVH && qo.mode != GWN_MODE_DIRECT) return fail(GWN_ERR_INVALID_ARG, "unknown mode");
    if (qo.precision < -1 || qo.precision > 2) return fail(GWN_ERR_INVALID_ARG, "unknown precision");
    if (qo.beta != 0.0 && !(qo.beta >= 2.0)) return fail(GWN_ERR_INVALID_ARG, "beta must be >= 2");
    if (qo.beta_leaf != 0.0 && !(qo.beta_leaf >= 2.0)) return fail(GWN_ERR_INVALID_ARG, "beta_leaf must be >= 2");
    if (!(qo.repair_band >= 0.0 && qo.repair_band < 0.5)) return fail(GWN_ERR_INVALID_ARG, "repair_band must be in [0, 0.5)");
    if (!(qo.local_ratio <= 0.0 || (qo.local_ratio >= 4.0 && qo.local_ratio < 1e6)))
        return fail(GWN_ERR_INVALID_ARG, "local_ratio must be <= 0 or in [4, 1e6)");
    DeviceGuard g(m->device);
    std::lock_guard<std::mutex> lk(m->mu);
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    size_t esz = dtype == GWN_F32 ? sizeof(float) : sizeof(double);
    size_t pbytes = n * m->dim * esz;
    size_t obytes = n * (sizeof(double) + sizeof(int32_t) + sizeof(uint32_t));
    gwn_status s = ensure_workspace(m, n, mem == GWN_MEM_HOST ? pbytes + obytes + 64 : 0);
    if (s != GWN_OK) return s;
    m->ws.list_points = (int)std::min(std::max<size_t>(n, 4096), kChunk);
    // calls on other streams share the model's workspace: start after the previous call's work
    if (!m->last) GWN_CUDA_TRY(cudaEventCreateWithFlags(&m->last, cudaEventDisableTiming));
    if (m->last_recorded) GWN_CUDA_TRY(cudaStreamWaitEvent(st, m->last, 0));
    // the end of whatever this call enqueued, also when a later enqueue fails:
    // the next call must not reuse the workspace under kernels already queued
    auto mark_last = [&]() {
        if (cudaEventRecord(m->last, st) == cudaSuccess) m->last_recorded = true;
    };
    if (mem == GWN_MEM_DEVICE) {
        s = gwn_enqueue_device(m, points, dtype, n, out_w, out_label, (uint32_t*)out_status, qo, st, m->ws);
        mark_last();
        return s;
    }
    // host buffers: stage through model-owned device memory
    char* base = reinterpret_cast<char*>(m->stage);
    void* dp = base;
    double* dw = reinterpret_cast<double*>(base + ((pbytes + 15) & ~size_t(15)));
    int32_t* dl = reinterpret_cast<int32_t*>(dw + n);
    uint32_t* ds = reinterpret_cast<uint32_t*>(dl + n);
    GWN_CUDA_TRY(cudaMemcpyAsync(dp, points, pbytes, cudaMemcpyHostToDevice, st));
    s = gwn_enqueue_device(m, dp, dtype, n, dw, out_label ? dl : nullptr, out_status ? ds : nullptr, qo, st, m->ws);
    if (s != GWN_OK) {
        mark_last();
        return s;
    }
    GWN_CUDA_TRY(cudaMemcpyAsync(out_w, dw, n * sizeof(double), cudaMemcpyDeviceToHost, st));
    if (out_label) GWN_CUDA_TRY(cudaMemcpyAsync(out_label, dl, n * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    if (out_status) GWN_CUDA_TRY(cudaMemcpyAsync(out_status, ds, n * sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
    GWN_CUDA_TRY(cudaEventRecord(m->last, st));
    m->last_recorded = true;
    GWN_CUDA_TRY(cudaStreamSynchronize(st));
    return GWN_OK;
}

}  // extern "C"

// ---------------------------------------------------------------- query without allocation
//
// gwn_query_noalloc runs the FP32 traversal with FP64 repair without asking the
// CUDA runtime for memory: its only scratch -- the list of points to repair
// and its counter -- is the file-scope device array below, which every GPU
// that loads this library holds until the process exits.  Host code cannot
// use g_noalloc_scratch's name as a device address; the address comes from
// cudaGetSymbolAddress, once per device, on the first call made with that
// device current.

static constexpr size_t kNoAllocMaxPoints = (size_t)1 << 20;   // points per call
static constexpr int kNoAllocHeader = 64;                      // counter, padded to 256 bytes
static __device__ __align__(256) int g_noalloc_scratch[kNoAllocHeader + kNoAllocMaxPoints];

namespace {
std::mutex g_noalloc_mu;
int* g_noalloc_addr[256] = {};
int g_noalloc_sms[256] = {};

// the array's device address and the device's SM count, looked up once per
// device (with that device current) and cached
gwn_status noalloc_scratch(int dev, int** out, int* sms) {
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (dev < 0 || dev >= 256) return fail(GWN_ERR_INVALID_ARG, "device ordinal out of range");
    if (!g_noalloc_addr[dev]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p)
            return fail(GWN_ERR_CUDA, std::string("cudaGetSymbolAddress(no-alloc scratch): ") + cudaGetErrorString(e));
        int n_sm = 0;
        e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess || n_sm <= 0)
            return fail(GWN_ERR_CUDA, std::string("cudaDeviceGetAttribute(SM count): ") + cudaGetErrorString(e));
        g_noalloc_sms[dev] = n_sm;
        g_noalloc_addr[dev] = reinterpret_cast<int*>(p);
    }
    *out = g_noalloc_addr[dev];
    *sms = g_noalloc_sms[dev];
    return GWN_OK;
}

// 2D, one thread per point: Algorithm 1 in FP32 with every leaf evaluated in place;
// points near a half-integer or flagged go to the repair list
__global__ void __launch_bounds__(128) k_query_noalloc2(DevTree t, const void* pts, int dtype, long long n, QueryParams p,
                                                        double* out_w, int* out_label, uint32_t* out_status, int* rlist,
                                                        int* rcount) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double qd[3];
    load_point(pts, dtype, 2, i, qd);
    uint32_t st = 0;
    double wd = (double)query2_32(t, (float)qd[0], (float)qd[1], p.beta2, st);
    if (near_half(wd, p.band) || (st & (GWN_QS_STACK_OVERFLOW | GWN_QS_UNRESOLVED))) rlist[atomicAdd(rcount, 1)] = (int)i;
    out_w[i] = wd;
    if (out_label) out_label[i] = (int)round(wd);
    if (out_status) out_status[i] = st;
}

// 3D: one warp per point with the far exact leaves in place (k_wide3), the near ones
// through a list, kNoAllocStep points at a time so that everything fits the
// fixed scratch: per point 16 bytes of position, 4 + 4 + 4 + 4 of sums, status and
// lists, 4 of FP64 status, 8 of near sums, 7 near pairs and 3 near-band pairs of 8 bytes (points
// with more are evaluated by one thread, k_overflow3; the repair's sums follow in the place of
// the third near-band pair): 124 bytes.  100,000
// points on 1.4k leaves, one thread per point with its leaves in place before: 44 ms.
constexpr size_t kNoAllocStep = 32768;
static_assert(kNoAllocStep * 124 + 4096 <= sizeof(int) * kNoAllocMaxPoints, "the no-alloc scratch holds one step");

gwn_status noalloc_3d(gwn_model_s* m, const QueryParams& p, const void* points, int dtype, size_t n, double* out_w,
                      int32_t* out_label, uint32_t* out_status, int* scratch, int sms, cudaStream_t st) {
    char* at = reinterpret_cast<char*>(scratch + kNoAllocHeader);
    auto carve = [&](size_t bytes) {
        char* r = at;
        at += (bytes + 255) & ~size_t(255);
        return r;
    };
    const size_t C = kNoAllocStep;
    Workspace ws{};
    ws.counters = scratch;
    ws.gcount = scratch + kCounterCount;
    ws.found = (unsigned long long*)(scratch + 2 * kCounterCount);
    ws.spos = (float4*)carve(C * 16);
    ws.near = (long long*)carve(C * 8);
    ws.pairs2 = (int2*)carve(C * 56);
    ws.slow_cap = (long long)C * 7;
    ws.pairs64 = (int2*)carve(C * 24);
    ws.rw = (double*)(ws.pairs64 + 2 * C);
    ws.wacc = (float*)carve(C * 4);
    ws.st = (uint32_t*)carve(C * 4);
    ws.rst = (uint32_t*)carve(C * 4);
    ws.olist2 = (int*)carve(C * 4);
    ws.rlist_g = (int*)carve(C * 4);
    const bool o3 = m->tree.order3 != 0;
    const int near_cap = (int)(3 * C);
    const size_t esz = (dtype == GWN_F32 ? sizeof(float) : sizeof(double)) * 3;
    const int B = 128;
    for (size_t off = 0; off < n; off += C) {
        const int c = (int)std::min(C, n - off);
        const unsigned nb = (unsigned)((c + B - 1) / B);
        const void* pts = reinterpret_cast<const char*>(points) + off * esz;
        double* w = out_w + off;
        int* label = out_label ? out_label + off : nullptr;
        uint32_t* status = out_status ? out_status + off : nullptr;
        // the array keeps the previous call's contents: the counters must start at zero
        GWN_CUDA_TRY(cudaMemsetAsync(scratch, 0, kNoAllocHeader * sizeof(int), st));
        k_scatter_points<3><<<nb, B, 0, st>>>(pts, dtype, c, nullptr, nullptr, ws.spos, ws.wacc, ws.st,
                                              ws.near);
        (o3 ? k_wide3<true, false, false> : k_wide3<false, false, false>)
            <<<(unsigned)std::min(((size_t)c + 3) / 4, (size_t)sms * 16), B, 0, st>>>(
                m->tree, ws.spos, c, nullptr, nullptr, p.beta2, p.beta2_leaf, ws, ws.pairs2, ws.slow_cap, ws.olist2, nullptr,
                Dense{nullptr, 0}, false);
        k_pair_eval<long long><<<(unsigned)(sms * kEvalBlocks), B, 0, st>>>(
            m->tree, ws.spos, ws.slow_cap, ws.counters + 8, ws.counters, ws.pairs2, ws.near, ws.st, ws.pairs64, near_cap,
            ws.olist2, nullptr);
        k_pair_eval64_warp<<<(unsigned)(sms * 2), B, 0, st>>>(m->tree, ws.spos, near_cap, ws.counters, ws.pairs64, ws.wacc,
                                                              ws.st, ws.near);
        k_overflow3<<<(unsigned)(sms * 2), B, 0, st>>>(m->tree, ws.spos, p.beta2, ws, ws.olist2, ws.near);
        k_finish<float><<<nb, B, 0, st>>>(c, ws.spos, ws.wacc, ws.st, p.precision, p.band, w, label, status, nullptr, nullptr,
                                          0, ws.rlist_g, ws.gcount, c, 0, ws.near);
        const RepairList R{ws.rlist_g, ws.gcount, c, ws.rw, ws.rst};
        k_rtrav_warp<true><<<(unsigned)(sms * 4), 32 * kRepairWarps, 0, st>>>(
            m->tree, pts, dtype, p.beta2_repair, R, p.beta2_repair, Rule64{kRatio64Repair, false}, false);
        k_rfinish<<<(unsigned)(sms * 2), B, 0, st>>>(R, w, label, status, true, GWN_QS_REPAIRED);
        GWN_CUDA_TRY(cudaGetLastError());
    }
    return GWN_OK;
}
}  // namespace

extern "C" gwn_status gwn_query_noalloc(gwn_model m, const void* points, int32_t dtype, size_t n, double* out_w,
                                        int32_t* out_label, uint32_t* out_status, void* stream) {
    if (!m) return fail(GWN_ERR_INVALID_ARG, "model is NULL");
    if (m->device == GWN_DEVICE_HOST_ONLY) return fail(GWN_ERR_INVALID_ARG, "model was built host-only");
    if (n == 0) return GWN_OK;
    if (!points || !out_w) return fail(GWN_ERR_INVALID_ARG, "points and out_w are required");
    if (dtype != GWN_F32 && dtype != GWN_F64) return fail(GWN_ERR_INVALID_ARG, "unknown points dtype");
    if (n > kNoAllocMaxPoints)
        return fail(GWN_ERR_INVALID_ARG, "gwn_query_noalloc takes at most " + std::to_string(kNoAllocMaxPoints) +
                                             " points per call (its scratch array has a fixed size); split the batch");
    DeviceGuard g(m->device);
    int* scratch = nullptr;
    int sms = 0;
    gwn_status s = noalloc_scratch(m->device, &scratch, &sms);
    if (s != GWN_OK) return s;
    int* rcount = scratch;
    int* rlist = scratch + kNoAllocHeader;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    QueryParams p{};
    p.work = nullptr;
    const double beta = m->opts.beta;
    const double beta_leaf = m->opts.beta_leaf > 0 ? m->opts.beta_leaf : beta;
    p.beta2 = (float)(beta * beta);
    p.beta2_leaf = (float)(beta_leaf * beta_leaf);
    double br = m->opts.beta_repair;
    if (br < 0) br = auto_beta_repair(m, beta);
    p.beta2_repair = br > 0 ? br * br : 0.0;
    p.band = (float)m->opts.repair_band;
    p.mode = GWN_MODE_BVH;
    p.precision = GWN_PREC_FP32_REPAIR;
    if (m->dim == 3) return noalloc_3d(m, p, points, dtype, n, out_w, out_label, out_status, scratch, sms, st);
    // the array keeps the previous call's contents: the counter must start at zero
    GWN_CUDA_TRY(cudaMemsetAsync(rcount, 0, sizeof(int), st));
    const int B = 128;
    const unsigned nb = (unsigned)((n + B - 1) / B);
    const unsigned rb = (unsigned)std::min<long long>(std::max<long long>(nb, sms * 4), (long long)sms * 8);
    k_query_noalloc2<<<nb, B, 0, st>>>(m->tree, points, dtype, (long long)n, p, out_w, out_label, out_status, rlist, rcount);
    k_repair2<<<rb, B, 0, st>>>(m->tree, points, dtype, p, out_w, out_label, out_status, rlist, rcount);
    GWN_CUDA_TRY(cudaGetLastError());
    return GWN_OK;
}

extern "C" {

gwn_status gwn_last_query_stats(gwn_model m, int64_t* out) {
    if (!m || !out) return fail(GWN_ERR_INVALID_ARG, "NULL argument");
    DeviceGuard g(m->device);
    std::lock_guard<std::mutex> lk(m->mu);
    unsigned long long c[kCounterCount] = {};
    unsigned long long wk[kWorkCount] = {};
    if (m->ws_mem) {
        GWN_CUDA_TRY(cudaDeviceSynchronize());
        GWN_CUDA_TRY(cudaMemcpy(c, m->ws.acc, sizeof(c), cudaMemcpyDeviceToHost));
        GWN_CUDA_TRY(cudaMemcpy(wk, m->ws.work, sizeof(wk), cudaMemcpyDeviceToHost));
    }
    for (int k = 0; k < kQueryStats; ++k) out[k] = 0;
    for (int k = 0; k < 4; ++k) out[k] = (int64_t)c[k];
    out[2] = (int64_t)c[2];           // near-band (FP64) pairs of both passes
    out[3] = (int64_t)(c[6] + c[3]);  // points whose pairs overflowed, in either pass
    for (int k = 0; k < 8; ++k) out[4 + k] = (int64_t)wk[k];
    out[14] = (int64_t)(c[8] + c[9]);  // pairs the full evaluator took (the rest came from the node tables)
    out[15] = (int64_t)wk[kWorkFastNodes];
    out[18] = (int64_t)wk[kWorkLocal];
    if (m->profiled) {
        double a = 0, b = 0, f = 0;
        for (int ch = 0; ch < m->prof_chunks; ++ch) {
            float x = 0, y = 0, z = 0;
            GWN_CUDA_TRY(cudaEventSynchronize(m->ev[ch][3]));
            GWN_CUDA_TRY(cudaEventElapsedTime(&x, m->ev[ch][0], m->ev[ch][1]));
            GWN_CUDA_TRY(cudaEventElapsedTime(&y, m->ev[ch][2], m->ev[ch][3]));
            GWN_CUDA_TRY(cudaEventElapsedTime(&z, m->ev[ch][2], m->ev[ch][4]));
            a += x;
            b += y;
            f += z;
        }
        out[12] = (int64_t)(a * 1000.0);
        out[13] = (int64_t)(b * 1000.0);
        out[16] = (int64_t)(f * 1000.0);
        out[17] = (int64_t)((b - f) * 1000.0);
    }
    return GWN_OK;
}

gwn_status gwn_model_info(gwn_model m, gwn_model_stats* s) {
    if (!m || !s) return fail(GWN_ERR_INVALID_ARG, "NULL argument");
    std::memset(s, 0, sizeof(*s));
    s->dim = m->dim;
    s->n_primitives = m->n_primitives;
    s->n_leaves = m->host.n_leaves;
    s->n_nodes = std::max(0, m->host.n_leaves - 1);
    s->max_depth = m->host.max_depth;
    s->device_bytes = (int64_t)m->device_bytes;
    s->build_ms = m->build_ms;
    s->beta = m->opts.beta;
    s->beta_repair = m->opts.beta_repair < 0 ? auto_beta_repair(m, m->opts.beta) : m->opts.beta_repair;
    s->repair_band = m->opts.repair_band;
    s->order = m->opts.order;
    s->eval_order = m->eval_order;
    s->local_ratio = m->dim == 3 ? m->local_ratio : 0.0;
    for (int k = 0; k < 3; ++k) {
        s->lo[k] = m->host.lo[k];
        s->hi[k] = m->host.hi[k];
    }
    s->beta_leaf = m->opts.beta_leaf > 0 ? m->opts.beta_leaf : m->opts.beta;
    s->device = m->device;
    s->bin_points_per_cell = m->dim == 3 ? m->bin_ppc : 0;
    s->stack_depth = m->stack_depth;
    {
        const double bl = m->opts.beta_leaf > 0 ? m->opts.beta_leaf : m->opts.beta;
        const double br = s->beta_repair;
        s->beta_repair_leaf = br > 0 ? (m->opts.beta_repair < 0 ? m->repair_leaf_factor * bl : br * bl / m->opts.beta)
                                     : 0.0;
    }
    return GWN_OK;
}

gwn_status gwn_model_leaves(gwn_model m, int64_t* prim, double* param) {
    if (!m) return fail(GWN_ERR_INVALID_ARG, "model is NULL");
    if (prim) std::memcpy(prim, m->host.leaf_prim.data(), m->host.leaf_prim.size() * sizeof(int64_t));
    if (param) std::memcpy(param, m->host.leaf_param.data(), m->host.leaf_param.size() * sizeof(double));
    return GWN_OK;
}

gwn_status gwn_model_tree(gwn_model m, int32_t* child, double* x0, double* r, double* mom) {
    if (!m) return fail(GWN_ERR_INVALID_ARG, "model is NULL");
    const HostModel& H = m->host;
    int ni = std::max(0, H.n_leaves - 1);
    if (child)
        for (int k = 0; k < ni; ++k) {
            child[2 * k] = H.child[k].x;
            child[2 * k + 1] = H.child[k].y;
        }
    if (x0) std::memcpy(x0, H.x0.data(), H.x0.size() * sizeof(double));
    if (r) std::memcpy(r, H.r.data(), H.r.size() * sizeof(double));
    if (mom) std::memcpy(mom, H.mom_c.data(), H.mom_c.size() * sizeof(double));
    return GWN_OK;
}

// ---------------------------------------------------------------- checkpoint
//
// A model file holds everything the device upload needs, so that a serving
// process can load a model without rebuilding it: a header (magic, format
// version, dimension, leaf mode, primitive count, build options after
// autotuning) and every host array of the model, each as a 64-bit element
// count followed by the raw elements.  Files are written and read on
// little-endian hosts (x86-64, aarch64) with the same struct layouts.

}  // extern "C"

namespace {
constexpr char kModelMagic[8] = {'G', 'W', 'N', 'M', 'O', 'D', 'E', 'L'};
constexpr uint32_t kModelVersion = 7;

template <typename V>
bool write_vec(FILE* f, const std::vector<V>& v) {
    const uint64_t n = v.size();
    return std::fwrite(&n, sizeof(n), 1, f) == 1 && (n == 0 || std::fwrite(v.data(), sizeof(V), n, f) == n);
}

// reads one array; `left` is the number of bytes of the file not read yet, so a
// corrupt count can neither allocate more than the file holds nor read past it
template <typename V>
bool read_vec(FILE* f, std::vector<V>* v, uint64_t* left) {
    uint64_t n = 0;
    if (*left < sizeof(n) || std::fread(&n, sizeof(n), 1, f) != 1) return false;
    *left -= sizeof(n);
    if (n > *left / sizeof(V)) return false;
    v->resize((size_t)n);
    if (n != 0 && std::fread(v->data(), sizeof(V), (size_t)n, f) != n) return false;
    *left -= n * sizeof(V);
    return true;
}

// Every array has the size the build gives it for the model's dimension and
// leaf count, every child index names a node or a leaf, each node and leaf
// except the root has exactly one parent (so the traversal ends), and every
// leaf's and boundary curve's ranges stay inside their tables.
bool host_model_consistent(const HostModel& H, int dim) {
    if (H.dim != dim || H.n_leaves < 1) return false;
    const size_t nl = (size_t)H.n_leaves, ni = nl - 1, d = (size_t)dim;
    const size_t fv = dim == 2 ? kMom2Vec : kMom3Vec, ff = dim == 2 ? kMom2F64 : kMom3F64;
    const size_t M = dim == 2 ? 2 + 4 + 8 : kLeafMom3;
    if (H.child.size() != ni || H.hdr.size() != ni || H.mom.size() != ni * fv || H.hdr64.size() != ni * 4 ||
        H.mom64.size() != ni * ff || H.lhdr.size() != nl || H.lmom.size() != nl * fv || H.lhdr64.size() != nl * 4 ||
        H.lmom64.size() != nl * ff || H.x0.size() != ni * d || H.r.size() != ni || H.mom_c.size() != ni * M ||
        H.leaf_prim.size() != nl || H.leaf_param.size() != nl * 4)
        return false;
    std::vector<unsigned char> parents(ni + nl, 0);
    for (size_t k = 0; k < ni; ++k)
        for (int c : {H.child[k].x, H.child[k].y}) {
            size_t slot;
            if (c >= 0) {
                if ((size_t)c >= ni || c == 0) return false;  // node 0 is the root
                slot = (size_t)c;
            } else {
                const long long li = ~(long long)c;
                if (li >= (long long)nl) return false;
                slot = ni + (size_t)li;
            }
            if (parents[slot]++) return false;
        }
    for (size_t k = 1; k < ni + nl; ++k)
        if (parents[k] != 1 && !(ni == 0 && k == 0)) return false;
    if (dim == 2) return H.leaf2.size() == nl * kLeaf2Vec && H.leaf2_64.size() == nl * kLeaf2F64;
    if (H.leaf3.size() != nl || H.net3.size() != nl * kNet3Vec || H.net3_64.size() != nl * 64 ||
        H.c3pts64.size() != H.c3pts.size() * 4 || H.c3n.size() != H.c3.size() * kC3NodeVec ||
        H.c3n64.size() != H.c3.size() * kC3Node64 ||
        H.c2.size() != H.c2mult.size() * kC2Vec ||
        H.c2_64.size() != H.c2mult.size() * 12)
        return false;
    for (const Curve3Info& c : H.c3)
        if (c.deg < 1 || c.deg > kMaxC3Deg || c.ctrl_off < 0 || c.min_level < 0 || c.min_level > kMaxMinLevel ||
            (size_t)c.ctrl_off + 2 * (2 * (size_t)c.deg + 1) > H.c3pts.size())
            return false;
    for (const Leaf3Info& I : H.leaf3)
        if (I.c3_off < 0 || I.c3_cnt < 0 || (size_t)I.c3_off + (size_t)I.c3_cnt > H.c3.size() || I.c2_off < 0 ||
            I.c2_cnt < 0 || (size_t)I.c2_off + (size_t)I.c2_cnt > H.c2mult.size())
            return false;
    return true;
}

// apply f to every array of the host model, in file order
template <typename F>
bool each_array(HostModel& H, F f) {
    return f(H.child) && f(H.hdr) && f(H.mom) && f(H.hdr64) && f(H.mom64) && f(H.lhdr) && f(H.lmom) &&
           f(H.lhdr64) && f(H.lmom64) && f(H.x0) && f(H.r) && f(H.mom_c) && f(H.leaf_prim) && f(H.leaf_param) &&
           f(H.leaf2) && f(H.leaf2_64) && f(H.leaf3) && f(H.net3) && f(H.net3_64) && f(H.c3) && f(H.c3pts) &&
           f(H.c3pts64) && f(H.c3n) && f(H.c3n64) && f(H.c2) && f(H.c2_64) && f(H.c2mult);
}
}  // namespace

extern "C" {

gwn_status gwn_model_save(gwn_model m, const char* path) {
    if (!m || !path) return fail(GWN_ERR_INVALID_ARG, "model and path are required");
    FILE* f = std::fopen(path, "wb");
    if (!f) return fail(GWN_ERR_INVALID_ARG, std::string("cannot open for writing: ") + path);
    const int32_t hdr[4] = {(int32_t)kModelVersion, m->dim, m->leaf_far, (int32_t)sizeof(gwn_build_opts)};
    const HostModel& H = m->host;
    const int32_t hm[5] = {H.dim, H.n_leaves, H.max_depth, m->bin_ppc, m->eval_order};
    const double rf[3] = {m->repair_node_factor, m->repair_leaf_factor, m->local_ratio};
    bool ok = std::fwrite(kModelMagic, 1, 8, f) == 8 && std::fwrite(hdr, sizeof(hdr), 1, f) == 1 &&
              std::fwrite(&m->n_primitives, sizeof(m->n_primitives), 1, f) == 1 &&
              std::fwrite(&m->opts, sizeof(gwn_build_opts), 1, f) == 1 && std::fwrite(hm, sizeof(hm), 1, f) == 1 &&
              std::fwrite(rf, sizeof(rf), 1, f) == 1 &&
              std::fwrite(H.lo, sizeof(H.lo), 1, f) == 1 && std::fwrite(H.hi, sizeof(H.hi), 1, f) == 1 &&
              each_array(const_cast<HostModel&>(H), [&](auto& v) { return write_vec(f, v); });
    ok = (std::fclose(f) == 0) && ok;
    return ok ? GWN_OK : fail(GWN_ERR_INTERNAL, std::string("write failed: ") + path);
}

gwn_status gwn_model_load(const char* path, int32_t device, gwn_model* out) {
    if (!path || !out) return fail(GWN_ERR_INVALID_ARG, "path and out are required");
    *out = nullptr;
    FILE* f = std::fopen(path, "rb");
    if (!f) return fail(GWN_ERR_INVALID_ARG, std::string("cannot open for reading: ") + path);
    gwn_model_s* m = new (std::nothrow) gwn_model_s();
    if (!m) {
        std::fclose(f);
        return fail(GWN_ERR_OOM, "host allocation failed");
    }
    char magic[8] = {};
    int32_t hdr[4] = {}, hm[5] = {};
    double rf[3] = {};
    bool ok = std::fread(magic, 1, 8, f) == 8 && std::memcmp(magic, kModelMagic, 8) == 0 &&
              std::fread(hdr, sizeof(hdr), 1, f) == 1 && hdr[0] == (int32_t)kModelVersion &&
              (hdr[1] == 2 || hdr[1] == 3) && hdr[3] == (int32_t)sizeof(gwn_build_opts) &&
              std::fread(&m->n_primitives, sizeof(m->n_primitives), 1, f) == 1 &&
              std::fread(&m->opts, sizeof(gwn_build_opts), 1, f) == 1 && std::fread(hm, sizeof(hm), 1, f) == 1 &&
              std::fread(rf, sizeof(rf), 1, f) == 1 &&
              std::fread(m->host.lo, sizeof(m->host.lo), 1, f) == 1 &&
              std::fread(m->host.hi, sizeof(m->host.hi), 1, f) == 1;
    try {
        // no array may hold more elements than the rest of the file has bytes
        long pos = ok ? std::ftell(f) : -1;
        struct stat sb;
        ok = ok && pos >= 0 && fstat(fileno(f), &sb) == 0 && (uint64_t)sb.st_size >= (uint64_t)pos;
        uint64_t left = ok ? (uint64_t)sb.st_size - (uint64_t)pos : 0;
        ok = ok && each_array(m->host, [&](auto& v) { return read_vec(f, &v, &left); });
        ok = ok && left == 0;  // nothing may follow the last array
    } catch (const std::bad_alloc&) {
        ok = false;
    }
    std::fclose(f);
    HostModel& H = m->host;
    if (ok) {
        m->dim = hdr[1];
        m->leaf_far = hdr[2] ? 1 : 0;
        H.dim = hm[0];
        H.n_leaves = hm[1];
        H.max_depth = hm[2];
        m->bin_ppc = hm[3];
        m->eval_order = hm[4];
        m->repair_node_factor = rf[0];
        m->repair_leaf_factor = rf[1];
        m->local_ratio = rf[2];
        ok = hm[3] >= 1 && hm[3] <= 4096 && rf[0] >= 1.0 && rf[0] <= 16.0 && rf[1] >= 1.0 && rf[1] <= 16.0 &&
             hm[4] >= 0 && hm[4] <= m->opts.order && (rf[2] == 0.0 || (rf[2] >= 4.0 && rf[2] < 1e6));
        // consistency of the arrays the kernels index
        ok = ok && host_model_consistent(H, m->dim);
    }
    if (!ok || check_opts(m->opts, m->dim) != GWN_OK) {
        delete m;
        return fail(GWN_ERR_INVALID_ARG, std::string("not a model file of this library version: ") + path);
    }
    m->opts.device = device;
    if (device == GWN_DEVICE_HOST_ONLY) {
        m->device = GWN_DEVICE_HOST_ONLY;
        *out = m;
        return GWN_OK;
    }
    auto t0 = std::chrono::steady_clock::now();
    DeviceGuard g(device);
    cudaGetDevice(&m->device);
    const bool tune = m->opts.beta == 0.0;  // saved from a host-only build: tune now
    if (tune) m->opts.beta = 2.0;
    gwn_status s = finish_build(m, out);
    if (s != GWN_OK) return s;
    if (tune) {
        s = autotune(m);
        if (s != GWN_OK) {
            gwn_release(m);
            *out = nullptr;
            return s;
        }
    }
    m->build_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    return GWN_OK;
}

gwn_status gwn_release(gwn_model m) {
    if (!m) return GWN_OK;
    if (m->device != GWN_DEVICE_HOST_ONLY) {
        DeviceGuard g(m->device);
        std::lock_guard<std::mutex> lk(m->mu);
        free_model_memory(m);
    }
    delete m;
    return GWN_OK;
}

const char* gwn_last_error(void) { return g_err.c_str(); }

const char* gwn_version(void) { return "gwn-gb300 0.1 (sm_103a)"; }

}  // extern "C"

gwn_status gwn_fail(gwn_status s, const std::string& msg) { return fail(s, msg); }

size_t gwn_workspace_bytes(int dim, int n_leaves, char* base, gwn::Workspace* ws) {
    return workspace_layout(dim, n_leaves, kChunk, base, ws);
}

size_t gwn_chunk_points() { return kChunk; }
