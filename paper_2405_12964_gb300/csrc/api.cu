// C ABI of the differential walk-on-spheres library: context, problem state,
// argument checks, device workspaces and the launch sequences of each call.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <unordered_map>
#include <vector>

#include "ctx.h"
#include "dwos_device.cuh"
#include "dwos_internal.h"

using namespace dwos;

namespace {

thread_local std::string g_create_err;

dwos_status fail(dwos_ctx* c, dwos_status s, const std::string& msg) {
    if (c) c->err = msg; else g_create_err = msg;
    return s;
}

// The search order a launch uses: the warp-wide one only where the tree supports it.
constexpr int kMaxRefits = 64;   // parameter updates between full BVH builds

constexpr int kStarWideMin = 128;

int effective_traversal(const dwos_ctx* c) {
    int t = c->opt.traversal;
    if (t < 0) t = 3;
    if (t == 1 && !c->bvh.cells_ok) return 0;   // a refit tree: its Morton cells no longer hold
    return ((t == 2 || t == 3) && !c->bvh.wide_ok) ? 0 : t;
}

dwos_status cuda_fail(dwos_ctx* c, cudaError_t e, const char* where) {
    std::string m = std::string(where) + ": " + cudaGetErrorString(e);
    cudaGetLastError();
    return fail(c, e == cudaErrorMemoryAllocation ? DWOS_ERR_OOM : DWOS_ERR_CUDA, m);
}

#define CK(call, where) do { cudaError_t e_ = (call); if (e_ != cudaSuccess) return cuda_fail(ctx, e_, where); } while (0)
#define CKC(c, call, where) do { cudaError_t e_ = (call); if (e_ != cudaSuccess) return cuda_fail(c, e_, where); } while (0)

template <typename T>
cudaError_t grow(T*& p, size_t& cap, size_t n) {
    if (n <= cap && p) return cudaSuccess;
    if (p) cudaFree(p);
    p = nullptr;
    cap = 0;
    size_t want = std::max<size_t>(n, 1);
    cudaError_t e = cudaMalloc(&p, want * sizeof(T));
    if (e == cudaSuccess) cap = want;
    return e;
}

// Copy n elements into device buffer `dst` from host or device `src`.
template <typename T>
cudaError_t to_device(dwos_ctx* ctx, T* dst, const T* src, size_t n, int mem) {
    if (n == 0) return cudaSuccess;
    return cudaMemcpyAsync(dst, src, n * sizeof(T), mem == DWOS_MEM_DEVICE ? cudaMemcpyDeviceToDevice
                                                                           : cudaMemcpyHostToDevice, ctx->stream);
}

template <typename T>
cudaError_t from_device(dwos_ctx* ctx, T* dst, const T* src, size_t n, int mem) {
    if (n == 0 || !dst) return cudaSuccess;
    return cudaMemcpyAsync(dst, src, n * sizeof(T), mem == DWOS_MEM_DEVICE ? cudaMemcpyDeviceToDevice
                                                                           : cudaMemcpyDeviceToHost, ctx->stream);
}

bool finite_all(const float* p, size_t n) {
    for (size_t i = 0; i < n; ++i) if (!std::isfinite(p[i])) return false;
    return true;
}

dwos_status check_mem(dwos_ctx* ctx, int mem) {
    if (mem != DWOS_MEM_HOST && mem != DWOS_MEM_DEVICE) return fail(ctx, DWOS_ERR_INVALID_ARG, "mem must be DWOS_MEM_HOST or DWOS_MEM_DEVICE");
    return DWOS_OK;
}

dwos_status check_device_ptr(dwos_ctx* ctx, const void* p, const char* name) {
    if (!p) return DWOS_OK;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) { cudaGetLastError(); return fail(ctx, DWOS_ERR_INVALID_ARG, std::string(name) + " is not a device pointer"); }
    if (a.type != cudaMemoryTypeDevice && a.type != cudaMemoryTypeManaged)
        return fail(ctx, DWOS_ERR_INVALID_ARG, std::string(name) + " is not device memory");
    if (a.device != ctx->device) return fail(ctx, DWOS_ERR_INVALID_ARG, std::string(name) + " lives on another device");
    return DWOS_OK;
}

dwos_status set_device(dwos_ctx* ctx) {
    CK(cudaSetDevice(ctx->device), "cudaSetDevice");
    return DWOS_OK;
}

// The counters of the current launch (of two buffers; the other one is kept
// zero for the next walk launch, which zeroes this one in turn).
inline DevCounters* cur_ctr(dwos_ctx* ctx) { return ctx->d_ctr + ctx->ctr_cur; }

// Normal cones of the silhouette candidates' tree.  A site (an endpoint in 2D,
// an edge in 3D) with its two normals n1, n2 oriented consistently across it
// is a silhouette from x only where n1 . (x - p) and n2 . (x - p) have
// opposite signs (the silhouette rule restated: 2D n = perp of the segment
// directions w -> v and v -> z, 3D n1 = (b - a) x (c - a), n2 = (z - a) x (b - a));
// a whole pair may be negated.  Each leaf's cone covers its sites' pairs,
// oriented so that the element's own normal is the same for all its sites;
// each node's cone covers its children's.  A site that ends the Neumann part,
// or any site when the part moves with theta, gets the whole sphere.
// The cones are built and tested from this many candidate elements up, for a
// Neumann part that does not move (walk kernel ms with / without them:
// icosphere of 200k triangles 0.97 s / 6.8 s, 20k 0.31 / 0.79 s; but 720
// triangles 41 / 35 ms, thermal slab 7.5 / 5.6 ms: the test costs more than
// it prunes on small trees).
constexpr int kConeMinSites = 1024;

struct Cone {
    double a[3] = {0, 0, 0};
    double t = 0;
    bool full = false, empty = true;
};

static void cone_add(Cone& c, const Cone& d) {
    if (d.empty || c.full) return;
    if (d.full) { c.full = true; c.empty = false; return; }
    if (c.empty) { c = d; return; }
    const double dot = c.a[0] * d.a[0] + c.a[1] * d.a[1] + c.a[2] * d.a[2];
    const double phi = std::acos(std::max(-1.0, std::min(1.0, dot)));
    if (phi + d.t <= c.t) return;
    if (phi + c.t <= d.t) { c = d; return; }
    const double t = 0.5 * (phi + c.t + d.t);
    if (t >= M_PI || phi >= M_PI - 1e-9) { c.full = true; return; }
    const double r = t - c.t;          // turn c's axis toward d's by r
    if (phi > 1e-12) {
        const double s0 = std::sin(phi - r) / std::sin(phi), s1 = std::sin(r) / std::sin(phi);
        double n = 0;
        for (int i = 0; i < 3; ++i) { c.a[i] = s0 * c.a[i] + s1 * d.a[i]; n += c.a[i] * c.a[i]; }
        n = std::sqrt(n);
        for (int i = 0; i < 3; ++i) c.a[i] /= n;
    }
    c.t = t;
}

static Cone cone_of(const double* n) {
    Cone c;
    const double l = std::sqrt(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
    if (!(l > 0)) { c.full = true; c.empty = false; return c; }
    for (int i = 0; i < 3; ++i) c.a[i] = n[i] / l;
    c.empty = false;
    return c;
}

static dwos_status build_silhouette_cones(dwos_ctx* ctx) {
    const int d = ctx->dim;
    const BvhBuffers& b = ctx->bvh_s;
    const int n_int = b.n_internal, n_leaf = b.n_tree + b.n_big;
    std::vector<Cone> leaf(n_leaf), node(std::max(n_int, 0));
    std::vector<int32_t> prim(n_leaf);
    CK(cudaMemcpy(prim.data(), b.prim_elem, sizeof(int32_t) * n_leaf, cudaMemcpyDeviceToHost), "copy leaves");
    const std::vector<float>& V = ctx->vert_neu_h;
    auto vx = [&](int v, int k) { return (double)V[(size_t)d * v + k]; };
    // the silhouette rule's collinear tolerance is relative to the distance from x to the
    // site's other vertices: as an angle about the perpendicular it reaches 1e-4 (distance) /
    // (segment length, 3D: triangle height over the edge); the smallest such length over the
    // candidates and the largest element size bound it in the walk kernel
    double h_min = INFINITY, l_max = 0;
    auto dist = [&](int p, int q) {
        double r = 0;
        for (int k = 0; k < d; ++k) r += (vx(p, k) - vx(q, k)) * (vx(p, k) - vx(q, k));
        return std::sqrt(r);
    };
    for (int l = 0; l < n_leaf; ++l) {
        Cone& c = leaf[l];
        if (ctx->neu_moving) { c.full = true; c.empty = false; continue; }
        const int site = ctx->sites_h[prim[l]];
        const int e = site >> 3, mask = site & 7;
        const int* t = ctx->elem_n_h.data() + (size_t)d * e;
        double ne[3] = {0, 0, 0};
        if (d == 2) {
            ne[0] = vx(t[1], 1) - vx(t[0], 1);
            ne[1] = -(vx(t[1], 0) - vx(t[0], 0));
        } else {
            double u[3], w[3];
            for (int k = 0; k < 3; ++k) { u[k] = vx(t[1], k) - vx(t[0], k); w[k] = vx(t[2], k) - vx(t[0], k); }
            ne[0] = u[1] * w[2] - u[2] * w[1]; ne[1] = u[2] * w[0] - u[0] * w[2]; ne[2] = u[0] * w[1] - u[1] * w[0];
        }
        cone_add(c, cone_of(ne));
        const double len_e = std::sqrt(ne[0] * ne[0] + ne[1] * ne[1] + ne[2] * ne[2]);
        for (int j = 0; j < d; ++j) l_max = std::max(l_max, dist(t[j], t[(j + 1) % d]));
        for (int j = 0; j < d; ++j) {
            if (!((mask >> j) & 1)) continue;
            const int nb = ctx->nadj_h[(size_t)d * e + j];
            if (nb < 0) { c.full = true; break; }
            if (d == 2) {
                h_min = std::min(h_min, std::min(len_e, dist(nb, t[j])));
                l_max = std::max(l_max, dist(nb, t[j]));
            } else {
                const double lab = dist(t[j], t[(j + 1) % 3]);
                double ab[3], az[3], cr[3];
                for (int k = 0; k < 3; ++k) { ab[k] = vx(t[(j + 1) % 3], k) - vx(t[j], k); az[k] = vx(nb, k) - vx(t[j], k); }
                cr[0] = az[1] * ab[2] - az[2] * ab[1]; cr[1] = az[2] * ab[0] - az[0] * ab[2]; cr[2] = az[0] * ab[1] - az[1] * ab[0];
                const double h2 = std::sqrt(cr[0] * cr[0] + cr[1] * cr[1] + cr[2] * cr[2]) / lab;
                h_min = std::min(h_min, std::min(len_e / lab, h2));
                l_max = std::max(l_max, std::max(dist(nb, t[j]), dist(nb, t[(j + 1) % 3])));
            }
            double n2[3] = {0, 0, 0};
            if (d == 2) {   // v -> z; the pair (perp(v - w), perp(z - v)) negated where perp(v - w) = -ne
                const int v = t[j];
                const double sgn = j == 1 ? 1.0 : -1.0;
                n2[0] = sgn * (vx(nb, 1) - vx(v, 1));
                n2[1] = -sgn * (vx(nb, 0) - vx(v, 0));
            } else {        // (z - a) x (b - a) for the edge a = t[j], b = t[j + 1]
                const int a = t[j], bb = t[(j + 1) % 3];
                double ab[3], az[3];
                for (int k = 0; k < 3; ++k) { ab[k] = vx(bb, k) - vx(a, k); az[k] = vx(nb, k) - vx(a, k); }
                n2[0] = az[1] * ab[2] - az[2] * ab[1]; n2[1] = az[2] * ab[0] - az[0] * ab[2]; n2[2] = az[0] * ab[1] - az[1] * ab[0];
            }
            cone_add(c, cone_of(n2));
        }
    }
    if (n_int > 0) {
        const int f4 = d == 2 ? BvhLayout<2>::kNodeF4 : BvhLayout<3>::kNodeF4;
        std::vector<float4> nodes((size_t)n_int * f4);
        CK(cudaMemcpy(nodes.data(), b.nodes, sizeof(float4) * nodes.size(), cudaMemcpyDeviceToHost), "copy nodes");
        // post-order over the tree from the root (node 0)
        std::vector<std::pair<int, int>> stack{{0, 0}};
        while (!stack.empty()) {
            auto& top = stack.back();
            const float4 m = nodes[(size_t)f4 * top.first + f4 - 1];
            int ch[2];
            std::memcpy(&ch[0], &m.x, sizeof(int));
            std::memcpy(&ch[1], &m.y, sizeof(int));
            if (top.second < 2) {
                const int c = ch[top.second++];
                if (c >= 0 && c != kEmptyChild) stack.push_back({c, 0});
                continue;
            }
            Cone& c = node[top.first];
            for (int k = 0; k < 2; ++k) {
                if (ch[k] == kEmptyChild) continue;
                cone_add(c, ch[k] >= 0 ? node[ch[k]] : leaf[~ch[k]]);
            }
            stack.pop_back();
        }
    }
    std::vector<float4> out((size_t)std::max(n_int, 0) + n_leaf);
    auto pack = [](const Cone& c) {
        if (c.full || c.empty) return make_float4(0.0f, 0.0f, 0.0f, 4.0f);
        return make_float4((float)c.a[0], (float)c.a[1], (float)c.a[2], (float)c.t + 1e-6f);
    };
    for (int i = 0; i < n_int; ++i) out[i] = pack(node[i]);
    for (int l = 0; l < n_leaf; ++l) out[(size_t)std::max(n_int, 0) + l] = pack(leaf[l]);
    ctx->cone_tol = h_min > 0 && std::isfinite(h_min) ? (float)(1e-4 / h_min) : 1e30f;
    ctx->cone_lmax = (float)l_max;
    if (ctx->sil_cones) cudaFree(ctx->sil_cones);
    ctx->sil_cones = nullptr;
    CK(cudaMalloc(&ctx->sil_cones, sizeof(float4) * out.size()), "alloc cones");
    CK(cudaMemcpy(ctx->sil_cones, out.data(), sizeof(float4) * out.size(), cudaMemcpyHostToDevice), "copy cones");
    return DWOS_OK;
}

// The Neumann data per compact Neumann element, on the device; none (NULL) when no data was
// given or it is zero on the whole Neumann part.
static dwos_status upload_neumann_data(dwos_ctx* ctx) {
    if (ctx->neu_data) cudaFree(ctx->neu_data);
    ctx->neu_data = nullptr;
    if (ctx->n_neumann == 0 || ctx->neu_data_h.size() != (size_t)ctx->n_elem) return DWOS_OK;
    std::vector<float> c(ctx->nmap_h.size());
    bool any = false;
    for (size_t i = 0; i < c.size(); ++i) {
        c[i] = ctx->neu_data_h[ctx->nmap_h[i]];
        any = any || c[i] != 0.0f;
    }
    if (!any) return DWOS_OK;
    CK(cudaMalloc(&ctx->neu_data, sizeof(float) * c.size()), "alloc Neumann data");
    CK(cudaMemcpy(ctx->neu_data, c.data(), sizeof(float) * c.size(), cudaMemcpyHostToDevice), "copy Neumann data");
    return DWOS_OK;
}

dwos_status rebuild(dwos_ctx* ctx) {
    ctx->inside_cached = -1;   // the inside flags belong to the old geometry
    ctx->refits = 0;
    if (ctx->n_neumann == 0) {
        CK(bvh_build(ctx->bvh, ctx->dim, ctx->vert, ctx->elem, ctx->n_elem, ctx->stream), "BVH build");
        return DWOS_OK;
    }
    // walk on stars: one tree over the Dirichlet part (distance queries), one over the Neumann part
    CK(bvh_build(ctx->bvh, ctx->dim, ctx->vert, ctx->elem_d, ctx->n_elem - ctx->n_neumann, ctx->stream), "BVH build");
    CK(bvh_build(ctx->bvh_n, ctx->dim, ctx->vert, ctx->elem_n, ctx->n_neumann, ctx->stream), "Neumann BVH build");
    if (ctx->n_sites > 0) {
        CK(bvh_build(ctx->bvh_s, ctx->dim, ctx->vert, ctx->elem_s, ctx->n_sites, ctx->stream), "silhouette BVH build");
        CK(cudaStreamSynchronize(ctx->stream), "synchronize");
        if (ctx->n_sites >= kConeMinSites && !ctx->neu_moving)
            if (dwos_status st = build_silhouette_cones(ctx)) return st;
    }
    DevNeumann N;
    N.nodes = ctx->bvh_n.nodes;
    N.prims = ctx->bvh_n.prims;
    N.prim_elem = ctx->bvh_n.prim_elem;
    N.n_internal = ctx->bvh_n.n_internal;
    N.n_tree = ctx->bvh_n.n_tree;
    N.n_big = ctx->bvh_n.n_big;
    N.pad = 0;
    N.elem = ctx->elem_n;
    N.adj = ctx->nadj;
    N.vert = ctx->vert;
    N.dmap = ctx->dmap;
    N.q_start = ctx->q_start;
    const bool sil = ctx->n_sites > 0;
    N.sil_nodes = sil ? ctx->bvh_s.nodes : nullptr;
    N.sil_prims = sil ? ctx->bvh_s.prims : nullptr;
    N.sil_prim = sil ? ctx->bvh_s.prim_elem : nullptr;
    N.sites = ctx->sites;
    N.sil_n_internal = sil ? ctx->bvh_s.n_internal : 0;
    N.sil_n_tree = sil ? ctx->bvh_s.n_tree : 0;
    N.sil_n_big = sil ? ctx->bvh_s.n_big : 0;
    N.n_sites = ctx->n_sites;
    const bool cones = sil && ctx->n_sites >= kConeMinSites && !ctx->neu_moving && ctx->sil_cones;
    N.sil_cone_node = cones ? ctx->sil_cones : nullptr;
    N.sil_cone_leaf = cones ? ctx->sil_cones + std::max(ctx->bvh_s.n_internal, 0) : nullptr;
    N.cone_tol = ctx->cone_tol;
    N.cone_lmax = ctx->cone_lmax;
    N.flux = ctx->neu_data;
    ctx->neu_host = N;
    CK(cudaMemcpyAsync(ctx->d_neu, &ctx->neu_host, sizeof(N), cudaMemcpyHostToDevice, ctx->stream),
       "copy Neumann part");
    CK(cudaStreamSynchronize(ctx->stream), "synchronize");
    return DWOS_OK;
}

__global__ void xor_flags_kernel(int n, const int* __restrict__ a, int* __restrict__ b) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] ^= a[i];
}

__global__ void map_ids_kernel(int n, const int* __restrict__ map, int* __restrict__ ids) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && ids[i] >= 0) ids[i] = map[ids[i]];
}

// Inside test by ray parity over the whole boundary: with a Neumann part the
// crossings of the two trees add up, so the parities combine by XOR.
cudaError_t inside_all(dwos_ctx* ctx, int n, const float* p, int* inside) {
    cudaError_t e = launch_inside(ctx->bvh, n, p, inside, ctx->stream);
    if (e != cudaSuccess || ctx->n_neumann == 0 || n <= 0) return e;
    e = grow(ctx->inside_tmp, ctx->inside_tmp_cap, (size_t)n);
    if (e == cudaSuccess) e = launch_inside(ctx->bvh_n, n, p, ctx->inside_tmp, ctx->stream);
    if (e != cudaSuccess) return e;
    xor_flags_kernel<<<(n + 255) / 256, 256, 0, ctx->stream>>>(n, ctx->inside_tmp, inside);
    return cudaGetLastError();
}

// Shared front half of every walk-running call: validate, stage the query
// points, optionally classify them, fill the problem descriptor, run the walks.
dwos_status run_walks(dwos_ctx* ctx, int n_query, const float* xq, int W, unsigned long long base,
                      int differential, int mem, uint32_t* trace_dev, dwos_walk_debug* dbg_dev,
                      float4* cv_sample = nullptr, float4* cv_end = nullptr, const float4* cv_elem = nullptr) {
    if (!ctx->have_boundary) return fail(ctx, DWOS_ERR_STATE, "no boundary: call dwos_set_boundary first");
    if (n_query < 0 || W < 1) return fail(ctx, DWOS_ERR_INVALID_ARG, "n_query must be >= 0 and walks_per_point >= 1");
    if (n_query > 0 && !xq) return fail(ctx, DWOS_ERR_INVALID_ARG, "xq is NULL");
    const unsigned long long total = (unsigned long long)n_query * (unsigned long long)W;
    if (total > (1ull << 40)) return fail(ctx, DWOS_ERR_INVALID_ARG, "too many walks in one call");
    if (mem == DWOS_MEM_HOST && n_query > 0 && !finite_all(xq, (size_t)n_query * ctx->dim))
        return fail(ctx, DWOS_ERR_INVALID_ARG, "query points must be finite");
    if (mem == DWOS_MEM_DEVICE) { dwos_status s = check_device_ptr(ctx, xq, "xq"); if (s) return s; }
    CK(grow(ctx->rec, ctx->rec_cap, (size_t)total), "alloc records");
    // device query points are read in place (stream order); host ones are staged
    const float* d_xq = xq;
    if (mem == DWOS_MEM_HOST) {
        CK(grow(ctx->xq, ctx->xq_cap, (size_t)n_query * ctx->dim), "alloc xq");
        CK(to_device(ctx, ctx->xq, xq, (size_t)n_query * ctx->dim, mem), "copy xq");
        d_xq = ctx->xq;
    }
    ctx->xq_in = d_xq;
    const int* valid = nullptr;
    if (ctx->n_neumann > 0) {
        if (ctx->opt.dudn_estimator != 0)
            return fail(ctx, DWOS_ERR_INVALID_ARG, "a Neumann part needs the backward-difference du/dn estimator");
        if (cv_sample || cv_end || cv_elem)
            return fail(ctx, DWOS_ERR_NOT_IMPLEMENTED, "control variates with a Neumann part");
    }
    if (ctx->opt.check_inside && n_query > 0) {
        CK(grow(ctx->valid, ctx->valid_cap, (size_t)n_query), "alloc inside flags");
        if (ctx->n_neumann == 0) {
            // the flags of points equal to the previous call's (same geometry) are kept
            CK(grow(ctx->xq_prev, ctx->xq_prev_cap, (size_t)n_query * ctx->dim), "alloc inside cache");
            const bool cached = ctx->inside_cached == n_query;
            ctx->inside_cached = -1;
            CK(launch_inside(ctx->bvh, n_query, d_xq, ctx->valid, ctx->stream, cached ? ctx->xq_prev : nullptr,
                             ctx->xq_prev), "inside test");
            ctx->inside_cached = n_query;
            ctx->launches += 1;
        } else {
            CK(inside_all(ctx, n_query, d_xq, ctx->valid), "inside test");
            ctx->launches += 3;
        }
        valid = ctx->valid;
    }
    if (ctx->n_neumann > 0 && n_query > 0) {
        // query points on the Neumann part (within 1e-3 eps) start their walks on it, the
        // element's normal oriented out of the domain by an inside test behind its centre
        CK(grow(ctx->q_start, ctx->q_start_cap, (size_t)n_query), "alloc start states");
        CK(grow(ctx->behind, ctx->behind_cap, (size_t)n_query * ctx->dim), "alloc start states");
        CK(grow(ctx->behind_in, ctx->behind_in_cap, (size_t)n_query), "alloc start states");
        if (ctx->neu_host.q_start != ctx->q_start) {
            ctx->neu_host.q_start = ctx->q_start;
            CK(cudaMemcpyAsync(ctx->d_neu, &ctx->neu_host, sizeof(DevNeumann), cudaMemcpyHostToDevice, ctx->stream),
               "copy Neumann part");
        }
        CK(launch_neumann_start(ctx->dim, n_query, d_xq, ctx->neu_host, 1e-3f * ctx->opt.eps, ctx->q_start,
                                ctx->behind, ctx->stream), "Neumann start");
        CK(inside_all(ctx, n_query, ctx->behind, ctx->behind_in), "Neumann start orientation");
        CK(launch_neumann_orient(n_query, ctx->behind_in, ctx->q_start,
                                 ctx->opt.check_inside ? ctx->valid : nullptr, ctx->stream), "Neumann start");
        ctx->launches += 5;
    }
    DevProblem P;
    std::memset(&P, 0, sizeof(P));
    P.nodes = ctx->bvh.nodes;
    P.prims = ctx->bvh.prims;
    P.prim_elem = ctx->bvh.prim_elem;
    P.elem = ctx->elem;
    P.g_vert = ctx->g_vert;
    P.root = 0;
    P.n_internal = ctx->bvh.n_internal;
    P.n_tree = ctx->bvh.n_tree;
    P.n_big = ctx->bvh.n_big;
    P.leaf_parent = ctx->bvh.leaf_parent;
    P.node_cell = ctx->bvh.node_cell;
    P.r_max = ctx->bvh.r_max;
    P.traversal = effective_traversal(ctx);
    P.wnodes = ctx->bvh.wnodes;
    P.n_wide = ctx->bvh.n_wide;
    P.data_kind = ctx->data_kind;
    P.differential = differential;
    for (int i = 0; i < 10; ++i) P.field[i] = (float)ctx->field[i];
    P.sqrt_sigma = std::sqrt(ctx->sigma);
    P.f = ctx->f;
    P.eps = ctx->opt.eps;
    P.h = ctx->opt.h;
    P.inv_h = 1.0f / ctx->opt.h;
    P.K = ctx->opt.K;
    P.max_steps = ctx->opt.max_steps;
    P.dudn_mode = ctx->opt.dudn_estimator;
    P.seed_lo = (uint32_t)ctx->opt.seed;
    P.seed_hi = (uint32_t)(ctx->opt.seed >> 32);
    P.xq = d_xq;
    P.valid = valid;
    P.walks = W;
    P.node_budget = ctx->node_budget;
    P.walk_id_base = base;
    P.work_begin = 0;
    P.work_end = total;
    P.rec = ctx->rec;
    P.trace = trace_dev;
    P.dbg = dbg_dev;
    P.cv_sample = cv_sample;
    P.cv_end = cv_end;
    P.cv_elem = cv_elem;
    P.neu = ctx->n_neumann > 0 ? ctx->d_neu : nullptr;
    // walk on stars, automatic order: the Dirichlet part's tree is searched per lane below
    // kStarWideMin elements (measured: 64-68 elements 23-28 % faster per lane, 128 and 256
    // elements 12 % and 3.3x faster warp-wide)
    if (P.neu && ctx->opt.traversal < 0 && ctx->n_elem - ctx->n_neumann < kStarWideMin) P.traversal = 0;
    if (cv_sample) CK(cudaMemsetAsync(cv_sample, 0xff, sizeof(float4) * total, ctx->stream), "init samples");
    // counters: this launch takes the zeroed buffer and zeroes the other for the next one
    if (!ctx->ctr_next_zero)
        CK(cudaMemsetAsync(ctx->d_ctr + (ctx->ctr_cur ^ 1), 0, sizeof(DevCounters), ctx->stream), "reset counters");
    ctx->ctr_cur ^= 1;
    ctx->ctr_next_zero = false;
    WalkLaunch L;
    L.dim = ctx->dim;
    L.block_size = ctx->opt.block_size > 0 ? ctx->opt.block_size : 256;
    L.blocks_per_sm = ctx->opt.blocks_per_sm;
    L.n_sm = ctx->n_sm;
    L.traversal = P.traversal;
    L.wide_depth = ctx->bvh.wide_depth;
    L.star = P.neu != nullptr;
    L.cones = L.star && ctx->neu_host.sil_cone_node != nullptr;
    L.data = L.star && ctx->neu_host.flux != nullptr;
    CK(cudaEventRecord(ctx->ev0, ctx->stream), "event");
    int blocks = 0;
    CK(launch_walks(L, nullptr, 1, total, cur_ctr(ctx), ctx->stream, &blocks, &P, ctx->d_ctr + (ctx->ctr_cur ^ 1)),
       "walk kernel");
    ctx->ctr_next_zero = true;
    ctx->launches += blocks > 0 ? 1 : 0;
    ctx->last_blocks = blocks;
    CK(cudaEventRecord(ctx->ev1, ctx->stream), "event");
    ctx->timed = true;
    return DWOS_OK;
}

// After a synchronous call: report device-side flags.
dwos_status finish_sync(dwos_ctx* ctx) {
    CK(cudaStreamSynchronize(ctx->stream), "synchronize");
    DevCounters c;
    CK(cudaMemcpy(&c, cur_ctr(ctx), sizeof(c), cudaMemcpyDeviceToHost), "read counters");
    if (c.error & 4) return fail(ctx, DWOS_ERR_INVALID_ARG, "a query point is not finite");
    if (c.error & 2) return fail(ctx, DWOS_ERR_OUTSIDE, "a query point lies outside the domain");
    if (c.error & 1) return fail(ctx, DWOS_ERR_STEP_LIMIT, "BVH traversal exceeded its iteration bound");
    return DWOS_OK;
}

// An element whose normal the walks cannot form: the squared length of a
// segment, or of a triangle's edge cross product, is zero (or not finite) in
// the FP32 arithmetic the walk kernel uses for it.
__host__ __device__ inline bool degenerate_element(int dim, const float* a, const float* b, const float* c) {
    float n2;
    if (dim == 2) {
        const float tx = b[0] - a[0], ty = b[1] - a[1];
        n2 = tx * tx + ty * ty;
    } else {
        const float e1[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]};
        const float e2[3] = {c[0] - a[0], c[1] - a[1], c[2] - a[2]};
        const float cr[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2], e1[0] * e2[1] - e1[1] * e2[0]};
        n2 = cr[0] * cr[0] + cr[1] * cr[1] + cr[2] * cr[2];
    }
    return !(n2 > 0.0f && n2 < __builtin_inff());
}

// Checks of boundary arrays that live on the device: bit 0 a vertex or Jacobian
// entry is not finite, bit 1 an element's vertex id is out of range, bit 2 an
// element is degenerate.
__global__ void validate_boundary_kernel(int dim, int n_vert, const float* __restrict__ vert, int n_elem,
                                         const int* __restrict__ elem, long long n_jac,
                                         const float* __restrict__ jac, int* __restrict__ flags) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    int bad = 0;
    for (long long i = i0; i < (long long)n_vert * dim; i += stride)
        if (!isfinite(vert[i])) bad |= 1;
    for (long long i = i0; i < n_jac; i += stride)
        if (!isfinite(jac[i])) bad |= 1;
    for (long long e = i0; e < n_elem; e += stride) {
        const int* ev = elem + (size_t)dim * e;
        bool in_range = true;
        for (int k = 0; k < dim; ++k) in_range = in_range && ev[k] >= 0 && ev[k] < n_vert;
        if (!in_range) { bad |= 2; continue; }
        const float* a = vert + (size_t)dim * ev[0];
        const float* b = vert + (size_t)dim * ev[1];
        const float* c = dim == 3 ? vert + (size_t)dim * ev[2] : a;
        if (degenerate_element(dim, a, b, c)) bad |= 4;
    }
    if (bad) atomicOr(flags, bad);
}

}  // namespace

extern "C" {

void dwos_default_options(dwos_options* o) {
    if (!o) return;
    o->eps = 1e-3f;
    o->h = 1e-2f;
    o->K = 1;
    o->B = 8;
    o->max_steps = 1 << 14;
    o->seed = 0x12964ull;
    o->check_inside = 1;
    o->block_size = 0;
    o->blocks_per_sm = 0;
    o->traversal = -1;
    o->dudn_estimator = 0;
}

dwos_status dwos_create(dwos_ctx** out, int device) {
    if (!out) return fail(nullptr, DWOS_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    int n = 0;
    cudaError_t e = cudaGetDeviceCount(&n);
    if (e != cudaSuccess) { cudaGetLastError(); return fail(nullptr, DWOS_ERR_CUDA, std::string("no CUDA device: ") + cudaGetErrorString(e)); }
    if (device < 0 || device >= n) return fail(nullptr, DWOS_ERR_INVALID_ARG, "device index out of range");
    dwos_ctx* ctx = new (std::nothrow) dwos_ctx();
    if (!ctx) return fail(nullptr, DWOS_ERR_OOM, "host allocation failed");
    ctx->device = device;
    dwos_default_options(&ctx->opt);
    cudaError_t ce = cudaSetDevice(device);
    if (ce == cudaSuccess) ce = cudaDeviceGetAttribute(&ctx->n_sm, cudaDevAttrMultiProcessorCount, device);
    if (ce == cudaSuccess) ce = cudaMalloc(&ctx->d_ctr, 2 * sizeof(DevCounters));
    if (ce == cudaSuccess) ce = cudaMalloc(&ctx->d_err, sizeof(int));
    if (ce == cudaSuccess) ce = cudaEventCreate(&ctx->ev0);
    if (ce == cudaSuccess) ce = cudaEventCreate(&ctx->ev1);
    if (ce == cudaSuccess) ce = cudaMemset(ctx->d_ctr, 0, 2 * sizeof(DevCounters));
    if (ce != cudaSuccess) {
        cudaGetLastError();
        g_create_err = std::string("context setup failed: ") + cudaGetErrorString(ce);
        dwos_destroy(ctx);
        return ce == cudaErrorMemoryAllocation ? DWOS_ERR_OOM : DWOS_ERR_CUDA;
    }
    *out = ctx;
    return DWOS_OK;
}

void dwos_destroy(dwos_ctx* ctx) {
    if (!ctx) return;
    cudaSetDevice(ctx->device);
    if (ctx->stream) cudaStreamSynchronize(ctx->stream);
    bvh_free(ctx->bvh);
    void* bufs[] = {ctx->vert_ref, ctx->vert, ctx->elem, ctx->jac, ctx->theta, ctx->g_vert, ctx->dg_vert, ctx->rec,
                    ctx->xq, ctx->valid, ctx->wvec, ctx->out, ctx->acc_vert, ctx->trace, ctx->dbg, ctx->misc_f,
                    ctx->misc_i, ctx->misc_u, ctx->xq_prev, ctx->d_ctr, ctx->d_err, ctx->pw, ctx->vert_active,
                    ctx->misc_d, ctx->elem_d, ctx->elem_n, ctx->dmap, ctx->nadj, ctx->d_neu, ctx->inside_tmp,
                    ctx->q_start, ctx->behind, ctx->behind_in, ctx->sites, ctx->elem_s, ctx->sil_cones,
                    ctx->neu_data};
    bvh_free(ctx->bvh_n);
    bvh_free(ctx->bvh_s);
    for (void* p : bufs) if (p) cudaFree(p);
    if (ctx->ev0) cudaEventDestroy(ctx->ev0);
    if (ctx->ev1) cudaEventDestroy(ctx->ev1);
    delete ctx;
}

dwos_status dwos_set_stream(dwos_ctx* ctx, void* stream) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    ctx->stream = (cudaStream_t)stream;
    return DWOS_OK;
}

const char* dwos_last_error(const dwos_ctx* ctx) {
    return ctx ? ctx->err.c_str() : g_create_err.c_str();
}

dwos_status dwos_sync(dwos_ctx* ctx) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    dwos_status s = set_device(ctx);
    if (s) return s;
    return finish_sync(ctx);
}

dwos_status dwos_set_options(dwos_ctx* ctx, const dwos_options* o) {
    if (!ctx || !o) return fail(ctx, DWOS_ERR_INVALID_ARG, "NULL argument");
    if (!(o->eps > 0.0f) || !std::isfinite(o->eps)) return fail(ctx, DWOS_ERR_INVALID_ARG, "eps must be > 0");
    if (!(o->h > 0.0f) || !std::isfinite(o->h)) return fail(ctx, DWOS_ERR_INVALID_ARG, "h must be > 0");
    if (o->K < 1 || o->K > 255) return fail(ctx, DWOS_ERR_INVALID_ARG, "K must be in [1, 255]");
    if (!(o->B == 2 || o->B == 4 || o->B == 8 || o->B == 16 || o->B == 32))
        return fail(ctx, DWOS_ERR_INVALID_ARG, "B must be 2, 4, 8, 16 or 32");
    if (o->max_steps < 1 || o->max_steps >= (1 << 24)) return fail(ctx, DWOS_ERR_INVALID_ARG, "max_steps must be in [1, 2^24)");
    if (o->block_size != 0 && (o->block_size < 32 || o->block_size > 256 || o->block_size % 32))
        return fail(ctx, DWOS_ERR_INVALID_ARG, "block_size must be 0 or a multiple of 32 in [32, 256]");
    if (o->blocks_per_sm < 0 || o->blocks_per_sm > 64) return fail(ctx, DWOS_ERR_INVALID_ARG, "blocks_per_sm must be in [0, 64]");
    if (o->dudn_estimator < 0 || o->dudn_estimator > 1)
        return fail(ctx, DWOS_ERR_INVALID_ARG, "dudn_estimator must be 0 or 1");
    if (o->traversal < -1 || o->traversal > 3)
        return fail(ctx, DWOS_ERR_INVALID_ARG, "traversal must be -1 (automatic), 0, 1, 2 or 3");
    ctx->opt = *o;
    return DWOS_OK;
}

dwos_status dwos_set_boundary(dwos_ctx* ctx, int dim, int n_vert, const float* vert_ref, int n_elem,
                              const int32_t* elem, int n_param, const float* vert_jac, int mem) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (dwos_status s = check_mem(ctx, mem)) return s;
    if (dim != 2 && dim != 3) return fail(ctx, DWOS_ERR_INVALID_ARG, "dim must be 2 or 3");
    if (n_vert < dim || n_elem < 1) return fail(ctx, DWOS_ERR_INVALID_ARG, "empty boundary");
    if (n_param < 0 || (n_param > 0 && !vert_jac)) return fail(ctx, DWOS_ERR_INVALID_ARG, "n_param > 0 needs vert_jac");
    if (!vert_ref || !elem) return fail(ctx, DWOS_ERR_INVALID_ARG, "NULL vertex or element array");
    if ((long long)n_elem >= (1ll << 30)) return fail(ctx, DWOS_ERR_INVALID_ARG, "too many elements");
    if (mem == DWOS_MEM_HOST) {
        if (!finite_all(vert_ref, (size_t)n_vert * dim)) return fail(ctx, DWOS_ERR_INVALID_ARG, "vertices must be finite");
        for (long long i = 0; i < (long long)n_elem * dim; ++i)
            if (elem[i] < 0 || elem[i] >= n_vert) return fail(ctx, DWOS_ERR_INVALID_ARG, "element vertex id out of range");
        for (long long e = 0; e < n_elem; ++e) {
            const int32_t* ev = elem + (size_t)dim * e;
            const float* a = vert_ref + (size_t)dim * ev[0];
            const float* b = vert_ref + (size_t)dim * ev[1];
            if (degenerate_element(dim, a, b, dim == 3 ? vert_ref + (size_t)dim * ev[2] : a))
                return fail(ctx, DWOS_ERR_INVALID_ARG, "element " + std::to_string(e) +
                                                           " is degenerate (zero length or area)");
        }
        if (n_param > 0 && !finite_all(vert_jac, (size_t)n_vert * dim * n_param))
            return fail(ctx, DWOS_ERR_INVALID_ARG, "Jacobian must be finite");
    } else {
        for (const void* p : {(const void*)vert_ref, (const void*)elem, (const void*)vert_jac})
            if (dwos_status s = check_device_ptr(ctx, p, "boundary array")) return s;
    }
    if (dwos_status s = set_device(ctx)) return s;
    CK(cudaStreamSynchronize(ctx->stream), "synchronize");
    for (void* p : {(void*)ctx->vert_ref, (void*)ctx->vert, (void*)ctx->elem, (void*)ctx->jac, (void*)ctx->theta,
                    (void*)ctx->g_vert, (void*)ctx->dg_vert}) if (p) cudaFree(p);
    ctx->vert_ref = ctx->vert = ctx->jac = ctx->theta = ctx->g_vert = ctx->dg_vert = nullptr;
    ctx->elem = nullptr;
    ctx->have_boundary = false;
    for (void* p : {(void*)ctx->elem_d, (void*)ctx->elem_n, (void*)ctx->dmap, (void*)ctx->nadj, (void*)ctx->sites,
                    (void*)ctx->elem_s, (void*)ctx->sil_cones}) if (p) cudaFree(p);
    ctx->elem_d = ctx->elem_n = ctx->dmap = ctx->nadj = ctx->sites = ctx->elem_s = nullptr;
    ctx->sil_cones = nullptr;
    ctx->n_neumann = 0;
    ctx->n_sites = 0;
    if (ctx->neu_data) cudaFree(ctx->neu_data);
    ctx->neu_data = nullptr;
    ctx->neu_data_h.clear();
    ctx->nmap_h.clear();
    const size_t nv = (size_t)n_vert * dim;
    CK(cudaMalloc(&ctx->vert_ref, nv * sizeof(float)), "alloc vertices");
    CK(cudaMalloc(&ctx->vert, nv * sizeof(float)), "alloc vertices");
    CK(cudaMalloc(&ctx->elem, (size_t)n_elem * dim * sizeof(int)), "alloc elements");
    CK(cudaMalloc(&ctx->g_vert, (size_t)n_vert * sizeof(float)), "alloc data");
    CK(cudaMalloc(&ctx->theta, (size_t)std::max(n_param, 1) * sizeof(float)), "alloc theta");
    if (n_param > 0) CK(cudaMalloc(&ctx->jac, nv * n_param * sizeof(float)), "alloc Jacobian");
    CK(to_device(ctx, ctx->vert_ref, vert_ref, nv, mem), "copy vertices");
    CK(cudaMemcpyAsync(ctx->vert, ctx->vert_ref, nv * sizeof(float), cudaMemcpyDeviceToDevice, ctx->stream), "copy vertices");
    CK(to_device(ctx, ctx->elem, elem, (size_t)n_elem * dim, mem), "copy elements");
    if (n_param > 0) CK(to_device(ctx, ctx->jac, vert_jac, nv * n_param, mem), "copy Jacobian");
    if (mem == DWOS_MEM_DEVICE) {   // the host checks above, run on the device copies
        CK(cudaMemsetAsync(ctx->d_err, 0, sizeof(int), ctx->stream), "reset flag");
        const long long work = std::max<long long>((long long)n_elem, (long long)nv * std::max(n_param, 1));
        const int blocks = (int)std::min<long long>((work + 255) / 256, 4096);
        validate_boundary_kernel<<<blocks, 256, 0, ctx->stream>>>(dim, n_vert, ctx->vert_ref, n_elem, ctx->elem,
                                                                 n_param > 0 ? (long long)nv * n_param : 0, ctx->jac,
                                                                 ctx->d_err);
        CK(cudaGetLastError(), "validate boundary");
        int flags = 0;
        CK(cudaMemcpyAsync(&flags, ctx->d_err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream), "read flag");
        CK(cudaStreamSynchronize(ctx->stream), "synchronize");
        ctx->launches += 1;
        if (flags & 1) return fail(ctx, DWOS_ERR_INVALID_ARG, "vertices and Jacobian must be finite");
        if (flags & 2) return fail(ctx, DWOS_ERR_INVALID_ARG, "element vertex id out of range");
        if (flags & 4) return fail(ctx, DWOS_ERR_INVALID_ARG, "an element is degenerate (zero length or area)");
    }
    CK(cudaMemsetAsync(ctx->g_vert, 0, (size_t)n_vert * sizeof(float), ctx->stream), "zero data");
    CK(cudaMemsetAsync(ctx->theta, 0, (size_t)std::max(n_param, 1) * sizeof(float), ctx->stream), "zero theta");
    ctx->dim = dim; ctx->n_vert = n_vert; ctx->n_elem = n_elem; ctx->n_param = n_param;
    ctx->data_kind = 0;
    ctx->active_stale = true;
    std::memset(ctx->field, 0, sizeof(ctx->field));
    if (dwos_status s = rebuild(ctx)) return s;
    CK(cudaStreamSynchronize(ctx->stream), "BVH build");
    ctx->have_boundary = true;
    return DWOS_OK;
}

dwos_status dwos_set_params(dwos_ctx* ctx, const float* theta, int mem) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (!ctx->have_boundary) return fail(ctx, DWOS_ERR_STATE, "no boundary");
    if (dwos_status s = check_mem(ctx, mem)) return s;
    if (ctx->n_param == 0) return DWOS_OK;
    if (!theta) return fail(ctx, DWOS_ERR_INVALID_ARG, "theta is NULL");
    if (mem == DWOS_MEM_HOST && !finite_all(theta, ctx->n_param)) return fail(ctx, DWOS_ERR_INVALID_ARG, "theta must be finite");
    if (mem == DWOS_MEM_DEVICE) if (dwos_status s = check_device_ptr(ctx, theta, "theta")) return s;
    if (dwos_status s = set_device(ctx)) return s;
    CK(to_device(ctx, ctx->theta, theta, ctx->n_param, mem), "copy theta");
    CK(launch_apply_params(ctx->vert_ref, ctx->jac, ctx->theta, ctx->vert, ctx->n_vert * ctx->dim, ctx->n_param,
                           ctx->stream), "apply theta");
    // the same elements moved: refit the trees' boxes (no host synchronisation), with a
    // full rebuild every kMaxRefits updates to restore the tree's quality, and for
    // search order 1, which needs the Morton cells of a fresh build
    if (ctx->refits < kMaxRefits && ctx->opt.traversal != 1) {
        ctx->inside_cached = -1;
        CK(bvh_refit(ctx->bvh, ctx->vert, ctx->n_neumann > 0 ? ctx->elem_d : ctx->elem, ctx->stream), "BVH refit");
        if (ctx->n_neumann > 0) CK(bvh_refit(ctx->bvh_n, ctx->vert, ctx->elem_n, ctx->stream), "Neumann BVH refit");
        if (ctx->n_sites > 0) CK(bvh_refit(ctx->bvh_s, ctx->vert, ctx->elem_s, ctx->stream), "silhouette BVH refit");
        ++ctx->refits;
        ctx->launches += 3;
        return DWOS_OK;
    }
    return rebuild(ctx);
}

dwos_status dwos_set_dirichlet_mapped(dwos_ctx* ctx, const float* g_vert, const float* dg_vert, int mem) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (!ctx->have_boundary) return fail(ctx, DWOS_ERR_STATE, "no boundary");
    if (dwos_status s = check_mem(ctx, mem)) return s;
    if (!g_vert) return fail(ctx, DWOS_ERR_INVALID_ARG, "g_vert is NULL");
    if (mem == DWOS_MEM_HOST) {
        if (!finite_all(g_vert, ctx->n_vert)) return fail(ctx, DWOS_ERR_INVALID_ARG, "g_vert must be finite");
        if (dg_vert && !finite_all(dg_vert, (size_t)ctx->n_vert * ctx->n_param))
            return fail(ctx, DWOS_ERR_INVALID_ARG, "dg_vert must be finite");
    }
    if (dg_vert && ctx->n_param == 0) return fail(ctx, DWOS_ERR_INVALID_ARG, "dg_vert given but n_param = 0");
    if (dwos_status s = set_device(ctx)) return s;
    CK(to_device(ctx, ctx->g_vert, g_vert, ctx->n_vert, mem), "copy g");
    if (ctx->dg_vert) { CK(cudaStreamSynchronize(ctx->stream), "synchronize"); cudaFree(ctx->dg_vert); ctx->dg_vert = nullptr; }
    if (dg_vert) {
        CK(cudaMalloc(&ctx->dg_vert, (size_t)ctx->n_vert * ctx->n_param * sizeof(float)), "alloc dg");
        CK(to_device(ctx, ctx->dg_vert, dg_vert, (size_t)ctx->n_vert * ctx->n_param, mem), "copy dg");
    }
    ctx->data_kind = 0;
    ctx->active_stale = true;
    return DWOS_OK;
}

dwos_status dwos_set_dirichlet_field(dwos_ctx* ctx, const double* coeffs) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (!coeffs) return fail(ctx, DWOS_ERR_INVALID_ARG, "coeffs is NULL");
    for (int i = 0; i < 10; ++i) if (!std::isfinite(coeffs[i])) return fail(ctx, DWOS_ERR_INVALID_ARG, "coeffs must be finite");
    std::memcpy(ctx->field, coeffs, sizeof(ctx->field));
    ctx->data_kind = 1;
    ctx->active_stale = true;
    return DWOS_OK;
}

dwos_status dwos_set_pde(dwos_ctx* ctx, float sigma, float f) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (!(sigma >= 0.0f) || !std::isfinite(sigma)) return fail(ctx, DWOS_ERR_INVALID_ARG, "sigma must be finite and >= 0");
    if (!std::isfinite(f)) return fail(ctx, DWOS_ERR_INVALID_ARG, "f must be finite");
    ctx->sigma = sigma;
    ctx->f = f;
    return DWOS_OK;
}

dwos_status dwos_set_neumann(dwos_ctx* ctx, const int32_t* flags, int mem) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (!ctx->have_boundary) return fail(ctx, DWOS_ERR_STATE, "no boundary: call dwos_set_boundary first");
    if (dwos_status s = check_mem(ctx, mem)) return s;
    if (mem == DWOS_MEM_DEVICE) if (dwos_status s = check_device_ptr(ctx, flags, "flags")) return s;
    if (dwos_status s = set_device(ctx)) return s;
    const int n = ctx->n_elem, d = ctx->dim;
    std::vector<int32_t> f(n, 0);
    if (flags) CK(cudaMemcpyAsync(f.data(), flags, sizeof(int32_t) * n, mem == DWOS_MEM_DEVICE ? cudaMemcpyDeviceToHost
                                                                                              : cudaMemcpyHostToHost,
                                  ctx->stream), "copy flags");
    std::vector<int32_t> el((size_t)n * d);
    CK(cudaMemcpyAsync(el.data(), ctx->elem, sizeof(int32_t) * el.size(), cudaMemcpyDeviceToHost, ctx->stream), "copy elements");
    CK(cudaStreamSynchronize(ctx->stream), "synchronize");
    std::vector<int32_t> ed, en, dmap;
    std::vector<int32_t> nmap;
    for (int e = 0; e < n; ++e) {
        if (f[e] != 0 && f[e] != 1) return fail(ctx, DWOS_ERR_INVALID_ARG, "flags must be 0 or 1");
        auto& dst = f[e] ? en : ed;
        for (int k = 0; k < d; ++k) dst.push_back(el[(size_t)d * e + k]);
        (f[e] ? nmap : dmap).push_back(e);
    }
    const int n_n = (int)(en.size() / d);
    if (n_n > 0 && n_n == n) return fail(ctx, DWOS_ERR_INVALID_ARG, "the boundary needs a Dirichlet part");
    for (void* p : {(void*)ctx->elem_d, (void*)ctx->elem_n, (void*)ctx->dmap, (void*)ctx->nadj, (void*)ctx->sites,
                    (void*)ctx->elem_s, (void*)ctx->sil_cones}) if (p) cudaFree(p);
    ctx->elem_d = ctx->elem_n = ctx->dmap = ctx->nadj = ctx->sites = ctx->elem_s = nullptr;
    ctx->sil_cones = nullptr;
    ctx->n_neumann = 0;
    ctx->n_sites = 0;
    ctx->nmap_h = nmap;
    if (n_n == 0) {                               // every element Dirichlet again
        if (dwos_status st = upload_neumann_data(ctx)) return st;
        return rebuild(ctx);
    }
    // neighbours across each endpoint (segments) or edge (triangles) within the Neumann part
    std::vector<int32_t> adj((size_t)n_n * d, -1);
    std::unordered_map<unsigned long long, std::vector<int>> at;
    auto key = [](int a, int b) {
        const unsigned lo = (unsigned)std::min(a, b), hi = (unsigned)std::max(a, b);
        return ((unsigned long long)hi << 32) | lo;
    };
    for (int c = 0; c < n_n; ++c)
        for (int j = 0; j < d; ++j) {
            const int* t = en.data() + (size_t)d * c;
            at[d == 2 ? (unsigned long long)(unsigned)t[j] : key(t[j], t[(j + 1) % 3])].push_back(c);
        }
    for (int c = 0; c < n_n; ++c) {
        const int* t = en.data() + (size_t)d * c;
        for (int j = 0; j < d; ++j) {
            const auto& list = at[d == 2 ? (unsigned long long)(unsigned)t[j] : key(t[j], t[(j + 1) % 3])];
            for (int o : list) {
                if (o == c) continue;
                const int* u = en.data() + (size_t)d * o;
                if (d == 2) adj[2 * (size_t)c + j] = u[0] == t[j] ? u[1] : u[0];
                else for (int i = 0; i < 3; ++i)
                    if (u[i] != t[j] && u[i] != t[(j + 1) % 3]) adj[3 * (size_t)c + j] = u[i];
                break;
            }
        }
    }
    // silhouette candidates: the sites where the Neumann part ends or does not run straight on
    // (a vertex between two segments whose directions agree, an edge between two coplanar
    // triangles is a silhouette from no point); every site one of whose vertices moves with
    // theta.  The walk kernel applies the same test with a relative 1e-6; a site is left out
    // here only if it is straight within 1e-7, so that rounding cannot leave out one the
    // kernel would keep.
    std::vector<float> vh((size_t)ctx->n_vert * d);
    CK(cudaMemcpy(vh.data(), ctx->vert, sizeof(float) * vh.size(), cudaMemcpyDeviceToHost), "copy vertices");
    std::vector<char> moves(ctx->n_vert, 0);
    if (ctx->n_param > 0 && ctx->jac) {
        std::vector<float> jh((size_t)ctx->n_vert * d * ctx->n_param);
        CK(cudaMemcpy(jh.data(), ctx->jac, sizeof(float) * jh.size(), cudaMemcpyDeviceToHost), "copy Jacobian");
        for (size_t v = 0; v < (size_t)ctx->n_vert; ++v)
            for (size_t q = 0; q < (size_t)d * ctx->n_param && !moves[v]; ++q)
                moves[v] = jh[v * d * ctx->n_param + q] != 0.0f;
    }
    auto vx = [&](int v, int k) { return (double)vh[(size_t)d * v + k]; };
    std::vector<int32_t> sites, elem_s;
    for (int c = 0; c < n_n; ++c) {
        const int* t = en.data() + (size_t)d * c;
        int mask = 0;
        for (int j = 0; j < d; ++j) {
            const int nb = adj[(size_t)d * c + j];
            bool straight = false;
            const bool moving = nb >= 0 && (moves[t[0]] || moves[t[1]] || (d == 3 && moves[t[2]]) || moves[nb]);
            if (nb >= 0 && !moving) {
                double u1[3] = {0, 0, 0}, u2[3] = {0, 0, 0};
                if (d == 2) {   // directions w -> v and v -> z at v = t[j]
                    for (int k = 0; k < 2; ++k) { u1[k] = vx(t[j], k) - vx(t[1 - j], k); u2[k] = vx(nb, k) - vx(t[j], k); }
                } else {        // normals (b - a) x (c - a) and (z - a) x (b - a) of the edge ab
                    const int a = t[j], b = t[(j + 1) % 3], cc = t[(j + 2) % 3];
                    double ab[3], ac[3], az[3];
                    for (int k = 0; k < 3; ++k) { ab[k] = vx(b, k) - vx(a, k); ac[k] = vx(cc, k) - vx(a, k); az[k] = vx(nb, k) - vx(a, k); }
                    u1[0] = ab[1] * ac[2] - ab[2] * ac[1]; u1[1] = ab[2] * ac[0] - ab[0] * ac[2]; u1[2] = ab[0] * ac[1] - ab[1] * ac[0];
                    u2[0] = az[1] * ab[2] - az[2] * ab[1]; u2[1] = az[2] * ab[0] - az[0] * ab[2]; u2[2] = az[0] * ab[1] - az[1] * ab[0];
                }
                const double dot = u1[0] * u2[0] + u1[1] * u2[1] + u1[2] * u2[2];
                const double n1 = u1[0] * u1[0] + u1[1] * u1[1] + u1[2] * u1[2];
                const double n2 = u2[0] * u2[0] + u2[1] * u2[1] + u2[2] * u2[2];
                straight = dot >= (1.0 - 1e-7) * std::sqrt(n1 * n2);
            }
            if (!straight) mask |= 1 << j;
        }
        if (!mask) continue;
        sites.push_back(8 * c + mask);
        for (int j = 0; j < d; ++j) elem_s.push_back(t[j]);
    }
    if (!sites.empty()) {
        CK(cudaMalloc(&ctx->sites, sizeof(int32_t) * sites.size()), "alloc silhouette sites");
        CK(cudaMalloc(&ctx->elem_s, sizeof(int32_t) * elem_s.size()), "alloc silhouette sites");
        CK(cudaMemcpy(ctx->sites, sites.data(), sizeof(int32_t) * sites.size(), cudaMemcpyHostToDevice), "copy");
        CK(cudaMemcpy(ctx->elem_s, elem_s.data(), sizeof(int32_t) * elem_s.size(), cudaMemcpyHostToDevice), "copy");
    }
    ctx->n_sites = (int)sites.size();
    ctx->elem_n_h = en;
    ctx->nadj_h = adj;
    ctx->sites_h = sites;
    ctx->vert_neu_h = vh;
    ctx->neu_moving = false;
    for (size_t i = 0; i < en.size() && !ctx->neu_moving; ++i) ctx->neu_moving = moves[en[i]] != 0;
    CK(cudaMalloc(&ctx->elem_d, sizeof(int32_t) * ed.size()), "alloc Dirichlet elements");
    CK(cudaMalloc(&ctx->elem_n, sizeof(int32_t) * en.size()), "alloc Neumann elements");
    CK(cudaMalloc(&ctx->dmap, sizeof(int32_t) * dmap.size()), "alloc element map");
    CK(cudaMalloc(&ctx->nadj, sizeof(int32_t) * adj.size()), "alloc neighbours");
    if (!ctx->d_neu) CK(cudaMalloc(&ctx->d_neu, sizeof(DevNeumann)), "alloc Neumann descriptor");
    CK(cudaMemcpy(ctx->elem_d, ed.data(), sizeof(int32_t) * ed.size(), cudaMemcpyHostToDevice), "copy");
    CK(cudaMemcpy(ctx->elem_n, en.data(), sizeof(int32_t) * en.size(), cudaMemcpyHostToDevice), "copy");
    CK(cudaMemcpy(ctx->dmap, dmap.data(), sizeof(int32_t) * dmap.size(), cudaMemcpyHostToDevice), "copy");
    CK(cudaMemcpy(ctx->nadj, adj.data(), sizeof(int32_t) * adj.size(), cudaMemcpyHostToDevice), "copy");
    ctx->n_neumann = n_n;
    if (dwos_status st = upload_neumann_data(ctx)) return st;
    return rebuild(ctx);
}

dwos_status dwos_set_neumann_data(dwos_ctx* ctx, const float* h, int mem) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (!ctx->have_boundary) return fail(ctx, DWOS_ERR_STATE, "no boundary: call dwos_set_boundary first");
    if (dwos_status s = check_mem(ctx, mem)) return s;
    if (mem == DWOS_MEM_DEVICE) if (dwos_status s = check_device_ptr(ctx, h, "h")) return s;
    if (dwos_status s = set_device(ctx)) return s;
    std::vector<float> hv;
    if (h) {
        hv.resize(ctx->n_elem);
        CK(cudaMemcpyAsync(hv.data(), h, sizeof(float) * hv.size(), mem == DWOS_MEM_DEVICE ? cudaMemcpyDeviceToHost
                                                                                           : cudaMemcpyHostToHost,
                           ctx->stream), "copy Neumann data");
        CK(cudaStreamSynchronize(ctx->stream), "synchronize");
        if (!finite_all(hv.data(), hv.size())) return fail(ctx, DWOS_ERR_INVALID_ARG, "Neumann data must be finite");
    }
    ctx->neu_data_h = hv;
    if (dwos_status st = upload_neumann_data(ctx)) return st;
    if (ctx->n_neumann > 0) {
        ctx->neu_host.flux = ctx->neu_data;
        CK(cudaMemcpyAsync(ctx->d_neu, &ctx->neu_host, sizeof(DevNeumann), cudaMemcpyHostToDevice, ctx->stream),
           "copy Neumann part");
        CK(cudaStreamSynchronize(ctx->stream), "synchronize");
    }
    return DWOS_OK;
}

dwos_status dwos_set_traversal_budget(dwos_ctx* ctx, int max_fetches) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (max_fetches < 0) return fail(ctx, DWOS_ERR_INVALID_ARG, "max_fetches must be >= 0");
    ctx->node_budget = max_fetches;
    return DWOS_OK;
}

dwos_status dwos_eval(dwos_ctx* ctx, int n_query, const float* xq, int W, double* u_mean, double* u_se,
                      double* du_mean, double* du_se, int mem) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (dwos_status s = check_mem(ctx, mem)) return s;
    if (!u_mean && n_query > 0) return fail(ctx, DWOS_ERR_INVALID_ARG, "u_mean is NULL");
    if (du_mean && ctx->n_param == 0) return fail(ctx, DWOS_ERR_INVALID_ARG, "derivatives requested but n_param = 0");
    if (mem == DWOS_MEM_DEVICE)
        for (const void* p : {(const void*)u_mean, (const void*)u_se, (const void*)du_mean, (const void*)du_se})
            if (dwos_status s = check_device_ptr(ctx, p, "output")) return s;
    if (dwos_status s = set_device(ctx)) return s;
    if (n_query == 0) return DWOS_OK;   // nothing to estimate
    const int diff = du_mean ? 1 : 0;
    if (dwos_status s = run_walks(ctx, n_query, xq, W, 0, diff, mem, nullptr, nullptr)) return s;
    const int N = ctx->n_param;
    const size_t need = 2 * (size_t)n_query + (diff ? 2 * (size_t)n_query * N : 0);
    CK(grow(ctx->out, ctx->out_cap, need), "alloc outputs");
    double* m = mem == DWOS_MEM_DEVICE ? u_mean : ctx->out;
    double* se = mem == DWOS_MEM_DEVICE ? u_se : ctx->out + n_query;
    if (!diff) {
        CK(launch_reduce_u(ctx->rec, n_query, W, m, se, ctx->stream), "reduce u");
    } else {
        double* dm = mem == DWOS_MEM_DEVICE ? du_mean : ctx->out + 2 * (size_t)n_query;
        double* ds = mem == DWOS_MEM_DEVICE ? du_se : ctx->out + 2 * (size_t)n_query + (size_t)n_query * N;
        CK(launch_reduce_udot(ctx->rec, ctx->elem, ctx->jac, ctx->dg_vert, ctx->dim, N, n_query, W, m, se, dm, ds,
                              ctx->n_sm, ctx->stream), "reduce udot");
    }
    ctx->launches += n_query > 0 ? 1 : 0;
    if (mem == DWOS_MEM_HOST) {
        CK(from_device(ctx, u_mean, ctx->out, n_query, mem), "copy u");
        CK(from_device(ctx, u_se, ctx->out + n_query, n_query, mem), "copy se");
        if (diff) {
            CK(from_device(ctx, du_mean, ctx->out + 2 * (size_t)n_query, (size_t)n_query * N, mem), "copy du");
            CK(from_device(ctx, du_se, ctx->out + 2 * (size_t)n_query + (size_t)n_query * N, (size_t)n_query * N, mem), "copy du se");
        }
        return finish_sync(ctx);
    }
    return DWOS_OK;
}

// Per-vertex flags: a nonzero Jacobian or dg row (recomputed after the boundary or the
// data changed).  The scatter skips unflagged vertices when only the parameter gradient
// is wanted: their accumulators meet zero rows in the adjoint GEMV.
static dwos_status ensure_vert_active(dwos_ctx* ctx) {
    if (!ctx->active_stale && ctx->vert_active) return DWOS_OK;
    CK(grow(ctx->vert_active, ctx->vert_active_cap, (size_t)std::max(ctx->n_vert, 1)), "alloc vertex flags");
    CK(launch_vertex_active(ctx->jac, ctx->dg_vert, ctx->n_vert, ctx->dim, ctx->n_param, ctx->vert_active,
                            ctx->stream), "vertex flags");
    ctx->launches += 1;
    ctx->active_stale = false;
    return DWOS_OK;
}

// mode 0: VJP with cotangent wv; 1: squared-loss gradient, U-statistic product; 2: correlated
// product; 3: uncorrelated product (wv = uref for modes 1-3).
static dwos_status reverse_common(dwos_ctx* ctx, int n_query, const float* xq, const float* wv, int W,
                                  unsigned long long base, int mode, double* loss, double* grad_param,
                                  double* grad_vert, int mem, const float* pweight = nullptr) {
    if (dwos_status s = check_mem(ctx, mem)) return s;
    if (!wv && n_query > 0) return fail(ctx, DWOS_ERR_INVALID_ARG, mode ? "uref is NULL" : "w is NULL");
    if (ctx->n_param > 0 && !grad_param) return fail(ctx, DWOS_ERR_INVALID_ARG, "grad_param is NULL");
    if (mode == 1 && W % ctx->opt.B) return fail(ctx, DWOS_ERR_INVALID_ARG, "walks_per_point must be a multiple of B");
    if (mode == 3 && (W < 2 || W % 2)) return fail(ctx, DWOS_ERR_INVALID_ARG, "walks_per_point must be even");
    if (mode >= 1 && !loss) return fail(ctx, DWOS_ERR_INVALID_ARG, "loss is NULL");
    if (mem == DWOS_MEM_HOST && wv && !finite_all(wv, n_query)) return fail(ctx, DWOS_ERR_INVALID_ARG, "weights must be finite");
    if (mem == DWOS_MEM_DEVICE)
        for (const void* p : {(const void*)wv, (const void*)loss, (const void*)grad_param, (const void*)grad_vert})
            if (dwos_status s = check_device_ptr(ctx, p, "argument")) return s;
    if (dwos_status s = set_device(ctx)) return s;
    if (dwos_status s = run_walks(ctx, n_query, xq, W, base, 1, mem, nullptr, nullptr)) return s;
    const int N = ctx->n_param;
    // device weights are read in place (stream order); host ones are staged
    const float* d_w = wv;
    if (mem == DWOS_MEM_HOST) {
        CK(grow(ctx->wvec, ctx->wvec_cap, (size_t)std::max(n_query, 1)), "alloc weights");
        CK(to_device(ctx, ctx->wvec, wv, (size_t)n_query, mem), "copy weights");
        d_w = ctx->wvec;
    }
    const float* d_pw = nullptr;
    if (pweight) {
        d_pw = pweight;
        if (mem == DWOS_MEM_HOST) {
            CK(grow(ctx->pw, ctx->pw_cap, (size_t)std::max(n_query, 1)), "alloc point weights");
            CK(to_device(ctx, ctx->pw, pweight, (size_t)n_query, mem), "copy point weights");
            d_pw = ctx->pw;
        }
    }
    // accumulators: per-vertex sums (and data sums), then the per-point sums of u (U-statistic mode)
    const size_t nvacc = (size_t)ctx->n_vert * ctx->dim + (size_t)ctx->n_vert;
    const size_t nacc = nvacc + (mode == 1 ? (size_t)n_query : 0);
    CK(grow(ctx->acc_vert, ctx->acc_cap, nacc), "alloc accumulators");
    CK(cudaMemsetAsync(ctx->acc_vert, 0, nacc * sizeof(double), ctx->stream), "zero accumulators");
    double* acc_g = ctx->dg_vert ? ctx->acc_vert + (size_t)ctx->n_vert * ctx->dim : nullptr;
    double* d_usum = mode == 1 ? ctx->acc_vert + nvacc : nullptr;
    const size_t need = 2 * (size_t)n_query + (size_t)std::max(N, 1) + 1;
    CK(grow(ctx->out, ctx->out_cap, need), "alloc outputs");
    double* d_umean = ctx->out + std::max(N, 1) + n_query + 1;   // per-point mean for the product weights
    if (mode == 2 || mode == 3) {
        CK(launch_reduce_u(ctx->rec, n_query, W, d_umean, nullptr, ctx->stream, nullptr, mode == 3 ? W / 2 : W),
           "reduce u");
        ctx->launches += n_query > 0 ? 1 : 0;
    }
    const unsigned char* active = nullptr;   // every vertex when the vertex gradient is returned
    if (!grad_vert) {
        if (dwos_status s = ensure_vert_active(ctx)) return s;
        active = ctx->vert_active;
    }
    double* d_grad = mem == DWOS_MEM_DEVICE ? grad_param : ctx->out;
    // the scatter also zeroes the parameter gradient the adjoint GEMV accumulates into
    CK(launch_scatter(ctx->rec, ctx->elem, ctx->dim, n_query, W, ctx->opt.B, mode, d_w, ctx->acc_vert, acc_g,
                      ctx->stream, nullptr, d_umean, d_pw, active, d_usum, N > 0 ? d_grad : nullptr, N), "scatter");
    ctx->launches += n_query > 0 ? 1 : 0;
    if (N > 0) {
        CK(launch_gemv(ctx->jac, ctx->dg_vert, ctx->acc_vert, acc_g, ctx->n_vert, ctx->dim, N, d_grad, ctx->stream), "adjoint gemv");
        ctx->launches += 1;
    }
    double* d_loss = nullptr;
    if (mode >= 1) {
        d_loss = mem == DWOS_MEM_DEVICE ? loss : ctx->out + std::max(N, 1) + n_query;
        if (mode == 1) {   // the means from the scatter's per-point sums
            CK(launch_loss(d_usum, d_w, n_query, d_loss, ctx->stream, d_pw, 1.0 / W), "loss");
            ctx->launches += 1;
        } else {
            double* d_mean = ctx->out + std::max(N, 1);
            CK(launch_reduce_u(ctx->rec, n_query, W, d_mean, nullptr, ctx->stream), "reduce u");
            CK(launch_loss(d_mean, d_w, n_query, d_loss, ctx->stream, d_pw), "loss");
            ctx->launches += n_query > 0 ? 2 : 1;
        }
    }
    if (grad_vert)
        CK(from_device(ctx, grad_vert, ctx->acc_vert, (size_t)ctx->n_vert * ctx->dim, mem), "copy vertex gradient");
    if (mem == DWOS_MEM_HOST) {
        if (N > 0) CK(from_device(ctx, grad_param, ctx->out, N, mem), "copy grad");
        if (mode >= 1) CK(from_device(ctx, loss, d_loss, 1, mem), "copy loss");
        return finish_sync(ctx);
    }
    return DWOS_OK;
}

dwos_status dwos_grad_l2_weighted(dwos_ctx* ctx, int n_query, const float* xq, const float* uref,
                                  const float* point_weight, int W, uint64_t walk_id_base, double* loss,
                                  double* grad_param, double* grad_vert, int mem) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (n_query > 0 && !point_weight) return fail(ctx, DWOS_ERR_INVALID_ARG, "point_weight is NULL");
    if (mem == DWOS_MEM_HOST && n_query > 0 && !finite_all(point_weight, n_query))
        return fail(ctx, DWOS_ERR_INVALID_ARG, "point weights must be finite");
    return reverse_common(ctx, n_query, xq, uref, W, walk_id_base, 1, loss, grad_param, grad_vert, mem,
                          point_weight);
}

dwos_status dwos_grad_l2_product(dwos_ctx* ctx, int n_query, const float* xq, const float* uref, int W,
                                 uint64_t walk_id_base, int product, double* loss, double* grad_param,
                                 double* grad_vert, int mem) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (product < 0 || product > 2) return fail(ctx, DWOS_ERR_INVALID_ARG, "product must be 0, 1 or 2");
    const int mode = product == 0 ? 1 : product + 1;
    return reverse_common(ctx, n_query, xq, uref, W, walk_id_base, mode, loss, grad_param, grad_vert, mem);
}

dwos_status dwos_vjp(dwos_ctx* ctx, int n_query, const float* xq, const float* w, int W,
                     uint64_t walk_id_base, double* grad_param, double* grad_vert, int mem) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    return reverse_common(ctx, n_query, xq, w, W, walk_id_base, 0, nullptr, grad_param, grad_vert, mem);
}

dwos_status dwos_grad_l2(dwos_ctx* ctx, int n_query, const float* xq, const float* uref, int W,
                         uint64_t walk_id_base, double* loss, double* grad_param, double* grad_vert, int mem) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    return reverse_common(ctx, n_query, xq, uref, W, walk_id_base, 1, loss, grad_param, grad_vert, mem);
}

dwos_status dwos_grad_l2_cv(dwos_ctx* ctx, int n_query, const float* xq, const float* uref, int W,
                            uint64_t walk_id_base, const float* cv_grad, int cv_whole_walk, const float* cv_elem,
                            float* samples, dwos_walk_debug* debug, double* loss, double* grad_param,
                            double* u_var) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (cv_elem && ctx->opt.dudn_estimator != 0)
        return fail(ctx, DWOS_ERR_INVALID_ARG, "the nested table corrects the backward-difference du/dn estimator");
    if (n_query < 1 || !uref || !loss) return fail(ctx, DWOS_ERR_INVALID_ARG, "bad arguments");
    if (ctx->n_param > 0 && !grad_param) return fail(ctx, DWOS_ERR_INVALID_ARG, "grad_param is NULL");
    if (W % ctx->opt.B) return fail(ctx, DWOS_ERR_INVALID_ARG, "walks_per_point must be a multiple of B");
    for (const void* p : {(const void*)xq, (const void*)uref, (const void*)cv_grad, (const void*)cv_elem,
                          (const void*)samples, (const void*)debug, (const void*)loss, (const void*)grad_param,
                          (const void*)u_var})
        if (dwos_status s = check_device_ptr(ctx, p, "argument")) return s;
    if (dwos_status s = set_device(ctx)) return s;
    const size_t total = (size_t)n_query * W;
    float4* smp = reinterpret_cast<float4*>(samples);
    float4* end = nullptr;
    const size_t need = (cv_grad && !smp ? 4 * total : 0) + (cv_grad && cv_whole_walk ? 4 * total : 0);
    if (need) CK(grow(ctx->misc_f, ctx->misc_f_cap, need), "alloc samples");
    if (!smp && cv_grad) smp = reinterpret_cast<float4*>(ctx->misc_f);
    if (cv_grad && cv_whole_walk) end = reinterpret_cast<float4*>(ctx->misc_f + (samples ? 0 : 4 * total));
    if (dwos_status s = run_walks(ctx, n_query, xq, W, walk_id_base, 1, DWOS_MEM_DEVICE, nullptr, debug, smp, end,
                                  reinterpret_cast<const float4*>(cv_elem)))
        return s;
    const CvView cv{smp, cv_grad, ctx->xq_in, ctx->dim, end};
    const CvView* cvp = cv_grad ? &cv : nullptr;
    const int N = ctx->n_param;
    CK(grow(ctx->wvec, ctx->wvec_cap, (size_t)n_query), "alloc weights");
    CK(cudaMemcpyAsync(ctx->wvec, uref, sizeof(float) * n_query, cudaMemcpyDeviceToDevice, ctx->stream), "copy uref");
    const size_t nacc = (size_t)ctx->n_vert * ctx->dim + (size_t)ctx->n_vert;
    CK(grow(ctx->acc_vert, ctx->acc_cap, nacc), "alloc accumulators");
    CK(cudaMemsetAsync(ctx->acc_vert, 0, nacc * sizeof(double), ctx->stream), "zero accumulators");
    double* acc_g = ctx->dg_vert ? ctx->acc_vert + (size_t)ctx->n_vert * ctx->dim : nullptr;
    if (dwos_status s = ensure_vert_active(ctx)) return s;
    CK(launch_scatter(ctx->rec, ctx->elem, ctx->dim, n_query, W, ctx->opt.B, 1, ctx->wvec, ctx->acc_vert, acc_g,
                      ctx->stream, cvp, nullptr, nullptr, ctx->vert_active), "scatter");
    if (N > 0) {
        CK(cudaMemsetAsync(grad_param, 0, (size_t)N * sizeof(double), ctx->stream), "zero grad");
        CK(launch_gemv(ctx->jac, ctx->dg_vert, ctx->acc_vert, acc_g, ctx->n_vert, ctx->dim, N, grad_param,
                       ctx->stream), "adjoint gemv");
    }
    CK(grow(ctx->out, ctx->out_cap, 2 * (size_t)n_query), "alloc outputs");
    double* mean = ctx->out;
    double* se = ctx->out + n_query;
    // u_var: per-point standard errors without and with the control variate
    CK(launch_reduce_u(ctx->rec, n_query, W, mean, u_var ? u_var + n_query : se, ctx->stream, cvp, 0, u_var),
       "reduce u");
    CK(launch_loss(mean, ctx->wvec, n_query, loss, ctx->stream), "loss");
    ctx->launches += 4 + (N > 0);
    if (samples) {
        CK(launch_pack_samples(ctx->rec, smp, (long long)total, ctx->stream), "pack samples");
        ctx->launches += 1;
    }
    return DWOS_OK;
}

namespace {

// Element centres of a 2D boundary (current vertices).
__global__ void cv_centres_kernel(const float* __restrict__ vert, const int* __restrict__ elem, int n_elem,
                                  float* __restrict__ centres) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n_elem) return;
    const int a = elem[2 * e], b = elem[2 * e + 1];
    centres[2 * e] = 0.5f * (vert[2 * a] + vert[2 * b]);
    centres[2 * e + 1] = 0.5f * (vert[2 * a + 1] + vert[2 * b + 1]);
}

struct FieldCoef { float c[10]; };

// (q, t) per element: q as given, t the tangential gradient of the Dirichlet
// data on the element: (g1 - g0) / |d|^2 d for mapped vertex data (d = v1 - v0),
// grad g - (grad g . n) n at the centre for field data.
__global__ void cv_table_kernel(const float* __restrict__ vert, const int* __restrict__ elem,
                                const float* __restrict__ g_vert, int data_kind, FieldCoef fc,
                                const float* __restrict__ q, int n_elem, float4* __restrict__ table) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n_elem) return;
    const int a = elem[2 * e], b = elem[2 * e + 1];
    const float dx = vert[2 * b] - vert[2 * a], dy = vert[2 * b + 1] - vert[2 * a + 1];
    const float l2 = dx * dx + dy * dy;
    float tx = 0.0f, ty = 0.0f;
    if (l2 > 0.0f) {
        if (data_kind == 1) {
            const float X = 0.5f * (vert[2 * a] + vert[2 * b]), Y = 0.5f * (vert[2 * a + 1] + vert[2 * b + 1]);
            const float gx = fc.c[1] + 2.0f * (fc.c[4] * X + fc.c[7] * Y);
            const float gy = fc.c[2] + 2.0f * (fc.c[7] * X + fc.c[5] * Y);
            const float s = (gx * dx + gy * dy) / l2;      // projection on the segment's direction
            tx = s * dx;
            ty = s * dy;
        } else {
            const float s = (g_vert[b] - g_vert[a]) / l2;
            tx = s * dx;
            ty = s * dy;
        }
    }
    table[e] = make_float4(q[e], tx, ty, 0.0f);
}

}  // namespace

namespace {
// Reads `words` float4 of an L2-resident buffer `reps` times (grid-stride,
// coalesced) and folds them into one value so the loads cannot be dropped.
__global__ void l2_read_kernel(const float4* __restrict__ buf, size_t words, int reps, float* sink) {
    float acc = 0.0f;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (int r = 0; r < reps; ++r)
        for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < words; i += stride) {
            const float4 v = __ldcg(buf + i);
            acc += v.x + v.y + v.z + v.w;
        }
    if (acc == 1.2345e-30f) *sink = acc;
}
}  // namespace

dwos_status dwos_probe_l2_read(int device, size_t bytes, int reps, double* gbs) {
    if (!gbs || bytes < 16 || reps < 1) return fail(nullptr, DWOS_ERR_INVALID_ARG, "bad arguments");
    cudaError_t e = cudaSetDevice(device);
    if (e != cudaSuccess) return fail(nullptr, DWOS_ERR_CUDA, cudaGetErrorString(e));
    int n_sm = 0;
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, device);
    const size_t words = bytes / 16;
    float4* buf = nullptr;
    float* sink = nullptr;
    cudaEvent_t a = nullptr, b = nullptr;
    float ms = 0.0f;
    e = cudaMalloc(&buf, words * 16);
    if (e == cudaSuccess) e = cudaMalloc(&sink, sizeof(float));
    if (e == cudaSuccess) e = cudaMemset(buf, 0, words * 16);
    if (e == cudaSuccess) e = cudaEventCreate(&a);
    if (e == cudaSuccess) e = cudaEventCreate(&b);
    if (e == cudaSuccess) {
        l2_read_kernel<<<n_sm * 8, 256>>>(buf, words, 1, sink);           // bring the buffer into L2
        cudaEventRecord(a);
        l2_read_kernel<<<n_sm * 8, 256>>>(buf, words, reps, sink);
        cudaEventRecord(b);
        e = cudaEventSynchronize(b);
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, a, b);
    }
    if (a) cudaEventDestroy(a);
    if (b) cudaEventDestroy(b);
    cudaFree(buf);
    cudaFree(sink);
    if (e != cudaSuccess) return fail(nullptr, DWOS_ERR_CUDA, cudaGetErrorString(e));
    *gbs = (double)words * 16.0 * reps / (ms * 1e-3) / 1e9;
    return DWOS_OK;
}

dwos_status dwos_get_vertices(const dwos_ctx* ctx, float* vert, int mem) {
    dwos_ctx* c = const_cast<dwos_ctx*>(ctx);
    if (!ctx || !vert) return fail(c, DWOS_ERR_INVALID_ARG, "NULL argument");
    if (!ctx->have_boundary) return fail(c, DWOS_ERR_STATE, "no boundary");
    if (dwos_status s = check_mem(c, mem)) return s;
    if (dwos_status s = set_device(c)) return s;
    const size_t n = (size_t)ctx->n_vert * ctx->dim;
    CKC(c, cudaMemcpyAsync(vert, ctx->vert, sizeof(float) * n,
                           mem == DWOS_MEM_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice, ctx->stream),
        "copy vertices");
    if (mem == DWOS_MEM_HOST) CKC(c, cudaStreamSynchronize(ctx->stream), "synchronize");
    return DWOS_OK;
}

dwos_status dwos_bvh_info(const dwos_ctx* ctx, int32_t* info) {
    if (!ctx || !info) return fail(nullptr, DWOS_ERR_INVALID_ARG, "NULL argument");
    if (!ctx->have_boundary) return fail(const_cast<dwos_ctx*>(ctx), DWOS_ERR_STATE, "no boundary");
    info[0] = ctx->n_elem;
    info[1] = ctx->bvh.n_tree;
    info[2] = ctx->bvh.n_big;
    info[3] = ctx->bvh.n_internal;
    info[4] = (int32_t)wide_units(ctx->dim, ctx->bvh.n_wide);
    info[5] = ctx->bvh.wide_depth;
    return DWOS_OK;
}

dwos_status dwos_cv_table(dwos_ctx* ctx, dwos_mlp* mlp, float* table) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (!mlp || !table) return fail(ctx, DWOS_ERR_INVALID_ARG, "NULL argument");
    if (!ctx->have_boundary) return fail(ctx, DWOS_ERR_STATE, "no boundary: call dwos_set_boundary first");
    if (ctx->dim != 2) return fail(ctx, DWOS_ERR_NOT_IMPLEMENTED, "the control-variate network is two-dimensional");
    if (dwos_status s = check_device_ptr(ctx, table, "table")) return s;
    if (dwos_status s = set_device(ctx)) return s;
    const int n = ctx->n_elem;
    CK(grow(ctx->misc_f, ctx->misc_f_cap, 3 * (size_t)n), "alloc");
    float* centres = ctx->misc_f;
    float* q = centres + 2 * (size_t)n;
    const int blocks = (n + 255) / 256;
    cv_centres_kernel<<<blocks, 256, 0, ctx->stream>>>(ctx->vert, ctx->elem, n, centres);
    CK(cudaGetLastError(), "centres");
    if (dwos_status s = dwos_mlp_set_stream(mlp, ctx->stream))
        return fail(ctx, s, std::string("network: ") + dwos_mlp_last_error(mlp));
    if (dwos_status s = dwos_mlp_eval(mlp, n, centres, nullptr, nullptr, q, DWOS_MEM_DEVICE))
        return fail(ctx, s, std::string("network: ") + dwos_mlp_last_error(mlp));
    FieldCoef fc;
    for (int i = 0; i < 10; ++i) fc.c[i] = (float)ctx->field[i];
    cv_table_kernel<<<blocks, 256, 0, ctx->stream>>>(ctx->vert, ctx->elem, ctx->g_vert, ctx->data_kind, fc, q, n,
                                                     reinterpret_cast<float4*>(table));
    CK(cudaGetLastError(), "table");
    ctx->launches += 3;
    return DWOS_OK;
}

dwos_status dwos_cv_training_set(dwos_ctx* ctx, long long n_walks, const float* samples, const dwos_walk_debug* debug,
                                 long long stride, long long offset, float q_weight, float* x, float* target,
                                 float* mask, long long* n_rows) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (n_walks < 0 || stride < 1 || offset < 0 || (n_walks > 0 && offset >= n_walks))
        return fail(ctx, DWOS_ERR_INVALID_ARG, "need n_walks >= 0, stride >= 1 and 0 <= offset < n_walks");
    if (!samples || !x || !target || !mask || !n_rows) return fail(ctx, DWOS_ERR_INVALID_ARG, "NULL argument");
    if (!(q_weight >= 0.0f) || !std::isfinite(q_weight)) return fail(ctx, DWOS_ERR_INVALID_ARG, "q_weight must be >= 0");
    for (const void* p : {(const void*)samples, (const void*)debug, (const void*)x, (const void*)target, (const void*)mask})
        if (dwos_status s = check_device_ptr(ctx, p, "argument")) return s;
    if (dwos_status s = set_device(ctx)) return s;
    const long long rows = n_walks > 0 ? (n_walks - offset + stride - 1) / stride : 0;
    *n_rows = rows * (debug ? 2 : 1);
    CK(grow(ctx->misc_d, ctx->misc_d_cap, 2), "alloc");
    CK(launch_cv_rows(reinterpret_cast<const float4*>(samples), debug, rows, offset, stride, ctx->opt.h, q_weight, x,
                      target, mask, ctx->misc_d, ctx->stream), "training rows");
    ctx->launches += debug ? 2 : 1;
    return DWOS_OK;
}

dwos_status dwos_walk_records(dwos_ctx* ctx, int n_query, const float* xq, int W, uint64_t walk_id_base,
                              int differential, dwos_record* records, uint32_t* trace, dwos_walk_debug* debug,
                              int mem) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (dwos_status s = check_mem(ctx, mem)) return s;
    if (!records) return fail(ctx, DWOS_ERR_INVALID_ARG, "records is NULL");
    if (mem == DWOS_MEM_DEVICE)
        for (const void* p : {(const void*)records, (const void*)trace, (const void*)debug})
            if (dwos_status s = check_device_ptr(ctx, p, "output")) return s;
    if (dwos_status s = set_device(ctx)) return s;
    const size_t total = (size_t)std::max(n_query, 0) * (size_t)std::max(W, 0);
    const int K1 = ctx->opt.K + 1;
    uint32_t* d_trace = nullptr;
    dwos_walk_debug* d_dbg = nullptr;
    if (trace) {
        if (mem == DWOS_MEM_DEVICE) d_trace = trace;
        else { CK(grow(ctx->trace, ctx->trace_cap, total * K1), "alloc trace"); d_trace = ctx->trace; }
        CK(cudaMemsetAsync(d_trace, 0xff, total * K1 * sizeof(uint32_t), ctx->stream), "init trace");
    }
    if (debug) {
        if (mem == DWOS_MEM_DEVICE) d_dbg = debug;
        else { CK(grow(ctx->dbg, ctx->dbg_cap, total), "alloc debug"); d_dbg = ctx->dbg; }
    }
    if (dwos_status s = run_walks(ctx, n_query, xq, W, walk_id_base, differential ? 1 : 0, mem, d_trace, d_dbg)) return s;
    CK(from_device(ctx, records, ctx->rec, total, mem), "copy records");
    if (trace && mem == DWOS_MEM_HOST) CK(from_device(ctx, trace, d_trace, total * K1, mem), "copy trace");
    if (debug && mem == DWOS_MEM_HOST) CK(from_device(ctx, debug, d_dbg, total, mem), "copy debug");
    if (mem == DWOS_MEM_HOST) return finish_sync(ctx);
    return DWOS_OK;
}

dwos_status dwos_last_stats(dwos_ctx* ctx, dwos_run_stats* out) {
    if (!ctx || !out) return fail(ctx, DWOS_ERR_INVALID_ARG, "NULL argument");
    if (dwos_status s = set_device(ctx)) return s;
    CK(cudaStreamSynchronize(ctx->stream), "synchronize");
    DevCounters c;
    CK(cudaMemcpy(&c, cur_ctr(ctx), sizeof(c), cudaMemcpyDeviceToHost), "read counters");
    out->steps_main = c.steps_main;
    out->steps_nested = c.steps_nested;
    out->walks = c.next_work;
    out->capped = c.capped;
    out->nodes_visited = c.nodes;
    out->prims_tested = c.prims;
    out->wide_nodes_visited = wide_units(ctx->dim, c.wnodes);
    out->launches = ctx->launches;
    out->blocks = ctx->last_blocks;
    float ms = 0.0f;
    if (ctx->timed && cudaEventElapsedTime(&ms, ctx->ev0, ctx->ev1) != cudaSuccess) { cudaGetLastError(); ms = 0.0f; }
    out->kernel_ms = ms;
    return DWOS_OK;
}

static dwos_status closest_common(dwos_ctx* ctx, int n, const float* p, const int32_t* hint, float* dist,
                                  int32_t* elem_out, float* bary, int mem) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (dwos_status s = check_mem(ctx, mem)) return s;
    if (!ctx->have_boundary) return fail(ctx, DWOS_ERR_STATE, "no boundary");
    if (n < 0 || (n > 0 && (!p || !dist || !elem_out || !bary))) return fail(ctx, DWOS_ERR_INVALID_ARG, "bad arguments");
    if (mem == DWOS_MEM_HOST && hint)
        for (int i = 0; i < n; ++i)
            if (hint[i] >= ctx->n_elem) return fail(ctx, DWOS_ERR_INVALID_ARG, "hint element out of range");
    if (dwos_status s = set_device(ctx)) return s;
    CK(grow(ctx->misc_f, ctx->misc_f_cap, (size_t)n * (ctx->dim + 3)), "alloc");
    CK(grow(ctx->misc_i, ctx->misc_i_cap, 2 * (size_t)std::max(n, 1)), "alloc");
    float* dp = ctx->misc_f;
    float* dd = dp + (size_t)n * ctx->dim;
    float* db = dd + n;
    int* dh = nullptr;
    CK(to_device(ctx, dp, p, (size_t)n * ctx->dim, mem), "copy points");
    if (hint) { dh = ctx->misc_i + std::max(n, 1); CK(to_device(ctx, dh, hint, (size_t)n, mem), "copy hints"); }
    CK(cudaMemsetAsync(ctx->d_err, 0, sizeof(int), ctx->stream), "reset");
    CK(cudaMemsetAsync(cur_ctr(ctx), 0, sizeof(DevCounters), ctx->stream), "reset counters");
    if (hint && ctx->n_neumann > 0) return fail(ctx, DWOS_ERR_NOT_IMPLEMENTED, "hinted queries with a Neumann part");
    CK(launch_closest(ctx->bvh, n, dp, dh, dd, ctx->misc_i, db, ctx->d_err, cur_ctr(ctx), effective_traversal(ctx),
                      ctx->stream), "closest point");
    ctx->launches += n > 0 ? 1 : 0;
    if (ctx->n_neumann > 0 && n > 0) {   // the Dirichlet tree numbers its own elements
        map_ids_kernel<<<(n + 255) / 256, 256, 0, ctx->stream>>>(n, ctx->dmap, ctx->misc_i);
        CK(cudaGetLastError(), "map element ids");
    }
    CK(from_device(ctx, dist, dd, n, mem), "copy");
    CK(from_device(ctx, elem_out, ctx->misc_i, n, mem), "copy");
    CK(from_device(ctx, bary, db, 2 * (size_t)n, mem), "copy");
    if (mem == DWOS_MEM_HOST) {
        CK(cudaStreamSynchronize(ctx->stream), "synchronize");
        int err = 0;
        CK(cudaMemcpy(&err, ctx->d_err, sizeof(int), cudaMemcpyDeviceToHost), "read flag");
        if (err) return fail(ctx, DWOS_ERR_STEP_LIMIT, "BVH traversal exceeded its iteration bound");
    }
    return DWOS_OK;
}

dwos_status dwos_closest_point(dwos_ctx* ctx, int n, const float* p, float* dist, int32_t* elem_out, float* bary,
                               int mem) {
    return closest_common(ctx, n, p, nullptr, dist, elem_out, bary, mem);
}

dwos_status dwos_closest_point_hint(dwos_ctx* ctx, int n, const float* p, const int32_t* hint_elem, float* dist,
                                    int32_t* elem_out, float* bary, int mem) {
    if (!hint_elem && n > 0) return fail(ctx, DWOS_ERR_INVALID_ARG, "hint_elem is NULL");
    return closest_common(ctx, n, p, hint_elem, dist, elem_out, bary, mem);
}

dwos_status dwos_inside(dwos_ctx* ctx, int n, const float* p, int32_t* inside, int mem) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (dwos_status s = check_mem(ctx, mem)) return s;
    if (!ctx->have_boundary) return fail(ctx, DWOS_ERR_STATE, "no boundary");
    if (n < 0 || (n > 0 && (!p || !inside))) return fail(ctx, DWOS_ERR_INVALID_ARG, "bad arguments");
    if (dwos_status s = set_device(ctx)) return s;
    CK(grow(ctx->misc_f, ctx->misc_f_cap, (size_t)n * ctx->dim), "alloc");
    CK(grow(ctx->misc_i, ctx->misc_i_cap, (size_t)std::max(n, 1)), "alloc");
    CK(to_device(ctx, ctx->misc_f, p, (size_t)n * ctx->dim, mem), "copy points");
    CK(inside_all(ctx, n, ctx->misc_f, ctx->misc_i), "inside test");
    CK(from_device(ctx, inside, ctx->misc_i, n, mem), "copy");
    if (mem == DWOS_MEM_HOST) CK(cudaStreamSynchronize(ctx->stream), "synchronize");
    return DWOS_OK;
}

dwos_status dwos_philox4x32_10(dwos_ctx* ctx, int n, const uint32_t* ctr, const uint32_t* key, uint32_t* out,
                               int mem) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (dwos_status s = check_mem(ctx, mem)) return s;
    if (n < 0 || (n > 0 && (!ctr || !key || !out))) return fail(ctx, DWOS_ERR_INVALID_ARG, "bad arguments");
    if (dwos_status s = set_device(ctx)) return s;
    uint32_t k[2];
    if (mem == DWOS_MEM_DEVICE) CK(cudaMemcpy(k, key, sizeof(k), cudaMemcpyDeviceToHost), "copy key");
    else { k[0] = key[0]; k[1] = key[1]; }
    CK(grow(ctx->misc_u, ctx->misc_u_cap, 8 * (size_t)std::max(n, 1)), "alloc");
    uint32_t* dc = ctx->misc_u;
    uint32_t* dout = dc + 4 * (size_t)n;
    CK(to_device(ctx, dc, ctr, 4 * (size_t)n, mem), "copy counters");
    CK(launch_philox(n, dc, k[0], k[1], dout, ctx->stream), "philox");
    CK(from_device(ctx, out, dout, 4 * (size_t)n, mem), "copy");
    if (mem == DWOS_MEM_HOST) CK(cudaStreamSynchronize(ctx->stream), "synchronize");
    return DWOS_OK;
}

dwos_status dwos_ball_weights(dwos_ctx* ctx, int dim, float sigma, int n, const float* d, const float* u,
                              float* source, float* alpha, int mem) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (dwos_status s = check_mem(ctx, mem)) return s;
    if (dim != 2 && dim != 3) return fail(ctx, DWOS_ERR_INVALID_ARG, "dim must be 2 or 3");
    if (!(sigma >= 0.0f) || !std::isfinite(sigma)) return fail(ctx, DWOS_ERR_INVALID_ARG, "sigma must be finite and >= 0");
    if (n < 0 || (n > 0 && (!d || !u || (!source && !alpha)))) return fail(ctx, DWOS_ERR_INVALID_ARG, "bad arguments");
    if (dwos_status s = set_device(ctx)) return s;
    if (n == 0) return DWOS_OK;
    CK(grow(ctx->misc_f, ctx->misc_f_cap, 4 * (size_t)n), "alloc");
    float* dd = ctx->misc_f;
    float* du = dd + n;
    float* ds = du + n;
    float* da = ds + n;
    CK(to_device(ctx, dd, d, (size_t)n, mem), "copy d");
    CK(to_device(ctx, du, u, (size_t)n, mem), "copy u");
    CK(launch_ball_weights(dim, std::sqrt(sigma), n, dd, du, source ? ds : nullptr, alpha ? da : nullptr,
                           ctx->stream), "ball weights");
    ctx->launches += 1;
    if (source) CK(from_device(ctx, source, ds, (size_t)n, mem), "copy source weights");
    if (alpha) CK(from_device(ctx, alpha, da, (size_t)n, mem), "copy recursive weights");
    if (mem == DWOS_MEM_HOST) CK(cudaStreamSynchronize(ctx->stream), "synchronize");
    return DWOS_OK;
}

static dwos_status bessel_k(dwos_ctx* ctx, int order, int n, const float* x, float* out, int mem) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (dwos_status s = check_mem(ctx, mem)) return s;
    if (n < 0 || (n > 0 && (!x || !out))) return fail(ctx, DWOS_ERR_INVALID_ARG, "bad arguments");
    if (dwos_status s = set_device(ctx)) return s;
    if (n == 0) return DWOS_OK;
    CK(grow(ctx->misc_f, ctx->misc_f_cap, 2 * (size_t)n), "alloc");
    CK(to_device(ctx, ctx->misc_f, x, (size_t)n, mem), "copy x");
    CK(launch_bessel_k(order, n, ctx->misc_f, ctx->misc_f + n, ctx->stream), "K");
    ctx->launches += 1;
    CK(from_device(ctx, out, ctx->misc_f + n, (size_t)n, mem), "copy K");
    if (mem == DWOS_MEM_HOST) CK(cudaStreamSynchronize(ctx->stream), "synchronize");
    return DWOS_OK;
}

dwos_status dwos_bessel_k0(dwos_ctx* ctx, int n, const float* x, float* out, int mem) {
    return bessel_k(ctx, 0, n, x, out, mem);
}

dwos_status dwos_bessel_k1(dwos_ctx* ctx, int n, const float* x, float* out, int mem) {
    return bessel_k(ctx, 1, n, x, out, mem);
}

dwos_status dwos_star_weight(dwos_ctx* ctx, int dim, float sigma, int n, const float* t, const float* R, float* out,
                             int mem) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (dwos_status s = check_mem(ctx, mem)) return s;
    if (dim != 2 && dim != 3) return fail(ctx, DWOS_ERR_INVALID_ARG, "dim must be 2 or 3");
    if (!(sigma >= 0.0f) || !std::isfinite(sigma)) return fail(ctx, DWOS_ERR_INVALID_ARG, "sigma must be finite and >= 0");
    if (n < 0 || (n > 0 && (!t || !R || !out))) return fail(ctx, DWOS_ERR_INVALID_ARG, "bad arguments");
    if (dwos_status s = set_device(ctx)) return s;
    if (n == 0) return DWOS_OK;
    CK(grow(ctx->misc_f, ctx->misc_f_cap, 3 * (size_t)n), "alloc");
    CK(to_device(ctx, ctx->misc_f, t, (size_t)n, mem), "copy t");
    CK(to_device(ctx, ctx->misc_f + n, R, (size_t)n, mem), "copy R");
    CK(launch_star_weight(dim, std::sqrt(sigma), n, ctx->misc_f, ctx->misc_f + n, ctx->misc_f + 2 * (size_t)n,
                          ctx->stream), "star weight");
    ctx->launches += 1;
    CK(from_device(ctx, out, ctx->misc_f + 2 * (size_t)n, (size_t)n, mem), "copy weights");
    if (mem == DWOS_MEM_HOST) CK(cudaStreamSynchronize(ctx->stream), "synchronize");
    return DWOS_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Allocation-free evaluation.
//
// Some callers cannot allocate device memory while they call us: hosts whose
// memory is owned by another allocator (a framework's caching pool, a fixed
// device budget set aside at start-up), or latency-sensitive loops where the
// implicit device synchronisation of cudaMalloc / cudaFree is unacceptable.  dwos_eval_static
// serves them: it runs the same walk, inside-test and reduction kernels as
// dwos_eval, but every byte of scratch (problem descriptor, counters, inside
// flags, per-walk records) lives in the fixed array below, so the call itself
// allocates nothing.  The context's boundary and BVH must already be set up.
// ---------------------------------------------------------------------------
namespace {

constexpr size_t kStaticHeader = 4096;     // problem descriptor (offset 0) + counters (offset 2048)
constexpr size_t kStaticCounters = 2048;
// One inside flag per query point; n_query reaches DWOS_STATIC_MAX_WALKS when
// walks_per_point = 1, so the region is sized for that worst case.
constexpr size_t kStaticFlags = (size_t)DWOS_STATIC_MAX_WALKS * sizeof(int);
constexpr size_t kStaticBytes = kStaticHeader + kStaticFlags + (size_t)DWOS_STATIC_MAX_WALKS * sizeof(dwos_record);
static_assert(sizeof(DevProblem) <= kStaticCounters, "the problem descriptor must end before the counters");
static_assert(kStaticCounters + sizeof(DevCounters) <= kStaticHeader, "the counters must fit in the header");

// Held by every GPU that loads the library, until the process exits.
static __device__ __align__(256) unsigned char g_static_scratch[kStaticBytes];

std::mutex g_static_mutex;
void* g_static_addr[64] = {nullptr};

// Device address of the scratch array on ctx's device (looked up once per
// device, with that device current; the host-side symbol is not an address).
// The address belongs to the device's primary context: a cudaDeviceReset in
// the caller's process ends that context, and the cached address with it.
dwos_status static_scratch(dwos_ctx* ctx, unsigned char** out) {
    if (ctx->device < 0 || ctx->device >= 64) return fail(ctx, DWOS_ERR_INVALID_ARG, "device index too large");
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_addr[ctx->device]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
        if (e != cudaSuccess || !p) return cuda_fail(ctx, e != cudaSuccess ? e : cudaErrorInvalidSymbol,
                                                     "cudaGetSymbolAddress(static scratch)");
        g_static_addr[ctx->device] = p;
    }
    *out = static_cast<unsigned char*>(g_static_addr[ctx->device]);
    return DWOS_OK;
}

// Stores the walk launch's problem descriptor into the scratch array: the
// descriptor travels as a kernel argument (copied at launch), so nothing is read
// from the host stack after the call returns.
__global__ void store_problem_kernel(DevProblem P, DevProblem* dst) {
    if (threadIdx.x == 0 && blockIdx.x == 0) *dst = P;
}

}  // namespace

extern "C" dwos_status dwos_eval_static(dwos_ctx* ctx, int n_query, const float* xq, int W, double* u_mean,
                                        double* u_se, double* du_mean, double* du_se) {
    if (!ctx) return fail(nullptr, DWOS_ERR_INVALID_ARG, "ctx is NULL");
    if (!ctx->have_boundary) return fail(ctx, DWOS_ERR_STATE, "no boundary: call dwos_set_boundary first");
    if (n_query < 0 || W < 1) return fail(ctx, DWOS_ERR_INVALID_ARG, "n_query must be >= 0 and walks_per_point >= 1");
    const unsigned long long total = (unsigned long long)n_query * (unsigned long long)W;
    if (total > (unsigned long long)DWOS_STATIC_MAX_WALKS)
        return fail(ctx, DWOS_ERR_INVALID_ARG,
                    "n_query * walks_per_point exceeds DWOS_STATIC_MAX_WALKS (262144) for dwos_eval_static");
    if (n_query == 0) return DWOS_OK;
    if (!xq || !u_mean) return fail(ctx, DWOS_ERR_INVALID_ARG, "xq and u_mean must be device pointers");
    if (du_mean && ctx->n_param == 0) return fail(ctx, DWOS_ERR_INVALID_ARG, "derivatives requested but n_param = 0");
    if (ctx->n_neumann > 0) return fail(ctx, DWOS_ERR_NOT_IMPLEMENTED, "dwos_eval_static with a Neumann part");
    for (const void* p : {(const void*)xq, (const void*)u_mean, (const void*)u_se, (const void*)du_mean,
                          (const void*)du_se})
        if (dwos_status s = check_device_ptr(ctx, p, "argument")) return s;
    if (dwos_status s = set_device(ctx)) return s;
    unsigned char* base = nullptr;
    if (dwos_status s = static_scratch(ctx, &base)) return s;
    DevProblem* d_prob = reinterpret_cast<DevProblem*>(base);
    DevCounters* d_ctr = reinterpret_cast<DevCounters*>(base + kStaticCounters);
    int* d_valid = reinterpret_cast<int*>(base + kStaticHeader);
    dwos_record* d_rec = reinterpret_cast<dwos_record*>(base + kStaticHeader + kStaticFlags);
    const int diff = du_mean ? 1 : 0;
    const int* valid = nullptr;
    if (ctx->opt.check_inside) {
        CK(launch_inside(ctx->bvh, n_query, xq, d_valid, ctx->stream), "inside test");
        valid = d_valid;
    }
    DevProblem P;
    std::memset(&P, 0, sizeof(P));
    P.nodes = ctx->bvh.nodes;
    P.prims = ctx->bvh.prims;
    P.prim_elem = ctx->bvh.prim_elem;
    P.elem = ctx->elem;
    P.g_vert = ctx->g_vert;
    P.root = 0;
    P.n_internal = ctx->bvh.n_internal;
    P.n_tree = ctx->bvh.n_tree;
    P.n_big = ctx->bvh.n_big;
    P.leaf_parent = ctx->bvh.leaf_parent;
    P.node_cell = ctx->bvh.node_cell;
    P.r_max = ctx->bvh.r_max;
    P.traversal = effective_traversal(ctx);
    P.wnodes = ctx->bvh.wnodes;
    P.n_wide = ctx->bvh.n_wide;
    P.data_kind = ctx->data_kind;
    P.differential = diff;
    for (int i = 0; i < 10; ++i) P.field[i] = (float)ctx->field[i];
    P.sqrt_sigma = std::sqrt(ctx->sigma);
    P.f = ctx->f;
    P.eps = ctx->opt.eps;
    P.h = ctx->opt.h;
    P.inv_h = 1.0f / ctx->opt.h;
    P.K = ctx->opt.K;
    P.max_steps = ctx->opt.max_steps;
    P.dudn_mode = ctx->opt.dudn_estimator;
    P.seed_lo = (uint32_t)ctx->opt.seed;
    P.seed_hi = (uint32_t)(ctx->opt.seed >> 32);
    P.xq = xq;
    P.valid = valid;
    P.walks = W;
    P.node_budget = ctx->node_budget;
    P.walk_id_base = 0;
    P.work_begin = 0;
    P.work_end = total;
    P.rec = d_rec;
    store_problem_kernel<<<1, 32, 0, ctx->stream>>>(P, d_prob);
    CK(cudaGetLastError(), "store problem");
    // the array keeps the previous call's contents: the work counter and statistics start at zero
    CK(cudaMemsetAsync(d_ctr, 0, sizeof(DevCounters), ctx->stream), "reset counters");
    WalkLaunch L;
    L.dim = ctx->dim;
    L.block_size = ctx->opt.block_size > 0 ? ctx->opt.block_size : 256;
    L.blocks_per_sm = ctx->opt.blocks_per_sm;
    L.n_sm = ctx->n_sm;
    L.traversal = P.traversal;
    L.wide_depth = ctx->bvh.wide_depth;
    int blocks = 0;
    CK(launch_walks(L, d_prob, 1, total, d_ctr, ctx->stream, &blocks), "walk kernel");
    if (!diff)
        CK(launch_reduce_u(d_rec, n_query, W, u_mean, u_se, ctx->stream), "reduce u");
    else
        CK(launch_reduce_udot(d_rec, ctx->elem, ctx->jac, ctx->dg_vert, ctx->dim, ctx->n_param, n_query, W, u_mean,
                              u_se, du_mean, du_se, ctx->n_sm, ctx->stream), "reduce udot");
    return DWOS_OK;
}
