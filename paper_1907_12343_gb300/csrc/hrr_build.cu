// Light hierarchy builder: Morton keys, stable radix sort, binary radix tree, refit.
//
// Sec. 1 of the paper asks for light vertices sorted by a hierarchy in which every node
// is a contiguous range [a_n, b_n) of leaf indices, and notes that a spatial sort lets the
// sequence index inherit the radical inverse's stratification. This file builds such a
// hierarchy on the device:
//   1. morton_kernel     63-bit Morton keys (21 bits per axis) and finiteness checks;
//   2. sort passes       stable radix sort of (key, original index), 8 bits each (hrr_sort.cuh);
//   3. gather_sorted     short runs put in order; sorted (x, y, z, intensity) as float4;
//   4. topology_kernel   binary radix tree over (key, sorted position) in parallel: every
//                        internal node finds its range and split from its neighbours'
//                        common-prefix lengths (Karras, HPG 2012);
//   5. the box pass      boxes, maximum intensities and the records (hrr_boxes.cuh).
#include <algorithm>

#include "hrr_boxes.cuh"
#include "hrr_internal.cuh"
#include "hrr_order.cuh"
#include "hrr_sort.cuh"
#include "hrr_split.cuh"

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ void store_slot(hrr_node *node, uint32_t slot, const float lo[3],
                                           const float hi[3], float imax) {
    float *f = reinterpret_cast<float *>(node) + (slot ? 8 : 0);
    f[0] = lo[0]; f[1] = lo[1]; f[2] = lo[2]; f[3] = imax;
    f[4] = hi[0]; f[5] = hi[1]; f[6] = hi[2];
}

// Refit for moved lights: the leaves keep their order, so thread i gathers the new light i of that
// order (flagging non-finite values) and sets the parent links of node i's children from its
// record; then the box pass runs again, and skips its work when the gather raised a flag, so the
// hierarchy is left as it was. The links need no clearing first: each is set by its one parent
// (and where a corrupt record left one unset, the box pass checks it like any other). In two
// kernels this took 16 us more for 2^20 lights.
__global__ void __launch_bounds__(kThreads) refit_gather_kernel(const float *__restrict__ x, const float *__restrict__ y,
                                                                const float *__restrict__ z,
                                                                const float *__restrict__ inten,
                                                                const uint32_t *__restrict__ perm,
                                                                const hrr_node *__restrict__ nodes, uint32_t n,
                                                                float4 *__restrict__ spos, BoxScratch s,
                                                                unsigned long long *flags) {
    chain_begin();
    const uint32_t i = blockIdx.x * kThreads + threadIdx.x;
    if (i >= n) return;
    const uint32_t v = perm[i];
    uint32_t split = 0, other = 0;
    if (i < n - 1) {
        split = nodes[i].split;
        other = nodes[i].other_end;
    }
    const float4 p = make_float4(x[v], y[v], z[v], inten[v]);
    if (!isfinite(p.x) || !isfinite(p.y) || !isfinite(p.z) || !isfinite(p.w)) atomicOr(flags, HRR_FLAG_NONFINITE);
    spos[i] = p;
    box_reset_counts(s, i, n);
    if (i < n - 1) {
        const uint32_t first = min(i, other), last = max(i, other);
        if (last >= n || split < first || split >= last) {
            atomicOr(flags, HRR_FLAG_TOPOLOGY);
            return;
        }
        const uint32_t code = i << 1;
        if (first == split) s.leaf_parent[split] = code; else s.int_parent[split] = code;
        if (last == split + 1) s.leaf_parent[split + 1] = code | 1u; else s.int_parent[split + 1] = code | 1u;
    }
}

// The hierarchy of one light: its record, its permutation and (unless `der` is empty) the records
// derived from it: the leaf in slot 0 of the width-four record and in both places of the paired
// one, the rest and the top slots empty.
__global__ void single_leaf_kernel(const float *x, const float *y, const float *z,
                                   const float *inten, hrr_node *node, uint32_t *perm, Derived der,
                                   unsigned long long *flags) {
    const float px = x[0], py = y[0], pz = z[0], w = inten[0];
    if (!isfinite(px) || !isfinite(py) || !isfinite(pz) || !isfinite(w)) {
        atomicOr(flags, HRR_FLAG_NONFINITE);
        return;  // a build fails; a refit leaves the record as it was
    }
    const float lo[3] = {px, py, pz};
    store_slot(node, 0, lo, lo, w);
    store_slot(node, 1, lo, lo, w);
    node->split = 0;
    node->other_end = 0;
    perm[0] = 0;
    if (!der.wide) return;
    const float4 *r = reinterpret_cast<const float4 *>(node);
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    if (der.pairs) store_pairs(der.pairs, r[0], r[1], r[0], r[1], 0u, 0u);
    for (int k = 0; k < 8; ++k) der.wide[k] = k < 2 ? r[k] : zero;
    for (uint32_t k = 0; k < 3 * HRR_TOP_SLOTS; ++k) reinterpret_cast<float4 *>(node)[4 + k] = zero;
}

}  // namespace

namespace {

// Sorts by the key bits from `shift` up (kTopShift, or 0 for all); with the paired records or without.
int build_attempt(hrr_ctx *ctx, const hrr_lights &L, uint32_t n, hrr_tree **out, int topology, uint32_t cost_depth,
                  int shift, bool paired) {
    cudaStream_t st = ctx->stream;
    hrr_tree *tree = new (std::nothrow) hrr_tree();
    if (!tree) return hrr_fail(ctx, HRR_ERR_OOM, "host allocation of the tree");
    tree->device = ctx->device;
    tree->n = n;
    auto fail = [&](int status) {
        if (tree->nodes) cudaFreeAsync(tree->nodes, st);
        if (tree->perm) cudaFreeAsync(tree->perm, st);
        if (tree->pairs) cudaFreeAsync(tree->pairs, st);
        if (tree->wide) cudaFreeAsync(tree->wide, st);
        delete tree;
        return status;
    };
    const uint32_t n_rec = n > 1 ? n - 1 : 1;
    cudaError_t e = hrr_alloc(ctx, &tree->nodes, sizeof(hrr_node) * (size_t)n_rec + HRR_TOP_BYTES);
    if (e == cudaSuccess) e = hrr_alloc(ctx, &tree->perm, sizeof(uint32_t) * (size_t)n);
    if (e == cudaSuccess && paired) e = hrr_alloc(ctx, &tree->pairs, 8 * sizeof(float4) * (size_t)n_rec);
    if (e == cudaSuccess) e = hrr_alloc(ctx, &tree->wide, 8 * sizeof(float4) * (size_t)n_rec);
    if (e != cudaSuccess) return fail(hrr_cuda_fail(ctx, e, "tree allocation"));
    unsigned long long *flags = ctx->counters + 2;
    if ((e = cudaMemsetAsync(flags, 0, sizeof(unsigned long long), st)) != cudaSuccess)
        return fail(hrr_cuda_fail(ctx, e, "flag reset"));

    if (n == 1) {
        single_leaf_kernel<<<1, 1, 0, st>>>(L.x, L.y, L.z, L.intensity, tree->nodes, tree->perm,
                                              Derived{tree->pairs, tree->wide}, flags);
        ++ctx->launches;
        if ((e = cudaGetLastError()) != cudaSuccess) return fail(hrr_cuda_fail(ctx, e, "single_leaf_kernel"));
        tree->height = 0;
    } else {
        const size_t bytes = 2 * pad256(sizeof(uint64_t) * (size_t)n) + pad256(sizeof(uint32_t) * (size_t)n) +
                             pad256(sort_scratch_bytes(n)) + pad256(sizeof(float4) * (size_t)n) + box_scratch_bytes(n, false);
        char *scratch = nullptr;
        if ((e = hrr_alloc(ctx, &scratch, bytes)) != cudaSuccess) return fail(hrr_cuda_fail(ctx, e, "build scratch"));
        char *p = scratch;
        uint64_t *keys0 = carve<uint64_t>(p, n), *keys1 = carve<uint64_t>(p, n);
        uint32_t *vals0 = carve<uint32_t>(p, n);
        const SortScratch ss = carve_sort(p, n);
        float4 *spos = carve<float4>(p, n);
        BoxScratch rs = carve_boxes(p, n, false);
        rs.child_height = reinterpret_cast<uint32_t *>(keys0);  // the gather is the last to read those keys

        const unsigned g = (n + kThreads - 1) / kThreads;
        int rc = HRR_OK;
        do {
            if ((e = cudaMemsetAsync(ss.hist, 0, sort_scratch_bytes(n), st)) != cudaSuccess) { rc = hrr_cuda_fail(ctx, e, "memset"); break; }
            const int passes = sort_passes(shift);
            morton_kernel<<<morton_grid(n), kThreads, 0, st>>>(L.x, L.y, L.z, L.intensity, n, keys0, shift, passes, ss.hist, flags);
            sort_enqueue(keys0, vals0, keys1, tree->perm, n, shift, ss, flags, st);
            launch_chained(shift ? gather_sorted_kernel<true> : gather_sorted_kernel<false>, g, kThreads, st,
                L.x, L.y, L.z, L.intensity, keys0, vals0, n, keys1, tree->perm, spos, rs, flags);
            ctx->launches += 2 + passes;
            const unsigned gi = (n - 1 + kThreads - 1) / kThreads;
            const bool groups = topology == HRR_TOPOLOGY_COST && n > kSubMax;  // what the cost splits need before the boxes
            if (groups) {
                groups_enqueue(PointLeaves{spos}, n, rs, st);
                ++ctx->launches;
            }
            if (topology == HRR_TOPOLOGY_COST) {
                if ((rc = cost_topology(ctx, spos, keys1, n, cost_depth, tree->nodes, rs, flags, st)) != HRR_OK) break;
            } else {
                launch_chained(topology_kernel, gi, kThreads, st, keys1, n, tree->nodes, rs.leaf_parent, rs.int_parent, flags);
                ++ctx->launches;
            }
            boxes_enqueue(PointLeaves{spos}, n, tree->nodes, {tree->pairs, tree->wide}, rs, flags, st, groups);
            ctx->launches += 2;
            if ((e = cudaGetLastError()) != cudaSuccess) { rc = hrr_cuda_fail(ctx, e, "build kernels"); break; }
            if ((e = cudaMemcpyAsync(&ctx->host_counters[4], rs.root_height, sizeof(uint32_t),
                                     cudaMemcpyDeviceToHost, st)) != cudaSuccess) { rc = hrr_cuda_fail(ctx, e, "height copy"); break; }
        } while (0);
        cudaFreeAsync(scratch, st);
        if (rc != HRR_OK) return fail(rc);
    }
    if ((e = cudaMemcpyAsync(&ctx->host_counters[2], flags, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st)) != cudaSuccess)
        return fail(hrr_cuda_fail(ctx, e, "flag copy"));
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return fail(hrr_cuda_fail(ctx, e, "build"));
    if (n > 1) tree->height = (uint32_t)(ctx->host_counters[4] & 0xFFFFFFFFull);
    if (ctx->host_counters[2] & HRR_FLAG_NONFINITE)
        return fail(hrr_fail(ctx, HRR_ERR_INVALID_ARG, "a light position or intensity is not finite"));
    if ((ctx->host_counters[2] & HRR_FLAG_RUNS) && shift) {  // many lights in few cells: every key bit sorted
        fail(HRR_OK);
        return build_attempt(ctx, L, n, out, topology, cost_depth, 0, paired);
    }
    if (ctx->host_counters[2] & HRR_FLAG_WAIT) return fail(hrr_fail(ctx, HRR_ERR_TIMEOUT, "a wait of the sort ran out"));
    if (ctx->host_counters[2] & HRR_FLAG_TOPOLOGY)
        return fail(hrr_fail(ctx, HRR_ERR_DEVICE, "inconsistent radix-tree links"));
    *out = tree;
    return HRR_OK;
}

}  // namespace

int hrr_build_impl(hrr_ctx *ctx, const hrr_lights &L, uint32_t n, hrr_tree **out, int topology, uint32_t cost_depth) {
    int rc = build_attempt(ctx, L, n, out, topology, cost_depth, kTopShift, true);
    if (rc == HRR_ERR_OOM)  // the paired records are what a hierarchy can do without
        rc = build_attempt(ctx, L, n, out, topology, cost_depth, kTopShift, false);
    return rc;
}

// ------------------------------------------------------------------------------------
// Refit for moved lights
// ------------------------------------------------------------------------------------

size_t hrr_refit_scratch_bytes(uint32_t n) { return pad256(sizeof(float4) * (size_t)n) + box_scratch_bytes(n); }

cudaError_t hrr_refit_enqueue(hrr_tree *tree, const hrr_lights &L, void *scratch_mem, unsigned long long *flags,
                              cudaStream_t st) {
    const uint32_t n = tree->n;
    // one leaf: rewrite the single record unless the light is not finite (checked there)
    if (n == 1) {
        single_leaf_kernel<<<1, 1, 0, st>>>(L.x, L.y, L.z, L.intensity, tree->nodes, tree->perm,
                                              Derived{tree->pairs, tree->wide}, flags);
        return cudaGetLastError();
    }
    char *p = static_cast<char *>(scratch_mem);
    float4 *spos = carve<float4>(p, n);
    const BoxScratch rs = carve_boxes(p, n);
    refit_gather_kernel<<<(n + kThreads - 1) / kThreads, kThreads, 0, st>>>(L.x, L.y, L.z, L.intensity, tree->perm,
                                                                           tree->nodes, n, spos, rs, flags);
    return boxes_enqueue(PointLeaves{spos}, n, tree->nodes, {tree->pairs, tree->wide}, rs, flags, st);
}

// ------------------------------------------------------------------------------------
// Build without allocation
// ------------------------------------------------------------------------------------
//
// hrr_build_light_tree_static runs the same kernels as hrr_build_light_tree, but takes
// its working memory from one file-scope device array instead of allocating, and writes
// the hierarchy into arrays the caller provides. Host code must not hand the array's name
// to a kernel (in host code it names a host-side stand-in); its device address is looked
// up once per device with cudaGetSymbolAddress and cached.

#include <cstdio>
#include <mutex>

namespace {

constexpr uint32_t kStaticMaxLights = HRR_STATIC_BUILD_MAX_LIGHTS;

constexpr size_t static_scratch_bytes(size_t n) {
    return 2 * pad256(sizeof(uint64_t) * n)                               // keys, ping-pong
           + pad256(sizeof(uint32_t) * n)                                 // second value buffer
           + pad256(sort_scratch_bytes(n))                                // digit counts, tile states
           + pad256(sizeof(float4) * n)                                   // sorted lights
           + box_scratch_bytes((uint32_t)n)                               // box pass
           + pad256(sizeof(unsigned long long));                          // error flags
}

// The shared working memory of every hrr_build_light_tree_static call on a device
// (about 3.7 MiB for 65536 lights), held by each device that loads the library.
static __device__ __align__(256) unsigned char g_static_build_scratch[static_scratch_bytes(kStaticMaxLights)];

std::mutex g_static_mutex;
void *g_static_scratch_ptr[128] = {};

void set_err(char *err, size_t len, const char *msg) {
    if (err && len) snprintf(err, len, "%s", msg);
}

}  // namespace

extern "C" int hrr_build_light_tree_static(hrr_lights L, uint32_t n, hrr_node *dev_nodes,
                                           uint32_t *dev_perm, uint32_t *out_height,
                                           void *cuda_stream, char *err, size_t err_len) {
    set_err(err, err_len, "");
    if (n == 0 || n > kStaticMaxLights) {
        char msg[160];
        snprintf(msg, sizeof msg, "n_lights = %u is outside [1, %u], the most this call's fixed "
                 "working memory holds; use hrr_build_light_tree for larger light sets", n, kStaticMaxLights);
        set_err(err, err_len, msg);
        return HRR_ERR_INVALID_ARG;
    }
    if (!L.x || !L.y || !L.z || !L.intensity || !dev_nodes || !dev_perm) {
        set_err(err, err_len, "a light, node or permutation array is NULL");
        return HRR_ERR_INVALID_ARG;
    }
    cudaStream_t st = (cudaStream_t)cuda_stream;
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= 128) {
        set_err(err, err_len, "no usable current CUDA device");
        return HRR_ERR_CUDA;
    }
    char *scratch = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_static_mutex);
        if (!g_static_scratch_ptr[dev]) {
            void *p = nullptr;
            e = cudaGetSymbolAddress(&p, g_static_build_scratch);
            if (e != cudaSuccess || !p) {
                set_err(err, err_len, "cudaGetSymbolAddress of the build working memory failed");
                return HRR_ERR_CUDA;
            }
            g_static_scratch_ptr[dev] = p;
        }
        scratch = static_cast<char *>(g_static_scratch_ptr[dev]);
    }
    char *p = scratch;
    uint64_t *keys0 = carve<uint64_t>(p, kStaticMaxLights), *keys1 = carve<uint64_t>(p, kStaticMaxLights);
    uint32_t *vals0 = carve<uint32_t>(p, kStaticMaxLights);
    const SortScratch ss = carve_sort(p, kStaticMaxLights);
    float4 *spos = carve<float4>(p, kStaticMaxLights);
    const BoxScratch rs = carve_boxes(p, kStaticMaxLights);
    unsigned long long *flags = carve<unsigned long long>(p, 1);

    // Every call reuses the array: clear what the kernels expect to start cleared.
    e = cudaMemsetAsync(flags, 0, sizeof(unsigned long long), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(rs.root_height, 0, sizeof(uint32_t), st);
    if (n == 1) {
        if (e == cudaSuccess) {
            single_leaf_kernel<<<1, 1, 0, st>>>(L.x, L.y, L.z, L.intensity, dev_nodes, dev_perm, Derived{nullptr, nullptr}, flags);
            e = cudaGetLastError();
        }
    } else {
        if (e == cudaSuccess) e = cudaMemsetAsync(ss.hist, 0, sort_scratch_bytes(n), st);
        if (e == cudaSuccess) {
            const unsigned g = (n + kThreads - 1) / kThreads;
            morton_kernel<<<morton_grid(n), kThreads, 0, st>>>(L.x, L.y, L.z, L.intensity, n, keys0, 0, kSortPasses, ss.hist, flags);
            sort_enqueue(keys0, vals0, keys1, dev_perm, n, 0, ss, flags, st);
            launch_chained(gather_sorted_kernel<false>, g, kThreads, st, L.x, L.y, L.z, L.intensity, keys0, vals0, n, keys1, dev_perm,
                                                                spos, rs, flags);
            const unsigned gi = (n - 1 + kThreads - 1) / kThreads;
            launch_chained(topology_kernel, gi, kThreads, st, keys1, n, dev_nodes, rs.leaf_parent, rs.int_parent, flags);
            boxes_enqueue(PointLeaves{spos}, n, dev_nodes, {nullptr, nullptr}, rs, flags, st);
            e = cudaGetLastError();
        }
    }
    uint32_t height = 0;
    unsigned long long host_flags = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&height, rs.root_height, sizeof height, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&host_flags, flags, sizeof host_flags, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        char msg[200];
        snprintf(msg, sizeof msg, "CUDA error in the build: %s", cudaGetErrorString(e));
        set_err(err, err_len, msg);
        return HRR_ERR_CUDA;
    }
    if (host_flags & HRR_FLAG_NONFINITE) {
        set_err(err, err_len, "a light position or intensity is not finite");
        return HRR_ERR_INVALID_ARG;
    }
    if (host_flags & HRR_FLAG_WAIT) {
        set_err(err, err_len, "a wait of the sort ran out");
        return HRR_ERR_TIMEOUT;
    }
    if (host_flags & HRR_FLAG_TOPOLOGY) {
        set_err(err, err_len, "inconsistent radix-tree links");
        return HRR_ERR_DEVICE;
    }
    if (out_height) *out_height = height;
    return HRR_OK;
}
