// build_tree: Morton-ordered octree with node mass, centre of mass and size
// (the gravity tree of Section 2.2.1, octree form).
//
// Rounding is fixed so that the result is the same bit for bit on any
// device: products and sums that feed the centre of mass and the node size
// use explicit round-to-nearest intrinsics (no fused multiply-add), leaves
// sum their particles in Morton order and internal nodes sum their children
// in octant order.
#include <algorithm>
#include <climits>

#include "common.cuh"
#include "tree_util.cuh"

namespace {

__global__ void k_morton(int64_t n, const double *__restrict__ x, const double *__restrict__ y,
                         const double *__restrict__ z, double xlo, double xhi, double ylo, double yhi, double zlo,
                         double zhi, uint64_t *__restrict__ key, int32_t *__restrict__ idx)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    key[i] = em::morton_key(x[i], y[i], z[i], xlo, xhi, ylo, yhi, zlo, zhi);
    idx[i] = (int32_t)i;
}

__global__ void k_gather4(int64_t n, const int32_t *__restrict__ perm, const double *__restrict__ x,
                          const double *__restrict__ y, const double *__restrict__ z, const double *__restrict__ m,
                          double *__restrict__ xs, double *__restrict__ ys, double *__restrict__ zs,
                          double *__restrict__ ms)
{
    int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= n) return;
    int32_t i = perm[k];
    xs[k] = x[i];
    ys[k] = y[i];
    zs[k] = z[i];
    if (m) ms[k] = m[i];
}

// The topology in one pass over the sorted keys instead of level by level.
// With cpl(a, b) the number of leading octal digits two keys share, position k
// starts a node of level L iff the keys k - 1 and k differ in their first L
// digits, L > d(k) = cpl(key[k-1], key[k]), and the level L - 1 node around k
// holds more than leaf_max particles: L - 1 <= m(k), the largest cpl(key[i],
// key[i + leaf_max]) of the leaf_max + 1 windows that cover k.  So each
// position emits the nodes of levels (d(k), min(m(k) + 1, 21)], in order of k,
// and a stable sort by level puts all nodes breadth first, each level in
// Morton order.  Level by level the build took three launches, a scan and a
// host read per level (13 levels at 1e6 particles): 1.98 ms for the whole tree,
// 0.54 ms for 2,000 particles; so 0.97 and 0.21.
__device__ __forceinline__ int common_digits(uint64_t a, uint64_t b)
{
    return a == b ? em::kMortonBits : (__clzll((long long)(a ^ b)) - 1) / 3;   // keys have 63 bits
}

constexpr int TREE_LEVELS = em::kMortonBits + 1;

// Per position: the first and last level of the nodes it starts (lev), their
// number (cnt), and the nodes per level (hist).
__global__ void k_node_levels(int64_t n, int leaf_max, const uint64_t *__restrict__ key, char2 *__restrict__ lev,
                              int32_t *__restrict__ cnt, unsigned *__restrict__ hist)
{
    __shared__ unsigned h[TREE_LEVELS];
    if (threadIdx.x < TREE_LEVELS) h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k < n) {
        const uint64_t kk = key[k];
        const int d = k ? common_digits(key[k - 1], kk) : -1;
        int m = -1;
        const int64_t i1 = k < n - 1 - leaf_max ? k : n - 1 - leaf_max;
        for (int64_t i = k > leaf_max ? k - leaf_max : 0; i <= i1; ++i)
            m = max(m, common_digits(key[i], key[i + leaf_max]));
        const int last = min(m + 1, em::kMortonBits);
        lev[k] = make_char2((char)(d + 1), (char)last);
        cnt[k] = max(0, last - d);
        for (int L = d + 1; L <= last; ++L) atomicAdd(&h[L], 1u);
    }
    __syncthreads();
    if (threadIdx.x < TREE_LEVELS && h[threadIdx.x]) atomicAdd(hist + threadIdx.x, h[threadIdx.x]);
}

__global__ void k_node_emit(int64_t n, const char2 *__restrict__ lev, const int32_t *__restrict__ ofs,
                            uint32_t *__restrict__ level, int32_t *__restrict__ first)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= n) return;
    const char2 l = lev[k];
    int32_t t = ofs[k];
    for (int L = l.x; L <= l.y; ++L, ++t) {
        level[t] = (uint32_t)L;
        first[t] = (int32_t)k;
    }
}

struct LevelOffsets {
    int32_t at[TREE_LEVELS + 2];   // first node of each level; the number of nodes from the last on
};

// First position in the ascending v[lo, hi) with v >= x.
__device__ __forceinline__ int32_t lower_bound(const int32_t *__restrict__ v, int32_t lo, int32_t hi, int32_t x)
{
    while (lo < hi) {
        const int32_t mid = lo + (hi - lo) / 2;
        if (v[mid] < x) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// The rest of a node from its level and first position: the end of its run of
// equal digits, and its parent and children by their first positions.
__global__ void k_node_topology(int32_t nn, int32_t n, int leaf_max, LevelOffsets off, const uint64_t *__restrict__ key,
                                const int32_t *__restrict__ level, const int32_t *__restrict__ first,
                                uint64_t *__restrict__ label, int32_t *__restrict__ parent,
                                int32_t *__restrict__ count, int32_t *__restrict__ first_child,
                                int32_t *__restrict__ nchild)
{
    const int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (a >= nn) return;
    const int L = level[a];
    const int32_t k = first[a];
    const int shift = 3 * (em::kMortonBits - L);
    const uint64_t p = key[k] >> shift;
    // end: the last probe known inside is lo, the first known outside hi
    int64_t lo = k, hi = n, step = 1;
    while (lo + step < hi) {
        if ((key[lo + step] >> shift) == p) lo += step;
        else hi = lo + step;
        step *= 2;
    }
    while (hi - lo > 1) {
        const int64_t mid = lo + (hi - lo) / 2;
        if ((key[mid] >> shift) == p) lo = mid;
        else hi = mid;
    }
    label[a] = (1ull << (3 * L)) | p;
    count[a] = (int32_t)(hi - k);
    parent[a] = L ? lower_bound(first, off.at[L - 1], off.at[L], k + 1) - 1 : -1;
    if (hi - k > leaf_max && L < em::kMortonBits) {
        const int32_t c0 = lower_bound(first, off.at[L + 1], off.at[L + 2], k);
        first_child[a] = c0;
        nchild[a] = lower_bound(first, c0, off.at[L + 2], (int32_t)hi) - c0;
    } else {
        first_child[a] = -1;
        nchild[a] = 0;
    }
}

// Mass, m x and centre of mass of every node in one launch: a thread sums a
// leaf, then climbs; the last of a node's children to arrive sums the node.
// Leaves add their particles in Morton order, nodes their children in octant
// order, whoever does it.
__global__ void k_node_sums(int64_t nnode, const int32_t *__restrict__ parent, const int32_t *__restrict__ first,
                            const int32_t *__restrict__ count, const int32_t *__restrict__ first_child,
                            const int32_t *__restrict__ nchild, const double *__restrict__ xs,
                            const double *__restrict__ ys, const double *__restrict__ zs,
                            const double *__restrict__ ms, int32_t *__restrict__ arrived, double *mass, double *mx,
                            double *my, double *mz, double *__restrict__ cx, double *__restrict__ cy,
                            double *__restrict__ cz)
{
    int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (a >= nnode || nchild[a] != 0) return;
    double sm = 0.0, sx = 0.0, sy = 0.0, sz = 0.0;
    for (int32_t k = first[a]; k < first[a] + count[a]; ++k) {
        const double mk = ms[k];
        sm = __dadd_rn(sm, mk);
        sx = __dadd_rn(sx, __dmul_rn(mk, xs[k]));
        sy = __dadd_rn(sy, __dmul_rn(mk, ys[k]));
        sz = __dadd_rn(sz, __dmul_rn(mk, zs[k]));
    }
    while (true) {
        __stcg(mass + a, sm);
        __stcg(mx + a, sx);
        __stcg(my + a, sy);
        __stcg(mz + a, sz);
        cx[a] = __ddiv_rn(sx, sm);
        cy[a] = __ddiv_rn(sy, sm);
        cz[a] = __ddiv_rn(sz, sm);
        const int32_t p = parent[a];
        if (p < 0) return;
        __threadfence();
        if (atomicAdd(arrived + p, 1) != nchild[p] - 1) return;
        __threadfence();
        a = p;
        sm = sx = sy = sz = 0.0;
        for (int32_t c = first_child[a]; c < first_child[a] + nchild[a]; ++c) {
            sm = __dadd_rn(sm, __ldcg(mass + c));
            sx = __dadd_rn(sx, __ldcg(mx + c));
            sy = __dadd_rn(sy, __ldcg(my + c));
            sz = __dadd_rn(sz, __ldcg(mz + c));
        }
    }
}

// s_node = max over constituents of |x - COM|.  Nodes of up to SIZE_SMALL
// constituents, nearly all, take a thread each.  The others are cut into chunks
// of SIZE_CHUNK constituents, one warp per chunk, so that the root's million
// particles do not fall to one warp; each chunk raises its node's r^2 with an
// atomic max on the bit pattern (non-negative doubles order like their bits).
// Every term is rounded alike and max does not depend on the order, so
// the result is the same bit for bit.
constexpr int SIZE_SMALL = 32, SIZE_CHUNK = 1024;

__device__ __forceinline__ double dist2_rn(double x, double y, double z, double ax, double ay, double az)
{
    const double dx = __dsub_rn(x, ax), dy = __dsub_rn(y, ay), dz = __dsub_rn(z, az);
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

__global__ void k_size_small(int64_t nnode, const int32_t *__restrict__ first, const int32_t *__restrict__ count,
                             const double *__restrict__ xs, const double *__restrict__ ys,
                             const double *__restrict__ zs, const double *__restrict__ cx,
                             const double *__restrict__ cy, const double *__restrict__ cz, double *__restrict__ size,
                             int64_t *__restrict__ nchunk)
{
    const int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (a >= nnode) return;
    const int32_t n = count[a], k0 = first[a];
    nchunk[a] = n > SIZE_SMALL ? (n + SIZE_CHUNK - 1) / SIZE_CHUNK : 0;
    double r2 = 0.0;
    if (n <= SIZE_SMALL) {
        const double ax = cx[a], ay = cy[a], az = cz[a];
        for (int32_t k = k0; k < k0 + n; ++k) {
            const double q = dist2_rn(xs[k], ys[k], zs[k], ax, ay, az);
            r2 = q > r2 ? q : r2;
        }
    }
    size[a] = r2;
}

__global__ void k_node_size(int64_t nnode, const int64_t *__restrict__ task_off, const int32_t *__restrict__ first,
                            const int32_t *__restrict__ count, const double *__restrict__ xs,
                            const double *__restrict__ ys, const double *__restrict__ zs,
                            const double *__restrict__ cx, const double *__restrict__ cy,
                            const double *__restrict__ cz, unsigned long long *__restrict__ r2bits)
{
    const int lane = threadIdx.x & 31;
    const int64_t ntask = task_off[nnode], warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; t < ntask; t += warps) {
        int64_t lo = 0, hi = nnode;   // task_off[lo] <= t < task_off[hi]
        while (hi - lo > 1) {
            const int64_t mid = (lo + hi) >> 1;
            if (task_off[mid] <= t) lo = mid;
            else hi = mid;
        }
        const int64_t a = lo;
        const int64_t c = t - task_off[a];
        const double ax = cx[a], ay = cy[a], az = cz[a];
        const int32_t k0 = first[a] + (int32_t)(c * SIZE_CHUNK);
        const int32_t k1 = min(first[a] + count[a], k0 + SIZE_CHUNK);
        double r2 = 0.0;
        for (int32_t k = k0 + lane; k < k1; k += 32) {
            const double q = dist2_rn(xs[k], ys[k], zs[k], ax, ay, az);
            r2 = q > r2 ? q : r2;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double q = __shfl_xor_sync(0xffffffffu, r2, o);
            r2 = q > r2 ? q : r2;
        }
        if (lane == 0) atomicMax(r2bits + a, (unsigned long long)__double_as_longlong(r2));
    }
}

__global__ void k_size_finish(int64_t nnode, double *__restrict__ size)
{
    const int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (a < nnode) size[a] = __dsqrt_rn(size[a]);   // the bits hold r^2 as a double
}

}  // namespace

// Morton sort of n points: keys and permutation (stable: ties by index).
int em_morton_sort(em_ctx *ctx, int64_t n, const double *x, const double *y, const double *z, const double *box,
                   uint64_t *key, int32_t *perm)
{
    k_morton<<<em_grid(n, 256), 256, 0, ctx->stream>>>(n, x, y, z, box[0], box[1], box[2], box[3], box[4], box[5],
                                                       key, perm);
    EM_LAUNCHED(ctx);
    return em_sort_pairs_u64(ctx, key, perm, n, 3 * em::kMortonBits);
}

int em_gather_sorted(em_ctx *ctx, int64_t n, const int32_t *perm, const double *x, const double *y,
                     const double *z, const double *m, double *xs, double *ys, double *zs, double *ms)
{
    k_gather4<<<em_grid(n, 256), 256, 0, ctx->stream>>>(n, perm, x, y, z, m, xs, ys, zs, ms);
    EM_LAUNCHED(ctx);
    return EM_OK;
}

static int build_tree_impl(em_ctx *ctx, em_tree *t, const double *d_x, const double *d_y, const double *d_z,
                           const double *d_m, int leaf_max)
{
    const int64_t n = t->n;
    cudaStream_t st = ctx->stream;
    DevArena &mem = t->mem;
    EM_TRY(mem.alloc(&t->key, n));
    EM_TRY(mem.alloc(&t->perm, n));
    EM_TRY(mem.alloc(&t->xs, n));
    EM_TRY(mem.alloc(&t->ys, n));
    EM_TRY(mem.alloc(&t->zs, n));
    EM_TRY(mem.alloc(&t->ms, n));
    EM_TRY(em_morton_sort(ctx, n, d_x, d_y, d_z, t->box, t->key, t->perm));
    EM_TRY(em_gather_sorted(ctx, n, t->perm, d_x, d_y, d_z, d_m, t->xs, t->ys, t->zs, t->ms));

    // topology: nodes per position, then breadth first by a sort on the level
    DevArena tmp(st, true);
    char2 *lev;
    int32_t *cnt, *ofs;
    unsigned *hist;
    EM_TRY(tmp.alloc(&lev, n));
    EM_TRY(tmp.alloc(&cnt, n));
    EM_TRY(tmp.alloc(&ofs, n));
    EM_TRY(tmp.alloc(&hist, TREE_LEVELS));
    EM_CUDA(cudaMemsetAsync(hist, 0, TREE_LEVELS * sizeof(unsigned), st));
    k_node_levels<<<em_grid(n, 256), 256, 0, st>>>(n, leaf_max, t->key, lev, cnt, hist);
    EM_LAUNCHED(ctx);
    EM_TRY(em_exclusive_scan_i32(ctx, cnt, ofs, n));
    unsigned h[TREE_LEVELS];
    EM_CUDA(cudaMemcpyAsync(h, hist, sizeof h, cudaMemcpyDeviceToHost, st));
    EM_CUDA(cudaStreamSynchronize(st));
    std::vector<int64_t> loff = {0};
    for (int L = 0; L < TREE_LEVELS && h[L]; ++L) loff.push_back(loff.back() + h[L]);
    if (loff.back() >= INT32_MAX) {
        em_set_error("build_tree: %lld nodes exceed the 2^31 limit", (long long)loff.back());
        return EM_ECAPACITY;
    }
    t->depth = (int)loff.size() - 2;
    t->nnode = loff.back();
    const int64_t nn = t->nnode;
    LevelOffsets off;
    for (int L = 0; L < TREE_LEVELS + 2; ++L) off.at[L] = (int32_t)(L < (int)loff.size() ? loff[L] : nn);
    EM_TRY(mem.alloc(&t->label, nn));
    EM_TRY(mem.alloc(&t->level, nn));
    EM_TRY(mem.alloc(&t->parent, nn));
    EM_TRY(mem.alloc(&t->first, nn));
    EM_TRY(mem.alloc(&t->count, nn));
    EM_TRY(mem.alloc(&t->first_child, nn));
    EM_TRY(mem.alloc(&t->nchild, nn));
    k_node_emit<<<em_grid(n, 256), 256, 0, st>>>(n, lev, ofs, (uint32_t *)t->level, t->first);
    EM_LAUNCHED(ctx);
    EM_TRY(em_sort_pairs_u32(ctx, (uint32_t *)t->level, t->first, nn, em_nbits(em::kMortonBits)));
    k_node_topology<<<em_grid(nn, 256), 256, 0, st>>>((int32_t)nn, (int32_t)n, leaf_max, off, t->key, t->level,
                                                      t->first, t->label, t->parent, t->count, t->first_child,
                                                      t->nchild);
    EM_LAUNCHED(ctx);
    EM_TRY(mem.alloc(&t->mass, nn));
    EM_TRY(mem.alloc(&t->mx, nn));
    EM_TRY(mem.alloc(&t->my, nn));
    EM_TRY(mem.alloc(&t->mz, nn));
    EM_TRY(mem.alloc(&t->cx, nn));
    EM_TRY(mem.alloc(&t->cy, nn));
    EM_TRY(mem.alloc(&t->cz, nn));
    EM_TRY(mem.alloc(&t->size, nn));
    int32_t *arrived;
    int64_t *nchunk, *task_off;
    EM_TRY(tmp.alloc(&arrived, nn));
    EM_TRY(tmp.alloc(&nchunk, nn + 1));
    EM_TRY(tmp.alloc(&task_off, nn + 1));
    EM_CUDA(cudaMemsetAsync(arrived, 0, nn * sizeof(int32_t), st));
    EM_CUDA(cudaMemsetAsync(nchunk + nn, 0, sizeof(int64_t), st));
    k_node_sums<<<em_grid(nn, 128), 128, 0, st>>>(nn, t->parent, t->first, t->count, t->first_child, t->nchild, t->xs,
                                                  t->ys, t->zs, t->ms, arrived, t->mass, t->mx, t->my, t->mz, t->cx,
                                                  t->cy, t->cz);
    EM_LAUNCHED(ctx);
    k_size_small<<<em_grid(nn, 128), 128, 0, st>>>(nn, t->first, t->count, t->xs, t->ys, t->zs, t->cx, t->cy, t->cz,
                                                   t->size, nchunk);
    EM_LAUNCHED(ctx);
    EM_TRY(em_exclusive_scan_i64(ctx, nchunk, task_off, nn + 1));
    k_node_size<<<(unsigned)std::min<int64_t>(em_grid(nn * 32, 256), 8 * (int64_t)ctx->nsm), 256, 0, st>>>(
        nn, task_off, t->first, t->count, t->xs, t->ys, t->zs, t->cx, t->cy, t->cz, (unsigned long long *)t->size);
    EM_LAUNCHED(ctx);
    k_size_finish<<<em_grid(nn, 256), 256, 0, st>>>(nn, t->size);
    EM_LAUNCHED(ctx);
    return EM_OK;
}

EM_EXPORT int build_tree(em_ctx *ctx, int64_t n, const double *d_x, const double *d_y, const double *d_z,
                         const double *d_m, const double *h_box, int leaf_max, em_tree **out)
{
    EM_CHECK_ARG(ctx && out && h_box && d_x && d_y && d_z && d_m);
    EM_CHECK_ARG(n >= 1 && n < INT32_MAX);
    EM_CHECK_ARG(leaf_max >= 1 && leaf_max <= 64);
    EM_CHECK_ARG(h_box[1] > h_box[0] && h_box[3] > h_box[2] && h_box[5] > h_box[4]);
    *out = nullptr;
    em_tree *t = new em_tree(ctx->stream);
    t->device = ctx->device;
    t->n = n;
    for (int k = 0; k < 6; ++k) t->box[k] = h_box[k];
    int rc = build_tree_impl(ctx, t, d_x, d_y, d_z, d_m, leaf_max);
    if (rc) {
        t->mem.release();
        delete t;
        return rc;
    }
    *out = t;
    return EM_OK;
}

// ---------------------------------------------------------------------------
// Chunk tree (32-ary boxes over Morton-ordered items)
// ---------------------------------------------------------------------------

namespace {

// One warp per box, a lane per item (or child box): a thread per box walked its
// 32 items serially, 22 us a call however few they were.
__device__ __forceinline__ void warp_box(float (&lo)[3], float (&hi)[3])
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            lo[c] = fminf(lo[c], __shfl_xor_sync(0xffffffffu, lo[c], o));
            hi[c] = fmaxf(hi[c], __shfl_xor_sync(0xffffffffu, hi[c], o));
        }
}

__global__ void k_chunk_leaf(int64_t nbox, int64_t n, const double *__restrict__ xs, const double *__restrict__ ys,
                             const double *__restrict__ zs, const double *__restrict__ r, double rscale,
                             float4 *__restrict__ lo, float4 *__restrict__ hi, float4 *__restrict__ pts)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, b = k >> 5;
    if (b >= nbox) return;   // whole warps
    float l[3] = {INFINITY, INFINITY, INFINITY}, h[3] = {-INFINITY, -INFINITY, -INFINITY};
    if (k < n) {
        const double x = xs[k], y = ys[k], z = zs[k], rr = r ? r[k] * rscale : 0.0;
        pts[k] = make_float4((float)x, (float)y, (float)z, __double2float_ru(rr));
        l[0] = fminf(l[0], __double2float_rd(x - rr));
        l[1] = fminf(l[1], __double2float_rd(y - rr));
        l[2] = fminf(l[2], __double2float_rd(z - rr));
        h[0] = fmaxf(h[0], __double2float_ru(x + rr));
        h[1] = fmaxf(h[1], __double2float_ru(y + rr));
        h[2] = fmaxf(h[2], __double2float_ru(z + rr));
    }
    warp_box(l, h);
    if ((threadIdx.x & 31) == 0) {
        lo[b] = make_float4(l[0], l[1], l[2], 0.f);
        hi[b] = make_float4(h[0], h[1], h[2], 0.f);
    }
}

__global__ void k_chunk_up(int64_t nbox, int64_t nchild, const float4 *__restrict__ clo, const float4 *__restrict__ chi,
                           float4 *__restrict__ lo, float4 *__restrict__ hi)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, b = k >> 5;
    if (b >= nbox) return;   // whole warps
    float l[3] = {INFINITY, INFINITY, INFINITY}, h[3] = {-INFINITY, -INFINITY, -INFINITY};
    if (k < nchild) {
        const float4 a = clo[k], c = chi[k];
        l[0] = fminf(l[0], a.x);
        l[1] = fminf(l[1], a.y);
        l[2] = fminf(l[2], a.z);
        h[0] = fmaxf(h[0], c.x);
        h[1] = fmaxf(h[1], c.y);
        h[2] = fmaxf(h[2], c.z);
    }
    warp_box(l, h);
    if ((threadIdx.x & 31) == 0) {
        lo[b] = make_float4(l[0], l[1], l[2], 0.f);
        hi[b] = make_float4(h[0], h[1], h[2], 0.f);
    }
}

}  // namespace

int em_chunk_tree_build(em_ctx *ctx, DevArena &mem, int64_t n, const double *xs, const double *ys, const double *zs,
                        const double *r, double rscale, em::ChunkTree *out)
{
    em::ChunkTree T;
    T.count[0] = n;
    for (int l = 0; l <= em::kMaxLevels; ++l) {
        T.lo[l] = nullptr;
        T.hi[l] = nullptr;
        if (l) T.count[l] = 0;
    }
    T.nlev = 0;
    T.pts = nullptr;
    if (n == 0) {
        *out = T;
        return EM_OK;
    }
    EM_TRY(mem.alloc(&T.pts, n));
    int l = 1;
    for (;; ++l) {
        if (l > em::kMaxLevels) {
            em_set_error("chunk tree: %lld items exceed %d levels", (long long)n, em::kMaxLevels);
            return EM_ECAPACITY;
        }
        T.count[l] = (T.count[l - 1] + 31) / 32;
        EM_TRY(mem.alloc(&T.lo[l], T.count[l]));
        EM_TRY(mem.alloc(&T.hi[l], T.count[l]));
        if (l == 1)
            k_chunk_leaf<<<em_grid(T.count[1] * 32, 128), 128, 0, ctx->stream>>>(T.count[1], n, xs, ys, zs, r, rscale,
                                                                                  T.lo[1], T.hi[1], T.pts);
        else
            k_chunk_up<<<em_grid(T.count[l] * 32, 128), 128, 0, ctx->stream>>>(T.count[l], T.count[l - 1], T.lo[l - 1],
                                                                                T.hi[l - 1], T.lo[l], T.hi[l]);
        EM_LAUNCHED(ctx);
        if (T.count[l] <= 32) break;
    }
    T.nlev = l;
    *out = T;
    return EM_OK;
}
