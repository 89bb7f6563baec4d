// Exact mapping (map_exact), cell densities, inverse mapping (map_back), and
// the import paths for cells and pair lists.
#include <algorithm>
#include <climits>
#include <cmath>
#include <mutex>

#include "common.cuh"
#include "exact.cuh"
#include "fp64.cuh"
#include "quad32.cuh"
#include "split.cuh"

using namespace em;

// ---------------------------------------------------------------------------
// Derived cell geometry in each generator's frame
// ---------------------------------------------------------------------------

// Per face (one thread each): the face's cell by binary search in the cell
// offsets, the plane records, and the face and cell ids of its vertices for
// the edge pass.
__global__ void k_prepare_faces(int64_t nface, int64_t ncell, const double *__restrict__ gen,
                                const int64_t *__restrict__ cfo, const int64_t *__restrict__ fvo,
                                const double *__restrict__ verts, const double *__restrict__ normals,
                                PlaneD *__restrict__ plane, PlaneF *__restrict__ plane_f,
                                PlaneF *__restrict__ plane_fl, int32_t *__restrict__ face_of_fv,
                                int32_t *__restrict__ cell_of_face)
{
    const int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (f >= nface) return;
    int64_t lo = 0, hi = ncell;   // cfo[lo] <= f < cfo[hi]
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (cfo[mid] <= f) lo = mid;
        else hi = mid;
    }
    const int64_t j = lo;
    const double gx = gen[3 * j], gy = gen[3 * j + 1], gz = gen[3 * j + 2];
    double nx = normals[3 * f], ny = normals[3 * f + 1], nz = normals[3 * f + 2], c = 0.0;
    const int64_t v0 = fvo[f], v1 = fvo[f + 1];
    if (v0 < v1) c = nx * (verts[3 * v0] - gx) + ny * (verts[3 * v0 + 1] - gy) + nz * (verts[3 * v0 + 2] - gz);
    else nx = ny = nz = 0.0;   // an imported face of no vertices lies nowhere and bounds nothing
    plane[f] = PlaneD{nx, ny, nz, c};
    // hi and low parts: the plane = hi + lo to about 2^-48 relative (float-float)
    PlaneF F, G;
    split_all<4>({nx, ny, nz, c}, {&F.x, &F.y, &F.z, &F.w}, {&G.x, &G.y, &G.z, &G.w});
    plane_f[f] = F;
    plane_fl[f] = G;
    cell_of_face[f] = (int32_t)j;
    for (int64_t k = v0; k < v1; ++k) face_of_fv[k] = (int32_t)f;
}

// Per face-vertex k, one thread each: the edge from vertex k to the next vertex
// of its face, in the generator's frame, as FP64 and FP32 hi/lo records.  Bound
// by the FP64 pipe (about 36 operations a vertex): 21.2 M vertices 3.01 ms with
// the splits' conversions if-converted (split.cuh: split_all) and the records
// written 80 and 48 B apart, 2.08 ms so.  The records, 176 B a thread, are put
// together in shared memory and written out by adjacent threads.  The cell
// radius is the largest |V - g| over its
// vertices: the largest of a warp's lanes on one cell (a cell's vertices lie
// together) raises the cell's r^2 with an atomic max on the bit pattern
// (non-negative doubles order like their bits), so the result does not depend
// on the order.
constexpr int PREP_EDGES = 128;   // threads per block
__global__ void __launch_bounds__(PREP_EDGES)
    k_prepare_edges(int64_t nfv, const double *__restrict__ gen, const int64_t *__restrict__ fvo,
                    const double *__restrict__ verts, const double *__restrict__ normals,
                    const int32_t *__restrict__ face_of_fv, const int32_t *__restrict__ cell_of_face,
                    unsigned long long *__restrict__ r2bits, EdgeD *__restrict__ edge, EdgeF *__restrict__ edge_f,
                    EdgeF *__restrict__ edge_fl)
{
    __shared__ EdgeD sd[PREP_EDGES];
    __shared__ EdgeF sf[2][PREP_EDGES];
    const int64_t kb = blockIdx.x * (int64_t)PREP_EDGES, k = min(kb + (int64_t)threadIdx.x, nfv - 1);
    const int64_t f = face_of_fv[k];
    const int64_t j = cell_of_face[f];
    const double gx = gen[3 * j], gy = gen[3 * j + 1], gz = gen[3 * j + 2];
    const double nx = normals[3 * f], ny = normals[3 * f + 1], nz = normals[3 * f + 2];
    const int64_t v0 = fvo[f], v1 = fvo[f + 1];
    int64_t k1 = (k + 1 < v1) ? k + 1 : v0;
    double ax = verts[3 * k] - gx, ay = verts[3 * k + 1] - gy, az = verts[3 * k + 2] - gz;
    double bx = verts[3 * k1] - gx, by = verts[3 * k1 + 1] - gy, bz = verts[3 * k1 + 2] - gz;
    double q = ax * ax + ay * ay + az * az;
    double ex = bx - ax, ey = by - ay, ez = bz - az;
    // L and 1/L from one reciprocal square root: an FP32 seed (on the bits,
    // split.cuh) and the series of (1 - e)^(-1/2), e = 1 - s2 r0^2 of at most
    // 2^-20, to e^2 (the next term is below 2^-61), within about an ulp, for
    // fewer FP64 instructions than a square root and a division
    const double s2 = ex * ex + ey * ey + ez * ez;
    double L = 0.0;
    EdgeD E;
    const int e2 = __double2hiint(s2) >> 20;   // the exponent: s2 >= 0 (a comparison would issue at the FP64 rate)
    if (e2 >= 1023 - 99 && e2 < 1023 + 99) {   // the seed in float's normal range
        const double r0 = f64_of(rsqrtf(f32_of(s2))), e = fma(-(s2 * r0), r0, 1.0);
        const double r = fma(r0 * e, fma(0.375, e, 0.5), r0);
        L = s2 * r;
        ex *= r;
        ey *= r;
        ez *= r;
    } else if (s2 > 0.0) {   // outside it: the plain operations
        L = sqrt(s2);
        ex /= L;
        ey /= L;
        ez /= L;
    }
    E.ex = ex;
    E.ey = ey;
    E.ez = ez;
    E.L = L;
    E.mx = ey * nz - ez * ny;   // e x n: in-plane outward normal
    E.my = ez * nx - ex * nz;
    E.mz = ex * ny - ey * nx;
    E.cm = E.mx * ax + E.my * ay + E.mz * az;
    E.ce = ex * ax + ey * ay + ez * az;
    E.pad = 0.0;
    sd[threadIdx.x] = E;
    // hi and low parts: E = hi + lo to about 2^-48 relative (float-float)
    EdgeF F, G;
    split_all<9>({E.mx, E.my, E.mz, E.cm, E.ex, E.ey, E.ez, E.ce, E.L},
                 {&F.mx, &F.my, &F.mz, &F.cm, &F.ex, &F.ey, &F.ez, &F.ce, &F.L},
                 {&G.mx, &G.my, &G.mz, &G.cm, &G.ex, &G.ey, &G.ez, &G.ce, &G.L});
    F.pad0 = F.pad1 = F.pad2 = 0.f;
    G.pad0 = G.pad1 = G.pad2 = 0.f;
    sf[0][threadIdx.x] = F;
    sf[1][threadIdx.x] = G;
    // the last threads past nfv repeat its vertex: they change no maximum
    const int lane = threadIdx.x & 31;
    unsigned long long qb = (unsigned long long)__double_as_longlong(q);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long qo = __shfl_down_sync(0xffffffffu, qb, o);
        const int jo = __shfl_down_sync(0xffffffffu, (int)j, o);
        if (lane + o < 32 && jo == (int)j) qb = max(qb, qo);
    }
    const int jp = __shfl_up_sync(0xffffffffu, (int)j, 1);
    if (lane == 0 || jp != (int)j) atomicMax(r2bits + j, qb);
    __syncthreads();
    const int n = (int)min((int64_t)PREP_EDGES, nfv - kb);
    constexpr int ND = sizeof(EdgeD) / 16, NF = sizeof(EdgeF) / 16;
    for (int i = threadIdx.x; i < n * ND; i += PREP_EDGES) ((float4 *)(edge + kb))[i] = ((const float4 *)sd)[i];
    for (int i = threadIdx.x; i < n * NF; i += PREP_EDGES) {
        ((float4 *)(edge_f + kb))[i] = ((const float4 *)sf[0])[i];
        ((float4 *)(edge_fl + kb))[i] = ((const float4 *)sf[1])[i];
    }
}

__global__ void k_radius_finish(int64_t ncell, double *__restrict__ radius)
{
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j >= ncell) return;
    radius[j] = sqrt(radius[j]);   // the bits hold r^2 as a double
}

int em_prepare_cells(em_ctx *ctx, em_voronoi *v)
{
    EM_TRY(v->mem.alloc(&v->radius, v->ncell));
    EM_TRY(v->mem.alloc(&v->plane, v->nface));
    EM_TRY(v->mem.alloc(&v->edge, v->nfv));
    EM_TRY(v->mem.alloc(&v->plane_f, v->nface));
    EM_TRY(v->mem.alloc(&v->plane_fl, v->nface));
    EM_TRY(v->mem.alloc(&v->edge_f, v->nfv));
    EM_TRY(v->mem.alloc(&v->edge_fl, v->nfv));
    if (v->ncell) {
        EM_CUDA(cudaMemsetAsync(v->radius, 0, v->ncell * sizeof(double), ctx->stream));
        if (v->nface) {
            DevArena tmp(ctx->stream, true);
            int32_t *face_of_fv, *cell_of_face;
            EM_TRY(tmp.alloc(&face_of_fv, v->nfv));
            EM_TRY(tmp.alloc(&cell_of_face, v->nface));
            k_prepare_faces<<<em_grid(v->nface, 128), 128, 0, ctx->stream>>>(
                v->nface, v->ncell, v->gen, v->cell_face_off, v->face_vert_off, v->verts, v->normals, v->plane,
                v->plane_f, v->plane_fl, face_of_fv, cell_of_face);
            EM_LAUNCHED(ctx);
            if (v->nfv) {   // its last threads repeat vertex nfv - 1
                k_prepare_edges<<<em_grid(v->nfv, PREP_EDGES), PREP_EDGES, 0, ctx->stream>>>(
                    v->nfv, v->gen, v->face_vert_off, v->verts, v->normals, face_of_fv, cell_of_face,
                    (unsigned long long *)v->radius, v->edge, v->edge_f, v->edge_fl);
                EM_LAUNCHED(ctx);
            }
        }
        k_radius_finish<<<em_grid(v->ncell, 256), 256, 0, ctx->stream>>>(v->ncell, v->radius);
        EM_LAUNCHED(ctx);
    }
    return EM_OK;
}

EM_EXPORT int voronoi_from_cells(em_ctx *ctx, int64_t ncell, int64_t nface, int64_t nfv, const double *d_gen,
                                 const int64_t *d_cell_face_off, const int64_t *d_face_vert_off,
                                 const double *d_verts, const double *d_normals, const int64_t *d_nbr,
                                 const double *d_volume, em_voronoi **out)
{
    EM_CHECK_ARG(ctx && out && ncell >= 0 && ncell < INT32_MAX && nface >= 0 && nfv >= 0);
    EM_CHECK_ARG(d_gen && d_cell_face_off && d_face_vert_off && d_verts && d_normals && d_volume);
    *out = nullptr;
    em_voronoi *v = new em_voronoi(ctx->stream);
    v->device = ctx->device;
    v->ncell = ncell;
    v->nface = nface;
    v->nfv = nfv;
    for (int k = 0; k < 6; ++k) v->box[k] = 0.0;
    int s = EM_OK;
    auto fail = [&](int st) {
        v->mem.release();
        delete v;
        return st;
    };
    if ((s = v->mem.alloc(&v->gen, 3 * ncell)) || (s = v->mem.alloc(&v->cell_face_off, ncell + 1)) ||
        (s = v->mem.alloc(&v->face_vert_off, nface + 1)) || (s = v->mem.alloc(&v->verts, 3 * nfv)) ||
        (s = v->mem.alloc(&v->normals, 3 * nface)) || (s = v->mem.alloc(&v->nbr, nface)) ||
        (s = v->mem.alloc(&v->volume, ncell)))
        return fail(s);
    cudaStream_t st = ctx->stream;
    cudaMemcpyAsync(v->gen, d_gen, 3 * ncell * sizeof(double), cudaMemcpyDeviceToDevice, st);
    cudaMemcpyAsync(v->cell_face_off, d_cell_face_off, (ncell + 1) * sizeof(int64_t), cudaMemcpyDeviceToDevice, st);
    cudaMemcpyAsync(v->face_vert_off, d_face_vert_off, (nface + 1) * sizeof(int64_t), cudaMemcpyDeviceToDevice, st);
    cudaMemcpyAsync(v->verts, d_verts, 3 * nfv * sizeof(double), cudaMemcpyDeviceToDevice, st);
    cudaMemcpyAsync(v->normals, d_normals, 3 * nface * sizeof(double), cudaMemcpyDeviceToDevice, st);
    if (d_nbr) cudaMemcpyAsync(v->nbr, d_nbr, nface * sizeof(int64_t), cudaMemcpyDeviceToDevice, st);
    else cudaMemsetAsync(v->nbr, 0xff, nface * sizeof(int64_t), st);
    cudaMemcpyAsync(v->volume, d_volume, ncell * sizeof(double), cudaMemcpyDeviceToDevice, st);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        em_set_error("voronoi_from_cells: %s", cudaGetErrorString(e));
        return fail(EM_ECUDA);
    }
    if ((s = em_prepare_cells(ctx, v))) return fail(s);
    *out = v;
    return EM_OK;
}

// ---------------------------------------------------------------------------
// Pair index: CSR offsets by cell and the (i, j)-ordered transpose
// ---------------------------------------------------------------------------

// off[c] = first position k with key[k] >= c, for c in [0, nseg]; key sorted.
__global__ void k_segment_offsets(int64_t n, const int32_t *__restrict__ key, int64_t nseg, int64_t *__restrict__ off,
                                  int *__restrict__ bad)
{
    int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k > n) return;
    int64_t prev = (k == 0) ? -1 : (int64_t)key[k - 1];
    int64_t cur = (k == n) ? nseg : (int64_t)key[k];
    if (k < n && (cur < 0 || cur >= nseg)) {
        atomicOr(bad, 1);
        return;
    }
    if (cur < prev) {
        atomicOr(bad, 2);
        return;
    }
    // (a negative key before this one is an error that its own thread raises)
    for (int64_t c = prev < -1 ? 0 : prev + 1; c <= cur; ++c) off[c] = k;
}

__global__ void k_iota_keys(int64_t n, const int32_t *__restrict__ src, uint32_t *__restrict__ key,
                            int32_t *__restrict__ val)
{
    int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= n) return;
    key[k] = (uint32_t)src[k];
    val[k] = (int32_t)k;
}

__global__ void k_check_within_cell(int64_t n, const int32_t *__restrict__ pi, const int32_t *__restrict__ pj,
                                    int64_t np, int *__restrict__ bad)
{
    int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= n) return;
    if (pi[k] < 0 || pi[k] >= np) atomicOr(bad, 4);
    if (k > 0 && pj[k] == pj[k - 1] && pi[k] <= pi[k - 1]) atomicOr(bad, 8);
}

// The rows of the transpose with more than EM_ROW_LONG pairs, which long_rows
// sums 32 at a time, longest first and like lengths together (four classes an
// octave; the order within one is of no account).  k_long_count: rows per class.
constexpr int ROW_CLASSES = 32, VERY_CLASS = 14;
constexpr int ROW_VERY = 1086, ROW_FEW = 8;   // EM_ROW_LONG 2^(VERY_CLASS / 4), rounded down; rows a block has of them
__device__ __forceinline__ int row_class(int64_t n)
{
    return ROW_CLASSES - 1 - min(ROW_CLASSES - 1, (int)(4.f * log2f((float)n * (1.f / EM_ROW_LONG))));
}

__global__ void k_long_count(int64_t np, const int64_t *__restrict__ off, int *__restrict__ count)
{
    __shared__ int c[ROW_CLASSES];
    if (threadIdx.x < ROW_CLASSES) c[threadIdx.x] = 0;
    __syncthreads();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t n = i < np ? off[i + 1] - off[i] : 0;
    if (n > EM_ROW_LONG) atomicAdd(&c[row_class(n)], 1);
    __syncthreads();
    if (threadIdx.x < ROW_CLASSES && c[threadIdx.x]) atomicAdd(count + threadIdx.x, c[threadIdx.x]);
}

// Into rows (of that capacity: the offsets of a list that is refused afterwards
// may be anything), with their number to nlong[0] and that of those of at least
// about ROW_VERY pairs to nlong[1].
__global__ void k_long_place(int64_t np, const int64_t *__restrict__ off, const int *__restrict__ count,
                             int *__restrict__ cursor, int capacity, int32_t *__restrict__ rows, int *__restrict__ nlong)
{
    __shared__ int c[ROW_CLASSES], base[ROW_CLASSES];
    const int t = threadIdx.x;
    if (t < ROW_CLASSES) c[t] = 0;
    __syncthreads();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + t;
    const int64_t n = i < np ? off[i + 1] - off[i] : 0;
    int k = 0, r = 0;
    if (n > EM_ROW_LONG) {
        k = row_class(n);
        r = atomicAdd(&c[k], 1);
    }
    __syncthreads();
    if (t < ROW_CLASSES) {   // one warp
        int first = count[t];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, first, o);
            if (t >= o) first += x;
        }
        if (blockIdx.x == 0 && t == ROW_CLASSES - 1) nlong[0] = min(first, capacity);
        if (blockIdx.x == 0 && t == ROW_CLASSES - 1 - VERY_CLASS) nlong[1] = min(first, capacity);
        base[t] = first - count[t] + (c[t] ? atomicAdd(cursor + t, c[t]) : 0);
    }
    __syncthreads();
    if (n > EM_ROW_LONG && base[k] + r < capacity) rows[base[k] + r] = (int32_t)i;
}
static_assert(ROW_CLASSES == 32, "one warp scans the classes");

// The (i, j)-ordered transpose of a list ordered by (j, i): a stable sort by i.
// bad (or null): raised where the sorted keys are out of range.
int em_build_transpose(em_ctx *ctx, em_pairs *pr, int *bad)
{
    const int64_t n = pr->npairs;
    DevArena tmp(ctx->stream, true);
    int *ignored;
    EM_TRY(tmp.alloc(&ignored, 1));
    EM_TRY(pr->mem.alloc(&pr->part_pair_off, pr->np + 1));
    EM_TRY(pr->mem.alloc(&pr->part_pair_idx, n));
    uint32_t *keys;
    EM_TRY(tmp.alloc(&keys, n));
    if (n) {
        k_iota_keys<<<em_grid(n, 256), 256, 0, ctx->stream>>>(n, pr->pair_i, keys, pr->part_pair_idx);
        EM_LAUNCHED(ctx);
        EM_TRY(em_sort_pairs_u32(ctx, keys, pr->part_pair_idx, n, em_nbits((uint64_t)pr->np)));
    }
    k_segment_offsets<<<em_grid(n + 1, 256), 256, 0, ctx->stream>>>(n, (const int32_t *)keys, pr->np,
                                                                      pr->part_pair_off, bad ? bad : ignored);
    EM_LAUNCHED(ctx);
    if (n > EM_ROW_LONG && pr->np) {
        int *count;   // and the cursors
        EM_TRY(tmp.alloc(&count, 2 * ROW_CLASSES));
        EM_CUDA(cudaMemsetAsync(count, 0, 2 * ROW_CLASSES * sizeof(int), ctx->stream));
        const int capacity = (int)(n / (EM_ROW_LONG + 1));
        EM_TRY(pr->mem.alloc(&pr->nlong, 2));
        EM_TRY(pr->mem.alloc(&pr->long_rows, capacity));
        k_long_count<<<em_grid(pr->np, 256), 256, 0, ctx->stream>>>(pr->np, pr->part_pair_off, count);
        EM_LAUNCHED(ctx);
        k_long_place<<<em_grid(pr->np, 256), 256, 0, ctx->stream>>>(pr->np, pr->part_pair_off, count,
                                                                     count + ROW_CLASSES, capacity, pr->long_rows,
                                                                     pr->nlong);
        EM_LAUNCHED(ctx);
    }
    return EM_OK;
}

// Cell offsets and transpose of a given list, which is checked.
int em_build_pair_index(em_ctx *ctx, em_pairs *pr)
{
    int64_t n = pr->npairs;
    DevArena tmp(ctx->stream, true);
    int *bad;
    EM_TRY(tmp.alloc(&bad, 1));
    EM_CUDA(cudaMemsetAsync(bad, 0, sizeof(int), ctx->stream));
    EM_TRY(pr->mem.alloc(&pr->cell_pair_off, pr->ncell + 1));
    k_segment_offsets<<<em_grid(n + 1, 256), 256, 0, ctx->stream>>>(n, pr->pair_j, pr->ncell, pr->cell_pair_off, bad);
    EM_LAUNCHED(ctx);
    if (n) {
        k_check_within_cell<<<em_grid(n, 256), 256, 0, ctx->stream>>>(n, pr->pair_i, pr->pair_j, pr->np, bad);
        EM_LAUNCHED(ctx);
    }
    EM_TRY(em_build_transpose(ctx, pr, bad));
    int hbad = 0;
    EM_CUDA(cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    EM_CUDA(cudaStreamSynchronize(ctx->stream));
    if (hbad) {
        em_set_error("pair list invalid (code %d): indices out of range or not sorted by (j, i)", hbad);
        return EM_EINVAL;
    }
    return EM_OK;
}

EM_EXPORT int pairs_from_list(em_ctx *ctx, int64_t npairs, const int32_t *d_pair_i, const int32_t *d_pair_j,
                              int64_t np, const em_voronoi *v, em_pairs **out)
{
    EM_CHECK_ARG(ctx && v && out && npairs >= 0 && npairs < INT32_MAX && np >= 0 && np < INT32_MAX);
    EM_CHECK_ARG(npairs == 0 || (d_pair_i && d_pair_j));
    *out = nullptr;
    em_pairs *pr = new em_pairs(ctx->stream);
    pr->device = ctx->device;
    pr->npairs = npairs;
    pr->np = np;
    pr->ncell = v->ncell;
    int s;
    if ((s = pr->mem.alloc(&pr->pair_i, npairs)) || (s = pr->mem.alloc(&pr->pair_j, npairs)) ||
        (s = pr->mem.alloc(&pr->near, npairs))) {
        pr->mem.release();
        delete pr;
        return s;
    }
    if (npairs) {
        cudaMemcpyAsync(pr->pair_i, d_pair_i, npairs * sizeof(int32_t), cudaMemcpyDeviceToDevice, ctx->stream);
        cudaMemcpyAsync(pr->pair_j, d_pair_j, npairs * sizeof(int32_t), cudaMemcpyDeviceToDevice, ctx->stream);
        cudaMemsetAsync(pr->near, 0, npairs, ctx->stream);
    }
    if ((s = em_build_pair_index(ctx, pr))) {
        pr->mem.release();
        delete pr;
        return s;
    }
    *out = pr;
    return EM_OK;
}

// ---------------------------------------------------------------------------
// Per-pair weight
// ---------------------------------------------------------------------------

template <class T>
struct GeomT;
template <>
struct GeomT<double> {
    using Plane = PlaneD;
    using Edge = EdgeD;
};
template <>
struct GeomT<float> {
    using Plane = PlaneF;
    using Edge = EdgeF;
};

// w for particle p (r = p - g, absolute units) and cell j; err returns the sum
// of magnitudes of the combined terms (in units of w).  ALWAYS_FULL selects
// the full form for every pair (the FP64 path).
template <class T, bool ALWAYS_FULL>
__device__ __forceinline__ T pair_weight(T rx, T ry, T rz, T h, T radius, int64_t f0, int64_t f1,
                                         const int64_t *__restrict__ fvo,
                                         const typename GeomT<T>::Plane *__restrict__ plane,
                                         const typename GeomT<T>::Edge *__restrict__ edge, T &err)
{
    const T ih = T(1) / h;
    bool inside = true;
    if (!ALWAYS_FULL) {
        for (int64_t f = f0; f < f1; ++f) {
            auto pl = plane[f];
            T s = pl.w - (pl.x * rx + pl.y * ry + pl.z * rz);
            inside = inside && !(s < T(0));
        }
    }
    T rr = em_sqrt(rx * rx + ry * ry + rz * rz);
    const bool full = ALWAYS_FULL || (inside && (rr + radius < T(2) * h));
    T acc = T(0), comp = T(0);   // compensated (Kahan) accumulation over faces
    err = (!full && inside) ? T(1) : T(0);
    T terr = T(0);
    for (int64_t f = f0; f < f1; ++f) {
        auto pl = plane[f];
        T s = pl.w - (pl.x * rx + pl.y * ry + pl.z * rz);
        T D = fabs(s) * ih;
        if (s == T(0) || (!full && D >= T(2))) continue;
        const T kd = full ? K_of<T>(D) : K_tilde<T>(D);
        T fs = T(0);
        int64_t e0 = fvo[f], e1 = fvo[f + 1];
        for (int64_t e = e0; e < e1; ++e) {
            auto E = edge[e];
            T a = E.cm - (E.mx * rx + E.my * ry + E.mz * rz);
            if (a == T(0)) continue;
            T A = fabs(a) * ih;
            T t0 = (E.ce - (E.ex * rx + E.ey * ry + E.ez * rz)) * ih;
            T t1 = t0 + E.L * ih;
            T c = full ? edge_full<T>(D, A, t0, t1, kd, terr) : edge_tilde<T>(D, A, t0, t1, kd, terr);
            fs += (a > T(0)) ? c : -c;
        }
        T term = (s > T(0)) ? fs : -fs;
        T y = term - comp;
        T t = acc + y;
        comp = (t - acc) - y;
        acc = t;
    }
    err += terr * Consts<T>::inv_pi;
    T w = acc * Consts<T>::inv_pi;
    return full ? w : ((inside ? T(1) : T(0)) - w);
}

// FP64 closed form, one warp per pair (both the FP64 mode and the recompute
// of the pairs the mixed pass flagged).
//
// An edge with signed in-plane distance a and range [T0, T1] along its line
// contributes sum_r int_{portion r} [K_r(Q) - K(D)] D a / (a^2 + tau^2) dtau
// over its portions in the kernel's regions r (Q < 1, Q < 2, beyond).  With
// K_r = sum_n c_n Q^n and Q^2 = D^2 + a^2 + tau^2, the antiderivatives reduce
// to two angles and one logarithm (see exact.cuh for J_n and U_n):
//     C_r(D) theta + S_r(D) psi + D a (E_r + H_r dash),
//     theta = atan(T1/a) - atan(T0/a), the angle of (a^2 + T0 T1, a (T1 - T0)),
//     psi = atan(D T1/(a Q1)) - atan(D T0/(a Q0)), the angle of
//           (a^2 Q0 Q1 + D^2 T0 T1, a D (T1 Q0 - T0 Q1)),
//     dash = asinh(T1/B) - asinh(T0/B), the log of a ratio of |T| + Q,
//     S_r = c_-1 + c_3 D^4 + c_5 D^6,  C_r = D (c_0 + c_2 D^2 + c_4 D^4) - D K(D),
// E_r a polynomial in T, Q.  So a portion takes two angles, a logarithm and
// no more square roots than its end points, where evaluating the six
// antiderivatives at every end point and every crossing took two angles, an
// asinh and two roots each; the rounding is that of the same terms, each at
// most ~1.  C_r and S_r are formed once per face (C_r = -S_r exactly where D
// lies in region r).
//
// Each lane takes an edge, cuts it at the region crossings and appends its
// portions to one of two per-warp queues, regions 1 and 2 or region 3 (angles
// alone); whenever a queue holds 32 entries the warp evaluates them, one per
// lane.  The kernel is bound by the number of FP64 instructions (one per ~20
// cycles per SM whatever its active lanes): region tests run in FP32 (a
// portion cut 1e-7 off moves the integral by the fifth power of that, since
// K's pieces agree to fourth order), and the transcendentals are fp64.cuh's.
// 4.68 M pairs of the 2e5-particle cloud: 109.9 ms (4.3e7 pairs/s), against
// 367.6 ms with the six antiderivatives; the FP64 pipe is 88% busy, issue 15%.
// Each lane adds what it evaluated; a fixed-order warp sum ends the pair.  The
// order of the evaluations depends on the pair alone, so the result is
// reproducible.  A cell with more than FW_MAXF faces (possible only for
// imported cells) is done by one lane with pair_weight.
//
// Entry t of list is k >= 0: pair k in the complement form (faces beyond 2h
// skipped; its rounding, about 1e-13, is far inside the mixed mode's
// tolerance), or ~k < 0: pair k in the full form (a particle in a face plane,
// for which such a face carries nothing).  Without a list, entry t is pair t
// in the full form (the FP64 mode).
constexpr int FW_WARPS = 4;
constexpr int FW_MAXF = 64;
constexpr int FQ = 64;   // ring capacity of each evaluation queue (a power of two, >= 63)

// Portions waiting for a full warp; code: the face's index | region << 8.
struct FwQueue {
    double a[FQ], T0[FQ], Q0[FQ], T1[FQ], Q1[FQ];
    int code[FQ];
};

// A warp's pair: per face D / h, its signed copy (orientation, and the
// complement form's sign), and the signed C_r and S_r.
struct FwPair {
    FwQueue near, far;
    double D[FW_MAXF], sD[FW_MAXF], C[3][FW_MAXF], S[3][FW_MAXF];
    int64_t E0[FW_MAXF];
    int pre[FW_MAXF + 1];
};

struct FwTab {
    double atan[65], log[64][2];
};

// theta and psi of a portion from a^2, D, D^2 and its ends
__device__ __forceinline__ void fw_angles(const FwTab &tb, double a, double a2, double D, double D2, double T0,
                                          double Q0, double T1, double Q1, double &theta, double &psi)
{
    const double tt = T0 * T1;
    theta = angle64(a * (T1 - T0), a2 + tt, tb.atan);
    psi = angle64((a * D) * fma(T1, Q0, -T0 * Q1), fma(a2, Q0 * Q1, D2 * tt), tb.atan);
}

__device__ __noinline__ double fw_eval_near(const FwPair &p, const FwTab &tb, int i)
{
    const FwQueue &q = p.near;
    const double a = q.a[i], T0 = q.T0[i], Q0 = q.Q0[i], T1 = q.T1[i], Q1 = q.Q1[i];
    const int f = q.code[i] & 255;
    const bool r1 = (q.code[i] >> 8) == 1;
    const double D = p.D[f], D2 = D * D, a2 = fma(a, a, 1e-280), B2 = a2 + D2;
    double theta, psi;
    fw_angles(tb, a, a2, D, D2, T0, Q0, T1, Q1, theta, psi);
    // asinh(T/B) = +-log((|T| + Q)/B)
    const bool s0 = __double2hiint(T0) < 0, s1 = __double2hiint(T1) < 0;
    const double e0 = fabs(T0) + Q0, e1 = fabs(T1) + Q1;
    const double ee = s0 != s1 ? e0 * e1 : 1.0;
    const double dash = log_ratio(s0 == s1 ? (s0 ? e0 : e1) : (s0 ? ee : B2), s0 == s1 ? (s0 ? e1 : e0) : (s0 ? B2 : ee),
                                  tb.log);
    const double c2 = r1 ? 1.0 / 6.0 : 1.0 / 3.0, c4 = r1 ? -3.0 / 40.0 : 3.0 / 40.0, c43 = r1 ? -0.025 : 0.025;
    const double c3 = r1 ? 0.0 : -0.25, c3h = r1 ? 0.0 : -0.125;
    const double c5 = r1 ? 0.025 : -1.0 / 120.0, c5h = r1 ? 0.0125 : -1.0 / 240.0, c54 = r1 ? 0.00625 : -1.0 / 480.0,
                 c538 = r1 ? 0.009375 : -0.003125;
    const double al = fma(c4, fma(2.0, D2, a2), c2), be = fma(c5h, fma(0.75, B2, D2), c3h);
    const double H = fma(D2, fma(c5, D2, c3), B2 * fma(c538, B2, fma(c5h, D2, c3h)));
    const double t0 = T0 * T0, t1 = T1 * T1;
    const double g0 = fma(Q0, fma(c54, B2 + t0, be), fma(c43, t0, al)), g1 = fma(Q1, fma(c54, B2 + t1, be), fma(c43, t1, al));
    const double E = fma(H, dash, fma(T1, g1, -T0 * g0));
    return fma(p.sD[f] * a, E, fma(r1 ? p.S[0][f] : p.S[1][f], psi, (r1 ? p.C[0][f] : p.C[1][f]) * theta));
}

__device__ __noinline__ double fw_eval_far(const FwPair &p, const FwTab &tb, int i, bool full)
{
    const FwQueue &q = p.far;
    const double a = q.a[i], T0 = q.T0[i], T1 = q.T1[i], a2 = fma(a, a, 1e-280);
    const int f = q.code[i] & 255;
    double theta, psi;
    if (!full) return p.C[2][f] * angle64(a * (T1 - T0), fma(T0, T1, a2), tb.atan);   // S_3 = 0
    const double D = p.D[f];
    fw_angles(tb, a, a2, D, D * D, T0, q.Q0[i], T1, q.Q1[i], theta, psi);
    return fma(p.S[2][f], psi, p.C[2][f] * theta);
}

// Append this lane's portion (if has) to ring q of n entries from head.
__device__ __forceinline__ void fw_push(FwQueue &q, int head, int &n, bool has, double a, double T0, double Q0,
                                        double T1, double Q1, int code)
{
    const unsigned m = __ballot_sync(0xffffffffu, has);
    if (has) {
        const int pos = (head + n + __popc(m & ((1u << (threadIdx.x & 31)) - 1u))) & (FQ - 1);
        q.a[pos] = a;
        q.T0[pos] = T0;
        q.Q0[pos] = Q0;
        q.T1[pos] = T1;
        q.Q1[pos] = Q1;
        q.code[pos] = code;
    }
    n += __popc(m);
}

// Evaluate the queues' full warps (every entry when last), lane by entry.
__device__ __forceinline__ void fw_drain(FwPair &p, const FwTab &tb, int &hb, int &nb, int &ha, int &na, bool full,
                                         bool last, double &acc)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();
    while (nb >= 32 || (last && nb > 0)) {
        if (lane < nb) acc += fw_eval_near(p, tb, (hb + lane) & (FQ - 1));
        const int d = min(nb, 32);
        hb = (hb + d) & (FQ - 1);
        nb -= d;
    }
    while (na >= 32 || (last && na > 0)) {
        if (lane < na) acc += fw_eval_far(p, tb, (ha + lane) & (FQ - 1), full);
        const int d = min(na, 32);
        ha = (ha + d) & (FQ - 1);
        na -= d;
    }
    __syncwarp();
}

// C_r and S_r of the face at distance D, signed by sg: the coefficients of
// theta and psi in region r (complement form: those of K_3 - K).
__device__ __forceinline__ void fw_face(FwPair &p, int f, double D, bool full, double sg)
{
    const double D2 = D * D, D4 = D2 * D2, D6 = D4 * D2;
    const double P[3] = {D * fma(-3.0 / 40.0, D4, D2 * (1.0 / 6.0)),
                         D * fma(3.0 / 40.0, D4, fma(1.0 / 3.0, D2, -1.0 / 20.0)), D * (7.0 / 20.0)};
    const double S[3] = {D6 * (1.0 / 40.0), fma(-1.0 / 120.0, D6, fma(-0.25, D4, 1.0 / 60.0)), -0.25};
    const int rD = D < 1.0 ? 0 : (D < 2.0 ? 1 : 2);
    const double kD = rD == 0 ? P[0] + S[0] : (rD == 1 ? P[1] + S[1] : P[2] + S[2]);   // D K(D)
    p.D[f] = D;
    p.sD[f] = full ? sg * D : -sg * D;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const double C = r == rD ? -S[r] : P[r] - kD;
        p.C[r][f] = sg * (full ? C : 0.25 - C);
        p.S[r][f] = sg * (full ? S[r] : -0.25 - S[r]);
    }
}

__device__ __forceinline__ void fp64_pairs_warp(int64_t n, const int32_t *__restrict__ list,
                                                const int32_t *__restrict__ pi, const int32_t *__restrict__ pj,
                                                const double *__restrict__ x, const double *__restrict__ y,
                                                const double *__restrict__ z, const double *__restrict__ h,
                                                const double *__restrict__ gen, const double *__restrict__ radius,
                                                const int64_t *__restrict__ cfo, const int64_t *__restrict__ fvo,
                                                const PlaneD *__restrict__ plane, const EdgeD *__restrict__ edge,
                                                double *__restrict__ w)
{
    __shared__ FwPair pairs[FW_WARPS];
    __shared__ FwTab tb;
    for (int t = threadIdx.x; t < 65 + 128; t += blockDim.x) {
        if (t < 65) tb.atan[t] = kAtanTab[t];
        else tb.log[(t - 65) >> 1][(t - 65) & 1] = kLogTab[(t - 65) >> 1][(t - 65) & 1];
    }
    __syncthreads();
    const int wi = threadIdx.x >> 5, lane = threadIdx.x & 31, wpb = blockDim.x >> 5;   // wpb <= FW_WARPS
    FwPair &p = pairs[wi];
    for (int64_t t = blockIdx.x * (int64_t)wpb + wi; t < n; t += (int64_t)gridDim.x * wpb) {
        const int32_t code = list ? list[t] : ~(int32_t)t;
        const int64_t k = code >= 0 ? code : ~code;
        const int i = pi[k], j = pj[k];
        const double rx = x[i] - gen[3 * j], ry = y[i] - gen[3 * j + 1], rz = z[i] - gen[3 * j + 2];
        const double hh = h[i], ih = 1.0 / hh;
        const int64_t f0 = cfo[j];
        const int nface = (int)(cfo[j + 1] - f0);
        if (nface > FW_MAXF) {
            if (lane == 0) {
                double err;
                w[k] = code >= 0 ? pair_weight<double, false>(rx, ry, rz, hh, radius[j], f0, f0 + nface, fvo, plane,
                                                              edge, err)
                                 : pair_weight<double, true>(rx, ry, rz, hh, radius[j], f0, f0 + nface, fvo, plane,
                                                             edge, err);
            }
            continue;
        }
        // inside test over all faces, then the form
        bool ins = nface > 0;   // nothing lies in a cell without faces: it weighs 0
        if (code >= 0)
            for (int f = lane; f < nface; f += 32) {
                const PlaneD pl = plane[f0 + f];
                ins = ins && !(pl.w - (pl.x * rx + pl.y * ry + pl.z * rz) < 0.0);
            }
        ins = __all_sync(0xffffffffu, ins);
        const bool full = code < 0 || (ins && sqrt(rx * rx + ry * ry + rz * rz) + radius[j] < 2.0 * hh);
        // faces: distance, coefficients, and how many edges each contributes
        if (lane == 0) p.pre[0] = 0;   // also where there is no face (a cell that a range build left out)
        __syncwarp();
        for (int base = 0; base < nface; base += 32) {
            const int f = base + lane;
            int cnt = 0;
            if (f < nface) {
                const PlaneD pl = plane[f0 + f];
                const double sd = pl.w - (pl.x * rx + pl.y * ry + pl.z * rz);
                const double D = fabs(sd) * ih;
                fw_face(p, f, D, full, sd > 0.0 ? 1.0 : -1.0);
                p.E0[f] = fvo[f0 + f];
                if (!(sd == 0.0 || (!full && D >= 2.0))) cnt = (int)(fvo[f0 + f + 1] - fvo[f0 + f]);
            }
            int xs = cnt;   // inclusive scan of the edge counts over these 32 faces
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, xs, o);
                if (lane >= o) xs += y;
            }
            const int carry = p.pre[base];
            if (f < nface) p.pre[f + 1] = carry + xs;
            __syncwarp();
        }
        const int ne = p.pre[nface];
        double acc = 0.0;
        int hb = 0, nb = 0, ha = 0, na = 0;
        for (int base = 0; base < ne; base += 32) {
            const int e = base + lane;
            double a = 0.0, T1 = 0.0, Q1 = 0.0, B2 = 0.0, cur = 0.0, Qc = 0.0;
            float t1f = 0.f, t2f = 0.f, T1f = 0.f;
            int f = 0;
            // where the rest of the edge starts: 0 before -t2, 1 before -t1,
            // 2 before t1, 3 before t2, 4 beyond; 5: nothing left
            int st = 5;
            if (e < ne) {
                int hi = nface;   // pre[f] <= e < pre[hi]
                while (hi - f > 1) {
                    const int mid = (f + hi) >> 1;
                    if (p.pre[mid] <= e) f = mid;
                    else hi = mid;
                }
                const EdgeD E = edge[p.E0[f] + (e - p.pre[f])];
                a = (E.cm - (E.mx * rx + E.my * ry + E.mz * rz)) * ih;
                cur = (E.ce - (E.ex * rx + E.ey * ry + E.ez * rz)) * ih;
                T1 = fma(E.L, ih, cur);
                const double D = p.D[f];
                B2 = fma(D, D, fma(a, a, 1e-280));
                Qc = sqrt64(fma(cur, cur, B2));
                Q1 = sqrt64(fma(T1, T1, B2));
                const float B2f = f32_cut(B2), T0f = f32_cut(cur);
                T1f = f32_cut(T1);
                t1f = B2f < 1.f ? sqrtf(1.f - B2f) : 0.f;
                t2f = B2f < 4.f ? sqrtf(4.f - B2f) : 0.f;
                if (a != 0.0 && E.L > 0.0)
                    st = T0f >= t2f ? 4 : (T0f >= t1f ? 3 : (T0f >= -t1f ? 2 : (T0f >= -t2f ? 1 : 0)));
            }
            // one portion per lane and pass, until every lane's edge is done
            while (__any_sync(0xffffffffu, st < 5)) {
                const bool has = st < 5;
                if (st == 0 && t2f == 0.f) st = 4;
                if (st == 1 && t1f == 0.f) st = 3;
                const int reg = st == 2 ? 1 : ((st == 1 || st == 3) ? 2 : 3);
                const float bpf = st == 0 ? -t2f : (st == 1 ? -t1f : (st == 2 ? t1f : t2f));
                const bool cross = st < 4 && bpf < T1f;
                double end = T1, Qe = Q1;
                if (cross) {
                    const bool at1 = st == 1 || st == 2;
                    const double tb2 = sqrt64(fmax((at1 ? 1.0 : 4.0) - B2, 0.0));
                    end = st < 2 ? -tb2 : tb2;
                    Qe = at1 ? 1.0 : 2.0;
                }
                fw_push(p.near, hb, nb, has && reg < 3, a, cur, Qc, end, Qe, f | (reg << 8));
                fw_push(p.far, ha, na, has && reg == 3, a, cur, Qc, end, Qe, f | (reg << 8));
                cur = end;
                Qc = Qe;
                st = cross ? st + 1 : 5;
                if (nb >= 32 || na >= 32) fw_drain(p, tb, hb, nb, ha, na, full, false, acc);
            }
        }
        fw_drain(p, tb, hb, nb, ha, na, full, true, acc);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) {
            const double s = acc * Consts<double>::inv_pi;
            w[k] = full ? s : ((ins ? 1.0 : 0.0) - s);
        }
        __syncwarp();
    }
}

// the flagged pairs of the mixed pass; the count is read on the device, so
// the launch needs no host synchronisation (grid-stride loop)
__global__ void __launch_bounds__(32 * FW_WARPS) k_map_fp64_flagged(
    const int *__restrict__ nflag, const int32_t *__restrict__ pi, const int32_t *__restrict__ pj,
    const double *__restrict__ x, const double *__restrict__ y, const double *__restrict__ z,
    const double *__restrict__ h, const double *__restrict__ gen, const double *__restrict__ radius,
    const int64_t *__restrict__ cfo, const int64_t *__restrict__ fvo, const PlaneD *__restrict__ plane,
    const EdgeD *__restrict__ edge, const int32_t *__restrict__ list, double *__restrict__ w)
{
    fp64_pairs_warp(*nflag, list, pi, pj, x, y, z, h, gen, radius, cfo, fvo, plane, edge, w);
}

// every pair, full form (the FP64 mode)
__global__ void __launch_bounds__(32 * FW_WARPS) k_map_fp64(
    int64_t npairs, const int32_t *__restrict__ pi, const int32_t *__restrict__ pj, const double *__restrict__ x,
    const double *__restrict__ y, const double *__restrict__ z, const double *__restrict__ h,
    const double *__restrict__ gen, const double *__restrict__ radius, const int64_t *__restrict__ cfo,
    const int64_t *__restrict__ fvo, const PlaneD *__restrict__ plane, const EdgeD *__restrict__ edge,
    double *__restrict__ w)
{
    fp64_pairs_warp(npairs, nullptr, pi, pj, x, y, z, h, gen, radius, cfo, fvo, plane, edge, w);
}

// FP32 bulk pass (quadrature form, see quad32.cuh).
//
// A warp maps 32 consecutive pairs (mostly of one cell, since pairs are
// sorted by cell), one pair per lane for the geometry: per face the plane
// distance D in float-float and an FP32 pass for the reference R = distance
// from p to the face polygon (any value used consistently for the face is
// exact when P is outside the polygon; inside, R = D), then R, 2 - R, K(R)
// and K(1) - K(R) in FP32; per edge A, T0, T1 and B^2 in float-float, and from
// them the segments' Q^2 - R^2 and 4 - Q^2, each rounded once to FP32.  The
// FP64 pipe runs at 1/64 of the FP32 rate, so nothing per face, edge or
// quadrature segment touches it: the pieces are summed in float-float.
//
// Each edge yields up to four quadrature segments (one for most), which the
// lane appends to its column of a per-warp queue in shared memory; whenever a
// lane's column may overflow, the warp evaluates all queued segments together,
// one 6-node slot (a 6-point segment, or half of a 12-point sub-piece) per
// lane, so that the node loop runs with the warp converged whatever the pairs'
// geometry.  Each lane then adds its own segments' results in a fixed order,
// which keeps the result bit-reproducible.  The queue is small (9 KB per
// warp) so that 12 two-warp blocks fit an SM: the pass is bound by instruction
// issue, and the warps hide its latencies.  The estimated error 8 eps times
// the sum of the magnitudes of the non-negative pieces flags the pair for the
// FP64 pass when it exceeds max(tol |w|, 1e-14) (relative accuracy tol for
// every weight above 1e-14 / tol, absolute 1e-14 below); so does a face plane
// through P.
//
// 24.06 M pairs of the 1e6-particle cloud: 63.8 ms (3.8e8 pairs/s), against
// 111 ms with 4- and 8-point rules in s = asinh(tau / A), an asinh per
// segment and an exponential per node, the two sides of every edge queued in
// turn, and correctly rounded or subnormal-safe reciprocals; the error against
// FP64 fell from 2.5e-7 to 2.4e-7 RMS.
namespace {

// factor of the FP32 pass's error estimate: fp32_err_ulps units of 2^-24
// (0 stands for the default 8)
double em_est_k(const em_params *p)
{
    return (double)(p->fp32_err_ulps > 0 ? p->fp32_err_ulps : 8) * 5.9604644775390625e-8;
}

// launch shape of the FP32 pass (build-time tuning knobs)
#ifndef EM_MQ_SLOTS
#define EM_MQ_SLOTS 6
#endif
#ifndef EM_MQ_WARPS
#define EM_MQ_WARPS 2
#endif
#ifndef EM_MQ_MINB
// minimum resident blocks per SM asked of the compiler (0: none): 12 two-warp
// blocks, 24 warps, is what the shared memory of 12 queues allows (18.2 KB a
// block), and caps the registers at 80 without spills
#define EM_MQ_MINB 12
#endif
constexpr int MQ_SLOTS = EM_MQ_SLOTS;   // segments a lane holds between evaluations (>= 5)
constexpr int MQ_WARPS = EM_MQ_WARPS;   // warps per block
constexpr int MQ_CHUNK = 64;            // sub-piece results a warp holds between accumulations
static_assert(MQ_SLOTS >= 5, "an edge queues up to four segments");
static_assert(MQ_CHUNK % 32 == 0, "whole rounds of the warp");
// a lane holds at most MQ_SLOTS segments of at most 2 x 28 slots each (m <= 28)
constexpr int MQ_NOSLOT = 4095;
static_assert(MQ_SLOTS * 56 < MQ_NOSLOT, "slot indices fit in 12 bits");
constexpr unsigned FULL_MASK = 0xffffffffu;
constexpr unsigned MQ_EDGE_DONE = 32;   // mq_edge: every segment of the edge is queued

struct SegQueue {
    float ts[MQ_SLOTS][32], len[MQ_SLOTS][32], A[MQ_SLOTS][32];
    float B2[MQ_SLOTS][32], c4s[MQ_SLOTS][32], es[MQ_SLOTS][32], Rr[MQ_SLOTS][32], vv[MQ_SLOTS][32];
    float add[MQ_SLOTS][32], scale[MQ_SLOTS][32];
    // m | piece1 | tilde | six (quad32.cuh) in the low 16 bits; during a
    // flush, the index of the segment's first slot among its lane's
    // in bits 16-27 (MQ_NOSLOT for an empty row)
    int meta[MQ_SLOTS][32];
    float vhi[MQ_CHUNK], vlo[MQ_CHUNK];   // scale * integral of each evaluated slot (float-float)
    int pre[33];
};

// Evaluate every queued segment of the warp and add each lane's results to
// its pair.  Called with the warp converged.  The work is spread by
// slot (6 quadrature nodes: a 6-point segment, or half of a 12-point
// sub-piece): lane L's segments hold M_L slots in queue order, the warp
// numbers all of them L by L and evaluates them 32 at a time, whoever owns
// them, so that a segment cut into many sub-pieces does not hold up the
// lanes.  Each result, times its segment's signed factor, is
// kept exactly as a float-float product; the owner then adds its own results
// in order into its float-float sum, which
// keeps the sum bit-reproducible, and their magnitudes in FP32: they only
// scale the error bound.
__device__ __forceinline__ void mq_flush(SegQueue &q, int lane, int cnt, emq::ff &acc, float &mag)
{
    int M = 0;
#pragma unroll
    for (int sl = 0; sl < MQ_SLOTS; ++sl) {
        const int mt = q.meta[sl][lane] & 0xffff;
        q.meta[sl][lane] = mt | ((sl < cnt ? M : MQ_NOSLOT) << 16);
        if (sl < cnt) M += (mt & emq::SEG_SIX) ? 1 : 2 * (mt & 255);   // 6-point: 1 slot, 12-point: 2 per sub-piece
    }
    int x = M;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(FULL_MASK, x, o);
        if (lane >= o) x += y;
    }
    const int total = __shfl_sync(FULL_MASK, x, 31);
    q.pre[lane + 1] = x;
    if (lane == 0) q.pre[0] = 0;
    __syncwarp();
    const int mine0 = x - M;   // this lane's slots are [mine0, x)
    for (int c0 = 0; c0 < total; c0 += MQ_CHUNK) {
        const int c1 = min(total, c0 + MQ_CHUNK);
        for (int t = c0 + lane; t < c1; t += 32) {
            int lo = 0, hi = 32;   // pre[lo] <= t < pre[hi]
#pragma unroll
            for (int it = 0; it < 5; ++it) {
                const int mid = (lo + hi) >> 1;
                if (q.pre[mid] <= t) lo = mid;
                else hi = mid;
            }
            const int r = t - q.pre[lo];
            int sl = 0;
#pragma unroll
            for (int k = 1; k < MQ_SLOTS; ++k) sl += (q.meta[k][lo] >> 16) <= r ? 1 : 0;
            const int mw = q.meta[sl][lo];
            const int rr = r - (mw >> 16);
            const int mt = mw & 0xffff;
            const bool six = (mt & emq::SEG_SIX) != 0;
            const float val = emq::slot_eval(six ? 0 : rr >> 1, six ? 0 : 1 + (rr & 1), q.ts[sl][lo], q.len[sl][lo],
                                             q.A[sl][lo], q.B2[sl][lo], q.c4s[sl][lo], q.es[sl][lo], q.Rr[sl][lo],
                                             q.vv[sl][lo], q.add[sl][lo], mt);
            const emq::ff v = emq::ff_two_prod(q.scale[sl][lo], val);
            q.vhi[t - c0] = v.hi;
            q.vlo[t - c0] = v.lo;
        }
        __syncwarp();
        const int e1 = min(x, c1);
        for (int t = max(mine0, c0); t < e1; ++t) {
            // (the low parts' sum needs no renormalisation: its rounding is 2^-48 of the magnitudes)
            const emq::ff s2 = emq::ff_two_sum(acc.hi, q.vhi[t - c0]);
            acc.hi = s2.hi;
            acc.lo += s2.lo + q.vlo[t - c0];
            mag += fabsf(q.vhi[t - c0]);
        }
        __syncwarp();
    }
}

// Face constants of the lane's current face.
struct FaceState {
    emq::ff D2, R2;             // D^2 and R^2 (float-float, units of h)
    float Df, R, v, KR, C1;     // v = 2 - R
    float sign;   // orientation of the face as seen from P (sign of the signed distance)
};

// Face constants from R^2 (float-float): R, v = 2 - R, K(R) (or K~(R)) and,
// for R < 1, K(1) - K(R), in FP32.  Each is written so that no sum cancels:
// 1 - R^2 and 4 - R^2 in float-float, and for R < 1 the polynomials in
// x = 1 - R with integer coefficients (times 120), where
//   K1(1) - K1(R) = (1 - R^2) P / 120,  P = 8 + 6x - 3x^3 + 3/(1 + R),
//   K1(R) = R^2 (14 + 9x - 3x^3) / 120,
//   K~1(1) - K~1(R) = (1 - R^2) N / (120 R (1 + R)),
//   N = 11 + 15x + 10x^2 - 9x^4 + 3x^5,
// sums whose terms are at most 1.6 times their value, so each constant comes
// out within a few ulp.
__device__ __forceinline__ void face_consts(emq::ff R2x, bool tilde, FaceState &fs)
{
    const float R2 = R2x.hi + R2x.lo;
    const float R = sqrtf(R2);
    const float iR = R > 0.f ? __frcp_rn(R) : 0.f;
    fs.R = R;
    if (R < 1.f) {
        const emq::ff omx = emq::ff_add(emq::ff{1.f, 0.f}, emq::ff_neg(R2x));
        const float om = (omx.hi + omx.lo) * (1.f / 120.f);
        const float x = 1.f - R;
        const float i1 = __frcp_rn(1.f + R);
        fs.v = 2.f - R;
        if (tilde) {
            const float N = fmaf(x, fmaf(x, fmaf(x * x, fmaf(3.f, x, -9.f), 10.f), 15.f), 11.f);
            const float c1 = om * (N * iR * i1);
            fs.C1 = c1;
            fs.KR = -(1.f / 60.f) - c1;
        } else {
            const float P = fmaf(x, fmaf(-3.f * x, x, 6.f), 8.f) + 3.f * i1;
            fs.C1 = om * P;
            fs.KR = R2 * fmaf(x, fmaf(-3.f * x, x, 9.f), 14.f) * (1.f / 120.f);
        }
        return;
    }
    fs.C1 = 0.f;
    // K(R) = 7/20 - 1/(4R) - K~2(R) for R >= 1, with 7/20 - 1/(4R) = (7R - 5)/(20R)
    const float k3 = fmaf(7.f, R, -5.f) * iR * 0.05f;
    if (R >= 2.f) {
        fs.v = 0.f;
        fs.KR = tilde ? 0.f : k3;
        return;
    }
    const emq::ff fmx = emq::ff_add(emq::ff{4.f, 0.f}, emq::ff_neg(R2x));
    const float v = (fmx.hi + fmx.lo) * __frcp_rn(2.f + R);
    const float v2 = v * v;
    const float kt2 = -(v2 * v2) * v * (1.f + R) * iR * (1.f / 120.f);
    fs.v = v;
    fs.KR = tilde ? kt2 : k3 - kt2;
}

// Queue one segment of an edge: tau from t (float-float) over length len (from
// accurate offsets, see mq_edge) on kernel piece `piece`, with signed factor sc.
// The nodes lie at offsets from t rounded to FP32, but Q^2 - Rr^2 and 4 - Q^2
// are taken at t itself: t's rounding, 6e-8, would shift a segment of length
// 0.05 against its neighbours by a millionth of itself.
__device__ __forceinline__ void mq_push(SegQueue &q, int lane, int sl, int piece, emq::ff t, float len, float A,
                                        float A2, float B2f, emq::ff B2, float sc, const FaceState &fs, bool tilde)
{
    const bool ref1 = piece == 2 && fs.R < 1.f;   // difference split at Q = 1
    // eta^2 = len^2 / r2 chooses the rule (quad32.cuh)
    const float ts = t.hi, r2 = fmaf(ts, ts, A2), l2 = len * len;
    const bool six = l2 <= emq::SIX_ETA * emq::SIX_ETA * r2;
    int m = 1;
    if (l2 > emq::TWELVE_ETA * emq::TWELVE_ETA * r2) {
        // m <= 28: A >= 1e-18, tau <= 2
        const float te = ts + len;
        const float e = __logf((te + emq::sqrt_nr(fmaf(te, te, A2))) * emq::rcp_a(ts + emq::sqrt_nr(r2)));
        m = max(1, min(28, (int)ceilf(e * (1.f / emq::SUB_LOG))));
    }
    // Q^2 at t, then Q^2 - Rr^2 and 4 - Q^2 there, each a float-float
    // difference rounded once
    emq::ff t2 = emq::ff_two_prod(ts, ts);
    t2.lo = fmaf(2.f * ts, t.lo, t2.lo);
    const emq::ff Q2 = emq::ff_add(B2, t2);
    q.ts[sl][lane] = ts;
    q.len[sl][lane] = len;
    q.A[sl][lane] = A;
    q.B2[sl][lane] = B2f;
    q.c4s[sl][lane] = emq::ff_diff(emq::ff{4.f, 0.f}, Q2);
    q.es[sl][lane] = emq::ff_diff(Q2, ref1 ? emq::ff{1.f, 0.f} : fs.R2);
    q.Rr[sl][lane] = ref1 ? 1.f : fs.R;
    q.vv[sl][lane] = ref1 ? 1.f : fs.v;
    q.add[sl][lane] = ref1 ? fs.C1 : 0.f;
    q.scale[sl][lane] = sc;
    q.meta[sl][lane] = m | (piece == 1 ? emq::SEG_PIECE1 : 0) | (tilde ? emq::SEG_TILDE : 0) | (six ? emq::SEG_SIX : 0);
}

// Queue the kernel pieces of (D/pi) int over tau in [T0, T1] of one edge, with
// the signed factor sc; the part beyond 2h is added directly.  The integrand
// is even in tau, so a range on one side of the foot is taken as [ua, ua + du],
// ua >= 0.  du is from an accurate difference (the edge length L/h, or |T| for
// a range that starts at the foot), and so is every segment's length: offsets
// of the breakpoints from ua, then differences of offsets.  Forming a length
// as a difference of two tau of size ~1 instead would carry an absolute error
// of 2^-24, tens of ulps of a short segment (a small face seen from afar).
// A breakpoint itself may be off by a few ulp: K's pieces agree to fourth
// order there, and both sides use the same offset.
// A range across the foot is taken as its two sides.  Most edges yield one
// segment: the loop runs once for each that the warp's busiest lane has, with
// the lanes converged.
__device__ __forceinline__ void mq_edge(SegQueue &q, int lane, int &cnt, unsigned &queued, emq::ff T0x,
                                        emq::ff T1x, float dT, float A, emq::ff B2, float sc, const FaceState &fs, bool tilde, emq::ff &acc,
                                        float &mag)
{
    const float A2 = A * A, B2f = fmaxf(B2.hi, A2);
    const float c1 = emq::ff_diff(emq::ff{1.f, 0.f}, B2), c4 = emq::ff_diff(emq::ff{4.f, 0.f}, B2);
    const float t1 = c1 > 1e-30f ? c1 * emq::rsqrt_a(c1) : 0.f;
    const float t2 = c4 > 1e-30f ? c4 * emq::rsqrt_a(c4) : 0.f;
    const float T0 = T0x.hi, T1 = T1x.hi;
    const bool foot = T0 < 0.f && T1 > 0.f;
    const float ua = foot ? 0.f : (T0 >= 0.f ? T0 : -T1), ualo = foot ? 0.f : (T0 >= 0.f ? T0x.lo : -T1x.lo);
    const float du = foot ? T1 : dT;      // this side, from ua
    const float xo = foot ? -T0 : 0.f;    // the other side of the foot, from 0
    const float o1 = t1 - ua, o2 = t2 - ua;
    // pieces: piece 1 on offsets [0, e1], piece 2 on [s2, e2]
    const float e1 = fminf(du, o1), s2 = fmaxf(0.f, o1), e2 = fminf(du, o2);
    // the other side's: piece 1 up to x1, piece 2 from t1 to x2
    const float x1 = fminf(xo, t1), x2 = fminf(xo, t2);
    unsigned todo = (e1 > 0.f ? 1u : 0u) | (e2 > s2 ? 2u : 0u) | (x1 > 0.f ? 4u : 0u) | (x2 > t1 ? 8u : 0u);
    const bool first = queued == 0;   // the part beyond 2h is added once
    todo &= ~queued;
    while (todo && cnt < MQ_SLOTS) {
        const int k = __ffs(todo) - 1;
        todo &= todo - 1;
        queued |= 1u << k;
        // start: ua, ua + s2, 0 or t1
        emq::ff t = emq::ff_two_sum(k < 2 ? ua : 0.f, k == 1 ? s2 : (k == 3 ? t1 : 0.f));
        if (k < 2) t.lo += ualo;
        const float len = k == 0 ? e1 : (k == 1 ? e2 - s2 : (k == 2 ? x1 : x2 - t1));
        mq_push(q, lane, cnt++, (k & 1) ? 2 : 1, t, len, A, A2, B2f, B2, sc, fs, tilde);
    }
    queued = todo ? queued | 16u : MQ_EDGE_DONE;
    if (tilde && first) {   // beyond 2h: K~(Q) = 0, the integrand is -K~(R) >= 0
        auto far = [&](float u, float l) {   // tau from u over length l
            const emq::ff v = emq::ff_two_prod(sc, -fs.KR * emq::angle_q1(l * A, fmaf(u, u + l, A2)));
            const emq::ff s = emq::ff_two_sum(acc.hi, v.hi);
            acc.hi = s.hi;
            acc.lo += s.lo + v.lo;
            mag += fabsf(v.hi);
        };
        if (du > o2) far(fmaxf(ua, t2), o2 > 0.f ? du - o2 : du);
        if (xo > t2) far(t2, xo - t2);
    }
}

}  // namespace

// Launch shapes of the FP32 pass (em_params.fp32_variant, map_autotune):
// warps per block and the minimum resident blocks per SM asked of the
// compiler (0: none).  Variant 0 is the default shape; the others trade
// registers (no minimum: 92-94) against warps per SM.
constexpr int MQ_NVARIANT = 4;
constexpr int MQ_VARIANT_WARPS[MQ_NVARIANT] = {MQ_WARPS, 1, 4, 2};
constexpr int MQ_VARIANT_MINB[MQ_NVARIANT] = {EM_MQ_MINB, 0, 6, 0};

template <int WARPS, int MINB>
__global__ void __launch_bounds__(32 * WARPS, MINB) k_map_fp32(int64_t npairs, const int32_t *__restrict__ pi,
                                                        const int32_t *__restrict__ pj, const double *__restrict__ x,
                                                        const double *__restrict__ y, const double *__restrict__ z,
                                                        const double *__restrict__ h, const double *__restrict__ gen,
                                                        const double *__restrict__ radius,
                                                        const int64_t *__restrict__ cfo, const int64_t *__restrict__ fvo,
                                                        const PlaneF *__restrict__ plane_f,
                                                        const PlaneF *__restrict__ plane_fl,
                                                        const EdgeF *__restrict__ edge_f,
                                                        const EdgeF *__restrict__ edge_fl, float tol, double est_k,
                                                        double *__restrict__ w, int32_t *__restrict__ flagged,
                                                        int *__restrict__ nflag)
{
    __shared__ SegQueue queues[WARPS];
    SegQueue &q = queues[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t k0 = (blockIdx.x * (int64_t)WARPS + (threadIdx.x >> 5)) * 32;
    if (k0 >= npairs) return;   // the whole warp
    const int64_t k = k0 + lane;
    const bool valid = k < npairs;

    double rx = 0.0, ry = 0.0, rz = 0.0, hh = 1.0, rad = 0.0;
    int64_t f = 0, f1 = 0;
    if (valid) {
        const int i = pi[k], j = pj[k];
        rx = x[i] - gen[3 * j];
        ry = y[i] - gen[3 * j + 1];
        rz = z[i] - gen[3 * j + 2];
        hh = h[i];
        f = cfo[j];
        f1 = cfo[j + 1];
        rad = radius[j];
    }
    const double ih = 1.0 / hh;
    // float-float copies of r = p - g and 1/h for the plane and edge geometry,
    // and their FP32 roundings
    const emq::ff rxx = emq::ff_from_double(rx), ryy = emq::ff_from_double(ry), rzz = emq::ff_from_double(rz);
    const emq::ff ihh = emq::ff_from_double(ih);
    const float rxf = rxx.hi, ryf = ryy.hi, rzf = rzz.hi, ihf = ihh.hi;
    // signed distance c - n.r of P from face g's plane (positive inside), in
    // float-float; the inside test and the faces' orientations below both
    // take their signs from this one value
    auto plane_dist = [&](int64_t g) {
        const PlaneF H = plane_f[g], Lo = plane_fl[g];
        return emq::ff_offset_dot(H.w, Lo.w, H.x, Lo.x, H.y, Lo.y, H.z, Lo.z, rxx, ryy, rzz);
    };
    // the full kernel applies when P is inside a cell that lies entirely
    // within 2h of it; otherwise the complement form, and whether P is inside
    // is read off the face loop's own plane distances
    bool inside = f1 > f, full = false;   // nothing lies in a cell without faces: it weighs 0
    if (valid && sqrt(rx * rx + ry * ry + rz * rz) + rad < 2.0 * hh) {
        for (int64_t g = f; g < f1; ++g) inside = inside && !(plane_dist(g).hi < 0.f);
        full = inside;
    }
    const bool tilde = !full;

    // the quadrature's results are added in the order of the lane's own
    // segments (mq_flush), the angles beyond 2h in the order of its edges, each
    // into its own sum: neither order depends on when the warp flushes, so a
    // pair's weight does not depend on the other pairs of its warp
    emq::ff acc{0.f, 0.f}, acc_far{0.f, 0.f};
    float mag = 0.f, mag_far = 0.f;
    bool force = false;   // the FP32 form does not apply: recompute in FP64
    int cnt = 0;   // segments queued by this lane
    const int nface = valid ? (int)(f1 - f) : 0;
    // faces and edges in lockstep across the warp: consecutive pairs mostly
    // share their cell, so the per-face geometry runs with the lanes converged
    // One pass more than the warp has faces, with one empty edge, evaluates
    // what is left: the flush has a single call site, so that a slot's result
    // cannot depend on which copy of the code (the compiler may round two
    // copies differently) evaluated it, that is on the other pairs of the warp.
    for (int fi = 0;; ++fi) {
        const bool last = !__any_sync(FULL_MASK, fi < nface);
        int64_t e0 = 0;
        int ne = 0;
        FaceState fs{};
        if (fi < nface) {
            const int64_t g = f + fi;
            const emq::ff sd = plane_dist(g);
            inside = inside && !(sd.hi < 0.f);
            const emq::ff D = emq::ff_mul(sd.hi < 0.f ? emq::ff_neg(sd) : sd, ihh);
            // P in (or next to) the face plane: in the complement form such a
            // face would carry half of the kernel
            if (tilde && D.hi < 1e-15f) force = true;
            const bool beyond = D.hi > 2.f || (D.hi == 2.f && D.lo >= 0.f);
            if (!(sd.hi == 0.f || (tilde && beyond))) {
                // reference distance to the polygon (FP32)
                const int64_t g0 = fvo[g], g1 = fvo[g + 1];
                bool inpoly = true;
                float rho2 = INFINITY;
                for (int64_t q1 = g0; q1 < g1; ++q1) {
                    EdgeF E = edge_f[q1];
                    float a = (E.cm - (E.mx * rxf + E.my * ryf + E.mz * rzf)) * ihf;
                    float t0 = (E.ce - (E.ex * rxf + E.ey * ryf + E.ez * rzf)) * ihf;
                    float t1 = t0 + E.L * ihf;
                    inpoly = inpoly && a > 0.f;
                    float tc = t0 > 0.f ? t0 : (t1 < 0.f ? t1 : 0.f);
                    rho2 = fminf(rho2, a * a + tc * tc);
                }
                const float rr2 = inpoly ? 0.f : rho2;
                fs.D2 = emq::ff_mul(D, D);
                fs.R2 = emq::ff_add(fs.D2, emq::ff{rr2, 0.f});
                const bool far = fs.R2.hi > 4.f || (fs.R2.hi == 4.f && fs.R2.lo >= 0.f);
                if (!(tilde && far)) {   // else the polygon lies entirely beyond 2h
                    fs.Df = D.hi;
                    face_consts(fs.R2, tilde, fs);
                    fs.sign = sd.hi > 0.f ? 1.f : -1.f;
                    e0 = g0;
                    ne = (int)(g1 - g0);
                }
            }
        }
        unsigned queued = 0;   // of the lane's current edge: the segments queued (mq_edge)
        for (int ei = 0; last ? ei == 0 : __any_sync(FULL_MASK, ei < ne);) {
            if (ei < ne && queued != MQ_EDGE_DONE) {
                // edge geometry in float-float (see quad32.cuh): A, T0, T1 and
                // B^2, each rounded once to FP32 where it is used so
                const EdgeF H = edge_f[e0 + ei], Lo = edge_fl[e0 + ei];
                const emq::ff2 at = emq::ff2_mul(emq::edge_offsets(H, Lo, rxx, ryy, rzz), ihh);
                const emq::ff a{at.hi.x, at.lo.x};
                if (a.hi != 0.f) {
                    const emq::ff t0{at.hi.y, at.lo.y};
                    const emq::ff lh = emq::ff_mul(emq::ff{H.L, Lo.L}, ihh);   // L/h
                    const emq::ff t1 = emq::ff_add(t0, lh);
                    // A below 1e-18 h changes the integral by ~1e-18 relative and would
                    // leave A^2 below FP32's normal range
                    const float A = fmaxf(fabsf(a.hi), 1e-18f);
                    // signed factor: D/pi, face orientation, side of the edge line
                    // (T1 >= T0: the edge runs along its direction)
                    const float sc = fs.sign * (a.hi > 0.f ? 1.f : -1.f) * fs.Df * 0.31830988618379067154f;
                    mq_edge(q, lane, cnt, queued, t0, t1, lh.hi, A, emq::ff_add(fs.D2, emq::ff_mul(a, a)), sc, fs,
                            tilde, acc_far, mag_far);
                } else {
                    queued = MQ_EDGE_DONE;
                }
            }
            // almost every edge queues one or two segments: the queue is evaluated
            // when a lane has no room for two (71.2 ms on the 1e6-particle cloud where
            // it was when a lane had no room for four, 70.2 so), and an edge that
            // found too little room is taken up again after that
            const bool rest = ei < ne && queued != MQ_EDGE_DONE;
            if (__any_sync(FULL_MASK, rest || cnt > (last ? 0 : MQ_SLOTS - 2))) {
                mq_flush(q, lane, cnt, acc, mag);
                cnt = 0;
            }
            if (!__any_sync(FULL_MASK, rest)) {
                queued = 0;
                ++ei;
            }
        }
        if (last) break;
    }
    bool flag = false;
    if (valid) {
        // the integrals were summed with their signs: w = sum (full kernel) or
        // [P inside] - sum (complement kernel)
        const emq::ff tot = emq::ff_add(acc, acc_far);
        const double sum = (double)tot.hi + (double)tot.lo;
        const double wk = full ? sum : ((inside ? 1.0 : 0.0) - sum);
        const double magd = (double)mag + (double)mag_far + ((inside && !full) ? 1.0 : 0.0);
        w[k] = wk;
        // error bound of the FP32 pass: est_k = (ulps) 2^-24 times the sum of
        // the non-negative pieces it summed.  With the default 8 ulps the
        // largest error against FP64 on the 1e5 and 1e6 clouds is 0.35 of the
        // bound where that is above 1e-5 |w|, 0.64 from 3e-6 to 1e-5 |w| (0.51
        // for tiny cells deep inside large kernels, h / V^(1/3) above 12); below
        // 1e-6 |w| it reaches 2.2 of it, 1.2e-6 |w|.  With 3 one of the 8e6
        // cloud's 145.6 M pairs misses the tolerance, with 4 none
        const double est = est_k * magd;
        flag = force || !(est <= fmax((double)tol * fabs(wk), 1e-14));
    }
    // one append per warp: the flagged pairs of a warp (mostly of one cell)
    // stay together in the list, which keeps the FP64 pass's warps coherent
    const unsigned fm = __ballot_sync(FULL_MASK, flag);
    if (fm) {
        int base = 0;
        if (lane == 0) base = atomicAdd(nflag, __popc(fm));
        base = __shfl_sync(FULL_MASK, base, 0);
        if (flag) flagged[base + __popc(fm & ((1u << lane) - 1u))] = force ? ~(int32_t)k : (int32_t)k;
    }
}

// rho_j = sum_i m_i w_ij / V_j over the cell's pairs (ascending i), one warp per cell
__global__ void k_cell_density(int64_t ncell, const int64_t *__restrict__ off, const int32_t *__restrict__ pi,
                               const double *__restrict__ w, const double *__restrict__ m,
                               const double *__restrict__ volume, double *__restrict__ rho)
{
    int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    if (warp >= ncell) return;
    double s = 0.0;
    for (int64_t k = off[warp] + lane; k < off[warp + 1]; k += 32) s += m[pi[k]] * w[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    // a cell without pairs has density 0 (also one a range build left without volume)
    if (lane == 0) rho[warp] = off[warp + 1] > off[warp] ? s / volume[warp] : 0.0;
}

// Sums over a particle's pairs, a row of the (i, j)-ordered transpose, in
// ascending j, each product and each sum rounded on its own (no fused
// multiply-add): den = sum w, and with f given, num = sum w f_j.  The order fixes
// the bits, so a row cannot be split.  MODE 0: out0 = den; 1: out0 = num / den;
// 2: out0 += num, out1 += den.
template <int MODE>
__device__ __forceinline__ void row_out(int64_t i, double num, double den, double *__restrict__ out0,
                                        double *__restrict__ out1)
{
    if (MODE == 0) out0[i] = den;
    else if (MODE == 1) out0[i] = num / den;
    else {
        out0[i] = __dadd_rn(out0[i], num);
        out1[i] = __dadd_rn(out1[i], den);
    }
}

// A row of up to EM_ROW_LONG pairs by one thread, PB pairs at a time in a
// pipeline: while one batch is added the next one's weights and values are on
// their way, and the cells and pair numbers of the two after that.  The two
// batches' registers take turns in the code: copying one that is still being
// loaded into another would wait for it.
constexpr int PB = 2;
template <int MODE>
__device__ __forceinline__ void short_row(int64_t i, int64_t k0, int n, const int32_t *__restrict__ idx,
                                          const int32_t *__restrict__ pj, const double *__restrict__ w,
                                          const double *__restrict__ f, double *__restrict__ out0,
                                          double *__restrict__ out1)
{
    constexpr bool WITH_F = MODE > 0;
    idx += k0;
    // the batch from c on; past the row's end its last pair is loaded again, and not added
    auto pairs = [&](int c, int32_t(&q)[PB]) {
#pragma unroll
        for (int u = 0; u < PB; ++u) q[u] = __ldg(idx + min(c + u, n - 1));
    };
    auto cells = [&](const int32_t(&q)[PB], int32_t(&j)[PB]) {
#pragma unroll
        for (int u = 0; u < PB; ++u) j[u] = WITH_F ? __ldg(pj + q[u]) : 0;
    };
    struct Batch {
        double w[PB], f[PB];
    };
    auto values = [&](const int32_t(&q)[PB], const int32_t(&j)[PB], Batch &x) {
#pragma unroll
        for (int u = 0; u < PB; ++u) {
            x.w[u] = __ldg(w + q[u]);
            x.f[u] = WITH_F ? __ldg(f + j[u]) : 0.0;
        }
    };
    double num = 0.0, den = 0.0;
    if (n > 0) {
        // the first batches' loads of a kind together: a row waits for three in all
        int32_t qa[PB], qb[PB], ja[PB], jb[PB], q0[PB], q1[PB], j[PB];
        Batch A, B;
        pairs(0, qa);
        pairs(PB, qb);
        pairs(2 * PB, q0);
        pairs(3 * PB, q1);
        cells(qa, ja);
        cells(qb, jb);
        cells(q0, j);
        values(qa, ja, A);
        values(qb, jb, B);
        // before the batch at c: q0, j of the one at c + 2 PB, q1 of the next
        auto step = [&](int c, Batch &x) {
#pragma unroll
            for (int u = 0; u < PB; ++u)
                if (c + u < n) {
                    if (WITH_F) num = __dadd_rn(num, __dmul_rn(x.w[u], x.f[u]));
                    den = __dadd_rn(den, x.w[u]);
                }
            if (c + 2 * PB < n) {
                values(q0, j, x);
                cells(q1, j);
#pragma unroll
                for (int u = 0; u < PB; ++u) q0[u] = q1[u];
                pairs(c + 4 * PB, q1);
            }
        };
#pragma unroll 1
        for (int c = 0; c < n; c += 2 * PB) {
            step(c, A);
            step(c + PB, B);
        }
    }
    row_out<MODE>(i, num, den, out0, out1);
}

// Up to 32 longer rows of like length (listed with the transpose) by a block.  An
// FP64 instruction takes a scheduler 64 cycles whatever its active lanes, so a
// long row among shorter ones, or a warp that both gathers and adds, is what
// makes a row of thousands of pairs the last to end.  One warp adds, each lane
// its own row's terms as they stand in shared memory; the other three gather a
// tile of LR_COLS pairs of every row at a time, multiply, and store it, with the
// next two tiles' weights and values, a third one's cells and a fourth one's pair
// numbers on their way.  The adding warp is another one from block to block,
// since a block's warps go to the four schedulers in turn.  It adds whole tiles
// without asking (with a test at every term 0.11 us a pair of the longest row, so
// 0.073, 0.062 of it the two additions' 128 cycles).
constexpr int SHORT_THREADS = 64, ROW_THREADS = 128, LR_COLS = 12, LR_PER = 4;
static_assert((ROW_THREADS - 32) * LR_PER == 32 * LR_COLS && (ROW_THREADS - 32) % LR_COLS == 0, "a tile's entries");
template <int MODE>
struct LongTile {
    double w[2][32][LR_COLS + 1];   // padded: lanes read down a column
    double p[MODE > 0 ? 2 : 1][MODE > 0 ? 32 : 1][LR_COLS + 1];
};
// the block's barrier, met by its two kinds of warps in different places
__device__ __forceinline__ void tile_sync() { asm volatile("bar.sync 0, %0;" ::"n"(ROW_THREADS) : "memory"); }
template <int MODE>
__device__ __forceinline__ void long_rows(LongTile<MODE> &sh, int nrow, const int32_t *__restrict__ rows,
                                          const int64_t *__restrict__ off, const int32_t *__restrict__ idx,
                                          const int32_t *__restrict__ pj, const double *__restrict__ w,
                                          const double *__restrict__ f, double *__restrict__ out0,
                                          double *__restrict__ out1)
{
    constexpr bool WITH_F = MODE > 0;
    const int lane = threadIdx.x & 31, adder = blockIdx.x & 3, wp = threadIdx.x >> 5;
    const int i = lane < nrow ? rows[lane] : -1;   // the same in every warp
    const int k0 = i >= 0 ? (int)off[i] : 0, n = i >= 0 ? (int)off[i + 1] - k0 : 0;   // pairs < 2^31
    const int tiles = (__reduce_max_sync(FULL_MASK, n) + LR_COLS - 1) / LR_COLS;
    if (wp == adder) {
        double num = 0.0, den = 0.0;
        tile_sync();
        for (int c = 0; c < tiles; ++c) {
            const int s = c & 1, m = n - c * LR_COLS;
            double wv[LR_COLS], pv[LR_COLS];
#pragma unroll
            for (int t = 0; t < LR_COLS; ++t) {
                wv[t] = sh.w[s][lane][t];
                pv[t] = WITH_F ? sh.p[s][lane][t] : 0.0;
            }
            if (m >= LR_COLS) {
#pragma unroll
                for (int t = 0; t < LR_COLS; ++t) {
                    if (WITH_F) num = __dadd_rn(num, pv[t]);
                    den = __dadd_rn(den, wv[t]);
                }
            } else if (m > 0) {
#pragma unroll
                for (int t = 0; t < LR_COLS; ++t)
                    if (t < m) {
                        if (WITH_F) num = __dadd_rn(num, pv[t]);
                        den = __dadd_rn(den, wv[t]);
                    }
            }
            tile_sync();
        }
        if (i >= 0) row_out<MODE>(i, num, den, out0, out1);
        return;
    }
    // entry u of this thread: row RSTEP u + sub, column col
    constexpr int RSTEP = (ROW_THREADS - 32) / LR_COLS;
    const int t = (wp - (wp > adder ? 1 : 0)) * 32 + lane, col = t % LR_COLS, sub = t / LR_COLS;
    int kr[LR_PER], nr[LR_PER];
#pragma unroll
    for (int u = 0; u < LR_PER; ++u) {
        kr[u] = __shfl_sync(FULL_MASK, k0, RSTEP * u + sub) + col;
        nr[u] = __shfl_sync(FULL_MASK, n, RSTEP * u + sub) - col;
    }
    // the tile's pair numbers (-1 past a row's end), their cells, weights and values
    auto pairs = [&](int c, int32_t(&q)[LR_PER]) {
#pragma unroll
        for (int u = 0; u < LR_PER; ++u) q[u] = c * LR_COLS < nr[u] ? __ldg(idx + kr[u] + c * LR_COLS) : -1;
    };
    auto cells = [&](const int32_t(&q)[LR_PER], int32_t(&j)[LR_PER]) {
#pragma unroll
        for (int u = 0; u < LR_PER; ++u) j[u] = WITH_F && q[u] >= 0 ? __ldg(pj + q[u]) : 0;
    };
    struct Part {
        double w[LR_PER], f[LR_PER];
    };
    auto values = [&](const int32_t(&q)[LR_PER], const int32_t(&j)[LR_PER], Part &x) {
#pragma unroll
        for (int u = 0; u < LR_PER; ++u) {
            x.w[u] = q[u] >= 0 ? __ldg(w + q[u]) : 0.0;
            x.f[u] = WITH_F && q[u] >= 0 ? __ldg(f + j[u]) : 0.0;
        }
    };
    int32_t qa[LR_PER], qb[LR_PER], ja[LR_PER], jb[LR_PER], q0[LR_PER], q1[LR_PER], j[LR_PER];
    Part A, B;   // take turns, as in short_row
    pairs(0, qa);
    pairs(1, qb);
    pairs(2, q0);
    pairs(3, q1);
    cells(qa, ja);
    cells(qb, jb);
    cells(q0, j);
    values(qa, ja, A);
    values(qb, jb, B);
    // before tile c: q0, j of tile c + 2, q1 of the next
    auto step = [&](int c, Part &x) {
        const int s = c & 1;
#pragma unroll
        for (int u = 0; u < LR_PER; ++u) {
            sh.w[s][RSTEP * u + sub][col] = x.w[u];
            if (WITH_F) sh.p[s][RSTEP * u + sub][col] = __dmul_rn(x.w[u], x.f[u]);
        }
        values(q0, j, x);
        cells(q1, j);
#pragma unroll
        for (int u = 0; u < LR_PER; ++u) q0[u] = q1[u];
        pairs(c + 4, q1);
        tile_sync();   // tile c is there; the adder has done with tile c - 1, whose place tile c + 1 takes
    };
#pragma unroll 1
    for (int c = 0; c < tiles; c += 2) {
        step(c, A);
        if (c + 1 < tiles) step(c + 1, B);
    }
    tile_sync();
}

// LONG: blocks below nlongb take the long rows, the longest first: 32 each, and
// ROW_FEW of those beyond ROW_VERY pairs, which then end sooner (24.04 M pairs
// with rows of up to 3,781: 569 us with 32 of any length, 466 so; 16.4 M with rows
// of up to 33,417: 2,834 and 2,451).
// SHORT: the other blocks take those of up to `longest` pairs, a row per thread.
template <int MODE, bool LONG, bool SHORT>
__global__ void __launch_bounds__(LONG ? ROW_THREADS : SHORT_THREADS, LONG ? 5 : 16)
    k_rows(int64_t np, int nlongb, int longest, const int *__restrict__ nlong, const int32_t *__restrict__ rows,
           const int64_t *__restrict__ off, const int32_t *__restrict__ idx, const int32_t *__restrict__ pj,
           const double *__restrict__ w, const double *__restrict__ f, double *__restrict__ out0,
           double *__restrict__ out1)
{
    if constexpr (LONG) {
        __shared__ LongTile<MODE> sh;
        if ((int)blockIdx.x < nlongb) {
            const int nl = nlong[0], nv = nlong[1], vb = (nv + ROW_FEW - 1) / ROW_FEW, b = blockIdx.x;
            const int g = b < vb ? b * ROW_FEW : nv + (b - vb) * 32, end = b < vb ? nv : nl;
            if (g < end)
                long_rows<MODE>(sh, min(b < vb ? ROW_FEW : 32, end - g), rows + g, off, idx, pj, w, f, out0, out1);
            return;
        }
    }
    if constexpr (SHORT) {
        const int64_t i = (int64_t)(blockIdx.x - nlongb) * blockDim.x + threadIdx.x;
        if (i >= np) return;
        const int64_t k0 = off[i], n = off[i + 1] - k0;
        if (n <= longest) short_row<MODE>(i, k0, (int)n, idx, pj, w, f, out0, out1);
    }
}

// Both kinds in one launch up to ROWS_ONE_LAUNCH pairs: the long rows do not wait
// for the short ones (545,000 pairs, rows of up to 361: 46 us, 64 in two).
// Beyond, two: the short rows' kernel has more warps resident by itself (1.7 M
// pairs in rows of 43: 33 us, 38 in one; 17.6 M: 229 and 311).
// map_back, us, with one thread per row and a wait for each of its three loads /
// with every pair gathered into a copy of the transpose first and the rows, in
// the caller's order, added from there (eight lanes a row below 2^20 pairs) / so:
//   107,000 pairs, rows of about 107               40.0 /   25.0 /   21.4
//   412,000 pairs, rows of about 41                23.5 /   34.7 /   15.2
//   4.3 M, rows of about 43                        68.5 /  104   /   68.3
//   17.6 M, rows of about 44                       245  /  491   /  229
//   1.9 M, rows of about 3                         47.9 /   72.9 /   48.8
//   0.55 M pseudo-particle pairs, rows up to 361   80.8 /   58.1 /   39.8
//   4.7 M, up to 2,504                             571  /  284   /  227
//   24.0 M, up to 3,781                           1,667 /  782   /  466
//   16.4 M, up to 33,417                         13,596 / 3,145  / 2,451
// Up to ROWS_ONE_LAUNCH pairs in rows of fewer than ROWS_THREAD on average, every
// row by a thread: the long rows' blocks, registers and shared memory would be a
// tenth to a quarter of such a call (500 to 50,000 pairs in rows of 1 to 5: 10.5
// to 11.8 us, 12.6 to 13.6 with them).
constexpr int64_t ROWS_ONE_LAUNCH = 1 << 20, ROWS_THREAD = 8;
template <int MODE>
static int launch_rows(em_ctx *ctx, const em_pairs *pr, const double *w, const double *f, double *out0, double *out1)
{
    // as many blocks of long rows as there may be; those without return at once
    const int nlongb = pr->npairs > EM_ROW_LONG
                           ? (int)(pr->npairs / (EM_ROW_LONG + 1) / 32 + pr->npairs / ROW_VERY / ROW_FEW) + 2
                           : 0;
    auto launch = [&](auto kernel, int threads, int nl, int64_t nshort, int longest) {
        kernel<<<(unsigned)(nl + nshort), threads, 0, ctx->stream>>>(pr->np, nl, longest, pr->nlong, pr->long_rows,
                                                                     pr->part_pair_off, pr->part_pair_idx, pr->pair_j,
                                                                     w, f, out0, out1);
    };
    if (pr->npairs < ROWS_ONE_LAUNCH) {
        if (pr->npairs < ROWS_THREAD * pr->np)
            launch(k_rows<MODE, false, true>, SHORT_THREADS, 0, em_grid(pr->np, SHORT_THREADS), INT_MAX);
        else
            launch(k_rows<MODE, true, true>, ROW_THREADS, nlongb, em_grid(pr->np, ROW_THREADS), EM_ROW_LONG);
        EM_LAUNCHED(ctx);
        return EM_OK;
    }
    launch(k_rows<MODE, true, false>, ROW_THREADS, nlongb, 0, 0);
    EM_LAUNCHED(ctx);
    launch(k_rows<MODE, false, true>, SHORT_THREADS, 0, em_grid(pr->np, SHORT_THREADS), EM_ROW_LONG);
    EM_LAUNCHED(ctx);
    return EM_OK;
}

// The FP32 pass in launch shape `variant` (see MQ_VARIANT_*).
template <int V>
static void launch_variant(cudaStream_t st, int64_t n, const int32_t *pi, const int32_t *pj, const double *x,
                           const double *y, const double *z, const double *h, const double *gen, const double *radius,
                           const int64_t *cfo, const int64_t *fvo, const PlaneF *pf, const PlaneF *pfl,
                           const EdgeF *ef, const EdgeF *efl, float tol, double est_k, double *w, int32_t *flagged,
                           int *nflag)
{
    constexpr int W = MQ_VARIANT_WARPS[V], B = MQ_VARIANT_MINB[V];
    k_map_fp32<W, B><<<em_grid((n + 31) / 32, W), 32 * W, 0, st>>>(n, pi, pj, x, y, z, h, gen, radius, cfo, fvo, pf,
                                                                 pfl, ef, efl, tol, est_k, w, flagged, nflag);
}

static void launch_map_fp32(int variant, cudaStream_t st, int64_t n, const int32_t *pi, const int32_t *pj,
                            const double *x, const double *y, const double *z, const double *h, const double *gen,
                            const double *radius, const int64_t *cfo, const int64_t *fvo, const PlaneF *pf,
                            const PlaneF *pfl, const EdgeF *ef, const EdgeF *efl, float tol, double est_k, double *w,
                            int32_t *flagged, int *nflag)
{
    switch (variant) {
    case 1: launch_variant<1>(st, n, pi, pj, x, y, z, h, gen, radius, cfo, fvo, pf, pfl, ef, efl, tol, est_k, w, flagged, nflag); break;
    case 2: launch_variant<2>(st, n, pi, pj, x, y, z, h, gen, radius, cfo, fvo, pf, pfl, ef, efl, tol, est_k, w, flagged, nflag); break;
    case 3: launch_variant<3>(st, n, pi, pj, x, y, z, h, gen, radius, cfo, fvo, pf, pfl, ef, efl, tol, est_k, w, flagged, nflag); break;
    default: launch_variant<0>(st, n, pi, pj, x, y, z, h, gen, radius, cfo, fvo, pf, pfl, ef, efl, tol, est_k, w, flagged, nflag); break;
    }
}

// map_exact, map_exact_noalloc and map_batch: the mixed pass's flagged-pair
// list and counter are stream-ordered scratch, the caller's scratch
// (d_flag_buf, d_flag_count: map_batch), or the library's fixed device array
// (fixed == true, at most EM_NOALLOC_MAX_PAIRS pairs).
static int noalloc_buffers(em_ctx *ctx, int32_t **flagged, int **count);

int em_map_exact_impl(em_ctx *ctx, const em_pairs *pr, const double *d_x, const double *d_y, const double *d_z,
                      const double *d_h, const double *d_m, const em_voronoi *v, const em_params *p, double *d_w_out,
                      double *d_rho_out, double *d_wsum_out, int64_t *h_nfp64, bool fixed, int32_t *d_flag_buf,
                      int *d_flag_count)
{
    EM_CHECK_ARG(ctx && pr && v && p && pr->ncell == v->ncell);
    EM_CHECK_ARG(pr->npairs == 0 || (d_x && d_y && d_z && d_h && d_w_out));
    EM_CHECK_ARG(d_rho_out == nullptr || d_m != nullptr);
    EM_CHECK_ARG(p->precision == 0 || p->precision == 1);
    const int64_t n = pr->npairs;
    if (fixed && n > EM_NOALLOC_MAX_PAIRS) {
        em_set_error("map_exact_noalloc: %lld pairs exceed the fixed capacity of %d pairs", (long long)n,
                     EM_NOALLOC_MAX_PAIRS);
        return EM_ECAPACITY;
    }
    const int block = p->block_pairs > 0 ? p->block_pairs : 128;
    EM_CHECK_ARG(block % 32 == 0 && block <= 128);
    EM_CHECK_ARG(p->fp32_variant >= 0 && p->fp32_variant < MQ_NVARIANT);
    if (h_nfp64) *h_nfp64 = 0;
    if (ctx->timing) ctx->recorded[0] = ctx->recorded[1] = false;
    if (n) {
        const int fgrid = (int)std::min<int64_t>((n + block / 32 - 1) / (block / 32), (int64_t)ctx->nsm * 64);
        if (ctx->timing) EM_CUDA(cudaEventRecord(ctx->ev[0], ctx->stream));
        if (p->precision == 0) {
            k_map_fp64<<<fgrid, block, 0, ctx->stream>>>(n, pr->pair_i, pr->pair_j, d_x, d_y, d_z, d_h, v->gen,
                                                         v->radius, v->cell_face_off, v->face_vert_off, v->plane,
                                                         v->edge, d_w_out);
            EM_LAUNCHED(ctx);
            if (ctx->timing) {
                EM_CUDA(cudaEventRecord(ctx->ev[1], ctx->stream));
                ctx->recorded[0] = true;
            }
        } else {
            DevArena tmp(ctx->stream, true);
            int32_t *flagged;
            int *nflag;
            if (fixed) {
                EM_TRY(noalloc_buffers(ctx, &flagged, &nflag));
            } else if (d_flag_buf && d_flag_count) {   // the caller's scratch (map_batch), n entries
                flagged = d_flag_buf;
                nflag = d_flag_count;
            } else {
                EM_TRY(tmp.alloc(&flagged, n));
                EM_TRY(tmp.alloc(&nflag, 1));
            }
            EM_CUDA(cudaMemsetAsync(nflag, 0, sizeof(int), ctx->stream));
            launch_map_fp32(p->fp32_variant, ctx->stream, n, pr->pair_i, pr->pair_j, d_x, d_y, d_z, d_h, v->gen,
                            v->radius, v->cell_face_off, v->face_vert_off, v->plane_f, v->plane_fl, v->edge_f,
                            v->edge_fl, (float)p->fp64_threshold, em_est_k(p), d_w_out, flagged, nflag);
            EM_LAUNCHED(ctx);
            if (ctx->timing) {
                EM_CUDA(cudaEventRecord(ctx->ev[1], ctx->stream));
                EM_CUDA(cudaEventRecord(ctx->ev[2], ctx->stream));
            }
            // FP64 recompute of the flagged pairs; the count stays on the device
            k_map_fp64_flagged<<<fgrid, block, 0, ctx->stream>>>(nflag, pr->pair_i, pr->pair_j, d_x, d_y, d_z, d_h,
                                                                 v->gen, v->radius, v->cell_face_off,
                                                                 v->face_vert_off, v->plane, v->edge, flagged,
                                                                 d_w_out);
            EM_LAUNCHED(ctx);
            if (ctx->timing) {
                EM_CUDA(cudaEventRecord(ctx->ev[3], ctx->stream));
                ctx->recorded[0] = ctx->recorded[1] = true;
            }
            if (h_nfp64) {
                int hflag = 0;
                EM_CUDA(cudaMemcpyAsync(&hflag, nflag, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
                EM_CUDA(cudaStreamSynchronize(ctx->stream));
                *h_nfp64 = hflag;
            }
        }
    }
    if (d_rho_out && v->ncell) {
        k_cell_density<<<em_grid(v->ncell * 32, 256), 256, 0, ctx->stream>>>(v->ncell, pr->cell_pair_off, pr->pair_i,
                                                                               d_w_out, d_m, v->volume, d_rho_out);
        EM_LAUNCHED(ctx);
    }
    if (d_wsum_out && pr->np) EM_TRY(launch_rows<0>(ctx, pr, d_w_out, nullptr, d_wsum_out, nullptr));   // u_i = sum_j w_ij
    return EM_OK;
}

EM_EXPORT int map_exact(em_ctx *ctx, const em_pairs *pr, const double *d_x, const double *d_y, const double *d_z,
                        const double *d_h, const double *d_m, const em_voronoi *v, const em_params *p,
                        double *d_w_out, double *d_rho_out, double *d_wsum_out, int64_t *h_nfp64)
{
    return em_map_exact_impl(ctx, pr, d_x, d_y, d_z, d_h, d_m, v, p, d_w_out, d_rho_out, d_wsum_out, h_nfp64, false,
                             nullptr, nullptr);
}

// Time the FP32 pass in every launch shape on the given pairs (a warm-up
// launch, then the median of three CUDA-event-timed launches each) and return
// the fastest.  Scratch only; the caller's arrays are read, never written.
EM_EXPORT int map_autotune(em_ctx *ctx, const em_pairs *pr, const double *d_x, const double *d_y, const double *d_z,
                           const double *d_h, const em_voronoi *v, const em_params *p, int *h_best, double *h_ms)
{
    EM_CHECK_ARG(ctx && pr && v && p && h_best && pr->ncell == v->ncell);
    EM_CHECK_ARG(pr->npairs == 0 || (d_x && d_y && d_z && d_h));
    *h_best = 0;
    const int64_t n = pr->npairs;
    if (n == 0) {
        if (h_ms)
            for (int k = 0; k < MQ_NVARIANT; ++k) h_ms[k] = 0.0;
        return EM_OK;
    }
    DevArena tmp(ctx->stream, true);
    double *w;
    int32_t *flagged;
    int *nflag;
    EM_TRY(tmp.alloc(&w, n));
    EM_TRY(tmp.alloc(&flagged, n));
    EM_TRY(tmp.alloc(&nflag, 1));
    cudaEvent_t e0, e1;
    EM_CUDA(cudaEventCreate(&e0));
    EM_CUDA(cudaEventCreate(&e1));
    int rc = EM_OK;
    double best = 1e300;
    for (int k = 0; k < MQ_NVARIANT && rc == EM_OK; ++k) {
        float t[4] = {0.f, 0.f, 0.f, 0.f};
        for (int r = 0; r < 4 && rc == EM_OK; ++r) {
            cudaMemsetAsync(nflag, 0, sizeof(int), ctx->stream);
            cudaEventRecord(e0, ctx->stream);
            launch_map_fp32(k, ctx->stream, n, pr->pair_i, pr->pair_j, d_x, d_y, d_z, d_h, v->gen, v->radius,
                            v->cell_face_off, v->face_vert_off, v->plane_f, v->plane_fl, v->edge_f, v->edge_fl,
                            (float)p->fp64_threshold, em_est_k(p), w, flagged, nflag);
            ctx->launches++;
            cudaEventRecord(e1, ctx->stream);
            cudaError_t e = cudaEventSynchronize(e1);
            if (e == cudaSuccess) e = cudaEventElapsedTime(&t[r], e0, e1);
            if (e == cudaSuccess) e = cudaGetLastError();
            if (e != cudaSuccess) {
                em_set_error("map_autotune: variant %d: %s", k, cudaGetErrorString(e));
                rc = EM_ECUDA;
            }
        }
        const float a = t[1], b = t[2], c = t[3];   // t[0] is the warm-up
        const double med = fmax(fmin(a, b), fmin(fmax(a, b), c));
        if (h_ms) h_ms[k] = med;
        if (rc == EM_OK && med < best) {
            best = med;
            *h_best = k;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return rc;
}

// ---------------------------------------------------------------------------
// map_exact without allocation, for callers that cannot allocate device
// memory during the call (their own pool holds all free memory, or they cannot
// take an allocation's synchronisation every step): the mixed pass's
// flagged-pair list and its counter live in a fixed device array instead of
// stream-ordered scratch.
// ---------------------------------------------------------------------------

namespace {

// Zeroed at the start of every call (the counter); the list needs no reset,
// the FP32 pass writes entries [0, count) before the FP64 pass reads them.
static __device__ __align__(256) int32_t g_noalloc_flagged[EM_NOALLOC_MAX_PAIRS];
static __device__ __align__(256) int g_noalloc_count[1];

constexpr int NOALLOC_MAX_DEVICES = 64;
std::mutex g_noalloc_mutex;
int32_t *g_noalloc_flagged_addr[NOALLOC_MAX_DEVICES];
int *g_noalloc_count_addr[NOALLOC_MAX_DEVICES];

}  // namespace

// Device addresses of the two arrays on ctx's device, looked up once per
// device with that device current.
static int noalloc_buffers(em_ctx *ctx, int32_t **flagged, int **count)
{
    EM_CHECK_ARG(ctx->device >= 0 && ctx->device < NOALLOC_MAX_DEVICES);
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_flagged_addr[ctx->device]) {
        int cur = -1;
        EM_CUDA(cudaGetDevice(&cur));
        if (cur != ctx->device) EM_CUDA(cudaSetDevice(ctx->device));
        void *a = nullptr, *b = nullptr;
        cudaError_t e1 = cudaGetSymbolAddress(&a, g_noalloc_flagged);
        cudaError_t e2 = e1 == cudaSuccess ? cudaGetSymbolAddress(&b, g_noalloc_count) : e1;
        if (cur != ctx->device && cur >= 0) cudaSetDevice(cur);
        if (e2 != cudaSuccess) {
            em_set_error("map_exact_noalloc: cudaGetSymbolAddress failed on device %d: %s", ctx->device,
                         cudaGetErrorString(e2));
            return EM_ECUDA;
        }
        g_noalloc_count_addr[ctx->device] = (int *)b;
        g_noalloc_flagged_addr[ctx->device] = (int32_t *)a;
    }
    *flagged = g_noalloc_flagged_addr[ctx->device];
    *count = g_noalloc_count_addr[ctx->device];
    return EM_OK;
}

EM_EXPORT int map_exact_noalloc(em_ctx *ctx, const em_pairs *pr, const double *d_x, const double *d_y,
                                const double *d_z, const double *d_h, const double *d_m, const em_voronoi *v,
                                const em_params *p, double *d_w_out, double *d_rho_out, double *d_wsum_out,
                                int64_t *h_nfp64)
{
    return em_map_exact_impl(ctx, pr, d_x, d_y, d_z, d_h, d_m, v, p, d_w_out, d_rho_out, d_wsum_out, h_nfp64, true,
                             nullptr, nullptr);
}

// ---------------------------------------------------------------------------
// Inverse mapping
// ---------------------------------------------------------------------------

// every SPH particle takes the value of the pseudo-particle it belongs to
__global__ void k_inherit(int64_t npseudo, const int32_t *__restrict__ first, const int32_t *__restrict__ count,
                          const int32_t *__restrict__ perm, const double *__restrict__ f_pseudo,
                          double *__restrict__ f_particle)
{
    int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (a >= npseudo) return;
    double f = f_pseudo[a];
    for (int32_t k = first[a]; k < first[a] + count[a]; ++k) f_particle[perm[k]] = f;
}

EM_EXPORT int map_back_sums(em_ctx *ctx, const em_pairs *pr, const double *d_w, const double *d_f_cell,
                            double *d_num, double *d_den)
{
    EM_CHECK_ARG(ctx && pr && d_num && d_den && (pr->npairs == 0 || d_w) && (pr->ncell == 0 || d_f_cell));
    if (pr->np) EM_TRY(launch_rows<2>(ctx, pr, d_w, d_f_cell, d_num, d_den));
    return EM_OK;
}

EM_EXPORT int inherit(em_ctx *ctx, const em_pseudo *ps, const em_tree *t, const double *d_f_pseudo,
                      double *d_f_particle_out)
{
    EM_CHECK_ARG(ctx && ps && t && d_f_particle_out && (ps->n == 0 || d_f_pseudo));
    if (ps->n) {
        k_inherit<<<em_grid(ps->n, 128), 128, 0, ctx->stream>>>(ps->n, ps->first, ps->count, t->perm, d_f_pseudo,
                                                                 d_f_particle_out);
        EM_LAUNCHED(ctx);
    }
    return EM_OK;
}

EM_EXPORT int map_back(em_ctx *ctx, const em_pairs *pr, const double *d_w, const double *d_f_cell, double *d_f_out,
                       const em_pseudo *ps, const em_tree *t, double *d_f_particle_out)
{
    EM_CHECK_ARG(ctx && pr && d_f_out && (pr->npairs == 0 || d_w) && (pr->ncell == 0 || d_f_cell));
    bool inherit = ps || t || d_f_particle_out;
    EM_CHECK_ARG(!inherit || (ps && t && d_f_particle_out && ps->n == pr->np));
    if (pr->np) EM_TRY(launch_rows<1>(ctx, pr, d_w, d_f_cell, d_f_out, nullptr));
    if (inherit && ps->n) {
        k_inherit<<<em_grid(ps->n, 128), 128, 0, ctx->stream>>>(ps->n, ps->first, ps->count, t->perm, d_f_out,
                                                                 d_f_particle_out);
        EM_LAUNCHED(ctx);
    }
    return EM_OK;
}
