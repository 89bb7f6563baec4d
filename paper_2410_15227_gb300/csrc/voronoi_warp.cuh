// Warp-cooperative Voronoi cell construction (one warp per cell, the cell
// in shared memory, in dual form: planes, and vertices as triangles of
// planes).  A clip removes the vertices beyond the bisector, keeps the
// others in order and appends the new vertices in the order (removed
// vertex, edge), so the vertex order is fixed by the clips alone.
// Candidates: every generator within a radius R of the site (found by a warp
// walk of the generators' box hierarchy), sorted by distance; the cell is
// exact once 2 R_max < R, otherwise the shell up to 2 R_max is clipped in as
// well.
//
// Arithmetic.  The planes are exact FP64 bisectors (g_k - g, |g_k - g|^2 / 2)
// and each vertex is the meet of its three planes.  During the construction a
// vertex is held in FP32 only, computed from the FP32 roundings of its planes
// by Cramer's rule together with a bound on its distance from the exact meet
// of the FP64 planes (meet32).  A side test in FP32 whose margin exceeds the
// bound it implies is exact; the few that do not decide take the vertex's
// FP64 meet (meet64).  The FP64 vertices of the finished cell are formed
// once, for its faces.  So the FP64 pipe, at 1/64 of the FP32 rate, carries
// the exact decisions and the output, not the construction.
#pragma once

#include <cstdint>

#include "split.cuh"
#include "tree_util.cuh"
#include "voronoi_cell.cuh"

namespace emw {

constexpr int WMAXP = emv::MAXP;
constexpr int WCAND = 256;   // candidate list (power of two for the bitonic sort)
constexpr float U32 = 5.9604645e-8f;   // 2^-24, the unit roundoff of FP32

// A cell under construction with room for NV vertices.  Plane q is the
// bisector of the site and generator sid[q] (its sorted index), or box wall
// -1 - sid[q]; its FP64 form is formed again from the generator positions
// wherever it is needed (plane64), its FP32 rounding is kept in pf[q].
template <int NV>
struct WCell {
    static constexpr int MAXV = NV;
    static_assert(NV <= 255, "vertex indices are bytes, 0xff marks a removed vertex");
    float4 vf[NV];     // FP32 vertex in the site's frame, w = |x| + |y| + |z|
    float ev[NV];      // bound on |vf - v| per coordinate, v the exact meet of its planes
    float4 pf[WMAXP];
    int sid[WMAXP];
    union {
        struct {
            float cd2[WCAND];   // sort keys of the candidates: squared distances rounded to FP32
            int cid[WCAND];
        } k;                    // while the cell is built
        double vx[NV][3];       // the FP64 vertices of the finished cell
    } u;
    uint8_t side[NV];       // clip in progress: the vertex's new index (0xff if removed)
    uint8_t out_list[NV];   // clip in progress: the removed vertices
    // clip in progress: the new vertex whose edge leaves plane p (a = p), and the
    // one whose edge ends at it (b = p)
    uint8_t of_a[WMAXP], of_b[WMAXP];
    uint32_t tri[2][NV];    // the vertex's three planes, one per byte (byte_of)
    // byte e of adj[t]: the vertex across edge e of vertex t, i.e. the one whose
    // triangle holds the reversed edge (tri e + 1, tri e)
    uint32_t adj[2][NV];
    int np, nt, cur;
};

__device__ __forceinline__ int byte_of(uint32_t w, int e) { return (int)((w >> (8 * e)) & 0xffu); }

// Bisector plane n.x <= d of the site g (at the origin of the cell's frame)
// and generator k: n = g_k - g, d = |n|^2 / 2.
__device__ __forceinline__ void bisector(const double *__restrict__ xs, const double *__restrict__ ys,
                                         const double *__restrict__ zs, int64_t k, double gx, double gy, double gz,
                                         double &nx, double &ny, double &nz, double &d)
{
    nx = __dsub_rn(xs[k], gx);
    ny = __dsub_rn(ys[k], gy);
    nz = __dsub_rn(zs[k], gz);
    d = __dmul_rn(0.5, __fma_rn(nz, nz, __fma_rn(ny, ny, __dmul_rn(nx, nx))));
}

// Box wall w (0..5: x-lo, x-hi, y-lo, y-hi, z-lo, z-hi) as n.x <= d in the
// site's frame.
__device__ __forceinline__ void wall_plane(const double *box, int w, double gx, double gy, double gz, double &nx,
                                           double &ny, double &nz, double &d)
{
    const int ax = w >> 1;
    const double g = ax == 0 ? gx : (ax == 1 ? gy : gz);
    nx = ax == 0 ? ((w & 1) ? 1.0 : -1.0) : 0.0;
    ny = ax == 1 ? ((w & 1) ? 1.0 : -1.0) : 0.0;
    nz = ax == 2 ? ((w & 1) ? 1.0 : -1.0) : 0.0;
    d = (w & 1) ? box[2 * ax + 1] - g : -(box[2 * ax] - g);
}

// Where the plane positions come from: the sorted generators, the box and
// the site.
struct Frame {
    const double *xs, *ys, *zs;
    const double *box;
    double gx, gy, gz;
};

__device__ __forceinline__ void plane64(const Frame &F, int sid, double &nx, double &ny, double &nz, double &d)
{
    if (sid >= 0) bisector(F.xs, F.ys, F.zs, sid, F.gx, F.gy, F.gz, nx, ny, nz, d);
    else wall_plane(F.box, -1 - sid, F.gx, F.gy, F.gz, nx, ny, nz, d);
}

// Meet of the planes A, B, C (n.x = d, FP32 roundings of FP64 planes) by
// Cramer's rule, x = (d_A (n_B x n_C) + d_B (n_C x n_A) + d_C (n_A x n_B)) / det,
// det = n_A.(n_B x n_C).  With s_P = |n_P|_1, each cross-product component is
// within 4u s s' of the exact one's over the FP64 planes (its own rounding
// and the inputs'), det within 8u S, S = s_A s_B s_C, and each numerator
// within 8u N, N = |d_A| s_B s_C + |d_B| s_C s_A + |d_C| s_A s_B; so while
// |det| >= 64u S every coordinate is within 16u (N + |x|_inf S) / |det| of the
// exact meet (10.2u by the first-order sum, the rest covering the rounding of
// the quotient and of |x|).  err = inf when |det| is below that or S leaves
// FP32's normal range.
__device__ __forceinline__ void meet32(float4 A, float4 B, float4 Cp, float &x, float &y, float &z, float &err)
{
    const float bcx = fmaf(B.y, Cp.z, -B.z * Cp.y), bcy = fmaf(B.z, Cp.x, -B.x * Cp.z),
                bcz = fmaf(B.x, Cp.y, -B.y * Cp.x);
    const float cax = fmaf(Cp.y, A.z, -Cp.z * A.y), cay = fmaf(Cp.z, A.x, -Cp.x * A.z),
                caz = fmaf(Cp.x, A.y, -Cp.y * A.x);
    const float abx = fmaf(A.y, B.z, -A.z * B.y), aby = fmaf(A.z, B.x, -A.x * B.z),
                abz = fmaf(A.x, B.y, -A.y * B.x);
    const float det = fmaf(A.x, bcx, fmaf(A.y, bcy, A.z * bcz));
    const float id = 1.f / det;
    x = fmaf(A.w, bcx, fmaf(B.w, cax, Cp.w * abx)) * id;
    y = fmaf(A.w, bcy, fmaf(B.w, cay, Cp.w * aby)) * id;
    z = fmaf(A.w, bcz, fmaf(B.w, caz, Cp.w * abz)) * id;
    const float sA = fabsf(A.x) + fabsf(A.y) + fabsf(A.z), sB = fabsf(B.x) + fabsf(B.y) + fabsf(B.z),
                sC = fabsf(Cp.x) + fabsf(Cp.y) + fabsf(Cp.z);
    const float S = sA * sB * sC;
    const float N = fabsf(A.w) * sB * sC + fabsf(B.w) * sC * sA + fabsf(Cp.w) * sA * sB;
    const float xm = fmaxf(fabsf(x), fmaxf(fabsf(y), fabsf(z)));
    const float ad = fabsf(det);
    err = (ad >= 64.f * U32 * S && S >= 1e-30f) ? 16.f * U32 * (N + xm * S) / ad : INFINITY;
}

// FP64 meet of three FP64 planes (Cramer's rule, as meet32).
__device__ __forceinline__ void meet64p(const double *A, const double *B, const double *Cp, double &x, double &y,
                                        double &z)
{
    const double bcx = B[1] * Cp[2] - B[2] * Cp[1], bcy = B[2] * Cp[0] - B[0] * Cp[2], bcz = B[0] * Cp[1] - B[1] * Cp[0];
    const double cax = Cp[1] * A[2] - Cp[2] * A[1], cay = Cp[2] * A[0] - Cp[0] * A[2], caz = Cp[0] * A[1] - Cp[1] * A[0];
    const double abx = A[1] * B[2] - A[2] * B[1], aby = A[2] * B[0] - A[0] * B[2], abz = A[0] * B[1] - A[1] * B[0];
    const double id = 1.0 / (A[0] * bcx + A[1] * bcy + A[2] * bcz);
    x = (A[3] * bcx + B[3] * cax + Cp[3] * abx) * id;
    y = (A[3] * bcy + B[3] * cay + Cp[3] * aby) * id;
    z = (A[3] * bcz + B[3] * caz + Cp[3] * abz) * id;
}

// FP64 meet of vertex t's three planes.
template <class C>
__device__ void meet64(const C &c, const Frame &F, int t, double &x, double &y, double &z)
{
    double P[3][4];
#pragma unroll 1
    for (int e = 0; e < 3; ++e) plane64(F, c.sid[byte_of(c.tri[c.cur][t], e)], P[e][0], P[e][1], P[e][2], P[e][3]);
    meet64p(P[0], P[1], P[2], x, y, z);
}

// FP32 copy of a vertex from its FP64 meet, and the bound of its rounding.
__device__ __forceinline__ void set_vf(float4 &vf, float &ev, double x, double y, double z)
{
    const float xf = (float)x, yf = (float)y, zf = (float)z;
    vf = make_float4(xf, yf, zf, fabsf(xf) + fabsf(yf) + fabsf(zf));
    ev = U32 * fmaxf(fabsf(xf), fmaxf(fabsf(yf), fabsf(zf)));
}

__device__ __forceinline__ unsigned lanemask_lt() { return (1u << (threadIdx.x & 31)) - 1u; }

// The box as the starting cell: walls 0..5 (x-lo, x-hi, y-lo, y-hi, z-lo,
// z-hi), and corner i (bits x, y, z of i: 0 for lo, 1 for hi) the meet of
// walls sx, 2 + sy, 4 + sz, ordered counter-clockwise seen from outside.  The
// corner across the edge (tri[e], tri[e + 1]) shares those two walls and
// differs in the axis of the third, tri[e + 2]: i with that axis' bit flipped.
// Lane w sets wall w, lane i corner i.
template <class C>
__device__ void wcell_box(C &c, const Frame &F)
{
    const int lane = threadIdx.x & 31;
    if (lane < 6) {
        c.sid[lane] = -1 - lane;
        double nx, ny, nz, d;
        wall_plane(F.box, lane, F.gx, F.gy, F.gz, nx, ny, nz, d);
        c.pf[lane] = make_float4((float)nx, (float)ny, (float)nz, (float)d);
    }
    if (lane < 8) {
        const int i = lane;
        const int sx = i & 1, sy = (i >> 1) & 1, sz = (i >> 2) & 1;
        const uint8_t X = (uint8_t)sx, Y = (uint8_t)(2 + sy), Z = (uint8_t)(4 + sz);
        const bool pos = ((sx ? 1 : -1) * (sy ? 1 : -1) * (sz ? 1 : -1)) > 0;
        const uint8_t t[3] = {X, pos ? Y : Z, pos ? Z : Y};
        uint32_t tw = 0, aw = 0;
        for (int e = 0; e < 3; ++e) {
            tw |= (uint32_t)t[e] << (8 * e);
            aw |= (uint32_t)(i ^ (1 << (t[(e + 2) % 3] >> 1))) << (8 * e);
        }
        c.tri[0][i] = tw;
        c.adj[0][i] = aw;
        set_vf(c.vf[i], c.ev[i], sx ? F.box[1] - F.gx : F.box[0] - F.gx, sy ? F.box[3] - F.gy : F.box[2] - F.gy,
               sz ? F.box[5] - F.gz : F.box[4] - F.gz);
    }
    if (lane == 0) {
        c.np = 6;
        c.nt = 8;
        c.cur = 0;
    }
    __syncwarp();
}

// Drop planes no vertex refers to (one lane; rare).
template <class C>
__device__ int wcompact(C &c)
{
    const int lane = threadIdx.x & 31;
    if (lane == 0) {
        int map[WMAXP];
#pragma unroll 1
        for (int q = 0; q < c.np; ++q) map[q] = -1;
        const int cur = c.cur;
#pragma unroll 1
        for (int t = 0; t < c.nt; ++t)
            for (int e = 0; e < 3; ++e) map[byte_of(c.tri[cur][t], e)] = 0;
        int n = 0;
#pragma unroll 1
        for (int q = 0; q < c.np; ++q) {
            if (map[q] < 0) continue;
            map[q] = n;
            c.sid[n] = c.sid[q];
            c.pf[n] = c.pf[q];
            ++n;
        }
#pragma unroll 1
        for (int t = 0; t < c.nt; ++t) {
            const uint32_t w = c.tri[cur][t];
            c.tri[cur][t] = (uint32_t)map[byte_of(w, 0)] | (uint32_t)map[byte_of(w, 1)] << 8 | (uint32_t)map[byte_of(w, 2)] << 16;
        }
        c.np = n;
    }
    __syncwarp();
    return c.np;
}

// The FP32 side of vertex (v, ev) of the plane P = (n, d): f = n.v - d from
// the FP32 vertex and plane differs from the exact f by at most |n|_1 ev (the
// vertex) + 5u (|n|_1 |v|_1 + |d|) (the plane's rounding and the FP32 sum);
// beyond the band, twice that, its sign is exact.
__device__ __forceinline__ void side32(float4 P, float nsum, float4 v, float ev, bool &out, bool &unsure)
{
    const float ff = fmaf(P.x, v.x, fmaf(P.y, v.y, fmaf(P.z, v.z, -P.w)));
    const float band = 2.f * (nsum * ev + 5.f * U32 * (nsum * v.w + fabsf(P.w)));
    out = ff > band;
    unsure = !out && !(ff < -band);
}

// Clip by the bisector P (rounded to FP32) of generator sid.  Returns 1
// changed, 0 unchanged, < 0 error (all lanes).
template <class C>
__device__ int wclip(C &c, const Frame &F, float4 P, int sid)
{
    const int lane = threadIdx.x & 31;
    const int cur = c.cur, nxt = cur ^ 1, nt = c.nt;
    // The side of each vertex (side32).  Inside the band the vertex's
    // FP64 meet decides, with the warp converged on the few that need it; a
    // vertex within 1e-13 of the plane's scale (above the rounding of the
    // FP64 meet and value) counts as on the plane and is kept, so that a plane
    // through existing vertices, as in degenerate (lattice) site sets, cuts
    // no sliver off.
    const float nsum = fabsf(P.x) + fabsf(P.y) + fabsf(P.z);
    // lane i holds round i's masks: the removed vertices, and those FP64 decides
    unsigned mo = 0, mu = 0, any = 0, anyu = 0;
#pragma unroll 1
    for (int it = 0; it * 32 < nt; ++it) {
        const int t = it * 32 + lane;
        bool out = false, unsure = false;
        if (t < nt) side32(P, nsum, c.vf[t], c.ev[t], out, unsure);
        const unsigned bo = __ballot_sync(0xffffffffu, out && !unsure), bu = __ballot_sync(0xffffffffu, unsure);
        if (lane == it) {
            mo = bo;
            mu = bu;
        }
        any |= bo;
        anyu |= bu;
    }
    if (anyu) {
#pragma unroll 1
        for (int it = 0; it * 32 < nt; ++it) {
            const int t = it * 32 + lane;
            bool out = false;
            if ((__shfl_sync(0xffffffffu, mu, it) >> lane) & 1u) {
                double nx, ny, nz, d, x, y, z;
                bisector(F.xs, F.ys, F.zs, sid, F.gx, F.gy, F.gz, nx, ny, nz, d);
                meet64(c, F, t, x, y, z);
                out = nx * x + ny * y + nz * z - d > 1e-13 * (double)(nsum * c.vf[t].w + fabsf(P.w));
            }
            const unsigned b = __ballot_sync(0xffffffffu, out);
            any |= b;
            if (lane == it) mo |= b;
        }
    }
    if (!any) return 0;
    if (c.np >= WMAXP && wcompact(c) >= WMAXP) return -emv::VS_CAPACITY;
    const int q = c.np;
    // new index of every kept vertex (order kept), in side[]; removed ones listed
    int nk = 0, nout = 0;
#pragma unroll 1
    for (int it = 0; it * 32 < nt; ++it) {
        const int t = it * 32 + lane, left = nt - it * 32;
        const unsigned m = __shfl_sync(0xffffffffu, mo, it);
        const unsigned mk = (left >= 32 ? 0xffffffffu : (1u << left) - 1u) & ~m;
        if (t < nt) {
            const bool out = (m >> lane) & 1u;
            c.side[t] = out ? (uint8_t)0xff : (uint8_t)(nk + __popc(mk & lanemask_lt()));
            if (out) c.out_list[nout + __popc(m & lanemask_lt())] = (uint8_t)t;
        }
        nk += __popc(mk);
        nout += __popc(m);
    }
    __syncwarp();
    if (nk == 0) return -emv::VS_TOPOLOGY;
    // kept vertices into the other buffer, their neighbours renumbered (those
    // across a cut edge are set below); the FP32 copy and its bound move
    // within their buffer (a vertex never moves up, and each round reads
    // before it writes)
#pragma unroll 1
    for (int it = 0; it * 32 < nt; ++it) {
        const int t = it * 32 + lane;
        const int pos = t < nt ? c.side[t] : 0xff;
        float4 v;
        float e = 0.f;
        if (pos != 0xff) {
            v = c.vf[t];
            e = c.ev[t];
            const uint32_t w = c.adj[cur][t];
            uint32_t a = 0;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int n = byte_of(w, k);
                a |= (uint32_t)(n < nt ? c.side[n] : (uint8_t)0xff) << (8 * k);
            }
            c.tri[nxt][pos] = c.tri[cur][t];
            c.adj[nxt][pos] = a;
        }
        __syncwarp();
        if (pos != 0xff) {
            c.vf[pos] = v;
            c.ev[pos] = e;
        }
        __syncwarp();
    }
    // one task per (removed vertex, edge): a new vertex where the neighbour
    // across the edge is kept, with the two linked to each other; the new
    // vertex is the meet of the edge's planes a, b and the new plane, in FP32
    // with its bound, or from the FP64 meet where the FP32 one is too
    // uncertain to be of use (planes near a common line)
    int nn = nk;
    bool bad = false;
#pragma unroll 1
    for (int base = 0; base < 3 * nout; base += 32) {
        const int k = base + lane;
        bool newv = false;
        int a = 0, b = 0, upos = 0, ue = 0;
        float px = 0.f, py = 0.f, pz = 0.f, perr = INFINITY;
        if (k < 3 * nout) {
            const int t = c.out_list[k / 3], e = k % 3;
            const uint32_t tw = c.tri[cur][t];
            a = byte_of(tw, e);
            b = byte_of(tw, e == 2 ? 0 : e + 1);
            const int u = byte_of(c.adj[cur][t], e);
            if (u >= nt) {
                bad = true;   // inconsistent neighbours: reported, never followed
            } else if (c.side[u] != 0xff) {
                newv = true;
                upos = c.side[u];
                // the edge of u that is (b, a)
                const uint32_t tu = c.tri[cur][u];
                ue = (byte_of(tu, 0) == b && byte_of(tu, 1) == a) ? 0 : ((byte_of(tu, 1) == b && byte_of(tu, 2) == a) ? 1 : 2);
                bad = bad || !(byte_of(tu, ue) == b && byte_of(tu, ue == 2 ? 0 : ue + 1) == a);
                meet32(c.pf[a], c.pf[b], P, px, py, pz, perr);
            }
        }
        const bool poor = newv && !(perr <= 1e-4f * (fabsf(px) + fabsf(py) + fabsf(pz)));
        if (__any_sync(0xffffffffu, poor)) {
            if (poor) {
                double PL[3][4];
                plane64(F, c.sid[a], PL[0][0], PL[0][1], PL[0][2], PL[0][3]);
                plane64(F, c.sid[b], PL[1][0], PL[1][1], PL[1][2], PL[1][3]);
                bisector(F.xs, F.ys, F.zs, sid, F.gx, F.gy, F.gz, PL[2][0], PL[2][1], PL[2][2], PL[2][3]);
                double x, y, z;
                meet64p(PL[0], PL[1], PL[2], x, y, z);
                px = (float)x;
                py = (float)y;
                pz = (float)z;
                // the FP64 meet's own error is far below the FP32 rounding
                // unless the planes nearly share a line, where the bound is
                // left infinite and every side test takes the FP64 meet
                perr = isfinite(x + y + z) ? 2.f * U32 * fmaxf(fabsf(px), fmaxf(fabsf(py), fabsf(pz))) : INFINITY;
            }
        }
        unsigned m = __ballot_sync(0xffffffffu, newv);
        if (newv) {
            int pos = nn + __popc(m & lanemask_lt());
            if (pos < C::MAXV) {
                c.tri[nxt][pos] = (uint32_t)a | (uint32_t)b << 8 | (uint32_t)q << 16;
                c.adj[nxt][pos] = (uint32_t)upos;   // the edges on the new face follow
                reinterpret_cast<uint8_t *>(&c.adj[nxt][upos])[ue] = (uint8_t)pos;
                c.vf[pos] = make_float4(px, py, pz, fabsf(px) + fabsf(py) + fabsf(pz));
                c.ev[pos] = perr;
                c.of_a[a] = (uint8_t)pos;
                c.of_b[b] = (uint8_t)pos;
            }
        }
        nn += __popc(m);
    }
    __syncwarp();
    // the new vertices around the new face q: (a, b, q) meets the one whose
    // a is this b across (b, q), and the one whose b is this a across (q, a);
    // entries of of_a and of_b that this clip did not write are told apart by
    // their vertex
    if (nn <= C::MAXV)
#pragma unroll 1
        for (int n = nk + lane; n < nn; n += 32) {
            const uint32_t tw = c.tri[nxt][n];
            const int an = byte_of(tw, 0), bn = byte_of(tw, 1);
            const int m1 = c.of_a[bn], m2 = c.of_b[an];
            bad = bad || m1 < nk || m1 >= nn || m2 < nk || m2 >= nn;
            if (!bad) {
                bad = byte_of(c.tri[nxt][m1], 0) != bn || byte_of(c.tri[nxt][m2], 1) != an;
                c.adj[nxt][n] |= (uint32_t)m1 << 8 | (uint32_t)m2 << 16;
            }
        }
    if (__any_sync(0xffffffffu, bad)) return -emv::VS_TOPOLOGY;
    if (nn > C::MAXV) return -emv::VS_CAPACITY;
    if (lane == 0) {
        c.sid[q] = sid;
        c.pf[q] = P;
        c.np = q + 1;
        c.nt = nn;
        c.cur = nxt;
    }
    __syncwarp();
    return 1;
}

// An upper bound of the squared distance from the site to the cell's
// farthest vertex: per vertex |vf|_2 + sqrt(3) ev (the exact vertex lies
// within ev per coordinate), squared, widened by 1e-5 for the FP32 rounding
// of the norm.  A vertex with no finite bound takes its FP64 meet.
template <class C>
__device__ double wrmax2(const C &c, const Frame &F)
{
    const int lane = threadIdx.x & 31;
    float r2 = 0.f;
    bool fp64 = false;
#pragma unroll 1
    for (int t = lane; t < c.nt; t += 32) {
        const float4 v = c.vf[t];
        const float r = sqrtf(v.x * v.x + v.y * v.y + v.z * v.z) + 1.7320509f * c.ev[t];
        if (isfinite(r)) r2 = fmaxf(r2, r * r);
        else fp64 = true;
    }
    double q2 = (double)r2 * (1.0 + 1e-5);
    if (__any_sync(0xffffffffu, fp64)) {
#pragma unroll 1
        for (int t = lane; t < c.nt; t += 32) {
            if (isfinite(c.ev[t])) continue;
            double x, y, z;
            meet64(c, F, t, x, y, z);
            q2 = fmax(q2, (x * x + y * y + z * z) * (1.0 + 1e-12));
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q2 = fmax(q2, __shfl_xor_sync(0xffffffffu, q2, o));
    return q2;
}

// Gather every generator k != s with lo2 <= d^2 < hi2 into the candidate
// list (sorted by (d^2, k) afterwards).  Returns the count, or -1 if it
// exceeds WCAND.
template <class C>
__device__ int gather(C &c, const em::ChunkTree &T, const double *__restrict__ xs, const double *__restrict__ ys,
                      const double *__restrict__ zs, int64_t s, double gx, double gy, double gz, double lo2,
                      double hi2, float margin, int &status)
{
    int n = 0;
    float R = (float)sqrt(hi2) + margin;
    // The window test runs in FP32 on the rounded positions and keeps every
    // point whose FP32 distance lies within the window widened by a band above
    // the rounding of the coordinates: a superset of the exact window, which
    // is all the callers need (every generator in the window gets clipped).
    // The sort key is the FP32 squared distance; only near-coincident points
    // are checked in FP64.
    const float gxf = (float)gx, gyf = (float)gy, gzf = (float)gz;
    const float gabs = fabsf(gxf) + fabsf(gyf) + fabsf(gzf);
    float rhi = sqrtf((float)hi2) * (1.f + 1e-5f) + 1e-5f * gabs;
    const float rlo = lo2 > 0.0 ? sqrtf((float)lo2) * (1.f - 1e-5f) - 1e-5f * gabs : -1.f;
    const float rtiny = 1e-5f * (gabs + rhi);
    em::warp_traverse(T, gxf, gyf, gzf, R * R, INT64_MAX, [&](int64_t k, bool valid) {
        bool hit = false;
        float d2f = 0.f;
        if (valid && k != s) {
            const float4 pk = T.pts[k];
            const float ex = pk.x - gxf, ey = pk.y - gyf, ez = pk.z - gzf;
            d2f = ex * ex + ey * ey + ez * ez;
            const float rf = sqrtf(d2f);
            hit = rf <= rhi && rf >= rlo;
            if (rf < rtiny) {   // possibly the same point
                const double dx = xs[k] - gx, dy = ys[k] - gy, dz = zs[k] - gz;
                if (dx * dx + dy * dy + dz * dz == 0.0) status |= emv::VS_COINCIDENT;
            }
        }
        unsigned m = __ballot_sync(0xffffffffu, hit);
        if (hit) {
            int pos = n + __popc(m & lanemask_lt());
            if (pos < WCAND) {
                c.u.k.cd2[pos] = d2f;
                c.u.k.cid[pos] = (int)k;
            }
        }
        n += __popc(m);
    });
    status = __reduce_or_sync(0xffffffffu, status);
    __syncwarp();
    return n > WCAND ? -1 : n;
}

// Bitonic sort of the first n candidates by (d^2 in FP32, index), padded with
// (inf, max) up to the next power of two (at most WCAND).
template <class C>
__device__ void sort_cand(C &c, int n)
{
    const int lane = threadIdx.x & 31;
    float *cd2 = c.u.k.cd2;
    int *cid = c.u.k.cid;
    int len = 2;
#pragma unroll 1
    while (len < n) len <<= 1;
#pragma unroll 1
    for (int i = n + lane; i < len; i += 32) {
        cd2[i] = INFINITY;
        cid[i] = 0x7fffffff;
    }
    __syncwarp();
#pragma unroll 1
    for (int size = 2; size <= len; size <<= 1) {
#pragma unroll 1
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
#pragma unroll 1
            for (int i = lane; i < len / 2; i += 32) {
                int lo = 2 * i - (i & (stride - 1));
                int hi = lo + stride;
                bool up = ((lo & size) == 0);
                const float a = cd2[lo], b = cd2[hi];
                int ia = cid[lo], ib = cid[hi];
                bool gt = (a > b) || (a == b && ia > ib);
                if (gt == up) {
                    cd2[lo] = b;
                    cd2[hi] = a;
                    cid[lo] = ib;
                    cid[hi] = ia;
                }
            }
            __syncwarp();
        }
    }
}

// Generators k != s whose bisector may cut the current cell (some vertex v
// may have f = r_k.v - |r_k|^2/2 > 0, r_k = g_k - g), excluding those nearer
// than sqrt(skip2) (already applied), up to the window's end hi2.  Boxes are
// skipped when every vertex is at least as close to the site as to the box.
// When the list would overflow, the walk keeps the candidates whose FP32 key
// is below the median key k and goes on with hi2 narrowed to the float p just
// below k: every generator with d2 < p has a key <= p, so none is lost, and a
// kept one a little beyond p is only applied early (the half-spaces commute;
// once applied it no longer cuts).  Returns the count with hi2 the window
// actually covered, or -1 if the window cannot narrow (ties at the median).
// A listed generator that does not cut costs a clip that changes nothing.
template <class C>
__device__ int gather_cutting(C &c, const em::ChunkTree &T, const double *__restrict__ xs,
                              const double *__restrict__ ys, const double *__restrict__ zs, int64_t s, double gx,
                              double gy, double gz, double skip2, double &hi2)
{
    const int lane = threadIdx.x & 31;
    const int nt = c.nt;
    float *cd2 = c.u.k.cd2;
    int *cid = c.u.k.cid;
    // The pruning tests run in FP32 with margins above the rounding of the
    // coordinates (S below is a bound on their magnitudes) and the vertices'
    // bounds ev: a box or point is dropped only where the exact test would
    // drop it too.
    const float gxf = (float)gx, gyf = (float)gy, gzf = (float)gz;
    const float gabs = fabsf(gxf) + fabsf(gyf) + fabsf(gzf);
    float rhi = sqrtf((float)hi2) * (1.f + 1e-5f) + 1e-5f * gabs;
    const float rlo = skip2 > 0.0 ? sqrtf((float)skip2) * (1.f - 1e-5f) - 1e-5f * gabs : -1.f;
    auto box_can_cut = [&](const float4 lo, const float4 hi) -> bool {
        const float babs = fabsf(lo.x) + fabsf(lo.y) + fabsf(lo.z) + fabsf(hi.x) + fabsf(hi.y) + fabsf(hi.z);
        const float lx = lo.x - gxf, ly = lo.y - gyf, lz = lo.z - gzf;
        const float hx = hi.x - gxf, hy = hi.y - gyf, hz = hi.z - gzf;
        {   // the whole box beyond the window's outer radius
            float dx = fmaxf(fmaxf(lx, -hx), 0.f), dy = fmaxf(fmaxf(ly, -hy), 0.f), dz = fmaxf(fmaxf(lz, -hz), 0.f);
            if (sqrtf(dx * dx + dy * dy + dz * dz) > rhi + 1e-5f * babs) return false;
        }
        // some vertex nearer to the box than to the site (the exact vertex
        // lies within 1.8 ev of vf, which moves both squared distances by at
        // most 3.6 ev (|d| + |g|) + 6.5 ev^2)
#pragma unroll 1
        for (int t = 0; t < nt; ++t) {
            const float4 v = c.vf[t];
            const float vx = v.x, vy = v.y, vz = v.z;
            float dx = fmaxf(fmaxf(lx - vx, vx - hx), 0.f);
            float dy = fmaxf(fmaxf(ly - vy, vy - hy), 0.f);
            float dz = fmaxf(fmaxf(lz - vz, vz - hz), 0.f);
            const float db = dx * dx + dy * dy + dz * dz;
            const float dg = vx * vx + vy * vy + vz * vz;
            const float S = gabs + babs + v.w;
            const float e = c.ev[t];
            if (!(db >= dg + 1e-5f * S * S + 7.2f * e * S + 6.5f * e * e)) return true;
        }
        return false;
    };
    // a level above the top, of one node, so that the box test has one call site
    uint32_t mask[em::kMaxLevels + 2];
    int64_t base[em::kMaxLevels + 2];
    const int top = T.nlev + 1;
    int n = 0;
    mask[top] = 1;
    base[top] = 0;
    int lvl = top;
    while (true) {
        if (mask[lvl] == 0) {
            if (lvl == top) break;
            ++lvl;
            continue;
        }
        int cidx = __ffs(mask[lvl]) - 1;
        mask[lvl] &= mask[lvl] - 1;
        int64_t node = base[lvl] * 32 + cidx;
        if (lvl == 1) {
            int64_t k = node * 32 + lane;
            double d2 = 0.0;
            bool hit = k < T.count[0] && k != s;
            if (hit) {
                // FP32: inside the window and some vertex possibly beyond the
                // bisector (margin above the rounding of the coordinates and
                // the vertex bounds)
                const float4 pk = T.pts[k];
                const float ex = pk.x - gxf, ey = pk.y - gyf, ez = pk.z - gzf;
                const float rf = sqrtf(ex * ex + ey * ey + ez * ez);
                hit = rf <= rhi && rf >= rlo;
                if (hit) {
                    const float df = 0.5f * rf * rf, rabs = fabsf(ex) + fabsf(ey) + fabsf(ez);
                    bool maybe = false;
#pragma unroll 1
                    for (int t = 0; t < nt && !maybe; ++t) {
                        const float4 vf = c.vf[t];
                        const float ff = ex * vf.x + ey * vf.y + ez * vf.z - df;
                        maybe = !(ff <= -(1e-5f * (gabs + rabs + vf.w) * (vf.w + rabs) + rabs * c.ev[t]));
                    }
                    hit = maybe;
                }
            }
            if (hit) {
                const double rx = xs[k] - gx, ry = ys[k] - gy, rz = zs[k] - gz;
                d2 = rx * rx + ry * ry + rz * rz;
                hit = d2 >= skip2 && d2 < hi2;
            }
            unsigned m = __ballot_sync(0xffffffffu, hit);
            if (n + __popc(m) > WCAND) {
                // narrow the window to the nearer half of the list (n <= WCAND here)
                sort_cand(c, n);
                const float kth = cd2[n / 2];
                const float pf = nextafterf(kth, 0.f);
                const double p2 = (double)pf;
                int keep = 0;   // the sorted prefix below the median key
#pragma unroll 1
                for (int b = 0; b < n; b += 32) {
                    const int i = b + lane;
                    keep += __popc(__ballot_sync(0xffffffffu, i < n && cd2[i] < kth));
                }
                if (!(kth > 0.f) || !(p2 > skip2) || !(p2 < hi2) || keep == 0) return -1;
                n = keep;
                hi2 = p2;
                rhi = sqrtf(pf) * (1.f + 1e-5f) + 1e-5f * gabs;
                hit = hit && d2 < hi2;
                m = __ballot_sync(0xffffffffu, hit);
            }
            if (hit) {
                int pos = n + __popc(m & lanemask_lt());
                if (pos < WCAND) {
                    cd2[pos] = em::f32_rn(d2);
                    cid[pos] = (int)k;
                }
            }
            n += __popc(m);
        } else {
            int64_t child = node * 32 + lane;
            bool hit = child < T.count[lvl - 1] && box_can_cut(T.lo[lvl - 1][child], T.hi[lvl - 1][child]);
            mask[lvl - 1] = __ballot_sync(0xffffffffu, hit);
            base[lvl - 1] = node;
            --lvl;
        }
    }
    __syncwarp();
    return n > WCAND ? -1 : n;
}

// Clip by the first nc (sorted) candidates, 32 at a time: each lane forms its
// candidate's FP64 bisector and rounds it to FP32 (an FP64 instruction costs
// the pipe the same on 32 lanes as on one), and the warp clips by the rounded
// planes in turn; the FP64 one is formed again by the few side tests and meets
// that need it.  After the first 32 few candidates still cut: each lane tests
// its own against the cell's vertices, and only those that some vertex does
// not clear are taken up (a cell only shrinks, so the test stays valid).
template <class C>
__device__ int clip_sorted(C &c, const Frame &F, int64_t n, int nc)
{
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int i0 = 0; i0 < nc; i0 += 32) {
        const int k = i0 + lane < nc ? c.u.k.cid[i0 + lane] : 0;
        if (__any_sync(0xffffffffu, k < 0 || k >= n)) return emv::VS_BOUNDS;
        double nx, ny, nz, d;
        bisector(F.xs, F.ys, F.zs, k, F.gx, F.gy, F.gz, nx, ny, nz, d);
        const float4 P = make_float4(em::f32_rn(nx), em::f32_rn(ny), em::f32_rn(nz), em::f32_rn(d));
        bool maybe = i0 + lane < nc;
        if (i0 > 0) {
            const float nsum = fabsf(P.x) + fabsf(P.y) + fabsf(P.z);
            bool cut = false;
            const int nt = c.nt;
#pragma unroll 1
            for (int t = 0; t < nt; ++t) {
                bool out, unsure;
                side32(P, nsum, c.vf[t], c.ev[t], out, unsure);
                cut = cut || out || unsure;
            }
            maybe = maybe && cut;
        }
        unsigned todo = __ballot_sync(0xffffffffu, maybe);
        while (todo) {
            const int l = __ffs(todo) - 1;
            todo &= todo - 1;
            const float4 Q = make_float4(__shfl_sync(0xffffffffu, P.x, l), __shfl_sync(0xffffffffu, P.y, l),
                                         __shfl_sync(0xffffffffu, P.z, l), __shfl_sync(0xffffffffu, P.w, l));
            const int r = wclip(c, F, Q, __shfl_sync(0xffffffffu, k, l));
            if (r < 0) return -r;
        }
    }
    return 0;
}

// Build the cell of sorted generator s.
// Stage 1: every generator within a radius R chosen from the local spacing
// (8th nearest of the site's 32-generator chunk), nearest first.  Stage 2
// (exact completion): generators whose bisector still cuts the cell, in
// distance windows [lo, hi) that shrink until they fit the candidate list,
// nearest first, until the window passes 2 R_max.  Every generator nearer
// than lo has been applied at each step.
template <class C>
__device__ int wbuild_cell(C &c, const em::ChunkTree &T, const Frame &F, int64_t s, int K, float margin)
{
    const int lane = threadIdx.x & 31;
    int status = 0;
    const double *xs = F.xs, *ys = F.ys, *zs = F.zs, *box = F.box;
    const double gx = F.gx, gy = F.gy, gz = F.gz;
    if (!(gx > box[0] && gx < box[1] && gy > box[2] && gy < box[3] && gz > box[4] && gz < box[5]))
        return emv::VS_OUTSIDE;
    wcell_box(c, F);
    const int64_t n = T.count[0];
    // local spacing: the 8th smallest distance to the other members of the
    // chunk (a starting radius only, so FP32 on the rounded positions)
    double R2;
    {
        int64_t k = (s / 32) * 32 + lane;
        float d2 = INFINITY;
        if (k < n && k != s) {
            const float4 pk = T.pts[k], ps = T.pts[s];
            const float dx = pk.x - ps.x, dy = pk.y - ps.y, dz = pk.z - ps.z;
            d2 = dx * dx + dy * dy + dz * dz;
        }
        float kthf = INFINITY;
#pragma unroll 1
        for (int r = 0; r < 8; ++r) {
            float m = d2;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) m = fminf(m, __shfl_xor_sync(0xffffffffu, m, o));
            kthf = m;
            unsigned who = __ballot_sync(0xffffffffu, d2 == m);
            if (lane == __ffs(who) - 1) d2 = INFINITY;
        }
        double kth = kthf;
        if (!(kth > 0.0 && kth < INFINITY)) {
            const double bx = box[1] - box[0], by = box[3] - box[2], bz = box[5] - box[4];
            kth = 0.01 * (bx * bx + by * by + bz * bz);
        }
        // the chunk's own 8th nearest overestimates the local spacing (its
        // members lie mostly to one side), hence the factor 1/4
        R2 = 0.25 * kth * cbrt(1.5 * K / 8.0) * cbrt(1.5 * K / 8.0);
    }
    // round -1 is stage 1, rounds 0.. stage 2; both clip through the one call
    // site below (one inlined copy of the clip keeps the code small)
    double skip2 = -1.0;
#pragma unroll 1
    for (int round = -1; round < 256; ++round) {
        int m = -1;
        double hi2 = 0.0;
        if (round < 0) {
            // stage 1: shrink or grow R until the candidates fit and number at least K
            double lo_ok = 0.0, hi_bad = INFINITY;
#pragma unroll 1
            for (int it = 0; it < 48; ++it) {
                m = gather(c, T, xs, ys, zs, s, gx, gy, gz, -1.0, R2, margin, status);
                if (status & emv::VS_COINCIDENT) return status;
                if (m < 0) {
                    hi_bad = R2;
                    R2 = lo_ok > 0.0 ? sqrt(lo_ok * hi_bad) : 0.3 * R2;
                    continue;
                }
                if (m < K && m < n - 1 && hi_bad == INFINITY && it < 40) {
                    lo_ok = R2;
                    R2 *= 2.0;
                    continue;
                }
                break;
            }
            hi2 = m >= 0 ? R2 : -1.0;   // every generator nearer than R gets applied
        } else {
            // stage 2: windows [skip2, hi2) of generators that still cut, nearest first
            const double lim2 = 4.0 * wrmax2(c, F) * (1.0 + 1e-12);   // no generator beyond 2 R_max can cut
            if (skip2 >= lim2) return status;
            hi2 = lim2;
#pragma unroll 1
            for (int h = 0; h < 64; ++h) {
                m = gather_cutting(c, T, xs, ys, zs, s, gx, gy, gz, skip2, hi2);
                if (m >= 0) break;
                hi2 = (skip2 > 0.0 ? skip2 : 0.0) + 0.5 * (hi2 - (skip2 > 0.0 ? skip2 : 0.0));
            }
            if (m < 0) return status | emv::VS_CANDIDATES;
        }
        if (m > 0) {
            sort_cand(c, m);
            int st = clip_sorted(c, F, n, m);
            if (st) return status | st;
        }
        skip2 = hi2;
    }
    return status | emv::VS_ROUNDS;
}

// The FP64 vertices of the finished cell (each the FP64 meet of its three
// planes), into c.u.vx; the candidate list is no longer needed.
template <class C>
__device__ void finish_vertices(C &c, const Frame &F)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();
#pragma unroll 1
    for (int t = lane; t < c.nt; t += 32) {
        double x, y, z;
        meet64(c, F, t, x, y, z);
        c.u.vx[t][0] = x;
        c.u.vx[t][1] = y;
        c.u.vx[t][2] = z;
    }
    __syncwarp();
}

// Face loop of plane q (one lane): vertex indices counter-clockwise seen from
// outside; returns the length (0 if the plane holds no vertex, -1 on error).
// From a vertex t holding q at position r, the next vertex around q is the
// one across t's edge (tri[t][r + 2], q).
template <class C>
__device__ int wface_loop(const C &c, int q, uint8_t *loop, int maxn)
{
    const int cur = c.cur, nt = c.nt;
    int t0 = -1;
#pragma unroll 1
    for (int t = 0; t < nt && t0 < 0; ++t) {
        const uint32_t w = c.tri[cur][t];
        if (byte_of(w, 0) == q || byte_of(w, 1) == q || byte_of(w, 2) == q) t0 = t;
    }
    if (t0 < 0) return 0;
    int n = 0, t = t0;
    do {
        if (n >= maxn) return -1;
        loop[n++] = (uint8_t)t;
        const uint32_t w = c.tri[cur][t];
        const int r = byte_of(w, 0) == q ? 0 : (byte_of(w, 1) == q ? 1 : 2);
        const int nx = byte_of(c.adj[cur][t], r == 0 ? 2 : r - 1);
        if (nx >= nt) return -1;
        t = nx;
    } while (t != t0);
    return n;
}

}  // namespace emw
