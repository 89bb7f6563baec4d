// make_pseudo_particles: adaptive tree-walk selection (Section 2.4.1, Eq. 4),
// node neighbour search and the node smoothing-length solver (Section 2.4.2,
// Eqs. 6-11).
//
// Selection is evaluated per node instead of by a sequential walk: a node is
// reached when every ancestor is opened; a reached internal node that is not
// opened, or a reached leaf outside r_part, becomes a pseudo-particle; a
// reached leaf inside r_part is replaced by its particles.  The predicates use
// explicit round-to-nearest products, so the selected set is bit-identical to
// a sequential walk with the same arithmetic.
//
// The neighbour search runs inside every solver iteration: a warp walks a
// 32-ary box hierarchy over the solver population (selected nodes plus the
// leaves of extracted particles, Morton order) with radius 2h, so the sum
// n(h) = sum_b W(r_ab, h) always covers every neighbour of the current h.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "split.cuh"
#include "tree_util.cuh"

namespace {

enum : uint8_t { F_LEAF = 1, F_EXTRACT = 2, F_OPEN = 4, F_REACHED = 8 };

__global__ void k_node_flags(int64_t nnode, const int32_t *__restrict__ nchild, const double *__restrict__ cx,
                             const double *__restrict__ cy, const double *__restrict__ cz,
                             const double *__restrict__ size, int nsrc, const double *__restrict__ src, double rp2,
                             double rl2, double th2, const uint8_t *__restrict__ force, uint8_t *__restrict__ flags)
{
    int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (a >= nnode) return;
    double r2 = INFINITY;
    for (int s = 0; s < nsrc; ++s) {
        double dx = __dsub_rn(cx[a], src[3 * s]), dy = __dsub_rn(cy[a], src[3 * s + 1]),
               dz = __dsub_rn(cz[a], src[3 * s + 2]);
        double q = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
        r2 = q < r2 ? q : r2;
    }
    uint8_t f = 0;
    // a node the refinement check found under-resolved (Eq. 5) is opened, or
    // if a leaf has its particles extracted
    const bool forced = force != nullptr && force[a] != 0;
    if (nchild[a] == 0) {
        f |= F_LEAF;
        if (r2 < rp2 || forced) f |= F_EXTRACT;
    } else {
        // open inside r_leaf, or when theta^2 < (s/r)^2 (Eq. 4)
        if (forced || r2 < rl2 || __dmul_rn(size[a], size[a]) > __dmul_rn(th2, r2)) f |= F_OPEN;
    }
    flags[a] = f;
}

__global__ void k_reached(int64_t nnode, const int32_t *__restrict__ parent, uint8_t *__restrict__ flags)
{
    int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (a >= nnode) return;
    bool r = true;
    for (int32_t p = parent[a]; p >= 0 && r; p = parent[p]) r = (flags[p] & F_OPEN) != 0;
    if (r) flags[a] |= F_REACHED;
}

// Mark Morton positions that start a pseudo-particle / a population entry.
__global__ void k_mark(int64_t nnode, const uint8_t *__restrict__ flags, const int32_t *__restrict__ first,
                       const int32_t *__restrict__ count, int32_t *__restrict__ start, int32_t *__restrict__ owner,
                       int32_t *__restrict__ popstart)
{
    int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (a >= nnode) return;
    uint8_t f = flags[a];
    if (!(f & F_REACHED)) return;
    bool leaf = f & F_LEAF;
    if (leaf && (f & F_EXTRACT)) {
        for (int32_t k = first[a]; k < first[a] + count[a]; ++k) {
            start[k] = 1;
            owner[k] = -1 - (int32_t)a;
        }
        popstart[first[a]] = 1;
    } else if (leaf || !(f & F_OPEN)) {
        start[first[a]] = 1;
        owner[first[a]] = (int32_t)a;
        popstart[first[a]] = 1;
    }
}

__global__ void k_emit(int64_t n, const int32_t *__restrict__ start, const int32_t *__restrict__ pidx,
                       const int32_t *__restrict__ owner, const int32_t *__restrict__ popstart,
                       const int32_t *__restrict__ popidx, const uint64_t *__restrict__ label,
                       const int32_t *__restrict__ first, const int32_t *__restrict__ count,
                       const double *__restrict__ mass, const double *__restrict__ cx, const double *__restrict__ cy,
                       const double *__restrict__ cz, const double *__restrict__ size, const double *__restrict__ xs,
                       const double *__restrict__ ys, const double *__restrict__ zs, const double *__restrict__ ms,
                       const int32_t *__restrict__ perm, const double *__restrict__ hpart, double h_fact,
                       double *__restrict__ px, double *__restrict__ py, double *__restrict__ pz,
                       double *__restrict__ ph, double *__restrict__ pm, int64_t *__restrict__ origin,
                       int32_t *__restrict__ pfirst, int32_t *__restrict__ pcount, int32_t *__restrict__ status,
                       int32_t *__restrict__ pnode, int32_t node_status, double *__restrict__ popx,
                       double *__restrict__ popy, double *__restrict__ popz)
{
    int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= n) return;
    if (start[k]) {
        int32_t q = pidx[k];
        int32_t a = owner[k];
        if (a >= 0) {
            px[q] = cx[a];
            py[q] = cy[a];
            pz[q] = cz[a];
            pm[q] = mass[a];
            origin[q] = (int64_t)label[a];
            pfirst[q] = first[a];
            pcount[q] = count[a];
            pnode[q] = a;
            status[q] = node_status;   // -1: to be solved; 2: takes h_0 without a solve
            // h_0 = h_fact (2 s_node) (Eq. 11); a one-particle node starts from its particle's h
            ph[q] = (count[a] == 1 || size[a] == 0.0) ? hpart[perm[first[a]]] : (2.0 * h_fact) * size[a];
        } else {
            px[q] = xs[k];
            py[q] = ys[k];
            pz[q] = zs[k];
            pm[q] = ms[k];
            origin[q] = -(int64_t)perm[k] - 1;
            pfirst[q] = (int32_t)k;
            pcount[q] = 1;
            pnode[q] = -1;
            status[q] = 3;
            ph[q] = hpart[perm[k]];
        }
    }
    if (popstart[k]) {
        // the population entry at this position is the node whose range starts here
        int32_t a = owner[k];
        if (a < 0) a = -1 - a;
        int32_t q = popidx[k];
        popx[q] = cx[a];
        popy[q] = cy[a];
        popz[q] = cz[a];
    }
}

struct Density {
    double n, dn;
};

// Neighbour candidates that pass the FP32 prefilter are collected in a
// per-warp buffer and summed in FP64 32 at a time, one per lane, so that the
// FP64 work (the costly part on GB300, whose FP64 rate is 1/64 of FP32) runs
// with every lane busy instead of on the few lanes of each 32-point chunk
// that hold a neighbour.
constexpr int HS_WARPS = 4;
constexpr float HS_FINE = 1e-16f;
constexpr int HS_BUF = 64;   // two batches: a chunk adds at most 32 to fewer than 32

// The FP32 prefilter: candidates clearly beyond 2h skip the FP64 work.  The
// band, 1e-5 of the coordinates' scale plus 2h, is far above the FP32 rounding
// of the positions, so no neighbour is dropped; nor where the squares are
// infinite (<=), or so small that they lose digits (HS_FINE).  Appends the warp's passing
// candidates to buf (nb entries, the same on every lane).
__device__ __forceinline__ void collect(const em::ChunkTree &T, int64_t k, bool valid, float xaf, float yaf,
                                        float zaf, float lim2, int32_t *buf, int &nb)
{
    const int lane = threadIdx.x & 31;
    bool cand = false;
    if (valid) {
        const float4 pk = T.pts[k];
        const float ex = pk.x - xaf, ey = pk.y - yaf, ez = pk.z - zaf;
        cand = ex * ex + ey * ey + ez * ez <= lim2;
    }
    const unsigned b = __ballot_sync(0xffffffffu, cand);
    if (cand) buf[nb + __popc(b & ((1u << lane) - 1u))] = (int32_t)k;
    __syncwarp();
    nb += __popc(b);
}

// Drop the first 32 entries of buf (already summed).
__device__ __forceinline__ void shift32(int32_t *buf, int &nb)
{
    const int lane = threadIdx.x & 31;
    const int32_t v = lane + 32 < nb ? buf[lane + 32] : 0;
    __syncwarp();
    if (lane + 32 < nb) buf[lane] = v;
    __syncwarp();
    nb -= 32;
}

// q = sqrt(q2) from an FP32 reciprocal square root (within 2^-22 relative)
// and one FP64 Newton step, which squares that error: within about 1e-13
// relative, far below the solver's tolerance on h and the 1e-12 to which h is
// held, at four FP64 instructions fewer than a second step; below 1e-30 q is 0
// (W then differs from W(0) by about 1e-30).  The conversions to and from
// float are done on the bits (split.cuh), which gives the same values off the
// FP64 pipe; q2 < 4 here.
__device__ __forceinline__ double q_of(double q2)
{
    if (!(q2 > 1e-30)) return 0.0;
    double r = em::f64_of(rsqrtf(em::f32_of(q2)));
    r = r * (1.5 - 0.5 * q2 * r * r);
    return q2 * r;
}

// 1/x for 2^-100 <= |x| < 2^100 (h and f' here): an FP32 reciprocal (its
// conversions on the bits, split.cuh) and two FP64 Newton steps, within about
// an ulp.  The solver's divisions have the same operands on every lane, so
// each FP64 instruction costs the pipe a full warp; this takes about half the
// FP64 instructions of a division.
__device__ __forceinline__ double rcp64(double x)
{
    // outside that range (zero, infinities, NaN included) the plain division;
    // the test reads the exponent's bits, off the FP64 pipe
    const int e = (int)(((unsigned long long)__double_as_longlong(x) >> 52) & 0x7ff);
    if (e < 923 || e >= 1123) return 1.0 / x;
    double r = em::f64_of(__frcp_rn(em::f32_of(x)));
    r = fma(r, fma(-x, r, 1.0), r);
    r = fma(r, fma(-x, r, 1.0), r);
    return r;
}

// The M4 spline w(q) and g(q) = 3 w(q) + q w'(q), the two sums of the
// solver, for q < 2 (q2 = q^2).
__device__ __forceinline__ void m4_wg(double q, double q2, double &w, double &g)
{
    if (q < 1.0) {
        w = 1.0 + q2 * (-1.5 + 0.75 * q);
        g = 3.0 + q2 * (-7.5 + 4.5 * q);
    } else {
        const double t = 2.0 - q, t2 = t * t;
        w = 0.25 * t2 * t;
        g = 0.75 * t2 * (t - q);
    }
}

// The solver's FP32 side.  Each FP64 evaluation of n(h) costs the FP64 pipe
// about 20 instructions per 32 neighbours and 75 on values every lane shares;
// the iterations that only approach the root, and the bisection's 50 signs,
// need none of that.  Population positions are float-float (T.pts and plo), so
// that a neighbour's offset is good to FP32 whatever the coordinates' size.
struct Population {
    const double *x, *y, *z;
    const float4 *lo;   // position - T.pts, rounded to FP32
};

constexpr int HS_LIST = 384;        // neighbours a warp keeps from its last walk
constexpr float HS_COVER = 1.08f;   // the walk's radius, in units of the 2h it serves
constexpr int HS_LEAVES = 4;        // 32-point leaves a walk reads together (their loads in flight at once)

// A node is solved by one warp or, where its 2h holds so much of the population
// that one warp's walk would outlast all others (HS_HEAVY batches), by a team
// of HS_TEAM: each warp of the team takes its share of every walk's leaves, and
// all add up and decide alike.  (1e6 particles: the longest node 11.5 M cycles
// against a mean of 0.12 M; tree, walk and h 8.6 ms without teams, 6.4 with.)
// The limit: a team redoes what the warp had done of the node, and FP64 sums,
// bound by the FP64 pipe, gain nothing from it until the other nodes have ended.
// make_pseudo_particles in us with h_tol 1e-2, 1e-8 and 1e-13, with 48 / 96 / 192
// batches / without a limit:
//   1e6 particles, theta 0.065   6750 9446 3377 / 6519 8949 3407 / 6736 9071 3370 / 9822 11987 4170
//   1e6, theta 0.25              1345 1933  730 / 1157 1515  480 / 1189 1489  487 / 1158  1523  495
//   3e5, theta 0.2                930 1465  509 /  877 1182  407 /  870 1177  406 /  875  1184  408
//   1e5, theta 0.1               1324 2098  819 / 1514 2092  821 / 1848 2035  801 / 1831  2071  822
// Teams of 4 instead of 8: 2% to 7% slower on the first with h_tol 1e-2, of 16: 6%
// with 1e-13.
constexpr int HS_TEAM = 8;
constexpr int HS_HEAVY = 96;   // batches of HS_LEAVES leaves: 12,288 entries

// A node under solution: its position, the neighbours of its last walk (every
// population entry within r of it if n >= 0; n = -1: more than the list holds),
// and this warp's part of the team.
struct HsList {
    double xa, ya, za;
    float xh, yh, zh, xl, yl, zl;
    float r;
    int n;
    int32_t *k;
    int32_t *buf;      // HS_BUF entries of the warp's own
    double (*red)[3];  // the team's partial sums
    int part;
    bool heavy;        // one warp alone: the walk was given up
};

// N values summed over the team's lanes, the same on all of them
template <int TEAM, int N, class Real>
__device__ __forceinline__ void team_sum(const HsList &L, Real (&v)[N])
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    if (TEAM > 1) {
        if ((threadIdx.x & 31) == 0)
            for (int i = 0; i < N; ++i) L.red[L.part][i] = (double)v[i];
        __syncthreads();
        for (int i = 0; i < N; ++i) {
            v[i] = Real(0);
            for (int t = 0; t < TEAM; ++t) v[i] += (Real)L.red[t][i];
        }
        __syncthreads();
    }
}

// The population within 2h of the node, 32 entries at a time from a compacted
// buffer: batch(k, in) on every lane, in false on the lanes without one; it
// returns false to end the walk (a warp-uniform value).  Returns false where
// the walk was ended or, by one warp alone, given up as heavy.
template <int TEAM, class Batch>
__device__ __forceinline__ bool walk_neighbours(const em::ChunkTree &T, HsList &L, double h, float margin,
                                                Batch &&batch)
{
    const int lane = threadIdx.x & 31;
    const float h2f = (float)(2.0 * h), R = h2f + margin;
    const float lim = fmaxf(h2f + 1e-5f * (fabsf(L.xh) + fabsf(L.yh) + fabsf(L.zh) + h2f), HS_FINE), lim2 = lim * lim;
    int nb = 0, visits = 0;
    const bool full = em::warp_traverse_batch<1>(T, L.xh, L.yh, L.zh, R * R, L.part, TEAM, [&](const int32_t(&k)[1]) {
        if (TEAM == 1 && ++visits > HS_HEAVY * HS_LEAVES) {
            L.heavy = true;
            return false;
        }
        collect(T, k[0], k[0] >= 0, L.xh, L.yh, L.zh, lim2, L.buf, nb);
        if (nb < 32) return true;
        const bool go = batch(L.buf[lane], true);
        shift32(L.buf, nb);
        return go;
    });
    if (!full) return false;
    batch(lane < nb ? L.buf[lane] : 0, lane < nb);
    __syncwarp();
    return true;
}

// w(q) and g(q) of entry k in FP64; false beyond 2h
__device__ __forceinline__ bool term64(const Population &P, const HsList &L, int32_t k, double ih2, double &w, double &g)
{
    const double dx = P.x[k] - L.xa, dy = P.y[k] - L.ya, dz = P.z[k] - L.za;
    const double q2 = (dx * dx + dy * dy + dz * dz) * ih2;
    if (!(q2 < 4.0)) return false;
    m4_wg(q_of(q2), q2, w, g);
    return true;
}

// n(h) and dn/dh in FP64 (the same on all lanes) by a walk: n = norm sum w,
// dn/dh = -norm sum g / h.
template <int TEAM>
__device__ Density warp_density(const em::ChunkTree &T, const Population &P, HsList &L, double h, float margin)
{
    double s[2] = {0.0, 0.0};
    const double ih = rcp64(h), ih2 = ih * ih, norm = ih2 * ih * 0.31830988618379067154;   // 1/(pi h^3)
    walk_neighbours<TEAM>(T, L, h, margin, [&](int32_t k, bool in) {
        double w, g;
        if (in && term64(P, L, k, ih2, w, g)) {
            s[0] += w;
            s[1] += g;
        }
        return true;
    });
    team_sum<TEAM>(L, s);
    return Density{s[0] * norm, -s[1] * norm * ih};
}

// Sign of f(h) = h_fact n(h)^(-1/3) - h (Eq. 8) for the bisection, which uses
// nothing else.  Every term of n is non-negative, so once a warp's running sum
// exceeds (h_fact / h)^3 (1 + 1e-9) the sign is negative whatever the rest of
// the sum; its walk stops there (checked after each batch of 32 terms).  This
// matters for the wide first brackets (h up to 1e2 h_0), whose 2h sphere
// holds a large share of the population.  Otherwise the full sum decides, as
// in warp_density.  Returns the sign of f (+1, 0 or -1).
template <int TEAM>
__device__ int warp_f_sign(const em::ChunkTree &T, const Population &P, HsList &L, double h, double h_fact,
                           float margin)
{
    double s[2] = {0.0, 0.0};   // the sum; warps that ended their walk
    const double ih = rcp64(h), ih2 = ih * ih, norm = ih2 * ih * 0.31830988618379067154;   // 1/(pi h^3)
    const double t = h_fact * ih, thr = t * t * t * (1.0 + 1e-9);
    // the sum of w; the walk stops once norm sum w exceeds thr
    const double thrw = thr * (3.14159265358979323846 * h * h * h);   // thr / norm
    const bool full = walk_neighbours<TEAM>(T, L, h, margin, [&](int32_t k, bool in) {
        double w, g;
        if (in && term64(P, L, k, ih2, w, g)) s[0] += w;
        double tot = s[0];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
        return !(tot > thrw);
    });
    if (!full) s[1] = 1.0;
    team_sum<TEAM>(L, s);
    if (s[1] > 0.0) return -1;
    const double f = h_fact * rcbrt(s[0] * norm) - h;   // n^(-1/3) as a reciprocal cube root
    return f > 0.0 ? 1 : (f < 0.0 ? -1 : 0);
}

// Sums of w, of g = 3 w + q w' and of e = q g': dS / dlog h = 3 S - G,
// dG / dlog h = -E.
struct Sum32 {
    float S, G, E;
};

// w, g and e of the M4 spline at q2 = q^2 < 4, branch-free
__device__ __forceinline__ void m4_wge32(float q2, float &w, float &g, float &e)
{
    const float q = q2 * rsqrtf(fmaxf(q2, 1e-30f));   // 0 at the particle itself
    const float t = 2.f - q, t2 = t * t;
    w = q < 1.f ? fmaf(q2, fmaf(0.75f, q, -1.5f), 1.f) : 0.25f * t2 * t;
    g = q < 1.f ? fmaf(q2, fmaf(4.5f, q, -7.5f), 3.f) : 0.75f * t2 * (t - q);
    e = q < 1.f ? q2 * fmaf(13.5f, q, -15.f) : q * t * fmaf(4.5f, q, -6.f);
}

// Add one entry's terms (none if !in).  No branches, so that the entries of a
// batch overlap: a lone warp walking a large node's 2 h_0, which may hold the
// whole population, is bound by the latency of this chain.
__device__ __forceinline__ void add32(const HsList &L, bool in, float4 p, float4 lo, float ih2, float (&s)[3])
{
    const float ex = (p.x - L.xh) + (lo.x - L.xl), ey = (p.y - L.yh) + (lo.y - L.yl), ez = (p.z - L.zh) + (lo.z - L.zl);
    const float q2 = fmaf(ex, ex, fmaf(ey, ey, ez * ez)) * ih2;
    float w, g, e;
    m4_wge32(q2, w, g, e);
    const bool add = in && q2 < 4.f;
    s[0] += add ? w : 0.f;
    s[1] += add ? g : 0.f;
    s[2] += add ? e : 0.f;
}

// The sums at h in FP32 (the same on every lane), from the list where it
// covers 2h, else by a walk that renews it.
template <int TEAM>
__device__ Sum32 warp_sum32(const em::ChunkTree &T, const Population &P, HsList &L, float h, float margin)
{
    const int lane = threadIdx.x & 31;
    const float ih2 = 1.f / (h * h);
    float s[3] = {0.f, 0.f, 0.f}, lost[3] = {0.f, 0.f, 0.f};
    if (L.n >= 0 && 2.0002f * h <= L.r) {
        for (int t = lane; t < L.n; t += 32) add32(L, true, T.pts[L.k[t]], P.lo[L.k[t]], ih2, s);
    } else {
        const float r = 2.f * HS_COVER * h;
        const float lim = r + 1e-5f * (fabsf(L.xh) + fabsf(L.yh) + fabsf(L.zh) + r), lim2 = lim * lim;
        int n = 0, visits = 0;
        em::warp_traverse_batch<HS_LEAVES>(T, L.xh, L.yh, L.zh, (r + margin) * (r + margin), L.part, TEAM,
                                           [&](const int32_t(&k)[HS_LEAVES]) {
            if (TEAM == 1 && ++visits > HS_HEAVY) {
                L.heavy = true;
                return false;
            }
            float4 p[HS_LEAVES], lo[HS_LEAVES];
            unsigned b[HS_LEAVES];
            float v[3] = {0.f, 0.f, 0.f};
#pragma unroll
            for (int u = 0; u < HS_LEAVES; ++u) {
                const int32_t kk = max(k[u], 0);
                p[u] = T.pts[kk];
                lo[u] = P.lo[kk];
            }
#pragma unroll
            for (int u = 0; u < HS_LEAVES; ++u) {
                const float ex = p[u].x - L.xh, ey = p[u].y - L.yh, ez = p[u].z - L.zh;
                const bool in = k[u] >= 0 && ex * ex + ey * ey + ez * ez < lim2;
                add32(L, in, p[u], lo[u], ih2, v);
                b[u] = __ballot_sync(0xffffffffu, in);
            }
            // a team's lanes add up thousands of terms: with what each addition rounds off
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const float t = s[i] + v[i];
                if (TEAM > 1) lost[i] += v[i] - (t - s[i]);
                s[i] = t;
            }
#pragma unroll
            for (int u = 0; u < HS_LEAVES; ++u) {
                const int pos = n + __popc(b[u] & ((1u << lane) - 1u));
                if (TEAM == 1 && ((b[u] >> lane) & 1u) && pos < HS_LIST) L.k[pos] = k[u];
                n += __popc(b[u]);
            }
            return true;
        });
        __syncwarp();
        L.r = r;
        L.n = TEAM == 1 && n <= HS_LIST && !L.heavy ? n : -1;
    }
    if (TEAM > 1)
        for (int i = 0; i < 3; ++i) s[i] += lost[i];
    team_sum<TEAM>(L, s);
    return Sum32{s[0], s[1], s[2]};
}

// Make the list the population within 2h and a margin for h's last digits, so
// that FP64 batches hold neighbours only.
template <int TEAM>
__device__ void settle_list(const em::ChunkTree &T, const Population &P, HsList &L, float h, float margin)
{
    const int lane = threadIdx.x & 31;
    if (TEAM > 1) return;   // a team keeps no list
    if (!(L.n >= 0 && 2.0002f * h <= L.r)) warp_sum32<TEAM>(T, P, L, h, margin);
    const float r = 2.004f * h;
    if (L.n < 0 || L.r <= r) return;
    const float lim = r + 1e-5f * (fabsf(L.xh) + fabsf(L.yh) + fabsf(L.zh) + r), lim2 = lim * lim;
    int n = 0;
    for (int t0 = 0; t0 < L.n; t0 += 32) {
        const int t = t0 + lane, k = t < L.n ? L.k[t] : 0;
        bool in = false;
        if (t < L.n) {
            const float4 p = T.pts[k];
            const float ex = p.x - L.xh, ey = p.y - L.yh, ez = p.z - L.zh;
            in = ex * ex + ey * ey + ez * ez < lim2;
        }
        const unsigned b = __ballot_sync(0xffffffffu, in);   // read before anything is written at or below t0
        if (in) L.k[n + __popc(b & ((1u << lane) - 1u))] = k;
        n += __popc(b);
        __syncwarp();
    }
    L.n = n;
    L.r = r;
}

// n(h) and dn/dh in FP64 from the list where it covers 2h, else by a walk.
template <int TEAM>
__device__ Density list_density(const em::ChunkTree &T, const Population &P, HsList &L, double h, float margin)
{
    if (!(L.n >= 0 && 2.0002f * (float)h <= L.r)) return warp_density<TEAM>(T, P, L, h, margin);
    double s[2] = {0.0, 0.0};
    const double ih = rcp64(h), ih2 = ih * ih, norm = ih2 * ih * 0.31830988618379067154;   // 1/(pi h^3)
    for (int t = threadIdx.x & 31; t < L.n; t += 32) {
        double w, g;
        if (term64(P, L, L.k[t], ih2, w, g)) {
            s[0] += w;
            s[1] += g;
        }
    }
    team_sum<TEAM>(L, s);
    return Density{s[0] * norm, -s[1] * norm * ih};
}

// The step f / f' of Newton's iteration (Eqs. 8-10: the next iterate is h less
// the step) from n and dn/dh at h.
__device__ __forceinline__ double newton_step(Density d, double h, double h_fact)
{
    // n^(-1/3) as a reciprocal cube root and n^(-4/3) as its fourth power:
    // the same values to an ulp or two, for a fraction of the FP64 work of
    // two general powers (every lane computes them, so each FP64
    // instruction costs the pipe a full warp)
    const double c = rcbrt(d.n);
    const double f = h_fact * c - h;                                              // Eq. 8
    const double fp = -h_fact * d.dn * ((c * c) * (c * c)) * (1.0 / 3.0) - 1.0;   // Eq. 9 (a product, not a division)
    return f * rcp64(fp);                                                         // Eq. 10
}

// Newton (Eq. 10) from h_0 (Eq. 11) until |dh|/h_0 < tol, every evaluation in
// FP64.  Returns false where an iterate leaves the bracket [1e-2 h_0, 1e2 h_0]
// or max_newton steps do not suffice: Newton failed.
template <int TEAM>
__device__ bool newton64(const em::ChunkTree &T, const Population &P, HsList &L, double h0, double h_fact,
                         double tol, int max_newton, float margin, double &hout)
{
    const double ih0 = rcp64(h0), blo = 1e-2 * h0, bhi = 1e2 * h0;
    double h = h0;
    for (int it = 0; it < max_newton; ++it) {
        const double hn = h - newton_step(warp_density<TEAM>(T, P, L, h, margin), h, h_fact);
        if (L.heavy) return false;
        if (!(hn >= blo && hn <= bhi)) return false;
        const double step = fabs(hn - h) * ih0;   // |dh| / h_0
        h = hn;
        if (step < tol) {
            hout = h;
            return true;
        }
    }
    return false;
}

// Bisection on [1e-2 h_0, 1e2 h_0] by signs (warp_f_sign), else h_0.
template <int TEAM>
__device__ double bisect64(const em::ChunkTree &T, const Population &P, HsList &L, double h0, double h_fact,
                           double tol, float margin, int &st)
{
    double lo = 1e-2 * h0, hi = 1e2 * h0;
    const int slo = warp_f_sign<TEAM>(T, P, L, lo, h_fact, margin);
    const int shi = warp_f_sign<TEAM>(T, P, L, hi, h_fact, margin);
    const bool plo = slo > 0;
    if (L.heavy) return h0;
    if (slo * shi > 0) {
        st = 2;
        return h0;
    }
    for (int k = 0; k < 200 && (hi - lo) > tol * h0 && !L.heavy; ++k) {
        const double mid = 0.5 * (lo + hi);
        if ((warp_f_sign<TEAM>(T, P, L, mid, h_fact, margin) > 0) == plo) lo = mid;
        else hi = mid;
    }
    st = 1;
    return 0.5 * (lo + hi);
}

// One Newton step from FP32 sums at h, in relative terms (x = log h,
// a = h_fact n^(-1/3) / h): f = h (a - 1), f' = c - 1, h f'' = dc/dx.
struct Step32 {
    float s;      // the step f / f', over h: the next iterate is h (1 - s)
    float c;      // f' + 1
    float K;      // h f'' / (2 f'): Newton's remaining error is K s^2
    // with h known to within e (relative) and the sums to within eps:
    float err;    // bound on the error of 1 - s
    float least;  // |s| is at least this, also where c - 1 may have either sign
};
__device__ __forceinline__ Step32 step32(Sum32 u, float hf, float e, float eps)
{
    const float a = hf * cbrtf(3.14159265f / u.S), iS = 1.f / (3.f * u.S);
    Step32 r;
    r.c = a * u.G * iS;
    const float i = 1.f / (r.c - 1.f);
    const float dc = (r.c - a) * u.G * iS - a * iS * (u.E + u.G * (3.f - u.G / u.S));
    r.s = (a - 1.f) * i;
    r.K = 0.5f * dc * i;
    // the next iterate's derivative by x, over h, carries e on; and the sums'
    // rounding: that of c is eps of 2.5 |c| + 2 a at most (the terms of G add up
    // to |G| + 6 S in magnitude, since the positive ones are below 3 w)
    const float M = 1.f - r.s, dM = (a - r.c + r.s * dc) * i, ce = eps * (2.5f * fabsf(r.c) + 2.f * a);
    r.err = e * fabsf(M + dM) + eps * (fabsf(M) + fabsf(i) * a) + ce * fabsf(i * r.s);
    r.least = (fabsf(a - 1.f) - e * fabsf(r.c - a) - eps * a) / (fabsf(r.c - 1.f) + e * fabsf(dc) + ce);
    return r;
}
// of the sums: a lane's adds up at most HS_HEAVY batches in a warp, and keeps what it rounds off in a team
constexpr float HS_EPS = 2e-6f;

// The root of f near h (an FP32 root, K of Step32 there) in FP64, to its
// rounding whatever the tolerance: Newton's step and the next term of its
// series, h K s^2, after which what is left is K^2 s^3 and s^2 times the change
// of K over the step.  So one evaluation suffices in nine cases of ten.
// Returns false where it does not settle at once.
template <int TEAM>
__device__ bool polish64(const em::ChunkTree &T, const Population &P, HsList &L, double &h, double h_fact, float K,
                         float margin)
{
    settle_list<TEAM>(T, P, L, (float)h, margin);
    for (int it = 0; it < 5; ++it) {
        const double d = newton_step(list_density<TEAM>(T, P, L, h, margin), h, h_fact);
        if (L.heavy) return false;
        const float s = (float)(d * rcp64(h)), q = K * s * s;
        if (!(fabsf(s) <= 1e-3f)) return false;
        h = h - d - h * (double)q;
        if (fabsf(q) <= 1e-13f && fabsf(s) <= 1e-5f) return true;
    }
    return false;
}

// For a tolerance that means "converged" (tol <= HS_WARM_TOL) the approach is
// made in FP32.  newton32: Newton's iterates from h_0 decide whether Newton
// converges (1; the root polished in FP64) or leaves the bracket (0).  A bound
// on how far each iterate may lie from FP64's goes along (Step32::err: near
// f' = 0 a step magnifies the rounding without limit); where it leaves a
// decision open, or grows beyond 1e-2, the step from the last iterate known in
// FP64 (hx, after itx steps) is taken again in FP64 and FP32 goes on from there.
// -1: not decided, which is also the answer where the tolerance is so near
// FP64's rounding of a step, about 1e-14 h / |f'|, that FP64's iterates may
// never meet it.  In a model of both on 6 x 10^7 random neighbourhoods (shells
// of 1 to 200 entries at 0.006 to 160 h_0) no decision differed; 55 of 3 x 10^6
// did where only iterates within 10% of the bracket's ends were left open.  1e6
// particles: a handful of nodes take a step again; FP64 iterates throughout for
// these, which may take them across the whole cloud, cost 1.2 ms of 5.9.
// FP32 sums need h and 100 h_0 with squares well inside FP32's range: they are
// used for h_0 between 1e-15 and 1e15 in the caller's unit of length (not for a
// cloud of parsecs in cm, say, whose nodes all take FP64 iterates with a walk
// each: the same statuses, 11.2 ms instead of 3.4 for 1e6 particles).
constexpr double HS_WARM_TOL = 1e-9;
constexpr float HS_WARM_MIN = 1e-15f, HS_WARM_MAX = 1e15f;
template <int TEAM>
__device__ int newton32(const em::ChunkTree &T, const Population &P, HsList &L, double h0, double h_fact, double tol,
                        int max_newton, float margin, double &hout)
{
    const float h0f = (float)h0, hf = (float)h_fact, blo = 1e-2f * h0f, bhi = 1e2f * h0f;
    if (!(h0f > HS_WARM_MIN && h0f < HS_WARM_MAX)) return -1;
    float h = h0f, e = 1e-7f;
    double hx = h0;
    int itx = 0;
    bool exact = false;   // take the next step in FP64
    // every step taken again moves itx on: at most max_newton of them (n bounds the loop whatever happens)
    for (int it = 0, n = 0; it + 4 < max_newton && n < 4 * max_newton; ++it, ++n) {
        if (exact) {
            exact = false;
            const double hn = hx - newton_step(list_density<TEAM>(T, P, L, hx, margin), hx, h_fact);
            if (L.heavy) return -1;
            if (!(hn >= 1e-2 * h0 && hn <= 1e2 * h0)) return 0;
            hx = hn;
            itx = it + 1;
            h = (float)hx;
            e = 1e-7f;
            continue;
        }
        const Sum32 u = warp_sum32<TEAM>(T, P, L, h, margin);
        if (L.heavy) return -1;
        const Step32 r = step32(u, hf, e, HS_EPS);
        const float hn = h * (1.f - r.s), dh = h * r.err;
        const bool finite = fabsf(hn) < 1e30f && dh < 1e30f;
        // left: below, above, or by a step so long that it leaves either way
        if ((finite && (hn + dh < 0.999f * blo || hn - dh > 1.001f * bhi)) || r.least > 1.f + 1.01f * bhi / h) return 0;
        e = r.err / (1.f - r.s);
        if (!(finite && hn - dh > 1.001f * blo && hn + dh < 0.999f * bhi && e < 1e-2f)) {
            it = itx - 1;
            exact = true;
            continue;
        }
        if (fabsf(r.s) < 3e-4f) {
            if (!(tol * h0 * (double)fabsf(r.c - 1.f) >= 1e-14 * (double)hn)) return -1;
            hout = hn - h * (r.K * r.s * r.s);
            return polish64<TEAM>(T, P, L, hout, h_fact, r.K, margin) ? 1 : -1;
        }
        h = hn;
    }
    return -1;
}

// bisect64's result where FP32 decides it (else false): f's sign is that of
// pi h_fact^3 - S(h), S = sum w increasing in h, so its one root r in the
// bracket is found by a bracketed Newton in log h, polished to FP64's rounding
// (about 1e-15 r / |f'|), and the bisection's decisions are comparisons with r;
// only a midpoint within ten times that of it takes an FP64 evaluation.
template <int TEAM>
__device__ bool bisect32(const em::ChunkTree &T, const Population &P, HsList &L, double h0, double h_fact, double tol,
                         float margin, double &hout, int &st)
{
    const float h0f = (float)h0, hf = (float)h_fact, blo = 1e-2f * h0f, bhi = 1e2f * h0f;
    const float target = 3.14159265f * hf * hf * hf;
    if (!(h0f > HS_WARM_MIN && h0f < HS_WARM_MAX)) return false;
    // the bracket's ends, each moved to the nearest point with the same sign
    float lo = blo, hi = h0f;
    auto sum = [&](float at) { return warp_sum32<TEAM>(T, P, L, at, margin); };
    Sum32 u = sum(h0f);
    if (L.heavy) return false;
    if (u.S < target) {
        lo = h0f;
        while (true) {
            hi = fminf(2.f * lo, bhi);
            u = sum(hi);
            if (L.heavy) return false;
            if (u.S > target) break;
            if (hi == bhi) {
                if (u.S > 0.999f * target) return false;
                hout = h0;   // no root below 1e2 h_0
                st = 2;
                return true;
            }
            lo = hi;
        }
        if (hi == bhi && u.S < 1.001f * target) return false;
    } else {
        u = sum(blo);
        if (L.heavy) return false;
        if (u.S > 0.999f * target) return false;
    }
    float h = sqrtf(lo * hi);
    for (int it = 0;; ++it) {
        if (it == 40) return false;
        u = sum(h);
        if (L.heavy) return false;
        if (u.S < target) lo = h;
        else hi = h;
        const float D = 3.f * u.S - u.G;   // dS / dlog h
        float hn = D > 0.f ? h * __expf(fminf(fmaxf((target - u.S) / D, -2.f), 2.f)) : 0.f;
        const bool in = hn > lo && hn < hi;
        if (!in) hn = sqrtf(lo * hi);
        const float d = fabsf(hn - h);
        h = hn;
        if ((in && d < 3e-4f * h) || hi - lo < 1e-6f * h) break;
    }
    double r = h;
    const Step32 v = step32(u, hf, 0.f, 0.f);   // within 3e-4 of the root, or so
    if (!polish64<TEAM>(T, P, L, r, h_fact, v.K, margin)) return false;
    double dlo = 1e-2 * h0, dhi = 1e2 * h0;
    const double near = 1e-14 * r * (1.0 + 1.0 / (double)fabsf(v.c - 1.f)), width = tol * h0;
    for (int k = 0; k < 200 && (dhi - dlo) > width && !L.heavy; ++k) {
        const double mid = 0.5 * (dlo + dhi), e = mid - r;
        const bool below = fabs(e) > near ? e < 0.0
                                          : warp_f_sign<TEAM>(T, P, L, mid, h_fact, margin) > 0;
        if (below) dlo = mid;
        else dhi = mid;
    }
    hout = 0.5 * (dlo + dhi);
    st = 1;
    return !L.heavy;
}

// Solve node a; a warp alone that meets a heavy walk leaves it (false).
template <int TEAM>
__device__ __forceinline__ bool solve_node(const em::ChunkTree &T, const Population &P, HsList &L, int64_t a,
                                           const double *__restrict__ px, const double *__restrict__ py,
                                           const double *__restrict__ pz, double h_fact, double tol, int max_newton,
                                           float margin, double *__restrict__ ph, int32_t *__restrict__ status)
{
    L.xa = px[a];
    L.ya = py[a];
    L.za = pz[a];
    em::split_all<3>({L.xa, L.ya, L.za}, {&L.xh, &L.yh, &L.zh}, {&L.xl, &L.yl, &L.zl});
    L.r = 0.f;
    L.n = -1;
    L.heavy = false;
    const double h0 = ph[a];
    double h = h0;
    int st = 0;
    const bool warm = tol <= HS_WARM_TOL;
    int ok = warm ? newton32<TEAM>(T, P, L, h0, h_fact, tol, max_newton, margin, h) : -1;
    if (ok < 0 && !L.heavy) ok = newton64<TEAM>(T, P, L, h0, h_fact, tol, max_newton, margin, h) ? 1 : 0;
    if (!ok && !L.heavy && !(warm && bisect32<TEAM>(T, P, L, h0, h_fact, tol, margin, h, st)) && !L.heavy)
        h = bisect64<TEAM>(T, P, L, h0, h_fact, tol, margin, st);
    if (L.heavy) return false;
    if (TEAM > 1) __syncthreads();   // every warp has read h_0
    if ((threadIdx.x & 31) == 0 && L.part == 0) {
        ph[a] = h;
        status[a] = st;
    }
    return true;
}

// One warp per pseudo-particle; the heavy ones are listed for k_h_solve_heavy.
// 1e6 particles (94,193 nodes, 5,733 of them bisected): 417,533 FP64
// evaluations of n(h) and 298,116 signs, each with its walk, took 11.2 ms; 1.1
// FP64 evaluations, 1.5 walks and 1.8 sums over a list per node take 2.2, and
// 0.9 the few nodes whose 2h holds thousands of the population (k_h_solve_heavy).
__global__ void __launch_bounds__(32 * HS_WARPS, 6) k_h_solve(
    int64_t npseudo, em::ChunkTree T, Population P, const double *__restrict__ px, const double *__restrict__ py,
    const double *__restrict__ pz, double h_fact, double tol, int max_newton, float margin, double *__restrict__ ph,
    int32_t *__restrict__ status, int *__restrict__ nheavy, int32_t *__restrict__ heavy)
{
    __shared__ int32_t bufs[HS_WARPS][HS_BUF], lists[HS_WARPS][HS_LIST];
    int64_t a = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (a >= npseudo) return;
    if (status[a] != -1) return;   // extracted particles keep their own h
    HsList L;
    L.k = lists[threadIdx.x >> 5];
    L.buf = bufs[threadIdx.x >> 5];
    L.red = nullptr;
    L.part = 0;
    if (!solve_node<1>(T, P, L, a, px, py, pz, h_fact, tol, max_newton, margin, ph, status) && (threadIdx.x & 31) == 0)
        heavy[atomicAdd(nheavy, 1)] = (int32_t)a;
}

// The listed nodes, a block of HS_TEAM warps each (grid-stride; the count is
// read on the device).
__global__ void __launch_bounds__(32 * HS_TEAM, 2) k_h_solve_heavy(
    em::ChunkTree T, Population P, const double *__restrict__ px, const double *__restrict__ py,
    const double *__restrict__ pz, double h_fact, double tol, int max_newton, float margin, double *__restrict__ ph,
    int32_t *__restrict__ status, const int *__restrict__ nheavy, const int32_t *__restrict__ heavy)
{
    __shared__ int32_t bufs[HS_TEAM][HS_BUF];
    __shared__ double red[HS_TEAM][3];
    HsList L;
    L.k = nullptr;
    L.buf = bufs[threadIdx.x >> 5];
    L.red = red;
    L.part = threadIdx.x >> 5;
    const int n = *nheavy;
    for (int t = blockIdx.x; t < n; t += gridDim.x) {
        solve_node<HS_TEAM>(T, P, L, heavy[t], px, py, pz, h_fact, tol, max_newton, margin, ph, status);
        __syncthreads();
    }
}

// Low parts of the population's positions (Population::lo).
__global__ void k_population_lo(int64_t n, const double *__restrict__ x, const double *__restrict__ y,
                                const double *__restrict__ z, float4 *__restrict__ lo)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= n) return;
    float h, lx, ly, lz;
    em::split_df(x[k], h, lx);
    em::split_df(y[k], h, ly);
    em::split_df(z[k], h, lz);
    lo[k] = make_float4(lx, ly, lz, 0.f);
}

__global__ void k_status_count(int64_t n, const int32_t *__restrict__ status, unsigned long long *__restrict__ cnt)
{
    int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (a >= n) return;
    int s = status[a];
    if (s >= 0 && s < 4) atomicAdd(&cnt[s], 1ull);
}

}  // namespace

static int pseudo_impl(em_ctx *ctx, const em_tree *t, const double *d_hp, int nsrc, const double *h_src,
                       const em_params *p, const uint8_t *d_force, em_pseudo *ps)
{
    cudaStream_t st = ctx->stream;
    const int64_t n = t->n, nn = t->nnode;
    DevArena tmp(st, true);
    double *src;
    uint8_t *flags;
    int32_t *start, *owner, *popstart, *pidx, *popidx;
    EM_TRY(tmp.alloc(&src, 3 * nsrc));
    EM_TRY(tmp.alloc(&flags, nn));
    EM_TRY(tmp.alloc(&start, n));
    EM_TRY(tmp.alloc(&owner, n));
    EM_TRY(tmp.alloc(&popstart, n));
    EM_TRY(tmp.alloc(&pidx, n));
    EM_TRY(tmp.alloc(&popidx, n));
    EM_CUDA(cudaMemcpyAsync(src, h_src, 3 * nsrc * sizeof(double), cudaMemcpyHostToDevice, st));
    EM_CUDA(cudaMemsetAsync(start, 0, n * sizeof(int32_t), st));
    EM_CUDA(cudaMemsetAsync(popstart, 0, n * sizeof(int32_t), st));
    const double rp2 = p->r_part * p->r_part, rl2 = p->r_leaf * p->r_leaf, th2 = p->theta * p->theta;
    k_node_flags<<<em_grid(nn, 256), 256, 0, st>>>(nn, t->nchild, t->cx, t->cy, t->cz, t->size, nsrc, src, rp2, rl2,
                                                   th2, d_force, flags);
    EM_LAUNCHED(ctx);
    k_reached<<<em_grid(nn, 256), 256, 0, st>>>(nn, t->parent, flags);
    EM_LAUNCHED(ctx);
    k_mark<<<em_grid(nn, 256), 256, 0, st>>>(nn, flags, t->first, t->count, start, owner, popstart);
    EM_LAUNCHED(ctx);
    EM_TRY(em_exclusive_scan_i32(ctx, start, pidx, n));
    EM_TRY(em_exclusive_scan_i32(ctx, popstart, popidx, n));
    int32_t h4[4];
    cudaMemcpyAsync(&h4[0], pidx + n - 1, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
    cudaMemcpyAsync(&h4[1], start + n - 1, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
    cudaMemcpyAsync(&h4[2], popidx + n - 1, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
    cudaMemcpyAsync(&h4[3], popstart + n - 1, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
    EM_CUDA(cudaStreamSynchronize(st));
    const int64_t np = (int64_t)h4[0] + h4[1], npop = (int64_t)h4[2] + h4[3];
    ps->n = np;
    ps->npop = npop;
    // more pseudo-particles than h0_above: every node keeps h_0, no neighbour
    // search and no solve (Section 2.4.2)
    const bool bypass = p->h0_above > 0 && np > (int64_t)p->h0_above;
    DevArena &m = ps->mem;
    EM_TRY(m.alloc(&ps->x, np));
    EM_TRY(m.alloc(&ps->y, np));
    EM_TRY(m.alloc(&ps->z, np));
    EM_TRY(m.alloc(&ps->h, np));
    EM_TRY(m.alloc(&ps->m, np));
    EM_TRY(m.alloc(&ps->origin, np));
    EM_TRY(m.alloc(&ps->first, np));
    EM_TRY(m.alloc(&ps->count, np));
    EM_TRY(m.alloc(&ps->status, np));
    EM_TRY(m.alloc(&ps->node, np));
    double *qx, *qy, *qz;
    EM_TRY(tmp.alloc(&qx, npop));
    EM_TRY(tmp.alloc(&qy, npop));
    EM_TRY(tmp.alloc(&qz, npop));
    k_emit<<<em_grid(n, 256), 256, 0, st>>>(n, start, pidx, owner, popstart, popidx, t->label, t->first, t->count,
                                            t->mass, t->cx, t->cy, t->cz, t->size, t->xs, t->ys, t->zs, t->ms,
                                            t->perm, d_hp, p->h_fact, ps->x, ps->y, ps->z, ps->h, ps->m, ps->origin,
                                            ps->first, ps->count, ps->status, ps->node, bypass ? 2 : -1, qx, qy,
                                            qz);
    EM_LAUNCHED(ctx);
    if (np && !bypass) {
        em::ChunkTree T;
        EM_TRY(em_chunk_tree_build(ctx, tmp, npop, qx, qy, qz, nullptr, 0.0, &T));
        double ext = 0.0;
        for (int k = 0; k < 6; ++k) ext = fmax(ext, fabs(t->box[k]));
        // float rounding of positions and boxes: widen the search radius
        const float margin = (float)(4e-7 * (ext + 1.0));
        float4 *plo;
        EM_TRY(tmp.alloc(&plo, npop));
        k_population_lo<<<em_grid(npop, 256), 256, 0, st>>>(npop, qx, qy, qz, plo);
        EM_LAUNCHED(ctx);
        int *nheavy;
        int32_t *heavy;
        EM_TRY(tmp.alloc(&nheavy, 1));
        EM_TRY(tmp.alloc(&heavy, np));
        EM_CUDA(cudaMemsetAsync(nheavy, 0, sizeof(int), st));
        const Population P{qx, qy, qz, plo};
        k_h_solve<<<em_grid(np * 32, 32 * HS_WARPS), 32 * HS_WARPS, 0, st>>>(np, T, P, ps->x, ps->y, ps->z, p->h_fact,
                                                                              p->h_tol, p->max_newton, margin, ps->h,
                                                                              ps->status, nheavy, heavy);
        EM_LAUNCHED(ctx);
        k_h_solve_heavy<<<(unsigned)std::min<int64_t>(np, 4 * (int64_t)ctx->nsm), 32 * HS_TEAM, 0, st>>>(
            T, P, ps->x, ps->y, ps->z, p->h_fact, p->h_tol, p->max_newton, margin, ps->h, ps->status, nheavy, heavy);
        EM_LAUNCHED(ctx);
    }
    unsigned long long *cnt;
    EM_TRY(tmp.alloc(&cnt, 4));
    EM_CUDA(cudaMemsetAsync(cnt, 0, 4 * sizeof(unsigned long long), st));
    if (np) {
        k_status_count<<<em_grid(np, 256), 256, 0, st>>>(np, ps->status, cnt);
        EM_LAUNCHED(ctx);
    }
    unsigned long long hc[4];
    EM_CUDA(cudaMemcpyAsync(hc, cnt, sizeof hc, cudaMemcpyDeviceToHost, st));
    EM_CUDA(cudaStreamSynchronize(st));
    for (int k = 0; k < 4; ++k) ps->nstatus[k] = (int64_t)hc[k];
    return EM_OK;
}

static int make_pseudo(em_ctx *ctx, const em_tree *t, const double *d_h_particle, int nsrc, const double *h_src,
                       const em_params *p, const uint8_t *d_force, em_pseudo **out)
{
    EM_CHECK_ARG(ctx && t && d_h_particle && h_src && p && out);
    EM_CHECK_ARG(nsrc >= 1 && nsrc <= 4096);
    EM_CHECK_ARG(p->theta >= 0.0 && p->r_part >= 0.0 && p->r_leaf >= 0.0 && p->h_fact > 0.0);
    EM_CHECK_ARG(p->h_tol > 0.0 && p->max_newton >= 0 && p->h0_above >= 0);
    *out = nullptr;
    em_pseudo *ps = new em_pseudo(ctx->stream);
    ps->device = ctx->device;
    int rc = pseudo_impl(ctx, t, d_h_particle, nsrc, h_src, p, d_force, ps);
    if (rc) {
        ps->mem.release();
        delete ps;
        return rc;
    }
    *out = ps;
    const bool bypass = p->h0_above > 0 && ps->n > (int64_t)p->h0_above;
    return ps->nstatus[2] && !bypass ? EM_ENOTCONV : EM_OK;
}

EM_EXPORT int make_pseudo_particles(em_ctx *ctx, const em_tree *t, const double *d_h_particle, int nsrc,
                                    const double *h_src, const em_params *p, em_pseudo **out)
{
    return make_pseudo(ctx, t, d_h_particle, nsrc, h_src, p, nullptr, out);
}

EM_EXPORT int make_pseudo_particles_forced(em_ctx *ctx, const em_tree *t, const double *d_h_particle, int nsrc,
                                           const double *h_src, const em_params *p, const uint8_t *d_force,
                                           em_pseudo **out)
{
    EM_CHECK_ARG(d_force);
    return make_pseudo(ctx, t, d_h_particle, nsrc, h_src, p, d_force, out);
}

namespace {

// Eq. 5 for every node pseudo-particle: under-resolved when its neutral
// fraction is below (K - s_root / s_node) / K (NaN, a pseudo-particle without
// pairs, does not fail; nor does a node of size 0).  cnt[1] counts the failing
// leaves.  A failing internal node not yet flagged, and a failing leaf when
// flag_leaves is set, gets its flag and is counted in cnt[0].
__global__ void k_refine_check(int64_t np, const int32_t *__restrict__ node, const int32_t *__restrict__ nchild,
                               const double *__restrict__ size, const double *__restrict__ f_neu, double K,
                               int flag_leaves, uint8_t *__restrict__ force, unsigned long long *__restrict__ cnt)
{
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= np) return;
    const int32_t a = node[q];
    if (a < 0 || !(size[a] > 0.0)) return;
    const double lim = (K - size[0] / size[a]) / K;
    if (!(f_neu[q] < lim)) return;
    const bool leaf = nchild[a] == 0;
    if (leaf) atomicAdd(&cnt[1], 1ull);
    if ((!leaf || flag_leaves) && !force[a]) {
        force[a] = 1;
        atomicAdd(&cnt[0], 1ull);
    }
}

}  // namespace

EM_EXPORT int refine_check(em_ctx *ctx, const em_pseudo *ps, const em_tree *t, const double *d_f_neu, double K,
                           int flag_leaves, uint8_t *d_force, int64_t *h_nnew, int64_t *h_nleaf)
{
    EM_CHECK_ARG(ctx && ps && t && d_f_neu && d_force && h_nnew);
    EM_CHECK_ARG(K > 1.0);
    EM_CHECK_ARG(flag_leaves == 0 || flag_leaves == 1);
    *h_nnew = 0;
    if (h_nleaf) *h_nleaf = 0;
    if (ps->n == 0 || t->nnode == 0) return EM_OK;
    DevArena tmp(ctx->stream, true);
    unsigned long long *cnt;
    EM_TRY(tmp.alloc(&cnt, 2));
    EM_CUDA(cudaMemsetAsync(cnt, 0, 2 * sizeof *cnt, ctx->stream));
    k_refine_check<<<em_grid(ps->n, 256), 256, 0, ctx->stream>>>(ps->n, ps->node, t->nchild, t->size, d_f_neu, K,
                                                                 flag_leaves, d_force, cnt);
    EM_LAUNCHED(ctx);
    unsigned long long h[2] = {0, 0};
    EM_CUDA(cudaMemcpyAsync(h, cnt, sizeof h, cudaMemcpyDeviceToHost, ctx->stream));
    EM_CUDA(cudaStreamSynchronize(ctx->stream));
    *h_nnew = (int64_t)h[0];
    if (h_nleaf) *h_nleaf = (int64_t)h[1];
    return EM_OK;
}
