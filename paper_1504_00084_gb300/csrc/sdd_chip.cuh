// Subdomain solves held in shared memory and registers (included by sdd_solve.cu).
//
// The same iteration as solve_body -- FP64 residual and refinement, conjugate gradients, one V-cycle
// as preconditioner -- for subdomains that fit on chip: one CTA, or a cluster of 2 to 16 CTAs that
// own contiguous strips of rows.  The passes of solve_body are a few microseconds of global-memory
// latency and a barrier each, about 50 of them per CG iteration; here a pass is shared-memory
// traffic and a barrier, a few hundred nanoseconds.  Measured (face coefficients and solve, from
// global memory / on chip): 16 subdomains of 63 x 63, 1.415 / 0.334 ms; 4 of 15 x 15 in FP64,
// 0.571 / 0.096; 16 of 31 x 31, 0.567 / 0.150; 4 of 127 x 127, 3.84 / 0.60; 4 of 255 x 255,
// 4.65 / 0.70.  What bounds it: at 63 x 63 half the time is the FP64 residual, which one SM's unit
// works at for 20 us a sweep; below that the chain of passes; in clusters the barriers, about 0.9 us
// each, which is why the team is the smallest that holds the subdomain.

// Storage.  Each level holds x (the correction), t (the residual; at level 0 the same array serves
// p between the cycles) and the face coefficients, diagonal and its reciprocal in shared memory, a
// row as two planes (even and odd columns), so that a half-sweep's lanes read consecutive words.
// Rims are zero, so that no pass tests for the boundary.  The right-hand side of a coarse level is
// in shared memory; at level 0 every thread owns fixed nodes (kSlots at most) whose residual,
// direction, product and correction stay in its registers.
// Clusters.  A level is split by rows over the CTAs while it has more than kShared nodes and every
// CTA a row; a thread that writes an edge row also writes the neighbour CTA's halo copy of it
// (distributed shared memory), so that every read is local, and the pass ends in a cluster barrier.
// Smaller levels are held and computed by every CTA, whole.
//
// FP32 arithmetic is solve_body's operation for operation: every product, sum and quotient rounds
// as there, quotients by the diagonal through its correctly rounded reciprocal and two residual
// corrections, which give the correctly rounded quotient (Markstein).  Dot products are compensated
// FP32 pairs (exact products, 48-bit sums) instead of FP64, whose unit would need 8 us for the 16
// thousand products of a 63 x 63 iteration; step lengths are their quotients rounded once to FP32.
// What these see is scaled by powers of two (chip_body), so that FP32's range is enough.
// In FP64 mode the vectors and dot products of the CG iteration are FP64, the V-cycle that
// preconditions it FP32.
#pragma once

#include <cooperative_groups.h>

#include <type_traits>

namespace {

namespace cg = cooperative_groups;

constexpr int kChipLevels = 9;   // sizes up to 256 rows and columns
constexpr int kShared = 300;     // levels of at most this many nodes are held whole by every CTA
constexpr int kChipWidth = 16;   // CTAs of the widest cluster
constexpr int kChipSmem = 232448 - 2048;  // dynamic shared memory a CTA may have beside its tables

// nodes a thread may own at level 0
template <typename TI> struct ChipSlots;
template <> struct ChipSlots<float> { static constexpr int n = 8; };
template <> struct ChipSlots<double> { static constexpr int n = 4; };

// What one thread works out for all: the squared norm at which a component is done, the components' scale, what
// the residual in hand has still to be multiplied with (a TI), and what comes next.
struct ChipScalars {
    double bn[2], goal[2], stop[2], more[2], rr[2];
    int scale[2], target, state;
};
enum { kChipSolve, kChipDone, kChipAgain };

// One level as a CTA holds it.  Offsets are bytes into the dynamic shared memory, alike in every CTA
// of a cluster.
struct ChipLevel {
    int nx, ny;              // the whole level
    int r0, nr;              // rows of this CTA
    int below;               // rows of the CTA before this one (a halo row's place there)
    int H, F, C;             // plane lengths: x and t; faces along xi; the other arrays
    int w2, kcs;             // log2 of the lanes of a warp, and of the warps, that share a row
    int dist;                // split over the cluster
    int x, t, p, b, ce, cn, dg, inv;  // p: level 0
};

__host__ __device__ inline int chip_lanes_log2(int nx)
{
    const int half = (nx + 1) / 2;
    int w = 0;
    while ((1 << w) < half && w < 5) ++w;
    return w;
}

// log2 of the warps that share a row.
__host__ __device__ inline int chip_chunks_log2(int ni)
{
    int k = 0;
    while ((32 << k) < (ni + 1) / 2) ++k;
    return k;
}
// Levels of an ni x nj interior over cw CTAs: sizes, offsets and the bytes they take.  `elem`: bytes
// of a component of p (level 0).
__host__ __device__ inline int chip_levels(int ni, int nj, int cw, int elem, ChipLevel* L, int* levels_out, int* p_off)
{
    const int levels = mg_levels(ni, nj);
    int off = 0;
    auto take = [&](int bytes) { const int o = off; off += (bytes + 15) / 16 * 16; return o; };
    int nx = ni, ny = nj, rows = (nj + cw - 1) / cw, least = nj / cw;
    bool dist = cw > 1;
    for (int l = 0; l < levels && l < kChipLevels; ++l) {
        if (l > 0) {
            nx = mg_coarse(nx);
            ny = mg_coarse(ny);
            rows = (rows + 1) / 2;  // a strip of n rows owns (n + 1) / 2 coarse ones at most
            least /= 2;
            if (dist && (nx * ny <= kShared || least < 1)) dist = false;
            if (!dist) rows = ny;
        }
        ChipLevel v{};
        v.nx = nx; v.ny = ny; v.dist = dist ? 1 : 0;
        v.H = (nx + 3) / 2; v.F = (nx + 2) / 2; v.C = (nx + 1) / 2;
        v.w2 = chip_lanes_log2(nx); v.kcs = chip_chunks_log2(nx);
        v.x = take((rows + 2) * 2 * v.H * 8);
        v.t = take((rows + 2) * 2 * v.H * 8);
        v.b = l > 0 ? take(rows * 2 * v.C * 8) : 0;
        v.ce = take(rows * 2 * v.F * 4);
        v.cn = take((rows + 1) * 2 * v.C * 4);
        v.dg = take(rows * 2 * v.C * 4);
        v.inv = take(rows * 2 * v.C * 4);
        if (l == 0) *p_off = elem == 4 ? v.t : take((rows + 2) * 2 * v.H * 16);
        L[l] = v;
    }
    *levels_out = levels;
    return off;
}

// Slots a thread needs at level 0 with nw warps a CTA (0: a step of rows would be odd).
__host__ __device__ inline int chip_slots(int ni, int nj, int cw, int nw)
{
    const int rows = (nj + cw - 1) / cw, step = (nw >> chip_chunks_log2(ni)) << (5 - chip_lanes_log2(ni));
    return step < 2 ? 0 : 2 * ((rows + step - 1) / step);
}

// Whether every level below 0 gives a thread at most one node of each colour with nw warps a CTA.
__host__ __device__ inline bool chip_levels_fit(const ChipLevel* L, int levels, int cw, int nw)
{
    int rows = (L[0].ny + cw - 1) / cw;
    for (int l = 1; l < levels; ++l) {
        rows = L[l].dist ? (rows + 1) / 2 : L[l].ny;
        if (((nw >> L[l].kcs) << (5 - L[l].w2)) < rows) return false;
    }
    return true;
}

// ---- compensated FP32 pairs ----------------------------------------------------------------
struct F2 { float h, l; };
__device__ __forceinline__ F2 ff_add(F2 a, F2 b)
{
    const float s = __fadd_rn(a.h, b.h), z = __fsub_rn(s, a.h);
    const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, z)), __fsub_rn(b.h, z));
    const float l = __fadd_rn(e, __fadd_rn(a.l, b.l));
    const float h = __fadd_rn(s, l);
    return F2{h, __fsub_rn(l, __fsub_rn(h, s))};
}
// a += x y, the product exact; the low part is not renormalised until ff_add
__device__ __forceinline__ void ff_mac(F2& a, float x, float y)
{
    const float p = __fmul_rn(x, y), pe = __fmaf_rn(x, y, -p);
    const float s = __fadd_rn(a.h, p), z = __fsub_rn(s, a.h);
    const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, z)), __fsub_rn(p, z));
    a.h = s;
    a.l = __fadd_rn(a.l, __fadd_rn(e, pe));
}
// a / b rounded to FP32 (b > 0)
__device__ __forceinline__ float ff_div(F2 a, F2 b)
{
    const float q = __fdiv_rn(a.h, b.h);
    const float r = __fadd_rn(__fmaf_rn(-q, b.h, a.h), __fmaf_rn(-q, b.l, a.l));
    return __fadd_rn(q, __fdiv_rn(r, b.h));
}
__device__ __forceinline__ bool ff_le(F2 a, F2 b) { return a.h < b.h || (a.h == b.h && a.l <= b.l); }

// Correctly rounded (ax, ay) / dg from inv = 1 / dg rounded: after one correction the quotient is
// within one unit in the last place, after the second it is the rounded one (Markstein).  Exact
// zeros stay zero; numerators below 2^-100, whose corrections would lose bits, are less than 2^-80 of
// the residual they come from, which is scaled to 2^-20 at least.
__device__ __forceinline__ float2 div_diag(float ax, float ay, float dg, float inv)
{
    float qx = __fmul_rn(ax, inv), qy = __fmul_rn(ay, inv);
    qx = __fmaf_rn(__fmaf_rn(-qx, dg, ax), inv, qx);
    qy = __fmaf_rn(__fmaf_rn(-qy, dg, ay), inv, qy);
    qx = __fmaf_rn(__fmaf_rn(-qx, dg, ax), inv, qx);
    qy = __fmaf_rn(__fmaf_rn(-qy, dg, ay), inv, qy);
    return make_float2(qx, qy);
}

template <typename V> __device__ __forceinline__ V* at(char* base, int off) { return reinterpret_cast<V*>(base + off); }

// The CTA's view of its team.
template <bool CL> struct Chip {
    char* sm;                 // dynamic shared memory
    char *dn, *up;            // the same of the CTAs before and after (CL)
    int rank, cw, warp, nw, lane;
    __device__ __forceinline__ void sync(int dist) const
    {
        if (CL && dist) cg::this_cluster().sync();
        else __syncthreads();
    }
};

// A thread's node of one colour at a level: row jl of this CTA, column c + 2 k, and its places in x and
// t (self, west neighbour; east is the next word after west), in the xi faces (west, east) and in the
// other arrays.  Below level 0 every level gives a thread at most one node of each colour
// (chip_levels_fit).
struct ChipAt { int self, w, fw, fe, c, jl, k, cc; bool on; };
__device__ __forceinline__ ChipAt chip_at(const ChipLevel& v, int colour, int warp, int nw, int lane)
{
    ChipAt o;
    const int kc = v.kcs;
    o.jl = ((warp >> kc) << (5 - v.w2)) + (lane >> v.w2);
    o.k = (lane & ((1 << v.w2) - 1)) + 32 * (warp & ((1 << kc) - 1));
    o.cc = (v.r0 + o.jl + colour) & 1;
    o.self = ((o.jl + 1) * 2 + 1 - o.cc) * v.H + o.k + o.cc;
    o.w = ((o.jl + 1) * 2 + o.cc) * v.H + o.k;
    o.fw = (o.jl * 2 + o.cc) * v.F + o.k;
    o.fe = (o.jl * 2 + 1 - o.cc) * v.F + o.k + o.cc;
    o.c = (o.jl * 2 + o.cc) * v.C + o.k;
    o.on = o.jl < v.nr && o.cc + 2 * o.k < v.nx;
    return o;
}
// Store to x or t (array offset `off`) and to the neighbour CTA's halo copy of an edge row.
template <bool CL>
__device__ __forceinline__ void put(const Chip<CL>& T, const ChipLevel& v, int off, const ChipAt& o, float2 val)
{
    at<float2>(T.sm, off)[o.self] = val;
    if (CL && v.dist) {
        if (o.jl == 0 && T.rank > 0) at<float2>(T.dn, off)[o.self + v.below * 2 * v.H] = val;
        if (o.jl == v.nr - 1 && T.rank + 1 < T.cw) at<float2>(T.up, off)[o.self - v.nr * 2 * v.H] = val;
    }
}
// sum over the neighbours of c_nb x_nb, west, east, south, north
__device__ __forceinline__ float2 offdiag(char* sm, const ChipLevel& v, const ChipAt& o)
{
    const float2* x = at<float2>(sm, v.x);
    const float* ce = at<float>(sm, v.ce);
    const float* cn = at<float>(sm, v.cn);
    const float cW = ce[o.fw], cE = ce[o.fe], cS = cn[o.c], cN = cn[o.c + 2 * v.C];
    const float2 w = x[o.w], e = x[o.w + 1], s = x[o.self - 2 * v.H], n = x[o.self + 2 * v.H];
    return make_float2(__fmaf_rn(cN, n.x, __fmaf_rn(cS, s.x, __fmaf_rn(cE, e.x, __fmul_rn(cW, w.x)))),
                       __fmaf_rn(cN, n.y, __fmaf_rn(cS, s.y, __fmaf_rn(cE, e.y, __fmul_rn(cW, w.y)))));
}

// The passes of a level below 0 at a thread's node.
template <bool CL>
__device__ __forceinline__ void chip_first(const Chip<CL>& T, const ChipLevel& v, const ChipAt& o)
{
    if (!o.on) return;
    const float2 b = at<float2>(T.sm, v.b)[o.c];
    put<CL>(T, v, v.x, o, div_diag(b.x, b.y, at<float>(T.sm, v.dg)[o.c], at<float>(T.sm, v.inv)[o.c]));
}
template <bool CL>
__device__ __forceinline__ void chip_sweep(const Chip<CL>& T, const ChipLevel& v, const ChipAt& o)
{
    if (!o.on) return;
    const float2 b = at<float2>(T.sm, v.b)[o.c], u = offdiag(T.sm, v, o);
    put<CL>(T, v, v.x, o, div_diag(__fadd_rn(b.x, u.x), __fadd_rn(b.y, u.y), at<float>(T.sm, v.dg)[o.c],
                                   at<float>(T.sm, v.inv)[o.c]));
}
template <bool CL>
__device__ __forceinline__ void chip_residual(const Chip<CL>& T, const ChipLevel& v, const ChipAt& o)
{
    if (!o.on) return;
    const float2 b = at<float2>(T.sm, v.b)[o.c], u = offdiag(T.sm, v, o), x = at<float2>(T.sm, v.x)[o.self];
    const float dg = at<float>(T.sm, v.dg)[o.c];
    put<CL>(T, v, v.t, o, make_float2(__fsub_rn(b.x, __fmaf_rn(dg, x.x, -u.x)), __fsub_rn(b.y, __fmaf_rn(dg, x.y, -u.y))));
}
// b of the next level: full weighting of t.  The coarse rows this CTA computes are those whose fine
// row 2 J + 1 it owns; a level held whole gets them from every CTA.
template <bool CL>
__device__ __forceinline__ void chip_restrict(const Chip<CL>& T, const ChipLevel& F, const ChipLevel& C, int warp, int nw)
{
    const float2* t = at<float2>(T.sm, F.t);
    const int J0 = F.r0 / 2, J1 = min((F.r0 + F.nr) / 2, C.ny);
    const int w2 = min(C.w2 + 1, 5), W = 1 << w2, rp = 32 >> w2;
    for (int J = J0 + warp * rp + (T.lane >> w2); J < J1; J += nw * rp)
        for (int I = T.lane & (W - 1); I < C.nx; I += W) {
            // fine node (2 I + 1, 2 J + 1): column 2 I + 1 is the odd column k = I; its neighbours the
            // even columns I and I + 1
            const int row = (2 * J + 1 - F.r0 + 1) * 2 * F.H;
            float2 a = make_float2(0.f, 0.f);
#pragma unroll
            for (int dj = -1; dj <= 1; ++dj) {
                const float2* r = t + row + dj * 2 * F.H;
                const float w1 = dj == 0 ? 0.125f : 0.0625f, w2_ = 2.f * w1;
                const float2 v0 = r[F.H + I], v1 = r[I + 1], v2 = r[F.H + I + 1];
                a.x = __fmaf_rn(w1, v0.x, a.x); a.y = __fmaf_rn(w1, v0.y, a.y);
                a.x = __fmaf_rn(w2_, v1.x, a.x); a.y = __fmaf_rn(w2_, v1.y, a.y);
                a.x = __fmaf_rn(w1, v2.x, a.x); a.y = __fmaf_rn(w1, v2.y, a.y);
            }
            const int o = ((J - C.r0) * 2 + (I & 1)) * C.C + (I >> 1);
            if (CL && F.dist && !C.dist) {
                for (int r = 0; r < T.cw; ++r) at<float2>(cg::this_cluster().map_shared_rank(T.sm, r), C.b)[o] = a;
            } else {
                at<float2>(T.sm, C.b)[o] = a;
            }
        }
}
// f + the bilinear interpolation of the next level's x at the colour-0 node of row j (whole level),
// column cc + 2 k; the other colour is overwritten by the half-sweep that follows before anything
// reads it.
__device__ __forceinline__ float2 prolonged(char* sm, const ChipLevel& C, float2 f, int j, int cc, int k)
{
    const float2* x = at<float2>(sm, C.x);
    // coarse node (I, J) is x[((J - r0 + 1) * 2 + 1 - (I & 1)) * H + (I + 1) / 2]
    auto val = [&](int I, int J) { return x[((J - C.r0 + 1) * 2 + 1 - (I & 1)) * C.H + ((I + 1) >> 1)]; };
    if (cc) {  // odd row, odd column: a coarse node
        const float2 v = val(k, (j - 1) / 2);
        return make_float2(__fadd_rn(f.x, v.x), __fadd_rn(f.y, v.y));
    }
    // even row and column: the four around it, column k - 1 before k, row j / 2 - 1 before j / 2
    const int J = j / 2;
    const float2 a = val(k - 1, J - 1), b = val(k - 1, J), d = val(k, J - 1), e = val(k, J);
    const float sx = __fmaf_rn(0.25f, e.x, __fmaf_rn(0.25f, d.x, __fmaf_rn(0.25f, b.x, 0.25f * a.x)));
    const float sy = __fmaf_rn(0.25f, e.y, __fmaf_rn(0.25f, d.y, __fmaf_rn(0.25f, b.y, 0.25f * a.y)));
    return make_float2(__fadd_rn(f.x, sx), __fadd_rn(f.y, sy));
}

// Levels 1 .. levels - 1 of the V-cycle: level 1's right-hand side is in place; its correction is
// left in x.  Levels lt .. are run by warp 0 alone, which needs no barrier between their passes.
template <bool CL>
__device__ __forceinline__ void chip_coarse_cycle(const Chip<CL>& T, const ChipLevel* L, int levels, int lt)
{
    const int last = levels - 1;
#pragma unroll 1
    for (int l = 1; l <= last; ++l) {
        const bool tail = l >= lt;
        if (tail && T.warp != 0) break;
        const ChipLevel v = L[l];
        const int w = tail ? 0 : T.warp, nw = tail ? 1 : T.nw;
        const ChipAt o0 = chip_at(v, 0, w, nw, T.lane), o1 = chip_at(v, 1, w, nw, T.lane);
        chip_first(T, v, o0);
        if (tail) __syncwarp(); else T.sync(v.dist);
        if (l == last) {
            // coarsest: symmetric sweeps, colours (0) 1 1 0 | 0 1 1 0 | ...; one node is solved already
            const int n = v.nx * v.ny == 1 ? 0 : 4 * kCoarseSweeps - 1;
#pragma unroll 1
            for (int m = 0; m < n; ++m) {
                if ((m + 2) & 2) chip_sweep(T, v, o1); else chip_sweep(T, v, o0);
                if (tail) __syncwarp(); else T.sync(v.dist);
            }
            break;
        }
        chip_sweep(T, v, o1);
        if (tail) __syncwarp(); else T.sync(v.dist);
        chip_residual(T, v, o0);
        chip_residual(T, v, o1);
        if (tail) __syncwarp(); else T.sync(v.dist);
        chip_restrict(T, v, L[l + 1], w, nw);
        if (tail) __syncwarp(); else T.sync(v.dist);
    }
#pragma unroll 1
    for (int l = last - 1; l >= 1; --l) {
        const bool tail = l >= lt;
        if (tail && T.warp != 0) continue;
        const ChipLevel v = L[l];
        const int w = tail ? 0 : T.warp, nw = tail ? 1 : T.nw;
        const ChipAt o0 = chip_at(v, 0, w, nw, T.lane), o1 = chip_at(v, 1, w, nw, T.lane);
        if (l == lt - 1 && lt <= last) __syncthreads();  // warp 0 has left the tail's correction
        if (o0.on) put<CL>(T, v, v.x, o0, prolonged(T.sm, L[l + 1], at<float2>(T.sm, v.x)[o0.self], v.r0 + o0.jl, o0.cc, o0.k));
        if (tail) __syncwarp(); else T.sync(v.dist);
        chip_sweep(T, v, o1);
        if (tail) __syncwarp(); else T.sync(v.dist);
        chip_sweep(T, v, o0);
        if (tail) __syncwarp(); else T.sync(v.dist);
    }
    if (lt <= 1) __syncthreads();
}

// Sums over the team, in a fixed order: a warp tree, the CTA's warps, the CTAs.  A cluster's CTAs
// send their totals to each other; the buffers alternate, so that one team barrier per sum suffices.
template <typename V> struct SumOf;
template <> struct SumOf<F2> {
    __device__ static F2 zero() { return F2{0.f, 0.f}; }
    __device__ static F2 add(F2 a, F2 b) { return ff_add(a, b); }
    __device__ static F2 shfl(F2 a, int o) { return F2{__shfl_xor_sync(kFull, a.h, o), __shfl_xor_sync(kFull, a.l, o)}; }
    __device__ static F2 from(F2 a, int lane) { return F2{__shfl_sync(kFull, a.h, lane), __shfl_sync(kFull, a.l, lane)}; }
    __device__ static F2 pick(bool c, F2 a, F2 b) { return F2{c ? a.h : b.h, c ? a.l : b.l}; }
};
template <> struct SumOf<double> {
    __device__ static double zero() { return 0.0; }
    __device__ static double add(double a, double b) { return a + b; }
    __device__ static double shfl(double a, int o) { return __shfl_xor_sync(kFull, a, o); }
    __device__ static double from(double a, int lane) { return __shfl_sync(kFull, a, lane); }
    __device__ static double pick(bool c, double a, double b) { return c ? a : b; }
};
constexpr int kRedBytes = 8 * 4 * (16 + 2 * 16);  // a warp's totals; two buffers of CTAs' totals
// Totals over the groups of 32 / NV lanes, lane group q holding value q: the values are spread over the
// lanes while they are halved, so that a warp adds 5 (NV = 2) or 6 pairs instead of 10 or 20.
template <int NV, typename V>
__device__ __forceinline__ V chip_spread(V (&v)[NV], int lane)
{
    if constexpr (NV == 4) {
        const bool hi = lane & 16;
        const V a = SumOf<V>::pick(hi, v[2], v[0]), b = SumOf<V>::pick(hi, v[3], v[1]);
        const V c = SumOf<V>::pick(hi, v[0], v[2]), d = SumOf<V>::pick(hi, v[1], v[3]);
        v[0] = SumOf<V>::add(a, SumOf<V>::shfl(c, 16));
        v[1] = SumOf<V>::add(b, SumOf<V>::shfl(d, 16));
    }
    constexpr int half = NV == 4 ? 8 : 16;
    const bool hi = lane & half;
    const V a = SumOf<V>::pick(hi, v[1], v[0]), c = SumOf<V>::pick(hi, v[0], v[1]);
    V t = SumOf<V>::add(a, SumOf<V>::shfl(c, half));
#pragma unroll
    for (int o = half / 2; o > 0; o >>= 1) t = SumOf<V>::add(t, SumOf<V>::shfl(t, o));
    return t;
}
// v[q] = sum of part[16 q .. 16 q + n), n <= 16, in every lane
template <int NV, typename V>
__device__ __forceinline__ void chip_gather(V (&v)[NV], const V* part, int n, int lane)
{
    constexpr int group = 32 / NV;
    const int q = lane / group, k = lane % group;
    V t = k < n ? part[q * 16 + k] : SumOf<V>::zero();
    if (NV == 4 && k + 8 < n) t = SumOf<V>::add(t, part[q * 16 + k + 8]);
#pragma unroll
    for (int o = group / 2; o > 0; o >>= 1) t = SumOf<V>::add(t, SumOf<V>::shfl(t, o));
#pragma unroll
    for (int p = 0; p < NV; ++p) v[p] = SumOf<V>::from(t, p * group);
}
// WARP0: the totals in the first warp alone (an FP64 addition costs an SM 16 clocks a warp).
template <bool CL, int NV, typename V, bool WARP0 = false>
__device__ __forceinline__ void chip_sum(const Chip<CL>& T, V (&v)[NV], char* red, int& turn)
{
    // without a cluster the warps' totals alternate instead
    V* part = reinterpret_cast<V*>(red) + (CL ? 0 : (turn & 1) * 64);
    V* team = reinterpret_cast<V*>(red) + 64 + (turn & 1) * 64;
    ++turn;
    const V own = chip_spread<NV>(v, T.lane);
    if (T.lane % (32 / NV) == 0) part[T.lane / (32 / NV) * 16 + T.warp] = own;
    __syncthreads();
    if constexpr (CL) {
        if (T.warp == 0) {
            chip_gather<NV>(v, part, T.nw, T.lane);
            if (T.lane < T.cw) {
                V* to = cg::this_cluster().map_shared_rank(team, T.lane);
#pragma unroll
                for (int q = 0; q < NV; ++q) to[q * 16 + T.rank] = v[q];
            }
        }
        T.sync(1);
        if (!WARP0 || T.warp == 0) chip_gather<NV>(v, team, T.cw, T.lane);
    } else {
        if (!WARP0 || T.warp == 0) chip_gather<NV>(v, part, T.nw, T.lane);
    }
}

// 2^k, |k| <= 1022
__device__ __forceinline__ double pow2(int k) { return __hiloint2double((1023 + k) << 20, 0); }
// Exponent of d: -1023 for zero and subnormal numbers, 1024 for what is not finite.
__device__ __forceinline__ int exponent(double d) { return ((__double2hiint(d) >> 20) & 0x7FF) - 1023; }
// d 2^k as a float, rounded to nearest even, |k| <= 1100: integer operations, no branch.  Below the normal range 0,
// above it an infinity; what is not finite becomes a NaN.
__device__ __forceinline__ float float_scaled(double d, int k)
{
    const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
    const int E = (int)((hi >> 20) & 0x7FFu);
    const uint64_t u = (((uint64_t)(hi + ((uint32_t)k << 20)) << 32) | lo) + 0x0FFFFFFFu + ((lo >> 29) & 1u);
    uint32_t v = (uint32_t)(u >> 29) + 0x40000000u;
    if ((uint32_t)(E + k) - 0x381u > 0xFCu) v = E + k < 0x381 ? 0u : 0x7F800000u;
    if (E == 0x7FF) v = 0x7FC00000u;
    return __uint_as_float(v | (hi & 0x80000000u));
}
// A coefficient as the V-cycle takes it.  FP32 mode: the solve's own.  FP64 mode: times 2^k, which puts those around the
// subdomain's middle near 1 (the cycle's result is then 2^-k times as large, which the iteration does not notice),
// and no further from it than FP32 holds over all levels; only the preconditioner sees the bounds.
template <typename TI> __device__ __forceinline__ float chip_face(const void* f, const double* f64, long id, int k)
{
    if constexpr (sizeof(TI) == 8) return fminf(fmaxf(float_scaled(f64[id], k), 0x1p-100f), 0x1p100f);
    else return static_cast<const float*>(f)[id];
}
template <typename TI> __device__ __forceinline__ float chip_mass(double d, int k)
{
    if constexpr (sizeof(TI) == 8) return fminf(float_scaled(d, k), 0x1p100f);
    else return (float)d;
}
// The largest exponent of the mass and the face coefficients at node id.
__device__ __forceinline__ int chip_exponent(const SolveParams& P, long id)
{
    return max(exponent(P.form == 0 ? 1.0 : P.om64[id]), max(exponent(P.ce64[id]), exponent(P.cn64[id])));
}
// v 2^k
template <typename TI> __device__ __forceinline__ TI to_inner(double v, int k)
{
    if constexpr (sizeof(TI) == 8) return v * pow2(k);
    else return float_scaled(v, k);
}
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// Coefficients of every level, level by level: a coarse face spans two fine faces (a quarter of their
// series combination), except the face to the rim after an even fine size, half of the one it
// spans.  A strip's outermost coarse faces may need its neighbours' fine ones, which it reads from
// their shared memory; a level held whole gets each CTA's part from it.
template <typename TI, bool CL>
__device__ __forceinline__ void chip_setup(const Chip<CL>& T, const SolveParams& P, const ChipLevel* L, int levels, int i0,
                                           int j0, int k)
{
    auto series = [](float a, float b) {
        const float m = __fmul_rn(0.5f * a, b), n = __fadd_rn(a, b);
        return m >= 0x1p-100f && m <= 0x1p120f ? __fdiv_rn(m, n) : 0.5f * a * __fdiv_rn(b, n);
    };
#pragma unroll 1
    for (int l = 0; l < levels; ++l) {
        const ChipLevel v = L[l], u = L[l > 0 ? l - 1 : 0];
        // the rows this CTA computes: its own, or (a whole level under a split one) those under its fine rows
        const bool spread = CL && u.dist && !v.dist;
        const int ja = spread ? u.r0 / 2 : v.r0, jb = spread ? min((u.r0 + u.nr) / 2, v.ny) : v.r0 + v.nr;
        // face row jb is the next CTA's too, except the last
        const int gb = spread && jb < v.ny ? jb - 1 : jb;
        auto store = [&](int off, int o, float c) {
            if (spread) {
                for (int r = 0; r < T.cw; ++r) at<float>(cg::this_cluster().map_shared_rank(T.sm, r), off)[o] = c;
            } else {
                at<float>(T.sm, off)[o] = c;
            }
        };
        for (int j = ja + T.warp; j < jb; j += T.nw)
            for (int f = T.lane; f <= v.nx; f += 32) {
                float c;
                if (l == 0) {
                    c = chip_face<TI>(P.ce, P.ce64, (long)(j0 + 1 + j) * P.nx + (i0 + f), k);
                } else {
                    const float* fe = at<float>(T.sm, u.ce) + (2 * j + 1 - u.r0) * 2 * u.F + f;  // face 2 f of row 2 j + 1
                    c = 2 * f + 1 > u.nx ? 0.5f * fe[0] : series(fe[0], fe[u.F]);
                }
                store(v.ce, ((j - v.r0) * 2 + (f & 1)) * v.F + (f >> 1), c);
            }
        for (int g = ja + T.warp; g <= gb; g += T.nw)
            for (int i = T.lane; i < v.nx; i += 32) {
                float c;
                if (l == 0) {
                    c = chip_face<TI>(P.cn, P.cn64, (long)(j0 + g) * P.nx + (i0 + 1 + i), k);
                } else {
                    auto fine = [&](int y) {  // face row y of the level above, column 2 i + 1
                        char* from = T.sm;
                        int row = y - u.r0;
                        if constexpr (CL) {
                            if (row < 0) { from = T.dn; row += u.below; }
                            else if (row > u.nr) { from = T.up; row -= u.nr; }
                        }
                        return at<float>(from, u.cn)[(row * 2 + 1) * u.C + i];
                    };
                    c = 2 * g + 1 > u.ny ? 0.5f * fine(2 * g) : series(fine(2 * g), fine(2 * g + 1));
                }
                store(v.cn, ((g - v.r0) * 2 + (i & 1)) * v.C + (i >> 1), c);
            }
        T.sync(u.dist);
    }
#pragma unroll 1
    for (int l = 0; l < levels; ++l) {
        const ChipLevel v = L[l];
        const float* ce = at<float>(T.sm, v.ce);
        const float* cn = at<float>(T.sm, v.cn);
        for (int j = T.warp; j < v.nr; j += T.nw)
            for (int i = T.lane; i < v.nx; i += 32) {
                const int o = (j * 2 + (i & 1)) * v.C + (i >> 1);
                double w = 1.0;
                if (P.form != 0)  // coarse node (I, J) is fine node ((I + 1) 2^l - 1, (J + 1) 2^l - 1)
                    w = P.om64[(long)(j0 + ((v.r0 + j + 1) << l)) * P.nx + (i0 + ((i + 1) << l))];
                const float d = chip_mass<TI>(w, k);
                const float dg = d + ce[(j * 2 + (i & 1)) * v.F + (i >> 1)] + ce[(j * 2 + ((i + 1) & 1)) * v.F + ((i + 1) >> 1)] +
                                 cn[o] + cn[o + 2 * v.C];
                at<float>(T.sm, v.dg)[o] = dg;
                at<float>(T.sm, v.inv)[o] = __frcp_rn(dg);
            }
    }
    T.sync(1);
}

template <typename TI> struct ChipVec;
template <> struct ChipVec<float> { typedef float2 V; typedef F2 Sum; };
template <> struct ChipVec<double> { typedef double2 V; typedef double Sum; };

__device__ __forceinline__ void mac(F2& a, float x, float y) { ff_mac(a, x, y); }
__device__ __forceinline__ void mac(double& a, double x, double y) { a = fma(x, y, a); }
__device__ __forceinline__ float ratio(F2 a, F2 b) { return b.h > 0.f ? ff_div(a, b) : 0.f; }
__device__ __forceinline__ double ratio(double a, double b) { return b > 0.0 ? a / b : 0.0; }
__device__ __forceinline__ F2 from_double(double t, F2) { const float h = (float)t; return F2{h, (float)(t - (double)h)}; }
__device__ __forceinline__ double from_double(double t, double) { return t; }
__device__ __forceinline__ bool at_most(F2 a, F2 b) { return ff_le(a, b); }
__device__ __forceinline__ bool at_most(double a, double b) { return a <= b; }
__device__ __forceinline__ float2 to_f2(float2 v) { return v; }
__device__ __forceinline__ float2 to_f2(double2 v) { return make_float2((float)v.x, (float)v.y); }

// d 2^k, d >= 0, by its exponent: 0 where d or the result is below the normal range
__device__ __forceinline__ double times_pow2(double d, int k)
{
    const int e = exponent(d);
    if (e == 1024) return d;
    if (e == -1023 || e + k < -1022) return 0.0;
    if (e + k > 1023) return INFINITY;
    return __hiloint2double(__double2hiint(d) + (int)((uint32_t)k << 20), __double2loint(d));
}
// 2^k: |k| <= 60 (float), <= 1022 (double)
template <typename TI> __device__ __forceinline__ TI pow2_of(int k)
{
    if constexpr (sizeof(TI) == 8) return pow2(k);
    else return __int_as_float((127 + k) << 23);
}

// From the squared norms r0, r1 of a sweep's residual (before its scale): whether the solve is done, what the residual
// in hand is still to be multiplied with, and where the sweep's iteration stops.  One thread: the FP64 unit would take
// microseconds for all of them.  Not inlined, which leaves the kernel's registers to the iteration (340 -> 336 us
// of 16 subdomains of 63 x 63; 334 with the norms' totals in one warp).
template <typename TI>
__device__ __noinline__ void chip_decide(ChipScalars* scal, double r0, double r1, double rtol)
{
    typedef typename ChipVec<TI>::Sum Sum;
    const double rr[2] = {r0, r1};
    bool fine = true;
    int state = kChipSolve;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const double goal = scal->goal[c];
        if (goal > 1e-290) fine = fine && rr[c] <= goal;
        else fine = fine && sqrt(scal->bn[c] > 0 ? rr[c] / scal->bn[c] : rr[c]) <= rtol;
        const int more = rr[c] > 0.0 ? scal->target - (exponent(rr[c]) >> 1) - scal->scale[c] : 0;
        const int k = scal->scale[c] + more;
        if (abs(more) > 60 && scal->state != kChipAgain) state = kChipAgain;
        *reinterpret_cast<TI*>(&scal->more[c]) = pow2_of<TI>(more);
        scal->scale[c] = k;
        // squared residual norm at which a component is done: half the target in FP64 (but not below 1e-14 of
        // the start), 1e-5 of the start in FP32
        const double st = sizeof(TI) == 8 ? fmin(0.25 * rr[c], fmax(0.25 * goal, 1e-28 * rr[c])) : 1e-10 * rr[c];
        *reinterpret_cast<Sum*>(&scal->stop[c]) = from_double(times_pow2(st, 2 * k), Sum{});
        scal->rr[c] = rr[c];
    }
    scal->state = fine ? kChipDone : state;
}

// Subdomain `sub` of the problem P by the calling CTA or cluster.
template <typename TI, bool CL, int NS>
__device__ __forceinline__ void chip_body(const SolveParams& P, int sub, ChipLevel* L, ChipScalars* scal, char* sm)
{
    typedef typename ChipVec<TI>::V V;
    typedef typename ChipVec<TI>::Sum Sum;
    Chip<CL> T;
    T.sm = sm;
    T.rank = 0; T.cw = 1; T.dn = T.up = nullptr;
    if constexpr (CL) {
        cg::cluster_group cl = cg::this_cluster();
        T.rank = (int)cl.block_rank();
        T.cw = (int)cl.num_blocks();
        if (T.rank > 0) T.dn = cl.map_shared_rank(sm, T.rank - 1);
        if (T.rank + 1 < T.cw) T.up = cl.map_shared_rank(sm, T.rank + 1);
    }
    T.warp = threadIdx.x >> 5; T.nw = blockDim.x >> 5; T.lane = threadIdx.x & 31;
    const int nx = P.nx;
    const int I = sub % P.px, J = sub / P.px;
    const int i0 = split_line(I, nx, P.px), i1 = split_line(I + 1, nx, P.px);
    const int j0 = split_line(J, P.ny, P.py), j1 = split_line(J + 1, P.ny, P.py);
    const int ni = i1 - i0 - 1, nj = j1 - j0 - 1;
    if (ni <= 0 || nj <= 0) {  // no interior: nothing to solve (a team of one CTA)
        if (threadIdx.x == 0) {
            P.stat_iters[sub] = 0; P.stat_outer[sub] = 0; P.stat_ok[sub] = 1; P.stat_res[sub] = 0.0;
        }
        return;
    }
    const int levels = mg_levels(ni, nj);
    if (threadIdx.x == 0) {  // the layout and this CTA's rows; the entry after the last: p's place and the bytes
        int lv, p_at;
        const int bytes = chip_levels(ni, nj, T.cw, (int)sizeof(TI), L, &lv, &p_at);
        int before = T.rank > 0 ? (int)((long)(T.rank - 1) * nj / T.cw) : 0;
        int a = (int)((long)T.rank * nj / T.cw), b = (int)((long)(T.rank + 1) * nj / T.cw);
        for (int l = 0; l < levels; ++l) {
            if (!L[l].dist) {
                L[l].r0 = 0; L[l].nr = L[l].ny; L[l].below = 0;
            } else {
                if (l > 0) { before /= 2; a /= 2; b = min(b / 2, L[l].ny); }
                L[l].r0 = a; L[l].nr = b - a; L[l].below = a - before;
            }
        }
        int lt = 1;
        while (lt < levels && (L[lt].dist || L[lt].kcs > 0 || (32 >> L[lt].w2) < L[lt].ny)) ++lt;  // one warp holds the rest
        L[kChipLevels].p = p_at;
        L[kChipLevels].x = bytes;
        L[kChipLevels].nx = lt;
    }
    __syncthreads();
    const int p_off = L[kChipLevels].p, bytes = L[kChipLevels].x, lt = L[kChipLevels].nx;
    char* red = sm + bytes;  // partial sums
    for (int k = threadIdx.x; k < bytes / 16; k += blockDim.x) reinterpret_cast<float4*>(sm)[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    T.sync(1);  // rims are zero, and nobody writes to a CTA that is still clearing
    const long mid = (long)(j0 + 1 + nj / 2) * nx + (i0 + 1 + ni / 2);
    chip_setup<TI, CL>(T, P, L, levels, i0, j0, sizeof(TI) == 8 ? -chip_exponent(P, mid) : 0);

    // The thread's nodes: slot s = 2 m + colour is row jl0 + m rstep, columns k0 of that colour (a row
    // wider than 64 is shared by 2^kcs warps).  A step of rows is even, so a column's parity depends on
    // the colour alone, and slots advance by constant steps in every array.
    const int H = L[0].H, F = L[0].F, C = L[0].C, w2 = L[0].w2, nr = L[0].nr, r0 = L[0].r0, d0 = L[0].dist;
    const int below = L[0].below;
    const int kcs = chip_chunks_log2(ni);
    const int rstep = (T.nw >> kcs) << (5 - w2);
    const int jl0 = ((T.warp >> kcs) << (5 - w2)) + (T.lane >> w2);
    const int k0 = (T.lane & ((1 << w2) - 1)) + 32 * (T.warp & ((1 << kcs) - 1));
    const int par = (r0 + jl0) & 1;  // column parity of colour 0
    unsigned vm = 0;                 // slots that are nodes
#pragma unroll
    for (int s = 0; s < NS; ++s)
        if (jl0 + (s >> 1) * rstep < nr && (par ^ (s & 1)) + 2 * k0 < ni) vm |= 1u << s;
    float2* const X = at<float2>(sm, L[0].x);
    float2* const R = at<float2>(sm, L[0].t);
    V* const Pv = at<V>(sm, p_off);
    const float* const CE = at<float>(sm, L[0].ce);
    const float* const CN = at<float>(sm, L[0].cn);
    const float* const DG = at<float>(sm, L[0].dg);
    const float* const IV = at<float>(sm, L[0].inv);
    // Place of slot `colour` and the step to the next row's.  Worked out anew by every pass (opaque): kept
    // over the passes, the places of all slots spill.
    struct At { int self, w, fw, fe, c, jl; long id; };
    const int sx = rstep * 2 * H, sf = rstep * 2 * F, sc = rstep * 2 * C;
    auto first = [&](int colour) -> At {
        int jl = jl0;
        asm volatile("" : "+r"(jl));
        const int cc = par ^ colour;
        At o;
        o.self = ((jl + 1) * 2 + 1 - cc) * H + k0 + cc;
        o.w = ((jl + 1) * 2 + cc) * H + k0;
        o.fw = (jl * 2 + cc) * F + k0;
        o.fe = (jl * 2 + 1 - cc) * F + k0 + cc;
        o.c = (jl * 2 + cc) * C + k0;
        o.jl = jl;
        o.id = (long)(j0 + 1 + r0 + jl) * nx + (i0 + 1 + cc + 2 * k0);
        return o;
    };
    auto next = [&](At& o) {
        o.self += sx; o.w += sx; o.fw += sf; o.fe += sf; o.c += sc; o.jl += rstep;
        o.id += (long)rstep * nx;
    };
// the thread's nodes of one colour: o their place, s their slot
#define CHIP_SLOTS(colour)                                                      \
    At o = first(colour);                                                       \
    _Pragma("unroll") for (int s = (colour); s < NS; s += 2, next(o)) if (vm >> s & 1)
    auto dP = [&](long id) -> double { return P.form == 0 ? 1.0 : P.om64[id]; };
    // store to an array of level 0 and to the neighbour CTA's halo copy of an edge row
    auto store = [&](auto* arr, const At& o, auto v) {
        arr[o.self] = v;
        if constexpr (CL) {
            typedef decltype(v) W;
            const int off = (int)(reinterpret_cast<char*>(arr) - sm);
            if (o.jl == 0 && T.rank > 0) at<W>(T.dn, off)[o.self + below * 2 * H] = v;
            if (o.jl == nr - 1 && T.rank + 1 < T.cw) at<W>(T.up, off)[o.self - nr * 2 * H] = v;
        }
    };
    auto off_sum = [&](const At& o) -> float2 {
        const float cW = CE[o.fw], cE = CE[o.fe], cS = CN[o.c], cN = CN[o.c + 2 * C];
        const float2 w = X[o.w], e = X[o.w + 1], so = X[o.self - 2 * H], n = X[o.self + 2 * H];
        return make_float2(__fmaf_rn(cN, n.x, __fmaf_rn(cS, so.x, __fmaf_rn(cE, e.x, __fmul_rn(cW, w.x)))),
                           __fmaf_rn(cN, n.y, __fmaf_rn(cS, so.y, __fmaf_rn(cE, e.y, __fmul_rn(cW, w.y)))));
    };

    V r[NS], p[NS], q[NS], e[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) r[s].x = r[s].y = p[s].x = p[s].y = q[s].x = q[s].y = e[s].x = e[s].y = (TI)0;

    // initial guess and ||b||
    const Sum none{};
    double bn[2] = {0.0, 0.0};
    // (the diagonals, which every residual needs, go to the workspace, which a solve of one CTA does not use)
    double* const diag64 = CL ? nullptr : reinterpret_cast<double*>(static_cast<char*>(P.mg) + (size_t)sub * P.mg_stride);
#pragma unroll
    for (int col = 0; col < 2; ++col) {
        double xc[NS / 2], yc[NS / 2];
        {
            CHIP_SLOTS(col) { xc[s / 2] = P.xcur[o.id]; yc[s / 2] = P.ycur[o.id]; }
        }
        {
            CHIP_SLOTS(col) {
                double bx = xc[s / 2], by = yc[s / 2];
                if (P.form != 0) { const double d = P.om64[o.id]; bx *= d; by *= d; }
                bn[0] += bx * bx;
                bn[1] += by * by;
            }
        }
        {
            CHIP_SLOTS(col) { P.xnew[o.id] = xc[s / 2]; P.ynew[o.id] = yc[s / 2]; }
        }
    }
    // the nodes next to the rim: (d x + rim terms)^2 - (d x)^2
    for (int k = T.rank * (int)blockDim.x + (int)threadIdx.x; k < 2 * (ni + nj); k += T.cw * (int)blockDim.x) {
        const bool row = k < 2 * ni;
        const int m = row ? k >> 1 : (k - 2 * ni) >> 1, far = k & 1;
        const int i = i0 + 1 + (row ? m : far ? ni - 1 : 0), j = j0 + 1 + (row ? (far ? nj - 1 : 0) : m);
        if (row ? far && nj == 1 : j == j0 + 1 || j == j1 - 1 || (far && ni == 1)) continue;  // counted once
        const long id = (long)j * nx + i;
        const double d = dP(id), bx = d * P.xcur[id], by = d * P.ycur[id];
        double ex = 0.0, ey = 0.0;
        if (i - 1 == i0) { ex += P.ce64[id - 1] * P.xnew[id - 1]; ey += P.ce64[id - 1] * P.ynew[id - 1]; }
        if (i + 1 == i1) { ex += P.ce64[id] * P.xnew[id + 1]; ey += P.ce64[id] * P.ynew[id + 1]; }
        if (j - 1 == j0) { ex += P.cn64[id - nx] * P.xnew[id - nx]; ey += P.cn64[id - nx] * P.ynew[id - nx]; }
        if (j + 1 == j1) { ex += P.cn64[id] * P.xnew[id + nx]; ey += P.cn64[id] * P.ynew[id + nx]; }
        bn[0] += ex * (2.0 * bx + ex);
        bn[1] += ey * (2.0 * by + ey);
    }
    int turn = 0;
    chip_sum<CL, 2, double>(T, bn, red, turn);  // its barrier also orders the guess before the residual

    // z = V-cycle(r): level 0's passes on the slots, the levels below in shared memory.  Ends without a
    // barrier: until the next one a thread reads the z of its own nodes only, which it wrote itself.
    auto sweep = [&](auto colour) {
        CHIP_SLOTS(colour.value) {
            const float2 b = to_f2(r[s]), u = off_sum(o);
            store(X, o, div_diag(__fadd_rn(b.x, u.x), __fadd_rn(b.y, u.y), DG[o.c], IV[o.c]));
        }
    };
    const std::integral_constant<int, 0> red0{};
    const std::integral_constant<int, 1> black{};
    auto cycle = [&]() {
        {
            CHIP_SLOTS(0) {
                const float2 b = to_f2(r[s]);
                store(X, o, div_diag(b.x, b.y, DG[o.c], IV[o.c]));
            }
        }
        if (levels == 1) {
            if (ni * nj == 1) return;
#pragma unroll 1
            for (int m = 0; m < 4 * kCoarseSweeps - 1; ++m) {  // colours (0) 1 1 0 | 0 1 1 0 | ...
                T.sync(d0);
                if ((m + 2) & 2) sweep(black); else sweep(red0);
            }
            return;
        }
        T.sync(d0);
        sweep(black);
        T.sync(d0);
#pragma unroll
        for (int col = 0; col < 2; ++col) {
            CHIP_SLOTS(col) {
                const float2 u = off_sum(o), x = X[o.self], b = to_f2(r[s]);
                const float dg = DG[o.c];
                store(R, o, make_float2(__fsub_rn(b.x, __fmaf_rn(dg, x.x, -u.x)), __fsub_rn(b.y, __fmaf_rn(dg, x.y, -u.y))));
            }
        }
        T.sync(d0);
        chip_restrict(T, L[0], L[1], T.warp, T.nw);
        T.sync(d0);
        chip_coarse_cycle<CL>(T, L, levels, lt);
        {
            const ChipLevel& C1 = L[1];
            CHIP_SLOTS(0) store(X, o, prolonged(sm, C1, X[o.self], r0 + o.jl, par, k0));
        }
        T.sync(d0);
        sweep(black);
        T.sync(d0);
        sweep(red0);
    };

    int iters = 0, outer = 0, ok = 0;
    // A sweep's residual is taken times 2^scale, a scale for each component, so that its norm is about the root of
    // the cycle's diagonal (by the exponents at the middle node; between 2^-20 and 2^50): squares, r.z, p.q and the cycle's
    // values then stay in FP32's range whatever the extents and the monitor's size are.  Powers of two change no
    // rounding.
    if (threadIdx.x == 0) {
        scal->target = sizeof(TI) == 8 ? 0 : max(-20, min(50, chip_exponent(P, mid) >> 1));
        scal->state = kChipSolve;
        for (int c = 0; c < 2; ++c) {
            scal->bn[c] = bn[c];
            scal->goal[c] = P.rtol * P.rtol * (bn[c] > 0 ? bn[c] : 1.0);
            scal->scale[c] = scal->target - (exponent(bn[c]) >> 1);  // a guess: of the size of b
        }
    }
    __syncthreads();
#pragma unroll 1
    for (outer = 0; outer < kMaxOuter;) {
        // FP64 residual of the current iterate and its squared norms; formed again (once) where the scale, that of
        // the sweep before, is so far off that entries may have left FP32's range.  The norms are sums of FP64 squares,
        // as the global-memory solver's: 4 of the 334 us of 16 subdomains of 63 x 63 against sums of FP32 pairs over
        // the rounded residual, which lose what is below 1e-23 and above 1e19.
        const int kx = scal->scale[0], ky = scal->scale[1];
        double rr[2] = {0.0, 0.0};
#pragma unroll
        for (int col = 0; col < 2; ++col) {
            CHIP_SLOTS(col) {
                const long id = o.id;
                const double cE = P.ce64[id], cW = P.ce64[id - 1], cN = P.cn64[id], cS = P.cn64[id - nx];
                double diag;
                if (CL || outer == 0) {
                    diag = dP(id) + cE + cW + cN + cS;
                    if (!CL) diag64[o.jl * ni + (par ^ col) + 2 * k0] = diag;
                } else {
                    diag = diag64[o.jl * ni + (par ^ col) + 2 * k0];
                }
                const double ax = fma_rn(-cS, P.xnew[id - nx], fma_rn(-cN, P.xnew[id + nx], fma_rn(-cW, P.xnew[id - 1],
                                  fma_rn(diag, P.xnew[id], -(cE * P.xnew[id + 1])))));
                const double ay = fma_rn(-cS, P.ynew[id - nx], fma_rn(-cN, P.ynew[id + nx], fma_rn(-cW, P.ynew[id - 1],
                                  fma_rn(diag, P.ynew[id], -(cE * P.ynew[id + 1])))));
                double rx, ry;
                if (P.form == 0) {
                    rx = P.xcur[id] - ax;
                    ry = P.ycur[id] - ay;
                } else {
                    rx = fma_rn(P.om64[id], P.xcur[id], -ax);
                    ry = fma_rn(P.om64[id], P.ycur[id], -ay);
                }
                r[s].x = to_inner<TI>(rx, kx);
                r[s].y = to_inner<TI>(ry, ky);
                mac(rr[0], rx, rx);
                mac(rr[1], ry, ry);
            }
        }
        chip_sum<CL, 2, double, true>(T, rr, red, turn);
        if (threadIdx.x == 0) chip_decide<TI>(scal, rr[0], rr[1], P.rtol);
        __syncthreads();
        if (scal->state == kChipAgain) continue;
        if (scal->state == kChipDone) {
            ok = 1;
            break;
        }
        if (iters >= P.max_iter) break;
        {
            const TI mx = *reinterpret_cast<const TI*>(&scal->more[0]), my = *reinterpret_cast<const TI*>(&scal->more[1]);
#pragma unroll
            for (int s = 0; s < NS; ++s) { r[s].x *= mx; r[s].y *= my; }
        }
        bool done0 = scal->rr[0] == 0.0, done1 = scal->rr[1] == 0.0;
        Sum rz[2] = {none, none};
#pragma unroll
        for (int s = 0; s < NS; ++s) e[s].x = e[s].y = p[s].x = p[s].y = (TI)0;
        // the first turn only preconditions: p = z + 0 p
#pragma unroll 1
        for (bool start = true;; start = false) {
            if (!start) {
                if (iters >= P.max_iter || (done0 && done1)) break;
                ++iters;
#pragma unroll
                for (int col = 0; col < 2; ++col) {
                    CHIP_SLOTS(col) store(Pv, o, p[s]);
                }
                T.sync(d0);
                Sum pq[2] = {none, none};
#pragma unroll
                for (int col = 0; col < 2; ++col) {
                    CHIP_SLOTS(col) {
                        const V pe = Pv[o.w + 1], pw = Pv[o.w], pn = Pv[o.self + 2 * H], pp = Pv[o.self - 2 * H];
                        TI cE, cW, cN, cS, d = (TI)1;
                        if constexpr (sizeof(TI) == 8) {
                            cE = P.ce64[o.id]; cW = P.ce64[o.id - 1]; cN = P.cn64[o.id]; cS = P.cn64[o.id - nx];
                        } else {
                            cW = CE[o.fw]; cE = CE[o.fe]; cS = CN[o.c]; cN = CN[o.c + 2 * C];
                        }
                        if (P.form != 0) d = (TI)P.om64[o.id];
                        const TI diag = d + cE + cW + cN + cS;
                        q[s].x = fma_rn(-cS, pp.x, fma_rn(-cN, pn.x, fma_rn(-cW, pw.x, fma_rn(diag, p[s].x, -(cE * pe.x)))));
                        q[s].y = fma_rn(-cS, pp.y, fma_rn(-cN, pn.y, fma_rn(-cW, pw.y, fma_rn(diag, p[s].y, -(cE * pe.y)))));
                        mac(pq[0], p[s].x, q[s].x);
                        mac(pq[1], p[s].y, q[s].y);
                    }
                }
                chip_sum<CL, 2, Sum>(T, pq, red, turn);
                const TI ax = !done0 ? ratio(rz[0], pq[0]) : (TI)0;
                const TI ay = !done1 ? ratio(rz[1], pq[1]) : (TI)0;
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    e[s].x = fma_rn(ax, p[s].x, e[s].x); e[s].y = fma_rn(ay, p[s].y, e[s].y);
                    r[s].x = fma_rn(-ax, q[s].x, r[s].x); r[s].y = fma_rn(-ay, q[s].y, r[s].y);
                }
            }
            cycle();
            Sum v[4] = {none, none, none, none};
#pragma unroll
            for (int col = 0; col < 2; ++col) {
                CHIP_SLOTS(col) {
                    const float2 z = X[o.self];
                    mac(v[0], r[s].x, (TI)z.x);
                    mac(v[1], r[s].y, (TI)z.y);
                    mac(v[2], r[s].x, r[s].x);
                    mac(v[3], r[s].y, r[s].y);
                }
            }
            chip_sum<CL, 4, Sum>(T, v, red, turn);  // its barrier: all are done with t, whose place p takes
            TI bx = (TI)0, by = (TI)0;
            if (!start) {
                if (!done0 && at_most(v[2], *reinterpret_cast<const Sum*>(&scal->stop[0]))) done0 = true;
                if (!done1 && at_most(v[3], *reinterpret_cast<const Sum*>(&scal->stop[1]))) done1 = true;
                bx = !done0 ? ratio(v[0], rz[0]) : (TI)0;
                by = !done1 ? ratio(v[1], rz[1]) : (TI)0;
            }
            rz[0] = v[0];
            rz[1] = v[1];
#pragma unroll
            for (int col = 0; col < 2; ++col) {
                CHIP_SLOTS(col) {
                    const float2 z = X[o.self];
                    p[s].x = fma_rn(bx, p[s].x, (TI)z.x);
                    p[s].y = fma_rn(by, p[s].y, (TI)z.y);
                }
            }
        }
        // x += e, the scale undone
        const double ux = pow2(-scal->scale[0]), uy = pow2(-scal->scale[1]);
#pragma unroll
        for (int col = 0; col < 2; ++col) {
            CHIP_SLOTS(col) {
                P.xnew[o.id] = fma_rn((double)e[s].x, ux, P.xnew[o.id]);
                P.ynew[o.id] = fma_rn((double)e[s].y, uy, P.ynew[o.id]);
            }
        }
        T.sync(1);
        ++outer;
    }
    if (T.rank == 0 && threadIdx.x == 0) {
        P.stat_iters[sub] = iters;
        P.stat_outer[sub] = outer;
        P.stat_ok[sub] = ok;
        const double rx = scal->rr[0], ry = scal->rr[1];
        const double bx = scal->bn[0], by = scal->bn[1];
        P.stat_res[sub] = fmax(sqrt(bx > 0 ? rx / bx : rx), sqrt(by > 0 ? ry / by : ry));
    }
#undef CHIP_SLOTS
    if constexpr (CL) cg::this_cluster().sync();  // no CTA leaves while another may still write to it
}

// items: (problem, subdomain) of each CTA or cluster; probs (null: the problem P) the records they
// index.
template <typename TI, bool CL, int NS>
__global__ void __launch_bounds__(512, 1) chip_kernel(const __grid_constant__ SolveParams P, const SolveParams* probs,
                                                      const int2* items)
{
    extern __shared__ __align__(16) char chip_sm[];
    __shared__ ChipLevel L[kChipLevels + 1];
    __shared__ ChipScalars scal;
    __shared__ SolveParams sp;
    int team = blockIdx.x;
    if constexpr (CL) team /= (int)cg::this_cluster().num_blocks();
    const int2 it = items[team];
    if (threadIdx.x == 0) sp = probs ? probs[it.x] : P;
    __syncthreads();
    if (sp.bad && *sp.bad) return;  // alike in every CTA of a cluster
    chip_body<TI, CL, NS>(sp, it.y, L, &scal, chip_sm);
}

// ---- forward Euler on chip ----------------------------------------------------------------
// The paper's local solver (fe_body's substeps) with the iterate in shared memory and each thread's
// nodes, with their weights c_nb / (S d), in registers; a subdomain is split by rows over a cluster
// whose edge rows are written to the neighbours' halo copies.  A substep is 18 FP64 operations a
// node (fe_body: 48 with its divisions) and a barrier; the FP64 unit bounds it until a CTA has few
// nodes, then the barrier.  Every node computes the same operations in any team, and the team is
// chosen by how many subdomains the launch has.  15 subdomains of 65 x 27, 60 substeps: 1.54 ms from
// global memory by a CTA each, 0.23 ms by clusters of eight.
constexpr int kFeThreads = 512, kFeSlots = 4;
__host__ __device__ inline int fe_chip_bytes(int ni, int nj, int cw)
{
    return 2 * ((nj + cw - 1) / cw + 2) * (ni + 2) * 16 + 128;
}

template <bool CL>
__device__ __forceinline__ void fe_chip_body(const SolveParams& P, int sub, char* sm)
{
    Chip<CL> T;
    T.sm = sm;
    T.rank = 0; T.cw = 1; T.dn = T.up = nullptr;
    if constexpr (CL) {
        cg::cluster_group cl = cg::this_cluster();
        T.rank = (int)cl.block_rank();
        T.cw = (int)cl.num_blocks();
        if (T.rank > 0) T.dn = cl.map_shared_rank(sm, T.rank - 1);
        if (T.rank + 1 < T.cw) T.up = cl.map_shared_rank(sm, T.rank + 1);
    }
    const int tid = threadIdx.x, nx = P.nx;
    const int I = sub % P.px, J = sub / P.px;
    const int i0 = split_line(I, nx, P.px), i1 = split_line(I + 1, nx, P.px);
    const int j0 = split_line(J, P.ny, P.py), j1 = split_line(J + 1, P.ny, P.py);
    const int ni = i1 - i0 - 1, nj = j1 - j0 - 1;
    if (ni <= 0 || nj <= 0) {  // no interior
        if (T.rank == 0 && tid == 0) {
            P.stat_iters[sub] = 1; P.stat_outer[sub] = 0; P.stat_ok[sub] = 1; P.stat_res[sub] = 0.0;
        }
        return;
    }
    const int r0 = (int)((long)T.rank * nj / T.cw), r1 = (int)((long)(T.rank + 1) * nj / T.cw), nr = r1 - r0;
    const int below = T.rank > 0 ? r0 - (int)((long)(T.rank - 1) * nj / T.cw) : 0;
    const int rows = (nj + T.cw - 1) / T.cw, W = ni + 2;
    double* red = reinterpret_cast<double*>(sm);                // 16: warps' maxima, then CTAs'
    double2* buf = reinterpret_cast<double2*>(sm + 128);        // two buffers of (rows + 2) x W
    const int cells = (rows + 2) * W;
    auto dP = [&](long id) -> double { return P.form == 0 ? 1.0 : P.om64[id]; };
    // own nodes: place in a buffer, coefficients, value
    int at_[kFeSlots];
    double aE[kFeSlots], aW[kFeSlots], aN[kFeSlots], aS[kFeSlots];
    double2 x[kFeSlots];
    double cmax = 0.0;
#pragma unroll
    for (int s = 0; s < kFeSlots; ++s) {
        const int k = tid + s * kFeThreads;
        at_[s] = -1;
        if (k >= nr * ni) continue;
        const int jl = k / ni, i = k % ni;
        const long id = (long)(j0 + 1 + r0 + jl) * nx + (i0 + 1 + i);
        at_[s] = (jl + 1) * W + i + 1;
        aE[s] = P.ce64[id]; aW[s] = P.ce64[id - 1]; aN[s] = P.cn64[id]; aS[s] = P.cn64[id - nx];
        x[s] = make_double2(P.xcur[id], P.ycur[id]);
        const double c = __dadd_rn(__dadd_rn(__dadd_rn(aE[s], aW[s]), aN[s]), aS[s]);
        cmax = fmax(cmax, P.form == 0 ? c : __ddiv_rn(c, P.om64[id]));
    }
    // largest over the team (the same value in any order)
    for (int o = 16; o > 0; o >>= 1) cmax = fmax(cmax, __shfl_xor_sync(kFull, cmax, o));
    if ((tid & 31) == 0) red[tid >> 5] = cmax;
    __syncthreads();
    cmax = red[0];
    for (int w = 1; w < kFeThreads / 32; ++w) cmax = fmax(cmax, red[w]);
    if constexpr (CL) {
        cg::this_cluster().sync();  // every CTA has read its warps' maxima
        if (tid < T.cw) cg::this_cluster().map_shared_rank(red, tid)[T.rank] = cmax;  // 8 CTAs at most
        cg::this_cluster().sync();
        cmax = red[0];
        for (int r = 1; r < T.cw; ++r) cmax = fmax(cmax, red[r]);
    }
    const double Sd = ceil(cmax) < 1.0 ? 1.0 : ceil(cmax);
    const bool solve = Sd <= (double)P.fe_max_substeps;
    const int S = solve ? (int)Sd : 0;
    // the rim cells of this CTA: the columns beside its rows, and the rows below the first and above the
    // last CTA's; cell k's place and node
    const int nrim = 2 * nr + (T.rank == 0 ? ni : 0) + (T.rank == T.cw - 1 ? ni : 0);
    auto rim = [&](int k, int& place, long& id) {
        int jl, i;
        if (k < 2 * nr) { jl = k >> 1; i = (k & 1) ? ni : -1; }
        else {
            k -= 2 * nr;
            const bool low = T.rank == 0 && k < ni;
            if (T.rank == 0 && !low) k -= ni;
            jl = low ? -1 : nr;
            i = k;
        }
        place = (jl + 1) * W + i + 1;
        id = (long)(j0 + 1 + r0 + jl) * nx + (i0 + 1 + i);
    };
    int rim_at = -1;             // the thread's first rim cell in registers, further ones from memory
    double2 rim_x = make_double2(0.0, 0.0), rim_d = rim_x;
    if (tid < nrim) {
        long id;
        rim(tid, rim_at, id);
        rim_x = make_double2(P.xcur[id], P.ycur[id]);
        rim_d = make_double2(__dsub_rn(P.xnew[id], rim_x.x), __dsub_rn(P.ynew[id], rim_x.y));
    }
    auto write_rim = [&](double2* b, double f) {  // x^n + f (x^{n+1} - x^n)
        if (rim_at >= 0)
            b[rim_at] = make_double2(__dadd_rn(rim_x.x, __dmul_rn(f, rim_d.x)), __dadd_rn(rim_x.y, __dmul_rn(f, rim_d.y)));
        for (int k = tid + kFeThreads; k < nrim; k += kFeThreads) {
            int place;
            long id;
            rim(k, place, id);
            const double px = P.xcur[id], py = P.ycur[id];
            b[place] = make_double2(__dadd_rn(px, __dmul_rn(f, __dsub_rn(P.xnew[id], px))),
                                    __dadd_rn(py, __dmul_rn(f, __dsub_rn(P.ynew[id], py))));
        }
    };
    auto write_node = [&](int which, int place, double2 v) {
        buf[which * cells + place] = v;
        if constexpr (CL) {
            if (T.rank > 0 && place < 2 * W) at<double2>(T.dn, 128)[which * cells + place + below * W] = v;
            if (T.rank + 1 < T.cw && place >= nr * W) at<double2>(T.up, 128)[which * cells + place - nr * W] = v;
        }
    };
#pragma unroll
    for (int s = 0; s < kFeSlots; ++s) {
        if (at_[s] < 0) continue;
        const int k = tid + s * kFeThreads;
        const long id = (long)(j0 + 1 + r0 + k / ni) * nx + (i0 + 1 + k % ni);
        const double w = __ddiv_rn(1.0, __dmul_rn(Sd, dP(id)));
        aE[s] *= w; aW[s] *= w; aN[s] *= w; aS[s] *= w;
        write_node(0, at_[s], x[s]);
    }
    write_rim(buf, 0.0);
    T.sync(1);
#pragma unroll 1
    for (int m = 0; m < S; ++m) {
        const double2* b = buf + (m & 1) * cells;
        const int to = (m + 1) & 1;
#pragma unroll
        for (int s = 0; s < kFeSlots; ++s) {
            if (at_[s] < 0) continue;
            const double2 e = b[at_[s] + 1], w = b[at_[s] - 1], n = b[at_[s] + W], so = b[at_[s] - W];
            const double dx = fma(aS[s], so.x - x[s].x, fma(aN[s], n.x - x[s].x, fma(aW[s], w.x - x[s].x, aE[s] * (e.x - x[s].x))));
            const double dy = fma(aS[s], so.y - x[s].y, fma(aN[s], n.y - x[s].y, fma(aW[s], w.y - x[s].y, aE[s] * (e.y - x[s].y))));
            x[s].x += dx;
            x[s].y += dy;
            write_node(to, at_[s], x[s]);
        }
        write_rim(buf + to * cells, (double)(m + 1) / Sd);
        T.sync(1);
    }
#pragma unroll
    for (int s = 0; s < kFeSlots; ++s) {
        if (at_[s] < 0) continue;
        const int k = tid + s * kFeThreads;
        const long id = (long)(j0 + 1 + r0 + k / ni) * nx + (i0 + 1 + k % ni);
        P.xnew[id] = x[s].x;  // x^n where the subdomain needs more substeps than allowed
        P.ynew[id] = x[s].y;
    }
    if (T.rank == 0 && tid == 0) {
        P.stat_iters[sub] = S; P.stat_outer[sub] = 0; P.stat_ok[sub] = solve ? 1 : 0; P.stat_res[sub] = 0.0;
    }
    if constexpr (CL) cg::this_cluster().sync();  // no CTA leaves while another may still write to it
}

template <bool CL>
__global__ void __launch_bounds__(kFeThreads, 1) fe_chip_kernel(const __grid_constant__ SolveParams P, const SolveParams* probs,
                                                                const int2* items)
{
    extern __shared__ __align__(16) char chip_sm[];
    __shared__ SolveParams sp;
    int team = blockIdx.x;
    if constexpr (CL) team /= (int)cg::this_cluster().num_blocks();
    const int2 it = items[team];
    if (threadIdx.x == 0) sp = probs ? probs[it.x] : P;
    __syncthreads();
    if (sp.bad && *sp.bad) return;  // alike in every CTA of a cluster
    fe_chip_body<CL>(sp, it.y, chip_sm);
}

// CTAs of the smallest team that holds a subdomain of ni x nj nodes (0: none of up to eight, or `widest`, does).
inline int fe_chip_team(int ni, int nj, int widest)
{
    if (ni <= 0 || nj <= 0) return 1;
    for (int cw = 1; cw <= 8 && cw <= widest; cw *= 2)
        if (nj >= cw && (int64_t)((nj + cw - 1) / cw) * ni <= kFeThreads * kFeSlots && ni <= 4096 &&
            fe_chip_bytes(ni, nj, cw) <= kChipSmem)
            return cw;
    return 0;
}

// Team of a subdomain of ni x nj interior nodes: CTAs (0: it does not fit), warps per CTA, slots of
// its kernel, dynamic shared memory.  The fewest CTAs that hold it -- a cluster barrier costs about a
// microsecond, ten times a CTA's -- as a function of the size (and of the widest cluster that the device takes)
// alone, so that a subdomain gives the same bits in every launch.  Warps: the fewest, from four, with half the slots, so that small
// subdomains share an SM and run the smaller kernel.
inline void chip_team(int ni, int nj, bool fp64, int widest, ChipLaunch* c)
{
    c->cw = c->nw = c->slots = c->smem = 0;
    const int most = fp64 ? ChipSlots<double>::n : ChipSlots<float>::n;
    if (ni <= 0 || nj <= 0) {
        c->cw = 1; c->nw = 4; c->slots = most / 2; c->smem = 1024;
        return;
    }
    if (ni > 512 || nj > 4096) return;
    for (int cw = 1; cw <= widest; cw *= 2) {
        if (cw > 1 && nj < 2 * cw) return;
        ChipLevel L[kChipLevels];
        int levels = 0, p_off = 0;
        const int bytes = chip_levels(ni, nj, cw, fp64 ? 8 : 4, L, &levels, &p_off) + kRedBytes;
        if (levels > kChipLevels || bytes > kChipSmem) continue;
        for (int slots = most / 2; slots <= most; slots *= 2)
            for (int nw = slots == most ? 16 : 4; nw <= 16; nw *= 2) {
                const int need = chip_slots(ni, nj, cw, nw);
                if (need == 0 || need > slots || !chip_levels_fit(L, levels, cw, nw)) continue;
                c->cw = cw; c->nw = nw; c->slots = slots; c->smem = bytes;
                return;
            }
    }
}

}  // namespace
