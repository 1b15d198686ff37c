// Monitor preparation, Dirichlet-data scatter and face coefficients: grid-sized, bound by memory traffic and,
// on large grids, by the FP64 unit (each kernel's comment has its figures).
//
//   prep_omega_kernel : omega at every node on the current mesh at t^n (Sec. 2, Sec. 3.2),
//                       FP64; periodic wrap nodes evaluate their canonical node so they
//                       repeat it bit for bit.
//   prep_pack_kernel  : finite-difference gradient of omega in the computational
//                       coordinates (Sec. 3.4), the packed {omega, omega_xi, omega_eta}
//                       records in the path precision (FP64: one per node; FP32: the four
//                       corners of every node's cell), and the previous mesh
//                       as a displacement from the identity.
//   solve_setup_kernel: the new mesh's Dirichlet data -- physical boundary (identity) and
//                       interface estimates with periodic offsets (Sec. 3.5) -- and the face
//                       coefficients of the backward-Euler subdomain systems.
//
// The prep arithmetic uses explicit round-to-nearest intrinsics (no fused multiply-add), so
// the FP64 monitor record is reproducible independently of compiler contraction choices.
#include <math.h>

#include "sdd_internal.cuh"

namespace sdd {

namespace {

constexpr int kMonGauss = 1, kMonFront = 2, kMonRings = 4;  // otherwise bumps (3) or nodal (0)

__device__ __forceinline__ double min_image(double d, double L, int periodic)
{
    return periodic ? d - L * floor(d / L + 0.5) : d;
}

__device__ double monitor_value(const PrepParams& P, double x, double y, double t)
{
    const double* q = P.params;
    if (P.kind == kMonGauss) {
        const double dx = min_image(x - q[2], P.Lx, P.periodic);
        const double dy = min_image(y - q[3], P.Ly, P.periodic);
        return sqrt(1.0 + q[0] * exp(-q[1] * (dx * dx + dy * dy)));
    }
    if (P.kind == kMonFront) {
        const double dx = min_image(x - q[4], P.Lx, P.periodic);
        const double dy = min_image(y - q[5], P.Ly, P.periodic);
        const double r = sqrt(dx * dx + dy * dy);
        const double u = tanh(q[1] * (r - q[2] - q[3] * t));
        const double g = q[1] * (1.0 - u * u);      // |grad u|
        return sqrt(1.0 + q[0] * g * g);
    }
    if (P.kind == kMonRings) {                       // sum of tanh rings (five-ring problem)
        double gx = 0.0, gy = 0.0;
        for (int b = 3; b + 1 < P.n_params; b += 2) {
            const double dx = min_image(x - q[b], P.Lx, P.periodic);
            const double dy = min_image(y - q[b + 1], P.Ly, P.periodic);
            const double uk = tanh(q[1] * (dx * dx + dy * dy - q[2]));
            const double f = q[1] * (1.0 - uk * uk) * 2.0;
            gx += f * dx;
            gy += f * dy;
        }
        return sqrt(1.0 + q[0] * (gx * gx + gy * gy));
    }
    double w = 1.0;                                  // bumps
    // 4097 x 4097 nodes, three bumps: 2.78 -> 1.68 ms without the divisions and the terms out of reach;
    // bound by the FP64 unit, most of it for the exponentials that remain
    for (int b = 0; b + 3 < P.n_params; b += 4) {
        const double dx = min_image(x - q[b + 2], P.Lx, P.periodic);
        const double dy = min_image(y - q[b + 3], P.Ly, P.periodic);
        const double r2 = dx * dx + dy * dy;
        if (r2 > P.bump_reach[b / 4]) continue;
        // r2 / w^2 rounded, by its reciprocal and two corrections (Markstein; r2 is bounded by the reach)
        const double W = P.bump_w2[b / 4], inv = P.bump_inv[b / 4];
        double z;
        if (inv > 0.0) {
            z = __dmul_rn(r2, inv);
            z = __fma_rn(__fma_rn(-z, W, r2), inv, z);
            z = __fma_rn(__fma_rn(-z, W, r2), inv, z);
        } else {
            z = r2 / W;
        }
        w += q[b] * exp(-z);
    }
    return w;
}

// Monitor on the current mesh at every node (the body of one block of blocks nb).
__device__ __forceinline__ void prep_omega_body(const PrepParams& P, int blk, int nb)
{
    const int n = P.nx * P.ny;
    const double t = P.t_dev ? *P.t_dev : P.t;
    for (int id = blk * blockDim.x + threadIdx.x; id < n; id += nb * blockDim.x) {
        const int i = id % P.nx, j = id / P.nx;
        const int ci = P.periodic ? i % (P.nx - 1) : i;
        const int cj = P.periodic ? j % (P.ny - 1) : j;
        const int c = cj * P.nx + ci;
        P.om64[id] = P.kind == 0 ? P.omega_in[c] : monitor_value(P, P.x[c], P.y[c], t);
    }
}

__global__ void prep_omega_kernel(const PrepParams P)
{
    if (blockIdx.x == 0 && threadIdx.x == 0 && P.bad) *P.bad = 0;  // before the pack launch
    prep_omega_body(P, blockIdx.x, gridDim.x);
}

// d f / d s along one grid line at index i of n nodes: central differences in the interior,
// one-sided second order at Dirichlet ends, wrapped when periodic; factor c = (n - 1) / 2.
__device__ __forceinline__ double fd_line(const double* f, long stride, int i, int n, int periodic, double c)
{
    if (periodic) {
        const int m = n - 1;
        const int ii = i % m;
        const int ip = (ii + 1) % m, im = (ii + m - 1) % m;
        return __dmul_rn(__dsub_rn(f[ip * stride], f[im * stride]), c);
    }
    if (i == 0)
        return __dmul_rn(__dsub_rn(__dadd_rn(__dmul_rn(-3.0, f[0]), __dmul_rn(4.0, f[stride])),
                                   f[2 * stride]), c);
    if (i == n - 1)
        return __dmul_rn(__dsub_rn(__dadd_rn(__dmul_rn(3.0, f[(long)(n - 1) * stride]),
                                             __dmul_rn(-4.0, f[(long)(n - 2) * stride])),
                                   -f[(long)(n - 3) * stride]), c);
    return __dmul_rn(__dsub_rn(f[(long)(i + 1) * stride], f[(long)(i - 1) * stride]), c);
}

// Gradient, packed records and displacement of a tile of kTileX x kTileY nodes.  FP32: the block forms the
// tile's node values and those of the column and row beyond it in shared memory, and each thread
// writes its whole cell record.  4097 x 4097 nodes: 0.74 ms, bound by 120 bytes a node of memory
// traffic (0.3 ms) and about 10 FP64 operations (0.3 ms); one thread a node that wrote its 16 bytes
// into four records and divided for its coordinates took 1.41 ms.
constexpr int kTileX = 32, kTileY = 8;

template <typename T>
__device__ __forceinline__ T rounded(double d)
{
    if constexpr (sizeof(T) == 4) return float_rn(d);
    else return d;
}

template <typename T>
__device__ __forceinline__ void prep_pack_tile(const PrepParams& P, int tile)
{
    __shared__ Mon4<T> rec[sizeof(T) == 4 ? kTileY + 1 : 1][sizeof(T) == 4 ? kTileX + 1 : 1];
    __shared__ double xi[kTileX], eta[kTileY];
    const int nx = P.nx, ny = P.ny, tiles_x = (nx + kTileX - 1) / kTileX;
    const int bx = tile % tiles_x * kTileX, by = tile / tiles_x * kTileY;
    const int tid = threadIdx.x, lx = tid % kTileX, ly = tid / kTileX;
    bool bad = false;
    if (tid < kTileX) {
        const int i = bx + tid;
        xi[tid] = (double)(P.periodic ? i % (nx - 1) : i) / (double)(nx - 1);
    } else if (tid < kTileX + kTileY) {
        const int j = by + tid - kTileX;
        eta[tid - kTileX] = (double)(P.periodic ? j % (ny - 1) : j) / (double)(ny - 1);
    }
    constexpr int W = sizeof(T) == 4 ? kTileX + 1 : kTileX, H = sizeof(T) == 4 ? kTileY + 1 : kTileY;
    for (int k = tid; k < W * H; k += kTileX * kTileY) {
        const int tx = k % W, ty = k / W;
        if (bx + tx > nx || by + ty > ny) continue;  // one beyond the grid is the corner clamped to it
        const int i = min(bx + tx, nx - 1), j = min(by + ty, ny - 1);
        const int id = j * nx + i;
        const double w = P.om64[id];
        const double wx = fd_line(P.om64 + (long)j * nx, 1, i, nx, P.periodic, P.gx);
        const double we = fd_line(P.om64 + i, nx, j, ny, P.periodic, P.gy);
        const Mon4<T> r{rounded<T>(w), rounded<T>(wx), rounded<T>(we), (T)0};
        const bool own = tx < kTileX && ty < kTileY && bx + tx < nx && by + ty < ny;
        if (own) {
            P.wxi64[id] = wx;
            P.weta64[id] = we;
            // the monitor must be positive and everything finite (Sec. 2: omega > 0)
            bad = bad || !(positive_bits(w) && finite_bits(w) && finite_bits(wx) && finite_bits(we));
        }
        if constexpr (sizeof(T) == 4) rec[ty][tx] = r;
        else if (own) static_cast<Mon4<T>*>(P.mon)[id] = r;
    }
    __syncthreads();
    const int i = bx + lx, j = by + ly;
    if (i < nx && j < ny) {
        const int id = j * nx + i;
        if constexpr (sizeof(T) == 4) {  // corners (i, j), (i + 1, j), (i, j + 1), (i + 1, j + 1)
            Mon4<T>* c = static_cast<Mon4<T>*>(P.mon) + 4 * (long)id;
            c[0] = rec[ly][lx];
            c[1] = rec[ly][lx + 1];
            c[2] = rec[ly + 1][lx];
            c[3] = rec[ly + 1][lx + 1];
        }
        const int c = P.periodic ? j % (ny - 1) * nx + i % (nx - 1) : id;
        const double X = __dsub_rn(P.x[c], __dmul_rn(P.Lx, xi[lx]));
        const double Y = __dsub_rn(P.y[c], __dmul_rn(P.Ly, eta[ly]));
        static_cast<Disp2<T>*>(P.disp)[id] = Disp2<T>{rounded<T>(X), rounded<T>(Y)};
        bad = bad || !(finite_bits(X) && finite_bits(Y));
    }
    if (P.bad && bad) atomicOr(P.bad, 1);
}

template <typename T>
__global__ void __launch_bounds__(kTileX * kTileY) prep_pack_kernel(const PrepParams P)
{
    prep_pack_tile<T>(P, blockIdx.x);
}

__global__ void shift_kernel(const int2* nodes, int M, int nx, const double* x, const double* y,
                             double* shift)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    const int2 ij = nodes[m];
    shift[2 * m] = x[(long)ij.y * nx + ij.x];
    shift[2 * m + 1] = y[(long)ij.y * nx + ij.x];
}

// Boundary node k of 2 (nx + ny): the rows eta = 0, 1, then the columns xi = 0, 1 (corners twice, alike).
__device__ __forceinline__ void scatter_boundary_one(int nx, int ny, double Lx, double Ly, double* xnew, double* ynew,
                                                     const double* bnd, int k)
{
    int i, j;
    if (k < 2 * nx) { i = k >> 1; j = (k & 1) ? ny - 1 : 0; }
    else if (k < 2 * (nx + ny)) { i = (k & 1) ? nx - 1 : 0; j = (k - 2 * nx) >> 1; }
    else return;
    const long id = (long)j * nx + i;
    double vx = Lx * ((double)i / (double)(nx - 1));
    double vy = Ly * ((double)j / (double)(ny - 1));
    if (bnd) {  // moving boundary: tangential components from the 1-D step
        if (j == 0) vx = bnd[i];
        else if (j == ny - 1) vx = bnd[nx + i];
        if (i == 0) vy = bnd[2 * nx + j];
        else if (i == nx - 1) vy = bnd[2 * nx + ny + j];
    }
    xnew[id] = vx;
    ynew[id] = vy;
}

// One backward-Euler step of the 1-D generator along side s of a Dirichlet domain (Sec. 2): the
// tangential coordinate b_k at its n nodes -- x along eta = 0 (s = 0) and eta = 1 (s = 1), y along
// xi = 0 (s = 2) and xi = 1 (s = 3) -- solves
//   d_k b_k + r sum_{nb = k +- 1} c_{k,nb} (b_k - b_nb) = d_k b^n_k,  k = 1 .. n-2,
//   c_{k,k+1} = (omega_k + omega_{k+1}) / 2 / h^2,  d_k = 1 (form 0) or omega_k (form 1),
// with the corner values fixed: a diagonally dominant M-matrix, by parallel cyclic reduction in shared
// memory (each of log2 n passes joins every row with the rows 2^p away), one block a side.  A serial
// elimination is a chain of two FP64 divisions a node: 467 us for the four sides of a 200 x 141 grid,
// against 13.  Sides longer than kSideMax nodes, which the shared memory does not hold, are eliminated serially.
// The method depends on the side's own length alone, so that a side's bits do not depend on the other sides of
// a launch; `cap` is how many nodes the launch has shared memory for, min(its longest side, kSideMax).
constexpr int kSideThreads = 512;
constexpr int kSideBytes = 48;               // A, C, D twice
constexpr int kSideMax = 200 * 1024 / kSideBytes;

template <typename T>
__device__ __forceinline__ void boundary_side(const PrepParams& P, int s, double* sm, int cap)
{
    const int nx = P.nx, ny = P.ny;
    const int n = s < 2 ? nx : ny;
    const long off = s == 0 ? 0 : s == 1 ? nx : s == 2 ? 2L * nx : 2L * nx + ny;
    auto id = [&](int k) -> long {
        return s == 0 ? k : s == 1 ? (long)(ny - 1) * nx + k : s == 2 ? (long)k * nx : (long)k * nx + nx - 1;
    };
    auto coord = [&](int k) -> double { return s < 2 ? P.x[id(k)] : P.y[id(k)]; };
    double* b = P.bnd64 + off;
    T* bt = static_cast<T*>(P.bnd) + off;
    const double h2 = (double)(n - 1) * (double)(n - 1);
    // row k: lower b_{k-1} + diag b_k + upper b_{k+1} = rhs
    auto row = [&](int k, double& lower, double& diag, double& upper, double& rhs) {
        const double w = P.om64[id(k)];
        const double cw = __dmul_rn(P.r, __dmul_rn(__dmul_rn(0.5, __dadd_rn(w, P.om64[id(k - 1)])), h2));
        const double ce = __dmul_rn(P.r, __dmul_rn(__dmul_rn(0.5, __dadd_rn(w, P.om64[id(k + 1)])), h2));
        const double d = P.form == 1 ? w : 1.0;
        diag = __dadd_rn(__dadd_rn(d, cw), ce);
        rhs = __dmul_rn(d, coord(k));
        lower = -cw;
        upper = -ce;
        if (k == 1) { rhs = __dadd_rn(rhs, __dmul_rn(cw, coord(0))); lower = 0.0; }
        if (k == n - 2) { rhs = __dadd_rn(rhs, __dmul_rn(ce, coord(n - 1))); upper = 0.0; }
    };
    if (threadIdx.x == 0) {
        b[0] = coord(0);
        b[n - 1] = coord(n - 1);
        bt[0] = (T)b[0];
        bt[n - 1] = (T)b[n - 1];
    }
    if (n > cap) {
        if (threadIdx.x != 0) return;
        double* cp = P.bnd_scratch + 2 * off;
        double* dp = cp + n;
        for (int k = 1; k <= n - 2; ++k) {
            double lower, diag, upper, rhs;
            row(k, lower, diag, upper, rhs);
            const double m = k == 1 ? diag : __dsub_rn(diag, __dmul_rn(lower, cp[k - 1]));
            cp[k] = __ddiv_rn(upper, m);
            dp[k] = __ddiv_rn(k == 1 ? rhs : __dsub_rn(rhs, __dmul_rn(lower, dp[k - 1])), m);
        }
        b[n - 2] = dp[n - 2];
        for (int k = n - 3; k >= 1; --k) b[k] = __dsub_rn(dp[k], __dmul_rn(cp[k], b[k + 1]));
        for (int k = 1; k <= n - 2; ++k) bt[k] = (T)b[k];
        return;
    }
    const int m = n - 2;
    double *A = sm, *C = sm + n, *Dv = sm + 2 * n, *A2 = sm + 3 * n, *C2 = sm + 4 * n, *D2 = sm + 5 * n;
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        double lower, diag, upper, rhs;
        row(i + 1, lower, diag, upper, rhs);
        const double inv = 1.0 / diag;
        A[i] = lower * inv;
        C[i] = upper * inv;
        Dv[i] = rhs * inv;
    }
    for (int st = 1; st < m; st *= 2) {
        __syncthreads();
        for (int i = threadIdx.x; i < m; i += blockDim.x) {
            const double a = A[i], c = C[i];
            double am = 0.0, cm = 0.0, dm = 0.0, ap = 0.0, cp = 0.0, dp = 0.0;
            if (i - st >= 0) { am = A[i - st]; cm = C[i - st]; dm = Dv[i - st]; }
            if (i + st < m) { ap = A[i + st]; cp = C[i + st]; dp = Dv[i + st]; }
            const double inv = 1.0 / fma(-a, cm, fma(-c, ap, 1.0));
            A2[i] = -a * am * inv;
            C2[i] = -c * cp * inv;
            D2[i] = fma(-a, dm, fma(-c, dp, Dv[i])) * inv;
        }
        double* t;
        t = A; A = A2; A2 = t;
        t = C; C = C2; C2 = t;
        t = Dv; Dv = D2; D2 = t;
    }
    for (int i = threadIdx.x; i < m; i += blockDim.x) {  // each thread's own rows
        b[i + 1] = Dv[i];
        bt[i + 1] = (T)Dv[i];
    }
}

template <typename T>
__global__ void __launch_bounds__(kSideThreads) boundary_kernel(const PrepParams P, int cap)
{
    extern __shared__ double side_sm[];
    boundary_side<T>(P, blockIdx.x, side_sm, cap);
}

__device__ __forceinline__ void scatter_iface_one(int nx, int ny, int periodic, double Lx, double Ly,
                                                  const int2* nodes, int m, const double* est, double* xnew,
                                                  double* ynew)
{
    const int2 ij = nodes[m];
    const double vx = est[2 * m], vy = est[2 * m + 1];
    const long id = (long)ij.y * nx + ij.x;
    xnew[id] = vx;
    ynew[id] = vy;
    if (periodic) {
        if (ij.x == 0) {
            xnew[id + nx - 1] = vx + Lx;
            ynew[id + nx - 1] = vy;
        }
        if (ij.y == 0) {
            const long w = (long)(ny - 1) * nx + ij.x;
            xnew[w] = vx;
            ynew[w] = vy + Ly;
        }
        if (ij.x == 0 && ij.y == 0) {
            const long w = (long)(ny - 1) * nx + nx - 1;
            xnew[w] = vx + Lx;
            ynew[w] = vy + Ly;
        }
    }
}

__device__ __forceinline__ void faces_body(const SolveParams& P, int inner_fp64, int blk, int nb)
{
    const int nx = P.nx, ny = P.ny;
    const long n = (long)nx * ny;
    // r (w + w')/2 / h^2, each step rounded; the half is taken into 1 / h^2, which is exact.  4097 x 4097
    // nodes: 0.45 -> 0.26 ms (44 bytes a node take 0.11) with fewer FP64 operations and conversions
    for (int id = blk * (int)blockDim.x + threadIdx.x; id < n; id += nb * (int)blockDim.x) {  // n <= 2^28
        const int j = id / nx, i = id - j * nx;
        const double w = P.om64[id];
        double e = 0.0, no = 0.0;
        if (i < nx - 1) e = __dmul_rn(P.r, __dmul_rn(__dadd_rn(w, P.om64[id + 1]), P.hx));
        if (j < ny - 1) no = __dmul_rn(P.r, __dmul_rn(__dadd_rn(w, P.om64[id + nx]), P.hy));
        P.ce64[id] = e;
        P.cn64[id] = no;
        if (inner_fp64) {
            static_cast<double*>(P.ce)[id] = e;
            static_cast<double*>(P.cn)[id] = no;
        } else {
            static_cast<float*>(P.ce)[id] = float_rn(e);
            static_cast<float*>(P.cn)[id] = float_rn(no);
        }
    }
}

// Everything a solve needs beside the monitor, in one launch: its blocks are face coefficients, then
// boundary nodes, then interface nodes.  Small grids are bound by the launches and their gaps, 3 to 4 us
// each: with the scatters as launches of their own a 257 x 257 solve call took 423 us, 409 so.
__global__ void solve_setup_kernel(const __grid_constant__ SolveParams P, int inner_fp64, int periodic, double Lx,
                                   double Ly, const int2* nodes, int M, const double* est, const double* bnd,
                                   int face_blocks, int rim_blocks)
{
    int blk = blockIdx.x;
    if (blk < face_blocks) {
        faces_body(P, inner_fp64, blk, face_blocks);
        return;
    }
    blk -= face_blocks;
    if (blk < rim_blocks) {
        scatter_boundary_one(P.nx, P.ny, Lx, Ly, P.xnew, P.ynew, bnd, blk * blockDim.x + threadIdx.x);
        return;
    }
    const int m = (blk - rim_blocks) * blockDim.x + threadIdx.x;
    if (m < M) scatter_iface_one(P.nx, P.ny, periodic, Lx, Ly, nodes, m, est, P.xnew, P.ynew);
}

// ---------------------------------------------------------------------------------------
// Batched forms: one launch over the problems of a batch.  Grid-sized work gives problem i the
// blocks blk_off[i] .. blk_off[i + 1] - 1 (each problem its own block count, as its single-problem
// launch would have); node work runs over the batch's concatenated nodes.  Every node computes
// what the single-problem kernels compute for it.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ int batch_problem_of_block(const int32_t* blk_off, int n, int b)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (blk_off[mid] <= b) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__global__ void prep_omega_batch_kernel(const BatchRec* R, const int32_t* blk_off, int n)
{
    const int i = batch_problem_of_block(blk_off, n, blockIdx.x);
    const int blk = blockIdx.x - blk_off[i], nb = blk_off[i + 1] - blk_off[i];
    if (blk == 0 && threadIdx.x == 0 && R[i].prep.bad) *R[i].prep.bad = 0;  // before the pack launch
    prep_omega_body(R[i].prep, blk, nb);
}

// Face coefficients of every problem of a batch in one launch.
__global__ void faces_batch_kernel(const SolveParams* probs, const int32_t* blk_off, int n, int inner_fp64)
{
    const int i = batch_problem_of_block(blk_off, n, blockIdx.x);
    faces_body(probs[i], inner_fp64, blockIdx.x - blk_off[i], blk_off[i + 1] - blk_off[i]);
}

template <typename T>
__global__ void __launch_bounds__(kTileX * kTileY) prep_pack_batch_kernel(const BatchRec* R, const int32_t* tile_off, int n)
{
    const int i = batch_problem_of_block(tile_off, n, blockIdx.x);
    prep_pack_tile<T>(R[i].prep, blockIdx.x - tile_off[i]);
}

template <typename T>
__global__ void __launch_bounds__(kSideThreads) boundary_batch_kernel(const BatchRec* R, int cap)
{
    extern __shared__ double side_sm[];
    const PrepParams& P = R[blockIdx.x / 4].prep;
    if (P.moving_boundary && !P.periodic) boundary_side<T>(P, blockIdx.x % 4, side_sm, cap);
}

__global__ void shift_batch_kernel(const BatchRec* R, const int32_t* node_prob, int M, double* shift)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= M) return;
    const BatchRec& r = R[node_prob[g]];
    const int2 ij = r.nodes[g - r.node_offset];
    shift[2 * g] = r.prep.x[(long)ij.y * r.prep.nx + ij.x];
    shift[2 * g + 1] = r.prep.y[(long)ij.y * r.prep.nx + ij.x];
}

__global__ void scatter_boundary_batch_kernel(const BatchRec* R, const int32_t* blk_off, int n)
{
    const int i = batch_problem_of_block(blk_off, n, blockIdx.x);
    const BatchRec& r = R[i];
    if (r.prep.periodic) return;
    const int threads = (blk_off[i + 1] - blk_off[i]) * (int)blockDim.x;
    for (int k = (blockIdx.x - blk_off[i]) * blockDim.x + threadIdx.x; k < 2 * (r.prep.nx + r.prep.ny); k += threads)
        scatter_boundary_one(r.prep.nx, r.prep.ny, r.prep.Lx, r.prep.Ly, r.xnew, r.ynew,
                             r.prep.moving_boundary ? r.prep.bnd64 : nullptr, k);
}

__global__ void scatter_iface_batch_kernel(const BatchRec* R, const int32_t* node_prob, int M, const double* est)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= M) return;
    const BatchRec& r = R[node_prob[g]];
    scatter_iface_one(r.prep.nx, r.prep.ny, r.prep.periodic, r.prep.Lx, r.prep.Ly, r.nodes, g - r.node_offset,
                      est + 2 * (size_t)r.node_offset, r.xnew, r.ynew);
}

// x <- x^{n+1}, y <- y^{n+1} of every problem (the step's last launch)
__global__ void copy_back_batch_kernel(const BatchRec* R, const int32_t* blk_off, int n)
{
    const int i = batch_problem_of_block(blk_off, n, blockIdx.x);
    const BatchRec& r = R[i];
    const int nb = blk_off[i + 1] - blk_off[i];
    const long N = (long)r.prep.nx * r.prep.ny;
    double* x = const_cast<double*>(r.prep.x);
    double* y = const_cast<double*>(r.prep.y);
    for (long id = (long)(blockIdx.x - blk_off[i]) * blockDim.x + threadIdx.x; id < N; id += (long)nb * blockDim.x) {
        x[id] = r.xnew[id];
        y[id] = r.ynew[id];
    }
}

// Geometric quality Q = tr(J^T J) / (2 |det J|) of every cell (Eq. 8), J from the mean of the
// cell's two xi-edges and two eta-edges; then the maximum and mean over the cells.
__global__ void quality_kernel(int nx, int ny, const double* x, const double* y, double* q)
{
    const long nc = (long)(nx - 1) * (ny - 1);
    for (long c = blockIdx.x * (long)blockDim.x + threadIdx.x; c < nc; c += (long)gridDim.x * blockDim.x) {
        const int i = (int)(c % (nx - 1)), j = (int)(c / (nx - 1));
        const long a = (long)j * nx + i, b = a + 1, d = a + nx, e = d + 1;
        const double x_xi = 0.5 * ((x[b] - x[a]) + (x[e] - x[d]));
        const double y_xi = 0.5 * ((y[b] - y[a]) + (y[e] - y[d]));
        const double x_eta = 0.5 * ((x[d] - x[a]) + (x[e] - x[b]));
        const double y_eta = 0.5 * ((y[d] - y[a]) + (y[e] - y[b]));
        const double tr = x_xi * x_xi + y_xi * y_xi + x_eta * x_eta + y_eta * y_eta;
        q[c] = 0.5 * tr / fabs(x_xi * y_eta - x_eta * y_xi);
    }
}

__global__ void max_mean_kernel(long n, const double* v, double* out)
{
    __shared__ double smax[32], ssum[32];
    double m = -INFINITY, s = 0.0;
    for (long k = threadIdx.x; k < n; k += blockDim.x) {
        m = fmax(m, v[k]);
        s += v[k];
    }
    for (int off = 16; off > 0; off >>= 1) {
        m = fmax(m, __shfl_xor_sync(0xffffffffu, m, off));
        s += __shfl_xor_sync(0xffffffffu, s, off);
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) { smax[w] = m; ssum[w] = s; }
    __syncthreads();
    if (threadIdx.x == 0) {  // holds warp 0's totals; add the other warps in order
        for (int k = 1; k < (int)(blockDim.x >> 5); ++k) { m = fmax(m, smax[k]); s += ssum[k]; }
        out[0] = m;
        out[1] = s / (double)n;
    }
}

// Nodes that a launch of the boundary kernels has shared memory for, n those of its longest side.
inline int side_cap(int n) { return n < kSideMax ? n : kSideMax; }
cudaError_t side_allow(const void* fn)
{
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSideMax * kSideBytes);
}

inline int blocks_for(long n, int threads) { return (int)((n + threads - 1) / threads); }

}  // namespace

int prep_tiles(int nx, int ny)
{
    return ((nx + kTileX - 1) / kTileX) * ((ny + kTileY - 1) / kTileY);
}

cudaError_t launch_prep(const PrepParams& P, cudaStream_t s)
{
    const long n = (long)P.nx * P.ny;
    // few nodes: blocks of one warp, which spread over the SMs (FP64 monitors are bound by each SM's unit)
    const int threads = n < 152 * 256 ? 32 : 256;
    // (a nodal monitor that is to be read where it is needs no copy)
    if (P.om64 != P.omega_in) prep_omega_kernel<<<blocks_for(n, threads), threads, 0, s>>>(P);
    if (P.precision == 0)
        prep_pack_kernel<double><<<prep_tiles(P.nx, P.ny), kTileX * kTileY, 0, s>>>(P);
    else
        prep_pack_kernel<float><<<prep_tiles(P.nx, P.ny), kTileX * kTileY, 0, s>>>(P);
    if (P.moving_boundary && !P.periodic) {
        const int cap = side_cap(P.nx > P.ny ? P.nx : P.ny);
        const auto fn = P.precision == 0 ? boundary_kernel<double> : boundary_kernel<float>;
        const cudaError_t e = side_allow(reinterpret_cast<const void*>(fn));
        if (e != cudaSuccess) return e;
        fn<<<4, kSideThreads, (size_t)cap * kSideBytes, s>>>(P, cap);
    }
    return cudaGetLastError();
}

cudaError_t launch_quality(int nx, int ny, const double* x, const double* y, double* q, double* stats,
                           cudaStream_t s)
{
    const long nc = (long)(nx - 1) * (ny - 1);
    quality_kernel<<<blocks_for(nc, 256), 256, 0, s>>>(nx, ny, x, y, q);
    max_mean_kernel<<<1, 1024, 0, s>>>(nc, q, stats);
    return cudaGetLastError();
}

cudaError_t launch_shift(const int2* nodes, int M, int nx, const double* x, const double* y,
                         double* shift, cudaStream_t s)
{
    shift_kernel<<<blocks_for(M, 256), 256, 0, s>>>(nodes, M, nx, x, y, shift);
    return cudaGetLastError();
}

cudaError_t launch_solve_setup(const SolveParams& P, int periodic, double Lx, double Ly, const int2* nodes, int M,
                               const double* est, const double* bnd64, bool fp64_inner, cudaStream_t s)
{
    const int faces = blocks_for((long)P.nx * P.ny, 256), rim = periodic ? 0 : blocks_for(2L * (P.nx + P.ny), 256);
    solve_setup_kernel<<<faces + rim + blocks_for(M, 256), 256, 0, s>>>(P, fp64_inner ? 1 : 0, periodic, Lx, Ly, nodes, M,
                                                                       est, bnd64, faces, rim);
    return cudaGetLastError();
}

}  // namespace sdd

namespace sdd {

int batch_blocks(long n_nodes) { return blocks_for(n_nodes, 256); }

void set_prep_consts(PrepParams& P)
{
    P.gx = 0.5 * (double)(P.nx - 1);
    P.gy = 0.5 * (double)(P.ny - 1);
    if (P.kind != 3) return;
    bool all = true;  // every amplitude finite and >= 0
    for (int b = 0; b + 3 < P.n_params; b += 4) all = all && P.params[b] >= 0.0 && isfinite(P.params[b]);
    for (int b = 0; b + 3 < P.n_params; b += 4) {
        const double W = P.params[b + 1] * P.params[b + 1];
        int e = 0;
        frexp(P.params[b], &e);
        P.bump_w2[b / 4] = W;
        P.bump_inv[b / 4] = all && W > 1e-100 && W < 1e100 ? 1.0 / W : 0.0;  // 0: the device divides
        P.bump_reach[b / 4] = all && W > 0.0 ? (56.0 + (e > -50 ? e : -50)) * 0.6931471805599454 * W : INFINITY;
    }
}

cudaError_t launch_prep_batch(const BatchRec* R, const int32_t* blk_off, const int32_t* tile_off, int n, int total_blocks,
                              int total_tiles, bool fp64, int moving_nodes, cudaStream_t s)
{
    prep_omega_batch_kernel<<<total_blocks, 256, 0, s>>>(R, blk_off, n);
    if (fp64)
        prep_pack_batch_kernel<double><<<total_tiles, kTileX * kTileY, 0, s>>>(R, tile_off, n);
    else
        prep_pack_batch_kernel<float><<<total_tiles, kTileX * kTileY, 0, s>>>(R, tile_off, n);
    if (moving_nodes > 0) {
        const int cap = side_cap(moving_nodes);
        const auto fn = fp64 ? boundary_batch_kernel<double> : boundary_batch_kernel<float>;
        const cudaError_t e = side_allow(reinterpret_cast<const void*>(fn));
        if (e != cudaSuccess) return e;
        fn<<<4 * n, kSideThreads, (size_t)cap * kSideBytes, s>>>(R, cap);
    }
    return cudaGetLastError();
}

cudaError_t launch_faces_batch(const SolveParams* probs, const int32_t* blk_off, int n, int total_blocks,
                               bool fp64_inner, cudaStream_t s)
{
    faces_batch_kernel<<<total_blocks, 256, 0, s>>>(probs, blk_off, n, fp64_inner ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_shift_batch(const BatchRec* R, const int32_t* node_prob, int M, double* shift, cudaStream_t s)
{
    if (M <= 0) return cudaSuccess;
    shift_batch_kernel<<<blocks_for(M, 256), 256, 0, s>>>(R, node_prob, M, shift);
    return cudaGetLastError();
}

cudaError_t launch_scatter_batch(const BatchRec* R, const int32_t* blk_off, int n, int total_blocks,
                                 const int32_t* node_prob, int M, const double* est, cudaStream_t s)
{
    scatter_boundary_batch_kernel<<<total_blocks, 256, 0, s>>>(R, blk_off, n);
    if (M > 0) scatter_iface_batch_kernel<<<blocks_for(M, 256), 256, 0, s>>>(R, node_prob, M, est);
    return cudaGetLastError();
}

cudaError_t launch_copy_back_batch(const BatchRec* R, const int32_t* blk_off, int n, int total_blocks, cudaStream_t s)
{
    copy_back_batch_kernel<<<total_blocks, 256, 0, s>>>(R, blk_off, n);
    return cudaGetLastError();
}

}  // namespace sdd
