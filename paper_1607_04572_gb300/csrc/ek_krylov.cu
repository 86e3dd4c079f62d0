// Poisson solve with an inhomogeneous permittivity and fixed-potential nodes
// by preconditioned conjugate gradients (FP64): a multigrid V-cycle as the
// preconditioner where the box can be coarsened, else Jacobi.
//
// The paper solves Eq. 3 (homogeneous permittivity) by FFT and leaves the
// general problem div(eps grad Phi) = -4 pi l_B q to iterative solvers such as
// SOR or Krylov subspace methods (Sec. III.C, the paragraph after Eq. 16).
// Discretisation: the 7-point operator of the periodic solve with face
// permittivities, the harmonic mean 2 eps_i eps_j / (eps_i + eps_j) of the
// face's two nodes; a free node satisfies sum_f eps_f (Phi_i - Phi_j) =
// 4 pi l_B q_i, a fixed node holds its given potential.  The operator on the
// free nodes is symmetric positive definite (semidefinite with no fixed node:
// then the charge's mean is removed and Phi is returned with mean 0, as by
// the FFT solve).
//
// Every reduction (the CG inner products) is a fixed-order sum: each thread
// of a fixed grid adds its grid-stride elements in order, the block adds its
// threads in a fixed tree, and the last block to finish adds the block sums in
// order and forms the scalar that needs them; so a solve is bit-reproducible.
// The scalars alpha and beta stay on the device; the host reads the residual
// every CG_CHECK (Jacobi) or PCG_CHECK (multigrid) iterations.
//
// What bounds it: the FP64 pipe (2 lanes per clock per SM) on the fine level,
// launches on the coarse ones.  So the smoother gathers (b + sum c_f x_f) / D
// with the stored diagonal D (7 FP64 instructions a node; differences
// c_f (x - x_f) take 13), residuals are formed only where they are not zero,
// and corrections are added only where they are read.  The outer operator keeps
// the differences: its rounding is the solution's.  128^3, dielectric sphere
// between electrodes, tol 1e-12 (GB300): 32 iterations of 0.60 ms (18.9 ms)
// with damped Jacobi V(2,2) cycles and a launch per scalar, 18 of 0.41 ms (7.3
// ms) with red-black Gauss-Seidel.  Of an iteration at 128^3 (launches one by
// one, cold L2) the fine level's half sweeps take 0.138 ms, the operator 0.065
// (FP64 pipe 43 us), the small levels 0.074, 64^3 0.054, the update 0.033,
// the restriction 0.029.
#include <math.h>

#include <algorithm>
#include <atomic>

#include <cooperative_groups.h>

#include "ek_internal.cuh"

namespace ek {

namespace cg = cooperative_groups;

namespace {

constexpr int CG_T = 256;         // threads per block
constexpr int CG_BLOCKS = 608;    // blocks of the grid-stride kernels (4 per SM: a block's FP64 sum is
                                  // spread over more nodes than with 8)
constexpr int CG_CHECK = 10;      // iterations between residual reads (Jacobi)
constexpr int PCG_CHECK = 2;      // with the multigrid V-cycle (an iteration costs several)

// scalars on the device: [0] r.z, [1] p.Ap, [2] alpha, [3] beta, [4] r.r,
// [5] b.b (then sum x), [6] sum q, [7] fixed-node count, [8] permittivities
// that are not positive and finite, [9] sum of D^-1, [10] mean of r to remove,
// [12] the counter of finished blocks
//
// Without fixed nodes the operator is singular (constants): b has mean 0, and
// so has r = b - A x in exact arithmetic, but rounding lets a constant
// component creep into r, which A cannot remove; once the rest of r has
// converged, p points along it, p.Ap vanishes and alpha blows up.  There the
// mean of r is removed every iteration (r.z and r.r are formed for the
// projected r from the partial sums of r and D^-1 r).
struct CGView {
  double* cf;       // 3N: permittivity of the +x, +y, +z face of each node
  double* dinv;     // N: 1 / diagonal on free nodes, 0 on fixed nodes
  double* r;        // N: residual
  double* p;        // N: search direction
  double* ap;       // N: A p
  double* part;     // 4 * CG_BLOCKS block sums
  double* sc;       // 16 scalars
};

size_t cg_layout(long long N, CGView* v, void* base) {
  size_t off = 0;
  auto take = [&](double** ptr, size_t count) {
    off = (off + 255) & ~(size_t)255;
    if (v) *ptr = (double*)((char*)base + off);
    off += count * sizeof(double);
  };
  double* dummy = nullptr;
  take(v ? &v->cf : &dummy, 3 * (size_t)N);
  take(v ? &v->dinv : &dummy, (size_t)N);
  take(v ? &v->r : &dummy, (size_t)N);
  take(v ? &v->p : &dummy, (size_t)N);
  take(v ? &v->ap : &dummy, (size_t)N);
  take(v ? &v->part : &dummy, 4 * CG_BLOCKS);
  take(v ? &v->sc : &dummy, 16);
  return off;
}

struct Box {
  int nx, ny, nz;
  long long N;
};

// harmonic mean; equal values (most faces of a piecewise constant medium) need
// no division, which costs some 20 FP64 instructions
__device__ __forceinline__ double harmonic(double a, double b) { return a == b ? a : 2.0 * a * b / (a + b); }

// v is zero (a fixed node's D^-1), from its bits: no FP64 instruction
__device__ __forceinline__ bool is_zero(double v) { return (__double_as_longlong(v) << 1) == 0; }

// the block's sum of v (every thread), in a fixed tree; valid in thread 0
__device__ __forceinline__ double block_total(double v) {
  __shared__ double ws[CG_T / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  __syncthreads();  // ws is reused by the next call
  if (lane == 0) ws[w] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < CG_T / 32; ++i) t += ws[i];
  return t;
}

// the sum of part[row * CG_BLOCKS + 0 .. nb) by one block: each thread adds
// its strided entries in order, then the fixed tree; valid in thread 0
__device__ __forceinline__ double row_total(const double* part, int row, int nb) {
  double t = 0.0;
  for (int i = threadIdx.x; i < nb; i += CG_T) t += part[row * CG_BLOCKS + i];
  return block_total(t);
}

// true in every thread of the last block of the grid to get here, with the
// other blocks' partial sums visible; the counter is left at zero
__device__ __forceinline__ bool last_block(const CGView& v) {
  __shared__ bool last;
  if (threadIdx.x == 0) {
    __threadfence();
    unsigned* count = reinterpret_cast<unsigned*>(v.sc + 12);
    const unsigned done = atomicAdd(count, 1u);
    last = done == gridDim.x - 1;
    if (last) {
      *count = 0u;
      __threadfence();
    }
  }
  __syncthreads();
  return last;
}

// the neighbours of node n = (x, y, z) across its +x, -x, +y, -y, +z, -z faces
__device__ __forceinline__ void neighbours(int nx, int ny, int nz, int n, int x, int y, int z, int (&m)[6]) {
  const int sy = nx, sz = nx * ny;
  m[0] = n + (x + 1 < nx ? 1 : 1 - nx);
  m[1] = n + (x > 0 ? -1 : nx - 1);
  m[2] = n + (y + 1 < ny ? sy : sy - sz);
  m[3] = n + (y > 0 ? -sy : sz - sy);
  m[4] = n + (z + 1 < nz ? sz : sz - sz * nz);
  m[5] = n + (z > 0 ? -sz : sz * nz - sz);
}
__device__ __forceinline__ void node_xyz(int nx, int ny, int n, int& x, int& y, int& z) {
  const unsigned row = (unsigned)n / (unsigned)nx;
  x = n - (int)row * nx;
  z = (int)(row / (unsigned)ny);
  y = (int)row - z * ny;
}

// face permittivities; the sum of q, the number of fixed nodes and of
// permittivities that are not positive and finite
__global__ void __launch_bounds__(CG_T) k_cg_faces(Box b, CGView v, const double* q, const double* eps,
                                                   const unsigned char* fixed) {
  double sq = 0.0;
  int nf = 0, ne = 0;
  for (long long i = blockIdx.x * (long long)CG_T + threadIdx.x; i < b.N; i += (long long)gridDim.x * CG_T) {
    const int n = (int)i;
    sq += q[n];
    if (fixed && fixed[n]) ++nf;
    double c0 = 1.0, c1 = 1.0, c2 = 1.0;
    if (eps) {
      int x, y, z, m[6];
      node_xyz(b.nx, b.ny, n, x, y, z);
      neighbours(b.nx, b.ny, b.nz, n, x, y, z, m);
      const double e = eps[n];
      if (!(e > 0.0 && e < INFINITY)) ++ne;
      c0 = harmonic(e, eps[m[0]]);
      c1 = harmonic(e, eps[m[2]]);
      c2 = harmonic(e, eps[m[4]]);
    }
    v.cf[n] = c0;
    v.cf[b.N + n] = c1;
    v.cf[2 * b.N + n] = c2;
  }
  sq = block_total(sq);
  const double df = block_total((double)nf), de = block_total((double)ne);
  if (threadIdx.x == 0) {
    v.part[blockIdx.x] = sq;
    v.part[CG_BLOCKS + blockIdx.x] = df;
    v.part[2 * CG_BLOCKS + blockIdx.x] = de;
  }
  if (!last_block(v)) return;
  const double a = row_total(v.part, 0, gridDim.x), c = row_total(v.part, 1, gridDim.x),
               d = row_total(v.part, 2, gridDim.x);
  if (threadIdx.x == 0) {
    v.sc[6] = a;
    v.sc[7] = c;
    v.sc[8] = d;
  }
}

// diagonal, right-hand side and the start x = 0 (free) / phi_fixed (fixed);
// r = b, p = D^-1 r (Jacobi); r.p, b.b and the sum of D^-1.  Without fixed
// nodes the mean charge is removed.
__global__ void __launch_bounds__(CG_T) k_cg_prep(Box b, CGView v, double* D, const double* q,
                                                  const unsigned char* fixed, const double* phi_fixed,
                                                  double* x, double scale) {
  const double qmean = v.sc[7] == 0.0 ? v.sc[6] / (double)b.N : 0.0;
  double rz = 0.0, bb = 0.0, sd = 0.0;
  for (long long i = blockIdx.x * (long long)CG_T + threadIdx.x; i < b.N; i += (long long)gridDim.x * CG_T) {
    const int n = (int)i;
    int xx, yy, zz, m[6];
    node_xyz(b.nx, b.ny, n, xx, yy, zz);
    neighbours(b.nx, b.ny, b.nz, n, xx, yy, zz, m);
    const double f[6] = {v.cf[n],           v.cf[m[1]],           v.cf[b.N + n],
                         v.cf[b.N + m[3]], v.cf[2 * b.N + n], v.cf[2 * b.N + m[5]]};
    const double d = ((f[0] + f[1]) + (f[2] + f[3])) + (f[4] + f[5]);
    D[n] = d;
    const bool fx = fixed && fixed[n];
    if (fx) {
      const double pv = phi_fixed ? phi_fixed[n] : 0.0;
      x[n] = pv;
      v.dinv[n] = 0.0;
      v.r[n] = 0.0;
      v.p[n] = 0.0;
      continue;
    }
    double rhs = scale * (q[n] - qmean);
    if (fixed) {
#pragma unroll
      for (int k = 0; k < 6; ++k)
        if (fixed[m[k]]) rhs += f[k] * (phi_fixed ? phi_fixed[m[k]] : 0.0);
    }
    const double di = 1.0 / d;
    x[n] = 0.0;
    v.dinv[n] = di;
    v.r[n] = rhs;
    v.p[n] = di * rhs;
    rz += di * rhs * rhs;
    bb += rhs * rhs;
    sd += di;
  }
  rz = block_total(rz);
  bb = block_total(bb);
  sd = block_total(sd);
  if (threadIdx.x == 0) {
    v.part[blockIdx.x] = rz;
    v.part[CG_BLOCKS + blockIdx.x] = bb;
    v.part[2 * CG_BLOCKS + blockIdx.x] = sd;
  }
  if (!last_block(v)) return;
  const double a = row_total(v.part, 0, gridDim.x), c = row_total(v.part, 1, gridDim.x),
               e = row_total(v.part, 2, gridDim.x);
  if (threadIdx.x == 0) {
    v.sc[0] = a;
    v.sc[5] = c;
    v.sc[9] = e;
  }
}

// Ap on the free nodes (p is 0 on fixed nodes); alpha = r.z / p.Ap.  The
// work items are the 32 x 8 tiles of every plane (tx x ty tiles per plane);
// block b takes items b, b + gridDim.x, ...: node coordinates come from the
// item, with no division per node.
__global__ void __launch_bounds__(CG_T) k_cg_apply(Box b, CGView v, int tx, int ty) {
  let_next_start();
  after_previous();
  const int N = (int)b.N, sy = b.nx, sz = b.nx * b.ny;
  const int items = tx * ty * b.nz;
  const double* __restrict__ cx = v.cf;
  const double* __restrict__ cy = v.cf + N;
  const double* __restrict__ cz = v.cf + 2 * (size_t)N;
  double pap = 0.0;
  for (int w = blockIdx.x; w < items; w += gridDim.x) {
    const int bx = w % tx, by = (w / tx) % ty, z = w / (tx * ty);
    const int x = bx * 32 + (threadIdx.x & 31), y = by * 8 + (threadIdx.x >> 5);
    if (x >= b.nx || y >= b.ny) continue;
    const int n = x + sy * y + sz * z;
    if (is_zero(v.dinv[n])) {
      v.ap[n] = 0.0;
      continue;
    }
    const int dxp = x + 1 < b.nx ? 1 : 1 - b.nx, dxm = x > 0 ? -1 : b.nx - 1;
    const int dyp = y + 1 < b.ny ? sy : sy - sz, dym = y > 0 ? -sy : sz - sy;
    const int dzp = z + 1 < b.nz ? sz : sz - N, dzm = z > 0 ? -sz : N - sz;
    const double pn = v.p[n];
    const double a = cx[n] * (pn - v.p[n + dxp]) + cx[n + dxm] * (pn - v.p[n + dxm]) +
                     cy[n] * (pn - v.p[n + dyp]) + cy[n + dym] * (pn - v.p[n + dym]) +
                     cz[n] * (pn - v.p[n + dzp]) + cz[n + dzm] * (pn - v.p[n + dzm]);
    v.ap[n] = a;
    pap += pn * a;
  }
  pap = block_total(pap);
  if (threadIdx.x == 0) v.part[blockIdx.x] = pap;
  if (!last_block(v)) return;
  pap = row_total(v.part, 0, gridDim.x);
  if (threadIdx.x == 0) {
    v.sc[1] = pap;
    v.sc[2] = pap > 0.0 ? v.sc[0] / pap : 0.0;
  }
}

// x += alpha p, r -= alpha Ap; r.z, r.r, and (for the projection) the sums of
// r and D^-1 r; then beta = r.z(new) / r.z(old), r.r for the convergence test
// and, with the projection (every node free), m = mean r and r.z, r.r of r - m
__global__ void __launch_bounds__(CG_T) k_cg_update(Box b, CGView v, double* x, int neutral) {
  let_next_start();
  after_previous();
  const double alpha = v.sc[2];
  double rz = 0.0, rr = 0.0, s1 = 0.0, s2 = 0.0;
  for (long long n = blockIdx.x * (long long)CG_T + threadIdx.x; n < b.N; n += (long long)gridDim.x * CG_T) {
    const double di = v.dinv[n];
    if (is_zero(di)) continue;
    x[n] += alpha * v.p[n];
    const double rn = v.r[n] - alpha * v.ap[n];
    v.r[n] = rn;
    rz += di * rn * rn;
    rr += rn * rn;
    if (neutral) {
      s1 += rn;
      s2 += di * rn;
    }
  }
  rz = block_total(rz);
  rr = block_total(rr);
  if (neutral) {
    s1 = block_total(s1);
    s2 = block_total(s2);
  }
  if (threadIdx.x == 0) {
    v.part[blockIdx.x] = rz;
    v.part[CG_BLOCKS + blockIdx.x] = rr;
    if (neutral) {
      v.part[2 * CG_BLOCKS + blockIdx.x] = s1;
      v.part[3 * CG_BLOCKS + blockIdx.x] = s2;
    }
  }
  if (!last_block(v)) return;
  const int nb = gridDim.x;
  rz = row_total(v.part, 0, nb);
  rr = row_total(v.part, 1, nb);
  if (neutral) {
    s1 = row_total(v.part, 2, nb);
    s2 = row_total(v.part, 3, nb);
  }
  if (threadIdx.x == 0) {
    double m = 0.0;
    if (neutral) {
      m = s1 / (double)b.N;
      rz = rz - 2.0 * m * s2 + m * m * v.sc[9];
      rr = rr - m * s1;
    }
    v.sc[10] = m;
    v.sc[3] = v.sc[0] > 0.0 ? rz / v.sc[0] : 0.0;
    v.sc[0] = rz;
    v.sc[4] = rr;
  }
}

// r -= m (the projection; m = 0 with fixed nodes), p = D^-1 r + beta p on
// the free nodes
__global__ void __launch_bounds__(CG_T) k_cg_direction(Box b, CGView v, int neutral) {
  let_next_start();
  after_previous();
  const double beta = v.sc[3], m = v.sc[10];
  const unsigned n = blockIdx.x * CG_T + threadIdx.x;
  if (n >= (unsigned)b.N) return;
  const double di = v.dinv[n];
  if (is_zero(di)) return;
  double rn = v.r[n];
  if (neutral) v.r[n] = rn -= m;
  v.p[n] = di * rn + beta * v.p[n];
}

// the sum of x (for the mean of a solution without fixed nodes)
__global__ void __launch_bounds__(CG_T) k_cg_sum(Box b, CGView v, const double* x) {
  double s = 0.0;
  for (long long n = blockIdx.x * (long long)CG_T + threadIdx.x; n < b.N; n += (long long)gridDim.x * CG_T)
    s += x[n];
  s = block_total(s);
  if (threadIdx.x == 0) v.part[blockIdx.x] = s;
  if (!last_block(v)) return;
  s = row_total(v.part, 0, gridDim.x);
  if (threadIdx.x == 0) v.sc[5] = s;
}

__global__ void __launch_bounds__(CG_T) k_cg_shift(Box b, double* x, const double* sc) {
  const double mean = sc[5] / (double)b.N;
  for (long long n = blockIdx.x * (long long)CG_T + threadIdx.x; n < b.N; n += (long long)gridDim.x * CG_T)
    x[n] -= mean;
}

// ---------------------------------------------------------------------------
// Multigrid preconditioner: one V-cycle z = M r of the same operator.  The next
// level halves every edge of at least 8 nodes (rounded up: the last coarse node
// of an odd edge covers one) and keeps the others; levels end when no edge is
// left to halve.  Coarse face permittivity: the fine faces it covers, summed,
// over the halving along the face's axis (the flux through them over a distance
// twice as long); a coarse node is fixed (zero correction) when one of its
// nodes is.  Restriction sums the residuals of a coarse node's nodes,
// prolongation copies its correction to them (the transpose).  Smoother: two
// red-black Gauss-Seidel sweeps before (red first) and after (black first, the
// adjoint) on levels whose edges are all even, else two sweeps of damped Jacobi
// (omega = 0.8: the colours of a periodic odd edge meet); the coarsest level
// takes a few Jacobi sweeps from zero.  Every part is symmetric, so the V-cycle is
// a symmetric positive definite preconditioner for CG.
//
// Iterations to 1e-12 (dielectric sphere, fixed planes): Jacobi V(2,2) 27 at
// 64^3, Gauss-Seidel V(1,1) 32 and V(2,2) 16, with trilinear transfers 17; a
// 53^3 box, which only takes Jacobi sweeps, 28 (650 without the V-cycle).
// ---------------------------------------------------------------------------
constexpr int MG_MAXLEV = 12;
constexpr double MG_OMEGA = 0.8;

struct MGLevel {
  int nx, ny, nz, n;
  int rb;          // all edges even: red-black Gauss-Seidel
  int fx, fy, fz;  // halving towards the next level (2 or 1 per axis)
  double* cf;      // 3n face permittivities (+x, +y, +z)
  double* dinv;    // n: 1 / diagonal, 0 on fixed nodes
  double* D;       // n: diagonal
  double* x;       // n: the level's correction
  double* xt;      // n: the other Jacobi buffer
  double* b;       // n: the level's right-hand side
};

// sweeps on the coarsest level: enough to cross its longest edge (4: 2, 7: 8;
// 40 sweeps save no iteration: 64^3, coarsest 4^3, 16 with 2 or 40; 48 x 88 x
// 104, coarsest 6 x 6 x 7, 17 with 8 or 40, 21 with 2)
__host__ __device__ inline int coarse_sweeps(int nx, int ny, int nz) {
  const int e = nx > ny ? (nx > nz ? nx : nz) : (ny > nz ? ny : nz);
  return e > 4 ? 2 * (e - 3) : 2;
}

// b + sum over the faces of c_f x_f at node n of level L (x is 0 on fixed nodes)
__device__ __forceinline__ double level_gather(const MGLevel& L, const double* x, int n, int xx, int yy, int zz) {
  int m[6];
  neighbours(L.nx, L.ny, L.nz, n, xx, yy, zz, m);
  const double* cy = L.cf + L.n;
  const double* cz = L.cf + 2 * (size_t)L.n;
  double s = fma(L.cf[n], x[m[0]], L.b[n]);
  s = fma(L.cf[m[1]], x[m[1]], s);
  s = fma(cy[n], x[m[2]], s);
  s = fma(cy[m[3]], x[m[3]], s);
  s = fma(cz[n], x[m[4]], s);
  return fma(cz[m[5]], x[m[5]], s);
}
// node j of a colour (x + y + z even: red, colour 0)
__device__ __forceinline__ int colour_node(const MGLevel& L, unsigned j, int colour, int& x, int& y, int& z) {
  const unsigned hx = (unsigned)L.nx >> 1, row = j / hx;
  z = (int)(row / (unsigned)L.ny);
  y = (int)row - z * L.ny;
  x = 2 * (int)(j - row * hx) + ((y + z + colour) & 1);
  return x + L.nx * (int)row;
}

// beta = r.z(new) / r.z(old) from the block sums of r.z (first: r.z only)
__device__ __forceinline__ void finish_beta(const CGView& v, double t, int first) {
  t = block_total(t);
  if (threadIdx.x == 0) v.part[blockIdx.x] = t;
  if (!last_block(v)) return;
  const double rz = row_total(v.part, 0, gridDim.x);
  if (threadIdx.x == 0) {
    v.sc[3] = (!first && v.sc[0] > 0.0) ? rz / v.sc[0] : 0.0;
    v.sc[0] = rz;
  }
}

// one half of a Gauss-Seidel sweep, in place: the nodes of one colour from
// their neighbours, which all have the other
__device__ __forceinline__ void half_node(const MGLevel& L, unsigned j, int colour) {
  int x, y, z;
  const int n = colour_node(L, j, colour, x, y, z);
  L.x[n] = L.dinv[n] * level_gather(L, L.x, n, x, y, z);
}
__global__ void __launch_bounds__(CG_T) k_mg_half(MGLevel L, int colour) {
  let_next_start();
  after_previous();
  const unsigned j = blockIdx.x * CG_T + threadIdx.x;
  if (j < (unsigned)L.n / 2) half_node(L, j, colour);
}
// the last half sweep (red) of the fine level, with b.x: a red node's
// neighbour x ^ 1 in the row is black and final
__global__ void __launch_bounds__(CG_T) k_mg_half_dot(MGLevel L, CGView v, int first) {
  let_next_start();
  after_previous();
  double t = 0.0;
  for (unsigned j = blockIdx.x * CG_T + threadIdx.x; j < (unsigned)L.n / 2; j += gridDim.x * CG_T) {
    int x, y, z;
    const int n = colour_node(L, j, 0, x, y, z);
    const double xn = L.dinv[n] * level_gather(L, L.x, n, x, y, z);
    L.x[n] = xn;
    const int o = n + 1 - 2 * (x & 1);
    t = fma(L.b[n], xn, fma(L.b[o], L.x[o], t));
  }
  finish_beta(v, t, first);
}

// one damped Jacobi sweep: out = in + omega D^-1 (b - A in); in == nullptr:
// from zero (out = omega D^-1 b)
__device__ __forceinline__ double jacobi_node(const MGLevel& L, const double* in, int n) {
  const double di = L.dinv[n];
  if (!in) return MG_OMEGA * di * L.b[n];
  if (is_zero(di)) return 0.0;
  int x, y, z;
  node_xyz(L.nx, L.ny, n, x, y, z);
  return fma(MG_OMEGA * di, level_gather(L, in, n, x, y, z), (1.0 - MG_OMEGA) * in[n]);
}
__global__ void __launch_bounds__(CG_T) k_mg_jacobi(MGLevel L, const double* in, double* out) {
  let_next_start();
  after_previous();
  const unsigned n = blockIdx.x * CG_T + threadIdx.x;
  if (n < (unsigned)L.n) out[n] = jacobi_node(L, in, (int)n);
}
// the last sweep of the fine level, with b.x
__global__ void __launch_bounds__(CG_T) k_mg_jacobi_dot(MGLevel L, const double* in, double* out, CGView v, int first) {
  let_next_start();
  after_previous();
  double t = 0.0;
  for (unsigned i = blockIdx.x * CG_T + threadIdx.x; i < (unsigned)L.n; i += gridDim.x * CG_T) {
    const int n = (int)i;
    const double xn = jacobi_node(L, in, n);
    out[n] = xn;
    t = fma(L.b[n], xn, t);
  }
  finish_beta(v, t, first);
}

// coarse right-hand side: the sum of the fine residuals (0 at fixed nodes).
// After a red-black sweep the residuals of the black nodes are zero (to
// rounding): only the red ones are formed.  On a red-black coarse level its
// first half sweep from zero, x = D^-1 b on the red nodes, comes along.
__device__ __forceinline__ void restrict_node(const MGLevel& F, const MGLevel& C, int n) {
  int X, Y, Z;
  node_xyz(C.nx, C.ny, n, X, Y, Z);
  const double di = C.dinv[n];
  double s = 0.0;
  auto residual = [&](int x, int y, int z) -> double {
    const int m = x + F.nx * (y + F.ny * z);
    const double v = fma(-F.D[m], F.x[m], level_gather(F, F.x, m, x, y, z));
    return is_zero(F.dinv[m]) ? 0.0 : v;
  };
  if (!is_zero(di)) {
    if (F.rb && F.fx + F.fy + F.fz == 6) {
      // the four red children, their loads in flight together
      const int x = 2 * X, y = 2 * Y, z = 2 * Z;
      const double r0 = residual(x, y, z), r1 = residual(x + 1, y + 1, z), r2 = residual(x + 1, y, z + 1),
                   r3 = residual(x, y + 1, z + 1);
      s = (r0 + r1) + (r2 + r3);
    } else {
      for (int c = 0; c < 8; ++c) {
        const int cx = c & 1, cy = (c >> 1) & 1, cz = c >> 2;
        if (cx >= F.fx || cy >= F.fy || cz >= F.fz) continue;
        const int x = F.fx * X + cx, y = F.fy * Y + cy, z = F.fz * Z + cz;
        if (x >= F.nx || y >= F.ny || z >= F.nz) continue;
        if (F.rb && ((x + y + z) & 1)) continue;
        s += residual(x, y, z);
      }
    }
  }
  C.b[n] = s;
  if (C.rb && !((X + Y + Z) & 1)) C.x[n] = di * s;
}
__global__ void __launch_bounds__(CG_T) k_mg_restrict(MGLevel F, MGLevel C) {
  let_next_start();
  after_previous();
  const unsigned n = blockIdx.x * CG_T + threadIdx.x;
  if (n < (unsigned)C.n) restrict_node(F, C, (int)n);
}

// fine x += the coarse correction (free fine nodes; on a red-black level only
// the red ones: the black half sweep that follows does not read the others)
__device__ __forceinline__ void prolong_node(const MGLevel& F, const MGLevel& C, unsigned j) {
  int x, y, z, n = (int)j;
  if (F.rb) n = colour_node(F, j, 0, x, y, z);
  else node_xyz(F.nx, F.ny, n, x, y, z);
  if (!is_zero(F.dinv[n]))
    F.x[n] += C.x[(x >> (F.fx - 1)) + C.nx * ((y >> (F.fy - 1)) + C.ny * (z >> (F.fz - 1)))];
}
__global__ void __launch_bounds__(CG_T) k_mg_prolong(MGLevel F, MGLevel C) {
  let_next_start();
  after_previous();
  const unsigned j = blockIdx.x * CG_T + threadIdx.x;
  if (j < (unsigned)(F.rb ? F.n / 2 : F.n)) prolong_node(F, C, j);
}

// the coarse level's faces and fixed nodes from the fine level
__global__ void __launch_bounds__(CG_T) k_mg_coarsen(MGLevel F, MGLevel C) {
  let_next_start();
  after_previous();
  const int n = (int)(blockIdx.x * CG_T + threadIdx.x);
  if ((unsigned)n >= (unsigned)C.n) return;
  int X, Y, Z;
  node_xyz(C.nx, C.ny, n, X, Y, Z);
  bool fixed = false;
  double fc[3] = {0.0, 0.0, 0.0};
  for (int c = 0; c < 8; ++c) {
    const int cx = c & 1, cy = (c >> 1) & 1, cz = c >> 2;
    if (cx >= F.fx || cy >= F.fy || cz >= F.fz) continue;
    const int x = F.fx * X + cx, y = F.fy * Y + cy, z = F.fz * Z + cz;
    if (x >= F.nx || y >= F.ny || z >= F.nz) continue;
    const int m = x + F.nx * (y + F.ny * z);
    fixed |= F.dinv[m] == 0.0;
    // the fine faces on the coarse node's + side: its last nodes along the axis
    if (cx == F.fx - 1 || x == F.nx - 1) fc[0] += F.cf[m];
    if (cy == F.fy - 1 || y == F.ny - 1) fc[1] += F.cf[F.n + m];
    if (cz == F.fz - 1 || z == F.nz - 1) fc[2] += F.cf[2 * (size_t)F.n + m];
  }
  C.cf[n] = F.fx == 2 ? 0.5 * fc[0] : fc[0];
  C.cf[C.n + n] = F.fy == 2 ? 0.5 * fc[1] : fc[1];
  C.cf[2 * (size_t)C.n + n] = F.fz == 2 ? 0.5 * fc[2] : fc[2];
  C.dinv[n] = fixed ? 0.0 : 1.0;  // marks the fixed nodes; the diagonal follows
}

__global__ void __launch_bounds__(CG_T) k_mg_diag(MGLevel C) {
  let_next_start();
  after_previous();
  const int n = (int)(blockIdx.x * CG_T + threadIdx.x);
  if ((unsigned)n >= (unsigned)C.n) return;
  int x, y, z, m[6];
  node_xyz(C.nx, C.ny, n, x, y, z);
  neighbours(C.nx, C.ny, C.nz, n, x, y, z, m);
  const double d = C.cf[n] + C.cf[m[1]] + C.cf[C.n + n] + C.cf[C.n + m[3]] + C.cf[2 * (size_t)C.n + n] +
                   C.cf[2 * (size_t)C.n + m[5]];
  C.D[n] = d;
  if (C.dinv[n] != 0.0) C.dinv[n] = 1.0 / d;
}

// The cycle below a level: the levels of at most MG_SMALL nodes in one launch
// of one cluster, whose CTAs meet at cluster barriers between the half sweeps.
// Each of these phases is short: as launches of their own (nine per level) they
// took 3 to 4 us each, most of an iteration at 64^3.  The FP64 pipes of 16 SMs
// hold up to 32^3 nodes (15 us); a part of a GPU that cannot place a cluster of 16
// (above the portable size) takes a smaller one, with the same result.  The coarsest level (every edge below 8: at
// most 343 nodes) is done by the first CTA, a node per thread with its faces in
// registers and x in shared memory.
constexpr int MG_COARSE_MAX = 343;
constexpr int MG_SMALL = 40000;
constexpr int MG_SMALL_T = 512;
constexpr int MG_SMALL_CTAS = 16;
struct MGSmall {
  MGLevel lev[MG_MAXLEV];  // the first is the caller's: its right-hand side (and first half sweep) is ready
  int n;
};
__device__ void coarse_solve(const MGLevel& C) {
  __shared__ double xs[2][MG_COARSE_MAX];
  const int n = threadIdx.x;
  const bool in = n < C.n;
  int m[6] = {0, 0, 0, 0, 0, 0};
  double c[6] = {}, wd = 0.0, wb = 0.0;
  if (in) {
    int x, y, z;
    node_xyz(C.nx, C.ny, n, x, y, z);
    neighbours(C.nx, C.ny, C.nz, n, x, y, z, m);
    wd = MG_OMEGA * C.dinv[n];
    wb = wd * C.b[n];
    c[0] = wd * C.cf[n];
    c[1] = wd * C.cf[m[1]];
    c[2] = wd * C.cf[C.n + n];
    c[3] = wd * C.cf[C.n + m[3]];
    c[4] = wd * C.cf[2 * C.n + n];
    c[5] = wd * C.cf[2 * C.n + m[5]];
    xs[0][n] = wb;
  }
  __syncthreads();
  const double keep = wd == 0.0 ? 0.0 : 1.0 - MG_OMEGA;
  double xn = wb;
  const int sweeps = coarse_sweeps(C.nx, C.ny, C.nz);
  for (int s = 1; s < sweeps; ++s) {
    const double* const cur = xs[(s + 1) & 1];
    if (in) {
      const double a = fma(c[0], cur[m[0]], fma(keep, xn, wb)), b = c[1] * cur[m[1]];
      const double d = fma(c[2], cur[m[2]], a), e = fma(c[3], cur[m[3]], b);
      xn = fma(c[4], cur[m[4]], d) + fma(c[5], cur[m[5]], e);
      xs[s & 1][n] = xn;
    }
    __syncthreads();
  }
  if (in) C.x[n] = xn;
}
__global__ void __launch_bounds__(MG_SMALL_T) k_mg_small(const __grid_constant__ MGSmall S) {
  let_next_start();
  after_previous();
  cg::cluster_group cl = cg::this_cluster();
  const unsigned first = blockIdx.x * MG_SMALL_T + threadIdx.x, step = gridDim.x * MG_SMALL_T;
  auto half = [&](const MGLevel& A, int colour) {
    for (unsigned j = first; j < (unsigned)A.n / 2; j += step) half_node(A, j, colour);
    cl.sync();
  };
  auto jacobi = [&](const MGLevel& A, const double* in, double* out) {
    for (unsigned n = first; n < (unsigned)A.n; n += step) out[n] = jacobi_node(A, in, (int)n);
    cl.sync();
  };
  for (int l = 0; l < S.n - 1; ++l) {
    const MGLevel& A = S.lev[l];
    const MGLevel& C = S.lev[l + 1];
    if (A.rb) {
      half(A, 1);
      half(A, 0);
      half(A, 1);
    } else {
      jacobi(A, nullptr, A.xt);
      jacobi(A, A.xt, A.x);
    }
    for (unsigned n = first; n < (unsigned)C.n; n += step) restrict_node(A, C, (int)n);
    cl.sync();
  }
  if (blockIdx.x == 0) coarse_solve(S.lev[S.n - 1]);
  cl.sync();
  for (int l = S.n - 2; l >= 0; --l) {
    const MGLevel& A = S.lev[l];
    for (unsigned j = first; j < (unsigned)(A.rb ? A.n / 2 : A.n); j += step) prolong_node(A, S.lev[l + 1], j);
    cl.sync();
    if (A.rb) {
      half(A, 1);
      half(A, 0);
      half(A, 1);
      half(A, 0);
    } else {
      jacobi(A, A.x, A.xt);
      jacobi(A, A.xt, A.x);
    }
  }
}

// x += alpha p, r -= alpha Ap; r.r and (for the projection) the mean of r.
// Without the projection the preconditioner's first half sweep from zero,
// z = D^-1 r on the red nodes, comes along.
__global__ void __launch_bounds__(CG_T) k_pcg_update(Box b, CGView v, double* x, MGLevel L, int neutral) {
  let_next_start();
  after_previous();
  const double alpha = v.sc[2];
  double rr = 0.0, s1 = 0.0;
  for (long long i = blockIdx.x * (long long)CG_T + threadIdx.x; i < b.N; i += (long long)gridDim.x * CG_T) {
    const int n = (int)i;
    const double di = v.dinv[n];
    double rn = 0.0;
    if (!is_zero(di)) {
      x[n] += alpha * v.p[n];
      rn = v.r[n] - alpha * v.ap[n];
      v.r[n] = rn;
      rr += rn * rn;
      if (neutral) s1 += rn;
    }
    if (!neutral && L.rb) {
      int xx, yy, zz;
      node_xyz(b.nx, b.ny, n, xx, yy, zz);
      if (!((xx + yy + zz) & 1)) L.x[n] = di * rn;
    }
  }
  rr = block_total(rr);
  if (neutral) s1 = block_total(s1);
  if (threadIdx.x == 0) {
    v.part[blockIdx.x] = rr;
    v.part[CG_BLOCKS + blockIdx.x] = s1;
  }
  if (!last_block(v)) return;
  rr = row_total(v.part, 0, gridDim.x);
  if (neutral) s1 = row_total(v.part, 1, gridDim.x);
  if (threadIdx.x == 0) {
    const double m = neutral ? s1 / (double)b.N : 0.0;
    v.sc[10] = m;
    v.sc[4] = neutral ? rr - m * s1 : rr;
  }
}

// r -= its mean (only without fixed nodes; before the first cycle m = 0), and
// the preconditioner's first half sweep from zero
__global__ void __launch_bounds__(CG_T) k_pcg_project(Box b, CGView v, MGLevel L, int shift) {
  let_next_start();
  after_previous();
  const double m = shift ? v.sc[10] : 0.0;
  for (long long i = blockIdx.x * (long long)CG_T + threadIdx.x; i < b.N; i += (long long)gridDim.x * CG_T) {
    const int n = (int)i;
    const double di = v.dinv[n];
    double rn = v.r[n];
    if (shift && !is_zero(di)) v.r[n] = rn -= m;
    if (L.rb) {
      int xx, yy, zz;
      node_xyz(b.nx, b.ny, n, xx, yy, zz);
      if (!((xx + yy + zz) & 1)) L.x[n] = di * rn;
    }
  }
}

// p = z + beta p on the free nodes
__global__ void __launch_bounds__(CG_T) k_pcg_direction(Box b, CGView v, const double* z) {
  let_next_start();
  after_previous();
  const double beta = v.sc[3];
  const unsigned n = blockIdx.x * CG_T + threadIdx.x;
  if (n < (unsigned)b.N && !is_zero(v.dinv[n])) v.p[n] = z[n] + beta * v.p[n];
}

// the multigrid levels of a box (one: the diagonal is the preconditioner): the
// edges of each, and the halving towards the next.  A rod, whose one long edge would
// be halved alone level after level, keeps the diagonal from 64 nodes on, or when
// another edge is 1: the coupling across it comes to outweigh the one along it, and
// the point sweeps no longer damp what the coarse level cannot hold (ms to 1e-10,
// diagonal and V-cycle, without fixed nodes: 1 x 1 x 100 1.3, 3.0; 7 x 7 x 64 2.2,
// 2.5; 7 x 7 x 32 1.5, 1.4; 6 x 6 x 64 2.2, 1.9; 9 x 9 x 64 2.5, 1.9).
int mg_levels(int nx, int ny, int nz, int (*dims)[6]) {
  int L = 0;
  int d[3] = {nx, ny, nz};
  while (L < MG_MAXLEV) {
    bool more = false;
    for (int k = 0; k < 3; ++k) {
      dims[L][k] = d[k];
      dims[L][3 + k] = d[k] >= 8 ? 2 : 1;
      more |= d[k] >= 8;
    }
    ++L;
    if (!more) break;
    for (int k = 0; k < 3; ++k) d[k] = d[k] >= 8 ? (d[k] + 1) / 2 : d[k];
  }
  const int longest = std::max(nx, std::max(ny, nz)), shortest = std::min(nx, std::min(ny, nz));
  if ((nx >= 8) + (ny >= 8) + (nz >= 8) == 1 && (longest >= 64 || shortest == 1)) return 1;
  const int* c = dims[L - 1];
  return c[0] * c[1] * c[2] <= MG_COARSE_MAX ? L : 1;
}

// the CG arrays, then the preconditioner's: z, the fine level's Jacobi buffer
// and diagonal, and each coarser level's faces, diagonal and its inverse, x,
// Jacobi buffer and right-hand side (8 values per node)
size_t full_layout(int nx, int ny, int nz, CGView* v, void* base, MGLevel* lev, int* nlev) {
  const long long N = (long long)nx * ny * nz;
  size_t off = cg_layout(N, v, base);
  auto take = [&](size_t count) {
    off = (off + 255) & ~(size_t)255;
    double* p = base ? (double*)((char*)base + off) : nullptr;
    off += count * sizeof(double);
    return p;
  };
  int dims[MG_MAXLEV][6];
  const int L = mg_levels(nx, ny, nz, dims);
  if (nlev) *nlev = L;
  for (int l = 0; l < L; ++l) {
    const int* d = dims[l];
    const int n = d[0] * d[1] * d[2];
    MGLevel g{d[0], d[1], d[2], n, !((d[0] | d[1] | d[2]) & 1), d[3], d[4], d[5],
              nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
    if (l > 0) {
      g.cf = take(3 * (size_t)n);
      g.dinv = take((size_t)n);
    } else if (v) {
      g.cf = v->cf;
      g.dinv = v->dinv;
    }
    g.D = take((size_t)n);
    g.x = take((size_t)n);
    g.xt = take((size_t)n);
    if (l > 0) g.b = take((size_t)n);
    else if (v) g.b = v->r;
    if (lev) lev[l] = g;
  }
  return off;
}

unsigned nblocks(int n) { return ((unsigned)n + CG_T - 1) / CG_T; }

// the small launch's configuration for a cluster of n CTAs
struct SmallLaunch {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  SmallLaunch(int n, cudaStream_t s, bool early) {
    cfg.gridDim = dim3(n);
    cfg.blockDim = dim3(MG_SMALL_T);
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = n;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = early ? 2 : 1;
  }
};

std::atomic<int> g_cluster_limit{0};  // ek_debug_cluster_limit

// CTAs of the small launch: the largest cluster that the device can place
cudaError_t small_ctas(cudaStream_t s, int& n) {
  cudaError_t e = cudaFuncSetAttribute(k_mg_small, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  const int limit = g_cluster_limit.load();
  for (n = MG_SMALL_CTAS; n > 1; n /= 2) {
    if (limit > 0 && n > limit) continue;
    SmallLaunch c(n, s, false);
    int fit = 0;
    if (cudaOccupancyMaxActiveClusters(&fit, k_mg_small, &c.cfg) == cudaSuccess && fit > 0) break;
    cudaGetLastError();
  }
  return cudaSuccess;
}

cudaError_t launch_small(const MGLevel* lev, int L, int ctas, cudaStream_t s) {
  MGSmall S;
  S.n = L;
  std::copy(lev, lev + L, S.lev);
  const SmallLaunch c(ctas, s, early_launch(s));
  return cudaLaunchKernelEx(&c.cfg, k_mg_small, S);
}

// z = M r: one V-cycle over the levels, then r.z and beta.  The first half
// sweep of a red-black level has been made where its right-hand side was.  The
// fine level is never in the small launch: its last sweep forms r.z.
cudaError_t vcycle(const MGLevel* lev, int L, int ctas, const CGView& v, int first, cudaStream_t s) {
  int small = 1;
  while (small < L - 1 && lev[small].n > MG_SMALL) ++small;
  for (int l = 0; l < small; ++l) {
    const MGLevel& A = lev[l];
    if (A.rb) {
      launch_next(k_mg_half, nblocks(A.n / 2), CG_T, 0, s, A, 1);
      launch_next(k_mg_half, nblocks(A.n / 2), CG_T, 0, s, A, 0);
      launch_next(k_mg_half, nblocks(A.n / 2), CG_T, 0, s, A, 1);
    } else {
      launch_next(k_mg_jacobi, nblocks(A.n), CG_T, 0, s, A, nullptr, A.xt);
      launch_next(k_mg_jacobi, nblocks(A.n), CG_T, 0, s, A, A.xt, A.x);
    }
    launch_next(k_mg_restrict, nblocks(lev[l + 1].n), CG_T, 0, s, A, lev[l + 1]);
  }
  const cudaError_t e = launch_small(lev + small, L - small, ctas, s);
  if (e != cudaSuccess) return e;
  for (int l = small - 1; l >= 0; --l) {
    const MGLevel& A = lev[l];
    const unsigned nb = std::min<unsigned>(CG_BLOCKS, nblocks(A.rb ? A.n / 2 : A.n));
    launch_next(k_mg_prolong, nblocks(A.rb ? A.n / 2 : A.n), CG_T, 0, s, A, lev[l + 1]);
    if (A.rb) {
      launch_next(k_mg_half, nblocks(A.n / 2), CG_T, 0, s, A, 1);
      launch_next(k_mg_half, nblocks(A.n / 2), CG_T, 0, s, A, 0);
      launch_next(k_mg_half, nblocks(A.n / 2), CG_T, 0, s, A, 1);
      if (l > 0) launch_next(k_mg_half, nblocks(A.n / 2), CG_T, 0, s, A, 0);
      else launch_next(k_mg_half_dot, nb, CG_T, 0, s, A, v, first);
    } else {
      launch_next(k_mg_jacobi, nblocks(A.n), CG_T, 0, s, A, A.x, A.xt);
      if (l > 0) launch_next(k_mg_jacobi, nblocks(A.n), CG_T, 0, s, A, A.xt, A.x);
      else launch_next(k_mg_jacobi_dot, nb, CG_T, 0, s, A, A.xt, A.x, v, first);
    }
  }
  return cudaGetLastError();
}

}  // namespace

void poisson_cg_cluster_limit(int n) { g_cluster_limit.store(n > 0 ? n : 0); }

size_t poisson_cg_scratch_bytes(int nx, int ny, int nz) {
  return full_layout(nx, ny, nz, nullptr, nullptr, nullptr, nullptr);
}

cudaError_t poisson_solve_cg(const double* q, const double* eps, const unsigned char* fixed,
                             const double* phi_fixed, double* phi, int nx, int ny, int nz, double bjerrum,
                             double tol, int max_iter, void* scratch, cudaStream_t s, int* iters,
                             double* residual, bool* bad_eps) {
  const Box b{nx, ny, nz, (long long)nx * ny * nz};
  CGView v;
  MGLevel lev[MG_MAXLEV];
  int nlev = 1;
  full_layout(nx, ny, nz, &v, scratch, lev, &nlev);
  const bool mg = nlev >= 2;
  int ctas = 1;  // of the cycle's small launch
  const int nb = (int)std::min<long long>(CG_BLOCKS, (b.N + CG_T - 1) / CG_T);
  const int tx = (nx + 31) / 32, ty = (ny + 7) / 8;
  const int na = (int)std::min<long long>(CG_BLOCKS, (long long)tx * ty * nz);  // operator blocks
  double h[16];
  *bad_eps = false;
  cudaError_t e = cudaMemsetAsync(v.sc, 0, 16 * sizeof(double), s);
  if (e == cudaSuccess && mg) e = small_ctas(s, ctas);
  if (e != cudaSuccess) return e;
  k_cg_faces<<<nb, CG_T, 0, s>>>(b, v, q, eps, fixed);
  // the invalid permittivities are counted before phi is written
  if (eps) {
    e = cudaMemcpyAsync(h, v.sc, 16 * sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    if (h[8] != 0.0) {
      *bad_eps = true;
      return cudaSuccess;
    }
  }
  k_cg_prep<<<nb, CG_T, 0, s>>>(b, v, lev[0].D, q, fixed, phi_fixed, phi, 4.0 * M_PI * bjerrum);
  e = cudaMemcpyAsync(h, v.sc, 16 * sizeof(double), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return e;
  const int neutral = h[7] == 0.0 ? 1 : 0;  // no fixed node: the mean charge was removed
  const double bnorm = sqrt(h[5]);
  int it = 0;
  double rel = 0.0;
  auto iterate = [&]() {
    launch_next(k_cg_apply, na, CG_T, 0, s, b, v, tx, ty);
    if (!mg) {
      launch_next(k_cg_update, nb, CG_T, 0, s, b, v, phi, neutral);
      launch_next(k_cg_direction, nblocks((int)b.N), CG_T, 0, s, b, v, neutral);
      return;
    }
    launch_next(k_pcg_update, nb, CG_T, 0, s, b, v, phi, lev[0], neutral);
    if (neutral) launch_next(k_pcg_project, nb, CG_T, 0, s, b, v, lev[0], 1);
    const cudaError_t ve = vcycle(lev, nlev, ctas, v, 0, s);
    if (e == cudaSuccess) e = ve;
    launch_next(k_pcg_direction, nblocks((int)b.N), CG_T, 0, s, b, v, lev[0].x);
  };
  if (mg && bnorm > 0.0) {
    // the coarse levels' operators, then p = z = M r and r.z
    for (int l = 1; l < nlev; ++l) {
      launch_next(k_mg_coarsen, nblocks(lev[l].n), CG_T, 0, s, lev[l - 1], lev[l]);
      launch_next(k_mg_diag, nblocks(lev[l].n), CG_T, 0, s, lev[l]);
    }
    if (lev[0].rb) launch_next(k_pcg_project, nb, CG_T, 0, s, b, v, lev[0], 0);
    e = vcycle(lev, nlev, ctas, v, 1, s);
    if (e != cudaSuccess) return e;
    launch_next(k_pcg_direction, nblocks((int)b.N), CG_T, 0, s, b, v, lev[0].x);
  }
  // the iterations between two residual reads as one graph (a caller stream
  // other than the legacy default stream can be captured); else the launches
  // one by one
  const int check = mg ? PCG_CHECK : CG_CHECK;
  cudaGraphExec_t graph = nullptr;
  if (s != nullptr && bnorm > 0.0 && max_iter >= check) {
    cudaGraph_t g = nullptr;
    if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
      for (int k = 0; k < check; ++k) iterate();
      if (cudaStreamEndCapture(s, &g) == cudaSuccess && g && e == cudaSuccess) {
        if (cudaGraphInstantiate(&graph, g, 0) != cudaSuccess) graph = nullptr;
      }
      if (g) cudaGraphDestroy(g);
    }
    cudaGetLastError();  // a failed capture leaves the launches one by one
    e = cudaSuccess;
  }
  if (bnorm > 0.0) {
    rel = 1.0;
    while (it < max_iter && rel > tol) {
      const int batch = std::min(check, max_iter - it);
      if (batch == check && graph) {
        e = cudaGraphLaunch(graph, s);
        if (e != cudaSuccess) break;
      } else {
        for (int k = 0; k < batch; ++k) iterate();
        if (e != cudaSuccess) break;
      }
      it += batch;
      e = cudaMemcpyAsync(h, v.sc, 16 * sizeof(double), cudaMemcpyDeviceToHost, s);
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
      if (e != cudaSuccess) break;
      rel = sqrt(h[4]) / bnorm;
      if (!(rel == rel)) break;  // not a number: reported to the caller
    }
  }
  if (graph) cudaGraphExecDestroy(graph);
  if (e != cudaSuccess) return e;
  if (neutral) {
    k_cg_sum<<<nb, CG_T, 0, s>>>(b, v, phi);
    k_cg_shift<<<nb, CG_T, 0, s>>>(b, phi, v.sc);
  }
  e = cudaStreamSynchronize(s);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (iters) *iters = it;
  if (residual) *residual = rel;
  return e;
}

}  // namespace ek
