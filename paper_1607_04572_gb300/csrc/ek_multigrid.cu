// Periodic Poisson solve of Eq. 3 by geometric multigrid: the same discrete
// problem the FFT solver of S1 solves (7-point Laplacian, periodic box,
// (6 phi - sum of the 6 neighbours) = 4 pi l_B (q - mean q), mean phi = 0),
// reached by V-cycles instead of a transform.  Levels: the box and its full
// coarsenings by 2 while every coarse edge stays even and >= 8 (coarse n_x a
// multiple of 2 for the real-to-complex transform) and the grid holds
// more than 4096 nodes; on level l the operator is 4^-l (6 phi - sum nb) (the
// same stencil on spacing 2^l).  Per V-cycle and level: two red-black
// Gauss-Seidel sweeps, the residual, full-weighting restriction, the coarser
// cycle, trilinear prolongation of the correction, two sweeps; the coarsest
// level is solved exactly by the FFT solver.  On the finest level the sweeps
// before the next cycle's residual follow the prolongation, so that one
// residual serves the convergence test and the restriction.  Red-black sweeps
// need even edges, which every level above the coarsest has.  All sums run in a
// fixed order.
//
// What bounds it: the FP64 pipe on the finest level, launches below.  So the
// right-hand side is kept as b / (6 c) (a half sweep is 5 additions and one FMA
// a node), residuals are formed on the red nodes only (those of the black ones,
// updated last, are zero to rounding, once that last half sweep divides by 6
// with both parts of 1/6: by the rounded 1/6 alone every black node kept a residual of
// 6 2^-54 phi, of one sign, which the cycles did not see; the residual that is
// returned is taken over all nodes), the restriction weighs the 13 red nodes of its 27, and the
// correction goes to the black nodes only (the red half sweep that follows does
// not read the others).  The coarse levels run while the host waits for the
// residual.  128^3 to 1e-12 (GB300): 13 cycles of 0.51 ms -> 13 of 0.26 ms.  Of
// a cycle (launches one by one, cold L2) the finest level's half sweeps take 8 x
// 15 us (FP64 pipe: 10 us), its residual, restriction and prolongation 41 us,
// 64^3 48 us, 32^3 35 us and the FFT of 16^3 50 us.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "ek_internal.cuh"

namespace ek {
namespace {

constexpr int MG_T = 256;          // threads per CTA of the grid kernels
constexpr int MG_COARSE = 4096;    // a level this small (or not coarsenable) is solved by FFT
constexpr int MG_RED_BLOCKS = 512; // partial sums of a reduction

struct Level {
  int nx, ny, nz;
  long long n;
  double* phi;      // level 0: the caller's output
  double* b;        // right-hand side over 6 4^-l
  double* r;        // residual over 4^-l, red nodes
};

__device__ __forceinline__ int wrap(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

// scalars of a solve on the device
struct Scalars {
  double sum, mean;
  unsigned long long max;  // bits of a maximum of absolute values
  unsigned count;          // finished blocks of a sum
};

// sum of x and its mean over n values: block partial sums (a grid-stride sum
// per thread, then a tree over the block), added in the same way by the last
// block to finish
__device__ __forceinline__ double block_sum(double s) {
  __shared__ double sh[MG_T];
  __syncthreads();
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int w = MG_T / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  return sh[0];
}
__global__ void k_mg_sum(const double* x, long long n, double* part, Scalars* out) {
  __shared__ bool last;
  double s = 0.0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    s += x[i];
  s = block_sum(s);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = s;
    __threadfence();
    last = atomicAdd(&out->count, 1u) == gridDim.x - 1;
    if (last) __threadfence();
  }
  __syncthreads();
  if (!last) return;
  s = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += MG_T) s += part[i];
  s = block_sum(s);
  if (threadIdx.x == 0) {
    out->sum = s;
    out->mean = s / (double)n;
    out->count = 0u;
  }
}

// 1/6 as a sum of two doubles
constexpr double SIXTH = 1.0 / 6.0, SIXTH_LO = 0x1.5555555555555p-57;

// the bits of |v| (they order as the values do); 0 for a NaN
__device__ __forceinline__ unsigned long long abs_bits(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffULL;
  return b > 0x7ff0000000000000ULL ? 0ULL : b;
}
// maximum over the grid (it does not depend on the order, and costs no FP64
// instruction)
__device__ __forceinline__ void grid_max(unsigned long long m, Scalars* out) {
  __shared__ unsigned long long sh[MG_T / 32];
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_down_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < MG_T / 32; ++w) m = max(m, sh[w]);
    atomicMax(&out->max, m);
  }
}

// node j of a colour (colour 0, red: x + y + z even; n_x even: half of every row)
__device__ __forceinline__ int colour_node(unsigned j, int nx, int ny, int colour, int& x, int& y, int& z) {
  const unsigned hx = (unsigned)nx / 2u, row = j / hx;
  z = (int)(row / (unsigned)ny);
  y = (int)row - z * ny;
  x = 2 * (int)(j - row * hx) + ((y + z + colour) & 1);
  return x + nx * (int)row;
}

// sum of the six neighbours of node i = (x, y, z) (32-bit indices: N < 2^31)
__device__ __forceinline__ double nb_sum(const double* phi, int i, int x, int y, int z, int nx,
                                         int ny, int nz) {
  const int sy = nx, sz = nx * ny;
  return ((phi[i - x + wrap(x - 1, nx)] + phi[i - x + wrap(x + 1, nx)]) +
          (phi[i + (wrap(y - 1, ny) - y) * sy] + phi[i + (wrap(y + 1, ny) - y) * sy])) +
         (phi[i + (wrap(z - 1, nz) - z) * sz] + phi[i + (wrap(z + 1, nz) - z) * sz]);
}

// b = s (q - mean q) / 6, and the first red half sweep from zero: phi = b on
// the red nodes, 0 on the black ones; the maximum of |6 b|
__global__ void __launch_bounds__(MG_T) k_mg_rhs(const double* q, double* phi, double* b, int nx, int ny, int nz,
                                                 double s, Scalars* sc) {
  const unsigned i = blockIdx.x * MG_T + threadIdx.x;
  unsigned long long m = 0;
  if (i < (unsigned)nx * (unsigned)ny * (unsigned)nz) {
    const unsigned row = i / (unsigned)nx;
    const int x = (int)(i - row * (unsigned)nx), y = (int)(row % (unsigned)ny), z = (int)(row / (unsigned)ny);
    const double v = s * (q[i] - sc->mean);  // read before phi, which may alias q, is written
    const double v6 = fma(v, SIXTH, v * SIXTH_LO);
    b[i] = v6;
    phi[i] = ((x + y + z) & 1) ? 0.0 : v6;
    m = abs_bits(v);
  }
  grid_max(m, sc);
}

// one colour of a red-black Gauss-Seidel sweep: phi = sum nb / 6 + b (FULL: both
// parts of 1/6)
template <bool FULL>
__global__ void __launch_bounds__(MG_T) k_mg_half(double* phi, const double* b, int nx, int ny, int nz, int colour) {
  let_next_start();
  after_previous();
  const unsigned j = blockIdx.x * MG_T + threadIdx.x;
  if (j >= (unsigned)nx / 2u * (unsigned)ny * (unsigned)nz) return;
  int x, y, z;
  const int i = colour_node(j, nx, ny, colour, x, y, z);
  const double s = nb_sum(phi, i, x, y, z, nx, ny, nz);
  phi[i] = fma(s, SIXTH, FULL ? fma(s, SIXTH_LO, b[i]) : b[i]);
}

// residual over 4^-l on the red nodes, r = sum nb - 6 (phi - b); with MAX the
// maximum of |r|
template <bool MAX>
__global__ void __launch_bounds__(MG_T) k_mg_resid(const double* phi, const double* b, double* r, int nx, int ny,
                                                   int nz, Scalars* sc) {
  let_next_start();
  after_previous();
  const unsigned j = blockIdx.x * MG_T + threadIdx.x;
  unsigned long long m = 0;
  if (j < (unsigned)nx / 2u * (unsigned)ny * (unsigned)nz) {
    int x, y, z;
    const int i = colour_node(j, nx, ny, 0, x, y, z);
    const double v = fma(-6.0, phi[i] - b[i], nb_sum(phi, i, x, y, z, nx, ny, nz));
    r[i] = v;
    if (MAX) m = abs_bits(v);
  }
  if (MAX) grid_max(m, sc);
}
// the maximum of |r| over all nodes
__global__ void __launch_bounds__(MG_T) k_mg_resid_max(const double* phi, const double* b, int nx, int ny, int nz,
                                                       Scalars* sc) {
  const unsigned i = blockIdx.x * MG_T + threadIdx.x;
  unsigned long long m = 0;
  if (i < (unsigned)nx * (unsigned)ny * (unsigned)nz) {
    const unsigned row = i / (unsigned)nx;
    const int x = (int)(i - row * (unsigned)nx), y = (int)(row % (unsigned)ny), z = (int)(row / (unsigned)ny);
    m = abs_bits(fma(-6.0, phi[i] - b[i], nb_sum(phi, (int)i, x, y, z, nx, ny, nz)));
  }
  grid_max(m, sc);
}

// full weighting: coarse node (X, Y, Z) sits on fine node (2X, 2Y, 2Z) and
// takes the weighted mean of the 27 fine residuals around it (weights 1, 1/2,
// 1/4, 1/8 by the number of offset axes; every fine node gives a total weight
// of 1, so the mean is kept), of which the 13 red ones (none or two offset
// axes) are not zero; over 6 4^-(l+1) that is (r_0 + sum r / 4) / 12.  The
// coarse level's first red half sweep from zero comes along.
__global__ void __launch_bounds__(MG_T) k_mg_restrict(const double* rf, int nx, int ny, int nz, double* bc,
                                                      double* phic) {
  let_next_start();
  after_previous();
  const int cx = nx / 2, cy = ny / 2, cz = nz / 2;
  const unsigned i = blockIdx.x * MG_T + threadIdx.x;
  if (i >= (unsigned)cx * (unsigned)cy * (unsigned)cz) return;
  const unsigned row = i / (unsigned)cx;
  const int X = (int)(i - row * (unsigned)cx), Y = (int)(row % (unsigned)cy), Z = (int)(row / (unsigned)cy);
  const int x[3] = {wrap(2 * X - 1, nx), 2 * X, 2 * X + 1};
  const int y[3] = {nx * wrap(2 * Y - 1, ny), nx * (2 * Y), nx * (2 * Y + 1)};
  const int sz = nx * ny, z[3] = {sz * wrap(2 * Z - 1, nz), sz * (2 * Z), sz * (2 * Z + 1)};
  const double a = (rf[x[0] + y[0] + z[1]] + rf[x[2] + y[0] + z[1]]) + (rf[x[0] + y[2] + z[1]] + rf[x[2] + y[2] + z[1]]);
  const double b = (rf[x[0] + y[1] + z[0]] + rf[x[2] + y[1] + z[0]]) + (rf[x[0] + y[1] + z[2]] + rf[x[2] + y[1] + z[2]]);
  const double c = (rf[x[1] + y[0] + z[0]] + rf[x[1] + y[2] + z[0]]) + (rf[x[1] + y[0] + z[2]] + rf[x[1] + y[2] + z[2]]);
  const double v = fma(0.25, (a + b) + c, rf[x[1] + y[1] + z[1]]) * (1.0 / 12.0);
  bc[i] = v;
  if (!((X + Y + Z) & 1)) phic[i] = v;
}

// trilinear prolongation of the coarse correction, added to the black nodes of
// the fine phi: per axis an even fine index lies on coarse node x / 2, an odd
// one half way between (x - 1) / 2 and (x + 1) / 2 (periodic); a black node has
// one odd axis or three
__global__ void __launch_bounds__(MG_T) k_mg_prolong(const double* phic, int nx, int ny, int nz, double* phif) {
  let_next_start();
  after_previous();
  const int cx = nx / 2, cy = ny / 2, cz = nz / 2;
  const unsigned j = blockIdx.x * MG_T + threadIdx.x;
  if (j >= (unsigned)nx / 2u * (unsigned)ny * (unsigned)nz) return;
  int x, y, z;
  const int i = colour_node(j, nx, ny, 1, x, y, z);
  const int x0 = x >> 1, y0 = (y >> 1) * cx, z0 = (z >> 1) * cx * cy;
  const int x1 = wrap(x0 + 1, cx), y1 = wrap((y >> 1) + 1, cy) * cx, z1 = wrap((z >> 1) + 1, cz) * cx * cy;
  const double a = phic[x0 + y0 + z0];
  if (y & z & 1) {
    const double s = ((a + phic[x1 + y0 + z0]) + (phic[x0 + y1 + z0] + phic[x1 + y1 + z0])) +
                     ((phic[x0 + y0 + z1] + phic[x1 + y0 + z1]) + (phic[x0 + y1 + z1] + phic[x1 + y1 + z1]));
    phif[i] = fma(0.125, s, phif[i]);
  } else {
    const double o = phic[(x & 1) ? x1 + y0 + z0 : (y & 1) ? x0 + y1 + z0 : x0 + y0 + z1];
    phif[i] = fma(0.5, a + o, phif[i]);
  }
}

// phi -= its mean
__global__ void __launch_bounds__(MG_T) k_sub_mean(double* phi, long long n, const Scalars* sc) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  phi[i] -= sc->mean;
}

unsigned blocks(long long n) { return (unsigned)((n + MG_T - 1) / MG_T); }

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

// the levels of a box: itself, then full coarsenings while every coarse edge
// stays >= 8 and even where it must be (n_x / 2 even for the coarse FFT), as
// long as the level holds more than MG_COARSE nodes
std::vector<Level> make_levels(int nx, int ny, int nz) {
  std::vector<Level> lv;
  Level l{nx, ny, nz, (long long)nx * ny * nz, nullptr, nullptr, nullptr};
  lv.push_back(l);
  while (l.n > MG_COARSE && l.nx % 4 == 0 && l.ny % 2 == 0 && l.nz % 2 == 0 && l.nx >= 16 &&
         l.ny >= 16 && l.nz >= 16) {
    l.nx /= 2;
    l.ny /= 2;
    l.nz /= 2;
    l.n = (long long)l.nx * l.ny * l.nz;
    lv.push_back(l);
  }
  return lv;
}

// scratch: b and r of level 0; phi, b, r of every coarser level; the
// coarsest level's spectrum; reduction slots
struct Layout {
  size_t b0, r0, coarse, spectrum, red, total;
};

Layout layout(const std::vector<Level>& lv) {
  Layout L;
  size_t off = 0;
  L.b0 = off;
  off += align256(lv[0].n * sizeof(double));
  L.r0 = off;
  off += align256(lv[0].n * sizeof(double));
  L.coarse = off;
  for (size_t k = 1; k < lv.size(); ++k) off += 3 * align256(lv[k].n * sizeof(double));
  L.spectrum = off;
  const Level& c = lv.back();
  off += align256(poisson_spectrum_bytes(c.nx, c.ny, c.nz));
  L.red = off;
  off += align256((MG_RED_BLOCKS + 4) * sizeof(double));
  L.total = off;
  return L;
}

struct Solver {
  std::vector<Level> lv;
  PoissonPlan coarse_plan;
  double2* spectrum;
  double* part;   // MG_RED_BLOCKS partial sums
  Scalars* sc;
  cudaStream_t s;
};

cudaError_t mean_of(const Solver& S, const double* x, long long n) {
  const int nb = (int)std::min<long long>(MG_RED_BLOCKS, (n + MG_T - 1) / MG_T);
  k_mg_sum<<<nb, MG_T, 0, S.s>>>(x, n, S.part, S.sc);
  return cudaGetLastError();
}

void half(const Solver& S, const Level& l, int colour, bool full = false) {
  launch_next(full ? k_mg_half<true> : k_mg_half<false>, blocks(l.n / 2), MG_T, 0, S.s, l.phi, l.b, l.nx, l.ny, l.nz,
              colour);
}
void restrict_to(const Solver& S, const Level& l, const Level& c) {
  launch_next(k_mg_restrict, blocks(c.n), MG_T, 0, S.s, l.r, l.nx, l.ny, l.nz, c.b, c.phi);
}
void prolong_to(const Solver& S, const Level& l, const Level& c) {
  launch_next(k_mg_prolong, blocks(l.n / 2), MG_T, 0, S.s, c.phi, l.nx, l.ny, l.nz, l.phi);
}

// one V-cycle from level k >= 1 down, from zero; the red nodes have had their
// first half sweep
cudaError_t vcycle(const Solver& S, size_t k) {
  const Level& l = S.lv[k];
  if (k + 1 == S.lv.size()) {
    // exact on the coarsest level: 6 phi - sum nb = 6 b is the FFT solver's
    // problem with 4 pi l_B = 6
    Phys ph;
    memset(&ph, 0, sizeof(ph));
    ph.bjerrum = 6.0 / (4.0 * M_PI);
    return poisson_solve(S.coarse_plan, l.b, nullptr, nullptr, nullptr, ph, l.phi, S.spectrum, S.s);
  }
  half(S, l, 1);
  half(S, l, 0);
  half(S, l, 1);
  launch_next(k_mg_resid<false>, blocks(l.n / 2), MG_T, 0, S.s, l.phi, l.b, l.r, l.nx, l.ny, l.nz, S.sc);
  restrict_to(S, l, S.lv[k + 1]);
  cudaError_t e = vcycle(S, k + 1);
  if (e != cudaSuccess) return e;
  prolong_to(S, l, S.lv[k + 1]);
  for (int sweep = 0; sweep < 2; ++sweep) {
    half(S, l, 0);
    half(S, l, 1);
  }
  return cudaGetLastError();
}

// the device's maximum, read on a stream of its own once `ready` has passed,
// while the solve's stream goes on
struct Reader {
  cudaStream_t s = nullptr;
  cudaEvent_t ready = nullptr;
  cudaError_t open() {
    cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    return e != cudaSuccess ? e : cudaEventCreateWithFlags(&ready, cudaEventDisableTiming);
  }
  ~Reader() {
    if (ready) cudaEventDestroy(ready);
    if (s) cudaStreamDestroy(s);
  }
  cudaError_t mark(cudaStream_t from) { return cudaEventRecord(ready, from); }
  cudaError_t read(const Scalars* sc, double& v) {
    unsigned long long bits = 0;
    cudaError_t e = cudaStreamWaitEvent(s, ready, 0);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&bits, &sc->max, sizeof(bits), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    memcpy(&v, &bits, sizeof(v));
    return e;
  }
};

}  // namespace

size_t poisson_mg_scratch_bytes(int nx, int ny, int nz) { return layout(make_levels(nx, ny, nz)).total; }

cudaError_t poisson_solve_mg(const PoissonPlan& coarse_plan, const double* q, double* phi, int nx,
                             int ny, int nz, double bjerrum, double tol, int max_cycles,
                             void* scratch, cudaStream_t s, int* cycles, double* residual) {
  Solver S;
  S.lv = make_levels(nx, ny, nz);
  const Layout L = layout(S.lv);
  unsigned char* base = static_cast<unsigned char*>(scratch);
  S.lv[0].phi = phi;
  S.lv[0].b = reinterpret_cast<double*>(base + L.b0);
  S.lv[0].r = reinterpret_cast<double*>(base + L.r0);
  size_t off = L.coarse;
  for (size_t k = 1; k < S.lv.size(); ++k) {
    const size_t sz = align256(S.lv[k].n * sizeof(double));
    S.lv[k].phi = reinterpret_cast<double*>(base + off);
    S.lv[k].b = reinterpret_cast<double*>(base + off + sz);
    S.lv[k].r = reinterpret_cast<double*>(base + off + 2 * sz);
    off += 3 * sz;
  }
  S.coarse_plan = coarse_plan;
  S.spectrum = reinterpret_cast<double2*>(base + L.spectrum);
  S.part = reinterpret_cast<double*>(base + L.red);
  S.sc = reinterpret_cast<Scalars*>(S.part + MG_RED_BLOCKS);
  S.s = s;
  Reader rd;
  cudaError_t e = rd.open();
  if (e != cudaSuccess) return e;
  const Level& f = S.lv[0];
  auto clear_max = [&]() { return cudaMemsetAsync(&S.sc->max, 0, sizeof(S.sc->max), s); };
  // the maximum so far, as soon as the kernels launched until now have run
  auto read_max = [&](double& v) -> cudaError_t {
    cudaError_t r = cudaGetLastError();
    if (r == cudaSuccess) r = rd.mark(s);
    return r != cudaSuccess ? r : rd.read(S.sc, v);
  };
  e = cudaMemsetAsync(S.sc, 0, sizeof(Scalars), s);
  // b = 4 pi l_B (q - mean q)
  if (e == cudaSuccess) e = mean_of(S, q, f.n);
  if (e != cudaSuccess) return e;
  k_mg_rhs<<<blocks(f.n), MG_T, 0, s>>>(q, phi, f.b, f.nx, f.ny, f.nz, 4.0 * M_PI * bjerrum, S.sc);
  double bmax = 0.0, rmax = 0.0;
  e = read_max(bmax);
  if (e != cudaSuccess) return e;
  int done = 0;
  if (S.lv.size() == 1 && bmax > 0.0) {
    // a box that cannot be coarsened: one FFT solve of the whole problem.  (Another
    // of the same right-hand side would give the same again, whatever the tolerance.)
    Phys ph;
    memset(&ph, 0, sizeof(ph));
    ph.bjerrum = 6.0 / (4.0 * M_PI);
    e = poisson_solve(S.coarse_plan, f.b, nullptr, nullptr, nullptr, ph, phi, S.spectrum, s);
    if (e == cudaSuccess) e = clear_max();
    if (e != cudaSuccess) return e;
    done = 1;
    k_mg_resid_max<<<blocks(f.n), MG_T, 0, s>>>(f.phi, f.b, f.nx, f.ny, f.nz, S.sc);
    e = read_max(rmax);
    if (e != cudaSuccess) return e;
  } else if (bmax > 0.0) {
    half(S, f, 1, true);  // the first sweep's black half
    for (;;) {
      e = clear_max();
      if (e != cudaSuccess) return e;
      k_mg_resid<true><<<blocks(f.n / 2), MG_T, 0, s>>>(f.phi, f.b, f.r, f.nx, f.ny, f.nz, S.sc);
      e = rd.mark(s);
      // the coarse correction does not touch phi: it runs while the host waits
      // for the residual (and for nothing when that has converged)
      const bool more = done < max_cycles;
      if (e == cudaSuccess && more) {
        restrict_to(S, f, S.lv[1]);
        e = vcycle(S, 1);
      }
      if (e == cudaSuccess && done > 0) e = rd.read(S.sc, rmax);
      if (e != cudaSuccess) return e;
      if (done > 0 && (!more || rmax <= tol * bmax)) {
        // the red nodes have converged (or no cycle is left): over all nodes
        e = clear_max();
        if (e != cudaSuccess) return e;
        k_mg_resid_max<<<blocks(f.n), MG_T, 0, s>>>(f.phi, f.b, f.nx, f.ny, f.nz, S.sc);
        e = read_max(rmax);
        if (e != cudaSuccess) return e;
        if (!more || rmax <= tol * bmax) break;
      }
      prolong_to(S, f, S.lv[1]);
      for (int sweep = 0; sweep < 4; ++sweep) {
        half(S, f, 0);
        half(S, f, 1, sweep == 3);
      }
      ++done;
    }
  }
  // the zero-mean solution (the periodic problem fixes phi up to a constant)
  if (bmax == 0.0) {
    e = cudaMemsetAsync(phi, 0, f.n * sizeof(double), s);
    if (e != cudaSuccess) return e;
  }
  e = mean_of(S, phi, f.n);
  if (e != cudaSuccess) return e;
  k_sub_mean<<<blocks(f.n), MG_T, 0, s>>>(phi, f.n, S.sc);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (cycles) *cycles = done;
  if (residual) *residual = bmax > 0.0 ? rmax / bmax : 0.0;
  return e;
}

int poisson_mg_levels(int nx, int ny, int nz, int coarse[3]) {
  const std::vector<Level> lv = make_levels(nx, ny, nz);
  coarse[0] = lv.back().nx;
  coarse[1] = lv.back().ny;
  coarse[2] = lv.back().nz;
  return (int)lv.size();
}

}  // namespace ek
