// S2 (Capuani link fluxes + coupling force fused with the TRT/BGK collision,
// Guo force term and push streaming with velocity bounce-back) and S3 (species
// update: flux divergence + volume-of-fluid advection), FP64 form.
//
// Node index x + nx*(y + ny*z).  Populations and species are
// structure-of-arrays (direction- / species-major), so every load and store of
// a warp touches consecutive x: coalesced 8-byte accesses.
#include <math.h>

#include <algorithm>

#include "ek_internal.cuh"

namespace ek {

namespace {

__device__ __forceinline__ long long nbr_index(int d, int x, int y, int z, const Nbr& b,
                                               int nx, int ny) {
  const int X = dcx(d) > 0 ? b.xp : (dcx(d) < 0 ? b.xm : x);
  const int Y = dcy(d) > 0 ? b.yp : (dcy(d) < 0 ? b.ym : y);
  const int Z = dcz(d) > 0 ? b.zp : (dcz(d) < 0 ? b.zm : z);
  return (long long)X + (long long)nx * ((long long)Y + (long long)ny * Z);
}

// Boundary velocity v_b = v + omega x (r_b - r) of particle p at wrapped node
// (xb, yb, zb) (Eq. 10).  The node is unwrapped into the particle's box
// [lo, lo + n) so that r_b - r is never taken across the periodic seam.
__device__ __forceinline__ void boundary_velocity(const DevParticle& P, int xb, int yb, int zb,
                                                  const Grid& g, double vb[3]) {
  const double X = (double)(P.lo[0] + wrapi(xb - P.lo[0], g.nx));
  const double Y = (double)(P.lo[1] + wrapi(yb - P.lo[1], g.ny));
  const double Z = (double)(P.lo[2] + wrapi(zb - P.lo[2], g.nz));
  const double dx = X - P.pos[0], dy = Y - P.pos[1], dz = Z - P.pos[2];
  vb[0] = P.vel[0] + (P.omega[1] * dz - P.omega[2] * dy);
  vb[1] = P.vel[1] + (P.omega[2] * dx - P.omega[0] * dz);
  vb[2] = P.vel[2] + (P.omega[0] * dy - P.omega[1] * dx);
}

// ---------------------------------------------------------------------------
// S2, FP64 form: 32 x 8 tiles marching through a segment of planes.
//
// The kernel is bound by the FP64 pipe (2 lanes per clock per SM), so it is
// laid out to spend as few FP64 instructions per node as it can; loads, integer
// work and shared memory are free beside them.  Each link flux is computed
// once, by the end whose link points up in z (or, in the plane, along (1,0),
// (0,1), (1,1), (1,-1)): the values of the nine links go to shared memory, from
// where the other end takes them with the opposite sign: what leaves one node
// enters the other up to the rounding of the sums.
// Where no node of the three planes is a boundary or partly covered (SIMPLE)
// the partial-volume factors drop out.  The collision is a pair form
// (lb64_collide).
//
// One thread per node with all 18 links evaluated at both ends took 900 FP64
// instructions per node, the pipe 87% busy: 3.30 ms at 128^3, 0.433 ms at 64^3.
// This form takes 350: 1.49 and 0.243 ms, the pipe 84% busy at 128^3 (barriers and
// the latency of the FP64 chains between them are the rest).
// ---------------------------------------------------------------------------
constexpr int HX = TILE_X + 2, HY = TILE_Y + 2, HP = HX * HY, TN = TILE_X * TILE_Y;

// the nine links a node computes: in the plane 1, 3, 7, 9; up 5, 11, 14, 15, 18
constexpr int NLINK = 9, NFLAT = 4;
__host__ __device__ constexpr int link_dir(int l) {
  return l == 0 ? 1 : l == 1 ? 3 : l == 2 ? 7 : l == 3 ? 9 : l == 4 ? 5 : l == 5 ? 11 : l == 6 ? 14 : l == 7 ? 15 : 18;
}
__host__ __device__ constexpr int link_off(int l) { return dcx(link_dir(l)) + HX * dcy(link_dir(l)); }

// constants of the collision, rounded once on the host
struct Coll64 {
  double hp, hm;    // (1 + lambda_e)/2, (1 + lambda_o)/2
  double gw, kw;    // 9/2 (2 + lambda_e)/36, -9/2 lambda_e/36
  double lo12;      // -lambda_o/12
  double g15, le1;  // -3/2 (2 + lambda_e), 1 + lambda_e
};

template <int K>
struct LB64Smem {
  static constexpr int NV = K >= 2 ? K + 1 : 1;  // values of a link: per species, and their sum
  double phi[3][HP], om[3][HP], rho[K > 0 ? K : 1][3][HP];  // plane p in slot p mod 3; om: 1 - Psi, rho: rho/om
  double link[K > 0 ? NLINK : 1][NV][HP];  // of the node at the halo-tile index
  int own[4][HP];                          // plane p in slot p & 3
};

__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}
// periodic coordinate of a tile-halo position v in [-1, n + 33): exact for
// every position a node of the box uses (at most n), inside the box for all
__device__ __forceinline__ int halo_wrap(int v, int n) {
  v = v < 0 ? v + n : (v >= n ? v - n : v);
  return min(v, n - 1);
}
__device__ __forceinline__ int wrap_plane(int z, int n) { return z < 0 ? z + n : (z >= n ? z - n : z); }
// not an infinity or a NaN, from the exponent bits (no FP64 instruction)
__device__ __forceinline__ bool finite_bits(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }
// sign code of v from its bits
__device__ __forceinline__ unsigned sign_bits(double v) {
  const long long b = __double_as_longlong(v);
  return (b << 1) == 0 ? 0u : (b < 0 ? 2u : 1u);
}

// one link from node e of plane slot s0 to node f of plane slot s1 (weight w:
// 1 on faces, 1/sqrt 2 on edges), Eq. 20 in units of D_k / A_0:
// s [(a - b) + z/2 (a + b) dPhi], a and b the densities over their 1 - Psi,
// s = (1 - Psi)(1 - Psi') w; 0 when one end is a boundary node
template <int K, bool SIMPLE, bool PV, bool UNIT>
__device__ __forceinline__ void link_flux(const LB64Smem<K>& t, const Phys& ph, int s0, int e, int s1, int f, double w,
                                          double ec, bool open, double (&T)[K > 0 ? K : 1], double& tsum) {
  const double dphi = (t.phi[s0][e] - t.phi[s1][f]) + ec;
  double sl = w;
  if (!SIMPLE && PV) sl = (t.om[s0][e] * t.om[s1][f]) * w;
  tsum = 0.0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const double ra = t.rho[k][s0][e], rb = t.rho[k][s1][f];
    double br = fma(ra + rb, ph.hz[k] * dphi, ra - rb);
    if (!UNIT || (!SIMPLE && PV)) br *= sl;
    if (!SIMPLE) br = open ? br : 0.0;
    T[k] = br;
    tsum = k == 0 ? br : tsum + br;
  }
}
template <int K>
__device__ __forceinline__ void link_put(LB64Smem<K>& t, int l, int e, const double (&T)[K > 0 ? K : 1], double tsum) {
#pragma unroll
  for (int k = 0; k < K; ++k) t.link[l][k][e] = T[k];
  if (K >= 2) t.link[l][LB64Smem<K>::NV - 1][e] = tsum;
}

// the links L0 .. L1 - 1 of the thread's node e0 (slots s0, s1: its plane and
// the next; o0, o1 their node classes), added to S and G and published
template <int K, bool SIMPLE, bool PV, int L0, int L1>
__device__ __forceinline__ void own_links(LB64Smem<K>& t, const Phys& ph, int s0, int s1, int o0, int o1, int e0,
                                          double (&S)[K > 0 ? K : 1], double (&G)[3]) {
  const bool here = SIMPLE || t.own[o0][e0] == FLUID;
#pragma unroll
  for (int l = L0; l < L1; ++l) {
    const int d = link_dir(l), f = e0 + link_off(l);
    const bool open = SIMPLE || (here && t.own[l < NFLAT ? o0 : o1][f] == FLUID);
    double T[K > 0 ? K : 1], ts;
    if (d < 7) link_flux<K, SIMPLE, PV, true>(t, ph, s0, e0, l < NFLAT ? s0 : s1, f, 1.0, ph.ec[d], open, T, ts);
    else link_flux<K, SIMPLE, PV, false>(t, ph, s0, e0, l < NFLAT ? s0 : s1, f, 0.70710678118654752, ph.ec[d], open, T, ts);
#pragma unroll
    for (int k = 0; k < K; ++k) S[k] += T[k];
    if (dcx(d)) G[0] += csgn(dcx(d), ts);
    if (dcy(d)) G[1] += csgn(dcy(d), ts);
    if (dcz(d)) G[2] += csgn(dcz(d), ts);
    link_put<K>(t, l, e0, T, ts);
  }
}
// the links L0 .. L1 - 1 that end at the thread's node (published by their
// source): the node's own link value is the negative, along the opposite
// direction, so S falls by it and G takes it with the source's direction
template <int K, int L0, int L1>
__device__ __forceinline__ void other_links(const LB64Smem<K>& t, int e0, double (&S)[K > 0 ? K : 1], double (&G)[3]) {
#pragma unroll
  for (int l = L0; l < L1; ++l) {
    const int d = link_dir(l), f = e0 - link_off(l);
#pragma unroll
    for (int k = 0; k < K; ++k) S[k] -= t.link[l][k][f];
    const double ts = t.link[l][LB64Smem<K>::NV - 1][f];
    if (dcx(d)) G[0] += csgn(dcx(d), ts);
    if (dcy(d)) G[1] += csgn(dcy(d), ts);
    if (dcz(d)) G[2] += csgn(dcz(d), ts);
  }
}

// The links whose source lies in the halo and whose other end in the tile: one
// thread each.  Per link the sources off the tile: a column of HY - 2 rows (at
// the left, for link 14 at the right), and a row (below, for the links with
// c_y < 0 above).  e: source (-1: none), l: link, off: to the other end.
struct HaloLink {
  int e, l, off, d;
};
__device__ __forceinline__ HaloLink halo_link(int tid) {
  HaloLink h{-1, 0, 0, 0};
  int t = tid;
  auto col = [&](int l, int x, int y0) {
    if (t >= 0 && t < TILE_Y) h = HaloLink{x + HX * (y0 + t), l, 0, 0};
    t -= TILE_Y;
  };
  auto row = [&](int l, int y, int n) {
    if (t >= 0 && t < n) h = HaloLink{1 + t + HX * y, l, 0, 0};
    t -= n;
  };
  col(0, 0, 1);                 // (1, 0): left column
  col(2, 0, 0);                 // (1, 1): left column from the corner, then the row below
  col(3, 0, 2);                 // (1, -1): left column to the upper corner, then the row above
  col(5, 0, 1);                 // (1, 0, 1)
  col(6, HX - 1, 1);            // (-1, 0, 1): right column
  row(1, 0, TILE_X);            // (0, 1)
  row(2, 0, TILE_X - 1);
  row(3, HY - 1, TILE_X - 1);
  row(7, 0, TILE_X);            // (0, 1, 1)
  row(8, HY - 1, TILE_X);       // (0, -1, 1)
  const int l = h.l;
  h.off = l == 0 ? link_off(0) : l == 1 ? link_off(1) : l == 2 ? link_off(2) : l == 3 ? link_off(3)
        : l == 5 ? link_off(5) : l == 6 ? link_off(6) : l == 7 ? link_off(7) : link_off(8);
  h.d = l == 0 ? 1 : l == 1 ? 3 : l == 2 ? 7 : l == 3 ? 9 : l == 5 ? 11 : l == 6 ? 14 : l == 7 ? 15 : 18;
  return h;
}
template <int K, bool SIMPLE, bool PV>
__device__ __forceinline__ void halo_links(LB64Smem<K>& t, const Phys& ph, const HaloLink& h, bool flat, int s0, int s1,
                                           int o0, int o1) {
  if (h.e < 0 || (!flat && h.l < NFLAT)) return;
  const int f = h.e + h.off, s = h.l < NFLAT ? s0 : s1;
  const bool open = SIMPLE || (t.own[o0][h.e] == FLUID && t.own[h.l < NFLAT ? o0 : o1][f] == FLUID);
  double T[K > 0 ? K : 1], ts;
  link_flux<K, SIMPLE, PV, false>(t, ph, s0, h.e, s, f, h.d < 7 ? 1.0 : 0.70710678118654752, ph.ec[h.d], open, T, ts);
  link_put<K>(t, h.l, h.e, T, ts);
}

// The collision of one node (Eqs. 8-9), TRT in pair form, in place.  With s, d
// the sum and difference of an opposite pair the two results are A + B and
// A - B, A = (1 + lambda_e)/2 s + Ep, B = (1 + lambda_o)/2 d + Em.  Ep is
// quadratic: with h = w (9/2 (2 + lambda_e) F - 9/2 lambda_e rho u) the edges
// x + y and x - y share b + u_x h_x + u_y h_y and differ in the sign of
// u_x h_y + u_y h_x; a face takes twice the edge weight 1/36.
__device__ __forceinline__ void lb64_collide(double (&f)[Q], const Coll64& c, double lam_e, double Fx, double Fy,
                                             double Fz, double& ux, double& uy, double& uz, double& rho, double& usq) {
  double s[9], d[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    s[i] = f[2 * i + 1] + f[2 * i + 2];
    d[i] = f[2 * i + 1] - f[2 * i + 2];
  }
  rho = f[0] + (((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7]))) + s[8];
  const double jx = d[0] + ((d[3] + d[4]) + (d[5] + d[6]));
  const double jy = d[1] + ((d[3] - d[4]) + (d[7] + d[8]));
  const double jz = d[2] + ((d[5] - d[6]) + (d[7] - d[8]));
  const double irho = 1.0 / rho;
  ux = fma(0.5, Fx, jx) * irho;
  uy = fma(0.5, Fy, jy) * irho;
  uz = fma(0.5, Fz, jz) * irho;
  usq = fma(uz, uz, fma(uy, uy, ux * ux));
  const double uF = fma(uz, Fz, fma(uy, Fy, ux * Fx));
  const double base = fma(c.g15, uF, (-lam_e * rho) * fma(-1.5, usq, 1.0));
  const double bw = base * (1.0 / 36.0), kw = c.kw * rho;
  const double hx = fma(kw, ux, c.gw * Fx), hy = fma(kw, uy, c.gw * Fy), hz = fma(kw, uz, c.gw * Fz);
  const double qx = fma(c.lo12, jx, (1.0 / 12.0) * Fx), qy = fma(c.lo12, jy, (1.0 / 12.0) * Fy),
               qz = fma(c.lo12, jz, (1.0 / 12.0) * Fz);
  const double bx = fma(ux, hx, bw), by = fma(uy, hy, bw), bz = fma(uz, hz, bw);
  const double bxy = fma(uy, hy, bx), bxz = fma(uz, hz, bx), byz = fma(uz, hz, by);
  const double mxy = fma(ux, hy, uy * hx), mxz = fma(ux, hz, uz * hx), myz = fma(uy, hz, uz * hy);
  f[0] = fma(c.le1, f[0], 12.0 * bw);
  const double Ep[9] = {bx + bx, by + by, bz + bz, bxy + mxy, bxy - mxy, bxz + mxz, bxz - mxz, byz + myz, byz - myz};
  const double Em[9] = {qx + qx, qy + qy, qz + qz, qx + qy, qx - qy, qx + qz, qx - qz, qy + qz, qy - qz};
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const double A = fma(c.hp, s[i], Ep[i]), B = fma(c.hm, d[i], Em[i]);
    f[2 * i + 1] = A + B;
    f[2 * i + 2] = A - B;
  }
}

// collision and push stream of the thread's node (plane z) once S and G are
// complete; iv takes the node's internal solute force on the fluid,
// i = f_ext - q_ions E (also stored in ifield)
template <int K, bool SIMPLE>
__device__ __forceinline__ void lb64_node(const LB64Smem<K>& t, const LBArgs& a, const Coll64& c, int x, int y, int z,
                                          int e0, const double (&S)[K > 0 ? K : 1], const double (&G)[3], double (&f)[Q],
                                          double (&iv)[3]) {
  double* f_out = (double*)a.f_out;
  const double* rho_in = (const double*)a.rho_in;
  double* rho_out = (double*)a.rho_out;
  double* u = (double*)a.u;
  double* ifield = (double*)a.ifield;
  const long long N = a.g.N;
  const int nx = a.g.nx, ny = a.g.ny;
  const long long n = node_index(a.g, x, y, z);
  if (!SIMPLE && t.own[z & 3][e0] != FLUID) {
    // boundary node: no fluid, no solute transport
    a.vsig[n] = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) rho_out[k * N + n] = rho_in[k * N + n];
    u[n] = 0.0;
    u[N + n] = 0.0;
    u[2 * N + n] = 0.0;
    ifield[n] = 0.0;
    ifield[N + n] = 0.0;
    ifield[2 * N + n] = 0.0;
    return;
  }
  const Nbr b = make_nbr(x, y, z, a.g);
  constexpr double HALF_INV_A0 = 0.13060193748187072;  // 1 / (2 (1 + 2 sqrt 2))
  double qion = 0.0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const double r = rho_in[k * N + n];
    rho_out[k * N + n] = fma(-a.ph.dcoef[k], S[k], r);
    qion = fma(a.ph.z[k], r, qion);
  }
  const double gx = G[0] * HALF_INV_A0, gy = G[1] * HALF_INV_A0, gz = G[2] * HALF_INV_A0;
  const double ix = fma(-qion, a.ph.E[0], gx), iy = fma(-qion, a.ph.E[1], gy), iz = fma(-qion, a.ph.E[2], gz);
  ifield[n] = ix;
  ifield[N + n] = iy;
  ifield[2 * N + n] = iz;
  iv[0] += ix;
  iv[1] += iy;
  iv[2] += iz;
  double ux, uy, uz, rho, usq;
  lb64_collide(f, c, a.ph.lam_e, gx + a.ph.g[0], gy + a.ph.g[1], gz + a.ph.g[2], ux, uy, uz, rho, usq);
  if (!finite_bits(rho) || !finite_bits(usq)) atomicOr(a.status, ST_NONFINITE);
  u[n] = ux;
  u[N + n] = uy;
  u[2 * N + n] = uz;
  a.vsig[n] = (unsigned char)(0x80u | sign_bits(ux) | (sign_bits(uy) << 2) | (sign_bits(uz) << 4));
  // ---- push stream with velocity bounce-back (Eq. 12) ----
  f_out[n] = f[0];
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    const int om = SIMPLE ? FLUID : t.own[(z + 4 + dcz(i)) & 3][e0 + dcx(i) + HX * dcy(i)];
    if (om == FLUID) {
      f_out[i * N + nbr_index(i, x, y, z, b, nx, ny)] = f[i];
    } else {
      double cvb = 0.0;
      if (om >= 0) {
        const int xb = dcx(i) > 0 ? b.xp : (dcx(i) < 0 ? b.xm : x);
        const int yb = dcy(i) > 0 ? b.yp : (dcy(i) < 0 ? b.ym : y);
        const int zb = dcz(i) > 0 ? b.zp : (dcz(i) < 0 ? b.zm : z);
        double vb[3];
        boundary_velocity(a.parts[om], xb, yb, zb, a.g, vb);
        cvb = cdot(i, vb[0], vb[1], vb[2]);
      }
      f_out[opp(i) * N + n] = f[i] - 6.0 * wgt(i) * a.ph.rho0 * cvb;
    }
  }
}

// Sum of three doubles over a block, fixed order; thread 0 writes it to
// ipart[3 * blk].
__device__ __forceinline__ void block_sum3(double (&v)[3], double* ipart, long long blk) {
  __shared__ double red[TN / 32][3];
  const int t = threadIdx.x + TILE_X * threadIdx.y;
  const int lane = t & 31, warp = t >> 5;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    double s = v[c];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) red[warp][c] = s;
  }
  __syncthreads();
  if (t == 0) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      double s = 0.0;
      for (int w = 0; w < TN / 32; ++w) s += red[w][c];
      ipart[3 * blk + c] = s;
    }
  }
}

// One block: tile column (bx, by), planes [z0, zend).  Per plane z: the links
// coming up from plane z - 1 are taken in; (barrier) the node's nine links and
// the halo's are computed and published; (barrier) the links of the plane are
// taken in and the node collides.  The fields of plane z + 2 are copied in
// meanwhile.
template <int K, bool PV>
__global__ void __launch_bounds__(256, K <= 2 ? 2 : 1) k_lb_fused(LBArgs a, Coll64 c) {
  extern __shared__ __align__(16) unsigned char lb64_smem[];
  LB64Smem<K>& t = *reinterpret_cast<LB64Smem<K>*>(lb64_smem);
  const int nx = a.g.nx, ny = a.g.ny, nz = a.g.nz;
  const long long N = a.g.N;
  const int x0 = blockIdx.x * TILE_X, y0 = blockIdx.y * TILE_Y;
  const int z0 = (int)((long long)blockIdx.z * nz / a.nzb);
  const int zend = (int)((long long)(blockIdx.z + 1) * nz / a.nzb);
  const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
  const int tid = threadIdx.x + TILE_X * threadIdx.y;
  const bool in_xy = x < nx && y < ny;
  const int e0 = threadIdx.x + 1 + HX * (threadIdx.y + 1);
  const HaloLink hl = halo_link(tid);
  int hoff[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int e = tid + q * TN, ey = e / HX, ex = e - ey * HX;
    hoff[q] = e < HP ? halo_wrap(x0 - 1 + ex, nx) + nx * halo_wrap(y0 - 1 + ey, ny) : -1;
  }
  auto slot = [](int z) { return (z + 3) % 3; };  // z >= -1
  auto stage = [&](int z) {
    const size_t pz = (size_t)nx * ny * wrap_plane(z, nz);
    const int s = slot(z);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (hoff[q] < 0) continue;
      const int e = tid + q * TN;
      const size_t m = hoff[q] + pz;
      cp_async4(&t.own[z & 3][e], a.owner + m);
      if (K > 0) {
        cp_async8(&t.phi[s][e], (const double*)a.phi + m);
        if (PV) cp_async8(&t.om[s][e], (const double*)a.psi + m);
      }
#pragma unroll
      for (int k = 0; k < K; ++k) cp_async8(&t.rho[k][s][e], (const double*)a.rho_in + k * N + m);
    }
  };
  // a landed plane: Psi to 1 - Psi and the species to rho / (1 - Psi), each
  // thread the elements that it copied; true where a node is a boundary or
  // partly covered
  auto land = [&](int z) -> int {
    const int s = slot(z);
    bool special = false;
    for (int e = tid; e < HP; e += TN) {
      const bool fl = t.own[z & 3][e] == FLUID;
      special |= !fl;
      if (K > 0 && PV) {
        const double psi = t.om[s][e];
        if ((__double_as_longlong(psi) << 1) == 0) {
          t.om[s][e] = 1.0;
        } else {
          special = true;
          const double om = 1.0 - psi;
          t.om[s][e] = om;
          if (fl) {
#pragma unroll
            for (int k = 0; k < K; ++k) t.rho[k][s][e] = t.rho[k][s][e] / om;
          }
        }
      }
    }
    return special ? 1 : 0;
  };
  double iv[3] = {0.0, 0.0, 0.0};
  stage(z0 - 1);
  stage(z0);
  stage(z0 + 1);
  cp_async_wait_all();
  int fm1 = __syncthreads_or(land(z0 - 1)), f0 = __syncthreads_or(land(z0)), fp1 = land(z0 + 1);
  if (K > 0) {
    // the links going up from plane z0 - 1 (of which only their upper end counts)
    double S[K > 0 ? K : 1] = {}, G[3] = {};
    const int s0 = slot(z0 - 1), s1 = slot(z0), o0 = (z0 - 1) & 3, o1 = z0 & 3;
    if (fm1 | f0) {
      own_links<K, false, PV, NFLAT, NLINK>(t, a.ph, s0, s1, o0, o1, e0, S, G);
      halo_links<K, false, PV>(t, a.ph, hl, false, s0, s1, o0, o1);
    } else {
      own_links<K, true, PV, NFLAT, NLINK>(t, a.ph, s0, s1, o0, o1, e0, S, G);
      halo_links<K, true, PV>(t, a.ph, hl, false, s0, s1, o0, o1);
    }
    __syncthreads();
  }
  for (int z = z0; z < zend; ++z) {
    double S[K > 0 ? K : 1] = {}, G[3] = {};
    if (K > 0) other_links<K, NFLAT, NLINK>(t, e0, S, G);
    fp1 = __syncthreads_or(fp1);  // the links from below are taken in; plane z + 1 has landed
    if (z + 1 < zend) stage(z + 2);
    const bool special = fm1 | f0 | fp1;
    if (K > 0) {
      const int s0 = slot(z), s1 = slot(z + 1), o0 = z & 3, o1 = (z + 1) & 3;
      if (special) {
        own_links<K, false, PV, 0, NLINK>(t, a.ph, s0, s1, o0, o1, e0, S, G);
        halo_links<K, false, PV>(t, a.ph, hl, true, s0, s1, o0, o1);
      } else {
        own_links<K, true, PV, 0, NLINK>(t, a.ph, s0, s1, o0, o1, e0, S, G);
        halo_links<K, true, PV>(t, a.ph, hl, true, s0, s1, o0, o1);
      }
    }
    double f[Q];
    if (in_xy) {
      const double* f_in = (const double*)a.f_in + node_index(a.g, x, y, z);
#pragma unroll
      for (int i = 0; i < Q; ++i) f[i] = f_in[i * N];
    }
    __syncthreads();
    if (K > 0) other_links<K, 0, NFLAT>(t, e0, S, G);
    if (in_xy) {
      if (special) lb64_node<K, false>(t, a, c, x, y, z, e0, S, G, f, iv);
      else lb64_node<K, true>(t, a, c, x, y, z, e0, S, G, f, iv);
    }
    fm1 = f0;
    f0 = fp1;
    cp_async_wait_all();
    fp1 = z + 1 < zend ? land(z + 2) : 0;
  }
  block_sum3(iv, a.ipart,
             blockIdx.x + (long long)gridDim.x * (blockIdx.y + (long long)gridDim.y * blockIdx.z));
}

// S3: rho' = (rho - div J) + volume-of-fluid advection.  rho_out holds
// rho - div J (written by S2) and is updated in place; rho_in is the species
// field at the start of the step (the advected one).  The cell displaced by
// u overlaps the neighbours at offsets s with s_a in {0, sign(u_a)}; the share
// of offset s is prod_a w_a, w_a = 1 - |u_a| (s_a = 0) or |u_a|.
//
// 32 x 8 tiles marching through a segment of planes.  The weights |u_a| and
// 1 - |u_a|, the species and the sign bytes of three planes with a one-node
// halo are in shared memory (a fourth slot takes the next plane), each weight
// formed once.  A node first marks the neighbours of which it receives a share
// (integer work on the sign bytes), then all lanes of the warp take their marked
// neighbours one after another: a branch per neighbour would be issued by the
// warp for every direction that any of its lanes receives from.  FP64
// instructions per node (K = 2): 4 for the weights, 28 for the shares sent, 4
// per share received (seven on average).  One thread per node with the
// neighbours' velocities from global memory took 0.51 ms at 128^3, 0.097 at 64^3.
template <int K>
struct Adv64Plane {
  double w[6][HP];    // |u_x|, |u_y|, |u_z|, then 1 - each
  double rho[K][HP];
  unsigned char sg[HP + 4];  // sign bytes of S2 (bit 7 fluid)
};
template <int K>
struct Adv64Smem {
  Adv64Plane<K> pl[4];  // plane p in slot p & 3
};

template <int K>
__global__ void __launch_bounds__(256, 2) k_advect(LBArgs a) {
  extern __shared__ __align__(16) unsigned char adv64_smem[];
  Adv64Smem<K>& t = *reinterpret_cast<Adv64Smem<K>*>(adv64_smem);
  const int nx = a.g.nx, ny = a.g.ny, nz = a.g.nz;
  const long long N = a.g.N;
  double* rho_out = (double*)a.rho_out;
  const int x0 = blockIdx.x * TILE_X, y0 = blockIdx.y * TILE_Y;
  const int z0 = (int)((long long)blockIdx.z * nz / a.advseg);
  const int zend = (int)((long long)(blockIdx.z + 1) * nz / a.advseg);
  const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
  const int tid = threadIdx.x + TILE_X * threadIdx.y;
  const bool in_xy = x < nx && y < ny;
  const int e0 = threadIdx.x + 1 + HX * (threadIdx.y + 1);
  int hoff[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int e = tid + q * TN, ey = e / HX, ex = e - ey * HX;
    hoff[q] = e < HP ? halo_wrap(x0 - 1 + ex, nx) + nx * halo_wrap(y0 - 1 + ey, ny) : -1;
  }
  auto stage = [&](int z) {
    Adv64Plane<K>& p = t.pl[z & 3];
    const size_t pz = (size_t)nx * ny * wrap_plane(z, nz);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (hoff[q] < 0) continue;
      const int e = tid + q * TN;
      const size_t m = hoff[q] + pz;
#pragma unroll
      for (int d = 0; d < 3; ++d) cp_async8(&p.w[d][e], (const double*)a.u + d * N + m);
#pragma unroll
      for (int k = 0; k < K; ++k) cp_async8(&p.rho[k][e], (const double*)a.rho_in + k * N + m);
      p.sg[e] = a.vsig[m];
    }
  };
  // a landed plane: the weights, each thread the elements that it copied
  auto land = [&](int z) {
    Adv64Plane<K>& p = t.pl[z & 3];
    for (int e = tid; e < HP; e += TN) {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const double v = __longlong_as_double(__double_as_longlong(p.w[d][e]) & 0x7fffffffffffffffLL);
        p.w[d][e] = v;
        p.w[3 + d][e] = 1.0 - v;
      }
    }
  };
  stage(z0 - 1);
  stage(z0);
  stage(z0 + 1);
  cp_async_wait_all();
  land(z0 - 1);
  land(z0);
  bool bad = false;
  for (int z = z0; z < zend; ++z) {
    const long long n = node_index(a.g, x, y, z);
    double acc[K];
    if (in_xy) {
#pragma unroll
      for (int k = 0; k < K; ++k) acc[k] = rho_out[k * N + n];  // S2's result, issued early
    }
    cp_async_wait_all();
    land(z + 1);
    __syncthreads();  // planes z - 1, z, z + 1 ready; plane z - 2 no longer read
    if (z + 1 < zend) stage(z + 2);
    const Adv64Plane<K>& P0 = t.pl[z & 3];
    const unsigned own = in_xy ? P0.sg[e0] : 0u;
    if (!(own & 0x80u)) continue;  // fluid bit of S2 (the flags may change meanwhile)
    // the neighbours that move here along every nonzero component of q
    unsigned from = 0;
#pragma unroll
    for (int c = 0; c < 27; ++c) {
      const int qx = c % 3 - 1, qy = c / 3 % 3 - 1, qz = c / 9 - 1;
      if (!qx && !qy && !qz) continue;
      const unsigned mask = 0x80u | (qx ? 3u : 0u) | (qy ? 12u : 0u) | (qz ? 48u : 0u);
      const unsigned want = 0x80u | (qx > 0 ? 1u : (qx < 0 ? 2u : 0u)) | (qy > 0 ? 4u : (qy < 0 ? 8u : 0u)) |
                            (qz > 0 ? 16u : (qz < 0 ? 32u : 0u));
      const unsigned sg = t.pl[(z + 4 - qz) & 3].sg[e0 - qx - HX * qy];
      if ((sg & mask) == want) from |= 1u << c;
    }
    // outflow: the shares that land on fluid nodes (one aimed at a boundary
    // stays; one along a component of zero velocity is zero)
    auto sign_of = [](unsigned v) { return v == 1u ? 1 : (v == 2u ? -1 : 0); };
    const int sx = sign_of(own & 3u), sy = sign_of((own >> 2) & 3u), sz = sign_of((own >> 4) & 3u);
    {
      const double ax = P0.w[0][e0], ay = P0.w[1][e0], az = P0.w[2][e0];
      const double bx = P0.w[3][e0], by = P0.w[4][e0], bz = P0.w[5][e0];
      const double wxy[4] = {bx * by, ax * by, bx * ay, ax * ay};
      const unsigned char* const f0 = P0.sg;
      const unsigned char* const f1 = t.pl[(z + 4 + sz) & 3].sg;
#pragma unroll
      for (int o = 1; o < 8; ++o) {
        const int e = e0 + ((o & 1) ? sx : 0) + ((o & 2) ? HX * sy : 0);
        if (!(((o & 4) ? f1 : f0)[e] & 0x80u)) continue;
        const double frac = wxy[o & 3] * ((o & 4) ? az : bz);
#pragma unroll
        for (int k = 0; k < K; ++k) acc[k] = fma(-P0.rho[k][e0], frac, acc[k]);
      }
    }
    while (from) {
      const int c = __ffs(from) - 1;
      from &= from - 1u;
      const int cz = c / 9, cy = (c - 9 * cz) / 3, cx = c - 9 * cz - 3 * cy;  // q + 1
      const Adv64Plane<K>& P = t.pl[(z + 5 - cz) & 3];
      const int e = e0 + 1 - cx + HX * (1 - cy);
      const double frac = P.w[cx == 1 ? 3 : 0][e] * P.w[cy == 1 ? 4 : 1][e] * P.w[cz == 1 ? 5 : 2][e];
#pragma unroll
      for (int k = 0; k < K; ++k) acc[k] = fma(P.rho[k][e], frac, acc[k]);
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
      rho_out[k * N + n] = acc[k];
      bad |= !finite_bits(acc[k]);
    }
  }
  cp_async_wait_all();
  if (bad) atomicOr(a.status, ST_NONFINITE);
}

__global__ void k_fill(Grid g, const int* owner, double* f, double* rho, int K, double rho0,
                       double b0, double b1, double b2, double b3) {
  const long long N = g.N;
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  const bool fl = owner[n] == FLUID;
  const double bk[4] = {b0, b1, b2, b3};
  for (int k = 0; k < K; ++k) rho[k * N + n] = fl ? bk[k] : 0.0;
#pragma unroll
  for (int i = 0; i < Q; ++i) f[i * N + n] = fl ? wgt(i) * rho0 : 0.0;
}

unsigned blocks_for(long long n, int threads) { return (unsigned)((n + threads - 1) / threads); }

}  // namespace

// shared memory above the 48 KB default, set once per context before any launch
// (in particular before a step is captured into a graph)
cudaError_t lb64_prepare() {
  cudaError_t e = cudaSuccess;
#define EK_ATTR(KK, PV)                                                                                      \
  if (e == cudaSuccess)                                                                                      \
    e = cudaFuncSetAttribute(k_lb_fused<KK, PV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(LB64Smem<KK>));
  EK_ATTR(0, true) EK_ATTR(1, true) EK_ATTR(2, true) EK_ATTR(3, true) EK_ATTR(4, true)
  EK_ATTR(0, false) EK_ATTR(1, false) EK_ATTR(2, false) EK_ATTR(3, false) EK_ATTR(4, false)
#undef EK_ATTR
#define EK_ATTR(KK)     \
  if (e == cudaSuccess) \
    e = cudaFuncSetAttribute(k_advect<KK>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Adv64Smem<KK>));
  EK_ATTR(1) EK_ATTR(2) EK_ATTR(3) EK_ATTR(4)
#undef EK_ATTR
  return e;
}

// Segments per tile column.  The FP64 pipes of the 152 SMs share the blocks,
// so a launch takes about ceil(blocks / 152) block times, and a block of p
// planes costs p and a quarter (the links up from the plane below it); two
// blocks per SM hide each other's barriers, so fewer than 304 are not taken
// where the box has more planes.  Measured on GB300 (ms per launch): 64^3 in
// 9 / 16 / 19 / 32 / 64 segments 0.291, 0.279, 0.244, 0.246, 0.238; 128^3 in
// 5 / 10 / 16 / 19 / 32 segments 2.02, 1.67, 1.50, 1.55, 1.54.
int lb64_segments(const Grid& g) {
  const long long cols = (long long)((g.nx + TILE_X - 1) / TILE_X) * ((g.ny + TILE_Y - 1) / TILE_Y);
  int best = g.nz;
  double cost = -1.0;
  for (int n = 1; n <= g.nz; ++n) {
    if (cols * n < 2 * 152 && n < g.nz) continue;
    const int p = (g.nz + n - 1) / n;
    const double c = (double)((cols * n + 151) / 152) * (p + 0.25);
    if (cost < 0.0 || c < cost) {
      cost = c;
      best = n;
    }
  }
  return best;
}

cudaError_t launch_lb_fused(const LBArgs& a, cudaStream_t s) {
  const Phys& ph = a.ph;
  const Coll64 c{0.5 * (1.0 + ph.lam_e), 0.5 * (1.0 + ph.lam_o), 4.5 * (2.0 + ph.lam_e) / 36.0, -4.5 * ph.lam_e / 36.0,
                 -ph.lam_o / 12.0, -1.5 * (2.0 + ph.lam_e), 1.0 + ph.lam_e};
  const bool pv = ph.pv != 0;
  const dim3 grid = lattice_grid32(a.g, a.nzb);
  switch (ph.K) {
#define EK_CASE(KK)                                                                                        \
  case KK:                                                                                                 \
    if (pv) k_lb_fused<KK, true><<<grid, lattice_block(), sizeof(LB64Smem<KK>), s>>>(a, c);                 \
    else k_lb_fused<KK, false><<<grid, lattice_block(), sizeof(LB64Smem<KK>), s>>>(a, c);                   \
    break;
    EK_CASE(0)
    EK_CASE(1)
    EK_CASE(2)
    EK_CASE(3)
    EK_CASE(4)
#undef EK_CASE
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// Segments per tile column of S3: 8 planes each (a segment loads the plane on
// each side of it as well), shorter while the grid has less than two rounds of
// the two blocks that fit on an SM.
int adv64_segments(const Grid& g) {
  const long long cols = (long long)((g.nx + TILE_X - 1) / TILE_X) * ((g.ny + TILE_Y - 1) / TILE_Y);
  int p = 8;
  while (p > 1 && cols * ((g.nz + p - 1) / p) < 2 * 2 * 152) p /= 2;
  return std::max(1, (g.nz + p - 1) / p);
}

cudaError_t launch_advection(const LBArgs& a, cudaStream_t s) {
  const dim3 grid = lattice_grid32(a.g, a.advseg);
  switch (a.ph.K) {
    case 0: return cudaSuccess;
#define EK_CASE(KK) \
  case KK: k_advect<KK><<<grid, lattice_block(), sizeof(Adv64Smem<KK>), s>>>(a); break;
    EK_CASE(1)
    EK_CASE(2)
    EK_CASE(3)
    EK_CASE(4)
#undef EK_CASE
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_fill(const Grid& g, const Phys& ph, const int* owner, double* f, double* rho,
                        const double* bulk_k, cudaStream_t s) {
  k_fill<<<blocks_for(g.N, 256), 256, 0, s>>>(g, owner, f, rho, ph.K, ph.rho0, bulk_k[0],
                                                 bulk_k[1], bulk_k[2], bulk_k[3]);
  return cudaGetLastError();
}

}  // namespace ek
