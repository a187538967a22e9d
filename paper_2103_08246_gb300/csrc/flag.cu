// Spring-network flag (Sec. II.B structural model), one launch per fluid
// step running all velocity-Verlet sub-steps with the fluid force held
// constant: k_flag_patch on the lattice (forces in double-single arithmetic,
// state FP64), k_flag over lists (FP64) for lattices whose patches do not fit
// shared memory.
//
// Energies: stretching springs E = k_s/2 (|x_b - x_a| - l0)^2 on lattice edges
// and both cell diagonals; bending hinges E = k_h (1 - n_A . n_B) between the
// two triangles (of one of the two overlaid triangulations) sharing an edge.
//
// The bending force is assembled per triangle. For triangle T = (p0, p1, p2)
// with N = (p1 - p0) x (p2 - p0) and n = N / |N|, every hinge h of T with
// neighbour normal m_h contributes k_h dn/dx^T m_h, and
// dn/dx^T m = dN/dx^T (m - (n . m) n) / |N| is linear in the bracket, so
//   G_T = sum_h k_h (m_h - (n . m_h) n) / |N|,
//   f1 = (p2 - p0) x G_T,  f2 = G_T x (p1 - p0),  f0 = -(f1 + f2)
// gives the whole bending force of T on its vertices with two cross products.
//
// Each force term is written to its own slot and every vertex sums its slots
// in a fixed order (CSR list), so the result does not depend on thread
// timing. The CTAs of one thread-block cluster share the work and meet at the
// cluster barrier (hardware) between phases. Data written by other CTAs is
// read with L2-only loads. (The list form, k_flag.)
#include <cooperative_groups.h>

#include <cmath>

#include "solver.h"

namespace cg = cooperative_groups;

namespace ibm {

struct D3 {
  double x, y, z;
};
__device__ inline D3 operator-(D3 a, D3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ inline D3 operator+(D3 a, D3 b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ inline D3 operator*(double s, D3 a) { return {s * a.x, s * a.y, s * a.z}; }
__device__ inline double dot(D3 a, D3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ inline D3 cross(D3 a, D3 b) {
  return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}
__device__ inline D3 ld3(const double* p, int v) {
  return {__ldcg(p + 3 * v), __ldcg(p + 3 * v + 1), __ldcg(p + 3 * v + 2)};
}
__device__ inline void st3(double* p, int q, D3 f) {
  p[3 * q] = f.x;
  p[3 * q + 1] = f.y;
  p[3 * q + 2] = f.z;
}

// 1 / sqrt(x) in FP64 from the FP32 estimate and one Newton-Raphson step for
// f(y) = 1/y^2 - x: y1 = y0 (3/2 - x y0^2 / 2). The FP32 estimate carries a
// relative error below ~2^-22, one step squares it (~1e-13), well inside the
// parity bound of the structural solve; FP64 work drops to a few multiplies.
__device__ inline double rsqrt_nr(double x) {
  const double y0 = (double)rsqrtf((float)x);
  return y0 * (1.5 - 0.5 * x * y0 * y0);
}

// unit normals of all triangles, stretching forces of all springs
__device__ void phase_normals_springs(const Flag& fl, int gt, int G) {
  for (int t = gt; t < fl.n_tri; t += G) {
    const int* tv = fl.tri + 3 * t;
    const D3 p0 = ld3(fl.X, tv[0]), p1 = ld3(fl.X, tv[1]), p2 = ld3(fl.X, tv[2]);
    const D3 N = cross(p1 - p0, p2 - p0);
    const double inv = rsqrt_nr(dot(N, N));
    st3(fl.tri_n, t, inv * N);
    fl.tri_inv[t] = inv;
  }
  const int base = 3 * fl.n_tri;
  for (int q = gt; q < fl.n_spring; q += G) {
    const int a = fl.spring[2 * q], b = fl.spring[2 * q + 1];
    const D3 d = ld3(fl.X, b) - ld3(fl.X, a);
    const double len2 = dot(d, d);
    const double il = rsqrt_nr(len2);
    const D3 f = (fl.k_s * (len2 * il - fl.l0[q]) * il) * d;   // pulls a towards b when stretched
    st3(fl.slot, base + 2 * q, f);
    st3(fl.slot, base + 2 * q + 1, -1.0 * f);
  }
}

// bending forces of every triangle from its hinges
__device__ void phase_bending(const Flag& fl, int gt, int G) {
  for (int t = gt; t < fl.n_tri; t += G) {
    const D3 n = ld3(fl.tri_n, t);
    D3 g = {0.0, 0.0, 0.0};
    for (int e = 0; e < 3; ++e) {
      const int nb = fl.tri_nb[3 * t + e];
      if (nb < 0) continue;
      const D3 m = ld3(fl.tri_n, nb);
      g = g + fl.tri_k[3 * t + e] * (m - dot(n, m) * n);
    }
    g = __ldcg(fl.tri_inv + t) * g;
    const int* tv = fl.tri + 3 * t;
    const D3 p0 = ld3(fl.X, tv[0]), p1 = ld3(fl.X, tv[1]), p2 = ld3(fl.X, tv[2]);
    const D3 f1 = cross(p2 - p0, g), f2 = cross(g, p1 - p0);
    st3(fl.slot, 3 * t, -1.0 * (f1 + f2));
    st3(fl.slot, 3 * t + 1, f1);
    st3(fl.slot, 3 * t + 2, f2);
  }
}

__device__ inline D3 gather_acc(const Flag& fl, int v) {
  D3 f = {fl.Ff[3 * v], fl.Ff[3 * v + 1], fl.Ff[3 * v + 2]};
  for (int e = fl.csr_off[v]; e < fl.csr_off[v + 1]; ++e) f = f + ld3(fl.slot, fl.csr_idx[e]);
  return fl.inv_mass[v] * f;
}

__global__ void __launch_bounds__(512) k_flag(Params* __restrict__ prm, Flag fl, int force) {
  cg::cluster_group cl = cg::this_cluster();
  if (!force && !prm->flag_pending) return;   // same value for every thread of the cluster
  const int gt = (int)cl.block_rank() * blockDim.x + threadIdx.x;
  const int G = (int)cl.num_blocks() * blockDim.x;
  const double dt = prm->flag_dt;
  const int nsub = prm->flag_nsub;
  const double hs = dt / nsub;
  phase_normals_springs(fl, gt, G);
  cl.sync();
  phase_bending(fl, gt, G);
  cl.sync();
  for (int v = gt; v < fl.nv; v += G) st3(fl.A, v, gather_acc(fl, v));
  for (int s = 0; s < nsub; ++s) {
    for (int v = gt; v < fl.nv; v += G) {
      D3 V = {fl.V[3 * v], fl.V[3 * v + 1], fl.V[3 * v + 2]};
      const D3 A = {fl.A[3 * v], fl.A[3 * v + 1], fl.A[3 * v + 2]};
      V = V + (0.5 * hs) * A;
      st3(fl.V, v, V);
      fl.X[3 * v] += hs * V.x;
      fl.X[3 * v + 1] += hs * V.y;
      fl.X[3 * v + 2] += hs * V.z;
    }
    cl.sync();
    phase_normals_springs(fl, gt, G);
    cl.sync();
    phase_bending(fl, gt, G);
    cl.sync();
    for (int v = gt; v < fl.nv; v += G) {
      const D3 a = gather_acc(fl, v);
      st3(fl.A, v, a);
      fl.V[3 * v] += 0.5 * hs * a.x;
      fl.V[3 * v + 1] += 0.5 * hs * a.y;
      fl.V[3 * v + 2] += 0.5 * hs * a.z;
    }
  }
  cl.sync();
  if (gt == 0) prm->flag_pending = 0;
}

// ---------------------------------------------------------------- lattice patches
// The same forces on the structured lattice, one CTA of the cluster per
// rectangular patch of vertices, one cluster barrier per sub-step.
//
// What bounds the kernel above is the FP64 pipe of the cluster's 16 SMs (two
// instructions per clock and SM: about 500 FP64 instructions per lattice cell
// and sub-step), then its three barriers and the trips through L2 between
// them. Here the forces are evaluated in double-single arithmetic (an
// unevaluated FP32 pair, 48 bits; sums and products after Knuth and Dekker) on
// the FP32 pipe, which issues 64 times as many instructions per clock;
// positions, velocities and the integration stay FP64. The error of a force
// against 64 bits is below that of the list form, whose rsqrt_nr carries up to
// 5e-14: 0.3 to 0.8 of it over lattices of 9 to 2100 points a side, strains to
// 1e-2 and bending to 0.1 (33 x 33: 5.9e-14 against 1.9e-13 rms), 0.97 where
// the springs are too weak to count. Edges are exact: each CTA publishes its
// positions once per sub-step as 64-bit fixed point (2^49 per scaled unit; the
// longest spring is 1/2 to 1 unit), and edges are integer differences. The
// origin is a multiple of 1024 units near the flag's corner, so that subtracting
// it rounds nothing that the FP64 position held above 2^-49. Positions reach
// 8192 units from it; the longest lattice with patches has a side of 2176
// points, at most a unit apart. Beyond that (a flag that has diverged) they
// saturate, and a patch that has seen such a position, or one that is not a
// number, leaves its vertices as NaN.
//
// Each CTA keeps its vertices and a halo of two lattice points (the reach of
// the hinge forces) in shared memory, pulls the halo from its neighbours'
// shared memory after the barrier, and recomputes the normals of the halo
// cells instead of exchanging them (a second barrier and exchange cost more
// than the FP32 work: the ring is 144 against 81 cells on a 9 x 9 patch).
// A lattice cell (a, b) has the corners v00, v10 (along s), v01 (along t),
// v11 and the edges S = v10 - v00, T = v01 - v00, T' = v11 - v10,
// D = v11 - v00, E = v01 - v10; triangulation A splits it into
// A0 = (v00, v10, v11), A1 = (v00, v11, v01), B into B0 = (v00, v10, v01),
// B1 = (v10, v11, v01). One thread takes one triangulation of one cell, with
// the springs S, D (A) or T, E (B); its forces on the four corners go to
// shared memory and every vertex sums its four cells in a fixed order.
struct DS {
  float h, l;
};
// the _rn intrinsics keep the compiler from contracting a product into the
// sums whose rounding errors are recovered here
__device__ __forceinline__ DS quick2(float a, float b) {
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ DS two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ DS operator-(DS a) { return {-a.h, -a.l}; }
__device__ __forceinline__ DS operator+(DS a, DS b) {
  const DS s = two_sum(a.h, b.h);
  return quick2(s.h, s.l + (a.l + b.l));
}
__device__ __forceinline__ DS operator-(DS a, DS b) { return a + (-b); }
__device__ __forceinline__ DS operator*(DS a, DS b) {
  const float p = __fmul_rn(a.h, b.h);
  return quick2(p, fmaf(a.h, b.l, fmaf(a.l, b.h, fmaf(a.h, b.h, -p))));
}
// a b + c
__device__ __forceinline__ DS ds_fma(DS a, DS b, DS c) {
  const float p = __fmul_rn(a.h, b.h);
  const float e = fmaf(a.h, b.l, fmaf(a.l, b.h, fmaf(a.h, b.h, -p)));
  const DS s = two_sum(p, c.h);
  return quick2(s.h, s.l + (e + c.l));
}
// a b - c d
__device__ __forceinline__ DS ds_det(DS a, DS b, DS c, DS d) {
  const float p = __fmul_rn(a.h, b.h), q = __fmul_rn(c.h, d.h);
  const float pe = fmaf(a.h, b.l, fmaf(a.l, b.h, fmaf(a.h, b.h, -p)));
  const float qe = fmaf(c.h, d.l, fmaf(c.l, d.h, fmaf(c.h, d.h, -q)));
  const DS s = two_sum(p, -q);
  return quick2(s.h, s.l + (pe - qe));
}
// 1 / sqrt(x) from the FP32 estimate: with r = 1 - x y0^2 (|r| < 2^-21) in two
// parts, r1 the exact leading difference and r2 the rest,
// y0 (1 + r / 2 + 3 r^2 / 8); r in one part rounds at 2^-46
__device__ __forceinline__ DS ds_rsqrt(DS x) {
  const float y = rsqrtf(x.h);
  const float p = __fmul_rn(x.h, y);
  const float pl = fmaf(x.l, y, fmaf(x.h, y, -p));
  const float q = __fmul_rn(p, y);
  const float r1 = __fsub_rn(1.0f, q), r2 = -fmaf(pl, y, fmaf(p, y, -q)), r = r1 + r2;
  const float t = __fmul_rn(y, 0.5f * r1);
  const DS s = quick2(y, t);
  return {s.h, s.l + fmaf(y, fmaf(0.375f * r, r, 0.5f * r2), fmaf(y, 0.5f * r1, -t))};
}
// 1 / x
__device__ __forceinline__ DS ds_rcp(DS x) {
  const float y = __frcp_rn(x.h);
  const float q = __fmul_rn(x.h, y);
  const float r = __fsub_rn(__fsub_rn(1.0f, q), fmaf(x.h, y, -q)) - x.l * y;
  return quick2(y, y * fmaf(r, r, r));
}
struct DV {
  DS x, y, z;
};
__device__ __forceinline__ DV operator-(DV a) { return {-a.x, -a.y, -a.z}; }
__device__ __forceinline__ DV operator+(DV a, DV b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ DV operator*(DS s, DV a) { return {s * a.x, s * a.y, s * a.z}; }
__device__ __forceinline__ DV axpy(DS s, DV a, DV c) {
  return {ds_fma(s, a.x, c.x), ds_fma(s, a.y, c.y), ds_fma(s, a.z, c.z)};
}
__device__ __forceinline__ DS dot(DV a, DV b) { return ds_fma(a.x, b.x, ds_fma(a.y, b.y, a.z * b.z)); }
__device__ __forceinline__ DV cross(DV a, DV b) {
  return {ds_det(a.y, b.z, a.z, b.y), ds_det(a.z, b.x, a.x, b.z), ds_det(a.x, b.y, a.y, b.x)};
}

// an edge from the difference of its ends' fixed-point positions (2^49 per
// scaled unit): upper word, next 23 bits and last 9 bits, each exact in FP32
// (the upper word for edges below 128 units; it cannot overflow). Every bit
// that the pair has room for is kept: with the lower bits rounded once to 24
// the forces' error was three to ten times as large (33 x 33: 0.1455 ms, 0.149
// with them).
__device__ __forceinline__ DS ds_edge(long long b, long long a) {
  const long long d = b - a;
  const unsigned low = (unsigned)d;
  const DS s = quick2((float)(int)(d >> 32) * 0x1p-17f, (float)(low >> 9) * 0x1p-40f);
  return {s.h, s.l + (float)(low & 511u) * 0x1p-49f};
}
constexpr long long PATCH_LIM = 1ll << 62;   // positions saturate here: differences stay in 64 bits
constexpr int PATCH_SIDE = 4096;             // points along a side, half of what the positions reach
constexpr size_t PATCH_SMEM_MAX = 220 * 1024;
constexpr int PATCH_MAXV = 2;        // vertices per thread
constexpr int PATCH_HALO = 2;
constexpr int PATCH_NS = 17;         // normals: 16 values per cell (A0, A1, B0, B1: n, 1/|N|), padded
constexpr int PATCH_FS = 25;         // forces: 2 triangulations x 4 corners x 3, padded
// split of n points over p patches: patch q holds [q n / p, (q + 1) n / p)
__host__ __device__ inline int patch_begin(int q, int n, int p) { return (int)((long long)q * n / p); }
__host__ __device__ inline int patch_owner(int a, int n, int p) { return (int)(((long long)(a + 1) * p - 1) / n); }

struct PatchSmem {
  int hm, wm;                        // largest patch: rows, columns
  __host__ __device__ int wv() const { return wm + 2 * PATCH_HALO; }                     // vertex row
  __host__ __device__ int nvert() const { return (hm + 2 * PATCH_HALO) * wv(); }
  __host__ __device__ int wn() const { return wm + 3; }                                  // cells [-2, w]
  __host__ __device__ int nnorm() const { return (hm + 3) * wn(); }
  __host__ __device__ int wf() const { return wm + 1; }                                  // cells [-1, w - 1]
  __host__ __device__ int nforce() const { return (hm + 1) * wf(); }
  __host__ __device__ int nhalo() const { return nvert(); }
  __host__ __device__ size_t bytes() const {
    return (size_t)nvert() * 48 + (size_t)nnorm() * PATCH_NS * 8 + (size_t)nforce() * PATCH_FS * 8 +
           (size_t)nhalo() * 8;
  }
};

__device__ __forceinline__ DV edge_of(const long long* X, int p, int q) {   // from point p to point q
  return {ds_edge(X[3 * q], X[3 * p]), ds_edge(X[3 * q + 1], X[3 * p + 1]), ds_edge(X[3 * q + 2], X[3 * p + 2])};
}
__device__ __forceinline__ void put_normal(DS* n, DV N) {
  const DS inv = ds_rsqrt(dot(N, N));
  n[0] = inv * N.x;
  n[1] = inv * N.y;
  n[2] = inv * N.z;
  n[3] = inv;
}
__device__ __forceinline__ DV get_normal(const DS* n) { return {n[0], n[1], n[2]}; }
// sum_h k_h m_h over the three hinges of a triangle, minus its part along n, over |N|
__device__ __forceinline__ DV hinge_vector(const DS* n, DV M) {
  const DV u = get_normal(n);
  return n[3] * axpy(-dot(u, M), u, M);
}
// spring coefficient k (len - l0) / len (scaled): len - l0 = (len^2 - l0^2) / (len + l0)
__device__ __forceinline__ DS spring_coef(DV d, float4 rest, DS k) {
  const DS l2 = dot(d, d), il = ds_rsqrt(l2);
  const DS delta = l2 - DS{rest.z, rest.w};
  const DS den = ds_fma(DS{rest.x, rest.y}, il, DS{1.0f, 0.0f});
  return (k * delta) * ((il * il) * ds_rcp(den));
}

__global__ void __launch_bounds__(512) k_flag_patch(Params* __restrict__ prm, Flag fl, int force) {
  extern __shared__ __align__(16) unsigned char fp_smem[];
  __shared__ int n_halo, lost;   // lost: a position of the patch or its halo is out of range or NaN
  cg::cluster_group cl = cg::this_cluster();
  if (!force && !prm->flag_pending) return;   // same value for every thread of the cluster
  const int rank = (int)cl.block_rank(), tid = threadIdx.x, nt_ = blockDim.x;
  const int ns = fl.ns, nt = fl.nt, pr = fl.patch_r, pc = fl.patch_c;
  const PatchSmem L{(ns + pr - 1) / pr, (nt + pc - 1) / pc};
  const int ri = rank / pc, ci = rank - ri * pc;
  const int a0 = patch_begin(ri, ns, pr), a1 = patch_begin(ri + 1, ns, pr);
  const int b0 = patch_begin(ci, nt, pc), b1 = patch_begin(ci + 1, nt, pc);
  const int wv = L.wv(), wn = L.wn(), wf = L.wf();
  long long* X0 = reinterpret_cast<long long*>(fp_smem);
  // positions: two buffers, because a neighbour may still pull those of one
  // evaluation while this CTA publishes the next
  DS* N = reinterpret_cast<DS*>(X0 + 6 * L.nvert());
  DS* F = N + (size_t)L.nnorm() * PATCH_NS;
  int2* halo = reinterpret_cast<int2*>(F + (size_t)L.nforce() * PATCH_FS);
  auto vloc = [&](int a, int b) { return (a - a0 + PATCH_HALO) * wv + (b - b0 + PATCH_HALO); };

  // halo list: local point, owner and the point in its owner's numbering
  if (tid == 0) n_halo = lost = 0;
  __syncthreads();
  const int ha = a1 - a0 + 2 * PATCH_HALO, hb = b1 - b0 + 2 * PATCH_HALO;
  for (int q = tid; q < ha * hb; q += nt_) {
    const int a = a0 - PATCH_HALO + q / hb, b = b0 - PATCH_HALO + q % hb;
    if (a < 0 || a >= ns || b < 0 || b >= nt || (a >= a0 && a < a1 && b >= b0 && b < b1)) continue;
    const int ra = patch_owner(a, ns, pr), rb = patch_owner(b, nt, pc);
    const int la = a - patch_begin(ra, ns, pr) + PATCH_HALO, lb = b - patch_begin(rb, nt, pc) + PATCH_HALO;
    halo[atomicAdd(&n_halo, 1)] = make_int2(vloc(a, b), ((ra * pc + rb) << 20) | (la * wv + lb));
  }

  const double dt = prm->flag_dt;
  const int nsub = prm->flag_nsub;
  const double hs = dt / nsub;
  const DS kS = {fl.k_edge[0].x, fl.k_edge[0].y}, kT = {fl.k_edge[1].x, fl.k_edge[1].y},
           kD = {fl.k_edge[2].x, fl.k_edge[2].y}, ks = {fl.k_edge[3].x, fl.k_edge[3].y};
  const double x0[3] = {fl.fix_x0[0], fl.fix_x0[1], fl.fix_x0[2]};   // scaled origin
  const double fix = fl.fix_scale, back = fl.force_scale;

  // this thread's vertices
  const int bw = b1 - b0, nown = (a1 - a0) * bw;
  int own[PATCH_MAXV], loc[PATCH_MAXV];
  double xv[PATCH_MAXV][3], vv[PATCH_MAXV][3], ff[PATCH_MAXV][3], im[PATCH_MAXV];
#pragma unroll
  for (int m = 0; m < PATCH_MAXV; ++m) {
    const int q = tid + m * nt_;
    own[m] = -1;
    if (q < nown) {
      const int a = a0 + q / bw, b = b0 + q % bw;
      own[m] = a * nt + b;
      loc[m] = vloc(a, b);
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        xv[m][e] = fl.X[3 * own[m] + e];
        vv[m][e] = fl.V[3 * own[m] + e];
        ff[m][e] = fl.Ff[3 * own[m] + e];
      }
      im[m] = fl.inv_mass[own[m]];
    }
  }
  auto publish = [&](long long* X) {
#pragma unroll
    for (int m = 0; m < PATCH_MAXV; ++m)
      if (own[m] >= 0)
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          // NaN converts to the lowest integer
          const long long q = min(max(__double2ll_rn(fma(xv[m][e], fix, -x0[e])), -PATCH_LIM), PATCH_LIM);
          X[3 * loc[m] + e] = q;
        }
  };
  const int na = a1 - a0, nb = b1 - b0;
  const int ncn = (na + 3) * (nb + 3);                  // cells [a0 - 2, a1] x [b0 - 2, b1]
  const int ncf = (na + 1) * (nb + 1);                  // cells [a0 - 1, a1) x [b0 - 1, b1)
  const int ncn32 = (ncn + 31) & ~31, ncf32 = (ncf + 31) & ~31;   // each triangulation in whole warps

  // accelerations of this thread's vertices from the published positions
  auto accelerate = [&](long long* X, double (&acc)[PATCH_MAXV][3]) {
    cl.sync();
    for (int q = tid; q < 3 * n_halo; q += nt_) {
      const int m = q / 3, e = q - 3 * m;
      const int2 hl = halo[m];
      const long long* src = cl.map_shared_rank(X, hl.y >> 20);
      X[3 * hl.x + e] = src[3 * (hl.y & 0xfffff) + e];
    }
    __syncthreads();
    for (int q = tid; q < 2 * ncn32; q += nt_) {
      const bool tb = q >= ncn32;
      const int cidx = tb ? q - ncn32 : q;
      const int la = cidx / (nb + 3), lb = cidx - la * (nb + 3);
      const int a = a0 - 2 + la, b = b0 - 2 + lb;
      if (cidx >= ncn || a < 0 || b < 0 || a >= ns - 1 || b >= nt - 1) continue;
      const int p00 = la * wv + lb, p10 = p00 + wv, p01 = p00 + 1, p11 = p10 + 1;
      DS* n = N + (size_t)(la * wn + lb) * PATCH_NS;
      if (!tb) {
        const DV S = edge_of(X, p00, p10), T = edge_of(X, p00, p01), D = edge_of(X, p00, p11);
        put_normal(n, cross(S, D));
        put_normal(n + 4, cross(D, T));
      } else {
        const DV S = edge_of(X, p00, p10), T = edge_of(X, p00, p01);
        put_normal(n + 8, cross(S, T));
        put_normal(n + 12, cross(edge_of(X, p10, p11), edge_of(X, p10, p01)));
      }
    }
    __syncthreads();
    for (int q = tid; q < 2 * ncf32; q += nt_) {
      const bool tb = q >= ncf32;
      const int cidx = tb ? q - ncf32 : q;
      const int la = cidx / (nb + 1), lb = cidx - la * (nb + 1);
      const int a = a0 - 1 + la, b = b0 - 1 + lb;
      if (cidx >= ncf || a < 0 || b < 0) continue;
      const bool full = a < ns - 1 && b < nt - 1;       // else only the lattice's last row or column of edges
      const int p00 = (la + 1) * wv + lb + 1, p10 = p00 + wv, p01 = p00 + 1, p11 = p10 + 1;
      const DS* n = N + (size_t)((la + 1) * wn + lb + 1) * PATCH_NS;
      const DS* n_bm = n - PATCH_NS;                    // cells b - 1, b + 1, a - 1, a + 1
      const DS* n_bp = n + PATCH_NS;
      const DS* n_am = n - (size_t)wn * PATCH_NS;
      const DS* n_ap = n + (size_t)wn * PATCH_NS;
      const bool lo_b = b > 0, hi_b = b < nt - 2, lo_a = a > 0, hi_a = a < ns - 2;
      const float4* rest = fl.lat + 4 * ((size_t)a * nt + b);   // S, T, D, E
      const DS zero = {0.0f, 0.0f};
      DV f00 = {zero, zero, zero}, f10 = f00, f01 = f00, f11 = f00;
      if (!tb) {
        if (a < ns - 1) {
          const DV S = edge_of(X, p00, p10);
          f10 = -(spring_coef(S, rest[0], ks) * S);
          if (full) {
            const DV T = edge_of(X, p00, p01), D = edge_of(X, p00, p11);
            f11 = -(spring_coef(D, rest[2], ks) * D);
            DV M0 = kD * get_normal(n + 4), M1 = kD * get_normal(n);
            if (lo_b) M0 = axpy(kS, get_normal(n_bm + 4), M0);
            if (hi_a) M0 = axpy(kT, get_normal(n_ap + 4), M0);
            if (hi_b) M1 = axpy(kS, get_normal(n_bp), M1);
            if (lo_a) M1 = axpy(kT, get_normal(n_am), M1);
            const DV G0 = hinge_vector(n, M0), G1 = hinge_vector(n + 4, M1);
            f10 = f10 + cross(D, G0);
            f11 = f11 + (cross(G0, S) + cross(T, G1));
            f01 = cross(G1, D);
          }
          f00 = -(f10 + (f11 + f01));
        }
      } else {
        if (b < nt - 1) {
          const DV T = edge_of(X, p00, p01);
          f01 = -(spring_coef(T, rest[1], ks) * T);
          if (full) {
            const DV S = edge_of(X, p00, p10), T1 = edge_of(X, p10, p11), E = edge_of(X, p10, p01);
            const DV sE = spring_coef(E, rest[3], ks) * E;
            DV M0 = kD * get_normal(n + 12), M1 = kD * get_normal(n + 8);
            if (lo_b) M0 = axpy(kS, get_normal(n_bm + 12), M0);
            if (lo_a) M0 = axpy(kT, get_normal(n_am + 12), M0);
            if (hi_a) M1 = axpy(kT, get_normal(n_ap + 8), M1);
            if (hi_b) M1 = axpy(kS, get_normal(n_bp + 8), M1);
            const DV G0 = hinge_vector(n + 8, M0), G1 = hinge_vector(n + 12, M1);
            const DV g = cross(G1, T1);
            f11 = cross(E, G1);
            f10 = sE + (cross(T, G0) + -(f11 + g));
            f01 = f01 + ((cross(G0, S) + g) + -sE);
          }
          f00 = -(f10 + (f11 + f01));
        }
      }
      DS* f = F + (size_t)cidx * PATCH_FS + (tb ? 12 : 0);
      f[0] = f00.x, f[1] = f00.y, f[2] = f00.z;
      f[3] = f10.x, f[4] = f10.y, f[5] = f10.z;
      f[6] = f01.x, f[7] = f01.y, f[8] = f01.z;
      f[9] = f11.x, f[10] = f11.y, f[11] = f11.z;
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < PATCH_MAXV; ++m) {
      if (own[m] < 0) continue;
      const int q = tid + m * nt_;
      const int la = q / bw, lb = q - la * bw;          // cell (a, b) of the vertex: (la + 1, lb + 1)
      const int a = a0 + la, b = b0 + lb;
      const DS* c00 = F + (size_t)((la + 1) * (nb + 1) + lb + 1) * PATCH_FS;
      const DS* c10 = c00 - (size_t)(nb + 1) * PATCH_FS;
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        DS s = c00[e] + c00[12 + e];
        if (a > 0) s = s + (c10[3 + e] + c10[15 + e]);
        if (b > 0) s = s + (c00[6 + e - PATCH_FS] + c00[18 + e - PATCH_FS]);
        if (a > 0 && b > 0) s = s + (c10[9 + e - PATCH_FS] + c10[21 + e - PATCH_FS]);
        acc[m][e] = im[m] * fma((double)s.h + (double)s.l, back, ff[m][e]);
      }
    }
  };

  double acc[PATCH_MAXV][3];
  publish(X0);
  accelerate(X0, acc);
  for (int s = 0; s < nsub; ++s) {
#pragma unroll
    for (int m = 0; m < PATCH_MAXV; ++m)
      if (own[m] >= 0)
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          vv[m][e] = fma(0.5 * hs, acc[m][e], vv[m][e]);
          xv[m][e] = fma(hs, vv[m][e], xv[m][e]);
        }
    long long* Xs = X0 + ((s + 1) & 1) * 3 * L.nvert();
    publish(Xs);
    accelerate(Xs, acc);
#pragma unroll
    for (int m = 0; m < PATCH_MAXV; ++m)
      if (own[m] >= 0)
#pragma unroll
        for (int e = 0; e < 3; ++e) vv[m][e] = fma(0.5 * hs, acc[m][e], vv[m][e]);
  }
  // the positions of the last sub-step, those of the halo among them
  const long long* Xl = X0 + (nsub & 1) * 3 * L.nvert();
  auto check = [&](int at) {
    for (int e = 0; e < 3; ++e)
      if (Xl[3 * at + e] == PATCH_LIM || Xl[3 * at + e] == -PATCH_LIM) lost = 1;
  };
  for (int q = tid; q < n_halo; q += nt_) check(halo[q].x);
#pragma unroll
  for (int m = 0; m < PATCH_MAXV; ++m)
    if (own[m] >= 0) check(loc[m]);
  __syncthreads();
#pragma unroll
  for (int m = 0; m < PATCH_MAXV; ++m)
    if (own[m] >= 0)
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        fl.X[3 * own[m] + e] = lost ? nan("") : xv[m][e];
        fl.V[3 * own[m] + e] = lost ? nan("") : vv[m][e];
      }
  cl.sync();   // no CTA leaves while a neighbour may still read its positions
  if (rank == 0 && tid == 0) prm->flag_pending = 0;
}

// te_mid (3), force (3), max strain (1)
__global__ void k_flag_stats(Flag fl, double* out) {
  __shared__ double scratch[32];
  double fx = 0, fy = 0, fz = 0, st = 0;
  for (int v = threadIdx.x; v < fl.nv; v += blockDim.x) {
    fx += fl.Ff[3 * v];
    fy += fl.Ff[3 * v + 1];
    fz += fl.Ff[3 * v + 2];
  }
  for (int q = threadIdx.x; q < fl.n_spring; q += blockDim.x) {
    const int a = fl.spring[2 * q], b = fl.spring[2 * q + 1];
    const double dx = fl.X[3 * b] - fl.X[3 * a], dy = fl.X[3 * b + 1] - fl.X[3 * a + 1],
                 dz = fl.X[3 * b + 2] - fl.X[3 * a + 2];
    st = fmax(st, fabs(sqrt(dx * dx + dy * dy + dz * dz) / fl.l0[q] - 1.0));
  }
  fx = block_sum(fx, scratch);
  __syncthreads();
  fy = block_sum(fy, scratch);
  __syncthreads();
  fz = block_sum(fz, scratch);
  __syncthreads();
  st = block_max(st, scratch);
  if (threadIdx.x == 0) {
    const int te = (fl.ns - 1) * fl.nt + fl.nt / 2;
    out[0] = fl.X[3 * te];
    out[1] = fl.X[3 * te + 1];
    out[2] = fl.X[3 * te + 2];
    out[3] = fx;
    out[4] = fy;
    out[5] = fz;
    out[6] = st;
  }
}

int flag_max_cluster() {
  // per device, so before the cached answer
  cudaFuncSetAttribute(k_flag, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  cudaFuncSetAttribute(k_flag_patch, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  cudaFuncSetAttribute(k_flag_patch, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PATCH_SMEM_MAX);
  static int cached = -1;
  if (cached > 0) return cached;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(16);
  cfg.blockDim = dim3(512);
  cfg.dynamicSmemBytes = PATCH_SMEM_MAX;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = 16;
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxPotentialClusterSize(&n, k_flag_patch, &cfg) != cudaSuccess || n < 1) {
    cudaGetLastError();
    n = 8;
  }
  cached = n > 16 ? 16 : n;
  return cached;
}

// patches of the lattice for a cluster of up to 16 CTAs: about 64 to 96 vertices
// each (a smaller patch is mostly halo), none when the largest would not fit in
// shared memory: 84 x 84 points fit, and so do 700 x 9 or 2100 x 2, which the
// fixed-point positions reach (PATCH_SIDE)
static PatchSmem patch_of(int ns, int nt, int pr, int pc) { return {(ns + pr - 1) / pr, (nt + pc - 1) / pc}; }
bool flag_patches(int ns, int nt, int* pr, int* pc) {
  const int most = flag_max_cluster();
  if (ns > PATCH_SIDE || nt > PATCH_SIDE) return false;
  int n = 1;
  while (2 * n <= most && (long long)ns * nt > 96ll * n) n *= 2;
  int best = 0;
  for (; n <= most && !best; n *= 2)
    for (int r = 1; r <= n; r *= 2) {
      if (r > ns || n / r > nt) continue;
      const PatchSmem L = patch_of(ns, nt, r, n / r);
      if (L.bytes() > PATCH_SMEM_MAX || L.hm * L.wm > PATCH_MAXV * 512) continue;
      if (!best || L.nnorm() < best) {
        best = L.nnorm();
        *pr = r;
        *pc = n / r;
      }
    }
  return best > 0;
}

void launch_flag(Params* prm, const Flag& fl, bool force, cudaStream_t s) {
  if (fl.nv == 0) return;
  // one CTA per lattice patch where the patches fit (65 x 65: 0.45 -> 0.128 ms
  // at 8 sub-steps, 33 x 33: 0.64 -> 0.150 ms at 17); the list form otherwise
  if (fl.patch_r) {
    const PatchSmem L = patch_of(fl.ns, fl.nt, fl.patch_r, fl.patch_c);
    const int tasks = 2 * ((L.nnorm() + 31) & ~31);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(fl.patch_r * fl.patch_c);
    cfg.blockDim = dim3(tasks < 512 ? tasks : 512);
    cfg.dynamicSmemBytes = L.bytes();
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = fl.patch_r * fl.patch_c;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_flag_patch, prm, fl, force ? 1 : 0);
    return;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(fl.cluster);
  cfg.blockDim = dim3(512);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = fl.cluster;
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k_flag, prm, fl, force ? 1 : 0);
}

void launch_flag_stats(const Flag& fl, double* out, cudaStream_t s) {
  if (fl.nv == 0) return;
  k_flag_stats<<<1, 1024, 0, s>>>(fl, out);
}

}  // namespace ibm
