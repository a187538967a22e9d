// Pressure Poisson equation L_h phi = D (Sec. II.B projection step): transforms
// in the periodic y and z directions, one tridiagonal (Thomas) solve along x
// per transverse wavenumber pair, inverse transforms.
//
// Transform: the discrete Hartley transform H x (k) = sum_j x_j cas(2 pi j k / N),
// cas = cos + sin. The periodic second difference is symmetric and circulant,
// so its eigenvalue lambda(k) = (2 cos(2 pi k / N) - 2) / h^2 is shared by
// cos and sin modes; the separable 2-D Hartley transform H_y H_z therefore
// diagonalises the y-z part of L_h exactly like the DFT, while every array
// stays real. H is its own inverse up to 1/N. Two real lines are packed into
// one complex FFT (radix-2, decimation in time, in shared memory) and
// separated afterwards:
//   Z = FFT(a + i b):  H a (k) = (Re Z_k - Im Z_k + Re Z_{N-k} + Im Z_{N-k}) / 2
//                      H b (k) = (Re Z_k + Im Z_k - Re Z_{N-k} + Im Z_{N-k}) / 2
//
// x solve, with the equation scaled by h^2 (Neumann ends phi_{-1} = phi_0,
// phi_nx = phi_{nx-1}):
//   phi_{i-1} + (-2 + lambda h^2) phi_i + phi_{i+1} = h^2 D_i,
// lambda h^2 = -4 sin^2(pi k_y / N_y) - 4 sin^2(pi k_z / N_z). The LU inverse
// pivots are tabulated once (FP64 arithmetic) at creation. lambda depends on
// k_y and k_z only through min(k, N - k), so the table holds the
// (N_y/2 + 1) x (N_z/2 + 1) distinct modes of every plane: a quarter of a
// field, which mostly stays in L2 between the two sweeps.
// Mode (0, 0) is singular: phi_0 = 0 is pinned, then the line mean removed,
// which sets mean(phi) = 0.
#include <cooperative_groups.h>

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "async_copy.cuh"
#include "solver.h"

namespace ibm {

namespace cg = cooperative_groups;

__device__ inline int bitrev(int x, int logn) { return (int)(__brev((unsigned)x) >> (32 - logn)); }

// Transform W real lines of length n held in `data` (global), in place.
// CONTIG: lines are contiguous (z) with consecutive lines nz apart;
// otherwise positions are `pstride` apart and consecutive lines adjacent (y).
template <class T, bool CONTIG>
__global__ void __launch_bounds__(256)
k_dht(T* __restrict__ data, int n, int logn, int W, int lines_per_group, size_t group_stride,
      size_t pstride, const T* __restrict__ tw) {
  using C2 = typename Vec2<T>::type;
  extern __shared__ unsigned char smem_raw[];
  C2* Z = reinterpret_cast<C2*>(smem_raw);   // [W/2][n]
  const int groups_per_outer = lines_per_group / W;
  const int outer = blockIdx.x / groups_per_outer;
  const int g = blockIdx.x - outer * groups_per_outer;
  T* base = data + (size_t)outer * group_stride + (size_t)g * W * (CONTIG ? (size_t)n : (size_t)1);
  const int tot = W * n;
  // load with bit reversal, pairing lines (2q, 2q+1) as (re, im) of complex line q
  for (int e = threadIdx.x; e < tot; e += blockDim.x) {
    int l, j;
    size_t gi;
    if (CONTIG) {
      l = e / n;
      j = e - l * n;
      gi = (size_t)l * n + j;
    } else {
      j = e / W;
      l = e - j * W;
      gi = (size_t)j * pstride + l;
    }
    const T val = base[gi];
    C2* zz = Z + (size_t)(l >> 1) * n + bitrev(j, logn);
    if (l & 1) zz->y = val; else zz->x = val;
  }
  __syncthreads();
  const int half = n >> 1;
  const int nb = (W >> 1) * half;
  for (int m = 1; m < n; m <<= 1) {
    const int tstep = n / (2 * m);
    for (int t = threadIdx.x; t < nb; t += blockDim.x) {
      const int q = t / half;
      const int b = t - q * half;
      const int pos = b & (m - 1);
      const int i1 = ((b - pos) << 1) + pos;
      const int i2 = i1 + m;
      C2* zq = Z + (size_t)q * n;
      const C2 wv = reinterpret_cast<const C2*>(tw)[pos * tstep];
      const C2 a = zq[i1], c = zq[i2];
      const T br = c.x * wv.x - c.y * wv.y;
      const T bi = c.x * wv.y + c.y * wv.x;
      zq[i1] = C2{a.x + br, a.y + bi};
      zq[i2] = C2{a.x - br, a.y - bi};
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < tot; e += blockDim.x) {
    int l, j;
    size_t gi;
    if (CONTIG) {
      l = e / n;
      j = e - l * n;
      gi = (size_t)l * n + j;
    } else {
      j = e / W;
      l = e - j * W;
      gi = (size_t)j * pstride + l;
    }
    const C2* zq = Z + (size_t)(l >> 1) * n;
    const C2 zk = zq[j];
    const C2 zr = zq[j == 0 ? 0 : n - j];
    const T hv = (l & 1) ? (zk.x + zk.y - zr.x + zr.y) : (zk.x - zk.y + zr.x + zr.y);
    base[gi] = (T)0.5 * hv;
  }
}

// ---- transforms in registers
template <class T>
struct Cx {
  T r, i;
};
template <class T>
__device__ inline Cx<T> cmul(Cx<T> a, Cx<T> b) {
  return {a.r * b.r - a.i * b.i, a.r * b.i + a.i * b.r};
}

// in-register 8-point DFT: out[p] = sum_m in[m] W8^{m p}
template <class T>
__device__ inline void dft8(Cx<T> (&x)[8]) {
  const T s = (T)0.70710678118654752440;
  // radix-2 DIF stages (distance 4, 2, 1), outputs bit-reversed, then reorder
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const Cx<T> a = x[m], b = x[m + 4];
    x[m] = {a.r + b.r, a.i + b.i};
    Cx<T> d = {a.r - b.r, a.i - b.i};
    // twiddle W8^m
    if (m == 1) d = {s * (d.r + d.i), s * (d.i - d.r)};
    if (m == 2) d = {d.i, -d.r};
    if (m == 3) d = {s * (d.i - d.r), -s * (d.r + d.i)};
    x[m + 4] = d;
  }
#pragma unroll
  for (int g = 0; g < 8; g += 4)
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      const Cx<T> a = x[g + m], b = x[g + m + 2];
      x[g + m] = {a.r + b.r, a.i + b.i};
      Cx<T> d = {a.r - b.r, a.i - b.i};
      if (m == 1) d = {d.i, -d.r};   // W4^1 = -i
      x[g + m + 2] = d;
    }
#pragma unroll
  for (int g = 0; g < 8; g += 2) {
    const Cx<T> a = x[g], b = x[g + 1];
    x[g] = {a.r + b.r, a.i + b.i};
    x[g + 1] = {a.r - b.r, a.i - b.i};
  }
  // bit-reversed (3 bits) -> natural order
  Cx<T> t = x[1];
  x[1] = x[4];
  x[4] = t;
  t = x[3];
  x[3] = x[6];
  x[6] = t;
}

template <class T>
__device__ inline void load_twiddles(Cx<T>* tw, const T* g) {
  for (int t = threadIdx.x; t < 128; t += blockDim.x) {
    tw[t] = {g[2 * t], g[2 * t + 1]};
    tw[t + 128] = {-g[2 * t], -g[2 * t + 1]};   // W^{t+128} = -W^t
  }
  __syncthreads();
}

// ---- FP32: both transforms of a 256 x 256 plane with thread-level radix-16
// FFTs. Four-step form N = 16 x 16 with n = j0 + 16 m, k = k1 + 16 k2:
//   Z(k1 + 16 k2) = sum_j0 W16^{j0 k2} W256^{j0 k1} sum_m z(j0 + 16 m) W16^{m k1}.
// A thread holds the 16 values m of one j0 in registers, runs the inner
// 16-point DFT there, applies W256^{j0 k1} and hands its outputs through one
// shared-memory transpose to the thread that owns k1; that thread runs the
// outer 16-point DFT over j0. No shuffles; every shared-memory access is a
// warp-contiguous row. Two real lines travel as z = a + i b and are
// separated with the Hartley identities of the file header, each thread
// producing the outputs k and N - k from the same two values.
//
// A cluster of four CTAs owns a plane (input and output planes may be the
// same or distinct). Phase y: CTA q transforms columns
// 64 q .. 64 q + 63 (complex pairs (64 q + p, 64 q + 32 + p)) along y,
// loading straight from global memory (lanes along z, coalesced), and
// stores the result in a permuted order inside the plane,
//   element (row r, column z) -> r/64 * 16384 + z/16 * 1024 + z%16 * 64 + (r/32)%2 * 32 + r%32,
// so that phase z finds its inputs (the 16 values m of one j0, for 32 row
// pairs across the lanes) as coalesced 128-byte rows. That region of the
// plane is read back from L2 at once. The permuted stores of one CTA land in
// every quarter of the plane, so in place the cluster waits until every CTA
// has consumed its phase-y loads before anyone stores (split barrier, hidden
// behind the transpose), and in every case again before phase z loads. Phase z: CTA q
// transforms rows 64 q .. 64 q + 63 (pairs (64 q + p, 64 q + 32 + p)) along
// z and stores them in natural order; the permuted block it reads is the
// block it overwrites, so no barrier follows. Plane read and written once in
// HBM; 64 bytes of shared-memory traffic per complex value.
constexpr int R16_CLUSTER = 4;
constexpr int R16_THREADS = 512;
constexpr int R16_ROW = 257;   // complex stride of the separation buffer [32][257]
constexpr size_t R16_SMEM = (size_t)32 * R16_ROW * sizeof(Cx<float>);   // >= the transpose's 16 x 16 x 32

template <class T>
__device__ __forceinline__ void dft4_cx(Cx<T>& a0, Cx<T>& a1, Cx<T>& a2, Cx<T>& a3) {
  const Cx<T> t0 = {a0.r + a2.r, a0.i + a2.i}, t1 = {a0.r - a2.r, a0.i - a2.i};
  const Cx<T> t2 = {a1.r + a3.r, a1.i + a3.i}, t3 = {a1.r - a3.r, a1.i - a3.i};
  a0 = {t0.r + t2.r, t0.i + t2.i};
  a2 = {t0.r - t2.r, t0.i - t2.i};
  a1 = {t1.r + t3.i, t1.i - t3.r};   // t1 - i t3
  a3 = {t1.r - t3.i, t1.i + t3.r};   // t1 + i t3
}

// (a + i b) W16^e for the exponents e = n2 k1 of the 4 x 4 split
template <class T>
__device__ __forceinline__ Cx<T> w16(Cx<T> a, int e) {
  const T C = (T)0.92387953251128675613, S = (T)0.38268343236508977173, R = (T)0.70710678118654752440;
  switch (e) {
    case 1: return {a.r * C + a.i * S, a.i * C - a.r * S};
    case 2: return {(a.r + a.i) * R, (a.i - a.r) * R};
    case 3: return {a.r * S + a.i * C, a.i * S - a.r * C};
    case 4: return {a.i, -a.r};
    case 6: return {(a.i - a.r) * R, -(a.r + a.i) * R};
    case 9: return {-a.r * C - a.i * S, a.r * S - a.i * C};
    default: return a;
  }
}

// in-register 16-point DFT, natural order in and out: n = 4 n1 + n2,
// k = k1 + 4 k2, a 4-point DFT over n1, twiddles W16^{n2 k1}, a 4-point DFT
// over n2
template <class T>
__device__ __forceinline__ void dft16(Cx<T> (&x)[16]) {
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) dft4_cx(x[n2], x[4 + n2], x[8 + n2], x[12 + n2]);
#pragma unroll
  for (int k1 = 1; k1 < 4; ++k1)
#pragma unroll
    for (int n2 = 1; n2 < 4; ++n2) x[4 * k1 + n2] = w16(x[4 * k1 + n2], n2 * k1);
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) dft4_cx(x[4 * k1], x[4 * k1 + 1], x[4 * k1 + 2], x[4 * k1 + 3]);
  // slot 4 k1 + k2 holds Z(k1 + 4 k2): transpose the 4 x 4 index
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = a + 1; b < 4; ++b) {
      const Cx<T> t = x[4 * a + b];
      x[4 * a + b] = x[4 * b + a];
      x[4 * b + a] = t;
    }
}

__device__ __forceinline__ int r16_perm(int row, int z) {
  return (row >> 6) * 16384 + (z >> 4) * 1024 + (z & 15) * 64 + ((row >> 5) & 1) * 32 + (row & 31);
}

__device__ __forceinline__ void cluster_arrive_release() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait_acquire() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Inner DFT of the thread's 16 values, the W256^{j0 k1} twiddles, the
// transpose, and the outer DFT: on return x[k2] = Z(k1 + 16 k2) of the lane's
// line pair, k1 = the warp index. `pre_wait` runs between the transpose's
// stores and loads (the cluster arrive of phase y).
template <class T, class F>
__device__ __forceinline__ void r16_fft(Cx<T> (&x)[16], const Cx<T>* tw, Cx<T>* buf, int w, int l,
                                        F pre_wait) {
  dft16(x);
#pragma unroll
  for (int k1 = 0; k1 < 16; ++k1) buf[(k1 * 16 + w) * 32 + l] = k1 ? cmul(x[k1], tw[w * k1]) : x[0];   // w k1 <= 225
  pre_wait();
  __syncthreads();
#pragma unroll
  for (int j0 = 0; j0 < 16; ++j0) x[j0] = buf[(w * 16 + j0) * 32 + l];
  dft16(x);
  __syncthreads();   // the transpose buffer is free for the separation buffer
}

// the mirrored pair of a separation: Z_k and Z_{N-k} give the Hartley values
// k and N - k of both packed lines (times two) from four sums
template <class T>
struct Sep {
  T ak, bk, am, bm;   // lines a, b at k, then at N - k
};
template <class T>
__device__ __forceinline__ Sep<T> separate(Cx<T> zk, Cx<T> zm) {
  const T sr = zk.r + zm.r, dr = zk.r - zm.r, si = zk.i + zm.i, di = zk.i - zm.i;
  return {sr - di, si + dr, sr + di, si - dr};
}
// k = 0 and N / 2 are their own mirrors; z0, zh their values: a, b at 0, then at N / 2
template <class T>
__device__ __forceinline__ Sep<T> separate_ends(Cx<T> z0, Cx<T> zh) {
  return {z0.r + z0.r, z0.i + z0.i, zh.r + zh.r, zh.i + zh.i};
}

__global__ void __cluster_dims__(R16_CLUSTER, 1, 1) __launch_bounds__(R16_THREADS, 2)
k_dht2d_r16(const float* in, float* out, const float* __restrict__ twy) {
  grid_ready(in, out);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Cx<float> tw[256];
  Cx<float>* buf = reinterpret_cast<Cx<float>*>(smem_raw);
  const int q = (int)(blockIdx.x % R16_CLUSTER);   // rank in the cluster (clusters are consecutive blocks)
  const size_t plane = (size_t)(blockIdx.x / R16_CLUSTER) * 65536;
  float* P = out + plane;
  const bool inplace = in == out;   // the same for the whole grid
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  Cx<float> x[16];
  // ---- phase y: columns (64 q + l, 64 q + 32 + l), rows w + 16 m
  {
    const float* col = in + plane + 64 * q + l;
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      const int r = w + 16 * m;
      x[m] = {__ldcg(col + r * 256), __ldcg(col + r * 256 + 32)};
    }
  }
  load_twiddles(tw, twy);   // includes __syncthreads
  r16_fft(x, tw, buf, w, l, [inplace] {
    if (inplace) cluster_arrive_release();   // every phase-y load consumed
  });
#pragma unroll
  for (int k2 = 0; k2 < 16; ++k2) buf[l * R16_ROW + w + 16 * k2] = x[k2];
  __syncthreads();
  if (inplace) cluster_wait_acquire();   // no CTA still needs an original value of this plane
#pragma unroll
  for (int pp = 0; pp < 2; ++pp) {
    const int p = 2 * w + pp;
    const Cx<float>* Zp = buf + p * R16_ROW;
    const int za = 64 * q + p, zb = za + 32;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int k = l + 32 * v;
      const int kr = k == 0 ? 128 : 256 - k;   // k = 0 and 128 are their own mirrors
      const Cx<float> zk = Zp[k], zr = Zp[kr];
      const Sep<float> o = k == 0 ? separate_ends(zk, zr) : separate(zk, zr);
      P[r16_perm(k, za)] = o.ak;
      P[r16_perm(k, zb)] = o.bk;
      P[r16_perm(kr, za)] = o.am;
      P[r16_perm(kr, zb)] = o.bm;
    }
  }
  cluster_arrive_release();
  cluster_wait_acquire();   // the whole plane holds the y transform (permuted)
  // ---- phase z: rows (64 q + l, 64 q + 32 + l), columns w + 16 m
  {
    const float* blk = P + q * 16384 + w * 64 + l;
#pragma unroll
    for (int m = 0; m < 16; ++m) x[m] = {__ldcg(blk + m * 1024), __ldcg(blk + m * 1024 + 32)};
  }
  r16_fft(x, tw, buf, w, l, [] {});
#pragma unroll
  for (int k2 = 0; k2 < 16; ++k2) buf[l * R16_ROW + w + 16 * k2] = x[k2];
  __syncthreads();
#pragma unroll
  for (int pp = 0; pp < 2; ++pp) {
    const int p = 2 * w + pp;
    const Cx<float>* Zp = buf + p * R16_ROW;
    float* ra = P + (size_t)(64 * q + p) * 256;
    float* rb = ra + 32 * 256;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int k = l + 32 * v;
      const int kr = k == 0 ? 128 : 256 - k;
      const Cx<float> zk = Zp[k], zr = Zp[kr];
      const Sep<float> o = k == 0 ? separate_ends(zk, zr) : separate(zk, zr);
      ra[k] = 0.25f * o.ak;   // a half for each direction's separation
      rb[k] = 0.25f * o.bk;
      ra[kr] = 0.25f * o.am;
      rb[kr] = 0.25f * o.bm;
    }
  }
}


// ---- one direction, lines of 4 to 256 points (FP64 always; FP32 beyond the planes below)
// A CTA transforms 2 P real lines as P complex ones, N = R1 R2 with radices up
// to 16: R1-point DFTs of the elements j0 + R2 m in registers, twiddles
// W^{j0 k1}, R2-point DFTs over j0 after one trip through shared memory, and
// the separation on the way back to global memory. Two barriers where the
// radix-2 form (k_dht) has log2 N + 1. In FP64 the transforms are bound by the
// FP64 pipe (two instructions per clock and SM): about 12 instructions per
// value and direction plus two for the separation, against 18 to 24 of k_dht
// and of the warp-level 256-point form that was here; the blocks are small, so
// several share an SM and all SMs get the same number. FP64, y + z: 512 planes of
// 256 x 256 2.26 -> 1.88 ms, 256 of 128 x 128 0.344 -> 0.230; 1.75 since the
// separation leaves its factor of two to the x solve.
template <class T, int R>
__device__ __forceinline__ void dft_r(Cx<T> (&x)[R]) {
  if constexpr (R == 16) dft16(x);
  else if constexpr (R == 8) dft8(x);
  else if constexpr (R == 4) dft4_cx(x[0], x[1], x[2], x[3]);
}
constexpr int DHT1_PAIRS = 16;
// the separation's values are twice the transform's. FP64 leaves the factor in
// (one instruction in 14.4 per value on the pipe that bounds the kernels); the
// x solve's right-hand side takes it out (poisson_rhs_scale), exactly
template <class T>
__device__ __forceinline__ T dht1_norm(T v) {
  return sizeof(T) == 8 ? v : (T)0.5 * v;
}
// y: columns of a plane (positions nz apart); pairs (c, c + P) of a tile of 2 P columns
template <class T, int R1, int R2>
__global__ void __launch_bounds__(256, 2) k_dht1_y(T* __restrict__ data, int nz, int P, const T* __restrict__ twg) {
  grid_ready(data);
  constexpr int N = R1 * R2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Cx<T>* S = reinterpret_cast<Cx<T>*>(smem_raw);   // [N][P], wavenumber k1 + R1 k2 at row k1 R2 + k2
  Cx<T>* tw = S + N * P;
  const int tiles = nz / (2 * P), lp = 31 - __clz(P);
  const int pl = blockIdx.x / tiles;
  T* base = data + (size_t)pl * N * nz + (size_t)(blockIdx.x - pl * tiles) * 2 * P;
  for (int q = threadIdx.x; q < N / 2; q += blockDim.x) {
    tw[q] = {twg[2 * q], twg[2 * q + 1]};
    tw[q + N / 2] = {-twg[2 * q], -twg[2 * q + 1]};
  }
  __syncthreads();
  for (int q = threadIdx.x; q < P * R2; q += blockDim.x) {
    const int c = q & (P - 1), j0 = q >> lp;
    const T* col = base + (size_t)j0 * nz + c;
    Cx<T> x[R1];
#pragma unroll
    for (int m = 0; m < R1; ++m) x[m] = {col[(size_t)(m * R2) * nz], col[(size_t)(m * R2) * nz + P]};
    dft_r<T, R1>(x);
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) S[(j0 + R2 * k1) * P + c] = k1 && j0 ? cmul(x[k1], tw[j0 * k1]) : x[k1];
  }
  __syncthreads();
  if constexpr (R2 > 1) {
    for (int q = threadIdx.x; q < P * R1; q += blockDim.x) {
      Cx<T>* s = S + (q >> lp) * R2 * P + (q & (P - 1));
      Cx<T> x[R2];
#pragma unroll
      for (int j = 0; j < R2; ++j) x[j] = s[j * P];
      dft_r<T, R2>(x);
#pragma unroll
      for (int j = 0; j < R2; ++j) s[j * P] = x[j];
    }
    __syncthreads();
  }
  for (int q = threadIdx.x; q < P * (N / 2); q += blockDim.x) {
    const int c = q & (P - 1), k = q >> lp, km = k ? N - k : N / 2;
    const Cx<T> zk = S[((k % R1) * R2 + k / R1) * P + c], zm = S[((km % R1) * R2 + km / R1) * P + c];
    const Sep<T> o = k ? separate(zk, zm) : separate_ends(zk, zm);
    T* a = base + (size_t)k * nz + c;
    T* b = base + (size_t)km * nz + c;
    a[0] = dht1_norm<T>(o.ak);
    a[P] = dht1_norm<T>(o.bk);
    b[0] = dht1_norm<T>(o.am);
    b[P] = dht1_norm<T>(o.bm);
  }
}
// z: contiguous lines; pairs (r, r + P) of 2 P consecutive rows
template <class T, int R1, int R2>
__global__ void __launch_bounds__(256, 2) k_dht1_z(T* __restrict__ data, int P, const T* __restrict__ twg) {
  grid_ready(data);
  constexpr int N = R1 * R2;
  constexpr int LD = N + (R2 > 1 ? R1 : 1);   // one slot of padding per R2
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Cx<T>* S = reinterpret_cast<Cx<T>*>(smem_raw);   // [P][LD], position p at p + p / R2
  Cx<T>* tw = S + LD * P;
  T* base = data + (size_t)blockIdx.x * 2 * P * N;
  auto at = [](int p) { return R2 > 1 ? p + p / R2 : p; };
  for (int q = threadIdx.x; q < N / 2; q += blockDim.x) {
    tw[q] = {twg[2 * q], twg[2 * q + 1]};
    tw[q + N / 2] = {-twg[2 * q], -twg[2 * q + 1]};
  }
  __syncthreads();
  for (int q = threadIdx.x; q < P * R2; q += blockDim.x) {
    const int j0 = q % R2, r = q / R2;
    const T* row = base + (size_t)r * N + j0;
    Cx<T> x[R1];
#pragma unroll
    for (int m = 0; m < R1; ++m) x[m] = {row[m * R2], row[(size_t)P * N + m * R2]};
    dft_r<T, R1>(x);
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) S[r * LD + at(j0 + R2 * k1)] = k1 && j0 ? cmul(x[k1], tw[j0 * k1]) : x[k1];
  }
  __syncthreads();
  if constexpr (R2 > 1) {
    for (int q = threadIdx.x; q < P * R1; q += blockDim.x) {
      Cx<T>* s = S + (q / R1) * LD + (q % R1) * (R2 + 1);
      Cx<T> x[R2];
#pragma unroll
      for (int j = 0; j < R2; ++j) x[j] = s[j];
      dft_r<T, R2>(x);
#pragma unroll
      for (int j = 0; j < R2; ++j) s[j] = x[j];
    }
    __syncthreads();
  }
  for (int q = threadIdx.x; q < P * (N / 2); q += blockDim.x) {
    const int k = q % (N / 2), r = q / (N / 2), km = k ? N - k : N / 2;
    const Cx<T> zk = S[r * LD + at((k % R1) * R2 + k / R1)], zm = S[r * LD + at((km % R1) * R2 + km / R1)];
    const Sep<T> o = k ? separate(zk, zm) : separate_ends(zk, zm);
    T* a = base + (size_t)r * N;
    T* b = a + (size_t)P * N;
    a[k] = dht1_norm<T>(o.ak);
    b[k] = dht1_norm<T>(o.bk);
    a[km] = dht1_norm<T>(o.am);
    b[km] = dht1_norm<T>(o.bm);
  }
}
// calls f with the radices of an n-point line as integral constants; false beyond 256 points
template <class F>
static bool with_radices(int n, F f) {
  using std::integral_constant;
  switch (n) {
    case 4: f(integral_constant<int, 4>(), integral_constant<int, 1>()); return true;
    case 8: f(integral_constant<int, 8>(), integral_constant<int, 1>()); return true;
    case 16: f(integral_constant<int, 16>(), integral_constant<int, 1>()); return true;
    case 32: f(integral_constant<int, 8>(), integral_constant<int, 4>()); return true;
    case 64: f(integral_constant<int, 8>(), integral_constant<int, 8>()); return true;
    case 128: f(integral_constant<int, 16>(), integral_constant<int, 8>()); return true;
    case 256: f(integral_constant<int, 16>(), integral_constant<int, 16>()); return true;
    default: return false;
  }
}
static int dht1_threads(int P, int r) { return std::max(32, P * r); }
// line pairs per block: 16 (whole 128-byte lines of FP64 columns), fewer where
// that leaves under four blocks per SM
static int dht1_pairs(long long pairs, int most) {
  int P = std::min(DHT1_PAIRS, most);
  while (P > 4 && pairs / P < 4 * 152) P /= 2;
  return P;
}

// ---- FP32: both transforms of planes that fit one SM's shared memory, one CTA per plane
// The separate kernels read and write the field twice per transform. Here a
// CTA holds the plane as complex column pairs (c, c + nz/2) in shared memory
// and every pass is an R-point DFT in registers, N = R1 R2, in place (a thread
// stores to the slots it loaded), so both directions take four passes and
// barriers:
//   y1: from global memory, rows j0 + R2 m -> W^{j0 k1} -> rows j0 + R2 k1
//   y2: rows k1 R2 + j0; wavenumber ky = k1 + R1 k2 ends at row k1 R2 + k2
//   z1: the packed rows of the z transform are ky and ny - ky, so the
//       separation of the y transform needs only Z_ky and Z_{ny-ky} of a
//       column pair, both at hand; column position p < nz/2 of row pair
//       (ky, ny - ky) lives in slot (row of ky, p), p >= nz/2 in (row of
//       ny - ky, p - nz/2), which are the slots the thread read
//   z2, then the separation of the row pairs on the way to global memory.
// Columns are padded by one slot per R2 of the z direction (conflict-free
// strides in z1, z2 and the last pass). Bound by shared memory and latency;
// sizes are template parameters, because index arithmetic on run-time strides
// cost a third of the time. 256 planes of 128 x 128: 0.072 (y, z) -> 0.014 ms.
template <int R1Y, int R2Y, int R1Z, int R2Z>
struct PlaneSize {
  static constexpr int NY = R1Y * R2Y, NZ = R1Z * R2Z, NZH = NZ / 2;
  static constexpr int LD = NZH + (R2Z > 1 ? NZH / R2Z : 0);
  static constexpr int THREADS = NZH * R2Y < 64 ? 64 : NZH * R2Y > 512 ? 512 : NZH * R2Y;   // one item of y1 each
  static constexpr size_t SMEM = ((size_t)NY * LD + NY + NZ) * sizeof(Cx<float>);
  static constexpr bool FITS = SMEM <= 200 * 1024;
};
template <int R1Y, int R2Y, int R1Z, int R2Z>
__global__ void __launch_bounds__((PlaneSize<R1Y, R2Y, R1Z, R2Z>::THREADS), (PlaneSize<R1Y, R2Y, R1Z, R2Z>::THREADS == 512 ? 2 : 1))
k_dht2d_plane(const float* in, float* out, const float* __restrict__ twy, const float* __restrict__ twz) {
  grid_ready(in, out);
  using G = PlaneSize<R1Y, R2Y, R1Z, R2Z>;
  using C = Cx<float>;
  constexpr int NY = G::NY, NZ = G::NZ, NZH = G::NZH, LD = G::LD, TH = G::THREADS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* S = reinterpret_cast<C*>(smem_raw);
  C* ty = S + NY * LD;
  C* tz = ty + NY;
  in += (size_t)blockIdx.x * NY * NZ;
  out += (size_t)blockIdx.x * NY * NZ;
  auto col = [](int c) { return R2Z > 1 ? c + c / R2Z : c; };
  // row slots of wavenumber pair rp: ky = rp and ny - rp (0 and ny / 2 for rp = 0)
  auto rows = [&](int rp, C*& a, C*& b) {
    const int kb = rp ? NY - rp : NY / 2;
    a = S + ((rp % R1Y) * R2Y + rp / R1Y) * LD;
    b = S + ((kb % R1Y) * R2Y + kb / R1Y) * LD;
  };
  const int tid = threadIdx.x;
  // the first pass's loads are issued before the twiddle tables are filled
  for (int q0 = 0; q0 < NZH * R2Y; q0 += TH) {
    const int q = q0 + tid, c = q % NZH, j0 = q / NZH;
    const bool on = NZH * R2Y % TH == 0 || q < NZH * R2Y;
    C x[R1Y];
    if (on) {
      const float* p = in + j0 * NZ + c;
#pragma unroll
      for (int m = 0; m < R1Y; ++m) x[m] = {__ldcg(p + m * R2Y * NZ), __ldcg(p + m * R2Y * NZ + NZH)};
    }
    if (q0 == 0) {
      for (int t = tid; t < NY / 2; t += TH) {
        ty[t] = {twy[2 * t], twy[2 * t + 1]};
        ty[t + NY / 2] = {-twy[2 * t], -twy[2 * t + 1]};
      }
      for (int t = tid; t < NZ / 2; t += TH) {
        tz[t] = {twz[2 * t], twz[2 * t + 1]};
        tz[t + NZ / 2] = {-twz[2 * t], -twz[2 * t + 1]};
      }
      __syncthreads();
    }
    if (on) {
      dft_r<float, R1Y>(x);
      C* s = S + j0 * LD + col(c);
#pragma unroll
      for (int k1 = 0; k1 < R1Y; ++k1) s[k1 * R2Y * LD] = R2Y > 1 && k1 ? cmul(x[k1], ty[j0 * k1]) : x[k1];
    }
  }
  __syncthreads();
  if constexpr (R2Y > 1) {
    for (int q = tid; q < NZH * R1Y; q += TH) {
      C* s = S + (q / NZH) * R2Y * LD + col(q % NZH);
      C x[R2Y];
#pragma unroll
      for (int j = 0; j < R2Y; ++j) x[j] = s[j * LD];
      dft_r<float, R2Y>(x);
#pragma unroll
      for (int j = 0; j < R2Y; ++j) s[j * LD] = x[j];
    }
    __syncthreads();
  }
  for (int q = tid; q < (NY / 2) * R2Z; q += TH) {
    const int j0 = q % R2Z, rp = q / R2Z;
    C *a, *b;
    rows(rp, a, b);
    C x[R1Z];
#pragma unroll
    for (int m = 0; m < R1Z / 2; ++m) {
      const int c = col(j0 + m * R2Z);
      const C za = a[c], zb = b[c];
      const Sep<float> o = rp ? separate(za, zb) : separate_ends(za, zb);
      x[m] = {o.ak, o.am};              // column c of rows ky, ny - ky
      x[m + R1Z / 2] = {o.bk, o.bm};    // column c + nz / 2
    }
    dft_r<float, R1Z>(x);
#pragma unroll
    for (int k1 = 0; k1 < R1Z; ++k1)
      (k1 < R1Z / 2 ? a : b)[col(j0 + (k1 % (R1Z / 2)) * R2Z)] = R2Z > 1 && k1 ? cmul(x[k1], tz[j0 * k1]) : x[k1];
  }
  __syncthreads();
  if constexpr (R2Z > 1) {
    for (int q = tid; q < (NY / 2) * R1Z; q += TH) {
      const int k1 = q % R1Z;
      C *a, *b;
      rows(q / R1Z, a, b);
      C* s = (k1 < R1Z / 2 ? a : b) + (k1 % (R1Z / 2)) * (R2Z + 1);
      C x[R2Z];
#pragma unroll
      for (int j = 0; j < R2Z; ++j) x[j] = s[j];
      dft_r<float, R2Z>(x);
#pragma unroll
      for (int j = 0; j < R2Z; ++j) s[j] = x[j];
    }
    __syncthreads();
  }
  for (int q = tid; q < (NY / 2) * NZH; q += TH) {
    const int k = q % NZH, rp = q / NZH, km = k ? NZ - k : NZH;
    C *a, *b;
    rows(rp, a, b);
    const int pk = (k % R1Z) * R2Z + k / R1Z, pm = (km % R1Z) * R2Z + km / R1Z;
    const C zk = (pk < NZH ? a : b)[col(pk % NZH)], zm = (pm < NZH ? a : b)[col(pm % NZH)];
    const Sep<float> o = k ? separate(zk, zm) : separate_ends(zk, zm);
    float* ra = out + rp * NZ;
    float* rb = out + (rp ? NY - rp : NY / 2) * NZ;
    ra[k] = 0.25f * o.ak;   // a half for each direction's separation
    rb[k] = 0.25f * o.bk;
    ra[km] = 0.25f * o.am;
    rb[km] = 0.25f * o.bm;
  }
}
// calls f with the PlaneSize of ny x nz planes; false where there is none that fits
template <class F>
static bool with_plane(int ny, int nz, F f) {
  bool fits = false;
  const bool known = with_radices(ny, [&](auto r1y, auto r2y) {
    fits = with_radices(nz, [&](auto r1z, auto r2z) {
      using G = PlaneSize<decltype(r1y)::value, decltype(r2y)::value, decltype(r1z)::value, decltype(r2z)::value>;
      if constexpr (G::FITS)
        f(G(), k_dht2d_plane<decltype(r1y)::value, decltype(r2y)::value, decltype(r1z)::value, decltype(r2z)::value>);
    });
  });
  return known && fits && !(ny == 256 && nz == 256);
}
bool dht2d_plane_supported(int ny, int nz) {
  return with_plane(ny, nz, [](auto, auto) {});
}

// Thomas solve along x per mode; rhs scaled by h^2 / (ny nz) (Hartley
// normalisation). One thread per mode walks x (coalesced across modes) in
// chunks of PF planes; the loads of the next chunk (right-hand side and
// inverse pivots) are issued before the current chunk's recursion, so each
// thread keeps up to 4 PF independent loads in flight. Past the row from
// which a mode's stored pivots equal their limit (a few rows for all but
// the lowest modes) the limit stays in a register and the chunks carry
// right-hand sides only, twice as many per chunk in FP32.
constexpr int PF = 16;
__host__ __device__ inline size_t ptab_plane(const Consts& c) {
  return (size_t)(c.ny / 2 + 1) * (c.nz / 2 + 1);
}
__device__ inline size_t ptab_index(const Consts& c, int jk) {
  const int ky = jk / c.nz, kz = jk - ky * c.nz;
  const int qy = ky <= c.ny / 2 ? ky : c.ny - ky, qz = kz <= c.nz / 2 ? kz : c.nz - kz;
  return (size_t)qy * (c.nz / 2 + 1) + qz;
}

// storage conversions: FP32 / FP64 fields, or bfloat16 (the mixed solve's correction)
template <class T, class S>
__device__ inline T from_store(S v) {
  if constexpr (std::is_same<S, __nv_bfloat16>::value) return __bfloat162float(v);
  else return (T)v;
}
template <class S, class T>
__device__ inline S to_store(T v) {
  if constexpr (std::is_same<S, __nv_bfloat16>::value) return __float2bfloat16_rn(v);
  else return (S)v;
}

// forward elimination over planes [i0, i1) in chunks of N planes, the next
// chunk's loads issued before the current chunk's recursion (two chunks in
// flight); TAB: inverse pivots from the table, else the converged limit
template <int N, bool TAB, class T, class LDF, class STF>
__device__ __forceinline__ void px_forward(LDF LD, STF ST, const T* iv, size_t PT, int P, T lim, T scale,
                                           bool zero_mode, int i0, int i1, T& y) {
  constexpr int NT = TAB ? N : 1;
  const int nch = (i1 - i0) / N;
  T rd[N], rt[NT];
  if (nch > 0) {
#pragma unroll
    for (int q = 0; q < N; ++q) {
      rd[q] = LD((size_t)(i0 + q) * P);
      if constexpr (TAB) rt[q] = iv[(size_t)(i0 + q) * PT];
    }
  }
  int i = i0;
  for (int ch = 0; ch < nch; ++ch, i += N) {
    T nd[N], nt[NT];
    if (ch + 1 < nch) {
#pragma unroll
      for (int q = 0; q < N; ++q) {
        nd[q] = LD((size_t)(i + N + q) * P);
        if constexpr (TAB) nt[q] = iv[(size_t)(i + N + q) * PT];
      }
    }
#pragma unroll
    for (int q = 0; q < N; ++q) {
      if constexpr (TAB) {
        const T rhs = (zero_mode && i + q == 0) ? (T)0 : rd[q] * scale;
        y = (rhs - y) * rt[q];
      } else {
        y = (rd[q] * scale - y) * lim;
      }
      ST((size_t)(i + q) * P, y);
    }
#pragma unroll
    for (int q = 0; q < N; ++q) {
      rd[q] = nd[q];
      if constexpr (TAB) rt[q] = nt[q];
    }
  }
  for (; i < i1; ++i) {   // the partial chunk
    const size_t o = (size_t)i * P;
    if constexpr (TAB) {
      const T rhs = (zero_mode && i == 0) ? (T)0 : LD(o) * scale;
      y = (rhs - y) * iv[(size_t)i * PT];
    } else {
      y = (LD(o) * scale - y) * lim;
    }
    ST(o, y);
  }
}

// back substitution over planes i1 - 1 down to i0 (x holds x_{i1} on entry),
// the partial chunk first, then chunks of N as above
template <int N, bool TAB, class T, class LDF, class STF>
__device__ __forceinline__ void px_backward(LDF LD, STF ST, const T* iv, size_t PT, int P, T lim, bool zero_mode,
                                            int i0, int i1, T& x) {
  constexpr int NT = TAB ? N : 1;
  int i = i1 - 1;
  const int rem = (i1 - i0) % N;
  for (int r = 0; r < rem; ++r, --i) {
    const size_t o = (size_t)i * P;
    T cp = lim;
    if constexpr (TAB) cp = (zero_mode && i == 0) ? (T)0 : iv[(size_t)i * PT];
    x = LD(o) - cp * x;
    ST(o, x);
  }
  const int nch = (i1 - i0) / N;   // full chunks below: planes i, i - 1, ..., i0
  T rd[N], rt[NT];
  if (nch > 0) {
#pragma unroll
    for (int q = 0; q < N; ++q) {
      rd[q] = LD((size_t)(i - q) * P);
      if constexpr (TAB) rt[q] = iv[(size_t)(i - q) * PT];
    }
  }
  for (int ch = 0; ch < nch; ++ch, i -= N) {
    T nd[N], nt[NT];
    if (ch + 1 < nch) {
#pragma unroll
      for (int q = 0; q < N; ++q) {
        nd[q] = LD((size_t)(i - N - q) * P);
        if constexpr (TAB) nt[q] = iv[(size_t)(i - N - q) * PT];
      }
    }
#pragma unroll
    for (int q = 0; q < N; ++q) {
      T cp = lim;
      if constexpr (TAB) cp = (zero_mode && i - q == 0) ? (T)0 : rt[q];
      x = rd[q] - cp * x;
      ST((size_t)(i - q) * P, x);
    }
#pragma unroll
    for (int q = 0; q < N; ++q) {
      rd[q] = nd[q];
      if constexpr (TAB) rt[q] = nt[q];
    }
  }
}

// Single pass over the converged rows of modes whose converged inverse pivot
// is at most 1/2 in magnitude (FP32 arithmetic): there the back substitution
// x_j = y_j - lim x_{j+1} equals sum_k (-lim)^k y_{j+k}, and the sum after
// PW terms is below lim^PW <= 2^-24 of x, the FP32 rounding. Each chunk of PW
// rows is emitted once the next chunk's forward values exist: its last row
// from the truncated sum, the others by the exact recursion downward. The
// forward values of those rows never go to memory (read once, written once
// instead of read, written, read, written). Rows below ia (table pivots) and
// the last chunk with the remaining rows keep the stored forward values and
// the exact back substitution.
constexpr int PW = 24;
template <class T, class LDF, class STF>
__device__ __forceinline__ void px_single(LDF LD, STF ST, const T* iv, size_t PT, int P, T lim, T scale, int ia,
                                          int nx) {
  T y = 0;
  for (int i = 0; i < ia; ++i) {   // head: table pivots, forward values stored
    const size_t o = (size_t)i * P;
    y = (LD(o) * scale - y) * iv[(size_t)i * PT];
    ST(o, y);
  }
  const int nch = (nx - 1 - ia) / PW;   // >= 1 (checked by the caller)
  T yc[PW], yp[PW], nd[PW];
#pragma unroll
  for (int q = 0; q < PW; ++q) nd[q] = LD((size_t)(ia + q) * P);
  T x_ia = 0;
  for (int ch = 0; ch < nch; ++ch) {
    const int i0 = ia + ch * PW;
#pragma unroll
    for (int q = 0; q < PW; ++q) yp[q] = yc[q];
#pragma unroll
    for (int q = 0; q < PW; ++q) yc[q] = nd[q];
    if (ch + 1 < nch) {
#pragma unroll
      for (int q = 0; q < PW; ++q) nd[q] = LD((size_t)(i0 + PW + q) * P);
    }
#pragma unroll
    for (int q = 0; q < PW; ++q) {
      y = (yc[q] * scale - y) * lim;
      yc[q] = y;
    }
    if (ch > 0) {   // emit the previous chunk
      T acc = yc[PW - 2];
#pragma unroll
      for (int k = PW - 3; k >= 0; --k) acc = yc[k] - lim * acc;
      T x = yp[PW - 1] - lim * acc;
      const int j0 = i0 - PW;
      ST((size_t)(j0 + PW - 1) * P, x);
#pragma unroll
      for (int q = PW - 2; q >= 0; --q) {
        x = yp[q] - lim * x;
        ST((size_t)(j0 + q) * P, x);
      }
      if (ch == 1) x_ia = x;
    }
  }
  // tail: the last chunk's forward values, the remaining rows and the last
  // row (its own pivot) stored; exact back substitution down to the last chunk
  const int it = ia + (nch - 1) * PW;
#pragma unroll
  for (int q = 0; q < PW; ++q) ST((size_t)(it + q) * P, yc[q]);
  for (int i = it + PW; i < nx - 1; ++i) {
    const size_t o = (size_t)i * P;
    y = (LD(o) * scale - y) * lim;
    ST(o, y);
  }
  {
    const size_t o = (size_t)(nx - 1) * P;
    y = (LD(o) * scale - y) * iv[(size_t)(nx - 1) * PT];
    ST(o, y);
  }
  T x = y;
  for (int i = nx - 2; i >= it; --i) {
    const size_t o = (size_t)i * P;
    x = LD(o) - lim * x;
    ST(o, x);
  }
  if (nch == 1) x_ia = x;
  x = x_ia;   // head: exact back substitution with the table pivots
  for (int i = ia - 1; i >= 0; --i) {
    const size_t o = (size_t)i * P;
    x = LD(o) - iv[(size_t)i * PT] * x;
    ST(o, x);
  }
}

// gauge mean(phi) = 0: the first warp takes the line mean of mode (0, 0) out
// of every plane, its lanes sharing the line (a launch of its own before)
template <class T, class S>
__device__ __forceinline__ void px_mean00(S* phi, int P, int nx, int lane, unsigned warp_mask) {
  __syncwarp(warp_mask);
  const int n = __popc(warp_mask);   // 32, or 16 for 4 x 4 planes
  double sum = 0.0;
  for (int i = lane; i < nx; i += n) sum += from_store<double>(phi[(size_t)i * P]);
  for (int o = n / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(warp_mask, sum, o);
  const double mean = sum / nx;
  for (int i = lane; i < nx; i += n) {
    S& v = phi[(size_t)i * P];
    v = to_store<S>(from_store<double>(v) - mean);
  }
}

// Whole lines in shared memory: one warp per 32 modes copies its columns of
// every plane with cp.async (each instruction one coalesced row, all of them
// in flight), runs the forward sweep in place and the back substitution straight to global memory.
// A line waits for memory once, where the register form (k_poisson_x) waits
// once per chunk of 16 to 32 planes and once per plane of its partial chunks.
// For grids whose warps fit the SMs together; the low modes, whose pivots
// converge only after a hundred rows or more, set the time of a small grid.
// 16,384 modes of 256 planes FP32 0.029 -> 0.0185 ms, 1,024 of 64 FP64 0.025 ->
// 0.016.
template <class T>
__global__ void __launch_bounds__(32) k_poisson_xs(Consts c, const T* __restrict__ tab, const int* __restrict__ conv,
                                                   T* __restrict__ phi, T scale) {
  grid_ready(tab, phi);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int P = c.ny * c.nz, nx = c.nx, lane = threadIdx.x;
  const int jk = blockIdx.x * 32 + lane;
  if (jk >= P) return;
  const unsigned warp_mask = __activemask();
  T* s = reinterpret_cast<T*>(smem_raw) + lane;   // row i at s[32 i]
  T* d = phi + jk;
  {
    const uint32_t sb = smem_u32(s);
#pragma unroll 4
    for (int i = 0; i < nx; ++i)
      asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(sb + (uint32_t)(i * 32 * sizeof(T))),
                   "l"(d + (size_t)i * P), "n"(sizeof(T))
                   : "memory");
    cp_async_commit();
  }
  const size_t mi = ptab_index(c, jk);
  const T* iv = tab + mi;
  const size_t PT = ptab_plane(c);
  const bool zero_mode = jk == 0;
  const int ia = min(max(__reduce_max_sync(warp_mask, conv[mi]), 1), nx - 1);   // as in k_poisson_x
  const T lim = iv[(size_t)(nx - 2) * PT], plast = iv[(size_t)(nx - 1) * PT];
  // rows in unguarded groups of U: the group's pivots are loaded first, and a
  // lone warp's issue rate counts (about 14 instructions per row and sweep pair)
  constexpr int U = sizeof(T) == 4 ? 32 : 16;
  const T p0 = iv[0];
  const int m = nx - 1;
  cp_async_wait<0>();
  T y = zero_mode ? (T)0 : s[0] * scale * p0;
  s[0] = y;
  int i = 1;
  const T* ivi = iv + PT;
  auto table_rows = [&](auto n) {
    T p[decltype(n)::value];
#pragma unroll
    for (int q = 0; q < n; ++q) p[q] = ivi[q * PT];
#pragma unroll
    for (int q = 0; q < n; ++q) {
      y = (s[32 * (i + q)] * scale - y) * p[q];
      s[32 * (i + q)] = y;
    }
    i += n;
    ivi += n * PT;
  };
  using std::integral_constant;
  while (i + U <= ia) table_rows(integral_constant<int, U>());
  while (i + 8 <= ia) table_rows(integral_constant<int, 8>());
  while (i < ia) table_rows(integral_constant<int, 1>());
#pragma unroll 16
  for (; i < m; ++i) {
    y = (s[32 * i] * scale - y) * lim;
    s[32 * i] = y;
  }
  T x = (s[32 * m] * scale - y) * plast;
  T* di = d + (size_t)m * P;
  *di = x;
  i = m - 1;
#pragma unroll 16
  for (; i >= ia; --i) {
    x = s[32 * i] - lim * x;
    di -= P;
    *di = x;
  }
  ivi = iv + (size_t)i * PT;
  auto table_back = [&](auto n) {
    T p[decltype(n)::value];
#pragma unroll
    for (int q = 0; q < n; ++q) p[q] = *(ivi - q * PT);
#pragma unroll
    for (int q = 0; q < n; ++q) {
      x = s[32 * (i - q)] - p[q] * x;
      di -= P;
      *di = x;
    }
    i -= n;
    ivi -= n * PT;
  };
  while (i >= U) table_back(integral_constant<int, U>());
  while (i >= 8) table_back(integral_constant<int, 8>());
  while (i >= 1) table_back(integral_constant<int, 1>());
  x = s[0] - (zero_mode ? (T)0 : p0) * x;
  d[0] = x;
  if (blockIdx.x == 0) px_mean00<T>(phi, P, nx, lane, warp_mask);
}

template <class T, class S>
__global__ void __launch_bounds__(128) k_poisson_x(Consts c, const T* __restrict__ tab, const int* __restrict__ conv,
                                                   S* __restrict__ phi, T scale) {
  grid_ready(tab, phi);
  const int P = c.ny * c.nz;
  const int jk = blockIdx.x * blockDim.x + threadIdx.x;
  if (jk >= P) return;
  const unsigned warp_mask = __activemask();
  const int nx = c.nx;
  S* d = phi + jk;
  auto LD = [d](size_t o) { return from_store<T>(d[o]); };
  auto ST = [d](size_t o, T v) { d[o] = to_store<S>(v); };
  const size_t mi = ptab_index(c, jk);
  const T* iv = tab + mi;
  const size_t PT = ptab_plane(c);
  const bool zero_mode = (jk == 0);
  // planes [0, ia) take the table's pivots, [ia, nx - 1) the converged
  // limit held in a register (bitwise the table's values there), plane
  // nx - 1 its own; ia is the largest convergence row of the warp's modes,
  // so the split is warp-uniform and the converged range spends every load
  // slot on the right-hand side (chunks of PB planes)
  const int ia = min(max(__reduce_max_sync(warp_mask, conv[mi]), 1), nx - 1);
  const T lim = iv[(size_t)(nx - 2) * PT];
  if constexpr (sizeof(T) == 4) {
    // every mode of the warp decays fast enough for the single pass (never mode (0, 0))
    if (nx - 1 - ia >= PW && __all_sync(warp_mask, fabsf(lim) <= 0.5f) && !zero_mode) {
      px_single<T>(LD, ST, iv, PT, P, lim, scale, ia, nx);
      return;
    }
  }
  constexpr int PB = sizeof(T) == 8 ? PF : 2 * PF;
  T y = 0;
  px_forward<PF, true>(LD, ST, iv, PT, P, lim, scale, zero_mode, 0, ia, y);
  px_forward<PB, false>(LD, ST, iv, PT, P, lim, scale, zero_mode, ia, nx - 1, y);
  {
    const size_t o = (size_t)(nx - 1) * P;
    y = (LD(o) * scale - y) * iv[(size_t)(nx - 1) * PT];
    ST(o, y);
  }
  T x = y;  // x_{nx-1} = dp_{nx-1}
  px_backward<PB, false>(LD, ST, iv, PT, P, lim, zero_mode, ia, nx - 1, x);
  px_backward<PF, true>(LD, ST, iv, PT, P, lim, zero_mode, 0, ia, x);
  if (jk < 32) px_mean00<T>(phi, P, nx, jk, warp_mask);
}

// inverse pivots 1 / (diag_i - c'_{i-1}) of every distinct mode, FP64 arithmetic
template <class T>
__global__ void k_poisson_table(Consts c, T* __restrict__ tab, int* __restrict__ conv) {
  const int qz_n = c.nz / 2 + 1;
  const int PT = (c.ny / 2 + 1) * qz_n;
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= PT) return;
  const int ky = m / qz_n, kz = m - ky * qz_n;
  const double sy = sin(M_PI * ky / c.ny), sz = sin(M_PI * kz / c.nz);
  const double lam = -4.0 * sy * sy - 4.0 * sz * sz;
  const bool pinned = (m == 0);
  const int nx = c.nx;
  double cp = 0.0;
  for (int i = 0; i < nx; ++i) {
    double diag = (i == 0 || i == nx - 1) ? -1.0 + lam : -2.0 + lam;
    double lower = i == 0 ? 0.0 : 1.0;
    if (pinned && i == 0) diag = 1.0;              // pinned phi_0 = 0
    const double prev_cp = (pinned && i == 1) ? 0.0 : cp;
    const double denom = diag - lower * prev_cp;
    const double inv = 1.0 / denom;
    tab[(size_t)i * PT + m] = (T)inv;
    cp = inv;  // upper = 1
  }
  // rows 1 .. nx - 2 share one recursion whose pivots converge to a limit;
  // the first row from which the stored pivots equal the stored limit
  const T lim = tab[(size_t)(nx - 2) * PT + m];
  int ic = nx - 2;
  while (ic > 0 && tab[(size_t)(ic - 1) * PT + m] == lim) --ic;
  conv[m] = ic;
}

template <class T>
void launch_dht_y(const Consts& c, const Fields<T>& f, cudaStream_t s) {
  const int n = c.ny;
  if (with_radices(n, [&](auto r1, auto r2) {
        constexpr int R1 = decltype(r1)::value, R2 = decltype(r2)::value;
        const int P = dht1_pairs((long long)c.nx * c.nz / 2, c.nz / 2);
        const size_t sh = (size_t)R1 * R2 * (P + 1) * sizeof(Cx<T>);
        launch_next(k_dht1_y<T, R1, R2>, c.nx * (c.nz / (2 * P)), dht1_threads(P, std::max(R1, R2)), sh, s, f.phi, c.nz, P, f.tw_y);
      }))
    return;
  const int logn = (int)std::lround(std::log2((double)n));
  const int W = c.nz < 16 ? c.nz : 16;
  const size_t sh = (size_t)(W / 2) * n * sizeof(typename Vec2<T>::type);
  // group = one x plane; lines = nz columns; positions nz apart
  k_dht<T, false><<<c.nx * (c.nz / W), 256, sh, s>>>(f.phi, n, logn, W, c.nz, plane(c),
                                                       (size_t)c.nz, f.tw_y);
}

template <class T>
void launch_dht_z(const Consts& c, const Fields<T>& f, cudaStream_t s) {
  const int n = c.nz;
  if (with_radices(n, [&](auto r1, auto r2) {
        constexpr int R1 = decltype(r1)::value, R2 = decltype(r2)::value;
        const int P = dht1_pairs((long long)c.nx * c.ny / 2, c.ny / 2);
        const size_t sh = ((size_t)(R1 * R2 + (R2 > 1 ? R1 : 1)) * P + R1 * R2) * sizeof(Cx<T>);
        launch_next(k_dht1_z<T, R1, R2>, c.nx * (c.ny / (2 * P)), dht1_threads(P, std::max(R1, R2)), sh, s, f.phi, P, f.tw_z);
      }))
    return;
  const int logn = (int)std::lround(std::log2((double)n));
  const int lines = c.nx * c.ny;
  int W = 16;
  while (lines % W) W >>= 1;   // ny is an even power of two, so W >= 2
  const size_t sh = (size_t)(W / 2) * n * sizeof(typename Vec2<T>::type);
  k_dht<T, true><<<lines / W, 256, sh, s>>>(f.phi, n, logn, W, lines, 0, 1, f.tw_z);
}

constexpr size_t PXS_MAX = 200 * 1024;

// h^2 / (ny nz) for the x solve's right-hand side; in FP64 also 1 / 4 for each
// direction that k_dht1_y, k_dht1_z transform (there and back, a factor 2 each)
double poisson_rhs_scale(const Consts& c, bool fp64) {
  double s = c.h * c.h / ((double)c.ny * c.nz);
  if (fp64)
    for (int n : {c.ny, c.nz})
      if (with_radices(n, [](auto, auto) {})) s *= 0.25;
  return s;
}

template <class T>
void launch_poisson_x_on(const Consts& c, const Fields<T>& f, T* buf, cudaStream_t s) {
  const int P = c.ny * c.nz;
  const T scale = (T)poisson_rhs_scale(c, sizeof(T) == 8);
  const size_t line = (size_t)c.nx * 32 * sizeof(T);
  if (line <= PXS_MAX && (P + 31) / 32 <= 152 * (int)(227 * 1024 / (line + 1024))) {
    launch_next(k_poisson_xs<T>, (P + 31) / 32, 32, line, s, c, f.ptab, f.pconv, buf, scale);
    return;
  }
  launch_next(k_poisson_x<T, T>, (P + 127) / 128, 128, 0, s, c, f.ptab, f.pconv, buf, scale);
}

// the same on bfloat16 storage (FP32 arithmetic)
void launch_poisson_x_bf16(const Consts& c, const Fields<float>& f, void* buf, cudaStream_t s) {
  const int P = c.ny * c.nz;
  const float scale = (float)(c.h * c.h / ((double)c.ny * c.nz));
  __nv_bfloat16* b = reinterpret_cast<__nv_bfloat16*>(buf);
  launch_next(k_poisson_x<float, __nv_bfloat16>, (P + 127) / 128, 128, 0, s, c, f.ptab, f.pconv, b, scale);
}

template <class T>
void launch_poisson_x(const Consts& c, const Fields<T>& f, cudaStream_t s) {
  launch_poisson_x_on(c, f, f.phi, s);
}

// FP32: both transforms of every x plane in one pass where a kernel has the
// shape, 256 x 256 in clusters, planes that fit shared memory one CTA each. FP64
// takes the directions one by one: its pipe bounds them either way, and the
// small blocks of k_dht1_y, k_dht1_z fill the SMs evenly (512 planes of 256 x
// 256: 2.06 ms in the cluster form, 1.75 here)
bool launch_dht2d_on(const Consts& c, const Fields<float>& f, const float* in, float* out, cudaStream_t s) {
  if (c.ny == 256 && c.nz == 256) {
    launch_next(k_dht2d_r16, c.nx * R16_CLUSTER, R16_THREADS, R16_SMEM, s, in, out, f.tw_y);
    return true;
  }
  return with_plane(c.ny, c.nz, [&](auto g, auto kernel) {
    launch_next(kernel, c.nx, decltype(g)::THREADS, decltype(g)::SMEM, s, in, out, f.tw_y, f.tw_z);
  });
}
template <class T>
bool launch_dht2d(const Consts& c, const Fields<T>& f, cudaStream_t s) {
  if constexpr (sizeof(T) == 4) return launch_dht2d_on(c, f, f.phi, f.phi, s);
  else return false;
}

// the same transform of `nplanes` 256 x 256 planes outside a solver state
// (the generator's spectral relaxation); tw: the 256-point twiddles
bool dht2d_planes_fp32(const float* in, float* out, int nplanes, const float* tw, cudaStream_t s) {
  if (nplanes <= 0) return true;
  launch_next(k_dht2d_r16, nplanes * R16_CLUSTER, R16_THREADS, R16_SMEM, s, in, out, tw);
  return cudaGetLastError() == cudaSuccess;
}

template <class T>
void launch_poisson(const Consts& c, const Fields<T>& f, cudaStream_t s) {
  if (launch_dht2d(c, f, s)) {
    launch_poisson_x(c, f, s);
    launch_dht2d(c, f, s);
    return;
  }
  launch_dht_y(c, f, s);
  launch_dht_z(c, f, s);
  launch_poisson_x(c, f, s);
  launch_dht_z(c, f, s);
  launch_dht_y(c, f, s);
}

size_t poisson_table_size(const Consts& c) { return (size_t)c.nx * ptab_plane(c); }
size_t poisson_modes(const Consts& c) { return ptab_plane(c); }

template <class T>
void launch_poisson_table(const Consts& c, const Fields<T>& f, cudaStream_t s) {
  const int PT = (int)ptab_plane(c);
  k_poisson_table<T><<<(PT + 127) / 128, 128, 0, s>>>(c, f.ptab, f.pconv);
}

template void launch_poisson<double>(const Consts&, const Fields<double>&, cudaStream_t);
template bool launch_dht2d<double>(const Consts&, const Fields<double>&, cudaStream_t);
template bool launch_dht2d<float>(const Consts&, const Fields<float>&, cudaStream_t);
template void launch_dht_y<double>(const Consts&, const Fields<double>&, cudaStream_t);
template void launch_dht_y<float>(const Consts&, const Fields<float>&, cudaStream_t);
template void launch_dht_z<double>(const Consts&, const Fields<double>&, cudaStream_t);
template void launch_dht_z<float>(const Consts&, const Fields<float>&, cudaStream_t);
template void launch_poisson_x<double>(const Consts&, const Fields<double>&, cudaStream_t);
template void launch_poisson_x_on<float>(const Consts&, const Fields<float>&, float*, cudaStream_t);
template void launch_poisson_x_on<double>(const Consts&, const Fields<double>&, double*, cudaStream_t);
template void launch_poisson_x<float>(const Consts&, const Fields<float>&, cudaStream_t);
template void launch_poisson<float>(const Consts&, const Fields<float>&, cudaStream_t);
template void launch_poisson_table<double>(const Consts&, const Fields<double>&, cudaStream_t);
template void launch_poisson_table<float>(const Consts&, const Fields<float>&, cudaStream_t);

// opt in to large dynamic shared memory for the transform kernels of ny x nz
// planes (setting it for every size loads every kernel: 0.4 ms of a process's first create)
void poisson_set_attributes(int ny, int nz) {
  cudaFuncSetAttribute(k_dht2d_r16, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)R16_SMEM);
  cudaFuncSetAttribute(k_poisson_xs<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PXS_MAX);
  cudaFuncSetAttribute(k_poisson_xs<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PXS_MAX);
  with_plane(ny, nz, [](auto g, auto kernel) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)decltype(g)::SMEM);
  });
  for (int n : {ny, nz})
    with_radices(n, [](auto r1, auto r2) {
      constexpr int R1 = decltype(r1)::value, R2 = decltype(r2)::value;
      cudaFuncSetAttribute(k_dht1_y<double, R1, R2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
      cudaFuncSetAttribute(k_dht1_z<double, R1, R2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
      cudaFuncSetAttribute(k_dht1_y<float, R1, R2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
      cudaFuncSetAttribute(k_dht1_z<float, R1, R2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
    });
  cudaFuncSetAttribute(k_dht<double, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  cudaFuncSetAttribute(k_dht<double, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  cudaFuncSetAttribute(k_dht<float, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  cudaFuncSetAttribute(k_dht<float, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
}

}  // namespace ibm
