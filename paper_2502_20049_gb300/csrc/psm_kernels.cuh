// CUDA kernels of the PSM hot path (arXiv 2502.20049), templated on the PDF
// storage type, the stencil, the streaming access pattern and the fluid
// collision.  Included by one translation unit per storage precision.
//
//   k_step    one fused time step: load (AA / two-grid), remap of the geometry
//             field onto eps (Sec. 3), moments, B (Eq. 5/6), u_s = omega x r + v,
//             Omega^F (Eq. 2 / TRT), Omega^S (Eq. 7/8/9), PSM blend (Eq. 4),
//             streamed store (Eq. 1), force/torque (Eq. 10/11) reduced in FP64
//             with a deterministic order (per-warp, per-block, k_reduce_slots).
//   k_import  write a natural state (or a uniform equilibrium) in a layout
//   k_export  read a state in its layout and write it natural, unshifted, FP64
//   k_macro   rho and u per cell (FP64)
//   k_mass    deterministic FP64 total mass
//   k_remap   eps per cell (remap only)
#pragma once

#include <cuda_bf16.h>
#include <algorithm>
#include <type_traits>
#include <cuda_fp16.h>

#include "psm_internal.h"

namespace psm {

// ---------------------------------------------------------------------------
// Lattice: D3Q27 velocities in the library's order; the first 19 are D3Q19.
// Pairs (2k-1, 2k) are opposite; 0 is the rest direction.
// ---------------------------------------------------------------------------
__host__ __device__ __forceinline__ constexpr int lat_cx(int i) {
  constexpr int t[27] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, -1, 1};
  return t[i];
}
__host__ __device__ __forceinline__ constexpr int lat_cy(int i) {
  constexpr int t[27] = {0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, -1, 1, 1, -1};
  return t[i];
}
__host__ __device__ __forceinline__ constexpr int lat_cz(int i) {
  constexpr int t[27] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1, 1, -1, -1, 1, 1, -1, 1, -1};
  return t[i];
}
__host__ __device__ __forceinline__ constexpr int lat_opp(int i) { return i == 0 ? 0 : ((i & 1) ? i + 1 : i - 1); }
template <int Q>
__host__ __device__ __forceinline__ constexpr double lat_w(int i) {
  // |c|^2 = 0, 1, 2, 3
  return Q == 19 ? (i == 0 ? 1.0 / 3.0 : (i < 7 ? 1.0 / 18.0 : 1.0 / 36.0))
                 : (i == 0 ? 8.0 / 27.0 : (i < 7 ? 2.0 / 27.0 : (i < 19 ? 1.0 / 54.0 : 1.0 / 216.0)));
}

// ---------------------------------------------------------------------------
// Storage conversions.  PDFs are stored shifted (f - w rho0).
// ---------------------------------------------------------------------------
template <class S>
struct Store;
template <>
struct Store<double> {
  using T = double;
  static __device__ __forceinline__ double ld(const double* p) { return *p; }
  static __device__ __forceinline__ void st(double* p, double v) { *p = v; }
  static __device__ __forceinline__ double from_double(double v) { return v; }
};
template <>
struct Store<float> {
  using T = float;
  static __device__ __forceinline__ float ld(const float* p) { return *p; }
  static __device__ __forceinline__ void st(float* p, float v) { *p = v; }
  static __device__ __forceinline__ float from_double(double v) { return (float)v; }
};
template <>
struct Store<__half> {
  using T = float;
  static __device__ __forceinline__ float ld(const __half* p) { return __half2float(*p); }
  static __device__ __forceinline__ void st(__half* p, float v) { *p = __float2half_rn(v); }
  static __device__ __forceinline__ __half from_double(double v) { return __double2half(v); }
};
template <>
struct Store<__nv_bfloat16> {
  using T = float;
  static __device__ __forceinline__ float ld(const __nv_bfloat16* p) { return __bfloat162float(*p); }
  static __device__ __forceinline__ void st(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
  static __device__ __forceinline__ __nv_bfloat16 from_double(double v) { return __double2bfloat16(v); }
};

// Two 16-bit values of neighbouring cells (x even, x + 1) as one 32-bit word:
// the lower half is the cell at the lower address (16-bit storage types only).
template <class S>
struct Pair16 {
  template <class T>
  static __device__ __forceinline__ void unpack(unsigned, T& a, T& b) { a = b = T(0); }
  template <class T>
  static __device__ __forceinline__ unsigned pack(T, T) { return 0u; }
};
template <>
struct Pair16<__half> {
  static __device__ __forceinline__ void unpack(unsigned w, float& a, float& b) {
    __half2 h;
    memcpy(&h, &w, 4);
    a = __low2float(h);
    b = __high2float(h);
  }
  static __device__ __forceinline__ unsigned pack(float a, float b) {
    const __half2 h = __floats2half2_rn(a, b);
    unsigned w;
    memcpy(&w, &h, 4);
    return w;
  }
};
template <>
struct Pair16<__nv_bfloat16> {
  static __device__ __forceinline__ void unpack(unsigned w, float& a, float& b) {
    __nv_bfloat162 h;
    memcpy(&h, &w, 4);
    a = __low2float(h);
    b = __high2float(h);
  }
  static __device__ __forceinline__ unsigned pack(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    unsigned w;
    memcpy(&w, &h, 4);
    return w;
  }
};

// ---------------------------------------------------------------------------
// Remap of one body onto one cell (Sec. 3).  The cell centre is taken into the
// body frame, X = Q_n^T (x_c - R_n); the 2^s sub-cells per axis whose block
// starts at the sub-grid point nearest to X - 1/2 are counted in the
// brick-packed field.  The start index a0_k = floor(r_k),
// r_k = ((X_k - 1/2) - lo_k) 2^s + 1/2, is the double evaluation of r_k with
// separately rounded operations in that order.  The kernel evaluates r_k in
// float from the exact-split affine form of remap_setup (high part exact, low
// part within rtol of the double value); a cell whose float r_k lies within
// rtol of an integer on some axis takes the double evaluation itself, so the
// decision always equals the double one (the fallback is rare: rtol is a few
// float round-offs, so about 6 rtol of the cells in a body's box take it).
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long low_bits(int w) { return w >= 64 ? ~0ull : ((1ull << w) - 1ull); }

static __device__ __noinline__ int3 remap_start_double(const DevBody& b, int x, int y, int z) {
  const double n = (double)(1 << b.s);
  const double xc[3] = {(double)x + 0.5, (double)y + 0.5, (double)z + 0.5};
  double d[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) d[k] = __dsub_rn(xc[k], b.R[k]);
  int a0[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double X = __dadd_rn(__dadd_rn(__dmul_rn(b.Qd[k], d[0]), __dmul_rn(b.Qd[3 + k], d[1])),
                               __dmul_rn(b.Qd[6 + k], d[2]));
    a0[k] = (int)floor(__dadd_rn(__dmul_rn(__dsub_rn(__dsub_rn(X, 0.5), b.lod[k]), n), 0.5));
  }
  return make_int3(a0[0], a0[1], a0[2]);
}

__device__ __forceinline__ float remap_eps(const DevBody& b, int x, int y, int z) {
  const int s = b.s;
  const int n = 1 << s;
  const float e0 = (float)(x - b.anchor[0]), e1 = (float)(y - b.anchor[1]), e2 = (float)(z - b.anchor[2]);
  int a0[3];
  bool near = false;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float hi = __fmaf_rn(b.Ghi[6 + k], e2, __fmaf_rn(b.Ghi[3 + k], e1, __fmaf_rn(b.Ghi[k], e0, b.Hhi[k])));
    const float lo = __fmaf_rn(b.Glo[6 + k], e2, __fmaf_rn(b.Glo[3 + k], e1, __fmaf_rn(b.Glo[k], e0, b.Hlo[k])));
    const float fh = floorf(hi);
    const float v = __fadd_rn(__fsub_rn(hi, fh), lo);  // hi - fh is exact
    const float fv = floorf(v);
    a0[k] = (int)fh + (int)fv;
    near = near || fminf(__fsub_rn(v, fv), __fsub_rn(__fadd_rn(fv, 1.0f), v)) <= b.rtol;
  }
  if (near) {
    const int3 a = remap_start_double(b, x, y, z);
    a0[0] = a.x;
    a0[1] = a.y;
    a0[2] = a.z;
  }
  // per axis up to two coarse cells: [o, n) of g and [0, o) of g + 1
  int gc[3], o[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    gc[k] = a0[k] >> s;  // arithmetic shift = floor division
    o[k] = a0[k] & (n - 1);
  }
  const int dims[3] = {b.gx, b.gy, b.gz};
  // quick reject: the whole block lies outside the stored box
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int glast = gc[k] + (o[k] ? 1 : 0);
    if (glast < 0 || gc[k] >= dims[k]) return 0.0f;
  }
  // the block touches coarse cells {gc, gc + 1}^3 at most: none holds a set bit
  // where the occupancy byte is zero (then eps is exactly 0); the block bit of
  // 8^3 occupancy bytes is tested first (a small array that stays in L1,
  // where the bytes come from L2 or memory)
  if (b.occ8) {
    const long long bi = ((long long)((gc[2] + 1) >> 3) * b.o8y + ((gc[1] + 1) >> 3)) * b.o8x + ((gc[0] + 1) >> 3);
    if (!((__ldg(b.occ8 + (bi >> 5)) >> (unsigned)(bi & 31)) & 1u)) return 0.0f;
  }
  if (b.occ) {
    const long long oi = ((long long)(gc[2] + 1) * (b.gy + 1) + (gc[1] + 1)) * (long long)(b.gx + 1) + (gc[0] + 1);
    if (!__ldg(b.occ + oi)) return 0.0f;
  }
  int count = 0;
  const int nn = n * n;
  // s <= 2 (one word per brick, bit (z n + y) n + x): rowrep has bit r n set
  // for every row r < n^2, layrep bit l n^2 for every layer l < n
  const unsigned long long rowrep = s == 2 ? 0x1111111111111111ull : (s == 1 ? 0x55ull : 1ull);
  const unsigned long long layrep = s == 2 ? 0x0001000100010001ull : (s == 1 ? 0x11ull : 1ull);
  for (int sz = 0; sz < 2; ++sz) {
    if (sz == 1 && o[2] == 0) break;
    const int gz = gc[2] + sz;
    if (gz < 0 || gz >= b.gz) continue;
    const int za = sz ? 0 : o[2], zb = sz ? o[2] : n;
    for (int sy = 0; sy < 2; ++sy) {
      if (sy == 1 && o[1] == 0) break;
      const int gy = gc[1] + sy;
      if (gy < 0 || gy >= b.gy) continue;
      const int ya = sy ? 0 : o[1], yb = sy ? o[1] : n;
      for (int sx = 0; sx < 2; ++sx) {
        if (sx == 1 && o[0] == 0) break;
        const int gx = gc[0] + sx;
        if (gx < 0 || gx >= b.gx) continue;
        const int xa = sx ? 0 : o[0], xb = sx ? o[0] : n;
        const unsigned long long* brick =
            b.bricks + ((long long)((long long)gz * b.gy + gy) * b.gx + gx) * b.wpb;
        const unsigned long long xm = low_bits(xb - xa) << xa;
        if (s <= 2) {
          const unsigned long long ym = (low_bits(n * (yb - ya)) << (n * ya)) * layrep;
          const unsigned long long zm = low_bits(nn * (zb - za)) << (nn * za);
          const unsigned long long m = (xm * rowrep) & ym & zm;
          count += __popcll(__ldg(brick) & m);
        } else {
          // s = 3: word = z layer, bit y * 8 + x
          const unsigned long long m = (xm * 0x0101010101010101ull) & (low_bits(8 * (yb - ya)) << (8 * ya));
          for (int w = za; w < zb; ++w) count += __popcll(__ldg(brick + w) & m);
        }
      }
    }
  }
  return (float)count * (1.0f / (float)(n * nn));
}

// eps (min(1, sum over bodies)) and owner (argmax, lower id on ties; -1 if none)
__device__ __forceinline__ float cell_eps(const DevBody* bodies, int nb, int x, int y, int z, int& owner) {
  float sum = 0.0f, best = 0.0f;
  owner = -1;
  for (int bi = 0; bi < nb; ++bi) {
    const DevBody& b = bodies[bi];
    if (x >= b.x0 && x < b.x1 && y >= b.y0 && y < b.y1 && z >= b.z0 && z < b.z1) {
      const float e = remap_eps(b, x, y, z);
      sum += e;
      if (e > best) {
        best = e;
        owner = bi;
      }
    }
  }
  return fminf(sum, 1.0f);
}

// ---------------------------------------------------------------------------
// Neighbour offsets of a cell (periodic x, y; periodic or bounded z)
// ---------------------------------------------------------------------------
struct Nbr {
  // 32-bit unsigned offsets: cell indices are < 2^32 and the sum cell + off
  // wraps modulo 2^32 onto the neighbour's index
  unsigned dxm, dxp, dym, dyp, dzm, dzp;
  bool zlo_out, zhi_out;  // z - 1 (resp. z + 1) lies outside (ghost plane)
  __device__ __forceinline__ void init(const Grid3& g, int x, int y, int z) {
    const unsigned nx = (unsigned)g.nx, plane = (unsigned)g.nx * (unsigned)g.ny;
    dxm = (x == 0) ? nx - 1u : 0u - 1u;
    dxp = (x == g.nx - 1) ? 0u - (nx - 1u) : 1u;
    dym = (y == 0) ? (unsigned)(g.ny - 1) * nx : 0u - nx;
    dyp = (y == g.ny - 1) ? 0u - (unsigned)(g.ny - 1) * nx : nx;
    dzm = (z == 0) ? (unsigned)(g.nz - 1) * plane : 0u - plane;
    dzp = (z == g.nz - 1) ? 0u - (unsigned)(g.nz - 1) * plane : plane;
    const bool ghost = g.bc_z == PSM_BC_EQ_INLET_OUTLET;
    zlo_out = ghost && z == 0;
    zhi_out = ghost && z == g.nz - 1;
  }
  __device__ __forceinline__ unsigned off(int dx, int dy, int dz) const {
    return (dx < 0 ? dxm : (dx > 0 ? dxp : 0u)) + (dy < 0 ? dym : (dy > 0 ? dyp : 0u)) +
           (dz < 0 ? dzm : (dz > 0 ? dzp : 0u));
  }
  // x - c_i lies in a ghost plane: population i enters from the ghost plane
  __device__ __forceinline__ bool from_ghost(int cz) const { return (cz > 0 && zlo_out) || (cz < 0 && zhi_out); }
  // x + c_i lies in a ghost plane: population i leaves the domain
  __device__ __forceinline__ bool to_ghost(int cz) const { return (cz > 0 && zhi_out) || (cz < 0 && zlo_out); }
};

// s a for a lattice component s in {-1, 0, 1}, without multiplying (IEEE
// arithmetic keeps 0 * a, so products with the zero components are avoided)
template <class T>
__device__ __forceinline__ T csign(int c, T a) {
  return c > 0 ? a : (c < 0 ? -a : T(0));
}
// c_i . v over the non-zero components of c_i only
template <class T>
__device__ __forceinline__ T cdot(int i, T vx, T vy, T vz) {
  T r = T(0);
  bool h = false;
  if (lat_cx(i)) {
    r = csign(lat_cx(i), vx);
    h = true;
  }
  if (lat_cy(i)) {
    r = h ? r + csign(lat_cy(i), vy) : csign(lat_cy(i), vy);
    h = true;
  }
  if (lat_cz(i)) r = h ? r + csign(lat_cz(i), vz) : csign(lat_cz(i), vz);
  return r;
}

// Eq. 3 (sign-corrected) minus the storage shift w rho0, for velocity v:
//   f^eq_i(rho, v) - w_i rho0 = w_i (drho + rho (3 c.v + 4.5 (c.v)^2 - 1.5 v.v))
template <int Q, class T>
__device__ __forceinline__ T feq_shifted(int i, T drho, T rho, T vx, T vy, T vz, T vv) {
  const T cv = T(lat_cx(i)) * vx + T(lat_cy(i)) * vy + T(lat_cz(i)) * vz;
  return T(lat_w<Q>(i)) * (drho + rho * (T(3) * cv + T(4.5) * cv * cv - T(1.5) * vv));
}
// the same over the non-zero components of c_i only (fewer instructions; the
// adjoint kernel's form)
template <int Q, class T>
__device__ __forceinline__ T feq_shifted_nz(int i, T drho, T rho, T vx, T vy, T vz, T vv) {
  const T cv = cdot(i, vx, vy, vz);
  return T(lat_w<Q>(i)) * (drho + rho * (T(3) * cv + T(4.5) * cv * cv - T(1.5) * vv));
}

template <class V>
__device__ __forceinline__ V warp_sum(V v) {
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
  return v;
}

// Type of one cell's force/torque contribution and of its warp partial sum:
// the compute precision (FP64 arithmetic for FP64 storage; FP32 otherwise).
// The per-warp partials are added into FP64 block slots, and the block and
// grid sums are FP64 (on GB300 an FP64 instruction costs about 64 FP32 ones,
// so the 32-cell partials stay in the arithmetic's own precision).
template <class T>
using ft_t = typename std::conditional<sizeof(T) == 8, double, float>::type;

// out[c] = sum over the G blocks' partials[j][c], c < ncomp, by one block of NT
// threads in a fixed order.  Bound by latency: the warps take the components
// side by side (several share one where there are fewer), and each lane loads
// up to 16 partials before it adds the first.
template <int NT>
__device__ __forceinline__ void sum_partials(const double* partials, int G, int ncomp, double* out) {
  constexpr int NW = NT / 32;
  __shared__ double red[NW];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int share = ncomp < NW ? NW / ncomp : 1;  // warps per component
  for (int c = warp / share; c < ncomp; c += NW / share) {
    double acc = 0.0;
    for (int j0 = (warp % share) * 32 + lane; j0 < G; j0 += share * 512) {
      double v[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const int j = j0 + k * share * 32;
        v[k] = j < G ? __ldcg(&partials[(long long)j * ncomp + c]) : 0.0;
      }
#pragma unroll
      for (int h = 8; h > 0; h >>= 1)
#pragma unroll
        for (int k = 0; k < h; ++k) v[k] += v[k + h];
      acc += v[0];
    }
    acc = warp_sum(acc);
    if (lane == 0) {
      if (share == 1) out[c] = acc;
      else red[warp] = acc;
    }
  }
  __syncthreads();
  if (share > 1 && (int)threadIdx.x < ncomp) {
    double v = red[threadIdx.x * share];
    for (int k = 1; k < share; ++k) v += red[threadIdx.x * share + k];
    out[threadIdx.x] = v;
  }
}

// Block-wide ordered reduction of per-block values v[0..ncomp) held in shared
// memory `blk` into partials[blockIdx.x]; the last block to finish sums all
// partials in a fixed order into out[0..ncomp).  Deterministic for a fixed grid.
template <int NT = PSM_THREADS>
__device__ __forceinline__ void grid_reduce(const double* blk, int ncomp, double* partials, unsigned int* ticket,
                                            double* out) {
  __shared__ unsigned int s_last;
  if ((int)threadIdx.x < ncomp) {
    partials[(long long)blockIdx.x * ncomp + threadIdx.x] = blk[threadIdx.x];
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) s_last = (atomicAdd(ticket, 1u) == gridDim.x - 1) ? 1u : 0u;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  sum_partials<NT>(partials, (int)gridDim.x, ncomp, out);
  if (threadIdx.x == 0) *ticket = 0u;
}

// The blocks' partials of a kernel whose sum is taken later (k_reduce_slots): the
// number of blocks, then [block][ncomp].
__device__ __forceinline__ void store_slot(double* slot, const double* blk, int ncomp) {
  if ((int)threadIdx.x < ncomp) slot[1 + (long long)blockIdx.x * ncomp + threadIdx.x] = blk[threadIdx.x];
  if (blockIdx.x == 0 && threadIdx.x == 0) slot[0] = (double)gridDim.x;
}

// ---------------------------------------------------------------------------
// The fused step kernel (persistent: blocks stride over row tiles).
// ---------------------------------------------------------------------------
// Resident blocks per SM the register allocation aims at (D3Q19 / D3Q27).
#ifndef PSM_MIN_BLOCKS_Q19
#define PSM_MIN_BLOCKS_Q19 3
#endif
#ifndef PSM_MIN_BLOCKS_Q27
#define PSM_MIN_BLOCKS_Q27 2
#endif
// Resident blocks per SM of a step kernel for storage S and stencil Q: FP64
// state needs twice the registers per PDF, so one block fewer (80 / 128 / 255
// registers per thread at 3 / 2 / 1 blocks of 256 threads).
// The cumulant operator (FL = 2, D3Q19) keeps about twice the values of
// BGK/TRT live: it aims at PSM_MIN_BLOCKS_CUM blocks (128 registers at 2),
// and FP64 at one.
#ifndef PSM_MIN_BLOCKS_CUM
#define PSM_MIN_BLOCKS_CUM 2
#endif
// Tiles of 256 cells with two x neighbours per thread (TMA kernel, 2-byte
// storage): a tile is four warps' work, and the block's two groups of warps take
// alternate tiles.  These steps are bound by instruction issue, and a pair shares
// shared-memory accesses, stores, addresses and the tile's bookkeeping.
//   AA odd, BGK/TRT: 539 -> 403 warp instructions per 32 cells (D3Q19, 256x256x240
//     with two rotors), 644 -> 527 (D3Q27, 256x256x320).  Two-row tiles for the pairs
//     halved the pipeline's depth; one-row tiles keep it.
//     1024x1024x960 D3Q19 FP16 14.11 -> 13.67 ms per AA step (even and odd
//     averaged), 512x512x640 D3Q27 3.456 -> 3.348.
//   Cumulant, every mode: the additions and multiply-adds of its arithmetic
//     are packed FP32 instructions as well (256^3: AA even 449 -> 302 warp
//     instructions per 32 cells, AA odd 530 -> 402, two-grid 491 -> 343); 128
//     registers without spills.  256^3 FP16 AA 296.8 -> 245.6 us a
//     step, two-grid 289.6 -> 242.1 (pairs alone: 277.5 and 274.4).
template <class S, int FL, int MODE>
__host__ __device__ constexpr bool tile_pairs() {
  // (tensor stores write one cell per thread)
  return sizeof(S) == 2 && MODE >= 0 && (FL == 2 || MODE == MODE_AA_ODD) && !(PSM_TMA_STORE && MODE == MODE_AA_EVEN);
}
template <class S, int Q, int FL = 0, int MODE = -1>
__host__ __device__ constexpr int step_min_blocks() {
  if (FL == 2) return sizeof(S) == 8 ? 1 : PSM_MIN_BLOCKS_CUM;
  if (tile_pairs<S, FL, MODE>()) return 2;
  return sizeof(S) == 8 ? (Q == 19 ? PSM_MIN_BLOCKS_Q19 - 1 : PSM_MIN_BLOCKS_Q27 - 1)
                        : (Q == 19 ? PSM_MIN_BLOCKS_Q19 : PSM_MIN_BLOCKS_Q27);
}

template <class T>
__device__ __forceinline__ const ConstT<T>& cst(const StepParams& p) {
  if constexpr (sizeof(T) == 4) return p.cf;
  else return p.cd;
}

// 1 / r: FP32 by rcp.approx refined with one Newton-Raphson step
// (a' = a + a (1 - r a)), within 1 ulp for the densities here (r near 1); FP64
// by IEEE division.
template <class T>
__device__ __forceinline__ T recip(T r) {
  if constexpr (sizeof(T) == 4) {
    float a;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(a) : "f"(r));
    return fmaf(a, fmaf(-r, a, 1.0f), a);
  } else {
    return T(1) / r;
  }
}

// |c_i|^2: the weight class of direction i (0 rest, 1 axis, 2 face diagonal, 3 corner)
__host__ __device__ __forceinline__ constexpr int lat_cls(int i) {
  return lat_cx(i) * lat_cx(i) + lat_cy(i) * lat_cy(i) + lat_cz(i) * lat_cz(i);
}

// Separately rounded operations (never contracted or reordered by the
// compiler): the fluid collision computes the same bits in every kernel that
// inlines it.
template <class T>
__device__ __forceinline__ T r_add(T a, T b) {
  if constexpr (sizeof(T) == 4) return __fadd_rn(a, b);
  else return __dadd_rn(a, b);
}
template <class T>
__device__ __forceinline__ T r_sub(T a, T b) {
  if constexpr (sizeof(T) == 4) return __fsub_rn(a, b);
  else return __dsub_rn(a, b);
}
template <class T>
__device__ __forceinline__ T r_mul(T a, T b) {
  if constexpr (sizeof(T) == 4) return __fmul_rn(a, b);
  else return __dmul_rn(a, b);
}
template <class T>
__device__ __forceinline__ T r_fma(T a, T b, T c) {
  if constexpr (sizeof(T) == 4) return __fmaf_rn(a, b, c);
  else return __fma_rn(a, b, c);
}
// a + s b for a lattice component s = +-1
template <class T>
__device__ __forceinline__ T r_addc(T a, int s, T b) {
  return s > 0 ? r_add(a, b) : r_sub(a, b);
}
template <class T>
__device__ __forceinline__ T r_div(T a, T b) {
  if constexpr (sizeof(T) == 4) return __fdiv_rn(a, b);
  else return __ddiv_rn(a, b);
}

// Two cells' FP32 values side by side: the packed FP32 instructions compute both
// with one issue, each lane rounded as the scalar operation.
struct F2 {
  float2 v;
  __device__ __forceinline__ F2() {}
  __device__ __forceinline__ F2(float a) : v(make_float2(a, a)) {}
  __device__ __forceinline__ F2(float a, float b) : v(make_float2(a, b)) {}
  __device__ __forceinline__ F2(float2 a) : v(a) {}
};
__device__ __forceinline__ F2 operator-(F2 a) { return F2(-a.v.x, -a.v.y); }
// Additions and fused multiply-adds are packed; multiplications stay scalar: the
// assembler contracts a packed one into the addition that follows it, its .rn
// notwithstanding (which would round otherwise than the scalar kernels).
__device__ __forceinline__ unsigned long long f2_bits(F2 a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.v.x), "f"(a.v.y));
  return r;
}
__device__ __forceinline__ F2 f2_of(unsigned long long b) {
  F2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.v.x), "=f"(r.v.y) : "l"(b));
  return r;
}
__device__ __forceinline__ F2 r_add(F2 a, F2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));
  return f2_of(r);
}
__device__ __forceinline__ F2 r_mul(F2 a, F2 b) { return F2(__fmul_rn(a.v.x, b.v.x), __fmul_rn(a.v.y, b.v.y)); }
__device__ __forceinline__ F2 r_fma(F2 a, F2 b, F2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)), "l"(f2_bits(c)));
  return f2_of(r);
}
__device__ __forceinline__ F2 r_sub(F2 a, F2 b) { return r_fma(b, F2(-1.0f), a); }  // a - b, rounded once
__device__ __forceinline__ F2 recip(F2 r) { return F2(recip(r.v.x), recip(r.v.y)); }

// Density deviation, density and velocity of one cell from its shifted PDFs,
// summed over opposite pairs (i, i + 1): drho = f_0 + sum (f_i + f_i+1),
// j = sum c_i (f_i - f_i+1).
template <class T, int Q>
__device__ __forceinline__ void moments(const T (&f)[Q], T rho0, T& drho, T& rho, T& ux, T& uy, T& uz, T& uu) {
  T d = f[0], jx = T(0), jy = T(0), jz = T(0);
  bool hx = false, hy = false, hz = false;  // compile-time after unrolling
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    const T sp = r_add(f[i], f[i + 1]), dm = r_sub(f[i], f[i + 1]);
    d = r_add(d, sp);
    if (lat_cx(i)) {
      jx = hx ? r_addc(jx, lat_cx(i), dm) : (lat_cx(i) > 0 ? dm : -dm);
      hx = true;
    }
    if (lat_cy(i)) {
      jy = hy ? r_addc(jy, lat_cy(i), dm) : (lat_cy(i) > 0 ? dm : -dm);
      hy = true;
    }
    if (lat_cz(i)) {
      jz = hz ? r_addc(jz, lat_cz(i), dm) : (lat_cz(i) > 0 ? dm : -dm);
      hz = true;
    }
  }
  drho = d;
  rho = r_add(rho0, d);
  const T inv_rho = recip(rho);
  ux = r_mul(jx, inv_rho);
  uy = r_mul(jy, inv_rho);
  uz = r_mul(jz, inv_rho);
  uu = r_fma(uz, uz, r_fma(uy, uy, r_mul(ux, ux)));
}

// c_i . u with separately rounded operations
template <class T>
__device__ __forceinline__ T c_dot(int i, T ux, T uy, T uz) {
  T cu = T(0);
  bool h = false;
  if (lat_cx(i)) {
    cu = lat_cx(i) > 0 ? ux : -ux;
    h = true;
  }
  if (lat_cy(i)) {
    cu = h ? r_addc(cu, lat_cy(i), uy) : (lat_cy(i) > 0 ? uy : -uy);
    h = true;
  }
  if (lat_cz(i)) cu = h ? r_addc(cu, lat_cz(i), uz) : (lat_cz(i) > 0 ? uz : -uz);
  return cu;
}

// feq_shifted with separately rounded operations (the PSM cells of the
// cumulant step): w_i (drho + rho (3 c.v + 4.5 (c.v)^2 - 1.5 v.v))
template <int Q, class T>
__device__ __forceinline__ T feq_shifted_r(int i, T drho, T rho, T vx, T vy, T vz, T vv) {
  const T cv = c_dot(i, vx, vy, vz);
  const T q = r_fma(r_mul(T(4.5), cv), cv, r_fma(T(3), cv, r_mul(T(-1.5), vv)));
  return r_mul(T(lat_w<Q>(i)), r_fma(rho, q, drho));
}

// Pure fluid cell: f* = f + Omega^F (TRT; BGK is the case omega+ = omega- =
// 1/tau).  Per opposite pair (i, j), c_j = -c_i, with s = f_i + f_j and
// d = f_i - f_j the shifted equilibrium splits into
//   even = w (drho + rho (4.5 (c.u)^2 - 1.5 u.u)),  odd = 3 w rho (c.u),
//   f^eq_i - w rho0 = even + odd,  f^eq_j - w rho0 = even - odd,
// and the relaxed pair is f*_i = p + m, f*_j = p - m with
//   p = (1 - omega+) s / 2 + omega+ even,  m = (1 - omega-) d / 2 + omega- odd.
// The products of omega+-, the weight and the numeric factors are host
// constants per weight class (ConstT pw, pk, pd); f_i and f_j are not needed
// once s and d are formed.
// (T: float, double, or F2 with the float constants)
template <class T, bool UNIT, class CT>
__device__ __forceinline__ void cumulant_relax(const CT& C, T (&f)[19], T drho, T rho, T ux, T uy, T uz);

template <class T, int Q, int FL, class CT>
__device__ __forceinline__ void fluid_relax(const CT& C, T (&f)[Q], T drho, T rho, T ux, T uy, T uz, T uu) {
  if constexpr (FL == 2) {
    static_assert(Q == 19, "the cumulant operator is defined for D3Q19");
    if (C.cum_unit) cumulant_relax<T, true>(C, f, drho, rho, ux, uy, uz);
    else cumulant_relax<T, false>(C, f, drho, rho, ux, uy, uz);
    return;
  }
  const T base = r_fma(T(-1.5), r_mul(rho, uu), drho);
  constexpr int NC = Q == 27 ? 4 : 3;
  T A[NC], K[NC], D[NC];  // per class: omega+ w base, 4.5 omega+ w rho, 3 omega- w rho
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    A[c] = r_mul(C.pw[c], base);
    K[c] = r_mul(C.pk[c], rho);
    D[c] = r_mul(C.pd[c], rho);
  }
  f[0] = r_fma(C.omp1, f[0], A[0]);
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    const int j = i + 1, c = lat_cls(i);
    const T cu = c_dot(i, ux, uy, uz);
    const T sp = r_add(f[i], f[j]), dm = r_sub(f[i], f[j]);
    const T pe = r_fma(C.hp1, sp, r_fma(K[c], r_mul(cu, cu), A[c]));
    const T mo = r_fma(C.hm1, dm, r_mul(D[c], cu));
    f[i] = r_add(pe, mo);
    f[j] = r_sub(pe, mo);
  }
}

// Cumulant collision of one D3Q19 cell (Geier et al. 2015: listed in Sec. 2.2,
// the operator of every performance run in Sec. 5.1), restricted to the 19
// moments D3Q19 resolves, from the shifted PDFs f (f - w rho0), in place.
//   raw moments of the shifted PDFs, plane by plane (D3Q19 has no corner
//     directions, so the x-y face diagonals alone carry c_x^2 c_y^2, c_x^2 c_y,
//     c_x c_y^2 and c_x c_y);
//   central moments k_abc about u, kept as deviations from the fluid at rest
//     (k^_200 = k_200 - rho/3, k^_220 = k_220 - rho/9): every term is then of
//     the size of u^2 or the non-equilibrium part, so FP32 loses nothing to
//     cancellation against rho/3 or rho/9;
//   relaxation: off-diagonal and deviatoric second order with 1 - 1/tau, the
//     trace with 1 - omega_bulk, third order with 1 - omega_3, the fourth-order
//     cumulants C_220 = k_220 - (k_200 k_020 + 2 k_110^2) / rho with
//     1 - omega_4 (host constants cum1[0..3]); with the default rates (bulk,
//     third and fourth order 1, UNIT) the trace, third- and fourth-order
//     cumulants are set to equilibrium without computing them;
//   raw moments of the result by the inverse shift, then the D3Q19 PDFs in
//     closed form: f(sx, sy, 0) = (m_220 + sx m_120 + sy m_210 + sx sy m_110) / 4,
//     f(s, 0, 0) = ((m_200 - m_220 - m_202) + s (m_100 - m_120 - m_102)) / 2,
//     f_0 = m_000 - m_200 - m_020 - m_002 + m_220 + m_202 + m_022.
// Operations are separately rounded (same bits in every kernel that inlines it).
template <class T, bool UNIT, class CT>
__device__ __forceinline__ void cumulant_relax(const CT& C, T (&f)[19], T drho, T rho, T ux, T uy, T uz) {
  auto ad = [](T a, T b) { return r_add(a, b); };
  auto sb = [](T a, T b) { return r_sub(a, b); };
  auto ml = [](T a, T b) { return r_mul(a, b); };
  auto fm = [](T a, T b, T c) { return r_fma(a, b, c); };
  const T third = T(1.0 / 3.0), ninth = T(1.0 / 9.0);
  // ---- raw moments of the shifted PDFs ----
  const T Ax = ad(f[1], f[2]), Bx = sb(f[1], f[2]);
  const T Ay = ad(f[3], f[4]), By = sb(f[3], f[4]);
  const T Az = ad(f[5], f[6]), Bz = sb(f[5], f[6]);
  T Sxy, Mxy, Xxy, Yxy, Sxz, Mxz, Xxz, Zxz, Syz, Myz, Yyz, Zyz;
  {
    // group (a, b) with f[k] = (+,+), f[k+1] = (-,-), f[k+2] = (+,-), f[k+3] = (-,+)
    auto group = [&](int k, T& S, T& M, T& A, T& B) {
      const T p1 = ad(f[k], f[k + 1]), m1 = sb(f[k], f[k + 1]);
      const T p2 = ad(f[k + 2], f[k + 3]), m2 = sb(f[k + 2], f[k + 3]);
      S = ad(p1, p2);  // sum c_a^2 c_b^2 f
      M = sb(p1, p2);  // sum c_a c_b f
      A = ad(m1, m2);  // sum c_a f (= sum c_a c_b^2 f)
      B = sb(m1, m2);  // sum c_b f (= sum c_a^2 c_b f)
    };
    group(7, Sxy, Mxy, Xxy, Yxy);
    group(11, Sxz, Mxz, Xxz, Zxz);
    group(15, Syz, Myz, Yyz, Zyz);
  }
  const T jx = ad(ad(Bx, Xxy), Xxz), jy = ad(ad(By, Yxy), Yyz), jz = ad(ad(Bz, Zxz), Zyz);
  const T m200 = ad(ad(Ax, Sxy), Sxz), m020 = ad(ad(Ay, Sxy), Syz), m002 = ad(ad(Az, Sxz), Syz);
  // ---- central moments (deviation form) ----
  const T dt = ml(drho, third), dn = ml(drho, ninth);
  const T rux = ml(rho, ux), ruy = ml(rho, uy), ruz = ml(rho, uz);
  const T k200 = sb(m200, fm(rux, ux, dt)), k020 = sb(m020, fm(ruy, uy, dt)), k002 = sb(m002, fm(ruz, uz, dt));
  const T k110 = sb(Mxy, ml(rux, uy)), k101 = sb(Mxz, ml(rux, uz)), k011 = sb(Myz, ml(ruy, uz));
  const T uxx = ml(ux, ux), uyy = ml(uy, uy), uzz = ml(uz, uz);
  const T s1 = C.cum1[0];
  const T inv_rho = recip(rho);
  const T p110 = ml(s1, k110), p101 = ml(s1, k101), p011 = ml(s1, k011);
  const T d1 = ml(s1, sb(k200, k020)), d2 = ml(s1, sb(k200, k002));
  // relaxed second-order (deviatoric with 1 - 1/tau, trace with 1 - omega_bulk),
  // third-order (k_aab) and fourth-order (k^_aabb) central moments
  T p200, p020, p002, p210 = T(0), p120 = T(0), p201 = T(0), p102 = T(0), p021 = T(0), p012 = T(0);
  T p220, p202, p022;
  // k^_aabb of a Gaussian-like closure: (p_aa + p_bb)/3 + (p_aa p_bb + 2 p_ab^2)/rho
  auto closure = [&](T paa, T pbb, T pab) {
    return fm(third, ad(paa, pbb), ml(fm(paa, pbb, ml(ml(T(2), pab), pab)), inv_rho));
  };
  if constexpr (UNIT) {
    // bulk, third- and fourth-order rates 1: trace, third-order and fourth-order
    // cumulants take their equilibrium values (0 in deviation form)
    p200 = ml(ad(d1, d2), third);
    p020 = ml(fm(T(-2), d1, d2), third);
    p002 = ml(fm(T(-2), d2, d1), third);
    p220 = closure(p200, p020, p110);
    p202 = closure(p200, p002, p101);
    p022 = closure(p020, p002, p011);
  } else {
    const T b1 = C.cum1[1], t1 = C.cum1[2], q1 = C.cum1[3];
    const T r0t = ml(C.rho0, third);
    const T M200 = ad(m200, r0t), M020 = ad(m020, r0t), M002 = ad(m002, r0t);  // full raw c_a^2 moments
    const T n2ux = ml(T(-2), ux), n2uy = ml(T(-2), uy), n2uz = ml(T(-2), uz);
    // k_aab = m_aab - u_b M_aa - 2 u_a k_ab
    const T k210 = fm(n2ux, k110, fm(-uy, M200, Yxy)), k120 = fm(n2uy, k110, fm(-ux, M020, Xxy));
    const T k201 = fm(n2ux, k101, fm(-uz, M200, Zxz)), k102 = fm(n2uz, k101, fm(-ux, M002, Xxz));
    const T k021 = fm(n2uy, k011, fm(-uz, M020, Zyz)), k012 = fm(n2uz, k011, fm(-uy, M002, Yyz));
    // k^_aabb = (m_aabb - drho/9) - 2 u_b k_aab - 2 u_a k_abb - 4 u_a u_b k_ab - u_b^2 k^_aa
    //           - u_a^2 k^_bb - rho (u_a^2 + u_b^2) / 3 - rho u_a^2 u_b^2
    auto k4 = [&](T S, T kaab, T kabb, T ua, T ub, T uaa, T ubb, T kab, T kaa, T kbb) {
      T r = sb(S, dn);
      r = fm(ml(T(-2), ub), kaab, r);
      r = fm(ml(T(-2), ua), kabb, r);
      r = fm(ml(T(-4), ml(ua, ub)), kab, r);
      r = fm(-ubb, kaa, r);
      r = fm(-uaa, kbb, r);
      r = fm(-ml(rho, third), ad(uaa, ubb), r);
      return fm(-ml(rho, uaa), ubb, r);
    };
    const T k220 = k4(Sxy, k210, k120, ux, uy, uxx, uyy, k110, k200, k020);
    const T k202 = k4(Sxz, k201, k102, ux, uz, uxx, uzz, k101, k200, k002);
    const T k022 = k4(Syz, k021, k012, uy, uz, uyy, uzz, k011, k020, k002);
    const T tr = ml(b1, ad(ad(k200, k020), k002));
    p200 = ml(ad(ad(tr, d1), d2), third);
    p020 = ml(ad(fm(T(-2), d1, tr), d2), third);
    p002 = ml(fm(T(-2), d2, ad(tr, d1)), third);
    p210 = ml(t1, k210), p120 = ml(t1, k120), p201 = ml(t1, k201);
    p102 = ml(t1, k102), p021 = ml(t1, k021), p012 = ml(t1, k012);
    // fourth order: C = k^_aabb - closure(k), relaxed with 1 - omega_4, plus closure(p)
    auto c4 = [&](T k, T kaa, T kbb, T kab) {
      return sb(fm(-third, ad(kaa, kbb), k), ml(fm(kaa, kbb, ml(ml(T(2), kab), kab)), inv_rho));
    };
    p220 = fm(q1, c4(k220, k200, k020, k110), closure(p200, p020, p110));
    p202 = fm(q1, c4(k202, k200, k002, k101), closure(p200, p002, p101));
    p022 = fm(q1, c4(k022, k020, k002, k011), closure(p020, p002, p011));
  }
  // ---- raw moments of the result (shifted PDFs) ----
  const T n200 = fm(rux, ux, ad(p200, dt)), n020 = fm(ruy, uy, ad(p020, dt)), n002 = fm(ruz, uz, ad(p002, dt));
  const T n110 = fm(rux, uy, p110), n101 = fm(rux, uz, p101), n011 = fm(ruy, uz, p011);
  const T rt = ml(rho, third);
  const T F200 = fm(rux, ux, ad(p200, rt)), F020 = fm(ruy, uy, ad(p020, rt)), F002 = fm(ruz, uz, ad(p002, rt));
  const T n2 = T(2);
  // m_aab = k_aab + u_b F_aa + 2 u_a k_ab
  auto b3 = [&](T paab, T ub, T Faa, T ua, T pab) {
    if constexpr (UNIT) return fm(ml(n2, ua), pab, ml(ub, Faa));
    else return fm(ml(n2, ua), pab, fm(ub, Faa, paab));
  };
  const T n210 = b3(p210, uy, F200, ux, p110), n120 = b3(p120, ux, F020, uy, p110);
  const T n201 = b3(p201, uz, F200, ux, p101), n102 = b3(p102, ux, F002, uz, p101);
  const T n021 = b3(p021, uz, F020, uy, p011), n012 = b3(p012, uy, F002, uz, p011);
  // m_aabb = k^_aabb + drho/9 + 2 u_b k_aab + 2 u_a k_abb + 4 u_a u_b k_ab + u_b^2 (k^_aa + rho/3)
  //          + u_a^2 (k^_bb + rho/3) + rho u_a^2 u_b^2
  auto b4 = [&](T k, T kaab, T kabb, T ua, T ub, T uaa, T ubb, T kab, T kaa, T kbb) {
    T r = ad(k, dn);
    if constexpr (!UNIT) {
      r = fm(ml(n2, ub), kaab, r);
      r = fm(ml(n2, ua), kabb, r);
    }
    r = fm(ml(T(4), ml(ua, ub)), kab, r);
    r = fm(ubb, ad(kaa, rt), r);
    r = fm(uaa, ad(kbb, rt), r);
    return fm(ml(rho, uaa), ubb, r);
  };
  const T n220 = b4(p220, p210, p120, ux, uy, uxx, uyy, p110, p200, p020);
  const T n202 = b4(p202, p201, p102, ux, uz, uxx, uzz, p101, p200, p002);
  const T n022 = b4(p022, p021, p012, uy, uz, uyy, uzz, p011, p020, p002);
  // ---- PDFs ----
  const T qtr = T(0.25), hf = T(0.5);
  auto ungroup = [&](int k, T S, T M, T A, T B) {
    const T a = ad(S, M), b = sb(S, M), p = ad(A, B), q = sb(A, B);
    f[k] = ml(qtr, ad(a, p));
    f[k + 1] = ml(qtr, sb(a, p));
    f[k + 2] = ml(qtr, ad(b, q));
    f[k + 3] = ml(qtr, sb(b, q));
  };
  ungroup(7, n220, n110, n120, n210);
  ungroup(11, n202, n101, n102, n201);
  ungroup(15, n022, n011, n012, n021);
  auto axis = [&](int k, T e, T o) {
    f[k] = ml(hf, ad(e, o));
    f[k + 1] = ml(hf, sb(e, o));
  };
  axis(1, sb(sb(n200, n220), n202), sb(sb(jx, n120), n102));
  axis(3, sb(sb(n020, n220), n022), sb(sb(jy, n210), n012));
  axis(5, sb(sb(n002, n202), n022), sb(sb(jz, n201), n021));
  f[0] = ad(ad(ad(sb(sb(sb(drho, n200), n020), n002), n220), n202), n022);
}

// One cell's PSM update in registers, from its pre-collision (shifted) PDFs f:
// remap (Sec. 3), B (Eq. 5/6), moments, u_s = omega x r + v, Omega^F (Eq. 2 /
// TRT), Omega^S (Eq. 7/8/9), blend (Eq. 4).  f becomes the post-collision
// state.  For a cell in contact with a body (B > 0) ft receives the force and
// torque on the body (minus Eq. 10 / 11 per cell, about R_n).  A cell with
// B = 0 takes exactly the arithmetic of fluid_relax.
template <class T, int Q, int FL>
__device__ __forceinline__ void psm_collide(const StepParams& p, const DevBody* bodies, T (&f)[Q], int x, int y,
                                            int z, unsigned cell, int& owner, bool& solid_cell, ft_t<T> (&ft)[6]) {
  // (x, y, z): world cell indices (z includes the slab offset); cell: this grid's index
  const ConstT<T>& C = cst<T>(p);
  const T om_a = C.om_a, om_b = C.om_b;
  const T inv_tau = C.inv_tau;
  // ---- remap (Sec. 3) and weighting (Eq. 5/6) ----
  // Every operation below is separately rounded (r_*): a PSM cell gets the
  // same bits in every kernel and loop shape that inlines this function.
  const float epsf = cell_eps(bodies, p.nbodies, x, y, z, owner);
  T eps = T(epsf);
  if (p.delta) eps = r_add(eps, T(p.delta[cell]));
  T Bw = eps;
  if (p.weighting == PSM_B_TAU_WEIGHTED && eps != T(0)) {  // eps = 0 gives B = eps exactly
    const T t = C.tmh;
    Bw = r_div(r_mul(eps, t), r_add(r_sub(T(1), eps), t));
  }
  T drho, rho, ux, uy, uz, uu;
  moments<T, Q>(f, C.rho0, drho, rho, ux, uy, uz, uu);
  solid_cell = Bw != T(0);
  if (!solid_cell) {
    fluid_relax<T, Q, FL>(C, f, drho, rho, ux, uy, uz, uu);
    return;
  }
  // ---- PSM cell: f* = f + (1 - B) Omega^F + B Omega^S (Eq. 4) ----
  T usx = 0, usy = 0, usz = 0;
  T rx = 0, ry = 0, rz = 0;  // lever arm x_c - R (Eq. 11)
  if (owner >= 0) {
    const DevBody& b = bodies[owner];
    T wx, wy, wz, vx, vy, vz;
    if constexpr (sizeof(T) == 4) {
      rx = r_sub(r_add(T(x), T(0.5)), b.Rf[0]);
      ry = r_sub(r_add(T(y), T(0.5)), b.Rf[1]);
      rz = r_sub(r_add(T(z), T(0.5)), b.Rf[2]);
      wx = b.omegaf[0], wy = b.omegaf[1], wz = b.omegaf[2];
      vx = b.vf[0], vy = b.vf[1], vz = b.vf[2];
    } else {
      rx = r_sub(r_add((double)x, 0.5), b.R[0]);
      ry = r_sub(r_add((double)y, 0.5), b.R[1]);
      rz = r_sub(r_add((double)z, 0.5), b.R[2]);
      wx = b.omega[0], wy = b.omega[1], wz = b.omega[2];
      vx = b.v[0], vy = b.v[1], vz = b.v[2];
    }
    // u_s = omega x r + v (Eq. 7-9)
    usx = r_add(r_sub(r_mul(wy, rz), r_mul(wz, ry)), vx);
    usy = r_add(r_sub(r_mul(wz, rx), r_mul(wx, rz)), vy);
    usz = r_add(r_sub(r_mul(wx, ry), r_mul(wy, rx)), vz);
  }
  const T usus = r_fma(usz, usz, r_fma(usy, usy, r_mul(usx, usx)));
  const T omB = r_sub(T(1), Bw);
  // cumulant: Omega^F = C(f) - f from the relaxed copy fc
  T fc[Q];
  if constexpr (FL == 2) {
#pragma unroll
    for (int i = 0; i < Q; ++i) fc[i] = f[i];
    fluid_relax<T, Q, FL>(C, fc, drho, rho, ux, uy, uz, uu);
  }
  T gx = 0, gy = 0, gz = 0;  // sum_i Omega^S_i c_i
  if constexpr (FL == 2) {
    {
      const T n0 = r_sub(f[0], feq_shifted_r<Q, T>(0, drho, rho, ux, uy, uz, uu));
      const T m0 = r_sub(f[0], feq_shifted_r<Q, T>(0, drho, rho, usx, usy, usz, usus));
      const T of = r_sub(fc[0], f[0]);
      T os;
      if (p.solid == PSM_SC1) os = r_sub(n0, m0);
      else if (p.solid == PSM_SC2) os = r_mul(-m0, inv_tau);
      else os = T(0);
      f[0] = r_fma(Bw, os, r_fma(omB, of, f[0]));
    }
#pragma unroll
    for (int i = 1; i < Q; i += 2) {
      const int j = i + 1;
      const T ni = r_sub(f[i], feq_shifted_r<Q, T>(i, drho, rho, ux, uy, uz, uu));
      const T nj = r_sub(f[j], feq_shifted_r<Q, T>(j, drho, rho, ux, uy, uz, uu));
      const T mi = r_sub(f[i], feq_shifted_r<Q, T>(i, drho, rho, usx, usy, usz, usus));
      const T mj = r_sub(f[j], feq_shifted_r<Q, T>(j, drho, rho, usx, usy, usz, usus));
      const T ofi = r_sub(fc[i], f[i]), ofj = r_sub(fc[j], f[j]);
      T osi, osj;
      if (p.solid == PSM_SC1) {
        osi = r_sub(nj, mi);
        osj = r_sub(ni, mj);
      } else if (p.solid == PSM_SC2) {
        osi = r_mul(-mi, inv_tau);
        osj = r_mul(-mj, inv_tau);
      } else {
        osi = r_sub(mj, mi);
        osj = r_sub(mi, mj);
      }
      f[i] = r_fma(Bw, osi, r_fma(omB, ofi, f[i]));
      f[j] = r_fma(Bw, osj, r_fma(omB, ofj, f[j]));
      // c_j = -c_i: sum_i Omega^S_i c_i over the pair
      const T d = r_sub(osi, osj);
      if (lat_cx(i)) gx = r_addc(gx, lat_cx(i), d);
      if (lat_cy(i)) gy = r_addc(gy, lat_cy(i), d);
      if (lat_cz(i)) gz = r_addc(gz, lat_cz(i), d);
    }
  } else {
    // BGK / TRT in pair form (c_j = -c_i).  With s = f_i + f_j, d = f_i - f_j
    // and the equilibria split into even and odd parts, f^eq_i,j - w rho0 =
    // ev +- od at u and evs +- ods at u_s, the half sums and differences
    //   n+ = s/2 - ev, n- = d/2 - od,  m+ = s/2 - evs, m- = d/2 - ods
    // give Omega^F_i,j = -omega+ n+ -+ omega- n- and
    //   SC1: Omega^S_i,j = n_j - m_i, n_i - m_j = (n+ - m+) +- (-n- - m-),
    //   SC2: -(m+ +- m-) / tau,   SC3: m_j - m_i, m_i - m_j = +-(-2 m-);
    // then f*_i,j = P +- M with P = s/2 + (1 - B) OmF+ + B OmS+ and
    // M = d/2 + (1 - B) OmF- + B OmS-, and the pair adds 2 OmS- c_i to
    // sum_i Omega^S_i c_i.
    const T wp = r_add(om_a, om_b), wm = r_sub(om_a, om_b);
    const T bu = r_fma(T(-1.5), r_mul(rho, uu), drho), bs = r_fma(T(-1.5), r_mul(rho, usus), drho);
    {
      const T w0 = T(lat_w<Q>(0));
      const T n0 = r_fma(-w0, bu, f[0]), m0 = r_fma(-w0, bs, f[0]);
      T os;
      if (p.solid == PSM_SC1) os = r_sub(n0, m0);
      else if (p.solid == PSM_SC2) os = r_mul(-m0, inv_tau);
      else os = T(0);
      f[0] = r_fma(Bw, os, r_fma(omB, r_mul(-wp, n0), f[0]));
    }
#pragma unroll
    for (int i = 1; i < Q; i += 2) {
      const int j = i + 1;
      const T w = T(lat_w<Q>(i));
      const T wr = r_mul(w, rho);
      const T cu = c_dot(i, ux, uy, uz), cs = c_dot(i, usx, usy, usz);
      const T k45 = r_mul(T(4.5), wr), k3 = r_mul(T(3), wr);
      const T ev = r_fma(k45, r_mul(cu, cu), r_mul(w, bu)), od = r_mul(k3, cu);
      const T evs = r_fma(k45, r_mul(cs, cs), r_mul(w, bs)), ods = r_mul(k3, cs);
      const T hs = r_mul(T(0.5), r_add(f[i], f[j])), hd = r_mul(T(0.5), r_sub(f[i], f[j]));
      const T np = r_sub(hs, ev), nm = r_sub(hd, od), mp = r_sub(hs, evs), mm = r_sub(hd, ods);
      T sp, sm;
      if (p.solid == PSM_SC1) {
        sp = r_sub(np, mp);
        sm = r_sub(-nm, mm);
      } else if (p.solid == PSM_SC2) {
        sp = r_mul(-mp, inv_tau);
        sm = r_mul(-mm, inv_tau);
      } else {
        sp = T(0);
        sm = r_mul(T(-2), mm);
      }
      const T P = r_fma(Bw, sp, r_fma(omB, r_mul(-wp, np), hs));
      const T M = r_fma(Bw, sm, r_fma(omB, r_mul(-wm, nm), hd));
      f[i] = r_add(P, M);
      f[j] = r_sub(P, M);
      const T d = r_mul(T(2), sm);
      if (lat_cx(i)) gx = r_addc(gx, lat_cx(i), d);
      if (lat_cy(i)) gy = r_addc(gy, lat_cy(i), d);
      if (lat_cz(i)) gz = r_addc(gz, lat_cz(i), d);
    }
  }
  if (owner >= 0) {
    // Eq. 10 / 11 per cell, in the arithmetic's precision (ft_t); the body
    // receives minus the solid's momentum transfer
    const T Gx = r_mul(Bw, gx), Gy = r_mul(Bw, gy), Gz = r_mul(Bw, gz);
    ft[0] = -Gx;
    ft[1] = -Gy;
    ft[2] = -Gz;
    ft[3] = -r_sub(r_mul(ry, Gz), r_mul(rz, Gy));
    ft[4] = -r_sub(r_mul(rz, Gx), r_mul(rx, Gz));
    ft[5] = -r_sub(r_mul(rx, Gy), r_mul(ry, Gx));
  }
}

// Streaming indices of one cell: the index of x + c for c in {-1, 0, 1}^3 is
// zc[cz + 1] + dy[cy + 1] + dx[cx + 1] (mod 2^32; cell indices are < 2^32),
// periodic in x and y, and in z (where z ends in ghost planes the callers
// drop the populations that cross them).
struct Stencil {
  unsigned zc[3], dy[3], dx[3];
  __device__ __forceinline__ void init(const Grid3& g, int x, int y, int z, unsigned cell) {
    const unsigned nx = (unsigned)g.nx, plane = (unsigned)g.nx * (unsigned)g.ny;
    dx[0] = (x == 0) ? nx - 1u : 0u - 1u;
    dx[1] = 0u;
    dx[2] = (x == g.nx - 1) ? 0u - (nx - 1u) : 1u;
    dy[0] = (y == 0) ? (unsigned)(g.ny - 1) * nx : 0u - nx;
    dy[1] = 0u;
    dy[2] = (y == g.ny - 1) ? 0u - (unsigned)(g.ny - 1) * nx : nx;
    zc[0] = cell + ((z == 0) ? (unsigned)(g.nz - 1) * plane : 0u - plane);
    zc[1] = cell;
    zc[2] = cell + ((z == g.nz - 1) ? 0u - (unsigned)(g.nz - 1) * plane : plane);
  }
  __device__ __forceinline__ unsigned at(int cx, int cy, int cz) const { return zc[cz + 1] + dy[cy + 1] + dx[cx + 1]; }
};

// Position of a z plane against the ghost planes (never set for periodic z).
struct ZGhost {
  bool lo, hi;  // z - 1 (resp. z + 1) lies in a ghost plane
  __device__ __forceinline__ void init(const Grid3& g, int z) {
    const bool ghost = g.bc_z == PSM_BC_EQ_INLET_OUTLET;
    lo = ghost && z == 0;
    hi = ghost && z == g.nz - 1;
  }
  // x - c_i lies in a ghost plane: population i enters from it
  __device__ __forceinline__ bool from(int cz) const { return (cz > 0 && lo) || (cz < 0 && hi); }
  // x + c_i lies in a ghost plane: population i leaves the domain
  __device__ __forceinline__ bool to(int cz) const { return (cz > 0 && hi) || (cz < 0 && lo); }
};

// Streamed store (Eq. 1) of one cell's post-collision PDFs:
//   AA even  own cell, slot opp(i);
//   AA odd   cell x + c_i, slot i;
//   TG       cell x + c_i, slot i of the other buffer;
// with GHOST, populations that leave the domain through a ghost plane are dropped.
template <class S, int Q, int MODE, bool GHOST, class T>
__device__ __forceinline__ void psm_store(const StepParams& p, const Stencil& sn, const ZGhost& zg, unsigned cell,
                                          const T (&f)[Q]) {
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    if (MODE == MODE_AA_EVEN) {
      Store<S>::st(static_cast<S*>(p.dst_slot[lat_opp(i)]) + cell, f[i]);
    } else if (!GHOST || !zg.to(lat_cz(i))) {
      Store<S>::st(static_cast<S*>(p.dst_slot[i]) + sn.at(lat_cx(i), lat_cy(i), lat_cz(i)), f[i]);
    }
  }
}

// Pre-collision PDFs of one cell with plain global loads (AA odd: population i
// of x was stored by x - c_i in slot opp(i); otherwise slot i of x); with
// GHOST, populations entering from a ghost plane take the ghost value.
template <class S, int Q, int MODE, bool GHOST, class T>
__device__ __forceinline__ void psm_load(const StepParams& p, const Stencil& sn, const ZGhost& zg, unsigned cell,
                                         T (&f)[Q]) {
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int cx = lat_cx(i), cy = lat_cy(i), cz = lat_cz(i);
    if (GHOST && zg.from(cz)) {
      f[i] = cst<T>(p).ghost[i];
    } else if (MODE == MODE_AA_ODD) {
      f[i] = Store<S>::ld(static_cast<const S*>(p.src_slot[lat_opp(i)]) + sn.at(-cx, -cy, -cz));
    } else {
      f[i] = Store<S>::ld(static_cast<const S*>(p.src_slot[i]) + cell);
    }
  }
}

// Per-warp force/torque accumulation into s_ft[warp] (fixed order: warp
// butterfly in the contribution's precision, then added in FP64 in tile
// order).  All 32 lanes must call it.
template <class V>
__device__ __forceinline__ void warp_ft(double (*s_ft)[PSM_MAX_BODIES * 6], int nb, bool contributes, int owner,
                                        const V (&ft)[6]) {
  if (nb == 0 || !__any_sync(0xffffffffu, contributes)) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int bi = 0; bi < nb; ++bi) {
    const bool mine = contributes && owner == bi;
    if (!__any_sync(0xffffffffu, mine)) continue;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const V v = warp_sum(mine ? ft[k] : V(0));
      if (lane == 0) s_ft[warp][bi * 6 + k] += (double)v;
    }
  }
}

// Block sum of the per-warp slots (fixed order), stored for k_reduce_slots.  A
// grid-wide sum by the last block of every step was a tail that nothing
// overlapped (fences, a ticket, one block's loads: about 5 us).
template <int NT = PSM_THREADS>
__device__ __forceinline__ void block_ft_finish(double (*s_ft)[PSM_MAX_BODIES * 6], const StepParams& p) {
  __syncthreads();
  const int c = (int)threadIdx.x, ncomp = p.nft * 6;
  if (c < ncomp) {
    double s = 0.0;
    for (int w = 0; w < NT / 32; ++w) s += s_ft[w][c];
    p.ft_slot[1 + (long long)blockIdx.x * ncomp + c] = s;
  }
  if (blockIdx.x == 0 && c == 0) p.ft_slot[0] = (double)gridDim.x;
}

// (tile index t -> (tx, ty, z)) and its increment by a decomposed step
__device__ __forceinline__ int4 tile_split(const Tiling& t, int tile) {
  return make_int4(tile % t.ntx, (tile / t.ntx) % t.nty, tile / t.ntx / t.nty, 0);
}
__device__ __forceinline__ int4 tile_advance(const Tiling& t, int4 cur, int4 step) {
  cur.x += step.x;
  int c = cur.x >= t.ntx;
  cur.x -= c ? t.ntx : 0;
  cur.y += step.y + c;
  c = cur.y >= t.nty;
  cur.y -= c ? t.nty : 0;
  cur.z += step.z + c;
  return cur;
}

// Programmatic dependent launch: when every block of a step kernel has finished
// its cells the next kernel may start, and does everything that needs no memory
// of earlier kernels (barriers, walks, the bodies of the launch parameters)
// before it waits for them to end.  Every thread of every block waits, so that a
// kernel ends after its predecessors, and what follows it in the stream is
// ordered after all of them.
__device__ __forceinline__ void grid_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The bodies of this step, copied to shared memory at block start: from the
// launch parameters, or, for bodies whose motion the device integrates
// (two-way coupling), from device memory.  The caller synchronises the block.
__device__ __forceinline__ void load_bodies(const StepParams& p, DevBody* s_body) {
  static_assert(sizeof(DevBody) % 4 == 0, "DevBody is copied in 4-byte words");
  constexpr int W = (int)(sizeof(DevBody) / 4);
  for (int k = threadIdx.x; k < p.nbodies * W; k += blockDim.x) {
    const int b = k / W, w = k % W;
    const DevBody* src = ((p.free_mask >> b) & 1u) ? &p.dbody[b] : &p.body[b];
    reinterpret_cast<unsigned*>(&s_body[b])[w] = reinterpret_cast<const unsigned*>(src)[w];
  }
}

// A tile (TX x TY cells of one z plane) takes the fluid-only path when no
// body's cell box meets it, no eps perturbation is set and its plane is not
// next to a ghost plane: every cell of such a tile has B = 0, and no
// population of it enters or leaves through a ghost plane.
__device__ __forceinline__ bool tile_general(const StepParams& p, const DevBody* bodies, int x0, int y0, int z, int TX,
                                             int TY) {
  bool gen = p.delta != nullptr || (p.g.bc_z == PSM_BC_EQ_INLET_OUTLET && (z == 0 || z == p.g.nz - 1));
  const int zw = z + p.g.z0;  // world z of the plane (the body boxes are in world cells)
#pragma unroll
  for (int bi = 0; bi < PSM_MAX_BODIES; ++bi) {
    if (bi < p.nbodies) {
      const DevBody& b = bodies[bi];
      gen = gen || (x0 < b.x1 && x0 + TX > b.x0 && y0 < b.y1 && y0 + TY > b.y0 && zw >= b.z0 && zw < b.z1);
    }
  }
  return gen;
}

template <bool B>
struct BoolC {
  static constexpr bool value = B;
};

// One cell of a fluid-only tile: moments and Omega^F (the arithmetic psm_collide
// takes for B = 0).
template <class T, int Q, int FL>
__device__ __forceinline__ void fluid_collide(const StepParams& p, T (&f)[Q]) {
  const ConstT<T>& C = cst<T>(p);
  T drho, rho, ux, uy, uz, uu;
  moments<T, Q>(f, C.rho0, drho, rho, ux, uy, uz, uu);
  fluid_relax<T, Q, FL>(C, f, drho, rho, ux, uy, uz, uu);
}

// Two cells of fluid-only tiles: the cumulant in packed FP32 instructions (see
// tile_pairs), BGK and TRT one cell after the other, the same bits either way
// (packed, D3Q19 took 13.85 ms at 1024x1024x960, one by one 13.67, and D3Q27 was
// no faster).
template <int Q, int FL>
__device__ __forceinline__ void fluid_collide2(const StepParams& p, F2 (&f)[Q]) {
  if constexpr (FL == 2) {
    F2 drho, rho, ux, uy, uz, uu;
    moments<F2, Q>(f, F2(p.cf.rho0), drho, rho, ux, uy, uz, uu);
    fluid_relax<F2, Q, FL>(p.cf, f, drho, rho, ux, uy, uz, uu);
  } else {
    float a[Q], b[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) a[i] = f[i].v.x, b[i] = f[i].v.y;
    fluid_collide<float, Q, FL>(p, a);
    fluid_collide<float, Q, FL>(p, b);
#pragma unroll
    for (int i = 0; i < Q; ++i) f[i] = F2(a[i], b[i]);
  }
}

// ---------------------------------------------------------------------------
// The fused step kernel with plain global loads, any grid shape.  A warp's unit
// of work is 32 neighbouring cells of one row (the last unit of a row holds the
// remainder), and the warps of the persistent blocks stride over the units in
// memory order: no lane is idle but in the rows' last units (blocks of whole
// 256-cell tiles left 21-25 % of the lanes idle on rows of 203 and 96 cells).
// y and z are the warp's, and advance by the stride's own decomposition, without
// divisions.  A warp takes the fluid-only path when its unit meets no body's
// cell box, lies in no plane next to a ghost plane and no eps perturbation is
// set (tile_general, for its 32 cells).  The force/torque partials are those of
// 32 x-neighbours whatever the block size; where the TMA kernel applies, blocks
// of 256 hold its tiles' cells in the same order, so that in FP32 and FP64
// storage the sums agree bit for bit (in 16-bit storage its warps hold other
// cells).  96x96x120 D3Q27 FP32 with two rotors: 67 us a step in whole-row tiles,
// 58 us in units; 203x117x151 FP16 88 and 85 us.
// ---------------------------------------------------------------------------
template <class S, int Q, int MODE, int FL, int NT>
__global__ void __launch_bounds__(NT, step_min_blocks<S, Q, FL>() * PSM_THREADS / NT)
    k_step(const __grid_constant__ StepParams p) {
  using T = typename Store<S>::T;
  __shared__ double s_ft[NT / 32][PSM_MAX_BODIES * 6];
  __shared__ DevBody s_body[PSM_MAX_BODIES];
  const int nb = p.nft;  // bodies whose loads are wanted
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int k = lane; k < PSM_MAX_BODIES * 6; k += 32) s_ft[warp][k] = 0.0;
  if (p.free_mask) grid_wait_previous();  // the previous kernel advances the free bodies
  load_bodies(p, s_body);
  __syncthreads();
  grid_wait_previous();

  auto cell_body = [&](auto gen_c, bool active, int x, int y, int z, unsigned cell) {
    constexpr bool GEN = decltype(gen_c)::value;
    int owner = -1;
    bool solid_cell = false;
    ft_t<T> ft[6] = {0, 0, 0, 0, 0, 0};
    if (active) {
      Stencil sn;
      sn.init(p.g, x, y, z, cell);
      ZGhost zg;
      zg.init(p.g, z);
      T f[Q];
      psm_load<S, Q, MODE, GEN>(p, sn, zg, cell, f);
      if (GEN) psm_collide<T, Q, FL>(p, s_body, f, x, y, z + p.g.z0, cell, owner, solid_cell, ft);
      else fluid_collide<T, Q, FL>(p, f);
      if (MODE == MODE_AA_ODD) {
        // rebuild the stencil for the stores rather than keep it live through
        // the collision (register pressure); the empty asm hides the equality
        // of the inputs from common-subexpression elimination
        int xs = x, ys = y, zs = z;
        unsigned cs = cell;
        asm volatile("" : "+r"(xs), "+r"(ys), "+r"(zs), "+r"(cs));
        Stencil sn2;
        sn2.init(p.g, xs, ys, zs, cs);
        psm_store<S, Q, MODE, GEN>(p, sn2, zg, cs, f);
      } else {
        psm_store<S, Q, MODE, GEN>(p, sn, zg, cell, f);
      }
    }
    if (GEN) warp_ft(s_ft, nb, active && solid_cell && owner >= 0, owner, ft);
  };

  // this warp's unit and the stride over units, both as (x unit, y, z)
  constexpr int NW = NT / 32;
  const unsigned nxu = ((unsigned)p.g.nx + 31u) / 32u, ny = (unsigned)p.g.ny;
  const unsigned long long units = (unsigned long long)nxu * ny * (unsigned)p.g.nz;
  const unsigned stride = gridDim.x * (unsigned)NW, u0 = blockIdx.x * (unsigned)NW + (unsigned)warp;
  int xu = (int)(u0 % nxu), y = (int)(u0 / nxu % ny), z = (int)(u0 / nxu / ny);
  const int gx = (int)(stride % nxu), gy = (int)(stride / nxu % ny), gz = (int)(stride / nxu / ny);
  for (unsigned long long u = u0; u < units; u += stride) {
    const int x0 = xu * 32, x = x0 + lane;
    const unsigned cell = ((unsigned)z * ny + (unsigned)y) * (unsigned)p.g.nx + (unsigned)x;
    if (tile_general(p, s_body, x0, y, z, 32, 1)) cell_body(BoolC<true>{}, x < p.g.nx, x, y, z, cell);
    else cell_body(BoolC<false>{}, x < p.g.nx, x, y, z, cell);
    xu += gx;
    int c = xu >= (int)nxu;
    xu -= c ? (int)nxu : 0;
    y += gy + c;
    c = y >= p.g.ny;
    y -= c ? p.g.ny : 0;
    z += gz + c;
  }
  grid_launch_next();
  if (nb == 0) return;
  block_ft_finish<NT>(s_ft, p);
}

// Most input stages of the TMA step kernel (the stage count follows from the
// shared memory per SM, see TmaLayout).
#ifndef PSM_TMA_MAX_STAGES
#define PSM_TMA_MAX_STAGES 8
#endif

__device__ __forceinline__ unsigned smem_u32(const void* ptr) {
  return (unsigned)__cvta_generic_to_shared(ptr);
}
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
  asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred P;\n mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 P, [%1], %2;\n selp.u32 %0, 1, 0, P;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0u;
}
// try_wait with a suspend-time hint: the thread may stop issuing until the
// phase completes or about `ns` nanoseconds have passed
__device__ __forceinline__ bool mbar_try_wait_sleep(unsigned long long* bar, unsigned parity, unsigned ns) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred P;\n mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 P, [%1], %2, %3;\n selp.u32 %0, 1, 0, P;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(ns)
      : "memory");
  return ok != 0u;
}
__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait for a phase: one poll, then suspended polls until the phase
// completes, 100 ms pass (global timer) or 2^22 polls were made; false if the
// phase did not complete.
__device__ __forceinline__ bool mbar_wait_bounded(unsigned long long* bar, unsigned parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = globaltimer_ns();
  for (unsigned it = 0; it < (1u << 22); ++it) {
    if (mbar_try_wait_sleep(bar, parity, 20000u)) return true;
    if (globaltimer_ns() - t0 > 100000000ull) return false;
  }
  return false;
}
__device__ __forceinline__ void tma_load_4d(void* dst, const void* map, int c0, int c1, int c2, int c3,
                                            unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
      "[%6];" ::"r"(smem_u32(dst)),
      "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void bulk_load_16(void* dst, const void* src, unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], 16, [%2];" ::"r"(smem_u32(dst)),
      "l"(src), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

__device__ __forceinline__ void tma_store_4d(const void* map, int c0, int c1, int c2, int c3, const void* src) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3, %4}], [%5];" ::"l"(map),
               "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(src))
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// output boxes per warp (AA even), where the shared memory allows it
#ifndef PSM_TMA_OUT_BUFS
#define PSM_TMA_OUT_BUFS 2
#endif


// Lattice components for a run-time direction index (the producer's copy
// jobs): c + 1 in two bits per direction.
__host__ __device__ constexpr unsigned long long lat_bits(int axis) {
  unsigned long long b = 0;
  for (int i = 0; i < 27; ++i)
    b |= (unsigned long long)((axis == 0 ? lat_cx(i) : (axis == 1 ? lat_cy(i) : lat_cz(i))) + 1) << (2 * i);
  return b;
}
constexpr unsigned long long kLatCX = lat_bits(0), kLatCY = lat_bits(1), kLatCZ = lat_bits(2);
__device__ __forceinline__ int lat_c_rt(unsigned long long bits, int i) { return (int)((bits >> (2 * i)) & 3ull) - 1; }

// Shared-memory layout of the TMA step kernel (bytes; every box 128-byte
// aligned): [barriers 128 B] [NST input stages] [NOUT output buffers].
//   input, own-cell modes (two-grid, AA even): one [Q][TY][TX] box per tile
//     (TX TY = 256 CPT): slot i of cell r of thread t at element
//     256 CPT i + 256 r + t;
//   input, AA odd (TX = 256, TY = 1): per direction i the 256 values of slot
//     opp(i) at x - c_i for the tile's cells at byte 128 + i ROW, preceded and
//     followed by a 16-byte x-edge chunk, so that cell lx reads element
//     lx - c_x of it with no branch;
//   output (AA even): per warp a [Q][32] box of its 32 cells (WBOX bytes),
//     written back by the warp's own TMA tensor store.
// The stage count NST fills the shared memory of the resident blocks the
// launch bounds aim at (228 KB per SM, less 1 KB per block reserved and the
// kernel's static shared memory), between 2 and PSM_TMA_MAX_STAGES: deeper
// pipelines for the narrower storage types keep more bytes in flight.  (The
// launch refuses a build whose static shared memory exceeds STATIC_SMEM.)
template <class S, int Q, int MODE, int FL = 0>
struct TmaLayout {
  static constexpr bool LOAD_OWN = MODE != MODE_AA_ODD;
  static constexpr bool STORE_TMA = PSM_TMA_STORE && MODE == MODE_AA_EVEN;
  // cells per thread and tile (tma_cells_per_thread: the host tiles alike)
  static constexpr int CPT = tma_cells_per_thread((int)sizeof(S), MODE, Q, FL);  // FL numbers the fluid like psm.h
  static constexpr int EP = 16 / (int)sizeof(S);  // elements per 16-byte edge chunk
  static constexpr int r128(int b) { return ((b + 127) / 128) * 128; }
  static constexpr int BOX_BYTES = Q * PSM_THREADS * CPT * (int)sizeof(S);
  static constexpr int BOX = r128(BOX_BYTES);
  // AA odd records: direction i's row of 256 values at byte 128 + i ROW of the
  // stage (128-byte aligned), its 16-byte edge chunks right before and after
  // it; ROW >= row + 32 bytes keeps the chunk after one row clear of the chunk
  // before the next (which sits in the last 16 bytes below that row)
  static constexpr int ROW = r128(PSM_THREADS * (int)sizeof(S) + 32);
  static constexpr int STAGE = LOAD_OWN ? BOX : r128(Q * ROW + 16);
  static constexpr int WBOX = r128(Q * 32 * (int)sizeof(S));
  static constexpr int OUT = STORE_TMA ? (PSM_THREADS / 32) * WBOX : 0;
  static constexpr int SM_SMEM = 233472;
  static constexpr int BLOCKS = step_min_blocks<S, Q, FL, MODE>();
  // per block: 1 KB reserved by the hardware and the kernel's static shared
  // memory (about 5 KB: force/torque slots, reduction scratch, the bodies of
  // the step, stage headers), allowed for with 6 KB
  static constexpr int STATIC_SMEM = 6144;
  static constexpr int BUDGET0 = (SM_SMEM - BLOCKS * (1024 + STATIC_SMEM)) / BLOCKS - 256;
  static constexpr int clamp_st(int n) { return n < 2 ? 2 : (n > PSM_TMA_MAX_STAGES ? PSM_TMA_MAX_STAGES : n); }
  // output boxes per warp: PSM_TMA_OUT_BUFS where that leaves at least 3 input stages, else 1
  static constexpr int NOUT = (PSM_TMA_OUT_BUFS > 1 && (BUDGET0 - PSM_TMA_OUT_BUFS * OUT) / STAGE >= 3) ? PSM_TMA_OUT_BUFS : 1;
  // a multiple of the groups of warps that take alternate tiles (tile_pairs): a
  // stage then always belongs to one group, whose own waits order its refills
  static constexpr int GROUPS = tile_pairs<S, FL, MODE>() ? 2 : 1;
  static constexpr int NST = clamp_st((BUDGET0 - NOUT * OUT) / STAGE) / GROUPS * GROUPS;
  // refill lag in tiles: a stage is refilled LAG tiles after it was read, so the
  // refilling warp seldom waits for the slowest warp; NST - LAG tiles stay ahead
  // (a multiple of the groups too: a warp refills stages that its own group has read)
#ifdef PSM_TMA_REFILL_LAG
  static constexpr int LAG0 = PSM_TMA_REFILL_LAG < NST - 1 ? PSM_TMA_REFILL_LAG : NST - 2;
#else
  static constexpr int LAG0 = NST >= 5 ? 2 : (NST >= 3 ? 1 : 0);
#endif
  static constexpr int LAG = LAG0 / GROUPS * GROUPS;
  // + 128 B of barriers, + 128 B of alignment slack
  static constexpr int SMEM = 256 + NST * STAGE + NOUT * OUT;
};

// ---------------------------------------------------------------------------
// TMA-staged step kernel.  Shapes: tiles of TX x TY = 256 CPT cells of one z
// plane with nx % TX == 0 and ny % TY == 0 (TX = min(256, nx), a power of
// two), TX * sizeof(S) a multiple of 16 bytes; the AA odd step needs TX = 256.
// Persistent blocks stride over tiles.  Warp 0 keeps NST tiles of
// pre-collision PDFs in flight in shared memory (two-grid and AA even: one
// cp.async.bulk.tensor box per tile; AA odd: one row per direction plus
// 16-byte cp.async.bulk edge chunks for x - c_x) while all threads collide the
// oldest staged tile from shared memory.  The producer classifies each tile
// (tile_general) and the block takes the fluid-only path or the general one
// for the whole tile.  The two-grid and AA odd steps store to x + c_i with
// st.global; the AA even step stores to the own cells' swapped slots (with
// two cells per thread, the fluid-only tiles' x-neighbour pairs with one
// 32-bit access per slot), or, built with PSM_TMA_STORE, through one TMA
// tensor store per warp.  With tile_pairs a tile is the work of every other warp
// of the block.  No block barrier inside the tile loop.
// ---------------------------------------------------------------------------
template <class S, int Q, int MODE, int FL>
__global__ void __launch_bounds__(PSM_THREADS, step_min_blocks<S, Q, FL, MODE>())
    k_step_tma(const __grid_constant__ StepParams p, const __grid_constant__ TmaMaps maps) {
  using T = typename Store<S>::T;
  using L = TmaLayout<S, Q, MODE, FL>;
  constexpr int NST = L::NST;
  constexpr int NOUT = L::NOUT;
  constexpr int LAG = L::LAG;
  constexpr int EP = L::EP;
  __shared__ double s_ft[PSM_THREADS / 32][PSM_MAX_BODIES * 6];
  __shared__ int s_abort;
  __shared__ int s_issued[NST];  // loads issued per stage (warp 0, lane 0)
  __shared__ int4 s_hdr[NST];    // per stage: tile origin x0, y0, z and the general-path flag
  __shared__ DevBody s_body[PSM_MAX_BODIES];
  extern __shared__ __align__(128) unsigned char smem_raw[];
  // dynamic shared memory is only guaranteed 16-byte alignment: align by hand
  unsigned char* base = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
  // barriers in the first 128 B: full[s] completes when stage s holds its tile
  // (the producer's arrival plus the copied bytes); empty[s] when every warp has
  // read it (one arrival per warp)
  unsigned long long* full = reinterpret_cast<unsigned long long*>(base);
  unsigned long long* empty = full + NST;
  static_assert(2 * NST * 8 <= 128, "stage barriers exceed their 128 bytes");
  constexpr int NW = PSM_THREADS / 32;
  // tile_pairs: the even warps take the block's even tiles and the odd warps its
  // odd ones, two x-neighbour cells per thread; otherwise all warps share each tile
  constexpr bool PAIRS = tile_pairs<S, FL, MODE>();
  constexpr int GROUPS = L::GROUPS;
  static_assert(NST >= GROUPS && NST % GROUPS == 0 && LAG % GROUPS == 0, "a warp refills stages that its own group has read");
  const int nb = p.nft;  // bodies whose loads are wanted
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int k = lane; k < PSM_MAX_BODIES * 6; k += 32) s_ft[warp][k] = 0.0;
  const int TX = p.t.tx, TY = p.t.ty;
  constexpr int CPT = L::CPT;
  if (p.free_mask || TX * TY != PSM_THREADS * CPT) grid_wait_previous();  // the previous kernel advances the free bodies
  if (TX * TY != PSM_THREADS * CPT) {
    // a tiling this instance was not built for: refuse before any wait or copy
    if (threadIdx.x == 0 && p.err) atomicExch(p.err, 2);
    return;
  }
  const int TYB = TY / CPT;  // rows of the tile covered by one cell per thread
  unsigned char* stages = base + 128;
  unsigned char* outs = stages + NST * L::STAGE;
  const int ntiles = (int)p.t.ntiles;

  if (threadIdx.x == 0) {
    s_abort = 0;
    for (int s = 0; s < NST; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], NW / GROUPS);
      s_issued[s] = 0;
    }
    fence_mbar_init();
  }
  load_bodies(p, s_body);
  __syncthreads();

  // producer: the 32 lanes of one warp stage the pre-collision PDFs of the
  // walk's current tile into stage `s`, one copy job per lane, and advance the
  // walk.  Warp 0 stages the first NST tiles; afterwards warp w refills the
  // stage of tile j when j = w (mod NW), so the producer work rotates over the
  // warps (its walk: tiles w + NST, w + NST + NW, ... of this block).
  // (kept in shared memory, not in registers across the tile loop)
  __shared__ int4 s_walk[NW];  // per warp: the next tile it refills (tx, ty, z)
  __shared__ int4 s_wstep;     // NW * gridDim.x, split like a tile index
  if (lane == 0) s_walk[warp] = tile_split(p.t, blockIdx.x + (warp + NST) * gridDim.x);
  if (threadIdx.x == 0) s_wstep = tile_split(p.t, NW * gridDim.x);
  __syncthreads();
  grid_wait_previous();
  auto produce = [&](const int4 cur, int s) {
    const int z = cur.z;
    const int x0 = cur.x * TX, y0 = cur.y * TY;
    unsigned char* st = stages + s * L::STAGE;
    unsigned long long* bar = &full[s];
    fence_proxy_async();
    if (L::LOAD_OWN) {
      if (lane == 0) {
        mbar_expect_tx(bar, (unsigned)L::BOX_BYTES);
        tma_load_4d(st, &maps.tile, x0, y0, z, 0, bar);
      }
    } else {
      for (int i = lane; i < Q; i += 32) {
        const int cx = lat_c_rt(kLatCX, i), cy = lat_c_rt(kLatCY, i), cz = lat_c_rt(kLatCZ, i);
        int zs = z - cz;
        if (zs < 0 || zs >= p.g.nz) {
          if (p.g.bc_z == PSM_BC_EQ_INLET_OUTLET) continue;  // ghost populations: no load
          zs = zs < 0 ? zs + p.g.nz : zs - p.g.nz;
        }
        int ys = y0 - cy;
        ys = ys < 0 ? ys + p.g.ny : (ys >= p.g.ny ? ys - p.g.ny : ys);
        const int slot = lat_opp(i);
        unsigned char* row = st + i * L::ROW + 128;
        mbar_expect_tx(bar, (unsigned)(PSM_THREADS * (int)sizeof(S)));
        tma_load_4d(row, &maps.row1, x0, ys, zs, slot, bar);
        if (cx != 0) {
          // cx = +1: cell x0 reads x0 - 1 (the chunk before the row, wrapped in x);
          // cx = -1: cell x0 + 255 reads x0 + 256 (the chunk after it)
          const int xe = cx > 0 ? (x0 == 0 ? p.g.nx - EP : x0 - EP) : (x0 + PSM_THREADS == p.g.nx ? 0 : x0 + PSM_THREADS);
          // slot k starts k ncell values after slot 0 (one uniform base for every lane)
          const S* src = static_cast<const S*>(p.src_slot[0]) +
                         (((long long)slot * p.g.nz + zs) * p.g.ny + ys) * p.g.nx + xe;
          mbar_expect_tx(bar, 16u);
          bulk_load_16(cx > 0 ? row - 16 : row + PSM_THREADS * (int)sizeof(S), src, bar);
        }
      }
    }
    if (lane == 0) s_hdr[s] = make_int4(x0, y0, z, tile_general(p, s_body, x0, y0, z, TX, TY) ? 1 : 0);
    __syncwarp();  // every lane's expected bytes are registered before the arrival
    if (lane == 0) {
      mbar_arrive(bar);
      s_issued[s] += 1;
    }
  };

  if (warp == 0) {
    int4 first = tile_split(p.t, blockIdx.x);
    const int4 g1 = tile_split(p.t, gridDim.x);
    for (int k = 0; k < NST; ++k) {
      const int tile = blockIdx.x + k * gridDim.x;
      if (tile < ntiles) produce(first, k);
      first = tile_advance(p.t, first, g1);
    }
  }

  const int lx = threadIdx.x % TX, ly = threadIdx.x / TX;
  const int px = threadIdx.x % (TX / 2), py = threadIdx.x / (TX / 2);

  // One staged tile, read from stage s after its full barrier.  Each warp
  // signals empty[s] once it holds its cells' PDFs in registers; warp 0 then
  // waits for all warps' signals before refilling the stage, so warps do not
  // wait for one another otherwise.  A wait that times out sets s_abort and
  // the warp leaves the tile loop.
  // After the warp holds its cells' PDFs of stage s in registers.
  auto stage_read = [&](int tile, int k, int s) {
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[s]);
    // refill the stage of tile j = k - LAG (read by every warp by now, as a
    // rule) with tile j + NST; warp j mod NW does it
    const int j = k - LAG;
    if (j >= 0 && warp == j % NW) {
      const int next = tile + (NST - LAG) * gridDim.x;
      if (next < ntiles) {
        const int sj = j % NST;
        // warp-uniform outcome (produce needs the whole warp)
        if (__all_sync(0xffffffffu, mbar_wait_bounded(&empty[sj], (unsigned)((j / NST) & 1)))) {
          const int4 cur = s_walk[warp];
          produce(cur, sj);
          if (lane == 0) s_walk[warp] = tile_advance(p.t, cur, s_wstep);
        } else {
          s_abort = 1;
        }
      }
    }
  };

  auto tile_body = [&](auto gen_c, int tile, int k, int s, const int4 hd) {
    constexpr bool GEN = decltype(gen_c)::value;
    const int z = hd.z;
    ZGhost zg;
    zg.init(p.g, z);
    const unsigned char* st = stages + s * L::STAGE;
    // fluid-only tiles of the AA even step in 16-bit storage: the thread's two
    // cells are x neighbours (x even, x + 1), so one 32-bit shared load and one
    // 32-bit store per slot serve both
    constexpr bool XPAIR = !GEN && CPT == 2 && MODE == MODE_AA_EVEN && sizeof(S) == 2 && FL != 2 && !L::STORE_TMA;
    if constexpr (XPAIR) {
      const unsigned* sw = reinterpret_cast<const unsigned*>(st) + (py * TX) / 2 + px;
      F2 f[Q];
#pragma unroll
      for (int i = 0; i < Q; ++i) Pair16<S>::unpack(sw[i * (CPT * PSM_THREADS / 2)], f[i].v.x, f[i].v.y);
      stage_read(tile, k, s);
      fluid_collide2<Q, FL>(p, f);
      const int x = hd.x + 2 * px, y = hd.y + py;
      const unsigned cell = ((unsigned)z * (unsigned)p.g.ny + (unsigned)y) * (unsigned)p.g.nx + (unsigned)x;
#pragma unroll
      for (int i = 0; i < Q; ++i)
        *reinterpret_cast<unsigned*>(static_cast<S*>(p.dst_slot[lat_opp(i)]) + cell) = Pair16<S>::pack(f[i].v.x, f[i].v.y);
      return;
    }
    if constexpr (PAIRS && !GEN) {
      // x neighbours, x even: where c_x = 0 one 32-bit shared load and one 32-bit
      // store serve both
      const int tg = (warp >> 1) * 32 + lane, xl = 2 * tg % TX;
      F2 f[Q];
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        if (L::LOAD_OWN) {
          Pair16<S>::unpack(reinterpret_cast<const unsigned*>(st)[i * (PSM_THREADS / 2) + tg], f[i].v.x, f[i].v.y);
        } else {
          const unsigned char* row = st + i * L::ROW + 128;
          if (lat_cx(i) == 0) {
            Pair16<S>::unpack(reinterpret_cast<const unsigned*>(row)[tg], f[i].v.x, f[i].v.y);
          } else {
            const S* e = reinterpret_cast<const S*>(row) + (2 * tg - lat_cx(i));
            f[i].v = make_float2(Store<S>::ld(e), Store<S>::ld(e + 1));
          }
        }
      }
      stage_read(tile, k, s);
      fluid_collide2<Q, FL>(p, f);
      const int x = hd.x + xl, y = hd.y + 2 * tg / TX;
      const unsigned cell = ((unsigned)z * (unsigned)p.g.ny + (unsigned)y) * (unsigned)p.g.nx + (unsigned)x;
      Stencil sn;
      sn.init(p.g, x, y, z, cell);
      // x + 2 of the second cell wraps at the row's end (x + 1 of the first never does)
      const unsigned dx2 = x + 2 == p.g.nx ? 0u - (unsigned)x : 2u;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const int cx = lat_cx(i), cy = lat_cy(i), cz = lat_cz(i);
        if (MODE == MODE_AA_EVEN) {
          *reinterpret_cast<unsigned*>(static_cast<S*>(p.dst_slot[lat_opp(i)]) + cell) =
              Pair16<S>::pack(f[i].v.x, f[i].v.y);
          continue;
        }
        S* d = static_cast<S*>(p.dst_slot[i]);
        const unsigned r = sn.at(0, cy, cz);
        if (cx == 0) {
          *reinterpret_cast<unsigned*>(d + r) = Pair16<S>::pack(f[i].v.x, f[i].v.y);
        } else if (cx > 0) {
          Store<S>::st(d + (unsigned)(r + 1u), f[i].v.x);
          Store<S>::st(d + (unsigned)(r + dx2), f[i].v.y);
        } else {
          Store<S>::st(d + (unsigned)(r + sn.dx[0]), f[i].v.x);
          Store<S>::st(d + r, f[i].v.y);
        }
      }
      return;
    }
    // the thread's cells r = 0 .. CELLS-1: (lx, ly + r TYB), one after the other
    // (paired: 128 cells of the tile apart, so that a warp's lanes are x neighbours)
    constexpr int CELLS = PAIRS ? 2 : CPT;
    auto one_cell = [&](int r) {
      const int c = PAIRS ? (warp >> 1) * 32 + lane + r * (PSM_THREADS / 2) : (int)threadIdx.x;
      const int xl = PAIRS ? c % TX : lx;
      const int x = hd.x + xl, y = hd.y + (PAIRS ? c / TX : ly + r * TYB);
      const unsigned cell = ((unsigned)z * (unsigned)p.g.ny + (unsigned)y) * (unsigned)p.g.nx + (unsigned)x;
      T f[Q];
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        if (GEN && zg.from(lat_cz(i))) {
          f[i] = cst<T>(p).ghost[i];
        } else if (L::LOAD_OWN) {
          f[i] = Store<S>::ld(reinterpret_cast<const S*>(st) + (PAIRS ? i : i * CPT + r) * PSM_THREADS + c);
        } else {
          f[i] = Store<S>::ld(reinterpret_cast<const S*>(st + i * L::ROW + 128) + (xl - lat_cx(i)));
        }
      }
      if (r == CELLS - 1) stage_read(tile, k, s);
      int owner = -1;
      bool solid_cell = false;
      ft_t<T> ft[6] = {0, 0, 0, 0, 0, 0};
      if (GEN) psm_collide<T, Q, FL>(p, s_body, f, x, y, z + p.g.z0, cell, owner, solid_cell, ft);
      else fluid_collide<T, Q, FL>(p, f);
      if constexpr (L::STORE_TMA) {
        static_assert(CPT == 1, "TMA stores write one cell per thread");
        // this warp's output box of tile k; lane 0 issued (and committed) the
        // warp's earlier stores: the one NOUT tiles back must have read it
        S* ow = reinterpret_cast<S*>(outs + (k % NOUT) * L::OUT + warp * L::WBOX);
        if (lane == 0) bulk_wait_read<NOUT - 1>();
        __syncwarp();
#pragma unroll
        for (int i = 0; i < Q; ++i) Store<S>::st(ow + lat_opp(i) * 32 + lane, f[i]);
        fence_proxy_async();  // the generic-proxy writes above become visible to the TMA store
        __syncwarp();
        if (lane == 0) {
          const int w0 = warp * 32;
          tma_store_4d(&maps.dstw, hd.x + w0 % TX, hd.y + w0 / TX, z, 0, ow);
          bulk_commit();
        }
      } else {
        Stencil sn;
        sn.init(p.g, x, y, z, cell);
        psm_store<S, Q, MODE, GEN>(p, sn, zg, cell, f);
      }
      if (GEN) warp_ft(s_ft, nb, solid_cell && owner >= 0, owner, ft);
    };
    if constexpr (MODE == MODE_AA_EVEN || PAIRS) {
      // only general tiles come here (the fluid-only ones took the pairs above):
      // one copy of the PSM code
#pragma unroll 1
      for (int r = 0; r < CELLS; ++r) one_cell(r);
    } else {
#pragma unroll
      for (int r = 0; r < CELLS; ++r) one_cell(r);
    }
  };

  int k = GROUPS == 1 ? 0 : warp % GROUPS;
  for (int tile = blockIdx.x + k * gridDim.x; tile < ntiles; tile += GROUPS * gridDim.x, k += GROUPS) {
    const int s = k % NST;
    // bounded wait for the stage, warp-uniform outcome (on time-out the block's
    // results are invalid: s_abort; the warp leaves the loop)
    if (!__all_sync(0xffffffffu, mbar_wait_bounded(&full[s], (unsigned)((k / NST) & 1)))) {
      s_abort = 1;
      break;
    }
    const int4 hd = s_hdr[s];
    if (hd.w) tile_body(BoolC<true>{}, tile, k, s, hd);
    else tile_body(BoolC<false>{}, tile, k, s, hd);
  }
  if (L::STORE_TMA && lane == 0) bulk_wait_all();
  __syncthreads();
  if (s_abort) {
    if (threadIdx.x == 0) {
      if (p.err) atomicExch(p.err, 1);
      // let the copies already issued finish before the block's shared memory is released
      for (int s2 = 0; s2 < NST; ++s2)
        if (s_issued[s2] > 0) mbar_wait_bounded(&full[s2], (unsigned)((s_issued[s2] - 1) & 1));
    }
    __syncthreads();
  }
  grid_launch_next();
  if (nb == 0) return;
  block_ft_finish(s_ft, p);
}

// ---------------------------------------------------------------------------
// Import / export / diagnostics (one thread per cell of planes [z_begin, z_end)).
// An FP64 instruction (conversions from and to double included) costs about
// 64 FP32 ones on GB300, so a kernel with more than about 20 of them per cell
// runs below the memory's rate: conversions between double and the narrower
// types are integer operations on the bits (exact, the same values as the
// conversion instructions), and k_macro sums in integers.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned io_plane(const IoParams& p) { return (unsigned)p.g.nx * (unsigned)p.g.ny; }

// The conversion instruction, for the values the bit operations leave out
// (out of line: inline, the compiler would run it for every value and select).
static __device__ __noinline__ double widen_rare(float f) { return (double)f; }

// double(f): sign, exponent and mantissa moved to their places
__device__ __forceinline__ double widen(float f) {
  const unsigned b = __float_as_uint(f), m = b & 0x7fffffffu;
  if (m - 1u < 0x007fffffu || m >= 0x7f800000u) return widen_rare(f);  // subnormals, infinities, NaN
  const unsigned hi = (b & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u);
  return __hiloint2double((int)hi, (int)(b << 29));
}
__device__ __forceinline__ double widen(double f) { return f; }

// d rounded to the storage type (to nearest, ties to even) as one rounding.
// In the float's normal range the float's bits are cut out of the double's:
// for float storage rounded to nearest even, for 16-bit storage with the
// discarded bits or-ed into the last one (24 bits rounded to odd, which rounds
// on to 11 or 8 bits as the double itself would).
template <class S>
__device__ __forceinline__ S narrow(double d) {
  const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d), m = hi & 0x7fffffffu;
  // exponents of [2^-126, 2^127): below the smallest normal float, or so large
  // that rounding could overflow, the conversion instruction decides
  if (m - 0x38100000u >= 0x0fd00000u) return Store<S>::from_double(d);
  const unsigned top = ((m - 0x38000000u) << 3) | (lo >> 29);
  if constexpr (sizeof(S) == 4) {
    const unsigned rest = lo << 3;  // the 29 discarded bits, left-justified
    const unsigned up = (rest > 0x80000000u || (rest == 0x80000000u && (top & 1u))) ? 1u : 0u;
    return __uint_as_float((hi & 0x80000000u) | (top + up));
  } else {
    S r;
    Store<S>::st(&r, __uint_as_float((hi & 0x80000000u) | top | ((lo << 3) ? 1u : 0u)));
    return r;
  }
}
template <>
__device__ __forceinline__ double narrow<double>(double d) { return d; }

template <class T>
__device__ __forceinline__ T io_ghost(const IoParams& p, int i) {
  if constexpr (sizeof(T) == 4) return p.ghostf[i];
  else return p.ghost[i];
}

// f_i(x) (shifted) of a state stored in `layout`, ghost value for populations
// entering from a ghost plane
template <class S, int Q>
__device__ __forceinline__ void read_state(const IoParams& p, const S* buf, unsigned cell,
                                           typename Store<S>::T (&f)[Q]) {
  using T = typename Store<S>::T;
  const long long N = p.g.ncell;
  const unsigned plane = io_plane(p);
  if (p.layout == LAYOUT_SWAPPED) {
    const unsigned z = cell / plane, r = cell - z * plane, y = r / (unsigned)p.g.nx;
    Nbr nbr;
    nbr.init(p.g, (int)(r - y * (unsigned)p.g.nx), (int)y, (int)z);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      if (nbr.from_ghost(lat_cz(i))) f[i] = io_ghost<T>(p, i);
      else
        f[i] = Store<S>::ld(buf + (long long)lat_opp(i) * N +
                            (unsigned)(cell + nbr.off(-lat_cx(i), -lat_cy(i), -lat_cz(i))));
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < Q; ++i) f[i] = Store<S>::ld(buf + (long long)i * N + cell);
  if (p.g.bc_z == PSM_BC_EQ_INLET_OUTLET) {
    const bool lo = cell < plane, hi = cell >= (unsigned)N - plane;
    if (lo || hi) {
#pragma unroll
      for (int i = 0; i < Q; ++i)
        if ((lat_cz(i) > 0 && lo) || (lat_cz(i) < 0 && hi)) f[i] = io_ghost<T>(p, i);
    }
  }
}

// f^eq_i(rho, u) - w_i rho0 in FP64 (initial states), separately rounded
__device__ __forceinline__ double eq_shifted(double w, double cu, double rho, double uu, double rho0) {
  const double e = __fma_rn(-1.5, uu, __fma_rn(__dmul_rn(4.5, cu), cu, __fma_rn(3.0, cu, 1.0)));
  return __fma_rn(-w, rho0, __dmul_rn(__dmul_rn(w, rho), e));
}
__device__ __forceinline__ double uu64(const double* u) {
  return __fma_rn(u[2], u[2], __fma_rn(u[1], u[1], __dmul_rn(u[0], u[0])));
}
__device__ __forceinline__ double cu64(int cx, int cy, int cz, const double* u) {
  return __dadd_rn(__dadd_rn((double)cx * u[0], (double)cy * u[1]), (double)cz * u[2]);
}

// Uniform equilibrium: slot blockIdx.y of the stored layout filled with its
// one value over the planes that are stored (populations entering from a ghost
// plane are not), 16 bytes per store.  Bound by the write bandwidth; one value
// per block instead of FP64 arithmetic per cell and direction took a 128^3
// FP32 D3Q19 state (160 MB) from 1990 us to 39 us a call.
constexpr unsigned FILL_BLOCK_BYTES = 65536;
template <class S, int Q>
__global__ void __launch_bounds__(PSM_THREADS) k_fill_uniform(const __grid_constant__ IoParams p) {
  const int slot = blockIdx.y;
  // the population a slot holds; swapped: that of x + c_i, so the planes shift by c_z
  const int i = p.layout == LAYOUT_SWAPPED ? lat_opp(slot) : slot;
  const int cx = lat_c_rt(kLatCX, i), cy = lat_c_rt(kLatCY, i), cz = lat_c_rt(kLatCZ, i);
  __shared__ S s_v;
  if (threadIdx.x == 0) {
    const int cls = cx * cx + cy * cy + cz * cz;
    const double w = cls == 0 ? lat_w<Q>(0) : (cls == 1 ? lat_w<Q>(1) : (cls == 2 ? lat_w<Q>(7) : lat_w<Q>(Q - 1)));
    s_v = Store<S>::from_double(eq_shifted(w, cu64(cx, cy, cz, p.u), p.rho, uu64(p.u), p.rho0));
  }
  __syncthreads();
  const S v = s_v;
  int z0 = 0, z1 = p.g.nz;
  if (p.g.bc_z == PSM_BC_EQ_INLET_OUTLET && cz != 0) {
    const bool drop_first = (cz > 0) != (p.layout == LAYOUT_SWAPPED);
    if (drop_first) z0 = 1;
    else z1 = p.g.nz - 1;
  }
  const unsigned long long plane = io_plane(p);
  unsigned char* a = reinterpret_cast<unsigned char*>(static_cast<S*>(p.f) + (unsigned long long)slot * p.g.ncell + z0 * plane);
  unsigned char* b = reinterpret_cast<unsigned char*>(static_cast<S*>(p.f) + (unsigned long long)slot * p.g.ncell + z1 * plane);
  union {
    uint4 q;
    S e[16 / sizeof(S)];
  } pk;
#pragma unroll
  for (int k = 0; k < (int)(16 / sizeof(S)); ++k) pk.e[k] = v;
  // 16-byte pieces counted from the boundary below the range; the first and
  // the last may hold values outside it
  unsigned char* base = a - (reinterpret_cast<unsigned long long>(a) & 15ull);
  for (unsigned long long blk = blockIdx.x;; blk += gridDim.x) {
    unsigned char* c = base + blk * FILL_BLOCK_BYTES;
    if (c >= b) return;
#pragma unroll 4
    for (unsigned o = threadIdx.x * 16u; o < FILL_BLOCK_BYTES; o += PSM_THREADS * 16u) {
      unsigned char* q = c + o;
      if (q >= a && q + 16 <= b) *reinterpret_cast<uint4*>(q) = pk.q;
      else
        for (int k = 0; k < (int)(16 / sizeof(S)); ++k)
          if (q + k * sizeof(S) >= a && q + (k + 1) * sizeof(S) <= b) reinterpret_cast<S*>(q)[k] = v;
    }
  }
}

// A natural, unshifted FP64 state (or equilibria of per-cell fields, FIELD)
// into the stored layout.  Bound by memory (8 Q bytes read, the storage type
// written) with one FP64 operation per value: psm_set_state of a 256x256x192
// FP32 state in device memory 496 us (2.9 GB), with the staging 6330 us.
template <class S, int Q, bool FIELD>
__global__ void __launch_bounds__(PSM_THREADS) k_import(const __grid_constant__ IoParams p) {
  S* buf = static_cast<S*>(p.f);
  const long long N = p.g.ncell;
  const unsigned plane = io_plane(p);
  const long long n = (long long)plane * (p.z_end - p.z_begin);
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
       idx += (long long)gridDim.x * blockDim.x) {
    const unsigned cell = (unsigned)p.z_begin * plane + (unsigned)idx;
    double v[Q];
    if constexpr (FIELD) {
      const double u[3] = {p.u_f[3 * idx], p.u_f[3 * idx + 1], p.u_f[3 * idx + 2]};
      const double rc = p.rho_f[idx], uu = uu64(u);
#pragma unroll
      for (int i = 0; i < Q; ++i)
        v[i] = eq_shifted(lat_w<Q>(i), cu64(lat_cx(i), lat_cy(i), lat_cz(i), u), rc, uu, p.rho0);
    } else {
#pragma unroll
      for (int i = 0; i < Q; ++i) v[i] = __ldcs(p.f_in + (long long)i * n + idx);
#pragma unroll
      for (int i = 0; i < Q; ++i) v[i] = __fma_rn(-lat_w<Q>(i), p.rho0, v[i]);
    }
    const bool ghost = p.g.bc_z == PSM_BC_EQ_INLET_OUTLET;
    const bool lo = ghost && cell < plane, hi = ghost && cell >= (unsigned)N - plane;
    if (p.layout == LAYOUT_SWAPPED) {
      const unsigned z = cell / plane, r = cell - z * plane, y = r / (unsigned)p.g.nx;
      Nbr nbr;
      nbr.init(p.g, (int)(r - y * (unsigned)p.g.nx), (int)y, (int)z);
#pragma unroll
      for (int i = 0; i < Q; ++i)
        if (!nbr.from_ghost(lat_cz(i)))  // such populations always read the ghost value
          buf[(long long)lat_opp(i) * N + (unsigned)(cell + nbr.off(-lat_cx(i), -lat_cy(i), -lat_cz(i)))] =
              narrow<S>(v[i]);
    } else {
#pragma unroll
      for (int i = 0; i < Q; ++i)
        if (!((lat_cz(i) > 0 && lo) || (lat_cz(i) < 0 && hi))) buf[(long long)i * N + cell] = narrow<S>(v[i]);
    }
  }
}

// Natural, unshifted FP64.  Bound by memory (the storage type read, 8 Q bytes
// written) with one FP64 operation per value: psm_get_state of a 256x256x192
// FP32 state to device memory 503 us (2.9 GB), with the staging 4290 us.
template <class S, int Q>
__global__ void __launch_bounds__(PSM_THREADS) k_export(const __grid_constant__ IoParams p) {
  using T = typename Store<S>::T;
  const S* buf = static_cast<const S*>(p.f);
  const unsigned plane = io_plane(p);
  const long long n = (long long)plane * (p.z_end - p.z_begin);
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
       idx += (long long)gridDim.x * blockDim.x) {
    T f[Q];
    read_state<S, Q>(p, buf, (unsigned)p.z_begin * plane + (unsigned)idx, f);
#pragma unroll
    for (int i = 0; i < Q; ++i) __stcs(p.f_out + (long long)i * n + idx, __fma_rn(lat_w<Q>(i), p.rho0, widen(f[i])));
  }
}

// Natural layout, shifted, storage precision (psm_get_pdfs): the stored
// values themselves (ghost-plane populations as the ghost value, rounded).
template <class S, int Q>
__global__ void __launch_bounds__(PSM_THREADS) k_export_raw(const __grid_constant__ IoParams p) {
  using T = typename Store<S>::T;
  const S* buf = static_cast<const S*>(p.f);
  S* out = static_cast<S*>(p.f_out_raw);
  const unsigned plane = io_plane(p);
  const long long n = (long long)plane * (p.z_end - p.z_begin);
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
       idx += (long long)gridDim.x * blockDim.x) {
    T f[Q];
    read_state<S, Q>(p, buf, (unsigned)p.z_begin * plane + (unsigned)idx, f);
#pragma unroll
    for (int i = 0; i < Q; ++i) Store<S>::st(out + (long long)i * n + idx, f[i]);
  }
}

// Natural, unshifted FP64 PDFs of listed cells: out[k][Q].
template <class S, int Q>
__global__ void k_get_cells(const __grid_constant__ IoParams p, const long long* cells, long long n, double* out) {
  using T = typename Store<S>::T;
  const S* buf = static_cast<const S*>(p.f);
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
    const long long cell = cells[k];
    if (cell < 0 || cell >= p.g.ncell) continue;  // the host validates; never read out of bounds
    T f[Q];
    read_state<S, Q>(p, buf, (unsigned)cell, f);
    for (int i = 0; i < Q; ++i) out[k * Q + i] = (double)f[i] + lat_w<Q>(i) * p.rho0;
  }
}

// Density and velocity with FP64 sums and divisions.
template <class T, int Q>
__device__ __forceinline__ void macro64(const T* f, double rho0, double& rho, double* u) {
  double drho = 0, j[3] = {0, 0, 0};
  for (int i = 0; i < Q; ++i) {
    const double v = (double)f[i];
    drho += v;
    j[0] += lat_cx(i) * v;
    j[1] += lat_cy(i) * v;
    j[2] += lat_cz(i) * v;
  }
  rho = rho0 + drho;
  for (int k = 0; k < 3; ++k) u[k] = j[k] / rho;
}

template <int Q>
static __device__ __noinline__ void macro64_rare(const float* f, double rho0, double* out) {
  macro64<float, Q>(f, rho0, out[0], out + 1);
}
static __device__ __noinline__ double add_tail(double x, int n) { return __fma_rn((double)n, 1.1920928955078125e-07, x); }

// The same from float populations with the sums in integers: 16 FP64
// operations per cell instead of about 100.  The populations are scaled by a
// power of two (exactly) so that the largest lies in [1, 2), and each is cut
// into three integers, multiples of 2^-21, 2^-44 and 2^-67, by adding 1.5 times
// the power of two whose last place that is (the sum's bits then count from the
// constant's).  Integer sums are exact, and so are drho and j, but for one rounding
// where the third cut is not empty; rho0 + drho is rounded once (FP64 sums round
// after every term at 2^-53).  u = j / rho: a reciprocal from rcp.approx with
// one Newton step, then the quotient corrected by its own remainder
// (Markstein's method), rounded as the division is but for ties in the 2^-27
// tail.
// false (nothing written) for cells that the cuts are not made for, which
// macro64 decides: a population below 2^-44 of the largest, whose last bits the
// third cut would drop (the momentum may consist of such values alone), a
// largest population of 2 or more (a scale below 1 could push small ones out of
// range) or below 2^-97, densities outside the range, infinities and NaN.
template <int Q>
__device__ __forceinline__ bool macro_int(const float (&f)[Q], double rho0, double& rho, double (&u)[3]) {
  unsigned big = 0u, small = ~0u;  // largest and smallest size (less one: zeros do not count as small)
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const unsigned m = __float_as_uint(f[i]) & 0x7fffffffu;
    big = max(big, m);
    small = min(small, m - 1u);
  }
  const int E = (int)(big >> 23);
  if (E < 30 || E > 127) {
    if (big != 0u) return false;
    rho = rho0;
    u[0] = u[1] = u[2] = 0.0;
    return rho0 > 0.0;
  }
  // 24 bits from 2^-44 of the largest on end above the last cut
  if (E > 44 && small < ((unsigned)(E - 44) << 23) - 1u) return false;
  const float scale = __uint_as_float((unsigned)(254 - E) << 23);  // 2^(127 - E)
  const float M1 = 6.0f, M2 = 7.152557373046875e-07f, M3 = 8.526512829121202e-14f;  // 1.5 2^2, 2^-21, 2^-44
  int n1[4] = {0, 0, 0, 0}, n2[4] = {0, 0, 0, 0}, n3[4] = {0, 0, 0, 0};  // sums: 1, c_x, c_y, c_z
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const float g = __fmul_rn(f[i], scale);
    const float t1 = __fadd_rn(g, M1), r1 = __fsub_rn(g, __fsub_rn(t1, M1));
    const float t2 = __fadd_rn(r1, M2), r2 = __fsub_rn(r1, __fsub_rn(t2, M2));
    const float t3 = __fadd_rn(r2, M3);
    const int a = __float_as_int(t1), b = __float_as_int(t2), c = __float_as_int(t3);
    const int s[4] = {1, lat_cx(i), lat_cy(i), lat_cz(i)};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (s[k] > 0) n1[k] = (int)((unsigned)n1[k] + (unsigned)a), n2[k] = (int)((unsigned)n2[k] + (unsigned)b), n3[k] = (int)((unsigned)n3[k] + (unsigned)c);
      if (s[k] < 0) n1[k] = (int)((unsigned)n1[k] - (unsigned)a), n2[k] = (int)((unsigned)n2[k] - (unsigned)b), n3[k] = (int)((unsigned)n3[k] - (unsigned)c);
    }
  }
  // the constants' own bits cancel in the sums over c (as many +1 as -1)
  n1[0] = (int)((unsigned)n1[0] - (unsigned)Q * __float_as_uint(M1));
  n2[0] = (int)((unsigned)n2[0] - (unsigned)Q * __float_as_uint(M2));
  n3[0] = (int)((unsigned)n3[0] - (unsigned)Q * __float_as_uint(M3));
  double X[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    // (n1 2^23 + n2) as a double, exactly: below 2^51 in size
    const long long v = (long long)n1[k] * (1ll << 23) + (long long)n2[k];
    X[k] = __dsub_rn(__longlong_as_double(0x4338000000000000ll + v), 6755399441055744.0);
  }
  if (n3[0] | n3[1] | n3[2] | n3[3]) {  // values below 2^-20 of the largest: n3 2^-23 more
#pragma unroll
    for (int k = 0; k < 4; ++k) X[k] = add_tail(X[k], n3[k]);
  }
  const int sh = E - 171;  // X counts in units of 2^(E - 127 - 44)
  const double rh = __fma_rn(X[0], __hiloint2double((1023 + sh) << 20, 0), rho0);
  const unsigned rb = (unsigned)__double2hiint(rh);
  if (rb - (923u << 20) >= (200u << 20)) return false;  // not in [2^-100, 2^100)
  rho = rh;
  float a;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(a) : "f"(__uint_as_float((rb - 0x38000000u) << 3)));
  const unsigned ab = __float_as_uint(a);
  const double inv0 = __hiloint2double((int)((ab >> 3) + 0x38000000u), (int)(ab << 29));
  const double inv = __fma_rn(inv0, __fma_rn(-rh, inv0, 1.0), inv0);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double q0 = __dmul_rn(X[k + 1], inv);
    const double q = __fma_rn(__fma_rn(-q0, rh, X[k + 1]), inv, q0);
    const int qh = __double2hiint(q), ql = __double2loint(q);
    // q 2^sh: |q| is 0 or lies in [2^-124, 2^151], so the exponent field stays in range
    u[k] = ((qh & 0x7fffffff) | ql) ? __hiloint2double(qh + (sh << 20), ql) : 0.0;
  }
  return true;
}

// Density and velocity (psm_get_macroscopic).  The velocities of a warp's
// cells pass through shared memory so that the stores are contiguous.  Bound by
// the FP64 pipe (16 instructions per cell): a 256x256x192 FP32 state to device
// memory in 403 us (1.4 GB; FP64 sums and divisions and a staging chunk: 3290 us).
template <class S, int Q>
__global__ void __launch_bounds__(PSM_THREADS) k_macro(const __grid_constant__ IoParams p) {
  using T = typename Store<S>::T;
  const S* buf = static_cast<const S*>(p.f);
  __shared__ double s_u[PSM_THREADS / 32][96];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned plane = io_plane(p);
  const long long n = (long long)plane * (p.z_end - p.z_begin);
  for (long long w0 = blockIdx.x * (long long)blockDim.x + warp * 32; w0 < n; w0 += (long long)gridDim.x * blockDim.x) {
    const long long idx = w0 + lane;
    if (idx < n) {
      T f[Q];
      read_state<S, Q>(p, buf, (unsigned)p.z_begin * plane + (unsigned)idx, f);
      double rho, u[3];
      if constexpr (sizeof(T) == 4) {
        if (!macro_int<Q>(f, p.rho0, rho, u)) {
          float g[Q];
          double r[4];
#pragma unroll
          for (int i = 0; i < Q; ++i) g[i] = f[i];
          macro64_rare<Q>(g, p.rho0, r);
          rho = r[0], u[0] = r[1], u[1] = r[2], u[2] = r[3];
        }
      } else {
        macro64<T, Q>(f, p.rho0, rho, u);
      }
      __stcs(p.rho_out + idx, rho);
#pragma unroll
      for (int k = 0; k < 3; ++k) s_u[warp][3 * lane + k] = u[k];
    }
    __syncwarp();
    const int m = (int)(n - w0 < 32 ? n - w0 : 32) * 3;
    for (int k = lane; k < m; k += 32) __stcs(p.u_out + 3 * w0 + k, s_u[warp][k]);
    __syncwarp();
  }
}

template <class S, int Q>
__global__ void __launch_bounds__(PSM_THREADS) k_mass(const __grid_constant__ IoParams p) {
  using T = typename Store<S>::T;
  const S* buf = static_cast<const S*>(p.f);
  double acc = 0.0;
  const unsigned plane = io_plane(p);
  const long long n = (long long)plane * (p.z_end - p.z_begin);
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
       idx += (long long)gridDim.x * blockDim.x) {
    T f[Q];
    read_state<S, Q>(p, buf, (unsigned)p.z_begin * plane + (unsigned)idx, f);
    double m = p.rho0;
    for (int i = 0; i < Q; ++i) m += (double)f[i];
    acc += m;
  }
  __shared__ double s_w[PSM_THREADS / 32];
  __shared__ double blk[1];
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < PSM_THREADS / 32; ++w) s += s_w[w];
    blk[0] = s;
  }
  __syncthreads();
  grid_reduce(blk, 1, p.partials, p.ticket, p.sum_out);
}

// One semi-implicit Euler step of a free body's rigid-body equations (two-way
// coupling) by one warp, from this step's force and torque on the body ft:
//   v += (F + Fext) / m,  R += v,  L += T + Text,
//   Q <- Rot(w*) Q, w* = Q Ib^-1 Q^T L,  w = Q Ib^-1 Q^T L,
// then the DevBody of the next step (kinematics, the cell box of the rotated
// geometry box widened by 2.5 cells, the remap's pose and its float form,
// remap_setup).  Run by the block that summed the loads: a chain of FP64
// operations that the next step waits for, so the components and matrix elements
// go to the lanes (one thread for all of it: 25 us a step; so about 7 us).
static __device__ __forceinline__ void body_update(BodyDyn* S, DevBody* d, const double* ft, int nx, int ny, int nz) {
  const unsigned all = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int k = lane % 3, r = (lane / 3) % 3;  // a vector's component; a matrix element (r, k) in lanes 0 .. 8
  auto get = [&](double v, int src) { return __shfl_sync(all, v, src); };
  auto sum3 = [](double a, double x, double b, double y, double c, double z) { return fma(a, x, fma(b, y, c * z)); };
  const double v = S->v[k] + (ft[k] + S->Fext[k]) / S->mass;
  const double R = S->R[k] + v;
  const double L = S->L[k] + (ft[3 + k] + S->Text[k]);
  double Q = S->Q[3 * r + k];
  const double I0 = S->Ibinv[3 * k], I1 = S->Ibinv[3 * k + 1], I2 = S->Ibinv[3 * k + 2];
  const double L0 = get(L, 0), L1 = get(L, 1), L2 = get(L, 2);
  // component k of Q Ib^-1 Q^T L in every lane
  auto spin = [&](double q) {
    const double a = sum3(get(q, k), L0, get(q, 3 + k), L1, get(q, 6 + k), L2);
    const double b = sum3(I0, get(a, 0), I1, get(a, 1), I2, get(a, 2));
    return sum3(get(q, 3 * k), get(b, 0), get(q, 3 * k + 1), get(b, 1), get(q, 3 * k + 2), get(b, 2));
  };
  const double ws = spin(Q);
  const double w0 = get(ws, 0), w1 = get(ws, 1), w2 = get(ws, 2);
  const double a = sqrt(sum3(w0, w0, w1, w1, w2, w2));
  if (a > 0.0) {  // the same in every lane
    const double n = ws / a;
    const double n0 = get(n, 0), n1 = get(n, 1), n2 = get(n, 2);
    double sn, cs;
    sincos(a, &sn, &cs);
    const double nr = r == 0 ? n0 : (r == 1 ? n1 : n2), nk = k == 0 ? n0 : (k == 1 ? n1 : n2);
    // Rodrigues: element (r, k) = cos d_rk + (1 - cos) n_r n_k + sin [n]x_rk
    const int o = 3 - r - k;  // the third axis where r != k
    const double no = o == 0 ? n0 : (o == 1 ? n1 : n2);
    const double sgn = (k == (r + 1) % 3) ? -sn : sn;
    const double Rm = r == k ? fma((1.0 - cs) * nr, nk, cs) : fma((1.0 - cs) * nr, nk, sgn * no);
    Q = sum3(get(Rm, 3 * r), get(Q, k), get(Rm, 3 * r + 1), get(Q, 3 + k), get(Rm, 3 * r + 2), get(Q, 6 + k));
  }
  const double w = spin(Q);
  if (lane < 3) {
    S->v[k] = v, S->R[k] = R, S->L[k] = L, S->w[k] = w;
    d->R[k] = R, d->v[k] = v, d->omega[k] = w;
    d->Rf[k] = (float)R, d->vf[k] = (float)v, d->omegaf[k] = (float)w;
  }
  if (lane < 9) {
    S->Q[lane] = Q;
    d->Qd[lane] = Q;
  }
  // hull of the rotated geometry box: corner c, component k (lanes 3 c + k and, for corners 8 .. 10, copies)
  const int c = (lane / 3) & 7;
  const double lo0 = S->lo[0], lo1 = S->lo[1], lo2 = S->lo[2];
  const double p0 = lo0 + ((c & 1) ? (double)S->gx : 0.0), p1 = lo1 + ((c & 2) ? (double)S->gy : 0.0),
               p2 = lo2 + ((c & 4) ? (double)S->gz : 0.0);
  const double wc = sum3(get(Q, 3 * k), p0, get(Q, 3 * k + 1), p1, get(Q, 3 * k + 2), p2) + R;
  double mn = wc, mx = wc;
#pragma unroll
  for (int q = 1; q < 8; ++q) {
    const double t = get(wc, (3 * q + lane) % 24);  // lanes 0 .. 23 hold the eight corners
    mn = fmin(mn, t);
    mx = fmax(mx, t);
  }
  // (lanes 24 .. 31 repeat lanes 0 .. 7)
  const int dim = k == 0 ? nx : (k == 1 ? ny : nz);
  double b0d = floor(mn - 2.5), b1d = ceil(mx + 2.5) + 1.0;
  if (b0d < 0.0) b0d = 0.0;
  if (b1d > (double)dim) b1d = (double)dim;
  if (b1d < b0d) b1d = b0d;
  const int b0 = (int)b0d, b1 = (int)b1d;
  if (lane < 3) {
    int* lo_ = k == 0 ? &d->x0 : (k == 1 ? &d->y0 : &d->z0);
    int* hi_ = k == 0 ? &d->x1 : (k == 1 ? &d->y1 : &d->z1);
    *lo_ = b0;
    *hi_ = b1;
  }
  // remap_setup with its components in the lanes
  const double n = (double)(1 << d->s);
  const double U = 5.9604644775390625e-08, Ud = 1.1102230246251565e-16;  // 2^-24, 2^-53
  const int last = b1 > b0 ? b1 - 1 : b0;
  const int anc = b0 + (last - b0) / 2;
  const double be = fmax(fabs((double)(b0 - anc)), fabs((double)(last - anc)));
  const double bd = fmax(fabs((double)b0 + 0.5 - R), fabs((double)last + 0.5 - R));
  const double lok = k == 0 ? lo0 : (k == 1 ? lo1 : lo2);
  const double Be = get(be, 0) + get(be, 1) + get(be, 2), Bd = get(bd, 0) + get(bd, 1) + get(bd, 2);
  const double lom = fmax(fabs(lo0), fmax(fabs(lo1), fabs(lo2)));
  const double ac = ((double)anc + 0.5) - R;
  const double X = sum3(get(Q, k), get(ac, 0), get(Q, 3 + k), get(ac, 1), get(Q, 6 + k), get(ac, 2));
  const double H = ((X - 0.5) - lok) * n + 0.5;
  const double Hmax = fmax(fabs(get(H, 0)), fmax(fabs(get(H, 1)), fabs(get(H, 2))));
  const double span = (Hmax + 1.0) + (n + 1.0) * Be;
  // the finest grid 2^-m, m <= 20, on which the high parts stay below 2^24 (every m below it does too)
  const unsigned fits = __ballot_sync(all, lane <= 20 && span * (double)(1 << min(lane, 20)) < 16777216.0);
  const bool form = fits != 0u && span < 1e30;
  const int m = form ? 31 - __clz(fits) : 0;
  const double sc = (double)(1 << m), isc = 1.0 / sc;
  const double G = Q * n, gh = floor(G * sc + 0.5) * isc, hh = floor(H * sc + 0.5) * isc;
  if (lane < 9) {
    d->Ghi[lane] = form ? (float)gh : 0.0f;
    d->Glo[lane] = form ? (float)(G - gh) : 0.0f;
  }
  if (lane < 3) {
    d->anchor[k] = anc;
    d->lod[k] = lok;
    d->Hhi[k] = form ? (float)hh : 0.0f;
    d->Hlo[k] = form ? (float)(H - hh) : 0.0f;
  }
  if (lane == 0) {
    const double Lb = 0.5 * isc * (1.0 + Be);
    const double ef = U * 0.5 * isc * (1.0 + Be) + 3.0 * U * Lb + U * (1.0 + Lb);
    const double ed = n * Ud * (7.0 * Bd + 3.0 * lom + 2.0) + Ud;
    d->rtol = form ? (float)(2.0 * (ef + 2.0 * ed) + U) : 2.0f;
  }
}

// Sums of stored partials, one block per slot: slot k into row (first + dir k)
// mod cap of out (rows of `row` doubles); then the free bodies of free_mask
// advance under the loads just summed (one slot then).
static __global__ void __launch_bounds__(PSM_THREADS)
    k_reduce_slots(const double* slots, long long slot, int ncomp, double* out, int row, long long first, int dir,
                   long long cap, unsigned free_mask, BodyDyn* dyn, DevBody* dbody, int nx, int ny, int nz) {
  grid_launch_next();
  grid_wait_previous();
  const double* s = slots + blockIdx.x * slot;
  double* o = out + ((first + dir * (long long)blockIdx.x) % cap) * row;
  // a step kernel that refused its launch wrote no slot: whatever is there, stay inside it
  const double most = (double)((slot - 1) / ncomp), G = s[0];
  sum_partials<PSM_THREADS>(s + 1, G >= 0.0 && G <= most ? (int)G : 0, ncomp, o);
  if (free_mask == 0u) return;
  __syncthreads();
  const int b = threadIdx.x >> 5;
  if (b < PSM_MAX_BODIES && ((free_mask >> b) & 1u)) body_update(dyn + b, dbody + b, o + 6 * b, nx, ny, nz);
}

// ---------------------------------------------------------------------------
// Launcher helpers
// ---------------------------------------------------------------------------
template <class K>
int persistent_blocks(K kernel, int threads = PSM_THREADS) {
  int dev = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0);
  if (per_sm < 1) per_sm = 1;
  return sms * per_sm > 0 ? sms * per_sm : 1;
}

inline int persistent_limit(int per_sm) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms * per_sm > 0 ? sms * per_sm : 1;
}

// Launch that may begin before the previous kernel of the stream ends
// (grid_wait_previous): 32^3 FP64 sphere 28.8 -> 25.8 us a step, 96x96x120 D3Q27
// rotors 54.2 -> 51.6, 203x117x151 FP16 80.4 -> 78.1, 256^3 FP32 421 -> 418.
template <class... P, class... A>
cudaError_t launch_overlapped(void (*kernel)(P...), int grid, int threads, size_t smem, cudaStream_t st, const A&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <class S, int Q, int MODE, int FL, int NT>
cudaError_t launch_step_nt(const StepParams& p, cudaStream_t st) {
  // no more blocks than the launch bounds aim at, so that blocks of 256 stride
  // like the TMA kernel's
  static const int blocks = std::min(persistent_blocks(k_step<S, Q, MODE, FL, NT>, NT),
                                     persistent_limit(step_min_blocks<S, Q, FL>() * PSM_THREADS / NT));
  const long long units = (long long)((p.g.nx + 31) / 32) * p.g.ny * p.g.nz, need = (units + NT / 32 - 1) / (NT / 32);
  return launch_overlapped(k_step<S, Q, MODE, FL, NT>, (int)(need < blocks ? need : blocks), NT, 0, st, p);
}

template <class S, int Q, int MODE, int FL>
cudaError_t launch_step_t(const StepParams& p, cudaStream_t st) {
  if constexpr (sizeof(S) == 8)
    if (p.fine) return launch_step_nt<S, Q, MODE, FL, PSM_FINE_THREADS>(p, st);
  return launch_step_nt<S, Q, MODE, FL, PSM_THREADS>(p, st);
}

template <class S, int Q, int MODE, int FL>
cudaError_t launch_step_tma_t(const StepParams& p, const TmaMaps& m, cudaStream_t st) {
  using L = TmaLayout<S, Q, MODE, FL>;
  // persistent grid: resident blocks per SM (registers and shared memory), at most 8 per SM
  // The stage count assumes at most L::STATIC_SMEM bytes of static shared
  // memory per block; a build that exceeds it refuses to launch rather than
  // silently losing resident blocks.
  static const int blocks = [] {
    cudaFuncAttributes fa{};
    if (cudaFuncGetAttributes(&fa, k_step_tma<S, Q, MODE, FL>) != cudaSuccess ||
        fa.sharedSizeBytes > (size_t)L::STATIC_SMEM)
      return 0;
    if (cudaFuncSetAttribute(k_step_tma<S, Q, MODE, FL>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::SMEM) !=
        cudaSuccess)
      return 0;
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_step_tma<S, Q, MODE, FL>, PSM_THREADS, L::SMEM);
    if (per_sm > 8) per_sm = 8;
    return sms * per_sm;
  }();
  if (blocks < 1) return cudaErrorInvalidConfiguration;
  const long long grid = p.t.ntiles < blocks ? p.t.ntiles : blocks;
  return launch_overlapped(k_step_tma<S, Q, MODE, FL>, (int)grid, PSM_THREADS, L::SMEM, st, p, m);
}

// fluid operator fl (PSM_BGK, PSM_TRT, PSM_CUMULANT) -> template argument FL;
// the cumulant kernels exist for D3Q19 only
template <class S, int Q, int MODE>
cudaError_t launch_step_tma_m(int fl, const StepParams& p, const TmaMaps& m, cudaStream_t st) {
  if (fl == PSM_TRT) return launch_step_tma_t<S, Q, MODE, 1>(p, m, st);
  if (fl == PSM_CUMULANT) {
    if constexpr (Q == 19) return launch_step_tma_t<S, Q, MODE, 2>(p, m, st);
    else return cudaErrorNotSupported;
  }
  return launch_step_tma_t<S, Q, MODE, 0>(p, m, st);
}

template <class S, int Q>
cudaError_t launch_step_tma_q(int mode, int fl, const StepParams& p, const TmaMaps& m, cudaStream_t st) {
  if (mode == MODE_TG) return launch_step_tma_m<S, Q, MODE_TG>(fl, p, m, st);
  if (mode == MODE_AA_EVEN) return launch_step_tma_m<S, Q, MODE_AA_EVEN>(fl, p, m, st);
  return launch_step_tma_m<S, Q, MODE_AA_ODD>(fl, p, m, st);
}

template <class S, int Q, int FL>
int tma_smem_f(int mode) {
  if (mode == MODE_TG) return TmaLayout<S, Q, MODE_TG, FL>::SMEM;
  if (mode == MODE_AA_EVEN) return TmaLayout<S, Q, MODE_AA_EVEN, FL>::SMEM;
  return TmaLayout<S, Q, MODE_AA_ODD, FL>::SMEM;
}

template <class S, int Q>
int tma_smem_q(int mode, int fl) {
  if constexpr (Q == 19)
    if (fl == PSM_CUMULANT) return tma_smem_f<S, Q, 2>(mode);
  return tma_smem_f<S, Q, 0>(mode);
}

// dynamic shared memory, stages, resident blocks aimed at, cells per thread
template <class L>
void tma_layout_of(int* out) {
  out[0] = L::SMEM;
  out[1] = L::NST;
  out[2] = L::BLOCKS;
  out[3] = L::CPT;
}
template <class S, int Q, int FL>
void tma_layout_f(int mode, int* out) {
  if (mode == MODE_TG) tma_layout_of<TmaLayout<S, Q, MODE_TG, FL>>(out);
  else if (mode == MODE_AA_EVEN) tma_layout_of<TmaLayout<S, Q, MODE_AA_EVEN, FL>>(out);
  else tma_layout_of<TmaLayout<S, Q, MODE_AA_ODD, FL>>(out);
}
template <class S, int Q>
void tma_layout_q(int mode, int fl, int* out) {
  if constexpr (Q == 19)
    if (fl == PSM_CUMULANT) return tma_layout_f<S, Q, 2>(mode, out);
  tma_layout_f<S, Q, 0>(mode, out);
}

template <class S, int Q, int MODE>
cudaError_t launch_step_m(int fl, const StepParams& p, cudaStream_t st) {
  if (fl == PSM_TRT) return launch_step_t<S, Q, MODE, 1>(p, st);
  if (fl == PSM_CUMULANT) {
    if constexpr (Q == 19) return launch_step_t<S, Q, MODE, 2>(p, st);
    else return cudaErrorNotSupported;
  }
  return launch_step_t<S, Q, MODE, 0>(p, st);
}

template <class S, int Q>
cudaError_t launch_step_q(int mode, int fl, const StepParams& p, cudaStream_t st) {
  if (mode == MODE_TG) return launch_step_m<S, Q, MODE_TG>(fl, p, st);
  if (mode == MODE_AA_EVEN) return launch_step_m<S, Q, MODE_AA_EVEN>(fl, p, st);
  return launch_step_m<S, Q, MODE_AA_ODD>(fl, p, st);
}

inline long long io_cells(const IoParams& p) { return (long long)p.g.nx * p.g.ny * (p.z_end - p.z_begin); }
inline int io_grid(const IoParams& p) {
  long long b = (io_cells(p) + PSM_THREADS - 1) / PSM_THREADS;
  if (b > (1 << 20)) b = 1 << 20;
  return (int)(b < 1 ? 1 : b);
}

template <class S, int Q>
cudaError_t launch_import_q(const IoParams& p, cudaStream_t st) {
  if (p.uniform) {
    const unsigned long long bytes = (unsigned long long)p.g.ncell * sizeof(S) + 16;
    unsigned long long b = (bytes + FILL_BLOCK_BYTES - 1) / FILL_BLOCK_BYTES;
    if (b > (1u << 20)) b = 1u << 20;
    k_fill_uniform<S, Q><<<dim3((unsigned)b, Q), PSM_THREADS, 0, st>>>(p);
  } else if (p.rho_f) {
    k_import<S, Q, true><<<io_grid(p), PSM_THREADS, 0, st>>>(p);
  } else {
    k_import<S, Q, false><<<io_grid(p), PSM_THREADS, 0, st>>>(p);
  }
  return cudaGetLastError();
}

}  // namespace psm

// One translation unit per storage precision defines its launchers with this.
#define PSM_DEFINE_STORAGE(NAME, S)                                                                     \
  namespace psm {                                                                                       \
  cudaError_t launch_step_##NAME(int Q, int mode, int fl, const StepParams& p, cudaStream_t st) {       \
    return Q == 19 ? launch_step_q<S, 19>(mode, fl, p, st) : launch_step_q<S, 27>(mode, fl, p, st);     \
  }                                                                                                     \
  cudaError_t launch_step_tma_##NAME(int Q, int mode, int fl, const StepParams& p, const TmaMaps& m,    \
                                     cudaStream_t st) {                                                 \
    return Q == 19 ? launch_step_tma_q<S, 19>(mode, fl, p, m, st) : launch_step_tma_q<S, 27>(mode, fl, p, m, st); \
  }                                                                                                     \
  int tma_smem_bytes_##NAME(int Q, int mode, int fl) {                                                  \
    return Q == 19 ? tma_smem_q<S, 19>(mode, fl) : tma_smem_q<S, 27>(mode, fl);                         \
  }                                                                                                     \
  void tma_layout_##NAME(int Q, int mode, int fl, int* out) {                                           \
    if (Q == 19) tma_layout_q<S, 19>(mode, fl, out);                                                    \
    else tma_layout_q<S, 27>(mode, fl, out);                                                            \
  }                                                                                                     \
  cudaError_t launch_import_##NAME(int Q, const IoParams& p, cudaStream_t st) {                         \
    return Q == 19 ? launch_import_q<S, 19>(p, st) : launch_import_q<S, 27>(p, st);                     \
  }                                                                                                     \
  cudaError_t launch_export_##NAME(int Q, const IoParams& p, cudaStream_t st) {                         \
    if (Q == 19) k_export<S, 19><<<io_grid(p), PSM_THREADS, 0, st>>>(p);                                \
    else k_export<S, 27><<<io_grid(p), PSM_THREADS, 0, st>>>(p);                                        \
    return cudaGetLastError();                                                                          \
  }                                                                                                     \
  cudaError_t launch_export_raw_##NAME(int Q, const IoParams& p, cudaStream_t st) {                     \
    if (Q == 19) k_export_raw<S, 19><<<io_grid(p), PSM_THREADS, 0, st>>>(p);                            \
    else k_export_raw<S, 27><<<io_grid(p), PSM_THREADS, 0, st>>>(p);                                    \
    return cudaGetLastError();                                                                          \
  }                                                                                                     \
  cudaError_t launch_macro_##NAME(int Q, const IoParams& p, cudaStream_t st) {                          \
    if (Q == 19) k_macro<S, 19><<<io_grid(p), PSM_THREADS, 0, st>>>(p);                                 \
    else k_macro<S, 27><<<io_grid(p), PSM_THREADS, 0, st>>>(p);                                         \
    return cudaGetLastError();                                                                          \
  }                                                                                                     \
  cudaError_t launch_get_cells_##NAME(int Q, const IoParams& p, const long long* cells, long long n,     \
                                      double* out, cudaStream_t st) {                                  \
    const int b = (int)((n + PSM_THREADS - 1) / PSM_THREADS < 1024 ? (n + PSM_THREADS - 1) / PSM_THREADS : 1024); \
    if (Q == 19) k_get_cells<S, 19><<<b < 1 ? 1 : b, PSM_THREADS, 0, st>>>(p, cells, n, out);         \
    else k_get_cells<S, 27><<<b < 1 ? 1 : b, PSM_THREADS, 0, st>>>(p, cells, n, out);                 \
    return cudaGetLastError();                                                                          \
  }                                                                                                     \
  cudaError_t launch_mass_##NAME(int Q, const IoParams& p, int blocks, cudaStream_t st) {               \
    if (Q == 19) k_mass<S, 19><<<blocks, PSM_THREADS, 0, st>>>(p);                                      \
    else k_mass<S, 27><<<blocks, PSM_THREADS, 0, st>>>(p);                                              \
    return cudaGetLastError();                                                                          \
  }                                                                                                     \
  }
