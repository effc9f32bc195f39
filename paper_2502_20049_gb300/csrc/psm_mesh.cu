// Voxelisation of a closed triangle mesh into the super-sampled binary
// geometry field of Sec. 3 (the paper voxelises the body's surface mesh once
// and keeps the binary field), on the GPU.
//
// A sub-cell is inside iff a ray from its centre in the +x direction crosses
// the surface an odd number of times, decided in exact integer arithmetic:
//   * field box [lo, lo + dims): lo = floor(min v) - 1, lo + dims = ceil(max v) + 1
//     per axis (whole cells), dims <= 2^(19 - s);
//   * vertex coordinates relative to lo quantised to integers in units of
//     2^-(s+8) cells, rounded half away from zero; the centre of sub-cell a is
//     at 256 a + 128;
//   * the ray hits a triangle's (y, z) projection when the three edge
//     orientations share one strict sign, where a zero orientation takes the
//     sign it would have with the centre moved by (delta^2, delta) in (y, z),
//     delta -> 0+ (a point on a shared edge or vertex falls on one side only);
//   * a hit counts when the crossing lies at or ahead of the centre in x.
// Work, all on the GPU (the host reads a few numbers between two phases):
//   * vertices: extent of the box, finiteness; later their quantised coordinates;
//   * triangles: index checks, and the closedness of the mesh: every directed
//     edge toggles its undirected edge's bit in a hash table, and a running
//     count of the odd ones ends at zero iff every edge is shared evenly;
//   * triangles are binned by the 16 x 16-row tiles their projection's bounding
//     box covers (count, scan, fill);
//   * one block per tile finds each hit's crossing (binary search on an exact,
//     monotone integer test: the first m of the row's centres see it), toggles
//     bit m - 1 of the row in shared memory, turns the toggles into parities by
//     a suffix XOR, and writes the tile's bricks whole, without atomics.
// 131,072 triangles at s = 2 on a 124 x 124 x 76 box: 1.2 ms, kernels 0.2 ms
// (rows 86 us, bound by the gathers of the triangles' vertices), the rest
// allocations, copies and the host field.  One thread per row over its tile's
// list with global atomics per row and cell took 714 us for the rows, and
// sorting the edges on the host made it 12.5 ms.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "psm_internal.h"

namespace psm {
int set_error(int code, const char* msg);
}

namespace {

constexpr int TILE = 16;       // rows per tile side
constexpr int MAX_HITS = 256;  // crossings one row may have
constexpr int NT = 256;        // threads per block (a tile's rows)
static_assert(TILE * TILE == NT, "one thread per row of a tile");
// bits of a row a block holds at once; rows beyond it take several passes
constexpr int CHUNK_MAX = 1024;

// What the first phase finds.
struct MeshInfo {
  unsigned mn[3], mx[3];  // coordinate extremes as ordered integers (order_bits)
  unsigned bad_index, degenerate, non_finite;
  unsigned long long odd_edges;  // undirected edges seen an odd number of times so far
  unsigned long long total;      // entries of the tile lists
  int hits_exceeded;
};

// floats as unsigned integers of the same order
__device__ __forceinline__ unsigned order_bits(float f) {
  const unsigned b = __float_as_uint(f);
  return (b & 0x80000000u) ? ~b : b | 0x80000000u;
}
float from_order_bits(unsigned u) {
  const unsigned b = (u & 0x80000000u) ? u & 0x7fffffffu : ~u;
  float f;
  std::memcpy(&f, &b, 4);
  return f;
}

__global__ void __launch_bounds__(NT) k_mesh_extent(const float* __restrict__ vert, long long nv, MeshInfo* info) {
  unsigned mn[3] = {~0u, ~0u, ~0u}, mx[3] = {0u, 0u, 0u};
  bool bad = false;
  for (long long i = blockIdx.x * (long long)NT + threadIdx.x; i < nv; i += (long long)gridDim.x * NT)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float f = vert[3 * i + k];
      bad = bad || !isfinite(f);
      const unsigned u = order_bits(f);
      mn[k] = min(mn[k], u);
      mx[k] = max(mx[k], u);
    }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const unsigned lo = __reduce_min_sync(0xffffffffu, mn[k]), hi = __reduce_max_sync(0xffffffffu, mx[k]);
    if ((threadIdx.x & 31) == 0) {
      atomicMin(&info->mn[k], lo);
      atomicMax(&info->mx[k], hi);
    }
  }
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) info->non_finite = 1u;
}

// Index checks and the parity of the undirected edges.  keys (0: free; an edge's
// key is never 0) and odd have `slots` entries, a power of two of at least four
// per triangle, so a probe always ends, and soon: a closed mesh has 1.5 edges
// per triangle, loose triangles 3 (at most three quarters of the slots, about
// 9 probes for the last ones; a table filled up by 349,525 loose triangles took
// 421 ms to refuse them, this one 0.4 ms).
__global__ void __launch_bounds__(NT) k_mesh_edges(const int* __restrict__ tri, long long nt, long long nv,
                                                   unsigned long long* keys, unsigned* odd, unsigned long long slots,
                                                   MeshInfo* info) {
  int delta = 0;
  bool bad = false, deg = false;
  for (long long e = blockIdx.x * (long long)NT + threadIdx.x; e < 3 * nt; e += (long long)gridDim.x * NT) {
    const long long t = e / 3;
    const int c = (int)(e - 3 * t), n = c == 2 ? 0 : c + 1;
    const int a = tri[e], b = tri[3 * t + n];
    if (a < 0 || a >= nv || b < 0 || b >= nv) {
      bad = true;
      continue;
    }
    if (a == b) {
      deg = true;
      continue;
    }
    const unsigned long long key = ((unsigned long long)(unsigned)min(a, b) << 32) | (unsigned)max(a, b);
    unsigned long long h = (key ^ (key >> 31)) * 0x9e3779b97f4a7c15ull;
    h = (h ^ (h >> 29)) & (slots - 1);
    for (unsigned long long probe = 0; probe < slots; ++probe, h = (h + 1) & (slots - 1)) {
      const unsigned long long old = atomicCAS(&keys[h], 0ull, key);
      if (old == 0ull || old == key) {
        delta += (atomicXor(&odd[h], 1u) & 1u) ? -1 : 1;
        break;
      }
    }
  }
  delta = __reduce_add_sync(0xffffffffu, delta);
  if ((threadIdx.x & 31) == 0 && delta != 0) atomicAdd(&info->odd_edges, (unsigned long long)(long long)delta);
  if (bad) info->bad_index = 1u;
  if (deg) info->degenerate = 1u;
}

// quantised coordinates of the vertices (below 2^27: the box has at most 2^19 sub-cells per axis)
__global__ void __launch_bounds__(NT) k_mesh_quantise(const float* __restrict__ vert, long long nv, double lo0,
                                                      double lo1, double lo2, double scale, int* __restrict__ q) {
  const double lo[3] = {lo0, lo1, lo2};
  for (long long i = blockIdx.x * (long long)NT + threadIdx.x; i < nv; i += (long long)gridDim.x * NT)
#pragma unroll
    for (int k = 0; k < 3; ++k) q[3 * i + k] = (int)llround(((double)vert[3 * i + k] - lo[k]) * scale);
}

struct Rows {
  int y0, y1, z0, z1;  // rows (sub-cell indices) a projection's bounding box covers, inclusive
};
// rows a whose centre 256 a + 128 lies in [mn, mx], clamped to [0, n)
__device__ __forceinline__ void row_range(int mn, int mx, int n, int& a0, int& a1) {
  a0 = max((mn - 128 + 255) >> 8, 0);  // ceil((mn - 128) / 256)
  a1 = min((mx - 128) >> 8, n - 1);    // floor((mx - 128) / 256)
}
__device__ __forceinline__ Rows rows_of(const int* __restrict__ q, const int* __restrict__ tri, long long t, int ny,
                                        int nz, int (&v)[3][3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const long long i = tri[3 * t + c];
#pragma unroll
    for (int k = 0; k < 3; ++k) v[c][k] = q[3 * i + k];
  }
  Rows r;
  row_range(min(v[0][1], min(v[1][1], v[2][1])), max(v[0][1], max(v[1][1], v[2][1])), ny, r.y0, r.y1);
  row_range(min(v[0][2], min(v[1][2], v[2][2])), max(v[0][2], max(v[1][2], v[2][2])), nz, r.z0, r.z1);
  return r;
}

// FILL 0: entries per tile into cnt; 1: the entries, at the positions cnt counts up from
template <int FILL>
__global__ void __launch_bounds__(NT) k_mesh_bin(const int* __restrict__ q, const int* __restrict__ tri, long long nt,
                                                 int ny, int nz, unsigned* __restrict__ cnt,
                                                 unsigned* __restrict__ list, int tiles_y) {
  for (long long t = blockIdx.x * (long long)NT + threadIdx.x; t < nt; t += (long long)gridDim.x * NT) {
    int v[3][3];
    const Rows r = rows_of(q, tri, t, ny, nz, v);
    if (r.y0 > r.y1 || r.z0 > r.z1) continue;
    for (int tz = r.z0 / TILE; tz <= r.z1 / TILE; ++tz)
      for (int ty = r.y0 / TILE; ty <= r.y1 / TILE; ++ty) {
        const unsigned pos = atomicAdd(&cnt[(long long)tz * tiles_y + ty], 1u);
        if (FILL) list[pos] = (unsigned)t;
      }
  }
}

// exclusive scan of cnt[0, n) into start[0, n] and back into cnt (the fill's cursors); one block
__global__ void __launch_bounds__(1024) k_mesh_scan(unsigned* __restrict__ cnt, unsigned* __restrict__ start,
                                                    long long n, MeshInfo* info) {
  __shared__ unsigned long long s_w[32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned long long base = 0;
  for (long long i0 = 0; i0 < n; i0 += 1024) {
    const long long i = i0 + threadIdx.x;
    const unsigned long long c = i < n ? cnt[i] : 0u;
    unsigned long long x = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, x, d);
      if (lane >= d) x += y;
    }
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    unsigned long long before = 0, all = 0;
    for (int w = 0; w < 32; ++w) {
      if (w < warp) before += s_w[w];
      all += s_w[w];
    }
    const unsigned long long at = base + before + x - c;
    if (i < n) {
      start[i] = (unsigned)at;
      cnt[i] = (unsigned)at;
    }
    base += all;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    start[n] = (unsigned)base;
    info->total = base;
  }
}

// sign of the (y, z) orientation of the centre against the directed edge
// a -> b, with the centre moved by (delta^2, delta)
__device__ __forceinline__ int edge_sign(const int* a, const int* b, int py, int pz) {
  const long long ey = b[1] - a[1], ez = b[2] - a[2];
  const long long o = ey * (pz - a[2]) - ez * (py - a[1]);
  if (o != 0) return o > 0 ? 1 : -1;
  if (ey != 0) return ey > 0 ? 1 : -1;
  if (ez != 0) return ez < 0 ? 1 : -1;
  return 0;
}

// Number of the row's centres i in [0, nxs) that see the triangle's crossing
// ahead (those with i < m), -1 if the row (j, k) misses the triangle.
__device__ __forceinline__ int crossing(const int (&v)[3][3], int j, int k, int nxs) {
  const int py = 256 * j + 128, pz = 256 * k + 128;
  const int *A = v[0], *B = v[1], *C = v[2];
  const int s1 = edge_sign(A, B, py, pz), s2 = edge_sign(B, C, py, pz), s3 = edge_sign(C, A, py, pz);
  if (s1 == 0 || s1 != s2 || s2 != s3) return -1;
  const long long e1[3] = {B[0] - A[0], B[1] - A[1], B[2] - A[2]};
  const long long e2[3] = {C[0] - A[0], C[1] - A[1], C[2] - A[2]};
  const long long nx = e1[1] * e2[2] - e1[2] * e2[1];
  const long long nyv = e1[2] * e2[0] - e1[0] * e2[2];
  const long long nzv = e1[0] * e2[1] - e1[1] * e2[0];
  // the crossing is at or ahead of centre i (x = 256 i + 128) iff
  // sgn(nx) (D0 - 256 nx i) >= 0 with D0 = n . (A - (128, py, pz)):
  // a - b i >= 0, decreasing in i; m = the number of such i in [0, nxs)
  const __int128 D0 = (__int128)nx * (A[0] - 128) + (__int128)nyv * (A[1] - py) + (__int128)nzv * (A[2] - pz);
  const __int128 a = nx > 0 ? D0 : -D0;
  const __int128 b = (__int128)(nx > 0 ? nx : -nx) * 256;
  int lo = -1, hi = nxs;  // invariant: a - b lo >= 0 (or lo = -1), a - b hi < 0 (or hi = nxs)
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (a - b * mid >= 0) lo = mid;
    else hi = mid;
  }
  return lo + 1;
}

// One block per tile of 16 x 16 rows, rows in passes of `chunk` bits (a multiple
// of 64, from the far end of x so that a pass's parity carries into the next).
// Dense tiles give each thread a triangle of the list and its few rows; tiles
// with few triangles, which may cover all their rows, give each thread a row.
__global__ void __launch_bounds__(NT) k_mesh_rows(const int* __restrict__ q, const int* __restrict__ tri,
                                                  const unsigned* __restrict__ start,
                                                  const unsigned* __restrict__ list, int nxs, int ny, int nz,
                                                  int tiles_y, int s, int chunk,
                                                  unsigned long long* __restrict__ bricks, int gx, int gy, int gz,
                                                  int wpb, MeshInfo* info) {
  extern __shared__ unsigned s_tog[];  // [256 rows][chunk / 32 + 1]: the odd stride spreads the rows over the banks
  __shared__ int s_hits[NT];
  const int tid = threadIdx.x, ty = blockIdx.x % tiles_y, tz = blockIdx.x / tiles_y;
  const int words = chunk / 32, stride = words + 1;
  const int j0 = ty * TILE, k0 = tz * TILE;
  const unsigned e0 = start[blockIdx.x], e1 = start[blockIdx.x + 1];
  const bool by_row = e1 - e0 < 64u;
  const int n = 1 << s, per = TILE >> s;  // brick rows per tile side
  s_hits[tid] = 0;
  unsigned carry = 0u;  // this thread's row: parity of the toggles beyond the pass
  for (int x0 = (nxs - 1) / chunk * chunk; x0 >= 0; x0 -= chunk) {
    const bool first = x0 + chunk >= nxs;
    for (int w = 0; w < stride; ++w) s_tog[w * NT + tid] = 0u;
    __syncthreads();
    auto hit = [&](int m, int row) {
      if (first && atomicAdd(&s_hits[row], 1) == MAX_HITS) info->hits_exceeded = 1;
      const int bit = m - 1 - x0;
      if (bit >= 0 && bit < chunk) atomicXor(&s_tog[row * stride + (bit >> 5)], 1u << (bit & 31));
    };
    if (by_row) {
      const int j = j0 + tid % TILE, k = k0 + tid / TILE;
      for (unsigned e = e0; e < e1; ++e) {
        int v[3][3];
        const Rows r = rows_of(q, tri, list[e], ny, nz, v);
        if (j < r.y0 || j > r.y1 || k < r.z0 || k > r.z1) continue;
        const int m = crossing(v, j, k, nxs);
        if (m >= 0) hit(m, tid);
      }
    } else {
      for (unsigned e = e0 + tid; e < e1; e += NT) {
        int v[3][3];
        const Rows r = rows_of(q, tri, list[e], ny, nz, v);
        const int ja = max(r.y0, j0), jb = min(r.y1, j0 + TILE - 1);
        const int ka = max(r.z0, k0), kb = min(r.z1, k0 + TILE - 1);
        for (int k = ka; k <= kb; ++k)
          for (int j = ja; j <= jb; ++j) {
            const int m = crossing(v, j, k, nxs);
            if (m >= 0) hit(m, (k - k0) * TILE + (j - j0));
          }
      }
    }
    __syncthreads();
    // bit i of the row = parity of the toggles at or beyond i
    for (int w = words - 1; w >= 0; --w) {
      unsigned y = s_tog[tid * stride + w];
      const unsigned odd = __popc(y) & 1u;
      y ^= y >> 1;
      y ^= y >> 2;
      y ^= y >> 4;
      y ^= y >> 8;
      y ^= y >> 16;
      s_tog[tid * stride + w] = y ^ (carry ? ~0u : 0u);
      carry ^= odd;
    }
    __syncthreads();
    // bricks of the pass: a word collects the n bits of its rows
    const int cx0 = x0 >> s, ncx = min(chunk >> s, gx - cx0);
    for (int b = tid; b < per * per * ncx * wpb; b += NT) {
      const int w = b % wpb, cx = (b / wpb) % ncx, r = b / wpb / ncx;
      const int cy = (j0 >> s) + r % per, cz = (k0 >> s) + r / per;
      if (cy >= gy || cz >= gz) continue;
      const int bit = cx << s;
      unsigned long long word = 0ull;
      // s = 3: word w is the layer sz = w; otherwise the one word holds all n layers
      const int za = wpb > 1 ? w : 0, zb = wpb > 1 ? w + 1 : n;
      for (int sz = za; sz < zb; ++sz)
        for (int sy = 0; sy < n; ++sy) {
          const int row = ((r / per) * n + sz) * TILE + (r % per) * n + sy;
          const unsigned long long bits = (s_tog[row * stride + (bit >> 5)] >> (bit & 31)) & ((1u << n) - 1u);
          word |= bits << (((sz - za) * n + sy) * n);
        }
      bricks[(((long long)cz * gy + cy) * gx + cx0 + cx) * wpb + w] = word;
    }
    __syncthreads();
  }
}

int mesh_fail(int code, const char* msg) { return psm::set_error(code, msg); }

// The argument checks without a GPU (the same findings as the first phase's).
int check_on_host(const float* vertices, int64_t nv, const int32_t* triangles, int64_t nt, int s) {
  for (int64_t i = 0; i < 3 * nt; ++i)
    if (triangles[i] < 0 || triangles[i] >= nv) return mesh_fail(PSM_ERR_ARG, "triangle vertex index out of range");
  std::vector<uint64_t> edges;
  edges.reserve((size_t)nt * 3);
  for (int64_t t = 0; t < nt; ++t)
    for (int c = 0; c < 3; ++c) {
      const uint32_t a = (uint32_t)triangles[3 * t + c], b = (uint32_t)triangles[3 * t + (c + 1) % 3];
      if (a == b) return mesh_fail(PSM_ERR_ARG, "degenerate triangle (repeated vertex index)");
      edges.push_back(((uint64_t)std::min(a, b) << 32) | std::max(a, b));
    }
  std::sort(edges.begin(), edges.end());
  for (size_t i = 0; i < edges.size();) {
    size_t k = i;
    while (k < edges.size() && edges[k] == edges[i]) ++k;
    if ((k - i) & 1) return mesh_fail(PSM_ERR_ARG, "mesh is not closed (an edge has an odd number of triangles)");
    i = k;
  }
  for (int k = 0; k < 3; ++k) {
    double mn = 1e300, mx = -1e300;
    for (int64_t i = 0; i < nv; ++i) {
      const double c = (double)vertices[3 * i + k];
      if (!std::isfinite(c)) return mesh_fail(PSM_ERR_ARG, "non-finite vertex coordinate");
      mn = std::min(mn, c);
      mx = std::max(mx, c);
    }
    if (!(std::ceil(mx) + 1.0 - (std::floor(mn) - 1.0) <= (double)((int64_t)1 << (19 - s))))
      return mesh_fail(PSM_ERR_ARG, "mesh extent exceeds 2^(19-s) cells");
  }
  return PSM_OK;
}

}  // namespace

extern "C" int psm_geom_voxelize_mesh(const float* vertices, int64_t nv, const int32_t* triangles, int64_t nt, int s,
                                      psm_geom_field* out) {
  if (!out) return mesh_fail(PSM_ERR_ARG, "psm_geom_voxelize_mesh: NULL output");
  out->bricks = nullptr;
  if (!vertices || !triangles) return mesh_fail(PSM_ERR_ARG, "psm_geom_voxelize_mesh: NULL argument");
  if (s < 0 || s > 3) return mesh_fail(PSM_ERR_ARG, "super-sampling depth s must be 0..3");
  if (nv < 3 || nt < 1 || nv > (1ll << 31) - 1 || nt > (1ll << 31) - 1)
    return mesh_fail(PSM_ERR_ARG, "mesh needs 3 <= vertices < 2^31 and 1 <= triangles < 2^31");
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev < 1) {
    cudaGetLastError();
    const int rc = check_on_host(vertices, nv, triangles, nt, s);
    return rc != PSM_OK ? rc : mesh_fail(PSM_ERR_CUDA, "mesh voxeliser setup failed");
  }
  // first phase: the mesh, its quantised vertices, the edge table, the tile
  // counts (for grids of up to 2^17 tiles) and the findings, in one allocation.
  // It stays below cudaMalloc's 2 MB pages for meshes of up to about 9,000
  // triangles (counts for 2^18 tiles made it larger for every mesh: a 20^3 cube
  // at s = 3 385 us a call, now 293); a second allocation costs 200 us, and a
  // grid of more tiles takes tens of milliseconds.
  unsigned long long slots = 64;
  while (slots < (unsigned long long)nt * 4) slots *= 2;
  constexpr size_t TILES0 = (size_t)1 << 17;
  size_t at = 0;
  auto part = [&](size_t bytes) {
    const size_t o = at;
    at += (bytes + 255) / 256 * 256;
    return o;
  };
  const size_t o_info = part(sizeof(MeshInfo)), o_keys = part(slots * 8), o_odd = part(slots * 4);
  const size_t o_v = part(sizeof(float) * 3 * (size_t)nv), o_t = part(sizeof(int) * 3 * (size_t)nt);
  const size_t o_q = part(sizeof(int) * 3 * (size_t)nv), o_cnt = part(TILES0 * 4), o_start = part((TILES0 + 1) * 4);
  char *m1 = nullptr, *m2 = nullptr, *m3 = nullptr;
  auto release = [&]() {
    cudaFree(m1);
    cudaFree(m2);
    cudaFree(m3);
  };
  auto failed = [&](cudaError_t err, const char* msg) {
    cudaGetLastError();
    release();
    return mesh_fail(err == cudaErrorMemoryAllocation ? PSM_ERR_OOM : PSM_ERR_CUDA, msg);
  };
  cudaError_t e = cudaMalloc(&m1, at);
  if (e != cudaSuccess) return failed(e, "mesh voxeliser setup failed");
  MeshInfo* info = reinterpret_cast<MeshInfo*>(m1 + o_info);
  float* dv = reinterpret_cast<float*>(m1 + o_v);
  int* dt = reinterpret_cast<int*>(m1 + o_t);
  int* dq = reinterpret_cast<int*>(m1 + o_q);
  e = cudaMemcpy(dv, vertices, sizeof(float) * 3 * (size_t)nv, cudaMemcpyDefault);
  if (e == cudaSuccess) e = cudaMemcpy(dt, triangles, sizeof(int) * 3 * (size_t)nt, cudaMemcpyDefault);
  if (e != cudaSuccess) return failed(e, "mesh read failed");
  e = cudaMemsetAsync(m1, 0, o_v);  // findings, keys, parities
  if (e == cudaSuccess) e = cudaMemsetAsync(info->mn, 0xff, sizeof info->mn);
  if (e != cudaSuccess) return failed(e, "mesh voxeliser setup failed");
  auto blocks = [](int64_t work) { return (int)std::min<int64_t>((work + NT - 1) / NT, 4096); };
  k_mesh_extent<<<std::min(blocks(nv), 304), NT>>>(dv, nv, info);
  k_mesh_edges<<<blocks(3 * nt), NT>>>(dt, nt, nv, reinterpret_cast<unsigned long long*>(m1 + o_keys),
                                       reinterpret_cast<unsigned*>(m1 + o_odd), slots, info);
  e = cudaGetLastError();
  MeshInfo hi;
  if (e == cudaSuccess) e = cudaMemcpy(&hi, info, sizeof hi, cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return failed(e, "mesh voxeliser kernels failed");
  auto refused = [&](const char* msg) {
    release();
    return mesh_fail(PSM_ERR_ARG, msg);
  };
  if (hi.bad_index) return refused("triangle vertex index out of range");
  if (hi.degenerate) return refused("degenerate triangle (repeated vertex index)");
  if (hi.odd_edges != 0) return refused("mesh is not closed (an edge has an odd number of triangles)");
  if (hi.non_finite) return refused("non-finite vertex coordinate");
  int64_t dims[3];
  double lo[3];
  for (int k = 0; k < 3; ++k) {
    lo[k] = std::floor((double)from_order_bits(hi.mn[k])) - 1.0;
    const double d = std::ceil((double)from_order_bits(hi.mx[k])) + 1.0 - lo[k];
    if (!(d <= (double)((int64_t)1 << (19 - s)))) return refused("mesh extent exceeds 2^(19-s) cells");
    dims[k] = (int64_t)d;
  }
  const int n = 1 << s;
  const int wpb = s == 3 ? 8 : 1;
  const int nxs = (int)(dims[0] * n), ny = (int)(dims[1] * n), nz = (int)(dims[2] * n);
  const int tiles_y = (ny + TILE - 1) / TILE, tiles_z = (nz + TILE - 1) / TILE;
  const size_t ntiles = (size_t)tiles_y * tiles_z;
  const size_t nwords = (size_t)dims[0] * dims[1] * dims[2] * wpb;
  // second phase: tile lists, then the rows
  unsigned* cnt = reinterpret_cast<unsigned*>(m1 + o_cnt);
  unsigned* start = reinterpret_cast<unsigned*>(m1 + o_start);
  if (ntiles > TILES0) {
    e = cudaMalloc(&m2, (2 * ntiles + 1) * 4);
    if (e != cudaSuccess) return failed(e, "mesh voxeliser setup failed");
    cnt = reinterpret_cast<unsigned*>(m2);
    start = cnt + ntiles;
  }
  e = cudaMemsetAsync(cnt, 0, ntiles * 4);
  if (e == cudaSuccess) {
    k_mesh_quantise<<<blocks(nv), NT>>>(dv, nv, lo[0], lo[1], lo[2], std::ldexp(1.0, s + 8), dq);
    k_mesh_bin<0><<<blocks(nt), NT>>>(dq, dt, nt, ny, nz, cnt, nullptr, tiles_y);
    k_mesh_scan<<<1, 1024>>>(cnt, start, (long long)ntiles, info);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(&hi, info, sizeof hi, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && hi.total > 0xffffffffull) e = cudaErrorInvalidValue;
  const size_t list_bytes = ((size_t)hi.total * 4 + 255) / 256 * 256;
  if (e == cudaSuccess) e = cudaMalloc(&m3, list_bytes + nwords * 8);
  if (e != cudaSuccess) return failed(e, "mesh voxeliser kernels failed");
  unsigned* list = reinterpret_cast<unsigned*>(m3);
  unsigned long long* dbr = reinterpret_cast<unsigned long long*>(m3 + list_bytes);
  const int chunk = std::min(CHUNK_MAX, (nxs + 63) / 64 * 64);
  k_mesh_bin<1><<<blocks(nt), NT>>>(dq, dt, nt, ny, nz, cnt, list, tiles_y);
  k_mesh_rows<<<(unsigned)ntiles, NT, (size_t)NT * (chunk / 32 + 1) * 4>>>(
      dq, dt, start, list, nxs, ny, nz, tiles_y, s, chunk, dbr, (int)dims[0], (int)dims[1], (int)dims[2], wpb, info);
  e = cudaGetLastError();
  uint64_t* bricks = static_cast<uint64_t*>(std::malloc(nwords * sizeof(uint64_t)));
  if (!bricks) {
    release();
    return mesh_fail(PSM_ERR_OOM, "geometry field allocation failed");
  }
  // the field's pages exist before the copy: into memory that the heap has only
  // just grown by, the copy of a 9.3 MB field took 7.6 ms instead of 0.2 (the
  // same call 0.6 or 8.2 ms by what else the process holds, now 0.6 or 0.8)
  for (size_t o = 0; o < nwords * sizeof(uint64_t); o += 4096) reinterpret_cast<volatile char*>(bricks)[o] = 0;
  if (e == cudaSuccess) e = cudaMemcpy(bricks, dbr, sizeof(uint64_t) * nwords, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(&hi, info, sizeof hi, cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) {
    std::free(bricks);
    return failed(e, "mesh voxeliser kernels failed");
  }
  release();
  if (hi.hits_exceeded) {
    std::free(bricks);
    return mesh_fail(PSM_ERR_UNSUPPORTED, "more than 256 surface crossings along one sub-cell row");
  }
  out->bricks = bricks;
  out->gx = dims[0];
  out->gy = dims[1];
  out->gz = dims[2];
  out->s = s;
  for (int k = 0; k < 3; ++k) out->lo[k] = lo[k];
  return PSM_OK;
}
