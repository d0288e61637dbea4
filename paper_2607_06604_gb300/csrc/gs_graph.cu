// Lattice quantisation and the device radius-search graph build (Sec. 2.1).
//
// Points are binned into a uniform cell grid, kx x ky x kz cells per E_nb
// cubed, so every neighbour lies in a stencil of (2 kx + 1)(2 ky + 1)(2 kz + 1)
// cells. Points are relabelled in cell order (x-major, caller index within a
// cell), which makes rows come out sorted when the stencil's cells are
// visited in increasing cell order, and keeps neighbour ids close to the hub
// id (good L2 locality for the counting kernels). Only the oriented half
// N+(i) = {j > i} is stored: every tuple is counted at its smallest label.
// Thin cells along x make N+(i) nearly the half ball ahead of i, so rows are
// of nearly equal length: with cells as wide as E_nb they varied by 75% about
// the mean with the hub's place in its cell, which cost the triangle kernel
// pair tests and the tetrahedron kernel its longest rows.
#include <algorithm>
#include <mutex>

#include "gs_host_copy.h"
#include "gs_internal.cuh"

namespace gs {
namespace {

constexpr int kMaxCellsPerAxis = 256;
constexpr int kRowThreads = 256;    // row pass: a warp per group of hubs
constexpr int kRowWarps = kRowThreads / 32;
constexpr int kRowHubs = 4;         // hubs of one cell that a warp takes together
constexpr int kMaxRuns = 96;        // id ranges of a stencil (9 x 5 columns, split in z)
constexpr int kBucketMax = 2048;    // squared-distance buckets of the bin lookup

struct GridDesc {
  int nc[3];
  int k[3];          // cells per E_nb along each axis
  int64_t lo[3];     // open box: grid origin
  int64_t width[3];  // open box: cell width
  int64_t box;       // periodic box side, 0 = open
};

__device__ inline int cell_axis(const GridDesc& G, int a, int x) {
  if (G.box) return (int)(((int64_t)x * G.nc[a]) / G.box);
  return (int)(((int64_t)x - G.lo[a]) / G.width[a]);
}

__global__ void k_quantize(const double* pos, int64_t n3, int64_t box_u, int periodic,
                           int32_t* out, int* err) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n3;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double s = pos[i] * 1024.0;  // exact: scaling by a power of two
    double f = floor(s);
    if (!(f > -9.0e15 && f < 9.0e15)) {  // not finite or beyond exact integers
      atomicOr(err, kErrRange);
      out[i] = 0;
      continue;
    }
    int64_t X = (int64_t)f;
    if (periodic) {
      X %= box_u;
      if (X < 0) X += box_u;
    } else if (X < 0 || X >= box_u) {
      atomicOr(err, kErrRange);
      X = 0;
    }
    out[i] = (int32_t)X;
  }
}

// Validates coordinates and computes the bounding box.
__global__ void k_check_bbox(const int32_t* xyz, int64_t n, int64_t box, int* bbox, int* err) {
  int mn[3] = {INT_MAX, INT_MAX, INT_MAX}, mx[3] = {INT_MIN, INT_MIN, INT_MIN};
  int bad = 0;
  const int64_t limit = box ? box : (int64_t(1) << 30);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    for (int a = 0; a < 3; ++a) {
      const int x = xyz[3 * i + a];
      if (x < 0 || (int64_t)x >= limit) bad = 1;
      mn[a] = min(mn[a], x);
      mx[a] = max(mx[a], x);
    }
  }
  for (int o = 16; o; o >>= 1) {
    for (int a = 0; a < 3; ++a) {
      mn[a] = min(mn[a], __shfl_xor_sync(0xffffffffu, mn[a], o));
      mx[a] = max(mx[a], __shfl_xor_sync(0xffffffffu, mx[a], o));
    }
    bad |= __shfl_xor_sync(0xffffffffu, bad, o);
  }
  if ((threadIdx.x & 31) == 0) {
    for (int a = 0; a < 3; ++a) {
      atomicMin(bbox + a, mn[a]);
      atomicMax(bbox + 3 + a, mx[a]);
    }
    if (bad) atomicOr(err, kErrRange);
  }
}

__global__ void k_cell_keys(const int32_t* xyz, int64_t n, GridDesc G, int32_t* key,
                            int32_t* count) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int cx = cell_axis(G, 0, xyz[3 * i]);
    const int cy = cell_axis(G, 1, xyz[3 * i + 1]);
    const int cz = cell_axis(G, 2, xyz[3 * i + 2]);
    const int c = (cx * G.nc[1] + cy) * G.nc[2] + cz;
    key[i] = c;
    atomicAdd(count + c, 1);
  }
}

// Groups points by cell (order inside a cell is arbitrary here).
__global__ void k_scatter(const int32_t* key, int64_t n, int32_t* cursor, int32_t* tmp) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int pos = atomicAdd(cursor + key[i], 1);
    tmp[pos] = (int32_t)i;
  }
}

// Orders each cell by caller index: slot s goes to cell_start + rank, rank =
// number of points of the same cell with a smaller caller index.
__global__ void k_rank_in_cell(const int32_t* key, const int32_t* tmp, int64_t n,
                               const int32_t* cell_start, const int32_t* xyz, int4* xyzp,
                               int32_t* cell) {
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n;
       s += (int64_t)gridDim.x * blockDim.x) {
    const int32_t me = tmp[s];
    const int c = key[me];
    const int b = cell_start[c], e = cell_start[c + 1];
    int r = 0;
    for (int t = b; t < e; ++t) r += tmp[t] < me;
    xyzp[b + r] = make_int4(xyz[3 * (int64_t)me], xyz[3 * (int64_t)me + 1],
                            xyz[3 * (int64_t)me + 2], me);
    cell[b + r] = c;
  }
}

// Id ranges of the later neighbours' cells: points [beg, end) seen at the
// periodic image code (two bits per axis: image + 1).
struct Run {
  int beg, end, code, pad;
};
constexpr int kNoShift = 1 | (1 << 2) | (1 << 4);

// The runs of hubs i0.. of the cell (cx, cy, cz): per column of the stencil
// the cells cz - kz .. cz + kz are consecutive ids (two runs where they wrap).
// Ids up to i0 are cut off. Runs come out in ascending order; at the faces of
// a periodic box they are ranked first. Returns their number.
__device__ inline int stencil_runs(const GridDesc& G, const int32_t* __restrict__ start, int cx,
                                   int cy, int cz, int i0, Run* run, Run* tmp) {
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  const bool per = G.box != 0;
  const bool faces = per && (cx < G.k[0] || cx >= G.nc[0] - G.k[0] || cy < G.k[1] ||
                             cy >= G.nc[1] - G.k[1] || cz < G.k[2] || cz >= G.nc[2] - G.k[2]);
  const int wy = 2 * G.k[1] + 1, ncol = (2 * G.k[0] + 1) * wy;
  Run* out = faces ? tmp : run;
  int n = 0;
  for (int q0 = 0; q0 < ncol; q0 += 32) {
    const int q = q0 + lane;
    int x = cx + q / wy - G.k[0], y = cy + q % wy - G.k[1];
    int code = kNoShift;
    bool ok = q < ncol;
    if (x < 0) {
      ok = ok && per;
      x += G.nc[0];
      code -= 1;
    } else if (x >= G.nc[0]) {
      ok = ok && per;
      x -= G.nc[0];
      code += 1;
    }
    if (y < 0) {
      ok = ok && per;
      y += G.nc[1];
      code -= 1 << 2;
    } else if (y >= G.nc[1]) {
      ok = ok && per;
      y -= G.nc[1];
      code += 1 << 2;
    }
    const int64_t col = ((int64_t)x * G.nc[1] + y) * G.nc[2];
    auto add = [&](bool use, int z0, int z1, int cd) {
      Run r{0, 0, cd, 0};
      if (use) {
        r.beg = max(start[col + z0], i0 + 1);
        r.end = start[col + z1 + 1];
      }
      const bool v = r.beg < r.end;
      const unsigned m = __ballot_sync(0xffffffffu, v);
      if (v) out[n + __popc(m & below)] = r;
      n += __popc(m);
    };
    const int z0 = cz - G.k[2], z1 = cz + G.k[2];
    add(ok, max(z0, 0), min(z1, G.nc[2] - 1), code);
    if (faces) {
      add(ok && z0 < 0, z0 + G.nc[2], G.nc[2] - 1, code - (1 << 4));
      add(ok && z1 >= G.nc[2], 0, z1 - G.nc[2], code + (1 << 4));
    }
  }
  __syncwarp();
  if (faces) {
    for (int q = lane; q < n; q += 32) {
      const Run r = tmp[q];
      int rank = 0;
      for (int t = 0; t < n; ++t) rank += tmp[t].beg < r.beg ? 1 : 0;
      run[rank] = r;
    }
    __syncwarp();
  }
  return n;
}

// Row pass: a warp takes up to kRowHubs consecutive hubs of one cell (they
// share the stencil) and tests every candidate of its runs against all of
// them, lanes over candidates (128-bit coalesced loads through L1/L2); a
// ballot compacts the hits, so rows come out sorted without a sort. The
// image of a run is fixed by its cell, so a candidate costs three
// subtractions and three 64-bit multiply-adds per hub.
// FILL = false counts |N+(i)| and takes the totals; FILL = true writes the
// packed words (and sums |N+(j)| over the edges). Only hubs in [h0, h1) are
// processed (chunked out-of-core builds).
// Bound by latency with 72 registers (59% of issue slots); the two passes over 3e6 uniform points (402
// edges a row, E_nb = 40 h^-1Mpc) take 19.5 ms against 48 ms for a CTA per
// cell of side E_nb with the stencil staged in shared memory (twice the
// candidates, one hub per warp at a time, per-candidate minimum images).
template <bool FILL>
__global__ void __launch_bounds__(kRowThreads) k_rows(
    const int4* __restrict__ xyzp, const int32_t* __restrict__ cell, GridDesc G,
    const int32_t* __restrict__ start, const int64_t* __restrict__ e2g, int nb, int bk_shift,
    int bk_n, int32_t* deg, const int64_t* __restrict__ ptr, uint32_t* __restrict__ adj,
    int64_t h0, int64_t h1, int64_t out_off, unsigned long long* totals) {
  __shared__ Run s_run[2][kRowWarps][kMaxRuns];
  __shared__ int64_t e2[kMaxBins + 1];
  __shared__ uint8_t s_bk[kBucketMax];
  for (int b = threadIdx.x; b <= nb; b += kRowThreads) e2[b] = e2g[b];
  if (FILL)
    for (int k = threadIdx.x; k < bk_n; k += kRowThreads) {
      const int64_t x = (int64_t)k << bk_shift;
      int b = 0;
      while (b + 1 < nb && e2g[b + 1] <= x) ++b;
      s_bk[k] = (uint8_t)b;
    }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned below = (1u << lane) - 1u;
  Run* run = s_run[0][warp];
  const unsigned long long e2lo = (unsigned long long)e2[0],
                           span = (unsigned long long)(e2[nb] - e2[0]);
  unsigned long long edges = 0, probe = 0;
  int longest = 0;
  const int64_t nblk = (h1 + kRowHubs - 1) / kRowHubs;
  for (int64_t q = h0 / kRowHubs + blockIdx.x * (int64_t)kRowWarps + warp; q < nblk;
       q += (int64_t)gridDim.x * kRowWarps) {
    int i = (int)max(q * kRowHubs, h0);
    const int iend = (int)min((q + 1) * kRowHubs, h1);
    while (i < iend) {
      const int c = cell[i];
      int H = 1;
      while (i + H < iend && cell[i + H] == c) ++H;
      const int cz = c % G.nc[2], cy = (c / G.nc[2]) % G.nc[1], cx = c / (G.nc[2] * G.nc[1]);
      const int nr = stencil_runs(G, start, cx, cy, cz, i, run, s_run[1][warp]);
      // hubs beyond H repeat the last one and keep nothing
      int4 P[kRowHubs];
      int px[kRowHubs], py[kRowHubs], pz[kRowHubs], cnt[kRowHubs];
      uint32_t* out[kRowHubs];
#pragma unroll
      for (int h = 0; h < kRowHubs; ++h) {
        P[h] = xyzp[min(i + h, i + H - 1)];
        px[h] = P[h].x, py[h] = P[h].y, pz[h] = P[h].z;
        cnt[h] = 0;
        out[h] = FILL ? adj + (ptr[min(i + h, i + H - 1)] - out_off) : nullptr;
      }
      int code = kNoShift;
      for (int r = 0; r < nr; ++r) {
        const Run R = run[r];
        if (R.code != code) {  // the hubs as seen from the run's image
          code = R.code;
          const unsigned sx = (unsigned)((code & 3) - 1) * (unsigned)G.box,
                         sy = (unsigned)(((code >> 2) & 3) - 1) * (unsigned)G.box,
                         sz = (unsigned)((code >> 4) - 1) * (unsigned)G.box;
#pragma unroll
          for (int h = 0; h < kRowHubs; ++h) {
            px[h] = (int)((unsigned)P[h].x - sx);
            py[h] = (int)((unsigned)P[h].y - sy);
            pz[h] = (int)((unsigned)P[h].z - sz);
          }
        }
        for (int t0 = R.beg; t0 < R.end; t0 += 32) {
          const int t = t0 + lane;
          const bool in = t < R.end;
          const int4 Q = in ? xyzp[t] : make_int4(0, 0, 0, 0);
          const int dt = FILL && in ? deg[t] : 0;
#pragma unroll
          for (int h = 0; h < kRowHubs; ++h) {
            if (h >= H) continue;  // uniform
            // modulo 2^32 on purpose: the true difference is a few cells
            const int x = (int)((unsigned)Q.x - (unsigned)px[h]),
                      y = (int)((unsigned)Q.y - (unsigned)py[h]),
                      z = (int)((unsigned)Q.z - (unsigned)pz[h]);
            const unsigned long long D2 = (unsigned long long)((long long)x * x + (long long)y * y +
                                                               (long long)z * z);
            const bool hit = in && t > i + h && D2 - e2lo < span;
            const unsigned m = __ballot_sync(0xffffffffu, hit);
            if (FILL && hit) {
              int b;
              if (bk_n) {
                b = s_bk[D2 >> bk_shift];
                b += (long long)D2 >= e2[b + 1] ? 1 : 0;
              } else {
                b = 0;
                int hi = nb;
                while (hi - b > 1) {
                  const int mid = (b + hi) >> 1;
                  if (e2[mid] <= (long long)D2) b = mid;
                  else hi = mid;
                }
              }
              out[h][cnt[h] + __popc(m & below)] = ((uint32_t)t << 8) | (uint32_t)b;
              probe += (unsigned long long)dt;
            }
            cnt[h] += __popc(m);
          }
        }
      }
#pragma unroll
      for (int h = 0; h < kRowHubs; ++h) {
        if (h >= H) continue;
        if (!FILL) {
          if (lane == 0) deg[i + h] = cnt[h];
          edges += (unsigned long long)cnt[h];
          longest = max(longest, cnt[h]);
        } else {
          const int pad = (int)pad_row(cnt[h]);
          if (cnt[h] + lane < pad) out[h][cnt[h] + lane] = kSentinel;
        }
      }
      __syncwarp();  // the runs are rewritten for the next group
      i += H;
    }
  }
  if (FILL) {
    for (int o = 16; o; o >>= 1) probe += __shfl_xor_sync(0xffffffffu, probe, o);
    if (lane == 0 && probe) atomicAdd(totals, probe);
  } else if (lane == 0) {
    if (edges) atomicAdd(totals + 1, edges);
    atomicMax((int*)(totals + 2), longest);
  }
}

__global__ void k_pad_lengths(const int32_t* deg, int64_t n, int64_t* len) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= n;
       i += (int64_t)gridDim.x * blockDim.x)
    len[i] = (i < n) ? pad_row(deg[i]) : 0;
}

int grid_blocks(int64_t work, int threads) {
  int64_t b = (work + threads - 1) / threads;
  return (int)std::max<int64_t>(1, std::min<int64_t>(b, 152 * 16));
}

}  // namespace

int quantize_device(const double* d_pos, int64_t n, int64_t box_u, int periodic, int32_t* d_xyz,
                    cudaStream_t s, Scratch& sc) {
  int* err = sc.alloc<int>(1);
  if (!err) return GS_ENOMEM;
  cudaMemsetAsync(err, 0, sizeof(int), s);
  { k_quantize<<<grid_blocks(3 * n, 256), 256, 0, s>>>(d_pos, 3 * n, box_u, periodic, d_xyz, err); note_launch(); }
  int h = 0;
  cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s);
  cudaError_t e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_status(e);
  return h ? GS_ERANGE : GS_OK;
}

int build_graph_device(const int32_t* d_xyz, int64_t n, int64_t box_u,
                       const std::vector<int64_t>& edges, const Opts& o, Graph* g) {
  cudaStream_t s = o.stream;
  cudaGetDevice(&g->device);
  g->n = n;
  g->nb = (int)edges.size() - 1;
  g->box_u = box_u;
  g->budget = o.budget;
  g->force_windows = std::max(0, o.force_windows);
  g->edges = edges;
  const int nb = g->nb;
  const int64_t rmax = edges[nb];
  std::vector<int64_t> e2(nb + 1);
  for (int b = 0; b <= nb; ++b) e2[b] = edges[b] * edges[b];
  auto dev_alloc = [&](void** p, size_t bytes, bool pooled = true) -> int {
    if (bytes == 0) bytes = 16;
    // small arrays from the library's pool (ready in the order of the build's
    // stream, which the build synchronises), large ones of their own
    cudaMemPool_t pool = memory_pool();
    cudaError_t e = pool && pooled && bytes <= kPoolKeep / 8
                        ? cudaMallocFromPoolAsync(p, bytes, pool, s)
                        : cudaMalloc(p, bytes);
    if (e != cudaSuccess) {
      cudaGetLastError();
      // give back what the pool keeps, and try again
      if (pool) {
        cudaStreamSynchronize(s);
        cudaMemPoolTrimTo(pool, 0);
      }
      if (cudaMalloc(p, bytes) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return GS_ENOMEM;
      }
    }
    g->device_bytes += (int64_t)bytes;
    return GS_OK;
  };
  // not from the pool: freeing it is how gs_free_graph waits for the device
  int st = dev_alloc((void**)&g->d_edges2, sizeof(int64_t) * (nb + 1), false);
  if (!st) st = dev_alloc((void**)&g->d_xyzp, sizeof(int4) * std::max<int64_t>(n, 1));
  if (!st) st = dev_alloc((void**)&g->d_deg, sizeof(int32_t) * std::max<int64_t>(n, 1));
  if (!st) st = dev_alloc((void**)&g->d_ptr, sizeof(int64_t) * (n + 1));
  if (st) return st;
  cudaMemcpyAsync(g->d_edges2, e2.data(), sizeof(int64_t) * (nb + 1), cudaMemcpyHostToDevice, s);
  if (n == 0) {
    cudaMemsetAsync(g->d_ptr, 0, sizeof(int64_t), s);
    g->h_ptr.assign(1, 0);
    return dev_alloc((void**)&g->d_adj, 16);
  }

  Scratch sc(s);
  int* flags = sc.alloc<int>(8);  // bbox min[3], max[3], err
  if (!flags) return GS_ENOMEM;
  const int init[8] = {INT_MAX, INT_MAX, INT_MAX, INT_MIN, INT_MIN, INT_MIN, 0, 0};
  cudaMemcpyAsync(flags, init, sizeof(init), cudaMemcpyHostToDevice, s);
  { k_check_bbox<<<grid_blocks(n, 256), 256, 0, s>>>(d_xyz, n, box_u, flags, flags + 6); note_launch(); }
  int h[8];
  cudaMemcpyAsync(h, flags, sizeof(h), cudaMemcpyDeviceToHost, s);
  cudaError_t ce = cudaStreamSynchronize(s);
  if (ce != cudaSuccess) return cuda_status(ce);
  if (h[6]) return GS_ERANGE;

  // Cells of side E_nb, split further where they hold enough points to fill a
  // warp's candidate loads: (4, 2, 2) from 32 points a cell on, where the
  // stencil's later half shrinks from 14 to 7.1 E_nb^3 and rows become even,
  // (2, 1, 1) from 8 on.
  GridDesc G;
  G.box = box_u;
  auto grid = [&](int kx, int ky, int kz) {
    const int k[3] = {kx, ky, kz};
    for (int a = 0; a < 3; ++a) {
      G.k[a] = k[a];
      if (box_u) {
        G.nc[a] = (int)std::max<int64_t>(1, std::min<int64_t>(box_u * k[a] / rmax,
                                                              (int64_t)kMaxCellsPerAxis * k[a]));
        G.lo[a] = 0;
        G.width[a] = 0;
      } else {
        const int64_t ext = (int64_t)h[3 + a] - h[a];
        G.lo[a] = h[a];
        G.width[a] = std::max<int64_t>((rmax + k[a] - 1) / k[a],
                                       ext / ((int64_t)kMaxCellsPerAxis * k[a]) + 1);
        G.nc[a] = (int)(ext / G.width[a] + 1);
      }
      g->cells[a] = G.nc[a];
    }
    return (int64_t)G.nc[0] * G.nc[1] * G.nc[2];
  };
  int64_t ncell = grid(1, 1, 1);
  if (n >= 32 * ncell) ncell = grid(4, 2, 2);
  else if (n >= 8 * ncell) ncell = grid(2, 1, 1);

  int32_t* key = sc.alloc<int32_t>(n);
  int32_t* tmp = sc.alloc<int32_t>(n);
  int32_t* start = sc.alloc<int32_t>(ncell + 1);
  int32_t* cursor = sc.alloc<int32_t>(ncell);
  int32_t* cell = sc.alloc<int32_t>(n);
  int64_t* len = sc.alloc<int64_t>(n + 1);
  if (!key || !tmp || !start || !cursor || !cell || !len) return GS_ENOMEM;
  cudaMemsetAsync(start, 0, sizeof(int32_t) * (ncell + 1), s);
  { k_cell_keys<<<grid_blocks(n, 256), 256, 0, s>>>(d_xyz, n, G, key, start); note_launch(); }
  st = scan_exclusive_i32(start, start, ncell + 1, nullptr, s, sc);
  if (st) return st;
  cudaMemcpyAsync(cursor, start, sizeof(int32_t) * ncell, cudaMemcpyDeviceToDevice, s);
  { k_scatter<<<grid_blocks(n, 256), 256, 0, s>>>(key, n, cursor, tmp); note_launch(); }
  { k_rank_in_cell<<<grid_blocks(n, 256), 256, 0, s>>>(key, tmp, n, start, d_xyz, g->d_xyzp, cell); note_launch(); }

  // squared-distance buckets no wider than the narrowest bin
  int bk_shift = 0, bk_n = 0;
  {
    int64_t gap = INT64_MAX;
    for (int b = 0; b < nb; ++b) gap = std::min(gap, e2[b + 1] - e2[b]);
    while (bk_shift < 62 && (int64_t(1) << (bk_shift + 1)) <= gap) ++bk_shift;
    const int64_t nbk = ((e2[nb] - 1) >> bk_shift) + 1;
    if (nbk <= kBucketMax) bk_n = (int)nbk;
  }
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  unsigned long long* tot = sc.alloc<unsigned long long>(3);  // probe words, edges, longest row
  if (!tot) return GS_ENOMEM;
  cudaMemsetAsync(tot, 0, sizeof(unsigned long long) * 3, s);
  auto rows = [&](bool fill, uint32_t* adj, int64_t h0, int64_t h1, int64_t off) {
    const int64_t groups = (h1 - h0 + kRowHubs - 1) / kRowHubs + 1;
    const int blocks = (int)std::min<int64_t>((groups + kRowWarps - 1) / kRowWarps, sms * 16);
    auto kern = fill ? k_rows<true> : k_rows<false>;
    kern<<<blocks, kRowThreads, 0, s>>>(g->d_xyzp, cell, G, start, g->d_edges2, nb, bk_shift, bk_n,
                                        g->d_deg, fill ? g->d_ptr : nullptr, adj, h0, h1, off, tot);
    note_launch();
  };
  KernelTimer timer(o.kernel_ms);
  timer.start(s);
  rows(false, nullptr, 0, n, 0);
  timer.stop(s);
  { k_pad_lengths<<<grid_blocks(n + 1, 256), 256, 0, s>>>(g->d_deg, n, len); note_launch(); }
  st = scan_exclusive_i64(len, g->d_ptr, n + 1, s, sc);
  if (st) return st;
  cudaMemcpyAsync(&g->slots, g->d_ptr + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
  ce = cudaStreamSynchronize(s);
  if (ce != cudaSuccess) return cuda_status(ce);
  const uint64_t edge_bytes = sizeof(uint32_t) * (uint64_t)g->slots;
  const bool out_of_core = o.force_windows > 0 || (o.budget && edge_bytes > o.budget);
  if (!out_of_core) {
    st = dev_alloc((void**)&g->d_adj, edge_bytes);
    if (st) return st;
    timer.start(s);
    rows(true, g->d_adj, 0, n, 0);
    timer.stop(s);
  } else {
    g->h_ptr.resize(n + 1);
    ce = cudaMemcpyAsync(g->h_ptr.data(), g->d_ptr, sizeof(int64_t) * (n + 1),
                         cudaMemcpyDeviceToHost, s);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
    if (ce != cudaSuccess) return cuda_status(ce);
    // Out of core: the edges live in pinned host memory. Rows are filled a
    // chunk of hubs at a time into a device staging buffer and copied out.
    ce = cudaHostAlloc((void**)&g->h_adj, std::max<uint64_t>(edge_bytes, 16), cudaHostAllocDefault);
    if (ce != cudaSuccess) {
      cudaGetLastError();
      g->h_adj = nullptr;
      return GS_ENOMEM;
    }
    int64_t chunk = o.budget ? (int64_t)(o.budget / (2 * sizeof(uint32_t))) : g->slots;
    if (o.force_windows > 0)
      chunk = std::min<int64_t>(chunk, (g->slots + o.force_windows - 1) / o.force_windows);
    chunk = std::max<int64_t>(chunk, 1 << 16);
    const int64_t max_row = [&]() {
      int64_t m = 0;
      for (int64_t i = 0; i < n; ++i) m = std::max<int64_t>(m, g->h_ptr[i + 1] - g->h_ptr[i]);
      return m;
    }();
    chunk = std::max(chunk, max_row);
    uint32_t* stage = sc.alloc<uint32_t>(chunk);
    if (!stage) return GS_ENOMEM;
    for (int64_t h0 = 0; h0 < n;) {
      int64_t h1 = h0;
      while (h1 < n && g->h_ptr[h1 + 1] - g->h_ptr[h0] <= chunk) ++h1;
      const int64_t off = g->h_ptr[h0];
      const int64_t words = g->h_ptr[h1] - off;
      timer.start(s);
      rows(true, stage, h0, h1, off);
      timer.stop(s);
      ce = cudaMemcpyAsync(g->h_adj + off, stage, sizeof(uint32_t) * words, cudaMemcpyDeviceToHost, s);
      if (ce != cudaSuccess) return cuda_status(ce);
      ce = cudaStreamSynchronize(s);  // the staging buffer is reused
      if (ce != cudaSuccess) return cuda_status(ce);
      h0 = h1;
    }
    std::vector<int32_t> hdeg(n);
    cudaMemcpy(hdeg.data(), g->d_deg, sizeof(int32_t) * n, cudaMemcpyDeviceToHost);
    // first id of the last E_nb in x (cells are x-major); open boxes: n
    g->wrap_start = n;
    if (box_u) {
      int32_t ws = 0;
      const int64_t c_last = (int64_t)(G.nc[0] - G.k[0]) * G.nc[1] * G.nc[2];
      cudaMemcpy(&ws, start + c_last, sizeof(int32_t), cudaMemcpyDeviceToHost);
      g->wrap_start = ws;
    }
    g->h_reach.resize(n);
    g->h_far.assign(n, 0);
    for (int64_t i = 0; i < n; ++i) {
      const uint32_t* r = g->h_adj + g->h_ptr[i];
      int d = hdeg[i];
      if (i < g->wrap_start) {  // split off the wrap-around neighbours
        int e = d;
        while (e > 0 && (int64_t)edge_id(r[e - 1]) >= g->wrap_start) --e;
        g->h_far[i] = (e < d) ? 1 : 0;
        d = e;
      }
      g->h_reach[i] = d ? (int32_t)edge_id(r[d - 1]) : (int32_t)i;
    }
    WindowPlan plan;
    st = plan_windows(*g, o, &plan, 0, n);
    if (st) return st;
    g->windows = (int)plan.h0.size();
  }
  unsigned long long ht[3];
  cudaMemcpyAsync(ht, tot, sizeof(ht), cudaMemcpyDeviceToHost, s);
  ce = cudaStreamSynchronize(s);
  if (ce != cudaSuccess) return cuda_status(ce);
  g->probe_words = (int64_t)ht[0];
  g->edges_total = (int64_t)ht[1];
  g->max_deg = (int)(ht[2] & 0xffffffffu);
  timer.publish();
  return cuda_status(cudaGetLastError());
}

namespace {
// walk[i] summed: for each edge (i, j), the words of N+(j) with id <= the
// largest id of N+(i).
__global__ void k_walk_words(const int32_t* __restrict__ deg, const int64_t* __restrict__ ptr,
                             const uint32_t* __restrict__ adj, int64_t adj_off, int64_t split,
                             int64_t adj_off2, int64_t h0, int64_t h1,
                             unsigned long long* total) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  unsigned long long acc = 0;
  for (int64_t i = h0 + blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); i < h1;
       i += warps) {
    const int d = deg[i];
    if (d == 0) continue;
    const uint32_t* r = row_at(adj, ptr, i, adj_off, split, adj_off2);
    const uint32_t hub_hi = edge_id(r[d - 1]);
    for (int k = lane; k < d; k += 32) {
      const uint32_t j = edge_id(r[k]);
      const uint32_t* rj = row_at(adj, ptr, j, adj_off, split, adj_off2);
      int lo = 0, hi = deg[j];
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (edge_id(rj[mid]) <= hub_hi) lo = mid + 1;
        else hi = mid;
      }
      acc += (unsigned long long)lo;
    }
  }
  for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) atomicAdd(total, acc);
}
}  // namespace

namespace {
// Triangles (i < j < k) and the sum over them of |N+(k)|: one warp per hub,
// lanes over the words of each spoke row N+(j); a word k is a triangle when
// a binary search finds it in N+(i).
__global__ void k_tri_words(const int32_t* __restrict__ deg, const int64_t* __restrict__ ptr,
                            const uint32_t* __restrict__ adj, int64_t adj_off, int64_t split,
                            int64_t adj_off2, int64_t h0, int64_t h1, unsigned long long* tri,
                            unsigned long long* words) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  unsigned long long nt = 0, nw = 0;
  for (int64_t i = h0 + blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); i < h1;
       i += warps) {
    const int d = deg[i];
    if (d < 2) continue;
    const uint32_t* r = row_at(adj, ptr, i, adj_off, split, adj_off2);
    for (int s = 0; s + 1 < d; ++s) {
      const uint32_t j = edge_id(r[s]);
      const uint32_t* rj = row_at(adj, ptr, j, adj_off, split, adj_off2);
      const int dj = deg[j];
      for (int t = lane; t < dj; t += 32) {
        const uint32_t k = edge_id(rj[t]);
        int lo = s + 1, hi = d;  // k > j, so only the hub row after j
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (edge_id(r[mid]) < k) lo = mid + 1;
          else hi = mid;
        }
        if (lo < d && edge_id(r[lo]) == k) {
          nt += 1;
          nw += (unsigned long long)deg[k];
        }
      }
    }
  }
  for (int o = 16; o; o >>= 1) {
    nt += __shfl_xor_sync(0xffffffffu, nt, o);
    nw += __shfl_xor_sync(0xffffffffu, nw, o);
  }
  if (lane == 0) {
    atomicAdd(tri, nt);
    atomicAdd(words, nw);
  }
}
}  // namespace

int tri_words_device(const Graph& g, int64_t* tri, int64_t* words) {
  *tri = *words = 0;
  if (g.n == 0 || g.slots == 0) return GS_OK;
  Opts o;
  Scratch sc(o.stream);
  unsigned long long* tot = sc.alloc<unsigned long long>(2);
  if (!tot) return GS_ENOMEM;
  cudaMemsetAsync(tot, 0, 2 * sizeof(unsigned long long), o.stream);
  int st = for_each_window(g, o, sc, [&](const WinView& v) -> int {
    { k_tri_words<<<grid_blocks((v.h1 - v.h0) * 32, 256), 256, 0, o.stream>>>(
        g.d_deg, g.d_ptr, v.adj, v.off1, v.split, v.off2, v.h0, v.h1, tot, tot + 1); note_launch(); }
    return cuda_status(cudaGetLastError());
  });
  if (st) return st;
  unsigned long long h[2] = {0, 0};
  cudaMemcpyAsync(h, tot, sizeof(h), cudaMemcpyDeviceToHost, o.stream);
  cudaError_t e = cudaStreamSynchronize(o.stream);
  if (e != cudaSuccess) return cuda_status(e);
  *tri = (int64_t)h[0];
  *words = (int64_t)h[1];
  return GS_OK;
}

int walk_words_device(Graph* g) {
  if (g->n == 0 || g->slots == 0) {
    g->walk_words = 0;
    return GS_OK;
  }
  Opts o;
  Scratch sc(o.stream);
  unsigned long long* tot = sc.alloc<unsigned long long>(1);
  if (!tot) return GS_ENOMEM;
  cudaMemsetAsync(tot, 0, sizeof(unsigned long long), o.stream);
  int st = for_each_window(*g, o, sc, [&](const WinView& v) -> int {
    { k_walk_words<<<grid_blocks((v.h1 - v.h0) * 32, 256), 256, 0, o.stream>>>(
        g->d_deg, g->d_ptr, v.adj, v.off1, v.split, v.off2, v.h0, v.h1, tot); note_launch(); }
    return cuda_status(cudaGetLastError());
  });
  if (st) return st;
  unsigned long long h = 0;
  cudaMemcpyAsync(&h, tot, sizeof(h), cudaMemcpyDeviceToHost, o.stream);
  cudaError_t e = cudaStreamSynchronize(o.stream);
  if (e != cudaSuccess) return cuda_status(e);
  g->walk_words = (int64_t)h;
  return GS_OK;
}

namespace {
std::mutex g_host_mu;

template <class T>
int host_copy_of(std::vector<T>& kept, const T* src, size_t count, cudaStream_t s, const T** out) {
  return host_copy(g_host_mu, kept, count, [&](T* dst) {
    const cudaError_t e =
        cudaMemcpyAsync(dst, src, sizeof(T) * count, cudaMemcpyDeviceToHost, s);
    const cudaError_t e2 = cudaStreamSynchronize(s);  // nothing may write to dst later
    if (e != cudaSuccess || e2 != cudaSuccess) cudaGetLastError();
    return cuda_status(e != cudaSuccess ? e : e2);
  }, out);
}
}  // namespace

int host_ptr(const Graph& g, cudaStream_t s, const int64_t** out) {
  return host_copy_of(g.h_ptr, g.d_ptr, (size_t)g.n + 1, s, out);
}
int host_deg(const Graph& g, cudaStream_t s, const int32_t** out) {
  return host_copy_of(g.h_deg, g.d_deg, (size_t)g.n, s, out);
}

int shard_range(const Graph& g, const Opts& o, int64_t* lo, int64_t* hi) {
  *lo = 0;
  *hi = g.n;
  if (o.shards <= 1 || g.n == 0) return GS_OK;
  // boundaries at equal shares of the edge words (row starts do not decrease)
  const int64_t* P = nullptr;
  const int st = host_ptr(g, o.stream, &P);
  if (st) return st;
  const int64_t total = P[g.n];
  auto bound = [&](int k) -> int64_t {
    if (k <= 0) return 0;
    if (k >= o.shards) return g.n;
    const int64_t target = (int64_t)((__int128)total * k / o.shards);
    return std::lower_bound(P, P + g.n, target) - P;
  };
  *lo = bound(o.shard);
  *hi = bound(o.shard + 1);
  return GS_OK;
}

int plan_windows(const Graph& g, const Opts& o, WindowPlan* plan, int64_t lo, int64_t hi) {
  const std::vector<int64_t>& P = g.h_ptr;
  const int64_t n = g.n, ws = g.wrap_start;
  const int64_t far_words = P[n] - P[ws];
  // a query without its own budget / window count uses the graph's
  const uint64_t budget = o.budget ? o.budget : g.budget;
  const int force = o.force_windows > 0 ? o.force_windows : g.force_windows;
  const int64_t cap = budget ? (int64_t)(budget / (2 * sizeof(uint32_t))) : INT64_MAX;
  const int64_t target = force > 0 ? (P[hi] - P[lo] + force - 1) / force : INT64_MAX;
  // words a window [h0, h1) with near reach r and far flag f needs
  auto need = [&](int64_t h0, int64_t r, bool f) -> int64_t {
    if (f && r >= ws) return P[n] - P[h0];  // the two ranges touch: one range
    return (P[r] - P[h0]) + (f ? far_words : 0);
  };
  plan->h0.clear();
  plan->h1.clear();
  plan->r1.clear();
  plan->far.clear();
  plan->max_words = 0;
  int64_t h0 = lo;
  while (h0 < hi) {
    int64_t h1 = h0, reach = h0 + 1;
    bool far = false;
    while (h1 < hi) {
      const int64_t nr =
          std::max<int64_t>(std::max<int64_t>(reach, (int64_t)g.h_reach[h1] + 1), h1 + 1);
      const bool nf = far || g.h_far[h1];
      const int64_t own = P[h1 + 1] - P[h0];
      if (h1 > h0 && (own > target || need(h0, nr, nf) > cap)) break;
      reach = nr;
      far = nf;
      ++h1;
    }
    const int64_t words = need(h0, reach, far);
    if (words > cap) return GS_ENOMEM;  // one hub's rows exceed a window buffer
    if (far && reach >= ws) {
      reach = n;
      far = false;
    }
    plan->h0.push_back(h0);
    plan->h1.push_back(h1);
    plan->r1.push_back(reach);
    plan->far.push_back(far ? 1 : 0);
    plan->max_words = std::max(plan->max_words, words);
    h0 = h1;
  }
  return GS_OK;
}

}  // namespace gs
