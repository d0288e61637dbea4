// Pieces of the tiled pair kernels (3pCF counts, mu-binned 3pCF): a hub's row
// dealt into tiles of at most 32 neighbours, single-precision distances with
// exact decisions near bin edges. See k_count3t for the scheme.
#pragma once

#include <cmath>
#include <vector>

#include "gs_internal.cuh"

namespace gs {

constexpr int kTThreads = 512;  // two CTAs per SM
constexpr int kTWarps = kTThreads / 32;
// Rows above this are left to the walk and pair kernels: C(8192, 2) < 2^25
// pairs per hub keep the shared counters below 2^31 between flushes.
constexpr int kTMaxDeg = 8192;
// Absent j's and k's stand at these x (in units): farther from every point,
// and from one another, than twice the largest E_nb (2^19).
constexpr float kFarJ = 4.0e6f, kFarK = -4.0e6f;

__device__ inline unsigned long long t_pack(float x, float y) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ inline void t_unpack(unsigned long long v, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
}
__device__ inline unsigned long long t_add(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ inline unsigned long long t_mul(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ inline unsigned long long t_fma(unsigned long long a, unsigned long long b,
                                           unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ inline float t_sqrt(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Relative error below 2^-22; |x| below 2^-126 counts as zero.
__device__ inline float t_rsqrt(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// u of a pair in bin b lies in [kTileM + b, kTileM + b + 1): 16 fraction bits.
constexpr float kTileM = 192.0f;
constexpr uint32_t kTileBits = 0x43400000u;  // bits of kTileM
constexpr int kTileMaxBins = 62;             // kTileM + nb + 1 below 256

// The bin that u says, nb when none, plus kBin0 (taken off in the cells' base
// address). LOWER: u may lie below kTileM.
template <bool LOWER>
constexpr uint32_t kBin0 = LOWER ? 0u : kTileBits >> 16;
template <bool LOWER>
__device__ inline uint32_t t_bin(float u, int nb) {
  const uint32_t bits = __float_as_uint(u);
  return min((LOWER ? bits - kTileBits : bits) >> 16, kBin0<LOWER> + (uint32_t)nb);
}

__device__ inline void t_red(uint32_t addr, uint32_t v) {
  asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ inline uint32_t t_atom(uint32_t addr, uint32_t v) {
  uint32_t old;
  asm volatile("atom.shared.add.u32 %0, [%1], %2;" : "=r"(old) : "r"(addr), "r"(v) : "memory");
  return old;
}

// Staged neighbours of one hub, one array per quantity: x, y, z (float);
// unweighted: p = b nb rows, q = b rows of nb + 1 cells; weighted: p =
// b (b + 1) / 2 rows, q = b rows, W. p and q as byte offsets of 32-bit cells.
struct Stage {
  float *x, *y, *z;
  int *p, *q, *W;
};
__host__ __device__ inline size_t stage_bytes(int64_t cap, bool weighted) {
  return (size_t)cap * (weighted ? 24 : 20);
}
__device__ inline Stage stage_at(unsigned char* b, int64_t cap) {
  Stage s;
  s.x = reinterpret_cast<float*>(b);
  s.y = s.x + cap;
  s.z = s.y + cap;
  s.p = reinterpret_cast<int*>(s.z + cap);
  s.q = s.p + cap;
  s.W = s.q + cap;
  return s;
}

// Minimum-image difference q - p of coordinates.
__device__ inline int t_min_image(int q, int p, int64_t box) {
  int64_t d = (int64_t)q - p;
  if (box) {
    if (2 * d >= box) d -= box;
    else if (2 * d < -box) d += box;
  }
  return (int)d;
}

// Global staging of `each` bytes per CTA for rows beyond the shared one, with
// as many CTAs of *grid as there is memory for (nullptr: not even one). Last of
// a call's allocations: it may leave nothing for others.
inline unsigned char* staging(Scratch& sc, size_t each, int* grid) {
  for (;; *grid = (*grid + 1) / 2) {
    unsigned char* p = sc.alloc<unsigned char>(each * *grid);
    if (p || *grid <= 1) return p;
  }
}

// Exact bin of a pair from its displacement (integers held in floats), nb
// when it is no edge.
__device__ inline int t_exact_bin(const int64_t* e2, int nb, float dx, float dy, float dz) {
  const long long x = (long long)(int)dx, y = (long long)(int)dy, z = (long long)(int)dz;
  const long long D2 = x * x + y * y + z * z;
  if (D2 < e2[0] || D2 >= e2[nb]) return nb;
  int b = 0, e = nb;
  while (e - b > 1) {
    const int mid = (b + e) >> 1;
    if (e2[mid] <= D2) b = mid;
    else e = mid;
  }
  return b;
}

// Binning constants for evenly spaced bins; ok = false when they are not (to
// within 1/128 of their width: edges rounded to the lattice are).
struct TileBins {
  bool ok = false;
  float c = 0.f, m = 0.f;  // u = sqrt(D2) c + m
  uint32_t amb = 0;        // ambiguous iff the low 16 bits of u are <= amb
  bool lower = false;      // bins start above zero
};
inline TileBins tile_bins(const std::vector<int64_t>& edges) {
  TileBins t;
  const int nb = (int)edges.size() - 1;
  if (nb > kTileMaxBins) return t;
  const double w = (double)(edges[nb] - edges[0]) / nb;
  double dev = 0.0;  // edges off the even spacing, in bin widths
  for (int b = 0; b <= nb; ++b)
    dev = std::max(dev, std::fabs((double)(edges[b] - edges[0]) / w - b));
  // D = sqrt(D2): relative error below 0.75 2^-21 from the squared distance
  // (three roundings, halved), the approximate square root (2^-23) and c
  // (2^-24), at most E_nb / w bin widths; m's rounding; half a unit for u
  const double off = (double)edges[0] / w, one = 65536.0;
  const double err = (double)edges[nb] / w * std::ldexp(0.75, -21) + dev +
                     std::max(kTileM + 1.0, off) * std::ldexp(1.0, -24);
  if (err > 1.0 / 128) return t;
  const int delta = (int)std::ceil(err * one + 0.75);
  t.c = (float)(1.0 / w);
  t.m = (float)(kTileM + delta / one - off);
  t.amb = 2u * (uint32_t)delta;
  t.lower = edges[0] > 0;
  t.ok = true;
  return t;
}

}  // namespace gs
