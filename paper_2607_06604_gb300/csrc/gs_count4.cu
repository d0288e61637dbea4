// Binned tetrahedron counts (Sec. 2.2) and the parity-decomposed channels
// (Sec. 3.2, Eq. volume), GB300 layout.
//
// A tetrahedron i < a < b < c is counted at its smallest vertex i. The m
// neighbours N+(i) of a hub are taken in any order that suits the kernel
// (the orbit and the volume's sign follow the labels, whatever they are):
// sorted by the hub edge's bin, or, for the pixelised parity, by caller
// index. A group of warps (a whole CTA down to one warp, by the size of the
// rows) takes one hub at a time and
//   1. stages the minimum-image displacement of every neighbour from i;
//   2. fills the triangular byte matrix B of the bins of all pairs of
//      neighbours (nb: no edge) from the staged displacements;
//   3. takes rows a: the columns of row a that are edges form a list L, and
//      every pair (b, c) of L with B(b, c) an edge is a tetrahedron. The b's
//      go through a shared chunk of 32 entries that holds what depends on
//      (i, a, b) only (the cross product d_a x d_b and the table row of the
//      bins b_01, b_02, b_12); the c's sit in the lanes, 32 at a time, with
//      what depends on (i, a, c) in registers. A step of the inner loop
//      therefore costs one broadcast, one byte of B per lane (32 near
//      bytes), one table entry, three multiply-adds and one histogram update.
// This is the three-way walk of Eq. (threeway) with the second and third
// lists intersected through B (the paper's per-hub connectivity matrix,
// Sec. 3.5.2, holding bins instead of bits).
//
// A table maps the raw bin tuple to its S4 orbit, the parity of one
// relabelling onto the orbit representative and the orbit's chirality. The
// volume V = (d_a x d_b) . d_c is formed in single precision; within its
// error bound of zero, exactly in integers. Counts use per-CTA
// shared-memory histograms flushed with 64-bit atomics, one cell per orbit
// and sign of V: even = V > 0 plus V < 0, odd = their difference (chiral
// orbits), so a tetrahedron updates one cell; those with V = 0 go to the two
// cells in turn (see take_turn). Hubs with more neighbours than the shared
// workspace holds run with their workspace in global scratch.
//
// What bounds it: the shared-memory pipe (90% of its wavefronts; 71% of issue
// slots, 24 instructions per step of 14 tetrahedra). Measured on one GB300
// against a kernel that queued (b, c) pairs per warp and gave every lane one of
// them (7.5 instructions and two random 16-byte loads per tetrahedron): parity
// on 2e5 clustered points (8.4e10 tetrahedra) 648 -> 171 ms, pixelised parity on
// 1e5 (4.2e10) 810 -> 140 ms, connected 4pCF of 5e4 + 5e4 points 520 -> 254 ms,
// 1e5 points with rows of 26 (mock, build included) 8.5 -> 1.83 ms.
//
// When the per-orbit counters of every orbit do not fit in shared memory
// beside the hub workspace (unweighted: many bins; weighted: see below),
// shared memory holds the `hot` orbits only: the orbit tables are relabelled
// so that the orbits met most often in a sample of hubs come first, and a
// tetrahedron of any other orbit goes to the global counters directly.
//
// Weighted sums (exact, fixed-point W): the hub's sums of x = W_a W_b W_c are
// kept per cell in three 32-bit words, one array per word (cells of 16 bytes in
// a row left an atomic eight of the 32 banks: 4.3 wavefronts each), and
// multiplied by W_i into the global sums when the hub ends (into limbs, see
// record_limbs, where the hub is small enough, else 192-bit sums); the rare
// carry out of the top word goes there at once. Shared memory holds the words
// (and the counts) only for the `hot` orbits, as above; a tetrahedron of any
// other orbit goes to the limbs with its full product. Volumes of zero have
// cells of their own where a sample finds many of them (ZERO). Pairs that are no
// edge update words of the lane's own bank.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>
#include <type_traits>

#include "gs_internal.cuh"
#include "gs_tiles.cuh"

namespace gs {
namespace {

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxSmemRow = 512;
// A hub's tetrahedra (at most C(m, 3)) may go to the shared counters when
// they are at most this many (m <= 738).
constexpr unsigned long long kMaxHubNeed = 1ull << 26;
// Squared-distance buckets for the bin lookup: bucket k covers
// [k 2^shift, (k + 1) 2^shift) with 2^shift no wider than the narrowest bin
// in squared distance, so a bucket holds at most one bin edge.
constexpr int kBucketMax = 2048;
// A pixel volume at or below this is degenerate: over all pixel triples the
// exact value is zero or above 5e-5 in magnitude, and the single-precision
// value (six products of components of unit vectors, each rounded) is
// within 2e-6 of it.
constexpr float kPixZero = 2e-5f;

struct Args {
  const int64_t* __restrict__ ptr;
  const int32_t* __restrict__ deg;
  const uint32_t* __restrict__ adj;  // row i at row_at(adj, ptr, i, adj_off, split, adj_off2)
  int64_t adj_off, split, adj_off2;
  // hubs: list[0..nlist), or hub_begin + k hub_stride below hub_end with at
  // most dmax neighbours (list = nullptr)
  int64_t hub_begin, hub_end, hub_stride;
  const int64_t* __restrict__ list;
  int64_t nlist;
  int dmax;
  const int4* __restrict__ xyzp;
  const int64_t* __restrict__ e2g;
  const void* __restrict__ ent;      // orbit table (see Ent)
  const uint8_t* __restrict__ chir;  // chirality per slot (parity)
  int64_t box;
  int nb, tab3;  // bins; table entries per (b_01, b_02, b_12): nb^2 (nb + 1)
  int cap;   // shared-memory workspace capacity (neighbours) of a group
  int gcap;  // global workspace capacity
  int group; // warps per group
  int bk_shift, bk_n;  // squared-distance buckets (bk_n = 0: binary search)
  int hot;             // orbits (slots) below this are accumulated in shared memory
  int even_hot;        // weighted parity, ZERO: slots below this have an even-only cell too
  float eps;           // volumes within eps of zero are decided in integers
  unsigned long long limit;  // tetrahedra between two flushes of the shared counters
  unsigned long long* even;
  unsigned long long* odd;
  unsigned long long* weven;  // [n_orbits][3] 192-bit
  unsigned long long* wodd;
  unsigned long long* limbs;  // weighted: see record_limbs
  uint32_t even_limbs;        // its first cell of the even channel alone
  int long_rows;              // see record_sum
  unsigned long long limb_need;  // tetrahedra of a hub whose sums times W_i fit the limbs
  const int64_t* __restrict__ W;
  const float4* __restrict__ pixu;  // pixelised parity: unit vectors of the pixel centres
  unsigned long long* hub_counter;
  unsigned char* gscratch;  // per-CTA global workspace
  size_t gscratch_stride;
};

// Table entries: twice the slot, plus 1 when the relabelling onto the
// representative of a chiral orbit is odd; the top bit marks chiral orbits.
// Two bytes when the slots fit 14 bits (nb <= 8): half the lines per gather.
// The last digit (b_23) has one value more, no edge, whose entries say slot
// n_orbits: the counters have a cell for it, so that updates need no predicate
// (a predicated shared atomic is compiled to a branch, four instructions).
template <class E>
struct Ent {
  static constexpr int kTop = sizeof(E) * 8 - 1;
  static constexpr uint32_t kMask = (1u << kTop) - 1u;
};

// A table entry, sign-extended (the chirality bit fills the top).
__device__ inline int load_entry(const uint16_t* p) {
  int v;
  asm("ld.global.nc.s16 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
__device__ inline int load_entry(const uint32_t* p) { return (int)__ldg(p); }

__device__ inline int64_t mi(int64_t d, int64_t box) {
  if (box) {
    if (2 * d >= box) d -= box;
    else if (2 * d < -box) d += box;
  }
  return d;
}

// Largest b with e2[b] <= D2 (the caller knows D2 is an edge): the bucket
// of D2 gives the bin of the bucket's start, and one comparison with the
// next edge finishes it; without buckets, a binary search.
template <class T>
__device__ inline int bin_of(T D2, const T* e2, int nb, const uint8_t* bk, int shift) {
  if (bk) {
    const int b = bk[(uint64_t)D2 >> shift];
    return b + (D2 >= e2[b + 1] ? 1 : 0);
  }
  int lo = 0, hi = nb;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (e2[mid] <= D2) lo = mid;
    else hi = mid;
  }
  return lo;
}

// det[da, db, dc] exactly (components below 2^19: the sum is below 2^60).
__device__ inline long long det3(const int4& da, const int4& db, const int4& dc) {
  return (long long)da.x * ((long long)db.y * dc.z - (long long)db.z * dc.y) -
         (long long)da.y * ((long long)db.x * dc.z - (long long)db.z * dc.x) +
         (long long)da.z * ((long long)db.x * dc.y - (long long)db.y * dc.x);
}

// Direction pixel of the pixelised parity channel (Sec. 3.2 stores one
// pixel byte per spoke and treats |V| < 1e-9 as degenerate; the scheme is
// fixed here as 256 equal-area pixels): 16 bands of width 1/8 in
// cos(theta) = z / |d| (a direction on a band edge belongs to the band
// above it) times 16 sectors of pi / 8 in phi = atan2(y, x) in [0, 2 pi)
// (an edge belongs to the sector above it; sector 0 on the z axis); pixel =
// 16 band + sector. Everything is decided with exact 64-bit integer
// comparisons: z / |d| against s / 8 through 64 z^2 against s^2 |d|^2, and
// phi within its quadrant against pi/8, pi/4, 3pi/8 through tan(pi/8) =
// sqrt(2) - 1 and tan(3pi/8) = sqrt(2) + 1 squared out.
__host__ __device__ inline int dir_pixel(int64_t x, int64_t y, int64_t z) {
  // band = 8 + floor(8 z / |d|), at most 15. On the device t = 8 z / |d| is
  // first formed in single precision (relative error below 8 2^-24 from the
  // conversions, products, sums and the reciprocal square root's 2 ulp, so
  // below 2^-18 absolutely): at least 2^-10 from every integer, its floor is
  // exact; otherwise (and for d = 0) the integer comparisons decide.
  int band = -1;
#ifdef __CUDA_ARCH__
  {
    // the components fit 32 bits (displacements below 2^20): 32-bit
    // conversions, not the FP64 pipe's 64-bit ones
    const float fx = (float)(int)x, fy = (float)(int)y, fz = (float)(int)z;
    const float t = 8.0f * fz * rsqrtf(fx * fx + fy * fy + fz * fz);
    if (fabsf(t - rintf(t)) >= 0.0009765625f) {
      const int f = 8 + (int)floorf(t);
      band = f < 0 ? 0 : (f > 15 ? 15 : f);
    }
  }
#endif
  if (band < 0) {
    const int64_t n2 = x * x + y * y + z * z, z64 = 64 * z * z;
    band = z >= 0 ? 8 : 0;
    for (int s = 1; s <= 7; ++s) {
      const int64_t edge = (int64_t)(s * s) * n2;
      // z >= 0: edges s/8 at or below z/|d|; z < 0: edges -s/8 at or below it
      band += (z >= 0 ? (z64 >= edge) : (z64 <= edge)) ? 1 : 0;
    }
  }
  int sector = 0;
  if (x != 0 || y != 0) {
    // turn by -pi/2 until the direction lies in [0, pi/2): a > 0, b >= 0
    int quarter;
    int64_t a, b;
    if (x > 0 && y >= 0) {
      quarter = 0, a = x, b = y;
    } else if (x <= 0 && y > 0) {
      quarter = 1, a = y, b = -x;
    } else if (x < 0 && y <= 0) {
      quarter = 2, a = -x, b = -y;
    } else {
      quarter = 3, a = -y, b = x;
    }
    // phi >= pi/8 iff b >= (sqrt 2 - 1) a, phi >= 3 pi/8 iff b >= (sqrt 2 + 1) a
    // (never equal for integers, a > 0); on the device b - k a is formed in
    // single precision (a, b below 2^21: error below 1/2) and decides when
    // at least 1 from zero; otherwise, and on the host, the squared integer
    // forms decide
    int e1 = -1, e3 = -1;
#ifdef __CUDA_ARCH__
    if (a < (int64_t(1) << 21) && b < (int64_t(1) << 21)) {
      const float fa = (float)(int)a, fb = (float)(int)b;
      const float g1 = fmaf(-0.41421356237f, fa, fb), g3 = fmaf(-2.41421356237f, fa, fb);
      if (fabsf(g1) >= 1.0f) e1 = g1 > 0.0f ? 1 : 0;
      if (fabsf(g3) >= 1.0f) e3 = g3 > 0.0f ? 1 : 0;
    }
#endif
    const int64_t a2 = 2 * a * a;
    if (e1 < 0) e1 = ((a + b) * (a + b) >= a2) ? 1 : 0;
    if (e3 < 0) e3 = (b > a && (b - a) * (b - a) >= a2) ? 1 : 0;
    sector = 4 * quarter + e1 + (b >= a ? 1 : 0) + e3;
  }
  return 16 * band + sector;
}

// A 192-bit two's complement value into three global 64-bit words.
__device__ inline void atomic_add_w192(unsigned long long* g, unsigned long long w0,
                                       unsigned long long w1, unsigned long long w2) {
  const unsigned long long o0 = atomicAdd(g, w0);
  const unsigned long long c0 = (o0 + w0 < o0) ? 1ull : 0ull;
  const unsigned long long s1 = w1 + c0;
  const unsigned long long c1a = (s1 < w1) ? 1ull : 0ull;  // w1 = 2^64 - 1 and a carry
  unsigned long long c1b = 0;
  if (s1) {
    const unsigned long long o1 = atomicAdd(g + 1, s1);
    c1b = (o1 + s1 < o1) ? 1ull : 0ull;
  }
  const unsigned long long s2 = w2 + c1a + c1b;
  if (s2) atomicAdd(g + 2, s2);
}

// S * Wi into a global 192-bit sum: S a signed 128-bit hub sum (lo, hi),
// |Wi| < 2^63.
__device__ inline void fold_i128(unsigned long long* g, unsigned long long lo,
                                 unsigned long long hi, long long Wi) {
  const bool sn = (long long)hi < 0, wn = Wi < 0;
  if (sn) {
    lo = ~lo + 1ull;
    hi = ~hi + (lo == 0ull ? 1ull : 0ull);
  }
  const unsigned long long v = wn ? (unsigned long long)(-Wi) : (unsigned long long)Wi;
  unsigned long long p0 = lo * v;
  const unsigned long long t = __umul64hi(lo, v);
  unsigned long long p1 = hi * v + t;
  unsigned long long p2 = __umul64hi(hi, v) + (p1 < t ? 1ull : 0ull);
  if (sn != wn) {
    p0 = ~p0 + 1ull;
    unsigned long long c = p0 == 0ull ? 1ull : 0ull;
    p1 = ~p1 + c;
    c = (c && p1 == 0ull) ? 1ull : 0ull;
    p2 = ~p2 + c;
  }
  atomic_add_w192(g, p0, p1, p2);
}

// A hub's workspace. DISP etc. per neighbour, B the strictly upper triangle
// of bins by rows (entry (b, c), c > b, at row_off(b, m + 1) + c; nb: no edge,
// as all of column m, which unused lanes read), and per warp the list of row
// a's edges.
template <class L>
struct Workspace {
  int4* disp;     // displacement from the hub, bin of the hub edge
  int* wv;        // weight (weighted sums)
  int* cid;       // caller index (pixelised parity, while sorting)
  uint8_t* hpix;  // pixel of the spoke from the hub (pixelised parity)
  uint8_t* B;
  L* list;        // per warp: cap entries
  uint8_t* lpix;  // per warp: pixels of the spokes from a (pixelised parity)
  int cap;
};

__host__ __device__ inline size_t pad16(size_t x) { return (x + 15) & ~(size_t)15; }

// Bytes of one group's workspace; list entries of lsize bytes.
__host__ __device__ inline size_t workspace_bytes(int64_t cap, int group, int lsize, bool weighted,
                                                  bool pix) {
  const size_t c = (size_t)cap;
  return (c + 1) * 16 + (weighted ? pad16(c * 4) : 0) + (pix ? pad16(c * 4) + pad16(c) : 0) +
         pad16(c * (c + 1) / 2 + 1) + pad16((size_t)group * c * lsize) +
         (pix ? pad16((size_t)group * c) : 0);
}

template <class L>
__device__ inline Workspace<L> carve(unsigned char* p, int64_t cap, int group, bool weighted,
                                     bool pix) {
  const size_t c = (size_t)cap;
  Workspace<L> w;
  w.disp = reinterpret_cast<int4*>(p);
  p += (c + 1) * 16;
  w.wv = reinterpret_cast<int*>(p);
  if (weighted) p += pad16(c * 4);
  w.cid = reinterpret_cast<int*>(p);
  if (pix) p += pad16(c * 4);
  w.hpix = p;
  if (pix) p += pad16(c);
  w.B = p;
  p += pad16(c * (c + 1) / 2 + 1);
  w.list = reinterpret_cast<L*>(p);
  p += pad16((size_t)group * c * sizeof(L));
  w.lpix = p;
  w.cap = (int)cap;
  return w;
}

// Row b of a triangle of side m starts so that entry (b, c) is at row_off + c.
template <class I>
__device__ inline I row_off(I b, I m) {
  return b * (2 * m - b - 1) / 2 - b;
}

// Barrier of one group: named barrier 1 + g (groups of two warps and more
// than 15 groups are not used), a warp barrier for a single warp.
__device__ inline void group_sync(int g, int threads) {
  if (threads == 32) __syncwarp();
  else asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(threads) : "memory");
}

// Per-CTA shared state beside the histograms and workspaces.
struct Shared {
  int64_t e2[kMaxBins4 + 1];
  uint8_t bk[kBucketMax];
  int64_t hub[kWarps];            // per group
  int row[kWarps];                // per group: next row a
  int flush[kWarps];
  int cur[kWarps * kMaxBins4];    // per group: counting sort by bin
  unsigned long long pending;     // tetrahedra the shared counters may hold
};

// Adds 1 to a counter at a shared address.
__device__ inline void inc_shared(uint32_t addr) {
  asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(addr) : "memory");
}

// Pairs of floats in one 64-bit register (low half first); each half is
// rounded as the scalar operation.
__device__ inline unsigned long long pack2(float x, float y) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ inline void unpack2(unsigned long long v, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
}
__device__ inline unsigned long long mul2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ inline unsigned long long fma2(unsigned long long a, unsigned long long b,
                                          unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// What a warp keeps of 32 b's of its row a: the cross product d_a x d_b (or
// of the pixel vectors), the row of B (GW: b itself) and the table row of
// (b_01, b_02, b_12). Arrays, so that one 128-bit broadcast serves four steps.
struct Chunk {
  float nx[32], ny[32], nz[32];
  int row[32];
  uint32_t tab[32];
};

// The counters of one CTA: cells of the slots below a.hot (parity: two per
// slot; ZERO: then one per slot below a.even_hot for what counts in the even
// channel only, V = 0 and achiral orbits), then a word per lane for no edge.
// Weighted: three more arrays, `stride`
// words apart, the low to high words of the hub's sums.
struct Hist {
  unsigned* cnt;
  uint32_t stride;
};
// The top word starts at half its range, so that sums of either sign stay clear
// of its carry (from zero, every change of a sum's sign carried: 2.5 ms of
// global atomics per 1e9 tetrahedra).
constexpr uint32_t kTopZero = 0x80000000u;
__host__ __device__ inline size_t hist_words(int64_t cells) { return (size_t)cells + 32; }

// The cell that the next V = 0 of a chiral orbit goes to, unweighted: the two
// cells of the orbit in turn, which leaves their difference alone, but for one
// when the number of them is odd. The top bit of the first cell says whose turn
// it is, and that much is taken off when the cells are emptied: every +1 there
// stands for one more such tetrahedron in the first cell than in the second,
// whichever flush takes which. (Global atomics for V = 0 cost planar catalogues
// more than all else: 2e4 points in a plane, 1.5e10 tetrahedra, 214 ms against
// 92.)
constexpr uint32_t kTurn = 0x80000000u;
__device__ inline uint32_t take_turn(const Hist& h, uint32_t slot) {
  return 2u * slot + (atomicXor(h.cnt + 2u * slot, kTurn) >> 31);
}

// One tetrahedron straight to the global counts. cell: twice the slot plus the
// sign (parity) or the slot; odd: of the odd channel too.
template <bool PARITY>
__device__ inline void record_global(const Args& a, uint32_t cell, bool odd) {
  const uint32_t slot = PARITY ? cell >> 1 : cell;
  atomicAdd(a.even + slot, 1ull);
  if (PARITY && odd) atomicAdd(a.odd + slot, (cell & 1u) ? ~0ull : 1ull);
}

// A weighted one, by cell (parity: 2 n_orbits + slot for the even channel alone):
// the count and the product (W_a W_b)(W_i W_c), below 2^120, in limbs of 25 bits
// (the top one is zero for weights within a factor of two), each to a word of its
// own. Nothing waits for a returned value, as carries
// between words would, and the two channels are told apart at the end (k_limbs):
// with few lanes of a warp at it, the round trips of 192-bit sums in both channels
// were the whole time (rows of 30, nb = 12, where few orbits have shared cells:
// 42 -> 15.7 ms).
constexpr int kLimbs = 5, kLimbBits = 25, kLimbWords = 1 + kLimbs;
// Additions that a word may take between two passes of k_limbs (it holds twice as
// many): launches are split to stay below.
constexpr double kLimbAdds = 274877906944.0;  // 2^38
__device__ inline void add_limbs(unsigned long long* L, long long lo, long long hi) {
#pragma unroll
  for (int k = 0; k < kLimbs; ++k) {
    // the lowest limb left; the top one keeps the sign
    const unsigned long long x = k + 1 < kLimbs
                                     ? (unsigned long long)lo & ((1ull << kLimbBits) - 1ull)
                                     : (unsigned long long)lo;
    if (x) atomicAdd(L + 1 + k, x);
    lo = (long long)(((unsigned long long)lo >> kLimbBits) |
                     ((unsigned long long)hi << (64 - kLimbBits)));
    hi >>= kLimbBits;
  }
}
__device__ inline void record_limbs(unsigned long long* limbs, uint32_t cell, int64_t Wi,
                                    int64_t Wab, int Wc) {
  unsigned long long* L = limbs + (size_t)cell * kLimbWords;
  long long lo, hi;
  mul_i128(Wab, Wi * (int64_t)Wc, &lo, &hi);
  atomicAdd(L, 1ull);
  add_limbs(L, lo, hi);
}

// The same straight to the count and the 192-bit sum of a slot, without parity:
// half the atomics, but each waits for the carry of the one before. Better where
// rows are long and more lanes have one (3e4 points, rows of 200, nb = 12: 339 ms
// against 373 to 411; rows of 30: 22 against 12.8).
__device__ inline void record_sum(const Args& a, uint32_t slot, int64_t Wi, int64_t Wab, int Wc) {
  long long lo, hi;
  atomicAdd(a.even + slot, 1ull);
  mul_i128(Wab, Wi * (int64_t)Wc, &lo, &hi);
  atomic_add_i192(a.weven + 3 * (size_t)slot, (unsigned long long)lo, (unsigned long long)hi);
}

// Two weighted tetrahedra with products Wc V[] in the cells at[] (shared
// addresses of their counts, `none` for the lane's unused words); cell[] for the
// carries out of the top word (about one in 2^21 for weights within a factor of
// two).
template <bool PARITY, bool ZERO>
__device__ inline void record_weighted(const Args& a, const uint32_t (&at)[2],
                                       const uint32_t (&cell)[2], uint32_t none, uint32_t stride,
                                       int64_t Wi, int Wc, const long long (&V)[2]) {
  uint32_t w0[2], w1[2], w2[2], o[2];
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    inc_shared(at[v]);
    // x = p1 2^32 + low word of p0
    const long long p0 = (long long)Wc * (long long)(V[v] & 0xFFFFFFFFll);
    const long long p1 = (long long)Wc * (int)(V[v] >> 32) + (p0 >> 32);
    w0[v] = (uint32_t)p0;
    w1[v] = (uint32_t)p1;
    w2[v] = (uint32_t)((unsigned long long)p1 >> 32);
    o[v] = t_atom(at[v] + stride, w0[v]);
  }
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    asm("{\n\t.reg .u32 s;\n\tadd.cc.u32 s, %2, %3;\n\taddc.cc.u32 %0, %0, 0;\n\t"
        "addc.u32 %1, %1, 0;\n\t}"
        : "+r"(w1[v]), "+r"(w2[v])
        : "r"(o[v]), "r"(w0[v]));
    o[v] = t_atom(at[v] + 2u * stride, w1[v]);
  }
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    asm("{\n\t.reg .u32 s;\n\tadd.cc.u32 s, %1, %2;\n\taddc.u32 %0, %0, 0;\n\t}"
        : "+r"(w2[v])
        : "r"(o[v]), "r"(w1[v]));
    o[v] = t_atom(at[v] + 3u * stride, w2[v]);
  }
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    uint32_t n, c;
    asm("add.cc.u32 %0, %2, %3;\n\taddc.u32 %1, 0, 0;" : "=&r"(n), "=r"(c) : "r"(o[v]), "r"(w2[v]));
    c -= w2[v] >> 31;  // sign extension
    if (c != 0u && at[v] != none) {
      // c 2^96 W_i
      const long long t = (long long)(int)c * Wi;
      const uint32_t cells2 = 2u * (uint32_t)a.hot;  // from here on the even-only ones
      const bool even = ZERO && cell[v] >= cells2;
      const uint32_t slot = even ? cell[v] - cells2 : PARITY ? cell[v] >> 1 : cell[v];
      atomic_add_w192(a.weven + 3 * (size_t)slot, 0ull, (unsigned long long)t << 32,
                      (unsigned long long)(t >> 32));
      if (PARITY && !even && a.chir[slot]) {
        const long long u = (cell[v] & 1u) ? -t : t;
        atomic_add_w192(a.wodd + 3 * (size_t)slot, 0ull, (unsigned long long)u << 32,
                        (unsigned long long)(u >> 32));
      }
    }
  }
}

// One hub by one group of warps. GW: the workspace is in global memory.
// gt: thread within the group; chunk (and wchunk): the warp's 32 entries.
// FAST: unweighted, every slot's cells in shared memory, workspace in shared
// memory; the inner loop is then free of branches. ZERO: weighted, with even-only
// cells (their few instructions in every loop cost 10% where V = 0 is rare).
template <bool PARITY, bool WEIGHTED, bool PIX, bool GW, bool FAST, bool ZERO, class E, class L>
__device__ inline void hub4(const Args& a, const Workspace<L>& w, Shared& s, const Hist& h,
                            const float4* pixu, Chunk* ch, long long* wchunk, int64_t i, int m,
                            int g, int gt) {
  const int lane = threadIdx.x & 31, wg = gt >> 5, group = a.group, gthreads = group * 32;
  const int nb = a.nb;
  const uint32_t* row = row_at(a.adj, a.ptr, i, a.adj_off, a.split, a.adj_off2);
  const int4 P = a.xyzp[i];
  int* cur = s.cur + g * kMaxBins4;
  auto place = [&](int pos, uint32_t word, uint32_t id, const int4& Q) {
    // the fourth component carries the hub edge's bin, so one 128-bit load
    // gives a vertex's displacement and b_i,vertex
    const int dx = (int)mi((int64_t)Q.x - P.x, a.box), dy = (int)mi((int64_t)Q.y - P.y, a.box),
              dz = (int)mi((int64_t)Q.z - P.z, a.box);
    w.disp[pos] = make_int4(dx, dy, dz, (int)edge_bin(word));
    if (PIX) w.hpix[pos] = (uint8_t)dir_pixel(dx, dy, dz);
    if (WEIGHTED) w.wv[pos] = (int)a.W[id];
  };
  if constexpr (PIX) {
    // by caller index: the position is the number of smaller indices
    for (int k = gt; k < m; k += gthreads) w.cid[k] = a.xyzp[edge_id(row[k])].w;
    group_sync(g, gthreads);
    for (int k = gt; k < m; k += gthreads) {
      const int me = w.cid[k];
      int pos = 0;
      for (int t = 0; t < m; ++t) pos += w.cid[t] < me ? 1 : 0;
      const uint32_t word = row[k], id = edge_id(word);
      place(pos, word, id, a.xyzp[id]);
    }
  } else if constexpr (ZERO) {
    // as they are: on a mesh or in a plane lanes with neighbouring c's of one bin
    // would all add to one orbit's cells
    for (int k = gt; k < m; k += gthreads) {
      const uint32_t word = row[k], id = edge_id(word);
      place(k, word, id, a.xyzp[id]);
    }
  } else {
    // by the hub edge's bin (counting sort): lanes with neighbouring c's then
    // share b_03, so their table entries lie in few lines
    for (int k = gt; k < m; k += gthreads) atomicAdd(cur + edge_bin(row[k]), 1);
    group_sync(g, gthreads);
    if (wg == 0) {
      const int v = lane < nb ? cur[lane] : 0;
      int incl = v;
      for (int o = 1; o < 16; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      if (lane < nb) cur[lane] = incl - v;
    }
    group_sync(g, gthreads);
    for (int k = gt; k < m; k += gthreads) {
      const uint32_t word = row[k], id = edge_id(word);
      place(atomicAdd(cur + edge_bin(word), 1), word, id, a.xyzp[id]);
    }
  }
  group_sync(g, gthreads);
  if (!PIX && !ZERO && gt < kMaxBins4) cur[gt] = 0;  // for the next hub (barriers below)
  using I = typename std::conditional<GW, int64_t, int>::type;
  // B: (a, c) is an edge iff E_0^2 <= |D_c - D_a|^2 < E_nb^2 on the staged
  // hub-relative displacements (4 E_nb < L makes their difference the pair's
  // minimum image)
  {
    const int64_t e2lo = s.e2[0], e2hi = s.e2[nb];
    const uint8_t* bk = a.bk_n ? s.bk : nullptr;
    if (gt == 0) w.disp[m] = make_int4(0, 0, 0, 0);  // unused lanes read it
    for (int sa = wg; sa < m; sa += group) {
      const int4 da = w.disp[sa];
      uint8_t* Ba = w.B + row_off<I>(sa, m + 1);
      for (int c = sa + 1 + lane; c <= m; c += 32) {
        if (c == m) {
          Ba[c] = (uint8_t)nb;
          break;
        }
        const int4 dc = w.disp[c];
        const int x = dc.x - da.x, y = dc.y - da.y, z = dc.z - da.z;
        const int64_t D2 = (int64_t)x * x + (int64_t)y * y + (int64_t)z * z;
        uint8_t b = (uint8_t)nb;
        if (D2 >= e2lo && D2 < e2hi) b = (uint8_t)bin_of(D2, s.e2, nb, bk, a.bk_shift);
        Ba[c] = b;
      }
    }
  }
  group_sync(g, gthreads);
  // pixelised parity: neighbours before the hub in caller order
  int nlow = 0;
  if (PIX) {
    for (int t0 = 0; t0 < m; t0 += 32)
      nlow += __popc(__ballot_sync(0xffffffffu, t0 + lane < m && w.cid[t0 + lane] < P.w));
  }
  const int64_t Wi = WEIGHTED ? a.W[i] : 0;
  const bool hist_ok = (unsigned long long)m * (unsigned long long)(m - 1) *
                           (unsigned long long)(m - 2) / 6 <= kMaxHubNeed;
  const E* __restrict__ ent = reinterpret_cast<const E*>(a.ent);
  L* list = w.list + (size_t)wg * w.cap;
  uint8_t* lpix = w.lpix + (size_t)wg * w.cap;
  // rows near the start carry most of the work: warps take them from a
  // shared counter (reset by the group's first thread before the hub began)
  for (int sa = -1;;) {
    if (group == 1) {
      ++sa;
    } else {
      if (lane == 0) sa = atomicAdd(s.row + g, 1);
      sa = __shfl_sync(0xffffffffu, sa, 0);
    }
    if (sa >= m - 2) break;
    const uint8_t* Ba = w.B + row_off<I>(sa, m + 1);
    const int4 da = w.disp[sa];
    const int b01 = da.w;
    const int64_t Wa = WEIGHTED ? (int64_t)w.wv[sa] : 0;
    // Pixelised parity. The neighbours are in caller order, so the spokes'
    // origin (the smallest caller index) is the hub or a. From the hub the
    // order is (hub, a, b, c) and the sign is that of V(u_a, u_b, u_c); from
    // a, with the hub anywhere after a, sorting (hub, a, b, c) and reordering
    // the spokes to (hub, b, c) together give one sign change:
    // -V(u_hub, u_b, u_c). A spoke of zero length gets a zero vector (V = 0).
    const bool from_a = PIX && sa < nlow;
    auto spoke = [&](const int4& d, int pix) -> float4 {
      const bool zero = from_a ? (d.x == da.x && d.y == da.y && d.z == da.z)
                               : ((d.x | d.y | d.z) == 0);
      return zero ? make_float4(0.f, 0.f, 0.f, 0.f) : pixu[pix];
    };
    float4 u1 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (PIX) {
      if (!from_a) {
        u1 = spoke(da, w.hpix[sa]);
      } else if ((da.x | da.y | da.z) != 0) {
        const float4 u = pixu[dir_pixel(-(int64_t)da.x, -(int64_t)da.y, -(int64_t)da.z)];
        u1 = make_float4(-u.x, -u.y, -u.z, 0.f);
      }
    }
    int n = 0;
    for (int c0 = sa + 1; c0 < m; c0 += 32) {
      const int c = c0 + lane;
      const bool e = c < m && Ba[c] < nb;
      const unsigned mask = __ballot_sync(0xffffffffu, e);
      if (e) {
        const int p = n + __popc(mask & ((1u << lane) - 1u));
        list[p] = (L)c;
        if (PIX) {
          const int4 dc = w.disp[c];
          lpix[p] = from_a ? (uint8_t)dir_pixel((int64_t)dc.x - da.x, (int64_t)dc.y - da.y,
                                                (int64_t)dc.z - da.z)
                           : w.hpix[c];
        }
      }
      n += __popc(mask);
    }
    for (int k0 = 0; k0 < n - 1; k0 += 32) {
      __syncwarp();  // the list is written; the chunk is no longer read
      {
        const int p = k0 + lane;
        int brow = 0;
        uint32_t tri = 0;
        float nx = 0.f, ny = 0.f, nz = 0.f;
        long long wab = 0;
        if (p < n) {
          const int b = (int)list[p];
          const int4 db = w.disp[b];
          tri = (uint32_t)((b01 * nb + db.w) * nb + Ba[b]) * (uint32_t)a.tab3;
          brow = GW ? b : row_off<int>(b, m + 1);
          if (PARITY) {
            if constexpr (PIX) {
              const float4 u2 = spoke(db, lpix[p]);
              nx = u1.y * u2.z - u1.z * u2.y;
              ny = u1.z * u2.x - u1.x * u2.z;
              nz = u1.x * u2.y - u1.y * u2.x;
            } else {
              nx = i40_to_float((long long)da.y * db.z - (long long)da.z * db.y);
              ny = i40_to_float((long long)da.z * db.x - (long long)da.x * db.z);
              nz = i40_to_float((long long)da.x * db.y - (long long)da.y * db.x);
            }
          }
          if (WEIGHTED) wab = Wa * w.wv[b];
        }
        ch->row[lane] = brow;
        ch->tab[lane] = tri;
        if (PARITY) {
          ch->nx[lane] = nx;
          ch->ny[lane] = ny;
          ch->nz[lane] = nz;
        }
        if (WEIGHTED) wchunk[lane] = wab;
      }
      __syncwarp();
      for (int t0 = k0; t0 < n; t0 += 32) {
        const int p = t0 + lane;
        const bool in = p < n;
        const int c = in ? (int)list[p] : m;  // column m: no edges
        const int4 dc = w.disp[c];
        const uint32_t lane_idx = (uint32_t)((dc.w * nb + (in ? (int)Ba[c] : 0)) * (nb + 1));
        const int Wc = WEIGHTED && in ? w.wv[c] : 0;
        float ux = 0.f, uy = 0.f, uz = 0.f;
        if constexpr (PIX) {
          const float4 u3 = spoke(dc, in ? lpix[p] : 0);
          ux = u3.x, uy = u3.y, uz = u3.z;
        } else if (PARITY) {
          // unused lanes: a volume far from zero
          ux = in ? (float)dc.x : 1e20f, uy = (float)dc.y, uz = (float)dc.z;
        }
        const int ns = t0 > k0 ? 32 : min(31, n - 1 - k0);
        if constexpr (FAST) {
          const uint8_t* Bc = w.B + c;
          const E* ent_c = ent + lane_idx;
          const uint32_t trash = (uint32_t)(PARITY ? 2 * a.hot : a.hot);
          const uint32_t cells = (uint32_t)__cvta_generic_to_shared(h.cnt);
          const unsigned long long ux2 = pack2(ux, ux), uy2 = pack2(uy, uy), uz2 = pack2(uz, uz);
          auto steps = [&](auto diag) {
            constexpr int U = 4;
            for (int s0 = 0; s0 < ns; s0 += U) {
              uint32_t b23[U];
              int en[U];
              float V[U] = {0.f, 0.f, 0.f, 0.f};
              const int4 r = *reinterpret_cast<const int4*>(ch->row + s0);
              const uint4 t = *reinterpret_cast<const uint4*>(ch->tab + s0);
              const int rr[U] = {r.x, r.y, r.z, r.w};
              const uint32_t tt[U] = {t.x, t.y, t.z, t.w};
#pragma unroll
              for (int u = 0; u < U; ++u) {
                b23[u] = (uint32_t)nb;
                if (!decltype(diag)::value || s0 + u < lane) b23[u] = Bc[rr[u]];
                en[u] = load_entry(ent_c + (tt[u] + b23[u]));
              }
              if (PARITY) {
                const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(ch->nx + s0);
                const ulonglong2 y = *reinterpret_cast<const ulonglong2*>(ch->ny + s0);
                const ulonglong2 z = *reinterpret_cast<const ulonglong2*>(ch->nz + s0);
                unpack2(fma2(z.x, uz2, fma2(y.x, uy2, mul2(x.x, ux2))), V[0], V[1]);
                unpack2(fma2(z.y, uz2, fma2(y.y, uy2, mul2(x.y, ux2))), V[2], V[3]);
              }
              // Signs are settled before any counter is touched: counters only
              // grow, so another group's flush may take them at any moment.
              if constexpr (PARITY && !PIX) {
                float vmin = 3.0e38f;
#pragma unroll
                for (int u = 0; u < U; ++u)
                  if (!decltype(diag)::value || s0 + u < lane) vmin = fminf(vmin, fabsf(V[u]));
                if (vmin < a.eps) {
                  // a volume within its error bound of zero: the exact sign, or
                  // the two cells in turn if V = 0
#pragma unroll
                  for (int u = 0; u < U; ++u) {
                    if (b23[u] >= (uint32_t)nb || !(fabsf(V[u]) < a.eps) || en[u] >= 0) continue;
                    const long long Vx = det3(da, w.disp[list[k0 + s0 + u]], dc);
                    V[u] = Vx < 0 ? -1.0f : 1.0f;
                    if (Vx == 0)
                      en[u] = (int)take_turn(h, ((uint32_t)en[u] & Ent<E>::kMask) >> 1);
                  }
                }
              }
#pragma unroll
              for (int u = 0; u < U; ++u) {
                uint32_t cell;
                if constexpr (PARITY) {
                  // V < 0 on a chiral orbit
                  const uint32_t neg = (__float_as_uint(V[u]) & (uint32_t)en[u]) >> 31;
                  cell = ((uint32_t)en[u] ^ neg) & Ent<E>::kMask;
                  // degenerate pixel volumes are a few percent: even channel
                  if (PIX && fabsf(V[u]) < a.eps && en[u] < 0) {
                    atomicAdd(a.even + (cell >> 1), 1ull);
                    cell = trash;
                  }
                } else {
                  cell = ((uint32_t)en[u] & Ent<E>::kMask) >> 1;
                }
                inc_shared(cells + 4u * cell);
              }
            }
          };
          if (t0 > k0) steps(std::false_type{});
          else steps(std::true_type{});
        } else if constexpr (WEIGHTED) {
          const uint8_t* Bc = w.B + c;
          const E* ent_c = ent + lane_idx;
          const uint32_t hotc = hist_ok ? (uint32_t)(PARITY ? 2 * a.hot : a.hot) : 0u;
          const uint32_t cells = (uint32_t)__cvta_generic_to_shared(h.cnt),
                         cells2 = (uint32_t)(PARITY ? 2 * a.hot : a.hot),
                         evenc = cells2 + (ZERO ? (uint32_t)a.even_hot : 0u),
                         hotce = hist_ok ? evenc : 0u,
                         none = cells + 4u * (evenc + lane);
          auto steps = [&](auto diag) {
            for (int s0 = 0; s0 < ns; s0 += 2) {
              uint32_t b23[2], cell[2], at[2];
              int en[2];
              float V[2] = {1.f, 1.f};
              long long wab[2];
              const int2 r = *reinterpret_cast<const int2*>(ch->row + s0);
              const uint2 t = *reinterpret_cast<const uint2*>(ch->tab + s0);
              const longlong2 w2 = *reinterpret_cast<const longlong2*>(wchunk + s0);
              wab[0] = w2.x, wab[1] = w2.y;
#pragma unroll
              for (int u = 0; u < 2; ++u) {
                const int ru = u ? r.y : r.x;
                b23[u] = (uint32_t)nb;
                if (!decltype(diag)::value || s0 + u < lane)
                  b23[u] = Bc[GW ? row_off<I>((I)ru, m + 1) : (I)ru];
                en[u] = load_entry(ent_c + ((u ? t.y : t.x) + b23[u]));
              }
              bool rare = false;
              if constexpr (PARITY) {
                const float2 x = *reinterpret_cast<const float2*>(ch->nx + s0),
                             y = *reinterpret_cast<const float2*>(ch->ny + s0),
                             z = *reinterpret_cast<const float2*>(ch->nz + s0);
                V[0] = fmaf(z.x, uz, fmaf(y.x, uy, x.x * ux));
                V[1] = fmaf(z.y, uz, fmaf(y.y, uy, x.y * ux));
              }
#pragma unroll
              for (int u = 0; u < 2; ++u) {
                if constexpr (PARITY) {
                  const uint32_t neg = (__float_as_uint(V[u]) & (uint32_t)en[u]) >> 31;
                  cell[u] = ((uint32_t)en[u] ^ neg) & Ent<E>::kMask;
                  rare |= fabsf(V[u]) < a.eps;
                } else {
                  cell[u] = ((uint32_t)en[u] & Ent<E>::kMask) >> 1;
                }
                const bool even = ZERO && en[u] >= 0;
                if (ZERO) cell[u] = even ? cells2 + (cell[u] >> 1) : cell[u];
                const bool hot = cell[u] < (even ? hotce : hotc);
                rare |= !hot && b23[u] < (uint32_t)nb;
                at[u] = hot ? cells + 4u * cell[u] : none;
              }
              if (rare) {
                // a volume near zero is decided in integers; what has no shared
                // cell goes to the global sums
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                  if (b23[u] >= (uint32_t)nb) continue;
                  bool deg = false;
                  if (PARITY && fabsf(V[u]) < a.eps && en[u] < 0) {
                    const long long Vx = PIX ? 0 : det3(da, w.disp[list[k0 + s0 + u]], dc);
                    deg = Vx == 0;
                    cell[u] = ((uint32_t)en[u] ^ (Vx < 0 ? 1u : 0u)) & Ent<E>::kMask;
                    at[u] = cell[u] < hotc && !deg ? cells + 4u * cell[u] : none;
                  }
                  if constexpr (ZERO) {
                    if (deg) {
                      cell[u] = cells2 + (cell[u] >> 1);
                      at[u] = cell[u] < hotce ? cells + 4u * cell[u] : none;
                    }
                    if (at[u] == none)
                      record_limbs(a.limbs,
                                   en[u] >= 0 || deg ? a.even_limbs + (cell[u] - cells2) : cell[u],
                                   Wi, wab[u], Wc);
                  } else if (deg || cell[u] >= hotc) {
                    if (!PARITY && a.long_rows)
                      record_sum(a, cell[u], Wi, wab[u], Wc);
                    else
                      record_limbs(a.limbs, deg ? a.even_limbs + (cell[u] >> 1) : cell[u], Wi,
                                   wab[u], Wc);
                  }
                }
              }
              record_weighted<PARITY, ZERO>(a, at, cell, none, 4u * h.stride, Wi, Wc, wab);
            }
          };
          if (t0 > k0) steps(std::false_type{});
          else steps(std::true_type{});
        } else {
          // entries [0, lim) of the chunk come before c
          const int lim = min(ns, in ? (t0 > k0 ? 32 : lane) : 0);
          const uint32_t hotc = hist_ok ? (uint32_t)(PARITY ? 2 * a.hot : a.hot) : 0u;
          constexpr int U = 2;  // two steps' loads before their updates
          for (int s0 = 0; s0 < lim; s0 += U) {
            uint32_t b23[U], e[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const I rb = GW ? row_off<I>((I)ch->row[s0 + u], m + 1) : (I)ch->row[s0 + u];
              b23[u] = (uint32_t)nb;
              if (s0 + u < lim) b23[u] = w.B[rb + c];
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
              e[u] = 0u;
              if (b23[u] < (uint32_t)nb) e[u] = ent[ch->tab[s0 + u] + lane_idx + b23[u]];
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
              if (b23[u] >= (uint32_t)nb) continue;
              uint32_t cell = e[u] & Ent<E>::kMask;
              bool deg = false;
              if constexpr (PARITY) {
                const float V = fmaf(ch->nz[s0 + u], uz,
                                     fmaf(ch->ny[s0 + u], uy, ch->nx[s0 + u] * ux));
                const uint32_t chiral = e[u] >> Ent<E>::kTop;
                uint32_t neg = __float_as_uint(V) >> 31;
                if (fabsf(V) < a.eps) {
                  const long long Vx = PIX ? 0 : det3(da, w.disp[list[k0 + s0 + u]], dc);
                  neg = Vx < 0 ? 1u : 0u;
                  deg = Vx == 0 && chiral;
                }
                cell ^= neg & chiral;
              } else {
                cell >>= 1;
              }
              if (PARITY && deg && cell < hotc) cell = take_turn(h, cell >> 1);
              if (cell < hotc) atomicAdd(h.cnt + cell, 1u);
              else record_global<PARITY>(a, cell, !deg && (e[u] >> Ent<E>::kTop));
            }
          }
        }
      }
    }
    __syncwarp();  // the list is rewritten for the next row
  }
}

// VARIANT: FAST of an unweighted launch, ZERO of a weighted one.
template <bool PARITY, bool WEIGHTED, bool PIX, bool VARIANT, class E>
__global__ void __launch_bounds__(kThreads, 1) k_count4(Args a) {
  constexpr bool FAST = !WEIGHTED && VARIANT, ZERO = WEIGHTED && VARIANT;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Shared s;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int group = a.group, gthreads = group * 32, g = warp / group, gt = tid - g * gthreads;
  unsigned char* sp = smem;
  Hist h;
  h.stride = (uint32_t)hist_words((PARITY ? 2 : 1) * a.hot + (ZERO ? a.even_hot : 0));
  h.cnt = reinterpret_cast<unsigned*>(sp);
  sp += pad16((size_t)h.stride * (WEIGHTED ? 16 : 4));
  float4* pixu = reinterpret_cast<float4*>(sp);
  if (PIX) sp += 256 * sizeof(float4);
  Chunk* ch = reinterpret_cast<Chunk*>(sp) + warp;
  sp += (size_t)kWarps * sizeof(Chunk);
  long long* wchunk = reinterpret_cast<long long*>(sp) + warp * 32;
  if (WEIGHTED) sp += (size_t)kThreads * sizeof(long long);
  const Workspace<uint16_t> ws_s = carve<uint16_t>(
      sp + (size_t)g * workspace_bytes(a.cap, group, sizeof(uint16_t), WEIGHTED, PIX), a.cap,
      group, WEIGHTED, PIX);

  for (uint32_t k = tid; k < h.stride * (WEIGHTED ? 4 : 1); k += kThreads)
    h.cnt[k] = k < 3 * h.stride ? 0u : kTopZero;
  for (int k = tid; k < kWarps * kMaxBins4; k += kThreads) s.cur[k] = 0;
  for (int b = tid; b <= a.nb; b += kThreads) s.e2[b] = a.e2g[b];
  for (int k = tid; k < a.bk_n; k += kThreads) {
    const int64_t x = (int64_t)k << a.bk_shift;
    int b = 0;
    while (b + 1 < a.nb && a.e2g[b + 1] <= x) ++b;
    s.bk[k] = (uint8_t)b;
  }
  if (PIX)
    for (int k = tid; k < 256; k += kThreads) pixu[k] = a.pixu[k];
  if (tid == 0) s.pending = 0;
  __syncthreads();

  // Adds the shared counters to the global counts and clears them. Exchanges,
  // so that one group can do it while the others count on.
  auto flush = [&](int t, int threads) {
    for (int k = t; k < a.hot; k += threads) {
      if (PARITY) {
        const unsigned c = atomicExch(h.cnt + 2 * k, 0u), n = atomicExch(h.cnt + 2 * k + 1, 0u);
        if (c | n) {
          const unsigned p = c & ~kTurn;
          const long long d = (long long)p - (long long)n - (long long)(c >> 31);
          if (p | n) atomicAdd(a.even + k, (unsigned long long)p + n);
          if (d && a.chir[k]) atomicAdd(a.odd + k, (unsigned long long)d);
        }
      } else {
        const unsigned p = atomicExch(h.cnt + k, 0u);
        if (p) atomicAdd(a.even + k, (unsigned long long)p);
      }
    }
    if (ZERO)
      for (int k = t; k < a.even_hot; k += threads) {
        const unsigned z = atomicExch(h.cnt + 2 * a.hot + k, 0u);
        if (z) atomicAdd(a.even + k, (unsigned long long)z);
      }
  };

  unsigned long long next = 0;  // the group's first thread: the next ticket, taken ahead
  if (gt == 0) next = atomicAdd(a.hub_counter, 1ull);
  for (;;) {
    if (gt == 0) {
      int64_t i = -1;
      for (;;) {
        const int64_t q = (int64_t)next;
        if (a.list) {
          if (q >= a.nlist) break;
          next = atomicAdd(a.hub_counter, 1ull);
          i = a.list[q];
          break;
        }
        const int64_t j = a.hub_begin + q * a.hub_stride;
        if (j >= a.hub_end) break;
        next = atomicAdd(a.hub_counter, 1ull);
        const int d = a.deg[j];
        if (d >= 3 && d <= a.dmax) {
          i = j;
          break;
        }
      }
      s.hub[g] = i;
      s.row[g] = 0;
      s.flush[g] = 0;
      if (i >= 0) {
        const unsigned long long m = (unsigned long long)a.deg[i];
        const unsigned long long need = m * (m - 1) * (m - 2) / 6;
        // The shared counters stay below 2^31: between two flushes they take
        // the hubs registered since the last reset (at most 2^28 and one
        // hub), those registered while a flush runs (the same) and those
        // under way at a reset (31 hubs). A hub is at most 2^26, and below 2^25
        // where a CTA has several groups (their rows are in shared memory).
        if (need <= kMaxHubNeed &&
            atomicAdd(&s.pending, need) + need > a.limit) {
          atomicExch(&s.pending, 0ull);
          s.flush[g] = 1;
        }
      }
    }
    group_sync(g, gthreads);
    const int64_t i = s.hub[g];
    if (i < 0) break;
    if (s.flush[g]) flush(gt, gthreads);
    const int m = a.deg[i];
    if (m > a.cap) {
      const Workspace<uint32_t> ws_g =
          carve<uint32_t>(a.gscratch + (size_t)blockIdx.x * a.gscratch_stride, a.gcap, group,
                          WEIGHTED, PIX);
      hub4<PARITY, WEIGHTED, PIX, true, false, ZERO, E>(a, ws_g, s, h, pixu, ch, wchunk, i, m, g, gt);
    } else {
      hub4<PARITY, WEIGHTED, PIX, false, FAST, ZERO, E>(a, ws_s, s, h, pixu, ch, wchunk, i, m, g, gt);
    }
    group_sync(g, gthreads);
    if (WEIGHTED) {
      // the hub's sums times W_i into the global 192-bit sums (weighted
      // launches have one group; the barrier at the top of the loop orders
      // the clearing before the next hub's additions)
      const long long Wi = a.W[i];
      // the words as a signed 96-bit number (carries out of it are in the
      // global sums already); cleared
      auto take = [&](int cell, unsigned long long& lo, unsigned long long& hi) {
        unsigned* c = h.cnt + h.stride + cell;
        const uint32_t w0 = c[0], w1 = c[h.stride], w2 = c[2 * h.stride];
        lo = ((unsigned long long)w1 << 32) | w0;
        hi = (unsigned long long)(long long)(int)(w2 ^ kTopZero);
        if (lo | hi) {
          c[0] = c[h.stride] = 0u;
          c[2 * h.stride] = kTopZero;
        }
      };
      // a hub of few tetrahedra: every cell's sum times W_i is below 2^124 and
      // goes to the limbs of its cell, which waits for nothing (1e5 points, rows
      // of 8, nb = 8: 5.9 -> 4.9 ms)
      const unsigned long long mm = (unsigned long long)m;
      if (mm * (mm - 1) * (mm - 2) / 6 <= a.limb_need) {
        const int n2 = (PARITY ? 2 : 1) * a.hot, all = n2 + (ZERO ? a.even_hot : 0);
        for (int k = gt; k < all; k += gthreads) {
          unsigned long long lo, hi;
          take(k, lo, hi);
          if (!(lo | hi)) continue;
          const unsigned long long v = (unsigned long long)Wi;
          add_limbs(a.limbs + (size_t)(k < n2 ? (uint32_t)k : a.even_limbs + (uint32_t)(k - n2)) *
                                  kLimbWords,
                    (long long)(lo * v),
                    (long long)(__umul64hi(lo, v) - (Wi < 0 ? lo : 0ull) + hi * v));
        }
        continue;
      }
      for (int k = gt; k < a.hot; k += gthreads) {
        unsigned long long elo, ehi;
        take(PARITY ? 2 * k : k, elo, ehi);
        if (PARITY) {
          // even = S+ + S-, odd = S+ - S-
          unsigned long long nlo, nhi;
          take(2 * k + 1, nlo, nhi);
          if (!(elo | ehi | nlo | nhi)) continue;
          const unsigned long long olo = elo - nlo, ohi = ehi - nhi - (elo < nlo ? 1ull : 0ull);
          elo += nlo;
          ehi += nhi + (elo < nlo ? 1ull : 0ull);
          if ((olo | ohi) && a.chir[k]) fold_i128(a.wodd + 3 * k, olo, ohi, Wi);
        }
        if (elo | ehi) fold_i128(a.weven + 3 * k, elo, ehi, Wi);
      }
      if (ZERO)
        for (int k = gt; k < a.even_hot; k += gthreads) {
          unsigned long long lo, hi;
          take(2 * a.hot + k, lo, hi);
          if (lo | hi) fold_i128(a.weven + 3 * k, lo, hi, Wi);
        }
    }
  }
  __syncthreads();
  flush(tid, kThreads);
}

}  // namespace

// 192-bit sums: x += y or x -= y.
__device__ inline void add_w192(unsigned long long (&x)[3], const unsigned long long (&y)[3],
                                bool minus) {
  unsigned long long c = minus ? 1ull : 0ull;
  for (int k = 0; k < 3; ++k) {
    const unsigned long long v = minus ? ~y[k] : y[k], s = x[k] + v;
    const unsigned long long t = s + c;
    c = (s < v ? 1ull : 0ull) + (t < s ? 1ull : 0ull);
    x[k] = t;
  }
}

// Adds the limbs (see record_limbs) of every slot to its counts and 192-bit sums
// and clears them. odd, wodd: nullptr without parity.
__global__ void k_limbs(unsigned long long* limbs, int64_t n, const uint8_t* chir,
                        unsigned long long* even, unsigned long long* odd,
                        unsigned long long* weven, unsigned long long* wodd) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    unsigned long long cnt[3] = {0, 0, 0}, sum[3][3] = {};
    const int cells = odd ? 3 : 1;
    bool any = false;
    for (int c = 0; c < cells; ++c) {
      unsigned long long* L =
          limbs + (size_t)(odd ? (c < 2 ? 2 * k + c : 2 * n + k) : k) * kLimbWords;
      unsigned long long l[kLimbs], some = cnt[c] = L[0];
      for (int q = 0; q < kLimbs; ++q) some |= l[q] = L[1 + q];
      if (!some) continue;
      any = true;
      for (int q = 0; q < kLimbWords; ++q) L[q] = 0ull;
      for (int q = 0; q < kLimbs; ++q) {
        const unsigned long long v = l[q];
        const unsigned long long ext = q + 1 == kLimbs && (long long)v < 0 ? ~0ull : 0ull;
        const int sh = q * kLimbBits, w = sh >> 6, r = sh & 63;
        unsigned long long y[3] = {0, 0, 0};
        const unsigned long long part[2] = {v << r, r ? (v >> (64 - r)) | (ext << r) : ext};
        for (int p = w; p < 3; ++p) y[p] = p - w < 2 ? part[p - w] : ext;
        add_w192(sum[c], y, false);
      }
    }
    if (!any) continue;
    even[k] += cnt[0] + cnt[1] + cnt[2];
    unsigned long long* E = weven + 3 * k;
    unsigned long long x[3] = {E[0], E[1], E[2]};
    for (int c = 0; c < cells; ++c) add_w192(x, sum[c], false);
    for (int q = 0; q < 3; ++q) E[q] = x[q];
    if (!odd || !chir[k]) continue;
    odd[k] += cnt[0] - cnt[1];
    unsigned long long* O = wodd + 3 * k;
    unsigned long long z[3] = {O[0], O[1], O[2]};
    add_w192(z, sum[0], false);
    add_w192(z, sum[1], true);
    for (int q = 0; q < 3; ++q) O[q] = z[q];
  }
}

__global__ void k_i192_to_double(const unsigned long long* acc, int64_t n, int scale, double* out);
__global__ void k_u64_to_double(const unsigned long long* c, int64_t n, double* out);
__global__ void k_i64_to_double(const long long* c, int64_t n, double* out) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x)
    out[k] = (double)c[k];
}

namespace {
// Unit vectors of the 256 pixel centres (band z_c = -1 + (band + 1/2) / 8,
// sector phi_c = (sector + 1/2) pi / 8), formed in FP64 on the host, kept per
// device.
std::mutex g_pix_mu;
float4* g_pix_dev[64] = {nullptr};

const float4* pixel_centres(int* status) {
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) {
    *status = GS_ERANGE;
    return nullptr;
  }
  std::lock_guard<std::mutex> lock(g_pix_mu);
  if (g_pix_dev[dev]) return g_pix_dev[dev];
  std::vector<float4> u(256);
  for (int p = 0; p < 256; ++p) {
    const double zc = (2.0 * (p >> 4) + 1.0) / 16.0 - 1.0;
    const double phi = M_PI * (2.0 * (p & 15) + 1.0) / 16.0;
    const double rho = std::sqrt((1.0 - zc) * (1.0 + zc));
    u[p] = make_float4((float)(rho * std::cos(phi)), (float)(rho * std::sin(phi)), (float)zc, 0.f);
  }
  float4* d = nullptr;
  cudaError_t e = cudaMalloc(&d, u.size() * sizeof(float4));
  if (e == cudaSuccess)
    e = cudaMemcpy(d, u.data(), u.size() * sizeof(float4), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    cudaGetLastError();
    if (d) cudaFree(d);
    *status = cuda_status(e);
    return nullptr;
  }
  g_pix_dev[dev] = d;
  return d;
}

// Table entries (see Ent) and chirality by slot from the orbit table: orbit o
// takes slot slot_of[o] (its own index when slot_of is null).
template <class E>
__global__ void k_entries(const uint32_t* __restrict__ lut, int64_t n, int nb, int n_orbits,
                          const int32_t* __restrict__ slot_of, E* out, uint8_t* chir) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = k / (nb + 1);
    const int b = (int)(k - row * (nb + 1));
    if (b == nb) {
      out[k] = (E)(n_orbits << 1);
      continue;
    }
    const uint32_t e = lut[row * nb + b], o = e & 0x3FFFFFFFu, chiral = e >> 31;
    const uint32_t slot = slot_of ? (uint32_t)slot_of[o] : o;
    out[k] = (E)((slot << 1) | ((e >> 30) & chiral) | (chiral << Ent<E>::kTop));
    chir[slot] = (uint8_t)chiral;  // every raw tuple of an orbit agrees
  }
}

// Per-slot results back to orbit order: dst[o] = src[slot_of[o]], `words`
// 64-bit words per entry.
__global__ void k_slots_to_orbits(const unsigned long long* __restrict__ src,
                                  const int32_t* __restrict__ slot_of, int64_t n, int words,
                                  unsigned long long* dst) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n * words;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t o = k / words;
    dst[k] = src[(int64_t)slot_of[o] * words + (k - o * words)];
  }
}

// Fraction of volumes of zero, estimated: triples of neighbours of random hubs,
// out[0] those with V = 0 (pixelised: of the pixels seen from the hub), out[1]
// all. Any sequence of numbers will do; the answer only decides a layout.
__global__ void k_zero_volumes(Args a, int pix, unsigned* out) {
  uint32_t r = (blockIdx.x * blockDim.x + threadIdx.x) * kHashMul + 12345u;
  auto next = [&](int n) {
    r = r * 1664525u + 1013904223u;
    return (int)__umulhi(r, (uint32_t)n);
  };
  const int64_t i = a.hub_begin + next((int)(a.hub_end - a.hub_begin));
  const int m = a.deg[i];
  if (m < 3) return;
  const uint32_t* row = row_at(a.adj, a.ptr, i, a.adj_off, a.split, a.adj_off2);
  const int4 P = a.xyzp[i];
  const int at[3] = {next(m), next(m), next(m)};
  if (at[0] == at[1] || at[0] == at[2] || at[1] == at[2]) return;
  int4 d[3];
  float4 u[3];
  for (int v = 0; v < 3; ++v) {
    const int4 Q = a.xyzp[edge_id(row[at[v]])];
    d[v] = make_int4((int)mi((int64_t)Q.x - P.x, a.box), (int)mi((int64_t)Q.y - P.y, a.box),
                     (int)mi((int64_t)Q.z - P.z, a.box), 0);
    if (pix) u[v] = a.pixu[dir_pixel(d[v].x, d[v].y, d[v].z)];
  }
  bool zero;
  if (pix) {
    const float V = (u[0].y * u[1].z - u[0].z * u[1].y) * u[2].x +
                    (u[0].z * u[1].x - u[0].x * u[1].z) * u[2].y +
                    (u[0].x * u[1].y - u[0].y * u[1].x) * u[2].z;
    zero = fabsf(V) < a.eps;
  } else {
    zero = det3(d[0], d[1], d[2]) == 0;
  }
  if (zero) atomicAdd(out, 1u);
  atomicAdd(out + 1, 1u);
}

__global__ void k_dir_pixels(const int32_t* d, int64_t n, uint8_t* out) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x)
    out[k] = (uint8_t)dir_pixel(d[3 * k], d[3 * k + 1], d[3 * k + 2]);
}
}  // namespace

int direction_pixels_device(const int32_t* d_dirs, int64_t n, uint8_t* d_out, cudaStream_t s) {
  if (n > 0) {
    const int blocks = (int)std::min<int64_t>((n + 255) / 256, 4096);
    k_dir_pixels<<<blocks, 256, 0, s>>>(d_dirs, n, d_out);
    note_launch();
  }
  return cuda_status(cudaGetLastError());
}

namespace {
// variant: unweighted with every slot in shared memory; weighted parity with
// cells for V = 0
template <class E>
void (*pick4(bool parity, bool weighted, bool pix, bool variant))(Args) {
#define GS_K4(P, X)                                                             \
  (weighted ? (P && variant ? k_count4<P, true, X, P, E> : k_count4<P, true, X, false, E>) \
   : variant ? k_count4<P, false, X, true, E>                                   \
             : k_count4<P, false, X, false, E>)
  if (parity && pix) return GS_K4(true, true);
  if (parity) return GS_K4(true, false);
  return GS_K4(false, false);
#undef GS_K4
}

// Shared memory of a launch: `cells` counters, chunks, pixel centres and the
// workspaces of 32 / group groups.
size_t launch_smem(int64_t cells, int cap, int group, bool weighted, bool pix) {
  return pad16(hist_words(cells) * (weighted ? 16 : 4)) + (pix ? 256 * sizeof(float4) : 0) +
         (size_t)kWarps * sizeof(Chunk) + (weighted ? (size_t)kThreads * 8 : 0) +
         (size_t)(kWarps / group) * workspace_bytes(cap, group, sizeof(uint16_t), weighted, pix);
}

// Largest row capacity (a multiple of 16, at most want) of a launch, 0 if
// not even 16 fit.
int fit_cap(int want, int64_t cells, int group, bool weighted, bool pix, size_t avail) {
  int cap = (want + 15) & ~15;
  while (cap >= 16 && launch_smem(cells, cap, group, weighted, pix) > avail) cap -= 16;
  return std::max(cap, 0);
}
}  // namespace

int count4_device(const Graph& g, const FixedW* fw, bool parity, uint64_t* d_even,
                  int64_t* d_odd, double* d_weven, double* d_wodd, const Opts& o, bool pix,
                  unsigned long long* weven_out, unsigned long long* wodd_out) {
  cudaStream_t s = o.stream;
  Scratch sc(s);  // given back on return: wide weights make five of these calls
  int st = GS_OK;
  pix = pix && parity;
  const float4* pixu = nullptr;
  if (pix) {
    pixu = pixel_centres(&st);
    if (!pixu) return st;
  }
  const Conf4Tables* t = conf4_tables(g.nb, &st);
  if (!t) return st;
  const int no = (int)t->n_orbits;
  const bool weighted = fw != nullptr;
  Args a;
  a.ptr = g.d_ptr;
  a.deg = g.d_deg;
  a.adj = nullptr;
  a.adj_off = 0;
  a.split = g.n;
  a.adj_off2 = 0;
  a.hub_begin = 0;
  a.hub_end = g.n;
  a.hub_stride = 1;
  a.list = nullptr;
  a.nlist = 0;
  a.xyzp = g.d_xyzp;
  a.e2g = g.d_edges2;
  a.box = g.box_u;
  a.nb = g.nb;
  a.tab3 = g.nb * g.nb * (g.nb + 1);
  a.even = reinterpret_cast<unsigned long long*>(d_even);
  a.odd = parity ? (d_odd ? reinterpret_cast<unsigned long long*>(d_odd)
                          : sc.alloc<unsigned long long>(no))
                 : nullptr;
  a.W = weighted ? fw->d_W : nullptr;
  a.pixu = pixu;
  // |V| <= E_nb^3; the single-precision volume is within 4 2^-24 E_nb^3 of
  // the exact one (one rounding of each component of the cross product and
  // three of the sum, each relative to at most |d_a x d_b| |d_c|)
  {
    const double r = (double)g.edges[g.nb];
    a.eps = pix ? kPixZero : (float)std::ldexp(r * r * r, -21);
  }
  // variant 1024: a flush before every hub (exercises flushes while other
  // groups count)
  a.limit = (o.variant & 1024) ? 0 : 1ull << 28;
  // weighted results land in the callers' 192-bit arrays (or scratch)
  unsigned long long* weven = weighted ? (weven_out ? weven_out : sc.alloc<unsigned long long>(3 * (size_t)no))
                                       : nullptr;
  unsigned long long* wodd = (weighted && parity) ? (wodd_out ? wodd_out : sc.alloc<unsigned long long>(3 * (size_t)no))
                                                  : nullptr;
  a.weven = weven;
  a.wodd = wodd;
  const size_t limb_words = weighted ? (size_t)(parity ? 3 : 1) * no * kLimbWords : 0;
  a.limbs = weighted ? sc.alloc<unsigned long long>(limb_words) : nullptr;
  a.even_limbs = 2u * (uint32_t)no;
  // (need) 2^(4 mag) < 2^124
  a.limb_need = weighted && fw->mag < 31 ? (1ull << std::min(40, 123 - 4 * fw->mag)) : 0;
  a.hub_counter = sc.alloc<unsigned long long>(1);
  if (!a.hub_counter || (parity && !a.odd) || (weighted && (!a.weven || !a.limbs)) ||
      (weighted && parity && !a.wodd))
    return GS_ENOMEM;

  int dev = 0, sms = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const size_t avail = (size_t)optin - sizeof(Shared) - 64;
  // two-byte entries hold slots below 2^14 (nb <= 8)
  const bool small_ent = no < 16384;
  // Launch 1: groups of `group` warps over every hub of at most `cap`
  // neighbours; launch 2 (when longer rows exist): whole CTAs over a list of
  // the longer ones, in shared memory up to cap2, else in global scratch.
  const int maxd = std::max(g.max_deg, 3);
  const double mean = g.n ? (double)g.edges_total / (double)g.n : 0.0;
  a.long_rows = mean > 100.0;
  int group = kWarps, cap = 0, cap2 = 0, nh = no;
  const int64_t per = parity ? 2 : 1;  // cells per slot
  int64_t room = 0;                   // cells that fit
  bool even_cells = false, probe = false;  // ZERO, and whether a sample of volumes decides on it
  a.even_hot = 0;
  const bool all_hot = !weighted && !(o.variant & 8) &&
                       fit_cap(std::min(256, maxd), per * no, kWarps, false, pix, avail) >=
                           std::min(256, (maxd + 15) & ~15);
  // few warps per hub where rows are short: a hub's barriers and its rows' ragged
  // ends cost the same however many warps wait for them
  auto warps_per_hub = [](double m) {
    return m <= 24 ? 1 : m <= 48 ? 4 : m <= 96 ? 8 : m <= 160 ? 16 : kWarps;
  };
  if (all_hot) {
    group = warps_per_hub(mean);
    const int want = std::min(maxd, std::max(48, (int)(2.0 * mean) + 32));
    for (;; group = group == 1 ? 4 : group * 2) {
      cap = fit_cap(maxd, per * no, group, false, pix, avail);
      if (cap >= want || group == kWarps) break;
    }
    cap2 = fit_cap(std::min(maxd, kMaxSmemRow), per * no, kWarps, false, pix, avail);
  } else {
    // as many slots as fit beside the workspace: of rows of up to 352 when
    // weighted (1e5 clustered points, nb = 8: rows beyond 256 took 114 of 400 ms
    // in global scratch; the 3,300 slots left hold all but 0.3% of tetrahedra),
    // longer ones where every slot fits all the same (a clump of 400, nb = 5: 38 ->
    // 25 ms)
    cap = std::min(weighted ? 352 : 256, (maxd + 15) & ~15);
    if (weighted)
      cap = std::max(cap, fit_cap(std::min(maxd, kMaxSmemRow), per * no, kWarps, true, pix, avail));
    // unweighted, groups as above while their workspaces take a quarter at most
    if (!weighted) {
      group = warps_per_hub(mean);
      while (group < kWarps &&
             (kWarps / group) * workspace_bytes(cap, group, sizeof(uint16_t), false, pix) > avail / 4)
        group = group == 1 ? 4 : group * 2;
    }
    room = (int64_t)((avail - launch_smem(0, cap, group, weighted, pix) - 32) / (weighted ? 16 : 4));
    cap2 = cap;
    // variant 8: only 64 shared slots (exercises the global path of the other
    // orbits on any input)
    if (o.variant & 8) room = std::min<int64_t>(room, 64 * 3);
    nh = (int)std::min<int64_t>(no, room / per);
    if (o.variant & 8) nh = std::min(nh, 64);
    if (weighted && parity) {
      probe = !(o.variant & 8);
      even_cells = !probe;
      if (even_cells) a.even_hot = nh;
    }
  }
  // variant 1 sends every hub to the global workspace (exercises it on any
  // input)
  if (o.variant & 1) cap = cap2 = 2;
  // with fewer slots than orbits the orbits are relabelled (most frequent
  // first) and the per-slot results mapped back at the end
  const bool relabel = nh < no || (probe && room < 3 * (int64_t)no);
  unsigned long long* s_even = a.even;
  unsigned long long* s_odd = a.odd;
  unsigned long long* const o_odd = a.odd;  // odd counts in orbit order (caller's or scratch)
  int32_t* d_slot = nullptr;
  const int64_t nl = (int64_t)t->lut.size() / g.nb * (g.nb + 1);
  void* d_ent = sc.alloc_bytes((size_t)nl * (small_ent ? 2 : 4));
  uint8_t* d_chir = sc.alloc<uint8_t>(no);
  unsigned* d_probe = probe ? sc.alloc<unsigned>(2) : nullptr;
  if (!d_ent || !d_chir || (probe && !d_probe)) return GS_ENOMEM;
  unsigned long long* d_sample = nullptr;  // counts of the sample that ranks the orbits
  if (relabel) {
    d_sample = sc.alloc<unsigned long long>(no);
    s_even = sc.alloc<unsigned long long>(no);
    s_odd = parity ? sc.alloc<unsigned long long>(no) : nullptr;
    if (weighted) {
      a.weven = sc.alloc<unsigned long long>(3 * (size_t)no);
      a.wodd = parity ? sc.alloc<unsigned long long>(3 * (size_t)no) : nullptr;
    }
    d_slot = sc.alloc<int32_t>(no);
    if (!s_even || (parity && !s_odd) || (weighted && (!a.weven || (parity && !a.wodd))) ||
        !d_slot || !d_sample)
      return GS_ENOMEM;
    // a call without hubs maps its zeros back by this (in range)
    cudaMemsetAsync(d_slot, 0, sizeof(int32_t) * no, s);
  }
  cudaMemsetAsync(s_even, 0, sizeof(uint64_t) * no, s);
  if (parity) cudaMemsetAsync(s_odd, 0, sizeof(uint64_t) * no, s);
  if (a.weven) cudaMemsetAsync(a.weven, 0, sizeof(unsigned long long) * 3 * no, s);
  if (a.wodd) cudaMemsetAsync(a.wodd, 0, sizeof(unsigned long long) * 3 * no, s);
  if (a.limbs) cudaMemsetAsync(a.limbs, 0, sizeof(unsigned long long) * limb_words, s);
  a.even = s_even;
  a.odd = s_odd;
  a.hot = nh;
  a.ent = d_ent;
  a.chir = d_chir;
  auto entries = [&](const int32_t* slot_of) {
    const int blocks = (int)std::min<int64_t>((nl + 255) / 256, 4096);
    if (small_ent)
      k_entries<uint16_t><<<blocks, 256, 0, s>>>(t->d_lut, nl, g.nb, no, slot_of, (uint16_t*)d_ent,
                                               d_chir);
    else
      k_entries<uint32_t><<<blocks, 256, 0, s>>>(t->d_lut, nl, g.nb, no, slot_of, (uint32_t*)d_ent,
                                               d_chir);
    note_launch();
  };
  entries(nullptr);

  // squared-distance buckets no wider than the narrowest bin (variant 4:
  // binary search instead)
  a.bk_shift = 0;
  a.bk_n = 0;
  if (!(o.variant & 4)) {
    int64_t gap = INT64_MAX;
    for (int b = 0; b < g.nb; ++b)
      gap = std::min(gap, g.edges[b + 1] * g.edges[b + 1] - g.edges[b] * g.edges[b]);
    int sh = 0;
    while (sh < 62 && (int64_t(1) << (sh + 1)) <= gap) ++sh;
    const int64_t top = g.edges[g.nb] * g.edges[g.nb];
    const int64_t nbk = ((top - 1) >> sh) + 1;
    if (gap >= 1 && nbk <= kBucketMax) {
      a.bk_shift = sh;
      a.bk_n = (int)nbk;
    }
  }
  a.gscratch = nullptr;
  a.gscratch_stride = 0;
  a.gcap = maxd;

  auto pick = [&](bool P, bool Wt, bool X, bool variant) {
    return small_ent ? pick4<uint16_t>(P, Wt, X, variant) : pick4<uint32_t>(P, Wt, X, variant);
  };
  auto launch = [&](void (*k)(Args), const Args& la, int grid, size_t smem) -> int {
    allow_shared(k, smem);
    cudaMemsetAsync(la.hub_counter, 0, sizeof(unsigned long long), s);
    k<<<grid, kThreads, smem, s>>>(la);
    note_launch();
    return cuda_status(cudaGetLastError());
  };

  // The same over the hubs of la, rows of at most `rows`, in as many launches as
  // the limbs of weighted sums allow.
  double added = 0.0;
  auto fold_limbs = [&]() -> int {
    if (!weighted) return GS_OK;
    k_limbs<<<(int)std::min<int64_t>((no + 255) / 256, 4096), 256, 0, s>>>(
        a.limbs, no, a.chir, a.even, parity ? a.odd : nullptr, a.weven, parity ? a.wodd : nullptr);
    note_launch();
    added = 0.0;
    return cuda_status(cudaGetLastError());
  };
  auto launch_hubs = [&](void (*k)(Args), const Args& la, int grid, size_t smem, int rows) -> int {
    if (!weighted) return launch(k, la, grid, smem);
    const double hub = std::max(1.0, (double)rows * (rows - 1.0) * (rows - 2.0) / 6.0);
    const int64_t n = la.list ? la.nlist : la.hub_end - la.hub_begin,
                  step = (o.variant & 1024) ? 256  // exercises the split
                                            : std::max<int64_t>(1, (int64_t)(kLimbAdds / hub));
    int ls = GS_OK;
    for (int64_t h = 0; h < n && !ls; h += step) {
      const int64_t m = std::min(step, n - h);
      if (added > 0.0 && (added + (double)m * hub > kLimbAdds || (o.variant & 1024))) ls = fold_limbs();
      Args part = la;
      if (la.list) {
        part.list = la.list + h;
        part.nlist = m;
      } else {
        part.hub_begin = la.hub_begin + h;
        part.hub_end = part.hub_begin + m;
      }
      added += (double)m * hub;
      if (!ls) ls = launch(k, part, grid, smem);
    }
    return ls;
  };

  // Weighted parity: even-only cells take instructions and room from the others,
  // worth it when more than one volume in 64 is zero (planes, meshes, pixels);
  // such a tetrahedron costs a global 192-bit sum otherwise. A third of the room,
  // or three quarters where most volumes are zero. 2e4 points in a plane, nb = 8:
  // 166 ms against 691 without.
  auto probe_zero = [&](const Args& wa) -> int {
    unsigned h[2] = {0, 0};
    cudaMemsetAsync(d_probe, 0, sizeof(h), s);
    k_zero_volumes<<<64, 256, 0, s>>>(wa, pix ? 1 : 0, d_probe);
    note_launch();
    cudaMemcpyAsync(h, d_probe, sizeof(h), cudaMemcpyDeviceToHost, s);
    const cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_status(e);
    if (64ull * h[0] > h[1]) {
      even_cells = true;
      a.even_hot = (int)std::min<int64_t>(no, 2ull * h[0] > h[1] ? room * 3 / 4 : room / 3);
      nh = (int)std::min<int64_t>(no, (room - a.even_hot) / 2);
    }
    return cuda_status(cudaGetLastError());
  };

  // Relabelling: count the tetrahedra of every orbit over an evenly strided
  // sample of about 2048 hubs of the first window (at most a quarter of them;
  // unweighted, all slots in shared memory, long rows skipped), rank the orbits by that count and
  // give the top nh the shared slots. Where that count kernel does not fit,
  // the orbits keep their order. The choice changes only the speed.
  auto relabel_orbits = [&](const Args& wa) -> int {
    std::vector<int32_t> slot_of(no);
    std::vector<int32_t> order(no);
    for (int k = 0; k < no; ++k) order[k] = k;
    const int cap_s = fit_cap(std::min(maxd, 256), no, kWarps, false, false, avail);
    if (nh < no && cap_s >= 16) {
      cudaMemsetAsync(d_sample, 0, sizeof(unsigned long long) * no, s);
      Args sa = wa;
      sa.group = kWarps;
      sa.cap = cap_s;
      sa.dmax = cap_s;
      sa.hot = no;
      sa.even_hot = 0;
      sa.even = d_sample;
      sa.odd = nullptr;
      sa.weven = sa.wodd = nullptr;
      sa.W = nullptr;
      sa.hub_stride = std::max<int64_t>(4, (wa.hub_end - wa.hub_begin) / 2048);
      int ls = launch(pick(false, false, false, true), sa, sms,
                      launch_smem(no, cap_s, kWarps, false, false));
      if (ls) return ls;
      std::vector<unsigned long long> cnt(no);
      cudaMemcpyAsync(cnt.data(), d_sample, sizeof(unsigned long long) * no,
                      cudaMemcpyDeviceToHost, s);
      const cudaError_t e = cudaStreamSynchronize(s);
      if (e != cudaSuccess) return cuda_status(e);
      std::stable_sort(order.begin(), order.end(),
                       [&](int x, int y) { return cnt[x] > cnt[y]; });
    }
    for (int k = 0; k < no; ++k) slot_of[order[k]] = k;
    cudaMemcpyAsync(d_slot, slot_of.data(), sizeof(int32_t) * no, cudaMemcpyHostToDevice, s);
    entries(d_slot);
    // the host vector must outlive the (pageable, hence synchronous) copy
    const cudaError_t e = cudaStreamSynchronize(s);
    return e == cudaSuccess ? cuda_status(cudaGetLastError()) : cuda_status(e);
  };

  KernelTimer timer(o.kernel_ms);
  timer.start(s);
  bool first = true;
  std::vector<int64_t> longer;  // hubs of rows beyond cap, their device copy and their CTAs
  int64_t* d_list = nullptr;
  int grid2 = 0;
  bool listed = false;
  const int32_t* deg = nullptr;
  // The hubs of longer rows, in ascending order, and the workspace of those beyond
  // the shared one, for all windows: of as many CTAs as there is memory for. After
  // the first launch, which hides the mapping of new memory (1e5 clustered points,
  // 58 MB, 10 ms).
  auto list_longer = [&]() -> int {
    listed = true;
    int64_t lo = 0, hi = 0;
    const int ls = shard_range(g, o, &lo, &hi);
    if (ls) return ls;
    bool global = false;
    for (int64_t h = lo; h < hi; ++h)
      if (deg[h] > std::max(cap, 2)) {
        longer.push_back(h);
        global = global || deg[h] > cap2;
      }
    if (longer.empty()) return GS_OK;
    d_list = sc.alloc<int64_t>(longer.size());
    if (!d_list) return GS_ENOMEM;
    // (pageable memory: copied out of `longer` when the call returns)
    const cudaError_t e = cudaMemcpyAsync(d_list, longer.data(), sizeof(int64_t) * longer.size(),
                                          cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return cuda_status(e);
    grid2 = (int)std::min<int64_t>(sms, (int64_t)longer.size());
    if (!global) return GS_OK;
    a.gscratch_stride =
        (workspace_bytes(maxd, kWarps, sizeof(uint32_t), weighted, pix) + 255) & ~(size_t)255;
    a.gscratch = staging(sc, a.gscratch_stride, &grid2);
    return a.gscratch ? GS_OK : GS_ENOMEM;
  };
  void (*kern)(Args) = pick(parity, weighted, pix, weighted ? even_cells : all_hot);
  st = for_each_window(g, o, sc, [&](const WinView& v) -> int {
    a.adj = v.adj;
    a.adj_off = v.off1;
    a.split = v.split;
    a.adj_off2 = v.off2;
    a.hub_begin = v.h0;
    a.hub_end = v.h1;
    a.group = group;
    a.cap = cap;
    a.dmax = cap;
    if (first && probe) {
      const int ps = probe_zero(a);
      if (ps) return ps;
      a.hot = nh;
      kern = pick(parity, weighted, pix, even_cells);
    }
    if (first && relabel) {
      const int rs = relabel_orbits(a);
      if (rs) return rs;
    }
    first = false;
    int ls = GS_OK;
    if (cap >= 3)
      ls = launch_hubs(kern, a, sms, launch_smem(per * nh + a.even_hot, cap, group, weighted, pix),
                       cap);
    if (ls || maxd <= cap) return ls;
    // the longer rows
    if (!listed) ls = list_longer();
    if (ls) return ls;
    const int64_t l0 = std::lower_bound(longer.begin(), longer.end(), v.h0) - longer.begin(),
                  l1 = std::lower_bound(longer.begin(), longer.end(), v.h1) - longer.begin();
    if (l0 == l1) return GS_OK;
    Args la = a;
    la.list = d_list + l0;
    la.nlist = l1 - l0;
    la.group = kWarps;
    la.cap = cap2;
    return launch_hubs(kern, la, (int)std::min<int64_t>(grid2, la.nlist),
                       launch_smem(per * nh + a.even_hot, cap2, kWarps, weighted, pix), maxd);
  }, [&]() -> int {
    // (a copy over the stream: not behind the first launch)
    return maxd > cap ? host_deg(g, s, &deg) : GS_OK;
  });
  if (!st) st = fold_limbs();
  if (st) return st;
  if (relabel) {
    auto back = [&](const unsigned long long* src, int words, unsigned long long* dst) {
      const int64_t n = (int64_t)no * words;
      k_slots_to_orbits<<<(int)std::min<int64_t>((n + 255) / 256, 4096), 256, 0, s>>>(src, d_slot,
                                                                                     no, words, dst);
      note_launch();
    };
    back(s_even, 1, reinterpret_cast<unsigned long long*>(d_even));
    if (parity) back(s_odd, 1, o_odd);
    if (weighted) back(a.weven, 3, weven);
    if (weighted && parity) back(a.wodd, 3, wodd);
  }
  timer.stop(s);
  if (d_weven) {
    if (weighted)
      { k_i192_to_double<<<(no + 255) / 256, 256, 0, s>>>(weven, no, 4 * fw->scale, d_weven); note_launch(); }
    else
      { k_u64_to_double<<<(no + 255) / 256, 256, 0, s>>>(reinterpret_cast<unsigned long long*>(d_even), no, d_weven); note_launch(); }
  }
  if (d_wodd && parity) {
    if (weighted)
      { k_i192_to_double<<<(no + 255) / 256, 256, 0, s>>>(wodd, no, 4 * fw->scale, d_wodd); note_launch(); }
    else
      { k_i64_to_double<<<(no + 255) / 256, 256, 0, s>>>(reinterpret_cast<const long long*>(o_odd), no,
                                                       d_wodd); note_launch(); }
  }
  cudaError_t e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_status(e);
  timer.publish();
  return GS_OK;
}

}  // namespace gs
