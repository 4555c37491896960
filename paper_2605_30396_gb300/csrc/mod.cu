// Dictionary update with the codes fixed (Sec. 2.1: alternating minimisation of
// Eq. 1), read as MOD: the least-squares minimiser of sum ||x_i - D alpha_i||^2
// in D, with a small ridge so that unused atoms keep it well posed:
//   G = A A^T, B = X A^T, lambda = 1e-6 trace(G)/K,
//   D~^T = (G + lambda I)^-1 (B + lambda D_old)^T, d_j = d~_j / ||d~_j||,
//   unused atoms refilled with the worst-fit signals.
//
// GPU design (deterministic, no floating-point atomics):
//   1. count_kernel     per-tile atom histograms (integer counts)
//   2. chunk_sum, layout, tile_offsets  per-atom totals, list offsets per
//                       (chunk of tiles, atom) and per (tile, atom), and the
//                       accumulation segments
//   3. scatter_kernel   one CTA per signal tile sorts its entries by atom in
//                       shared memory and writes (signal, coef, nnz) into the
//                       atom-major list in signal order (a counting sort)
//   4. accum_b_kernel, accum_g_kernel  column j of B and row j of G (entries
//                       k >= j; G is symmetric, and its lower triangle is
//                       mirrored from the upper one after the reduction), per
//                       segment of an atom's list; the segments run in signal
//                       order, so that what they gather stays in L2.  Sums are
//                       float-float (exact FMA products, two-sum accumulation:
//                       about FP64 accuracy on the FP32 pipe, since GB300's
//                       FP64 units are slow), added up in a fixed order.
//                       N = 3M, K = 1024, s = 8 (us): one kernel for both,
//                       atom by atom, took 2326; now B 552 (L1 85 % busy,
//                       9 TB/s of L2 reads) and G 726; sort 536 -> 250.
//   5. mixed-precision solve of (G + lambda I) D~^T = (B + lambda D_old)^T:
//      Jacobi scaling S = diag^-1/2 (unit diagonal); one cooperative kernel
//      factors S (G + lambda I) S = L L^T in FP32 and inverts L on the way
//      (right-looking steps over [A | I], one grid barrier per step);
//      each FP32 solve is then two triangular products with W = L^-1, and
//      iterative refinement uses the residual of the scaled system computed
//      in float-float
//   6. normalise, then refill unused atoms (argmax passes over resid_sq)
//
// The same file holds the other reading of the D-step, the approximate K-SVD
// sweep (dlsh_ksvd_update): it reuses the counting sort (1-3, with each
// record's code slot), then runs the atoms in order on one cooperative kernel,
// and refills unused atoms as in 6.
#include <math.h>

#include "common.cuh"
#include "host.hpp"
#include "internal.hpp"

namespace dlsh {
namespace mod {

constexpr int CH = 64;          // counting-sort tiles per chunk
constexpr int SEGG = 8192;      // list entries per accumulation segment of G at most (about half on average)
constexpr int NB = 32;         // Cholesky block
constexpr int RW = 48;         // padded RHS width (45 used)
constexpr int MAX_K = 4096;    // shared-memory G-row partials limit
constexpr int SMEM_LIMIT = 232448;
constexpr double RIDGE_REL = 1e-6;
constexpr int kRefine = 3;     // FP32 solves (two float-float residual corrections)

// The counting sort of the codes by atom, shared by both dictionary updates.
struct Sort {
  int* cnt;         // T x K: entries of each (tile, atom), then their list offsets
  int* csum;        // P x K: entries of each (chunk, atom)
  int* segtot;      // P x ceil(K / 256): first B segment of each (chunk, 256 atoms)
  int* cstart;      // P x K: list offset of each (chunk, atom)
  int* atom_start;  // K + 1
  int* segb_start;  // P x K + 1: first B segment of each (chunk, atom)
  int* segg_start;  // PG x K + 1: first G segment of each (group of gc chunks, atom)
  uint2* list;      // N*s atom-major records: (signal | nnz << 26, coefficient bits)
  int ts, T, P;     // signals per tile, tiles, chunks
  int segb;         // list entries per B segment
  int gc, PG;       // chunks per group of G segments, groups
  int threads;      // of a scatter CTA
  uint32_t sdiv;    // e / s = umulhi(e, sdiv) for e < 65536, s >= 2
};

inline size_t scatter_smem(int K, int s, int ts, int threads);

// Tiles of 1024 signals on 16 warps where they fill the GPU and two CTAs fit an
// SM, else 512 on 8.  (Longer tiles give longer runs of list slots per atom.)
// B segments: enough for 32 warps on every SM, 64 to 1024 entries each.
static void sort_shape(int K, int s, int64_t N, Sort& so) {
  const bool big = N >= 2 * 152 * 1024 && scatter_smem(K, s, 1024, 512) <= 114 * 1024;
  so.ts = big ? 1024 : 512;
  so.threads = big ? 512 : 256;
  so.T = static_cast<int>(N > 0 ? (N + so.ts - 1) / so.ts : 1);
  so.P = (so.T + CH - 1) / CH;
  const int64_t per = N * s / (152 * 32);
  so.segb = static_cast<int>(per < 64 ? 64 : (per > 1024 ? 1024 : per));
  // groups of chunks in which an atom has about SEGG / 2 entries
  const int64_t gc = static_cast<int64_t>(SEGG / 2) * K / (static_cast<int64_t>(s) * CH * so.ts);
  so.gc = static_cast<int>(gc < 1 ? 1 : (gc > so.P ? so.P : gc));
  so.PG = (so.P + so.gc - 1) / so.gc;
  so.sdiv = s >= 2 ? static_cast<uint32_t>((uint64_t(1) << 32) / static_cast<uint64_t>(s) + 1) : 0u;
}
static void carve_sort(Carver& c, int K, int s, int64_t N, Sort& so) {
  sort_shape(K, s, N, so);
  so.cnt = c.take<int>(static_cast<size_t>(K) * so.T);
  so.csum = c.take<int>(static_cast<size_t>(K) * so.P);
  so.segtot = c.take<int>(static_cast<size_t>((K + 255) / 256) * so.P);
  so.cstart = c.take<int>(static_cast<size_t>(K) * so.P);
  so.atom_start = c.take<int>(K + 1);
  so.segb_start = c.take<int>(static_cast<size_t>(K) * so.P + 1);
  so.segg_start = c.take<int>(static_cast<size_t>(K) * so.PG + 1);
  so.list = c.take<uint2>(static_cast<size_t>(N) * s + 1);
}
inline int64_t max_segb(const Sort& so, int K, int s, int64_t N) {
  return N * s / so.segb + static_cast<int64_t>(so.P) * K;
}
inline int64_t max_segg(const Sort& so, int K, int s, int64_t N) {
  return N * s / SEGG + static_cast<int64_t>(so.PG) * K;
}

struct Ws {
  uint32_t* status;
  Sort so;         // the atom-major list
  double* M;       // K x K: G (FP64, entries k >= j of row j)
  double* Z;       // K x RW: B^T
  double* lam;     // [0] lambda
  double* dsc;     // K: Jacobi scale 1 / sqrt(M_jj + lambda)
  float2* S;       // K x K: the scaled matrix, float-float
  float* A32;      // K x K: the same in FP32 (lower), destroyed by the factorisation
  float* Rh32;     // K x K: its right-hand sides
  float* W32;      // K x K: L^-1 (lower)
  float* Yg;       // two 32 x 32 blocks: inverse of the factor's diagonal block
  float* Y32;      // K x RW: W r, between the two triangular products
  unsigned* gbar;  // grid barrier of the factorisation: arrivals
  float2* Zs;      // K x RW: scaled right-hand side
  float2* Xs;      // K x RW: solution of the scaled system
  float* R32;      // K x RW: current residual of the scaled system
  int* dead;       // K
  double* Gp;      // G segments x K partial rows
  double* Bp;      // B segments x RW partial columns
};

static size_t carve(void* base, int K, int s, int64_t N, Ws& w) {
  Carver c(base);
  w.status = c.take<uint32_t>(64);
  carve_sort(c, K, s, N, w.so);
  w.M = c.take<double>(static_cast<size_t>(K) * K);
  w.Z = c.take<double>(static_cast<size_t>(K) * RW);
  w.lam = c.take<double>(4);
  w.dsc = c.take<double>(K);
  w.S = c.take<float2>(static_cast<size_t>(K) * K);
  w.A32 = c.take<float>(static_cast<size_t>(K) * K);
  w.Rh32 = c.take<float>(static_cast<size_t>(K) * K);
  w.Yg = c.take<float>(2 * NB * NB);
  w.W32 = c.take<float>(static_cast<size_t>(K) * K);
  w.Y32 = c.take<float>(static_cast<size_t>(K) * RW);
  w.gbar = c.take<unsigned>(64);
  w.Zs = c.take<float2>(static_cast<size_t>(K) * RW);
  w.Xs = c.take<float2>(static_cast<size_t>(K) * RW);
  w.R32 = c.take<float>(static_cast<size_t>(K) * RW);
  w.dead = c.take<int>(K);
  w.Gp = c.take<double>(static_cast<size_t>(max_segg(w.so, K, s, N)) * K);
  w.Bp = c.take<double>(static_cast<size_t>(max_segb(w.so, K, s, N)) * RW);
  return c.size();
}

// ---- float-float accumulation -------------------------------------------------
// (h, l) += (p, pl), renormalised: about 48 bits.
__device__ __forceinline__ void ff_add(float& h, float& l, float p, float pl) {
  const float s = __fadd_rn(h, p);
  const float v = __fadd_rn(s, -h);
  const float e = __fadd_rn(__fadd_rn(h, -__fadd_rn(s, -v)), __fadd_rn(p, -v));
  const float t = __fadd_rn(e, __fadd_rn(l, pl));
  h = __fadd_rn(s, t);
  l = __fadd_rn(t, -__fadd_rn(h, -s));
}

// The same on pairs of values (Blackwell's packed FP32 instructions: one issue
// slot for two lanes' worth of work).  sub(a, b) = a - b as an FMA by -1, which
// rounds once like the subtraction.
struct f2 {
  uint64_t v;
};
__device__ __forceinline__ f2 f2_make(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2_get(f2 x, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x.v));
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) { return f2_fma(b, f2_make(-1.f, -1.f), a); }
// (h, l) += a x: the product exact as p + pe, h + p by a two-sum whose error and
// pe go to l.  l is renormalised into h by f2_norm (every few hundred steps at
// most: l stays near 2^-24 of the partial sums, so its own rounding errors are
// those of the renormalised form).
__device__ __forceinline__ void f2_acc(f2& h, f2& l, f2 a, f2 na, f2 x) {
  const f2 p = f2_mul(a, x);
  const f2 npe = f2_fma(na, x, p);  // p - a x = -pe, exact
  const f2 s = f2_add(h, p);
  const f2 v = f2_sub(s, h);
  const f2 e = f2_add(f2_sub(h, f2_sub(s, v)), f2_sub(p, v));
  l = f2_sub(f2_add(l, e), npe);
  h = s;
}
__device__ __forceinline__ void f2_norm(f2& h, f2& l) {
  const f2 s = f2_add(h, l);
  const f2 v = f2_sub(s, h);
  l = f2_add(f2_sub(h, f2_sub(s, v)), f2_sub(l, v));
  h = s;
}

// Whether two active lanes of the warp hold the same place: each has read the
// place's value, writes its lane number there and looks whether it is still
// there; the caller then writes the new values.  (match-any answers the same
// but takes about a hundred cycles when the places differ.)
template <class T>
__device__ __forceinline__ bool any_shared(T* place, bool active, T tag) {
  __syncwarp();
  if (active) *place = tag;
  __syncwarp();
  const bool lost = active && *const_cast<volatile T*>(place) != tag;
  return __any_sync(0xffffffffu, lost);
}

// ---- 1. per-tile histograms, cnt[tile][atom] -----------------------------------
// Two 16-bit counters per word (a tile has fewer than 65,536 entries), integer
// atomics in shared memory.
__global__ void __launch_bounds__(256) count_kernel(const uint16_t* idx, const uint8_t* nnz,
                                                   int s, uint32_t sdiv, int64_t N, int K, int ts,
                                                   int* __restrict__ cnt, uint32_t* status) {
  depend();
  extern __shared__ unsigned hist[];  // [(K + 1) / 2]
  const int nw = (K + 1) / 2;
  for (int j = threadIdx.x; j < nw; j += blockDim.x) hist[j] = 0;
  __syncthreads();
  const int64_t i0 = static_cast<int64_t>(blockIdx.x) * ts;
  const int nt = static_cast<int>(N - i0 < ts ? N - i0 : ts);  // signals in this tile
  const uint16_t* tidx = idx + i0 * s;
  bool bad = false;
  auto one = [&](int e, unsigned j) {
    const int q = s == 1 ? e : static_cast<int>(__umulhi(static_cast<uint32_t>(e), sdiv));
    int nz = nnz[i0 + q];
    bad |= nz > s;
    if (e - q * s < nz) {
      if (j < static_cast<unsigned>(K)) atomicAdd(&hist[j >> 1], (j & 1u) ? 65536u : 1u);
      else bad = true;
    }
  };
  const int ne = nt * s;
  int done = 0;
  if ((reinterpret_cast<uintptr_t>(tidx) & 15u) == 0) {  // eight indices per load
    const int nv = ne / 8;
    for (int v = threadIdx.x; v < nv; v += blockDim.x) {
      const uint4 w = reinterpret_cast<const uint4*>(tidx)[v];
      const unsigned u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        one(8 * v + 2 * k, u[k] & 0xffffu);
        one(8 * v + 2 * k + 1, u[k] >> 16);
      }
    }
    done = nv * 8;
  }
  for (int e = done + threadIdx.x; e < ne; e += blockDim.x) one(e, tidx[e]);
  __syncthreads();
  int* row = cnt + static_cast<size_t>(blockIdx.x) * K;
  for (int j = threadIdx.x; j < K; j += blockDim.x) row[j] = (hist[j >> 1] >> (16 * (j & 1))) & 0xffffu;
  if (bad) flag_status(status, ST_BAD_INPUT);
}

// ---- 2. offsets -------------------------------------------------------------------
// Chunks of CH tiles, 256 atoms per CTA.  chunk_sum: entries of each (chunk,
// atom) and how many segments of B (at most segb entries each) its 256 atoms
// need.  layout (one CTA): atom starts, G segments (SEGG entries of one atom),
// and the first B segment of each (chunk, 256 atoms).  tile_offsets: list offset
// of each (tile, atom), in place of its count, and of each (chunk, atom), and
// its first B segment.  Only what needs one CTA runs on one (everything in one
// took 38 us at 46 chunks and 84 at 92: one SM's bandwidth).
// Exclusive prefix over the block (whole warps) and the total; sm: 32 ints.
__device__ __forceinline__ int block_scan(int v, int* sm, int& total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += u;
  }
  if (lane == 31) sm[w] = x;
  __syncthreads();
  int y = lane < static_cast<int>(blockDim.x >> 5) ? sm[lane] : 0;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, y, o);
    if (lane >= o) y += u;
  }
  total = __shfl_sync(0xffffffffu, y, 31);
  const int before = w > 0 ? __shfl_sync(0xffffffffu, y, w - 1) : 0;
  __syncthreads();
  return before + x - v;
}

__global__ void __launch_bounds__(256) chunk_sum_kernel(const int* cnt, int T, int K, int segb,
                                                       int* __restrict__ csum, int* __restrict__ segtot) {
  depend();
  __shared__ int sm[32];
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int t0 = blockIdx.y * CH, t1 = t0 + CH < T ? t0 + CH : T;
  int acc = 0;
  if (j < K) {
#pragma unroll 8
    for (int t = t0; t < t1; ++t) acc += cnt[static_cast<size_t>(t) * K + j];
    csum[static_cast<size_t>(blockIdx.y) * K + j] = acc;
  }
  int all = 0;
  block_scan((acc + segb - 1) / segb, sm, all);
  if (threadIdx.x == 0) segtot[blockIdx.y * gridDim.x + blockIdx.x] = all;
}

__global__ void __launch_bounds__(1024) layout_kernel(const int* csum, int P, int K, int gc, int PG,
                                                      int nseg, int* __restrict__ segtot, int* __restrict__ atom_start,
                                                      int* __restrict__ segg_start, int* __restrict__ segb_end) {
  depend();
  __shared__ int sm[32];
  int carry = 0;
  for (int base = 0; base < K; base += 1024) {
    const int j = base + threadIdx.x;
    int tot = 0;
    if (j < K)
      for (int pg = 0; pg < PG; ++pg) {  // entries per group of chunks, then of the atom
        int g = 0;
        const int p1 = (pg + 1) * gc < P ? (pg + 1) * gc : P;
#pragma unroll 8
        for (int p = pg * gc; p < p1; ++p) g += csum[static_cast<size_t>(p) * K + j];
        segg_start[static_cast<size_t>(pg) * K + j] = (g + SEGG - 1) / SEGG;
        tot += g;
      }
    int all = 0;
    const int st = carry + block_scan(tot, sm, all);
    if (j < K) atom_start[j] = st;
    carry += all;
  }
  auto scan = [&](int* v, int n) {  // exclusive scan in place, the total returned
    int c = 0;
    __syncthreads();
    for (int base = 0; base < n; base += 4096) {  // four consecutive per thread
      const int q = base + 4 * threadIdx.x;
      int x[4], tot = 0, all = 0;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        x[u] = q + u < n ? v[q + u] : 0;
        tot += x[u];
      }
      int st = c + block_scan(tot, sm, all);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (q + u < n) v[q + u] = st;
        st += x[u];
      }
      c += all;
    }
    return c;
  };
  const int nb = scan(segtot, nseg);
  const int ng = scan(segg_start, PG * K);
  if (threadIdx.x == 0) {
    atom_start[K] = carry;
    segg_start[PG * K] = ng;
    *segb_end = nb;
  }
}

__global__ void __launch_bounds__(256) tile_offsets_kernel(int* __restrict__ cnt, int T, int K, int segb,
                                                          const int* csum, const int* segtot,
                                                          const int* atom_start, int* __restrict__ cstart,
                                                          int* __restrict__ segb_start) {
  depend();
  __shared__ int sm[32];
  const int j = blockIdx.x * blockDim.x + threadIdx.x, p = blockIdx.y;
  const int n = j < K ? csum[static_cast<size_t>(p) * K + j] : 0;
  int all = 0;
  const int sb = segtot[p * gridDim.x + blockIdx.x] + block_scan((n + segb - 1) / segb, sm, all);
  if (j >= K) return;
  int run = atom_start[j];
#pragma unroll 8
  for (int q = 0; q < p; ++q) run += csum[static_cast<size_t>(q) * K + j];
  cstart[static_cast<size_t>(p) * K + j] = run;
  segb_start[static_cast<size_t>(p) * K + j] = sb;
  const int t0 = p * CH, t1 = t0 + CH < T ? t0 + CH : T;
  for (int tb = t0; tb < t1; tb += 8) {  // eight loads, then their stores
    int c[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) c[u] = tb + u < t1 ? cnt[static_cast<size_t>(tb + u) * K + j] : 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (tb + u < t1) cnt[static_cast<size_t>(tb + u) * K + j] = run;
      run += c[u];
    }
  }
}

// ---- 3. counting-sort scatter, one CTA per tile, signal order ------------------
// The tile's indices, counts and coefficients are staged in shared memory by
// coalesced loads; its entries are sorted by atom there, and the records then
// leave in sorted order, so that a warp's store covers a few runs of
// consecutive list slots (written straight from signal order, every record was
// a 32-byte L2 write of its own: 397 us at 24M entries against 190).
// Warp w owns a contiguous range of the tile's entries.  Pass 1 counts each atom
// per warp (integer atomics); the counts become per-warp bases in tile order;
// pass 2 ranks each entry among the earlier ones of its atom (warps in order,
// then lanes in order).
// SLOT: the record's upper 6 bits hold the entry's code slot t instead of nnz.
inline size_t scatter_smem(int K, int s, int ts, int threads) {
  const size_t ne = static_cast<size_t>(ts) * s;
  const size_t kp = (static_cast<size_t>(K) + 1) / 2 * 2;
  return ne * 8 + ts + 16 + kp * 2 * (threads / 32) + static_cast<size_t>(K) * 4 + 128;
}
template <bool SLOT>
__global__ void __launch_bounds__(512) scatter_kernel(const uint16_t* idx, const float* coef,
                                                      const uint8_t* nnz, int s, uint32_t sdiv, int64_t N,
                                                      int K, int ts, const int* off,
                                                      uint2* __restrict__ list) {
  depend();
  extern __shared__ __align__(16) uint8_t scb[];
  const int ncap = ts * s;
  const int kp = (K + 1) / 2 * 2;
  const int nthr = blockDim.x, nwarps = nthr >> 5;
  float* scoef = reinterpret_cast<float*>(scb);                             // [ts s]
  uint16_t* sidx = reinterpret_cast<uint16_t*>(scoef + ncap);               // [ts s] atom, 0xFFFF = no entry
  uint16_t* sorted = sidx + ncap;                                           // [ts s] entries by atom
  uint8_t* snz = reinterpret_cast<uint8_t*>(sorted + ncap);                 // [ts]
  int* toff = reinterpret_cast<int*>(scb + (static_cast<size_t>(ncap) * 8 + ts + 15) / 16 * 16);  // [K] list offset - local start
  uint16_t* wc = reinterpret_cast<uint16_t*>(toff + K);                     // [warps][kp] counts, then bases
  __shared__ int wsum[32];
  const int b = blockIdx.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t t0 = static_cast<int64_t>(b) * ts;
  const int nt = static_cast<int>(N - t0 < ts ? N - t0 : ts);  // signals in this tile
  const int ne = nt * s;
  auto div_s = [&](int e) { return s == 1 ? e : static_cast<int>(__umulhi(static_cast<uint32_t>(e), sdiv)); };
  for (int q = tid; q < nt; q += nthr) snz[q] = nnz[t0 + q];
  for (int j = tid; j < kp / 2 * nwarps; j += nthr) reinterpret_cast<unsigned*>(wc)[j] = 0u;
  {
    // 16-byte loads where the tile's rows are 16-byte aligned, the rest one by one
    const float* cs = coef + t0 * s;
    int done = 0;
    if ((reinterpret_cast<uintptr_t>(cs) & 15u) == 0) {
      const int nv = ne / 4;
      for (int v = tid; v < nv; v += nthr)
        reinterpret_cast<float4*>(scoef)[v] = reinterpret_cast<const float4*>(cs)[v];
      done = nv * 4;
    }
    for (int e = done + tid; e < ne; e += nthr) scoef[e] = cs[e];
  }
  __syncthreads();
  {
    const uint16_t* src = idx + t0 * s;
    auto live = [&](int e, unsigned j) -> unsigned {
      const int q = div_s(e);
      return (e - q * s < snz[q] && j < static_cast<unsigned>(K)) ? j : 0xffffu;
    };
    int done = 0;
    if ((reinterpret_cast<uintptr_t>(src) & 15u) == 0) {
      const int nv = ne / 8;
      for (int v = tid; v < nv; v += nthr) {
        const uint4 w = reinterpret_cast<const uint4*>(src)[v];
        unsigned u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int k = 0; k < 4; ++k)
          u[k] = live(8 * v + 2 * k, u[k] & 0xffffu) | live(8 * v + 2 * k + 1, u[k] >> 16) << 16;
        reinterpret_cast<uint4*>(sidx)[v] = make_uint4(u[0], u[1], u[2], u[3]);
      }
      done = nv * 8;
    }
    for (int e = done + tid; e < ne; e += nthr) sidx[e] = static_cast<uint16_t>(live(e, src[e]));
  }
  __syncthreads();
  // the warp's entries, a multiple of 32 but for the last warp's
  const int per = (ne + 32 * nwarps - 1) / (32 * nwarps) * 32;
  const int e0 = warp * per < ne ? warp * per : ne;
  const int e1 = e0 + per < ne ? e0 + per : ne;
  uint16_t* mine = wc + static_cast<size_t>(warp) * kp;
  const unsigned lt = (1u << lane) - 1u;
  // pass 1: counts
  for (int e = e0 + lane; e < e1; e += 32) {
    const unsigned j = sidx[e];
    if (j != 0xffffu) atomicAdd(reinterpret_cast<unsigned*>(mine) + (j >> 1), (j & 1u) ? 65536u : 1u);
  }
  __syncthreads();
  // local starts (atoms in order) and per-warp bases (warps in order)
  int carry = 0;
  for (int base = 0; base < K; base += nthr) {
    const int j = base + tid;
    int tot = 0;
    if (j < K)
      for (int w = 0; w < nwarps; ++w) tot += wc[static_cast<size_t>(w) * kp + j];
    int x = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += u;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    int before = 0, all = 0;
    for (int w = 0; w < nwarps; ++w) {
      if (w < warp) before += wsum[w];
      all += wsum[w];
    }
    __syncthreads();
    if (j < K) {
      int run = carry + before + x - tot;
      toff[j] = off[static_cast<size_t>(b) * K + j] - run;
      for (int w = 0; w < nwarps; ++w) {
        const int c = wc[static_cast<size_t>(w) * kp + j];
        wc[static_cast<size_t>(w) * kp + j] = static_cast<uint16_t>(run);
        run += c;
      }
    }
    carry += all;
  }
  __syncthreads();
  // pass 2: ranks
  for (int eb = e0; eb < e1; eb += 32) {
    const int e = eb + lane;
    const unsigned j = e < e1 ? sidx[e] : 0xffffu;
    const bool on = j != 0xffffu;
    uint16_t* place = mine + (on ? j : 0u);
    unsigned pos = *place;
    bool last = true;
    if (any_shared<uint16_t>(place, on, static_cast<uint16_t>(lane))) {
      const unsigned m = __match_any_sync(0xffffffffu, j);
      pos += __popc(m & lt);
      last = (m >> lane) == 1u;
    }
    if (on) sorted[pos] = static_cast<uint16_t>(e);
    __syncwarp();
    if (on && last) *place = static_cast<uint16_t>(pos + 1);
    __syncwarp();
  }
  __syncthreads();
  // the records in sorted order
  for (int p = tid; p < carry; p += nthr) {
    const int e = sorted[p];
    const int j = sidx[e];
    const int q = div_s(e);
    unsigned f = SLOT ? static_cast<unsigned>(e - q * s) : snz[q];
    if (!SLOT && f > static_cast<unsigned>(s)) f = s;
    list[toff[j] + p] = make_uint2(static_cast<uint32_t>(t0 + q) | (f << 26), __float_as_uint(scoef[e]));
  }
}

// ---- 4a. column j of B: B_j = sum a_ij x_i ---------------------------------------
// One warp per segment (entries of one atom within one chunk of signals), four
// entries at a time: eight lanes take an entry's row, lane l its dimensions l,
// l + 8, .., in packed float-float registers, with the rows of 16 entries in
// flight per warp.  The segments run chunk by chunk, so that the rows of the
// chunks in flight (about 12 MB each) come from HBM once and stay in L2 for the
// s entries that use them (0.7 GB of HBM reads at 3M instead of 5.7).  Bound by
// those L2 gathers (208 bytes of sectors per entry) and the FP32 pipe together.
constexpr int BQ = 6;  // dimensions per lane (48, 45 used)
__global__ void __launch_bounds__(256, 4) accum_b_kernel(const float* __restrict__ X, int K, int P,
                                                        const int* __restrict__ cstart,
                                                        const int* __restrict__ atom_start,
                                                        const int* __restrict__ segb_start, int segb,
                                                        const uint2* __restrict__ list, double* __restrict__ Bp) {
  depend();
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, sub = lane & 7, grp = lane >> 3;
  const int seg = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (seg >= segb_start[P * K]) return;
  // the segment's (chunk, atom): the largest pj with segb_start[pj] <= seg
  int lo = 0, hi = P * K - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (segb_start[mid] <= seg) lo = mid; else hi = mid - 1;
  }
  const int p = lo / K, j = lo - p * K;
  const int q0 = cstart[lo] + (seg - segb_start[lo]) * segb;
  const int end = p + 1 < P ? cstart[lo + K] : atom_start[j + 1];
  const int q1 = q0 + segb < end ? q0 + segb : end;
  const float* Xl = X + sub;
  const int last = sub + 8 * (BQ - 1) < DLSH_D ? 8 * (BQ - 1) : 0;  // offset of the sixth dimension, if any
  f2 h[BQ / 2], l[BQ / 2];
#pragma unroll
  for (int q = 0; q < BQ / 2; ++q) h[q] = l[q] = f2_make(0.f, 0.f);
  constexpr int U = 4;  // steps of four entries whose loads are in flight
  uint2 next = q0 + lane < q1 ? __ldg(list + q0 + lane) : make_uint2(0u, 0u);
  for (int eb = q0; eb < q1; eb += 32) {
    const uint2 rec = next;
    if (eb + 32 + lane < q1) next = __ldg(list + eb + 32 + lane);
    const bool whole = eb + 32 <= q1;
#pragma unroll 1
    for (int i0 = 0; i0 < 8; i0 += U) {
      if (eb + 4 * i0 >= q1) break;
      float x[U][BQ];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int src = 4 * (i0 + u) + grp;
        const unsigned sig = __shfl_sync(FULL, rec.x, src) & 0x3FFFFFFu;
        const float* xr = Xl + static_cast<size_t>(sig) * DLSH_D;
        const bool on = whole || eb + src < q1;  // past the end: x = 0
#pragma unroll
        for (int q = 0; q < BQ; ++q) x[u][q] = on ? __ldg(xr + (q + 1 < BQ ? 8 * q : last)) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float a = __uint_as_float(__shfl_sync(FULL, rec.y, 4 * (i0 + u) + grp));
        const f2 aa = f2_make(a, a), na = f2_make(-a, -a);
#pragma unroll
        for (int q = 0; q < BQ / 2; ++q) f2_acc(h[q], l[q], aa, na, f2_make(x[u][2 * q], x[u][2 * q + 1]));
      }
    }
#pragma unroll
    for (int q = 0; q < BQ / 2; ++q) f2_norm(h[q], l[q]);
  }
  double* out = Bp + static_cast<size_t>(seg) * RW;
#pragma unroll
  for (int q = 0; q < BQ; ++q) {
    float h0, h1, l0, l1;
    f2_get(h[q / 2], h0, h1);
    f2_get(l[q / 2], l0, l1);
    float vh = (q & 1) ? h1 : h0, vl = (q & 1) ? l1 : l0;
#pragma unroll
    for (int o = 8; o < 32; o <<= 1) {
      const float h2 = __shfl_xor_sync(FULL, vh, o), l2 = __shfl_xor_sync(FULL, vl, o);
      ff_add(vh, vl, h2, l2);
    }
    const int d = sub + 8 * q;
    if (grp == 0) out[d] = d < DLSH_D ? static_cast<double>(vh) + static_cast<double>(vl) : 0.0;
  }
}

// ---- 4b. row j of G (entries k >= j; k < j come from row k, mirrored later) --------
// One CTA per segment (entries of one atom within a group of chunks, so that the
// codes gathered meanwhile stay in L2), its warps on fixed slices.  Eight lanes
// take one entry, lane t its code slots t, t + 8, ..: each adds a_ij a_ik into
// the warp's float-float row in shared memory where k > j (the diagonal stays
// in registers).  A signal's atoms are distinct, so two lanes seldom meet on one
// k: any_shared finds out, and then they update it one after the other in lane
// order.
// Bound by the update's shared-memory latency at the warps that the rows leave
// room for (28 per SM at K = 1024).  SG = slots per lane.
template <int SG>
__global__ void __launch_bounds__(128) accum_g_kernel(const uint16_t* __restrict__ idx, const float* __restrict__ coef,
                                                     int s, int K, int P, int gc, int PG,
                                                     const int* __restrict__ cstart, const int* __restrict__ atom_start,
                                                     const int* __restrict__ segg_start,
                                                     const uint2* __restrict__ list, double* __restrict__ Gp) {
  depend();
  extern __shared__ __align__(16) float2 grow[];  // [warps][K] (hi, lo)
  const int seg = blockIdx.x;
  if (seg >= segg_start[PG * K]) return;
  const int nw = blockDim.x >> 5;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned FULL = 0xffffffffu;
  // the segment's (chunk group, atom): the largest pj with segg_start[pj] <= seg
  int lo = 0, hi = PG * K - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (segg_start[mid] <= seg) lo = mid; else hi = mid - 1;
  }
  const int pg = lo / K, j = lo - pg * K;
  float2* row = grow + static_cast<size_t>(warp) * K;
  for (int k = j + lane; k < K; k += 32) row[k] = make_float2(0.f, 0.f);
  __syncwarp();
  const int e0 = cstart[static_cast<size_t>(pg) * gc * K + j] + (seg - segg_start[lo]) * SEGG;
  const int end = (pg + 1) * gc < P ? cstart[static_cast<size_t>(pg + 1) * gc * K + j] : atom_start[j + 1];
  const int len = (e0 + SEGG < end ? e0 + SEGG : end) - e0;
  const int q0 = e0 + static_cast<int>(static_cast<long long>(len) * warp / nw);
  const int q1 = e0 + static_cast<int>(static_cast<long long>(len) * (warp + 1) / nw);
  const int sub = lane & 7, grp = lane >> 3;
  float dh = 0.f, dl = 0.f;  // G[j][j]: each entry's a_ij^2 on the lane that loads its record
  constexpr int U = SG == 1 ? 4 : 2;  // steps of four entries whose codes are in flight
  // record of lane's entry in a block of 32, the next block's loaded ahead
  uint2 next = q0 + lane < q1 ? __ldg(list + q0 + lane) : make_uint2(0u, 0u);
  for (int eb = q0; eb < q1; eb += 32) {
    const uint2 rec = next;
    next = eb + 32 + lane < q1 ? __ldg(list + eb + 32 + lane) : make_uint2(0u, 0u);
    {
      const float a = __uint_as_float(rec.y);
      const float ph = __fmul_rn(a, a);
      if (eb + lane < q1) ff_add(dh, dl, ph, __fmaf_rn(a, a, -ph));
    }
#pragma unroll 1
    for (int i0 = 0; i0 < 8; i0 += U) {
      if (eb + 4 * i0 >= q1) break;
      int kk[U][SG];
      float cc[U][SG], aa[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int src = 4 * (i0 + u) + grp;
        const unsigned rx = __shfl_sync(FULL, rec.x, src);
        aa[u] = __uint_as_float(__shfl_sync(FULL, rec.y, src));
        const int nz = eb + src < q1 ? static_cast<int>(rx >> 26) : 0;
        const size_t c0 = static_cast<size_t>(rx & 0x3FFFFFFu) * s + sub;
#pragma unroll
        for (int g = 0; g < SG; ++g) {
          const bool on = sub + 8 * g < nz;
          kk[u][g] = on ? static_cast<int>(__ldg(idx + c0 + 8 * g)) : -1;
          cc[u][g] = on ? __ldg(coef + c0 + 8 * g) : 0.f;
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        int selves = 0;  // slots that hold atom j, over the step's entries
#pragma unroll
        for (int g = 0; g < SG; ++g) {
          const int k = kk[u][g];
          const float ph = __fmul_rn(aa[u], cc[u][g]);
          const float pl = __fmaf_rn(aa[u], cc[u][g], -ph);
          const bool upd = k > j && k < K;
          float2* place = row + (upd ? k : j);
          float2 r = *place;
          const bool shared = any_shared<float>(&place->x, upd, __int_as_float(lane));
          ff_add(r.x, r.y, ph, pl);
          if (!shared) {
            if (upd) *place = r;
          } else {  // lanes that share a k, in lane order
            const unsigned peers = __match_any_sync(FULL, upd ? k : -1 - lane);
            const int rank = upd ? __popc(peers & ((1u << lane) - 1u)) : 0;
            const int most = __reduce_max_sync(FULL, rank);
            if (upd && rank == 0) *place = r;
            for (int q = 1; q <= most; ++q) {
              __syncwarp();
              if (upd && rank == q) {
                r = *place;
                ff_add(r.x, r.y, ph, pl);
                *place = r;
              }
            }
          }
          __syncwarp();
          selves += __popc(__ballot_sync(FULL, k == j));
        }
        // a code that names atom j more than once: the other slots' a_ij a_ij'
        const int here = q1 - eb - 4 * (i0 + u);  // entries of this step
        if (selves != (here < 4 ? (here > 0 ? here : 0) : 4)) {
#pragma unroll
          for (int g = 0; g < SG; ++g)
            if (kk[u][g] == j) {
              const float ph = __fmul_rn(aa[u], cc[u][g]);
              ff_add(dh, dl, ph, __fmaf_rn(aa[u], cc[u][g], -ph));
            }
          if (sub == 0 && grp < here) {  // its own square is counted already
            const float ph = __fmul_rn(-aa[u], aa[u]);
            ff_add(dh, dl, ph, __fmaf_rn(-aa[u], aa[u], -ph));
          }
        }
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float h2 = __shfl_xor_sync(FULL, dh, o);
    const float l2 = __shfl_xor_sync(FULL, dl, o);
    ff_add(dh, dl, h2, l2);
  }
  if (lane == 0) row[j] = make_float2(dh, dl);
  // the warps' rows in order, one conversion to FP64 per atom
  __syncthreads();
  for (int k = j + threadIdx.x; k < K; k += blockDim.x) {
    float2 r = grow[k];
    for (int w = 1; w < nw; ++w) {
      const float2 o = grow[static_cast<size_t>(w) * K + k];
      ff_add(r.x, r.y, o.x, o.y);
    }
    Gp[static_cast<size_t>(seg) * K + k] = static_cast<double>(r.x) + static_cast<double>(r.y);
  }
}

// Row j of G (entries k >= j) and column j of B: the atom's segment partials
// summed in order, chunk (group) by chunk (group).
__global__ void __launch_bounds__(256) seg_reduce_kernel(const int* segg_start, const int* segb_start,
                                                        const double* Gp, const double* Bp,
                                                        int K, int P, int PG, double* __restrict__ M,
                                                        double* __restrict__ Z) {
  depend();
  const int j = blockIdx.x;
  for (int k = j + threadIdx.x; k < K; k += blockDim.x) {
    double acc = 0.0;
#pragma unroll 4
    for (int p = 0; p < PG; ++p) {
      const int g0 = segg_start[static_cast<size_t>(p) * K + j], g1 = segg_start[static_cast<size_t>(p) * K + j + 1];
      for (int sg = g0; sg < g1; ++sg) acc += Gp[static_cast<size_t>(sg) * K + k];
    }
    M[static_cast<size_t>(j) * K + k] = acc;
  }
  // B: four groups of threads take every fourth chunk, summed in group order
  __shared__ double red[4][RW];
  const int g = threadIdx.x >> 6, q = threadIdx.x & 63;
  if (q < RW) {
    double acc = 0.0;
    for (int p = g; p < P; p += 4)
      for (int sg = segb_start[static_cast<size_t>(p) * K + j]; sg < segb_start[static_cast<size_t>(p) * K + j + 1]; ++sg)
        acc += Bp[static_cast<size_t>(sg) * RW + q];
    red[g][q] = acc;
  }
  __syncthreads();
  if (threadIdx.x < RW) {
    const int t = threadIdx.x;
    Z[static_cast<size_t>(j) * RW + t] = ((red[0][t] + red[1][t]) + red[2][t]) + red[3][t];
  }
}

static int accum_warps(int K, size_t* smem) {
  for (int nw = 4; nw >= 1; --nw) {
    const size_t b = static_cast<size_t>(nw) * K * sizeof(float2);
    if (b <= static_cast<size_t>(SMEM_LIMIT)) {
      *smem = b;
      return nw;
    }
  }
  return 0;
}

// ---- 5a. lambda = 1e-6 trace(G)/K and the Jacobi scale 1 / sqrt(M_jj + lambda) ----
__global__ void __launch_bounds__(1024) ridge_kernel(const double* M, int K, double* lam_out,
                                                     double* __restrict__ dsc) {
  depend();
  __shared__ double part[1024];
  double acc = 0.0;
  for (int j = threadIdx.x; j < K; j += blockDim.x) acc += M[static_cast<size_t>(j) * K + j];
  part[threadIdx.x] = acc;
  __syncthreads();
  for (int w = 512; w > 0; w >>= 1) {  // fixed-order tree (blockDim.x = 1024)
    if (static_cast<int>(threadIdx.x) < w) part[threadIdx.x] += part[threadIdx.x + w];
    __syncthreads();
  }
  const double tr = part[0];
  const double lam = tr > 0.0 ? RIDGE_REL * tr / K : RIDGE_REL;
  if (threadIdx.x == 0) *lam_out = lam;
  for (int j = threadIdx.x; j < K; j += blockDim.x) dsc[j] = 1.0 / sqrt(M[static_cast<size_t>(j) * K + j] + lam);
}

// ---- 5b. the scaled system: S = diag(d) (M + lambda I) diag(d) from M's upper
// triangle (row j of G holds the entries k >= j), whole, as float-float pairs for
// the residuals, and its lower triangle in FP32 for the factorisation; right-hand
// side Zs = d (Z + lambda D_old).  One CTA per 32 x 32 tile on or above the
// diagonal, its mirror image written through shared memory.  S has a unit
// diagonal, which keeps the FP32 factorisation well scaled.
__device__ __forceinline__ float2 ff_split(double x) {
  const float h = static_cast<float>(x);
  return make_float2(h, static_cast<float>(x - static_cast<double>(h)));
}
constexpr int MT = 32;
__global__ void __launch_bounds__(MT * 8) scale_kernel(const double* M, const double* Z,
                                                       const float* D_old,
                                                       const double* lamp,
                                                       const double* dsc, int K, float2* __restrict__ S,
                                                       float* __restrict__ A, float2* __restrict__ Zs,
                                                       float* __restrict__ R32, float2* __restrict__ Xs) {
  depend();
  __shared__ float2 t[MT][MT + 1];
  const int rb = blockIdx.y, cb = blockIdx.x;  // tile: rows rb, columns cb >= rb
  if (cb < rb) return;
  const double lam = *lamp;
  const int x = threadIdx.x % MT, y0 = threadIdx.x / MT;
  for (int y = y0; y < MT; y += 8) {
    const int r = rb * MT + y, c = cb * MT + x;
    float2 v = make_float2(0.f, 0.f);
    if (r < K && c < K && r <= c) {
      const double m = M[static_cast<size_t>(r) * K + c] + (r == c ? lam : 0.0);
      v = ff_split(dsc[c] * m * dsc[r]);
      S[static_cast<size_t>(r) * K + c] = v;
    }
    t[y][x] = v;
  }
  __syncthreads();
  for (int y = y0; y < MT; y += 8) {
    const int r = cb * MT + y, c = rb * MT + x;
    if (r < K && c < K && r >= c) {
      const float2 v = t[x][y];
      if (r > c) S[static_cast<size_t>(r) * K + c] = v;
      A[static_cast<size_t>(r) * K + c] = v.x;
    }
  }
  if (rb == cb)
    for (int f = threadIdx.x; f < MT * RW; f += MT * 8) {
      const int r = rb * MT + f / RW, c = f % RW;
      if (r >= K) break;
      const size_t o = static_cast<size_t>(r) * RW + c;
      const double z =
          c < DLSH_D ? dsc[r] * (Z[o] + lam * static_cast<double>(D_old[static_cast<size_t>(r) * DLSH_D + c])) : 0.0;
      Zs[o] = ff_split(z);
      R32[o] = static_cast<float>(z);
      Xs[o] = make_float2(0.f, 0.f);
    }
}

// ---- 5c. W = L^-1 of the FP32 Cholesky factor of A = L L^T -------------------------
// One cooperative launch (every CTA resident) walks the 32-column steps of a
// right-looking factorisation of the augmented matrix [A | I]; a step needs only
// Y_k = L_kk^-1, so that one grid barrier per step is enough:
//   every CTA but 0  takes 64 x 64 tiles of the trailing matrix and of the
//            right-hand sides, forms the panels it needs itself (P = A_ik Y_k^T,
//            V = Y_k R_k) and applies A_ij -= P_i P_j^T and R_i -= P_i V; V is
//            the finished row block of W
//   CTA 0    meanwhile updates the next diagonal block, factors and inverts it
//            and publishes Y_(k+1) before the barrier
// L itself is not stored: every later solve is two triangular products with W.
// Bound by the chain of CTA 0 and the barrier, 8 us a step (K = 1024: 32 steps,
// 638 -> 253 us).  With the panel and the update as two phases, two barriers and the
// block factored by every CTA before the panel, a step took 20 us.
constexpr int CH_T = 256;   // threads per CTA
constexpr int CH_TILE = 64;

// The CTA inverts the factor of the 32 x 32 block B (symmetric, both triangles;
// rows past the matrix padded with the identity): Y = L^-1, zeros above the
// diagonal.  Thread (i, g) = (tid / 8, tid % 8) holds columns 4 g .. 4 g + 3 of
// row i of [B | I], where column c of the right half takes the place of column c
// of the left half once that is eliminated.  Per column, row c goes through
// shared memory (buf, two rows in turn) and every other row i > c subtracts
// b_ci / b_cc of it; by symmetry row c holds column c too.  Row i is scaled by
// b_ii^-1/2 at the end.  About 120 cycles per column: one barrier, one
// shared-memory read, one hardware reciprocal (the refinement of the solve
// absorbs its last-bit error).  (One warp with the rows in registers and
// shuffles took 340 to 500 cycles per column.)
__device__ __forceinline__ bool factor_diag(const float (*B)[NB + 1], float (*Y)[NB + 1], float (*buf)[NB]) {
  const int i = threadIdx.x >> 3, g = threadIdx.x & 7;
  float a[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) a[m] = B[i][4 * g + m];
  bool bad = false;
  float di = 1.f;  // the row's own pivot
#pragma unroll 1
  for (int c4 = 0; c4 < NB; c4 += 4) {
#pragma unroll
    for (int cc = 0; cc < 4; ++cc) {
      const int c = c4 + cc;
      float* row = buf[cc & 1];
      if (i == c) *reinterpret_cast<float4*>(row + 4 * g) = make_float4(a[0], a[1], a[2], a[3]);
      __syncthreads();
      float d = row[c];
      const float bi = row[i];
      const float4 v = *reinterpret_cast<const float4*>(row + 4 * g);
      if (!(d > 0.f)) {
        bad = true;
        d = 1e-30f;
      }
      const float f = i > c ? -bi * __fdividef(1.f, d) : 0.f;
      di = i == c ? d : di;
      const bool own = 4 * g == c4;  // this thread holds column c: its right half begins
      const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        if (m == cc && own) a[m] = i == c ? 1.f : (i > c ? f : 0.f);
        else a[m] = fmaf(f, x[m], a[m]);
      }
    }
  }
  const float r = rsqrtf(di);
#pragma unroll
  for (int m = 0; m < 4; ++m) Y[i][4 * g + m] = 4 * g + m <= i ? a[m] * r : 0.f;
  return bad;
}

// The 64 x nb panel rows [r0, r0 + 64) of A's columns [k0, k0 + nb), transposed.
__device__ __forceinline__ void stage_panel(const float* __restrict__ A, int K, int r0, int k0, int nb,
                                            float (*raw)[CH_TILE + 1]) {
#pragma unroll
  for (int u = 0; u < CH_TILE * NB / CH_T; ++u) {
    const int f = threadIdx.x + u * CH_T, r = f / NB, q = f % NB;
    raw[q][r] = (r0 + r < K && q < nb) ? A[static_cast<size_t>(r0 + r) * K + k0 + q] : 0.f;
  }
}

// Pt[c][r] = sum_q Y[c][q] raw[q][r]: 32 x 64.
__device__ __forceinline__ void times_y(const float (*Y)[NB + 1], const float (*raw)[CH_TILE + 1],
                                        float (*Pt)[CH_TILE + 1]) {
  const int tr = threadIdx.x % 16, tc = threadIdx.x / 16;  // columns tr + 16 i, rows tc, tc + 16
  float acc[2][4] = {};
#pragma unroll 8
  for (int q = 0; q < NB; ++q) {
    const float y0 = Y[tc][q], y1 = Y[tc + 16][q];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float v = raw[q][tr + 16 * i];
      acc[0][i] = fmaf(v, y0, acc[0][i]);
      acc[1][i] = fmaf(v, y1, acc[1][i]);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    Pt[tc][tr + 16 * i] = acc[0][i];
    Pt[tc + 16][tr + 16 * i] = acc[1][i];
  }
}

// v[i][j] -= sum_q Pt[q][r] Qt[q][c] at r = tid / 16 + 16 i, c = tid % 16 + 16 j.  The
// products are summed by themselves and subtracted at once: they are small beside
// what is left of a nearly singular matrix's diagonal, which one rounding per step
// of 32 keeps and 32 would not (condition 6e4, K = 1024: the refined solution 2.6e-8
// off against 2.0e-7).
__device__ __forceinline__ void tile_product(const float (*Pt)[CH_TILE + 1], const float (*Qt)[CH_TILE + 1],
                                             float (&v)[4][4]) {
  const int tr = threadIdx.x / 16, tc = threadIdx.x % 16;
  float acc[4][4] = {};
#pragma unroll 8
  for (int q = 0; q < NB; ++q) {
    float pi[4], qj[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) pi[i] = Pt[q][tr + 16 * i];
#pragma unroll
    for (int j = 0; j < 4; ++j) qj[j] = Qt[q][tc + 16 * j];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(pi[i], qj[j], acc[i][j]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) v[i][j] -= acc[i][j];
}

// A: the matrix (lower, destroyed).  R: K x K scratch, the right-hand sides below
// the current step.  Yg: two 32 x 32 blocks, Y of the even and odd steps.
__global__ void __launch_bounds__(CH_T) chol_inv_kernel(float* __restrict__ A, float* __restrict__ R,
                                                        float* __restrict__ W, float* __restrict__ Yg, int K,
                                                        unsigned* __restrict__ bar, uint32_t* __restrict__ status,
                                                        long long budget) {
  __shared__ float Y[NB][NB + 1];
  __shared__ float Dg[NB][NB + 1];
  __shared__ __align__(16) float buf[2][NB];
  __shared__ float raw[2][NB][CH_TILE + 1];
  __shared__ float Pt[NB][CH_TILE + 1];
  __shared__ float Qt[NB][CH_TILE + 1];
  const int tid = threadIdx.x;
  const int nblk = (K + NB - 1) / NB;
  unsigned arrived = 0;  // barriers passed
  // CTA 0: the diagonal block in Dg -> Y, published for step kb
  auto publish = [&](int kb) {
    __syncthreads();
    if (factor_diag(Dg, Y, buf) && tid == 0) flag_status(status, ST_BAD_INPUT);
    __syncthreads();
    for (int f = tid; f < NB * NB; f += CH_T) Yg[(kb & 1) * NB * NB + f] = Y[f / NB][f % NB];
  };
  // entry (r, c) of the diagonal block at k0 (c <= r), identity past the matrix
  auto diag_at = [&](int r, int c, int k0) {
    return (k0 + r < K && k0 + c < K) ? A[static_cast<size_t>(k0 + r) * K + k0 + c] : (r == c ? 1.f : 0.f);
  };
  if (blockIdx.x == 0) {
    for (int f = tid; f < NB * NB; f += CH_T) {
      const int r = f / NB, c = f % NB;
      Dg[r][c] = c <= r ? diag_at(r, c, 0) : diag_at(c, r, 0);
    }
    publish(0);
  }
  if (!grid_barrier_count(bar, ++arrived, budget, status)) return;
  for (int kb = 0; kb < nblk; ++kb) {
    const int k0 = kb * NB, nb = K - k0 < NB ? K - k0 : NB, k1 = k0 + nb;
    for (int f = tid; f < NB * NB; f += CH_T) Y[f / NB][f % NB] = Yg[(kb & 1) * NB * NB + f];
    const int rest = K - k1;  // > 0 only when nb = NB (a partial block is the last)
    if (blockIdx.x == 0 && rest > 0) {
      // the next diagonal block: D - P P^T over its 32 rows
      float dv[NB * NB / CH_T];
#pragma unroll
      for (int u = 0; u < NB * NB / CH_T; ++u) {
        const int f = tid + u * CH_T, r = f / NB, c = f % NB;
        dv[u] = c <= r ? diag_at(r, c, k1) : diag_at(c, r, k1);
      }
      stage_panel(A, K, k1, k0, nb, raw[0]);
      __syncthreads();
      times_y(Y, raw[0], Pt);
      __syncthreads();
#pragma unroll
      for (int u = 0; u < NB * NB / CH_T; ++u) {
        const int f = tid + u * CH_T, r = f / NB, c = f % NB;
        float acc = 0.f;
#pragma unroll
        for (int q = 0; q < NB; ++q) acc = fmaf(Pt[q][r], Pt[q][c], acc);  // rows past the matrix are zero
        Dg[r][c] = dv[u] - acc;
      }
      publish(kb + 1);
      __syncthreads();
      if (gridDim.x == 1)
        for (int f = tid; f < NB * NB; f += CH_T) Y[f / NB][f % NB] = Yg[(kb & 1) * NB * NB + f];
    }
    const int T1 = (rest + CH_TILE - 1) / CH_TILE;
    const int T2 = (k1 + CH_TILE - 1) / CH_TILE;
    const int nsyrk = T1 * (T1 + 1) / 2;
    const int total = nsyrk + (T1 > 0 ? T1 : 1) * T2;
    const int workers = gridDim.x > 1 ? gridDim.x - 1 : 1;
    const int first = gridDim.x > 1 ? static_cast<int>(blockIdx.x) - 1 : 0;
    const int tr = tid / 16, tc = tid % 16;
    if (first >= 0)
      for (int t = first; t < total; t += workers) {
        // the tile's values are loaded first: their latency hides behind the panels
        float acc[4][4];
        __syncthreads();  // Y is there, and the previous tile's panels are consumed
        if (t < nsyrk) {
          int bi = static_cast<int>((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
          while (bi * (bi + 1) / 2 > t) --bi;
          while ((bi + 1) * (bi + 2) / 2 <= t) ++bi;
          const int bj = t - bi * (bi + 1) / 2;
          const int r0 = k1 + bi * CH_TILE, c0 = k1 + bj * CH_TILE;
          // (the next diagonal block is CTA 0's, and is not read again)
          auto mine = [&](int gr, int gc) { return gr < K && gc <= gr && !(gr < k1 + NB && gc < k1 + NB); };
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int gr = r0 + tr + 16 * i, gc = c0 + tc + 16 * j;
              acc[i][j] = mine(gr, gc) ? A[static_cast<size_t>(gr) * K + gc] : 0.f;
            }
          stage_panel(A, K, r0, k0, nb, raw[0]);
          if (bi != bj) stage_panel(A, K, c0, k0, nb, raw[1]);
          __syncthreads();
          times_y(Y, raw[0], Pt);
          if (bi != bj) times_y(Y, raw[1], Qt);
          __syncthreads();
          tile_product(Pt, bi != bj ? Qt : Pt, acc);
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int gr = r0 + tr + 16 * i, gc = c0 + tc + 16 * j;
              if (mine(gr, gc)) A[static_cast<size_t>(gr) * K + gc] = acc[i][j];
            }
        } else {
          const int u = t - nsyrk;
          const int bi = u / T2, bc = u % T2;
          const int r0 = k1 + bi * CH_TILE, c0 = bc * CH_TILE;
          // this step's own columns start from zero
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int gr = r0 + tr + 16 * i, gc = c0 + tc + 16 * j;
              acc[i][j] = gr < K && gc < k0 ? R[static_cast<size_t>(gr) * K + gc] : 0.f;
            }
          // R_k (32 x 64 columns; the identity in its own columns) and the panel
#pragma unroll
          for (int v = 0; v < NB * CH_TILE / CH_T; ++v) {
            const int f = tid + v * CH_T, p = f / CH_TILE, c = f % CH_TILE, gc = c0 + c;
            raw[1][p][c] = (p < nb && gc < k0) ? R[static_cast<size_t>(k0 + p) * K + gc] : (gc == k0 + p ? 1.f : 0.f);
          }
          if (rest > 0) stage_panel(A, K, r0, k0, nb, raw[0]);
          __syncthreads();
          times_y(Y, raw[1], Qt);  // V = Y R_k: the finished rows of W
          if (rest > 0) times_y(Y, raw[0], Pt);
          __syncthreads();
          if (bi == 0)
#pragma unroll
            for (int v = 0; v < NB * CH_TILE / CH_T; ++v) {
              const int f = tid + v * CH_T, q = f / CH_TILE, c = f % CH_TILE;
              if (q < nb && c0 + c < k1) W[static_cast<size_t>(k0 + q) * K + c0 + c] = Qt[q][c];
            }
          if (rest > 0) {
            tile_product(Pt, Qt, acc);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const int gr = r0 + tr + 16 * i, gc = c0 + tc + 16 * j;
                if (gr < K && gc < k1) R[static_cast<size_t>(gr) * K + gc] = acc[i][j];
              }
          }
        }
      }
    if (kb + 1 < nblk && !grid_barrier_count(bar, ++arrived, budget, status)) return;
  }
}

// ---- 5d, 5e. products with the 48-column right-hand sides -------------------------
// Eight output rows per CTA, their matrix entries staged in shared memory, the
// inner index dealt to 16 warps; in a warp lane (row, g) = (lane / 4, lane % 4)
// keeps the row's columns 12 g .. 12 g + 11, and the warps' sums are added in
// order.  K / 8 CTAs: latency and the L2 reads of the right-hand side bound
// them.  At K = 1024 a triangular product takes 15 us and a residual 44 (one warp
// per row with 48 sums per lane: 33 to 46; the residual in FP64: 155 to 190, of
// which its arithmetic alone 80).
constexpr int PR = 8;              // rows per CTA
constexpr int PT = 512;            // threads per CTA
constexpr int PKC = 1024;          // inner indices staged at once
constexpr int PS = PKC + 4;        // row stride of the stage: the rows start on different banks

// FP32 solve of (L L^T) c = r with W = L^-1: y = W r (TRANS = false), then
// c = W^T y and X += c in float-float.  W's upper triangle is zero.
template <bool TRANS>
__global__ void __launch_bounds__(PT) trmm_kernel(const float* W, int K, const float* in,
                                                  float* __restrict__ out, float2* __restrict__ Xs) {
  depend();
  extern __shared__ __align__(16) float psm[];  // [PR][PS], then the warps' sums
  const int j0 = blockIdx.x * PR;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = lane >> 2, c0 = (lane & 3) * 12;
  const int kb = TRANS ? j0 : 0, ke = TRANS ? K : (j0 + PR < K ? j0 + PR : K);
  float acc[12];
#pragma unroll
  for (int c = 0; c < 12; ++c) acc[c] = 0.f;
  for (int k0 = kb; k0 < ke; k0 += PKC) {
    const int kn = ke - k0 < PKC ? ke - k0 : PKC;
    __syncthreads();
    for (int f = threadIdx.x; f < PR * kn; f += PT) {
      const int r = TRANS ? f % PR : f / kn, k = TRANS ? f / PR : f % kn;
      psm[r * PS + k] = j0 + r < K ? (TRANS ? W[static_cast<size_t>(k0 + k) * K + j0 + r]
                                            : W[static_cast<size_t>(j0 + r) * K + k0 + k])
                                   : 0.f;
    }
    __syncthreads();
#pragma unroll 4
    for (int k = warp; k < kn; k += PT / 32) {
      const float w = psm[row * PS + k];
      const float4* v = reinterpret_cast<const float4*>(in + static_cast<size_t>(k0 + k) * RW + c0);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const float4 x = v[q];
        acc[4 * q] = fmaf(w, x.x, acc[4 * q]);
        acc[4 * q + 1] = fmaf(w, x.y, acc[4 * q + 1]);
        acc[4 * q + 2] = fmaf(w, x.z, acc[4 * q + 2]);
        acc[4 * q + 3] = fmaf(w, x.w, acc[4 * q + 3]);
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < 12; ++c) psm[(warp * PR + row) * RW + c0 + c] = acc[c];
  __syncthreads();
  if (threadIdx.x < PR * RW && j0 + threadIdx.x / RW < K) {
    float sum = 0.f;
#pragma unroll
    for (int w = 0; w < PT / 32; ++w) sum += psm[w * PR * RW + threadIdx.x];
    const size_t o = static_cast<size_t>(j0) * RW + threadIdx.x;
    if (TRANS) {
      float2 x = Xs[o];
      ff_add(x.x, x.y, sum, 0.f);
      Xs[o] = x;
    } else {
      out[o] = sum;
    }
  }
}

// Residual of the scaled system, R = Zs - S X, in float-float (products exact,
// about 48 bits; FP64 runs at 1/64 of the FP32 rate here), as FP32.
__global__ void __launch_bounds__(PT) residual_kernel(const float2* S, int K,
                                                      const float2* Zs, const float2* Xs,
                                                      float* __restrict__ R32) {
  depend();
  extern __shared__ __align__(16) float2 rsm[];  // [PR][PS], then the warps' sums
  const int j0 = blockIdx.x * PR;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = lane >> 2, c0 = (lane & 3) * 12;
  f2 h[6], l[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) h[c] = l[c] = f2_make(0.f, 0.f);
  for (int k0 = 0; k0 < K; k0 += PKC) {
    const int kn = K - k0 < PKC ? K - k0 : PKC;
    __syncthreads();
    for (int f = threadIdx.x; f < PR * kn; f += PT) {
      const int r = f / kn, k = f % kn;
      rsm[r * PS + k] = j0 + r < K ? S[static_cast<size_t>(j0 + r) * K + k0 + k] : make_float2(0.f, 0.f);
    }
    __syncthreads();
#pragma unroll 2
    for (int k = warp; k < kn; k += PT / 32) {
      const float2 m = rsm[row * PS + k];
      const f2 mh = f2_make(m.x, m.x), nmh = f2_make(-m.x, -m.x), ml = f2_make(m.y, m.y);
      const float4* v = reinterpret_cast<const float4*>(Xs + static_cast<size_t>(k0 + k) * RW + c0);
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        const float4 x = v[c];  // (hi, lo) of two columns
        const f2 xh = f2_make(x.x, x.z);
        f2_acc(h[c], l[c], mh, nmh, xh);
        l[c] = f2_fma(mh, f2_make(x.y, x.w), f2_fma(ml, xh, l[c]));
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    f2_norm(h[c], l[c]);
    float h0, h1, l0, l1;
    f2_get(h[c], h0, h1);
    f2_get(l[c], l0, l1);
    rsm[(warp * PR + row) * RW + c0 + 2 * c] = make_float2(h0, l0);
    rsm[(warp * PR + row) * RW + c0 + 2 * c + 1] = make_float2(h1, l1);
  }
  __syncthreads();
  if (threadIdx.x < PR * RW && j0 + threadIdx.x / RW < K) {
    const size_t o = static_cast<size_t>(j0) * RW + threadIdx.x;
    float2 r = Zs[o];
    for (int w = 0; w < PT / 32; ++w) {
      const float2 p = rsm[w * PR * RW + threadIdx.x];
      ff_add(r.x, r.y, -p.x, -p.y);
    }
    R32[o] = r.x;
  }
}
constexpr int PSM32 = PR * PS * 4 > (PT / 32) * PR * RW * 4 ? PR * PS * 4 : (PT / 32) * PR * RW * 4;
constexpr int PSM64 = 2 * PSM32;

// ---- 6a. normalise; mark dead atoms ----------------------------------------------
__global__ void normalise_kernel(const float2* Xs, const double* dsc,
                                 const int* atom_start,
                                 int K, float* __restrict__ D_new, const float* D_old,
                                 int* __restrict__ dead) {
  depend();
  const int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (j >= K) return;
  // D~^T = diag(d) Xs
  const float2 x0 = Xs[static_cast<size_t>(j) * RW + lane];
  const float2 x1 = lane < DLSH_D - 32 ? Xs[static_cast<size_t>(j) * RW + 32 + lane] : make_float2(0.f, 0.f);
  const double z0 = dsc[j] * (static_cast<double>(x0.x) + static_cast<double>(x0.y));
  const double z1 = dsc[j] * (static_cast<double>(x1.x) + static_cast<double>(x1.y));
  double n2 = z0 * z0 + z1 * z1;
  for (int o = 16; o > 0; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
  const bool unused = atom_start[j + 1] == atom_start[j];
  const bool isdead = unused || !(n2 > 0.0);
  if (lane == 0) dead[j] = isdead ? 1 : 0;
  const double inv = isdead ? 0.0 : 1.0 / sqrt(n2);
  float* dr = D_new + static_cast<size_t>(j) * DLSH_D;
  const float* dold = D_old + static_cast<size_t>(j) * DLSH_D;
  dr[lane] = isdead ? dold[lane] : static_cast<float>(z0 * inv);
  if (lane < DLSH_D - 32) dr[32 + lane] = isdead ? dold[32 + lane] : static_cast<float>(z1 * inv);
}

// ---- 6b. refill dead atoms in increasing j with the largest-residual signals -----
// Picks come in the order (resid desc, index asc); each pass takes the best key
// strictly after the previous pick.  Signals with x = 0 are skipped.
__global__ void __launch_bounds__(1024)
    refill_kernel(const float* X, const float* resid, int64_t N, int K,
                  const int* dead, float* __restrict__ D_new) {
  depend();
  __shared__ float bv[1024];
  __shared__ long long bi[1024];
  __shared__ int dl[MAX_K];   // the dead atoms, increasing
  __shared__ int wcount[32];
  __shared__ float prev_v;
  __shared__ long long prev_i;
  __shared__ int found, ndead;
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  if (tid == 0) {
    prev_v = INFINITY;
    prev_i = -1;
    ndead = 0;
  }
  __syncthreads();
  // ordered compaction of the dead flags (one pass of ballots per 1024 atoms)
  for (int base = 0; base < K; base += 1024) {
    const bool d = base + tid < K && dead[base + tid] != 0;
    const unsigned m = __ballot_sync(0xffffffffu, d);
    if (lane == 0) wcount[wp] = __popc(m);
    __syncthreads();
    int before = ndead;
    for (int q = 0; q < wp; ++q) before += wcount[q];
    if (d) dl[before + __popc(m & ((1u << lane) - 1u))] = base + tid;
    __syncthreads();
    if (tid == 0)
      for (int q = 0; q < 32; ++q) ndead += wcount[q];
    __syncthreads();
  }
  for (int t = 0; t < ndead; ++t) {
    const int j = dl[t];
    while (true) {
      const float pv = prev_v;
      const long long pi = prev_i;
      float best = -1.f;
      long long besti = -1;
      for (int64_t i = tid; i < N; i += blockDim.x) {
        const float v = resid[i];
        const bool after = (v < pv) || (v == pv && i > pi);
        if (after && (v > best || (v == best && (besti < 0 || i < besti)))) {
          best = v;
          besti = i;
        }
      }
      bv[tid] = best;
      bi[tid] = besti;
      __syncthreads();
      for (int w = 512; w > 0; w >>= 1) {
        if (tid < w) {
          const float v2 = bv[tid + w];
          const long long i2 = bi[tid + w];
          if (i2 >= 0 && (bi[tid] < 0 || v2 > bv[tid] || (v2 == bv[tid] && i2 < bi[tid]))) {
            bv[tid] = v2;
            bi[tid] = i2;
          }
        }
        __syncthreads();
      }
      const long long pick = bi[0];
      if (pick < 0) {
        if (tid == 0) found = 0;
        __syncthreads();
        break;
      }
      // norm of the picked signal
      if (tid < 32) {
        const float x0 = X[pick * DLSH_D + tid];
        const float x1 = tid < DLSH_D - 32 ? X[pick * DLSH_D + 32 + tid] : 0.f;
        double n2 = static_cast<double>(x0) * x0 + static_cast<double>(x1) * x1;
        for (int o = 16; o > 0; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
        if (n2 > 0.0) {
          const double inv = 1.0 / sqrt(n2);
          D_new[static_cast<size_t>(j) * DLSH_D + tid] = static_cast<float>(x0 * inv);
          if (tid < DLSH_D - 32) D_new[static_cast<size_t>(j) * DLSH_D + 32 + tid] = static_cast<float>(x1 * inv);
        }
        if (tid == 0) {
          found = n2 > 0.0 ? 1 : 2;
          prev_v = bv[0];
          prev_i = pick;
        }
      }
      __syncthreads();
      if (found == 1) break;
    }
    __syncthreads();
    if (found == 0) break;  // no signals left
  }
}

// ---- approximate K-SVD (the alternative D-update) ------------------------------
// A sweep over the atoms in order; atom j and the coefficients that use it are
// refitted with one power step from the current coefficients g (Rubinstein,
// Zibulevsky and Elad, 2008):
//   E = R_w + g d_j^T (R = X - D A, kept current),  d = E^T g / ||E^T g||,
//   g' = E d,  R_w <- E - g' d^T,  d_j <- d,  A[j, w] <- g'.
// R lives in the workspace, rows padded to 48 floats (16-byte loads).  One
// cooperative kernel runs the sweep.  A CTA owns a range of signals (whole tiles
// of the counting sort), so that the rows it reads and writes are its own and
// atom after atom needs no barrier for them; per atom the CTAs only exchange
// their sums of g R_i and g^2:
//   phase 1  sixteen lanes take one entry of the CTA's part of the list (a
//            float4 of its row each); the sums go through shared memory to 16
//            words of 16 bytes, three values and the exchange's number in
//            each, written and read by single 128-bit accesses, so that a
//            word's arrival is its own flag
//   phase 2  every CTA sums all words in the same order, forms d, and updates
//            its rows (up to KS_KEEP passes still in registers), coefficients
//            and, on CTA 0, the atom
// Two sets of words alternate from one exchange to the next (an unused atom has
// none, so they go by the exchanges done, not by the atom's number): a CTA writes
// the words of an exchange only after it has read all of the previous one's, which
// the others write only after they have read the one before, so no word is
// overwritten before its readers are through.  Every sum runs in a fixed order.
// Bound by latency: the row gather, one L2 round trip of the words and the
// reductions, 3.0 us per atom (N = 400k, K = 512, s = 8; with two grid barriers per
// atom and one thread per entry 12.4 us; with the words waited for one after the
// other 3.4).
constexpr int KS_T = 512;          // threads per sweep CTA
constexpr int KS_E = KS_T / 16;    // entries per pass
constexpr int KS_KEEP = 5;         // passes kept in registers between the phases
constexpr int KS_WORDS = 16;       // 16-byte words of a CTA's sums: 45 of g R_i, then g^2
constexpr int RROW = 48;           // residual row stride in floats

struct KsWs {
  uint32_t* status;
  Sort so;         // records carry the entry's code slot
  float* R;        // N x 48 residual (45 used)
  uint4* part;     // 2 x grid x KS_WORDS: the CTAs' sums
  int* dead;
};

constexpr int KS_MAX_GRID = 1024;

static size_t carve_ksvd(void* base, int K, int s, int64_t N, KsWs& w) {
  Carver c(base);
  w.status = c.take<uint32_t>(64);
  carve_sort(c, K, s, N, w.so);
  w.R = c.take<float>(static_cast<size_t>(N) * RROW);
  w.part = c.take<uint4>(static_cast<size_t>(2) * KS_MAX_GRID * KS_WORDS);
  w.dead = c.take<int>(K);
  return c.size();
}

// R = X - D A with the input codes; one warp per signal, lane d owning
// dimensions d and d + 32 (and the zero padding 45..47).
__global__ void __launch_bounds__(256) ksvd_resid_kernel(const float* X, const float* D,
                                                         int K, const uint16_t* idx,
                                                         const float* coef,
                                                         const uint8_t* nnz, int s, int64_t N,
                                                         float* __restrict__ R) {
  depend();
  const int lane = threadIdx.x & 31;
  const int64_t i = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (i >= N) return;
  const bool hi = lane < DLSH_D - 32;
  float r0 = X[i * DLSH_D + lane];
  float r1 = hi ? X[i * DLSH_D + 32 + lane] : 0.f;
  int nz = nnz[i];
  nz = nz > s ? s : nz;
  const int jl = lane < nz ? idx[i * s + lane] : 0;
  const float al = lane < nz ? coef[i * s + lane] : 0.f;
  for (int t = 0; t < nz; ++t) {
    const int j = __shfl_sync(0xffffffffu, jl, t);
    const float a = __shfl_sync(0xffffffffu, al, t);
    if (j >= K) continue;
    const float* dr = D + static_cast<size_t>(j) * DLSH_D;
    r0 = fmaf(-a, dr[lane], r0);
    if (hi) r1 = fmaf(-a, dr[32 + lane], r1);
  }
  R[i * RROW + lane] = r0;
  if (lane < RROW - 32) R[i * RROW + 32 + lane] = r1;
}

__global__ void __launch_bounds__(KS_T, 1) ksvd_sweep_kernel(const int* __restrict__ off, int T,
                                                             const int* __restrict__ atom_start,
                                                             const uint2* __restrict__ list, int K, int s,
                                                             float* __restrict__ coef, const float* __restrict__ D_old,
                                                             float* __restrict__ D_new, float* __restrict__ R,
                                                             uint4* __restrict__ part, int* __restrict__ dead,
                                                             uint32_t* status, long long budget) {
  __shared__ float4 wsum[KS_T / 32][16];
  __shared__ float tsum[KS_T / 32][3 * KS_WORDS];
  __shared__ __align__(16) float dsm[KS_T / 32][RROW];
  const unsigned FULL = 0xffffffffu;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int l = tid & 15, slot = tid >> 4;  // the thread's float4 of a row, its entry in a pass
  const int G = gridDim.x;
  const int t0 = static_cast<int>(static_cast<long long>(T) * blockIdx.x / G);
  const int t1 = static_cast<int>(static_cast<long long>(T) * (blockIdx.x + 1) / G);
  const bool rl = l < RROW / 4;
  // what is read ahead of the next atom: the CTA's range of its list, the
  // thread's first record, and its part of the atom
  auto lo_of = [&](int j) { return off[static_cast<size_t>(t0) * K + j]; };
  auto hi_of = [&](int j) { return t1 < T ? off[static_cast<size_t>(t1) * K + j] : atom_start[j + 1]; };
  auto old_of = [&](int j) {
    const float* d = D_old + static_cast<size_t>(j) * DLSH_D + 4 * l;
    return make_float4(4 * l < DLSH_D ? __ldg(d) : 0.f, 4 * l + 1 < DLSH_D ? __ldg(d + 1) : 0.f,
                       4 * l + 2 < DLSH_D ? __ldg(d + 2) : 0.f, 4 * l + 3 < DLSH_D ? __ldg(d + 3) : 0.f);
  };
  int a0 = atom_start[0], a1 = atom_start[1];
  int lo = lo_of(0), hi = hi_of(0);
  uint2 first = lo + slot < hi ? list[lo + slot] : make_uint2(0u, 0u);
  float4 dj = rl ? old_of(0) : make_float4(0.f, 0.f, 0.f, 0.f);
  unsigned turn = 0;  // exchanges begun, the same in every CTA; the words' tag
  for (int j = 0; j < K; ++j) {
    const bool used = a1 > a0;  // the same decision in every CTA
    const int clo = lo, chi = hi;
    const uint2 rec0 = first;
    const float4 d = dj;
    if (blockIdx.x == 0 && tid == 0) dead[j] = used ? 0 : 1;
    uint2 rec[KS_KEEP];
    float4 r[KS_KEEP];
    if (used) {
      ++turn;
      // ---- phase 1: sum g R_i (lanes 0..11) and g^2 (lane 12) over the CTA's entries
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int p = 0; p < KS_KEEP; ++p) {
        const int e = clo + p * KS_E + slot;
        rec[p] = p == 0 ? rec0 : (e < chi ? __ldg(list + e) : make_uint2(0u, 0u));
      }
#pragma unroll
      for (int p = 0; p < KS_KEEP; ++p) {
        r[p] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (rl && clo + p * KS_E + slot < chi)
          r[p] = __ldcg(reinterpret_cast<const float4*>(R + static_cast<size_t>(rec[p].x & 0x3FFFFFFu) * RROW) + l);
      }
      auto add = [&](float g, float4 x) {
        if (l == RROW / 4) x.x = g;
        v.x = fmaf(g, x.x, v.x);
        v.y = fmaf(g, x.y, v.y);
        v.z = fmaf(g, x.z, v.z);
        v.w = fmaf(g, x.w, v.w);
      };
#pragma unroll
      for (int p = 0; p < KS_KEEP; ++p) add(__uint_as_float(rec[p].y), r[p]);  // no entry: g = 0, r = 0
      for (int e = clo + KS_KEEP * KS_E + slot; e < chi; e += KS_E) {
        const uint2 q = __ldg(list + e);
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (rl) x = __ldcg(reinterpret_cast<const float4*>(R + static_cast<size_t>(q.x & 0x3FFFFFFu) * RROW) + l);
        add(__uint_as_float(q.y), x);
      }
      v.x += __shfl_xor_sync(FULL, v.x, 16);
      v.y += __shfl_xor_sync(FULL, v.y, 16);
      v.z += __shfl_xor_sync(FULL, v.z, 16);
      v.w += __shfl_xor_sync(FULL, v.w, 16);
      if (lane < 16) wsum[warp][lane] = v;
      __syncthreads();
      // the warps' sums in order; word w carries values 3 w .. 3 w + 2 (45 of
      // g R_i, then g^2, which sits at value 48 of wsum)
      if (tid < KS_WORDS) {
        float t3[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const int val = 3 * tid + q < DLSH_D ? 3 * tid + q : (3 * tid + q == DLSH_D ? RROW : RROW + 1);
          float sum = 0.f;
#pragma unroll
          for (int w = 0; w < KS_T / 32; ++w) sum += reinterpret_cast<const float*>(&wsum[w][0])[val];
          t3[q] = sum;
        }
        st_word(part + (static_cast<size_t>(turn & 1u) * G + blockIdx.x) * KS_WORDS + tid, t3[0], t3[1], t3[2], turn);
      }
    }
    // ---- the next atom's reads, while the words travel
    a0 = a1;
    if (j + 1 < K) {
      a1 = atom_start[j + 2 <= K ? j + 2 : K];
      lo = lo_of(j + 1);
      hi = hi_of(j + 1);
      first = lo + slot < hi ? list[lo + slot] : make_uint2(0u, 0u);
      if (rl) dj = old_of(j + 1);
    }
    if (!used) {
      if (blockIdx.x == 0 && warp == 0 && rl && lane < 16) {
        const float x[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (4 * l + q < DLSH_D) D_new[static_cast<size_t>(j) * DLSH_D + 4 * l + q] = x[q];
      }
      continue;
    }
    // ---- every CTA's words, summed CTA by CTA within a slot, then slot by slot
    {
      float t3[3] = {0.f, 0.f, 0.f};
      bool ok = true;
      const uint4* base = part + static_cast<size_t>(turn & 1u) * G * KS_WORDS + (tid & 15);
      constexpr int B = 5;  // words in flight per thread: all of 152 CTAs' in one go
      for (int c0 = slot; c0 < G && ok; c0 += B * KS_E) {
        uint4 w[B];  // zeros past the last CTA
        ok = wait_words(base + static_cast<size_t>(c0) * KS_WORDS, KS_E * KS_WORDS, (G - c0 + KS_E - 1) / KS_E, turn, w,
                        budget, status);
#pragma unroll
        for (int b = 0; b < B; ++b) {
          t3[0] += __uint_as_float(w[b].x);
          t3[1] += __uint_as_float(w[b].y);
          t3[2] += __uint_as_float(w[b].z);
        }
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) t3[q] += __shfl_xor_sync(FULL, t3[q], 16);
      if (lane < 16)
#pragma unroll
        for (int q = 0; q < 3; ++q) tsum[warp][3 * lane + q] = t3[q];
      if (__syncthreads_or(!ok)) return;
    }
    // ---- phase 2, every warp for itself: d = E^T g = sum g R_i + d_j sum g^2
    float u0 = 0.f, u1 = 0.f, gg = 0.f;
#pragma unroll
    for (int w = 0; w < KS_T / 32; ++w) {
      u0 += tsum[w][lane];
      if (lane < RROW - 32) u1 += tsum[w][32 + lane];
      gg += tsum[w][DLSH_D];
    }
    {
      // d_j in the lanes' order (dimension lane and 32 + lane)
      if (lane < 16 && rl) *reinterpret_cast<float4*>(&dsm[warp][4 * l]) = d;
      __syncwarp();
      const float o0 = dsm[warp][lane], o1 = lane < DLSH_D - 32 ? dsm[warp][32 + lane] : 0.f;
      const float v0 = fmaf(o0, gg, u0);
      const float v1 = lane < DLSH_D - 32 ? fmaf(o1, gg, u1) : 0.f;
      float n2 = fmaf(v0, v0, v1 * v1);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) n2 += __shfl_xor_sync(FULL, n2, o);
      const bool zero = !(n2 > 0.f);
      const float inv = zero ? 0.f : rsqrtf(n2);
      u0 = v0 * inv;
      u1 = v1 * inv;
      float dd = fmaf(o0, u0, o1 * u1);  // d_j . d, of the atom as it is rounded
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) dd += __shfl_xor_sync(FULL, dd, o);
      if (blockIdx.x == 0 && warp == 0) {
        float* out = D_new + static_cast<size_t>(j) * DLSH_D;
        out[lane] = zero ? o0 : u0;
        if (lane < DLSH_D - 32) out[32 + lane] = zero ? o1 : u1;
      }
      __syncwarp();
      dsm[warp][lane] = u0;
      if (lane < RROW - 32) dsm[warp][32 + lane] = lane < DLSH_D - 32 ? u1 : 0.f;
      __syncwarp();
      if (!zero) {
        const float4 u = rl ? *reinterpret_cast<const float4*>(&dsm[warp][4 * l]) : make_float4(0.f, 0.f, 0.f, 0.f);
        // E_i . d = R_i . d + g (d_j . d); R_i <- R_i + g d_j - g' d
        auto refit = [&](uint2 q, float4 x, bool on) {
          const float g = __uint_as_float(q.y);
          float e = fmaf(x.x, u.x, fmaf(x.y, u.y, fmaf(x.z, u.z, x.w * u.w)));
#pragma unroll
          for (int o = 8; o > 0; o >>= 1) e += __shfl_xor_sync(FULL, e, o);
          const float gn = fmaf(g, dd, e);
          if (!on) return;
          const size_t i = q.x & 0x3FFFFFFu;
          if (rl) {
            float4 y;
            y.x = fmaf(-gn, u.x, fmaf(g, d.x, x.x));
            y.y = fmaf(-gn, u.y, fmaf(g, d.y, x.y));
            y.z = fmaf(-gn, u.z, fmaf(g, d.z, x.z));
            y.w = fmaf(-gn, u.w, fmaf(g, d.w, x.w));
            __stcg(reinterpret_cast<float4*>(R + i * RROW) + l, y);
          }
          if (l == RROW / 4) coef[i * s + static_cast<int>(q.x >> 26)] = gn;
        };
#pragma unroll
        for (int p = 0; p < KS_KEEP; ++p)
          if (clo + p * KS_E + 2 * warp < chi) refit(rec[p], r[p], clo + p * KS_E + slot < chi);  // uniform per warp
        for (int e = clo + KS_KEEP * KS_E + 2 * warp; e < chi; e += KS_E) {
          const bool on = e + (lane >> 4) < chi;
          const uint2 q = on ? __ldg(list + e + (lane >> 4)) : make_uint2(0u, 0u);
          float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
          if (rl && on) x = __ldcg(reinterpret_cast<const float4*>(R + static_cast<size_t>(q.x & 0x3FFFFFFu) * RROW) + l);
          refit(q, x, on);
        }
      }
    }
    __syncthreads();  // the rows are written before the next atom's phase 1 reads them
  }
}

}  // namespace mod

size_t mod_ws_bytes(int K, int s, int64_t N) {
  mod::Ws w;
  return mod::carve(nullptr, K, s, N, w);
}

namespace mod {
// Enqueues the counting sort: the atom-major list and its offsets.
template <bool SLOT>
static int sort_enqueue(const uint16_t* idx, const float* coef, const uint8_t* nnz, int s, int64_t N, int K,
                        const Sort& so, uint32_t* status, cudaStream_t st, const char* call) {
  if (N > 0) {
    launch_dependent(count_kernel, so.T, 256, (K + 1) / 2 * sizeof(unsigned), st, idx, nnz, s, so.sdiv, N, K, so.ts,
                     so.cnt, status);
  } else {
    DLSH_CUDA_TRY(cudaMemsetAsync(so.cnt, 0, sizeof(int) * K * so.T, st), call);
  }
  const dim3 g((K + 255) / 256, so.P);
  launch_dependent(chunk_sum_kernel, g, 256, 0, st, so.cnt, so.T, K, so.segb, so.csum, so.segtot);
  launch_dependent(layout_kernel, 1, 1024, 0, st, so.csum, so.P, K, so.gc, so.PG, static_cast<int>(g.x * g.y),
                   so.segtot, so.atom_start, so.segg_start, so.segb_start + static_cast<size_t>(so.P) * K);
  launch_dependent(tile_offsets_kernel, g, 256, 0, st, so.cnt, so.T, K, so.segb, so.csum, so.segtot, so.atom_start,
                   so.cstart, so.segb_start);
  count_launches((N > 0 ? 1 : 0) + 3);
  if (N > 0) {
    const size_t smem = scatter_smem(K, s, so.ts, so.threads);
    DLSH_CUDA_TRY(cudaFuncSetAttribute(scatter_kernel<SLOT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       SMEM_LIMIT - 512),
                  call);
    launch_dependent(scatter_kernel<SLOT>, so.T, so.threads, smem, st, idx, coef, nnz, s, so.sdiv, N, K, so.ts,
                     so.cnt, so.list);
    count_launches(1);
  }
  return check_launch(call);
}
}  // namespace mod

// Enqueues one MOD update (no host synchronisation; capturable).
int mod_enqueue(const float* X, int64_t N, int K, const uint16_t* idx, const float* coef,
                const uint8_t* nnz, int s, const float* D_old, const float* resid,
                float* D_new, void* ws, cudaStream_t st, uint32_t** status_out) {
  using namespace mod;
  if (N >= (int64_t(1) << 26))
    return set_error(DLSH_ERR_UNSUPPORTED,
                     "dlsh_mod_update: N must be < 2^26 (the atom lists pack signal and nnz in 32 bits)");
  Ws w;
  carve(ws, K, s, N, w);
  if (status_out) *status_out = w.status;
  size_t acc_smem = 0;
  const int acc_nw = accum_warps(K, &acc_smem);
  if (acc_nw == 0)
    return set_error(DLSH_ERR_UNSUPPORTED, "dlsh_mod_update: K=%d s=%d does not fit", K, s);
  DLSH_CUDA_TRY(cudaMemsetAsync(w.status, 0, sizeof(uint32_t), st), "dlsh_mod_update: reset");
  int launches = 0;
  const Sort& so = w.so;
  const int src = sort_enqueue<false>(idx, coef, nnz, s, N, K, so, w.status, st, "dlsh_mod_update: sort");
  if (src) return src;
  {
    const int64_t nb = (max_segb(so, K, s, N) + 7) / 8;
    // (launched normally: started early, these two lose more than a launch. With
    // accum_b beside the scatter's last CTAs the update of 3M signals takes 2360 us
    // instead of 2040, with accum_g beside accum_b that of 10,000 220 instead of 201)
    accum_b_kernel<<<static_cast<int>(nb > 0 ? nb : 1), 256, 0, st>>>(X, K, so.P, so.cstart, so.atom_start,
                                                                      so.segb_start, so.segb, so.list, w.Bp);
    void (*accum)(const uint16_t*, const float*, int, int, int, int, int, const int*, const int*, const int*,
                  const uint2*, double*) =
        s <= 8 ? accum_g_kernel<1> : (s <= 16 ? accum_g_kernel<2> : accum_g_kernel<4>);
    DLSH_CUDA_TRY(cudaFuncSetAttribute(accum, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(acc_smem)),
                  "dlsh_mod_update: attribute");
    accum<<<static_cast<int>(max_segg(w.so, K, s, N)), acc_nw * 32, acc_smem, st>>>(
        idx, coef, s, K, so.P, so.gc, so.PG, so.cstart, so.atom_start, so.segg_start, so.list, w.Gp);
  }
  launch_dependent(seg_reduce_kernel, K, 256, 0, st, so.segg_start, so.segb_start, w.Gp, w.Bp, K, so.P, so.PG, w.M,
                   w.Z);
  launch_dependent(ridge_kernel, 1, 1024, 0, st, w.M, K, w.lam, w.dsc);
  // mixed-precision solve: FP32 Cholesky of the Jacobi-scaled matrix, then
  // kRefine FP32 solves with float-float residuals in between
  {
    const int nb = (K + MT - 1) / MT;
    launch_dependent(scale_kernel, dim3(nb, nb), MT * 8, 0, st, w.M, w.Z, D_old, w.lam, w.dsc, K, w.S, w.A32, w.Zs,
                     w.R32, w.Xs);
  }
  launches += 5;
  {
    static PerDevice<int> coop;
    int coop_grid = 0;
    const int crc = coop.get(&coop_grid, [](int& g) {
      int per_sm = 0;
      DLSH_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, chol_inv_kernel, CH_T, 0),
                    "dlsh_mod_update: occupancy");
      int sms = device_sm_count();
      if (sms <= 0) sms = 1;
      if (per_sm < 1) return set_error(DLSH_ERR_CUDA, "dlsh_mod_update: factorisation kernel does not fit");
      g = sms;  // one CTA per SM: fewer arrivals at each grid barrier
      return DLSH_OK;
    });
    if (crc) return crc;
    DLSH_CUDA_TRY(cudaMemsetAsync(w.gbar, 0, 2 * sizeof(unsigned), st), "dlsh_mod_update: barrier");
    float* A32 = w.A32;
    float* Rh32 = w.Rh32;
    float* W32 = w.W32;
    float* Yg = w.Yg;
    int Kk = K;
    unsigned* gb = w.gbar;
    uint32_t* stw = w.status;
    long long budget = kWaitBudget;
    void* args[] = {&A32, &Rh32, &W32, &Yg, &Kk, &gb, &stw, &budget};
    DLSH_CUDA_TRY(cudaLaunchCooperativeKernel(reinterpret_cast<void*>(chol_inv_kernel), dim3(coop_grid),
                                              dim3(CH_T), args, 0, st),
                  "dlsh_mod_update: factorisation");
    ++launches;
  }
  DLSH_CUDA_TRY(cudaFuncSetAttribute(residual_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, PSM64),
                "dlsh_mod_update: attribute");
  const int rows = (K + PR - 1) / PR;
  for (int it = 0; it < kRefine; ++it) {
    if (it > 0) {
      launch_dependent(residual_kernel, rows, PT, PSM64, st, w.S, K, w.Zs, w.Xs, w.R32);
      ++launches;
    }
    launch_dependent(trmm_kernel<false>, rows, PT, PSM32, st, w.W32, K, w.R32, w.Y32, nullptr);
    launch_dependent(trmm_kernel<true>, rows, PT, PSM32, st, w.W32, K, w.Y32, nullptr, w.Xs);
    launches += 2;
  }
  launch_dependent(normalise_kernel, (K + 7) / 8, 256, 0, st, w.Xs, w.dsc, so.atom_start, K, D_new, D_old, w.dead);
  ++launches;
  if (resid && N > 0) {
    launch_dependent(refill_kernel, 1, 1024, 0, st, X, resid, N, K, w.dead, D_new);
    ++launches;
  }
  count_launches(launches);
  return check_launch("dlsh_mod_update: launch");
}

size_t ksvd_ws_bytes(int K, int s, int64_t N) {
  mod::KsWs w;
  return mod::carve_ksvd(nullptr, K, s, N, w);
}

// Enqueues one approximate K-SVD sweep (no host synchronisation).
int ksvd_enqueue(const float* X, int64_t N, int K, const uint16_t* idx, float* coef, const uint8_t* nnz, int s,
                 const float* D_old, const float* resid, float* D_new, void* ws, cudaStream_t st,
                 uint32_t** status_out) {
  using namespace mod;
  if (N >= (int64_t(1) << 26))
    return set_error(DLSH_ERR_UNSUPPORTED, "dlsh_ksvd_update: N must be < 2^26");
  KsWs w;
  carve_ksvd(ws, K, s, N, w);
  if (status_out) *status_out = w.status;
  DLSH_CUDA_TRY(cudaMemsetAsync(w.status, 0, sizeof(uint32_t), st), "dlsh_ksvd_update: reset");
  int launches = 0;
  const int src = sort_enqueue<true>(idx, coef, nnz, s, N, K, w.so, w.status, st, "dlsh_ksvd_update: sort");
  if (src) return src;
  if (N > 0) {
    launch_dependent(ksvd_resid_kernel, static_cast<int>((N + 7) / 8), 256, 0, st, X, D_old, K, idx, coef, nnz, s, N,
                     w.R);
    launches += 1;
  }
  {
    static PerDevice<int> coop;
    int coop_grid = 0;
    const int crc = coop.get(&coop_grid, [](int& grid) {
      int per_sm = 0;
      int sms = device_sm_count();
      if (sms <= 0) sms = 1;
      DLSH_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ksvd_sweep_kernel, KS_T, 0),
                    "dlsh_ksvd_update: occupancy");
      if (per_sm < 1) return set_error(DLSH_ERR_CUDA, "dlsh_ksvd_update: sweep kernel does not fit");
      grid = sms < KS_MAX_GRID ? sms : KS_MAX_GRID;  // one CTA per SM
      return DLSH_OK;
    });
    if (crc) return crc;
    if (coop_grid > w.so.T) coop_grid = w.so.T;  // each CTA owns at least a tile
    DLSH_CUDA_TRY(cudaMemsetAsync(w.part, 0, sizeof(uint4) * 2 * coop_grid * KS_WORDS, st), "dlsh_ksvd_update: words");
    const int* of = w.so.cnt;
    int T = w.so.T;
    const int* as = w.so.atom_start;
    const uint2* li = w.so.list;
    int Kk = K, ss = s;
    float* cf = coef;
    const float* Do = D_old;
    float* Dn = D_new;
    float* Rr = w.R;
    uint4* pt = w.part;
    int* dd = w.dead;
    uint32_t* stw = w.status;
    long long budget = kWaitBudget;
    void* args[] = {&of, &T, &as, &li, &Kk, &ss, &cf, &Do, &Dn, &Rr, &pt, &dd, &stw, &budget};
    DLSH_CUDA_TRY(cudaLaunchCooperativeKernel(reinterpret_cast<void*>(ksvd_sweep_kernel), dim3(coop_grid),
                                              dim3(KS_T), args, 0, st),
                  "dlsh_ksvd_update: sweep");
    ++launches;
  }
  if (resid && N > 0) {
    launch_dependent(refill_kernel, 1, 1024, 0, st, X, resid, N, K, w.dead, D_new);
    ++launches;
  }
  count_launches(launches);
  return check_launch("dlsh_ksvd_update: launch");
}

}  // namespace dlsh

extern "C" {

size_t dlsh_mod_workspace_size(int K, int d, int s, int64_t N) {
  if (d != DLSH_D || K < 1 || K > dlsh::mod::MAX_K || s < 1 || s > DLSH_MAX_S || N < 0) return 0;
  return dlsh::mod_ws_bytes(K, s, N);
}

int dlsh_mod_update(const float* X, int64_t N, int d, int K, const uint16_t* idx,
                    const float* coef, const uint8_t* nnz, int s, const float* D_old,
                    const float* resid_sq, float* D_new, void* ws, size_t ws_bytes, void* stream,
                    int flags) {
  using namespace dlsh;
  clear_error();
  if (d != DLSH_D) return set_error(DLSH_ERR_UNSUPPORTED, "dlsh_mod_update: d must be 45");
  if (K < 1 || K > mod::MAX_K)
    return set_error(DLSH_ERR_UNSUPPORTED, "dlsh_mod_update: K must be in [1, 4096], got %d", K);
  if (s < 1 || s > DLSH_MAX_S)
    return set_error(DLSH_ERR_UNSUPPORTED, "dlsh_mod_update: s must be in [1, 32]");
  if (N < 0 || N * s >= (1LL << 31))
    return set_error(DLSH_ERR_UNSUPPORTED, "dlsh_mod_update: N*s must be < 2^31");
  if (!D_old || !D_new) return set_error(DLSH_ERR_INVALID_ARG, "dlsh_mod_update: NULL D");
  if (reinterpret_cast<uintptr_t>(idx) % 4 != 0)
    return set_error(DLSH_ERR_INVALID_ARG, "dlsh_mod_update: idx must be 4-byte aligned");
  if (N > 0 && (!X || !idx || !coef || !nnz))
    return set_error(DLSH_ERR_INVALID_ARG, "dlsh_mod_update: NULL array");
  int rc = check_workspace(ws, ws_bytes, mod_ws_bytes(K, s, N), "dlsh_mod_update");
  if (rc) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint32_t* status = nullptr;
  rc = mod_enqueue(X, N, K, idx, coef, nnz, s, D_old, resid_sq, D_new, ws, st, &status);
  if (rc) return rc;
  return finish(st, status, flags, "dlsh_mod_update");
}

size_t dlsh_ksvd_workspace_size(int K, int d, int s, int64_t N) {
  if (d != DLSH_D || K < 1 || K > dlsh::mod::MAX_K || s < 1 || s > DLSH_MAX_S || N < 0) return 0;
  return dlsh::ksvd_ws_bytes(K, s, N);
}

int dlsh_ksvd_update(const float* X, int64_t N, int d, int K, const uint16_t* idx, float* coef,
                     const uint8_t* nnz, int s, const float* D_old, const float* resid_sq, float* D_new,
                     void* ws, size_t ws_bytes, void* stream, int flags) {
  using namespace dlsh;
  clear_error();
  if (d != DLSH_D) return set_error(DLSH_ERR_UNSUPPORTED, "dlsh_ksvd_update: d must be 45");
  if (K < 1 || K > mod::MAX_K)
    return set_error(DLSH_ERR_UNSUPPORTED, "dlsh_ksvd_update: K must be in [1, 4096], got %d", K);
  if (s < 1 || s > DLSH_MAX_S) return set_error(DLSH_ERR_UNSUPPORTED, "dlsh_ksvd_update: s must be in [1, 32]");
  if (N < 0 || N * s >= (1LL << 31))
    return set_error(DLSH_ERR_UNSUPPORTED, "dlsh_ksvd_update: N*s must be < 2^31");
  if (!D_old || !D_new) return set_error(DLSH_ERR_INVALID_ARG, "dlsh_ksvd_update: NULL D");
  if (D_old == D_new) return set_error(DLSH_ERR_INVALID_ARG, "dlsh_ksvd_update: D_new must not alias D_old");
  if (reinterpret_cast<uintptr_t>(idx) % 4 != 0)
    return set_error(DLSH_ERR_INVALID_ARG, "dlsh_ksvd_update: idx must be 4-byte aligned");
  if (N > 0 && (!X || !idx || !coef || !nnz))
    return set_error(DLSH_ERR_INVALID_ARG, "dlsh_ksvd_update: NULL array");
  int rc = check_workspace(ws, ws_bytes, ksvd_ws_bytes(K, s, N), "dlsh_ksvd_update");
  if (rc) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint32_t* status = nullptr;
  rc = ksvd_enqueue(X, N, K, idx, coef, nnz, s, D_old, resid_sq, D_new, ws, st, &status);
  if (rc) return rc;
  return finish(st, status, flags, "dlsh_ksvd_update");
}

}  // extern "C"
