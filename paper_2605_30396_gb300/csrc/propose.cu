// Fused inference of the support-proposal network: for every signal, the m
// atoms with the largest logits of the 45 -> 256 -> 256 -> K GELU MLP, ordered
// by decreasing logit (ties to the smaller atom index), or the logits
// themselves, in one persistent kernel.  Activations never leave the SM.
//
// Per tile of 128 signals (one TMEM lane per signal):
//   epilogue warps  stage the unit-norm BF16 signals as the A operand
//   MMA warp        layer 1 (N = 256, K = 64) into a 256-column TMEM buffer
//   epilogue warps  bias + GELU -> BF16 hidden activations, written over the
//                   A operand in the canonical K-major layout
//   MMA warp        layer 2 (K = 256) into the other TMEM buffer; same epilogue
//   MMA warp        layer 3, 256 atoms per job, TMEM buffers alternating so the
//                   epilogue of one block overlaps the MMAs of the next; in
//                   top-m mode twice, but for two blocks that stay in TMEM
//   epilogue warps  each thread owns one signal and a quarter of every job's
//                   columns (16 warps over the 4 TMEM lane quadrants): 16 of each
//                   64, so that a layer's activations are handed on in four parts
//                   and the next MMAs run beside the rest of the GELUs
//   producer warp   streams the weights, pre-packed into 16 KB operand chunks
//                   in their consumption order, through a 4-stage ring
// The MMAs (M = 128, N = 256, K = 16, FP32 accumulation) take k in the order of
// the layer-by-layer training GEMM and the element-wise steps share its code, so
// the logits agree with it bit for bit.
//
// Top-m (exact, ties to the smaller atom index):
//   pass A  the maxima of 16 interleaved column groups per quarter row; the m-th
//           largest of the row's 64 group maxima is a lower bound T of its
//           m-th largest logit (64 distinct logits reach their group maxima)
//   pass B  only logits >= T are queued (shared memory): about m + m^2/128 per
//           row.  Blocks 0 and 1 come last in pass A and are still in TMEM.
//   rank    a row's queues become one list; a candidate's place is the number of
//           those before it, counted by the row's four threads
//
// What bounds it: instruction issue of the epilogue warps and, in pass A, of the
// single thread that issues the MMAs.  At K = 1024, m = 16 a tile takes 57,000
// cycles: two GELU layers 21,000, pass B 14,000, pass A 15,000 (3500 a block, where
// the tensor pipe needs 2050), ranks 5000.
// 500,001 signals 1235 -> 897 us, m = 32 1760 -> 1357; 10,000 signals at K = 128
// 82 -> 68.  What it took: 16 epilogue warps instead of 8 (1235 -> 1106); biases in
// shared memory, read one job ahead (a miss cost every step of a pass 600 cycles),
// and activations handed on in parts (1042); candidates queued once and ranked
// instead of inserted one by one into a register list of m (897; a lane's insertion
// held up the other 31).  A cluster of two that shares the weights' stream (1000
// beside 987 without) and one pass with T from two blocks (twice the candidates)
// were slower.
#include <cuda_bf16.h>
#include <math.h>

#include "common.cuh"
#include "host.hpp"
#include "internal.hpp"
#include "mlp.cuh"

namespace dlsh {
namespace prop {

using mlp::HID;
using mlp::XIN;

constexpr int TM = 128;                          // signals per tile (MMA M)
constexpr int NC = 256;                          // columns per accumulation job
constexpr int KC = 32;                           // k per operand chunk (two k-steps of 16)
constexpr uint32_t CHUNK_BYTES = NC * KC * 2;    // 16 KB
constexpr int NST = 4;                           // operand ring stages
constexpr int NEPI = 512;                        // epilogue threads (16 warps)
constexpr int NQ = NEPI / TM;                    // threads per signal, a column quarter of each job each
constexpr int QW = NC / NQ;                      // columns of a quarter
constexpr int PARTS = QW / 16;                   // parts in which a layer's activations are handed on
constexpr int NG = 64 / NQ;                      // column groups per quarter (pass A)
constexpr int NTHREADS = NEPI + 64;              // + MMA warp + producer warp
constexpr uint32_t Q_BYTES = 30 * NEPI * 6;      // queues: 21 entries of 8 bytes per thread, or 30 of 6
constexpr int QS = 4;                            // columns between two looks at the queues
constexpr uint32_t A_BYTES = TM * HID * 2;       // 64 KB: X, then H1, then H2
constexpr uint32_t OFF_A = 0;
constexpr uint32_t OFF_Q = OFF_A + A_BYTES;        // queues
constexpr uint32_t OFF_RING = OFF_Q + Q_BYTES;
constexpr uint32_t OFF_BIAS = OFF_RING + NST * CHUNK_BYTES;  // the job's biases, a copy per warp
constexpr uint32_t OFF_T = OFF_BIAS + (NEPI / 32) * QW * 4;  // threshold per signal
constexpr uint32_t OFF_CN = OFF_T + TM * 4;  // candidates of each thread
constexpr uint32_t OFF_BAR = OFF_CN + NEPI;
constexpr uint32_t OFF_OUT = 32768;  // of the ranked atoms, from the queues' start
constexpr uint32_t SMEM_BYTES = OFF_BAR + 256;
static_assert(SMEM_BYTES <= 232448, "shared memory");
static_assert(Q_BYTES >= (64 + 32) * TM * 4, "the queues hold the sorted group maxima");

// Packed weights: W1, then W2, by k-range, then for each 256-atom block j the
// eight k-ranges of W3 rows [256 j, 256 j + 256) (rows past K are zero).  Chunk layout: canonical K-major, no swizzle: element
// (n, k) at byte (k / 8) * (NC * 16) + n * 16 + (k % 8) * 2.
inline int n_blocks(int K) { return (K + NC - 1) / NC; }
constexpr int C1 = XIN / KC, C2 = HID / KC;  // chunks of W1 and of W2 or a block of W3
inline int n_chunks(int K) { return C1 + C2 + C2 * n_blocks(K); }

struct Ws {
  uint32_t* status;
  uint8_t* img;
  float* b1;
  float* b2;
  float* b3;  // padded to whole blocks with -inf
};
inline size_t carve(void* base, int K, Ws& w) {
  Carver c(base);
  w.status = c.take<uint32_t>(64);
  w.img = c.take<uint8_t>(static_cast<size_t>(n_chunks(K)) * CHUNK_BYTES);
  w.b1 = c.take<float>(HID);
  w.b2 = c.take<float>(HID);
  w.b3 = c.take<float>(static_cast<size_t>(n_blocks(K)) * NC);
  return c.size();
}

// One thread per 16-byte unit of the image (8 consecutive k of one row).
__global__ void pack_kernel(const __nv_bfloat16* __restrict__ Pb, const float* __restrict__ P, int K,
                            int nblk, uint8_t* __restrict__ img, float* __restrict__ b1,
                            float* __restrict__ b2, float* __restrict__ b3) {
  const mlp::Layout L = mlp::layout(K);
  const long long u = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  const long long units = static_cast<long long>(C1 + C2 + C2 * nblk) * (CHUNK_BYTES / 16);
  if (u < units) {
    const int c = static_cast<int>(u / (CHUNK_BYTES / 16));
    const int w = static_cast<int>(u % (CHUNK_BYTES / 16));
    const int kb = w / NC, n = w % NC;
    const __nv_bfloat16* src;
    long long row;
    int ld, k0;
    bool valid = true;
    if (c < C1) {
      src = Pb + L.W1;
      ld = XIN;
      row = n;
      k0 = c * KC;
    } else if (c < C1 + C2) {
      src = Pb + L.W2;
      ld = HID;
      row = n;
      k0 = (c - C1) * KC;
    } else {
      const int j = (c - C1 - C2) / C2, kc = (c - C1 - C2) % C2;
      src = Pb + L.W3;
      ld = HID;
      row = static_cast<long long>(j) * NC + n;
      k0 = kc * KC;
      valid = row < K;
    }
    uint4 v = make_uint4(0, 0, 0, 0);
    if (valid) v = *reinterpret_cast<const uint4*>(src + row * ld + k0 + kb * 8);
    *reinterpret_cast<uint4*>(img + static_cast<size_t>(c) * CHUNK_BYTES + kb * (NC * 16) + n * 16) = v;
  }
  if (u < HID) {
    b1[u] = P[L.b1 + u];
    b2[u] = P[L.b2 + u];
  }
  if (u < static_cast<long long>(nblk) * NC) b3[u] = u < K ? P[L.b3 + u] : -INFINITY;
}

struct Args {
  const float* X;
  long long N;
  const uint8_t* img;
  const float* b1;
  const float* b2;
  const float* b3;
  int nblk, K;
  uint16_t* cand;   // top-m mode: N x m
  float* logits;    // logits mode: N x K, row-major
  uint32_t* status;
  long long budget;
};

// n += x > y ? 1 : 0 and n += x >= y ? 1 : 0, as a compare and an addition under
// its predicate (the select between them would cost as much as either).
__device__ __forceinline__ void count_if_greater(float& n, float x, float y) {
  asm("{\n\t.reg .pred p;\n\tsetp.gt.f32 p, %1, %2;\n\t@p add.f32 %0, %0, 0f3F800000;\n\t}" : "+f"(n) : "f"(x), "f"(y));
}
__device__ __forceinline__ void count_if_not_less(float& n, float x, float y) {
  asm("{\n\t.reg .pred p;\n\tsetp.ge.f32 p, %1, %2;\n\t@p add.f32 %0, %0, 0f3F800000;\n\t}" : "+f"(n) : "f"(x), "f"(y));
}

// LOGITS = false: the top-M atoms per signal into a.cand.  LOGITS = true: the
// logits themselves into a.logits (the inference forward), same arithmetic.
template <int M, bool LOGITS>
__global__ void __launch_bounds__(NTHREADS, 1) propose_kernel(const __grid_constant__ Args a) {
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t* A = smem + OFF_A;
  uint8_t* ring = smem + OFF_RING;
  // The queues: logit and atom in one word, or for M = 32 in two planes.
  constexpr bool PLANES = M > 16;
  constexpr int QC = PLANES ? 30 : 21;  // queued logits per thread
  static_assert(QC * NEPI * (PLANES ? 6 : 8) <= static_cast<int>(Q_BYTES), "queues");
  uint8_t* Q = smem + OFF_Q;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + OFF_BAR);
  uint64_t* full = bars;              // [NST] chunk landed
  uint64_t* empty = bars + NST;       // [NST] chunk consumed by the MMAs
  uint64_t* tfull = bars + 2 * NST;   // [2] accumulation job done
  uint64_t* tempty = tfull + 2;       // [2] TMEM buffer drained
  uint64_t* abar = tempty + 2;        // [PARTS] A operand (a part of it) written
  uint64_t* mdone = abar + PARTS;         // every MMA of the issuer complete (exit)
  uint32_t* tslot = reinterpret_cast<uint32_t*>(mdone + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long ntiles = (a.N + TM - 1) / TM;
  const int nkeep = LOGITS ? a.nblk : a.nblk < 2 ? a.nblk : 2;  // blocks 0 and 1 are computed once
  const int nseq = 2 * a.nblk - nkeep;                          // jobs of layer 3
  // block of the s-th job of layer 3: nkeep ..., 0, 1, then nkeep ... again
  auto block = [&](int s) {
    return s < a.nblk - nkeep ? s + nkeep : s < a.nblk ? s - (a.nblk - nkeep) : s - a.nblk + nkeep;
  };

  if (tid == 0) {
    for (int q = 0; q < NST; ++q) {
      mbar_init(&full[q], 1);
      mbar_init(&empty[q], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], NEPI / 32);
    }
    for (int p = 0; p < PARTS; ++p) mbar_init(&abar[p], NEPI / 32);
    mbar_init(mdone, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(tslot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;

  if (warp == NEPI / 32 + 1) {
    // ------------------------------------------------------ producer
    if (lane == 0) {
      long long ri = 0;
      bool ok = true;
      for (long long tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
        for (int c = 0; c < C1 + C2 + C2 * nseq; ++c, ++ri) {
          const int s = (c - C1 - C2) / C2;
          const int ci = c < C1 + C2 ? c : C1 + C2 + C2 * block(s) + (c - C1 - C2) % C2;
          const int st = static_cast<int>(ri % NST);
          if (!mbar_wait(&empty[st], static_cast<uint32_t>((ri / NST) & 1) ^ 1u, a.budget)) {
            flag_status(a.status, ST_TIMEOUT);
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(&full[st], CHUNK_BYTES);
          bulk_g2s(ring + st * CHUNK_BYTES, a.img + static_cast<size_t>(ci) * CHUNK_BYTES, CHUNK_BYTES,
                   &full[st]);
        }
      }
      // every issued copy has landed before the CTA may exit
      for (long long f = ri > NST ? ri - NST : 0; f < ri; ++f)
        if (!mbar_wait(&full[f % NST], static_cast<uint32_t>((f / NST) & 1), a.budget))
          flag_status(a.status, ST_TIMEOUT);
    }
  } else if (warp == NEPI / 32) {
    // ------------------------------------------------------ MMA issuer
    if (lane == 0) {
      constexpr uint32_t idesc = umma_idesc(1, 1, TM, NC);
      // operand descriptors differ in the address alone (16-byte units, low bits)
      const uint64_t a_desc = umma_smem_desc(smem_u32(A), TM * 16, 128);
      const uint64_t r_desc = umma_smem_desc(smem_u32(ring), NC * 16, 128);
      int st = 0;
      uint32_t sph = 0, job = 0;
      uint32_t aph = 0;
      bool ok = true, issued = false;
      for (long long tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
        for (int L = 0; L < 2 + nseq && ok; ++L, ++job) {
          const int b = static_cast<int>(job & 1);
          if (!mbar_wait(&tempty[b], ((job >> 1) & 1u) ^ 1u, a.budget)) {
            flag_status(a.status, ST_TIMEOUT);
            ok = false;
            break;
          }
          tc_fence_after();
          const int nk = L == 0 ? C1 : C2;
          for (int kc = 0; kc < nk; ++kc) {
            // a new A operand: the signals for layer 1; a part of the activations at
            // a time for layer 2 and the first block of layer 3
            if (L == 0 ? kc == 0 : L <= 2 && kc % (C2 / PARTS) == 0) {
              const int p = L == 0 ? 0 : kc / (C2 / PARTS);
              if (!mbar_wait(&abar[p], (aph >> p) & 1u, a.budget)) {
                flag_status(a.status, ST_TIMEOUT);
                ok = false;
                break;
              }
              aph ^= 1u << p;
              tc_fence_after();
            }
            if (!mbar_wait(&full[st], sph, a.budget)) {
              flag_status(a.status, ST_TIMEOUT);
              ok = false;
              break;
            }
            tc_fence_after();
#pragma unroll
            for (int ks = 0; ks < KC / 16; ++ks) {
              const uint64_t ad = a_desc + static_cast<uint32_t>(kc * (KC / 8) + ks * 2) * TM;
              const uint64_t bd = r_desc + (static_cast<uint32_t>(st) * CHUNK_BYTES >> 4) + ks * 2 * NC;
              umma_bf16(tmem + static_cast<uint32_t>(b * NC), ad, bd, idesc, (kc | ks) ? 1u : 0u);
            }
            issued = true;
            tc_commit(&empty[st]);
            if (++st == NST) {
              st = 0;
              sph ^= 1u;
            }
          }
          if (ok) tc_commit(&tfull[b]);
        }
      }
      if (issued) {  // no MMA may still write TMEM when it is released
        tc_commit(mdone);
        if (!mbar_wait(mdone, 0, a.budget)) flag_status(a.status, ST_TIMEOUT);
      }
    }
  } else {
    // ------------------------------------------------------ epilogue warps
    const int q4 = warp & 3;             // TMEM lane quadrant
    const int h = warp >> 2;             // column quarter of each 256-column job
    const int r = q4 * 32 + lane;        // the thread's signal within the tile
    const uint32_t tl = tmem + (static_cast<uint32_t>(q4 * 32) << 16);
    // The candidates of every row, [place][128]: logits, and atoms (behind
    // them, or for M = 32 in the queues' place once these are read).
    constexpr int PER = M > QC ? M : QC;  // candidates a thread may hand on
    constexpr bool LATE = NQ * PER * TM * 6 > static_cast<int>(A_BYTES);
    static_assert(NQ * PER * TM * 4 <= static_cast<int>(A_BYTES) && NQ * PER * TM * 2 <= static_cast<int>(OFF_OUT), "");
    static_assert(OFF_OUT + TM * M * 2 <= Q_BYTES, "the ranked atoms lie in the queues' place");
    float* LV = reinterpret_cast<float*>(A);
    uint16_t* LJ = reinterpret_cast<uint16_t*>(LATE ? Q : A + NQ * PER * TM * 4);
    uint16_t* OUT = reinterpret_cast<uint16_t*>(Q + OFF_OUT);
    uint8_t* CN = smem + OFF_CN;
    constexpr uint32_t QSTEP = NEPI * (PLANES ? 4 : 8);  // bytes from an entry to the next
    const uint32_t q0 = smem_u32(Q) + tid * (PLANES ? 4 : 8);
    const uint32_t qa0 = smem_u32(Q) + QC * NEPI * 4 + tid * 2;
    auto queue_get = [&](int e, float& z, int& j) {
      if constexpr (PLANES) {
        z = reinterpret_cast<const float*>(Q)[e * NEPI + tid];
        j = reinterpret_cast<const uint16_t*>(Q + QC * NEPI * 4)[e * NEPI + tid];
      } else {
        const float2 v = reinterpret_cast<const float2*>(Q)[e * NEPI + tid];
        z = v.x;
        j = __float_as_int(v.y);
      }
    };
    // A job's biases of this warp's columns: read from memory one job ahead, two
    // per lane, and spread through shared memory.
    float* slot = reinterpret_cast<float*>(smem + OFF_BIAS) + warp * QW;
    float2 bnext;
    const int lcol = (lane >> 3) * 64 + h * 16 + (lane & 7) * 2;
    auto fetch_bias = [&](const float* b) { bnext = __ldg(reinterpret_cast<const float2*>(b + lcol)); };
    auto put_bias = [&]() {
      __syncwarp();
      reinterpret_cast<float2*>(slot)[lane] = bnext;
      __syncwarp();
    };
    const float4* bs = reinterpret_cast<const float4*>(slot);
    uint32_t job = 0;
    bool ok = true;
    constexpr int RW = TM / (NEPI / 32);  // signals staged per warp
    float x0[RW], x1[RW];                 // the next tile's, loaded while this one is ranked
    auto load_signals = [&](long long tile) {
#pragma unroll
      for (int rr = 0; rr < RW; ++rr) {
        const long long g = tile * TM + warp * RW + rr;
        x0[rr] = g < a.N ? a.X[g * DLSH_D + lane] : 0.f;
        x1[rr] = (g < a.N && lane < DLSH_D - 32) ? a.X[g * DLSH_D + 32 + lane] : 0.f;
      }
    };
    load_signals(blockIdx.x);
    fetch_bias(a.b1);
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
      // ---- signals -> unit-norm BF16 rows of A (k < 64); warp w: rows 8w..8w+7
      {
#pragma unroll
        for (int rr = 0; rr < RW; ++rr) {
          __nv_bfloat16 y0, y1;
          mlp::normalise_pair(x0[rr], x1[rr], y0, y1);
          const int row = warp * RW + rr;
          *reinterpret_cast<__nv_bfloat16*>(A + (lane >> 3) * (TM * 16) + row * 16 + (lane & 7) * 2) = y0;
          *reinterpret_cast<__nv_bfloat16*>(A + ((32 + lane) >> 3) * (TM * 16) + row * 16 + (lane & 7) * 2) = y1;
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&abar[0]);
      }
      // ---- layers 1 and 2: bias + GELU, BF16 activations over A
#pragma unroll 1
      for (int layer = 0; layer < 2; ++layer, ++job) {
        const int b = static_cast<int>(job & 1);
        if (ok && !mbar_wait(&tfull[b], (job >> 1) & 1u, a.budget)) {
          flag_status(a.status, ST_TIMEOUT);
          ok = false;
        }
        tc_fence_after();
        put_bias();
        if (layer == 0) fetch_bias(a.b2);
        else fetch_bias(a.b3 + static_cast<size_t>(block(0)) * NC);
#pragma unroll 1
        for (int p = 0; p < PARTS; ++p) {
          if (ok) {
            const int c0 = p * (16 * NQ) + h * 16;
            float v[16];
            tmem_ld16(tl + static_cast<uint32_t>(b * NC + c0), v);
#pragma unroll
            for (int g8 = 0; g8 < 2; ++g8) {
              const float4 bA = bs[4 * p + 2 * g8], bB = bs[4 * p + 2 * g8 + 1];
              const float bb[8] = {bA.x, bA.y, bA.z, bA.w, bB.x, bB.y, bB.z, bB.w};
              uint32_t pk[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const __nv_bfloat16 lo =
                    __float2bfloat16(mlp::gelu_f(mlp::add_bias(v[g8 * 8 + 2 * e], bb[2 * e])));
                const __nv_bfloat16 hi =
                    __float2bfloat16(mlp::gelu_f(mlp::add_bias(v[g8 * 8 + 2 * e + 1], bb[2 * e + 1])));
                pk[e] = static_cast<uint32_t>(__bfloat16_as_ushort(lo)) |
                        (static_cast<uint32_t>(__bfloat16_as_ushort(hi)) << 16);
              }
              *reinterpret_cast<uint4*>(A + ((c0 >> 3) + g8) * (TM * 16) + r * 16) =
                  make_uint4(pk[0], pk[1], pk[2], pk[3]);
            }
          }
          // the accumulators are drained with the last part; each part of the
          // activations goes to the next layer's MMAs by itself
          tc_fence_before();
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            if (p == PARTS - 1) mbar_arrive(&tempty[b]);
            mbar_arrive(&abar[p]);
          }
        }
      }
      // ---- layer 3
      float T = -INFINITY;
      if constexpr (!LOGITS) {
        // pass A: maxima of 16 interleaved groups (column mod 16) of the thread's
        // quarter row
        float gmax[NG];
#pragma unroll
        for (int i = 0; i < NG; ++i) gmax[i] = -INFINITY;
        for (int s = 0; s < a.nblk; ++s) {
          const uint32_t jb = job + static_cast<uint32_t>(s);
          const int b = static_cast<int>(jb & 1);
          if (ok && !mbar_wait(&tfull[b], (jb >> 1) & 1u, a.budget)) {
            flag_status(a.status, ST_TIMEOUT);
            ok = false;
          }
          tc_fence_after();
          put_bias();
          fetch_bias(a.b3 + static_cast<size_t>(s + 1 < a.nblk ? block(s + 1) : 0) * NC);
          if (ok) {
            const uint32_t tb = tl + static_cast<uint32_t>(b * NC + h * 16);
#pragma unroll 1
            for (int p = 0; p < PARTS; p += 2) {
              float v[2][16];
              tmem_ld16(tb + p * 64, v[0]);
              tmem_ld16(tb + p * 64 + 64, v[1]);
#pragma unroll
              for (int i4 = 0; i4 < 8; ++i4) {
                const float4 bq = bs[4 * p + i4];
                const float bb[4] = {bq.x, bq.y, bq.z, bq.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  const int i = (i4 * 4 + e) % 16;
                  gmax[i] = fmaxf(gmax[i], mlp::add_bias(v[i4 / 4][i], bb[e]));
                }
              }
            }
          }
          if (s < a.nblk - nkeep) {  // the last ones stay for pass B
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[b]);
          }
        }
        job += static_cast<uint32_t>(a.nblk - nkeep);
        // sort the maxima (bitonic network, decreasing), publish them and merge
        // them: the top NT of quarters 0 and 1 and of 2 and 3 are the elementwise
        // maxima of one list and the other reversed (a bitonic sequence, sorted
        // again), and the M-th of both is the smallest of max(c[i], d[M - 1 - i])
#pragma unroll
        for (int k = 2; k <= NG; k <<= 1) {
#pragma unroll
          for (int jj = k >> 1; jj > 0; jj >>= 1) {
#pragma unroll
            for (int i = 0; i < NG; ++i) {
              const int l = i ^ jj;
              if (l > i) {
                const float x = gmax[i], y = gmax[l];
                const bool dec = (i & k) == 0;
                gmax[i] = dec ? fmaxf(x, y) : fminf(x, y);
                gmax[l] = dec ? fminf(x, y) : fmaxf(x, y);
              }
            }
          }
        }
        float* S = reinterpret_cast<float*>(Q);  // [quarter * NG + rank][128]
        float* S2 = S + 64 * TM;                 // [rank][128]
        float* Ts = reinterpret_cast<float*>(smem + OFF_T);
        constexpr int NT = M > NG ? 2 * NG : NG;
#pragma unroll
        for (int i = 0; i < NG; ++i) S[(h * NG + i) * TM + r] = gmax[i];
        named_bar_sync(1, NEPI);
        if (h < 2) {
          float c[NT];
#pragma unroll
          for (int i = 0; i < NG; ++i) {
            const float x = S[(2 * h * NG + i) * TM + r], y = S[((2 * h + 1) * NG + NG - 1 - i) * TM + r];
            c[i] = fmaxf(x, y);
            if constexpr (NT > NG) c[NG + i] = fminf(x, y);
          }
#pragma unroll
          for (int jj = NG / 2; jj > 0; jj >>= 1) {
#pragma unroll
            for (int i = 0; i < NT; ++i) {
              const int l = i ^ jj;
              if (l > i) {
                const float x = c[i], y = c[l];
                c[i] = fmaxf(x, y);
                c[l] = fminf(x, y);
              }
            }
          }
          if (h == 1) {
#pragma unroll
            for (int i = 0; i < M; ++i) S2[i * TM + r] = c[i];
          }
          named_bar_sync(2, NEPI / 2);
          if (h == 0) {
            float t = INFINITY;
#pragma unroll
            for (int i = 0; i < M; ++i) t = fminf(t, fmaxf(c[i], S2[(M - 1 - i) * TM + r]));
            Ts[r] = t;
          }
        }
        named_bar_sync(1, NEPI);
        T = Ts[r];
      }
      // pass B (the only pass in logits mode)
      // T is finite: -inf (the atoms past K) and NaN are never candidates; the rows
      // past N have none
      T = tile * TM + r < a.N ? fmaxf(T, -3.402823466e38f) : INFINITY;
      // the place of the thread's next queued logit, and of its atom
      uint32_t qz = q0, qa = qa0;
      // predicated by hand: a branch around the store costs more than its issue slots
      auto queue_push = [&](float z, int j) {
        if constexpr (PLANES)
          asm volatile(
              "{\n\t.reg .pred p;\n\t.reg .b16 h;\n\tsetp.ge.f32 p, %2, %3;\n\tcvt.u16.u32 h, %4;\n\t"
              "@p st.shared.f32 [%0], %2;\n\t@p st.shared.u16 [%1], h;\n\t"
              "@p add.u32 %0, %0, %5;\n\t@p add.u32 %1, %1, %6;\n\t}"
              : "+r"(qz), "+r"(qa)
              : "f"(z), "f"(T), "r"(j), "n"(QSTEP), "n"(QSTEP / 2));
        else
          asm volatile(
              "{\n\t.reg .pred p;\n\tsetp.ge.f32 p, %1, %2;\n\t"
              "@p st.shared.v2.f32 [%0], {%1, %3};\n\t@p add.u32 %0, %0, %4;\n\t}"
              : "+r"(qz)
              : "f"(z), "f"(T), "f"(__int_as_float(j)), "n"(QSTEP));
      };
      // queued logits, with the stores before this ordered before the reads after it
      auto queued = [&]() {
        asm volatile("" ::: "memory");
        return static_cast<int>((qz - q0) / QSTEP);
      };
      int nl = 0;   // and those in its list, used once the queue has run over
      float lz[M];
      int lj[M];
      // Moves the queue into the list (decreasing logit, equal logits in the order of
      // arrival, which is that of the atoms).
      auto flush = [&]() {
#pragma unroll 1
        for (int e = 0, cnt = queued(); e < cnt; ++e) {
          float z;
          int j;
          queue_get(e, z, j);
          if (nl == M && !(z > lz[M - 1])) continue;
          int q = nl < M ? nl++ : M - 1;
#pragma unroll 1
          for (; q > 0 && z > lz[q - 1]; --q) {
            lz[q] = lz[q - 1];
            lj[q] = lj[q - 1];
          }
          lz[q] = z;
          lj[q] = j;
        }
        qz = q0;
        qa = qa0;
        if (nl == M) T = fmaxf(T, nextafterf(lz[M - 1], INFINITY));  // a later equal one ranks behind
      };
      for (int j = 0; j < a.nblk; ++j, ++job) {
        const int b = static_cast<int>(job & 1);
        if (ok && !mbar_wait(&tfull[b], (job >> 1) & 1u, a.budget)) {
          flag_status(a.status, ST_TIMEOUT);
          ok = false;
        }
        tc_fence_after();
        const uint32_t tb = tl + static_cast<uint32_t>(b * NC + h * 16);
        put_bias();
        if (j + 1 < a.nblk) fetch_bias(a.b3 + static_cast<size_t>(j + 1) * NC);
        else fetch_bias(a.b1);
        if (ok && LOGITS) {
          const long long g = tile * TM + r;
#pragma unroll 1
          for (int p = 0; p < PARTS; ++p) {
            float v[16];
            tmem_ld16(tb + p * 64, v);
            const int a0 = j * NC + p * 64 + h * 16;
            if (g < a.N) {
              float* out = a.logits + g * a.K + a0;
#pragma unroll
              for (int i = 0; i < 16; ++i)
                if (a0 + i < a.K) out[i] = mlp::add_bias(v[i], slot[p * 16 + i]);
            }
          }
        } else if (ok) {
          // queue the logits >= T; a queue that could run over within the next 16
          // columns is looked at every QS, and goes to its thread's list before it does
#pragma unroll 1
          for (int p = 0; p < PARTS; ++p) {
            float v[16];
            tmem_ld16(tb + p * 64, v);
            const int a0 = j * NC + p * 64 + h * 16;
            auto push4 = [&](int i4) {
              const float4 bq = bs[4 * p + i4];
              const float bb[4] = {bq.x, bq.y, bq.z, bq.w};
              float z[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) z[e] = mlp::add_bias(v[4 * i4 + e], bb[e]);
#pragma unroll
              for (int e = 0; e < 4; ++e) queue_push(z[e], a0 + 4 * i4 + e);
            };
            if (!__any_sync(0xffffffffu, qz > q0 + (QC - 16) * QSTEP)) {
#pragma unroll
              for (int i4 = 0; i4 < 4; ++i4) push4(i4);
            } else {
#pragma unroll
              for (int i4 = 0; i4 < 4; ++i4) {
                if (__any_sync(0xffffffffu, qz > q0 + (QC - QS) * QSTEP)) {
                  if (qz > q0 + (QC - QS) * QSTEP) flush();
                  __syncwarp();
                }
                push4(i4);
              }
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[b]);
      }
      // ---- rank the candidates of a row (A is free: every MMA of the tile is done;
      // in logits mode it takes the next signals right away)
      if constexpr (!LOGITS) {
        if (nl > 0) flush();
        CN[tid] = static_cast<uint8_t>(nl + queued());
      }
      if (named_bar_or(1, NEPI, !ok)) break;
      if constexpr (!LOGITS) {
        // one list per row: the quarters' candidates one after the other
        int off = 0, tot = 0;
#pragma unroll
        for (int l = 0; l < NQ; ++l) {
          const int c = CN[l * TM + r];
          off += l < h ? c : 0;
          tot += c;
        }
        auto put = [&](int e, float z, int j) {
          LV[(off + e) * TM + r] = z;
          if constexpr (!LATE) LJ[(off + e) * TM + r] = static_cast<uint16_t>(j);
        };
        const int cnt = queued();
        int qj[QC];
#pragma unroll
        for (int e = 0; e < QC; ++e) {
          if (e < cnt) {
            float z;
            queue_get(e, z, qj[e]);
            put(e, z, qj[e]);
          }
        }
#pragma unroll 1
        for (int e = 0; e < nl; ++e) put(e, lz[e], lj[e]);
        load_signals(tile + gridDim.x);
        named_bar_sync(1, NEPI);
        if constexpr (LATE) {  // the atoms take the place of the queues
#pragma unroll
          for (int e = 0; e < QC; ++e)
            if (e < cnt) LJ[(off + e) * TM + r] = static_cast<uint16_t>(qj[e]);
#pragma unroll 1
          for (int e = 0; e < nl; ++e) LJ[(off + e) * TM + r] = static_cast<uint16_t>(lj[e]);
          named_bar_sync(1, NEPI);
        }
        // rank = candidates before it, by (logit desc, atom asc); every fourth
        // candidate of the row is this thread's, RK at a time in registers.  Larger
        // and equal logits are counted; the atoms are looked at for one that has an
        // equal besides itself.
        constexpr int RK = M <= 8 ? 4 : M <= 16 ? 6 : 13;
        const int most = __reduce_max_sync(0xffffffffu, tot);
#pragma unroll 1
        for (int c = h; c < most; c += RK * NQ) {
          float key[RK], above[RK], from[RK];
#pragma unroll
          for (int k = 0; k < RK; ++k) {
            const int o = c + NQ * k;
            key[k] = o < tot ? LV[o * TM + r] : INFINITY;
            above[k] = from[k] = 0.f;
          }
#pragma unroll 4
          for (int o = 0; o < most; ++o) {
            const float x = o < tot ? LV[o * TM + r] : -INFINITY;
#pragma unroll
            for (int k = 0; k < RK; ++k) {
              count_if_greater(above[k], x, key[k]);
              count_if_not_less(from[k], x, key[k]);
            }
          }
#pragma unroll
          for (int k = 0; k < RK; ++k) {
            const int o = c + NQ * k;
            if (o < tot) {
              const int j = LJ[o * TM + r];
              int q = static_cast<int>(above[k]);
              if (from[k] > above[k] + 1.f) {
#pragma unroll 1
                for (int e = 0; e < tot; ++e) q += LV[e * TM + r] == key[k] && LJ[e * TM + r] < j ? 1 : 0;
              }
              if (q < M) OUT[r * M + q] = static_cast<uint16_t>(j);
            }
          }
        }
        for (int q = tot + h; q < M; q += NQ) OUT[r * M + q] = 0xffffu;  // fewer than M logits above -inf
        named_bar_sync(1, NEPI);
        const long long rows = a.N - tile * TM;
        const int words = static_cast<int>(rows < TM ? rows : TM) * (M / 2);
        uint32_t* out = reinterpret_cast<uint32_t*>(a.cand + tile * TM * M);
        for (int q = tid; q < words; q += NEPI) out[q] = reinterpret_cast<const uint32_t*>(OUT)[q];
      } else {
        load_signals(tile + gridDim.x);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

}  // namespace prop

size_t propose_ws_bytes(int K) {
  prop::Ws w;
  return prop::carve(nullptr, K, w);
}

// Packs the weights, then launches the fused kernel: top-m into cand (m > 0)
// or the logits into `logits` (m = 0).
static int fused_enqueue(const void* mlp_blob, int K, const float* X, long long N, int m,
                         uint16_t* cand, float* logits, void* ws, uint32_t* status, cudaStream_t st,
                         const char* call) {
  using namespace prop;
  if (reinterpret_cast<uintptr_t>(ws) % 256)
    return set_error(DLSH_ERR_INVALID_ARG, "%s: workspace must be 256-byte aligned", call);
  mlp::Blob b;
  mlp::carve_blob(const_cast<void*>(mlp_blob), K, b);
  Ws w;
  carve(ws, K, w);
  const int nblk = n_blocks(K);
  const long long units = static_cast<long long>(n_chunks(K)) * (CHUNK_BYTES / 16);
  pack_kernel<<<static_cast<int>((units + 255) / 256), 256, 0, st>>>(b.Pb, b.P, K, nblk, w.img, w.b1,
                                                                     w.b2, w.b3);
  count_launches(1);
  int rc = check_launch(call);
  if (rc) return rc;
  Args a;
  a.X = X;
  a.N = N;
  a.img = w.img;
  a.b1 = w.b1;
  a.b2 = w.b2;
  a.b3 = w.b3;
  a.nblk = nblk;
  a.K = K;
  a.cand = cand;
  a.logits = logits;
  a.status = status;
  a.budget = kWaitBudget;
  const long long ntiles = (N + TM - 1) / TM;
  const int grid = static_cast<int>(ntiles < device_sm_count() ? ntiles : device_sm_count());
#define LAUNCH(MM, LG)                                                                             \
  do {                                                                                             \
    static PerDevice<int> attr;                                                                    \
    int attr_ok = 0;                                                                               \
    const int arc = attr.get(&attr_ok, [&](int& v) {                                               \
      DLSH_CUDA_TRY(cudaFuncSetAttribute(propose_kernel<MM, LG>,                                   \
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES), \
                    call);                                                                         \
      v = 1;                                                                                       \
      return DLSH_OK;                                                                              \
    });                                                                                            \
    if (arc) return arc;                                                                           \
    propose_kernel<MM, LG><<<grid, NTHREADS, SMEM_BYTES, st>>>(a);                                 \
  } while (0)
  switch (m) {
    case 0: LAUNCH(2, true); break;
    case 2: LAUNCH(2, false); break;
    case 4: LAUNCH(4, false); break;
    case 8: LAUNCH(8, false); break;
    case 16: LAUNCH(16, false); break;
    default: LAUNCH(32, false); break;
  }
#undef LAUNCH
  count_launches(1);
  return check_launch(call);
}

int propose_enqueue(const void* mlp_blob, int K, const float* X, long long N, int m, uint16_t* cand,
                    void* ws, uint32_t* status, cudaStream_t st) {
  if (m != 2 && m != 4 && m != 8 && m != 16 && m != 32)
    return set_error(DLSH_ERR_UNSUPPORTED, "dlsh_mlp_propose: m must be 2, 4, 8, 16 or 32");
  if (N <= 0) return DLSH_OK;
  if (reinterpret_cast<uintptr_t>(cand) % (2 * m < 16 ? 2 * m : 16))
    return set_error(DLSH_ERR_INVALID_ARG, "dlsh_mlp_propose: cand must be aligned to min(16, 2m) bytes");
  return fused_enqueue(mlp_blob, K, X, N, m, cand, nullptr, ws, status, st, "dlsh_mlp_propose");
}

int infer_logits_enqueue(const void* mlp_blob, int K, const float* X, long long N, float* logits,
                         void* ws, uint32_t* status, cudaStream_t st) {
  if (N <= 0) return DLSH_OK;
  return fused_enqueue(mlp_blob, K, X, N, 0, nullptr, logits, ws, status, st, "dlsh_mlp_forward");
}

}  // namespace dlsh
