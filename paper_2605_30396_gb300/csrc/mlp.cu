// Learned support proposal: a 45 -> 256 -> 256 -> K MLP (GELU, BF16 weights,
// FP32 accumulation) trained on (signal, OMP support) pairs that the codec
// itself produces, whose 2s largest logits name candidate atoms for an OMP
// restricted to them; plain OMP (Sec. 2.1) remains the fallback.
//
// GPU design:
//   train_gemm_kernel  tcgen05 BF16 GEMM, C = A B^T with FP32 accumulation in
//                   TMEM, 128 x 128 tiles.  An operand is read in place by
//                   TMA, K-major or MN-major (the transposed activations and
//                   weights of the backward pass need no copies).  Each epilogue
//                   does the element-wise work that follows the product: bias +
//                   GELU, BCE gradient + loss + column sums, GELU backward +
//                   column sums, or the FP32 partial of a weight gradient.  The
//                   weight gradients of all three layers are one launch, split
//                   over the batch.
//   reduce_kernel   adds the split partials and the column sums in a fixed
//                   order (gradients), and applies Adam in a training step
// Batch 8192, K = 1024 (us of device time): logits with the BCE work 34 + 67 -> 29,
// dH2 with the GELU backward 103 -> 15, weight gradients 479 -> 12; the whole
// gradient call 810 -> 157, of which about 90 are the seven launches.
#include <cuda.h>
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "host.hpp"
#include "internal.hpp"
#include "mlp.cuh"

namespace dlsh {
namespace mlp {

constexpr int GM = 128;  // tile rows = MMA M
constexpr int GN = 128;  // tile cols = MMA N
constexpr int GK = 64;   // k-tile: four MMAs of K = 16
constexpr int GT = 256;  // threads per GEMM CTA (warp w: TMEM lanes of quarter w & 3, columns of half w >> 2)
// Operand tiles in shared memory, 128 rows (M or N) x 64 k, 16 KB, as TMA
// writes them with the 128-byte swizzle (16-byte word c of 128-byte line l sits
// at word c ^ (l & 7)):
//   K-major   one box: line = row, 64 k; eight-row groups 1024 bytes apart
//   MN-major  two boxes of 64 rows: line = k, 64 rows; eight-k groups 1024
//             bytes apart, the boxes 8 KB apart
// (With 16-byte cp.async into the unswizzled layout each word was an L2 request
// of its own: twice the bytes and 3 to 4 times the time of the k-loops.)
constexpr uint32_t OPER = GM * GK * 2;
constexpr uint32_t STAGE = 2 * OPER;
// Operand stages NS: three where the grid gives every SM two CTAs, six where it
// gives only one.
constexpr uint32_t gemm_smem(int ns) { return ns * STAGE + 1024; }

enum : int { EPI_GELU = 0, EPI_BCE = 1, EPI_GELU_BWD = 2, EPI_PART = 3 };

// One product of a launch: M x N over k [0, Kd), its tiles numbered from tile0.
// The operands' tensor maps: K-major maps have k as the inner dimension,
// MN-major ones the rows; what lies outside reads as zero.
struct Prod {
  CUtensorMap A, B;
  int M, N, Kd, tiles_n, tile0;
  float* C;  // FP32 output (EPI_PART: partial z at C + z * zstride), row stride ldc
  int ldc;
};

struct GemmArgs {
  Prod p[3];
  int nprod;
  int M;                // valid rows of the batch (all epilogues but EPI_PART)
  int klen;             // k range per split (multiple of GK)
  long long zstride;
  const float* bias;    // N (EPI_GELU, EPI_BCE)
  const float* Z;       // EPI_GELU_BWD: the layer's pre-activations, row stride HID
  __nv_bfloat16* H;     // BF16 output (activations or dZ), row stride ldh
  int ldh;
  float* colpart;       // column sums of the FP32 values per 128-row tile, [tile][ldh]
  const float* X;       // EPI_GELU with XA: the signals (A is their unit-norm BF16 form)
  __nv_bfloat16* Xn;    // and where that form is kept for the weight gradient
  const uint16_t* idx;  // EPI_BCE: the targets
  const uint8_t* nnz;
  int s;
  float inv_bk;
  double* loss_part;    // EPI_BCE: one loss sum per CTA
  uint32_t* status;
  long long budget;
};

// 32 bytes to global memory in one store (32-byte aligned).
__device__ __forceinline__ void st32(void* p, const uint32_t (&v)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]),
               "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
// 32 consecutive FP32 / BF16 values of one row (32-byte aligned).
__device__ __forceinline__ void store_f32(float* p, const float (&v)[32]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint32_t w[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) w[e] = __float_as_uint(v[8 * q + e]);
    st32(p + 8 * q, w);
  }
}
__device__ __forceinline__ void store_bf16(__nv_bfloat16* p, const float (&v)[32]) {
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    uint32_t w[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const __nv_bfloat162 b = __floats2bfloat162_rn(v[16 * q + 2 * e], v[16 * q + 2 * e + 1]);
      w[e] = *reinterpret_cast<const uint32_t*>(&b);
    }
    st32(p + 16 * q, w);
  }
}

// Hardware reciprocal (about 1 ulp; 0 for infinity).
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Sums of the warp's 32 rows: lane l returns the sum of v[l] over the lanes
// (a transposing butterfly, the same order on every run).
__device__ __forceinline__ float col_sums(float (&v)[32]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int m = 32, o = 16; o > 0; m >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int k = 0; k < m / 2; ++k) {
      const float send = up ? v[k] : v[k + m / 2];
      const float keep = up ? v[k + m / 2] : v[k];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  return v[0];
}

// C = A B^T tile by tile, and the layer's element-wise work on the result.
// Warp 0 streams the operands by TMA, warp 1 issues the MMAs, then all eight
// warps share the epilogue; a second CTA on the SM runs its k-loop meanwhile.
template <int EPI, bool AMN, bool BMN, bool XA, int NS>
__global__ void __launch_bounds__(GT, NS > 3 ? 1 : 2) train_gemm_kernel(const __grid_constant__ GemmArgs g) {
  extern __shared__ __align__(1024) uint8_t smem[];
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + NS * STAGE);  // [NS] operands landed
  uint64_t* empty = full + NS;                                       // [NS] consumed by the MMAs
  uint64_t* done = empty + NS;                                       // every MMA complete
  uint32_t* tslot = reinterpret_cast<uint32_t*>(done + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int pi = 0;
  if (EPI == EPI_PART)
    while (pi + 1 < g.nprod && static_cast<int>(blockIdx.x) >= g.p[pi + 1].tile0) ++pi;
  const Prod& P = g.p[pi];
  const int tile = static_cast<int>(blockIdx.x) - P.tile0;
  const int tm = tile / P.tiles_n;
  const int m0 = tm * GM, n0 = (tile - tm * P.tiles_n) * GN;
  const int kbeg = blockIdx.y * g.klen;
  const int kend = kbeg + g.klen < P.Kd ? kbeg + g.klen : P.Kd;
  const int nkt = kend > kbeg ? (kend - kbeg + GK - 1) / GK : 0;
  if (tid == 0) {
    for (int q = 0; q < NS; ++q) {
      mbar_init(&full[q], 1);
      mbar_init(&empty[q], 1);
    }
    mbar_init(done, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(tslot, GN);
    tmem_relinquish();
  }
  depend();  // nothing above touches global memory
  constexpr uint32_t idesc =
      umma_idesc(1, 1, GM, GN) | (AMN ? 1u << 15 : 0u) | (BMN ? 1u << 16 : 0u);  // bits 15, 16: MN-major
  if (XA) {
    // A = the signals at unit norm, one k-tile (Kd = XIN = GK); warp w stages
    // rows 16 w .. 16 w + 15
    float x0[16], x1[16];
#pragma unroll
    for (int rr = 0; rr < 16; ++rr) {
      const long long r = m0 + warp * 16 + rr;
      x0[rr] = r < g.M ? g.X[r * DLSH_D + lane] : 0.f;
      x1[rr] = (r < g.M && lane < DLSH_D - 32) ? g.X[r * DLSH_D + 32 + lane] : 0.f;
    }
#pragma unroll
    for (int rr = 0; rr < 16; ++rr) {
      const int row = warp * 16 + rr;
      __nv_bfloat16 y0, y1;
      normalise_pair(x0[rr], x1[rr], y0, y1);
      uint8_t* d = smem + row * 128 + (lane & 7) * 2;
      *reinterpret_cast<__nv_bfloat16*>(d + (((lane >> 3) ^ (row & 7)) << 4)) = y0;
      *reinterpret_cast<__nv_bfloat16*>(d + (((4 + (lane >> 3)) ^ (row & 7)) << 4)) = y1;
      if (n0 == 0 && m0 + row < g.M) {
        g.Xn[static_cast<size_t>(m0 + row) * XIN + lane] = y0;
        g.Xn[static_cast<size_t>(m0 + row) * XIN + 32 + lane] = y1;
      }
    }
    fence_proxy_async_smem();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  bool ok = true;
  if (tid == 0) {
    int issued = 0;
    for (int t = 0; t < nkt; ++t) {
      const int sl = t % NS, k0 = kbeg + t * GK;
      if (!mbar_wait(&empty[sl], static_cast<uint32_t>((t / NS) & 1) ^ 1u, g.budget)) {
        flag_status(g.status, ST_TIMEOUT);
        ok = false;
        break;
      }
      uint8_t* d = smem + sl * STAGE;
      mbar_arrive_expect_tx(&full[sl], XA ? OPER : STAGE);
      if (!XA) {
        if (AMN) {
          tma_load_2d(d, &P.A, m0, k0, &full[sl]);
          tma_load_2d(d + OPER / 2, &P.A, m0 + 64, k0, &full[sl]);
        } else {
          tma_load_2d(d, &P.A, k0, m0, &full[sl]);
        }
      }
      d += OPER;
      if (BMN) {
        tma_load_2d(d, &P.B, n0, k0, &full[sl]);
        tma_load_2d(d + OPER / 2, &P.B, n0 + 64, k0, &full[sl]);
      } else {
        tma_load_2d(d, &P.B, k0, n0, &full[sl]);
      }
      issued = t + 1;
    }
    // every issued copy has landed before the CTA may exit
    for (int t = issued > NS ? issued - NS : 0; t < issued; ++t)
      if (!mbar_wait(&full[t % NS], static_cast<uint32_t>((t / NS) & 1), g.budget)) {
        flag_status(g.status, ST_TIMEOUT);
        ok = false;
      }
  } else if (tid == 32) {
    const uint32_t s0 = smem_u32(smem);
    for (int t = 0; t < nkt; ++t) {
      const int sl = t % NS;
      if (!mbar_wait(&full[sl], static_cast<uint32_t>((t / NS) & 1), g.budget)) {
        flag_status(g.status, ST_TIMEOUT);
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t a = s0 + static_cast<uint32_t>(sl) * STAGE, b = a + OPER;
#pragma unroll
      for (int ks = 0; ks < GK / 16; ++ks) {
        // 16 k: two words further into each line (K-major), two groups of
        // eight lines further (MN-major)
        const uint64_t ad = umma_smem_desc_sw128(a + ks * (AMN ? 2048u : 32u), OPER / 2, 1024);
        const uint64_t bd = umma_smem_desc_sw128(b + ks * (BMN ? 2048u : 32u), OPER / 2, 1024);
        umma_bf16(tmem, ad, bd, idesc, (t > 0 || ks > 0) ? 1u : 0u);
      }
      tc_commit(&empty[sl]);
    }
    tc_commit(done);
  }
  __syncwarp();
  if (!mbar_wait(done, 0, 2 * g.budget)) {
    flag_status(g.status, ST_TIMEOUT);
    ok = false;
  }
  ok = !__syncthreads_or(!ok);
  tc_fence_after();
  // ---- epilogue: thread = one row, 64 columns in two groups of 32 (TMEM lane
  // quarter and column half of its warp).  A row's 32 values are whole 32-byte
  // sectors, stored straight from the registers.
  const int q4 = warp & 3, h = warp >> 2;
  const int row = m0 + q4 * 32 + lane;
  float* csum = reinterpret_cast<float*>(smem);  // [4][128] column sums of the quarters (the stages are free)
  double* lsum = reinterpret_cast<double*>(smem + 4 * GN * 4);
  if (ok) {
    unsigned long long tgt = 0;  // EPI_BCE: bit c = column n0 + 64 h + c is a target of the row
    float lh = 0.f, ll = 0.f;    // the row's loss, float-float
    double big = 0.0;            // and the part of it that FP32 cannot hold
    if (EPI == EPI_BCE && row < g.M) {
      int nz = g.nnz[row];
      nz = nz > g.s ? g.s : nz;
#pragma unroll 4
      for (int t = 0; t < nz; ++t) {
        const int c = static_cast<int>(g.idx[static_cast<size_t>(row) * g.s + t]) - (n0 + 64 * h);
        if (c >= 0 && c < 64) tgt |= 1ull << c;
      }
    }
#pragma unroll 1
    for (int cg = 0; cg < 2; ++cg) {
      const int cb = h * 64 + cg * 32, col = n0 + cb;
      float v[32];
      if (nkt > 0) {
        tmem_ld32(tmem + (static_cast<uint32_t>(q4 * 32) << 16) + cb, v);
      } else {
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = 0.f;
      }
      if (EPI == EPI_PART) {
        if (row < P.M && col < P.N)  // N is a multiple of 32
          store_f32(P.C + blockIdx.y * g.zstride + static_cast<size_t>(row) * P.ldc + col, v);
        continue;
      }
      if (EPI == EPI_GELU) {
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = add_bias(v[k], g.bias[col + k]);
        if (row < g.M) {
          store_f32(P.C + static_cast<size_t>(row) * P.ldc + col, v);
#pragma unroll
          for (int k = 0; k < 32; ++k) v[k] = gelu_f(v[k]);
          store_bf16(g.H + static_cast<size_t>(row) * g.ldh + col, v);
        }
        continue;
      }
      if (EPI == EPI_BCE) {
        // BCE(z, y) = max(y ? -z : z, 0) + log(1 + e^-|z|); the group's logs are
        // taken once, of the float-float product of its 1 + e^-|z| (at most
        // 2^32), each 1 + e^-|z| exact as a pair, and the max terms are summed in
        // float-float.  1 / (1 + e^-z) is the hardware reciprocal after one Newton
        // step (__frcp_rn gives the same gradients and takes 5 % longer over the
        // call).  A NaN logit leaves a NaN in the gradient and in the loss.
        const unsigned y32 = static_cast<unsigned>(tgt >> (32 * cg));
        float ph = 1.f, pl = 0.f;
        const float lh0 = lh, ll0 = ll;
        auto elem = [&](int k, float bias) {
          const float z = add_bias(v[k], bias);
          const bool y = (y32 >> k) & 1u;
          const float e = expf(-z), d = 1.f + e, r0 = rcp_approx(d);
          // (an infinite d keeps its reciprocal 0; a NaN is one in r0)
          const float r = fmaf(r0, fmaf(-fminf(d, 3.402823466e38f), r0, 1.f), r0);
          v[k] = (r - (y ? 1.f : 0.f)) * g.inv_bk;
          const float q = z < 0.f ? rcp_approx(e) : e;  // e^-|z|
          const float f = 1.f + q, fl = q - (f - 1.f);
          const float np = ph * f;
          pl = fmaf(pl, f, fmaf(ph, fl, fmaf(ph, f, -np)));
          ph = np;
          const float lz = fmaxf(y ? -z : z, 0.f);
          const float t = lh + lz, bb = t - lh;
          ll += (lh - (t - bb)) + (lz - bb);
          lh = t;
        };
        if (row < g.M && col + 32 <= P.N) {
#pragma unroll
          for (int k = 0; k < 32; ++k) elem(k, g.bias[col + k]);
        } else {
#pragma unroll
          for (int k = 0; k < 32; ++k) {
            if (row < g.M && col + k < P.N) elem(k, g.bias[col + k]);
            else v[k] = 0.f;
          }
        }
        // infinite logits, or a sum beyond FP32's range: the max terms from the accumulators
        // again, in FP64
        if (__any_sync(0xffffffffu, !(lh < INFINITY))) {
          double lin = 0.0;
#pragma unroll 1
          for (int c0 = 0; c0 < 32; c0 += 16) {
            float w[16];
            tmem_ld16(tmem + (static_cast<uint32_t>(q4 * 32) << 16) + cb + c0, w);
#pragma unroll
            for (int k = 0; k < 16; ++k)
              if (row < g.M && col + c0 + k < P.N) {
                const float z = add_bias(w[k], g.bias[col + c0 + k]);
                lin += fmaxf((y32 >> (c0 + k)) & 1u ? -z : z, 0.f);
              }
          }
          if (!(lh < INFINITY)) {
            big += lin;
            lh = lh0;
            ll = ll0;
          }
        }
        ll += logf(ph) + __fdividef(pl, ph);
      } else {
        float4 z4[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
          z4[k] = row < g.M ? *reinterpret_cast<const float4*>(g.Z + static_cast<size_t>(row) * HID + col + 4 * k)
                            : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          v[4 * k + 0] *= gelu_grad_f(z4[k].x);
          v[4 * k + 1] *= gelu_grad_f(z4[k].y);
          v[4 * k + 2] *= gelu_grad_f(z4[k].z);
          v[4 * k + 3] *= gelu_grad_f(z4[k].w);
        }
      }
      if (row < g.M && col < g.ldh) store_bf16(g.H + static_cast<size_t>(row) * g.ldh + col, v);
      csum[q4 * GN + cb + lane] = col_sums(v);
    }
    if (EPI == EPI_BCE) {
      double l = static_cast<double>(lh) + static_cast<double>(ll);
      if (big != 0.0) l += big;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
      if (lane == 0) lsum[warp] = l;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (ok && (EPI == EPI_BCE || EPI == EPI_GELU_BWD)) {
    if (tid < GN && n0 + tid < g.ldh)
      g.colpart[static_cast<size_t>(tm) * g.ldh + n0 + tid] =
          (csum[tid] + csum[GN + tid]) + (csum[2 * GN + tid] + csum[3 * GN + tid]);
    if (EPI == EPI_BCE && tid == 0) {
      double l = 0.0;
      for (int w = 0; w < GT / 32; ++w) l += lsum[w];
      g.loss_part[blockIdx.x] = l;
    }
  }
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, GN);
  }
}

// ---- gradients from the partials, and Adam -------------------------------------
struct ReduceArgs {
  const float* part;  // [splits][zstride] weight gradients at their parameter offsets
  long long zstride;
  int splits;
  const float* cp1;   // column sums per 128-row tile (bias gradients): [tiles][256], [tiles][256], [tiles][ldk]
  const float* cp2;
  const float* cp3;
  int tiles, ldk;
  const double* loss_part;
  int nloss;
  double inv_bk;
  float* loss;        // may be NULL
  float* G;           // gradients out (ADAM = false)
  Blob b;             // parameters and moments (ADAM = true)
  Layout L;
  float lr, beta1, beta2, eps, bc1, bc2;
};

template <bool ADAM>
__global__ void __launch_bounds__(256) reduce_kernel(const __grid_constant__ ReduceArgs a) {
  depend();
  // The first block takes the mean loss (a fixed-order sum), the others the
  // parameters from the last on, so that the longest sums (b3) begin first.
  if (blockIdx.x == 0) {
    __shared__ double red[256];
    double acc = 0.0;
    for (int q = threadIdx.x; q < a.nloss; q += 256) acc += a.loss_part[q];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
      if (static_cast<int>(threadIdx.x) < w) red[threadIdx.x] += red[threadIdx.x + w];
      __syncthreads();
    }
    if (threadIdx.x == 0 && a.loss) *a.loss = static_cast<float>(red[0] * a.inv_bk);
    return;
  }
  const long long i = static_cast<long long>(gridDim.x - 1 - blockIdx.x) * 256 + threadIdx.x;
  if (i >= a.L.n) return;
  const float* src = a.part + i;
  long long stride = a.zstride;
  int n = a.splits;
  if (i >= a.L.b3) {
    src = a.cp3 + (i - a.L.b3);
    stride = a.ldk;
    n = a.tiles;
  } else if (i >= a.L.b2 && i < a.L.W3) {
    src = a.cp2 + (i - a.L.b2);
    stride = HID;
    n = a.tiles;
  } else if (i >= a.L.b1 && i < a.L.W2) {
    src = a.cp1 + (i - a.L.b1);
    stride = HID;
    n = a.tiles;
  }
  float m = 0.f, v = 0.f, p = 0.f;  // Adam's operands, in flight beside the partials
  if (ADAM) {
    m = a.b.m1[i];
    v = a.b.m2[i];
    p = a.b.P[i];
  }
  float g = 0.f;
  if (stride == a.zstride) {
#pragma unroll 8
    for (int z = 0; z < n; ++z) g += src[z * stride];
  } else {  // eight sums side by side: a hundred tiles in a row would cost a bias gradient a bit
    // (32 of them in flight: the chain of loads is what this kernel takes)
    float c[8] = {};
    for (int z = 0; z < n; z += 32) {
      float x[32];
#pragma unroll
      for (int u = 0; u < 32; ++u) x[u] = z + u < n ? src[(z + u) * stride] : 0.f;
#pragma unroll
      for (int u = 0; u < 32; ++u) c[u & 7] += x[u];
    }
    g = ((c[0] + c[1]) + (c[2] + c[3])) + ((c[4] + c[5]) + (c[6] + c[7]));
  }
  if (!ADAM) {
    a.G[i] = g;
    return;
  }
  m = a.beta1 * m + (1.f - a.beta1) * g;
  v = a.beta2 * v + (1.f - a.beta2) * g * g;
  a.b.m1[i] = m;
  a.b.m2[i] = v;
  p = p - a.lr * (m / a.bc1) / (sqrtf(v / a.bc2) + a.eps);
  a.b.P[i] = p;
  a.b.Pb[i] = __float2bfloat16(p);
}

__global__ void mirror_kernel(const float* __restrict__ P, __nv_bfloat16* __restrict__ Pb, long long n) {
  const long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i < n) Pb[i] = __float2bfloat16(P[i]);
}

}  // namespace mlp
}  // namespace dlsh

// ===========================================================================
// Host side
// ===========================================================================
namespace dlsh {
namespace mlp {

// cuTensorMapEncodeTiled, taken from the driver at run time
using PFN_encodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                     const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                     CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

constexpr int kSms = 152;  // SMs of a GB300

// Training workspace for batches of up to B rows.
struct TWs {
  uint32_t* status;
  __nv_bfloat16* Xn;    // B x 64
  float* Z1;            // B x 256 pre-activations
  float* Z2;
  __nv_bfloat16* H1;    // B x 256 activations
  __nv_bfloat16* H2;
  __nv_bfloat16* dZ1;   // B x 256
  __nv_bfloat16* dZ2;
  __nv_bfloat16* dZ3;   // B x ldk (zeros past K)
  float* part;          // splits x zstride weight-gradient partials
  float* cp1;           // column sums per 128-row tile
  float* cp2;
  float* cp3;
  double* loss_part;    // one per CTA of the logits product
  int ldk;
  int splits, klen;     // split of the batch in the weight gradients
  int tiles_m, tiles_w;
  long long zstride;
};

// Batch split of the weight gradients: their 128 x 128 tiles (22 at K = 1024)
// times the splits fill two CTAs per SM once, each split at least four k-tiles
// long (shorter ones are mostly prologue and epilogue).
static void split_batch(int K, long long B, TWs& w) {
  w.tiles_m = static_cast<int>((B + GM - 1) / GM);
  w.tiles_w = ((K + GM - 1) / GM) * (HID / GN) + (HID / GM) * (HID / GN) + HID / GM;
  const long long kt = (B + GK - 1) / GK;
  long long splits = 2LL * kSms / w.tiles_w;
  splits = std::max<long long>(1, std::min<long long>(splits, kt / 4));
  const long long per = (kt + splits - 1) / splits;
  w.klen = static_cast<int>(per * GK);
  w.splits = static_cast<int>((kt + per - 1) / per);
}

static size_t carve_t(void* base, int K, long long B, TWs& w) {
  const Layout L = layout(K);
  split_batch(K, B, w);
  w.ldk = (K + 63) / 64 * 64;
  w.zstride = (L.n + 63) / 64 * 64;
  Carver c(base);
  w.status = c.take<uint32_t>(64);
  w.Xn = c.take<__nv_bfloat16>(B * XIN);
  w.Z1 = c.take<float>(B * HID);
  w.Z2 = c.take<float>(B * HID);
  w.H1 = c.take<__nv_bfloat16>(B * HID);
  w.H2 = c.take<__nv_bfloat16>(B * HID);
  w.dZ1 = c.take<__nv_bfloat16>(B * HID);
  w.dZ2 = c.take<__nv_bfloat16>(B * HID);
  w.dZ3 = c.take<__nv_bfloat16>(B * w.ldk);
  w.part = c.take<float>(w.zstride * w.splits);
  w.cp1 = c.take<float>(static_cast<size_t>(w.tiles_m) * HID);
  w.cp2 = c.take<float>(static_cast<size_t>(w.tiles_m) * HID);
  w.cp3 = c.take<float>(static_cast<size_t>(w.tiles_m) * w.ldk);
  w.loss_part = c.take<double>(static_cast<size_t>(w.tiles_m) * ((K + GN - 1) / GN));
  return c.size();
}

// A BF16 matrix of `lines` lines of `inner` elements (line stride ld elements,
// a multiple of 8) as a 128-byte-swizzled tensor map with boxes of 64 elements
// x box_lines lines.
static int tensor_map(CUtensorMap* m, const __nv_bfloat16* p, int inner, int lines, int ld, int box_lines) {
  static PerDevice<PFN_encodeTiled> entry;
  PFN_encodeTiled enc = nullptr;
  const int rc = entry.get(&enc, [](PFN_encodeTiled& v) {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    DLSH_CUDA_TRY(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q),
                  "dlsh_mlp: cuTensorMapEncodeTiled");
    if (!f || q != cudaDriverEntryPointSuccess)
      return set_error(DLSH_ERR_CUDA, "dlsh_mlp: the driver has no cuTensorMapEncodeTiled");
    v = reinterpret_cast<PFN_encodeTiled>(f);
    return DLSH_OK;
  });
  if (rc) return rc;
  const cuuint64_t dim[2] = {static_cast<cuuint64_t>(inner), static_cast<cuuint64_t>(lines)};
  const cuuint64_t stride[1] = {static_cast<cuuint64_t>(ld) * 2};
  const cuuint32_t box[2] = {64, static_cast<cuuint32_t>(box_lines)};
  const cuuint32_t one[2] = {1, 1};
  const CUresult e = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16*>(p), dim, stride, box, one,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (e != CUDA_SUCCESS)
    return set_error(DLSH_ERR_CUDA, "dlsh_mlp: tensor map of %d x %d: error %d", lines, inner, static_cast<int>(e));
  return DLSH_OK;
}
// rows x k operands: K-major (rows are the lines) and MN-major (k are the lines)
static int kmajor(CUtensorMap* m, const __nv_bfloat16* p, int rows, int k, int ld) {
  return tensor_map(m, p, k, rows, ld, GM);
}
static int mnmajor(CUtensorMap* m, const __nv_bfloat16* p, int rows, int k, int ld) {
  return tensor_map(m, p, rows, k, ld, GK);
}

template <int EPI, bool AMN, bool BMN, bool XA, int NS>
static int launch_gemm_ns(const GemmArgs& g, int tiles, int splits, cudaStream_t st) {
  static PerDevice<int> attr;
  int attr_ok = 0;
  const int arc = attr.get(&attr_ok, [](int& v) {
    DLSH_CUDA_TRY(cudaFuncSetAttribute(train_gemm_kernel<EPI, AMN, BMN, XA, NS>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, gemm_smem(NS)),
                  "dlsh_mlp: attribute");
    v = 1;
    return DLSH_OK;
  });
  if (arc) return arc;
  launch_dependent(train_gemm_kernel<EPI, AMN, BMN, XA, NS>, dim3(tiles, splits), GT, gemm_smem(NS), st, g);
  count_launches(1);
  return check_launch("dlsh_mlp: gemm");
}

template <int EPI, bool AMN, bool BMN, bool XA>
static int launch_gemm(const GemmArgs& g, int tiles, int splits, cudaStream_t st) {
  // one k-tile (XA) needs no depth; the logits' and the weight gradients' grids
  // give two CTAs per SM but on the smallest batches
  if constexpr (!XA && (EPI == EPI_GELU || EPI == EPI_GELU_BWD))
    if (tiles <= kSms) return launch_gemm_ns<EPI, AMN, BMN, XA, 6>(g, tiles, splits, st);
  return launch_gemm_ns<EPI, AMN, BMN, XA, 3>(g, tiles, splits, st);
}

// The products of a training step on batches of M rows in the workspace w,
// tensor maps included: built once per call, whatever the number of steps.
struct Plan {
  GemmArgs l1, l2, l3, d2, d1, wg;
};
static int make_plan(const Blob& b, int K, int M, const TWs& w, int s, Plan& t) {
  const Layout L = layout(K);
  GemmArgs g{};
  g.nprod = 1;
  g.M = M;
  g.s = s;
  g.inv_bk = static_cast<float>(1.0 / (static_cast<double>(M) * K));
  g.status = w.status;
  g.budget = kWaitBudget;
  t.l1 = t.l2 = t.l3 = t.d2 = t.d1 = t.wg = g;
  auto prod = [&](GemmArgs& a, int q, int Mr, int N, int Kd, float* C, int ldc) {
    Prod& p = a.p[q];
    p.M = Mr;
    p.N = N;
    p.Kd = Kd;
    p.tiles_n = (N + GN - 1) / GN;
    p.tile0 = q ? a.p[q - 1].tile0 + (a.p[q - 1].M + GM - 1) / GM * a.p[q - 1].tiles_n : 0;
    p.C = C;
    p.ldc = ldc;
    a.klen = (Kd + GK - 1) / GK * GK;
  };
  int rc = DLSH_OK;
  auto map = [&](int r) { rc = rc ? rc : r; };
  // layer 1 (A: the signals, normalised as they are staged) and layer 2
  prod(t.l1, 0, M, HID, XIN, w.Z1, HID);
  map(kmajor(&t.l1.p[0].B, b.Pb + L.W1, HID, XIN, XIN));
  t.l1.Xn = w.Xn;
  t.l1.bias = b.P + L.b1;
  t.l1.H = w.H1;
  t.l1.ldh = HID;
  prod(t.l2, 0, M, HID, HID, w.Z2, HID);
  map(kmajor(&t.l2.p[0].A, w.H1, M, HID, HID));
  map(kmajor(&t.l2.p[0].B, b.Pb + L.W2, HID, HID, HID));
  t.l2.bias = b.P + L.b2;
  t.l2.H = w.H2;
  t.l2.ldh = HID;
  // logits -> dZ3, column sums (b3) and loss
  prod(t.l3, 0, M, K, HID, nullptr, 0);
  map(kmajor(&t.l3.p[0].A, w.H2, M, HID, HID));
  map(kmajor(&t.l3.p[0].B, b.Pb + L.W3, K, HID, HID));
  t.l3.bias = b.P + L.b3;
  t.l3.H = w.dZ3;
  t.l3.ldh = w.ldk;
  t.l3.colpart = w.cp3;
  t.l3.loss_part = w.loss_part;
  // dZ2 = (dZ3 W3) * gelu'(Z2), dZ1 = (dZ2 W2) * gelu'(Z1); the weights are
  // read MN-major (their rows are the k of these products)
  prod(t.d2, 0, M, HID, K, nullptr, 0);
  map(kmajor(&t.d2.p[0].A, w.dZ3, M, w.ldk, w.ldk));
  map(mnmajor(&t.d2.p[0].B, b.Pb + L.W3, HID, K, HID));
  t.d2.Z = w.Z2;
  t.d2.H = w.dZ2;
  t.d2.ldh = HID;
  t.d2.colpart = w.cp2;
  prod(t.d1, 0, M, HID, HID, nullptr, 0);
  map(kmajor(&t.d1.p[0].A, w.dZ2, M, HID, HID));
  map(mnmajor(&t.d1.p[0].B, b.Pb + L.W2, HID, HID, HID));
  t.d1.Z = w.Z1;
  t.d1.H = w.dZ1;
  t.d1.ldh = HID;
  t.d1.colpart = w.cp1;
  // dW = dZ^T A_in of the three layers, both operands MN-major (k = the batch)
  t.wg.nprod = 3;
  prod(t.wg, 0, K, HID, M, w.part + L.W3, HID);
  map(mnmajor(&t.wg.p[0].A, w.dZ3, w.ldk, M, w.ldk));
  map(mnmajor(&t.wg.p[0].B, w.H2, HID, M, HID));
  prod(t.wg, 1, HID, HID, M, w.part + L.W2, HID);
  map(mnmajor(&t.wg.p[1].A, w.dZ2, HID, M, HID));
  map(mnmajor(&t.wg.p[1].B, w.H1, HID, M, HID));
  prod(t.wg, 2, HID, XIN, M, w.part + L.W1, XIN);
  map(mnmajor(&t.wg.p[2].A, w.dZ1, HID, M, HID));
  map(mnmajor(&t.wg.p[2].B, w.Xn, XIN, M, XIN));
  t.wg.klen = w.klen;
  t.wg.zstride = w.zstride;
  return rc;
}

// Forward and backward of one batch: weight-gradient partials, column sums and
// loss sums in the workspace.
static int backward(Plan& t, const float* X, const uint16_t* idx, const uint8_t* nnz, const TWs& w,
                    cudaStream_t st) {
  t.l1.X = X;
  t.l3.idx = idx;
  t.l3.nnz = nnz;
  auto tiles = [&](const GemmArgs& g) { return g.p[0].tiles_n * w.tiles_m; };
  int rc = launch_gemm<EPI_GELU, false, false, true>(t.l1, tiles(t.l1), 1, st);
  if (!rc) rc = launch_gemm<EPI_GELU, false, false, false>(t.l2, tiles(t.l2), 1, st);
  if (!rc) rc = launch_gemm<EPI_BCE, false, false, false>(t.l3, tiles(t.l3), 1, st);
  if (!rc) rc = launch_gemm<EPI_GELU_BWD, false, true, false>(t.d2, tiles(t.d2), 1, st);
  if (!rc) rc = launch_gemm<EPI_GELU_BWD, false, true, false>(t.d1, tiles(t.d1), 1, st);
  if (!rc) rc = launch_gemm<EPI_PART, true, true, false>(t.wg, w.tiles_w, w.splits, st);
  return rc;
}

static ReduceArgs reduce_args(int K, long long B, const TWs& w, float* loss) {
  ReduceArgs a{};
  a.part = w.part;
  a.zstride = w.zstride;
  a.splits = w.splits;
  a.cp1 = w.cp1;
  a.cp2 = w.cp2;
  a.cp3 = w.cp3;
  a.tiles = w.tiles_m;
  a.ldk = w.ldk;
  a.loss_part = w.loss_part;
  a.nloss = w.tiles_m * ((K + GN - 1) / GN);
  a.inv_bk = 1.0 / (static_cast<double>(B) * K);
  a.loss = loss;
  a.L = layout(K);
  return a;
}

// Gradients of the batch's mean loss into grads, the loss into *loss (device,
// may be NULL).
static int gradients(Plan& t, int K, const float* X, long long B, const uint16_t* idx, const uint8_t* nnz,
                     const TWs& w, float* grads, float* loss, cudaStream_t st) {
  const int rc = backward(t, X, idx, nnz, w, st);
  if (rc) return rc;
  ReduceArgs a = reduce_args(K, B, w, loss);
  a.G = grads;
  launch_dependent(reduce_kernel<false>, static_cast<int>((a.L.n + 255) / 256) + 1, 256, 0, st, a);
  count_launches(1);
  return check_launch("dlsh_mlp: reduce");
}

// The same, followed by Adam's step number `step` (from 1).
static int train_step(Plan& t, const Blob& b, int K, const float* X, long long B, const uint16_t* idx,
                      const uint8_t* nnz, const TWs& w, float lr, long long step, float* loss, cudaStream_t st) {
  const int rc = backward(t, X, idx, nnz, w, st);
  if (rc) return rc;
  ReduceArgs a = reduce_args(K, B, w, loss);
  a.b = b;
  a.lr = lr;
  a.beta1 = 0.9f;
  a.beta2 = 0.999f;
  a.eps = 1e-8f;
  a.bc1 = static_cast<float>(1.0 - pow(0.9, static_cast<double>(step)));
  a.bc2 = static_cast<float>(1.0 - pow(0.999, static_cast<double>(step)));
  launch_dependent(reduce_kernel<true>, static_cast<int>((a.L.n + 255) / 256) + 1, 256, 0, st, a);
  count_launches(1);
  return check_launch("dlsh_mlp: adam");
}

}  // namespace mlp

size_t mlp_train_ws_bytes(int K, long long B) {
  mlp::TWs w;
  return mlp::carve_t(nullptr, K, B, w);
}

}  // namespace dlsh

extern "C" {

long long dlsh_mlp_num_params(int K) { return K >= 1 ? dlsh::mlp::layout(K).n : 0; }

size_t dlsh_mlp_size(int K) {
  if (K < 1 || K > DLSH_MAX_K) return 0;
  dlsh::mlp::Blob b;
  return dlsh::mlp::carve_blob(nullptr, K, b);
}

size_t dlsh_mlp_workspace_size(int K, int64_t B) {
  if (K < 1 || K > DLSH_MAX_K || B < 1) return 0;
  return std::max(dlsh::mlp_train_ws_bytes(K, B), dlsh::propose_ws_bytes(K));
}

int dlsh_mlp_init(void* mlp, int K, const float* params, void* stream, int flags) {
  using namespace dlsh;
  clear_error();
  if (!mlp || !params || K < 1 || K > DLSH_MAX_K)
    return set_error(DLSH_ERR_INVALID_ARG, "dlsh_mlp_init: bad arguments");
  if (reinterpret_cast<uintptr_t>(mlp) % 256)
    return set_error(DLSH_ERR_INVALID_ARG, "dlsh_mlp_init: blob must be 256-byte aligned");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  mlp::Blob b;
  mlp::carve_blob(mlp, K, b);
  const long long n = mlp::layout(K).n;
  DLSH_CUDA_TRY(cudaMemcpyAsync(b.P, params, n * sizeof(float), cudaMemcpyDeviceToDevice, st),
                "dlsh_mlp_init: copy");
  DLSH_CUDA_TRY(cudaMemsetAsync(b.m1, 0, n * sizeof(float), st), "dlsh_mlp_init: m1");
  DLSH_CUDA_TRY(cudaMemsetAsync(b.m2, 0, n * sizeof(float), st), "dlsh_mlp_init: m2");
  DLSH_CUDA_TRY(cudaMemsetAsync(b.step, 0, 2 * sizeof(long long), st), "dlsh_mlp_init: step");
  mlp::mirror_kernel<<<static_cast<int>((n + 255) / 256), 256, 0, st>>>(b.P, b.Pb, n);
  count_launches(1);
  return finish(st, nullptr, flags, "dlsh_mlp_init");
}

int dlsh_mlp_params(const void* mlp, int K, float* params, void* stream, int flags) {
  using namespace dlsh;
  clear_error();
  if (!mlp || !params || K < 1) return set_error(DLSH_ERR_INVALID_ARG, "dlsh_mlp_params: bad arguments");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  mlp::Blob b;
  mlp::carve_blob(const_cast<void*>(mlp), K, b);
  DLSH_CUDA_TRY(cudaMemcpyAsync(params, b.P, mlp::layout(K).n * sizeof(float),
                                cudaMemcpyDeviceToDevice, st),
                "dlsh_mlp_params: copy");
  return finish(st, nullptr, flags, "dlsh_mlp_params");
}

static int mlp_common_checks(const char* call, const void* mlp, int K, const float* X, int64_t B,
                             void* ws, size_t ws_bytes) {
  using namespace dlsh;
  if (!mlp || K < 1 || K > DLSH_MAX_K) return set_error(DLSH_ERR_INVALID_ARG, "%s: bad blob or K", call);
  if (B < 1 || !X) return set_error(DLSH_ERR_INVALID_ARG, "%s: bad batch", call);
  return check_workspace(ws, ws_bytes, dlsh_mlp_workspace_size(K, B), call);
}

int dlsh_mlp_forward(const void* mlp, int K, const float* X, int64_t B, float* logits, void* ws,
                     size_t ws_bytes, void* stream, int flags) {
  using namespace dlsh;
  clear_error();
  int rc = mlp_common_checks("dlsh_mlp_forward", mlp, K, X, B, ws, ws_bytes);
  if (rc) return rc;
  if (!logits) return set_error(DLSH_ERR_INVALID_ARG, "dlsh_mlp_forward: NULL logits");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint32_t* status = static_cast<uint32_t*>(ws);  // both workspace layouts open with it
  DLSH_CUDA_TRY(cudaMemsetAsync(status, 0, 4, st), "dlsh_mlp_forward: reset");
  rc = infer_logits_enqueue(mlp, K, X, B, logits, ws, status, st);
  if (rc) return rc;
  return finish(st, status, flags, "dlsh_mlp_forward");
}

int dlsh_mlp_gradients(const void* mlp, int K, const float* X, int64_t B, const uint16_t* idx,
                       const uint8_t* nnz, int s, float* grads, float* loss, void* ws,
                       size_t ws_bytes, void* stream, int flags) {
  using namespace dlsh;
  clear_error();
  int rc = mlp_common_checks("dlsh_mlp_gradients", mlp, K, X, B, ws, ws_bytes);
  if (rc) return rc;
  if (!idx || !nnz || !grads || s < 1 || s > DLSH_MAX_S)
    return set_error(DLSH_ERR_INVALID_ARG, "dlsh_mlp_gradients: bad targets");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  mlp::Blob b;
  mlp::carve_blob(const_cast<void*>(mlp), K, b);
  mlp::TWs w;
  mlp::carve_t(ws, K, B, w);
  DLSH_CUDA_TRY(cudaMemsetAsync(w.status, 0, 4, st), "dlsh_mlp_gradients: reset");
  mlp::Plan plan;
  rc = mlp::make_plan(b, K, static_cast<int>(B), w, s, plan);
  if (rc) return rc;
  rc = mlp::gradients(plan, K, X, B, idx, nnz, w, grads, loss, st);
  if (rc) return rc;
  return finish(st, w.status, flags, "dlsh_mlp_gradients");
}

int dlsh_mlp_train_step(void* mlp, int K, const float* X, int64_t B, const uint16_t* idx,
                        const uint8_t* nnz, int s, float lr, int64_t step, float* loss, void* ws,
                        size_t ws_bytes, void* stream, int flags) {
  using namespace dlsh;
  clear_error();
  int rc = mlp_common_checks("dlsh_mlp_train_step", mlp, K, X, B, ws, ws_bytes);
  if (rc) return rc;
  if (!idx || !nnz || s < 1 || s > DLSH_MAX_S || step < 1)
    return set_error(DLSH_ERR_INVALID_ARG, "dlsh_mlp_train_step: bad arguments");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  mlp::Blob b;
  mlp::carve_blob(mlp, K, b);
  mlp::TWs w;
  mlp::carve_t(ws, K, B, w);
  DLSH_CUDA_TRY(cudaMemsetAsync(w.status, 0, 4, st), "dlsh_mlp_train_step: reset");
  mlp::Plan plan;
  rc = mlp::make_plan(b, K, static_cast<int>(B), w, s, plan);
  if (rc) return rc;
  rc = mlp::train_step(plan, b, K, X, B, idx, nnz, w, lr, step, loss, st);
  if (rc) return rc;
  return finish(st, w.status, flags, "dlsh_mlp_train_step");
}

int dlsh_mlp_train(void* mlp, int K, const float* X, int64_t N, const uint16_t* idx,
                   const uint8_t* nnz, int s, int epochs, int64_t batch, float lr,
                   float* loss_per_step, void* ws, size_t ws_bytes, void* stream, int flags) {
  using namespace dlsh;
  clear_error();
  if (batch < 1 || N < batch || epochs < 1)
    return set_error(DLSH_ERR_INVALID_ARG, "dlsh_mlp_train: need epochs >= 1 and N >= batch >= 1");
  int rc = mlp_common_checks("dlsh_mlp_train", mlp, K, X, batch, ws, ws_bytes);
  if (rc) return rc;
  if (!idx || !nnz || s < 1 || s > DLSH_MAX_S)
    return set_error(DLSH_ERR_INVALID_ARG, "dlsh_mlp_train: bad targets");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  mlp::Blob b;
  mlp::carve_blob(mlp, K, b);
  mlp::TWs w;
  mlp::carve_t(ws, K, batch, w);
  DLSH_CUDA_TRY(cudaMemsetAsync(w.status, 0, 4, st), "dlsh_mlp_train: reset");
  mlp::Plan plan;
  rc = mlp::make_plan(b, K, static_cast<int>(batch), w, s, plan);
  if (rc) return rc;
  const long long per_epoch = N / batch;
  const long long total = per_epoch * epochs;
  long long step = 0;
  for (int e = 0; e < epochs; ++e) {
    for (long long q = 0; q < per_epoch; ++q) {
      ++step;
      // cosine decay from lr to 0 over all steps
      const double frac = static_cast<double>(step - 1) / static_cast<double>(total);
      const float lr_t = static_cast<float>(0.5 * lr * (1.0 + cos(M_PI * frac)));
      const long long off = q * batch;
      rc = mlp::train_step(plan, b, K, X + off * DLSH_D, batch, idx + off * s, nnz + off, w, lr_t, step,
                           loss_per_step ? loss_per_step + (step - 1) : nullptr, st);
      if (rc) return rc;
    }
  }
  return finish(st, w.status, flags, "dlsh_mlp_train");
}

}  // extern "C"
