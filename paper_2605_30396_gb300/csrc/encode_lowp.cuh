// Batch-OMP with BF16 or FP8 correlations, s <= 8: two tiles per CTA with the
// warps split by task, as in the FP32 split encoder.
//
// Included by encode_core.cuh after encode_pair.cuh, whose plan, chunk width (64
// atoms), candidate keys and arithmetic it shares: the codes are bitwise those
// of the two-group kernel, which serves these precisions where there are fewer
// than four chunks.  There each group of eight warps selects and then solves its
// own tile, so that the ALU-bound top-4 network and the load-bound solver of a
// tile take turns (23,000 cycles per tile and iteration on an SM at K = 1024).  Here
//   warps 0-7   select: warp w reads tensor-memory lane quarter w & 3 and the
//               column half w >> 2 of every chunk, one job ahead of the solver;
//   warps 8-15  re-score the candidates in FP32 and solve, two lanes per row;
//   warp 16     issues the MMAs (A in shared memory, one operand per tile slot)
//               into a ring of eight 64-column accumulator buffers;
//   warp 17     streams the dictionary.
// N = 1M, K = 1024, s = 8, BF16: 4590 -> 4393 us; N = 10,000, K = 256 (a tile per
// SM): 159 -> 94.  Bound by the selection: about 1340 cycles per chunk on two
// warps per scheduler, whose min/max network fills the integer pipe to 77 % and
// is a chain of a dozen dependent steps.  (Halves of a chunk with the next load
// in flight: 4456 us; minima as multiply-adds on the other pipe: 4610.)

constexpr int LBUF = 8;  // accumulator buffers (all 512 tensor-memory columns)

template <int PREC, bool T4>
__global__ void __launch_bounds__(NTHREADS, 1) encode_lowp_kernel(const __grid_constant__ PairArgs a) {
  static_assert(PREC != 0, "low-precision correlations");
  extern __shared__ __align__(1024) uint8_t smem[];
  const PairPlan& p = a.p;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long NS = a.n_dev ? *a.n_dev : a.N;
  const int ntiles = static_cast<int>((NS + TILE_M - 1) / TILE_M);
  const int Gd = static_cast<int>(gridDim.x), bidx = static_cast<int>(blockIdx.x);
  const int s = p.s, K = p.K, nchunks = p.nchunks;
  // rounds k in which tile slot t has a tile (tiles b + (2 k + t) Gd), K0 >= K1
  const int K0 = bidx < ntiles ? (ntiles - bidx + 2 * Gd - 1) / (2 * Gd) : 0;
  const int K1 = bidx + Gd < ntiles ? (ntiles - bidx - Gd + 2 * Gd - 1) / (2 * Gd) : 0;
  auto slots_in = [&](int k) { return k < K1 ? 2 : 1; };
  auto tile_of = [&](int t, int k) -> long long { return static_cast<long long>(bidx) + (2LL * k + t) * Gd; };

  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + p.off_bar);
  uint64_t* bar_a = bars;                    // [2] a slot's A operand is written
  uint64_t* bar_full = bars + 2;             // [LBUF] a buffer holds a chunk's correlations
  uint64_t* bar_empty = bar_full + LBUF;     // [LBUF] it has been read
  uint64_t* cand_full = bar_empty + LBUF;    // [2] a slot's candidates are written
  uint64_t* cand_empty = cand_full + 2;      // [2] the solver has read them
  uint64_t* bar_dfull = cand_empty + 2;      // [stages]
  uint64_t* bar_dempty = bar_dfull + p.stages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_dempty + p.stages);

  if (tid == 0) {
    for (int t = 0; t < 2; ++t) {
      mbar_init(&bar_a[t], 1);
      mbar_init(&cand_full[t], SPW);
      mbar_init(&cand_empty[t], SVT / 32);
    }
    for (int b = 0; b < LBUF; ++b) {
      mbar_init(&bar_full[b], 1);
      mbar_init(&bar_empty[b], SPW);
    }
    for (int q = 0; q < p.stages; ++q) {
      mbar_init(&bar_dfull[q], 1);
      mbar_init(&bar_dempty[q], 1);
    }
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  if constexpr (PREC == 2) {
    float* sig = reinterpret_cast<float*>(smem + p.off_sig);
    for (int j = tid; j < p.Kp; j += NTHREADS) sig[j] = a.sigma[j];
    // FP8 rows hold 64 bytes: bytes 48..63 are zero padding, written once
    for (int row = tid; row < 2 * TILE_M; row += NTHREADS)
      *reinterpret_cast<uint4*>(smem + p.off_a[row / TILE_M] + 3 * TILE_M * 16 + (row % TILE_M) * 16) =
          make_uint4(0, 0, 0, 0);
    fence_proxy_async_smem();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const uint32_t ring_addr = smem_u32(smem + p.off_ring);

  if (warp == NEPI / 32 + 1) {
    // ------------------------------------------------ TMA producer
    if (lane == 0) {
      const long long njobs = static_cast<long long>(s) * (K0 + K1);
      long long n = 0;
      int st = 0;
      uint32_t par = 1u;
      bool ok = true;
      for (long long j = 0; j < njobs && ok; ++j)
        for (int c = 0; c < nchunks; ++c, ++n) {
          if (!mbar_wait(&bar_dempty[st], par, a.budget)) {
            flag_status(a.status, ST_TIMEOUT);
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(&bar_dfull[st], p.chunk_bytes);
          bulk_g2s(smem + p.off_ring + static_cast<size_t>(st) * p.chunk_bytes,
                   a.img + static_cast<size_t>(c) * p.chunk_bytes, p.chunk_bytes, &bar_dfull[st]);
          if (++st == p.stages) {
            st = 0;
            par ^= 1u;
          }
        }
      // every stage's last fill has been consumed before the CTA exits
      for (long long f = n > p.stages ? n - p.stages : 0; ok && f < n; ++f)
        if (!mbar_wait(&bar_dempty[f % p.stages], static_cast<uint32_t>((f / p.stages) & 1), a.budget)) {
          flag_status(a.status, ST_TIMEOUT);
          ok = false;
        }
    }
  } else if (warp == NEPI / 32) {
    // ------------------------------------------------ MMA issuer
    if (lane == 0) {
      uint32_t aph[2] = {0u, 0u};
      int st = 0, buf = 0;
      uint32_t dpar = 0u, epar = 1u;
      bool ok = true;
      for (int k = 0; k < K0 && ok; ++k)
        for (int it = 0; it < s && ok; ++it)
          for (int t = 0; t < slots_in(k) && ok; ++t) {
            if (!mbar_wait(&bar_a[t], aph[t], a.budget)) {
              flag_status(a.status, ST_TIMEOUT);
              ok = false;
              break;
            }
            aph[t] ^= 1u;
            const uint32_t aa = smem_u32(smem + p.off_a[t]);
            for (int c = 0; c < nchunks; ++c) {
              if (!mbar_wait(&bar_dfull[st], dpar, a.budget) || !mbar_wait(&bar_empty[buf], epar, a.budget)) {
                flag_status(a.status, ST_TIMEOUT);
                ok = false;
                break;
              }
              tc_fence_after();
              issue_chunk<PREC, PBN>(tmem_base + static_cast<uint32_t>(buf) * PBN, aa,
                                     ring_addr + static_cast<uint32_t>(st) * p.chunk_bytes);
              tc_commit(&bar_full[buf]);
              tc_commit(&bar_dempty[st]);
              if (++st == p.stages) {
                st = 0;
                dpar ^= 1u;
              }
              if (++buf == LBUF) {
                buf = 0;
                epar ^= 1u;
              }
            }
          }
    }
  } else if (warp < SPW) {
    // ------------------------------------------------ selection, one job ahead of the solver
    const int wq = warp & 3, h = warp >> 2;
    const int R1 = 32 * wq + lane;
    const uint32_t trow = tmem_base + (static_cast<uint32_t>(32 * wq) << 16) + static_cast<uint32_t>(h * PQC);
    const float* sig = reinterpret_cast<const float*>(smem + p.off_sig);
    int sbuf = 0;
    uint32_t spar = 0u, epar = 3u;  // bit t of epar: cand_empty parity to wait for (the first pass is free)
    bool ok = true;
    for (int k = 0; k < K0 && ok; ++k)
      for (int it = 0; it < s && ok; ++it)
        for (int t = 0; t < slots_in(k) && ok; ++t) {
          uint32_t best = 0;
          int bestc = 0;
          const uint32_t vmask = 0x7fffffffu & ~((1u << p.ib) - 1u);
          uint32_t run[4] = {0u, 0u, 0u, 0u};
          for (int c = 0; c < nchunks; ++c) {
            const int buf = sbuf;
            const uint32_t par = spar;
            if (++sbuf == LBUF) {
              sbuf = 0;
              spar ^= 1u;
            }
            if (!mbar_wait(&bar_full[buf], par, a.budget)) {
              flag_status(a.status, ST_TIMEOUT);
              ok = false;
              break;
            }
            tc_fence_after();
            __syncwarp();
            uint32_t rr[PQC];
            tmem_ld32_issue(trow + static_cast<uint32_t>(buf * PBN), rr);
            tmem_ld32_wait(rr);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_empty[buf]);
            if constexpr (PREC == 2) {
              const int j0 = c * PBN + h * PQC;
#pragma unroll
              for (int q = 0; q < PQC; ++q) rr[q] = __float_as_uint(__uint_as_float(rr[q]) * sig[j0 + q]);
            }
            if constexpr (T4) {
#pragma unroll
              for (int q = 0; q < PQC; ++q) rr[q] = (rr[q] & vmask) | static_cast<uint32_t>(31 - q);
              uint32_t ct[4];
              top4_of8(rr, ct);
#pragma unroll
              for (int o = 8; o < PQC; o += 8) {
                uint32_t t8[4];
                top4_of8(rr + o, t8);
                merge_top4(ct, t8);
              }
              const uint32_t cf = ((1u << p.ib) - 32u) - static_cast<uint32_t>(c) * 32u;
#pragma unroll
              for (int i = 0; i < 4; ++i) ct[i] |= cf;
              merge_top4(run, ct);
            } else {
              uint32_t m0 = 0, m1 = 0;
#pragma unroll
              for (int q = 0; q < PQC; q += 2) {
                m0 = max(m0, (rr[q] & 0x7fffffe0u) | static_cast<uint32_t>(31 - q));
                m1 = max(m1, (rr[q + 1] & 0x7fffffe0u) | static_cast<uint32_t>(30 - q));
              }
              const uint32_t m = max(m0, m1);
              if ((m & ~31u) > (best & ~31u)) {
                best = m;
                bestc = c;
              }
            }
          }
          if (!ok) break;
          if (!mbar_wait(&cand_empty[t], (epar >> t) & 1u, a.budget)) {
            flag_status(a.status, ST_TIMEOUT);
            ok = false;
            break;
          }
          epar ^= 1u << t;
          if constexpr (T4) {
            uint32_t* ckeys = reinterpret_cast<uint32_t*>(smem + p.off_cand[t]);  // [128][2][4]
            *reinterpret_cast<uint4*>(ckeys + (R1 * 2 + h) * 4) = make_uint4(run[0], run[1], run[2], run[3]);
          } else {
            float* cv = reinterpret_cast<float*>(smem + p.off_cand[t]);  // [128][2]
            int* cj = reinterpret_cast<int*>(smem + p.off_cand[t] + TILE_M * 2 * 4);
            cv[R1 * 2 + h] = __uint_as_float(best & ~31u);
            cj[R1 * 2 + h] = bestc * PBN + h * PQC + 31 - static_cast<int>(best & 31u);
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(&cand_full[t]);
        }
  } else {
    // ------------------------------------------------ solver: two lanes per row
    const int vt = tid - SPW * 32, vw = vt >> 5;
    const int R2 = 16 * vw + (lane >> 1), u = lane & 1;
    const float eps2 = a.eps * a.eps;
    uint32_t fpar = 0u;  // bit t: cand_full parity to wait for at slot t
    bool ok = true;
    // per-slot row state: ||r||^2, ||x||, atoms taken (bit 8: the row has stopped)
    auto st_rn2 = [&](int t) { return reinterpret_cast<float*>(smem + p.off_row[t]); };
    auto st_xn = [&](int t) { return reinterpret_cast<float*>(smem + p.off_row[t]) + TILE_M; };
    auto st_tc = [&](int t) { return reinterpret_cast<int*>(smem + p.off_row[t]) + 2 * TILE_M; };
    auto rows_of = [&](long long tl) -> int {
      const long long g0 = tl * TILE_M;
      return static_cast<int>(NS - g0 < TILE_M ? NS - g0 : TILE_M);
    };
    // the signals of tile tl are slot t's first A operand and residual
    auto stage_x = [&](int t, long long tl) {
      const bool in = R2 < rows_of(tl);
      const float* xr = a.X + (tl * TILE_M + R2) * DLSH_D + 24 * u;
      float x[24];
#pragma unroll
      for (int q = 0; q < 24; ++q) x[q] = (in && 24 * u + q < DLSH_D) ? __ldg(xr + q) : 0.f;
      float part = 0.f;
#pragma unroll
      for (int q = 0; q < 24; ++q) part = fmaf(x[q], x[q], part);
      float inv = 1.f;
      if constexpr (PREC == 2) {
        float mx = 0.f;
#pragma unroll
        for (int q = 0; q < 24; ++q) mx = fmaxf(mx, fabsf(x[q]));
        mx = pair_max(mx);
        inv = mx > 0.f ? FP8_MAX / mx : 1.f;
      }
      write_a_part24<PREC>(smem + p.off_a[t], R2, u, x, inv);
      float* rsm = reinterpret_cast<float*>(smem + p.off_r[t]);
#pragma unroll
      for (int q = 0; q < 24; ++q) rsm[q * PGT + vt] = x[q];
      const float rn2 = pair_sum(part);
      st_rn2(t)[R2] = rn2;
      st_xn(t)[R2] = sqrtf(rn2);
      st_tc(t)[R2] = in ? 0 : 0x100;
    };
#pragma unroll 1
    for (int t = 0; t < 2; ++t)
      if ((t == 0 ? K0 : K1) > 0) {
        stage_x(t, tile_of(t, 0));
        fence_proxy_async_smem();
        named_bar_sync(1, SVT);
        if (vt == 0) mbar_arrive(&bar_a[t]);
      }
    for (int k = 0; k < K0 && ok; ++k)
      for (int it = 0; it < s && ok; ++it)
#pragma unroll 1
        for (int t = 0; t < slots_in(k); ++t) {
          if (!mbar_wait(&cand_full[t], (fpar >> t) & 1u, a.budget)) {
            flag_status(a.status, ST_TIMEOUT);
            ok = false;
          }
          fpar ^= 1u << t;
          uint8_t* A = smem + p.off_a[t];
          float* Ls = reinterpret_cast<float*>(smem + p.off_L[t]);
          int* sel = reinterpret_cast<int*>(smem + p.off_sel[t]);
          float* ys = reinterpret_cast<float*>(smem + p.off_y[t]);
          float* gs = reinterpret_cast<float*>(smem + p.off_g[t]);
          float* idg = reinterpret_cast<float*>(smem + p.off_idg[t]);
          float* rsm = reinterpret_cast<float*>(smem + p.off_r[t]);  // [24][256]
#define LS(rr, cc2) Ls[(((rr) * ((rr) + 1)) / 2 + (cc2)) * TILE_M + R2]
#define IDG(rr) idg[(rr) * TILE_M + R2]
          // this lane's candidates into registers, then release the area
          uint4 keys = make_uint4(0u, 0u, 0u, 0u);
          int cw0 = 0, cw1 = 0;
          if constexpr (T4) {
            keys = *reinterpret_cast<const uint4*>(smem + p.off_cand[t] + static_cast<size_t>((R2 * 2 + u) * 4) * 4);
          } else {
            const int* cj = reinterpret_cast<const int*>(smem + p.off_cand[t] + TILE_M * 2 * 4);
            cw0 = cj[R2 * 2 + 0];
            cw1 = cj[R2 * 2 + 1];
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(&cand_empty[t]);
          const long long tl = tile_of(t, k);
          const int64_t g0 = tl * TILE_M;
          const bool in_tile = R2 < rows_of(tl);
          const float* xr = a.X + (g0 + R2) * DLSH_D + 24 * u;
          auto load_x = [&](float (&x)[24]) {
#pragma unroll
            for (int q = 0; q < 24; ++q) x[q] = (in_tile && 24 * u + q < DLSH_D) ? __ldg(xr + q) : 0.f;
          };
          float rn2c = st_rn2(t)[R2];
          const float xnorm = st_xn(t)[R2];
          const int stc = st_tc(t)[R2];
          int tcc = stc & 0xff;
          bool act = ok && (stc & 0x100) == 0;
          if (act && rn2c <= eps2) act = false;
          if (act) {
            float r[24];
            int sl[8];
#pragma unroll
            for (int m = 0; m < 8; ++m) sl[m] = m < tcc ? sel[m * TILE_M + R2] : 0;
            int js = -1;
            float best = -1.f;
#pragma unroll
            for (int q = 0; q < 24; ++q) r[q] = rsm[q * PGT + vt];
            // candidates: T4, the row's exact low-precision top 4 (sub-lane u
            // reads half u's list, one butterfly round); else the winner of
            // each column half
            int cjr[4];
            if constexpr (T4) {
              const uint32_t imask = (1u << p.ib) - 1u;
              unsigned long long lst[4];
              const uint32_t kv[4] = {keys.x, keys.y, keys.z, keys.w};
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const uint32_t key = kv[i];
                const uint32_t col = imask - (key & imask);
                const uint32_t j = (col >> 5) * PBN + static_cast<uint32_t>(u * PQC) + (col & 31u);
                lst[i] = key == 0u ? 0ull
                                   : (static_cast<unsigned long long>(key & ~imask & 0x7fffffffu) << 32) |
                                         static_cast<unsigned long long>(0xFFFFFFFFu - j);
              }
              unsigned long long oth[4];
#pragma unroll
              for (int i = 0; i < 4; ++i) oth[i] = __shfl_xor_sync(pair_mask(), lst[i], 1);
              merge_top4(lst, oth);
#pragma unroll
              for (int i = 0; i < 4; ++i)
                cjr[i] = lst[i] == 0ull ? 0x7fffffff
                                        : static_cast<int>(0xFFFFFFFFu - static_cast<uint32_t>(lst[i]));
            } else {
              cjr[0] = cw0;
              cjr[1] = cw1;
              cjr[2] = cjr[3] = 0x7fffffff;
            }
#pragma unroll
            for (int qq = 0; qq < 4; ++qq) {
              const int j = cjr[qq];
              float c0 = 0.f;
              if (j < K) {
                const float4* dr = reinterpret_cast<const float4*>(a.D32p + static_cast<size_t>(j) * DPAD + 24 * u);
#pragma unroll
                for (int w4 = 0; w4 < 6; ++w4) {
                  const float4 dv = __ldg(dr + w4);
                  c0 = fmaf(r[4 * w4 + 0], dv.x, c0);
                  c0 = fmaf(r[4 * w4 + 1], dv.y, c0);
                  c0 = fmaf(r[4 * w4 + 2], dv.z, c0);
                  c0 = fmaf(r[4 * w4 + 3], dv.w, c0);
                }
              }
              c0 = fabsf(pair_sum(c0));
              if (j < K && (c0 > best || (c0 == best && j < js))) {
                best = c0;
                js = j;
              }
            }
            // an atom already in the support has the largest |c| only when every
            // correlation is at rounding level: the row stops
            bool dup = false;
#pragma unroll
            for (int m = 0; m < 8; ++m) dup |= (m < tcc && sl[m] == js);
            if (dup) js = -1;
            if (js < 0 || !(best > CORR_STOP_REL * xnorm)) {
              act = false;
            } else {
            // the step for a support of t atoms, compiled once per t
            auto step = [&](auto tag) {
              constexpr int T = decltype(tag)::value;
              constexpr int TA = T > 0 ? T : 1;
              const float* Grow = a.G + static_cast<size_t>(js) * K;
              float gv[TA];
#pragma unroll
              for (int m = 0; m < T; ++m) gv[m] = __ldg(Grow + sl[m]);
              const float gjj = __ldg(Grow + js);
              float4 dj[6];
              {
                const float4* dr = reinterpret_cast<const float4*>(a.D32p + static_cast<size_t>(js) * DPAD + 24 * u);
#pragma unroll
                for (int w4 = 0; w4 < 6; ++w4) dj[w4] = __ldg(dr + w4);
              }
              load_x(r);  // r holds x until the residual is formed
              float w[TA];
              float wn2 = 0.f;
#pragma unroll
              for (int m = 0; m < T; ++m) {
                float acc = gv[m];
#pragma unroll
                for (int q = 0; q < m; ++q) acc = fmaf(-LS(m, q), w[q], acc);
                w[m] = acc * IDG(m);
                wn2 = fmaf(w[m], w[m], wn2);
              }
              const float ell2 = gjj - wn2;
              if (!(ell2 > PIVOT_MIN * gjj)) {
                act = false;
                return;
              }
              const float ell = sqrtf(ell2);
              const float iell = 1.f / ell;
#pragma unroll
              for (int m = 0; m < T; ++m) LS(T, m) = w[m];  // both sub-lanes store identical values
              LS(T, T) = ell;
              IDG(T) = iell;
              float bp = 0.f;
#pragma unroll
              for (int w4 = 0; w4 < 6; ++w4) {
                bp = fmaf(dj[w4].x, r[4 * w4 + 0], bp);
                bp = fmaf(dj[w4].y, r[4 * w4 + 1], bp);
                bp = fmaf(dj[w4].z, r[4 * w4 + 2], bp);
                bp = fmaf(dj[w4].w, r[4 * w4 + 3], bp);
              }
              float yv[TA];
#pragma unroll
              for (int m = 0; m < T; ++m) yv[m] = ys[m * TILE_M + R2];
              float yt = pair_sum(bp);
#pragma unroll
              for (int m = 0; m < T; ++m) yt = fmaf(-w[m], yv[m], yt);
              yt *= iell;
              ys[T * TILE_M + R2] = yt;
              sel[T * TILE_M + R2] = js;
              const float gt = yt * iell;
              float gam[TA];
#pragma unroll
              for (int m = T - 1; m >= 0; --m) {
                float acc = yv[m];
#pragma unroll
                for (int q = m + 1; q < T; ++q) acc = fmaf(-LS(q, m), gam[q], acc);
                acc = fmaf(-w[m], gt, acc);
                gam[m] = acc * IDG(m);
              }
#pragma unroll
              for (int m = 0; m < T; ++m) gs[m * TILE_M + R2] = gam[m];
              gs[T * TILE_M + R2] = gt;
              // residual r = x - D_I gamma on this sub-lane's 24 dims
              // the support atoms' rows in groups of up to 2, all loads of a
              // group issued before its FMAs (one L2 round trip per group)
#pragma unroll
              for (int m0 = 0; m0 < T; m0 += 2) {
                float4 dv[2][6];
#pragma unroll
                for (int mm = 0; mm < 2; ++mm)
                  if (m0 + mm < T) {
                    const float4* da =
                        reinterpret_cast<const float4*>(a.D32p + static_cast<size_t>(sl[m0 + mm]) * DPAD + 24 * u);
#pragma unroll
                    for (int w4 = 0; w4 < 6; ++w4) dv[mm][w4] = __ldg(da + w4);
                  }
#pragma unroll
                for (int mm = 0; mm < 2; ++mm)
                  if (m0 + mm < T) {
                    const float gm = gam[m0 + mm];
#pragma unroll
                    for (int w4 = 0; w4 < 6; ++w4) {
                      r[4 * w4 + 0] = fmaf(-gm, dv[mm][w4].x, r[4 * w4 + 0]);
                      r[4 * w4 + 1] = fmaf(-gm, dv[mm][w4].y, r[4 * w4 + 1]);
                      r[4 * w4 + 2] = fmaf(-gm, dv[mm][w4].z, r[4 * w4 + 2]);
                      r[4 * w4 + 3] = fmaf(-gm, dv[mm][w4].w, r[4 * w4 + 3]);
                    }
                  }
              }
#pragma unroll
              for (int w4 = 0; w4 < 6; ++w4) {
                r[4 * w4 + 0] = fmaf(-gt, dj[w4].x, r[4 * w4 + 0]);
                r[4 * w4 + 1] = fmaf(-gt, dj[w4].y, r[4 * w4 + 1]);
                r[4 * w4 + 2] = fmaf(-gt, dj[w4].z, r[4 * w4 + 2]);
                r[4 * w4 + 3] = fmaf(-gt, dj[w4].w, r[4 * w4 + 3]);
              }
              tcc = T + 1;
              float pr = 0.f;
#pragma unroll
              for (int q = 0; q < 24; ++q) pr = fmaf(r[q], r[q], pr);
              rn2c = pair_sum(pr);
              if (it + 1 < s) {
                float inv = 1.f;
                if constexpr (PREC == 2) {
                  float mx = 0.f;
#pragma unroll
                  for (int q = 0; q < 24; ++q) mx = fmaxf(mx, fabsf(r[q]));
                  mx = pair_max(mx);
                  inv = mx > 0.f ? FP8_MAX / mx : 1.f;
                }
                write_a_part24<PREC>(A, R2, u, r, inv);
              }
#pragma unroll
              for (int q = 0; q < 24; ++q) rsm[q * PGT + vt] = r[q];
            };
              if (tcc < 8)
                with_t<8>(tcc, step);
              else
                act = false;
            }
          }
          st_rn2(t)[R2] = rn2c;
          st_tc(t)[R2] = tcc | (act ? 0 : 0x100);
          const bool last = it + 1 == s;
          const bool next = k + 1 < (t == 0 ? K0 : K1);
          if (last) {  // the tile's codes, then the slot's next tile
            if (in_tile) {
              const int64_t gi = g0 + R2;
              for (int mm = u; mm < s; mm += 2) {
                a.idx[gi * s + mm] = mm < tcc ? static_cast<uint16_t>(sel[mm * TILE_M + R2]) : static_cast<uint16_t>(0);
                a.coef[gi * s + mm] = mm < tcc ? gs[mm * TILE_M + R2] : 0.f;
              }
              if (u == 0) {
                a.nnz[gi] = static_cast<uint8_t>(tcc);
                if (a.resid_sq) a.resid_sq[gi] = rn2c;
              }
            }
            if (next && ok) stage_x(t, tile_of(t, k + 1));
          }
#undef LS
#undef IDG
          fence_proxy_async_smem();
          if (named_bar_or(1, SVT, !ok)) {
            ok = false;
            break;
          }
          if ((!last || next) && vt == 0) mbar_arrive(&bar_a[t]);
        }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}
