// Tied-array beams on the tensor cores (Eq. bp_max_arbitrary as a GEMM) when the E-W axis
// is on the FFT-beam grid (pad_x < 2 nx - 1, at most 4 E-W beams): per channel f,
//   out[j, s] = sum_B wx[s, A_s] wy[s, B] P[j, f, A_s, B],
// a [pointings x beams] x [beams x windows] product for each E-W beam A. Operands are
// split FP16 pairs, x = 2^-e (hi + lo) with hi = fp16(2^e x), lo = fp16(2^e x - hi), and
// each K step accumulates hi*hi + hi*lo + lo*hi in FP32 (tcgen05.mma kind::f16, TMEM), which
// keeps FP32 accuracy; e scales every weight row and every beam row so that its largest
// magnitude lies in [2^14, 2^15) (inside the FP16 range, with the residuals normal), and the
// epilogue divides by 2^(e_s + e_j) exactly. Both split operands are stored in global
// memory already cut into tiles (128 pointings or 64 windows x 32 beams, the canonical K-major
// layout, zero rows past the ends). A CTA computes 128 pointings x 64 windows of one channel: one
// thread stages each K chunk as four bulk copies completing on a full-mbarrier (four stages),
// another issues its MMAs and commits them to the stage's empty-mbarrier; one TMEM accumulator
// of 64 columns per E-W beam used by the tile's pointings, and each pointing (TMEM lane) reads
// its own beam's accumulator. Every wait is bounded; a timeout sets the
// plan's error word.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>

#include "internal.cuh"
#include "tc_ptx.cuh"

namespace fftbf {

namespace ttc {
constexpr int TM = 128, KC = 32;               // pointings, beams per K chunk
constexpr int LBO = 128, SBO = 512;            // canonical K-major tile: 4 K blocks per row group
constexpr int TILE = TM * KC * 2;              // bytes of one 128 x 32 FP16 tile
constexpr int NT = 256;                        // warps w and w + 4 share TMEM lane quarter w % 4
constexpr int MAXA = 4;                        // E-W beams (one accumulator each)
// Windows per CTA. 64, because two CTAs then fit on an SM, so that one's set-up and scattered stores
// run under the other's products; the second window tile of a channel finds the weights in L2.
// 256 channels x 2048 pointings, whose split weights are 1.07 GB per call (156 us at the copy rate),
// against tiles of 128 windows with one CTA per SM: 245 for 482 us at 64 windows, 416 for 482 at 128,
// 783 for 921 at 256; 64 channels x 300 pointings x 128 windows of 4x64: 21 for 28 us.
constexpr int TN = 64;
constexpr int PT = TN * KC * 2;                // bytes of one TN x 32 beam tile
constexpr int STAGE = 2 * TILE + 2 * PT;       // W hi, W lo, P hi, P lo
// Staging buffers. Chunks of 32 beams in four rather than of 64 in two: a stage is given back sooner,
// so more of the buffers are in flight (336 -> 245 us at 64 windows, with the copy thread).
constexpr int NS = 4;
constexpr uint32_t TMEM_COLS = MAXA * TN;
constexpr uint64_t WAIT_NS = 1000000000ull;
}  // namespace ttc

// e such that 2^e m lies in [2^14, 2^15) (0 for a zero row)
__device__ __forceinline__ int split_exp(float m) { return m > 0.f ? 14 - ilogbf(m) : 0; }

// Half offset of element (row r < 128, k) of a row tile: tile (k / 32) of the row tile's
// chunks, canonical K-major layout inside.
__device__ __forceinline__ int64_t tiled_off(int64_t tile0, int r, int k) {
  return (tile0 + k / ttc::KC) * (ttc::TILE / 2) +
         (int64_t)(tc::kmajor_off(r, k % ttc::KC, ttc::LBO, ttc::SBO) >> 1);
}

// Split one row x (one warp): hi and lo written at tiled_off(tile0, r, k), the row exponent
// returned; a null x writes a zero row.
__device__ __forceinline__ int split_row_tiled(const float* x, float scale_in, int n, __half* hi,
                                               __half* lo, int64_t tile0, int r, int lane) {
  float m = 0.f;
  if (x)
    for (int b = lane; b < n; b += 32) m = fmaxf(m, fabsf(scale_in * x[b]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  const int e = split_exp(m);
  for (int b = lane; b < n; b += 32) {
    const float v = x ? ldexpf(scale_in * x[b], e) : 0.f;
    const __half h = __float2half_rn(v);
    const int64_t o = tiled_off(tile0, r, b);
    hi[o] = h;
    lo[o] = __float2half_rn(v - __half2float(h));
  }
  return e;
}

// Weight tables in tiles: per channel, pointing tiles of 128 sorted slots (zero rows past
// n_tied), each [my / 32] chunks of 128 x 32. Also the row's E-W beam A_s (the largest
// |wx|) and exponent; the row is wx[s, A_s] wy[s, :].
__global__ void tied_tc_table_kernel(const float* __restrict__ wx, const float* __restrict__ wy,
                                     int nfreq, int n_tied, int mx, int my, __half* wyh,
                                     __half* wyl, int* wye, int* wa) {
  const int lane = threadIdx.x & 31;
  const int nts = (n_tied + ttc::TM - 1) / ttc::TM, kcs = my / ttc::KC;
  const int64_t nrows = (int64_t)nfreq * nts * ttc::TM;
  const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t rp = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); rp < nrows; rp += nw) {
    const int f = (int)(rp / ((int64_t)nts * ttc::TM));
    const int slot = (int)(rp - (int64_t)f * nts * ttc::TM);
    const int64_t tile0 = ((int64_t)f * nts + (slot >> 7)) * kcs;
    if (slot >= n_tied) {
      split_row_tiled(nullptr, 0.f, my, wyh, wyl, tile0, slot & 127, lane);
      continue;
    }
    const int64_t r = (int64_t)f * n_tied + slot;
    int A = 0;
    float best = -1.f;
    for (int a = 0; a < mx; ++a) {
      const float v = fabsf(wx[r * mx + a]);
      if (v > best) { best = v; A = a; }
    }
    const int e = split_row_tiled(wy + r * my, wx[r * mx + A], my, wyh, wyl, tile0, slot & 127, lane);
    if (lane == 0) {
      wye[r] = e;
      wa[r] = A;
    }
  }
}

// x 2^e, rounded once as ldexpf does.
__device__ __forceinline__ float scale_pow2(float x, int e) {
  return e >= -126 && e <= 127 ? x * __int_as_float((127 + e) << 23) : ldexpf(x, e);
}

// Beam rows P[j, f, A, :] split the same way (per call), in tiles per (channel, E-W beam) of 64
// windows (zero rows past nwin); exponents at pe[(j nfreq + f) mx + A]. `wpg` warps take eight
// windows: lane (g, r) holds eight beams of window r at a time, so 128 contiguous bytes are read
// per window, and the eight windows' 16-byte pieces of one K block are the 128 bytes of a core
// matrix: every store of a warp is 512 contiguous bytes. A warp keeps its share of the rows in
// registers between the row maximum and the split (up to kHold blocks of 32 beams; what is past
// those is read again). Bound by memory: 134 MB read and 134 MB written for 64 windows x 256
// channels x 4 x 512 beams in 59 us (4.6 TB/s); with the rows read
// twice instead it took 80 us.
constexpr int kPrepWarps = 8, kHold = 2;
__global__ void __launch_bounds__(32 * kPrepWarps) tied_tc_prep_kernel(
    const float* __restrict__ P, int64_t nwin, int nfreq, int mx, int my, __half* ph, __half* pl,
    int* pe, int wpg, int vec) {
  __shared__ float s_max[kPrepWarps][8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, r = lane & 7, g = lane >> 3;
  const int sub = warp % wpg, grp = warp / wpg;
  using ttc::TN;
  const int ntj = (int)((nwin + TN - 1) / TN), nb = my / ttc::KC;
  const int64_t per_fa = (int64_t)ntj * (TN / 8);        // groups of eight windows
  const int64_t gp = (int64_t)blockIdx.x * (kPrepWarps / wpg) + grp;
  const int64_t fa = gp / per_fa;                        // f mx + A
  const int64_t j8 = gp - fa * per_fa, j = 8 * j8 + r;
  const bool have = fa < (int64_t)nfreq * mx, live = have && j < nwin;
  const int f = (int)(fa / mx), A = (int)(fa - (int64_t)f * mx);
  const float* x = P + ((live ? j * nfreq + f : 0) * mx + (live ? A : 0)) * my + 8 * g;
  auto load = [&](int b, float (&v)[8]) {                // beams 32 b + 8 g .. + 7
    if (vec) {
      const float4 a = *reinterpret_cast<const float4*>(x + 32 * b);
      const float4 c = *reinterpret_cast<const float4*>(x + 32 * b + 4);
      v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
      v[4] = c.x; v[5] = c.y; v[6] = c.z; v[7] = c.w;
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = x[32 * b + i];
    }
  };
  float hold[kHold][8];
  float m = 0.f;
#pragma unroll
  for (int q = 0; q < kHold; ++q) {
#pragma unroll
    for (int i = 0; i < 8; ++i) hold[q][i] = 0.f;
    if (live && sub + q * wpg < nb) load(sub + q * wpg, hold[q]);
  }
#pragma unroll
  for (int q = 0; q < kHold; ++q)
#pragma unroll
    for (int i = 0; i < 8; ++i) m = fmaxf(m, fabsf(hold[q][i]));
  if (live)
    for (int b = sub + kHold * wpg; b < nb; b += wpg) {
      float v[8];
      load(b, v);
#pragma unroll
      for (int i = 0; i < 8; ++i) m = fmaxf(m, fabsf(v[i]));
    }
  m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 8));
  m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 16));
  if (g == 0) s_max[warp][r] = m;
  __syncthreads();
  for (int w = 0; w < wpg; ++w) m = fmaxf(m, s_max[grp * wpg + w][r]);
  if (!have) return;
  const int e = split_exp(m);
  // this group's rows in the tile of chunk 0 (halves)
  const int jt = (int)(8 * j8 / TN), row = (int)(8 * j8 - (int64_t)jt * TN);
  const int64_t base = (fa * ntj + jt) * nb * (TN * ttc::KC) + (row >> 3) * (ttc::SBO / 2) + lane * 8;
  auto put = [&](int b, const float (&v)[8]) {
    __half2 h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float a = scale_pow2(v[2 * i], e), c = scale_pow2(v[2 * i + 1], e);
      h[i] = __halves2half2(__float2half_rn(a), __float2half_rn(c));
      l[i] = __halves2half2(__float2half_rn(a - __low2float(h[i])), __float2half_rn(c - __high2float(h[i])));
    }
    const int64_t o = base + (int64_t)b * (TN * ttc::KC);
    *reinterpret_cast<uint4*>(ph + o) = *reinterpret_cast<const uint4*>(h);
    *reinterpret_cast<uint4*>(pl + o) = *reinterpret_cast<const uint4*>(l);
  };
#pragma unroll
  for (int q = 0; q < kHold; ++q)
    if (sub + q * wpg < nb) put(sub + q * wpg, hold[q]);
  for (int b = sub + kHold * wpg; b < nb; b += wpg) {
    float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (live) load(b, v);
    put(b, v);
  }
  if (live && g == 0 && sub == 0) pe[(j * nfreq + f) * mx + A] = e;
}

__global__ void __launch_bounds__(ttc::NT, 2) tied_tc_kernel(
    const __half* __restrict__ wyh, const __half* __restrict__ wyl, const int* __restrict__ wye,
    const int* __restrict__ wa, const int* __restrict__ perm, const __half* __restrict__ ph,
    const __half* __restrict__ pl, const int* __restrict__ pe, float* __restrict__ out,
    int64_t nwin, int nfreq, int n_tied, int mx, int my, int* err) {
  using ttc::NS, ttc::PT, ttc::STAGE, ttc::TN;
  extern __shared__ __align__(1024) unsigned char smem_t[];
  __shared__ uint64_t full[NS], empty[NS];
  __shared__ uint32_t taddr;
  __shared__ int s_mask, s_ok;
  __shared__ int s_pe[ttc::MAXA][TN];
  const int tid = threadIdx.x, warp = tid >> 5;
  const int f = blockIdx.z;
  // pointing tiles run fastest, window tiles next, channels last
  const int nts = (n_tied + ttc::TM - 1) / ttc::TM;
  const int jt = (int)(blockIdx.x / (unsigned)nts), pt_i = (int)(blockIdx.x - (unsigned)jt * nts);
  const int s0 = pt_i * ttc::TM;
  const int64_t j0 = (int64_t)jt * TN;
  const int64_t fs0 = (int64_t)f * n_tied;
  if (warp == 0) {
    tc::tmem_alloc(&taddr, ttc::TMEM_COLS);
    tc::tmem_relinquish();
  }
  const int kcs = my / ttc::KC;
  const int64_t wt0 = ((int64_t)f * nts + pt_i) * kcs;   // first weight tile
  if (tid == 0) {
    for (int i = 0; i < NS; ++i) {
      tc::mbar_init(&full[i], 1);
      tc::mbar_init(&empty[i], 1);
    }
    tc::mbar_init_fence();
    s_mask = 0;
    s_ok = 1;
  }
  const int row = tid & (ttc::TM - 1);           // TMEM lane / pointing of this thread
  const int s = s0 + row;
  const bool srow = s < n_tied;
  const int my_a = srow ? wa[fs0 + s] : 0;
  const int my_e = srow ? wye[fs0 + s] : 0;
  const int dst_s = srow ? perm[fs0 + s] : 0;
  __syncthreads();
  if (srow && tid < ttc::TM) atomicOr(&s_mask, 1 << my_a);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const int mask = s_mask;
  int nact = 0, my_ai = 0;
  for (int A = 0; A < mx; ++A)
    if ((mask >> A) & 1) {
      if (A == my_a) my_ai = nact;
      ++nact;
    }
  // exponents of the tile's windows, per E-W beam in use (warps 0 and 1 start on the pipeline)
  for (int i = tid - 64; i >= 0 && i < nact * TN; i += ttc::NT - 64) {
    const int ai = i / TN, jj = i - ai * TN;
    int A = 0;
    for (int a = 0, c = -1; a < mx; ++a)
      if ((mask >> a) & 1 && ++c == ai) A = a;
    const int64_t j = j0 + jj;
    s_pe[ai][jj] = j < nwin ? pe[(j * nfreq + f) * mx + A] : 0;
  }
  const uint32_t tbase = taddr;
  const int total = nact * kcs;
  const uint32_t idesc = tc::idesc_f16(ttc::TM, TN, false);
  // Chunk t = (E-W beam in use number t / kcs, K chunk t % kcs) goes to stage t % NS. Thread 32
  // stages the chunks as four bulk copies each, completing on full[stage]; thread 0 issues their
  // MMAs and commits them to empty[stage], after which the stage takes chunk t + NS. One thread
  // for both held each refill back until the next chunk's MMAs were issued. The other threads
  // wait at the CTA barrier. Every wait is bounded.
  if (tid == 32) {
    const int ntj = (int)((nwin + TN - 1) / TN);
    bool ok = true;
    int t = 0;
    for (int A = 0; A < mx && ok; ++A) {
      if (!((mask >> A) & 1)) continue;
      const int64_t pt0 = (((int64_t)f * mx + A) * ntj + jt) * kcs;
      for (int kc = 0; kc < kcs; ++kc, ++t) {
        const int st = t % NS;
        if (t >= NS) ok = tc::mbar_wait(&empty[st], (uint32_t)((t / NS - 1) & 1), ttc::WAIT_NS);
        if (!ok) break;
        unsigned char* stg = smem_t + st * STAGE;
        const int64_t wt = (wt0 + kc) * (ttc::TILE / 2), pt = (pt0 + kc) * (PT / 2);
        tc::mbar_arrive_expect_tx(&full[st], (uint32_t)STAGE);
        tc::bulk_g2s(stg, wyh + wt, ttc::TILE, &full[st]);
        tc::bulk_g2s(stg + ttc::TILE, wyl + wt, ttc::TILE, &full[st]);
        tc::bulk_g2s(stg + 2 * ttc::TILE, ph + pt, PT, &full[st]);
        tc::bulk_g2s(stg + 2 * ttc::TILE + PT, pl + pt, PT, &full[st]);
      }
    }
    if (!ok) {
      atomicExch(&s_ok, 0);
      // copies in flight must have landed before the CTA gives back its memory
      for (int c = t > NS ? t - NS : 0; c < t; ++c)
        tc::mbar_wait(&full[c % NS], (uint32_t)((c / NS) & 1), ttc::WAIT_NS);
    }
  } else if (tid == 0) {
    bool ok = true;
    int t = 0;
    for (; t < total; ++t) {
      const int st = t % NS;
      ok = tc::mbar_wait(&full[st], (uint32_t)((t / NS) & 1), ttc::WAIT_NS);
      if (!ok) break;
      tc::fence_after_sync();
      const uint32_t sa = tc::smem_u32(smem_t + st * STAGE);
      const uint32_t d = tbase + (uint32_t)((t / kcs) * TN);
      const int kc = t % kcs;
#pragma unroll
      for (int ks = 0; ks < ttc::KC / 16; ++ks) {
        const uint32_t ko = (uint32_t)(ks * 2 * ttc::LBO);
        const uint64_t dwh = tc::smem_desc(sa + ko, ttc::LBO, ttc::SBO);
        const uint64_t dwl = tc::smem_desc(sa + ttc::TILE + ko, ttc::LBO, ttc::SBO);
        const uint64_t dph = tc::smem_desc(sa + 2 * ttc::TILE + ko, ttc::LBO, ttc::SBO);
        const uint64_t dpl = tc::smem_desc(sa + 2 * ttc::TILE + PT + ko, ttc::LBO, ttc::SBO);
        tc::mma_f16(d, dwh, dph, idesc, (kc > 0 || ks > 0) ? 1u : 0u);
        tc::mma_f16(d, dwh, dpl, idesc, 1u);
        tc::mma_f16(d, dwl, dph, idesc, 1u);
      }
      tc::mma_commit(&empty[st]);
    }
    if (t > 0) {                                    // the last commit covers every MMA issued
      const int tl = t - 1;
      ok = tc::mbar_wait(&empty[tl % NS], (uint32_t)((tl / NS) & 1), ttc::WAIT_NS) && ok;
    }
    if (!ok) atomicExch(&s_ok, 0);
  }
  tc::fence_before_sync();
  __syncthreads();
  const bool ok = s_ok != 0;
  tc::fence_after_sync();
  if (ok && total > 0) {
    // warp w reads TMEM lanes 32 (w % 4) .. + 31 (its pointings) and half w / 4 of the windows
    const uint32_t lane_off = (uint32_t)(32 * (warp & 3)) << 16;
    const int c = warp >> 2;
    for (int a2 = 0; a2 < nact; ++a2) {
      uint32_t r[32];
      tc::tmem_ld32(tbase + lane_off + (uint32_t)(a2 * TN + 32 * c), r);
      tc::tmem_wait_ld();
      if (a2 == my_ai && srow) {
#pragma unroll
        for (int q = 0; q < 32; ++q) {
          const int64_t j = j0 + 32 * c + q;
          if (j < nwin) {
            // D 2^-E: a power-of-two product (exact) while 2^-E is a normal float
            const int E = my_e + s_pe[a2][32 * c + q];
            const float d = __uint_as_float(r[q]);
            out[(j * nfreq + f) * (int64_t)n_tied + dst_s] =
                (E > -127 && E < 127) ? d * __int_as_float((127 - E) << 23) : ldexpf(d, -E);
          }
        }
      }
    }
  } else if (!ok && tid == 0) {
    atomicExch(err, FFTBF_ETIMEOUT);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tbase, ttc::TMEM_COLS);
}

// ------------------------------------------------------------------------------ host --
bool tied_tc_eligible(bool dense_x, int mx, int my) {
  const char* env = getenv("FFTBF_TIED_TC");
  if (env && env[0] == '0') return false;
  return !dense_x && mx <= ttc::MAXA && my >= 64 && my % 64 == 0;
}

int tied_tc_build(TiedTables& tt, int64_t nuv, int mx, int my, cudaStream_t st) {
  cudaFree(tt.wyh);
  cudaFree(tt.wyl);
  cudaFree(tt.wye);
  cudaFree(tt.wa);
  tt.wyh = tt.wyl = nullptr;
  tt.wye = tt.wa = nullptr;
  const int n_tied = tt.tc_n_tied;
  const int nfreq = (int)(nuv / n_tied);
  const int64_t nts = (n_tied + ttc::TM - 1) / ttc::TM;
  const size_t halves = (size_t)nfreq * nts * ttc::TM * my;      // padded to whole tiles
  // test hook: FFTBF_TEST_TIED_TC_NOMEM=1 makes the split tables look unallocatable, so
  // that the fallback to the CUDA-core GEMM can be exercised without exhausting the device
  const char* nomem = getenv("FFTBF_TEST_TIED_TC_NOMEM");
  if (nomem && nomem[0] == '1') return set_error(FFTBF_ENOMEM, "split tied-beam tables (test hook)");
  bool ok = cudaMalloc(&tt.wyh, halves * sizeof(__half)) == cudaSuccess &&
            cudaMalloc(&tt.wyl, halves * sizeof(__half)) == cudaSuccess &&
            cudaMalloc(&tt.wye, nuv * sizeof(int)) == cudaSuccess &&
            cudaMalloc(&tt.wa, nuv * sizeof(int)) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    cudaFree(tt.wyh);
    cudaFree(tt.wyl);
    cudaFree(tt.wye);
    cudaFree(tt.wa);
    tt.wyh = tt.wyl = nullptr;
    tt.wye = tt.wa = nullptr;
    return set_error(FFTBF_ENOMEM, "cannot allocate the split tied-beam tables");
  }
  const int64_t rows = (int64_t)nfreq * nts * ttc::TM;
  const unsigned blocks = (unsigned)std::min<int64_t>((rows + 7) / 8, 1 << 20);
  tied_tc_table_kernel<<<blocks, 256, 0, st>>>(tt.wx, tt.wy, nfreq, n_tied, mx, my,
                                               reinterpret_cast<__half*>(tt.wyh),
                                               reinterpret_cast<__half*>(tt.wyl), tt.wye, tt.wa);
  FFTBF_CUDA_TRY(cudaGetLastError());
  tt.tc = 1;
  return FFTBF_OK;
}

int tied_tc_launch(TiedTables& tt, const float* beams, int64_t nwin, int nfreq, int mx, int my,
                   float* out, cudaStream_t st) {
  using ttc::TN;
  const int64_t ntj = (nwin + TN - 1) / TN;
  const int64_t nts = (tt.n_tied + ttc::TM - 1) / ttc::TM;
  if ((nwin + 127) / 128 > 65535 || nfreq > 65535 || nts * ntj > INT32_MAX)
    return set_error(FFTBF_EUNSUPPORTED, "tied beams: too many windows or channels per call");
  const int64_t prow = (int64_t)nfreq * mx * ntj * TN;             // padded beam rows
  // scratch rows and exponents for the next whole 128 windows: a call of a few more windows than
  // an earlier one, possibly under capture, then seldom has to allocate
  const int64_t crow = (int64_t)nfreq * mx * ((nwin + 127) / 128) * 128;
  if ((size_t)crow > tt.p_cap) {
    cudaStreamSynchronize(st);                  // the old scratch may still be read
    cudaFree(tt.ph);
    cudaFree(tt.pl);
    cudaFree(tt.pe);
    tt.ph = tt.pl = nullptr;
    tt.pe = nullptr;
    tt.p_cap = 0;
    bool ok = cudaMalloc(&tt.ph, crow * my * sizeof(__half)) == cudaSuccess &&
              cudaMalloc(&tt.pl, crow * my * sizeof(__half)) == cudaSuccess &&
              cudaMalloc(&tt.pe, crow * sizeof(int)) == cudaSuccess;
    if (!ok) {
      cudaGetLastError();
      cudaFree(tt.ph);
      cudaFree(tt.pl);
      cudaFree(tt.pe);
      tt.ph = tt.pl = nullptr;
      tt.pe = nullptr;
      return set_error(FFTBF_ENOMEM, "cannot allocate the split beam scratch");
    }
    tt.p_cap = (size_t)crow;
  }
  // two blocks of 32 beams per warp where the row is long enough, so that a warp's loads are all
  // in flight at once and a short call still has many warps
  const int wpg = my >= 512 ? 8 : my >= 256 ? 4 : my >= 128 ? 2 : 1;
  const int64_t gpb = kPrepWarps / wpg, pblocks = (prow / 8 + gpb - 1) / gpb;
  const int vec = (reinterpret_cast<uintptr_t>(beams) & 15) == 0;   // rows are multiples of 64 beams
  tied_tc_prep_kernel<<<(unsigned)pblocks, 32 * kPrepWarps, 0, st>>>(
      beams, nwin, nfreq, mx, my, reinterpret_cast<__half*>(tt.ph),
      reinterpret_cast<__half*>(tt.pl), tt.pe, wpg, vec);
  FFTBF_CUDA_TRY(cudaGetLastError());
  const size_t smem = ttc::NS * (size_t)ttc::STAGE;
  FFTBF_CUDA_TRY(cudaFuncSetAttribute(tied_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)smem));
  dim3 grid((unsigned)(nts * ntj), 1, nfreq);
  tied_tc_kernel<<<grid, ttc::NT, smem, st>>>(
      reinterpret_cast<const __half*>(tt.wyh), reinterpret_cast<const __half*>(tt.wyl), tt.wye,
      tt.wa, tt.perm, reinterpret_cast<const __half*>(tt.ph), reinterpret_cast<const __half*>(tt.pl),
      tt.pe, out, nwin, nfreq, tt.n_tied, mx, my, tt.err);
  FFTBF_CUDA_TRY(cudaGetLastError());
  return FFTBF_OK;
}

}  // namespace fftbf
