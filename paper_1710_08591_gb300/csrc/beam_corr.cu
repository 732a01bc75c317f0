// FP32 form of the FFT-beam hot path on the FP8 tensor cores, through the feed covariance.
//
// The integrated intensity of a beam (Eq. fftbeamform, Eq. bf) is a quadratic form in the
// covariance of the voltages, R_ab = sum over the window's snapshots of x_a x_b^* (Eq. Vab):
//   P[A,B] = sum_{a,b} w_a w_b^* R_ab exp(-2 pi i (A (ix_a - ix_b)/Mx + B (iy_a - iy_b)/My))
//          = Re sum_{kappa, lambda} V[kappa][lambda] exp(-2 pi i (A kappa/Mx + B lambda/My)),
// with V the weighted covariance summed over the feed pairs of one separation (the stacked
// visibilities of Eq. b_V_delta, kappa = (ix_a - ix_b) mod Mx, lambda = iy_a - iy_b). It holds
// for every padding, the cyclic co-adding of pad < n included.
// The voltages are 4-bit integers, which FP8 (e4m3) holds exactly (integer k <= 15 is the bit
// pattern k: the subnormals and the first binade are one linear scale of 2^-9), and the
// tensor cores sum their products in FP32: R is exact while 128 snapshots <= 2^24. So one
// FP8 product per pair replaces the FP32 transform of every snapshot; the weights and the
// transform are applied once per window, to exact sums: in FP32 with every product's rounding
// error kept, V in fixed point of about 2^-38 of the largest product, the transform in two floats,
// because a weak beam beside a strong source is a small difference of large terms.
//
// Work split: one pair of CTAs (a cluster, tcgen05 cta_group::2) owns a work item (window,
// channel) and walks the upper-triangle tiles of R, 256 feeds x up to 256 feeds, one tile in
// tensor memory at a time (256 columns of real parts, 256 of imaginary parts, 128 rows per
// CTA), so an item's voltages are read from HBM once and re-read from L2, and no covariance
// leaves the SM. Feeds are held in slots ix * nyp + iy, nyp = ny rounded up to a multiple of
// 16 (zeros between), so a group of 16 slots lies in one E-W row. Roles (18 of 20 warps per CTA):
//   warps 0-7    epilogue: weights x covariance, summed along the diagonals of the tile,
//                added to V in shared memory (each warp at its own pace); after the last tile the
//                transform of V to beams;
//   warps 8-15   producers: voltages of this CTA's 128 row slots and its half of the column
//                slots, 64 snapshots per stage, nibbles to e4m3 (both MN-major operands);
//   warp 17      one thread stages the voltages with TMA (64 snapshots x 128 feeds a tile);
//   warps 16, 18 one thread each of the pair's first CTA issue the MMAs of the real and of the
//                imaginary half: per 32 snapshots
//                and off-diagonal tile Re += Xr Yr^T + Xi Yi^T, Im += Xi Yr^T - Xr Yi^T
//                (M = 256, N <= 256, K = 32 each). A tile and its mirror image are conjugate,
//                so off-diagonal tiles count twice and the real part is taken at the end; on
//                a diagonal tile C = Xi Yr^T alone gives the imaginary part (Im R = C - C^T, and
//                the mirror of C under the real part is -C^T), three products instead of four.
// The real and imaginary halves are handed over separately, each with its own issuing thread
// (a tcgen05.mma holds its thread for about 100 cycles, so one thread cannot keep the tensor
// cores busy), so the real products of the next tile run while the epilogue reads this tile's
// imaginary half, ahead by as many stages as the operand ring holds. Every wait is bounded by
// one second of device time.
// What bounds it: the producers' integer unpacking and shared memory beside the MMAs (per stage of an
// off-diagonal tile the MMAs read 64 KB, the producers write 32 KB and the staging moves 32 KB:
// about 128 bytes per cycle), and between tiles the epilogue, about 4500 cycles per half with real
// weights: a third its products, a third the gather of the lags. Measured on a GB300 (the FFT
// kernels; this one with products and sums rounded to FP32; this one): 4x256, 2 polarisations,
// 4096 windows x channels of 768 snapshots 8.57, 5.20, 6.16 ms (the MMAs alone would need 3.3 ms, 540
// tiles of 6.1 us in turn); 16 such items 608, 104, 119 us; 8x64 with complex gains, 2048 items of 512
// snapshots 3.44, 0.90, 1.19 ms; 3x37 onto 5x73 beams, 360 items of 100 snapshots 1267, 143, 139 us.
// Largest error of a beam beside a source of amplitude 7 over noise of 0.3, 4x256 with half-sine
// weights: 2e-6, 1e-4, 6e-8.
// An item's sums are whole numbers or taken in an order that depends on the item alone, so its
// beams are bit-identical whatever else the launch carries.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>

#include "beam_fp32.cuh"
#include "beam_fp32_warp.cuh"
#include "corr.cuh"
#include "tc_ptx.cuh"

namespace fftbf {

namespace corr {
constexpr int NT = 640;                  // 20 warps (warps are allocated by fours): 96 registers
constexpr int EPI = 256, PROD = 256;     // threads of the epilogue and the producers
constexpr int KS = kCorrSteps;           // snapshots per stage: two K = 32 MMA steps
constexpr int NE = KS / 16;              // units per thread, stage and operand
constexpr int TILE = 128 * KS;           // one operand component: 128 slots x 64 snapshots, e4m3
constexpr int STAGE = 4 * TILE;          // rows re, rows im, columns re, columns im
constexpr int LBO = 1024, SBO = 128;     // MN-major: 8 snapshots apart, 16 slots apart
constexpr int VMAX = 2048;               // entries of V (E-W separations x N-S lags)
constexpr int DS = 72;                   // pairs per staged diagonal (8 x 8, conflict-free gather)
constexpr float GRID = 12582912.f;       // 1.5 2^23: sums started here are whole numbers
constexpr int MAXNS = 6, MAXNR = 3;
constexpr int RAW = KS * 128;            // staged voltages of one operand: 64 snapshots x 128 feeds
constexpr int SMEM_MAX = 227 * 1024 - 1024;   // dynamic; static: the barriers
constexpr uint64_t WAIT_NS = 1000000000ull;
// barriers: FULL/EMPTY per stage; accumulators done (RD, ID) and drained (RF, IF), V of
// the other CTA ready (PV) and read by it (PE); raw voltages staged and read (RAWF, RAWE); the
// MMAs of an issuer that gave up (LR, LI)
enum { RD = 0, ID, RF, IF, PV, PE, FULL, EMPTY = FULL + MAXNS, RAWF = EMPTY + MAXNS,
       RAWE = RAWF + MAXNR, LR = RAWE + MAXNR, LI, NBAR };
}  // namespace corr

namespace {

using namespace corr;

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_rank(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
// Arrive on a barrier of either CTA: of an operand or tensor-memory hand-over (ordered by the
// proxy and tcgen05 fences; a release at cluster scope would wait for every load in flight),
// and of shared memory written for the other CTA's threads.
__device__ __forceinline__ void arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];\n" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void arrive_release_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];\n" ::"r"(cluster_addr)
               : "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.aligned;\n barrier.cluster.wait.aligned;\n" ::: "memory");
}
// Bounded wait: a non-blocking test first, then suspended (20 us hint; the arrival wakes it), so
// that waiting warps take no issue slots. ACQ: also sees what the other CTA's threads released
// at cluster scope.
template <bool ACQ = false>
__device__ __forceinline__ bool wait_pair(uint64_t* bar, uint32_t parity, volatile int* abort) {
  const uint32_t a = tc::smem_u32(bar);
  if (!ACQ && tc::mbar_test(bar, parity)) return true;
  uint64_t t0 = 0;
  for (uint32_t i = 0;; ++i) {
    uint32_t ok;
    if constexpr (ACQ)
      asm volatile(
          "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n"
          " selp.u32 %0, 1, 0, p;\n}\n"
          : "=r"(ok)
          : "r"(a), "r"(parity), "r"(20000u)
          : "memory");
    else
      asm volatile(
          "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
          " selp.u32 %0, 1, 0, p;\n}\n"
          : "=r"(ok)
          : "r"(a), "r"(parity), "r"(20000u)
          : "memory");
    if (ok) return true;
    if (*abort) return false;
    const uint64_t t = tc::globaltimer_ns();
    if (i == 0) t0 = t;
    else if (t - t0 > WAIT_NS) return false;
  }
}
__device__ __forceinline__ void mma_f8_pair(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive on the barrier at this offset in both CTAs once every MMA issued so far is done.
__device__ __forceinline__ void commit_pair(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n" ::"r"(
          tc::smem_u32(bar)),
      "h"((uint16_t)3)
      : "memory");
}

// The epilogue's 256 threads: a barrier, and one that tells whether `ok` held on all of them.
__device__ __forceinline__ void bar_epi() { tc::named_sync(1, 256); }
__device__ __forceinline__ bool bar_epi_all(bool ok) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.and.pred.aligned q, 1, 256, p;\n"
      " selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)ok)
      : "memory");
  return r != 0;
}

// TMEM -> registers, 16 lanes x 8 NB columns: thread t gets, for every 8-column block n,
// r[4n], r[4n+1] = row t/4, columns 8n + 2(t%4), +1 and r[4n+2], r[4n+3] = row t/4 + 8.
template <int NB> __device__ __forceinline__ void tmem_ld16x256(uint32_t taddr, uint32_t* r);
template <> __device__ __forceinline__ void tmem_ld16x256<1>(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}
template <> __device__ __forceinline__ void tmem_ld16x256<2>(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
// TMA tile: `rows` of 128 bytes from feed x of channel f, time t on, all polarisations (snapshots in
// order), 128-byte swizzle; zeros past the feeds and past the last sample.
__device__ __forceinline__ void tma_volts(uint32_t dst, const CUtensorMap* map, int x, int f, int t,
                                          uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, "
      "{%2, %3, %4, %5}], [%6];\n" ::"r"(dst),
      "l"(map), "r"(x), "r"(0), "r"(f), "r"(t), "r"(tc::smem_u32(bar))
      : "memory");
}

// A tensor map in global memory was written by a copy (generic proxy): before its first use by TMA
// the writes are acquired for the tensor-map proxy, or a descriptor cached from the table's earlier
// contents could be used. Maps in kernel parameters need no fence.
__device__ __forceinline__ void acquire_map(const CUtensorMap* map) {
  asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;\n" ::"l"(map) : "memory");
}

// The first `cnt` of 16 bytes at any address: aligned words where they lie inside
// [begin, end), single bytes at the ends of the buffer.
__device__ __noinline__ uint4 load16_any(const uint8_t* p, int cnt, const uint8_t* begin,
                                         const uint8_t* end) {
  uint32_t x[4] = {0u, 0u, 0u, 0u};
  const int sh = (int)(reinterpret_cast<uintptr_t>(p) & 3);
  const uint8_t* q = p - sh;
  if (cnt > 0 && q >= begin && q + 20 <= end) {
    uint32_t w[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) w[i] = __ldg(reinterpret_cast<const uint32_t*>(q) + i);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int n = cnt - 4 * i;                       // live bytes of this word
      x[i] = __funnelshift_r(w[i], w[i + 1], 8 * sh) & (n >= 4 ? ~0u : n > 0 ? (1u << (8 * n)) - 1u : 0u);
    }
  } else {
#pragma unroll 1
    for (int b = 0; b < cnt; ++b) {
      const uint32_t v = (uint32_t)__ldg(p + b) << (8 * (b & 3));
#pragma unroll
      for (int i = 0; i < 4; ++i) x[i] |= (b >> 2) == i ? v : 0u;
    }
  }
  return make_uint4(x[0], x[1], x[2], x[3]);
}

// Four signed nibbles as e4m3 bytes: sign and magnitude, where magnitude k <= 15 is the bit
// pattern k (value k 2^-9). n: the nibbles in bits 0-3 of each byte, s: their signs in bit 7 of
// each byte (other bits of both ignored). x + 8 = n ^ 8, and |x| is its distance from 8.
__device__ __forceinline__ uint32_t nibbles_e4m3(uint32_t n, uint32_t s) {
  return __vabsdiffu4((n & 0x0F0F0F0Fu) ^ 0x08080808u, 0x08080808u) | (s & 0x80808080u);
}
// 16 voltage bytes -> 16 real and 16 imaginary e4m3 values
__device__ __forceinline__ void unpack16(const uint4& v, uint4& re, uint4& im) {
  auto one = [](uint32_t w, uint32_t& r, uint32_t& i) {
    i = nibbles_e4m3(w, w << 4);
    r = nibbles_e4m3(w >> 4, w);
  };
  one(v.x, re.x, im.x);
  one(v.y, re.y, im.y);
  one(v.z, re.z, im.z);
  one(v.w, re.w, im.w);
}

// ---- two-float arithmetic on complex pairs (value h + l, |l| <= ulp(h) / 2). A beam far from a
// strong source is a small difference of large stacked visibilities, so V is summed and
// transformed to about twice FP32 precision (sums: Knuth's TwoSum; products: Dekker's, by FMA).
struct Cdd { float2 h, l; };
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ Cdd renorm(float2 s, float2 e) {
  Cdd r;
  r.h = cadd(s, e);
  r.l = csub(e, csub(r.h, s));
  return r;
}
__device__ __forceinline__ Cdd dd_add(Cdd a, Cdd b) {
  const float2 s = cadd(a.h, b.h), t = csub(s, a.h);
  const float2 e = cadd(csub(a.h, csub(s, t)), csub(b.h, t));
  return renorm(s, cadd(e, cadd(a.l, b.l)));
}
__device__ __forceinline__ Cdd dd_sub(const Cdd& a, const Cdd& b) {
  Cdd n;
  n.h = neg2(b.h);
  n.l = neg2(b.l);
  return dd_add(a, n);
}
// a x (c + i s), the factor as float4 (c hi, c lo, s hi, s lo)
__device__ __forceinline__ Cdd dd_cmul(Cdd a, float4 w) {
  const float2 ch = make_float2(w.x, w.x), cl = make_float2(w.y, w.y);
  const float2 sh = make_float2(w.z, w.z), sl = make_float2(w.w, w.w);
  const float2 rh = make_float2(-a.h.y, a.h.x), rl = make_float2(-a.l.y, a.l.x);   // i a
  Cdd p, q;
  p.h = __fmul2_rn(a.h, ch);
  p.l = __ffma2_rn(a.l, ch, __ffma2_rn(a.h, cl, __ffma2_rn(a.h, ch, neg2(p.h))));
  q.h = __fmul2_rn(rh, sh);
  q.l = __ffma2_rn(rl, sh, __ffma2_rn(rh, sl, __ffma2_rn(rh, sh, neg2(q.h))));
  return dd_add(p, q);
}
__device__ __forceinline__ Cdd dd_zero() { return Cdd{make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }

// The job of a work item; k: the job of this role's last item (items only grow).
__device__ __forceinline__ const CorrJob& find_job(const CorrParams& p, int64_t item, int& k) {
  if (!p.table) return p.one;
  while (k + 1 < p.njobs && item >= p.table[k + 1].item0) ++k;
  return p.table[k];
}
// A wait that ran out: every role of the CTA leaves, and the launch's error words are set.
__device__ __forceinline__ void corr_fail(const CorrParams& p, volatile int* abort_sm) {
  *abort_sm = 1;
  if (p.err) atomicExch(p.err, FFTBF_ETIMEOUT);
  else if (!p.table) atomicExch(p.one.a.err, FFTBF_ETIMEOUT);
  else
    for (int k = 0; k < p.njobs; ++k) atomicExch(p.table[k].a.err, FFTBF_ETIMEOUT);
}
// Column slots of tile column J (a multiple of 32)
__device__ __forceinline__ int tile_cols(int np, int J) {
  const int left = np - 256 * J;
  return left < 256 ? (left + 31) & ~31 : 256;
}

// What the epilogue needs of a job, in registers.
struct JobRegs { int nx, ny, nyp, np, nt, mx, mode; float rscale, lscale; };

struct Lay {                             // shared-memory offsets (bytes)
  int ring, raw, w, v, stg, tab, total;
};
__host__ __device__ inline Lay lay_of(const CorrSizes& s) {
  Lay L;
  int o = 0;
  auto take = [&](int bytes) { int r = o; o += (bytes + 127) & ~127; return r; };
  L.raw = take(s.nr * 2 * RAW);          // 1024-byte aligned tiles (128-byte swizzle)
  L.ring = take(s.ns * STAGE);
  L.w = take(s.wslots * 4 * (s.cplx ? 2 : 1));
  L.v = take(s.vlen * 16);
  L.stg = take(s.stg * 8 * 4);           // 8 warps; also the transform's buffer
  L.tab = take(s.tab * 16);
  L.total = o;
  return L;
}

// Floats of one warp's staged diagonals, (whole, rest) pairs of c components: the G + 1 of a step, the
// last one copied to the front for the next, or where there is room (c = 1) and several steps a ring
// of 2 G, its first one held behind the last as well so that a step's lie in order.
__host__ __device__ constexpr int stg_rows(int G, int CR, int c) { return c == 1 && CR > G ? 2 * G + 1 : G + 1; }
__host__ __device__ constexpr int stg_floats(int G, int CR, int c) { return 2 * c * (4 / G) * stg_rows(G, CR, c) * DS; }

// a x, exactly: the product and its rounding error with the sign changed (nx = -x)
__device__ __forceinline__ float2 mul_exact(float2 a, float2 x, float2 nx, float2& nerr) {
  const float2 p = __fmul2_rn(a, x);
  nerr = __ffma2_rn(a, nx, p);
  return p;
}
// grid += a x in whole numbers; returns what that rounds away (|.| <= 1/2)
__device__ __forceinline__ float2 fma_grid(float2 a, float2 x, float2& grid) {
  const float2 t = __ffma2_rn(a, x, grid), d = csub(grid, t);
  grid = t;
  return __ffma2_rn(a, x, d);
}

// ---- epilogue of a tile, one warp: 32 rows x 128 columns of one half (real or imaginary), or with
// complex weights of both. Slots are in runs of G 8-row groups (rows) and CR 8-column groups
// (columns) that each lie in one E-W row. A thread holds, of every 8 x 8 block, row r = lane/4 and
// two adjacent columns; it sums w_a R_ab w_b of the blocks on one block diagonal, d = j - i, in
// registers. A weak beam beside a strong source is a small difference of these products, so none of
// their bits is dropped: the weights are scaled by powers of two so that no product exceeds 2^19,
// each is added to a sum that starts at 1.5 2^23 and so takes whole numbers only, and what that
// leaves (an exact difference) goes to a second sum, with the products' own rounding errors: seven
// packed instructions per two elements where rounded products took two, and 37 for 9 with complex
// weights, whose z = w_b^* R is put on such a grid first. Both sums of G diagonals at a time go to
// shared memory, each lane gathers one lag b - a of them and adds it to V in fixed point, whole
// numbers and 2^-19 (1 / lscale) units in two words: integer additions, so V does not depend on their order and
// the warps need no barrier between tiles.
template <int G, int CR, bool CPLX>
__device__ __forceinline__ void corr_phase(uint32_t tacc, int cols, int row0, int col0, float scale,
                                           int ws0, int wslots, int stg0, int v0, int nv, int half,
                                           int nx, int ny, int nyp, int mx, float lscale, bool diag,
                                           uint32_t drained, uint32_t drained2) {
  extern __shared__ __align__(1024) unsigned char smem_corr[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = warp & 3, h = warp >> 2;
  const float* ws = reinterpret_cast<const float*>(smem_corr + ws0);
  constexpr int NC = CPLX ? 2 : 1;                     // staged components: re, im
  constexpr int SG = 4 / G, ROWS = stg_rows(G, CR, NC);
  constexpr bool RING = ROWS > G + 1;
  constexpr int NST = ROWS * DS, CST = SG * NST;       // pairs of a row run, of a component
  float2* stg = reinterpret_cast<float2*>(smem_corr + stg0 + warp * 4 * stg_floats(G, CR, NC));
  int* v = reinterpret_cast<int*>(smem_corr + v0);
  constexpr int JB = CPLX ? 1 : 2;                     // 8-column blocks per load
  const int r = lane >> 2, c2 = 2 * (lane & 3);
  const float2 grid0 = make_float2(GRID, GRID), zero = make_float2(0.f, 0.f);
  float wr[4], wi[4];                                  // rows 8 i + r of the warp's 32
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int s = row0 + 32 * q + 8 * i + r;
    wr[i] = ws[s] * scale;
    wi[i] = CPLX ? ws[wslots + s] * scale : 0.f;
  }
  const float rs = CPLX && diag ? 0.5f : 1.f;          // complex: real half of a diagonal tile once
  // gather of lag u = 8 G step + ul: one term per r, c = (u + 1 + r) mod 8 of staged diagonal
  // (u + 1 + r) / 8
  const int ul = lane & (8 * G - 1), sgl = G == 4 ? 0 : lane >> 4;
  const float2* gat[8];
#pragma unroll
  for (int rr = 0; rr < 8; ++rr) {
    const int k = ul + 1 + rr;
    gat[rr] = stg + sgl * NST + (k >> 3) * DS + 8 * rr + (k & 7);
  }
  float2* put = stg + 2 * lane;
  const int rowl = row0 + 32 * q + 8 * G * sgl;        // first slot of this lane's row run
  const int ia = rowl / nyp, ya = rowl - ia * nyp;
  // the accumulators go back to the MMAs once the last of them is in registers
  const int runs = cols > 128 * h ? min(16 / CR, (cols - 128 * h + 8 * CR - 1) / (8 * CR)) : 0;
  auto release = [&]() {
    tc::fence_before_sync();
    __syncwarp();
    if (lane == 0) {
      arrive_cluster(drained);
      if (CPLX) arrive_cluster(drained2);
    }
  };
  if (runs == 0) release();
  // Lags ul + 8 G step of a step's staged diagonals (rows from `at` on) to V: iy_a - iy_b = lam, and
  // -lam of the conjugate; kap -1 where no feeds are.
  auto gather = [&](int at, int lam, int kap) {
    __syncwarp();
    float2 x[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      float2 t[8];
#pragma unroll
      for (int rr = 0; rr < 8; ++rr) t[rr] = gat[rr][c * CST + at * DS];
      x[c] = cadd(cadd(cadd(t[0], t[1]), cadd(t[2], t[3])), cadd(cadd(t[4], t[5]), cadd(t[6], t[7])));
    }
    __syncwarp();
    const bool mir = lam < 0;
    if (mir) {
      lam = -lam;
      kap = kap > 0 ? mx - kap : kap;
    }
    if (kap < 0 || lam >= ny) return;
    int* o = v + kap * ny + lam;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const bool im = CPLX ? c == 1 : half == 1;
      if (im && mir) x[c] = neg2(x[c]);
      atomicAdd(o + (im ? 2 * nv : 0), __float2int_rn(x[c].x));
      atomicAdd(o + (im ? 3 * nv : nv), __float2int_rn(x[c].y * lscale));
    }
  };
#pragma unroll 1
  for (int run = 0; run < runs; ++run) {
    const int cc = 128 * h + 8 * CR * run;             // first column of the run in the tile
    const int ib = (col0 + cc) / nyp, yb = col0 + cc - ib * nyp;
    int kap = (ia - ib) % mx;
    kap = ia < nx && ib < nx ? (kap < 0 ? kap + mx : kap) : -1;
    float2 acc[SG][G], low[SG][G], aci[SG][G], lowi[SG][G];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      acc[i / G][i % G] = aci[i / G][i % G] = grid0;
      low[i / G][i % G] = lowi[i / G][i % G] = zero;
    }
    const int lam0 = ya - yb - ul + 8 * G - 1;
    auto stage = [&](int sg, int row, float2 a, float2 l, float2 ai, float2 li) {
      float2* o = put + sg * NST + row * DS;
      a = csub(a, grid0);
      *reinterpret_cast<float4*>(o) = make_float4(a.x, l.x, a.y, l.y);
      if constexpr (CPLX) {
        ai = csub(ai, grid0);
        *reinterpret_cast<float4*>(o + CST) = make_float4(ai.x, li.x, ai.y, li.y);
      }
    };
    auto stage_zero = [&](int row) {                   // before the first diagonal and after the last
#pragma unroll
      for (int sg = 0; sg < SG; ++sg) stage(sg, row, grid0, zero, grid0, zero);
    };
    auto carry = [&]() {
#pragma unroll
      for (int k = 0; k < SG * NC; ++k) {
        float2* o = put + k * NST;                     // CST = SG NST
        *reinterpret_cast<float4*>(o) = *reinterpret_cast<const float4*>(o + G * DS);
      }
    };
    stage_zero(0);
#pragma unroll(CPLX ? (CR > G ? 2 : 1) : CR / G)
    for (int j0 = 0; j0 < CR; j0 += G) {
      const int at = RING ? j0 & G : 0;                // row before the step's first diagonal
      if (!RING && CR > G && j0 > 0) carry();
#pragma unroll
      for (int jb = 0; jb < G; jb += JB) {
        uint32_t w[2][4 * JB], wim[2][4 * JB];         // 32 rows x 8 JB columns
        const uint32_t ta = tacc + ((uint32_t)(32 * q) << 16) + cc + 8 * (j0 + jb);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          tmem_ld16x256<JB>(ta + ((uint32_t)(16 * i) << 16), w[i]);
          if (CPLX) tmem_ld16x256<JB>(ta + 256 + ((uint32_t)(16 * i) << 16), wim[i]);
        }
        float2 br[JB], bi[JB];
#pragma unroll
        for (int j = 0; j < JB; ++j) {
          const int sc = col0 + cc + 8 * (j0 + jb + j) + c2;
          br[j] = *reinterpret_cast<const float2*>(ws + sc);
          if (CPLX) bi[j] = *reinterpret_cast<const float2*>(ws + wslots + sc);
        }
        tc::tmem_wait_ld();
        if (run == runs - 1 && j0 + G == CR && jb + JB == G) release();
#pragma unroll
        for (int j = 0; j < JB; ++j) {
          const int jj = jb + j, done = (jj + 1) % G;  // block diagonal j0 + jj - (G - 1) completes
          const float2 nb = CPLX ? neg2(bi[j]) : neg2(br[j]);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint32_t* x = &w[i >> 1][4 * j + 2 * (i & 1)];
            const float2 R = make_float2(__uint_as_float(x[0]), __uint_as_float(x[1]));
            const int sg = i / G, d = (jj - i % G + G) % G;
            const float2 ar = make_float2(wr[i], wr[i]), na = make_float2(-wr[i], -wr[i]);
            if constexpr (!CPLX) {
              float2 ne;
              const float2 p = mul_exact(R, br[j], nb, ne);
              const float2 l = fma_grid(p, ar, acc[sg][d]);
              low[sg][d] = cadd(low[sg][d], __ffma2_rn(ne, na, l));
            } else {                                   // w_a w_b^* (R + i X)
              const float2 ai = make_float2(wi[i], wi[i]), nai = make_float2(-wi[i], -wi[i]);
              const uint32_t* y = &wim[i >> 1][4 * j + 2 * (i & 1)];
              const float2 X = make_float2(__uint_as_float(y[0]), __uint_as_float(y[1]));
              const float2 S = __fmul2_rn(R, make_float2(rs, rs));
              float2 zr = grid0, zi = grid0;
              const float2 zrl = cadd(fma_grid(S, br[j], zr), fma_grid(X, bi[j], zr));
              const float2 zil = cadd(fma_grid(X, br[j], zi), fma_grid(S, nb, zi));
              zr = csub(zr, grid0);
              zi = csub(zi, grid0);
              float2 l = cadd(fma_grid(zr, ar, acc[sg][d]), fma_grid(zi, nai, acc[sg][d]));
              low[sg][d] = cadd(low[sg][d], __ffma2_rn(zil, nai, __ffma2_rn(zrl, ar, l)));
              l = cadd(fma_grid(zi, ar, aci[sg][d]), fma_grid(zr, ai, aci[sg][d]));
              lowi[sg][d] = cadd(lowi[sg][d], __ffma2_rn(zrl, ai, __ffma2_rn(zil, ar, l)));
            }
          }
#pragma unroll
          for (int sg = 0; sg < SG; ++sg) {
            stage(sg, at + 1 + jj, acc[sg][done], low[sg][done], aci[sg][done], lowi[sg][done]);
            if (RING && jj == G - 1 && at == G) stage(sg, 0, acc[sg][done], low[sg][done], aci[sg][done], lowi[sg][done]);
            acc[sg][done] = aci[sg][done] = grid0;
            low[sg][done] = lowi[sg][done] = zero;
          }
        }
      }
      gather(at, lam0 - 8 * j0, kap);
    }
    constexpr int AT = RING ? CR & G : 0;
    if (!RING) carry();
#pragma unroll
    for (int sg = 0; sg < SG; ++sg) {
#pragma unroll
      for (int e = 1; e < G; ++e)                      // diagonals CR - G + 1 .. CR - 1
        stage(sg, AT + e, acc[sg][e % G], low[sg][e % G], aci[sg][e % G], lowi[sg][e % G]);
    }
    stage_zero(AT + G);
    gather(AT, lam0 - 8 * CR, kap);
  }
}
// The same as a function of its own, whose registers do not add to the other splits': inlined, the four
// splits of complex weights and the four of real ones beside them in a launch spill inside the loops
// (8x64 with gains 1363 us, with calls 1227).
template <int G, int CR, bool CPLX>
__device__ __noinline__ void corr_phase_call(uint32_t tacc, int cols, int row0, int col0, float scale,
                                             int ws0, int wslots, int stg0, int v0, int nv, int half,
                                             int nx, int ny, int nyp, int mx, float lscale,
                                             bool diag, uint32_t drained, uint32_t drained2) {
  corr_phase<G, CR, CPLX>(tacc, cols, row0, col0, scale, ws0, wslots, stg0, v0, nv, half, nx, ny, nyp,
                          mx, lscale, diag, drained, drained2);
}

// Entries of a twiddle table that a transform of n reads: half of them where n is a power of two.
__host__ __device__ inline int tw_len(int n) { return (n & (n - 1)) == 0 && n > 1 ? n >> 1 : n; }

// ---- transform of an item's V to beams (256 threads of each CTA of the pair; the first takes the
// even pairs of E-W beams, the second the odd ones): over kappa in
// place when mx is a power of two (decimation in frequency: E-W beam A ends in row brev(A)), by
// the definition otherwise; then over lambda, two E-W beams per complex transform of length my
// (their spectra are real): z = H_A0 + i H_A1 with H_A[m] the Hermitian part of the sum of
// lambda = m (mod my).
__device__ void corr_beams(const CorrJob& J, int64_t item, int rank, float* v, int nv, float4* z,
                           const float4* tw, int tid) {
  const BeamArgs& a = J.a;
  const int ny = J.ny, mx = a.mx, my = a.my;
  const float4* ew = tw + tw_len(my);                  // exp(-2 pi i k / mx), after exp(-2 pi i k / my)
  const int np2 = ((mx + 1) / 2 - rank + 1) / 2;       // pairs of this CTA: u = 2 i + rank
  if (np2 <= 0) return;
  auto log2_of = [](int n) { return 31 - __clz(n); };
  const int lgx = log2_of(mx), lgy = log2_of(my);
  const bool pow2x = (1 << lgx) == mx, pow2y = (1 << lgy) == my;
  auto get = [&](int o) {
    return Cdd{make_float2(v[o], v[2 * nv + o]), make_float2(v[nv + o], v[3 * nv + o])};
  };
  auto put = [&](int o, const Cdd& x) {
    v[o] = x.h.x;
    v[nv + o] = x.l.x;
    v[2 * nv + o] = x.h.y;
    v[3 * nv + o] = x.l.y;
  };
  if (pow2x) {
    for (int st = lgx - 1; st >= 0; --st) {
      const int half = 1 << st;
      for (int o = tid; o < (mx >> 1) * ny; o += EPI) {
        const int b = o / ny, lam = o - b * ny;
        const int k = b & (half - 1), i0 = (((b >> st) << (st + 1)) + k) * ny + lam, i1 = i0 + half * ny;
        const Cdd x = get(i0), y = get(i1);
        const Cdd d = dd_sub(x, y);
        put(i0, dd_add(x, y));
        put(i1, k == 0 ? d : dd_cmul(d, ew[k << (lgx - 1 - st)]));
      }
      bar_epi();
    }
  }
  // sum over lambda = m (mod my) of E-W beam A
  auto beam_lag = [&](int A, int m) {
    Cdd s = dd_zero();
    for (int lam = m; lam < ny; lam += my) {
      if (pow2x) {
        s = dd_add(s, get((lgx ? (int)(__brev((unsigned)A) >> (32 - lgx)) : 0) * ny + lam));
      } else {
        int k = 0;
        for (int kap = 0; kap < mx; ++kap) {
          s = dd_add(s, dd_cmul(get(kap * ny + lam), ew[k]));
          k += A;
          if (k >= mx) k -= mx;
        }
      }
    }
    return s;
  };
  const bool simple = pow2x && my >= 2 * ny - 1;       // every lag alone in its residue
  auto hermitian = [&](int A, int m) {                 // (H[m] + conj H[-m]) / 2
    if (simple) {
      const int lam = m < ny ? m : my - m;
      if (lam >= ny) return dd_zero();
      Cdd x = get((lgx ? (int)(__brev((unsigned)A) >> (32 - lgx)) : 0) * ny + lam);
      const float c = m == 0 ? 0.f : m < ny ? 0.5f : -0.5f, e = m == 0 ? 1.f : 0.5f;
      return Cdd{make_float2(e * x.h.x, c * x.h.y), make_float2(e * x.l.x, c * x.l.y)};
    }
    Cdd g = beam_lag(A, m == 0 ? 0 : my - m);
    g.h.y = -g.h.y;
    g.l.y = -g.l.y;
    Cdd s = dd_add(beam_lag(A, m), g);
    s.h = make_float2(0.5f * s.h.x, 0.5f * s.h.y);
    s.l = make_float2(0.5f * s.l.x, 0.5f * s.l.y);
    return s;
  };
  auto zget = [&](int i) {
    const float4 t = z[i];
    return Cdd{make_float2(t.x, t.y), make_float2(t.z, t.w)};
  };
  auto zput = [&](int i, const Cdd& x) { z[i] = make_float4(x.h.x, x.h.y, x.l.x, x.l.y); };
  for (int o = tid; o < np2 * my; o += EPI) {
    const int u = o / my, m = o - u * my, A0 = 2 * (2 * u + rank);
    Cdd p = dd_zero();
#pragma unroll 1
    for (int A = min(A0 + 1, mx - 1); A >= A0; --A) {
      p = Cdd{make_float2(-p.h.y, p.h.x), make_float2(-p.l.y, p.l.x)};      // i x the odd beam
      p = dd_add(p, hermitian(A, m));
    }
    zput(u * my + (pow2y && lgy > 0 ? (int)(__brev((unsigned)m) >> (32 - lgy)) : m), p);
  }
  bar_epi();
  if (pow2y) {
    for (int st = 0; st < lgy; ++st) {                 // in place, decimation in time
      const int half = 1 << st;
      for (int o = tid; o < np2 * (my >> 1); o += EPI) {
        const int u = o >> (lgy - 1), b = o & ((my >> 1) - 1);
        const int k = b & (half - 1), i0 = u * my + ((b >> st) << (st + 1)) + k;
        const Cdd x = zget(i0), y = dd_cmul(zget(i0 + half), tw[k << (lgy - 1 - st)]);
        zput(i0, dd_add(x, y));
        zput(i0 + half, dd_sub(x, y));
      }
      bar_epi();
    }
  }
  float* dst = a.beams + item * (int64_t)(mx * my);
  for (int o = tid; o < np2 * my; o += EPI) {
    const int u = o / my, B = o - u * my, A0 = 2 * (2 * u + rank);
    float2 y;
    if (pow2y) {
      const float4 t = z[o];
      y = make_float2(t.x, t.y);
    } else {
      Cdd s = dd_zero();
      int k = 0;
      for (int m = 0; m < my; ++m) {
        s = dd_add(s, dd_cmul(zget(u * my + m), tw[k]));
        k += B;
        if (k >= my) k -= my;
      }
      y = s.h;
    }
    // intensities are sums of squares: rounding may leave a beam without power just below 0
    dst[A0 * my + B] = y.x < 0.f ? 0.f : ldexpf(y.x, J.out_exp);
    if (A0 + 1 < mx) dst[(A0 + 1) * my + B] = y.y < 0.f ? 0.f : ldexpf(y.y, J.out_exp);
  }
}

// ---- producers (256 threads): voltages of this CTA's row slots and its half of the column slots,
// 64 snapshots per stage, as e4m3 into the operand ring. Four warps fill a stage and the other four
// the next, so that one half's waits run under the other's stores. A thread takes one 16-slot
// unit of the rows and one of the columns at every 16th snapshot of the stage; eight lanes hold the eight snapshots of a core matrix, so a quarter-warp's 16-byte
// stores fill 128 bytes.
__device__ __forceinline__ void store_units(const uint4 (&x)[NE], unsigned char* st) {
#pragma unroll
  for (int e = 0; e < NE; ++e) {
    uint4 re, im;
    unpack16(x[e], re, im);
    *reinterpret_cast<uint4*>(st + e * 2 * LBO) = re;
    *reinterpret_cast<uint4*>(st + e * 2 * LBO + TILE) = im;
  }
}
// Columns that are the rows themselves (a full diagonal tile) are not staged again.
__device__ __forceinline__ bool separate_cols(int I, int J, int cols) { return I != J || cols != 256; }

// Where a producer stands: the operand stage (slot, par) and whose turn it is, the staged voltages
// (rs, rpar).
struct ProdState {
  int slot = 0, turn = 0, rs = 0;
  uint32_t par = 1, rpar = 0;
};

// An item's stages from voltages staged by TMA: the 128-byte swizzle moves 16-byte unit fb of row k to
// fb ^ (k & 7), so eight lanes reading one unit of eight rows touch 128 distinct bytes.
__device__ __forceinline__ bool produce_staged(const CorrParams& P, const CorrJob& J,
                                               const unsigned char* raw, unsigned char* ring,
                                               uint64_t* bars, volatile int* abort_sm, int t,
                                               uint32_t full0, ProdState& S) {
  const int lane = t & 31, grp = t >> 7, k = (t & 7) + 8 * ((t >> 6) & 1), fb = (t >> 3) & 7;
  raw += k * 128 + ((fb ^ (k & 7)) << 4);
  const int nt = J.nt, np = J.np, nsnap = J.a.n_int * J.a.npol;
  for (int I = 0; I < nt; ++I)
    for (int Jc = I; Jc < nt; ++Jc) {
      const int cols = tile_cols(np, Jc);
      const bool hasb = separate_cols(I, Jc, cols) && 16 * fb < cols / 2;
      for (int left = nsnap; left > 0; left -= KS) {
        if (S.turn == grp) {
          const bool ok = wait_pair(bars + RAWF + S.rs, S.rpar, abort_sm) &&
                          wait_pair(bars + EMPTY + S.slot, S.par, abort_sm);
          if (!ok) corr_fail(P, abort_sm);
          if (!__all_sync(0xffffffffu, ok)) return false;
          const unsigned char* src = raw + S.rs * (2 * RAW);
          unsigned char* dst = ring + S.slot * STAGE;
          uint4 x[NE], y[NE];
#pragma unroll
          for (int e = 0; e < NE; ++e) {
            x[e] = *reinterpret_cast<const uint4*>(src + e * (RAW / NE));
            if (hasb) y[e] = *reinterpret_cast<const uint4*>(src + RAW + e * (RAW / NE));
            if (k + 16 * e >= left) x[e] = y[e] = make_uint4(0u, 0u, 0u, 0u);   // the next window's
          }
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(bars + RAWE + S.rs);
          store_units(x, dst);
          if (hasb) store_units(y, dst + 2 * TILE);
          tc::fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) arrive_cluster(full0 + 8 * S.slot);
        }
        S.turn ^= 1;
        if (++S.slot == P.s.ns) { S.slot = 0; S.par ^= 1; }
        if (++S.rs == P.s.nr) { S.rs = 0; S.rpar ^= 1; }
      }
    }
  return true;
}
// One thread: the TMA tiles of every stage of the jobs that take them, rows and (if separate) columns.
__device__ __forceinline__ void stage_volts(const CorrParams& P, unsigned char* raw, uint64_t* bars,
                                            volatile int* abort_sm, uint32_t rank, int64_t pair,
                                            int64_t npairs) {
  const int NR = P.s.nr;
  const uint32_t raw0 = tc::smem_u32(raw);
  int rs = 0;
  uint32_t rpar = 1;
  int64_t n = 0;                                       // stages issued
  int job = 0;
  bool ok = true;
  const CorrJob* last = nullptr;
  for (int64_t item = pair; item < P.total && ok; item += npairs) {
    const CorrJob& J = find_job(P, item, job);
    if (!J.tma) continue;
    if (P.table && &J != last) acquire_map(&J.map);
    last = &J;
    const int nt = J.nt, np = J.np, npol = J.a.npol, nch = J.nch;
    const int64_t jw = (item - J.item0) / J.a.nfreq;
    const int f = (int)(item - J.item0 - jw * J.a.nfreq), t0 = (int)(jw * J.a.n_int);
    for (int I = 0; I < nt && ok; ++I)
      for (int Jc = I; Jc < nt && ok; ++Jc) {
        const int cols = tile_cols(np, Jc);
        const bool sep = separate_cols(I, Jc, cols);
        const int xa = 256 * I + 128 * (int)rank, xb = 256 * Jc + (int)rank * (cols / 2);
        for (int c = 0; c < nch && ok; ++c, ++n) {
          ok = wait_pair(bars + RAWE + rs, rpar, abort_sm);
          if (!ok) break;
          tc::mbar_arrive_expect_tx(bars + RAWF + rs, sep ? 2 * RAW : RAW);
          const int t = t0 + c * KS / npol;
          tma_volts(raw0 + rs * (2 * RAW), &J.map, xa, f, t, bars + RAWF + rs);
          if (sep) tma_volts(raw0 + rs * (2 * RAW) + RAW, &J.map, xb, f, t, bars + RAWF + rs);
          if (++rs == NR) { rs = 0; rpar ^= 1; }
        }
      }
  }
  if (!ok) corr_fail(P, abort_sm);
  // every copy issued must have landed before the CTA exits
  volatile int never = 0;
  for (int64_t i = n > NR ? n - NR : 0; i < n; ++i)
    wait_pair(bars + RAWF + (int)(i % NR), (uint32_t)((i / NR) & 1), &never);
}

// From global memory, byte by byte where the lattice or the pointer is not a multiple of 16 bytes.
__device__ __forceinline__ bool produce_direct(const CorrParams& P, const CorrJob& J, int64_t item,
                                               unsigned char* ring, uint64_t* bars,
                                               volatile int* abort_sm, int t, uint32_t rank,
                                               uint32_t full0, ProdState& S) {
  const int lane = t & 31, grp = t >> 7, k = (t & 7) + 8 * ((t >> 6) & 1), fb = (t >> 3) & 7;
  const BeamArgs& a = J.a;
  const int nt = J.nt, np = J.np, nsnap = a.n_int * a.npol, nyp = J.nyp, ny = J.ny, nx = a.nx;
  const uint8_t* begin = a.volts;
  const uint8_t* end = begin + a.nwin * a.n_int * a.nfreq * a.npol * (int64_t)J.nant;
  const uint8_t* ivol = item_volts(a, item - J.item0, J.nant);
  for (int I = 0; I < nt; ++I)
    for (int Jc = I; Jc < nt; ++Jc) {
      const int cols = tile_cols(np, Jc);
      const bool hasb = separate_cols(I, Jc, cols) && 16 * fb < cols / 2;
      int off[2] = {0, 0}, cnt[2] = {0, 0};            // feed offset and live feeds of the units
      auto unit = [&](int s, int b) {
        const int ix = s / nyp, iy = s - ix * nyp;
        off[b] = ix * ny + iy;
        cnt[b] = ix < nx ? max(0, min(16, ny - iy)) : 0;
      };
      unit(256 * I + 128 * (int)rank + 16 * fb, 0);
      if (hasb) unit(256 * Jc + (int)rank * (cols / 2) + 16 * fb, 1);
      for (int g = k; g - k < nsnap; g += KS) {
        if (S.turn == grp) {
          const bool ok = wait_pair(bars + EMPTY + S.slot, S.par, abort_sm);
          if (!ok) corr_fail(P, abort_sm);
          if (!__all_sync(0xffffffffu, ok)) return false;
#pragma unroll 1
          for (int b = 0; b < (hasb ? 2 : 1); ++b) {
            uint4 x[NE];
#pragma unroll
            for (int e = 0; e < NE; ++e) {
              const int ge = g + 16 * e;
              x[e] = load16_any(ivol + snap_offset(a, ge, J.nant) + (b ? off[1] : off[0]),
                                ge < nsnap ? (b ? cnt[1] : cnt[0]) : 0, begin, end);
            }
            store_units(x, ring + S.slot * STAGE + b * (2 * TILE));
          }
          tc::fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) arrive_cluster(full0 + 8 * S.slot);
        }
        S.turn ^= 1;
        if (++S.slot == P.s.ns) { S.slot = 0; S.par ^= 1; }
      }
    }
  return true;
}

// Each item by the way its own job allows: an array whose voltages cannot come by TMA does not slow
// the others of its launch.
__device__ __forceinline__ void produce(const CorrParams& P, const unsigned char* raw, unsigned char* ring,
                                        uint64_t* bars, volatile int* abort_sm, int t, uint32_t rank,
                                        int64_t pair, int64_t npairs) {
  ring += (t & 7) * 16 + ((t >> 6) & 1) * LBO + ((t >> 3) & 7) * SBO;
  const uint32_t full0 = map_rank(tc::smem_u32(bars + FULL), 0);
  ProdState S;
  int job = 0;
  bool ok = true;
  for (int64_t item = pair; item < P.total && ok; item += npairs) {
    const CorrJob& J = find_job(P, item, job);
    ok = J.tma ? produce_staged(P, J, raw, ring, bars, abort_sm, t, full0, S)
               : produce_direct(P, J, item, ring, bars, abort_sm, t, rank, full0, S);
  }
}

}  // namespace

template <bool CPLX>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(corr::NT, 1)
    beams_corr_kernel(const __grid_constant__ CorrParams P) {
  extern __shared__ __align__(1024) unsigned char smem_corr[];
  __shared__ uint64_t bars[NBAR];
  __shared__ uint32_t taddr_sm;
  __shared__ int abort_flag;
  unsigned char* smem = smem_corr;
  volatile int* abort_sm = &abort_flag;
  const Lay Y = lay_of(P.s);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t rank = cluster_rank();
  const int64_t pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const int NS = P.s.ns;

  if (warp == 16) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     tc::smem_u32(&taddr_sm)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;\n");
  }
  if (tid == 0) {
    for (int i = 0; i < NBAR; ++i) {
      uint32_t c = 1;                                  // MMA commits, PV, PE
      if (i == RF || i == IF) c = 2 * EPI / 32;         // warps of both CTAs
      if (i >= FULL && i < FULL + MAXNS) c = 2 * PROD / 64;      // half of the producers
      if (i >= EMPTY && i < EMPTY + MAXNS) c = 2;      // commits of both issuers
      if (i >= RAWE && i < RAWE + MAXNR) c = PROD / 64;
      tc::mbar_init(bars + i, c);
    }
    tc::mbar_init_fence();
    abort_flag = 0;
  }
  {
    int* v = reinterpret_cast<int*>(smem + Y.v);
    for (int i = tid; i < 4 * P.s.vlen; i += NT) v[i] = 0;
  }
  tc::fence_before_sync();
  cluster_sync();
  tc::fence_after_sync();
  const uint32_t tbase = taddr_sm;
  auto fail = [&]() { corr_fail(P, abort_sm); };
  auto wait_one = [&](int bar, uint32_t parity) -> bool {
    if (wait_pair(bars + bar, parity, abort_sm)) return true;
    fail();
    return false;
  };
  auto wait_warp = [&](int bar, uint32_t parity) -> bool {
    return __all_sync(0xffffffffu, wait_one(bar, parity)) != 0;
  };

  if (warp < 8) {
    // ================================================= epilogue
    float* ws = reinterpret_cast<float*>(smem + Y.w);
    int* vv = reinterpret_cast<int*>(smem + Y.v);
    float* stg = reinterpret_cast<float*>(smem + Y.stg);
    float4* tab = reinterpret_cast<float4*>(smem + Y.tab);
    const int wslots = P.s.wslots;
    const uint32_t rf = map_rank(tc::smem_u32(bars + RF), 0), imf = map_rank(tc::smem_u32(bars + IF), 0);
    const CorrJob* last = nullptr;
    int64_t item = pair;
    int job = 0;
    uint32_t ph = 0, iph = 0;                          // tile and item parities
    bool ok = true;
    while (item < P.total && ok) {
      const CorrJob& J = find_job(P, item, job);
      const JobRegs R{J.a.nx, J.ny, J.nyp, J.np, J.nt, J.a.mx, J.mode + (CPLX && !J.a.real_w ? 4 : 0),
                      J.rscale, J.lscale};
      const int nv = R.mx * R.ny;
      if (&J != last) {                                // weights in slot order, zeros between
        bar_epi();
        for (int s = tid; s < wslots; s += EPI) {
          const int ix = s / J.nyp, iy = s - ix * J.nyp;
          float2 w = make_float2(0.f, 0.f);
          if (ix < J.a.nx && iy < J.ny) w = J.a.w[ix * J.ny + iy];
          ws[s] = ldexpf(w.x, J.w_exp);
          if (CPLX) ws[wslots + s] = ldexpf(w.y, J.w_exp);
        }
        const int ty = tw_len(J.a.my), tx = tw_len(J.a.mx);
        for (int i = tid; i < ty + tx; i += EPI) tab[i] = J.a.cw[i < ty ? i : J.a.my + i - ty];
        last = &J;
        bar_epi();
      }
      for (int I = 0; I < R.nt && ok; ++I)
        for (int Jc = I; Jc < R.nt && ok; ++Jc) {
          const int cols = tile_cols(R.np, Jc);
          const int row0 = 256 * I + 128 * (int)rank, col0 = 256 * Jc;
          // off the diagonal a tile stands for its mirror too
          if (CPLX && (R.mode & 4)) {                  // complex weights: both halves at once
            ok = wait_warp(RD, ph) && wait_warp(ID, ph);
            if (ok) {
              tc::fence_after_sync();
#define FFTBF_PHASE(F, G, CR)                                                                           \
  F<G, CR, CPLX>(tbase, cols, row0, col0, 2.f * R.rscale, Y.w, wslots, Y.stg, Y.v, nv, 0, R.nx, R.ny,    \
                 R.nyp, R.mx, R.lscale, I == Jc, rf, imf)
              switch (R.mode & 3) {
                case 3: FFTBF_PHASE(corr_phase_call, 4, 16); break;
                case 0: FFTBF_PHASE(corr_phase_call, 4, 8); break;
                case 1: FFTBF_PHASE(corr_phase_call, 4, 4); break;
                default: FFTBF_PHASE(corr_phase, 2, 2); break;
              }
#undef FFTBF_PHASE
            }
          } else {
#pragma unroll 1
            for (int half = 0; half < 2 && ok; ++half) {
              ok = wait_warp(half ? ID : RD, ph);
              if (!ok) break;
              tc::fence_after_sync();
#define FFTBF_PHASE(F, G, CR)                                                                         \
  F<G, CR, false>(tbase + 256 * half, cols, row0, col0, half == 0 && I == Jc ? R.rscale : 2.f * R.rscale, \
                  Y.w, 0, Y.stg, Y.v, nv, half, R.nx, R.ny, R.nyp, R.mx, R.lscale, false,                 \
                  half ? imf : rf, 0)
#define FFTBF_REAL(G, CR)                                                                             \
  if constexpr (CPLX) FFTBF_PHASE(corr_phase_call, G, CR);                                              \
  else FFTBF_PHASE(corr_phase, G, CR)
              switch (R.mode) {
                case 3: FFTBF_REAL(4, 16); break;
                case 0: FFTBF_REAL(4, 8); break;
                case 1: FFTBF_REAL(4, 4); break;
                default: FFTBF_REAL(2, 2); break;
              }
#undef FFTBF_REAL
#undef FFTBF_PHASE
            }
          }
          ph ^= 1;
        }
      ok = bar_epi_all(ok);                            // the warps leave together or not at all
      if (!ok) break;
      // ---- item complete: each CTA adds the other's part of V to its own and transforms its share
      // of the beams; V is cleared once the other has read it. One thread releases and acquires
      // at cluster scope for all (the CTA's barriers carry it to the others).
      if (tid == 0) {
        arrive_release_cluster(map_rank(tc::smem_u32(bars + PV), rank ^ 1));
        ok = wait_pair<true>(bars + PV, iph, abort_sm);
        if (!ok) fail();
      }
      ok = bar_epi_all(ok);
      if (!ok) break;
      const uint32_t peer = map_rank(tc::smem_u32(vv), rank ^ 1);
      float* u = stg;                                  // the sum, then the transform's buffer after it
#pragma unroll 1
      for (int i0 = tid; i0 < nv; i0 += 4 * EPI) {
        int p[4][4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int i = min(i0 + k * EPI, nv - 1);
#pragma unroll
          for (int c = 0; c < 4; ++c)
            asm volatile("ld.shared::cluster.b32 %0, [%1];\n" : "=r"(p[k][c]) : "r"(peer + 4 * (c * nv + i)) : "memory");
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int i = i0 + k * EPI;
          if (i >= nv) break;
          // whole numbers and 2^-19 units, each to a float and its remainder
          const int re = vv[i] + p[k][0], rl = vv[nv + i] + p[k][1];
          const int im = vv[2 * nv + i] + p[k][2], il = vv[3 * nv + i] + p[k][3];
          auto two = [](int x, int y, float s) {
            const float fx = (float)x, fy = (float)y;
            return Cdd{make_float2(s * fx, s * fy),
                       make_float2(s * (float)(x - (int)fx), s * (float)(y - (int)fy))};
          };
          const Cdd t = dd_add(two(re, im, 1.f), two(rl, il, 1.f / R.lscale));
          u[i] = t.h.x;
          u[nv + i] = t.l.x;
          u[2 * nv + i] = t.h.y;
          u[3 * nv + i] = t.l.y;
        }
      }
      bar_epi();
      if (tid == 0) arrive_release_cluster(map_rank(tc::smem_u32(bars + PE), rank ^ 1));
      corr_beams(J, item - J.item0, (int)rank, u, nv, reinterpret_cast<float4*>(u + 4 * nv), tab, tid);
      if (tid == 0) {
        ok = wait_pair<true>(bars + PE, iph, abort_sm);   // the other CTA has read this one's V
        if (!ok) fail();
      }
      ok = bar_epi_all(ok);
      if (!ok) break;
      for (int i = tid; i < 4 * nv; i += EPI) vv[i] = 0;
      bar_epi();
      iph ^= 1;
      item += npairs;
    }
  } else if (warp < 8 + PROD / 32) {
    // ================================================= producers
    produce(P, smem + Y.raw, smem + Y.ring, bars, abort_sm, tid - EPI, rank, pair, npairs);
  } else if (warp == 17 && lane == 0 && P.s.tma) {
    stage_volts(P, smem + Y.raw, bars, abort_sm, rank, pair, npairs);
  } else if ((warp == 16 || warp == 18) && rank == 0 && lane == 0) {
    // ================================================= MMA issue: real (16), imaginary half (18)
    const bool im = warp == 18;
    const uint64_t desc0 = tc::smem_desc(tc::smem_u32(smem + Y.ring), LBO, SBO);
    const uint32_t acc = tbase + (im ? 256 : 0);
    const int done = im ? ID : RD, drained = im ? IF : RF;
    int slot = 0;
    uint32_t par = 0, tph = 1;                         // tph: parity of the drained barrier
    int job = 0;
    bool ok = true, issued = false;
    for (int64_t item = pair; item < P.total && ok; item += npairs) {
      const CorrJob& J = find_job(P, item, job);
      const int nt = J.nt, np = J.np, nsnap = J.a.n_int * J.a.npol;
      for (int I = 0; I < nt && ok; ++I)
        for (int Jc = I; Jc < nt && ok; ++Jc) {
          const int cols = tile_cols(np, Jc);
          const bool diag = I == Jc;
          const uint32_t id = (1u << 4) | (1u << 15) | (1u << 16) | ((uint32_t)(cols >> 3) << 17) | (16u << 24);
          // first product Xr Yr^T or Xi Yr^T, second Xi Yi^T or -Xr Yi^T (negated column operand;
          // none on the diagonal)
          const uint64_t dt = TILE >> 4, db = separate_cols(I, Jc, cols) ? 2 * dt : 0;
          const uint64_t a1 = im ? dt : 0, a2 = im ? 0 : dt;
          const uint32_t id2 = im ? id | (1u << 14) : id;
          const bool second = !im || !diag;
          ok = wait_one(drained, tph);
          if (!ok) break;
          tc::fence_after_sync();
          issued = true;
          for (int left = nsnap; left > 0; left -= KS) {
            ok = wait_one(FULL + slot, par);
            if (!ok) break;
            tc::fence_after_sync();
            const uint64_t d = desc0 + (uint64_t)(slot * (STAGE >> 4));
            constexpr uint64_t K32 = (4 * LBO) >> 4;   // the second K = 32 step of the stage
            mma_f8_pair(acc, d + a1, d + db, id, left < nsnap);
            if (second) mma_f8_pair(acc, d + a2, d + db + dt, id2, 1u);
            if (left > 32) {
              mma_f8_pair(acc, d + a1 + K32, d + db + K32, id, 1u);
              if (second) mma_f8_pair(acc, d + a2 + K32, d + db + dt + K32, id2, 1u);
            }
            commit_pair(bars + EMPTY + slot);
            if (++slot == NS) { slot = 0; par ^= 1; }
          }
          if (!ok) break;
          commit_pair(bars + done);
          tph ^= 1;
        }
    }
    // every MMA issued, those of a tile given up half-way included, must have completed before the
    // pair frees its memory
    if (issued) {
      volatile int never = 0;
      commit_pair(bars + (im ? LI : LR));
      wait_pair(bars + (im ? LI : LR), 0, &never);
    }
  }
  __syncwarp();
  tc::fence_before_sync();
  cluster_sync();
  tc::fence_after_sync();
  if (warp == 16)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;\n" ::"r"(tbase), "r"(512u));
}

// ------------------------------------------------------------------------- host side --
// Split of a lattice into slots: nyp and the (G, CR) of the epilogue.
static void corr_split(int ny, int* nyp, int* mode) {
  auto up = [&](int m) { return (ny + m - 1) / m * m; };
  // multiples of 16 stay as they are (slots = feeds, staged by TMA); others are rounded up, to
  // the longer runs where the padding is small
  if (ny % 16 == 0) *nyp = ny;
  else *nyp = up(ny >= 192 ? 64 : ny >= 96 ? 32 : 16);
  // the longest column runs that divide a row: 128, 64, 32 or 16 slots (a run of n 8-slot groups has
  // n / 4 + 1 gathers; 4x256, 1024 work items: 1614 us at 128 slots, 1720 at 64)
  const int n = *nyp;
  *mode = n % 128 == 0 ? 3 : n % 64 == 0 ? 0 : n % 32 == 0 ? 1 : 2;
}

bool corr_make_job(const BeamArgs& a, CorrJob* J) {
  CorrJob j{};
  j.a = a;
  j.ny = a.ny;
  j.nant = a.nx * a.ny;
  corr_split(a.ny, &j.nyp, &j.mode);
  j.np = a.nx * j.nyp;
  j.nt = (j.np + 255) / 256;
  const int64_t nsnap = (int64_t)a.n_int * a.npol;
  j.nch = (int)((nsnap + corr::KS - 1) / corr::KS);
  // TMA coordinates are 32 bits wide: a call of more samples loads them directly
  j.tma = (a.ny & 15) == 0 && (reinterpret_cast<uintptr_t>(a.volts) & 15) == 0 && KS % a.npol == 0 &&
          a.nwin * a.n_int <= INT32_MAX - KS;
  j.nitems = a.nwin * a.nfreq;
  // Units of V. With weights below 2 (w_exp) a product with its mirror is below 2 128 4 2^ns; a unit
  // is 2^-19 of that, and with n = nx ny ceil(nx / mx) feed pairs of one separation above 1024 2^e
  // times it (n <= 1024 2^e): V stays below 2^30 units. What lies below a unit, at most 1/2 + 2^-5 a
  // product and 1.4 with complex weights, sums over up to 2 n of them to 1.4 2^(11 + e) units at most,
  // and is kept in 2^-(19 - e) of one: below 2^31. With e = 4 that is 2^-30 of the largest product,
  // rounded once for every 16 or more of them; lattices folded further take the transform.
  auto clog2 = [](int64_t n) { int l = 0; while (((int64_t)1 << l) < n) ++l; return l; };
  const int ns = clog2(nsnap), e = std::max(0, clog2((int64_t)j.nant * ((a.nx + a.mx - 1) / a.mx)) - 10);
  const int z = a.real_w ? 0 : 31 - ns, w = a.w_exp == kNoExp ? 0 : a.w_exp;
  j.w_exp = z - w;                                     // complex: z = w_b^* R up to 2^21
  j.rscale = ldexpf(1.f, 27 - ns - e - 2 * z);         // R carries 2^-18
  j.lscale = ldexpf(1.f, 19 - e);
  j.out_exp = ns - 9 + e + 2 * w;
  *J = j;
  // sums stay exact to 128 * 2^16 snapshots with room; V and the transform fit beside the ring
  return a.cw && a.w_exp != kNoExp && e <= 4 && j.np <= 2048 && nsnap <= 65536 &&
         (int64_t)a.mx * a.ny <= corr::VMAX &&
         (int64_t)((a.mx + 1) / 2) * a.my <= 2048;
}

// Shared-memory sizes that hold every job of a launch; false if they do not fit.
bool corr_sizes(const CorrJob* jobs, int n, CorrSizes* out) {
  CorrSizes s{};
  for (int i = 0; i < n; ++i) {
    s.cplx |= !jobs[i].a.real_w;
    s.tma |= jobs[i].tma;
  }
  for (int i = 0; i < n; ++i) {
    const CorrJob& j = jobs[i];
    const int m = j.mode, c = j.a.real_w ? 1 : 2;
    const int G = m == 2 ? 2 : 4, CR = m == 3 ? 16 : m == 0 ? 8 : m == 1 ? 4 : 2;
    s.wslots = std::max(s.wslots, 256 * j.nt);
    s.vlen = std::max(s.vlen, j.a.mx * j.ny);
    s.stg = std::max({s.stg, stg_floats(G, CR, c), (4 * j.a.mx * j.ny + ((j.a.mx + 1) / 2 + 1) / 2 * j.a.my * 4 + 7) / 8});
    s.tab = std::max(s.tab, tw_len(j.a.my) + tw_len(j.a.mx));
  }
  s.stg = (s.stg + 3) & ~3;
  // the voltages' ring first (their latency is the longest), then operand stages
  s.nr = s.tma ? 2 : 0;
  s.ns = corr::MAXNS;
  while (s.ns >= 2 && lay_of(s).total > corr::SMEM_MAX) --s.ns;
  *out = s;
  return s.ns >= 2;
}

// Tensor map of a job's voltages: feeds, polarisations, channels, samples; tiles of 128 feeds x all
// polarisations x one channel x 64 snapshots, 128-byte swizzle.
static int corr_map(CorrJob* j) {
  using Encode = decltype(&cuTensorMapEncodeTiled);
  static const Encode encode = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<Encode>(f);
  }();
  if (!encode) return set_error(FFTBF_ECUDA, "the driver has no cuTensorMapEncodeTiled");
  const BeamArgs& a = j->a;
  const cuuint64_t dims[4] = {(cuuint64_t)j->nant, (cuuint64_t)a.npol, (cuuint64_t)a.nfreq,
                              (cuuint64_t)(a.nwin * a.n_int)};
  const cuuint64_t strides[3] = {(cuuint64_t)j->nant, (cuuint64_t)j->nant * a.npol,
                                 (cuuint64_t)j->nant * a.npol * a.nfreq};
  const cuuint32_t box[4] = {128, (cuuint32_t)a.npol, 1, (cuuint32_t)(KS / a.npol)};
  const cuuint32_t one[4] = {1, 1, 1, 1};
  auto make = [&] {
    return encode(&j->map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<uint8_t*>(a.volts), dims, strides,
                  box, one, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  };
  CUresult r = make();
  if (r == CUDA_ERROR_INVALID_CONTEXT) {               // a thread's first call: the runtime binds its
    int dev = 0;                                       // context only with work of its own
    FFTBF_CUDA_TRY(cudaGetDevice(&dev));
    FFTBF_CUDA_TRY(cudaSetDevice(dev));
    r = make();
  }
  if (r != CUDA_SUCCESS) return set_error(FFTBF_ECUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
  return FFTBF_OK;
}

// Prepare the tensor maps of the jobs that take them.
int corr_maps(CorrJob* jobs, int n) {
  for (int i = 0; i < n; ++i) {
    if (!jobs[i].tma) continue;
    const int rc = corr_map(jobs + i);
    if (rc != FFTBF_OK) return rc;
  }
  return FFTBF_OK;
}

int corr_launch(CorrParams& p, int nsm, cudaStream_t st) {
  if (p.total <= 0) return FFTBF_OK;
  const int smem = std::max(lay_of(p.s).total, 120 * 1024);   // one CTA per SM: all tensor memory
  auto kern = p.s.cplx ? beams_corr_kernel<true> : beams_corr_kernel<false>;
  // The limit belongs to the kernel, not to this launch: every thread sets the same one, so that none
  // takes it below what another is about to launch with.
  FFTBF_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, corr::SMEM_MAX));
  const int64_t pairs = std::min<int64_t>(p.total, nsm / 2);
  kern<<<(unsigned)(2 * pairs), corr::NT, smem, st>>>(p);
  FFTBF_CUDA_TRY(cudaGetLastError());
  return FFTBF_OK;
}

// Whether the covariance is taken rather than the transform of every snapshot: an estimate of both in
// microseconds for 608 work items (eight per CTA pair) on a GB300,
//   covariance  34 us per tile and 55 us per item, 1.4 times that with complex weights (epilogue
//               and transform of V, whatever the window), and from there 0.021 us per snapshot and
//               MMA unit (a 256 x 256 product of the chunk: 3 a diagonal tile, 4 another), three
//               times that where the voltages cannot come by TMA;
//   transform   us per snapshot and 1000 beams: 0.8 the 512-beam kernels (4x256: 829 us at 512),
//               0.6 the 32-beam kernel, 1.1 those of 1024 and 2048 beams, 1.9 the other FFT
//               kernels (8x64: 979 us at 512); the direct DFT 1.0 for every N-S feed. The
//               split-FP16 kernel (split) 1.3 (4x256: 2060 us at 768).
// So 4x256 changes over near 300 snapshots, 8x64 near 90, 16x16 near 400. These are the costs of the
// covariance with its products rounded to FP32; with their errors kept it takes longer (4x256 470 us
// and up for 398, 8x64 205 for 160, 16x16 152 for 107; complex weights 820, 281, 174) and the times
// meet near 420, 110 and 570 snapshots, 4x256 with complex weights near 770. The line stays where it
// was: between the two the covariance costs up to 1.35 times the transform (complex 1.6), for an error
// of 3e-8 in place of 1e-7 to 6e-7 (2-norm), and nothing that had the smaller error loses it. Only the
// plan's sizes enter, never the number of windows or the pointer: a window's beams do not depend on
// its call.
bool corr_preferred(const BeamArgs& a, bool split) {
  CorrJob j;
  CorrSizes s;
  if (!corr_make_job(a, &j) || !corr_sizes(&j, 1, &s)) return false;
  const char* force = std::getenv("FFTBF_FP32_PATH");  // tests: "cov" or "fft"
  if (force && (force[0] == 'c' || force[0] == 'f')) return force[0] == 'c';
  const double nsnap = (double)a.n_int * a.npol, nout = (double)a.mx * a.my;
  double tiles = 0, units = 0;
  for (int c = 0; c < j.nt; ++c) {
    const double w = std::min(256, j.np - 256 * c) / 256.0;
    tiles += c + 1;
    units += w * (3 + 4 * c);
  }
  const double fixed = (34.0 * tiles + 55.0) * (a.real_w ? 1.0 : 1.4);
  const double cov = std::max(fixed, 0.6 * fixed + 0.021 * (j.ny % 16 == 0 && corr::KS % a.npol == 0 ? 1 : 3) * units * nsnap);
  double per;                                          // us per snapshot
  if (split) per = 1.3e-3 * nout;
  else if (fp32_n512_supported(a)) per = 0.8e-3 * nout;
  else if (fp32_warp_supported(a)) per = (a.my == 32 ? 0.6e-3 : a.my >= 1024 ? 1.1e-3 : 1.9e-3) * nout;
  else if (fp32_fft_supported(a.mx, a.my)) per = 1.9e-3 * std::max<double>(nout, j.nant);
  else per = 1e-3 * nout * a.nyf;
  return cov < per * nsnap;
}

int launch_beams_corr(const BeamArgs& a, int nsm, cudaStream_t st) {
  CorrParams p{};
  if (!corr_make_job(a, &p.one) || !corr_sizes(&p.one, 1, &p.s))
    return set_error(FFTBF_EUNSUPPORTED, "lattice too large for the covariance kernel");
  const int rc = corr_maps(&p.one, 1);
  if (rc != FFTBF_OK) return rc;
  p.total = p.one.nitems;
  p.njobs = 1;
  return corr_launch(p, nsm, st);
}

// Cut a list of jobs (d_table: its device copy) into launches whose shared memory fits, usually
// one, costliest items first, and number each launch's items.
int corr_plan_jobs(std::vector<CorrJob>& jobs, const CorrJob* d_table, int* err,
                   std::vector<CorrParams>* out) {
  out->clear();
  auto cost = [](const CorrJob& j) { return (j.tma ? 1.0 : 3.0) * j.np * j.np * j.nch; };
  std::stable_sort(jobs.begin(), jobs.end(),
                   [&](const CorrJob& x, const CorrJob& y) { return cost(x) > cost(y); });
  for (size_t i = 0; i < jobs.size();) {
    CorrParams p{};
    size_t n = 1;
    CorrSizes s;
    if (!corr_sizes(&jobs[i], 1, &p.s))
      return set_error(FFTBF_EUNSUPPORTED, "lattice too large for the covariance kernel");
    while (i + n < jobs.size() && corr_sizes(&jobs[i], (int)n + 1, &s)) {
      p.s = s;
      ++n;
    }
    const int rc = corr_maps(&jobs[i], (int)n);
    if (rc != FFTBF_OK) return rc;
    for (size_t k = i; k < i + n; ++k) {
      jobs[k].item0 = p.total;
      p.total += jobs[k].nitems;
    }
    p.table = d_table + i;
    p.njobs = (int)n;
    p.err = err;
    out->push_back(p);
    i += n;
  }
  return FFTBF_OK;
}

}  // namespace fftbf

// How a call of nwin windows at address `volts` would bring its voltages (tests; host only): 1 by TMA,
// 0 by direct loads, -1 if the kernel does not take the lattice.
extern "C" int fftbf_corr_staging(int nx, int ny, int pad_x, int pad_y, int npol, int nfreq, int n_int,
                                  int64_t nwin, uint64_t volts) {
  fftbf::BeamArgs a{};
  float4 here;
  a.cw = &here;
  a.nx = nx; a.ny = ny; a.mx = pad_x; a.my = pad_y;
  a.npol = npol; a.nfreq = nfreq; a.n_int = n_int;
  a.nyf = std::min(ny, pad_y);
  a.real_w = 1;
  a.nwin = nwin;
  a.volts = reinterpret_cast<const uint8_t*>(volts);
  fftbf::CorrJob j;
  return fftbf::corr_make_job(a, &j) ? j.tma : -1;
}
