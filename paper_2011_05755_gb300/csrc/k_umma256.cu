// Precision-split path, M = 256 angles (rings up to 40): spectrum
// contraction on warp-level tensor cores (mma.sync), inverse angular DFT on
// the 5th-generation tensor cores (tcgen05.mma, FP32 accumulation in TMEM).
//
// Contraction (Alg. 1, CC step).  With q = Re X - Im X, p = Re X + Im X for a
// particle ring bin and v = Re Y - Im Y, u = Re Y + Im Y for a weighted
// reference bin, one m16n8k16 per k-step of 16 rings (A: q and p of 8 rows,
// B: v and u of 4 references) leaves in one lane, for one (row, reference)
// pair and one frequency f,
//     d0 = sum q v,  d1 = sum q u,  d2 = sum p v,  d3 = sum p u,
// and with C = conj(X) Y summed over the rings (unmirrored correlation) and
// C' = X Y (mirrored, up to a half-turn):
//     2 Re C = d0 + d3,  2 Im C = d1 - d2,  2 Re C' = d1 + d2,  2 Im C' = d3 - d0.
//
// Inverse angular DFT (Alg. 1, inverse-FFT step).  Both correlations are
// real, so each is a cosine sum over 2 Re C and a sine sum over 2 Im C.
// Splitting the frequencies by parity gives four sums per angle j < 64,
//     Ee, Eo = sum over even / odd f of   2 Re C(f) cos(2 pi f j / 256),
//     Oe, Oo = sum over even / odd f of - 2 Im C(f) sin(2 pi f j / 256),
// from which four angles follow by symmetry:
//     c(j), c(256 - j) = (Ee + Eo) +- (Oe + Oo),
//     c(128 + j), c(128 - j) = (Ee - Eo) +- (Oe - Oo),
// so the largest of the four is max(Ee + Eo + |Oe + Oo|, Ee - Eo + |Oe - Oo|).
// The sums are matrix products over (pair, correlation) rows: D[128 x 64] =
// A[128 x 64] W[64 x 64], 64 pairs x {C, C'} rows, K = 64 frequencies of one
// parity and part, N = 64 angles; four of them fill 256 TMEM columns.  The
// operands are BF16 (one rounding of 2 Re C, 2 Im C and of the matrices), the
// sums FP32; no intermediate is rounded in between, and the whole angular
// state never exists outside TMEM.  The zero frequency is added after the
// maximum (a constant over the angles, FP32).  Angles 64 and 192 need Ee and Oo
// at j = 64: column 0 of Oo, empty at j = 0 (sin 0), holds -sum 2 Im C sin(pi f
// / 2), and Ee(64) is an alternating sum of the even 2 Re C that the contraction
// warps form in FP32, each over its own frequencies, and the f = 0 warp adds up
// (a fifth product for it took a fifth of the MMAs).
//
// What bounds it, and why this split.  Each (row, reference) pair needs all
// 129 frequencies on chip at once, so a tile cannot exceed the pairs whose
// angular state fits; here that state is the FP32 accumulators (256 KB of
// TMEM hold 64 pairs twice, so one tile's maxima are read while the next
// tile accumulates).  A tile is 8 rows x 8 references; the row fragments
// (KS x 512 bytes) stay on chip over all reference tiles, in the registers of
// the warps that use them (rings up to 36) or in shared memory, and the
// reference fragments stream from L2 into a register ring ahead of their use.
// Measured (GB300, 12,000 images of the 76-pixel, 100-reference, 81-shift
// workload, contraction stage): 20.0 ms, against 66.9 ms for cc_tc256_kernel
// (all mma.sync, angular state in shared memory, whole chunks of both
// operands staged behind CTA barriers) and about 77 ms for a tcgen05 kernel
// that ran the contraction on tcgen05 as well (four frequencies block-diagonal
// per MMA, two 16-point inverse-DFT stages with a TMEM drain each).  Bound:
// shared-memory / L1 bandwidth, tensor issue and the contraction warps'
// latency together.  With Ee(64) as a fifth product it took 20.7 ms, of which
// the reference loads hid all but 1.0, 16 of the 20 MMAs all but 3.7, and both
// together all but 7.3.  Steps measured on the way: rows in shared memory
// instead of registers 29.4 ms; one operand stage per parity instead of per
// tile 23.6; references through a per-warp TMA buffer in shared memory 27.4;
// L1::no_allocate on the reference loads 22.2; ring of 4 / 5 / 6 / 7 k-steps
// 20.7 / 20.3 / 20.0 / 20.1.
//
// Roles (16 warps, one persistent CTA per SM):
//   warps 0-7    contract: warp w holds, for each parity, 8 frequencies
//                (slots) dealt so that every warp has the same k-step count
//                and its k-steps lie side by side in both fragment layouts
//                (k-step n0 + (2 w + parity) steps + i), and writes core
//                column w (8 K-values, 16 bytes per row) of the parity's two
//                operands;
//   warps 8-11   read the accumulators of their TMEM lane quarter and write
//                the row maxima;
//   warp 12      issues every tcgen05.mma (one lane);
//   warp 13      contracts f = 0 and adds up Ee(64);
//   warp 14      copies the row fragments to shared memory (when they are
//                there).
// All waits are bounded; a wait that gives up raises a CTA abort flag and
// the device error flag, every role leaves its loop, the copying lane waits
// for its copies in flight, the issuer for its MMAs, and the TMEM is
// released.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "../../include/mra.h"
#include "dev_util.cuh"
#include "mra_internal.h"
#include "smem_limit.cuh"
#include "umma.cuh"

namespace mra {

namespace u256 {
constexpr int kThreads = 512;
constexpr int kContract = 8;                     // contraction warps
constexpr uint32_t kOperand = 128 * 64 * 2;      // one operand of a parity: 128 rows x 64 frequencies
constexpr uint32_t kZStage = 2 * kOperand;       // real and imaginary parts
constexpr uint32_t kW = 64 * 64 * 2;             // one DFT matrix
constexpr uint32_t kWBytes = kHyb256Mats * kW;   // Ee, Oe, Eo, Oo
constexpr int kNumBars = 16;  // zfull[2] zempty[2] dfull[2] dempty[2] x0full[2] afull[2] aempty[2] fin, spare
// matrices, f = 0 terms, Ee(64) and its parts (two tiles each), barriers
constexpr uint32_t kMisc = kWBytes + 2 * (64 + 128 + kContract * 128) * 4 + kNumBars * 8 + 16;
// Operand stages: both parities of a tile together, two of them, when the row
// fragments are in registers (one synchronisation per tile); beside row
// fragments in shared memory there is room for one parity.
__host__ __device__ constexpr int z_parities(int pattern) { return pattern == 0 ? 2 : 1; }
__host__ __device__ constexpr int z_stages(int pattern) { return pattern == 0 ? 2 : 1; }
}  // namespace u256

template <bool FP16>
__device__ __forceinline__ void mma_frag(float (&d)[4], const uint4 &a, uint32_t b0, uint32_t b1) {
  if constexpr (FP16)
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
  else
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t pack_bf2u(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t *>(&h);
}

__device__ __forceinline__ uint4 load_frag(const unsigned char *p) {
  uint4 v;
  asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// The k-steps of the 8 slots of a warp and parity (fewer are padded with
// zero fragments): pattern 0 = {3,2,2,2,1,1,1,1}, 1 = {3,3,2,2,2,2,2,2}.
template <int PATTERN>
struct HybPattern {
  static constexpr int kSteps = PATTERN == 0 ? 13 : 18;
  static constexpr int KS = kHyb256N0 + 16 * kSteps;
  __host__ __device__ static constexpr int cap(int s) { return s <= PATTERN ? 3 : (PATTERN == 1 || s < 4 ? 2 : 1); }
  __host__ __device__ static constexpr int first(int s) {
    int n = 0;
    for (int i = 0; i < s; ++i) n += cap(i);
    return n;
  }
};

// One parity of one tile by one contraction warp.  fa(i) and fb(i) are the
// row and reference fragments of k-step i, done(i) is called after their use.
// out[part * 2 + correlation][block][word]; with SUM, ee[block][correlation] is
// the sum of 2 Re C over the slots, the last slot's times `last`.
template <class P, bool FP16, bool SUM, class FA, class FB, class Done>
__device__ __forceinline__ void contract_parity(FA &&fa, FB &&fb, Done &&done, uint32_t (&out)[4][2][4],
                                                float (&ee)[2][2], float last) {
  float keep[2][4];
  sfor<0, 8>([&](auto ss) {
    constexpr int s = decltype(ss)::value;
    float d[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    sfor<0, P::cap(s)>([&](auto jj) {
      constexpr int i = P::first(s) + decltype(jj)::value;
      const uint4 af = fa(i), bf = fb(i);
      mma_frag<FP16>(d[0], af, bf.x, bf.y);
      mma_frag<FP16>(d[1], af, bf.z, bf.w);
      done(i);
    });
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float v[4] = {d[k][0] + d[k][3], d[k][1] + d[k][2], d[k][1] - d[k][2], d[k][3] - d[k][0]};
      if constexpr (SUM) {
#pragma unroll
        for (int e = 0; e < 2; ++e)
          ee[k][e] = s == 0 ? v[e] : (s < 7 ? ee[k][e] + v[e] : fmaf(v[e], last, ee[k][e]));
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if constexpr (s & 1)
          out[e][k][s >> 1] = pack_bf2u(keep[k][e], v[e]);
        else
          keep[k][e] = v[e];
      }
    }
  });
}

// Every angle of the 32 rows of a warp's TMEM lane quarter into the debug table (dst null: no store).
__device__ __noinline__ void hybrid_debug_row(uint32_t d, int corr, float x0, float e64, float *dst) {
#pragma unroll 1
  for (int n = 0; n < 64; ++n) {
    uint32_t r[4];
    for (int i = 0; i < 4; ++i) tmem_ld1(d + i * 64 + n, r[i]);
    tmem_ld_wait();
    const float E = __uint_as_float(r[0]), F = __uint_as_float(r[1]);
    const float G = n ? __uint_as_float(r[2]) : e64, H = __uint_as_float(r[3]);
    const float c[4] = {n ? (E + F) + (G + H) : E + F, n ? (E + F) - (G + H) : G + H,
                        n ? (E - F) + (G - H) : E - F, n ? (E - F) - (G - H) : G - H};
    const int at[4] = {n, n ? 256 - n : 64, 128 + n, n ? 128 - n : 192};
    if (dst)  // mirrored row: angle n of the transform is angle n + 128 of the table
      for (int i = 0; i < 4; ++i) dst[(at[i] + corr * 128) & 255] = c[i] + x0;
  }
}

template <int PATTERN, bool FP16>
__global__ void __launch_bounds__(u256::kThreads, 1)
    cc_hybrid256_kernel(Geometry g, TcArgs a, int ref_tiles, int per_unit, int splits, int64_t units) {
  using namespace u256;
  using P = HybPattern<PATTERN>;
  constexpr int T = P::kSteps;
  constexpr bool kRegs = PATTERN == 0;                     // row fragments in registers (104 per thread)
  constexpr int kZp = z_parities(PATTERN), kZs = z_stages(PATTERN);
  constexpr int PF = kRegs ? 6 : 9;                        // k-steps of references in the register ring
  constexpr uint32_t kTile16 = P::KS * 512u;               // fragment bytes of a row or reference tile
  extern __shared__ __align__(1024) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned char *sZ = smem;                                // [kZs][kZp] operands of a parity
  unsigned char *sW = sZ + kZs * kZp * kZStage;            // DFT matrices
  unsigned char *sF = sW + kWBytes;                        // row fragments [KS][512] (pattern 1)
  float *s_x0 = reinterpret_cast<float *>(sF + (kRegs ? 0u : kTile16));  // [2][64] zero-frequency terms
  float *s_e = s_x0 + 2 * 64;                              // [2][128] Ee(64)
  float *s_part = s_e + 2 * 128;                           // [2][8 warps][128] its parts
  uint64_t *bars = reinterpret_cast<uint64_t *>(s_part + 2 * kContract * 128);
  uint64_t *zfull = bars, *zempty = bars + 2, *dfull = bars + 4, *dempty = bars + 6, *x0full = bars + 8,
           *afull = bars + 10, *aempty = bars + 12, *fin = bars + 14;
  uint32_t *s_tmem = reinterpret_cast<uint32_t *>(bars + kNumBars);
  volatile int *abort = reinterpret_cast<volatile int *>(s_tmem + 1);

  // ---- set-up: DFT matrices, barriers, TMEM ----
  for (int i = tid; i < static_cast<int>(kWBytes / 16); i += kThreads)
    reinterpret_cast<uint4 *>(sW)[i] = __ldg(reinterpret_cast<const uint4 *>(g.hyb_w) + i);
  if (tid == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(zfull + s, kContract);
      mbar_init(zempty + s, 2);  // the MMAs have read the operands, warp 13 the parts of Ee(64)
      mbar_init(dfull + s, 1);
      mbar_init(dempty + s, 4);
      mbar_init(x0full + s, 1);
      mbar_init(afull + s, 1);
      mbar_init(aempty + s, s == 0 ? kContract + 1 : kContract);  // f = 0 is in the even part
    }
    mbar_init(fin, 1);
    *abort = (smem_u32(smem) & 127u) ? 1 : 0;  // descriptors and copies assume an aligned base
    if (*abort) atomicOr(a.err, 2);
  }
  if (warp == 12) tmem_alloc(s_tmem, 512);
  mbar_init_fence();
  fence_proxy_async();  // the DFT matrices written above are read by the tensor cores
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *s_tmem;
  const unsigned char *gA = reinterpret_cast<const unsigned char *>(a.A16);
  const unsigned char *gB = reinterpret_cast<const unsigned char *>(a.B16);
  const uint32_t limit = a.wait_limit;
  // the first reference tile of unit u; a unit's row tile is u / splits
  auto first_tile = [&](int64_t u) { return static_cast<int>(u % splits) * per_unit; };

  // registers per thread: 128 at launch; the contraction keeps its row
  // fragments, the other roles need few (2 x 200 + 64 + 48 = 4 x 128)
  if (warp < kContract) {
    // ---------------- contraction ----------------
    asm volatile("setmaxnreg.inc.sync.aligned.u32 200;");
    const uint32_t woff = (kHyb256N0 + warp * 2 * T) * 512 + lane * 16;  // this warp's first even k-step
    unsigned char *zl = sZ + warp * 2048 + lane * 16;
    const int64_t u0 = blockIdx.x;
    const unsigned char *bw = gB + static_cast<size_t>(first_tile(u0)) * kTile16 + woff;
    uint4 b[PF];
    uint4 ra[kRegs ? 2 * T : 1];
#pragma unroll
    for (int i = 0; i < PF; ++i) b[i] = load_frag(bw + i * 512);
    if constexpr (kRegs) {
      const unsigned char *aw = gA + static_cast<size_t>(u0 / splits) * kTile16 + woff;
#pragma unroll
      for (int i = 0; i < 2 * T; ++i) ra[i] = load_frag(aw + i * 512);
    }
    uint32_t t = 0, un = 0;  // tiles, units
    bool ok = !*abort;
    for (int64_t u = u0; u < units && ok; u += gridDim.x, ++un) {
      const int k0 = first_tile(u), k1 = min(k0 + per_unit, ref_tiles);
      const int64_t nu = u + gridDim.x < units ? u + gridDim.x : u;
      const unsigned char *an = gA + static_cast<size_t>(nu / splits) * kTile16 + woff;  // the next unit's row fragments
      for (int kt = k0; kt < k1 && ok; ++kt, ++t) {
        const bool last = kt + 1 == k1;
        const unsigned char *bn = last ? gB + static_cast<size_t>(first_tile(nu)) * kTile16 + woff : bw + kTile16;
        auto parity = [&](auto pp) {
          constexpr int p = decltype(pp)::value;
          uint32_t out[4][2][4];
          float ee[2][2];
          // even f = 2 (8 s + warp) + 2; the last, f = 128, is its own mirror image
          const float lastw = warp == 7 ? 0.5f : 1.f;
          // register ring: entry i % PF holds k-step i; refilled on use with
          // k-step i + PF, or with the first ones of the next parity
          const unsigned char *cur = bw + p * T * 512, *next = p ? bn : cur + T * 512;
          auto fb = [&](int i) { return b[i % PF]; };
          auto refill = [&](int i) { b[i % PF] = load_frag(i + PF < T ? cur + (i + PF) * 512 : next + i % PF * 512); };
          if constexpr (kRegs) {
            contract_parity<P, FP16, p == 0>([&](int i) { return ra[p * T + i]; }, fb,
                                             [&](int i) {
                                               refill(i);
                                               if (last) ra[p * T + i] = load_frag(an + (p * T + i) * 512);
                                             },
                                             out, ee, lastw);
          } else {
            if (kt == k0 && !warp_wait_or_abort(afull + p, un & 1, limit, abort, a.err)) return false;
            const unsigned char *sa = sF + woff + p * T * 512;
            contract_parity<P, FP16, p == 0>([&](int i) { return *reinterpret_cast<const uint4 *>(sa + i * 512); }, fb,
                                             refill, out, ee, lastw);
            if (last) {
              __syncwarp();
              if (lane == 0) mbar_arrive(aempty + p);
            }
          }
          // operand stage: (tile, parity) number c; stages of kZp parities, kZs of them in turn
          const uint32_t c = 2 * t + p, st = c / kZp, slot = st % kZs, use = st / kZs;
          if (p % kZp == 0 && use > 0 && !warp_wait_or_abort(zempty + slot, (use - 1) & 1, limit, abort, a.err)) return false;
          unsigned char *z = zl + (slot * kZp + p % kZp) * kZStage;
#pragma unroll
          for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int k = 0; k < 2; ++k)  // row = correlation * 64 + block * 32 + lane
              *reinterpret_cast<uint4 *>(z + (e >> 1) * kOperand + (e & 1) * 1024 + k * 512) =
                  make_uint4(out[e][k][0], out[e][k][1], out[e][k][2], out[e][k][3]);
          if constexpr (p == 0) {  // cos(pi f / 2) = (-1)^(f / 2): + on odd warps
            const float sg = (warp & 1) ? 1.f : -1.f;
            float *part = s_part + ((t & 1) * kContract + warp) * 128 + lane;
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
              for (int e = 0; e < 2; ++e) part[e * 64 + k * 32] = sg * ee[k][e];
          }
          if (p % kZp == kZp - 1) {
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(zfull + slot);
          }
          return true;
        };
        ok = parity(std::integral_constant<int, 0>{}) && parity(std::integral_constant<int, 1>{});
        bw = bn;
      }
    }
  } else if (warp < 12) {
    // ---------------- row maxima ----------------
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    const int q = warp & 3;
    const uint32_t lanes = static_cast<uint32_t>(q * 32) << 16;
    const int refl = (lane & 3) + 4 * (q & 1), corr = q >> 1;
    uint32_t t = 0;
    bool ok = !*abort;
    for (int64_t u = blockIdx.x; u < units && ok; u += gridDim.x) {
      const int64_t rt = u / splits;
      const int k0 = first_tile(u), k1 = min(k0 + per_unit, ref_tiles);
      const int64_t row = rt * 8 + (lane >> 2);
      const int64_t img = static_cast<uint32_t>(row) / static_cast<uint32_t>(g.S);  // rows < 2^31
      const int64_t rb = img * a.K * g.S + (row - img * g.S);
      for (int kt = k0; kt < k1; ++kt, ++t) {
        const uint32_t buf = t & 1, ph = (t >> 1) & 1;
        if (!warp_wait_or_abort(x0full + buf, ph, limit, abort, a.err) ||
            !warp_wait_or_abort(dfull + buf, ph, limit, abort, a.err)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const float x0 = s_x0[buf * 64 + (q & 1) * 32 + lane], e64 = s_e[buf * 128 + q * 32 + lane];
        const int ref = kt * 8 + refl;
        const bool valid = row < a.rows && ref < a.K;
        const int64_t at = rb + static_cast<int64_t>(ref) * g.S;
        if (a.dbg_cc)
          hybrid_debug_row(tmem + lanes + buf * 256, corr, x0, e64, valid ? a.dbg_cc + at * 512 + corr * 256 : nullptr);
        float best = -INFINITY;
        // 8 angles of each sum at a time; the loop is kept short (the roles
        // run different code at the same time and share the instruction
        // cache: unrolled over all 64 angles the kernel took 39.2 instead of
        // 29.6 ms per 12,000 images of the 76-pixel, 100-reference workload)
#pragma unroll 1
        for (int j0 = 0; j0 < 64; j0 += 8) {
          uint32_t ee[8], eo[8], oe[8], oo[8];
          const uint32_t d = tmem + lanes + buf * 256 + j0;
          tmem_ld8(d, ee);
          tmem_ld8(d + 64, eo);
          tmem_ld8(d + 128, oe);
          tmem_ld8(d + 192, oo);
          tmem_ld_wait();
          if (j0 == 56) {  // the accumulators are free as soon as they are in registers
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(dempty + buf);
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float E = __uint_as_float(ee[j]), F = __uint_as_float(eo[j]);
            const float G = __uint_as_float(oe[j]), H = __uint_as_float(oo[j]);
            float v = (E + F) + fabsf(G + H), w = (E - F) + fabsf(G - H);
            if (j == 0 && j0 == 0) {  // angles 0, 128; H is Oo at angle 64
              v = E + fabsf(F);
              w = e64 + fabsf(H);
            }
            best = fmaxf(best, fmaxf(v, w));
          }
        }
        if (valid) a.rowmax[at * 2 + corr] = corr && !g.mirror ? -INFINITY : best + x0;
      }
    }
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 48;");
    if (warp == 12) {
      // ---------------- inverse DFT: MMA issue ----------------
      if (lane == 0 && !*abort) {
        const uint32_t idesc = umma_idesc(128, 64, true);
        const uint32_t zb = smem_u32(sZ), wb = smem_u32(sW);
        uint32_t t = 0;
        bool ok = true;
        for (int64_t u = blockIdx.x; u < units && ok; u += gridDim.x) {
          const int k0 = first_tile(u), k1 = min(k0 + per_unit, ref_tiles);
          for (int kt = k0; kt < k1 && ok; ++kt, ++t) {
            const uint32_t buf = t & 1, dcol = tmem + buf * 256;
            if (t >= 2 && !spin_or_abort(dempty + buf, ((t >> 1) - 1) & 1, limit, abort, a.err)) {
              ok = false;
              break;
            }
#pragma unroll 1
            for (int p = 0; p < 2; ++p) {
              const uint32_t c = 2 * t + p, st = c / kZp, slot = st % kZs;
              if (p % kZp == 0 &&
                  !spin_or_abort(zfull + slot, (st / kZs) & 1, c ? limit : a.first_wait_limit, abort, a.err)) {
                ok = false;
                break;
              }
              tc_fence_after();
              // core columns of 8 frequencies: 2048 bytes apart in an operand, 1024 in a matrix
              const uint64_t zr = umma_sdesc(zb + (slot * kZp + p % kZp) * kZStage, 2048, 128), zi = zr + (kOperand >> 4);
              const uint64_t w0 = umma_sdesc(wb + p * 2 * kW, 1024, 128), w1 = w0 + (kW >> 4);
#pragma unroll
              for (int ks = 0; ks < 4; ++ks) {
                umma_ss(dcol + p * 64, zr + ks * 256, w0 + ks * 128, idesc, ks > 0);        // Ee | Eo
                umma_ss(dcol + 128 + p * 64, zi + ks * 256, w1 + ks * 128, idesc, ks > 0);  // Oe | Oo
              }
              if (p % kZp == kZp - 1) umma_commit(zempty + slot);
            }
            if (ok) umma_commit(dfull + buf);
          }
        }
        // every MMA issued has completed before the TMEM and the operands are released
        umma_commit(fin);
        mbar_wait_bounded(fin, 0, limit);
      }
    } else if (warp == 13) {
      // ---------------- zero frequency: k-steps 0..n0-1 ----------------
      uint32_t t = 0, un = 0;
      bool ok = !*abort;
      for (int64_t u = blockIdx.x; u < units && ok; u += gridDim.x, ++un) {
        const int k0 = first_tile(u), k1 = min(k0 + per_unit, ref_tiles);
        const unsigned char *aw = gA + static_cast<size_t>(u / splits) * kTile16 + lane * 16;
        uint4 af[kHyb256N0];
        if constexpr (kRegs) {
#pragma unroll
          for (int j = 0; j < kHyb256N0; ++j) af[j] = load_frag(aw + j * 512);
        }
        for (int kt = k0; kt < k1; ++kt, ++t) {
          const uint32_t buf = t & 1;
          const unsigned char *bp = gB + static_cast<size_t>(kt) * kTile16 + lane * 16;
          uint4 b[kHyb256N0];
#pragma unroll
          for (int j = 0; j < kHyb256N0; ++j) b[j] = load_frag(bp + j * 512);
          if (!kRegs && kt == k0) {
            if (!warp_wait_or_abort(afull, un & 1, limit, abort, a.err)) {
              ok = false;
              break;
            }
#pragma unroll
            for (int j = 0; j < kHyb256N0; ++j) af[j] = *reinterpret_cast<const uint4 *>(sF + j * 512 + lane * 16);
            __syncwarp();
            if (lane == 0) mbar_arrive(aempty);
          }
          if (t >= 2 && !warp_wait_or_abort(dempty + buf, ((t >> 1) - 1) & 1, limit, abort, a.err)) {
            ok = false;
            break;
          }
          float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int j = 0; j < kHyb256N0; ++j) {
            mma_frag<FP16>(d0, af[j], b[j].x, b[j].y);
            mma_frag<FP16>(d1, af[j], b[j].z, b[j].w);
          }
          s_x0[buf * 64 + lane] = d0[0];
          s_x0[buf * 64 + 32 + lane] = d1[0];
          // the parts of Ee(64): written with the even operands of the stage(s) of this tile
#pragma unroll
          for (int p = 0; p < 2 && ok; p += kZp) {
            const uint32_t st = (2 * t + p) / kZp, slot = st % kZs;
            ok = warp_wait_or_abort(zfull + slot, (st / kZs) & 1, limit, abort, a.err);
            if (ok && p == 0) {
              const float *part = s_part + buf * kContract * 128 + lane;
#pragma unroll
              for (int r = 0; r < 4; ++r) {
                float e = 0.f;
#pragma unroll
                for (int w = 0; w < kContract; ++w) e += part[w * 128 + r * 32];
                s_e[buf * 128 + r * 32 + lane] = e;
              }
            }
            __syncwarp();
            if (lane == 0) {
              mbar_arrive(zempty + slot);
              if (p == 0) mbar_arrive(x0full + buf);
            }
          }
          if (!ok) break;
        }
      }
    } else if (warp == 14 && !kRegs) {
      // ---------------- row fragments to shared memory ----------------
      // lane w < 8: warp w's even or odd k-steps; lane 8: f = 0 (even)
      uint32_t un = 0;
      int issued[2] = {0, 0};
      bool ok = !*abort;
      for (int64_t u = blockIdx.x; u < units && ok; u += gridDim.x, ++un) {
        const unsigned char *src = gA + static_cast<size_t>(u / splits) * kTile16;
        for (int p = 0; p < 2 && ok; ++p) {
          if (un > 0 && !warp_wait_or_abort(aempty + p, (un - 1) & 1, limit, abort, a.err)) {
            ok = false;
            break;
          }
          if (lane == 0) mbar_arrive_expect_tx(afull + p, (kContract * T + (p ? 0 : kHyb256N0)) * 512u);
          __syncwarp();
          fence_proxy_async();  // earlier reads of these fragments are done (aempty)
          const uint32_t off = lane < kContract ? (kHyb256N0 + (2 * lane + p) * T) * 512u : 0u;
          if (lane < kContract || (lane == kContract && !p))
            bulk_g2s(sF + off, src + off, (lane < kContract ? T : kHyb256N0) * 512u, afull + p);
          ++issued[p];
        }
      }
      // every copy issued lands before the CTA's shared memory goes
      for (int p = 0; p < 2; ++p)
        if (issued[p]) mbar_wait_bounded(afull + p, (issued[p] - 1) & 1, limit);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 12) tmem_dealloc(tmem, 512);
}

// Units of work are (row tile, range of reference tiles): `splits` ranges
// per row tile, chosen to minimise the time of the fullest SM,
// waves x (tiles per unit + the unit's load of its row fragments, about one
// tile).  One range when the row tiles fill many waves (each row tile's
// fragments are then loaded once); more when the stack is so small that
// whole row tiles would leave SMs idle.
static int pick_splits(int64_t row_tiles, int ref_tiles, int sms) {
  int best = 1;
  int64_t best_cost = INT64_MAX;
  for (int s = 1; s <= ref_tiles; ++s) {
    const int per = (ref_tiles + s - 1) / s;
    if ((ref_tiles + per - 1) / per != s) continue;  // ranges must not be empty
    const int64_t cost = (row_tiles * s + sms - 1) / sms * (per + 1);
    if (cost < best_cost) {
      best_cost = cost;
      best = s;
    }
  }
  return best;
}

template <int PATTERN, bool FP16>
static cudaError_t launch_hybrid_t(const Geometry &g, const TcArgs &a, cudaStream_t st) {
  static SmemLimit granted;
  constexpr size_t smem = u256::z_stages(PATTERN) * u256::z_parities(PATTERN) * u256::kZStage + u256::kMisc +
                          (PATTERN == 0 ? 0 : HybPattern<PATTERN>::KS * 512);
  static_assert(smem <= kMaxSmemPerBlock, "row fragments must fit");
  if (g.KS != HybPattern<PATTERN>::KS) return cudaErrorInvalidValue;
  cudaError_t e = raise_smem_limit(cc_hybrid256_kernel<PATTERN, FP16>, smem, granted);
  if (e != cudaSuccess) return e;
  int sms = 0;
  e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  const int64_t row_tiles = (a.rows + kTile - 1) / kTile;
  const int ref_tiles = (a.K + kTile - 1) / kTile;
  if (row_tiles <= 0) return cudaSuccess;
  const int splits = pick_splits(row_tiles, ref_tiles, sms);
  const int per = (ref_tiles + splits - 1) / splits;
  const int64_t units = row_tiles * splits;
  const int grid = static_cast<int>(units < sms ? units : sms);
  cc_hybrid256_kernel<PATTERN, FP16><<<grid, u256::kThreads, smem, st>>>(g, a, ref_tiles, per, splits, units);
  return cudaGetLastError();
}

cudaError_t launch_cc_hybrid256(const Geometry &g, const TcArgs &a, bool fp16, cudaStream_t st) {
  if (g.M != 256 || !g.hyb_w) return cudaErrorInvalidValue;
  if (g.hyb_pattern == 0) return fp16 ? launch_hybrid_t<0, true>(g, a, st) : launch_hybrid_t<0, false>(g, a, st);
  return fp16 ? launch_hybrid_t<1, true>(g, a, st) : launch_hybrid_t<1, false>(g, a, st);
}

}  // namespace mra
