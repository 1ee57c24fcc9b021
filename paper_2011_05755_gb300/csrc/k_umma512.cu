// Precision-split path, M = 512 angles (rings up to 81): spectrum
// contraction on warp-level tensor cores (mma.sync), inverse angular DFT on
// tcgen05.mma with the angular sums accumulated in TMEM.
//
// The sums are those of the M = 256 kernel (k_umma256.cu) at twice the length:
// for angles j = 0..127
//     Ee, Eo = sum over even / odd f of   2 Re C(f) cos(2 pi f j / 512),
//     Oe, Oo = sum over even / odd f of - 2 Im C(f) sin(2 pi f j / 512),
//     c(j), c(512 - j) = (Ee + Eo) +- (Oe + Oo),
//     c(256 + j), c(256 - j) = (Ee - Eo) +- (Oe - Oo),
// as products D[128 x 128] = A[128 x 128] W[128 x 128] over 64 pairs x {C, C'}
// rows; the four fill the 512 TMEM columns.  For odd f
//     sin(2 pi f j / 512) = s_f cos(2 pi f (128 - j) / 512),  s_f = sin(pi f / 2) = +-1,
// so Oo uses the matrix of Eo on sign-flipped data and its column k is the
// angle 128 - k (three matrices, 96 KB, instead of four; column 0 is Oo(128),
// which angles 128 and 384 need).  Their other half, Ee(128), is an
// alternating sum of the even 2 Re C: each contraction warp adds its own
// frequencies in FP32 and the f = 0 warp adds the warps.
//
// What bounds it.  A tile is 8 rows x 8 references (the FP32 sums of 64 pairs
// fill TMEM), neither operand of its KS k-steps (708 at rings 1..60) fits on
// an SM beside the matrices, and a tile streams both from L2: KS x 1 KB, 18,000
// cycles at the ~40 bytes per cycle and SM that L2 delivers to all SMs at once.
// Everything else (contraction, MMAs, reading the sums) runs under that stream.
// The kernel it replaced kept the pair spectra in shared memory, staged whole
// chunks of frequencies behind CTA barriers and took 38,000 cycles a tile.
//
// Roles (24 warps, one persistent CTA per SM):
//   warps 0-15   contract: warp w holds 8 frequencies (slots) of each parity,
//                its k-steps side by side in both fragment layouts (even
//                slots, then odd), streamed by per-lane asynchronous copies
//                through a ring of kRing k-steps in shared memory (a lane
//                reads back only what it copied: no barrier), and writes core
//                column w of the parity's two operands;
//   warps 16-19  read the sums of their TMEM lane quarter, write row maxima;
//   warp 20      issues every tcgen05.mma (one lane);
//   warp 21      contracts f = 0 and adds up Ee(128).
// All waits are bounded; a wait that gives up raises a CTA abort flag and the
// device error flag, every role leaves its loop, the copies and MMAs in
// flight are waited for, and the TMEM is released.
#include "../../include/mra.h"
#include "dev_util.cuh"
#include "hybrid.cuh"
#include "mra_internal.h"
#include "smem_limit.cuh"
#include "umma.cuh"

namespace mra {

namespace u512 {
constexpr int kContract = 16;
constexpr int kThreads = 32 * (kContract + 8);
constexpr int kRing = 3;                          // k-steps in flight per warp
constexpr uint32_t kOperand = 128 * 128 * 2;      // one operand of a parity: 128 rows x 128 frequencies
constexpr uint32_t kStage = 2 * kOperand;         // real and imaginary parts
constexpr uint32_t kW = 128 * 128 * 2;
constexpr uint32_t kWBytes = kHyb512Mats * kW;    // Ee, Oe, Eo
constexpr uint32_t kRingBytes = kContract * kRing * 1024;
constexpr int kNumBars = 12;  // zfull zfree efull pfree dfull dempty[2] x0full[2] fin, spare
constexpr uint32_t kSmem = kWBytes + kStage + kRingBytes + kContract * 128 * 4 + 2 * (64 + 128) * 4 + kNumBars * 8 + 16;
static_assert(kSmem <= kMaxSmemPerBlock, "M = 512 kernel exceeds 227 KB of shared memory");
}  // namespace u512

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Every angle of the 32 rows of a warp's TMEM lane quarter into the debug table (dst null: no store).
__device__ __noinline__ void hybrid512_debug_row(uint32_t d, int corr, float x0, float e128, float *dst) {
#pragma unroll 1
  for (int n = 0; n <= 128; ++n) {
    uint32_t r[4];
    tmem_ld1(d + (n < 128 ? n : 0), r[0]);
    tmem_ld1(d + 128 + (n < 128 ? n : 0), r[1]);
    tmem_ld1(d + 256 + (n < 128 ? n : 0), r[2]);
    tmem_ld1(d + 384 + (n ? 128 - n : 0), r[3]);
    tmem_ld_wait();
    const float E = n < 128 ? __uint_as_float(r[0]) : e128, F = n < 128 ? __uint_as_float(r[1]) : 0.f;
    const float G = n < 128 ? __uint_as_float(r[2]) : 0.f, H = n ? __uint_as_float(r[3]) : 0.f;
    const float c[4] = {(E + F) + (G + H), (E + F) - (G + H), (E - F) + (G - H), (E - F) - (G - H)};
    const int at[4] = {n, 512 - n, 256 + n, 256 - n};
    if (dst)  // mirrored row: angle n of the transform is angle n + 256 of the table
      for (int i = 0; i < (n < 128 ? 4 : 2); ++i) dst[(at[i] + corr * 256) & 511] = c[i] + x0;
  }
}

template <bool FP16>
__global__ void __launch_bounds__(u512::kThreads, 1)
    cc_hybrid512_kernel(Geometry g, TcArgs a, int ref_tiles, int per_unit, int splits, int64_t units) {
  using namespace u512;
  extern __shared__ __align__(1024) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned char *sW = smem, *sZ = sW + kWBytes, *sR = sZ + kStage;
  float *s_part = reinterpret_cast<float *>(sR + kRingBytes);  // [16 warps][128 rows] parts of Ee(128)
  float *s_x0 = s_part + kContract * 128;                      // [2][64] zero-frequency terms
  float *s_e = s_x0 + 2 * 64;                                  // [2][128] Ee(128)
  uint64_t *bars = reinterpret_cast<uint64_t *>(s_e + 2 * 128);
  uint64_t *zfull = bars, *zfree = bars + 1, *efull = bars + 2, *pfree = bars + 3, *dfull = bars + 4, *dempty = bars + 5,
           *x0full = bars + 7, *fin = bars + 9;
  uint32_t *s_tmem = reinterpret_cast<uint32_t *>(bars + kNumBars);
  volatile int *abort = reinterpret_cast<volatile int *>(s_tmem + 1);

  // ---- set-up: DFT matrices, barriers, TMEM ----
  for (int i = tid; i < static_cast<int>(kWBytes / 16); i += kThreads)
    reinterpret_cast<uint4 *>(sW)[i] = __ldg(reinterpret_cast<const uint4 *>(g.hyb_w) + i);
  if (tid == 0) {
    mbar_init(zfull, kContract);
    mbar_init(zfree, 1);
    mbar_init(efull, kContract);
    mbar_init(pfree, 1);
    mbar_init(dfull, 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(dempty + s, 4);
      mbar_init(x0full + s, 1);
    }
    mbar_init(fin, 1);
    *abort = (smem_u32(smem) & 127u) ? 1 : 0;  // descriptors assume an aligned base
    if (*abort) atomicOr(a.err, 2);
  }
  if (warp == 20) tmem_alloc(s_tmem, 512);
  mbar_init_fence();
  fence_proxy_async();  // the DFT matrices written above are read by the tensor cores
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *s_tmem;
  const unsigned char *gA = reinterpret_cast<const unsigned char *>(a.A16);
  const unsigned char *gB = reinterpret_cast<const unsigned char *>(a.B16);
  const size_t tile_bytes = static_cast<size_t>(g.KS) * 512;
  const uint32_t limit = a.wait_limit;
  auto first_tile = [&](int64_t u) { return static_cast<int>(u % splits) * per_unit; };

  // registers per thread: 80 at launch (4 x 88 + 2 x 64 = 6 x 80)
  if (warp < kContract) {
    // ---------------- contraction ----------------
    asm volatile("setmaxnreg.inc.sync.aligned.u32 88;");
    // this warp's first k-step, its k-steps per tile, and 4 bits of k-steps per slot
    const int4 sched = __ldg(g.hyb_sched + warp);
    const size_t woff = static_cast<size_t>(sched.x) * 512 + lane * 16;
    const uint32_t ring = smem_u32(sR) + warp * kRing * 1024 + lane * 16;
    unsigned char *zl = sZ + warp * 2048 + lane * 16;
    // the copies run kRing k-steps ahead of the use: their own unit, tile and k-step
    int64_t cu = blockIdx.x;
    int ckt = first_tile(cu), left = sched.y;
    const unsigned char *pa = gA + static_cast<size_t>(cu / splits) * tile_bytes + woff;
    const unsigned char *pb = gB + static_cast<size_t>(ckt) * tile_bytes + woff;
    uint32_t put = 0, get = 0;  // ring slots, in bytes
    auto copy = [&]() {
      if (cu < units) {
        cp_async16(ring + put, pa);
        cp_async16(ring + put + 512, pb);
        pa += 512;
        pb += 512;
        if (--left == 0) {
          left = sched.y;
          if (++ckt == min(first_tile(cu) + per_unit, ref_tiles)) {
            cu += gridDim.x;
            ckt = first_tile(cu);
          }
          pa = gA + static_cast<size_t>(cu / splits) * tile_bytes + woff;
          pb = gB + static_cast<size_t>(ckt) * tile_bytes + woff;
        }
      }
      cp_async_commit();  // a group per k-step, empty past the end
      put = put == (kRing - 1) * 1024 ? 0 : put + 1024;
    };
    for (int i = 0; i < kRing; ++i) copy();
    uint32_t t = 0;
    bool ok = !*abort;
    for (int64_t u = blockIdx.x; u < units && ok; u += gridDim.x) {
      const int k0 = first_tile(u), k1 = min(k0 + per_unit, ref_tiles);
      for (int kt = k0; kt < k1 && ok; ++kt, ++t) {
#pragma unroll 1
        for (int p = 0; p < 2; ++p) {
          const uint32_t counts = p ? static_cast<uint32_t>(sched.w) : static_cast<uint32_t>(sched.z);
          uint32_t out[4][2][4];
          float keep[2][4], ee[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
          sfor<0, 8>([&](auto ss) {
            constexpr int s = decltype(ss)::value;
            float d[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll 1
            for (uint32_t n = (counts >> (4 * s)) & 15u; n > 0; --n) {
              cp_async_wait<kRing - 1>();
              uint4 af, bf;
              asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                           : "=r"(af.x), "=r"(af.y), "=r"(af.z), "=r"(af.w) : "r"(ring + get) : "memory");
              asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                           : "=r"(bf.x), "=r"(bf.y), "=r"(bf.z), "=r"(bf.w) : "r"(ring + get + 512) : "memory");
              get = get == (kRing - 1) * 1024 ? 0 : get + 1024;
              mma_frag<FP16>(d[0], af, bf.x, bf.y);
              mma_frag<FP16>(d[1], af, bf.z, bf.w);
              copy();
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              float v[4];
              pair_sums(d[k], v);
              // even f = 2 (16 s + warp) + 2; the last, f = 256, is its own mirror image
              const float half = s == 7 && warp == 15 ? 0.5f : 1.f;
              ee[k][0] = fmaf(v[0], half, ee[k][0]);
              ee[k][1] = fmaf(v[1], half, ee[k][1]);
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                if constexpr (s & 1)
                  out[e][k][s >> 1] = pack_bf2u(keep[k][e], v[e]);
                else
                  keep[k][e] = v[e];
              }
            }
          });
          if (p && !(warp & 1)) {  // odd f = 2 (16 s + warp) + 1: s_f = +1 on even warps, the data is - s_f 2 Im C
#pragma unroll
            for (int i = 0; i < 16; ++i) out[2 + (i >> 3)][(i >> 2) & 1][i & 3] ^= 0x80008000u;
          }
          const uint32_t c = 2 * t + p;  // uses of the operand stage
          if ((c > 0 && !warp_wait_or_abort(zfree, (c - 1) & 1, limit, abort, a.err)) ||
              (!p && t > 0 && !warp_wait_or_abort(pfree, (t - 1) & 1, limit, abort, a.err))) {
            ok = false;
            break;
          }
#pragma unroll
          for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int k = 0; k < 2; ++k)  // row = correlation * 64 + block * 32 + lane
              *reinterpret_cast<uint4 *>(zl + (e >> 1) * kOperand + (e & 1) * 1024 + k * 512) =
                  make_uint4(out[e][k][0], out[e][k][1], out[e][k][2], out[e][k][3]);
          if (!p) {  // cos(pi f / 2) = (-1)^(f / 2): + on odd warps
            const float sg = (warp & 1) ? 1.f : -1.f;
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
              for (int e = 0; e < 2; ++e) s_part[warp * 128 + e * 64 + k * 32 + lane] = sg * ee[k][e];
          }
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(zfull);
            if (!p) mbar_arrive(efull);
          }
        }
      }
    }
    cp_async_wait<0>();
  } else if (warp < kContract + 4) {
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
        const uint32_t buf = t & 1;
        if (!warp_wait_or_abort(x0full + buf, (t >> 1) & 1, limit, abort, a.err) ||
            !warp_wait_or_abort(dfull, t & 1, limit, abort, a.err)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const float x0 = s_x0[buf * 64 + (q & 1) * 32 + lane], e128 = s_e[buf * 128 + q * 32 + lane];
        const int ref = kt * 8 + refl;
        const bool valid = row < a.rows && ref < a.K;
        const int64_t at = rb + static_cast<int64_t>(ref) * g.S;
        if (a.dbg_cc)
          hybrid512_debug_row(tmem + lanes, corr, x0, e128, valid ? a.dbg_cc + at * 1024 + corr * 512 : nullptr);
        float best = -INFINITY, carry = 0.f;  // carry: Oo at angle j0 (0 at angle 0)
#pragma unroll 1
        for (int j0 = 0; j0 < 128; j0 += 8) {
          uint32_t ee[8], eo[8], oe[8], oo[8];
          const uint32_t d = tmem + lanes + j0;
          tmem_ld8(d, ee);
          tmem_ld8(d + 128, eo);
          tmem_ld8(d + 256, oe);
          tmem_ld8(tmem + lanes + 384 + 120 - j0, oo);  // angles j0 + 8 down to j0 + 1
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float E = __uint_as_float(ee[j]), F = __uint_as_float(eo[j]);
            const float G = __uint_as_float(oe[j]), H = j ? __uint_as_float(oo[8 - j]) : carry;
            best = fmaxf(best, fmaxf((E + F) + fabsf(G + H), (E - F) + fabsf(G - H)));
          }
          carry = __uint_as_float(oo[0]);
        }
        best = fmaxf(best, e128 + fabsf(carry));  // angles 128 and 384
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(dempty + buf);
        if (valid) a.rowmax[at * 2 + corr] = corr && !g.mirror ? -INFINITY : best + x0;
      }
    }
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    if (warp == 20) {
      // ---------------- inverse DFT: MMA issue ----------------
      if (lane == 0 && !*abort) {
        const uint32_t idesc = umma_idesc(128, 128, true);
        const uint32_t zb = smem_u32(sZ), wb = smem_u32(sW);
        uint32_t t = 0;
        bool ok = true;
        for (int64_t u = blockIdx.x; u < units && ok; u += gridDim.x) {
          const int k0 = first_tile(u), k1 = min(k0 + per_unit, ref_tiles);
          for (int kt = k0; kt < k1 && ok; ++kt, ++t) {
#pragma unroll 1
            for (int p = 0; p < 2; ++p) {
              const uint32_t c = 2 * t + p;
              if (!spin_or_abort(zfull, c & 1, c ? limit : a.first_wait_limit, abort, a.err) ||
                  (!p && t > 0 && !spin_or_abort(dempty + ((t - 1) & 1), ((t - 1) >> 1) & 1, limit, abort, a.err))) {
                ok = false;
                break;
              }
              tc_fence_after();
              // core columns of 8 frequencies are 2048 bytes apart in an operand and in a matrix
              const uint64_t zr = umma_sdesc(zb, 2048, 128), zi = zr + (kOperand >> 4);
              const uint64_t wr = umma_sdesc(wb + (p ? 2 * kW : 0), 2048, 128);
              const uint64_t wi = umma_sdesc(wb + (p ? 2 * kW : kW), 2048, 128);
#pragma unroll
              for (int ks = 0; ks < 8; ++ks) {
                umma_ss(tmem + p * 128, zr + ks * 256, wr + ks * 256, idesc, ks > 0);        // Ee | Eo
                umma_ss(tmem + 256 + p * 128, zi + ks * 256, wi + ks * 256, idesc, ks > 0);  // Oe | Oo
              }
              umma_commit(zfree);
            }
            if (ok) umma_commit(dfull);
          }
        }
        // every MMA issued has completed before the TMEM and the operands are released
        umma_commit(fin);
        mbar_wait_bounded(fin, 0, limit);
      }
    } else if (warp == 21) {
      // ---------------- zero frequency (k-steps 0..n0-1) and Ee(128) ----------------
      const int n0 = (g.NR + 15) / 16;  // every ring has f = 0
      uint32_t t = 0;
      bool ok = !*abort;
      for (int64_t u = blockIdx.x; u < units && ok; u += gridDim.x) {
        const int k0 = first_tile(u), k1 = min(k0 + per_unit, ref_tiles);
        const unsigned char *ap = gA + static_cast<size_t>(u / splits) * tile_bytes + lane * 16;
        for (int kt = k0; kt < k1; ++kt, ++t) {
          const uint32_t buf = t & 1;
          const unsigned char *bp = gB + static_cast<size_t>(kt) * tile_bytes + lane * 16;
          float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
          for (int j = 0; j < n0; ++j) {
            const uint4 af = load_frag(ap + j * 512), bf = load_frag(bp + j * 512);
            mma_frag<FP16>(d0, af, bf.x, bf.y);
            mma_frag<FP16>(d1, af, bf.z, bf.w);
          }
          if ((t >= 2 && !warp_wait_or_abort(dempty + buf, ((t >> 1) - 1) & 1, limit, abort, a.err)) ||
              !warp_wait_or_abort(efull, t & 1, limit, abort, a.err)) {
            ok = false;
            break;
          }
          s_x0[buf * 64 + lane] = d0[0];
          s_x0[buf * 64 + 32 + lane] = d1[0];
#pragma unroll 1
          for (int r = lane; r < 128; r += 32) {
            float e = 0.f;
#pragma unroll
            for (int w = 0; w < kContract; ++w) e += s_part[w * 128 + r];
            s_e[buf * 128 + r] = e;
          }
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(pfree);
            mbar_arrive(x0full + buf);
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 20) tmem_dealloc(tmem, 512);
}

template <bool FP16>
static cudaError_t launch_hybrid512_t(const Geometry &g, const TcArgs &a, cudaStream_t st) {
  static size_t granted = 0;
  cudaError_t e = raise_smem_limit(cc_hybrid512_kernel<FP16>, u512::kSmem, granted);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int64_t row_tiles = (a.rows + kTile - 1) / kTile;
  const int ref_tiles = (a.K + kTile - 1) / kTile;
  if (row_tiles <= 0) return cudaSuccess;
  const int splits = pick_splits(row_tiles, ref_tiles, sms);
  const int per = (ref_tiles + splits - 1) / splits;
  const int64_t units = row_tiles * splits;
  const int grid = static_cast<int>(units < sms ? units : sms);
  cc_hybrid512_kernel<FP16><<<grid, u512::kThreads, u512::kSmem, st>>>(g, a, ref_tiles, per, splits, units);
  return cudaGetLastError();
}

cudaError_t launch_cc_hybrid512(const Geometry &g, const TcArgs &a, bool fp16, cudaStream_t st) {
  if (g.M != 512 || !g.hyb_w || !g.hyb_sched) return cudaErrorInvalidValue;
  return fp16 ? launch_hybrid512_t<true>(g, a, st) : launch_hybrid512_t<false>(g, a, st);
}

}  // namespace mra
