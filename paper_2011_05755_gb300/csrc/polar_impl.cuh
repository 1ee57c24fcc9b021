// Polar resampling and ring FFT (Alg. 1, shift-loop conversion step: each
// particle is resampled on the rings about its shifted centre and every ring
// is Fourier transformed; the references get the same with no shift,
// followed by the ring weights of the Sec. 2 quadrature).
//
// A CTA stages one image in shared memory and walks groups of R consecutive
// rows (row = image * rows_per_img + shift): the groups blockIdx.x,
// blockIdx.x + gridDim.x, ...  Per group, phase 1 writes the bilinear
// samples of its rows into shared memory; phase 2
// gives each warp one (row, ring) job: an in-place N/2-point complex FFT of
// the ring's real samples packed as z_q = x_{2q} + i x_{2q+1}, then the
// split into the N/2 + 1 real-input bins X(f), written straight into the
// frequency-major tiled layout [row / 8][bin][row % 8] (FP32 path), or, for
// the 16-bit tensor-core paths, into the mma.sync A-fragment order: per tile
// of 8 rows and k-step of 16 rings of one frequency, lane 4g + t of a warp
// holds {q[g][2t..2t+1], p[g][2t..2t+1], q[g][2t+8..9], p[g][2t+8..9]} with
// q = Re X - Im X and p = Re X + Im X (rows 0-7 of the MMA are the q values of
// the 8 tile rows, rows 8-15 their p values).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "dev_util.cuh"
#include "mra_internal.h"
#include "ring_fft.cuh"
#include "smem_limit.cuh"
#include "tma.cuh"

namespace mra {

// Row stride of the sample buffer (NSb floats a row): 16 floats off a
// multiple of 32, so the ring-FFT jobs of consecutive rows start in opposite
// halves of the shared-memory banks.
__host__ __device__ inline int sample_stride(int NSb) { return NSb + ((16 - NSb) & 31); }

// Output layouts of the polar kernel: FP32 frequency-major tiles, or the
// 16-bit q / p planes (BF16 or FP16) that phase 3 turns into mma.sync
// fragments.
enum PolarOut { kOutF32 = 0, kOut16 = 1 };

// (q, p) of one bin packed as a 16-bit pair word: q low, p high.
__device__ __forceinline__ uint32_t pack_qp(float q, float p, bool fp16) {
  if (fp16) {
    const __half2 h = __floats2half2_rn(q, p);  // .x (low half) = q
    return *reinterpret_cast<const uint32_t *>(&h);
  }
  const __nv_bfloat162 h = __floats2bfloat162_rn(q, p);
  return *reinterpret_cast<const uint32_t *>(&h);
}

// Position of word w (k-step w / 16, word w % 16) in a row of the (q, p)
// planes: the word index inside the k-step is XORed with (k-step & 14), so
// that the stores of one ring's consecutive frequencies (k-steps 1, 2 or 3
// apart, same word) fall in different banks.  The XOR keeps word pairs
// (2j, 2j + 1) adjacent.
__device__ __forceinline__ int plane_swz(int w) { return w ^ ((w >> 4) & 14); }

// One bin of a particle or reference row into the path's output layout
// (weights for references, the debug copy, FP32 tiles or 16-bit words).
template <int OUT>
__device__ __forceinline__ void put_bin(const Geometry &g, const PolarArgs &a, uint32_t *planes_row, const int *s_kpos,
                                        int ring, int bin0, int64_t row, int k, float2 X) {
  if (OUT == kOutF32 && a.weighted) {  // references and debug copies take the FP32 output
    const float w = g.bweight[bin0 + k];
    X.x *= w;
    X.y *= w;
  }
  if (OUT == kOutF32 && a.dbg_spec) a.dbg_spec[row * g.NBIN + bin0 + k] = X;
  if constexpr (OUT == kOutF32) {
    if (a.out) a.out[((row >> 3) * g.NB + s_kpos[k] + ring) * kTile + (row & 7)] = X;
  } else {
    const int w = s_kpos[k] + ring;  // k-step w / 16, word w % 16 of it
    planes_row[plane_swz(w)] = pack_qp(X.x - X.y, X.x + X.y, a.fp16);
  }
}

// All (ring, row) jobs of one ring-length class c of a CTA: forward
// FFT of the packed samples, real split, weights, and the spectrum written in
// the layout the path needs (FP32 tiled, 16-bit q/p words, debug).  s_kpos
// holds the per-frequency base of the output layout: bin (ring, k) goes to
// s_kpos[k] + ring.
template <int H, int R, int OUT, int NWARPS>
__device__ __forceinline__ int ring_class(const Geometry &g, const PolarArgs &a, float *smem, uint32_t *planes,
                                          int NB16, const float2 *tws, const int *s_kpos, const RingClass &c, int nrows,
                                          int64_t row0, int warp, int lane, int first_warp) {
  constexpr int T = GroupFft<H>::T;
  constexpr int JPW = 32 / T;  // jobs per warp pass
  const int njobs = (c.i1 - c.i0) * nrows;
  const int t = lane % T;
  // warp passes of this class start after the previous class's last pass
  const int wslot = (warp - first_warp) & (NWARPS - 1);
  for (int j0 = wslot * JPW; j0 < njobs; j0 += NWARPS * JPW) {
    const int job = j0 + lane / T;
    const bool active = job < njobs;
    const int jc = active ? job : j0;
    // (ring, row) of the job; nrows is R except in an image's last group
    const int rc = nrows == R ? jc / R : jc / nrows, ring = c.i0 + rc;
    const int i = nrows == R ? jc % R : jc % nrows;
    const int bin0 = c.bin + rc * (H + 1);
    float2 *z = reinterpret_cast<float2 *>(smem + i * sample_stride(g.NSb) + c.off + rc * c.stride);
    group_fft<H>(z, t, active, tws, g.M);
    if (active) {
      const int wstep = g.M / (2 * H);
      const int64_t row = row0 + i;
      uint32_t *prow = planes + i * NB16;
      // bins k and H - k from one pair of loads and one twiddle
      for (int k = t; 2 * k <= H; k += T) {
        float2 xk, xhk;
        real_split_pair(z, H, k, tws[k * wstep], xk, xhk);
        put_bin<OUT>(g, a, prow, s_kpos, ring, bin0, row, k, xk);
        if (2 * k != H) put_bin<OUT>(g, a, prow, s_kpos, ring, bin0, row, H - k, xhk);
      }
    }
    __syncwarp();
  }
  return (first_warp + (njobs + JPW - 1) / JPW) & (NWARPS - 1);  // first warp of the next class
}

// Shared-memory image: the bare image, sampled with bounds checks
// (kPolarBare), or the image inside a zero border of g.pad pixels with rows
// of g.pitch floats, where every neighbour of every sample is in the buffer:
// integer shift grids (kPolarInt), whose bilinear weights do not depend on
// the shift, and other grids (kPolarFrac).
__host__ __device__ inline int image_floats(const Geometry &g, int mode) {
  const int n = mode == kPolarBare ? g.L * g.L : (g.L + 2 * g.pad) * g.pitch;
  return (n + 3) & ~3;
}

// Threads of a CTA: with a bordered image one CTA of 16 warps fills an SM and
// takes as many rows as fit, unless the box is small or the image has one row
// (launch_polar_t); otherwise two of 8 warps.
__host__ __device__ constexpr int polar_threads(int mode) { return mode != kPolarBare ? 512 : 256; }

// Bilinear interpolation with the fused multiply-adds written out: left to
// the compiler, instantiations with different row counts fuse differently,
// and an image's last bits would depend on the size of its call.
__device__ __forceinline__ float bilerp(float fx, float fy, float gx, float gy, float t0, float t1, float b0, float b1) {
  const float t = fmaf(gx, t0, __fmul_rn(fx, t1)), b = fmaf(gx, b0, __fmul_rn(fx, b1));
  return fmaf(gy, t, __fmul_rn(fy, b));
}

template <int R, int MODE, int OUT, int NT>
__global__ void __launch_bounds__(NT, 512 / NT) polar_fft_kernel(Geometry g, const __grid_constant__ PolarArgs a) {
  extern __shared__ float4 smem_f4[];
  const int L = g.L, NS = g.NS, M = g.M;
  const int NSp = sample_stride(g.NSb);
  const int LL = L * L;
  const int64_t img = blockIdx.y;
  float *im = reinterpret_cast<float *>(smem_f4);       // the image (with its zero border unless kPolarBare)
  uint64_t *ibar = reinterpret_cast<uint64_t *>(im + image_floats(g, MODE));  // image copy barrier (16 B)
  float2 *tws = reinterpret_cast<float2 *>(im + image_floats(g, MODE) + 4);  // [M] forward twiddles
  int *s_kpos = reinterpret_cast<int *>(tws + M);       // [M/2 + 1] output bases (padded to even)
  float *smem = reinterpret_cast<float *>(s_kpos + ((M / 2 + 2) & ~1));  // [R][NSp] samples, then ring FFTs
  const float c0 = 0.5f * static_cast<float>(L);
  // 16-bit paths: (q, p) words [row][NB16] after the samples; the padding
  // words are zeroed once, every group rewrites the same non-padding words
  const int NB16 = g.KS * 16;
  uint32_t *planes = reinterpret_cast<uint32_t *>(smem + R * NSp);
  if constexpr (OUT != kOutF32)
    for (int idx = threadIdx.x; idx < R * NB16 / 2; idx += NT)
      reinterpret_cast<uint2 *>(planes)[idx] = make_uint2(0u, 0u);
  {
    const int *kp = OUT == kOutF32 ? g.kpos : g.kpos16;
    for (int k = threadIdx.x; k <= M / 2; k += NT) s_kpos[k] = kp[k];
  }
  const float *src = a.imgs + img * LL;
  const bool vec = (L & 3) == 0 && (reinterpret_cast<uintptr_t>(src) & 15) == 0;
  // TMA staging: one tensor copy of the image (and, where it has one, its zero
  // border from the map's out-of-bounds fill), issued by thread 0 while the
  // CTA loads its tables; the destination must be 128-byte aligned
  const bool tma = a.tma && (smem_u32(im) & 127u) == 0;
  if (tma) {
    if (threadIdx.x == 0) {
      mbar_init(ibar, 1);
      mbar_init_fence();
      const int pad = MODE ? g.pad : 0;
      mbar_arrive_expect_tx(ibar, static_cast<uint32_t>(MODE ? (L + 2 * pad) * g.pitch : LL) * 4u);
      tma_load_3d(im, &a.tmap, -pad, -pad, static_cast<int>(img), ibar);
    }
  } else if constexpr (MODE != kPolarBare) {
    // zero the bordered buffer, then copy the interior (pad is a multiple of 4)
    const int Lp = g.pitch;
    for (int i = threadIdx.x; i < image_floats(g, MODE) / 4; i += NT)
      reinterpret_cast<float4 *>(im)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    float *dst = im + g.pad * Lp + g.pad;
    if (vec) {
      const int W = L / 4;
      for (int i = threadIdx.x; i < L * W; i += NT) {
        const int y = i / W, x4 = i - y * W;
        reinterpret_cast<float4 *>(dst + y * Lp)[x4] = __ldg(reinterpret_cast<const float4 *>(src + y * L) + x4);
      }
    } else {
      for (int i = threadIdx.x; i < LL; i += NT) {
        const int y = i / L, x = i - y * L;
        dst[y * Lp + x] = __ldg(src + i);
      }
    }
  } else {
    if (vec) {
      const float4 *s4 = reinterpret_cast<const float4 *>(src);
      for (int i = threadIdx.x; i < LL / 4; i += NT) reinterpret_cast<float4 *>(im)[i] = __ldg(s4 + i);
    } else {
      for (int i = threadIdx.x; i < LL; i += NT) im[i] = __ldg(src + i);
    }
  }
  for (int i = threadIdx.x; i < M; i += NT) tws[i] = g.fwd_tw[i];
  if (tma) {
    __syncthreads();  // the barrier's initialisation is visible to every thread
    const bool ok = mbar_wait_bounded(ibar, 0, a.wait_limit);
    if (__syncthreads_or(!ok)) {  // uniform: every thread leaves
      if (threadIdx.x == 0) {
        atomicOr(a.err, 1);
        mbar_wait_bounded(ibar, 0, a.wait_limit);  // the copy must land before the CTA's memory goes
      }
      return;
    }
  }
  __syncthreads();

  // Sample-table entries of the next pass over the samples, loaded while this
  // one is sampled (and those of a group's first pass during the previous
  // group's copy-out): 12,000 images of 76 px 16.77 -> 15.75 ms, 128 px 8.42 ->
  // 8.25 ms; four or six entries a thread instead of eight: 16.3 ms.
  constexpr int QU = 8;
  float4 tn[QU];
  auto load_taps = [&](int q0) {
#pragma unroll
    for (int u = 0; u < QU; ++u) {
      const int q = q0 + u * NT;
      tn[u] = q < NS ? __ldg(g.taps + q) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  if constexpr (MODE == kPolarInt) load_taps(threadIdx.x);
  for (int s0 = blockIdx.x * R; s0 < a.rows_per_img; s0 += gridDim.x * R) {
    const int nrows = min(R, a.rows_per_img - s0);
    const int64_t row0 = img * a.rows_per_img + s0;
    // Phase 1: samples x_r(theta_q) = I(c0 + s + r (cos theta_q, sin theta_q)).
    // The table lists the samples in patches of up to 5 adjacent rings x 8
    // angles, which spread the reads of a warp over the banks better than 32
    // samples along one ring (1.8 to 2.0 wavefronts per read against 2.4 to
    // 2.8, counted over the table's batches), with each sample's place in the
    // buffer (low 16 bits) and its number in ring order (high 16 bits).
    if constexpr (MODE == kPolarInt) {
      // integer shifts: the bilinear weights of a sample do not depend on the
      // shift, which only moves the neighbourhood inside the bordered image
      const int Lp = g.pitch;
      int soff[R];        // shift s = iy nx + ix is (smin + ix sstep, smin + iy sstep)
      uint32_t step = 0;  // bit i: row i's shift is row i - 1's plus one pixel along x
      {
        int iy = s0 / g.nx, ix = s0 - iy * g.nx;
#pragma unroll
        for (int i = 0; i < R; ++i) {
          soff[i] = a.use_shifts ? (g.smin + iy * g.sstep) * Lp + g.smin + ix * g.sstep : 0;
          if (i > 0 && ix > 0 && g.sstep == 1) step |= 1u << i;
          if (++ix == g.nx) {
            ix = 0;
            ++iy;
          }
        }
      }
      // QU samples per thread and pass; the next pass's table entries load meanwhile
      for (int q0 = threadIdx.x; q0 < NS; q0 += QU * NT) {
        float4 tp[QU];
#pragma unroll
        for (int u = 0; u < QU; ++u) tp[u] = tn[u];
        if (q0 + QU * NT < NS) load_taps(q0 + QU * NT);
#pragma unroll
        for (int u = 0; u < QU; ++u) {
          const int q = q0 + u * NT;
          if (q < NS) {
            const int at = __float_as_int(tp[u].w);
            const float fx = tp[u].y, fy = tp[u].z, gx = 1.f - fx, gy = 1.f - fy;
            const float *p = im + __float_as_int(tp[u].x);
            float *dst = smem + (at & 0xffff);
            auto put = [&](int i, float v) {
              dst[i * NSp] = v;
              if (OUT == kOutF32 && a.dbg_samples) a.dbg_samples[(row0 + i) * NS + (at >> 16)] = v;
            };
            float t1 = 0.f, b1 = 0.f;  // the right-hand pixels of the row before
#pragma unroll
            for (int i = 0; i < R; ++i) {
              if (i < nrows) {
                const float *pi = p + soff[i];
                // a row whose shift is one pixel further along x starts at the columns the row before ended at
                const bool next = (step >> i) & 1u;
                const float t0 = next ? t1 : pi[0], b0 = next ? b1 : pi[Lp];
                t1 = pi[1];
                b1 = pi[Lp + 1];
                put(i, bilerp(fx, fy, gx, gy, t0, t1, b0, b1));
              }
            }
          }
        }
      }
    } else {
      float cx[R], cy[R];
#pragma unroll
      for (int i = 0; i < R; ++i) {
        cx[i] = c0;
        cy[i] = c0;
        if (a.use_shifts && i < nrows) {
          const float2 sh = g.shifts[s0 + i];
          cx[i] += sh.x;
          cy[i] += sh.y;
        }
      }
      if constexpr (MODE == kPolarFrac) {
        const int Lp = g.pitch;
        const float *im0 = im + g.pad * Lp + g.pad;  // pixel (0, 0)
        for (int q = threadIdx.x; q < NS; q += NT) {
          const float4 tp = __ldg(g.taps + q);  // {place, offset x, offset y}
          const int at = __float_as_int(tp.x);
#pragma unroll
          for (int i = 0; i < R; ++i) {
            if (i < nrows) {
              const float x = cx[i] + tp.y, y = cy[i] + tp.z;
              const float xf = floorf(x), yf = floorf(y);
              const float fx = x - xf, fy = y - yf, gx = 1.f - fx, gy = 1.f - fy;
              const float *p = im0 + static_cast<int>(yf) * Lp + static_cast<int>(xf);
              const float v = bilerp(fx, fy, gx, gy, p[0], p[1], p[Lp], p[Lp + 1]);
              smem[i * NSp + (at & 0xffff)] = v;
              if (OUT == kOutF32 && a.dbg_samples) a.dbg_samples[(row0 + i) * NS + (at >> 16)] = v;
            }
          }
        }
      } else {
        for (int q = threadIdx.x; q < NS; q += NT) {
          const float2 o = g.offs[q];  // the bare mode's buffer is in ring order
#pragma unroll
          for (int i = 0; i < R; ++i) {
            if (i < nrows) {
              const float v = bilinear_smem(im, L, cx[i] + o.x, cy[i] + o.y);
              smem[i * NSp + q] = v;
              if (OUT == kOutF32 && a.dbg_samples) a.dbg_samples[(row0 + i) * NS + q] = v;
            }
          }
        }
      }
    }
    __syncthreads();

    // Phase 2: ring FFTs.  Rings of equal length form a contiguous class; the
    // (ring, row) jobs of a class are spread over the warps, 32 / T jobs per
    // warp, each transformed by a group of T threads (group_fft).
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int fw = 0;  // warp that takes the first pass of the next class
    sfor<0, kRingClasses>([&](auto kk) {  // longest first; a class the geometry lacks has no jobs
      constexpr int k = decltype(kk)::value;
      fw = ring_class<(256 >> k), R, OUT, NT / 32>(g, a, smem, planes, NB16, tws, s_kpos, g.cls[k], nrows, row0, warp,
                                                   lane, fw);
    });

    if constexpr (MODE == kPolarInt) load_taps(threadIdx.x);
    // Phase 3 (16-bit paths): copy-out in the layout of the tensor-core
    // kernel, 16 bytes per store.
    if constexpr (OUT != kOutF32) {
      __syncthreads();
      const int per_k = nrows * 4;
      for (int idx = threadIdx.x; idx < g.KS * per_k; idx += NT) {
        const int kk = nrows == R ? idx / (4 * R) : idx / per_k;
        const int rem = idx - kk * per_k;
        const int i = rem >> 2, t = rem & 3;
        const int64_t row = row0 + i;
        const int lane16 = 4 * static_cast<int>(row & 7) + t;
        const uint32_t *w = planes + i * NB16 + kk * 16;
        const uint2 w01 = *reinterpret_cast<const uint2 *>(w + ((2 * t) ^ (kk & 14)));
        const uint2 w89 = *reinterpret_cast<const uint2 *>(w + ((2 * t + 8) ^ (kk & 14)));
        const uint32_t w0 = w01.x, w1 = w01.y, w8 = w89.x, w9 = w89.y;
        // {q[2t], q[2t+1]}, {p[2t], p[2t+1]}, {q[2t+8], q[2t+9]}, {p[2t+8], p[2t+9]}
        a.out16[((row >> 3) * g.KS + kk) * 32 + lane16] =
            make_uint4(__byte_perm(w0, w1, 0x5410), __byte_perm(w0, w1, 0x7632), __byte_perm(w8, w9, 0x5410),
                       __byte_perm(w8, w9, 0x7632));
      }
      // the next group's phase 2 rewrites the planes only after the barrier
      // that follows its phase 1
    } else {
      __syncthreads();  // the next group's phase 1 overwrites the samples
    }
  }
}

template <int R, int MODE, int OUT, int NT = polar_threads(MODE)>
static cudaError_t launch_polar_r(const Geometry &g, const PolarArgs &a, size_t smem, cudaStream_t st) {
  static SmemLimit granted;
  cudaError_t e = raise_smem_limit(polar_fft_kernel<R, MODE, OUT, NT>, smem, granted);
  if (e != cudaSuccess) return e;
  // CTAs per image (each walks its share of the image's shift groups and
  // stages the image once): four of the small CTAs, so that the last wave
  // stays small, one of those that fill an SM; more when the images are too
  // few for four waves.
  int sms = 0;
  e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  constexpr int kPerSm = 512 / NT;
  const int64_t groups = (a.rows_per_img + R - 1) / R;
  const int64_t want = (static_cast<int64_t>(4 * kPerSm) * sms + a.n_imgs - 1) / a.n_imgs;
  int64_t per_img = kPerSm > 1 && smem + 1024 <= 232448 / 2 ? 4 : 1;
  if (per_img < want) per_img = want;
  if (per_img > groups) per_img = groups;
  dim3 grid(static_cast<unsigned>(per_img), static_cast<unsigned>(a.n_imgs));
  polar_fft_kernel<R, MODE, OUT, NT><<<grid, NT, smem, st>>>(g, a);
  return cudaGetLastError();
}

// Shared memory of a CTA with R rows: the staged image, its copy barrier,
// the twiddles, the output bases, then per row the samples and (16-bit
// output) the planes.
inline size_t polar_smem_bytes(const Geometry &g, int mode, bool out16, int R) {
  const size_t fixed = static_cast<size_t>(image_floats(g, mode)) * sizeof(float) + 16 + g.M * sizeof(float2) +
                       static_cast<size_t>((g.M / 2 + 2) & ~1) * sizeof(int);
  size_t per_row = static_cast<size_t>(sample_stride(g.NSb)) * sizeof(float);
  if (out16) per_row += static_cast<size_t>(g.KS) * 16 * sizeof(uint32_t);
  return fixed + per_row * R;
}

// Most rows (shifts) per CTA: with a bordered image as many as fit an SM, at
// most 8; otherwise as many as let two CTAs fit (~110 KB), else as many as
// fit in 200 KB, at most 4.
inline int polar_cta_rows(const Geometry &g, int mode, bool out16) {
  const size_t fixed = polar_smem_bytes(g, mode, out16, 0);
  const size_t per_row = polar_smem_bytes(g, mode, out16, 1) - fixed;
  auto fit = [&](size_t bytes) { return static_cast<int>((bytes > fixed ? bytes - fixed : 0) / per_row); };
  int R = mode != kPolarBare ? fit(kMaxSmemPerBlock) : fit(112640);
  if (R < 1) R = fit(204800);
  const int most = mode != kPolarBare ? 8 : 4;
  return R < 1 ? 1 : (R > most ? most : R);
}

// Rows per CTA with a bordered image.  A group of R rows takes about
// R + 2.5 row times (its phases' latency and barriers; fitted to R = 2..8 on
// the 76-, 90- and 128-pixel workloads: 12,000 images of 76 px, 81 shifts,
// 16-bit output: R = 2 28.4 ms, 3 23.8, 4 20.0, 5 19.0, and 21.4 for two CTAs
// of 8 warps with 2 rows each; 5,003 images of 32 px on a half-pixel grid of
// 49: 4 rows 1.92 ms, 6 1.47, 8 1.35, two small CTAs with 4 rows each 1.77), so
// large groups win on long stacks, where they also share table entries and
// pixel columns, and one row per CTA on calls whose rows do not fill the SMs.
// (With the warp count and table loads as they are now: 5 rows 15.8 ms, 8 rows
// of 32 px 1.16 ms; bound by the shared-memory data pipe, 81 % of its peak.)
inline int polar_bordered_rows(const PolarArgs &a, int most, int sms) {
  int best = 1;
  double best_cost = 1e300;
  for (int R = 1; R <= most; ++R) {
    if (R == 7) continue;  // not instantiated
    const int64_t groups = a.n_imgs * ((a.rows_per_img + R - 1) / R);
    const double cost = static_cast<double>((groups + sms - 1) / sms) * (R + 2.5);
    if (cost < best_cost) {
      best_cost = cost;
      best = R;
    }
  }
  return best;
}

template <int MODE, int OUT>
static cudaError_t launch_polar_t(const Geometry &g, const PolarArgs &a, cudaStream_t st) {
  int R = polar_cta_rows(g, MODE, OUT != kOutF32);
  if (R > a.rows_per_img) R = a.rows_per_img;
  if constexpr (MODE != kPolarBare) {
    int sms = 0;
    const cudaError_t e = sm_count(&sms);
    if (e != cudaSuccess) return e;
    // CTAs of 8 warps, two per SM, where one of 16 leaves its warps or the SM
    // idle (us, 16 warps / 8):
    // * one row per image (no shifts, or references), nothing for the other
    //   CTA's latency to hide behind: 300 images of 12, 60, 76 px 14.3 / 10.1,
    //   20.9 / 14.1, 22.4 / 15.0; 8,000 of 12, 76 px 194 / 98, 359 / 259 (and
    //   128 px, where only one CTA fits either way, 207 / 228: not taken);
    // * boxes whose rings hold fewer samples than the large CTA has threads
    //   (last ring up to 10), 4 rows a CTA: 2,000 images of 12, 24 px with 25
    //   shifts 228 / 168, 317 / 276;
    // * up to twice that where the images are so few that each is staged by
    //   several CTAs, or have 4 rows: 300 images of 32 px, 25 shifts 79 / 64, but
    //   2,000 392 / 460; 2,000 with 4 shifts 82 / 53.
    const size_t smem1 = polar_smem_bytes(g, MODE, OUT != kOutF32, 1);
    if (a.rows_per_img == 1 && 2 * (smem1 + 1024) <= kSmemPerSm)
      return launch_polar_r<1, MODE, OUT, 256>(g, a, smem1, st);
    const size_t smem4 = polar_smem_bytes(g, MODE, OUT != kOutF32, 4);
    if (R >= 4 && 2 * (smem4 + 1024) <= kSmemPerSm &&
        (g.NS < 512 || (g.NS < 1024 && (a.n_imgs < 4 * static_cast<int64_t>(sms) || a.rows_per_img == 4))))
      return launch_polar_r<4, MODE, OUT, 256>(g, a, smem4, st);
    R = polar_bordered_rows(a, R, sms);
    const size_t smem = polar_smem_bytes(g, MODE, OUT != kOutF32, R);
    switch (R) {
      case 1: return launch_polar_r<1, MODE, OUT>(g, a, smem, st);
      case 2: return launch_polar_r<2, MODE, OUT>(g, a, smem, st);
      case 3: return launch_polar_r<3, MODE, OUT>(g, a, smem, st);
      case 4: return launch_polar_r<4, MODE, OUT>(g, a, smem, st);
      case 5: return launch_polar_r<5, MODE, OUT>(g, a, smem, st);
      case 6: return launch_polar_r<6, MODE, OUT>(g, a, smem, st);
      default: return launch_polar_r<8, MODE, OUT>(g, a, smem, st);
    }
  } else {
    if (R == 3) R = 2;
    const size_t smem = polar_smem_bytes(g, MODE, OUT != kOutF32, R);
    switch (R) {
      case 1: return launch_polar_r<1, MODE, OUT>(g, a, smem, st);
      case 2: return launch_polar_r<2, MODE, OUT>(g, a, smem, st);
      default: return launch_polar_r<4, MODE, OUT>(g, a, smem, st);
    }
  }
}

template <int OUT>
static cudaError_t launch_polar_out(const Geometry &g, const PolarArgs &a, cudaStream_t st) {
  switch (g.mode) {
    case kPolarInt: return launch_polar_t<kPolarInt, OUT>(g, a, st);
    case kPolarFrac: return launch_polar_t<kPolarFrac, OUT>(g, a, st);
    default: return launch_polar_t<kPolarBare, OUT>(g, a, st);
  }
}

}  // namespace mra
