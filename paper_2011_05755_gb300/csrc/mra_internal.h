// Internal declarations shared by the C-ABI layer (mra_api.cpp) and the
// kernel translation units.  Not part of the public interface.
#pragma once

#include <cstdint>
#include <cuda.h>  // CUtensorMap (type only: the library does not link libcuda)
#include <cuda_runtime.h>

#include "../../include/mra.h"

namespace mra {

// Rows of the particle-spectrum layout and columns of the reference-spectrum
// layout are grouped in tiles of this many; within a tile the 8 values of one
// bin are contiguous (float2 each), so one bin of a tile is 64 bytes.
constexpr int kTile = 8;

// Rings [i0, i1) of one length 2 H: ring i's samples start at float
// off + (i - i0) stride of a row's sample buffer, its bins at natural-order
// bin + (i - i0) (H + 1).
struct RingClass {
  int i0, i1, H, off, stride, bin;
};

constexpr int kRingClasses = 7;

enum PolarMode { kPolarBare = 0, kPolarInt = 1, kPolarFrac = 2 };

// Geometry tables on the device (built in FP64 on the host, stored FP32).
struct Geometry {
  int L;            // box size
  int M;            // angles = largest ring length
  int NR;           // rings
  int NS;           // samples = sum N_r
  int NBIN;         // natural bins = sum (N_r/2 + 1)
  int NB;           // bins in the padded frequency-major layout
  int S;            // shifts
  int mirror;       // 0/1
  const float2 *offs;     // [NS]  r (cos theta_q, sin theta_q)
  // Polar kernel (PolarMode): where the image fits shared memory inside a zero
  // border of `pad` (4 or 8) pixels, rows of `pitch` floats, a table of the
  // samples in the order they are taken.  kPolarInt: {index of the top-left
  // neighbour of the unshifted position (int bits), fx, fy, place (int bits)};
  // kPolarFrac: {place, offset x, offset y, -}; place = offset in the sample
  // buffer | number in ring order << 16.
  const float4 *taps;     // [NS], null for kPolarBare
  int mode, pad, pitch;
  int nx, smin, sstep;    // kPolarInt: shift s = iy nx + ix is (smin + ix sstep, smin + iy sstep)
  // rings of length 512, 256, ..., 8 (i0 = i1: none), passed by value: walking
  // the ring table in memory for the class boundaries was a chain of NR
  // dependent loads per group of rows (12 % of the kernel)
  RingClass cls[kRingClasses];
  int NSb;                // floats of a row's sample buffer
  const int4 *rings;      // [NR]  {N_r, sample offset, natural-bin offset, log2(N_r/2)}
  const int *binpos;      // [NBIN] padded position of (ring, f), ring-major natural order
  const float *bweight;   // [NBIN] reference-side weight of (ring, f)
  const float2 *fwd_tw;   // [M]   exp(-2 pi i q / M)
  const float2 *inv_tw;   // [M]   exp(+2 pi i t k / M) at [k * T + t] (T threads per pair)
  const float2 *shifts;   // [S]   (sx, sy)
  const float2 *angles;   // [M]   (cos phi_j, sin phi_j)
  const int2 *fseg;       // [M/2 + 1] {segment offset, padded segment length} per frequency
  // 16-bit tensor-core layouts: frequency f owns k-steps [kso[f], kso[f+1]) of
  // 16 rings each; ksinfo[kk] = {f, k-step index within f}.
  int KS;                 // total k-steps
  const int *kso;         // [M/2 + 2]
  const int2 *ksinfo;     // [KS]
  const int *kpos;        // [M/2 + 1] binpos of (ring i, f) = kpos[f] + i
  const int *kpos16;      // [M/2 + 1] 16-bit position of (ring i, f) = kpos16[f] + i
  // BF16 mma fragments of the two 16-point DFT stages of the tensor-core
  // inverse angular DFT (kernels with an mma.sync inverse DFT only): [0, 512) stage-1 A, [512, 1024) stage-2 B,
  // each [32 lanes][16 words].
  const uint32_t *dft16;
  // Staging chunks of the M = 256 and M = 512 tensor-core kernels: chunk c
  // holds the whole frequencies [chunk_f[c], chunk_f[c + 1]), at most
  // kTc256ChunkKs (M = 256) or kTc512ChunkKs (M = 512) k-steps.
  int NCH;
  const int *chunk_f;     // [NCH + 1]
  // M = 256 kernel with the tcgen05 inverse DFT (null unless the handle uses
  // it; its k-steps are then ordered by contraction warp and parity): the
  // four BF16 DFT matrices Ee, Oe, Eo, Oo (64 angles x 64 frequencies,
  // canonical K-major core matrices).
  const uint32_t *hyb_w;   // [kHyb256Mats * 2048]
  int hyb_pattern;         // k-steps per slot: 0 = {3,2,2,2,1,1,1,1}, 1 = {3,3,2,2,2,2,2,2}
};

constexpr int kHyb256N0 = 3;    // k-steps of f = 0
constexpr int kHyb256Mats = 4;

constexpr int kTc256ChunkKs = 22;
constexpr int kTc512ChunkKs = 44;
constexpr int kTc512MaxKsPerF = 6;  // rings with N_r <= 512 have r <= 81: at most 6 k-steps of 16 per frequency

struct PolarArgs {
  const float *imgs;   // [n][L][L]
  int64_t n_imgs;
  int rows_per_img;    // S for particles, 1 for references
  bool use_shifts;     // false for references (s = 0)
  bool weighted;       // multiply bins by bweight (references)
  float2 *out;         // tiled spectra [ceil(rows/8)][NB][8] (may be null in debug)
  uint4 *out16;        // 16-bit A fragments [ceil(rows/8)][KS][32 lanes], or null
  bool fp16;           // out16 element type: FP16 (true) or BF16 (false)
  float *dbg_samples;  // [rows][NS] or null
  float2 *dbg_spec;    // [rows][NBIN] or null
  // Image staging by one TMA tensor copy per CTA (tma true): a 3-D map over
  // imgs ({L, L, n_imgs} FP32) whose box is the image in its zero border
  // ({L + 2 pad, L + 2 pad, 1}, loaded from (-pad, -pad, image); the border
  // is the map's zero fill) or the bare image (pad 0) of the path's layout.
  // tma false: plain loads.
  CUtensorMap tmap;
  bool tma;
  int *err;              // device flag: bit 0 = the staging wait timed out
  uint32_t wait_limit;   // polls before that wait gives up
};

struct CCArgs {
  const float2 *A;               // tiled particle spectra [row tiles][NB][8]
  const float2 *B;               // tiled weighted reference spectra [ref tiles][NB][8]
  int64_t rows;                  // images_in_chunk * S
  int K;                         // references
  unsigned long long *best;      // [images_in_chunk] argmax keys (pre-set to 0)
  float *dbg_cc;                 // [n][K][S][2][M] full table, or null
  int seg_max;                   // longest padded frequency segment (bins)
  int *err;                      // device flag: bit 0 = a bounded wait timed out
  uint32_t wait_limit;           // polls before a barrier wait gives up
  uint32_t first_wait_limit;     // same for each warp's first wait (tests shorten it)
};

// Precision-split path (16-bit tensor-core contraction + FP32 rescore).
constexpr int kTopRows = 8;  // candidate rows per image rescored in FP32

struct TcArgs {
  const uint4 *A16;              // [row tiles][KS][32 lanes] A fragments
  const uint4 *B16;              // [ref tiles of 8][KS][32 lanes] B fragments of both 4-reference blocks
  int64_t rows;                  // images_in_chunk * S
  int K;
  float *rowmax;                 // [images_in_chunk][K][S][2] row maxima over angles
  float *dbg_cc;                 // [n][K][S][2][M] full (16-bit-contraction) table, or null
  int ks_max;                    // most k-steps of any frequency
  int *err;
  uint32_t wait_limit, first_wait_limit;
};

struct RescoreArgs {
  const float *imgs;             // [n][L][L] images of the chunk
  int64_t n;
  const int *cand;               // [n][kTopRows] row ids (k * S + s) * 2 + m, or -1
  const float2 *B;               // FP32 weighted reference spectra, tiled
  unsigned long long *best;      // [n] argmax keys (zero on entry)
};

cudaError_t launch_refs16(const Geometry &g, const float2 *B, int ktiles, uint4 *B16, bool fp16, cudaStream_t st);
// M = 256: mma.sync contraction with the tcgen05 inverse DFT.
cudaError_t launch_cc_hybrid256(const Geometry &g, const TcArgs &a, bool fp16, cudaStream_t st);
cudaError_t launch_cc_tc(const Geometry &g, const TcArgs &a, bool fp16, cudaStream_t st);
cudaError_t launch_top8(const float *rowmax, int64_t n, int nrows, int *cand, unsigned long long *best,
                        cudaStream_t st);  // (clears best)
cudaError_t launch_rescore(const Geometry &g, const RescoreArgs &a, cudaStream_t st);
size_t rescore_smem(const Geometry &g);
int rescore_ctas_per_sm(const Geometry &g);  // resident rescore CTAs per SM (0 if unknown)
// Shared memory of one CTA of the polar kernel with one row, of the FP32
// contraction kernel, and the per-CTA opt-in limit of the device.
size_t polar_smem_one_row(const Geometry &g, int mode, bool out16);
int polar_rows_per_cta(const Geometry &g, int mode, bool out16);
size_t cc_fp32_smem(int M, int seg_max);
constexpr size_t kMaxSmemPerBlock = 232448;  // 227 KB
constexpr size_t kSmemPerSm = 233472;        // 228 KB, of which each resident CTA takes 1 KB more than it asks for
// Every check mra_create makes on a configuration, without CUDA calls or heap
// use: MRA_OK, MRA_EINVAL or MRA_EUNSUPPORTED with a message in why.
int check_config(const mra_config_t *c, char *why, size_t why_len);

// Ring classes of a geometry with NR rings (ascending lengths), `gap` floats
// between consecutive rings in the sample buffer; sets cls and NSb.
inline void set_ring_classes(Geometry &g, const int4 *rings, int NR, int gap) {
  for (int k = 0; k < kRingClasses; ++k) g.cls[k] = RingClass{0, 0, 256 >> k, 0, 0, 0};
  for (int i = 0; i < NR; ++i) {
    const int N = rings[i].x;
    int k = 0;
    while (512 >> k > N) ++k;
    if (g.cls[k].i1 == 0) g.cls[k] = RingClass{i, i, N / 2, rings[i].y + gap * i, N + gap, rings[i].z};
    g.cls[k].i1 = i + 1;
  }
  g.NSb = rings[NR - 1].y + rings[NR - 1].x + gap * NR;
}

// Launchers (return cudaGetLastError() of the launch).
cudaError_t launch_polar(const Geometry &g, const PolarArgs &a, cudaStream_t st);
cudaError_t launch_cc_fp32(const Geometry &g, const CCArgs &a, cudaStream_t st);
cudaError_t launch_decode(const Geometry &g, const unsigned long long *best, int64_t n, int K,
                          void *poses, cudaStream_t st);
int cc_threads_per_pair(int M);

// Class averaging.
struct AvgWork {
  int *hist;          // [K * nblk]
  int *scan;          // [K * nblk]
  int *perm;          // [n]
  int *chunk_class;   // [max_chunks]
  int *chunk_begin;   // [max_chunks]
  int *chunk_count;   // [max_chunks]
  int *n_chunks;      // [1]
  int *class_counts;  // [K]
  int *class_first_chunk; // [K + 1]
  float *part_sum;    // [max_chunks][L*L]
  float *part_comp;   // [max_chunks][L*L]
  int max_chunks;
};
constexpr int kClassSumLaunches = 6;  // kernels launched by launch_class_sums
constexpr int kAvgBlock = 256;   // images per histogram block
constexpr int kAvgChunk = 64;    // images per partial-sum chunk
cudaError_t launch_class_sums(const Geometry &g, const float *imgs, const void *poses, int64_t n,
                              int K, const AvgWork &w, float *sum, float *comp, int *counts,
                              bool accumulate, cudaStream_t st);
cudaError_t launch_refresh_refs(int L, float *refs, const int *counts, int K, const int *reseed, const float *imgs,
                                int64_t n, cudaStream_t st);
cudaError_t launch_average_finalize(const Geometry &g, int K, const float *sum, const float *comp,
                                    const int *counts, float *avg, cudaStream_t st);

}  // namespace mra
