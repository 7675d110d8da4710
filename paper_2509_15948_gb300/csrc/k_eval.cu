// Evaluation metrics of the matched mix against the target (Sec. 5.3): SI-SDR over the stereo signal and the
// MIR feature distances of Eq. (27) over disjoint 8 s segments: RMS and crest factor per channel, stereo
// width ||l - r|| / ||l + r||, stereo imbalance (||l||^2 - ||r||^2) / (||l||^2 + ||r||^2), and the 24-band
// Zwicker Bark spectrum of the mid signal (l + r) / 2 from Hann-windowed 8192-sample frames with hop 8192
// (mean power per band, in dB).  A song shorter than 8 s is one segment.
//
// A segment is cut into pieces of two Bark frames (16,384 samples), two CTAs per piece: CTA 0 takes the Bark spectrum
// of the estimate (the two frames packed as one complex FFT) and the statistics and SI-SDR sums of the piece's first
// half, CTA 1 the spectrum of the reference and the second half; the last segment of a song has further pieces, for
// the SI-SDR sums of the samples after it.  A per-segment kernel adds the pieces in order and forms the feature
// differences, a per-song kernel combines the segments (double precision, fixed order).
// The sums are double (FP64 runs at a 64th of FP32's rate here), so the work has to reach every SM: with one CTA per
// segment a 19 s song (2 segments) took 4.42 ms + 0.14 ms; with 104 CTAs it is latency of one FFT and 16 samples per
// thread.
#include "mg_fftp.cuh"

namespace mg {

namespace {
constexpr int kEvThreads = 512;
constexpr int kBarkFrame = 8192;
constexpr int kBarkLog = 13;
constexpr int kBands = 24;
constexpr int kPiece = kEvalPiece;
static_assert(kPiece == 2 * kBarkFrame, "a piece is two Bark frames");
// a part (one CTA's sums, doubles): 0-7 energies of the half piece (estimate, then reference: l^2, r^2, (l-r)^2,
// (l+r)^2), 8-10 the SI-SDR sums <e,r>, <r,r>, <e,e>, 11-14 peaks, 16-39 band powers of its signal
constexpr int kPartStride = kEvalPart;
// a segment (doubles): 0-4 sums of squared feature differences (RMS, crest factor, width, imbalance, Bark), 5-7 SI-SDR
constexpr int kSegStride = kEvalSeg;

template <int NV>
__device__ __forceinline__ void block_reduce_d(double (&v)[NV], double* red) {
  // sum over the block, result in thread 0
#pragma unroll
  for (int k = 0; k < NV; ++k)
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  __syncthreads();
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < NV; ++k) red[w * NV + k] = v[k];
  __syncthreads();
  if (threadIdx.x == 0)
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      double s = 0.0;
      for (int j = 0; j < nw; ++j) s += red[j * NV + k];
      v[k] = s;
    }
  __syncthreads();
}

__device__ __forceinline__ float warp_max(float v) {
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_down_sync(0xffffffffu, v, o));
  return v;
}
}  // namespace

// item = (song, segment, 2 piece + signal, -); band_lo/band_hi: [24] bin range of each Bark band
__global__ void __launch_bounds__(kEvThreads) k_eval_part(const SongDev* __restrict__ songs, const int4* __restrict__ items,
                                                          int seg_len, const int* __restrict__ band_lo,
                                                          const int* __restrict__ band_hi, double* __restrict__ out,
                                                          const float2* __restrict__ ptw) {
  extern __shared__ float2 sm[];
  __shared__ double red[16 * 11];
  __shared__ float mred[4][16];
  const int4 it = items[blockIdx.x];
  const SongDev& S = songs[it.x];
  const int nseg = S.L < seg_len ? 1 : S.L / seg_len, piece = it.z >> 1, sig = it.z & 1;
  const int s0 = it.y * (S.L < seg_len ? 0 : seg_len);
  const int s1 = S.L < seg_len ? S.L : s0 + seg_len;
  const int s2 = it.y == nseg - 1 ? S.L : s1;      // SI-SDR sums run to the end of the song on the last segment
  const float* el = S.mix;
  const float* er = S.mix + S.ld;
  const float* rl = S.target;
  const float* rr = S.target + S.ld;
  double acc[11] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
  float pk[4] = {0.f, 0.f, 0.f, 0.f};
  const int h0 = s0 + piece * kPiece + sig * kBarkFrame, h1 = min(h0 + kBarkFrame, s2);
  for (int s = h0 + threadIdx.x; s < h1; s += blockDim.x) {
    const float a = el[s], b = er[s], c = rl[s], d = rr[s];
    acc[8] += (double)a * c + (double)b * d;
    acc[9] += (double)c * c + (double)d * d;
    acc[10] += (double)a * a + (double)b * b;
    if (s < s1) {
      acc[0] += (double)a * a;
      acc[1] += (double)b * b;
      acc[2] += (double)(a - b) * (a - b);
      acc[3] += (double)(a + b) * (a + b);
      acc[4] += (double)c * c;
      acc[5] += (double)d * d;
      acc[6] += (double)(c - d) * (c - d);
      acc[7] += (double)(c + d) * (c + d);
      pk[0] = fmaxf(pk[0], fabsf(a));
      pk[1] = fmaxf(pk[1], fabsf(b));
      pk[2] = fmaxf(pk[2], fabsf(c));
      pk[3] = fmaxf(pk[3], fabsf(d));
    }
  }
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float m = warp_max(pk[k]);
    if (lane == 0) mred[k][w] = m;
  }
  block_reduce_d<11>(acc, red);
  double* o = out + (size_t)blockIdx.x * kPartStride;
  if (threadIdx.x == 0)
    for (int k = 0; k < 11; ++k) o[k] = acc[k];
  if (threadIdx.x < 4) {
    float m = 0.f;
    for (int j = 0; j < nw; ++j) m = fmaxf(m, mred[threadIdx.x][j]);
    o[11 + threadIdx.x] = m;
  }
  // Bark spectrum: frames 2 piece and 2 piece + 1 of one signal travel packed as one complex FFT (signals of very
  // different level are never mixed); a warp per band
  const int nfr = (s1 - s0) / kBarkFrame, f = 2 * piece;
  if (f >= nfr) return;   // the whole block: nothing of a Bark frame in this piece (its band sums are not read)
  const bool two = f + 1 < nfr;
  const float* xl = sig ? rl : el;
  const float* xr = sig ? rr : er;
  const int b0 = s0 + f * kBarkFrame;
  fft_p_io<false>(sm, kBarkLog, 1, pstride(kBarkFrame), ptw, [=](int, int j) {
    const float win = 0.5f * (1.f - cospif(2.f * j / kBarkFrame));
    const int s = b0 + j;
    const float a = 0.5f * (xl[s] + xr[s]) * win;
    const float b = two ? 0.5f * (xl[s + kBarkFrame] + xr[s + kBarkFrame]) * win : 0.f;
    return make_float2(a, b);
  });
  for (int b = w; b < kBands; b += nw) {
    double p = 0.0;
    for (int k = band_lo[b] + lane; k < band_hi[b]; k += 32) {
      const float2 z = sm[pidx(k)], zm = sm[pidx((kBarkFrame - k) & (kBarkFrame - 1))];
      const float ar = 0.5f * (z.x + zm.x), ai = 0.5f * (z.y - zm.y);      // frame f
      const float br = 0.5f * (z.y + zm.y), bi = 0.5f * (zm.x - z.x);      // frame f + 1
      p += (double)ar * ar + (double)ai * ai + (double)br * br + (double)bi * bi;
    }
#pragma unroll
    for (int o2 = 16; o2 > 0; o2 >>= 1) p += __shfl_down_sync(0xffffffffu, p, o2);
    if (lane == 0) o[16 + b] = p;
  }
}

// One CTA per segment: the parts of its pieces (parts[seg_begin[s]] .. parts[seg_begin[s + 1]]) added in order, then the
// squared feature differences of Eq. (27).
__global__ void __launch_bounds__(64) k_eval_seg(const SongDev* __restrict__ songs, const int2* __restrict__ segs,
                                                 const int* __restrict__ seg_begin, int seg_len,
                                                 const double* __restrict__ parts, double* __restrict__ out) {
  __shared__ double v[11 + 4 + 2 * kBands], bark[kBands];
  const int2 sg = segs[blockIdx.x];
  const SongDev& S = songs[sg.x];
  const int len = S.L < seg_len ? S.L : seg_len, nfr = len / kBarkFrame, npair = (nfr + 1) / 2;
  const int p0 = seg_begin[blockIdx.x], p1 = seg_begin[blockIdx.x + 1], t = threadIdx.x;
  if (t < 15) {
    double s = 0.0;
#pragma unroll 4
    for (int p = p0; p < p1; ++p) {
      const double x = parts[(size_t)p * kPartStride + t];
      s = t < 11 ? s + x : fmax(s, x);
    }
    v[t] = s;
  } else if (t >= 16 && t < 16 + 2 * kBands) {
    const int sig = (t - 16) / kBands, b = (t - 16) % kBands;
    double s = 0.0;
#pragma unroll 4
    for (int p = 0; p < npair; ++p) s += parts[(size_t)(p0 + 2 * p + sig) * kPartStride + 16 + b];
    v[15 + t - 16] = nfr ? s / nfr : 0.0;
  }
  __syncthreads();
  if (t < kBands) {
    const double d = 10.0 * log10(v[15 + t] + 1e-12) - 10.0 * log10(v[15 + kBands + t] + 1e-12);
    bark[t] = d * d;
  }
  __syncthreads();
  if (t != 0) return;
  auto q = [](double n, double d) { return d != 0.0 ? n / d : 0.0; };
  const double n = len;
  double* o = out + (size_t)blockIdx.x * kSegStride;
  double fe[6], fr[6];
  for (int h = 0; h < 2; ++h) {
    const double* e = v + 4 * h;
    double* f = h ? fr : fe;
    f[0] = sqrt(e[0] / n);
    f[1] = sqrt(e[1] / n);
    f[2] = q(v[11 + 2 * h], f[0]);
    f[3] = q(v[12 + 2 * h], f[1]);
    f[4] = q(sqrt(e[2]), sqrt(e[3]));
    f[5] = q(e[0] - e[1], e[0] + e[1]);
  }
  o[0] = (fe[0] - fr[0]) * (fe[0] - fr[0]) + (fe[1] - fr[1]) * (fe[1] - fr[1]);
  o[1] = (fe[2] - fr[2]) * (fe[2] - fr[2]) + (fe[3] - fr[3]) * (fe[3] - fr[3]);
  o[2] = (fe[4] - fr[4]) * (fe[4] - fr[4]);
  o[3] = (fe[5] - fr[5]) * (fe[5] - fr[5]);
  double s = 0.0;
  for (int b = 0; b < kBands; ++b) s += bark[b];
  o[4] = s;
  for (int k = 0; k < 3; ++k) o[5 + k] = v[8 + k];
}

// out_song [n][6]: SI-SDR (dB), d_rms, d_cf, d_sw, d_si, d_bs (Eq. 27; -inf when the features agree exactly)
__global__ void k_eval_finalize(const int* __restrict__ item_begin,
                                const double* __restrict__ seg, float* __restrict__ out_song) {
  const int si = blockIdx.x, t = threadIdx.x;
  const int a = item_begin[si], b = item_begin[si + 1];
  if (t == 0) {
    double dot = 0.0, rr = 0.0, ee = 0.0;
    for (int i = a; i < b; ++i) {
      const double* o = seg + (size_t)i * kSegStride;
      dot += o[5];
      rr += o[6];
      ee += o[7];
    }
    // SI-SDR: ||alpha r||^2 / ||alpha r - e||^2 with ||alpha r - e||^2 = ||e||^2 - alpha <e, r>, alpha = <e,r>/||r||^2
    const double alpha = rr != 0.0 ? dot / rr : 0.0;
    const double tgt = alpha * alpha * rr, res = ee - alpha * dot;
    out_song[si * 6 + 0] = (float)(10.0 * log10(tgt / res));
  } else if (t % 32 == 0 && t / 32 <= 5) {   // a warp per feature: double logarithms of one warp run in turn
    const int k = t / 32 - 1;
    double acc = 0.0;
    for (int i = a; i < b; ++i) acc += seg[(size_t)i * kSegStride + k];
    const int cnt = (b - a) * (k < 2 ? 2 : (k < 4 ? 1 : kBands));
    out_song[si * 6 + 1 + k] = acc > 0.0 ? (float)log10(acc / cnt) : -INFINITY;
  }
}

void launch_eval(cudaStream_t st, const SongDev* songs, int n_songs, const int4* parts, int n_parts, const int2* segs,
                 int n_segs, const int* seg_begin, const int* item_begin, int seg_len, const int* band_lo,
                 const int* band_hi, double* part_out, double* seg_out, float* out_song, const float2* ptw) {
  if (!n_segs) return;
  k_eval_part<<<n_parts, kEvThreads, pstride(kBarkFrame) * sizeof(float2), st>>>(songs, parts, seg_len, band_lo,
                                                                                   band_hi, part_out, ptw);
  k_eval_seg<<<n_segs, 64, 0, st>>>(songs, segs, seg_begin, seg_len, part_out, seg_out);
  k_eval_finalize<<<n_songs, 192, 0, st>>>(item_begin, seg_out, out_song);
}

void init_eval_attributes() {
  cudaFuncSetAttribute(k_eval_part, cudaFuncAttributeMaxDynamicSharedMemorySize, pstride(kBarkFrame) * (int)sizeof(float2));
}

}  // namespace mg
