// Multi-resolution STFT loss of Sec. 5.1 (Eqs. 20-21) and its adjoint.
// Per resolution: frames t hop .. t hop + n_fft of the stereo mix (periodic Hann, no centre padding) are
// transformed as one packed complex FFT z = left + i right; per bin the channel spectra are
// X_L = (Z[k] + conj Z[-k]) / 2, X_R = (Z[k] - conj Z[-k]) / 2i, X_M = X_L + X_R, X_S = X_L - X_R;
// magnitudes sqrt(A_k^2 |X|^2 + 1e-8) (A-weighting per bin) are projected on the Mel triangles (CSR by
// band, fixed summation order), compared with the cached target spectrograms, and reduced per work item
// (deterministic partial sums, no atomics).
// Adjoint: the same frames are re-transformed, dL/dY_hat per band goes back to the bins through the
// transposed Mel CSR, to the complex bins through |X|, to the packed Hermitian spectrum, and through one
// inverse FFT to the windowed frame; a gather kernel overlap-adds the frames of all resolutions.
//
// What bounds it: issue and latency of 32 warps per SM (two CTAs of 64 registers a thread and 95 KB; issue slots half
// used).  Before, the Mel sums and the adjoint's band values went one (frame, band) after the other, each waiting for its
// own table and target loads and for 20 shuffles, 45 us per wave of CTAs whatever the resolution and a launch for each.
// All resolutions are one launch now, the sums go band by band with a weight for four channels, and the loss terms are one
// coalesced pass (a 30 s mix: forward 242 -> 203 us, adjoint 190 -> 183 by the last two).  Every sum keeps its order, so the
// losses and gradients keep their bits.
// The band buffer is the largest resolution's in every mode.  Where it passes 43 KB (linear bins; 96 bands at n_fft 256, 512
// at 1,024) one CTA fills an SM in the forward too, which the kernel before, with no buffer there, did not; it is the
// faster one all the same (events, 30 s mix: 512/2048/8192 linear 490 -> 427 us, 256/1024/4096 with 96 bands 355 -> 271,
// 1024/2048/8192 with 512 bands 425 -> 332; 2 s: 127 -> 33, 106 -> 25, 124 -> 33).
#include "mg_fftp.cuh"

namespace mg {

namespace {
constexpr int kLossThreads = 512;
constexpr float kLogEps = 1e-5f;
constexpr float kMagEps = 1e-8f;
// frames of one item live in a padded layout: frame f, sample j at sm[f * pstride(n) + pidx(j)];
// an item holds 8192 samples (8192 / n_fft <= 128 frames), so the buffer needs 8192 + 512 + 128 entries.
constexpr int kFrameBuf = kLossFrameBuf;

// channel magnitudes^2 of bin k (|X_L|^2, |X_R|^2, |X_M|^2, |X_S|^2) and the complex X_L, X_R
__device__ __forceinline__ void bin_spectra(const float2* Z, int k, int n, float2& XL, float2& XR) {
  const float2 a = Z[pidx(k)], b = Z[pidx((n - k) & (n - 1))];
  XL = make_float2(0.5f * (a.x + b.x), 0.5f * (a.y - b.y));
  // (a - conj b) / 2i
  const float2 d = make_float2(a.x - b.x, a.y + b.y);
  XR = make_float2(0.5f * d.y, -0.5f * d.x);
}

__device__ __forceinline__ float2 chan(int c, float2 XL, float2 XR) {
  if (c == 0) return XL;
  if (c == 1) return XR;
  if (c == 2) return cadd(XL, XR);
  return csub(XL, XR);
}

// After the magnitude pass a frame holds, for bin k in [0, n/2], the weighted magnitudes
// sqrt(A_k^2 |X_c|^2 + 1e-8) of channels 0, 1 at slot pidx(k) and of channels 2, 3 at mag_slot2(k): the
// mirror slot pidx(n - k), or for the self-mirrored bins 0 and n/2 two padding slots no element uses
// (pidx(n) = the last slot of the padded frame, and slot 16).
__device__ __forceinline__ int mag_slot2(int k, int n) { return k == (n >> 1) ? 16 : pidx(n - k); }

__device__ __forceinline__ float4 bin_mags(const LossRes& R, const float2* Z, int k) {
  float2 XL, XR;
  bin_spectra(Z, k, R.nfft, XL, XR);
  const float a = R.aw2[k];
  float m[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const float2 X = chan(c, XL, XR);
    m[c] = sqrtf(a * (X.x * X.x + X.y * X.y) + kMagEps);
  }
  return make_float4(m[0], m[1], m[2], m[3]);
}
}  // namespace

// item (song, res, first frame, frames); mode 0: write target spectrogram + partial sum Y^2 per set;
// mode 1: partial sums of |dlog| and (Y - Yhat)^2 per set; mode 3: mode 1 that also keeps the frame spectra
// (in dF, which the adjoint overwrites frame by frame) and the band values Yhat (training forward);
// mode 2: adjoint frames to dF from the kept spectra and band values.
template <int mode>
__global__ void __launch_bounds__(kLossThreads, 2) k_loss_frames(LaunchCtx c, const SongDev* __restrict__ songs,
                                                              const LossRes* __restrict__ resv,
                                                              const int4* __restrict__ items) {
  extern __shared__ float2 sm[];
  __shared__ float red[6 * 32];
  const int4 it = items[blockIdx.x];
  const SongDev& S = songs[it.x];
  const LossRes& R = resv[it.y];
  const int t0 = it.z, nb = it.w, n = R.nfft, nbands = R.nbands, bs = pstride(n);
  const float* x = mode == 0 ? S.target : S.mix;
  float2* Zk = reinterpret_cast<float2*>(S.dF[it.y]);     // frame spectra kept between mode 3 and mode 2
  if constexpr (mode == 2) {
    const float4* zi = reinterpret_cast<const float4*>(Zk + (size_t)t0 * n);
#pragma unroll 4
    for (int e = threadIdx.x; e < nb * n / 2; e += blockDim.x) {
      const int f = e >> (R.log_nfft - 1), j = 2 * e & (n - 1);
      const float4 z = zi[e];
      sm[f * bs + pidx(j)] = make_float2(z.x, z.y);
      sm[f * bs + pidx(j + 1)] = make_float2(z.z, z.w);
    }
  } else {
    // the windowed frames go straight from global memory into the first pass of the transform
    const int L = S.L, ld = S.ld, hop = R.hop;
    const float* win = R.win;
    fft_p_io<false>(sm, R.log_nfft, nb, bs, c.tab.ptw, [=](int f, int j) {
      const int s = (t0 + f) * hop + j;
      const float w = win[j];
      return s < L ? make_float2(x[s] * w, x[ld + s] * w) : make_float2(0.f, 0.f);
    });
  }
  float* Yt = S.Y[it.y];
  float* Yk = S.Yh[it.y];
  if constexpr (mode != 2) {
    // magnitudes of the four channels per bin, in place (each thread owns the pair k, n - k; the thread of
    // k = 0 also takes k = n/2); mode 3 keeps the spectrum on the way
    const int half = n >> 1, lh = R.log_nfft - 1;
#pragma unroll 2
    for (int e = threadIdx.x; e < nb << lh; e += blockDim.x) {
      const int f = e >> lh, k = e & (half - 1);
      float2* Z = sm + f * bs;
      if (mode == 3) {
        float2* zo = Zk + (size_t)(t0 + f) * n;
        const int k2 = k == 0 ? half : n - k;
        zo[k] = Z[pidx(k)];
        zo[k2] = Z[pidx(k2)];
      }
      if (k == 0) {
        const float4 m0 = bin_mags(R, Z, 0), mh = bin_mags(R, Z, half);
        Z[pidx(0)] = make_float2(m0.x, m0.y);
        Z[mag_slot2(0, n)] = make_float2(m0.z, m0.w);
        Z[pidx(half)] = make_float2(mh.x, mh.y);
        Z[mag_slot2(half, n)] = make_float2(mh.z, mh.w);
      } else {
        const float4 m = bin_mags(R, Z, k);
        Z[pidx(k)] = make_float2(m.x, m.y);
        Z[pidx(n - k)] = make_float2(m.z, m.w);
      }
    }
    __syncthreads();
    // Band values Y[f][b][channel] of the item into shared memory, then one pass over them for the loss terms.  The
    // pairs (frame, band) go band by band, so that the threads of a warp run over equally long bands and read the same
    // weights, and a weight and its bin serve all four channels.  (One thread per value, resp. one warp per pair with 20
    // entries on average for its 32 lanes, was 60 % of the kernel's instructions.)
    const bool wide = R.band_beg[nbands] >= 16 * nbands;
    float* yv = reinterpret_cast<float*>(sm + kFrameBuf);
    const int pairs = nb * nbands;
    const float inv_nb = 1.f / (float)nb;   // e / nb = floor((e + 1/2) inv_nb): pairs < 2^16
    // pair (f, b) is quad f nbands + (b + f mod 8) mod nbands: the frames of one band fall in distinct banks
    const int rot = nbands >= 8 ? 7 : 0;
    auto quad_of = [&](int f, int b) {
      const int r = b + (f & rot);
      return f * nbands + (r >= nbands ? r - nbands : r);
    };
    if (wide) {
      // wide bands: eight lanes per pair.  Lane l holds the sums of entries l + 8 i (mod 32), i < 4, which are then added
      // as a warp would over its lanes with xor 16, 8, 4, 2, 1.
      const int l8 = threadIdx.x & 7;
      const bool h4 = l8 & 4, h2 = l8 & 2;
      for (int e0 = threadIdx.x >> 5 << 2; e0 < pairs; e0 += blockDim.x >> 3) {
        const int e = e0 + ((threadIdx.x >> 3) & 3);
        const bool live = e < pairs;
        const int bd = live ? (int)((e + 0.5f) * inv_nb) : 0, f = live ? e - bd * nb : 0;
        const int beg = R.band_beg[bd], len = live ? R.band_beg[bd + 1] - beg : 0;
        const int k0 = len ? R.band_bin[beg] : 0;
        const float2* Zf = sm + f * bs;
        float y4[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int ch = 0; ch < 4; ++ch) y4[i][ch] = 0.f;
        for (int q0 = l8; q0 < len; q0 += 32) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int q = q0 + 8 * i;
            if (q < len) {
              const float wq = R.band_w[beg + q];
              const float2 lr = Zf[pidx(k0 + q)], ms = Zf[mag_slot2(k0 + q, n)];
              y4[i][0] = fmaf(wq, lr.x, y4[i][0]);
              y4[i][1] = fmaf(wq, lr.y, y4[i][1]);
              y4[i][2] = fmaf(wq, ms.x, y4[i][2]);
              y4[i][3] = fmaf(wq, ms.y, y4[i][3]);
            }
          }
        }
        float y[4];
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) y[ch] = (y4[0][ch] + y4[2][ch]) + (y4[1][ch] + y4[3][ch]);
        // after xor 4 a lane keeps two channels, after xor 2 one
        const float s0 = __shfl_xor_sync(0xffffffffu, h4 ? y[0] : y[2], 4);
        const float s1 = __shfl_xor_sync(0xffffffffu, h4 ? y[1] : y[3], 4);
        const float a0 = (h4 ? y[2] : y[0]) + s0, a1 = (h4 ? y[3] : y[1]) + s1;
        float v = (h2 ? a1 : a0) + __shfl_xor_sync(0xffffffffu, h2 ? a0 : a1, 2);
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        if (live && !(l8 & 1)) yv[4 * quad_of(f, bd) + (l8 >> 1)] = v;
      }
    } else {
      for (int e = threadIdx.x; e < pairs; e += blockDim.x) {
        const int bd = (int)((e + 0.5f) * inv_nb), f = e - bd * nb;
        const int beg = R.band_beg[bd], len = R.band_beg[bd + 1] - beg;
        const int k0 = len ? R.band_bin[beg] : 0;
        const float2* Zf = sm + f * bs;
        float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (int q = 0; q < len; ++q) {
          const float wq = R.band_w[beg + q];
          const float2 lr = Zf[pidx(k0 + q)], ms = Zf[mag_slot2(k0 + q, n)];
          y.x = fmaf(wq, lr.x, y.x);
          y.y = fmaf(wq, lr.y, y.y);
          y.z = fmaf(wq, ms.x, y.z);
          y.w = fmaf(wq, ms.y, y.w);
        }
        reinterpret_cast<float4*>(yv)[quad_of(f, bd)] = y;
      }
    }
    __syncthreads();
    // the values in frame order, target and kept values coalesced.  The sums go in fixed chains of one channel each: narrow
    // bands, thread t adds values t, t + 512, ...; wide ones, lane c < 4 of a warp adds channel c of every 16th pair,
    // after all threads have put the terms where the frames were.
    const int row = nbands * 4, total = nb * row;
    float *t0v = reinterpret_cast<float*>(sm), *t1v = t0v + total;   // wide: total <= 2,048
    float acc0 = 0.f, acc1 = 0.f;
    const int mych = threadIdx.x & 3;
    {
      const float inv_row = 1.f / (float)row;
      const size_t base = (size_t)t0 * row;
      constexpr int kAhead = 4;
      for (int e0 = threadIdx.x; e0 < total; e0 += kAhead * blockDim.x) {
        float yt[kAhead];
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
          const int e = e0 + j * blockDim.x;
          yt[j] = mode != 0 && e < total ? Yt[base + e] : 0.f;
        }
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
          const int e = e0 + j * blockDim.x, f = (int)((e + 0.5f) * inv_row);
          if (e >= total) continue;
          const int r = e - f * row + 4 * (f & rot);
          const float yh = yv[f * row + (r >= row ? r - row : r)];
          if (mode == 3) Yk[base + e] = yh;
          if (mode == 0) {
            Yt[base + e] = yh;
            if (wide) t0v[e] = yh;
            else acc0 += yh * yh;
          } else {
            const float dl = fabsf(logf(yt[j] + kLogEps) - logf(yh + kLogEps)), d = yt[j] - yh;
            if (wide) {
              t0v[e] = dl;
              t1v[e] = d;
            } else {
              acc0 += dl;
              acc1 += d * d;
            }
          }
        }
      }
    }
    if (wide) {
      __syncthreads();
      if ((threadIdx.x & 31) < 4) {
#pragma unroll 4
        for (int e = threadIdx.x >> 5; e < pairs; e += blockDim.x >> 5) {
          const float x0 = t0v[4 * e + mych];
          if (mode == 0) {
            acc0 += x0 * x0;
          } else {
            const float x1 = t1v[4 * e + mych];
            acc0 += x0;
            acc1 += x1 * x1;
          }
        }
      }
    }
    float acc[6];
    {
      const int set = mych < 2 ? 0 : mych - 1;
#pragma unroll
      for (int k = 0; k < 6; ++k) acc[k] = mode == 0 ? (k == set ? acc0 : 0.f) : (k == 2 * set ? acc0 : (k == 2 * set + 1 ? acc1 : 0.f));
    }
    float out[6];
    block_sum<6>(acc, red, out);
    if (threadIdx.x == 0) {
      // partial row: the items of one (song, resolution) cover consecutive groups of R.per frames
      const int row = (t0 - S.first_frame[it.y]) / R.per;
      for (int j = 0; j < 6; ++j) S.lpart[((size_t)it.y * S.lcap + row) * 6 + j] = out[j];
    }
  } else {
  // ---- adjoint ----
  float* dY = reinterpret_cast<float*>(sm + kFrameBuf);   // [nb][nbands][4]
  const float* coef = S.coef + it.y * 6;                    // per set: (alpha / count, alpha / (|Y - Yh| |Y|))
  {
    // item-contiguous band values: entry e of the item is value e of its first frame's row
    const float *yk = Yk + (size_t)t0 * nbands * 4, *yt = Yt + (size_t)t0 * nbands * 4;
    const int ch = threadIdx.x & 3, set = ch < 2 ? 0 : ch - 1;
    const float c0 = coef[2 * set], c1 = coef[2 * set + 1];
#pragma unroll 4
    for (int e = threadIdx.x; e < nb * nbands * 4; e += blockDim.x) {
      const float yh = yk[e], y = yt[e];
      // sign of the difference of the logarithms; 1e-5 apart it is the values' own (logf is good to 2e-6 here)
      const float ph = yh + kLogEps, pt = y + kLogEps;
      float dl = ph - pt;
      if (!(fabsf(dl) > 1e-5f * pt)) dl = logf(ph) - logf(pt);
      const float sg = dl > 0.f ? 1.f : (dl < 0.f ? -1.f : 0.f);
      dY[e] = c0 * sg / ph + c1 * (yh - y);
    }
  }
  __syncthreads();
  // bins -> packed Hermitian spectrum, in place (thread owns the pair k, n - k)
  const int half = n >> 1;
  const float inv_bins = 1.f / (float)(half + 1);   // e / (half + 1) = floor((e + 1/2) inv_bins): e < 2^14
  for (int e = threadIdx.x; e < nb * (half + 1); e += blockDim.x) {
    const int f = (int)((e + 0.5f) * inv_bins), k = e - f * (half + 1);
    float2* Z = sm + f * bs;
    float2 XL, XR;
    bin_spectra(Z, k, n, XL, XR);
    const float* dYf = dY + (size_t)f * nbands * 4;
    float2 gl = make_float2(0.f, 0.f), gr = gl;
    float dmv[4] = {0.f, 0.f, 0.f, 0.f};
    const int qe = R.bin_beg[k + 1];
    for (int q = R.bin_beg[k]; q < qe; ++q) {   // the four channels of a band together
      const float wq = R.bin_w[q];
      const float4 d = reinterpret_cast<const float4*>(dYf)[R.bin_band[q]];
      dmv[0] = fmaf(wq, d.x, dmv[0]);
      dmv[1] = fmaf(wq, d.y, dmv[1]);
      dmv[2] = fmaf(wq, d.z, dmv[2]);
      dmv[3] = fmaf(wq, d.w, dmv[3]);
    }
    const float aw2 = R.aw2[k];
#pragma unroll
    for (int ch = 0; ch < 4; ++ch) {
      const float dm = dmv[ch];
      const float2 X = chan(ch, XL, XR);
      const float mag = sqrtf(aw2 * (X.x * X.x + X.y * X.y) + kMagEps);
      const float2 g = cscale(X, dm * aw2 / mag);
      if (ch == 0) gl = cadd(gl, g);
      else if (ch == 1) gr = cadd(gr, g);
      else if (ch == 2) { gl = cadd(gl, g); gr = cadd(gr, g); }
      else { gl = cadd(gl, g); gr = csub(gr, g); }
    }
    if (k == 0 || k == half) {
      Z[pidx(k)] = make_float2(gl.x, gr.x);
    } else {
      // G_L[k] = gl/2, G_L[n-k] = conj(gl)/2 (same for R); packed P = G_L + i G_R
      Z[pidx(k)] = make_float2(0.5f * (gl.x - gr.y), 0.5f * (gl.y + gr.x));
      Z[pidx(n - k)] = make_float2(0.5f * (gl.x + gr.y), 0.5f * (gr.x - gl.y));
    }
  }
  __syncthreads();
  // the last pass of the inverse writes the windowed frame gradients
  float2* dF = reinterpret_cast<float2*>(S.dF[it.y]) + (size_t)t0 * n;
  const float* win = R.win;
  fft_p_io<true>(sm, R.log_nfft, nb, bs, c.tab.ptw, fftp::SmemIO(),
                 [=](int f, int j, float2 v) { dF[(size_t)f * n + j] = cscale(v, win[j]); });
  }
}

// dmix[c][s] = sum over resolutions and covering frames of dF (overlap-add, fixed order).  One sample per thread, up to
// four frames of every resolution in flight: on short mixes the kernel is latency (four samples per thread in turn, one
// load after the other, before), on long ones the frames' 96 bytes per sample (60 s: 52 us either way).
__global__ void __launch_bounds__(kGatherTile) k_loss_gather(const SongDev* __restrict__ songs,
                                                             const LossRes* __restrict__ resv, int nres,
                                                             const Item* __restrict__ items) {
  const Item it = items[blockIdx.x];
  const SongDev& S = songs[it.proc];
  const int s = it.idx * kGatherTile + threadIdx.x;
  if (s >= S.L) return;
  constexpr int kRes = 3, kFrames = 4;
  float2 v[kRes][kFrames];
  int left[kRes];
  const float2* at[kRes];      // the sample in the first covering frame; the next frame is step further on
  int step[kRes];
#pragma unroll
  for (int r = 0; r < kRes; ++r) {
    left[r] = 0;
    if (r >= nres) continue;
    const LossRes& R = resv[r];
    const int n = R.nfft, hop = R.hop;
    const int tlast = min(S.nframes[r] - 1, s / hop);
    const int tfirst = max(s - n + 1 <= 0 ? 0 : (s - n + hop) / hop, S.first_frame[r]);
    left[r] = max(0, tlast - tfirst + 1);
    at[r] = reinterpret_cast<const float2*>(S.dF[r]) + ((size_t)tfirst * n + (s - tfirst * hop));
    step[r] = n - hop;
#pragma unroll
    for (int f = 0; f < kFrames; ++f)
      if (f < left[r]) v[r][f] = at[r][(size_t)f * step[r]];
  }
  float al = 0.f, ar = 0.f;
#pragma unroll
  for (int r = 0; r < kRes; ++r) {
#pragma unroll
    for (int f = 0; f < kFrames; ++f)
      if (f < left[r]) {
        al += v[r][f].x;
        ar += v[r][f].y;
      }
    for (int f = kFrames; f < left[r]; ++f) {   // hops below a quarter of the transform
      const float2 x = at[r][(size_t)f * step[r]];
      al += x.x;
      ar += x.y;
    }
  }
  S.dmix[s] = al;
  S.dmix[S.ld + s] = ar;
}

void launch_loss_frames(const LaunchCtx& c, const SongDev* songs, const LossRes* res, const int4* items, int n,
                        int mode, int max_dy) {
  if (!n) return;
  const size_t smem = kFrameBuf * sizeof(float2) + (size_t)max_dy * sizeof(float);
  switch (mode) {
    case 0: k_loss_frames<0><<<n, kLossThreads, smem, c.stream>>>(c, songs, res, items); break;
    case 1: k_loss_frames<1><<<n, kLossThreads, smem, c.stream>>>(c, songs, res, items); break;
    case 2: k_loss_frames<2><<<n, kLossThreads, smem, c.stream>>>(c, songs, res, items); break;
    default: k_loss_frames<3><<<n, kLossThreads, smem, c.stream>>>(c, songs, res, items);
  }
}

void launch_loss_gather(const LaunchCtx& c, const SongDev* songs, const LossRes* res, int nres, const Item* items,
                        int n) {
  if (n) k_loss_gather<<<n, kGatherTile, 0, c.stream>>>(songs, res, nres, items);
}

void init_loss_attributes() {
  const int most = kFrameBuf * sizeof(float2) + kLossMaxDy * (int)sizeof(float);
  cudaFuncSetAttribute(k_loss_frames<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  cudaFuncSetAttribute(k_loss_frames<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  cudaFuncSetAttribute(k_loss_frames<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  cudaFuncSetAttribute(k_loss_frames<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
}

}  // namespace mg
