// Equalizer (Sec. 3.3, Eqs. 7-8) by single-pass overlap-save in shared memory.
// The 2047-tap zero-phase FIR is short against an 8192-point FFT, so every block of B = 6146 output samples is
// computed by one CTA from its input segment [s0 - 1023, s0 + B + 1023) without any global FFT scratch:
//   forward:  segment -> FFT -> x H -> IFFT -> B valid outputs, fused with the dry/wet blend and the L_g
//             energies; the wet signal y_bar is kept for the backward;
//   backward: per block D = FFT(dL/dy_bar on the segment) with dL/dy_bar = w dy + c1 y_bar_mid from the kept y_bar,
//             Ub = FFT(u on the block only), du = IFFT(D H) on the block (h is even, so the correlation adjoint is
//             the same convolution).
//             dL/dh[j] = sum_n dL/dy_bar[n] u[n - j] = sum_m u[m] dL/dy_bar[m + j] is split over the blocks by the
//             input position m: a block contributes IFFT(D conj(Ub)) at lags |j| <= 1023 (m + j stays inside the
//             segment, no wrap-around), so the segment spectrum D serves both gradients.  The blocks' spectra are
//             added per node in a fixed order and one inverse FFT gives dL/dh at lags -1023..1023 summed over both
//             channels.
// H is real (h real and even); both channels travel packed as one complex signal.
#include "mg_fftp.cuh"

namespace mg {

namespace {
constexpr int kOsLog = 13;
constexpr int kOsM = 1 << kOsLog;
constexpr int kOsThreads = 512;
constexpr int kOsP = pstride(kOsM);   // padded buffer stride
}  // namespace

// Spectrum of the FIR on the 8192-point grid: one CTA per node.
__global__ void __launch_bounds__(kOsThreads) k_eq_spec(LaunchCtx c, const int* __restrict__ procs) {
  extern __shared__ float2 sm[];
  const ProcDev& P = c.procs[procs[blockIdx.x]];
  for (int j = threadIdx.x; j < kOsM; j += blockDim.x) {
    // tap time n = j for j < 1024, n = j - M for j > M - 1024 (circular placement of n in [-1023, 1023])
    int n = j < kOsM / 2 ? j : j - kOsM;
    float v = 0.f;
    if (n >= -kEqHalf && n <= kEqHalf) v = P.taps[n + kEqHalf];
    sm[pidx(j)] = make_float2(v, 0.f);
  }
  __syncthreads();
  fft_p<false>(sm, kOsLog, 1, kOsP, c.tab.ptw);
  for (int k = threadIdx.x; k < kOsM; k += blockDim.x) P.hspec[k] = sm[pidx(k)].x;
}

// item = (node, block): outputs [s0, s0 + 6146).
__global__ void __launch_bounds__(kOsThreads, 2) k_eq_os_fwd(LaunchCtx c, const Item* __restrict__ items) {
  extern __shared__ float2 sm[];
  __shared__ float red[2 * 32];
  const Item it = items[blockIdx.x];
  const ProcDev& P = c.procs[it.proc];
  constexpr int B = kOsM - 2 * kEqHalf;
  const int s0 = it.idx * B, seg = s0 - kEqHalf, L = P.L, ld = P.ld;
  const float* u = P.u;
  // the segment goes straight from global memory into the first pass of the transform
  fft_p_io<false>(sm, kOsLog, 1, kOsP, c.tab.ptw, [=](int, int j) {
    const int s = seg + j;
    return (s >= 0 && s < L) ? make_float2(u[s], u[ld + s]) : make_float2(0.f, 0.f);
  });
  for (int k = threadIdx.x; k < kOsM; k += blockDim.x) sm[pidx(k)] = cscale(sm[pidx(k)], P.hspec[k]);
  __syncthreads();
  const float w = dry_wet_w(c, P.qidx), wd = dry_wet_d(c, P.qidx);
  const float inv = 1.f / kOsM;
  float acc[2] = {0.f, 0.f};
  float* ybar = P.ybar;
  float* y = P.y;
  // the last pass of the inverse writes the B valid outputs, blended with the dry signal
  fft_p_io<true>(sm, kOsLog, 1, kOsP, c.tab.ptw, fftp::SmemIO(), [&](int, int j, float2 v) {
    const int t = j - kEqHalf, s = s0 + t;
    if (t < 0 || t >= B || s >= L) return;
    const float2 yb = cscale(v, inv);
    ybar[s] = yb.x;
    ybar[ld + s] = yb.y;
    const float ul = u[s], ur = u[ld + s];
    y[s] = w * yb.x + wd * ul;
    y[ld + s] = w * yb.y + wd * ur;
    const float ym = yb.x + yb.y, um = ul + ur;
    acc[0] += ym * ym;
    acc[1] += um * um;
  });
  float out[2];
  block_sum<2>(acc, red, out);
  if (threadIdx.x == 0) {
    P.fpart[it.idx * kNPart + 0] = out[0];
    P.fpart[it.idx * kNPart + 1] = out[1];
  }
}

// item = (node, block): everything the backward does with one block of B = 6146 samples, in one 70 KB buffer.
//   Ub = FFT(u on the block only)                 -> the block's row of eqg (read back below, from L2)
//   D  = FFT(dL/dy_bar on the segment)            -> shared memory; accumulates dL/dw of the block
//   Y[k] = (X[k] + conj X[-k]) / 2, X = D conj(Ub) -> over Ub's row, bins 0..4096 (bin 4096 in the imaginary part of
//                                                    bin 0): the spectrum of the real part of IFFT(X), which is the
//                                                    tap gradient of both channels, so half the bins are enough
//   du = IFFT(D H) on the block plus the dry path and the loudness-gain term (h even: the adjoint of the
//   convolution is the same convolution).
// A CTA per block keeps two CTAs on every SM from the shortest signal on.  With eight blocks per CTA one after the
// other (and du in a second kernel that read D H back) a launch took 142 us whenever it had fewer items than SMs.
__global__ void __launch_bounds__(kOsThreads, 2) k_eq_os_bwd(LaunchCtx c, const Item* __restrict__ items) {
  extern __shared__ float2 sm[];
  __shared__ float red[32];
  const Item it = items[blockIdx.x];
  const ProcDev& P = c.procs[it.proc];
  constexpr int B = kOsM - 2 * kEqHalf;   // 6146
  float2* g = P.eqg + (size_t)it.idx * kOsM;
  const int s0 = it.idx * B, seg = s0 - kEqHalf, L = P.L, ld = P.ld;
  const float *u = P.u, *ybar = P.ybar, *dy = P.dy;
  fft_p_io<false>(sm, kOsLog, 1, kOsP, c.tab.ptw, [=](int, int j) {
    const int t = j - kEqHalf, s = s0 + t;
    return (t >= 0 && t < B && s < L) ? make_float2(u[s], u[ld + s]) : make_float2(0.f, 0.f);
  }, [=](int, int k, float2 v) { g[k] = v; });
  __syncthreads();   // the buffer is free, and the spectrum in g visible to the block
  float dwacc[1] = {0.f};
  {
    const float w = dry_wet_w(c, P.qidx);
    const float c1 = P.stats[2];
    fft_p_io<false>(sm, kOsLog, 1, kOsP, c.tab.ptw, [&](int, int j) {
      const int s = seg + j;
      if (s < 0 || s >= L) return make_float2(0.f, 0.f);
      const float yl = ybar[s], yr = ybar[ld + s];
      const float gl = dy[s], gr = dy[ld + s];
      const float gm = c1 * (yl + yr);
      if (j >= kEqHalf && j < kEqHalf + B) dwacc[0] += gl * (yl - u[s]) + gr * (yr - u[ld + s]);
      return make_float2(w * gl + gm, w * gr + gm);
    });
  }
  // bins k and -k belong to one thread: it reads both of Ub before it writes Y[k] over them
  const float* hs = P.hspec;
  constexpr int kPer = 4;
#pragma unroll 1
  for (int k0 = threadIdx.x; k0 < kOsM / 2; k0 += kPer * kOsThreads) {
    float2 ua[kPer], ub[kPer];
    float ha[kPer], hb[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      const int k = k0 + j * kOsThreads, m = k ? kOsM - k : kOsM / 2;   // the thread of bin 0 takes bin 4096 along
      ua[j] = g[k];
      ub[j] = g[m];
      ha[j] = hs[k];
      hb[j] = hs[m];
    }
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      const int k = k0 + j * kOsThreads, m = k ? kOsM - k : kOsM / 2;
      const float2 a = sm[pidx(k)], b = sm[pidx(m)];
      const float2 xa = cmulc(a, ua[j]), xb = cmulc(b, ub[j]);
      g[k] = k ? make_float2(0.5f * (xa.x + xb.x), 0.5f * (xa.y - xb.y)) : make_float2(xa.x, xb.x);
      sm[pidx(k)] = cscale(a, ha[j]);
      sm[pidx(m)] = cscale(b, hb[j]);
    }
  }
  float out[1];
  block_sum<1>(dwacc, red, out);   // also the barrier before the transform
  if (threadIdx.x == 0) P.bpart[it.idx * kNPart] = out[0];
  fft_p<true>(sm, kOsLog, 1, kOsP, c.tab.ptw);
  const float wd = dry_wet_d(c, P.qidx), c2 = P.stats[3];
  const float inv = 1.f / kOsM;
  // two samples per thread and step (s0 is even, the rows are 256-byte aligned), the loads of four steps together
  float* du = P.du;
  constexpr int kPairs = B / 2, kBatch = 4;
  for (int q0 = threadIdx.x; q0 < kPairs; q0 += kBatch * kOsThreads) {
    float2 gl[kBatch], gr[kBatch], ul[kBatch], ur[kBatch];
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      const int q = q0 + j * kOsThreads, s = s0 + 2 * q;
      if (q < kPairs && s < L) {   // the row stride is even: the sample after an odd length's last one is padding
        gl[j] = *reinterpret_cast<const float2*>(dy + s);
        gr[j] = *reinterpret_cast<const float2*>(dy + ld + s);
        ul[j] = *reinterpret_cast<const float2*>(u + s);
        ur[j] = *reinterpret_cast<const float2*>(u + ld + s);
      }
    }
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      const int q = q0 + j * kOsThreads, s = s0 + 2 * q;
      if (q >= kPairs || s >= L) continue;
      const float2 d0 = cscale(sm[pidx(kEqHalf + 2 * q)], inv), d1 = cscale(sm[pidx(kEqHalf + 2 * q + 1)], inv);
      const float u0 = c2 * (ul[j].x + ur[j].x), u1 = c2 * (ul[j].y + ur[j].y);
      const float2 l = make_float2(wd * gl[j].x + d0.x + u0, wd * gl[j].y + d1.x + u1);
      const float2 r = make_float2(wd * gr[j].x + d0.y + u0, wd * gr[j].y + d1.y + u1);
      if (s + 1 < L) {
        *reinterpret_cast<float2*>(du + s) = l;
        *reinterpret_cast<float2*>(du + ld + s) = r;
      } else {
        du[s] = l.x;
        du[ld + s] = r.x;
      }
    }
  }
}

// Sum over a node's blocks of the half spectra Y (see k_eq_os_bwd): 64 bins per CTA as 32 pairs, the blocks split over
// eight groups of threads, each adding its blocks in order with eight loads in flight, the groups added in order.
// The sum goes over the first block's row.
constexpr int kDhSlice = 64, kDhGroups = 8;
__global__ void __launch_bounds__(32 * kDhGroups) k_eq_dh_sum(LaunchCtx c, const int* __restrict__ procs) {
  __shared__ float4 part[kDhGroups][32];
  const ProcDev& P = c.procs[procs[blockIdx.x]];
  const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5, n = P.nbpart;
  const size_t row = kOsM / 2;   // a row of eqg in float4
  float4* src = reinterpret_cast<float4*>(P.eqg) + blockIdx.y * (kDhSlice / 2) + lane;
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  constexpr int kBatch = 8;
  for (int b0 = grp; b0 < n; b0 += kBatch * kDhGroups) {
    float4 v[kBatch];
#pragma unroll
    for (int j = 0; j < kBatch; ++j)
      if (b0 + j * kDhGroups < n) v[j] = src[(size_t)(b0 + j * kDhGroups) * row];
#pragma unroll
    for (int j = 0; j < kBatch; ++j)
      if (b0 + j * kDhGroups < n) s = make_float4(s.x + v[j].x, s.y + v[j].y, s.z + v[j].z, s.w + v[j].w);
  }
  part[grp][lane] = s;
  __syncthreads();
  if (grp == 0) {
#pragma unroll
    for (int j = 1; j < kDhGroups; ++j) {
      const float4 p = part[j][lane];
      s = make_float4(s.x + p.x, s.y + p.y, s.z + p.z, s.w + p.w);
    }
    src[0] = s;
  }
}

// dL/dh (both channels summed into row 0, row 1 zero): one inverse FFT of the summed spectrum, lags n = -1023..1023
// at circular positions n mod 8192.
__global__ void __launch_bounds__(kOsThreads) k_eq_dh_taps(LaunchCtx c, const int* __restrict__ procs) {
  extern __shared__ float2 sm[];
  const ProcDev& P = c.procs[procs[blockIdx.x]];
  const float2* y = P.eqg;
  fft_p_io<true>(sm, kOsLog, 1, kOsP, c.tab.ptw, [=](int, int k) {
    const float2 v = y[k <= kOsM / 2 ? k & (kOsM / 2 - 1) : kOsM - k];
    if ((k & (kOsM / 2 - 1)) == 0) return make_float2(k ? v.y : v.x, 0.f);
    return k < kOsM / 2 ? v : cconj(v);
  });
  const float inv = 1.f / kOsM;
  for (int j = threadIdx.x; j < kEqTaps; j += blockDim.x) {
    P.dtaps[j] = sm[pidx((j - kEqHalf) & (kOsM - 1))].x * inv;
    P.dtaps[P.Nh + j] = 0.f;
  }
}

void launch_eq_spec(const LaunchCtx& c, const int* procs, int n) {
  if (n) k_eq_spec<<<n, kOsThreads, kOsP * sizeof(float2), c.stream>>>(c, procs);
}
void launch_eq_os_fwd(const LaunchCtx& c, const Item* items, int n) {
  if (n) k_eq_os_fwd<<<n, kOsThreads, kOsP * sizeof(float2), c.stream>>>(c, items);
}
void launch_eq_os_bwd(const LaunchCtx& c, const Item* items, int n) {
  if (n) k_eq_os_bwd<<<n, kOsThreads, kOsP * sizeof(float2), c.stream>>>(c, items);
}
void launch_eq_dh_reduce(const LaunchCtx& c, const int* procs, int n) {
  if (!n) return;
  k_eq_dh_sum<<<dim3(n, kOsM / 2 / kDhSlice), 32 * kDhGroups, 0, c.stream>>>(c, procs);
  k_eq_dh_taps<<<n, kOsThreads, kOsP * sizeof(float2), c.stream>>>(c, procs);
}
void init_eqos_attributes() {
  cudaFuncSetAttribute(k_eq_spec, cudaFuncAttributeMaxDynamicSharedMemorySize, kOsP * (int)sizeof(float2));
  cudaFuncSetAttribute(k_eq_os_fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, kOsP * (int)sizeof(float2));
  cudaFuncSetAttribute(k_eq_os_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, kOsP * (int)sizeof(float2));
  cudaFuncSetAttribute(k_eq_dh_taps, cudaFuncAttributeMaxDynamicSharedMemorySize, kOsP * (int)sizeof(float2));
}

}  // namespace mg
