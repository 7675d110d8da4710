// Elementwise processors (gain/panning Eq. 4, stereo imager Eqs. 5-6) fused with the dry/wet blend
// (Eq. 2b), their adjoints, the mix / output sums (Eq. 3) and source ingest (input node i).
// HBM-bound: one read of u and one write of y per sample in the forward pass; one read of dy and u
// and one write of du in the backward pass; float4 accesses on 256-byte aligned planar rows.
#include "mg_fft.cuh"

namespace mg {

__global__ void __launch_bounds__(256) k_gs_fwd(LaunchCtx c, const Item* __restrict__ items) {
  const Item it = items[blockIdx.x];
  const ProcDev& P = c.procs[it.proc];
  const float w = dry_wet_w(c, P.qidx), wd = dry_wet_d(c, P.qidx);
  const float4* ul = reinterpret_cast<const float4*>(P.u);
  const float4* ur = reinterpret_cast<const float4*>(P.u + P.ld);
  float4* yl = reinterpret_cast<float4*>(P.y);
  float4* yr = reinterpret_cast<float4*>(P.y + P.ld);
  const int v0 = it.idx * (c.elem_tile / 4);
  const int vend = min(v0 + c.elem_tile / 4, (P.L + 3) >> 2);
  if (P.type == T_G) {
    const float gl = expf(P.p[0]), gr = expf(P.p[1]);
    for (int v = v0 + threadIdx.x; v < vend; v += blockDim.x) {
      const float4 a = ul[v], b = ur[v];
      float4 oa, ob;
      oa.x = w * (gl * a.x) + wd * a.x; oa.y = w * (gl * a.y) + wd * a.y;
      oa.z = w * (gl * a.z) + wd * a.z; oa.w = w * (gl * a.w) + wd * a.w;
      ob.x = w * (gr * b.x) + wd * b.x; ob.y = w * (gr * b.y) + wd * b.y;
      ob.z = w * (gr * b.z) + wd * b.z; ob.w = w * (gr * b.w) + wd * b.w;
      yl[v] = oa;
      yr[v] = ob;
    }
  } else {  // stereo imager
    const float e = expf(P.p[0]);
    for (int v = v0 + threadIdx.x; v < vend; v += blockDim.x) {
      const float4 a = ul[v], b = ur[v];
      float4 oa, ob;
#define MG_IMG(X)                                         \
  {                                                       \
    const float m = a.X + b.X, s = e * (a.X - b.X);       \
    oa.X = w * ((m + s) * 0.5f) + wd * a.X;        \
    ob.X = w * ((m - s) * 0.5f) + wd * b.X;        \
  }
      MG_IMG(x) MG_IMG(y) MG_IMG(z) MG_IMG(w)
#undef MG_IMG
      yl[v] = oa;
      yr[v] = ob;
    }
  }
}

// Adjoints.  g: du_c = (1-w) dy_c + w e^{p_c} dy_c; partials S_c = sum dy_c u_c give
// dp_c = w e^{p_c} S_c and dw = sum_c (e^{p_c} - 1) S_c.
// s: du from the transposed 2x2 mixing matrix; partial S = sum (u_l - u_r)(dy_l - dy_r) gives
// dp = w e^p S / 2 and dw = (e^p - 1) S / 2.
__global__ void __launch_bounds__(256) k_gs_bwd(LaunchCtx c, const Item* __restrict__ items) {
  __shared__ float red[2 * 32];
  const Item it = items[blockIdx.x];
  const ProcDev& P = c.procs[it.proc];
  const float w = dry_wet_w(c, P.qidx), wd = dry_wet_d(c, P.qidx);
  const float4* ul = reinterpret_cast<const float4*>(P.u);
  const float4* ur = reinterpret_cast<const float4*>(P.u + P.ld);
  const float4* gl4 = reinterpret_cast<const float4*>(P.dy);
  const float4* gr4 = reinterpret_cast<const float4*>(P.dy + P.ld);
  float4* dl = reinterpret_cast<float4*>(P.du);
  float4* dr = reinterpret_cast<float4*>(P.du + P.ld);
  const int v0 = it.idx * (c.elem_tile / 4);
  const int vend = min(v0 + c.elem_tile / 4, (P.L + 3) >> 2);
  float acc[2] = {0.f, 0.f};
  if (P.type == T_G) {
    const float kl = wd + w * expf(P.p[0]), kr = wd + w * expf(P.p[1]);
    for (int v = v0 + threadIdx.x; v < vend; v += blockDim.x) {
      const float4 a = ul[v], b = ur[v], ga = gl4[v], gb = gr4[v];
      acc[0] += ga.x * a.x + ga.y * a.y + ga.z * a.z + ga.w * a.w;
      acc[1] += gb.x * b.x + gb.y * b.y + gb.z * b.z + gb.w * b.w;
      dl[v] = make_float4(kl * ga.x, kl * ga.y, kl * ga.z, kl * ga.w);
      dr[v] = make_float4(kr * gb.x, kr * gb.y, kr * gb.z, kr * gb.w);
    }
  } else {
    const float e = expf(P.p[0]);
    for (int v = v0 + threadIdx.x; v < vend; v += blockDim.x) {
      const float4 a = ul[v], b = ur[v], ga = gl4[v], gb = gr4[v];
      float4 oa, ob;
#define MG_IMGB(X)                                                   \
  {                                                                  \
    const float bl = w * ga.X, br = w * gb.X;                        \
    const float sm = 0.5f * (bl + br), df = 0.5f * e * (bl - br);    \
    oa.X = wd * ga.X + sm + df;                               \
    ob.X = wd * gb.X + sm - df;                               \
    acc[0] += (a.X - b.X) * (ga.X - gb.X);                           \
  }
      MG_IMGB(x) MG_IMGB(y) MG_IMGB(z) MG_IMGB(w)
#undef MG_IMGB
      dl[v] = oa;
      dr[v] = ob;
    }
  }
  float out[2];
  block_sum<2>(acc, red, out);
  if (threadIdx.x == 0) {
    P.bpart[it.idx * kNPart + 0] = out[0];
    P.bpart[it.idx * kNPart + 1] = out[1];
  }
}

// Imager s and gain/pan g right after it in a chain, in one pass over the signal.  Both are bound by HBM: apart they move
// 32 bytes per stereo sample forward and 48 backward, together 24 (y_s is stored for the backward and the scorer) and 24
// (g's input is formed again from s's, and g's input adjoint, a constant times dL/dy per channel, is not stored).
// Forward and backward of 24 tracks x 30 s: 473 -> 291 us.
__device__ __forceinline__ void imager(float w, float wd, float e, float l, float r, float& yl, float& yr) {
  const float m = l + r, s = e * (l - r);
  yl = w * ((m + s) * 0.5f) + wd * l;
  yr = w * ((m - s) * 0.5f) + wd * r;
}

__global__ void __launch_bounds__(256) k_sg_fwd(LaunchCtx c, const Item* __restrict__ items) {
  const Item it = items[blockIdx.x];
  const ProcDev& S = c.procs[it.proc];
  const ProcDev& G = c.procs[S.pair];
  const float ws = dry_wet_w(c, S.qidx), wds = dry_wet_d(c, S.qidx), e = expf(S.p[0]);
  const float wg = dry_wet_w(c, G.qidx), wdg = dry_wet_d(c, G.qidx), gl = expf(G.p[0]), gr = expf(G.p[1]);
  const float4* ul = reinterpret_cast<const float4*>(S.u);
  const float4* ur = reinterpret_cast<const float4*>(S.u + S.ld);
  float4* sl = reinterpret_cast<float4*>(S.y);
  float4* sr = reinterpret_cast<float4*>(S.y + S.ld);
  float4* yl = reinterpret_cast<float4*>(G.y);
  float4* yr = reinterpret_cast<float4*>(G.y + G.ld);
  const int v0 = it.idx * (c.elem_tile / 4);
  const int vend = min(v0 + c.elem_tile / 4, (S.L + 3) >> 2);
  for (int v = v0 + threadIdx.x; v < vend; v += blockDim.x) {
    const float4 a = ul[v], b = ur[v];
    float4 p, q, oa, ob;
#define MG_SG(X)                                                 \
  {                                                              \
    imager(ws, wds, e, a.X, b.X, p.X, q.X);                      \
    oa.X = wg * (gl * p.X) + wdg * p.X;                          \
    ob.X = wg * (gr * q.X) + wdg * q.X;                          \
  }
    MG_SG(x) MG_SG(y) MG_SG(z) MG_SG(w)
#undef MG_SG
    sl[v] = p;
    sr[v] = q;
    yl[v] = oa;
    yr[v] = ob;
  }
}

__global__ void __launch_bounds__(256) k_sg_bwd(LaunchCtx c, const Item* __restrict__ items) {
  __shared__ float red[3 * 32];
  const Item it = items[blockIdx.x];
  const ProcDev& S = c.procs[it.proc];
  const ProcDev& G = c.procs[S.pair];
  const float ws = dry_wet_w(c, S.qidx), wds = dry_wet_d(c, S.qidx), e = expf(S.p[0]);
  const float wg = dry_wet_w(c, G.qidx), wdg = dry_wet_d(c, G.qidx);
  const float kl = wdg + wg * expf(G.p[0]), kr = wdg + wg * expf(G.p[1]);
  const float4* ul = reinterpret_cast<const float4*>(S.u);
  const float4* ur = reinterpret_cast<const float4*>(S.u + S.ld);
  const float4* gl4 = reinterpret_cast<const float4*>(G.dy);
  const float4* gr4 = reinterpret_cast<const float4*>(G.dy + G.ld);
  float4* dl = reinterpret_cast<float4*>(S.du);
  float4* dr = reinterpret_cast<float4*>(S.du + S.ld);
  const int v0 = it.idx * (c.elem_tile / 4);
  const int vend = min(v0 + c.elem_tile / 4, (S.L + 3) >> 2);
  float acc[3] = {0.f, 0.f, 0.f};
  for (int v = v0 + threadIdx.x; v < vend; v += blockDim.x) {
    const float4 a = ul[v], b = ur[v], ga = gl4[v], gb = gr4[v];
    float4 p, q, oa, ob;
#define MG_SG(X) imager(ws, wds, e, a.X, b.X, p.X, q.X);
    MG_SG(x) MG_SG(y) MG_SG(z) MG_SG(w)
#undef MG_SG
    acc[0] += ga.x * p.x + ga.y * p.y + ga.z * p.z + ga.w * p.w;
    acc[1] += gb.x * q.x + gb.y * q.y + gb.z * q.z + gb.w * q.w;
#define MG_SGB(X)                                                    \
  {                                                                  \
    const float hl = kl * ga.X, hr = kr * gb.X;                      \
    const float bl = ws * hl, br = ws * hr;                          \
    const float sm = 0.5f * (bl + br), df = 0.5f * e * (bl - br);    \
    oa.X = wds * hl + sm + df;                                       \
    ob.X = wds * hr + sm - df;                                       \
    acc[2] += (a.X - b.X) * (hl - hr);                               \
  }
    MG_SGB(x) MG_SGB(y) MG_SGB(z) MG_SGB(w)
#undef MG_SGB
    dl[v] = oa;
    dr[v] = ob;
  }
  float out[3];
  block_sum<3>(acc, red, out);
  if (threadIdx.x == 0) {
    G.bpart[it.idx * kNPart + 0] = out[0];
    G.bpart[it.idx * kNPart + 1] = out[1];
    S.bpart[it.idx * kNPart + 0] = out[2];
    S.bpart[it.idx * kNPart + 1] = 0.f;
    if (it.idx == 0) {
      G.stats[kStatPairGain] = kl;
      G.stats[kStatPairGain + 1] = kr;
    }
  }
}

// Eq. (3) sums: out[s] = sum over its inputs (mix node m and output node o), in input order.  A thread makes one quad of
// one channel (blockIdx.y: channel and 1,024-sample part of the tile) with the loads of eight inputs together: with
// four quads of both channels per thread, one input after the other, the output sum of 5 chains x 10 s took 16 us on 108
// CTAs; now 8 (24 tracks x 30 s are at HBM rate either way, 52 us).
__global__ void __launch_bounds__(256) k_sum(float* const* outs, const float* const* ins, const int* in_beg,
                                             const int* Ls, const int* lds, const Item* items, int tile) {
  const Item it = items[blockIdx.x];
  const int s = it.proc, L = Ls[s], ld = lds[s];
  const int beg = in_beg[s], end = in_beg[s + 1];
  const int v = it.idx * (tile / 4) + (blockIdx.y >> 1) * 256 + threadIdx.x;
  if (v >= (L + 3) >> 2) return;
  const int64_t o = (int64_t)(blockIdx.y & 1) * ld;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  constexpr int kAhead = 8;
  for (int j0 = beg; j0 < end; j0 += kAhead) {
    float4 a[kAhead];
#pragma unroll
    for (int j = 0; j < kAhead; ++j)
      if (j0 + j < end) a[j] = reinterpret_cast<const float4*>(ins[j0 + j] + o)[v];
#pragma unroll
    for (int j = 0; j < kAhead; ++j)
      if (j0 + j < end) {
        acc.x += a[j].x; acc.y += a[j].y; acc.z += a[j].z; acc.w += a[j].w;
      }
  }
  reinterpret_cast<float4*>(outs[s] + o)[v] = acc;
}

__global__ void k_ingest(const float* __restrict__ mono, float* __restrict__ st, int L, int ld) {
  for (int n = blockIdx.x * blockDim.x + threadIdx.x; n < L; n += gridDim.x * blockDim.x) {
    const float x = mono[n];
    st[n] = x;
    st[ld + n] = x;
  }
}

// All K mono sources of one song ([K][L], device-readable: device memory or mapped pinned host memory) into
// both rows of their tracks' input buffers, one launch: blockIdx.y is the track.
__global__ void k_ingest_song(const float* __restrict__ mono, float* const* __restrict__ dst, int L, int ld) {
  const float* src = mono + (size_t)blockIdx.y * L;
  float* st = dst[blockIdx.y];
  for (int n = blockIdx.x * blockDim.x + threadIdx.x; n < L; n += gridDim.x * blockDim.x) {
    const float x = src[n];
    st[n] = x;
    st[ld + n] = x;
  }
}

// Mixes to the caller's rows, which may start at any sample: four samples of both channels of a thread in flight.
constexpr int kCopyPer = 4;
__global__ void __launch_bounds__(256) k_copy_mix(const SongDev* songs, int nsongs, float* out, const int64_t* offs) {
  const int s = blockIdx.y;
  const SongDev& S = songs[s];
  const int L = S.L, ld = S.ld, step = gridDim.x * blockDim.x;
  const float* mix = S.mix;
  float* o = out + offs[s];
  for (int n0 = blockIdx.x * blockDim.x + threadIdx.x; n0 < L; n0 += kCopyPer * step) {
    float a[kCopyPer], b[kCopyPer];
#pragma unroll
    for (int j = 0; j < kCopyPer; ++j)
      if (n0 + (int64_t)j * step < L) {
        a[j] = mix[n0 + j * step];
        b[j] = mix[ld + n0 + j * step];
      }
#pragma unroll
    for (int j = 0; j < kCopyPer; ++j)
      if (n0 + (int64_t)j * step < L) {
        o[n0 + j * step] = a[j];
        o[L + n0 + j * step] = b[j];
      }
  }
}

void launch_gs_fwd(const LaunchCtx& c, const Item* items, int n) {
  if (n) k_gs_fwd<<<n, 256, 0, c.stream>>>(c, items);
}
void launch_gs_bwd(const LaunchCtx& c, const Item* items, int n) {
  if (n) k_gs_bwd<<<n, 256, 0, c.stream>>>(c, items);
}
void launch_sg_fwd(const LaunchCtx& c, const Item* items, int n) {
  if (n) k_sg_fwd<<<n, 256, 0, c.stream>>>(c, items);
}
void launch_sg_bwd(const LaunchCtx& c, const Item* items, int n) {
  if (n) k_sg_bwd<<<n, 256, 0, c.stream>>>(c, items);
}
void launch_sum(cudaStream_t st, float* const* outs, const float* const* ins, const int* in_beg, const int* L,
                const int* ld, const Item* items, int n, int tile) {
  if (n) k_sum<<<dim3(n, 2 * (tile / 1024)), 256, 0, st>>>(outs, ins, in_beg, L, ld, items, tile);   // tile: 1,024 m
}
void launch_ingest(cudaStream_t st, const float* mono, float* stereo, int L, int ld) {
  k_ingest<<<min(1024, (L + 255) / 256), 256, 0, st>>>(mono, stereo, L, ld);
}
void launch_ingest_song(cudaStream_t st, const float* mono, float* const* dst, int K, int L, int ld) {
  if (K > 0 && L > 0) k_ingest_song<<<dim3(std::min(256, (L + 255) / 256), K), 256, 0, st>>>(mono, dst, L, ld);
}
void launch_copy_mix(cudaStream_t st, const SongDev* songs, int nsongs, float* out, const int64_t* offs) {
  if (nsongs) k_copy_mix<<<dim3(256, nsongs), 256, 0, st>>>(songs, nsongs, out, offs);
}

}  // namespace mg
