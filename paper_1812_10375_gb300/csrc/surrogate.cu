// Training and inference kernels of the sweep surrogate (include/hlb_surrogate.h).
// Small FP32 network: three strided conv1d layers over the early wall-flux
// history, mean pooling, and a three-layer MLP.  Batches are at most a few
// hundred samples, so plain SIMT kernels (shared-memory tiled for the linear
// layers) are used; every step of forward, backward and Adam runs here.
#include <math.h>
#include <stdint.h>

#include "hlb_surrogate.h"

#include <cuda_runtime.h>

namespace {

struct Dims {
  int L0, C1, C2, C3, K, S, NS, H, NOUT, L1, L2, L3;
};

bool dims_of(const hlb_sur_config* c, Dims* d) {
  if (!c) return false;
  if (c->L0 < 1 || c->C1 < 1 || c->C2 < 1 || c->C3 < 1 || c->K < 1 || c->S < 1 || c->NS < 0 || c->H < 1 ||
      c->NOUT < 2)
    return false;
  d->L0 = c->L0; d->C1 = c->C1; d->C2 = c->C2; d->C3 = c->C3; d->K = c->K; d->S = c->S;
  d->NS = c->NS; d->H = c->H; d->NOUT = c->NOUT;
  if (c->L0 < c->K) return false;
  d->L1 = (c->L0 - c->K) / c->S + 1;
  if (d->L1 < c->K) return false;
  d->L2 = (d->L1 - c->K) / c->S + 1;
  if (d->L2 < c->K) return false;
  d->L3 = (d->L2 - c->K) / c->S + 1;
  return true;
}

struct Offsets {  // parameter offsets (floats)
  size_t W1, b1, W2, b2, W3, b3, F1, c1, F2, c2, F3, c3, total;
};

Offsets param_offsets(const Dims& d) {
  Offsets o;
  size_t p = 0;
  o.W1 = p; p += (size_t)d.C1 * d.K;
  o.b1 = p; p += d.C1;
  o.W2 = p; p += (size_t)d.C2 * d.C1 * d.K;
  o.b2 = p; p += d.C2;
  o.W3 = p; p += (size_t)d.C3 * d.C2 * d.K;
  o.b3 = p; p += d.C3;
  o.F1 = p; p += (size_t)d.H * (d.C3 + d.NS);
  o.c1 = p; p += d.H;
  o.F2 = p; p += (size_t)d.H * d.H;
  o.c2 = p; p += d.H;
  o.F3 = p; p += (size_t)d.NOUT * d.H;
  o.c3 = p; p += d.NOUT;
  o.total = p;
  return o;
}

size_t al(size_t n) { return (n + 63) & ~(size_t)63; }  // 256-byte aligned float counts

// What the per-sample kernels (below) need of a network.
constexpr int SK = 5, SS = 2, ST = 512;  // taps, stride, threads

template <class I>
struct SampleLayout {  // shared-memory offsets (floats); rows of odd length
  I s1, s2, s3, p2, p3;
  I x, w1, wt2, wt3, a1, a2, a3, d2, d1, h0, a4, a5, z, g, total;
};

// I = int for networks that fit, whose sums do.
template <class I>
__host__ __device__ inline SampleLayout<I> sample_layout(const Dims& d, bool train) {
  SampleLayout<I> L;
  L.s1 = d.L1 | 1;
  L.s2 = d.L2 | 1;
  L.s3 = d.L3 | 1;
  L.p2 = (d.C2 + 7) & ~7;
  L.p3 = (d.C3 + 7) & ~7;
  I o = 0;
  auto take = [&](I n) {
    const I at = o;
    o += (n + 3) & ~3;
    return at;
  };
  L.wt2 = take((I)d.C1 * SK * L.p2);
  L.wt3 = take((I)d.C2 * SK * L.p3);
  L.x = take(d.L0);
  L.w1 = take((I)d.C1 * SK);
  L.a1 = take(d.C1 * L.s1);
  L.a2 = take(d.C2 * L.s2);
  L.a3 = take(d.C3 * L.s3);
  L.d2 = train ? take(d.C2 * L.s2) : o;
  L.d1 = train ? take(d.C1 * L.s1) : o;
  L.h0 = take((I)d.C3 + d.NS);
  L.a4 = take(d.H);
  L.a5 = take(d.H);
  L.z = take(d.NOUT > d.H ? d.NOUT : d.H);
  const int widest = d.H > d.C3 + d.NS ? d.H : d.C3 + d.NS;
  L.g = train ? take(4 * ST > widest ? 4 * ST : widest) : o;
  L.total = o;
  return L;
}

constexpr int SAMPLE_SMEM = 200 * 1024;

bool sample_fits(const Dims& d, bool train) {
  if (d.K != SK || d.S != SS) return false;
  // every size is at least an array's; after that no product leaves 64 bits
  constexpr int MOST = SAMPLE_SMEM / (int)sizeof(float);
  for (const int n : {d.L0, d.C1, d.C2, d.C3, d.NS, d.H, d.NOUT})
    if (n > MOST) return false;
  return sample_layout<long long>(d, train).total <= MOST;
}

// Whether a call runs by samples.  One CTA reads all linear weights for one sample and
// stages all convolution weights: that pays while the linear layers are narrow and,
// for many samples, the convolutions long.  Layers' time over samples' time on either
// side of the lines (conv, lin: multiply-adds of a sample; channels 16/32/32 unless
// short: conv = 4k):
//  - training, lin: 1 sample, H = 1024 1.00, H = 1280 0.61; 256 samples, lin = 7 conv 1.39,
//    15 conv 0.92.  4,096 samples, short: H = 512 1.00, H = 768 0.86.
//  - training, rows of F2 that are not whole 16-byte pieces (read by 4 bytes): 153
//    samples, H = 256 1.52, H = 512 0.74.
//  - forward, lin: 1 sample, H = 1280 1.31 (short 1.23), H = 2048 0.97 (0.76); 64 samples,
//    H = 2048 1.52 (1.28), 153 samples, short, H = 3072 0.99.
//  - forward, conv: 1,024 samples, 106k 1.10, short 0.86; 4,096 samples, 306k 1.58,
//    106k 0.83.
//  - forward, NOUT = 1000 1.59, 8,000 0.59.
constexpr int SAMPLE_BATCH = 512;
bool by_samples(const Dims& d, int B, bool train) {
  if (!sample_fits(d, train)) return false;
  const long long conv = (long long)SK * (d.C1 * d.L1 + (long long)d.C1 * d.C2 * d.L2 + (long long)d.C2 * d.C3 * d.L3);
  const long long lin = (long long)d.H * (d.C3 + d.NS + d.H + d.NOUT);
  const bool whole = d.H % 4 == 0 && param_offsets(d).F2 % 4 == 0, many = B > SAMPLE_BATCH;
  if (!train) {
    if (d.NOUT > 1024 || (many && conv < 100000) || (B > 2 * SAMPLE_BATCH && conv < 300000)) return false;
    return lin <= 1700000 || (B >= 64 && lin <= 5000000 && whole);
  }
  if (!whole) return lin <= 80000 && !(many && conv < 100000);
  if (many && conv < 100000) return lin <= 300000;
  return lin <= 1100000 || (B >= 256 && lin <= 8 * conv);
}

struct Acts {  // workspace offsets (floats)
  size_t z1, a1, z2, a2, z3, a3, h0, z4, a4, z5, a5, y, dy, dz5, dz4, dh0, dz3, dz2, dz1, loss, part, total;
};

Acts act_offsets(const Dims& d, int B) {
  Acts a;
  size_t p = 0;
  const size_t n1 = (size_t)B * d.C1 * d.L1, n2 = (size_t)B * d.C2 * d.L2, n3 = (size_t)B * d.C3 * d.L3;
  const size_t nh0 = (size_t)B * (d.C3 + d.NS), nh = (size_t)B * d.H, ny = (size_t)B * d.NOUT;
  a.z1 = p; p += al(n1);
  a.a1 = p; p += al(n1);
  a.z2 = p; p += al(n2);
  a.a2 = p; p += al(n2);
  a.z3 = p; p += al(n3);
  a.a3 = p; p += al(n3);
  a.h0 = p; p += al(nh0);
  a.z4 = p; p += al(nh);
  a.a4 = p; p += al(nh);
  a.z5 = p; p += al(nh);
  a.a5 = p; p += al(nh);
  a.y = p; p += al(ny);
  a.dy = p; p += al(ny);
  a.dz5 = p; p += al(nh);
  a.dz4 = p; p += al(nh);
  a.dh0 = p; p += al(nh0);
  a.dz3 = p; p += al(n3);
  a.dz2 = p; p += al(n2);
  a.dz1 = p; p += al(n1);
  // by samples: a pair of loss terms and the convolutions' partial gradients of each.  (A
  // workspace for B serves every smaller batch; one beyond SAMPLE_BATCH may run by
  // layers where those up to it run by samples.)
  const int most = by_samples(d, B, true) ? B : B < SAMPLE_BATCH ? B : SAMPLE_BATCH;
  const bool samples = by_samples(d, most, true);
  a.loss = p; p += al(samples ? 2 * (size_t)most : 2);
  a.part = p; p += samples ? al((size_t)most * param_offsets(d).F1) : 0;
  a.total = p;
  return a;
}

// z[b,o,t] = bias[o] + sum_{c,k} W[o,c,k] x[b,c,S t + k];  a = max(z, 0)
__global__ void k_conv_fwd(const float* __restrict__ x, int Cin, int Lin, const float* __restrict__ W,
                           const float* __restrict__ bias, int Cout, int K, int S, int Lout, int B,
                           float* __restrict__ z, float* __restrict__ a) {
  const long long n = (long long)B * Cout * Lout;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const int t = (int)(e % Lout);
    const int o = (int)((e / Lout) % Cout);
    const int b = (int)(e / ((long long)Lout * Cout));
    float s = bias[o];
    const float* xb = x + (long long)b * Cin * Lin + (long long)S * t;
    const float* wo = W + (long long)o * Cin * K;
    for (int c = 0; c < Cin; ++c)
      for (int k = 0; k < K; ++k) s += wo[c * K + k] * xb[(long long)c * Lin + k];
    z[e] = s;
    a[e] = fmaxf(s, 0.f);
  }
}

// dx[b,c,u] = sum over (o, k, t) with S t + k = u of W[o,c,k] dz[b,o,t]; times (zprev > 0)
__global__ void k_conv_bwd_data(const float* __restrict__ dz, const float* __restrict__ W, int B, int Cin, int Lin,
                                int Cout, int K, int S, int Lout, const float* __restrict__ zprev,
                                float* __restrict__ dx) {
  const long long n = (long long)B * Cin * Lin;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const int u = (int)(e % Lin);
    const int c = (int)((e / Lin) % Cin);
    const int b = (int)(e / ((long long)Lin * Cin));
    float s = 0.f;
    for (int k = 0; k < K; ++k) {
      const int v = u - k;
      if (v < 0 || v % S != 0) continue;
      const int t = v / S;
      if (t >= Lout) continue;
      for (int o = 0; o < Cout; ++o) s += W[((long long)o * Cin + c) * K + k] * dz[((long long)b * Cout + o) * Lout + t];
    }
    dx[e] = zprev ? (zprev[e] > 0.f ? s : 0.f) : s;
  }
}

template <int NT>
__device__ __forceinline__ float block_sum(float v) {
  __shared__ float red[NT / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float t = 0.f;
  if (threadIdx.x == 0)
    for (int w = 0; w < NT / 32; ++w) t += red[w];
  return t;
}

// One block per weight (o, c, k): dW = sum_{b,t} dz[b,o,t] x[b,c,S t + k];
// the last Cout blocks compute db[o] = sum_{b,t} dz[b,o,t].
__global__ void __launch_bounds__(256) k_conv_bwd_w(const float* __restrict__ dz, const float* __restrict__ x, int B,
                                                    int Cin, int Lin, int Cout, int K, int S, int Lout,
                                                    float* __restrict__ dW, float* __restrict__ db) {
  const int nw = Cout * Cin * K;
  const int id = blockIdx.x;
  const long long n = (long long)B * Lout;
  float s = 0.f;
  if (id < nw) {
    const int k = id % K, c = (id / K) % Cin, o = id / (K * Cin);
    for (long long e = threadIdx.x; e < n; e += blockDim.x) {
      const int t = (int)(e % Lout), b = (int)(e / Lout);
      s += dz[((long long)b * Cout + o) * Lout + t] * x[((long long)b * Cin + c) * Lin + (long long)S * t + k];
    }
    s = block_sum<256>(s);
    if (threadIdx.x == 0) dW[id] = s;
  } else {
    const int o = id - nw;
    for (long long e = threadIdx.x; e < n; e += blockDim.x) {
      const int t = (int)(e % Lout), b = (int)(e / Lout);
      s += dz[((long long)b * Cout + o) * Lout + t];
    }
    s = block_sum<256>(s);
    if (threadIdx.x == 0) db[o] = s;
  }
}

// h0[b, c] = mean_t a[b, c, t] for c < C; h0[b, C + j] = scal[b, j]
__global__ void k_pool_concat(const float* __restrict__ a, int B, int C, int L, const float* __restrict__ scal, int NS,
                              float* __restrict__ h0) {
  const int W = C + NS;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < B * W; e += gridDim.x * blockDim.x) {
    const int b = e / W, c = e % W;
    if (c < C) {
      float s = 0.f;
      const float* p = a + ((long long)b * C + c) * L;
      for (int t = 0; t < L; ++t) s += p[t];
      h0[e] = s / (float)L;
    } else {
      h0[e] = scal[b * NS + (c - C)];
    }
  }
}

// dz3[b,c,t] = dh0[b,c] / L * (z3 > 0)
__global__ void k_pool_bwd(const float* __restrict__ dh0, int ldh, const float* __restrict__ z, int B, int C, int L,
                           float* __restrict__ dzo) {
  const long long n = (long long)B * C * L;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const int c = (int)((e / L) % C), b = (int)(e / ((long long)L * C));
    dzo[e] = z[e] > 0.f ? dh0[(long long)b * ldh + c] / (float)L : 0.f;
  }
}

constexpr int TL = 16;

// z[b,n] = bias[n] + sum_k x[b,k] F[n,k]; a = relu(z) (if a != null).  16x16 tiles.
__global__ void k_linear_fwd(const float* __restrict__ x, int B, int Nin, const float* __restrict__ F,
                             const float* __restrict__ bias, int Nout, float* __restrict__ z, float* __restrict__ a) {
  __shared__ float xs[TL][TL + 1], fs[TL][TL + 1];
  const int b = blockIdx.y * TL + threadIdx.y;
  const int n = blockIdx.x * TL + threadIdx.x;
  float s = 0.f;
  for (int k0 = 0; k0 < Nin; k0 += TL) {
    const int kx = k0 + threadIdx.x;
    xs[threadIdx.y][threadIdx.x] = (b < B && kx < Nin) ? x[(long long)b * Nin + kx] : 0.f;
    const int nf = blockIdx.x * TL + threadIdx.y;
    fs[threadIdx.y][threadIdx.x] = (nf < Nout && kx < Nin) ? F[(long long)nf * Nin + kx] : 0.f;
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < TL; ++kk) s += xs[threadIdx.y][kk] * fs[threadIdx.x][kk];
    __syncthreads();
  }
  if (b < B && n < Nout) {
    s += bias[n];
    z[(long long)b * Nout + n] = s;
    if (a) a[(long long)b * Nout + n] = fmaxf(s, 0.f);
  }
}

// dx[b,k] = sum_n dz[b,n] F[n,k], times (zprev[b,k] > 0) if zprev != null
__global__ void k_linear_bwd_data(const float* __restrict__ dz, int B, int Nout, const float* __restrict__ F, int Nin,
                                  const float* __restrict__ zprev, float* __restrict__ dx) {
  __shared__ float ds[TL][TL + 1], fs[TL][TL + 1];
  const int b = blockIdx.y * TL + threadIdx.y;
  const int k = blockIdx.x * TL + threadIdx.x;
  float s = 0.f;
  for (int n0 = 0; n0 < Nout; n0 += TL) {
    const int nx = n0 + threadIdx.x;
    ds[threadIdx.y][threadIdx.x] = (b < B && nx < Nout) ? dz[(long long)b * Nout + nx] : 0.f;
    const int ny = n0 + threadIdx.y;
    fs[threadIdx.y][threadIdx.x] = (ny < Nout && k < Nin) ? F[(long long)ny * Nin + k] : 0.f;
    __syncthreads();
#pragma unroll
    for (int nn = 0; nn < TL; ++nn) s += ds[threadIdx.y][nn] * fs[nn][threadIdx.x];
    __syncthreads();
  }
  if (b < B && k < Nin) {
    const long long e = (long long)b * Nin + k;
    dx[e] = zprev ? (zprev[e] > 0.f ? s : 0.f) : s;
  }
}

// dF[n,k] = sum_b dz[b,n] x[b,k]; dc[n] = sum_b dz[b,n] (column k = Nin of the grid)
__global__ void k_linear_bwd_w(const float* __restrict__ dz, const float* __restrict__ x, int B, int Nout, int Nin,
                               float* __restrict__ dF, float* __restrict__ dc) {
  __shared__ float ds[TL][TL + 1], xs[TL][TL + 1];
  const int n = blockIdx.y * TL + threadIdx.y;
  const int k = blockIdx.x * TL + threadIdx.x;
  float s = 0.f;
  for (int b0 = 0; b0 < B; b0 += TL) {
    const int bx = b0 + threadIdx.x;
    const int nd = blockIdx.y * TL + threadIdx.y;
    ds[threadIdx.y][threadIdx.x] = (bx < B && nd < Nout) ? dz[(long long)bx * Nout + nd] : 0.f;
    const int by = b0 + threadIdx.y;
    xs[threadIdx.y][threadIdx.x] =
        (by < B && k < Nin + 1) ? (k < Nin ? x[(long long)by * Nin + k] : 1.f) : 0.f;
    __syncthreads();
#pragma unroll
    for (int bb = 0; bb < TL; ++bb) s += ds[threadIdx.y][bb] * xs[bb][threadIdx.x];
    __syncthreads();
  }
  if (n < Nout) {
    if (k < Nin) dF[(long long)n * Nin + k] = s;
    else if (k == Nin) dc[n] = s;
  }
}

// Loss terms and dL/dy (one block; B <= blockDim.x * iterations).
__global__ void __launch_bounds__(256) k_loss(const float* __restrict__ y, int B, int NOUT,
                                              const float* __restrict__ target, const int* __restrict__ label,
                                              float* __restrict__ dy, float* __restrict__ loss) {
  float mse = 0.f, ce = 0.f;
  const float invB = 1.f / (float)B;
  for (int b = threadIdx.x; b < B; b += blockDim.x) {
    const float* yb = y + (long long)b * NOUT;
    float* db = dy + (long long)b * NOUT;
    const float r = yb[0] - target[b];
    mse += r * r;
    db[0] = 2.f * r * invB;
    float m = yb[1];
    for (int q = 2; q < NOUT; ++q) m = fmaxf(m, yb[q]);
    float se = 0.f;
    for (int q = 1; q < NOUT; ++q) se += expf(yb[q] - m);
    const int lb = label[b];
    ce += logf(se) + m - yb[1 + lb];
    for (int q = 1; q < NOUT; ++q) db[q] = (expf(yb[q] - m) / se - (q - 1 == lb ? 1.f : 0.f)) * invB;
  }
  mse = block_sum<256>(mse);
  __syncthreads();
  ce = block_sum<256>(ce);
  if (threadIdx.x == 0) {
    loss[0] = mse * invB;
    loss[1] = ce * invB;
  }
}

__global__ void k_adam(long long n, float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, float lr, float b1, float b2, float eps, float bc1, float bc2) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const float gi = g[e];
    const float mi = b1 * m[e] + (1.f - b1) * gi;
    const float vi = b2 * v[e] + (1.f - b2) * gi * gi;
    m[e] = mi;
    v[e] = vi;
    p[e] -= lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
  }
}

// ------------------------------------------------- one CTA per sample
// Forward pass, loss and data gradients of one sample in one CTA, with every
// activation in shared memory, for the framework's kernel size and stride (K = 5,
// S = 2) and networks that fit and are narrow enough (by_samples).  The layer-by-layer
// kernels above take any other sizes; on a batch of 64 their 21 launches cost more than their arithmetic (243
// MFLOP), and the convolutions' inner loops read every operand from L1.  Here a
// thread forms eight output channels of one position from one input value and two
// broadcast 16-byte weight loads per tap, so that the FP32 pipe and shared memory
// are about equally busy.  The convolutions' weight gradients leave the CTA as
// per-sample partials (in the layout of the parameters), which k_sample_grads adds,
// and with them forms the linear layers' products.  Default
// network: a training step of 64 samples 317 -> 70 us (k_sample 55 of them: one CTA
// on each of 64 SMs, bound by the latency of its dozen dependent phases), a forward
// call of 96 samples 77 -> 27 us.

// W (Cout, Cin, 5) -> wt[(c 5 + k) Cp + o], zero-padded to Cp channels (coalesced
// reads, four in flight per thread; the scattered stores stay in shared memory)
__device__ __forceinline__ void stage_weights(const float* __restrict__ W, int Cin, int Cout, int Cp, float* wt) {
  const int row = Cin * SK, n = Cout * row;
  for (int e0 = threadIdx.x; e0 < n; e0 += 4 * ST) {
    float v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = e0 + j * ST < n ? __ldg(W + e0 + j * ST) : 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int e = e0 + j * ST;
      if (e < n) wt[(e % row) * Cp + e / row] = v[j];
    }
  }
  for (int e = threadIdx.x; e < row * (Cp - Cout); e += ST) wt[(e / (Cp - Cout)) * Cp + Cout + e % (Cp - Cout)] = 0.f;
}

// out = relu(bias + conv(in)): eight channels of one position per thread and pass
__device__ __forceinline__ void sample_conv(const float* in, int Cin, int sin, const float* wt, int Cp,
                                            const float* __restrict__ bias, int Cout, int Lout, float* out, int sout) {
  const int n = (Cp / 8) * Lout;
  for (int e = threadIdx.x; e < n; e += ST) {
    const int t = e % Lout, o0 = 8 * (e / Lout);
    float s[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) s[j] = o0 + j < Cout ? __ldg(bias + o0 + j) : 0.f;
    const float* x = in + SS * t;
    const float* w = wt + o0;
    for (int c = 0; c < Cin; ++c) {
#pragma unroll
      for (int k = 0; k < SK; ++k) {
        const float v = x[c * sin + k];
        const float4 w0 = *reinterpret_cast<const float4*>(w + (c * SK + k) * Cp);
        const float4 w1 = *reinterpret_cast<const float4*>(w + (c * SK + k) * Cp + 4);
        s[0] += w0.x * v, s[1] += w0.y * v, s[2] += w0.z * v, s[3] += w0.w * v;
        s[4] += w1.x * v, s[5] += w1.y * v, s[6] += w1.z * v, s[7] += w1.w * v;
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (o0 + j < Cout) out[(o0 + j) * sout + t] = fmaxf(s[j], 0.f);
  }
}

// din[c,u] = (act[c,u] > 0) sum over (o, k, t) with 2 t + k = u of W[o,c,k] dz[o,t]:
// four input channels of one position per thread (a dz value serves all four); even
// and odd positions, which meet different taps, in separate stretches of threads
__device__ __forceinline__ void sample_conv_bwd(const float* dz, int Cout, int Lout, int sout, const float* wt, int Cp,
                                                const float* act, int Cin, int Lin, int sin, float* din) {
  const int half = (Lin + 1) / 2, quads = (Cin + 3) / 4, n = 2 * quads * half;
  for (int e = threadIdx.x; e < n; e += ST) {
    const int m = e % half, rest = e / half, c0 = 4 * (rest % quads), par = rest / quads, u = 2 * m + par;
    if (u >= Lin) continue;
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    const float* w0[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) w0[j] = wt + min(c0 + j, Cin - 1) * SK * Cp;
    for (int k = par; k < SK; k += 2) {
      const int t = m - (k - par) / 2;
      if (t < 0 || t >= Lout) continue;
      const float* d = dz + t;
      int o = 0;
      for (; o + 4 <= Cout; o += 4) {
        const float d0 = d[o * sout], d1 = d[(o + 1) * sout], d2 = d[(o + 2) * sout], d3 = d[(o + 3) * sout];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 w = *reinterpret_cast<const float4*>(w0[j] + k * Cp + o);
          s[j] += w.x * d0;
          s[j] += w.y * d1;
          s[j] += w.z * d2;
          s[j] += w.w * d3;
        }
      }
      for (; o < Cout; ++o) {
#pragma unroll
        for (int j = 0; j < 4; ++j) s[j] += w0[j][k * Cp + o] * d[o * sout];
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (c0 + j < Cin) din[(c0 + j) * sin + u] = act[(c0 + j) * sin + u] > 0.f ? s[j] : 0.f;
  }
}

// gW[o,c,k] = sum_t dz[o,t] in[c,2t+k] for two output channels o and one c per thread
__device__ __forceinline__ void sample_conv_w(const float* dz, int Cout, int Lout, int sout, const float* in, int Cin,
                                              int sin, float* __restrict__ gW) {
  const int n = ((Cout + 1) / 2) * Cin;
#pragma unroll 1
  for (int e = threadIdx.x; e < n; e += ST) {
    const int c = e % Cin, o = 2 * (e / Cin), o1 = o + 1 < Cout ? o + 1 : o;
    float a[SK] = {0.f, 0.f, 0.f, 0.f, 0.f}, b[SK] = {0.f, 0.f, 0.f, 0.f, 0.f};
    const float* x = in + c * sin;
    float x0 = x[0], x1 = x[1], x2 = x[2];
#pragma unroll 4
    for (int t = 0; t < Lout; ++t) {
      const float x3 = x[2 * t + 3], x4 = x[2 * t + 4];
      const float da = dz[o * sout + t], db = dz[o1 * sout + t];
      a[0] += da * x0, a[1] += da * x1, a[2] += da * x2, a[3] += da * x3, a[4] += da * x4;
      b[0] += db * x0, b[1] += db * x1, b[2] += db * x2, b[3] += db * x3, b[4] += db * x4;
      x0 = x2, x1 = x3, x2 = x4;
    }
#pragma unroll
    for (int k = 0; k < SK; ++k) {
      gW[((long long)o * Cin + c) * SK + k] = a[k];
      if (o1 != o) gW[((long long)o1 * Cin + c) * SK + k] = b[k];
    }
  }
}

// gb[o] = sum_t dz[o,t], one warp per channel
__device__ __forceinline__ void sample_bias_grad(const float* dz, int C, int L, int s, float* __restrict__ gb) {
  const int lane = threadIdx.x & 31;
  for (int o = threadIdx.x >> 5; o < C; o += ST / 32) {
    float v = 0.f;
    for (int t = lane; t < L; t += 32) v += dz[o * s + t];
#pragma unroll
    for (int q = 16; q > 0; q >>= 1) v += __shfl_xor_sync(0xffffffffu, v, q);
    if (lane == 0) gb[o] = v;
  }
}

// z[n] = bias[n] + sum_k F[n,k] x[k], four rows per warp at a time (relu optional)
__device__ __forceinline__ void sample_linear(const float* __restrict__ F, const float* __restrict__ bias,
                                              const float* x, int Nin, int Nout, float* z, bool relu) {
  const int lane = threadIdx.x & 31;
  const bool vec = (Nin & 3) == 0 && ((uintptr_t)F & 15) == 0;  // (x is 16-byte aligned)
  for (int n0 = 4 * (threadIdx.x >> 5); n0 < Nout; n0 += 4 * (ST / 32)) {
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    const float* row[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) row[j] = F + (long long)min(n0 + j, Nout - 1) * Nin;
    if (vec) {
      for (int k = 4 * lane; k < Nin; k += 128) {
        const float4 v = *reinterpret_cast<const float4*>(x + k);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 w = __ldg(reinterpret_cast<const float4*>(row[j] + k));
          s[j] += w.x * v.x + w.y * v.y + (w.z * v.z + w.w * v.w);
        }
      }
    } else {
      for (int k = lane; k < Nin; k += 32) {
#pragma unroll
        for (int j = 0; j < 4; ++j) s[j] += __ldg(row[j] + k) * x[k];
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
      for (int q = 16; q > 0; q >>= 1) s[j] += __shfl_xor_sync(0xffffffffu, s[j], q);
      if (lane == j && n0 + j < Nout) {
        const float v = s[j] + __ldg(bias + n0 + j);
        z[n0 + j] = relu ? fmaxf(v, 0.f) : v;
      }
    }
  }
}

// dx[k] = (act[k] > 0, if act) sum_n dz[n] F[n,k]; g: scratch of max(4 ST, Nin) floats.
// Columns across threads (coalesced rows of F, 16 bytes a thread where they allow
// it), the rows dealt to groups of threads.
__device__ __forceinline__ void sample_linear_bwd(const float* __restrict__ F, const float* dz, int Nout, int Nin,
                                                  const float* act, float* dx, float* g) {
  const bool vec = (Nin & 3) == 0 && ((uintptr_t)F & 15) == 0;
  int ng;
  if (vec) {
    const int cols = Nin / 4;
    ng = cols < ST ? ST / cols : 1;
    for (int e = threadIdx.x; e < ng * cols; e += ST) {
      const int k = 4 * (e % cols), part = e / cols;
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
      for (int n = part; n < Nout; n += ng) {
        const float4 w = __ldg(reinterpret_cast<const float4*>(F + (long long)n * Nin + k));
        const float d = dz[n];
        s.x += d * w.x, s.y += d * w.y, s.z += d * w.z, s.w += d * w.w;
      }
      *reinterpret_cast<float4*>(g + part * Nin + k) = s;
    }
  } else {
    ng = Nin < ST ? ST / Nin : 1;
    for (int e = threadIdx.x; e < ng * Nin; e += ST) {
      const int k = e % Nin, part = e / Nin;
      float s = 0.f;
#pragma unroll 8
      for (int n = part; n < Nout; n += ng) s += dz[n] * __ldg(F + (long long)n * Nin + k);
      g[e] = s;
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < Nin; k += ST) {
    float s = 0.f;
    for (int part = 0; part < ng; ++part) s += g[part * Nin + k];
    dx[k] = act && !(act[k] > 0.f) ? 0.f : s;
  }
  __syncthreads();
}

struct SampleOut {  // what k_sample leaves for k_sample_grads (all per sample)
  float *h0, *a4, *dz4, *a5, *dz5, *dy, *part, *loss;
};

template <bool TRAIN>
__global__ void __launch_bounds__(ST, 1) k_sample(const Dims d, const Offsets o, const float* __restrict__ P,
                                                  const float* __restrict__ hist, const float* __restrict__ scal,
                                                  float* __restrict__ y, const float* __restrict__ target,
                                                  const int* __restrict__ label, const SampleOut out) {
  extern __shared__ __align__(16) float sm[];
  const SampleLayout<int> L = sample_layout<int>(d, TRAIN);
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, W0 = d.C3 + d.NS;
  float *x = sm + L.x, *w1 = sm + L.w1, *wt2 = sm + L.wt2, *wt3 = sm + L.wt3, *a1 = sm + L.a1, *a2 = sm + L.a2,
        *a3 = sm + L.a3, *h0 = sm + L.h0, *a4 = sm + L.a4, *a5 = sm + L.a5, *z = sm + L.z;
  float tgt = 0.f;
  int lb = 0;
  if (TRAIN && tid == 0) {
    tgt = target[b];
    lb = label[b];
  }
  for (int e = tid; e < d.L0; e += ST) x[e] = __ldg(hist + (long long)b * d.L0 + e);
  for (int e = tid; e < d.C1 * SK; e += ST) w1[e] = __ldg(P + o.W1 + e);
  stage_weights(P + o.W2, d.C1, d.C2, L.p2, wt2);
  stage_weights(P + o.W3, d.C2, d.C3, L.p3, wt3);
  __syncthreads();
  for (int e = tid; e < d.C1 * d.L1; e += ST) {
    const int t = e % d.L1, c = e / d.L1;
    float s = __ldg(P + o.b1 + c);
#pragma unroll
    for (int k = 0; k < SK; ++k) s += w1[c * SK + k] * x[SS * t + k];
    a1[c * L.s1 + t] = fmaxf(s, 0.f);
  }
  __syncthreads();
  sample_conv(a1, d.C1, L.s1, wt2, L.p2, P + o.b2, d.C2, d.L2, a2, L.s2);
  __syncthreads();
  sample_conv(a2, d.C2, L.s2, wt3, L.p3, P + o.b3, d.C3, d.L3, a3, L.s3);
  __syncthreads();
  for (int c = warp; c < d.C3; c += ST / 32) {
    float s = 0.f;
    for (int t = lane; t < d.L3; t += 32) s += a3[c * L.s3 + t];
#pragma unroll
    for (int q = 16; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
    if (lane == 0) h0[c] = s / (float)d.L3;
  }
  for (int j = tid; j < d.NS; j += ST) h0[d.C3 + j] = scal[(long long)b * d.NS + j];
  __syncthreads();
  sample_linear(P + o.F1, P + o.c1, h0, W0, d.H, a4, true);
  __syncthreads();
  sample_linear(P + o.F2, P + o.c2, a4, d.H, d.H, a5, true);
  __syncthreads();
  sample_linear(P + o.F3, P + o.c3, a5, d.H, d.NOUT, z, false);
  __syncthreads();
  if constexpr (!TRAIN) {
    for (int n = tid; n < d.NOUT; n += ST) y[(long long)b * d.NOUT + n] = z[n];
    return;
  }
  float *d2 = sm + L.d2, *d1 = sm + L.d1, *g = sm + L.g;
  for (int k = tid; k < W0; k += ST) out.h0[(long long)b * W0 + k] = h0[k];
  for (int k = tid; k < d.H; k += ST) {
    out.a4[(long long)b * d.H + k] = a4[k];
    out.a5[(long long)b * d.H + k] = a5[k];
  }
  if (tid == 0) {  // loss terms and dL/dy of the sample, y in place
    const float invB = 1.f / (float)gridDim.x;
    const float r = z[0] - tgt;
    float m = z[1];
    for (int q = 2; q < d.NOUT; ++q) m = fmaxf(m, z[q]);
    float se = 0.f;
    for (int q = 1; q < d.NOUT; ++q) se += expf(z[q] - m);
    out.loss[2 * b] = r * r;
    out.loss[2 * b + 1] = logf(se) + m - z[1 + lb];
    z[0] = 2.f * r * invB;
    for (int q = 1; q < d.NOUT; ++q) z[q] = (expf(z[q] - m) / se - (q - 1 == lb ? 1.f : 0.f)) * invB;
    for (int q = 0; q < d.NOUT; ++q) out.dy[(long long)b * d.NOUT + q] = z[q];
  }
  __syncthreads();
  sample_linear_bwd(P + o.F3, z, d.NOUT, d.H, a5, a5, g);  // a5 becomes dz5
  sample_linear_bwd(P + o.F2, a5, d.H, d.H, a4, a4, g);    // a4 becomes dz4
  for (int k = tid; k < d.H; k += ST) {
    out.dz5[(long long)b * d.H + k] = a5[k];
    out.dz4[(long long)b * d.H + k] = a4[k];
  }
  sample_linear_bwd(P + o.F1, a4, d.H, W0, nullptr, h0, g);
  for (int e = tid; e < d.C3 * d.L3; e += ST) {  // a3 becomes dz3
    const int t = e % d.L3, c = e / d.L3;
    float* p = a3 + c * L.s3 + t;
    *p = *p > 0.f ? h0[c] / (float)d.L3 : 0.f;
  }
  __syncthreads();
  sample_conv_bwd(a3, d.C3, d.L3, L.s3, wt3, L.p3, a2, d.C2, d.L2, L.s2, d2);
  float* part = out.part + (long long)b * o.F1;
  sample_conv_w(a3, d.C3, d.L3, L.s3, a2, d.C2, L.s2, part + o.W3);
  sample_bias_grad(a3, d.C3, d.L3, L.s3, part + o.b3);
  __syncthreads();
  sample_conv_bwd(d2, d.C2, d.L2, L.s2, wt2, L.p2, a1, d.C1, d.L1, L.s1, d1);
  sample_conv_w(d2, d.C2, d.L2, L.s2, a1, d.C1, L.s1, part + o.W2);
  sample_bias_grad(d2, d.C2, d.L2, L.s2, part + o.b2);
  __syncthreads();
  for (int c = warp; c < d.C1; c += ST / 32) {
    float s[SK + 1] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int t = lane; t < d.L1; t += 32) {
      const float v = d1[c * L.s1 + t];
#pragma unroll
      for (int k = 0; k < SK; ++k) s[k] += v * x[SS * t + k];
      s[SK] += v;
    }
#pragma unroll
    for (int k = 0; k <= SK; ++k) {
#pragma unroll
      for (int q = 16; q > 0; q >>= 1) s[k] += __shfl_xor_sync(0xffffffffu, s[k], q);
      if (lane == 0) part[k < SK ? o.W1 + c * SK + k : o.b1 + c] = s[k];
    }
  }
}

// One 16 x 16 tile of dF[n,k] = sum_b dz[b,n] x[b,k] (column Nin: the bias gradient)
__device__ __forceinline__ void linear_grad_tile(const float* __restrict__ dz, const float* __restrict__ x, int B,
                                                 int Nout, int Nin, int bx, int by, float* __restrict__ dF,
                                                 float* __restrict__ dc) {
  __shared__ float ds[TL][TL + 1], xs[TL][TL + 1];
  const int tx = threadIdx.x % TL, ty = threadIdx.x / TL;
  const int n = by * TL + ty, k = bx * TL + tx;
  float s = 0.f;
  for (int b0 = 0; b0 < B; b0 += TL) {
    // rows of both operands are read along their columns
    const int b = b0 + ty, nd = by * TL + tx;
    ds[tx][ty] = (b < B && nd < Nout) ? dz[(long long)b * Nout + nd] : 0.f;
    xs[ty][tx] = b < B && k <= Nin ? (k < Nin ? x[(long long)b * Nin + k] : 1.f) : 0.f;
    __syncthreads();
#pragma unroll
    for (int bb = 0; bb < TL; ++bb) s += ds[ty][bb] * xs[bb][tx];
    __syncthreads();
  }
  if (n < Nout && k <= Nin) (k < Nin ? dF[(long long)n * Nin + k] : dc[n]) = s;
}

// Parameter gradients from the samples' results: tiles of the three linear layers,
// the sums of the convolutions' partials, and the loss (last block).
__global__ void __launch_bounds__(256) k_sample_grads(const Dims d, const Offsets o, int B, const SampleOut w,
                                                      float* __restrict__ G, float* __restrict__ loss) {
  const int W0 = d.C3 + d.NS, th = (d.H + TL - 1) / TL, th1 = (d.H + TL) / TL, tw1 = (W0 + TL) / TL,
            to = (d.NOUT + TL - 1) / TL;
  int id = blockIdx.x;
  if (id < th1 * th) {
    linear_grad_tile(w.dz5, w.a4, B, d.H, d.H, id % th1, id / th1, G + o.F2, G + o.c2);
    return;
  }
  id -= th1 * th;
  if (id < tw1 * th) {
    linear_grad_tile(w.dz4, w.h0, B, d.H, W0, id % tw1, id / tw1, G + o.F1, G + o.c1);
    return;
  }
  id -= tw1 * th;
  if (id < th1 * to) {
    linear_grad_tile(w.dy, w.a5, B, d.NOUT, d.H, id % th1, id / th1, G + o.F3, G + o.c3);
    return;
  }
  id -= th1 * to;
  const int n = (int)o.F1, nb = (n + 255) / 256;
  if (id < nb) {
    const int e = id * 256 + threadIdx.x;
    if (e >= n) return;
    // groups of 64 samples in eight chains and a tree, the groups with their rounding
    // errors.  One chain of B additions rounded more than the layer kernels do: root
    // mean square error of W2's gradient (512-entry histories, H = 64) for 256 samples
    // of one sign 2.5e-7, 7e-8 so, 8e-8 by layers.  The loads bound it: 32 in flight take
    // 11.5 us for 256 samples (whole kernel), eight 14.3.
    const float* p = w.part + e;
    float hi = 0.f, lo = 0.f;
    for (int b0 = 0; b0 < B; b0 += 64) {
      float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      const int b1 = min(b0 + 64, B);
      int b = b0;
#pragma unroll 1
      for (; b + 32 <= b1; b += 32) {  // 32 loads in flight
        float v[32];
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = p[(long long)(b + k) * n];
#pragma unroll
        for (int k = 0; k < 32; ++k) s[k & 7] += v[k];
      }
#pragma unroll 8
      for (; b < b1; ++b) s[0] += p[(long long)b * n];
      const float g = ((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7]));
      const float t = hi + g, v = t - hi;
      lo += (hi - (t - v)) + (g - v);
      hi = t;
    }
    G[e] = lo == lo ? hi + lo : hi;  // (an infinite sum has no rounding error)
    return;
  }
  float mse = 0.f, ce = 0.f;
  for (int b = threadIdx.x; b < B; b += 256) {
    mse += w.loss[2 * b];
    ce += w.loss[2 * b + 1];
  }
  mse = block_sum<256>(mse);
  __syncthreads();
  ce = block_sum<256>(ce);
  if (threadIdx.x == 0) {
    loss[0] = mse / (float)B;
    loss[1] = ce / (float)B;
  }
}

int sample_grad_blocks(const Dims& d, const Offsets& o) {
  const int W0 = d.C3 + d.NS, th = (d.H + TL - 1) / TL, th1 = (d.H + TL) / TL, tw1 = (W0 + TL) / TL,
            to = (d.NOUT + TL - 1) / TL;
  return th1 * th + tw1 * th + th1 * to + ((int)o.F1 + 255) / 256 + 1;
}

// Launch k_sample on B samples.  The shared memory a kernel may take is one value per
// function and device, seen by every host thread: each call sets the most that any
// network takes (sample_fits), so that no call lowers it between another thread's
// setting and its launch.
template <bool TRAIN>
hlb_status launch_sample(const Dims& d, const Offsets& o, const float* P, const float* hist, const float* scal, int B,
                         float* y, const float* target, const int* label, const SampleOut& out, cudaStream_t s) {
  const size_t smem = (size_t)sample_layout<int>(d, TRAIN).total * sizeof(float);
  if (cudaFuncSetAttribute(k_sample<TRAIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, SAMPLE_SMEM) != cudaSuccess)
    return HLB_ECUDA;
  k_sample<TRAIN><<<B, ST, smem, s>>>(d, o, P, hist, scal, y, target, label, out);
  return HLB_OK;
}

int grid_for(long long n) {
  long long g = (n + 255) / 256;
  return (int)(g > 4096 ? 4096 : (g < 1 ? 1 : g));
}

bool ws_ok(const Dims& d, int B, void* ws, size_t bytes) {
  if (!ws || ((uintptr_t)ws & 255)) return false;
  return bytes >= act_offsets(d, B).total * sizeof(float);
}

void forward(const Dims& d, const Offsets& o, const Acts& A, const float* P, const float* hist, const float* scal,
             int B, float* w, cudaStream_t s) {
  k_conv_fwd<<<grid_for((long long)B * d.C1 * d.L1), 256, 0, s>>>(hist, 1, d.L0, P + o.W1, P + o.b1, d.C1, d.K, d.S,
                                                                  d.L1, B, w + A.z1, w + A.a1);
  k_conv_fwd<<<grid_for((long long)B * d.C2 * d.L2), 256, 0, s>>>(w + A.a1, d.C1, d.L1, P + o.W2, P + o.b2, d.C2, d.K,
                                                                  d.S, d.L2, B, w + A.z2, w + A.a2);
  k_conv_fwd<<<grid_for((long long)B * d.C3 * d.L3), 256, 0, s>>>(w + A.a2, d.C2, d.L2, P + o.W3, P + o.b3, d.C3, d.K,
                                                                  d.S, d.L3, B, w + A.z3, w + A.a3);
  const int W0 = d.C3 + d.NS;
  k_pool_concat<<<grid_for((long long)B * W0), 256, 0, s>>>(w + A.a3, B, d.C3, d.L3, scal, d.NS, w + A.h0);
  const dim3 blk(TL, TL);
  k_linear_fwd<<<dim3((d.H + TL - 1) / TL, (B + TL - 1) / TL), blk, 0, s>>>(w + A.h0, B, W0, P + o.F1, P + o.c1, d.H,
                                                                            w + A.z4, w + A.a4);
  k_linear_fwd<<<dim3((d.H + TL - 1) / TL, (B + TL - 1) / TL), blk, 0, s>>>(w + A.a4, B, d.H, P + o.F2, P + o.c2, d.H,
                                                                            w + A.z5, w + A.a5);
  k_linear_fwd<<<dim3((d.NOUT + TL - 1) / TL, (B + TL - 1) / TL), blk, 0, s>>>(w + A.a5, B, d.H, P + o.F3, P + o.c3,
                                                                               d.NOUT, w + A.y, nullptr);
}

}  // namespace

extern "C" {

void hlb_sur_config_default(hlb_sur_config* c) {
  if (!c) return;
  c->L0 = 500;
  c->C1 = 16;
  c->C2 = 32;
  c->C3 = 32;
  c->K = 5;
  c->S = 2;
  c->NS = 2;
  c->H = 256;
  c->NOUT = 6;
}

size_t hlb_sur_param_count(const hlb_sur_config* c) {
  Dims d;
  if (!dims_of(c, &d)) return 0;
  return param_offsets(d).total;
}

size_t hlb_sur_workspace_bytes(const hlb_sur_config* c, int B) {
  Dims d;
  if (!dims_of(c, &d) || B < 1 || B > 4096) return 0;
  return act_offsets(d, B).total * sizeof(float);
}

hlb_status hlb_sur_forward(const hlb_sur_config* c, const float* d_params, const float* d_hist, const float* d_scal,
                           int B, float* d_out, void* d_ws, size_t ws_bytes, void* stream) {
  Dims d;
  if (!dims_of(c, &d) || B < 1 || B > 4096 || !d_params || !d_hist || (d.NS > 0 && !d_scal) || !d_out)
    return HLB_EINVAL;
  if (!ws_ok(d, B, d_ws, ws_bytes)) return HLB_EINVAL;
  const Offsets o = param_offsets(d);
  const Acts A = act_offsets(d, B);
  float* w = (float*)d_ws;
  cudaStream_t s = (cudaStream_t)stream;
  if (by_samples(d, B, false)) {
    const hlb_status st = launch_sample<false>(d, o, d_params, d_hist, d_scal, B, d_out, nullptr, nullptr, SampleOut{}, s);
    if (st != HLB_OK) return st;
    return cudaGetLastError() == cudaSuccess ? HLB_OK : HLB_ECUDA;
  }
  forward(d, o, A, d_params, d_hist, d_scal, B, w, s);
  if (cudaMemcpyAsync(d_out, w + A.y, sizeof(float) * (size_t)B * d.NOUT, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
    return HLB_ECUDA;
  return cudaGetLastError() == cudaSuccess ? HLB_OK : HLB_ECUDA;
}

hlb_status hlb_sur_loss_grad(const hlb_sur_config* c, const float* d_params, const float* d_hist,
                             const float* d_scal, const float* d_target, const int* d_label, int B, float* d_grad,
                             float* d_loss, void* d_ws, size_t ws_bytes, void* stream) {
  Dims d;
  if (!dims_of(c, &d) || B < 1 || B > 4096 || !d_params || !d_hist || (d.NS > 0 && !d_scal) || !d_target ||
      !d_label || !d_grad || !d_loss)
    return HLB_EINVAL;
  if (!ws_ok(d, B, d_ws, ws_bytes)) return HLB_EINVAL;
  const Offsets o = param_offsets(d);
  const Acts A = act_offsets(d, B);
  float* w = (float*)d_ws;
  const float* P = d_params;
  float* G = d_grad;
  cudaStream_t s = (cudaStream_t)stream;
  if (by_samples(d, B, true)) {
    const SampleOut out = {w + A.h0, w + A.a4, w + A.dz4, w + A.a5, w + A.dz5, w + A.dy, w + A.part, w + A.loss};
    const hlb_status st = launch_sample<true>(d, o, P, d_hist, d_scal, B, nullptr, d_target, d_label, out, s);
    if (st != HLB_OK) return st;
    k_sample_grads<<<sample_grad_blocks(d, o), 256, 0, s>>>(d, o, B, out, G, d_loss);
    return cudaGetLastError() == cudaSuccess ? HLB_OK : HLB_ECUDA;
  }
  forward(d, o, A, P, d_hist, d_scal, B, w, s);
  k_loss<<<1, 256, 0, s>>>(w + A.y, B, d.NOUT, d_target, d_label, w + A.dy, w + A.loss);
  const dim3 blk(TL, TL);
  const int W0 = d.C3 + d.NS;
  // layer 6 (output)
  k_linear_bwd_w<<<dim3((d.H + 1 + TL - 1) / TL, (d.NOUT + TL - 1) / TL), blk, 0, s>>>(w + A.dy, w + A.a5, B, d.NOUT,
                                                                                      d.H, G + o.F3, G + o.c3);
  k_linear_bwd_data<<<dim3((d.H + TL - 1) / TL, (B + TL - 1) / TL), blk, 0, s>>>(w + A.dy, B, d.NOUT, P + o.F3, d.H,
                                                                                w + A.z5, w + A.dz5);
  // layer 5
  k_linear_bwd_w<<<dim3((d.H + 1 + TL - 1) / TL, (d.H + TL - 1) / TL), blk, 0, s>>>(w + A.dz5, w + A.a4, B, d.H, d.H,
                                                                                   G + o.F2, G + o.c2);
  k_linear_bwd_data<<<dim3((d.H + TL - 1) / TL, (B + TL - 1) / TL), blk, 0, s>>>(w + A.dz5, B, d.H, P + o.F2, d.H,
                                                                                w + A.z4, w + A.dz4);
  // layer 4
  k_linear_bwd_w<<<dim3((W0 + 1 + TL - 1) / TL, (d.H + TL - 1) / TL), blk, 0, s>>>(w + A.dz4, w + A.h0, B, d.H, W0,
                                                                                  G + o.F1, G + o.c1);
  k_linear_bwd_data<<<dim3((W0 + TL - 1) / TL, (B + TL - 1) / TL), blk, 0, s>>>(w + A.dz4, B, d.H, P + o.F1, W0,
                                                                               nullptr, w + A.dh0);
  // pooling and conv layers
  k_pool_bwd<<<grid_for((long long)B * d.C3 * d.L3), 256, 0, s>>>(w + A.dh0, W0, w + A.z3, B, d.C3, d.L3, w + A.dz3);
  k_conv_bwd_w<<<d.C3 * d.C2 * d.K + d.C3, 256, 0, s>>>(w + A.dz3, w + A.a2, B, d.C2, d.L2, d.C3, d.K, d.S, d.L3,
                                                        G + o.W3, G + o.b3);
  k_conv_bwd_data<<<grid_for((long long)B * d.C2 * d.L2), 256, 0, s>>>(w + A.dz3, P + o.W3, B, d.C2, d.L2, d.C3, d.K,
                                                                      d.S, d.L3, w + A.z2, w + A.dz2);
  k_conv_bwd_w<<<d.C2 * d.C1 * d.K + d.C2, 256, 0, s>>>(w + A.dz2, w + A.a1, B, d.C1, d.L1, d.C2, d.K, d.S, d.L2,
                                                        G + o.W2, G + o.b2);
  k_conv_bwd_data<<<grid_for((long long)B * d.C1 * d.L1), 256, 0, s>>>(w + A.dz2, P + o.W2, B, d.C1, d.L1, d.C2, d.K,
                                                                      d.S, d.L2, w + A.z1, w + A.dz1);
  k_conv_bwd_w<<<d.C1 * 1 * d.K + d.C1, 256, 0, s>>>(w + A.dz1, d_hist, B, 1, d.L0, d.C1, d.K, d.S, d.L1, G + o.W1,
                                                     G + o.b1);
  if (cudaMemcpyAsync(d_loss, w + A.loss, 2 * sizeof(float), cudaMemcpyDeviceToDevice, s) != cudaSuccess)
    return HLB_ECUDA;
  return cudaGetLastError() == cudaSuccess ? HLB_OK : HLB_ECUDA;
}

hlb_status hlb_sur_adam(long long n, float* d_params, const float* d_grad, float* d_m, float* d_v, float lr,
                        float beta1, float beta2, float eps, int t, void* stream) {
  if (n < 1 || !d_params || !d_grad || !d_m || !d_v || t < 1) return HLB_EINVAL;
  const float bc1 = 1.f - powf(beta1, (float)t);
  const float bc2 = 1.f - powf(beta2, (float)t);
  k_adam<<<grid_for(n), 256, 0, (cudaStream_t)stream>>>(n, d_params, d_grad, d_m, d_v, lr, beta1, beta2, eps, bc1, bc2);
  return cudaGetLastError() == cudaSuccess ? HLB_OK : HLB_ECUDA;
}

}  // extern "C"
