// Learned initial guess for the Poisson solve (an addition to the paper's
// method; the plain solver still iterates to the same tolerance afterwards).
//
// A small periodic 3-D convolutional network maps the residual of the
// warm-start potential, r = s - A psi(t-1), to a correction:
//   x0 = r / sigma_r (sigma_r: rms of r over fluid cells), x1 = fluid mask
//   h_c = tanh(b_c + sum_{ci, o in 3x3x3} W1[c][ci][o] x_ci(cell + o))
//   y   = sum_{c, o} W2[c][o] h_c(cell + o),   delta psi = sigma_r y (fluid)
// Training pairs come from the solver itself: the initial residual of each
// step and the correction the plain solve found, A dpsi* = r.  The loss is
// the normalised residual left after the guess,
//   L = sum_fluid (x0 - A y)^2 / sum_fluid x0^2  = ||A (dpsi* - dpsi)||^2 / ||r||^2,
// with A the finite-volume operator of the Poisson solve.  Forward, backward
// (weight gradients as correlations) and Adam run in the kernels below;
// inference stores weights and activations in FP16 with FP32 accumulation.
#include <cuda_fp16.h>
#include <math.h>

#include <algorithm>
#include <random>
#include <string>
#include <vector>

#include "lbm_internal.cuh"

namespace lbm_gb300 {

struct NNet {
  int C = 8;                 // hidden channels
  static constexpr int CI = 2;
  int np = 0;                // parameter count
  float* p = nullptr;        // FP32 master parameters [W1 | b1 | W2]
  float* g = nullptr;        // gradients
  float* m = nullptr;        // Adam first moment
  float* v = nullptr;        // Adam second moment
  __half* ph = nullptr;      // FP16 copy for inference
  int adam_t = 0;
  float* x0 = nullptr;       // normalised residual (N)
  float* hid = nullptr;      // hidden activations (C x N), FP32 (training)
  __half* hid16 = nullptr;   // hidden activations (C x N), FP16 (inference)
  float* y = nullptr;        // output (N)
  float* res = nullptr;      // x0 - A y (N)
  float* gy = nullptr;       // dL/dy (N)
  float* ga = nullptr;       // dL/d(pre-activation) (C x N)
  double* red = nullptr;     // reductions [0] sum x0^2 [1] sum res^2
  double* hred = nullptr;    // pinned mirror
  // collected training residuals (ring buffer of full lattice fields)
  float* pool = nullptr;
  int cap = 0, count = 0, next = 0;
  bool collect = false, use = false;
  // inference on channel pairs: input packed per cell as (x0, fluid mask),
  // hidden activations stored per cell ([N][C] halves), and a host copy of
  // the parameters for the kernels' arguments (stale after training)
  __half2* xin = nullptr;
  std::vector<float> hp;
  bool hp_stale = true;
  // statistics of the guesses applied by the solver
  long long tried = 0, accepted = 0;
  double sum_ratio = 0.0;    // sum of residual ratio after/before over accepted guesses
};

namespace {

inline unsigned nb(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

struct Geo {
  int nx, ny, nz;
  int64_t N;
  const uint32_t* links;  // NULL: all fluid
};

__device__ __forceinline__ void xyz(int64_t i, const Geo& G, int& x, int& y, int& z) {
  const int64_t t = i / G.nx;
  x = (int)(i - t * G.nx);
  z = (int)(t / G.ny);
  y = (int)(t - (int64_t)z * G.ny);
}

// The 27 neighbours of a cell from six wrapped axis offsets (no modulo per
// tap): offset of (dx, dy, dz) = ox[dx+1] + oy[dy+1] + oz[dz+1].
struct Taps {
  int ox[3], oy[3], oz[3];
};
__device__ __forceinline__ Taps taps_of(const Geo& G, int x, int y, int z) {
  Taps t;
  const int nxy = G.nx * G.ny;
  t.ox[0] = x == 0 ? G.nx - 1 : -1;
  t.ox[1] = 0;
  t.ox[2] = x == G.nx - 1 ? -(G.nx - 1) : 1;
  t.oy[0] = (y == 0 ? G.ny - 1 : -1) * G.nx;
  t.oy[1] = 0;
  t.oy[2] = (y == G.ny - 1 ? -(G.ny - 1) : 1) * G.nx;
  t.oz[0] = (z == 0 ? G.nz - 1 : -1) * nxy;
  t.oz[1] = 0;
  t.oz[2] = (z == G.nz - 1 ? -(G.nz - 1) : 1) * nxy;
  return t;
}

__device__ __forceinline__ bool fluid_at(const Geo& G, int64_t i) {
  return !G.links || !(G.links[i] & LINK_SOLID);
}

// (A v)_i over open faces (face open iff both cells fluid).
__device__ float apply_A(const float* v, const Geo& G, int64_t i, int x, int y, int z) {
  const float vc = v[i];
  const Taps T = taps_of(G, x, y, z);
  const int d[6] = {T.ox[2], T.ox[0], T.oy[2], T.oy[0], T.oz[2], T.oz[0]};
  float acc = 0.f;
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    const int64_t j = i + d[f];
    if (d[f] != 0 && fluid_at(G, j)) acc += vc - v[j];
  }
  return acc;
}

// x0 = r / sigma (fluid), 0 at wall nodes.  The residual of a trimmed
// multigrid box covers planes [zlo, zlo + nzb); with hx > 0 it is stored
// colour-split: cell (x, y, zb) of colour q = (x + y + zb) mod 2 at
// q H + (zb ny + y) hx + floor(x / 2), H = nzb ny hx.
// When xin is given, the same input packed for inference: (x0, fluid mask)
// as one FP16 pair per cell.
__global__ void k_nn_input(const float* __restrict__ r, int zlo, int nzb, int hx, float inv_sigma,
                           Geo G, float* __restrict__ x0, __half2* __restrict__ xin) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= G.N) return;
  const int64_t nxy = (int64_t)G.nx * G.ny;
  const int z = (int)(i / nxy);
  const bool fl = fluid_at(G, i);
  float v = 0.f;
  if (z >= zlo && z < zlo + nzb && fl) {
    int64_t j = i - (int64_t)zlo * nxy;
    if (hx > 0) {
      const int zb = z - zlo;
      const int64_t rem = i - (int64_t)z * nxy;
      const int y = (int)(rem / G.nx), x = (int)(rem - (int64_t)y * G.nx);
      const int64_t H = (int64_t)nzb * G.ny * hx;
      j = (((x + y + zb) & 1) ? H : 0) + ((int64_t)zb * G.ny + y) * hx + (x >> 1);
    }
    v = r[j] * inv_sigma;
  }
  x0[i] = v;
  if (xin) xin[i] = __floats2half2_rn(v, fl ? 1.f : 0.f);
}

__global__ void k_sum_sq(const float* __restrict__ a, int64_t n, double* out) {
  __shared__ float red[8];
  float v = 0.f;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    v += a[i] * a[i];
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    atomicAdd(out, t);
  }
}

// The FP32 kernels of the training pass are instantiated for up to 4, 8 and
// 16 channels (CM), so that the sums over channels stay in registers; the
// weights come from shared memory, the channels of one tap side by side.
// With a run-time channel count the sums lived in local memory and every tap
// wrapped its index with three divisions (64^3, 8 channels: layer 1 56 us,
// layer 2 45 us, its transpose 42 us; now 15, 29 and 11 us).
template <int CM>
__device__ __forceinline__ void stage_taps(float* w, const float* __restrict__ p, int C, int stride) {
  // w[o * CM + c] = p[c * stride + o], zero for c >= C
  for (int k = threadIdx.x; k < 27 * CM; k += blockDim.x) {
    const int o = k / CM, c = k - o * CM;
    w[k] = c < C ? p[c * stride + o] : 0.f;
  }
}

// Layer 1 (FP32): hid[c][i] = tanh(b1[c] + sum W1[c][ci][o] x_ci(i + o)).
template <int CM>
__global__ void __launch_bounds__(256) k_nn_layer1(const float* __restrict__ x0, const float* __restrict__ p,
                                                   int C, Geo G, float* __restrict__ hid) {
  __shared__ __align__(16) float wx[27 * CM], wm[27 * CM];
  stage_taps<CM>(wx, p, C, 54);
  stage_taps<CM>(wm, p + 27, C, 54);
  __syncthreads();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= G.N) return;
  int x, y, z;
  xyz(i, G, x, y, z);
  const Taps T = taps_of(G, x, y, z);
  float acc[CM];
#pragma unroll
  for (int c = 0; c < CM; ++c) acc[c] = c < C ? p[C * 2 * 27 + c] : 0.f;
#pragma unroll
  for (int o = 0; o < 27; ++o) {
    const int64_t j = i + T.ox[o % 3] + T.oy[(o / 3) % 3] + T.oz[o / 9];
    const float a0 = x0[j];
    const float a1 = fluid_at(G, j) ? 1.f : 0.f;
#pragma unroll
    for (int c = 0; c < CM; ++c) acc[c] += wx[o * CM + c] * a0 + wm[o * CM + c] * a1;
  }
#pragma unroll
  for (int c = 0; c < CM; ++c)
    if (c < C) hid[(int64_t)c * G.N + i] = tanhf(acc[c]);
}

// Layer 2 (FP32): y = sum W2[c][o] hid_c(i + o), zero at wall nodes.
template <int CM>
__global__ void __launch_bounds__(256) k_nn_layer2(const float* __restrict__ hid, const float* __restrict__ p,
                                                   int C, Geo G, float* __restrict__ y) {
  __shared__ __align__(16) float w2[27 * CM];
  stage_taps<CM>(w2, p + C * 2 * 27 + C, C, 27);
  __syncthreads();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= G.N) return;
  if (!fluid_at(G, i)) {
    y[i] = 0.f;
    return;
  }
  int x, yy, z;
  xyz(i, G, x, yy, z);
  const Taps T = taps_of(G, x, yy, z);
  // channels outside: the taps of one channel are neighbours in the cache
  float acc = 0.f;
  for (int c = 0; c < C; ++c) {
    const float* __restrict__ hc = hid + (int64_t)c * G.N + i;
    float v[27];
#pragma unroll
    for (int o = 0; o < 27; ++o) v[o] = hc[T.ox[o % 3] + T.oy[(o / 3) % 3] + T.oz[o / 9]];
#pragma unroll
    for (int o = 0; o < 27; ++o) acc += w2[o * CM + c] * v[o];
  }
  y[i] = acc;
}

// FP16 inference: the same two layers with half weights and activations,
// FP32 accumulation; writes the fixed-point correction sigma * y to dpsi.
__global__ void __launch_bounds__(256) k_nn_infer1(const float* __restrict__ x0, const __half* __restrict__ ph,
                                                   int C, Geo G, __half* __restrict__ hid) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= G.N) return;
  int x, y, z;
  xyz(i, G, x, y, z);
  const Taps T = taps_of(G, x, y, z);
  float acc[16];
  for (int c = 0; c < C; ++c) acc[c] = __half2float(ph[C * 2 * 27 + c]);
#pragma unroll
  for (int o = 0; o < 27; ++o) {
    const int64_t j = i + T.ox[o % 3] + T.oy[(o / 3) % 3] + T.oz[o / 9];
    const __half a0 = __float2half(x0[j]);
    const __half a1 = __float2half(fluid_at(G, j) ? 1.f : 0.f);
    for (int c = 0; c < C; ++c)
      acc[c] += __half2float(__hfma(ph[(c * 2 + 0) * 27 + o], a0, __hmul(ph[(c * 2 + 1) * 27 + o], a1)));
  }
  for (int c = 0; c < C; ++c) hid[(int64_t)c * G.N + i] = __float2half(tanhf(acc[c]));
}

__global__ void __launch_bounds__(256) k_nn_infer2(const __half* __restrict__ hid, const __half* __restrict__ ph,
                                                   int C, Geo G, float sigma, float* __restrict__ dpsi) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= G.N) return;
  if (!fluid_at(G, i)) {
    dpsi[i] = 0.f;
    return;
  }
  int x, yy, z;
  xyz(i, G, x, yy, z);
  const Taps T = taps_of(G, x, yy, z);
  const __half* W2 = ph + C * 2 * 27 + C;
  float acc = 0.f;
#pragma unroll
  for (int o = 0; o < 27; ++o) {
    const int64_t j = i + T.ox[o % 3] + T.oy[(o / 3) % 3] + T.oz[o / 9];
    for (int c = 0; c < C; ++c) acc += __half2float(__hmul(W2[c * 27 + o], hid[(int64_t)c * G.N + j]));
  }
  dpsi[i] = sigma * acc;
}

// Inference on channel pairs (C even, up to 16): the weights are kernel
// arguments (constant-bank operands of the FP16 pair FMAs, no loads), the
// input is one (x0, mask) pair per cell, the hidden activations one vector
// of C halves per cell.  Same network as k_nn_infer1/2: layer 1 with bias
// and tanh (the hardware's approximate tanh of FP16 pairs), layer 2
// accumulated per channel pair in FP16 and over pairs in FP32.
template <int C>
struct InferW {
  __half2 w1x[27][C / 2];  // W1[c][0][o] for c = 2k, 2k + 1
  __half2 w1m[27][C / 2];  // W1[c][1][o]
  __half2 b1[C / 2];
  __half2 w2[27][C / 2];   // W2[c][o]
};

template <int C>
struct HidVec {  // the C hidden halves of one cell
  __half2 v[C / 2];
};

__device__ __forceinline__ __half2 tanh_approx_h2(__half2 x) {
  uint32_t r;
  asm("tanh.approx.f16x2 %0, %1;" : "=r"(r) : "r"(*reinterpret_cast<const uint32_t*>(&x)));
  return *reinterpret_cast<const __half2*>(&r);
}

template <int C>
__global__ void __launch_bounds__(256) k_nn_fast1(const __half2* __restrict__ xin, const InferW<C> w,
                                                  Geo G, HidVec<C>* __restrict__ hid) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= G.N) return;
  int x, y, z;
  xyz(i, G, x, y, z);
  const Taps T = taps_of(G, x, y, z);
  __half2 acc[C / 2];
#pragma unroll
  for (int k = 0; k < C / 2; ++k) acc[k] = w.b1[k];
#pragma unroll
  for (int o = 0; o < 27; ++o) {
    const __half2 v = xin[i + T.ox[o % 3] + T.oy[(o / 3) % 3] + T.oz[o / 9]];
    const __half2 xx = __low2half2(v), mm = __high2half2(v);
#pragma unroll
    for (int k = 0; k < C / 2; ++k) acc[k] = __hfma2(w.w1m[o][k], mm, __hfma2(w.w1x[o][k], xx, acc[k]));
  }
  HidVec<C> out;
#pragma unroll
  for (int k = 0; k < C / 2; ++k) out.v[k] = tanh_approx_h2(acc[k]);
  hid[i] = out;
}

// Layer 2 and the correction: dpsi = sigma y on fluid cells (kept for a
// revert), psi += round(dpsi) in fixed point.
template <int C>
__global__ void __launch_bounds__(256) k_nn_fast2(const HidVec<C>* __restrict__ hid, const InferW<C> w,
                                                  Geo G, float sigma, float* __restrict__ dpsi,
                                                  int64_t* __restrict__ psi) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= G.N) return;
  if (!fluid_at(G, i)) {
    dpsi[i] = 0.f;
    return;
  }
  int x, y, z;
  xyz(i, G, x, y, z);
  const Taps T = taps_of(G, x, y, z);
  __half2 acc[C / 2];
#pragma unroll
  for (int k = 0; k < C / 2; ++k) acc[k] = __float2half2_rn(0.f);
#pragma unroll
  for (int o = 0; o < 27; ++o) {
    const HidVec<C> h = hid[i + T.ox[o % 3] + T.oy[(o / 3) % 3] + T.oz[o / 9]];
#pragma unroll
    for (int k = 0; k < C / 2; ++k) acc[k] = __hfma2(w.w2[o][k], h.v[k], acc[k]);
  }
  float yv = 0.f;
#pragma unroll
  for (int k = 0; k < C / 2; ++k) {
    const float2 f = __half22float2(acc[k]);
    yv += f.x + f.y;
  }
  const float d = sigma * yv;
  dpsi[i] = d;
  psi[i] += f32_to_i64_rn(d * PSI_SCALE_F);
}

template <int C>
InferW<C> infer_weights(const std::vector<float>& p) {
  InferW<C> w;
  const int b1 = C * 2 * 27, w2 = b1 + C;
  for (int o = 0; o < 27; ++o)
    for (int k = 0; k < C / 2; ++k) {
      const int c0 = 2 * k, c1 = 2 * k + 1;
      w.w1x[o][k] = __floats2half2_rn(p[(c0 * 2 + 0) * 27 + o], p[(c1 * 2 + 0) * 27 + o]);
      w.w1m[o][k] = __floats2half2_rn(p[(c0 * 2 + 1) * 27 + o], p[(c1 * 2 + 1) * 27 + o]);
      w.w2[o][k] = __floats2half2_rn(p[w2 + c0 * 27 + o], p[w2 + c1 * 27 + o]);
    }
  for (int k = 0; k < C / 2; ++k) w.b1[k] = __floats2half2_rn(p[b1 + 2 * k], p[b1 + 2 * k + 1]);
  return w;
}

template <int C>
cudaError_t fast_infer(NNet* n, const Geo& G, float sigma, int64_t* psi, cudaStream_t st) {
  const InferW<C> w = infer_weights<C>(n->hp);
  const unsigned b = nb(G.N, 256);
  HidVec<C>* hid = reinterpret_cast<HidVec<C>*>(n->hid16);
  k_nn_fast1<C><<<b, 256, 0, st>>>(n->xin, w, G, hid);
  k_nn_fast2<C><<<b, 256, 0, st>>>(hid, w, G, sigma, n->y, psi);
  return cudaGetLastError();
}

// res = x0 - A y and its squared sum.
__global__ void k_nn_res(const float* __restrict__ x0, const float* __restrict__ y, Geo G,
                         float* __restrict__ res, double* red) {
  __shared__ float sm[8];
  float v = 0.f;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < G.N;
       i += (int64_t)gridDim.x * blockDim.x) {
    float rv = 0.f;
    if (fluid_at(G, i)) {
      int x, yy, z;
      xyz(i, G, x, yy, z);
      rv = x0[i] - apply_A(y, G, i, x, yy, z);
    }
    res[i] = rv;
    v += rv * rv;
  }
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sm[w];
    atomicAdd(red + 1, t);
  }
}

// dL/dy = -2 A res / sum x0^2 (A symmetric), zero at wall nodes.
__global__ void k_nn_gy(const float* __restrict__ res, Geo G, const double* __restrict__ red,
                        float* __restrict__ gy) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= G.N) return;
  float v = 0.f;
  if (fluid_at(G, i)) {
    int x, yy, z;
    xyz(i, G, x, yy, z);
    v = -2.0f / (float)red[0] * apply_A(res, G, i, x, yy, z);
  }
  gy[i] = v;
}

// dL/d(pre-activation)_c = (1 - h_c^2) sum_o W2[c][o] gy(i - o).
template <int CM>
__global__ void __launch_bounds__(256) k_nn_ga(const float* __restrict__ gy, const float* __restrict__ hid,
                                               const float* __restrict__ p, int C, Geo G,
                                               float* __restrict__ ga) {
  __shared__ __align__(16) float w2[27 * CM];
  stage_taps<CM>(w2, p + C * 2 * 27 + C, C, 27);
  __syncthreads();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= G.N) return;
  int x, yy, z;
  xyz(i, G, x, yy, z);
  const Taps T = taps_of(G, x, yy, z);
  float acc[CM];
#pragma unroll
  for (int c = 0; c < CM; ++c) acc[c] = 0.f;
#pragma unroll
  for (int o = 0; o < 27; ++o) {
    // the opposite tap: i - o
    const int64_t j = i + T.ox[2 - o % 3] + T.oy[2 - (o / 3) % 3] + T.oz[2 - o / 9];
    const float gj = gy[j];
#pragma unroll
    for (int c = 0; c < CM; ++c) acc[c] += w2[o * CM + c] * gj;
  }
#pragma unroll
  for (int c = 0; c < CM; ++c)
    if (c < C) {
      const float h = hid[(int64_t)c * G.N + i];
      ga[(int64_t)c * G.N + i] = acc[c] * (1.f - h * h);
    }
}

// Weight gradients as correlations over cells:
//   g[W1 c,ci,o] = sum_i ga_c(i) x_ci(i + o),  g[b1 c] = sum_i ga_c(i),
//   g[W2 c,o]    = sum_i gy(i) hid_c(i + o).
// A CTA takes one channel c and one tap plane dz (blockIdx.y) and a share of
// the (z, x block) columns (blockIdx.x); each of its warps takes a run of
// rows y: lane = cell of a block of 32 x, the warp walks y with the three
// rows y - 1 .. y + 1 of x0, the mask and hid_c at z + dz in registers, so
// that a row costs 11 loads for 27 products, each summed per lane in a
// register.  One reduction per product over the warp and the CTA at the end,
// then one atomic.  (With a five-step warp sum for every product of every
// 32 cells, in CTAs of one warp, 64^3 and 8 channels took 4.38 ms; now 55
// us.)
constexpr int WG_WARPS = 8;

__global__ void __launch_bounds__(32 * WG_WARPS) k_nn_wgrad(const float* __restrict__ gy,
                                                            const float* __restrict__ ga,
                                                            const float* __restrict__ hid,
                                                            const float* __restrict__ x0, int C,
                                                            Geo G, int nwork,
                                                            float* __restrict__ g) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int c = blockIdx.y / 3, dz = blockIdx.y % 3 - 1;
  const int nx = G.nx, ny = G.ny, nz = G.nz;
  const int xb = (nx + 31) / 32;
  const float* __restrict__ gac = ga + (int64_t)c * G.N;
  const float* __restrict__ hc = hid + (int64_t)c * G.N;
  float ax[9], am[9], ah[9], ab = 0.f;
#pragma unroll
  for (int k = 0; k < 9; ++k) ax[k] = am[k] = ah[k] = 0.f;
  const int rows = (ny + WG_WARPS - 1) / WG_WARPS;
  const int y0 = wid * rows, y1 = min(y0 + rows, ny);
  for (int wk = blockIdx.x; wk < nwork; wk += gridDim.x) {
    const int z = wk / xb, x = (wk - z * xb) * 32 + lane;
    const bool ok = x < nx;
    const int xc = ok ? x : nx - 1;
    int zt = z + dz;
    zt = zt < 0 ? nz - 1 : (zt == nz ? 0 : zt);
    const int xi[3] = {xc == 0 ? nx - 1 : xc - 1, xc, xc == nx - 1 ? 0 : xc + 1};
    // rows y - 1 .. y + 2 of the taps' plane: two rows of cells at a time
    float vx[4][3], vm[4][3], vh[4][3];
    auto load = [&](int y, float (&px)[3], float (&pm)[3], float (&ph)[3]) {
      int yw = y < 0 ? ny - 1 : (y >= ny ? y - ny : y);  // y <= ny + 1
      if (yw >= ny) yw -= ny;
      const uint32_t row = (uint32_t)(zt * ny + yw) * (uint32_t)nx;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const uint32_t j = row + (uint32_t)xi[d];
        px[d] = x0[j];
        pm[d] = (float)(1u - (G.links ? G.links[j] & LINK_SOLID : 0u));
        ph[d] = hc[j];
      }
    };
    if (y0 < y1) {
      load(y0 - 1, vx[0], vm[0], vh[0]);
      load(y0, vx[1], vm[1], vh[1]);
    }
    for (int y = y0; y < y1; y += 2) {
      const bool two = y + 1 < y1;
      load(y + 1, vx[2], vm[2], vh[2]);
      load(y + 2, vx[3], vm[3], vh[3]);
      float ga_i[2], gy_i[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const uint32_t i = (uint32_t)(z * ny + min(y + u, ny - 1)) * (uint32_t)nx + (uint32_t)xc;
        const bool in = ok && (u == 0 || two);
        ga_i[u] = in ? gac[i] : 0.f;
        gy_i[u] = in ? gy[i] : 0.f;
      }
      ab += ga_i[0] + ga_i[1];
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int dy = 0; dy < 3; ++dy)
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            ax[dy * 3 + d] = fmaf(ga_i[u], vx[dy + u][d], ax[dy * 3 + d]);
            am[dy * 3 + d] = fmaf(ga_i[u], vm[dy + u][d], am[dy * 3 + d]);
            ah[dy * 3 + d] = fmaf(gy_i[u], vh[dy + u][d], ah[dy * 3 + d]);
          }
#pragma unroll
      for (int dy = 0; dy < 2; ++dy)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          vx[dy][d] = vx[dy + 2][d];
          vm[dy][d] = vm[dy + 2][d];
          vh[dy][d] = vh[dy + 2][d];
        }
    }
  }
  __shared__ float red[WG_WARPS][28];
  auto wsum = [](float v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    return v;
  };
#pragma unroll
  for (int k = 0; k < 28; ++k) {
    const float t = wsum(k < 9 ? ax[k] : (k < 18 ? am[k - 9 < 9 ? k - 9 : 0] : (k < 27 ? ah[k >= 18 ? k - 18 : 0] : ab)));
    if (lane == 0) red[wid][k] = t;
  }
  __syncthreads();
  if (threadIdx.x < 28) {
    const int k = threadIdx.x;
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < WG_WARPS; ++w) t += red[w][k];
    const int o = (dz + 1) * 9 + k % 9;
    if (k < 9) atomicAdd(g + (c * 2 + 0) * 27 + o, t);
    else if (k < 18) atomicAdd(g + (c * 2 + 1) * 27 + o, t);
    else if (k < 27) atomicAdd(g + C * 2 * 27 + C + c * 27 + o, t);
    else if (dz == 0) atomicAdd(g + C * 2 * 27 + c, t);
  }
}

__global__ void k_adam(float* p, const float* g, float* m, float* v, int n, float lr, float b1,
                       float b2, float eps, int t, __half* ph) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const float gk = g[k];
  const float mk = b1 * m[k] + (1.f - b1) * gk;
  const float vk = b2 * v[k] + (1.f - b2) * gk * gk;
  m[k] = mk;
  v[k] = vk;
  const float mh = mk / (1.f - powf(b1, (float)t));
  const float vh = vk / (1.f - powf(b2, (float)t));
  p[k] -= lr * mh / (sqrtf(vh) + eps);
  ph[k] = __float2half(p[k]);
}

__global__ void k_to_half(const float* p, __half* ph, int n) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) ph[k] = __float2half(p[k]);
}

// psi += round(dpsi) on fluid nodes (fixed point), or -= to revert.
__global__ void k_nn_apply(int64_t* psi, const float* __restrict__ dpsi, int64_t n, int sign) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t d = f32_to_i64_rn(dpsi[i] * PSI_SCALE_F);
  psi[i] += sign > 0 ? d : -d;
}

Geo geo_of(const lbm_t* h) {
  Geo G;
  G.nx = h->cfg.nx;
  G.ny = h->cfg.ny;
  G.nz = h->cfg.nz;
  G.N = h->N;
  G.links = h->links;
  return G;
}

// Forward + loss (+ backward into nn.g when grad) on the field in nn.x0.
// Returns the loss.
lbm_status loss_grad(lbm_t* h, bool grad, double* loss) {
  NNet& n = *h->nn;
  const Geo G = geo_of(h);
  const unsigned b = nb(G.N, 256);
  const unsigned gr = (unsigned)std::min<int64_t>(b, h->grid_cap);
  LBM_CUDA_TRY(h, cudaMemsetAsync(n.red, 0, 2 * sizeof(double), h->st));
  k_sum_sq<<<gr, 256, 0, h->st>>>(n.x0, G.N, n.red);
#define LBM_NN_C(KERNEL, ...)                                               \
  do {                                                                      \
    if (n.C <= 4) KERNEL<4><<<b, 256, 0, h->st>>>(__VA_ARGS__);             \
    else if (n.C <= 8) KERNEL<8><<<b, 256, 0, h->st>>>(__VA_ARGS__);        \
    else KERNEL<16><<<b, 256, 0, h->st>>>(__VA_ARGS__);                     \
  } while (0)
  LBM_NN_C(k_nn_layer1, n.x0, n.p, n.C, G, n.hid);
  LBM_NN_C(k_nn_layer2, n.hid, n.p, n.C, G, n.y);
  k_nn_res<<<gr, 256, 0, h->st>>>(n.x0, n.y, G, n.res, n.red);
  h->launches += 4;
  if (grad) {
    k_nn_gy<<<b, 256, 0, h->st>>>(n.res, G, n.red, n.gy);
    LBM_NN_C(k_nn_ga, n.gy, n.hid, n.p, n.C, G, n.ga);
    LBM_CUDA_TRY(h, cudaMemsetAsync(n.g, 0, n.np * sizeof(float), h->st));
    // a few waves of CTAs, at most one per column of 32 x
    const int nwork = G.nz * ((G.nx + 31) / 32);
    const int per = std::max(1, std::min(nwork, (2 * h->grid_cap + 3 * n.C - 1) / (3 * n.C)));
    k_nn_wgrad<<<dim3((unsigned)per, (unsigned)(3 * n.C)), 32 * WG_WARPS, 0, h->st>>>(
        n.gy, n.ga, n.hid, n.x0, n.C, G, nwork, n.g);
    h->launches += 3;
  }
#undef LBM_NN_C
  LBM_CUDA_TRY(h, cudaGetLastError());
  LBM_CUDA_TRY(h, cudaMemcpyAsync(n.hred, n.red, 2 * sizeof(double), cudaMemcpyDeviceToHost, h->st));
  LBM_CUDA_TRY(h, cudaStreamSynchronize(h->st));
  *loss = n.hred[0] > 0 ? n.hred[1] / n.hred[0] : 0.0;
  return LBM_OK;
}

}  // namespace

void nn_free(lbm_t* h) {
  NNet* n = h->nn;
  if (!n) return;
  cudaFree(n->p);
  cudaFree(n->g);
  cudaFree(n->m);
  cudaFree(n->v);
  cudaFree(n->ph);
  cudaFree(n->x0);
  cudaFree(n->hid);
  cudaFree(n->hid16);
  cudaFree(n->xin);
  cudaFree(n->y);
  cudaFree(n->res);
  cudaFree(n->gy);
  cudaFree(n->ga);
  cudaFree(n->red);
  cudaFree(n->pool);
  if (n->hred) cudaFreeHost(n->hred);
  delete n;
  h->nn = nullptr;
}

lbm_status nn_init(lbm_t* h, int hidden, uint64_t seed) {
  if (hidden < 1 || hidden > 16) {
    h->err = "hidden channels must be in 1..16";
    return LBM_EINVAL;
  }
  nn_free(h);
  NNet* n = new NNet();
  h->nn = n;
  n->C = hidden;
  n->np = hidden * 2 * 27 + hidden + hidden * 27;
  const int64_t N = h->N;
  bool ok = cudaMalloc(&n->p, n->np * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&n->g, n->np * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&n->m, n->np * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&n->v, n->np * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&n->ph, n->np * sizeof(__half)) == cudaSuccess &&
            cudaMalloc(&n->x0, N * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&n->hid, (size_t)hidden * N * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&n->hid16, (size_t)hidden * N * sizeof(__half)) == cudaSuccess &&
            cudaMalloc(&n->xin, N * sizeof(__half2)) == cudaSuccess &&
            cudaMalloc(&n->y, N * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&n->res, N * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&n->gy, N * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&n->ga, (size_t)hidden * N * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&n->red, 2 * sizeof(double)) == cudaSuccess &&
            cudaMallocHost(&n->hred, 2 * sizeof(double)) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    nn_free(h);
    h->err = "network allocation failed";
    return LBM_ENOMEM;
  }
  // He-style uniform initialisation, seeded; small output layer
  std::mt19937_64 rng(seed);
  std::uniform_real_distribution<float> U(-1.f, 1.f);
  std::vector<float> p(n->np, 0.f);
  const float a1 = sqrtf(3.f / (2.f * 27.f)), a2 = 0.1f * sqrtf(3.f / (hidden * 27.f));
  for (int k = 0; k < hidden * 2 * 27; ++k) p[k] = a1 * U(rng);
  for (int k = 0; k < hidden * 27; ++k) p[hidden * 2 * 27 + hidden + k] = a2 * U(rng);
  LBM_CUDA_TRY(h, cudaMemcpyAsync(n->p, p.data(), n->np * sizeof(float), cudaMemcpyHostToDevice, h->st));
  LBM_CUDA_TRY(h, cudaMemsetAsync(n->m, 0, n->np * sizeof(float), h->st));
  LBM_CUDA_TRY(h, cudaMemsetAsync(n->v, 0, n->np * sizeof(float), h->st));
  k_to_half<<<nb(n->np, 256), 256, 0, h->st>>>(n->p, n->ph, n->np);
  LBM_CUDA_TRY(h, cudaGetLastError());
  LBM_CUDA_TRY(h, cudaStreamSynchronize(h->st));
  return LBM_OK;
}

lbm_status nn_collect(lbm_t* h, int capacity) {
  NNet* n = h->nn;
  if (!n) {
    h->err = "network not initialised";
    return LBM_EINVAL;
  }
  if (capacity <= 0) {
    n->collect = false;
    return LBM_OK;
  }
  if (capacity != n->cap) {
    cudaFree(n->pool);
    n->pool = nullptr;
    if (cudaMalloc(&n->pool, (size_t)capacity * h->N * sizeof(float)) != cudaSuccess) {
      cudaGetLastError();
      n->cap = 0;
      h->err = "training pool allocation failed";
      return LBM_ENOMEM;
    }
    n->cap = capacity;
    n->count = n->next = 0;
  }
  n->collect = true;
  return LBM_OK;
}

// Called by the solver with the initial residual (FP32, box-indexed: planes
// [zlo, zlo + nzb); colour-split when hx > 0) and its rms.  Stores it when collecting; applies the
// learned correction when in use.  Returns the relative change of the
// residual norm the caller must verify (the caller reverts on failure).
lbm_status nn_before_solve(lbm_t* h, const float* r, int zlo, int nzb, int hx, double rms,
                           bool* applied, float** dpsi_out) {
  *applied = false;
  NNet* n = h->nn;
  if (!n || rms <= 0.0 || !isfinite(rms)) return LBM_OK;
  const Geo G = geo_of(h);
  const unsigned b = nb(G.N, 256);
  const bool fast = n->C == 2 || n->C == 4 || n->C == 8 || n->C == 16;
  if (n->collect || n->use) {
    k_nn_input<<<b, 256, 0, h->st>>>(r, zlo, nzb, hx, (float)(1.0 / rms), G, n->x0,
                                      n->use && fast ? n->xin : nullptr);
    ++h->launches;
  }
  if (n->collect && n->cap > 0) {
    LBM_CUDA_TRY(h, cudaMemcpyAsync(n->pool + (size_t)n->next * G.N, n->x0, G.N * sizeof(float),
                                    cudaMemcpyDeviceToDevice, h->st));
    n->next = (n->next + 1) % n->cap;
    n->count = std::min(n->count + 1, n->cap);
  }
  if (n->use) {
    if (fast) {
      if (n->hp_stale) {
        n->hp.resize(n->np);
        LBM_CUDA_TRY(h, cudaMemcpyAsync(n->hp.data(), n->p, n->np * sizeof(float), cudaMemcpyDeviceToHost,
                                        h->st));
        LBM_CUDA_TRY(h, cudaStreamSynchronize(h->st));
        n->hp_stale = false;
      }
      int64_t* psi = h->ps.psi[h->ps.cur];
      cudaError_t e = n->C == 2   ? fast_infer<2>(n, G, (float)rms, psi, h->st)
                      : n->C == 4 ? fast_infer<4>(n, G, (float)rms, psi, h->st)
                      : n->C == 8 ? fast_infer<8>(n, G, (float)rms, psi, h->st)
                                  : fast_infer<16>(n, G, (float)rms, psi, h->st);
      LBM_CUDA_TRY(h, e);
      h->launches += 2;
    } else {
      k_nn_infer1<<<b, 256, 0, h->st>>>(n->x0, n->ph, n->C, G, n->hid16);
      k_nn_infer2<<<b, 256, 0, h->st>>>(n->hid16, n->ph, n->C, G, (float)rms, n->y);
      k_nn_apply<<<b, 256, 0, h->st>>>(h->ps.psi[h->ps.cur], n->y, G.N, +1);
      h->launches += 3;
    }
    LBM_CUDA_TRY(h, cudaGetLastError());
    *applied = true;
    *dpsi_out = n->y;
    ++n->tried;
  }
  return LBM_OK;
}

lbm_status nn_revert(lbm_t* h, const float* dpsi) {
  k_nn_apply<<<nb(h->N, 256), 256, 0, h->st>>>(h->ps.psi[h->ps.cur], dpsi, h->N, -1);
  ++h->launches;
  LBM_CUDA_TRY(h, cudaGetLastError());
  return LBM_OK;
}

bool nn_active(const lbm_t* h) { return h->nn && (h->nn->collect || h->nn->use); }

void nn_stats(const lbm_t* h, double* out) {
  const NNet* n = h->nn;
  out[0] = n ? (double)n->tried : 0.0;
  out[1] = n ? (double)n->accepted : 0.0;
  out[2] = (n && n->accepted) ? n->sum_ratio / n->accepted : 0.0;
  out[3] = n ? (double)n->count : 0.0;
  out[4] = n ? (double)n->np : 0.0;
}

lbm_status nn_set_use(lbm_t* h, int enable) {
  if (!h->nn) {
    h->err = "network not initialised";
    return LBM_EINVAL;
  }
  h->nn->use = enable != 0;
  return LBM_OK;
}

void nn_record(lbm_t* h, double ratio) {
  if (!h->nn) return;
  h->nn->accepted += 1;
  h->nn->sum_ratio += ratio;
}

lbm_status nn_train(lbm_t* h, int epochs, double lr, double* losses) {
  NNet* n = h->nn;
  if (!n || n->count == 0) {
    h->err = "no network or no collected training residuals";
    return LBM_EINVAL;
  }
  for (int e = 0; e < epochs; ++e) {
    double tot = 0.0;
    for (int k = 0; k < n->count; ++k) {
      LBM_CUDA_TRY(h, cudaMemcpyAsync(n->x0, n->pool + (size_t)k * h->N, h->N * sizeof(float),
                                      cudaMemcpyDeviceToDevice, h->st));
      double L = 0.0;
      lbm_status s = loss_grad(h, true, &L);
      if (s != LBM_OK) return s;
      tot += L;
      ++n->adam_t;
      k_adam<<<nb(n->np, 256), 256, 0, h->st>>>(n->p, n->g, n->m, n->v, n->np, (float)lr, 0.9f,
                                                0.999f, 1e-8f, n->adam_t, n->ph);
      n->hp_stale = true;
      ++h->launches;
      LBM_CUDA_TRY(h, cudaGetLastError());
    }
    if (losses) losses[e] = tot / n->count;
  }
  LBM_CUDA_TRY(h, cudaStreamSynchronize(h->st));
  return LBM_OK;
}

lbm_status nn_loss_grad_host(lbm_t* h, const float* x0_host, double* loss, float* grad_host) {
  NNet* n = h->nn;
  if (!n) {
    h->err = "network not initialised";
    return LBM_EINVAL;
  }
  LBM_CUDA_TRY(h, cudaMemcpyAsync(n->x0, x0_host, h->N * sizeof(float), cudaMemcpyHostToDevice, h->st));
  lbm_status s = loss_grad(h, grad_host != nullptr, loss);
  if (s != LBM_OK) return s;
  if (grad_host) {
    LBM_CUDA_TRY(h, cudaMemcpy(grad_host, n->g, n->np * sizeof(float), cudaMemcpyDeviceToHost));
  }
  return LBM_OK;
}

lbm_status nn_infer_host(lbm_t* h, const float* x0_host, float* y_host) {
  NNet* n = h->nn;
  if (!n) {
    h->err = "network not initialised";
    return LBM_EINVAL;
  }
  const Geo G = geo_of(h);
  const unsigned b = nb(G.N, 256);
  const bool fast = n->C == 2 || n->C == 4 || n->C == 8 || n->C == 16;
  LBM_CUDA_TRY(h, cudaMemcpyAsync(n->x0, x0_host, h->N * sizeof(float), cudaMemcpyHostToDevice, h->st));
  // the same packing as for a solver residual (sigma 1, every plane)
  k_nn_input<<<b, 256, 0, h->st>>>(n->x0, 0, h->cfg.nz, 0, 1.0f, G, n->x0, fast ? n->xin : nullptr);
  ++h->launches;
  if (fast) {
    int64_t* scratch = nullptr;
    LBM_CUDA_TRY(h, cudaMalloc(&scratch, h->N * sizeof(int64_t)));
    cudaMemsetAsync(scratch, 0, h->N * sizeof(int64_t), h->st);
    if (n->hp_stale) {
      n->hp.resize(n->np);
      cudaMemcpyAsync(n->hp.data(), n->p, n->np * sizeof(float), cudaMemcpyDeviceToHost, h->st);
      cudaStreamSynchronize(h->st);
      n->hp_stale = false;
    }
    cudaError_t e = n->C == 2   ? fast_infer<2>(n, G, 1.0f, scratch, h->st)
                    : n->C == 4 ? fast_infer<4>(n, G, 1.0f, scratch, h->st)
                    : n->C == 8 ? fast_infer<8>(n, G, 1.0f, scratch, h->st)
                                : fast_infer<16>(n, G, 1.0f, scratch, h->st);
    cudaStreamSynchronize(h->st);
    cudaFree(scratch);
    LBM_CUDA_TRY(h, e);
    h->launches += 2;
  } else {
    k_nn_infer1<<<b, 256, 0, h->st>>>(n->x0, n->ph, n->C, G, n->hid16);
    k_nn_infer2<<<b, 256, 0, h->st>>>(n->hid16, n->ph, n->C, G, 1.0f, n->y);
    h->launches += 2;
    LBM_CUDA_TRY(h, cudaGetLastError());
  }
  LBM_CUDA_TRY(h, cudaMemcpyAsync(y_host, n->y, h->N * sizeof(float), cudaMemcpyDeviceToHost, h->st));
  LBM_CUDA_TRY(h, cudaStreamSynchronize(h->st));
  return LBM_OK;
}

lbm_status nn_params(lbm_t* h, float* get, const float* set, int* np) {
  NNet* n = h->nn;
  if (!n) {
    h->err = "network not initialised";
    return LBM_EINVAL;
  }
  if (np) *np = n->np;
  if (get) {
    LBM_CUDA_TRY(h, cudaMemcpyAsync(get, n->p, n->np * sizeof(float), cudaMemcpyDeviceToHost, h->st));
    LBM_CUDA_TRY(h, cudaStreamSynchronize(h->st));
  }
  if (set) {
    LBM_CUDA_TRY(h, cudaMemcpyAsync(n->p, set, n->np * sizeof(float), cudaMemcpyHostToDevice, h->st));
    n->hp_stale = true;
    k_to_half<<<nb(n->np, 256), 256, 0, h->st>>>(n->p, n->ph, n->np);
    LBM_CUDA_TRY(h, cudaGetLastError());
    LBM_CUDA_TRY(h, cudaStreamSynchronize(h->st));
  }
  return LBM_OK;
}

}  // namespace lbm_gb300
