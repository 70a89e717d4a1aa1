// Learned subgrid closure for coarse-order runs: per-element order projection, a small MLP
// (135 -> 128 -> 128 -> 135, SiLU, BF16 weights, FP32 accumulation) with forward, backward and Adam
// kernels, and its use inside the residual / RK path.  The paper names subgrid-scale modelling as
// future work (Section 8); the network and its training data are defined by the workload.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <numeric>
#include <random>
#include <vector>

#include "chorus.h"
#include "closure.h"
#include "internal.h"
#include "sd_tables.h"

namespace chorus {

// ------------------------------------------------------------------ record layout

size_t closure_record_bytes() { return (size_t)ClosureLayout::total_bytes; }

// ------------------------------------------------------------------ projection matrix (host)

// 1D L2 projection from Nf to Nc solution points on [0,1] (reference cube, unweighted):
// P = M_c^{-1} B with M_c[a][b] = int h^c_a h^c_b, B[a][s] = int h^c_a h^f_s (Gauss-Legendre).
std::vector<double> projection_matrix(int Nf, int Nc) {
  const Tables1D tf = make_tables(Nf), tc = make_tables(Nc);
  const int G = Nf + Nc;
  const double pi = 3.14159265358979323846;
  std::vector<double> gx(G), gw(G);
  for (int k = 1; k <= G; ++k) {
    double t = std::cos(pi * (k - 0.25) / (G + 0.5));
    for (int it = 0; it < 100; ++it) {
      double v, d;
      legendre(G, t, &v, &d);
      const double dt = v / d;
      t -= dt;
      if (std::fabs(dt) < 1e-17) break;
    }
    double v, d;
    legendre(G, t, &v, &d);
    gx[k - 1] = 0.5 * (t + 1.0);
    gw[k - 1] = 1.0 / ((1.0 - t * t) * d * d);
  }
  std::vector<double> M(Nc * Nc, 0.0), B(Nc * Nf, 0.0);
  for (int g = 0; g < G; ++g) {
    for (int a = 0; a < Nc; ++a) {
      const double ha = lag(tc.Xs, a, gx[g]);
      for (int b = 0; b < Nc; ++b) M[a * Nc + b] += gw[g] * ha * lag(tc.Xs, b, gx[g]);
      for (int s = 0; s < Nf; ++s) B[a * Nf + s] += gw[g] * ha * lag(tf.Xs, s, gx[g]);
    }
  }
  // solve M P = B by Gauss-Jordan elimination with partial pivoting
  for (int c = 0; c < Nc; ++c) {
    int piv = c;
    for (int r = c + 1; r < Nc; ++r)
      if (std::fabs(M[r * Nc + c]) > std::fabs(M[piv * Nc + c])) piv = r;
    if (piv != c) {
      for (int k = 0; k < Nc; ++k) std::swap(M[c * Nc + k], M[piv * Nc + k]);
      for (int k = 0; k < Nf; ++k) std::swap(B[c * Nf + k], B[piv * Nf + k]);
    }
    const double d = M[c * Nc + c];
    for (int k = 0; k < Nc; ++k) M[c * Nc + k] /= d;
    for (int k = 0; k < Nf; ++k) B[c * Nf + k] /= d;
    for (int r = 0; r < Nc; ++r) {
      if (r == c) continue;
      const double f = M[r * Nc + c];
      for (int k = 0; k < Nc; ++k) M[r * Nc + k] -= f * M[c * Nc + k];
      for (int k = 0; k < Nf; ++k) B[r * Nf + k] -= f * B[c * Nf + k];
    }
  }
  return B;
}

// ------------------------------------------------------------------ projection kernel

struct ProjArg {
  double P[kMaxN][kMaxN];  // [Nc][Nf]
  int Nf, Nc;
};

// Qc[e] = Pi(Qf[e]) along the three axes; `add_f`/`sub_c` add the fine background before and
// subtract the coarse one after (perturbation storage), all in FP64.
template <class R>
__global__ void k_project(int64_t E, ProjArg pa, const R* __restrict__ Qf, R* __restrict__ Qc,
                          const double* __restrict__ add_f, const double* __restrict__ sub_c, int nvar) {
  const int64_t e = blockIdx.x;
  if (e >= E) return;
  const int Nf = pa.Nf, Nc = pa.Nc;
  const int N3f = Nf * Nf * Nf, N3c = Nc * Nc * Nc;
  __shared__ double a[kMaxN * kMaxN * kMaxN], b[kMaxN * kMaxN * kMaxN], c[kMaxN * kMaxN * kMaxN];
  for (int v = 0; v < nvar; ++v) {
    for (int i = threadIdx.x; i < N3f; i += blockDim.x) {
      double x = (double)Qf[(e * nvar + v) * N3f + i];
      if (add_f) x += add_f[(e * nvar + v) * N3f + i];
      a[i] = x;
    }
    __syncthreads();
    // along i: b[k][j][ci] = sum_s P[ci][s] a[k][j][s]
    for (int t = threadIdx.x; t < Nf * Nf * Nc; t += blockDim.x) {
      const int ci = t % Nc, kj = t / Nc;
      double s = 0;
      for (int q = 0; q < Nf; ++q) s += pa.P[ci][q] * a[kj * Nf + q];
      b[kj * Nc + ci] = s;
    }
    __syncthreads();
    // along j: c[k][cj][ci]
    for (int t = threadIdx.x; t < Nf * Nc * Nc; t += blockDim.x) {
      const int ci = t % Nc, cj = (t / Nc) % Nc, k = t / (Nc * Nc);
      double s = 0;
      for (int q = 0; q < Nf; ++q) s += pa.P[cj][q] * b[(k * Nf + q) * Nc + ci];
      c[(k * Nc + cj) * Nc + ci] = s;
    }
    __syncthreads();
    // along k
    for (int t = threadIdx.x; t < N3c; t += blockDim.x) {
      const int ij = t % (Nc * Nc), ck = t / (Nc * Nc);
      double s = 0;
      for (int q = 0; q < Nf; ++q) s += pa.P[ck][q] * c[q * Nc * Nc + ij];
      if (sub_c) s -= sub_c[(e * nvar + v) * N3c + t];
      Qc[(e * nvar + v) * N3c + t] = (R)s;
    }
    __syncthreads();
  }
}

ProjArg proj_arg(int Nf, int Nc) {
  ProjArg pa{};
  pa.Nf = Nf;
  pa.Nc = Nc;
  const std::vector<double> P = projection_matrix(Nf, Nc);
  for (int a = 0; a < Nc; ++a)
    for (int s = 0; s < Nf; ++s) pa.P[a][s] = P[a * Nf + s];
  return pa;
}

cudaError_t launch_project(int64_t E, int Nf, int Nc, int prec, const void* Qf, void* Qc, const double* add_f,
                           const double* sub_c, int nvar, cudaStream_t st) {
  const ProjArg pa = proj_arg(Nf, Nc);
  if (prec == 0)
    k_project<double><<<(unsigned)E, 128, 0, st>>>(E, pa, (const double*)Qf, (double*)Qc, add_f, sub_c, nvar);
  else
    k_project<float><<<(unsigned)E, 128, 0, st>>>(E, pa, (const float*)Qf, (float*)Qc, add_f, sub_c, nvar);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ network kernels

namespace {

constexpr int NI = ClosureLayout::NI, NH = ClosureLayout::NH, NO = ClosureLayout::NO;
// Row strides of the tiles in shared memory, in words: multiples of 4 (16-byte loads along a row), the
// rows of a weight matrix an odd number of 8-byte units apart (a warp reads 32 of them at once).
constexpr int SX = 136;                      // inputs and outputs (135, the last column zero)
constexpr int SH = 132;                      // hidden layers (128)
constexpr int SW1 = 140, SW2 = 132;          // BF16: W1; W2 and W3
constexpr int kWords = NH * SW1 > (NO + 1) * SW2 ? NH * SW1 : (NO + 1) * SW2;

struct Rec {
  const __nv_bfloat16* W1;
  const __nv_bfloat16* W2;
  const __nv_bfloat16* W3;
  const float* b1;
  const float* b2;
  const float* b3;
  const float* in_scale;
  const float* out_scale;
};

__host__ __device__ inline Rec rec_of(const void* w) {
  const unsigned char* p = (const unsigned char*)w;
  Rec r;
  r.W1 = (const __nv_bfloat16*)(p + ClosureLayout::oW1);
  r.W2 = (const __nv_bfloat16*)(p + ClosureLayout::oW2);
  r.W3 = (const __nv_bfloat16*)(p + ClosureLayout::oW3);
  r.b1 = (const float*)(p + ClosureLayout::ob1);
  r.b2 = (const float*)(p + ClosureLayout::ob2);
  r.b3 = (const float*)(p + ClosureLayout::ob3);
  r.in_scale = (const float*)(p + ClosureLayout::oin);
  r.out_scale = (const float*)(p + ClosureLayout::oout);
  return r;
}

__device__ __forceinline__ float silu_f(float z) { return z / (1.0f + expf(-z)); }
__device__ __forceinline__ float silu_g(float z) {
  const float s = 1.0f / (1.0f + expf(-z));
  return s * (1.0f + z * (1.0f - s));
}

// The tile of a CTA: TB samples, TB / 4 warps; a warp's lanes share four sample rows.
template <int TB>
struct Tile {
  static constexpr int threads = 8 * TB;
  float X[TB * SX];
  float z1[TB * SH];  // pre-activations, then (backward) dL/dz
  float z2[TB * SH];
  float h[TB * SH];   // the activations in use
  float y[TB * SX];   // output, then dL/dy
  __nv_bfloat16 W[kWords];
};

// W1 ([NH][NI], rows of odd length) into shared memory at row stride SW1, its columns past NI zero.
template <int TB>
__device__ __forceinline__ void stage_w1(const __nv_bfloat16* __restrict__ Wg, __nv_bfloat16* sW) {
  const int lane = threadIdx.x & 31;
  const unsigned short* src = reinterpret_cast<const unsigned short*>(Wg);
  for (int c = threadIdx.x >> 5; c < NH; c += TB / 4)
#pragma unroll
    for (int k = lane; k < SW1; k += 32)
      reinterpret_cast<unsigned short*>(sW)[c * SW1 + k] = k < NI ? __ldg(src + c * NI + k) : (unsigned short)0;
}

// W2 or W3 ([ROWS][NH], a warp a row) at row stride SW2; a zero row after an odd number of rows.  The
// record needs the 4-byte alignment of its FP32 fields only: rows that do not start on an 8-byte boundary
// (the same for all of a matrix) are read in 4-byte halves.
template <int TB, int ROWS>
__device__ __forceinline__ void stage_w(const __nv_bfloat16* __restrict__ Wg, __nv_bfloat16* sW) {
  static_assert(ClosureLayout::oW2 % 8 == 0 && ClosureLayout::oW3 % 8 == 0 && NH == 128, "rows of 32 8-byte units");
  const int lane = threadIdx.x & 31;
  const bool v8 = ((uintptr_t)Wg & 7u) == 0;
  for (int c = threadIdx.x >> 5; c < ROWS + ROWS % 2; c += TB / 4) {
    uint2 v = make_uint2(0u, 0u);
    if (c < ROWS) {
      if (v8) {
        v = __ldg(reinterpret_cast<const uint2*>(Wg + c * NH) + lane);
      } else {
        const unsigned* h = reinterpret_cast<const unsigned*>(Wg + c * NH) + 2 * lane;
        v = make_uint2(__ldg(h), __ldg(h + 1));
      }
    }
    *reinterpret_cast<uint2*>(sW + c * SW2 + 4 * lane) = v;
  }
}

__device__ __forceinline__ void bf16x4(const __nv_bfloat16* p, float w[4]) {
  const uint2 v = *reinterpret_cast<const uint2*>(p);
  w[0] = __uint_as_float(v.x << 16);
  w[1] = __uint_as_float(v.x & 0xffff0000u);
  w[2] = __uint_as_float(v.y << 16);
  w[3] = __uint_as_float(v.y & 0xffff0000u);
}

__device__ __forceinline__ void load4(const float* p, float v[4]) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  v[0] = t.x;
  v[1] = t.y;
  v[2] = t.z;
  v[3] = t.w;
}

// out[r][c] = bias[c] + sum_k A[r][k] W[c][k], k in order, for the warp's rows: four rows by the columns
// lane + 32 j a thread (16 sums; per four k four broadcast and four 8-byte loads for 64 products), the
// columns past 128 one sum a lane.
template <int K, int stride, int NCOL>
__device__ __forceinline__ void dense(const float* A, int lda, const __nv_bfloat16* sW, const float* __restrict__ bias,
                                      float* out, int ldo) {
  const int lane = threadIdx.x & 31, r0 = 4 * (threadIdx.x >> 5);
  float acc[4][4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float b = __ldg(bias + lane + 32 * j);
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i][j] = b;
  }
#pragma unroll 2
  for (int k = 0; k < K; k += 4) {
    float a[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) load4(A + (r0 + i) * lda + k, a[i]);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float w[4];
      bf16x4(sW + (lane + 32 * j) * stride + k, w);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int t = 0; t < 4; ++t) acc[i][j] = fmaf(a[i][t], w[t], acc[i][j]);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) out[(r0 + i) * ldo + lane + 32 * j] = acc[i][j];
  constexpr int X = NCOL - 128;
  if (X > 0 && lane < 4 * X) {
    const int r = r0 + lane / (X > 0 ? X : 1), c = 128 + lane % (X > 0 ? X : 1);
    float s = __ldg(bias + c);
#pragma unroll 4
    for (int k = 0; k < K; k += 4) {
      float a[4], w[4];
      load4(A + r * lda + k, a);
      bf16x4(sW + c * stride + k, w);
#pragma unroll
      for (int t = 0; t < 4; ++t) s = fmaf(a[t], w[t], s);
    }
    out[r * ldo + c] = s;
  }
}

// h = SiLU(z) for the warp's rows
__device__ __forceinline__ void activate(const float* z, float* h) {
  const int lane = threadIdx.x & 31, r0 = 4 * (threadIdx.x >> 5);
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) h[(r0 + i) * SH + lane + 32 * j] = silu_f(z[(r0 + i) * SH + lane + 32 * j]);
}

// Rows r0 .. of [..][135] samples into the tile (zero past `rows` and in the last column).
template <int TB>
__device__ __forceinline__ void load_rows(const float* __restrict__ X, int64_t r0, int rows, float* dst) {
  for (int i = threadIdx.x; i < TB * SX; i += Tile<TB>::threads) {
    const int r = i / SX, k = i % SX;
    dst[i] = r < rows && k < NI ? __ldg(X + (r0 + r) * NI + k) : 0.f;
  }
}

// Forward pass of the tile's samples: leaves z1, z2, h = SiLU(z2) and y.  A warp computes its own rows
// of every layer; only the weights in shared memory are common.
template <int TB>
__device__ __forceinline__ void forward_tile(const Rec& w, Tile<TB>& s) {
  stage_w1<TB>(w.W1, s.W);
  __syncthreads();
  dense<NI + 1, SW1, NH>(s.X, SX, s.W, w.b1, s.z1, SH);
  __syncwarp();
  activate(s.z1, s.h);
  __syncthreads();
  stage_w<TB, NH>(w.W2, s.W);
  __syncthreads();
  dense<NH, SW2, NH>(s.h, SH, s.W, w.b2, s.z2, SH);
  __syncwarp();
  activate(s.z2, s.h);
  __syncthreads();
  stage_w<TB, NO>(w.W3, s.W);
  __syncthreads();
  dense<NH, SW2, NO>(s.h, SH, s.W, w.b3, s.y, SX);
}

// z[r][k] <- (sum_c D[r][c] W[c][k]) SiLU'(z[r][k]), c in order to C (a multiple of four), for the warp's
// rows (zero past `rows`): four rows by four consecutive columns a thread.
template <int C>
__device__ __forceinline__ void backward_data(const float* D, int ldd, const __nv_bfloat16* sW, float* z, int rows) {
  const int lane = threadIdx.x & 31, r0 = 4 * (threadIdx.x >> 5);
  float acc[4][4] = {};
#pragma unroll 2
  for (int c = 0; c < C; c += 4) {
    float d[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) load4(D + (r0 + i) * ldd + c, d[i]);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      float w[4];
      bf16x4(sW + (c + t) * SW2 + 4 * lane, w);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[i][u] = fmaf(d[i][t], w[u], acc[i][u]);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float v[4];
    load4(z + (r0 + i) * SH + 4 * lane, v);
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = r0 + i < rows ? acc[i][u] * silu_g(v[u]) : 0.f;
    *reinterpret_cast<float4*>(z + (r0 + i) * SH + 4 * lane) = make_float4(v[0], v[1], v[2], v[3]);
  }
}

// gW[c][k] += sum_r D[r][c] A[r][k] over the tile, c < NC, k < NK: up to 128 x 128 eight c by four
// consecutive k a thread (32 sums; per sample two broadcast and one 16-byte load), the rows and columns
// past that one sum a thread; gb[c] += sum_r D[r][c].  v4: the rows of gW are 16-byte aligned (vector
// atomics).
template <int TB, int NC, int NK>
__device__ __forceinline__ void backward_weights(const float* D, int ldd, const float* A, int lda, float* gW, float* gb,
                                                 bool v4) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int c0 = 8 * warp; c0 < 128; c0 += 2 * TB) {
    float acc[8][4] = {};
#pragma unroll 4
    for (int r = 0; r < TB; ++r) {
      float d[8], a[4];
      load4(D + r * ldd + c0, d);
      load4(D + r * ldd + c0 + 4, d + 4);
      load4(A + r * lda + 4 * lane, a);
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[i][u] = fmaf(d[i], a[u], acc[i][u]);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float* g = gW + (size_t)(c0 + i) * NK + 4 * lane;
      if (v4) {
        atomicAdd(reinterpret_cast<float4*>(g), make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]));
      } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) atomicAdd(g + u, acc[i][u]);
      }
    }
  }
  constexpr int XC = NC - 128, XK = NK - 128;
  static_assert(XC == 0 || XK == 0, "one of the two is 128");
  for (int i = threadIdx.x; i < XC * 128 + XK * 128; i += Tile<TB>::threads) {
    const int c = XC > 0 ? 128 + i / 128 : i / (XK > 0 ? XK : 1), k = XC > 0 ? i % 128 : 128 + i % (XK > 0 ? XK : 1);
    float s = 0.f;
#pragma unroll 8
    for (int r = 0; r < TB; ++r) s = fmaf(D[r * ldd + c], A[r * lda + k], s);
    atomicAdd(gW + (size_t)c * NK + k, s);
  }
  for (int c = threadIdx.x; c < NC; c += Tile<TB>::threads) {
    float s = 0.f;
#pragma unroll 8
    for (int r = 0; r < TB; ++r) s += D[r * ldd + c];
    atomicAdd(gb + c, s);
  }
}

}  // namespace

// Y = MLP(X) for n samples ([n][135] FP32, row-major).
template <int TB>
__global__ void __launch_bounds__(Tile<TB>::threads)
    k_mlp_forward(const void* weights, const float* __restrict__ X, float* __restrict__ Y, int64_t n) {
  extern __shared__ __align__(16) unsigned char smraw[];
  Tile<TB>& s = *reinterpret_cast<Tile<TB>*>(smraw);
  const Rec w = rec_of(weights);
  const int64_t r0 = (int64_t)blockIdx.x * TB;
  const int rows = (int)((n - r0) < TB ? (n - r0) : TB);
  load_rows<TB>(X, r0, rows, s.X);
  forward_tile<TB>(w, s);
  __syncthreads();
  for (int i = threadIdx.x; i < rows * NO; i += Tile<TB>::threads) Y[r0 * NO + i] = s.y[(i / NO) * SX + i % NO];
}

// Training pairs: X = q'_c / in_scale, Y = (P R_f - R_c) / out_scale per element.
template <class R>
__global__ void k_make_pairs(const void* weights, const R* __restrict__ Qc, const double* __restrict__ Q0,
                             const R* __restrict__ PRf, const R* __restrict__ Rc, float* __restrict__ X,
                             float* __restrict__ Y, int64_t E) {
  const Rec w = rec_of(weights);
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= E * NI) return;
  const int v = (int)(i % NI) / 27;
  double q = (double)Qc[i];
  if (Q0) q -= Q0[i];
  X[i] = (float)(q / (double)w.in_scale[v]);
  Y[i] = (float)(((double)PRf[i] - (double)Rc[i]) / (double)w.out_scale[v]);
}

// Gradient of L = sum (y - t)^2 / (2 n_total) over the CTA's samples, accumulated into
// grad (FP32, layout of ClosureLayout::master) with atomics; loss partial into *loss.  FP32 products
// (bound by the FMA rate: 2.5 GFLOP for 8,192 samples, 32 us at 78 TFLOP/s): register tiles of 16 and 32
// sums a thread, everything between the global inputs and the atomics in shared memory.
template <int TB>
__global__ void __launch_bounds__(Tile<TB>::threads)
    k_mlp_backward(const void* weights, const float* __restrict__ X, const float* __restrict__ T, int64_t row0,
                   int64_t rows_total, float* __restrict__ grad, double* __restrict__ loss) {
  extern __shared__ __align__(16) unsigned char smraw[];
  Tile<TB>& s = *reinterpret_cast<Tile<TB>*>(smraw);
  const Rec w = rec_of(weights);
  const int64_t r0 = row0 + (int64_t)blockIdx.x * TB;
  const int64_t left = row0 + rows_total - r0;
  const int rows = (int)(left < 0 ? 0 : (left < TB ? left : TB));
  load_rows<TB>(X, r0, rows, s.X);
  forward_tile<TB>(w, s);
  __syncthreads();
  // dY = (y - t) / n_total, loss partial (y's last column becomes zero)
  const double inv_n = 1.0 / ((double)rows_total * NO);
  double lp = 0.0;
  for (int i = threadIdx.x; i < TB * SX; i += Tile<TB>::threads) {
    const int r = i / SX, k = i % SX;
    float d = 0.f;
    if (r < rows && k < NO) {
      const float diff = s.y[i] - __ldg(T + (r0 + r) * NO + k);
      lp += 0.5 * (double)diff * diff;
      d = (float)(diff * inv_n);
    }
    s.y[i] = d;  // y now holds dY
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) lp += __shfl_xor_sync(0xffffffffu, lp, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(loss, lp * inv_n);
  __syncthreads();
  const bool v4 = ((uintptr_t)grad & 15u) == 0;
  static_assert(ClosureLayout::mW2 % 4 == 0 && ClosureLayout::mW3 % 4 == 0, "aligned rows of W2, W3");
  // dW3 = dY^T h2, db3; dz2 = (dY W3) SiLU'(z2) in place (W3 is still staged)
  backward_weights<TB, NO, NH>(s.y, SX, s.h, SH, grad + ClosureLayout::mW3, grad + ClosureLayout::mb3, v4);
  backward_data<NO + 1>(s.y, SX, s.W, s.z2, rows);
  __syncthreads();
  // dW2 = dz2^T h1, db2; dz1 = (dz2 W2) SiLU'(z1) in place
  activate(s.z1, s.h);
  stage_w<TB, NH>(w.W2, s.W);
  __syncthreads();
  backward_weights<TB, NH, NH>(s.z2, SH, s.h, SH, grad + ClosureLayout::mW2, grad + ClosureLayout::mb2, v4);
  backward_data<NH>(s.z2, SH, s.W, s.z1, rows);
  __syncthreads();
  // dW1 = dz1^T X, db1 (rows of 135: scalar atomics)
  backward_weights<TB, NH, NI>(s.z1, SH, s.X, SX, grad + ClosureLayout::mW1, grad + ClosureLayout::mb1, false);
}

// Adam update of the FP32 master parameters; writes the BF16 weights and FP32 biases of the record.
__global__ void k_adam(float* __restrict__ master, float* __restrict__ m1, float* __restrict__ m2,
                       const float* __restrict__ grad, void* weights, float lr, float b1, float b2, float eps, float c1,
                       float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ClosureLayout::n_params) return;
  const float g = grad[i];
  const float a = b1 * m1[i] + (1.f - b1) * g;
  const float b = b2 * m2[i] + (1.f - b2) * g * g;
  m1[i] = a;
  m2[i] = b;
  const float p = master[i] - lr * (a / c1) / (sqrtf(b / c2) + eps);
  master[i] = p;
  closure_store_param(weights, i, p);
}

// master <- record (BF16 weights widened, FP32 biases)
__global__ void k_load_master(const void* weights, float* __restrict__ master) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ClosureLayout::n_params) return;
  master[i] = closure_load_param(weights, i);
}

template __global__ void k_make_pairs<float>(const void*, const float*, const double*, const float*, const float*,
                                             float*, float*, int64_t);
template __global__ void k_make_pairs<double>(const void*, const double*, const double*, const double*,
                                              const double*, float*, float*, int64_t);

namespace {

template <int TB>
cudaError_t forward_tb(const void* weights, const float* X, float* Y, int64_t n, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(k_mlp_forward<TB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Tile<TB>));
  if (e != cudaSuccess) return e;
  k_mlp_forward<TB><<<(unsigned)((n + TB - 1) / TB), Tile<TB>::threads, sizeof(Tile<TB>), st>>>(weights, X, Y, n);
  return cudaGetLastError();
}

template <int TB>
cudaError_t backward_tb(const void* weights, const float* X, const float* T, int64_t row0, int64_t rows, float* grad,
                        double* loss, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(k_mlp_backward<TB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Tile<TB>));
  if (e != cudaSuccess) return e;
  k_mlp_backward<TB><<<(unsigned)((rows + TB - 1) / TB), Tile<TB>::threads, sizeof(Tile<TB>), st>>>(weights, X, T, row0,
                                                                                                  rows, grad, loss);
  return cudaGetLastError();
}

// Samples per CTA: one CTA per SM either way (its shared memory), so the largest tile, which stages the
// weights and adds the gradients the fewest times, once its CTAs fill half the chip; below that smaller
// tiles, so that a batch of a thousand still spreads over the SMs.  The gradient's error is that of adding
// one partial sum a tile with atomics, which grows with the square root of their number: 16 samples a tile
// only where it is no larger than with 32 (100 samples: 86 instead of 98 us, error 1.95e-7 instead of 2.0e-7;
// 2,400 samples: 98 us either way, but 1.86e-7 instead of 1.38e-7).
constexpr int64_t kWide = 64 * 76, kMid = 32 * 76, kSmall = 128;

}  // namespace

cudaError_t mlp_forward(const void* weights, const float* X, float* Y, int64_t n, cudaStream_t st) {
  return n >= kWide  ? forward_tb<64>(weights, X, Y, n, st)
         : n >= kMid ? forward_tb<32>(weights, X, Y, n, st)
                     : forward_tb<16>(weights, X, Y, n, st);
}

cudaError_t mlp_backward(const void* weights, const float* X, const float* T, int64_t n, int64_t row0, int64_t rows,
                         float* grad, double* loss, cudaStream_t st) {
  return rows >= kWide   ? backward_tb<64>(weights, X, T, row0, rows, grad, loss, st)
         : rows > kSmall ? backward_tb<32>(weights, X, T, row0, rows, grad, loss, st)
                         : backward_tb<16>(weights, X, T, row0, rows, grad, loss, st);
}

cudaError_t make_pairs(int prec, const void* weights, const void* Qc, const double* Q0, const void* PRf,
                       const void* Rc, float* X, float* Y, int64_t E, cudaStream_t st) {
  const int64_t n = E * NI;
  const unsigned nb = (unsigned)((n + 255) / 256);
  if (prec == 0)
    k_make_pairs<double><<<nb, 256, 0, st>>>(weights, (const double*)Qc, Q0, (const double*)PRf, (const double*)Rc, X,
                                             Y, E);
  else
    k_make_pairs<float><<<nb, 256, 0, st>>>(weights, (const float*)Qc, Q0, (const float*)PRf, (const float*)Rc, X, Y,
                                            E);
  return cudaGetLastError();
}

cudaError_t adam(float* master, float* m1, float* m2, const float* grad, void* weights, float lr, float b1, float b2,
                 float eps, int64_t t, cudaStream_t st) {
  const float c1 = 1.f - std::pow(b1, (float)t), c2 = 1.f - std::pow(b2, (float)t);
  k_adam<<<(ClosureLayout::n_params + 255) / 256, 256, 0, st>>>(master, m1, m2, grad, weights, lr, b1, b2, eps, c1,
                                                                c2);
  return cudaGetLastError();
}

cudaError_t load_master(const void* weights, float* master, cudaStream_t st) {
  k_load_master<<<(ClosureLayout::n_params + 255) / 256, 256, 0, st>>>(weights, master);
  return cudaGetLastError();
}

// Seeded host initialisation of a record: uniform weights scaled by sqrt(3 / fan_in) (output layer
// by 0.1), zero biases, given input and output scales.
std::vector<unsigned char> init_record(uint64_t seed, const float* in_scale, const float* out_scale) {
  std::vector<unsigned char> rec(ClosureLayout::total_bytes, 0);
  std::mt19937_64 gen(seed);
  std::uniform_real_distribution<double> uni(-1.0, 1.0);
  auto fill = [&](size_t off, int n_out, int n_in, double scale) {
    __nv_bfloat16* w = (__nv_bfloat16*)(rec.data() + off);
    const double lim = scale * std::sqrt(3.0 / n_in);
    for (int i = 0; i < n_out * n_in; ++i) w[i] = __float2bfloat16_rn((float)(lim * uni(gen)));
  };
  fill(ClosureLayout::oW1, NH, NI, 1.0);
  fill(ClosureLayout::oW2, NH, NH, 1.0);
  fill(ClosureLayout::oW3, NO, NH, 0.1);
  std::memcpy(rec.data() + ClosureLayout::oin, in_scale, 5 * sizeof(float));
  std::memcpy(rec.data() + ClosureLayout::oout, out_scale, 5 * sizeof(float));
  return rec;
}

}  // namespace chorus
