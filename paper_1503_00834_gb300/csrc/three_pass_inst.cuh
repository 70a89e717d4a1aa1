// Launchers of the three-pass kernels for one order N (three_pass.cuh).
#pragma once
#include "three_pass.cuh"

namespace chorus {

// EPB, EPBR: elements per CTA of the FP32 trace and lifting kernels, and of the FP32 residual kernel;
// EPB64: of the FP64 kernels.
template <int N, int EPB, int EPBR, int EPB64>
struct ThreePassInst {
  template <class R>
  using Args = three_pass::KArgs<R>;
  template <int B, class R>
  static cudaError_t trace(const MeshArg<R>& m, const OpsArg<R>& ops, const R* q, R* T, cudaStream_t st) {
    if (m.E == 0) return cudaSuccess;
    three_pass::k_trace<N, R, B><<<(m.E + B - 1) / B, B * N * N, 0, st>>>(m, ops, q, T);
    return cudaGetLastError();
  }
  template <int B, bool KR, class R>
  static cudaError_t grad(const Args<R>& A, cudaStream_t st) {
    constexpr bool PERT = sizeof(R) == 4;
    if (A.m.E == 0) return cudaSuccess;
    const size_t sm = (size_t)three_pass::Layout<N, PERT, R, B>::total_grad * sizeof(R);
    auto* k = three_pass::k_grad<N, PERT, R, B, KR>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k<<<(A.m.E + B - 1) / B, B * N * N, sm, st>>>(A);
    return cudaGetLastError();
  }
  template <class R>
  static cudaError_t face(const Args<R>& A, const int2* faces, int nf, int nw, cudaStream_t st) {
    if (nf + nw == 0) return cudaSuccess;
    const int64_t n = (int64_t)(nf + nw) * N * N;
    three_pass::k_face<N, sizeof(R) == 4, R><<<(unsigned)((n + 63) / 64), 64, 0, st>>>(A, faces, nf, nw);
    return cudaGetLastError();
  }
  template <int B, int MODE, bool KR, class R>
  static cudaError_t resid(const Args<R>& A, cudaStream_t st) {
    constexpr bool PERT = sizeof(R) == 4;
    if (A.m.E == 0) return cudaSuccess;
    const size_t sm = (size_t)three_pass::Layout<N, PERT, R, B, true>::total_resid * sizeof(R);
    auto* k = three_pass::k_resid<N, PERT, R, B, MODE, KR>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k<<<(A.m.E + B - 1) / B, B * N * N, sm, st>>>(A);
    return cudaGetLastError();
  }

  static cudaError_t grad32(const MeshArg<float>& m, const OpsArg<float>& ops, const PhysArg<float>& ph,
                            const BgArg& bg, const float* q, const float* T, float* Tv, float* G, unsigned* err,
                            cudaStream_t st) {
    Args<float> A{};
    A.m = m; A.ops = ops; A.ph = ph; A.bg = bg; A.q = q; A.T = T; A.Tv_out = Tv; A.G_out = G; A.err = err;
    return m.kr != nullptr ? grad<EPB, true>(A, st) : grad<EPB, false>(A, st);
  }
  static cudaError_t face32(const MeshArg<float>& m, const PhysArg<float>& ph, const BgArg& bg, const int2* faces,
                            int nf, int nw, const float* T, const float* Tv, float* Fc, cudaStream_t st) {
    Args<float> A{};
    A.m = m; A.ph = ph; A.bg = bg; A.T = T; A.Tv = Tv; A.Fc_out = Fc;
    return face(A, faces, nf, nw, st);
  }
  static cudaError_t stage32(const MeshArg<float>& m, const OpsArg<float>& ops, const PhysArg<float>& ph,
                             const BgArg& bg, const float* q, const float* G, const float* Fc, float* out,
                             float* T_out, const RkCoef<float>& rk, float dt, unsigned* err, cudaStream_t st) {
    Args<float> A{};
    A.m = m; A.ops = ops; A.ph = ph; A.bg = bg; A.q = q; A.out = out; A.T_out = T_out; A.G_in = G; A.Fc = Fc;
    A.un = rk.un; A.a = rk.a; A.b = rk.b; A.c = rk.c;
    A.un2 = rk.un2; A.out2 = rk.out2; A.a2 = rk.a2; A.b2 = rk.b2; A.c2 = rk.c2; A.radd = rk.radd;
    A.dt = dt; A.err = err;
    return m.kr != nullptr ? resid<EPBR, kModeRK, true>(A, st) : resid<EPBR, kModeRK, false>(A, st);
  }
  // traces, lifted density gradient and residual of an FP64 state
  static cudaError_t background64(const MeshArg<double>& m, const OpsArg<double>& ops, const PhysArg<double>& ph,
                                  const int2* faces, int nf, int nw, const double* q, double* T, double* Tv,
                                  double* grad_rho, double* G, double* Fc, double* R, unsigned* err, cudaStream_t st) {
    Args<double> A{};
    A.m = m; A.ops = ops; A.ph = ph; A.q = q; A.T = T; A.Tv_out = Tv; A.Tv = Tv; A.grad_rho_out = grad_rho;
    A.G_out = G; A.G_in = G; A.Fc_out = Fc; A.Fc = Fc; A.out = R; A.err = err;
    cudaError_t e = trace<EPB64>(m, ops, q, T, st);
    if (e == cudaSuccess) e = grad<EPB64, true>(A, st);
    if (e == cudaSuccess) e = face(A, faces, nf, nw, st);
    if (e == cudaSuccess) e = resid<EPB64, kModeResidual, true>(A, st);
    return e;
  }
  static ThreePassSet set() { return ThreePassSet{trace<EPB, float>, grad32, face32, stage32, background64}; }
};

}  // namespace chorus
