// Launchers of the residual kernels for one order N, for the FP64 total-state form and the FP32
// perturbation form.  Each kern_p<p>.cu instantiates this header once.
#pragma once
#include "sd_kernels.cuh"

namespace chorus {

// EPB64, EPB32: elements per CTA of the volume kernel; EPBU: of the update and trace kernels (the
// kernels share no shared-memory layout, only the per-element arrays in global memory).
template <int N, int EPB64, int EPB32, int EPBU>
struct Inst {
  template <bool PERT, class R, int EPB>
  static cudaError_t trace(const MeshArg<R>& m, const OpsArg<R>& ops, const R* q, R* T, cudaStream_t st) {
    return Launch<N, PERT, R, EPB>::trace(m, ops, q, T, st);
  }
  static cudaError_t vol64(const MeshArg<double>& m, const OpsArg<double>& ops, const PhysArg<double>& ph,
                           const double* q, const double* T, double* Tv, double* part, int* skip, unsigned* err,
                           cudaStream_t st) {
    KArgs<double> A{};
    A.m = m; A.ops = ops; A.ph = ph; A.q = q; A.T = T; A.Tv_out = Tv; A.part_out = part;
    A.skip_out = skip; A.err = err;
    return Launch<N, false, double, EPB64>::vol(A, st);
  }
  static cudaError_t vol32(const MeshArg<float>& m, const OpsArg<float>& ops, const PhysArg<float>& ph,
                           const BgArg& bg, const float* q, const float* T, float* Tv, float* part, int* skip,
                           unsigned* err, cudaStream_t st) {
    KArgs<float> A{};
    A.m = m; A.ops = ops; A.ph = ph; A.bg = bg; A.q = q; A.T = T; A.Tv_out = Tv; A.part_out = part;
    A.skip_out = skip; A.err = err;
    return Launch<N, true, float, EPB32>::vol(A, st);
  }
  static cudaError_t face64(const MeshArg<double>& m, const PhysArg<double>& ph, const int2* faces, int nf, int nw,
                            const double* T, const double* Tv, double* Fc, cudaStream_t st) {
    KArgs<double> A{};
    A.m = m; A.ph = ph; A.T = T; A.Tv = Tv; A.Fc_out = Fc;
    return Launch<N, false, double, EPB64>::face(A, faces, nf, nw, st);
  }
  static cudaError_t face32(const MeshArg<float>& m, const PhysArg<float>& ph, const BgArg& bg, const int2* faces,
                            int nf, int nw, const float* T, const float* Tv, float* Fc, cudaStream_t st) {
    KArgs<float> A{};
    A.m = m; A.ph = ph; A.bg = bg; A.T = T; A.Tv = Tv; A.Fc_out = Fc;
    return Launch<N, true, float, EPB32>::face(A, faces, nf, nw, st);
  }
  template <bool PERT, class R, int EPB>
  static cudaError_t update(const MeshArg<R>& m, const OpsArg<R>& ops, const R* q, const R* part, const R* Fc, R* out,
                            R* T_out, const RkCoef<R>& rk, const R* r0, R dt, int mode, const int* skip,
                            cudaStream_t st) {
    using L = Launch<N, PERT, R, EPB>;
    KArgs<R> A{};
    A.m = m; A.ops = ops; A.q = q; A.part = part; A.Fc = Fc; A.out = out; A.T_out = T_out;
    A.un = rk.un; A.a = rk.a; A.b = rk.b; A.c = rk.c;
    A.un2 = rk.un2; A.out2 = rk.out2; A.a2 = rk.a2; A.b2 = rk.b2; A.c2 = rk.c2;
    A.radd = rk.radd; A.r0 = r0; A.dt = dt; A.skip = skip;
    return mode == kModeRK ? L::template update<kModeRK>(A, st) : L::template update<kModeResidual>(A, st);
  }
  static LaunchSet set() {
    return LaunchSet{trace<false, double, EPB64>, vol64, face64, update<false, double, EPB64>,
                     trace<true, float, EPBU>,    vol32, face32, update<true, float, EPBU>,
                     EPB32};
  }
};

}  // namespace chorus
