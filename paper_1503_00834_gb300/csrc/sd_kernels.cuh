// Spectral-difference residual kernels for one order N = p + 1 (paper Sections 3 and 5).
//
// A residual (and an RK stage) is three kernels:
//   k_vol     everything an element can do alone once its neighbours' traces are known: the lifted
//             gradients, the one-sided viscous flux of every face point (written for both sides), the
//             fluxes at the interior flux points, their part of the divergence and the sources.
//             Writes the residual without the two end-point fluxes of each line (at p = 2 without R(Q0)
//             either: late_background).
//   k_face    the common flux of every face point, once per face, from both sides' traces.
//   k_update  adds the end-point fluxes' part of the divergence, forms the RK combination and writes the
//             new state's traces.
// The gradient record never leaves the SM, and the metrics and the background are read once a stage.
// The state is read again by k_update, so that the new state is rounded once, from the whole residual:
// with the combination in k_vol and the end-point fluxes added to its rounded result (one read of the state
// less; p = 3, 331,776 elements: 1.82 against 1.87 ms a stage) a step was 7 to 17 % further from the 64-bit
// one, at every order.
//
// k_vol: one CTA processes EPB elements; each element is handled by N*N threads, thread `ln` owning
// the line (a, b) = (ln % N, ln / N) of every direction (xi-line (j,k), eta-line (i,k), zeta-line
// (i,j)).  A thread does the 1D work of its line in registers: interpolation to the N+1 flux points
// (Eq. 17), fluxes, and the derivative back to the N solution points (Eq. 18).  Shared memory links
// the directional sweeps.
//
// Shared memory per element: the staged state and background tables (bulk TMA copies), and one block
// of 16 components per solution point that holds in turn the raw derivatives of the lifting (two
// directions x 8), then the 11-entry gradient record and the 5 divergence sums.  The directions are
// lifted in the order zeta, eta, xi and their fluxes swept in the order eta, xi, zeta, so that two
// buffers of one direction's metrics each, refilled by bulk copies while the other is in use, always
// hold the next sweep's (stage_metrics).  At N = 4 in FP32
// element blocks are padded so that the two elements of a warp use opposite halves of the banks, and
// the computed arrays are XOR-swizzled so that xi-, eta- and zeta-line accesses are conflict free.
#pragma once
#include <utility>
#include <utility>

#include "sd_device.cuh"
#include "sd_physics.cuh"

namespace chorus {

// ------------------------------------------------------------------ tuning

// Resident warps per SM asked of the compiler for k_vol (the register cap: 128 registers a thread at 16
// warps, 168 at 12, 200 at 10), timed per order on the shells of the workloads.
template <int N>
__host__ __device__ constexpr int vol_warps() {
  return N == 3 ? 16 : N == 5 ? 12 : 10;
}
template <int N, int EPB>
__host__ __device__ constexpr int vol_min_blocks() {
  return vol_warps<N>() / warps_per_cta<N, EPB>() > 0 ? vol_warps<N>() / warps_per_cta<N, EPB>() : 1;
}

// How k_vol's flux sweep holds a line.  FB = 1: one flux point at a time, the line's components in
// registers (reg_lines) or read from shared memory for each flux point; FB >= 2: the flux points in
// two blocks of at most FB from either end of the line, the line read once for each block.  In
// registers the line takes 21 N words: it fits at N = 4 (as blocks of three or four points it ran 9 % and
// 18 % slower there); two blocks hold 21 FB values instead.
template <int N, class R>
__host__ __device__ constexpr int flux_block() {
  return sizeof(R) == 8 || N == 4 ? 1 : N / 2 + 1;
}
// Whether the two blocks take the interpolation weights from the constant bank instead of shared memory:
// the weights of the flux points counted from the line's far end are those from the near end with the
// line reversed, so one set serves both.  At N = 6 four points' weights as pairs (48 registers) do not
// fit beside their 84 values; the scalar products with constants are 11 % faster there, 1-3 % slower at
// N = 3 and 5.
template <int N>
__host__ __device__ constexpr bool const_weights() { return N == 6; }
template <int N, class R>
__host__ __device__ constexpr bool reg_lines() { return sizeof(R) == 4 && flux_block<N, R>() == 1; }

// The threads that share staging barriers and element arrays.  At N = 4 a warp holds two whole
// elements: it stages them itself and a warp barrier orders its sweeps, so the warps of a CTA never
// wait for one another.  At the other orders elements straddle warps and the unit is the CTA.
template <int N>
__host__ __device__ constexpr bool warp_local() { return 32 % (N * N) == 0; }
template <int N>
__device__ __forceinline__ void unit_sync() {
  if constexpr (warp_local<N>()) __syncwarp();
  else __syncthreads();
}
template <int N, int EPB>
__host__ __device__ constexpr int unit_elems() { return warp_local<N>() ? 32 / (N * N) : EPB; }
template <int N, int EPB>
__host__ __device__ constexpr int unit_threads() { return warp_local<N>() ? 32 : EPB * N * N; }

// Whether the metrics are staged in shared memory (FP32, N = 3 and 4, where two directions' buffers
// fit beside twelve warps' elements); else each sweep loads its flux points' metrics from global
// memory.
template <int N, class R>
__host__ __device__ constexpr bool stage_metrics() { return sizeof(R) == 4 && N <= 4; }

// Whether the epilogue's inputs (R(Q0), x) are staged too, by bulk copies into the record's and a
// metric buffer's space once the last sweep has its lines in registers, so that they arrive during
// that sweep: left to register loads after it, they were the longest stall of the kernel (0.41 of
// 1.79 ms at p = 3, 331,776 elements).
template <int N, class R>
__host__ __device__ constexpr bool stage_epilogue() { return warp_local<N>() && reg_lines<N, R>() && stage_metrics<N, R>(); }

// Whether k_update adds R(Q0) (FP32), to the whole perturbation residual, rather than k_vol to the part
// without the end points.  A coarse p = 2 shell's residual is mostly R(Q0), and the part would be rounded at
// that size once more (288 and 450 elements: 6 to 7 % further from the 64-bit residual than the three-pass
// kernels'; late, as far as theirs; 98,304 elements take 334 us a stage either way).  From p = 3 on the early
// sum is the closer one, by 2 to 3 %.
template <int N, class R>
__host__ __device__ constexpr bool late_background() { return sizeof(R) == 4 && N == 3; }

template <int N, bool PERT, class R, int EPB>
struct Layout {
  static constexpr int N2 = N * N, N3 = N * N * N;
  static constexpr int V = 16 / (int)sizeof(R);  // words of a 16-byte bulk-copy unit
  // N = 4 FP32: padded element blocks, one bulk copy each; else the CTA's elements as in global memory,
  // one bulk copy for all of them, from the 16-byte boundary at or before the first
  static constexpr bool padded = N == 4 && sizeof(R) == 4;
  static constexpr int stride(int n) { return padded ? pad_stride<R>(n) : n; }
  static constexpr int block(int n) { return padded ? EPB * stride(n) : (EPB * n + 2 * V + V - 1) / V * V; }
  static constexpr bool SM = stage_metrics<N, R>();
  static constexpr int SQ = stride(5 * N3), SBG = stride(2 * N3), SGR0 = stride(3 * N3);
  // N = 3 FP32: 443 words, 27 mod 32, so that the xi lines of a warp's elements start in 32 different
  // banks (0.206 -> 0.193 ms at 98,304 elements); no stride measured better at N = 5 and 6
  static constexpr int SG = padded ? pad_stride<R>(16 * N3) : 16 * N3 + (N == 3 && sizeof(R) == 4 ? 11 : 0);
  // interpolation I[f][s], then derivative D[i][f] as [f][i], as pairs of equal values, indexed by rolled
  // loops (stage_tables)
  static constexpr int TAB = 4 * (N + 1) * N;
  static constexpr int units = (EPB + unit_elems<N, EPB>() - 1) / unit_elems<N, EPB>();
  static constexpr int oI = 0;
  static constexpr int oQ = (oI + TAB + 31) / 32 * 32;
  static constexpr int oBG = oQ + block(5 * N3);
  static constexpr int oGR0 = oBG + (PERT ? block(2 * N3) : 0);
  static constexpr int oG = oGR0 + (PERT ? block(3 * N3) : 0);
  // staged 1/|J| and metrics (one direction's [3][N+1][N2] an element in each of two buffers)
  static constexpr int SIJ = stride(N3), SS = 3 * (N + 1) * N2;
  static constexpr int oIJ = (oG + EPB * SG + V - 1) / V * V;
  static constexpr int oS0 = oIJ + (SM ? block(N3) : 0);
  static constexpr int oS1 = oS0 + (SM ? EPB * SS : 0);
  static constexpr int total = oS1 + (SM ? EPB * SS : 0);
  static_assert(!SM || (SS * (int)sizeof(R)) % 16 == 0, "a metric block is a multiple of the bulk-copy unit");
  static_assert(kG + 5 == 16, "the record and the divergence share the lifting's sixteen components");
};

// ------------------------------------------------------------------ kernel arguments

template <class R>
struct KArgs {
  MeshArg<R> m;
  OpsArg<R> ops;
  PhysArg<R> ph;
  BgArg bg;            // perturbation form only
  const R* q;          // state (form variables); k_update: in RK mode
  const R* T;          // face traces of q, [E][6][5][N2] (trace_slot)
  const R* Tv;         // one-sided viscous fluxes along the outward S [E][6][4][N2] (k_face input)
  R* Tv_out;           // k_vol output
  R* part_out;         // k_vol output: the residual without the end-point fluxes [E][5][N3]
  const R* part;       // k_update input
  R* out;              // k_update: residual or new state
  R* T_out;            // k_update: traces of the new state (RK mode)
  const R* un;         // first extra state of the RK combination
  R a, b, c, dt;       // out = a un + b q + c dt R
  const R* un2;        // optional second output: out2 = a2 un2 + b2 q + c2 dt R
  R* out2;
  R a2, b2, c2;
  const R* r0;         // k_update: R(Q0) [E][5][N3] where it adds it (late_background), or null
  const R* radd;       // k_update: optional additive residual correction [E][5][N3]
  R* Fc_out;           // k_face output: common fluxes along the owner's outward S [faces][5][N2]
  const R* Fc;         // k_update input
  int* skip_out;       // k_vol: per element, 1 if its staging gave up (nothing stored for it), else 0
  const int* skip;     // k_update: the same; elements with 1 are left as they are
  unsigned* err;       // k_vol: error flags and wait limit
};

// Face traces are kept where they are read: slot (e, F) of a trace array holds, at element e's own
// points of its face F, the neighbour's trace (on a wall the element's own).  The kernels that make a
// state's traces write each into the neighbour's slot, with the neighbour's point numbering, so that
// the volume kernel reads its neighbours' traces as one contiguous block with no table look-up before
// it (gathered there, they cost it 0.14 of 1.45 ms at p = 3, 331,776 elements).

// Where own face point ln of the face with table entries (k, c) goes, of element e (its index in the
// whole mesh) and face F: the word of variable 0 in [E][6][5][N2].
template <int N>
__device__ __forceinline__ size_t trace_slot(int64_t e, int F, int k, int c, int ln) {
  constexpr int N2 = N * N;
  return k >= 0 ? ((size_t)k * 6 + (c >> 3)) * 5 * N2 + map_face_pt<N>(ln, c & 7) : ((size_t)e * 6 + F) * 5 * N2 + ln;
}

// An element's neighbour or face-code table entries (six each).
__device__ __forceinline__ void load_six(const int* __restrict__ t, int64_t e, int out[6]) {
#pragma unroll
  for (int F = 0; F < 6; F += 2) {
    const int2 v = __ldg(reinterpret_cast<const int2*>(t + e * 6 + F));
    out[F] = v.x;
    out[F + 1] = v.y;
  }
}

// the traces on the other side of one face point
template <class R>
struct NbFace {
  int kind;  // >= 0 interior, -1 inner wall, -2 outer wall
  R q[5];
};

// Global-memory inputs of one lifting sweep, loaded ahead of their use so that their latency
// overlaps the preceding work: the neighbours' traces, and where the metrics are not staged (SM false)
// the line's metrics and 1/|J| too.
template <int N, class R, bool SM>
struct LiftPre {
  R S[SM ? 1 : 3][N + 1];  // S^D_n at the N+1 flux points of the line
  R ij[SM ? 1 : N];        // 1/|J| at the line's solution points
  NbFace<R> nb[2];
};

// nbr: the element's neighbour table entries.
template <int N, class R, int D, bool SM>
__device__ __forceinline__ void lift_prefetch(const KArgs<R>& A, int e, int ln, LiftPre<N, R, SM>& p, const int* nbr) {
  constexpr int N2 = N * N, N3 = N * N * N;
  if constexpr (!SM) {
    const R* Sl = A.m.Sf + ((size_t)e * 3 + D) * 3 * (N + 1) * N2;
#pragma unroll
    for (int n = 0; n < 3; ++n)
#pragma unroll
      for (int f = 0; f <= N; ++f) p.S[n][f] = __ldg(Sl + (n * (N + 1) + f) * N2 + ln);
#pragma unroll
    for (int i = 0; i < N; ++i) p.ij[i] = __ldg(A.m.invJ + (size_t)e * N3 + line_pt<N, D>(ln, i));
  }
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    const R* Te = A.T + ((size_t)e * 6 + 2 * D + side) * 5 * N2 + ln;
    p.nb[side].kind = nbr[2 * D + side];
#pragma unroll
    for (int v = 0; v < 5; ++v) p.nb[side].q[v] = ld_written(Te + v * N2);
  }
}

// Radiative diffusivity at flux point f of line ln (direction D): from the mesh's flux-point table
// (the interpolant of its solution-point values) when a profile is active, else the constant.  KR
// false compiles the lookup out (the FP32 kernels are built both ways).
template <int N, int D, bool KR, class R>
__device__ __forceinline__ R kr_at(const KArgs<R>& A, int e, int ln, int f) {
  if constexpr (!KR) return A.ph.kappa_r;
  if (A.m.kr == nullptr) return A.ph.kappa_r;
  return __ldg(A.m.kr + (((size_t)e * 3 + D) * (N + 1) + f) * (N * N) + ln);
}

// ------------------------------------------------------------------ trace kernel

// Traces of tile `tile` (elements tile * EPB ...), one thread per (element, line); threads beyond
// EPB * N^2 idle.
template <int N, class R, int EPB>
__device__ __forceinline__ void trace_tile(const MeshArg<R>& m, const OpsArg<R>& ops, const R* __restrict__ q,
                                           R* __restrict__ T, int64_t tile) {
  constexpr int N2 = N * N, N3 = N * N * N;
  const int el = threadIdx.x / N2, ln = threadIdx.x % N2;
  const int64_t e = tile * EPB + el;
  if (el >= EPB || e >= m.E) return;
  const R* qe = q + (size_t)e * 5 * N3;
  int nbr[6], code[6];
  load_six(m.nbr, e, nbr);
  load_six(m.code, e, code);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    R* T0 = T + trace_slot<N>(m.e0 + e, 2 * d, nbr[2 * d], code[2 * d], ln);
    R* T1 = T + trace_slot<N>(m.e0 + e, 2 * d + 1, nbr[2 * d + 1], code[2 * d + 1], ln);
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      R lo = R(0), hi = R(0);
#pragma unroll
      for (int s = 0; s < N; ++s) {
        const int pt = d == 0 ? line_pt<N, 0>(ln, s) : (d == 1 ? line_pt<N, 1>(ln, s) : line_pt<N, 2>(ln, s));
        const R val = qe[v * N3 + pt];
        lo += ops.I[0][s] * val;
        hi += ops.I[N][s] * val;
      }
      T0[v * N2] = lo;
      T1[v * N2] = hi;
    }
  }
}

template <int N, class R, int EPB>
__global__ void __launch_bounds__(EPB * N * N) k_trace(const MeshArg<R> m, const OpsArg<R> ops, const R* __restrict__ q,
                                                      R* __restrict__ T) {
  trace_tile<N, R, EPB>(m, ops, q, T, blockIdx.x);
}

// ------------------------------------------------------------------ staging

// One array of PER words an element, staged for a unit's elements e0 .. e0 + ne - 1 of `total`
// elements.  Unpadded blocks are copied as they lie in global memory, from the 16-byte unit that
// holds the first word (the elements start `shift` words into the block) to the end of the last
// unit; the array's own last, partial unit is left to plain loads (`tail` words from word t0).
template <class L, class R, int PER, bool PADDED>
struct Span {
  int64_t a0;       // first word copied
  int n, shift;     // words copied, first element's word in the block
  int64_t t0;
  int tail;
  bool bulk;
  __device__ __forceinline__ Span(const R* src, int e0, int ne, int64_t total) {
    constexpr int V = L::V;
    const int64_t w0 = (int64_t)e0 * PER, w1 = w0 + (int64_t)ne * PER;
    bulk = ((uintptr_t)src & 15u) == 0 && (!PADDED || PER % V == 0);
    shift = PADDED || PER % V == 0 || !bulk ? 0 : (int)(w0 % V);
    a0 = w0 - shift;
    const int64_t lim = total * PER / V * V;
    const int64_t up = (w1 + V - 1) / V * V;
    const int64_t a1 = PER % V == 0 || up <= lim ? up : lim;
    n = (int)(a1 - a0);
    t0 = a1;
    tail = a1 < w1 ? (int)(w1 - a1) : 0;
  }
  // issued by one thread; returns the bytes that will arrive
  __device__ __forceinline__ uint32_t bytes(int ne) const {
    return !bulk ? 0u : (uint32_t)((PADDED ? ne * PER : n) * sizeof(R));
  }
  __device__ __forceinline__ void issue(R* dst, const R* src, int e0, int ne, int stride, uint64_t* bar) const {
    if (!bulk) return;
    if constexpr (PADDED) {
      for (int el = 0; el < ne; ++el)
        bulk_g2s(dst + el * stride, src + (size_t)(e0 + el) * PER, PER * sizeof(R), bar);
    } else if (n > 0) {
      bulk_g2s(dst, src + a0, (uint32_t)(n * sizeof(R)), bar);
    }
  }
  // the part that does not go by bulk copy, all nt threads of the unit
  __device__ __forceinline__ void rest(R* dst, const R* src, int e0, int ne, int stride, int tid, int nt) const {
    if (!bulk) {
      for (int i = tid; i < ne * PER; i += nt) dst[(i / PER) * stride + i % PER] = src[(size_t)e0 * PER + i];
    } else if (!PADDED && tid < tail) {
      dst[t0 - a0 + tid] = src[t0 + tid];
    }
  }
};

// Where a unit's elements start in their staged blocks.
struct Shift {
  int q, bg, gr0, ij;
};

// Direction d's metric blocks of a unit's elements into buffer `dst` (one thread).
template <int N, class R, class L>
__device__ __forceinline__ void issue_metrics(const R* Sf, int e0, int ne, int d, R* dst, uint64_t* bar) {
  for (int j = 0; j < ne; ++j)
    bulk_g2s(dst + j * L::SS, Sf + ((size_t)(e0 + j) * 3 + d) * L::SS, L::SS * sizeof(R), bar);
}

// Stages a unit's elements e0 .. e0 + ne - 1, at element u0 of the CTA's blocks: state, background, and
// where staged 1/|J| and the metrics of the first two sweeps (zeta, eta).  tid of nt: the thread in its
// unit.  `between` runs after the copies are issued and before the wait (it issues the first sweep's
// global loads so that both latencies overlap).  The copies complete the phase of `bar` whose parity
// is `parity` (flipped here whenever the barrier was used).  Returns false, the same in every thread of
// the unit, when the bounded wait for the copies ran out (the flag is set in *A.err and the copies in
// flight have been waited for): the caller then skips its computation and every global store.
template <int N, bool PERT, class R, int EPB, class Between>
__device__ __forceinline__ bool stage_elements(const KArgs<R>& A, R* sm, uint64_t* bar, uint32_t& parity, int e0, int ne,
                                               int u0, int tid, int nt, Shift& sh, uint32_t polls, Between&& between) {
  using L = Layout<N, PERT, R, EPB>;
  constexpr int N3 = N * N * N;
  const Span<L, R, 5 * N3, L::padded> sq(A.q, e0, ne, A.m.E);
  R* dq = sm + L::oQ + u0 * L::SQ;
  sh = Shift{sq.shift, 0, 0, 0};
  uint32_t bytes = sq.bytes(ne);
  if constexpr (PERT) {
    const Span<L, R, 2 * N3, L::padded> sb(A.bg.bg, e0, ne, A.m.E);
    const Span<L, R, 3 * N3, L::padded> sg(A.bg.grho0, e0, ne, A.m.E);
    const Span<L, R, N3, L::padded> si(A.m.invJ, e0, ne, A.m.E);
    R *db = sm + L::oBG + u0 * L::SBG, *dg = sm + L::oGR0 + u0 * L::SGR0, *di = sm + L::oIJ + u0 * L::SIJ;
    sh.bg = sb.shift;
    sh.gr0 = sg.shift;
    sh.ij = si.shift;
    bytes += sb.bytes(ne) + sg.bytes(ne);
    if (L::SM) bytes += si.bytes(ne) + 2 * ne * L::SS * sizeof(R);
    if (tid == 0 && bytes > 0) {
      mbar_expect_tx(bar, bytes);
      if constexpr (L::SM) {
        issue_metrics<N, R, L>(A.m.Sf, e0, ne, 2, sm + L::oS0 + u0 * L::SS, bar);
        si.issue(di, A.m.invJ, e0, ne, L::SIJ, bar);
        issue_metrics<N, R, L>(A.m.Sf, e0, ne, 1, sm + L::oS1 + u0 * L::SS, bar);
      }
      sb.issue(db, A.bg.bg, e0, ne, L::SBG, bar);
      sg.issue(dg, A.bg.grho0, e0, ne, L::SGR0, bar);
    }
    sb.rest(db, A.bg.bg, e0, ne, L::SBG, tid, nt);
    sg.rest(dg, A.bg.grho0, e0, ne, L::SGR0, tid, nt);
    if (L::SM) si.rest(di, A.m.invJ, e0, ne, L::SIJ, tid, nt);
  } else if (tid == 0 && bytes > 0) {
    mbar_expect_tx(bar, bytes);
  }
  pdl_wait();  // the mesh's own data above; the state and its traces come from the kernels before
  if (tid == 0) sq.issue(dq, A.q, e0, ne, L::SQ, bar);
  sq.rest(dq, A.q, e0, ne, L::SQ, tid, nt);
  between();
  bool ok = true;
  if (bytes > 0) {
    ok = mbar_wait(bar, parity, A.err, polls);
    parity ^= 1u;
  }
  if constexpr (warp_local<N>()) {
    ok = __all_sync(0xffffffffu, ok) != 0;
    __syncwarp();  // the warp's own plain stores
    return ok;
  } else return __syncthreads_and(ok) != 0;
}

// ------------------------------------------------------------------ element views

// The staged and computed arrays of one element.
template <class R>
struct Elem {
  const R* q;    // [5][N3], linear order
  const R* bg;   // [2][N3], background order
  const R* gr0;  // [3][N3], background order
  R* g;          // [16][N3], computed arrays' order: the record, then the divergence at 11..15
  const R* ij;   // [N3], linear order (where staged)
  const R* S0;   // the two metric buffers [3][N+1][N2] (where staged)
  const R* S1;
};

// The N values of one component along line ln of direction D: state (linear order), background or
// computed arrays.  xi lines are contiguous: one 16-byte load at N = 4, 8-byte loads at N = 6 (FP32).
enum Order { kLinear, kBackground, kComputed };
template <int N, int D, Order O, class R>
__device__ __forceinline__ void load_line(const R* base, int ln, R out[N]) {
  if constexpr (D == 0 && N == 4 && sizeof(R) == 4) {
    const float4 v = *reinterpret_cast<const float4*>(base + (O == kLinear ? 4 * ln : line_sidx<N, 0, R>(ln, 0)));
    out[0] = v.x;
    out[1] = v.y;
    out[2] = v.z;
    out[3] = v.w;
  } else if constexpr (D == 0 && N == 6 && sizeof(R) == 4) {
#pragma unroll
    for (int s = 0; s < N; s += 2) {
      const float2 v = *reinterpret_cast<const float2*>(base + 6 * ln + s);
      out[s] = v.x;
      out[s + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int s = 0; s < N; ++s)
      out[s] = base[O == kLinear ? line_pt<N, D>(ln, s) : O == kBackground ? line_bg<N, D, R>(ln, s)
                                                                         : line_sidx<N, D, R>(ln, s)];
  }
}

// Component c of the values a flux point needs: 0..4 the state, 5..15 the gradient record, 16, 17 the
// background rho, E, 18..20 the background density gradient (perturbation form).
template <int N, int D, class R>
__device__ __forceinline__ void load_comp(const Elem<R>& x, int c, int ln, R out[N]) {
  constexpr int N3 = N * N * N;
  if (c < 5) load_line<N, D, kLinear>(x.q + c * N3, ln, out);
  else if (c < 16) load_line<N, D, kComputed>(x.g + (c - 5) * N3, ln, out);
  else if (c < 18) load_line<N, D, kBackground>(x.bg + (c - 16) * N3, ln, out);
  else load_line<N, D, kBackground>(x.gr0 + (c - 18) * N3, ln, out);
}

// ------------------------------------------------------------------ lifting, one direction

// d q / d xi_D along the thread's D-line with common face values (BR1-like averaging, Section 3;
// walls Section 5) and grad xi_D = S^D / |J| at its points.  Directions 2 and 1 store both (eight raw
// values a point); direction 0 forms the conserved gradients from all three and leaves the gradient
// record in place (its line's points are touched by no other thread in this phase).
template <int N, bool PERT, class R, int D, bool SM>
__device__ __forceinline__ void lift_dir(const KArgs<R>& A, const Elem<R>& x, int ln, int e,
                                         const LiftPre<N, R, SM>& pre) {
  constexpr int N2 = N * N, N3 = N * N * N;
  constexpr bool LAST = D == 0;
  constexpr bool V4 = D == 0 && N == 4 && sizeof(R) == 4;  // 16-byte shared-memory accesses along the line
  const PhysArg<R>& ph = A.ph;
  R qv[5][N];
#pragma unroll
  for (int v = 0; v < 5; ++v) load_line<N, D, kLinear>(x.q + v * N3, ln, qv[v]);
  R S[3][N + 1], ij[N];
  if constexpr (SM) {
    const R* sS = (D == 1 ? x.S1 : x.S0) + ln;
#pragma unroll
    for (int n = 0; n < 3; ++n)
#pragma unroll
      for (int f = 0; f <= N; ++f) S[n][f] = sS[(n * (N + 1) + f) * N2];
    load_line<N, D, kLinear>(x.ij, ln, ij);
  } else {
#pragma unroll
    for (int n = 0; n < 3; ++n)
#pragma unroll
      for (int f = 0; f <= N; ++f) S[n][f] = pre.S[n][f];
#pragma unroll
    for (int i = 0; i < N; ++i) ij[i] = pre.ij[i];
  }

  R gx[3][N];
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      R acc = R(0);
#pragma unroll
      for (int f = 0; f <= N; ++f) acc += A.ops.Lfs[i][f] * S[n][f];
      gx[n][i] = acc * ij[i];
    }
  // what needs no neighbour data first: its loads are still in flight at the first sweep
  R dv[5][N];
#pragma unroll
  for (int v = 0; v < 5; ++v)
#pragma unroll
    for (int i = 0; i < N; ++i) {
      R acc = A.ops.Dsol[i][0] * qv[v][0];
#pragma unroll
      for (int s = 1; s < N; ++s) acc += A.ops.Dsol[i][s] * qv[v][s];
      dv[v][i] = acc;
    }
  R dq[5][2];  // common state minus own trace at the two ends
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    const int f = side ? N : 0;
    const NbFace<R>& nb = pre.nb[side];
    R qe[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      R acc = R(0);
#pragma unroll
      for (int s = 0; s < N; ++s) acc += A.ops.I[f][s] * qv[v][s];
      qe[v] = acc;
    }
    if (nb.kind >= 0) {
#pragma unroll
      for (int v = 0; v < 5; ++v) dq[v][side] = R(0.5) * (nb.q[v] - qe[v]);
    } else {
      R rho0e = R(0), E0e = R(0);
      if constexpr (PERT) {
        R l[N];
        load_line<N, D, kBackground>(x.bg, ln, l);
#pragma unroll
        for (int s = 0; s < N; ++s) rho0e += A.ops.I[f][s] * l[s];
        load_line<N, D, kBackground>(x.bg + N3, ln, l);
#pragma unroll
        for (int s = 0; s < N; ++s) E0e += A.ops.I[f][s] * l[s];
      }
      // wall common state: zero normal velocity, interior density, interior pressure (inner wall)
      // or p = R rho T_top (outer wall)
      const R Sn[3] = {S[0][f], S[1][f], S[2][f]};
      const R i2 = qrcp(dot3(Sn, Sn));
      const Pt<R> st = point_state<PERT>(qe, rho0e, E0e, ph);
      const R mn = dot3(qe + 1, Sn) * i2;
      const R mc[3] = {qe[1] - mn * Sn[0], qe[2] - mn * Sn[1], qe[3] - mn * Sn[2]};
      const R pc = nb.kind == -2 ? ph.Rgas * qe[0] * ph.T_top : st.p;
      const R Ec = pc * qrcp(ph.gm1) + R(0.5) * dot3(mc, mc) * st.ir;
      dq[0][side] = R(0);
      dq[1][side] = mc[0] - qe[1];
      dq[2][side] = mc[1] - qe[2];
      dq[3][side] = mc[2] - qe[3];
      dq[4][side] = Ec - qe[4];
    }
  }
#pragma unroll
  for (int v = 0; v < 5; ++v)
#pragma unroll
    for (int i = 0; i < N; ++i) dv[v][i] += A.ops.D[i][0] * dq[v][0] + A.ops.D[i][N] * dq[v][1];
  if constexpr (!LAST) {
    constexpr int o = D == 2 ? 0 : 8;  // slot: the five derivatives, then grad xi_D
#pragma unroll
    for (int c = 0; c < 8; ++c)
#pragma unroll
      for (int i = 0; i < N; ++i)
        x.g[(o + c) * N3 + line_sidx<N, D, R>(ln, i)] = c < 5 ? dv[c < 5 ? c : 0][i] : gx[c < 5 ? 0 : c - 5][i];
  } else {
    // conserved gradients, then the record, the line's points in groups of one shared-memory access
    R l0[PERT ? 5 : 1][N];  // rho0, E0, grad rho0 along the line
    if constexpr (PERT) {
#pragma unroll
      for (int c = 0; c < 2; ++c) load_line<N, D, kBackground>(x.bg + c * N3, ln, l0[c]);
#pragma unroll
      for (int c = 0; c < 3; ++c) load_line<N, D, kBackground>(x.gr0 + c * N3, ln, l0[2 + c]);
    }
    R gq[V4 ? N : 1][15], rec[V4 ? kG : 1][V4 ? N : 1];
    if constexpr (V4) {
#pragma unroll
      for (int v = 0; v < 5; ++v)
#pragma unroll
        for (int n = 0; n < 3; ++n)
#pragma unroll
          for (int i = 0; i < N; ++i) gq[i][3 * v + n] = dv[v][i] * gx[n][i];
#pragma unroll
      for (int o = 0; o < 16; o += 8) {
        R gr[3][N];
#pragma unroll
        for (int n = 0; n < 3; ++n) load_line<N, D, kComputed>(x.g + (o + 5 + n) * N3, ln, gr[n]);
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          R dr[N];
          load_line<N, D, kComputed>(x.g + (o + v) * N3, ln, dr);
#pragma unroll
          for (int n = 0; n < 3; ++n)
#pragma unroll
            for (int i = 0; i < N; ++i) gq[i][3 * v + n] += dr[i] * gr[n][i];
        }
      }
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int si = line_sidx<N, D, R>(ln, i);
      R(&gp)[15] = gq[V4 ? i : 0];
      if constexpr (!V4) {
        R raw[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) raw[c] = x.g[c * N3 + si];
#pragma unroll
        for (int v = 0; v < 5; ++v)
#pragma unroll
          for (int n = 0; n < 3; ++n)
            gp[3 * v + n] = dv[v][i] * gx[n][i] + raw[v] * raw[5 + n] + raw[8 + v] * raw[13 + n];
      }
      R q[5], gr0[3] = {R(0), R(0), R(0)}, g[kG], r0 = R(0), E0 = R(0);
#pragma unroll
      for (int v = 0; v < 5; ++v) q[v] = qv[v][i];
      if constexpr (PERT) {
        r0 = l0[0][i];
        E0 = l0[1][i];
#pragma unroll
        for (int n = 0; n < 3; ++n) gr0[n] = l0[2 + n][i];
      }
      const Pt<R> st = point_state<PERT>(q, r0, E0, ph);
      grad_prim<PERT>(st, gp, gr0, ph, g);
#pragma unroll
      for (int c = 0; c < kG; ++c) {
        if constexpr (V4) rec[c][i] = g[c];
        else x.g[c * N3 + si] = g[c];
      }
    }
    if constexpr (V4) {
#pragma unroll
      for (int c = 0; c < kG; ++c)
        *reinterpret_cast<float4*>(x.g + c * N3 + line_sidx<N, 0, R>(ln, 0)) =
            make_float4(rec[c][0], rec[c][1], rec[c][2], rec[c][3]);
    }
  }
}

// ------------------------------------------------------------------ flux sweep, one direction

// Conductive energy flux f.S through the outer wall with the temperature imposed there (Section 5):
// T = T_top in f = -kappa rho T grad S - kappa_r rho C_p grad T written in rho and p.
template <class R>
__device__ __forceinline__ R wall_conduction(const R g[kG], const R S[3], R kr, const PhysArg<R>& ph) {
  return -ph.CpR * ((ph.kappa_g + kr) * dot3(g + 8, S) - (ph.kappa + kr) * ph.Rgas * ph.T_top * dot3(g, S));
}

// Transformed fluxes at the interior flux points of the thread's D-line (Eq. 12) and their part of the
// derivative back to the solution points (Eq. 18), left in acc; at the two end points the one-sided
// viscous flux along the outward S, written for k_face: Tv[e][F][0..2] = tau S, Tv[e][F][3] = u.tau S -
// f.S (on a wall side f.S with the top temperature imposed instead).
// kind: the neighbours (or wall codes) of the line's two faces.  sS: the direction's staged metrics.
// loaded: called once the line is in registers (reg_lines).
template <int N, bool PERT, class R, int D, bool KR, class Loaded>
__device__ __forceinline__ void flux_dir(const KArgs<R>& A, const Elem<R>& x, const R* tab, int ln, int e,
                                         const int kind[2], const R* sS, R (&acc)[5][N], Loaded&& loaded) {
  constexpr int N2 = N * N;
  constexpr int NC = PERT ? 21 : 16, NP = (NC + 1) / 2;
  constexpr int FB = flux_block<N, R>();
  constexpr bool REG = reg_lines<N, R>();
  const PhysArg<R>& ph = A.ph;
  constexpr bool SM = stage_metrics<N, R>();
  const R* Sl = SM ? sS + ln : A.m.Sf + ((size_t)e * 3 + D) * 3 * (N + 1) * N2 + ln;
  auto metric = [&](int n, int f) { return SM ? Sl[(n * (N + 1) + f) * N2] : __ldg(Sl + (n * (N + 1) + f) * N2); };
  const Pair<R>* tI = reinterpret_cast<const Pair<R>*>(tab);
  const Pair<R>* tD = tI + (N + 1) * N;
  Pair<R> a01[N], a23[N];
  R a4[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    a01[i] = a23[i] = Pair<R>{R(0), R(0)};
    a4[i] = R(0);
  }
  // the line's components as pairs (2k, 2k+1)
  auto load_pair = [&](int k, R (&u)[N], R (&w)[N]) {
    load_comp<N, D>(x, 2 * k, ln, u);
    if (2 * k + 1 < NC) load_comp<N, D>(x, 2 * k + 1, ln, w);
    else {
#pragma unroll
      for (int s = 0; s < N; ++s) w[s] = R(0);
    }
  };
  // the point values from the pairs
  struct Vals {
    R q[5], g[kG], r0, E0, gr0[3];
  };
  auto unpack = [&](const Pair<R> (&P)[NP]) {
    Vals v;
    auto c = [&](int i) { return i & 1 ? P[i / 2].y : P[i / 2].x; };
#pragma unroll
    for (int i = 0; i < 5; ++i) v.q[i] = c(i);
#pragma unroll
    for (int i = 0; i < kG; ++i) v.g[i] = c(5 + i);
    v.r0 = v.E0 = v.gr0[0] = v.gr0[1] = v.gr0[2] = R(0);
    if constexpr (PERT) {
      v.r0 = c(16);
      v.E0 = c(17);
#pragma unroll
      for (int i = 0; i < 3; ++i) v.gr0[i] = c(18 + i);
    }
    return v;
  };
  auto interior = [&](const Vals& v, const R s[3], int f) {
    const Pt<R> st = point_state<PERT>(v.q, v.r0, v.E0, ph);
    R Fi[5], Fv[4];
    flux_inv(v.q, st, s, Fi);
    flux_visc<PERT>(st, v.q, v.g, v.gr0, v.r0, v.E0, s, ph, kr_at<N, D, KR>(A, e, ln, f), Fv);
    const Pair<R> F01{Fi[0], Fi[1] - Fv[0]}, F23{Fi[2] - Fv[1], Fi[3] - Fv[2]};
    const R F4 = Fi[4] - Fv[3];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const Pair<R> d = tD[f * N + i];
      a01[i] = fma2(d, F01, a01[i]);
      a23[i] = fma2(d, F23, a23[i]);
      a4[i] += d.x * F4;
    }
  };
  auto end = [&](const Vals& v, const R s[3], int side) {
    const R sg = side ? R(1) : R(-1);
    const R So[3] = {sg * s[0], sg * s[1], sg * s[2]};
    const Pt<R> st = point_state<PERT>(v.q, v.r0, v.E0, ph);
    const R kr = kr_at<N, D, KR>(A, e, ln, side ? N : 0);
    R Fv[4];
    flux_visc<PERT>(st, v.q, v.g, v.gr0, v.r0, v.E0, So, ph, kr, Fv);
    if ((side ? kind[1] : kind[0]) < 0) Fv[3] = wall_conduction(v.g, So, kr, ph);
    R* o = A.Tv_out + ((size_t)e * 6 + 2 * D + side) * 4 * N2 + ln;
#pragma unroll
    for (int c = 0; c < 4; ++c) o[c * N2] = Fv[c];
  };

  if constexpr (FB == 1) {
    Pair<R> lines[REG ? NP : 1][N];
    if constexpr (REG) {
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        R u[N], w[N];
        load_pair(k, u, w);
#pragma unroll
        for (int s = 0; s < N; ++s) lines[k][s] = Pair<R>{u[s], w[s]};
      }
    }
    loaded();
    R sn[3];
#pragma unroll
    for (int n = 0; n < 3; ++n) sn[n] = metric(n, 0);
#pragma unroll 1
    for (int f = 0; f <= N; ++f) {
      R s3[3];
#pragma unroll
      for (int n = 0; n < 3; ++n) s3[n] = sn[n];
      if (f < N) {  // the next flux point's metrics
#pragma unroll
        for (int n = 0; n < 3; ++n) sn[n] = metric(n, f + 1);
      }
      Pair<R> w[N], P[NP];
#pragma unroll
      for (int s = 0; s < N; ++s) w[s] = tI[f * N + s];
      if constexpr (REG) {  // independent products side by side
#pragma unroll
        for (int k = 0; k < NP; ++k) P[k] = mul2(w[0], lines[REG ? k : 0][0]);
#pragma unroll
        for (int s = 1; s < N; ++s)
#pragma unroll
          for (int k = 0; k < NP; ++k) P[k] = fma2(w[s], lines[REG ? k : 0][s], P[k]);
      } else {
#pragma unroll
        for (int k = 0; k < NP; ++k) {
          R u[N], y[N];
          load_pair(k, u, y);
          P[k] = mul2(w[0], Pair<R>{u[0], y[0]});
#pragma unroll
          for (int s = 1; s < N; ++s) P[k] = fma2(w[s], Pair<R>{u[s], y[s]}, P[k]);
        }
      }
      const Vals v = unpack(P);
      if (f > 0 && f < N) interior(v, s3, f);
      else end(v, s3, f == N);
    }
  } else {
    static_assert(2 * FB >= N + 1 && FB <= N, "two blocks cover the line");
#pragma unroll 1
    for (int b = 0; b < 2; ++b) {
      const int cnt = b ? N + 1 - FB : FB;
      R s3[FB][3];
#pragma unroll
      for (int j = 0; j < FB; ++j) {
        const int f = b ? N - j : j;
        if (FB == N + 1 - FB || j < cnt) {
#pragma unroll
          for (int n = 0; n < 3; ++n) s3[j][n] = metric(n, f);
        }
      }
      Pair<R> P[FB][NP];
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        R u[N], y[N];
        load_pair(k, u, y);
        if constexpr (const_weights<N>()) {
          if (b) {
#pragma unroll
            for (int s = 0; s < N / 2; ++s) {
              const R a = u[s], c = y[s];
              u[s] = u[N - 1 - s];
              y[s] = y[N - 1 - s];
              u[N - 1 - s] = a;
              y[N - 1 - s] = c;
            }
          }
#pragma unroll
          for (int j = 0; j < FB; ++j) {
            Pair<R> t{A.ops.I[j][0] * u[0], A.ops.I[j][0] * y[0]};
#pragma unroll
            for (int s = 1; s < N; ++s) t = Pair<R>{t.x + A.ops.I[j][s] * u[s], t.y + A.ops.I[j][s] * y[s]};
            P[j][k] = t;
          }
        } else {
#pragma unroll
          for (int j = 0; j < FB; ++j) {
            Pair<R> t{R(0), R(0)};
#pragma unroll
            for (int s = 0; s < N; ++s) t = fma2(tI[(b ? N - j : j) * N + s], Pair<R>{u[s], y[s]}, t);
            P[j][k] = t;
          }
        }
      }
      end(unpack(P[0]), s3[0], b);
#pragma unroll
      for (int j = 1; j < FB; ++j)
        if (FB == N + 1 - FB || j < cnt) interior(unpack(P[j]), s3[j], b ? N - j : j);
    }
  }
#pragma unroll
  for (int i = 0; i < N; ++i) {
    acc[0][i] = a01[i].x;
    acc[1][i] = a01[i].y;
    acc[2][i] = a23[i].x;
    acc[3][i] = a23[i].y;
    acc[4][i] = a4[i];
  }
}

// Adds (or, FIRST, stores) the line's derivative into the divergence sums.
template <int N, class R, int D, bool FIRST>
__device__ __forceinline__ void add_div(const Elem<R>& x, int ln, const R (&acc)[5][N]) {
  constexpr int N3 = N * N * N;
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    R* d = x.g + (kG + v) * N3;
    if constexpr (D == 0 && N == 4 && sizeof(R) == 4) {
      float4* p = reinterpret_cast<float4*>(d + line_sidx<N, 0, R>(ln, 0));
      const float4 o = FIRST ? make_float4(0.f, 0.f, 0.f, 0.f) : *p;
      *p = make_float4(o.x + acc[v][0], o.y + acc[v][1], o.z + acc[v][2], o.w + acc[v][3]);
    } else {
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const int si = line_sidx<N, D, R>(ln, i);
        if (FIRST) d[si] = acc[v][i];
        else d[si] += acc[v][i];
      }
    }
  }
}

// ------------------------------------------------------------------ volume kernel

// Bound by instruction issue and the latency of dependent instructions at the warps that registers
// allow: at p = 3 in FP32 (331,776 elements) 1.14 ms for 12.2 KB of DRAM traffic an element, 58 % of the
// issue slots at 12 warps per SM, DRAM at 43 %; the lifting and residual kernels that it replaces took 1.97 ms,
// 28.9 KB and 1.5 times the instructions.  p = 2 (98,304 elements) 0.52 -> 0.18 ms, p = 4 (111,078) 2.92 ->
// 0.97 ms (shared-memory pipe 63 %), p = 5 (98,304) 3.34 -> 1.85 ms; FP64 at p = 3 43.7 -> 31.9 ms, at the
// FP64 units' rate.

// Barriers of a unit: the staging, the two refills of the metric buffers, and the epilogue's inputs.
constexpr int kVolBars = 4;

// The operator tables of a CTA's tiles, each value as a pair; a CTA barrier follows before the tiles read
// them.  (A table for each staging unit, stored in vol_tile, needs no barrier but measured slower: p = 3,
// 4,800 elements 38.1 -> 39.4 us a stage, 98,304 elements 575 -> 578.)  NT: threads of the CTA.
template <int N, bool PERT, class R, int EPB, int NT>
__device__ __forceinline__ void stage_tables(const KArgs<R>& A) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  R* tab = reinterpret_cast<R*>(smem_raw) + Layout<N, PERT, R, EPB>::oI;
  for (int i = threadIdx.x; i < 2 * (N + 1) * N; i += NT) {
    const R w = __ldg(A.m.tab + i);
    *reinterpret_cast<Pair<R>*>(tab + 2 * i) = Pair<R>{w, w};
  }
}

// Tile `tile` (elements tile * EPB ...; threads beyond EPB * N^2 idle but take part in the barriers).
// bars: the CTA's barriers, kVolBars for each unit (initialised), pbar: the parity of their next phase.
template <int N, bool PERT, class R, int EPB, bool KR>
__device__ __forceinline__ void vol_tile(const KArgs<R>& A, int64_t tile, uint64_t* bars, uint32_t& pbar) {
  using L = Layout<N, PERT, R, EPB>;
  constexpr int N2 = N * N, N3 = N * N * N;
  constexpr int UE = unit_elems<N, EPB>(), UT = unit_threads<N, EPB>();
  extern __shared__ __align__(128) unsigned char smem_raw[];
  R* sm = reinterpret_cast<R*>(smem_raw);
  const int el = threadIdx.x / N2, ln = threadIdx.x % N2;
  const int unit = warp_local<N>() ? threadIdx.x / 32 : 0, tid = warp_local<N>() ? threadIdx.x % 32 : threadIdx.x;
  if (EPB % UE == 0 && unit >= EPB / UE) return;  // a whole idle warp of a wider launch
  const int u0 = unit * UE;
  const int e0 = (int)(tile * EPB) + u0;
  const int ne = max(0, min(UE, A.m.E - e0));
  const int e = e0 + el - u0;
  const bool active = el - u0 < ne;
  uint64_t* bar = bars + unit * kVolBars;
  if (ne == 0) return;  // the same in every thread of the unit
  const uint32_t polls = wait_polls(A.err);
  const uint32_t par = pbar;
  const R* tab = sm + L::oI;
  LiftPre<N, R, L::SM> pre[L::SM ? 3 : 1];
  int nbr[6] = {0, 0, 0, 0, 0, 0};
  if (active) load_six(A.m.nbr, e, nbr);
  Shift sh;
  if (!stage_elements<N, PERT, R, EPB>(A, sm, bar, pbar, e0, ne, u0, tid, UT, sh, polls, [&] {
        if (!active) return;
        lift_prefetch<N, R, 2, L::SM>(A, e, ln, pre[0], nbr);
        if constexpr (L::SM) {
          lift_prefetch<N, R, 1, L::SM>(A, e, ln, pre[1], nbr);
          lift_prefetch<N, R, 0, L::SM>(A, e, ln, pre[2], nbr);
        }
      })) {
    if (active && ln == 0) A.skip_out[e] = 1;
    return;
  }
  const R *S0 = sm + L::oS0 + u0 * L::SS, *S1 = sm + L::oS1 + u0 * L::SS;  // the unit's metric buffers
  const Elem<R> x{sm + L::oQ + sh.q + el * L::SQ,
                  sm + L::oBG + sh.bg + el * L::SBG,
                  sm + L::oGR0 + sh.gr0 + el * L::SGR0,
                  sm + L::oG + el * L::SG,
                  sm + L::oIJ + sh.ij + el * L::SIJ,
                  sm + L::oS0 + el * L::SS,
                  sm + L::oS1 + el * L::SS};
  // refills a metric buffer that every thread of the unit has finished with
  auto refill = [&](int d, const R* dst, uint64_t* b) {
    if constexpr (L::SM) {
      if (tid == 0) {
        fence_async_smem();  // its previous contents were read by the generic proxy
        mbar_expect_tx(b, ne * L::SS * sizeof(R));
        issue_metrics<N, R, L>(A.m.Sf, e0, ne, d, const_cast<R*>(dst), b);
      }
    }
  };
  bool failed = false;
  if (active) lift_dir<N, PERT, R, 2, L::SM>(A, x, ln, e, pre[0]);
  if constexpr (L::SM) {
    unit_sync<N>();
    refill(0, S0, bar + 1);
  } else if (active) {
    lift_prefetch<N, R, 1, L::SM>(A, e, ln, pre[0], nbr);
  }
  if (active) lift_dir<N, PERT, R, 1, L::SM>(A, x, ln, e, pre[L::SM ? 1 : 0]);
  if constexpr (L::SM) failed |= !mbar_wait(bar + 1, par, A.err, polls);
  else if (active) lift_prefetch<N, R, 0, L::SM>(A, e, ln, pre[0], nbr);
  unit_sync<N>();
  if (active) lift_dir<N, PERT, R, 0, L::SM>(A, x, ln, e, pre[L::SM ? 2 : 0]);
  unit_sync<N>();
  R acc[5][N];
  if (active) {
    const int kind[2] = {nbr[2], nbr[3]};
    flux_dir<N, PERT, R, 1, KR>(A, x, tab, ln, e, kind, x.S1, acc, [] {});
    add_div<N, R, 1, true>(x, ln, acc);
  }
  unit_sync<N>();
  refill(2, S1, bar + 2);
  if (active) {
    const int kind[2] = {nbr[0], nbr[1]};
    flux_dir<N, PERT, R, 0, KR>(A, x, tab, ln, e, kind, x.S0, acc, [] {});
    add_div<N, R, 0, false>(x, ln, acc);
  }
  if constexpr (L::SM) failed |= !mbar_wait(bar + 2, par, A.err, polls);
  unit_sync<N>();
  // the epilogue's inputs: staged (SE) into the record's space (R(Q0)) and the free metric buffer (x)
  constexpr bool SE = PERT && stage_epilogue<N, R>();
  const bool want_r0 = PERT && !late_background<N, R>() && A.bg.R0 != nullptr;
  const unsigned lanes = SE ? __ballot_sync(0xffffffffu, active) : 0u;
  if constexpr (PERT && !SE) {
    if (tid == 0) {
      prefetch_l2(A.m.x + (size_t)e0 * 3 * N3, ne * 3 * N3 * sizeof(R));
      if (want_r0) prefetch_l2(A.bg.R0 + (size_t)e0 * 5 * N3, ne * 5 * N3 * sizeof(R));
    }
  }
  auto stage_late = [&] {
    if constexpr (SE) {
      __syncwarp(lanes);  // the lines of the warp's elements are in registers
      if (tid == 0) {
        fence_async_smem();
        constexpr uint32_t b5 = 5 * N3 * sizeof(R), b3 = 3 * N3 * sizeof(R);
        mbar_expect_tx(bar + 3, ne * ((want_r0 ? b5 : 0) + b3));
        for (int j = 0; j < ne; ++j) {
          if (want_r0) bulk_g2s(sm + L::oG + (u0 + j) * L::SG, A.bg.R0 + (size_t)(e0 + j) * 5 * N3, b5, bar + 3);
          bulk_g2s(const_cast<R*>(S0) + j * L::SS, A.m.x + (size_t)(e0 + j) * 3 * N3, b3, bar + 3);
        }
      }
    }
  };
  if (active) {
    const int kind[2] = {nbr[4], nbr[5]};
    flux_dir<N, PERT, R, 2, KR>(A, x, tab, ln, e, kind, x.S1, acc, stage_late);
  }
  // a refill that gave up (flag set, copies drained): the unit stores none of its elements
  if constexpr (SE) failed |= !mbar_wait(bar + 3, par, A.err, polls);
  if constexpr (L::SM) failed = warp_local<N>() ? __any_sync(0xffffffffu, failed) : __syncthreads_or(failed);
  if (!active) return;
  if (ln == 0) A.skip_out[e] = failed;
  if (failed) return;

  // Thread ln holds its zeta-line's points ln + N^2 i (i < N): consecutive threads read consecutive words
  // of each array.  Inputs that are not staged are loaded one point ahead.
  struct In {
    R x[3], ij, r0[5];
  };
  auto load_in = [&](int i) {
    In v;
    const int pt = ln + N2 * i;
#pragma unroll
    for (int n = 0; n < 3; ++n) v.x[n] = SE ? x.S0[n * N3 + pt] : __ldg(A.m.x + ((size_t)e * 3 + n) * N3 + pt);
    v.ij = L::SM ? x.ij[pt] : __ldg(A.m.invJ + (size_t)e * N3 + pt);
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      if constexpr (SE) v.r0[c] = want_r0 ? x.g[c * N3 + pt] : R(0);
      else v.r0[c] = want_r0 ? (R)__ldg(A.bg.R0 + ((size_t)e * 5 + c) * N3 + pt) : R(0);
    }
    return v;
  };
  // residual dQ/dt = -div/|J| - M (Eqs. 4, 11) without the end points, sources of Eqs. 2-3
  const PhysArg<R>& ph = A.ph;
  In cur, nxt = load_in(0);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    cur = nxt;
    if (i + 1 < N) nxt = load_in(i + 1);
    const int pt = ln + N2 * i;
    const int si = sidx<N, R>(ln % N, ln / N, i);
    R q[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) q[v] = x.q[v * N3 + pt];
    R gr = ph.GM;  // g3 points outward (the source uses -rho g_vec); FP32: x holds x / |x|^3
    if constexpr (sizeof(R) == 8) {
      const R r2 = dot3(cur.x, cur.x);
      gr *= qrcp(r2 * sqrt(r2));
    }
    const R g3[3] = {gr * cur.x[0], gr * cur.x[1], gr * cur.x[2]};
    R M[5];
    M[0] = R(0);
    M[1] = q[0] * g3[0] - ph.twoOmega * q[2];
    M[2] = q[0] * g3[1] + ph.twoOmega * q[1];
    M[3] = q[0] * g3[2];
    M[4] = q[1] * g3[0] + q[2] * g3[1] + q[3] * g3[2];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      R Rv = -(x.g[(kG + v) * N3 + si] + acc[v][i]) * cur.ij - M[v];
      if (PERT && !late_background<N, R>()) Rv += cur.r0[v];
      const size_t oi = ((size_t)e * 5 + v) * N3 + pt;
      A.part_out[oi] = Rv;
    }
  }
}

template <int N, bool PERT, class R, int EPB, bool KR>
__global__ void __launch_bounds__(EPB * N * N, sizeof(R) == 4 ? vol_min_blocks<N, EPB>() : 1) k_vol(const KArgs<R> A) {
  constexpr int units = Layout<N, PERT, R, EPB>::units;
  __shared__ __align__(8) uint64_t bars[units * kVolBars];
  pdl_trigger();
  if (threadIdx.x < units * kVolBars) mbar_init(&bars[threadIdx.x]);
  stage_tables<N, PERT, R, EPB, EPB * N * N>(A);
  __syncthreads();
  uint32_t ph = 0;
  vol_tile<N, PERT, R, EPB, KR>(A, blockIdx.x, bars, ph);
}

// ------------------------------------------------------------------ face kernel

// Common flux of every interior face point, once per face (Section 3: Rusanov inviscid flux with the
// wave speed of both sides, average of the two one-sided viscous fluxes from the volume kernel).
// One thread per (face, point) of the face list (element, local face) of owner sides.  |S| F_n along the
// owner's outward S, at the owner's points, is written once, in face order; both elements read it (one
// with the other sign: the two sides' fluxes are exactly opposite), which for all but the first reader
// hits L2.  Bound by DRAM: 6.4 KB an element at p = 3, 97 % of the copy rate (0.322 ms at 331,776
// elements).  (Written in both elements' own numbering: k_face 0.354 instead of 0.322 ms, k_update 0.318
// instead of 0.310, at p = 3 and 331,776 elements.)
//
// Wall faces follow the interior ones in the list (entries nf..nf+nw-1): their common flux (Section 5)
// is formed from the element's own trace and the volume kernel's wall data (the viscous traction
// tau S and the conductive flux with the top temperature imposed).
// One thread's face point g (of (nf + nw) * N^2).
template <int N, bool PERT, class R>
__device__ __forceinline__ void face_point(const KArgs<R>& A, const int2* __restrict__ faces, int nf, int nw, int64_t g) {
  constexpr int N2 = N * N;
  if (g < 0 || g >= (int64_t)(nf + nw) * N2) return;
  const int t = (int)(g % N2);
  const int2 fc = faces[g / N2];
  const int e = fc.x, F = fc.y, D = F >> 1, side = F & 1;
  const int k = __ldg(A.m.nbr + e * 6 + F), code = __ldg(A.m.code + e * 6 + F);
  const R sgn = side ? R(1) : R(-1);
  const bool wall = k < 0;
  // own slot: the other side's traces and background (a wall's own), own one-sided viscous flux; the
  // neighbour's slot: own traces and background, the neighbour's viscous flux
  const size_t oL = (size_t)e * 6 + F;
  const int Fn = wall ? F : code >> 3, tp = wall ? t : map_face_pt<N>(t, code & 7);
  const size_t oR = wall ? oL : (size_t)k * 6 + Fn;
  R qL[5], tvL[4], So[3], qR[5], tvR[4];
#pragma unroll
  for (int n = 0; n < 3; ++n)
    So[n] = sgn * __ldg(A.m.Sf + (((size_t)e * 3 + D) * 3 * (N + 1) + n * (N + 1) + (side ? N : 0)) * N2 + t);
  R r0L = R(0), E0L = R(0), r0R = R(0), E0R = R(0);
  if (PERT) {
    r0R = (R)__ldg(A.bg.bgT + (oL * 2) * N2 + t);
    E0R = (R)__ldg(A.bg.bgT + (oL * 2 + 1) * N2 + t);
    r0L = (R)__ldg(A.bg.bgT + (oR * 2) * N2 + tp);
    E0L = (R)__ldg(A.bg.bgT + (oR * 2 + 1) * N2 + tp);
  }
  pdl_wait();
#pragma unroll
  for (int v = 0; v < 5; ++v) qR[v] = ld_written(A.T + (oL * 5 + v) * N2 + t);
#pragma unroll
  for (int v = 0; v < 4; ++v) tvL[v] = ld_written(A.Tv + (oL * 4 + v) * N2 + t);
  if (wall) {  // exact inviscid flux (0, p S, 0) minus the normal viscous traction; energy: f.S
    const Pt<R> st = point_state<PERT>(qR, r0R, E0R, A.ph);
    const R mag2 = dot3(So, So);
    const R pn = st.p - dot3(tvL, So) * qrcp(mag2);
    R Fh[5] = {R(0), pn * So[0], pn * So[1], pn * So[2], tvL[3]};
    if (k != -2) Fh[4] = PERT ? R(0) : -A.ph.bottom_flux * sqrt(mag2);
#pragma unroll
    for (int v = 0; v < 5; ++v) A.Fc_out[((g / N2) * 5 + v) * N2 + t] = Fh[v];
    return;
  }
#pragma unroll
  for (int v = 0; v < 5; ++v) qL[v] = ld_written(A.T + (oR * 5 + v) * N2 + tp);
#pragma unroll
  for (int v = 0; v < 4; ++v) tvR[v] = ld_written(A.Tv + (oR * 4 + v) * N2 + tp);
  const Pt<R> sL = point_state<PERT>(qL, r0L, E0L, A.ph);
  const Pt<R> sR = point_state<PERT>(qR, r0R, E0R, A.ph);
  R Fh[5];
  rusanov<PERT>(qL, sL, r0L, E0L, qR, sR, r0R, E0R, So, sqrt(dot3(So, So)), A.ph, Fh);
#pragma unroll
  for (int v = 1; v < 5; ++v) Fh[v] -= R(0.5) * (tvL[v - 1] - tvR[v - 1]);  // tvR is along -S
#pragma unroll
  for (int v = 0; v < 5; ++v) A.Fc_out[((g / N2) * 5 + v) * N2 + t] = Fh[v];
}

template <int N, bool PERT, class R>
__global__ void __launch_bounds__(64) k_face(const KArgs<R> A, const int2* __restrict__ faces, int nf, int nw) {
  pdl_trigger();
  face_point<N, PERT, R>(A, faces, nf, nw, blockIdx.x * (int64_t)blockDim.x + threadIdx.x);
}

// ------------------------------------------------------------------ update kernel

// Shared memory of the update kernel: the common fluxes of the xi and eta faces and the new state.
template <int N, class R, int EPB>
struct UpLayout {
  static constexpr int N2 = N * N, N3 = N * N * N;
  static constexpr int SF = N == 4 ? pad_stride<R>(20 * N2) : 20 * N2;
  static constexpr int SW = N == 4 ? pad_stride<R>(5 * N3) : 5 * N3;
  static constexpr int oF = 0, oW = EPB * SF;
  static constexpr int total = oW + EPB * SW;
};

// The end-point fluxes' part of the divergence, added to the volume kernel's partial residual; in RK mode
// the stage's combination and the traces of the new state.  ADD: with an additive correction.  Thread ln takes the points ln + N^2 i of its
// element.  An element for which the volume kernel gave up a wait is left as it is.  Bound by DRAM: at p = 3,
// 331,776 elements, 7.5 KB an element in 0.410 ms, 89 % of the copy rate.  One point's inputs are loaded while the
// point before is worked on: all of them ahead took 96 registers, which slowed the kernel (0.590 ms) and, no
// room being left for its early start, a stage of 1,470 elements too (20.4 -> 26.2 us).
template <int N, class R, int EPB, int MODE, bool ADD>
__device__ __forceinline__ void update_tile(const KArgs<R>& A, int64_t tile) {
  using L = UpLayout<N, R, EPB>;
  constexpr int N2 = N * N, N3 = N * N * N;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  R* sm = reinterpret_cast<R*>(smem_raw);
  const int el = threadIdx.x / N2, ln = threadIdx.x % N2;
  const int64_t e = tile * EPB + el;
  bool active = el < EPB && e < A.m.E;
  R* sF = sm + L::oF + el * L::SF;
  R* sW = sm + L::oW + el * L::SW;
  constexpr int NI = MODE == kModeRK ? 5 : 1;
  R Fz[2][5];
  int nbr[6], code[6], fid[6];
  if (active) {
    load_six(A.m.nbr, e, nbr);
    load_six(A.m.code, e, code);
    load_six(A.m.fid, e, fid);
  }
  constexpr bool LATE = late_background<N, R>();
  pdl_wait();
  const int skip = active ? ld_written(A.skip + e) : 1;
  // A point's inputs, loaded one point ahead.
  struct In {
    R ij, part[5], q[NI], un[NI], add[ADD ? 5 : 1], r0[LATE ? 5 : 1];
  };
  auto load_in = [&](int i) {
    In in;
    in.ij = __ldg(A.m.invJ + (size_t)e * N3 + ln + N2 * i);
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const size_t oi = ((size_t)e * 5 + v) * N3 + ln + N2 * i;
      in.part[v] = ld_written(A.part + oi);
      if constexpr (ADD) in.add[v] = ld_written(A.radd + oi);
      if constexpr (LATE) in.r0[v] = A.r0 != nullptr ? __ldg(A.r0 + oi) : R(0);
      if constexpr (MODE == kModeRK) {
        in.q[v] = ld_written(A.q + oi);
        in.un[v] = A.a != R(0) ? ld_written(A.un + oi) : R(0);  // a stage without a u^n term does not read it
      }
    }
    return in;
  };
  In nxt;
  if (active) {
    // the faces' common fluxes at own points, along xi_d: the owner is the lower-numbered element
    R Fxy[20];
#pragma unroll
    for (int F = 0; F < 6; ++F) {
      const bool own = nbr[F] < 0 || nbr[F] > A.m.e0 + e;
      const R* Ff = A.Fc + (size_t)fid[F] * 5 * N2 + (own ? ln : map_face_pt<N>(ln, code[F] & 7));
      const R sg = own == ((F & 1) != 0) ? R(1) : R(-1);
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        const R f = sg * ld_written(Ff + v * N2);
        if (F < 4) Fxy[F < 4 ? 5 * F + v : 0] = f;
        else Fz[F < 4 ? 0 : F - 4][v] = f;
      }
    }
    nxt = load_in(0);
#pragma unroll
    for (int c = 0; c < 20; ++c) sF[c * N2 + ln] = Fxy[c];
  }
  unit_sync<N>();
  active = skip == 0;
  if (active) {
    const int a = ln % N, b = ln / N;
    const R d0a = A.ops.D[a][0], dNa = A.ops.D[a][N], d0b = A.ops.D[b][0], dNb = A.ops.D[b][N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int pt = ln + N2 * i, si = sidx<N, R>(a, b, i);
      const In in = nxt;
      if (i + 1 < N) nxt = load_in(i + 1);
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        R s = A.ops.D[i][0] * Fz[0][v] + A.ops.D[i][N] * Fz[1][v];
        s += d0a * sF[v * N2 + b + N * i] + dNa * sF[(5 + v) * N2 + b + N * i];
        s += d0b * sF[(10 + v) * N2 + a + N * i] + dNb * sF[(15 + v) * N2 + a + N * i];
        s *= in.ij;
        const size_t oi = ((size_t)e * 5 + v) * N3 + pt;
        R w = in.part[v] - s;
        if constexpr (LATE) w += in.r0[v];
        if constexpr (ADD) w += in.add[v];  // the whole residual
        if constexpr (MODE == kModeRK) {
          const R dR = A.dt * w, bq = A.b * in.q[v];
          if (A.out2) A.out2[oi] = fma_rn(A.c2, dR, fma_rn(A.a2, A.un2[oi], A.b2 * in.q[v]));
          w = fma_rn(A.c, dR, A.a != R(0) ? fma_rn(A.a, in.un[v], bq) : bq);  // the new state
          sW[v * N3 + si] = w;
        }
        A.out[oi] = w;
      }
    }
  }
  if constexpr (MODE == kModeRK) {
    if (A.T_out == nullptr) return;
    unit_sync<N>();
    if (!active) return;
    load_six(A.m.nbr, e, nbr);  // again: kept in registers over the points they cost a CTA per SM
    load_six(A.m.code, e, code);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      R* T0 = A.T_out + trace_slot<N>(A.m.e0 + e, 2 * d, nbr[2 * d], code[2 * d], ln);
      R* T1 = A.T_out + trace_slot<N>(A.m.e0 + e, 2 * d + 1, nbr[2 * d + 1], code[2 * d + 1], ln);
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        R l[N];
        if (d == 0) load_line<N, 0, kComputed>(sW + v * N3, ln, l);
        else if (d == 1) load_line<N, 1, kComputed>(sW + v * N3, ln, l);
        else load_line<N, 2, kComputed>(sW + v * N3, ln, l);
        R lo = R(0), hi = R(0);
#pragma unroll
        for (int s = 0; s < N; ++s) {
          lo += A.ops.I[0][s] * l[s];
          hi += A.ops.I[N][s] * l[s];
        }
        T0[v * N2] = lo;
        T1[v * N2] = hi;
      }
    }
  }
}

template <int N, class R, int EPB, int MODE, bool ADD>
__global__ void __launch_bounds__(EPB * N * N) k_update(const KArgs<R> A) {
  pdl_trigger();
  update_tile<N, R, EPB, MODE, ADD>(A, blockIdx.x);
}

// ------------------------------------------------------------------ launch helpers

// Launch of a stage kernel that may start while the kernel before it on the stream drains (programmatic
// dependent launch): every stage kernel lets its successor start at once (pdl_trigger) and reads what its
// predecessor wrote only after pdl_wait, which returns once that kernel has completed and its writes are
// visible.  A kernel completes only after its own wait, so the order reaches back along the stream.
template <class... P, class... Q>
cudaError_t launch_dependent(bool early, void (*k)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, Q&&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = early ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k, std::forward<Q>(args)...);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <int N, bool PERT, class R, int EPB>
struct Launch {
  static constexpr int threads = EPB * N * N;
  static int blocks(int E) { return (E + EPB - 1) / EPB; }
  // Early launches (launch_dependent) pay where a stage is a few tens of microseconds: at 12,288 elements
  // they took 8, 5, 4 and 1 % off a stage at p = 2..5 (p = 3, 288 elements: 23.1 -> 16.7 us), from 28,800
  // they cost p = 2 and 3 1 to 9 % and the others gain nothing.
  static bool early(int E) { return E <= 16384; }

  static cudaError_t trace(const MeshArg<R>& m, const OpsArg<R>& ops, const R* q, R* T, cudaStream_t st) {
    if (m.E == 0) return cudaSuccess;
    k_trace<N, R, EPB><<<blocks(m.E), threads, 0, st>>>(m, ops, q, T);
    return cudaGetLastError();
  }
  static cudaError_t face(const KArgs<R>& A, const int2* faces, int nf, int nw, cudaStream_t st) {
    if (nf + nw == 0) return cudaSuccess;
    if (A.Fc_out == nullptr || A.T == nullptr || A.Tv == nullptr) return cudaErrorInvalidValue;
    const int64_t n = (int64_t)(nf + nw) * N * N;
    // 64-thread CTAs (p = 3: 1 % faster than 128, 2.5 % faster than 256)
    return launch_dependent(early(A.m.E), k_face<N, PERT, R>, (unsigned)((n + 63) / 64), 64, 0, st, A, faces, nf, nw);
  }
  static cudaError_t vol(const KArgs<R>& A, cudaStream_t st) {
    if (A.m.E == 0) return cudaSuccess;
    if (A.Tv_out == nullptr || A.T == nullptr || A.part_out == nullptr || A.skip_out == nullptr) return cudaErrorInvalidValue;
    // the radiative-diffusivity profile is a compile-time option of the FP32 kernels (FP64 checks it
    // at run time)
    if constexpr (sizeof(R) == 8) {
      return vol_kr<true>(A, st);
    } else {
      return A.m.kr != nullptr ? vol_kr<true>(A, st) : vol_kr<false>(A, st);
    }
  }
  template <bool KR>
  static cudaError_t vol_kr(const KArgs<R>& A, cudaStream_t st) {
    const size_t sm = (size_t)Layout<N, PERT, R, EPB>::total * sizeof(R);
    cudaError_t e =
        cudaFuncSetAttribute(k_vol<N, PERT, R, EPB, KR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    return launch_dependent(early(A.m.E), k_vol<N, PERT, R, EPB, KR>, blocks(A.m.E), threads, sm, st, A);
  }
  template <int MODE>
  static cudaError_t update(const KArgs<R>& A, cudaStream_t st) {
    if (A.m.E == 0) return cudaSuccess;
    if (A.Fc == nullptr || A.part == nullptr || A.out == nullptr || A.skip == nullptr) return cudaErrorInvalidValue;
    if (MODE == kModeRK && (A.q == nullptr || (A.a != R(0) && A.un == nullptr))) return cudaErrorInvalidValue;
    // the learned closure's order; a kernel of its own, since a test of radd at each point kept the loads of the
    // next from starting early (331,776 elements at p = 3: 1.87 -> 1.99 ms a stage)
    if constexpr (N == 3) {
      if (A.radd != nullptr) return update_add<MODE, true>(A, st);
    }
    return A.radd != nullptr ? cudaErrorInvalidValue : update_add<MODE, false>(A, st);
  }
  template <int MODE, bool ADD>
  static cudaError_t update_add(const KArgs<R>& A, cudaStream_t st) {
    const size_t sm = (size_t)UpLayout<N, R, EPB>::total * sizeof(R);
    auto* k = k_update<N, R, EPB, MODE, ADD>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    return launch_dependent(early(A.m.E), k, blocks(A.m.E), threads, sm, st, A);
  }
};

}  // namespace chorus
