// Kernel templates of the ADG right-hand side, parameterised by dimension D, nodes per
// direction N = degree + 1 and the arithmetic type R of the operator (double, float or
// the FP32-pair type of df64.cuh).  The solution w is FP64 in every variant; the RK
// register (r or q) is stored in the operator's storage type.
//
// Per Runge-Kutta stage the solver runs two kernels:
//   flux_kernel : one thread per (direction, face, face node): numerical flux of Eq. 8-9
//                 from the two stored traces; on faces between subdomains it applies the
//                 delayed / AT rules of Algorithms 2-3 (Eq. 13-14) against a ring buffer.
//   vol_kernel (FP64: vol_kernel_fp64) : a tile of elements per block, one thread per node (FP32
//                 sweeps and traces: per line): pointwise Euler flux (Eq. 2), sum-factorised
//                 weak derivative along each direction, face lift, inverse mass (diagonal for
//                 collocated Gauss points; folded into the tables), the low-storage RK update
//                 (Eq. 10 or the 2N form), and the face traces of the next stage input.
// or one kernel:
//   vol_faces_kernel(_fp64) : the volume kernel with each element evaluating the numerical flux
//                 on its own faces from the stored traces (no face-flux array).
// Node and ring indices are 32-bit: the host rejects meshes with 2^31 or more degrees of freedom and
// rings of 2^31 or more values.  The traces (2 D / N values per degree of freedom) and the face fluxes
// (D / N) may be larger: their offsets are 64-bit (TraceLay).
#pragma once
#include <type_traits>
#include <cuda_runtime.h>
#include <stdint.h>

#include "adg_internal.h"
#include "arith.cuh"
#include "fixline.cuh"

namespace adg {

template <int B, int E>
struct IPow { static constexpr int value = B * IPow<B, E - 1>::value; };
template <int B>
struct IPow<B, 0> { static constexpr int value = 1; };

// Element tile of the volume kernel: about TT threads per block, one thread per node.
template <int D, int N, int TT = 128>
struct Tile {
  static constexpr int ND = IPow<N, D>::value;
  static constexpr int NF = ND / N;
  static constexpr int NV = D + 2;
  static constexpr int EPB = (TT / ND) > 0 ? (TT / ND) : 1;
  static constexpr int THREADS = EPB * ND;
};

// floor(e / m.n[i]) for 0 <= e < 2^31 (multiply-high by the precomputed inverse)
__device__ __forceinline__ int mesh_div(const MeshArgs& m, int i, int e) {
  return m.n[i] == 1 ? e : (int)(__umulhi((unsigned)e, m.divm[i]) >> m.divs[i]);
}

// Blocks per SM that leave `regs` registers per thread (0: no budget): each of the 4 SM
// sub-partitions holds 16384 registers and a whole number of warps.
constexpr int min_blocks_for(int regs, int threads) {
  if (regs == 0) return 1;
  if (threads <= 64 && regs < 48) regs = 48;
  const int warps = (threads + 31) / 32;
  const int b = (16384 / (regs * 32)) * 4 / warps;
  return b < 1 ? 1 : (b > 32 ? 32 : b);
}

__device__ __forceinline__ void elem_coords(const MeshArgs& m, int e, int* c) {
  const int q = mesh_div(m, 0, e);
  c[0] = e - q * m.n[0];
  c[2] = mesh_div(m, 1, q);
  c[1] = q - c[2] * m.n[1];
}

// index of the neighbour of element e (coordinates c) one step s (+1/-1) along d, periodic
// (selects instead of indexing c by a runtime d keep c in registers)
__device__ __forceinline__ int elem_shift(const MeshArgs& m, int e, const int* c, int d, int s) {
  const int cd = d == 0 ? c[0] : (d == 1 ? c[1] : c[2]);
  int k = cd + s;
  if (k < 0) k += m.n[d];
  if (k >= m.n[d]) k -= m.n[d];
  return e + (k - cd) * (int)m.es[d];
}

// Pointwise Euler flux columns F_d(w), d < D (Eq. 2-3, no source).
template <int D, typename R>
__device__ __forceinline__ void euler_flux_all(const R (&w)[D + 2], R gm1, R (&F)[D][D + 2]) {
  const R irho = r_rcp(w[0]);
  R u[D];
  typename Arith<R>::Acc kacc = acc_zero(typename Arith<R>::Acc());
#pragma unroll
  for (int d = 0; d < D; ++d) {
    u[d] = w[1 + d] * irho;
    kacc = acc_fma(w[1 + d], u[d], kacc);
  }
  const R kin2 = acc_result(kacc);
  const R p = gm1 * sub_half(w[D + 1], kin2);
  const R ep = w[D + 1] + p;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    F[d][0] = w[1 + d];
#pragma unroll
    for (int c = 0; c < D; ++c)  // rho u_c u_d is symmetric: each product once
      F[d][1 + c] = c < d ? F[c][1 + d] : (c == d ? r_fma(w[1 + c], u[d], p) : w[1 + c] * u[d]);
    F[d][D + 1] = ep * u[d];
  }
}

// Velocity along e_d, pressure and |u|^2 + c^2 of one trace state (d is a runtime direction;
// selects instead of indexing keep everything in registers).
template <int D, typename R>
__device__ __forceinline__ void side_state(const R (&w)[D + 2], int d, R gamma, R gm1, R& ud, R& p,
                                           R& s2) {
  const R irho = r_rcp(w[0]);
  R k2 = R(0.0f);
  ud = R(0.0f);
#pragma unroll
  for (int c = 0; c < D; ++c) {
    const R uc = w[1 + c] * irho;
    k2 = r_fma(w[1 + c], uc, k2);  // rho |u|^2
    if (c == d) ud = uc;
  }
  p = gm1 * sub_half(w[D + 1], k2);  // (gamma - 1) (E - rho |u|^2 / 2)
  s2 = r_fma(gamma, p, k2) * irho;   // |u|^2 + gamma p / rho
}

// Flux column along e_d and |u|^2 + c^2 of one trace state.
template <int D, typename R>
__device__ __forceinline__ void side_flux(const R (&w)[D + 2], int d, R gamma, R gm1,
                                          R (&fd)[D + 2], R& s2) {
  R ud, p;
  side_state<D, R>(w, d, gamma, gm1, ud, p, s2);
  fd[0] = w[1];
#pragma unroll
  for (int c = 0; c < D; ++c) {
    if (c == d) fd[0] = w[1 + c];
    fd[1 + c] = c == d ? r_fma(w[1 + c], ud, p) : w[1 + c] * ud;
  }
  fd[D + 1] = (w[D + 1] + p) * ud;
}

// Twice the Rusanov flux along +e_d (Eq. 8) with lambda = 1/2 max(sqrt(|u|^2 + c^2))
// (Eq. 9): f = F(w-) + F(w+) + lambda (w- - w+).  The factor 1/2 is folded into the lift
// coefficients of the volume kernel (one operation less per value; scaling by two is
// exact, so the results equal those of the halved form).  Stored fluxes, the ring of
// subdomain-face levels and their AT combinations all carry the factor two.
template <int D, typename R>
__device__ __forceinline__ void llf_flux(const R (&wm)[D + 2], const R (&wp)[D + 2], int d,
                                         R gamma, R gm1, R (&f)[D + 2]) {
  constexpr int NV = D + 2;
  if constexpr (std::is_same<R, double>::value) {
    // Bound by the FP64 pipe, 2D 46 and 3D 54 operations (from about 78 and 81): the square
    // root takes 6, the larger speed is found by integer comparison, and the two sides'
    // products are summed as they are formed.  256^2 p=4: 81 -> 69 us per launch; 48^3 p=3:
    // 677 -> 558 us.
    double um, up, pm, pp, sm, sp;
    side_state<D, double>(wm, d, gamma, gm1, um, pm, sm);
    side_state<D, double>(wp, d, gamma, gm1, up, pp, sp);
    const double lam = half_sqrt(speed_max(sm, sp)), psum = pm + pp;
    double mm = wm[1], mp = wp[1];  // normal momentum
#pragma unroll
    for (int c = 1; c < D; ++c) {
      mm = c == d ? wm[1 + c] : mm;
      mp = c == d ? wp[1 + c] : mp;
    }
    f[0] = fma(lam, wm[0] - wp[0], mm + mp);
#pragma unroll
    for (int c = 0; c < D; ++c) {
      const double s = fma(wm[1 + c], um, c == d ? psum : 0.0);
      f[1 + c] = fma(lam, wm[1 + c] - wp[1 + c], fma(wp[1 + c], up, s));
    }
    f[D + 1] = fma(lam, wm[D + 1] - wp[D + 1], fma(wp[D + 1] + pp, up, (wm[D + 1] + pm) * um));
  } else {
    R fm[NV], fp[NV], sm, sp;
    if constexpr (std::is_same<R, df64>::value) {
      // FP32 pairs: both sides in the two lanes of packed FP32x2 instructions
      df64x2 w2[NV], f2[NV], s2;
#pragma unroll
      for (int v = 0; v < NV; ++v) w2[v] = df64x2_of(wm[v], wp[v]);
      side_flux<D, df64x2>(w2, d, df64x2_of(gamma, gamma), df64x2_of(gm1, gm1), f2, s2);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        fm[v] = df64x2_lane(f2[v], 0);
        fp[v] = df64x2_lane(f2[v], 1);
      }
      sm = df64x2_lane(s2, 0);
      sp = df64x2_lane(s2, 1);
    } else {
      side_flux<D, R>(wm, d, gamma, gm1, fm, sm);
      side_flux<D, R>(wp, d, gamma, gm1, fp, sp);
    }
    const R lam = scale_pow2(r_sqrt(r_max(sm, sp)), 0.5f);
#pragma unroll
    for (int v = 0; v < NV; ++v) f[v] = r_fma(lam, wm[v] - wp[v], fm[v] + fp[v]);
  }
}

// Transverse coordinates of face node j of a face normal to d -> base node index of the
// line of nodes along d through it.
template <int D, int N>
__device__ __forceinline__ int line_base(int d, int j) {
  int base = 0, stride = 1, t = j;
#pragma unroll
  for (int c = 0; c < D; ++c) {
    if (c != d) {
      base += (t % N) * stride;
      t /= N;
    }
    stride *= N;
  }
  return base;
}

// Face node index of volume node (ix) on a face normal to d.
template <int D, int N>
__device__ __forceinline__ int face_index(int d, const int* ix) {
  int j = 0, stride = 1;
#pragma unroll
  for (int c = 0; c < D; ++c) {
    if (c != d) {
      j += ix[c] * stride;
      stride *= N;
    }
  }
  return j;
}

// Asynchronous 4- and 8-byte copies global -> shared memory (cp.async; sm_80 and later).
// The issuing thread waits for its own copies with cp_async_wait<n> (at most n of its
// committed groups still pending); nothing spins.
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int n>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(n) : "memory");
}

// Programmatic dependent launch: a stage's kernels may be launched as soon as the blocks of the
// previous kernel of the stream have exited, before its grid has completed and its writes are
// visible; a kernel waits for that here, before it touches anything another kernel writes.
// This hides most of the launch latency: 16^2 p=2 FP64 14.7 -> 10.2 us per stage, FP32 7.0 ->
// 5.4; 64^2 p=2 FP64 16.6 -> 12.6; 256^2 p=4 FP64 176 -> 172, pairs 134 -> 129, FP32 57.4 ->
// 54.6.  (Letting the next grid launch earlier, griddepcontrol.launch_dependents, places its
// blocks while the previous grid is still spread unevenly: 64^2 p=2 FP64 16.5 to 23 us.)
__device__ __forceinline__ void grid_dependency() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ---- mbarrier and TMA bulk copies (PTX) -----------------------------------------------
__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Waits for phase `parity` of the barrier for at most `limit` SM clock cycles.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, unsigned parity, long long limit) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > limit) return false;
  }
  return true;
}
// 1D bulk copy global -> shared by the TMA engine (both addresses 16-byte aligned, size a
// multiple of 16 bytes), completion counted on the mbarrier
__device__ __forceinline__ void bulk_load(void* dst, const void* src, unsigned bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// about one second at the GB300 SM clock
constexpr long long kWaitLimitCycles = 2000000000ll;

// Arithmetic of the trace interpolation for an operator arithmetic R: the FP32-pair kernels
// interpolate in native FP64 (the RK update hands over the FP64 stage input), the others in R
// itself.  These chains are about half of the pair kernels' FP64 operations, whose pipe is 78 % busy
// (256^2 p=4); in fixed point they cost 15 % more time, as the kernels are bound by issue as well.
template <typename R> struct TraceCompute { using C = R; };
template <> struct TraceCompute<df64> { using C = double; };

__device__ __forceinline__ void store_trace(double* p, double v) { *p = v; }
__device__ __forceinline__ void store_trace(float* p, float v) { *p = v; }
__device__ __forceinline__ void store_trace(float2* p, double v) {
  const df64 q = d2df_int(v);
  *p = make_float2(q.hi, q.lo);
}
__device__ __forceinline__ void store_trace(float2* p, df64 v) { *p = make_float2(v.hi, v.lo); }

// Layout of the trace arrays: [d][side][v][e][j], in the FP32 operator [d][side][e][j][v] -- the
// variables of a face node together, so that a 2D node's traces are one 16-byte access (in 3D
// five accesses from one address).
template <int D, int N, typename R>
struct TraceLay {
  static constexpr int NF = IPow<N, D - 1>::value, NV = D + 2;
  static constexpr bool kTogether = std::is_same<R, float>::value;
  // ds = 2 d + side (side 1: the element's +d face).  64 bits from the last product on: 2 D NV ne and
  // 2 D ne NF are at most NV ne ND < 2^31.  (Us per volume launch with the other one of
  // the last two forms: pairs 48^3 p=3 824 for 745, 32^3 p=5 918 for 867; FP64 48^3 772 for 763.)
  __device__ static __forceinline__ int64_t at(int ne, int ds, int v, int e, int j) {
    if (kTogether) return (int64_t)((ds * ne + e) * NF + j) * NV + v;
    if (std::is_same<R, df64>::value) return (int64_t)(ds * NV + v) * (ne * NF) + (e * NF + j);
    return (int64_t)((ds * NV + v) * ne + e) * NF + j;
  }
};

// Layout of the face-flux array: [d][v][e][j], in the FP32 operator [d][e][j][v].
template <int D, int N, typename R>
struct FluxLay {
  __device__ static __forceinline__ int64_t at(int ne, int d, int v, int e, int j) {
    return TraceLay<D, N, R>::at(ne, d, v, e, j);
  }
};

// The traces of one face node.
template <int D, int N, typename R>
__device__ __forceinline__ void load_traces(const typename Arith<R>::S* tr, int ne, int ds, int e, int j,
                                            R (&w)[D + 2]) {
  using Lay = TraceLay<D, N, R>;
  if constexpr (Lay::kTogether && D == 2) {
    const float4 q = __ldg(reinterpret_cast<const float4*>(tr + Lay::at(ne, ds, 0, e, j)));
    w[0] = q.x;
    w[1] = q.y;
    w[2] = q.z;
    w[3] = q.w;
  } else if constexpr (Lay::kTogether) {
    const float* q = tr + Lay::at(ne, ds, 0, e, j);
#pragma unroll
    for (int v = 0; v < D + 2; ++v) w[v] = __ldg(q + v);
  } else {
#pragma unroll
    for (int v = 0; v < D + 2; ++v) w[v] = Arith<R>::load(tr + Lay::at(ne, ds, v, e, j));
  }
}

// The fluxes of one face node (FP32 operator).
template <int D, int N>
__device__ __forceinline__ void load_flux(const float* fl, int ne, int d, int e, int j, float (&f)[D + 2]) {
  const float* p = fl + FluxLay<D, N, float>::at(ne, d, 0, e, j);
  if constexpr (D == 2) {
    const float4 q = __ldg(reinterpret_cast<const float4*>(p));
    f[0] = q.x;
    f[1] = q.y;
    f[2] = q.z;
    f[3] = q.w;
  } else {
#pragma unroll
    for (int v = 0; v < D + 2; ++v) f[v] = __ldg(p + v);
  }
}

// Shared-memory array of the values of all variables at a node in the FP32 operator: four as
// one float4, the fifth (3D) in an array of its own behind the CNT float4.
template <int D, int CNT>
struct NodeArray {
  static constexpr size_t BYTES = (CNT * (sizeof(float4) + (D == 3 ? sizeof(float) : 0)) + 15) / 16 * 16;
  float4* a;
  __device__ explicit NodeArray(unsigned char* p) : a(reinterpret_cast<float4*>(p)) {}
  __device__ __forceinline__ float* b() const { return reinterpret_cast<float*>(a + CNT); }
  __device__ __forceinline__ void store(int i, const float (&f)[D + 2]) const {
    a[i] = make_float4(f[0], f[1], f[2], f[3]);
    if constexpr (D == 3) b()[i] = f[4];
  }
  // variables 2 pair and 2 pair + 1 of node i
  __device__ __forceinline__ float2& pair(int i, int p) const { return reinterpret_cast<float2*>(a)[2 * i + p]; }
  __device__ __forceinline__ void load(int i, float (&f)[D + 2]) const {
    const float4 q = a[i];
    f[0] = q.x;
    f[1] = q.y;
    f[2] = q.z;
    f[3] = q.w;
    if constexpr (D == 3) f[4] = b()[i];
  }
};

// A NodeArray over the nodes of a tile: x-lines of 4 or 8 nodes are padded by one value, so that
// the lines that the lanes of a warp read start in different banks (unpadded a warp's access
// along x takes 4 or 8 passes: 160^2 p=7 48 against 40 us; 2 and 6 nodes take 2 passes, and
// padding them costs more in occupancy: 96^3 p=1 418 against 398 us).
template <int D, int N, int TT>
struct TileNodes : NodeArray<D, Tile<D, N, TT>::THREADS / N * (N + (N % 4 == 0 ? 1 : 0))> {
  static constexpr int PN = N + (N % 4 == 0 ? 1 : 0);
  using NodeArray<D, Tile<D, N, TT>::THREADS / N * PN>::NodeArray;
  __device__ static __forceinline__ int at(int node) { return node + (PN - N) * (node / N); }
};

// Sweep table of the FP32 operator as a kernel argument (each weight twice, for packed
// instructions): entries have compile-time addresses in the constant bank.  The other
// operators read theirs from memory.
template <int D, int N>
struct PackTab {
  float2 q[D][N * N];
};
struct NoTab {};
template <int D, int N, typename R>
using SweepArg = std::conditional_t<std::is_same<R, float>::value, PackTab<D, N>, NoTab>;
template <int D, int N, typename R>
SweepArg<D, N, R> sweep_arg(const VolArgs& a) {
  SweepArg<D, N, R> t;
  if constexpr (std::is_same<R, float>::value) {
    for (int d = 0; d < D; ++d)
      for (int i = 0; i < N * N; ++i) t.q[d][i] = (a.scaled ? a.tab_host->qps : a.tab_host->qp)[d][i];
  }
  return t;
}

// Threads of a volume-kernel block: the FP32 form's line phases stride by whole warps.
template <typename R>
constexpr int vol_block(int threads) {
  return std::is_same<R, float>::value ? (threads + 31) / 32 * 32 : threads;
}

// First value and stride of line r (= el * NF + j) along d of a tile of elements whose x-lines
// take PN values each (PN = N: the nodes as they are; PN > N: padded).
template <int D, int N, int PN>
__device__ __forceinline__ int tile_line(int d, int r, int& st) {
  constexpr int NF = IPow<N, D - 1>::value, NDP = PN * NF;
  st = 1;
  if (d == 0) return r * PN;
  const int el = r / NF, j = r - el * NF;
  const int base = el * NDP + j;
  st = PN;
  if constexpr (D == 3) {
    const int c = j / N;  // j = (a, c): z for d = 1, y for d = 2
    if (d == 1) return base + c * (PN * N - N);
    st = PN * N;
    return base + c * (PN - N);
  } else {
    return base;
  }
}

// FP32 traces of a tile of elements (node i of the tile in x) -> tr: one thread per (direction,
// line) interpolates all variables at both ends of its line, two variables per instruction.
template <int D, int N, int TT>
__device__ __forceinline__ void write_traces_fp32(const MeshArgs& m, const FixedTrace& ft,
                                                  const TileNodes<D, N, TT>& x, int e0,
                                                  float* tr) {
  using T = Tile<D, N, TT>;
  using Nodes = TileNodes<D, N, TT>;
  using Lay = TraceLay<D, N, float>;
  constexpr int NF = T::NF, NV = T::NV, LINES = T::EPB * NF;
  const int ne = (int)m.ne;
  const int last = (ne - e0) * NF;  // lines of the tile's elements inside the mesh
  for (int g = threadIdx.x; g < D * LINES; g += blockDim.x) {
    const int d = g / LINES, r = g - d * LINES;  // r = el * NF + j
    if (r >= last) continue;
    int st;
    const int base = tile_line<D, N, Nodes::PN>(d, r, st);
    float2 lo[D], hi[D];
#pragma unroll
    for (int i = 0; i < D; ++i) lo[i] = hi[i] = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int a = 0; a < N; ++a) {
      const float4 q = x.a[base + a * st];
      const float2 q0 = make_float2(q.x, q.y), q1 = make_float2(q.z, q.w);
      lo[0] = __ffma2_rn(ft.w[0][a], q0, lo[0]);
      lo[1] = __ffma2_rn(ft.w[0][a], q1, lo[1]);
      hi[0] = __ffma2_rn(ft.w[1][a], q0, hi[0]);
      hi[1] = __ffma2_rn(ft.w[1][a], q1, hi[1]);
      if constexpr (D == 3) {
        const float f = x.b()[base + a * st];
        lo[2].x = fmaf(ft.w[0][a].x, f, lo[2].x);
        hi[2].x = fmaf(ft.w[1][a].x, f, hi[2].x);
      }
    }
    float* dst = tr + Lay::at(ne, 2 * d, 0, e0, 0) + r * NV;
    const int side = ne * NF * NV;
    if constexpr (D == 2) {
      *reinterpret_cast<float4*>(dst) = make_float4(lo[0].x, lo[0].y, lo[1].x, lo[1].y);
      *reinterpret_cast<float4*>(dst + side) = make_float4(hi[0].x, hi[0].y, hi[1].x, hi[1].y);
    } else {
#pragma unroll
      for (int o = 0; o < 2; ++o) {
        const float2(&f)[D] = o ? hi : lo;
        dst[o * side] = f[0].x;
        dst[o * side + 1] = f[0].y;
        dst[o * side + 2] = f[1].x;
        dst[o * side + 3] = f[1].y;
        dst[o * side + 4] = f[D - 1].x;
      }
    }
  }
}

// FP64 traces of a tile of elements in shared memory (value (el, v, node) at v * VS + el * ND +
// node) -> tr: one thread per (direction, variable, line) interpolates both ends of
// its line in fixed point (fixline.cuh).
template <int D, int N, int TT>
__device__ __forceinline__ void write_traces_fp64(const MeshArgs& m, const FixedTrace& ft,
                                                  const OpTables* tab, const double* sX, int VS,
                                                  int e0, double* tr) {
  using T = Tile<D, N, TT>;
  constexpr int NF = T::NF, NV = T::NV, EPB = T::EPB, LINES = EPB * NF;
  const int ne = (int)m.ne;
  const int last = (ne - e0) * NF;  // lines of the tile's elements inside the mesh
  for (int g = threadIdx.x; g < D * NV * LINES; g += blockDim.x) {
    const int dv = g / LINES, r = g - dv * LINES;  // r = el * NF + j
    const int d = dv / NV, v = dv - d * NV;
    if (r >= last) continue;
    int st;
    const double* x = sX + v * VS + tile_line<D, N, N>(d, r, st);
    double val[N], lo, hi;
#pragma unroll
    for (int a = 0; a < N; ++a) val[a] = x[a * st];
    line_traces<N>(ft, tab, val, lo, hi);
    double* dst = tr + TraceLay<D, N, double>::at(ne, 2 * d, v, e0, r);
    dst[0] = lo;
    dst[NV * ne * NF] = hi;
  }
}

// Traces of a tile of elements held in shared memory sX[el][v][node] (compute type C, element
// stride SXS) -> tr, FP32-pair operator: a thread owns one (direction, side,
// variable, face node) combination, so its line of nodes, stride and interpolation weights
// are set up once, and interpolates it for a run of the tile's elements (the runs split the
// elements when the block has threads to spare); this halves the instruction count of this
// phase.  (The pair kernels are bound by issue as much as by the FP64 pipe: fixed-point lines
// as in the FP64 operator cost them 15 %.)
template <int D, int N, typename R, int TT, typename C, int SXS>
__device__ __forceinline__ void write_traces(const MeshArgs& m, const OpTables* tab, const C* sX,
                                             int e0, typename Arith<R>::S* tr) {
  using T = Tile<D, N, TT>;
  constexpr int ND = T::ND, NF = T::NF, NV = T::NV, EPB = T::EPB;
  const int ne = (int)m.ne;
  constexpr int CT = 2 * D * NV * NF;                            // combinations
  constexpr int CH = T::THREADS / CT > 0 ? T::THREADS / CT : 1;  // element runs
  constexpr int RUN = (EPB + CH - 1) / CH;                       // elements per run
  for (int g = threadIdx.x; g < CT * CH; g += blockDim.x) {
    const int c = g % CT, ch = g / CT;
    const int j = c % NF, rest = c / NF;  // rest = (d*2 + side)*NV + v
    const int v = rest % NV, ds = rest / NV;
    const int d = ds >> 1, side = ds & 1;
    const int base = line_base<D, N>(d, j);
    const int stride = d == 0 ? 1 : (d == 1 ? N : N * N);
    const double* tw = side ? tab->Tp : tab->Tm;
    const float2* twf = side ? tab->Tpf : tab->Tmf;
    C t[N];
#pragma unroll
    for (int a = 0; a < N; ++a) t[a] = Arith<C>::tab(tw, twf, a);
    const int el0 = ch * RUN;
    const int el1 = el0 + RUN < EPB ? el0 + RUN : EPB;
    typename Arith<R>::S* dst = tr + TraceLay<D, N, R>::at(ne, ds, v, e0, j);
    for (int el = el0; el < el1 && e0 + el < ne; ++el) {
      const C* x = sX + el * SXS + v * ND + base;
      typename Arith<C>::Acc acc = acc_zero(typename Arith<C>::Acc());
#pragma unroll
      for (int a = 0; a < N; ++a) acc = acc_fma(t[a], x[a * stride], acc);
      store_trace(dst + el * NF, acc_result(acc));
    }
  }
}

template <int D, int N, typename R>
__global__ void __launch_bounds__(Tile<D, N>::THREADS) trace_kernel(const TraceArgs A) {
  using T = Tile<D, N>;
  using C = typename TraceCompute<R>::C;
  constexpr int ND = T::ND, NV = T::NV, EPB = T::EPB;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* sX = reinterpret_cast<C*>(smem_raw);
  using Nodes = TileNodes<D, N, 128>;
  const Nodes sN(smem_raw);  // FP32 operator
  const int el = threadIdx.x / ND, node = threadIdx.x - el * ND;
  const int e0 = blockIdx.x * EPB;
  const int e = e0 + el;
  const int ne = (int)A.m.ne;
  if (e < ne) {
    C u[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) u[v] = Arith<C>::from_double(A.u[(v * ne + e) * ND + node]);
    if constexpr (std::is_same<R, float>::value) {
      sN.store(Nodes::at(threadIdx.x), u);
    } else {
#pragma unroll
      for (int v = 0; v < NV; ++v)
        sX[std::is_same<R, double>::value ? v * T::THREADS + (int)threadIdx.x
                                          : (el * NV + v) * ND + node] = u[v];
    }
  }
  __syncthreads();
  typename Arith<R>::S* tr = reinterpret_cast<typename Arith<R>::S*>(A.tr);
  if constexpr (std::is_same<R, double>::value)
    write_traces_fp64<D, N, 128>(A.m, A.ft, A.tab, sX, T::THREADS, e0, tr);
  else if constexpr (std::is_same<R, float>::value)
    write_traces_fp32<D, N, 128>(A.m, A.ft, sN, e0, tr);
  else
    write_traces<D, N, R, 128, C, NV * ND>(A.m, A.tab, sX, e0, tr);
}

// ---- Runge-Kutta update of one node -------------------------------------------------
// Native FP64: everything in FP64.  FP32 / FP32 pair: the RK register and the stage input
// stay in the operator arithmetic; only the accumulation into w is FP64 (one or two DADD).
__device__ __forceinline__ double add_increment(double w0, double d) { return w0 + d; }
__device__ __forceinline__ double add_increment(double w0, float d) { return w0 + f2d_int(d); }
__device__ __forceinline__ double add_increment(double w0, df64 d) {
  return (w0 + f2d_int(d.hi)) + f2d_int(d.lo);
}

// Value of the next stage input handed to the trace interpolation (compute type C): the
// operator's own value, or the FP64 one for the FP32-pair kernels.
template <typename C, typename R>
__device__ __forceinline__ C trace_value(double, R xr) { return xr; }
template <>
__device__ __forceinline__ double trace_value<double, df64>(double xd, df64) { return xd; }

template <typename R>
struct Update {
  using S = typename Arith<R>::S;
  // returns the next stage input at this node/variable; xd receives it in FP64 where the
  // update has it in FP64 (the FP32-pair traces use it)
  // pre: the solution w0 and the 2N register q at this index were staged in advance (pw0,
  // pq) by the volume kernel
  __device__ static __forceinline__ R apply(const VolArgs& A, int idx, R k, R u_in, double& xd,
                                            bool pre = false, double pw0 = 0.0, R pq = R(0.0f)) {
    if (A.mode == kModeRHS) {
      A.kout[idx] = Arith<R>::to_double(k);
      xd = Arith<R>::to_double(u_in);
      return u_in;
    }
    const double w0 = pre ? pw0 : A.w[idx];
    S* x = reinterpret_cast<S*>(A.x);
    if (A.mode == kMode2R) {
      const R cb = Arith<R>::pair(A.cb, A.cbf), ca = Arith<R>::pair(A.ca, A.caf);
      const double w1 = add_increment(w0, cb * k);
      A.w[idx] = w1;
      if (A.last) {
        xd = w1;
        return Arith<R>::from_double(w1);
      }
      const double r1d = add_increment(w0, ca * k);
      const R r1 = Arith<R>::from_double(r1d);
      Arith<R>::store(x + idx, r1);
      xd = r1d;
      return r1;
    }
    const R cA = Arith<R>::pair(A.ca, A.caf), cB = Arith<R>::pair(A.cb, A.cbf);
    const R dtk = A.scaled ? k : Arith<R>::pair(A.dt, A.dtf) * k;
    const R q1 = (A.stage > 0) ? r_fma(cA, pre ? pq : Arith<R>::load(x + idx), dtk) : dtk;
    const double w1 = add_increment(w0, cB * q1);
    A.w[idx] = w1;
    if (!A.last) Arith<R>::store(x + idx, q1);
    xd = w1;
    if constexpr (std::is_same<R, float>::value) {
      // FP32 operator: the next stage input (stage input u_in = w0 in FP32, plus the
      // increment) within an FP32 ulp of float(w1), without a conversion
      return r_fma(cB, q1, u_in);
    } else {
      return Arith<R>::from_double(w1);
    }
  }
};

// FP64: w0 is the solution and q the 2N register at this index.
template <>
struct Update<double> {
  __device__ static __forceinline__ double apply(const VolArgs& A, int idx, double k, double w0,
                                                 double q) {
    if (A.mode == kModeRHS) {
      A.kout[idx] = k;
      return k;
    }
    double* x = reinterpret_cast<double*>(A.x);
    if (A.mode == kMode2R) {
      const double w1 = fma(A.cb, k, w0);
      A.w[idx] = w1;
      if (A.last) return w1;
      const double r1 = fma(A.ca, k, w0);
      x[idx] = r1;
      return r1;
    }
    // (the 2N scheme takes the dt-scaled tables: k is dt times the right-hand side)
    const double q1 = A.stage > 0 ? fma(A.ca, q, k) : k;
    const double w1 = fma(A.cb, q1, w0);
    A.w[idx] = w1;
    if (!A.last) x[idx] = q1;
    return w1;
  }
};

// Pointwise fluxes of a tile in shared memory.  FP32: D NodeArrays of the tile's nodes (then in
// place the contributions of the direction's sweep and lift, then in the first one the next
// stage input).  FP32 pairs: [EPB][D][NV][ND] of R, in 2D pairs of variables
// together for the packed sweeps, [EPB][D][NV/2][ND] of float4 {hi_v, hi_v+1, lo_v, lo_v+1}
// (in 3D the odd variable count and the larger tiles cost more registers than the packing
// saves); the trace epilogue reuses them.
template <int D, typename R> struct PackedSweeps { static constexpr bool value = false; };
template <> struct PackedSweeps<2, df64> { static constexpr bool value = true; };
template <int D, int N, typename R, int TT>
constexpr size_t vol_flux_bytes() {
  using T = Tile<D, N, TT>;
  using C = typename TraceCompute<R>::C;
  if (std::is_same<R, float>::value) return D * TileNodes<D, N, TT>::BYTES;
  const size_t f = PackedSweeps<D, R>::value ? sizeof(float4) * T::EPB * D * ((T::NV + 1) / 2) * T::ND
                                             : sizeof(R) * T::EPB * D * T::NV * T::ND;
  const size_t x = sizeof(C) * T::EPB * T::NV * T::ND;  // reused for the next input
  return f > x ? f : x;
}

// Shared memory of the volume kernel: the pointwise fluxes of the tile, then (kStage) the
// per-thread staging slots of the RK operands (FP64 solution; stage register in the
// operator's storage type), then (kFaces) the numerical fluxes on every face of every
// element of the tile, [EPB][D][side][NV][NF] values of R (FP32: a NodeArray over
// [EPB][D][side][NF]).
template <int D, int N, typename R, int TT, bool kStage, bool kFaces = false>
struct VolSmem {
  using T = Tile<D, N, TT>;
  static constexpr size_t FLUX = (vol_flux_bytes<D, N, R, TT>() + 15) / 16 * 16;
  static constexpr size_t W_OFF = FLUX;
  static constexpr size_t Q_OFF = W_OFF + sizeof(double) * T::NV * T::THREADS;
  static constexpr size_t STAGED =
      kStage ? Q_OFF + sizeof(typename Arith<R>::S) * T::NV * T::THREADS : FLUX;
  static constexpr size_t FACE_OFF = (STAGED + 15) / 16 * 16;
  static constexpr size_t FACES = std::is_same<R, float>::value
                                      ? NodeArray<D, T::EPB * 2 * D * T::NF>::BYTES
                                      : sizeof(R) * T::EPB * 2 * D * T::NV * T::NF;
  static constexpr size_t BYTES = kFaces ? FACE_OFF + FACES : STAGED;
};

// Where the volume kernel takes the numerical fluxes of its elements' faces from.
// SplitFaces: the global flux array the face-flux launch wrote (each face once).
// ElementFaces: every element evaluates the numerical flux on each of its own faces from
// the stored traces of the current stage input (each interior face is then evaluated by
// both of its elements, with the same arguments and code, hence the same bits; ring
// stores come from the face's low element only).  The next stage's traces then go to a
// second trace buffer, since neighbouring blocks still read the current ones.
struct SplitFaces {};
struct ElementFaces {
  const FluxArgs& f;  // face rules of the stage (ring, subdomain slots, AT weights)
  const void* tr;     // traces of the current stage input [d][side][v][e][j]
  int* err;           // set to 2 when a wait for the tile's bulk copies gave up
};

// The FP32 and FP32-pair forms wait on memory more than on their pipes: they stage their
// stage input, solution and 2N register through shared memory with asynchronous copies
// issued at the start, so the reads of the RK update are in flight during the volume work
// instead of after it (512^2 p=4: FP32 210 -> 187 us, pairs 8 % faster).  (FP64:
// vol_body_fp64.)
template <typename R> struct VolStages { static constexpr bool value = false; };
template <> struct VolStages<float> { static constexpr bool value = true; };
template <> struct VolStages<df64> { static constexpr bool value = true; };

// asynchronous copy of one stored value (FP32: 4 bytes, FP32 pair: 8 bytes)
__device__ __forceinline__ void cp_async_val(float* smem, const float* gmem) { cp_async4(smem, gmem); }
__device__ __forceinline__ void cp_async_val(float2* smem, const float2* gmem) { cp_async8(smem, gmem); }
__device__ __forceinline__ float from_stored(float v) { return v; }
__device__ __forceinline__ df64 from_stored(float2 v) { return df64(v.x, v.y); }

// One element tile (tile index `tile`) of the volume/update kernel.  A is read through a
// reference so the batched kernels can pass per-instance arguments kept in device memory.
template <int D, int N, typename R, int TT>
__device__ __forceinline__ void element_face_fluxes(const ElementFaces& F, const MeshArgs& m,
                                                    int e, const int* ec, int el, int node,
                                                    bool active, unsigned char* face_smem);

template <int D, int N, typename R, int TT, bool kStage = false, typename Faces = SplitFaces>
__device__ __forceinline__ void vol_body(const VolArgs& A, const SweepArg<D, N, R>& tab, int tile,
                                         unsigned char* smem_raw, const Faces& faces = Faces()) {
  using T = Tile<D, N, TT>;
  using S = typename Arith<R>::S;
  constexpr bool kFaces = std::is_same<Faces, ElementFaces>::value;
  using SM = VolSmem<D, N, R, TT, kStage, kFaces>;
  // element path with staged operands in 3D: whole tiles are staged by TMA bulk copies (one
  // per variable row, issued by one thread; rows of whole 16-byte units) instead of one
  // asynchronous copy per thread and value (64^3 p=3 FP32: 850 -> 832 us per stage).  In 2D
  // p=4 the rows align only for 16-element tiles, which cost more than the copies save
  // (205 -> 253 us at 512^2).
  constexpr bool kBulk = kFaces && kStage && D == 3 && (Tile<D, N, TT>::THREADS % 4 == 0);
  uint64_t* vbar = nullptr;  // completion barriers of the two copy groups
  if constexpr (kBulk) {
    __shared__ __align__(8) uint64_t bars[2];
    vbar = bars;
  }
  constexpr int ND = T::ND, NF = T::NF, NV = T::NV, EPB = T::EPB;
  constexpr bool kF32 = std::is_same<R, float>::value;
  constexpr int SFS = D * NV * ND, SXS = NV * ND;  // element strides of sF and sX
  using Nodes = TileNodes<D, N, TT>;
  R* sF = reinterpret_cast<R*>(smem_raw);  // [EPB][D][NV][ND] (packed sweeps: sF4 below; FP32: Nodes)
  double* sW = reinterpret_cast<double*>(smem_raw + SM::W_OFF);  // [NV][THREADS] (kStage)
  S* sQ = reinterpret_cast<S*>(smem_raw + SM::Q_OFF);            // [NV][THREADS] (kStage)
  const int el = threadIdx.x / ND, node = threadIdx.x - el * ND;
  const int e0 = tile * EPB;
  const int ne = (int)A.m.ne;
  const int e = e0 + el;
  // (the test of el where the block has no spare threads costs the 3D pairs 6 %: 48^3 p=3 788 ->
  // 835 us)
  const bool active = (vol_block<R>(T::THREADS) == T::THREADS || el < EPB) && e < ne;

  int ix[3] = {node % N, (node / N) % N, node / (N * N)};
  int ec[3] = {0, 0, 0};
  if (active) elem_coords(A.m, e, ec);

  // 1. stage input at this node and its pointwise fluxes
  R u[NV];
  const bool from_r = (A.mode == kMode2R && A.stage > 0);
  const S* rin = reinterpret_cast<const S*>(A.r_in);
  const int tid = threadIdx.x;
  bool bulk = false, group2 = false;  // block-uniform
  if constexpr (kStage) {
    // group 1: the stage input (FP64 solution, or the 2R register r into the q slots);
    // group 2: the solution when the input was r, and the 2N register q
    const bool upd = active && A.mode != kModeRHS;
    const bool want_q = upd && A.mode == kMode2N && A.stage > 0;
    if constexpr (kBulk) bulk = A.bulk && e0 + EPB <= ne;  // a whole tile, aligned rows
    group2 = upd && (from_r || want_q);
    if (bulk) {
      if (tid == 0) {
        mbar_init(vbar, 1);
        mbar_init(vbar + 1, 1);
      }
      __syncthreads();
      if (tid == 0) {
        constexpr unsigned RW = sizeof(double) * T::THREADS, RS = sizeof(S) * T::THREADS;
        const S* xin = reinterpret_cast<const S*>(A.x);
        mbar_expect_tx(vbar, NV * (from_r ? RS : RW));
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const int row = (v * ne + e0) * ND;
          if (from_r) bulk_load(sQ + v * T::THREADS, rin + row, RS, vbar);
          else bulk_load(sW + v * T::THREADS, A.w_in + row, RW, vbar);
        }
        if (group2) {
          mbar_expect_tx(vbar + 1, NV * ((from_r ? RW : 0u) + (want_q ? RS : 0u)));
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            const int row = (v * ne + e0) * ND;
            if (from_r) bulk_load(sW + v * T::THREADS, A.w + row, RW, vbar + 1);
            if (want_q) bulk_load(sQ + v * T::THREADS, xin + row, RS, vbar + 1);
          }
        }
      }
    } else if (active) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const int idx = (v * ne + e) * ND + node;
        if (from_r) cp_async_val(sQ + v * T::THREADS + tid, rin + idx);
        else cp_async8(sW + v * T::THREADS + tid, A.w_in + idx);
      }
    }
    if (!bulk) cp_async_commit();
    if (!bulk && upd && (from_r || want_q)) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const int idx = (v * ne + e) * ND + node;
        if (from_r) cp_async8(sW + v * T::THREADS + tid, A.w + idx);
        if (want_q) cp_async_val(sQ + v * T::THREADS + tid, reinterpret_cast<const S*>(A.x) + idx);
      }
    }
    if (!bulk) cp_async_commit();
    if constexpr (kFaces) element_face_fluxes<D, N, R, TT>(faces, A.m, e, ec, el, node, active, smem_raw + SM::FACE_OFF);
    if (!bulk) {
      cp_async_wait<1>();
    } else if constexpr (kBulk) {
      // a wait that runs out flags the results as invalid and waits once more (bounded)
      // for the copies, so that none is in flight when the block's shared memory is reused
      if (!mbar_wait_bounded(vbar, 0, kWaitLimitCycles)) {
        atomicOr(faces.err, 2);
        mbar_wait_bounded(vbar, 0, kWaitLimitCycles);
      }
    }
#pragma unroll
    for (int v = 0; v < NV; ++v)
      u[v] = !active ? R(1.0f)
                     : (from_r ? from_stored(sQ[v * T::THREADS + tid])
                               : Arith<R>::from_double(sW[v * T::THREADS + tid]));
  } else {
    if constexpr (kFaces) element_face_fluxes<D, N, R, TT>(faces, A.m, e, ec, el, node, active, smem_raw + SM::FACE_OFF);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int idx = (v * ne + e) * ND + node;
      u[v] = !active ? R(1.0f) : (from_r ? Arith<R>::load(rin + idx) : Arith<R>::from_double(A.w_in[idx]));
    }
  }
  constexpr int NP = (NV + 1) / 2;  // variable pairs of the packed sweeps
  float4* sF4 = reinterpret_cast<float4*>(smem_raw);  // [EPB][D][NP][ND] (packed sweeps)
  {
    R F[D][NV];
    euler_flux_all<D, R>(u, Arith<R>::pair(A.gm1, A.gm1f), F);
    if constexpr (kF32) {
      if (active) {
#pragma unroll
        for (int d = 0; d < D; ++d) Nodes(smem_raw + d * Nodes::BYTES).store(Nodes::at(tid), F[d]);
      }
    } else if constexpr (PackedSweeps<D, R>::value) {
#pragma unroll
      for (int d = 0; d < D; ++d)
#pragma unroll
        for (int pr = 0; pr < NP; ++pr) {
          const R f0 = F[d][2 * pr];
          const R f1 = 2 * pr + 1 < NV ? F[d][2 * pr + 1] : R(0.0f);
          sF4[((el * D + d) * NP + pr) * ND + node] = make_float4(f0.hi, f1.hi, f0.lo, f1.lo);
        }
    } else {
#pragma unroll
      for (int d = 0; d < D; ++d)
#pragma unroll
        for (int v = 0; v < NV; ++v) sF[el * SFS + (d * NV + v) * ND + node] = F[d][v];
    }
  }
  __syncthreads();

  // 2. weak derivative (sum factorisation: one 1D contraction per direction) + face lift
  using Acc = typename Arith<R>::Acc;
  Acc acc[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = acc_zero(Acc());
  const S* fl = reinterpret_cast<const S*>(A.fl);
  if constexpr (kF32) {
    // One direction after the other, in place in the first one's NodeArray: one thread per
    // (line, variable pair), the pairs of a line in neighbouring lanes, with the table in the
    // constant bank (one thread per node would read every value N times and its table rows:
    // the shared-memory data pipe, which bounds this kernel, moves about half as much).  The
    // lift follows per node.  Every sum keeps the order of one thread per node (directions,
    // then lifts), and with it its bits.  Us per stage, element path, against that form with
    // one 4-byte access per value and variable: 256^2 p=4 54.6 -> 47.7, 432^2 p=2 67 -> 56,
    // 320^2 p=3 58 -> 43, 160^2 p=7 68 -> 41; 64^3 p=2 474 -> 424, 48^3 p=3 350 -> 289, 32^3
    // p=5 423 -> 329.
    constexpr int LINES = EPB * NF, BLOCK = vol_block<R>(T::THREADS), USED = (2 * LINES + 31) / 32 * 32;
    const int last = (ne - e0) * NF;
    const Nodes Y(smem_raw);
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const Nodes X(smem_raw + d * Nodes::BYTES);
      for (int g = tid; g < 2 * LINES; g += BLOCK) {
        const int r = g >> 1, pr = g & 1;
        if (r >= last) continue;
        int st;
        const int base = tile_line<D, N, Nodes::PN>(d, r, st);
        float2 x[N];
#pragma unroll
        for (int a = 0; a < N; ++a) x[a] = X.pair(base + a * st, pr);
#pragma unroll
        for (int i = 0; i < N; ++i) {
          float2 s = d > 0 ? Y.pair(base + i * st, pr) : make_float2(0.0f, 0.0f);
#pragma unroll
          for (int a = 0; a < N; ++a) s = __ffma2_rn(tab.q[d][i * N + a], x[a], s);
          Y.pair(base + i * st, pr) = s;
        }
      }
      if constexpr (D == 3) {  // the fifth variable, from the warp after the pairs' last one on
        int g = tid - USED % BLOCK;
        if (g < 0) g += BLOCK;
        for (; g < LINES; g += BLOCK) {
          if (g >= last) continue;
          int st;
          const int base = tile_line<D, N, Nodes::PN>(d, g, st);
          float x[N];
#pragma unroll
          for (int a = 0; a < N; ++a) x[a] = X.b()[base + a * st];
#pragma unroll
          for (int i = 0; i < N; ++i) {
            float s = d > 0 ? Y.b()[base + i * st] : 0.0f;
#pragma unroll
            for (int a = 0; a < N; ++a) s = fmaf(tab.q[d][i * N + a].x, x[a], s);
            Y.b()[base + i * st] = s;
          }
        }
      }
      __syncthreads();
    }
    if (active) {
      Y.load(Nodes::at(tid), acc);
      const NodeArray<D, EPB * 2 * D * NF> G(smem_raw + SM::FACE_OFF);  // face fluxes (kFaces)
#pragma unroll
      for (int d = 0; d < D; ++d) {
        const int j = face_index<D, N>(d, ix);
        const float lm = (A.scaled ? A.tab->Lmsf[d] : A.tab->Lmf[d])[ix[d]].x;
        const float lp = (A.scaled ? A.tab->Lpsf[d] : A.tab->Lpf[d])[ix[d]].x;
        float flo[NV], fhi[NV];
        if constexpr (kFaces) {
          G.load((el * 2 * D + 2 * d) * NF + j, flo);
          G.load((el * 2 * D + 2 * d + 1) * NF + j, fhi);
        } else {
          load_flux<D, N>(fl, ne, d, elem_shift(A.m, e, ec, d, -1), j, flo);
          load_flux<D, N>(fl, ne, d, e, j, fhi);
        }
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] = fmaf(-lp, fhi[v], fmaf(lm, flo[v], acc[v]));
      }
    }
  } else if (active) {
    df64acc2 acc2[NP];  // packed sweeps: lane k of pair pr accumulates variable 2 pr + k
#pragma unroll
    for (int pr = 0; pr < NP; ++pr) acc2[pr] = acc2_zero();
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const int stride = d == 0 ? 1 : (d == 1 ? N : N * N);
      const int base = node - ix[d] * stride;
      const double* Qd = (A.scaled ? A.tab->Qs[d] : A.tab->Q[d]) + ix[d] * N;
      const float2* Qdf = (A.scaled ? A.tab->Qsf[d] : A.tab->Qf[d]) + ix[d] * N;
      if constexpr (PackedSweeps<D, R>::value) {
#pragma unroll
        for (int a = 0; a < N; ++a) {
          const float2 q = Qdf[a];
          const float2 qh = make_float2(q.x, q.x), ql = make_float2(q.y, q.y);
          const float2 nqh = make_float2(-q.x, -q.x);
#pragma unroll
          for (int pr = 0; pr < NP; ++pr) {
            const float4 f = sF4[((el * D + d) * NP + pr) * ND + base + a * stride];
            acc2[pr] = acc2_fma(qh, ql, nqh, make_float2(f.x, f.y), make_float2(f.z, f.w), acc2[pr]);
          }
        }
      } else {
#pragma unroll
        for (int a = 0; a < N; ++a) {
          const R q = Arith<R>::tab(Qd, Qdf, a);
#pragma unroll
          for (int v = 0; v < NV; ++v)
            acc[v] = acc_fma(q, sF[el * SFS + (d * NV + v) * ND + base + a * stride], acc[v]);
        }
      }
    }
    if constexpr (PackedSweeps<D, R>::value) {
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] = acc2_lane(acc2[v / 2], v & 1);
    }
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const int j = face_index<D, N>(d, ix);
      const int elo = elem_shift(A.m, e, ec, d, -1);
      const R lp = Arith<R>::tab(A.scaled ? A.tab->Lps[d] : A.tab->Lp[d],
                                 A.scaled ? A.tab->Lpsf[d] : A.tab->Lpf[d], ix[d]);
      const R lm = Arith<R>::tab(A.scaled ? A.tab->Lms[d] : A.tab->Lm[d],
                                 A.scaled ? A.tab->Lmsf[d] : A.tab->Lmf[d], ix[d]);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        R fhi, flo;
        if constexpr (kFaces) {
          const R* sFace = reinterpret_cast<const R*>(smem_raw + SM::FACE_OFF);
          fhi = sFace[(((el * D + d) * 2 + 1) * NV + v) * NF + j];
          flo = sFace[(((el * D + d) * 2 + 0) * NV + v) * NF + j];
        } else {
          fhi = Arith<R>::load(fl + FluxLay<D, N, R>::at(ne, d, v, e, j));
          flo = Arith<R>::load(fl + FluxLay<D, N, R>::at(ne, d, v, elo, j));
        }
        acc[v] = acc_fma(lm, flo, acc[v]);
        acc[v] = acc_fma(-lp, fhi, acc[v]);
      }
    }
  }

  // 3. Runge-Kutta update; xnext = input of the next stage
  using C = typename TraceCompute<R>::C;
  C xnext[NV];
  if constexpr (kStage) {
    if (!bulk) {
      cp_async_wait<0>();
    } else if constexpr (kBulk) {
      if (group2 && !mbar_wait_bounded(vbar + 1, 0, kWaitLimitCycles)) {
        atomicOr(faces.err, 2);
        mbar_wait_bounded(vbar + 1, 0, kWaitLimitCycles);
      }
    }
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const int idx = (v * ne + e) * ND + node;
    double xd = 0.0;
    R xr = R(0.0f);
    if (active) {
      if constexpr (kStage) {
        // from_r (2R, stage > 0) the q slots hold r, which the 2R update does not read
        xr = Update<R>::apply(A, idx, acc_result(acc[v]), u[v], xd, A.mode != kModeRHS,
                              sW[v * T::THREADS + tid], from_stored(sQ[v * T::THREADS + tid]));
      } else {
        xr = Update<R>::apply(A, idx, acc_result(acc[v]), u[v], xd);
      }
    }
    xnext[v] = trace_value<C, R>(xd, xr);
  }

  // 4. traces of the next stage input
  if constexpr (kF32) {
    if (A.write_traces) {
      const Nodes sX(smem_raw);  // over this thread's own values
      if (active) sX.store(Nodes::at(tid), xnext);
      __syncthreads();
      write_traces_fp32<D, N, TT>(A.m, A.ft, sX, e0, reinterpret_cast<float*>(A.tr));
    }
  } else if (A.write_traces) {
    __syncthreads();
    C* sX = reinterpret_cast<C*>(smem_raw);  // reuse: [EPB][NV][ND], element stride SXS
#pragma unroll
    for (int v = 0; v < NV; ++v) sX[el * SXS + v * ND + node] = xnext[v];
    __syncthreads();
    write_traces<D, N, R, TT, C, SXS>(A.m, A.tab, sX, e0, reinterpret_cast<S*>(A.tr));
  }
}

// ---- FP64 volume/update work --------------------------------------------------------

// Limbs of a value in its place.
__device__ __forceinline__ double fixed_bits(double x, int es) {
  const int2 f = fixed_limbs(x, es);
  return __hiloint2double(f.x, f.y);
}
__device__ __forceinline__ int2 fixed_of_bits(double b) {
  return make_int2(__double2hiint(b), __double2loint(b));
}

// Row i of direction d over a line in FP64: k + the sweep over x (a line of nodes with a stride)
// and the lift of its two face fluxes.
template <int N>
__device__ __forceinline__ double chain_line(const OpTables& tab, int scaled, int d, int i, const double* x,
                                             int stride, double lo, double hi, double k) {
  const double* q = (scaled ? tab.Qs[d] : tab.Q[d]) + i * N;
#pragma unroll 1
  for (int a = 0; a < N; ++a) k = fma(q[a], x[a * stride], k);
  k = fma((scaled ? tab.Lms[d] : tab.Lm[d])[i], lo, k);
  return fma(-(scaled ? tab.Lps[d] : tab.Lp[d])[i], hi, k);
}

// Shared memory of the FP64 volume kernel: pointwise fluxes [D][NV][THREADS] and face fluxes
// [EPB][D][side][NV][NF] (as limbs, or FP64 for the FP64 chain), the staged solution and
// Runge-Kutta register [NV][THREADS] (the solution's place then takes the next stage input),
// the fixed-point sweep tables, and the exponents of every line of nodes [D][EPB * NF].
template <int D>
struct __align__(D == 2 ? 8 : 16) LineExp {  // one per variable, two in a word
  unsigned w[D == 2 ? 2 : 4];
};
template <int D, int N, int TT>
struct VolSmem64 {
  using T = Tile<D, N, TT>;
  static constexpr int BLOCK = (T::THREADS + 31) / 32 * 32;  // threads, in whole warps
  static constexpr size_t FACE_OFF = sizeof(double) * D * T::NV * T::THREADS;
  static constexpr size_t W_OFF = FACE_OFF + sizeof(double) * T::EPB * 2 * D * T::NV * T::NF;
  static constexpr size_t Q_OFF = W_OFF + sizeof(double) * T::NV * T::THREADS;
  static constexpr size_t TAB_OFF = Q_OFF + sizeof(double) * T::NV * T::THREADS;
  static constexpr size_t C_OFF = TAB_OFF + sizeof(int2) * D * N * (N + 2);
  static constexpr size_t EXP_OFF = (C_OFF + sizeof(long long) * D * N + 15) / 16 * 16;
  static constexpr size_t BYTES = EXP_OFF + sizeof(LineExp<D>) * D * T::EPB * T::NF;
};

// One element tile of the FP64 volume/update kernel.  Everything the tile reads is copied to
// shared memory asynchronously at the start; one thread per node evaluates the pointwise
// fluxes, one per line of nodes turns them and the face fluxes into fixed point, one per node
// forms the sweeps with the lift (fixline.cuh) and the Runge-Kutta update; one thread per line
// interpolates the traces of the next stage input.
// Bound: the FP64 pipe retires 2 operations per clock and SM, so whatever is a contraction runs
// on the integer pipe (2D p=4: 23 FP64 operations per node instead of 97); the pointwise fluxes
// and the update stay in FP64.  Against chains of FP64 fused multiply-adds: 256^2 p=4 295 -> 117
// us, 320^2 p=3 265 -> 107, 160^2 p=7 349 -> 117, 48^3 p=3 1874 -> 760, 32^3 p=5 2291 -> 880.
// Every line of nodes has an exponent of its own and every direction a table scale of its own,
// as a node's error has to be that of the lines through it.  (One exponent per element and
// variable and one scale for all directions: 48^3 687 us, 256^2 114 us, but a node whose lines
// are 10^-6 of the element's largest value was wrong from the eleventh digit on, and so was the
// flow along the sides of an element 10^6 times as long as wide.)
template <int D, int N, int TT, typename Faces = SplitFaces>
__device__ __forceinline__ void vol_body_fp64(const VolArgs& A, int tile, unsigned char* smem_raw,
                                              const Faces& faces = Faces()) {
  using T = Tile<D, N, TT>;
  constexpr bool kFaces = std::is_same<Faces, ElementFaces>::value;
  using SM = VolSmem64<D, N, TT>;
  constexpr int ND = T::ND, NF = T::NF, NV = T::NV, EPB = T::EPB, M = N + 2;
  constexpr int THREADS = T::THREADS, BLOCK = SM::BLOCK, LINES = EPB * NF;
  const int tid = threadIdx.x;
  double* sF = reinterpret_cast<double*>(smem_raw);
  double* sFace = reinterpret_cast<double*>(smem_raw + SM::FACE_OFF);
  double* sW = reinterpret_cast<double*>(smem_raw + SM::W_OFF) + tid;
  double* sQ = reinterpret_cast<double*>(smem_raw + SM::Q_OFF) + tid;
  int2* sTab = reinterpret_cast<int2*>(smem_raw + SM::TAB_OFF);  // [D][N][M]
  long long* sC = reinterpret_cast<long long*>(smem_raw + SM::C_OFF);  // [D][N]
  LineExp<D>* sExp = reinterpret_cast<LineExp<D>*>(smem_raw + SM::EXP_OFF);  // [D][LINES]
  const int el = tid / ND, node = tid - el * ND;
  const int e0 = tile * EPB;
  const int ne = (int)A.m.ne;
  const int e = e0 + el;
  const bool active = el < EPB && e < ne;
  const FixedSweep* tab = A.scaled ? &A.tab->fxs : &A.tab->fx;

  // copies: stage input (group 1); the register q, or the solution where the input is r, the
  // face fluxes and the tables (group 2)
  const bool from_r = (A.mode == kMode2R && A.stage > 0);
  if (active) {
    const double* in = from_r ? reinterpret_cast<const double*>(A.r_in) : A.w_in;
    const double* in2 = from_r ? A.w
                               : (A.mode == kMode2N && A.stage > 0 ? reinterpret_cast<const double*>(A.x)
                                                                   : nullptr);
#pragma unroll
    for (int v = 0; v < NV; ++v)
      cp_async8((from_r ? sQ : sW) + v * THREADS, in + (v * ne + e) * ND + node);
    cp_async_commit();
    if (in2) {
#pragma unroll
      for (int v = 0; v < NV; ++v)
        cp_async8((from_r ? sW : sQ) + v * THREADS, in2 + (v * ne + e) * ND + node);
    }
    int ec[3];
    elem_coords(A.m, e, ec);
    if constexpr (!kFaces) {
      const double* fl = reinterpret_cast<const double*>(A.fl);
      for (int q = node; q < 2 * D * NF; q += ND) {
        const int ds = q / NF, j = q - ds * NF;
        const int d = ds >> 1;
        const int lo = (ds & 1) ? e : elem_shift(A.m, e, ec, d, -1);
#pragma unroll
        for (int v = 0; v < NV; ++v)
          cp_async8(sFace + ((el * 2 * D + ds) * NV + v) * NF + j, fl + FluxLay<D, N, double>::at(ne, d, v, lo, j));
      }
    } else {
      element_face_fluxes<D, N, double, TT>(faces, A.m, e, ec, el, node, active, smem_raw + SM::FACE_OFF);
    }
  } else {
    cp_async_commit();
  }
  for (int i = tid; i < D * N * M; i += BLOCK) cp_async8(sTab + i, &tab->q[i / (N * M)][i % (N * M)]);
  if (tid < D * N) cp_async8(sC + tid, &tab->c[tid / N][tid % N]);
  cp_async_commit();

  // 1. pointwise fluxes
  cp_async_wait<1>();
  if (active) {
    double F[D][NV], u[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) u[v] = (from_r ? sQ : sW)[v * THREADS];
    euler_flux_all<D, double>(u, A.gm1, F);
#pragma unroll
    for (int d = 0; d < D; ++d)
#pragma unroll
      for (int v = 0; v < NV; ++v) sF[(d * NV + v) * THREADS + tid] = F[d][v];
  }
  cp_async_wait<0>();
  __syncthreads();

  // 2. fixed point, one thread per line of nodes with its two face fluxes: a thread takes the
  // same line of several (direction, variable) pairs.  With an even number of nodes their order
  // does not matter here: where it is a power of two, lines that start in the same bank are
  // walked in different orders (without: 320^2 p=3 114 against 109 us, 160^2 p=7 125 against 116,
  // 48^3 p=3 797 against 783).  Two pairs at a time: 48^3 774 against 775, 40^3 p=4 896 against
  // 906 us; four: 807 and 903.
  {
    constexpr int GROUPS = BLOCK / LINES;
    constexpr bool kPow2 = (N & (N - 1)) == 0;
    const int r = tid % LINES, le = r / NF, j = r - le * NF;  // r = el * NF + j
    FixedScale sc = tab->s[0];
    const int eout[3] = {sc.eout, tab->s[1].eout, tab->s[2].eout};
    if (tid < GROUPS * LINES && e0 + le < ne) {
#pragma unroll 2
      for (int dv = tid / LINES; dv < D * NV; dv += GROUPS) {
        const int d = dv / NV, v = dv - d * NV;
        int st, es;
        const int base = tile_line<D, N, N>(d, r, st);
        const int turn = kPow2 ? ((base >> 4) + (base >> 6)) & (N - 1) : 0;
        double* x = sF + dv * THREADS + base;
        double* f = sFace + ((le * D + d) * 2 * NV + v) * NF + j;
        double val[M];
#pragma unroll
        for (int a = 0; a < N; ++a) val[a] = x[(a ^ turn) * st];
        val[N] = f[0];
        val[N + 1] = f[NV * NF];
        sc.eout = d == 0 ? eout[0] : (d == 1 ? eout[1] : eout[2]);
        const int ex = line_exponent<N>(val, sc, es);
        unsigned short* out = reinterpret_cast<unsigned short*>(sExp[d * LINES + r].w) + v;
        if (D == 3 && v == NV - 1) *reinterpret_cast<unsigned*>(out) = (unsigned)ex;
        else *out = (unsigned short)ex;
        if (ex != kChainLine) {
#pragma unroll
          for (int a = 0; a < N; ++a) x[(a ^ turn) * st] = fixed_bits(val[a], es);
          f[0] = fixed_bits(val[N], es);
          f[NV * NF] = fixed_bits(val[N + 1], es);
        }
      }
    }
  }
  __syncthreads();

  // 3. weak derivative (one contraction per direction) and face lift, Runge-Kutta update
  if (active) {
    const int ix[3] = {node % N, (node / N) % N, node / (N * N)};
    constexpr int NW = (NV + 1) / 2;
    unsigned lx[D][NW], any = 0;  // exponents of the node's lines
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const LineExp<D> q = sExp[d * LINES + el * NF + face_index<D, N>(d, ix)];
#pragma unroll
      for (int w = 0; w < NW; ++w) any |= lx[d][w] = q.w[w];
    }
    auto line_ex = [&](int d, int v) { return (int)((lx[d][v >> 1] >> (16 * (v & 1))) & 0xFFFF); };
    const bool chain = any & (kChainLine * 0x10001u);
    if (!chain) {
      long long sum[NV];
      int ex[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        sum[v] = 0;
        ex[v] = line_ex(0, v);
#pragma unroll
        for (int d = 1; d < D; ++d) ex[v] = max(ex[v], line_ex(d, v));
      }
#pragma unroll
      for (int d = 0; d < D; ++d) {
        const int stride = d == 0 ? 1 : (d == 1 ? N : N * N);
        const double* f = sF + d * NV * THREADS + tid - ix[d] * stride;
        const double* g = sFace + (el * D + d) * 2 * NV * NF + face_index<D, N>(d, ix);
        const int2* q = sTab + (d * N + ix[d]) * M;
        const long long c = sC[d * N + ix[d]];
        FixedAcc acc[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] = FixedAcc{0, c};
#pragma unroll
        for (int a = 0; a < N; ++a) {
          const int2 w = q[a];
#pragma unroll
          for (int v = 0; v < NV; ++v) fixed_fma(w, fixed_of_bits(f[v * THREADS + a * stride]), acc[v]);
        }
#pragma unroll
        for (int side = 0; side < 2; ++side) {
          const int2 w = q[N + side];
#pragma unroll
          for (int v = 0; v < NV; ++v) fixed_fma(w, fixed_of_bits(g[(side * NV + v) * NF]), acc[v]);
        }
#pragma unroll
        for (int v = 0; v < NV; ++v) add_line(acc[v], line_ex(d, v), ex[v], sum[v]);
      }
#pragma unroll
      for (int v = 0; v < NV; ++v)
        sW[v * THREADS] = Update<double>::apply(A, (v * ne + e) * ND + node, line_result(sum[v], ex[v]),
                                                sW[v * THREADS], sQ[v * THREADS]);
    } else {  // line by line
#pragma unroll 1
      for (int v = 0; v < NV; ++v) {
        double k = 0.0;
#pragma unroll
        for (int d = 0; d < D; ++d) {
          const int stride = d == 0 ? 1 : (d == 1 ? N : N * N);
          const double* f = sF + (d * NV + v) * THREADS + tid - ix[d] * stride;
          const double* g = sFace + ((el * D + d) * 2 * NV + v) * NF + face_index<D, N>(d, ix);
          const int ex = reinterpret_cast<const unsigned short*>(
              sExp[d * LINES + el * NF + face_index<D, N>(d, ix)].w)[v];
          if (ex == kChainLine) {
            k = chain_line<N>(*A.tab, A.scaled, d, ix[d], f, stride, g[0], g[NV * NF], k);
          } else {
            const int2* q = sTab + (d * N + ix[d]) * M;
            FixedAcc acc{0, sC[d * N + ix[d]]};
#pragma unroll 1
            for (int a = 0; a < N; ++a) fixed_fma(q[a], fixed_of_bits(f[a * stride]), acc);
            fixed_fma(q[N], fixed_of_bits(g[0]), acc);
            fixed_fma(q[N + 1], fixed_of_bits(g[NV * NF]), acc);
            k += line_result(fixed_sum<kSweepFrac>(acc), ex);
          }
        }
        sW[v * THREADS] = Update<double>::apply(A, (v * ne + e) * ND + node, k, sW[v * THREADS],
                                                sQ[v * THREADS]);
      }
    }
  }

  // 4. traces of the next stage input
  if (A.write_traces) {
    __syncthreads();
    write_traces_fp64<D, N, TT>(A.m, A.ft, A.tab, sW - tid, THREADS, e0,
                                reinterpret_cast<double*>(A.tr));
  }
}

// Register budget of the single-instance volume kernel (an explicit budget also keeps the
// compiler from trading occupancy for registers).  The FP32 form is latency-bound and
// wants every warp slot.
template <int D, int N, typename R> struct VolKernelRegs {
  static constexpr int value = (D == 2 && (N == 2 || N == 8)) ? 64 : 56;  // at most 4 bytes spill (ptxas)
};
template <int D, int N> struct VolKernelRegs<D, N, double> {
  // us at 48, 56, 64 registers: 256^2 p=4 118.0, 117.3, 118.4; 640^2 p=1 151, 143, 141; 160^2 p=7
  // 116, 117, 121.  At 64, 72, 80: 48^3 p=3 783, 774, 759; 64^3 p=2 984, 923, 917; 32^3 p=5 889,
  // 894, 939, but at 56 875.
  static constexpr int value = D == 2 ? 56 : (N == 6 ? 56 : 80);
};
template <int D, int N> struct VolKernelRegs<D, N, float> {
  // 2D: 40 registers are 1 to 4 % slower (N = 8: 1 % faster); 3D: 32 spill (2 to 4 % slower),
  // 48 cost up to 8 %
  static constexpr int value = D == 2 && N != 8 ? 32 : 40;
};

template <int D, int N, typename R, int TT = 128>
__global__ void __launch_bounds__(vol_block<R>(Tile<D, N, TT>::THREADS),
                                  min_blocks_for(VolKernelRegs<D, N, R>::value,
                                                 vol_block<R>(Tile<D, N, TT>::THREADS)))
vol_kernel(const __grid_constant__ VolArgs A, const __grid_constant__ SweepArg<D, N, R> tab) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  grid_dependency();
  vol_body<D, N, R, TT, VolStages<R>::value>(A, tab, blockIdx.x, smem_raw);
}

// (64, 192 and 256 threads: 2 to 25 % slower than 128 over the degrees)
template <int D, int N, int TT = 128>
__global__ void __launch_bounds__(VolSmem64<D, N, TT>::BLOCK,
                                  min_blocks_for(VolKernelRegs<D, N, double>::value,
                                                 VolSmem64<D, N, TT>::BLOCK))
vol_kernel_fp64(const __grid_constant__ VolArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  grid_dependency();
  vol_body_fp64<D, N, TT>(A, blockIdx.x, smem_raw);
}

// Random-delay draw (same definition as the host schedule).
__device__ __forceinline__ uint64_t splitmix64_dev(uint64_t x) {
  uint64_t z = x + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Numerical flux (twice Eq. 8) on face (d, e) -- between element e and its +d neighbour --
// at face node j, from e's trace wm on its +d side and the neighbour's trace wp on its -d
// side.  slot >= 0 marks a face between subdomains (the delayed / AT rules of Algorithms 2-3,
// Eq. 13-14, against the ring of stored levels; stores into the ring at stage 0 of a
// storing step when `owner`).  Shared by the face-flux kernel and the fused kernel, so both
// produce the same bits for the same face.
template <int D, int N, typename R>
__device__ __forceinline__ void face_flux(const FluxArgs& A, int d, int slot, int j,
                                          const R (&wm)[D + 2], const R (&wp)[D + 2], bool owner,
                                          R (&f)[D + 2]) {
  using S = typename Arith<R>::S;
  constexpr int NF = IPow<N, D - 1>::value, NV = D + 2;
  const R gamma = Arith<R>::pair(A.gamma, A.gammaf), gm1 = Arith<R>::pair(A.gm1, A.gm1f);
  if (slot < 0) {
    llf_flux<D, R>(wm, wp, d, gamma, gm1, f);
    return;
  }
  S* ring = reinterpret_cast<S*>(A.ring);
  const bool traces = (A.flux_kind >= 3);  // AT on traces, and the learned mode
  const int npe = (int)A.npe;
  const int lvl_stride = (traces ? 2 : 1) * NV * npe * NF;
  auto at = [=](int v) { return (v * npe + slot) * NF + j; };  // of side and variable v in a level
  int kt = A.uniform_delay;
  if (A.random) {
    const int iface = A.pe_iface[slot];
    const uint64_t ctr = (uint64_t)A.step * (uint64_t)A.n_iface + (uint64_t)iface;
    kt = (int)(splitmix64_dev(A.seed ^ ctr) % (uint64_t)(A.dmax + 1));
    const int64_t need = (A.nterms == 1) ? kt : kt + A.np;
    if (A.step - need < 0) kt = 0;
  }
  if (A.store && traces && owner) {
    S* dst = ring + A.head * lvl_stride;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      Arith<R>::store(dst + at(v), wm[v]);
      Arith<R>::store(dst + at(NV + v), wp[v]);
    }
  }
  if (kt == 0 || (A.store && !traces)) {
    R fr[NV];
    llf_flux<D, R>(wm, wp, d, gamma, gm1, fr);
    if (A.store && !traces && owner) {
      S* dst = ring + A.head * lvl_stride;
#pragma unroll
      for (int v = 0; v < NV; ++v) Arith<R>::store(dst + at(v), fr[v]);
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) f[v] = fr[v];
  }
  if (kt != 0) {
    const int off = A.random ? kt : 0;
    using Acc = typename Arith<R>::Acc;
    Acc am[NV], ap[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) { am[v] = acc_zero(Acc()); ap[v] = acc_zero(Acc()); }
    for (int l = 0; l < A.nterms; ++l) {
      int lvl = (A.head - off - l) % A.depth;
      if (lvl < 0) lvl += A.depth;
      const R c = Arith<R>::pair(A.ctab[kt][l], A.ctabf[kt][l]);
      const S* src = ring + lvl * lvl_stride;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        am[v] = acc_fma(c, Arith<R>::load(src + at(v)), am[v]);
        if (traces) ap[v] = acc_fma(c, Arith<R>::load(src + at(NV + v)), ap[v]);
      }
    }
    if (traces) {
      R em[NV], ep[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) { em[v] = acc_result(am[v]); ep[v] = acc_result(ap[v]); }
      llf_flux<D, R>(em, ep, d, gamma, gm1, f);
    } else {
#pragma unroll
      for (int v = 0; v < NV; ++v) f[v] = acc_result(am[v]);
    }
  }
}

// One block of face-flux threads: block bx over (element, face node) of direction d.
template <int D, int N, typename R>
__device__ __forceinline__ void flux_body(const FluxArgs& A, int bx, int d) {
  using S = typename Arith<R>::S;
  constexpr int NF = IPow<N, D - 1>::value, NV = D + 2;
  const int ne = (int)A.m.ne;
  const int g = bx * blockDim.x + threadIdx.x;
  if (g >= ne * NF) return;
  const int e = g / NF;
  const int j = g - e * NF;
  int ec[3];
  elem_coords(A.m, e, ec);
  const int ehi = elem_shift(A.m, e, ec, d, +1);
  const S* tr = reinterpret_cast<const S*>(A.tr);
  R wm[NV], wp[NV], f[NV];
  load_traces<D, N, R>(tr, ne, d * 2 + 1, e, j, wm);
  load_traces<D, N, R>(tr, ne, d * 2, ehi, j, wp);
  const int slot = A.pe_mode ? A.pe_slot[d * ne + e] : -1;
  face_flux<D, N, R>(A, d, slot, j, wm, wp, true, f);
  S* fl = reinterpret_cast<S*>(A.fl);
  using Lay = FluxLay<D, N, R>;
  if constexpr (TraceLay<D, N, R>::kTogether && D == 2) {
    *reinterpret_cast<float4*>(fl + Lay::at(ne, d, 0, e, j)) = make_float4(f[0], f[1], f[2], f[3]);
  } else {
#pragma unroll
    for (int v = 0; v < NV; ++v) Arith<R>::store(fl + Lay::at(ne, d, v, e, j), f[v]);
  }
}

// Numerical fluxes on the 2D faces of element e (tile slot el) into shared memory
// [el][d][side][v][j]: the thread of node `node` takes the face nodes node, node + ND, ...
// Face (d, lo) lies between element lo and its +d neighbour hi; its flux is evaluated from
// lo's +d trace and hi's -d trace exactly as the face-flux launch evaluates it, so both
// elements of the face obtain the same value.
template <int D, int N, typename R, int TT>
__device__ __forceinline__ void element_face_fluxes(const ElementFaces& F, const MeshArgs& m,
                                                    int e, const int* ec, int el, int node,
                                                    bool active, unsigned char* face_smem) {
  using T = Tile<D, N, TT>;
  using S = typename Arith<R>::S;
  constexpr int ND = T::ND, NF = T::NF, NV = T::NV;
  if (!active) return;
  const int ne = (int)m.ne;
  const S* tr = reinterpret_cast<const S*>(F.tr);
  R* sFace = reinterpret_cast<R*>(face_smem) + el * (2 * D * NV * NF);
  for (int q = node; q < 2 * D * NF; q += ND) {
    const int ds = q / NF, j = q - ds * NF;  // ds = 2 d + side (side 1: the +d face)
    const int d = ds >> 1, side = ds & 1;
    const int nb = elem_shift(m, e, ec, d, side ? 1 : -1);
    const int lo = side ? e : nb, hi = side ? nb : e;
    R wm[NV], wp[NV], f[NV];
    load_traces<D, N, R>(tr, ne, d * 2 + 1, lo, j, wm);
    load_traces<D, N, R>(tr, ne, d * 2, hi, j, wp);
    const int slot = F.f.pe_mode ? F.f.pe_slot[d * ne + lo] : -1;
    face_flux<D, N, R>(F.f, d, slot, j, wm, wp, side == 1, f);
    if constexpr (std::is_same<R, float>::value) {
      NodeArray<D, T::EPB * 2 * D * NF>(face_smem).store((el * 2 * D + ds) * NF + j, f);
    } else {
#pragma unroll
      for (int v = 0; v < NV; ++v) sFace[(ds * NV + v) * NF + j] = f[v];
    }
  }
}

// One launch per RK stage without the face-flux launch: the volume kernel with every
// element evaluating the numerical fluxes on its own faces (ElementFaces).  Register
// budgets: no spills (ptxas sm_103a; FP64 3D p=5: 16 bytes); the FP32 form measured best at 48
// over the degrees (40: up to 30 % slower, 56: 1 to 5 %).
template <int D, int N, typename R> struct VolFacesRegs { static constexpr int value = D == 2 ? 64 : 80; };
template <int D, int N> struct VolFacesRegs<D, N, float> { static constexpr int value = 48; };
template <int D, int N> struct VolFacesRegs<D, N, double> { static constexpr int value = D == 2 ? 72 : 80; };

template <int D, int N, typename R, int TT = 128>
__global__ void __launch_bounds__(vol_block<R>(Tile<D, N, TT>::THREADS),
                                  min_blocks_for(VolFacesRegs<D, N, R>::value,
                                                 vol_block<R>(Tile<D, N, TT>::THREADS)))
vol_faces_kernel(const __grid_constant__ FusedArgs A, const __grid_constant__ SweepArg<D, N, R> tab) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  grid_dependency();
  vol_body<D, N, R, TT, VolStages<R>::value, ElementFaces>(A.v, tab, blockIdx.x, smem_raw,
                                                           ElementFaces{A.f, A.tr_in, A.err});
}

template <int D, int N, int TT = 128>
__global__ void __launch_bounds__(VolSmem64<D, N, TT>::BLOCK,
                                  min_blocks_for(VolFacesRegs<D, N, double>::value,
                                                 VolSmem64<D, N, TT>::BLOCK))
vol_faces_kernel_fp64(const __grid_constant__ FusedArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  grid_dependency();
  vol_body_fp64<D, N, TT, ElementFaces>(A.v, blockIdx.x, smem_raw,
                                        ElementFaces{A.f, A.tr_in, A.err});
}

// Face-flux blocks of 64 threads: a small mesh spreads over more SMs (the FP64 pipe of an SM
// works off one warp per 64 clocks and instruction whatever its lanes hold; 16^2 p=2 17.4 ->
// 14.7 us per stage against 256 threads), and the pair form's last wave is fuller (256^2 p=4
// 29.6 -> 27.3 us, 48^3 p=3 217 -> 203 us).
constexpr int kFluxThreads = 64;
// Register budget of the face-flux kernel (no spills, ptxas sm_103a).
template <int D, typename R> struct FluxKernelRegs { static constexpr int value = D == 2 ? 64 : 72; };
template <int D> struct FluxKernelRegs<D, float> { static constexpr int value = 48; };
template <int D> struct FluxKernelRegs<D, df64> { static constexpr int value = 64; };

// grid: x over (element, face node) of one direction, y = direction d
template <int D, int N, typename R>
__global__ void __launch_bounds__(kFluxThreads, min_blocks_for(FluxKernelRegs<D, R>::value, kFluxThreads))
flux_kernel(const FluxArgs A) {
  grid_dependency();
  flux_body<D, N, R>(A, blockIdx.x, blockIdx.y);
}

// ------------------------------------------------------------------------------------
// Launch helpers instantiated per arithmetic in the kernel translation units.
// ------------------------------------------------------------------------------------
template <int D, int N, typename R>
cudaError_t launch_trace_t(const TraceArgs& a, cudaStream_t s) {
  using T = Tile<D, N>;
  const int64_t blocks = (a.m.ne + T::EPB - 1) / T::EPB;
  const size_t smem = std::is_same<R, float>::value ? TileNodes<D, N, 128>::BYTES
                                                    : sizeof(R) * T::EPB * T::NV * T::ND;
  trace_kernel<D, N, R><<<(unsigned)blocks, T::THREADS, smem, s>>>(a);
  return cudaGetLastError();
}

// Launch that may start while the previous kernel of the stream runs (grid_dependency).
template <typename... A>
cudaError_t launch_dependent(void (*kernel)(A...), unsigned gx, unsigned gy, int threads, size_t smem,
                             cudaStream_t s, const A&... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(gx, gy);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Opt-in for more than 48 KB of dynamic shared memory.
template <typename K>
cudaError_t allow_smem(K kernel, size_t smem) {
  return smem > 48 * 1024 ? cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)smem)
                          : cudaSuccess;
}

template <int D, int N, typename R>
cudaError_t launch_vol_t(const VolArgs& a, cudaStream_t s) {
  constexpr bool k64 = std::is_same<R, double>::value;
  constexpr int TT = 128;
  using T = Tile<D, N, TT>;
  const unsigned blocks = (unsigned)((a.m.ne + T::EPB - 1) / T::EPB);
  cudaError_t err;
  if constexpr (k64) {
    const size_t smem = VolSmem64<D, N, TT>::BYTES;
    if ((err = allow_smem(vol_kernel_fp64<D, N>, smem)) != cudaSuccess) return err;
    return launch_dependent(vol_kernel_fp64<D, N>, blocks, 1, VolSmem64<D, N, TT>::BLOCK, smem, s, a);
  } else {
    const size_t smem = VolSmem<D, N, R, TT, VolStages<R>::value>::BYTES;
    if ((err = allow_smem(vol_kernel<D, N, R>, smem)) != cudaSuccess) return err;
    return launch_dependent(vol_kernel<D, N, R>, blocks, 1, vol_block<R>(T::THREADS), smem, s, a,
                            sweep_arg<D, N, R>(a));
  }
}

template <int D, int N, typename R>
cudaError_t launch_vol_faces_t(const FusedArgs& a, cudaStream_t s) {
  constexpr bool k64 = std::is_same<R, double>::value;
  constexpr int TT = 128;  // tiles of about 128 threads, as on the split path
  using T = Tile<D, N, TT>;
  const unsigned blocks = (unsigned)((a.v.m.ne + T::EPB - 1) / T::EPB);
  cudaError_t err;
  if constexpr (k64) {
    const size_t smem = VolSmem64<D, N, TT>::BYTES;
    if ((err = allow_smem(vol_faces_kernel_fp64<D, N>, smem)) != cudaSuccess) return err;
    return launch_dependent(vol_faces_kernel_fp64<D, N>, blocks, 1, VolSmem64<D, N, TT>::BLOCK, smem, s, a);
  } else {
    const size_t smem = VolSmem<D, N, R, TT, VolStages<R>::value, true>::BYTES;
    if ((err = allow_smem(vol_faces_kernel<D, N, R, TT>, smem)) != cudaSuccess) return err;
    return launch_dependent(vol_faces_kernel<D, N, R, TT>, blocks, 1, vol_block<R>(T::THREADS), smem, s,
                            a, sweep_arg<D, N, R>(a.v));
  }
}

template <int D, int N, typename R>
cudaError_t launch_flux_t(const FluxArgs& a, cudaStream_t s) {
  constexpr int NF = IPow<N, D - 1>::value;
  const int64_t per_dir = a.m.ne * NF;
  return launch_dependent(flux_kernel<D, N, R>, (unsigned)((per_dir + kFluxThreads - 1) / kFluxThreads),
                          D, kFluxThreads, 0, s, a);
}

// Dispatch over (dim, N) for one arithmetic R.
template <typename R>
struct Dispatch {
  static cudaError_t run_trace(int dim, int N, const TraceArgs& a, cudaStream_t s);
  static cudaError_t run_flux(int dim, int N, const FluxArgs& a, cudaStream_t s);
  static cudaError_t run_vol(int dim, int N, const VolArgs& a, cudaStream_t s);
  static cudaError_t run_vol_faces(int dim, int N, const FusedArgs& a, cudaStream_t s);
};

#define ADG_DISPATCH_BODY(FN, ARGS)                                  \
  if (dim == 2) {                                                    \
    switch (N) {                                                     \
      case 2: return FN<2, 2, R>(ARGS, s);                           \
      case 3: return FN<2, 3, R>(ARGS, s);                           \
      case 4: return FN<2, 4, R>(ARGS, s);                           \
      case 5: return FN<2, 5, R>(ARGS, s);                           \
      case 6: return FN<2, 6, R>(ARGS, s);                           \
      case 7: return FN<2, 7, R>(ARGS, s);                           \
      case 8: return FN<2, 8, R>(ARGS, s);                           \
    }                                                                \
  } else if (dim == 3) {                                             \
    switch (N) {                                                     \
      case 2: return FN<3, 2, R>(ARGS, s);                           \
      case 3: return FN<3, 3, R>(ARGS, s);                           \
      case 4: return FN<3, 4, R>(ARGS, s);                           \
      case 5: return FN<3, 5, R>(ARGS, s);                           \
      case 6: return FN<3, 6, R>(ARGS, s);                           \
    }                                                                \
  }                                                                  \
  return cudaErrorInvalidValue;

template <typename R>
cudaError_t Dispatch<R>::run_trace(int dim, int N, const TraceArgs& a, cudaStream_t s) {
  ADG_DISPATCH_BODY(launch_trace_t, a)
}
template <typename R>
cudaError_t Dispatch<R>::run_flux(int dim, int N, const FluxArgs& a, cudaStream_t s) {
  ADG_DISPATCH_BODY(launch_flux_t, a)
}
template <typename R>
cudaError_t Dispatch<R>::run_vol(int dim, int N, const VolArgs& a, cudaStream_t s) {
  ADG_DISPATCH_BODY(launch_vol_t, a)
}
template <typename R>
cudaError_t Dispatch<R>::run_vol_faces(int dim, int N, const FusedArgs& a, cudaStream_t s) {
  ADG_DISPATCH_BODY(launch_vol_faces_t, a)
}

}  // namespace adg
