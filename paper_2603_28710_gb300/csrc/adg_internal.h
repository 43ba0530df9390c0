// Internal declarations shared by the host side and the kernels of the ADG library.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace adg {

constexpr int kMaxN = 8;        // nodes per direction (degree <= 7)
constexpr int kMaxN3D = 6;      // 3D builds degree <= 5
constexpr int kMaxRing = 24;    // ring levels (random_delay_max + np + 1 <= 15 + 7 + 1)
constexpr int kMaxCoefDelay = 16;

// Fixed-point operator tables of the FP64 contractions (fixline.cuh).  eout: exponent of a
// result relative to that of its values; elo, ehi: value exponents the tables cover (none if
// ehi < 0).
struct FixedScale {
  int eout, elo, ehi;
};
constexpr int kFixedValueBits = 61;  // bits of a fixed-point value below its exponent
constexpr int kFixedMinExp = 61;     // smallest value exponent (the lowest bit stays normal)
constexpr int kSweepFrac = 1, kTraceFrac = 2;  // fractional bits that a result keeps
constexpr int fixed_out(int frac) { return 65 - frac; }  // eout plus the table's exponent
constexpr long long fixed_half(int frac) { return 1ll << (30 - frac); }  // half of the last bit kept
struct FixedTrace {  // rows l_a(-1) and l_a(+1), the limbs of an entry side by side
  int2 t[2][kMaxN];
  long long c[2];  // start values of the middle limb sums (fixline.cuh)
  FixedScale s;
  float2 w[2][kMaxN];  // the rows in FP32, each value twice (packed FP32 operator)
};
struct FixedSweep {  // direction d, row i: N flux weights, low-face and high-face weight
  int2 q[3][kMaxN * (kMaxN + 2)];  // entry [i*(N+2) + k]
  long long c[3][kMaxN];           // start value of the middle limb sum per row (fixline.cuh)
  FixedScale s[3];                 // per direction; elo and ehi are the same in all of them
};

// Operator tables in FP64; kernels convert entries to their arithmetic type.
struct OpTables {
  double Q[3][kMaxN * kMaxN];  // (2/h_d) omega_a l_i'(xi_a) / omega_i, entry [i*N + a]
  double Lp[3][kMaxN];         // (1/h_d) l_i(+1) / omega_i: half the lift (the stored
  double Lm[3][kMaxN];         // (1/h_d) l_i(-1) / omega_i   face fluxes are doubled)
  double Tp[kMaxN];            // l_a(+1): trace at the high face
  double Tm[kMaxN];            // l_a(-1): trace at the low face
  double xi[kMaxN];            // Gauss nodes on [-1, 1]
  double wq[kMaxN];            // Gauss weights
  double xe[kMaxN + 1];        // (N+1)-point Gauss nodes for error integrals
  double we[kMaxN + 1];
  double Le[(kMaxN + 1) * kMaxN];  // l_a(xe_p), entry [p*N + a]
  // the same operator tables split into FP32 pairs (hi, lo) for the FP32 and pair kernels
  float2 Qf[3][kMaxN * kMaxN];
  float2 Lpf[3][kMaxN];
  float2 Lmf[3][kMaxN];
  float2 Tpf[kMaxN];
  float2 Tmf[kMaxN];
  // the operator tables times the time step (2N scheme: the volume kernel then produces
  // dt * k directly); filled once dt is known
  double Qs[3][kMaxN * kMaxN];
  double Lps[3][kMaxN];
  double Lms[3][kMaxN];
  float2 Qsf[3][kMaxN * kMaxN];
  float2 Lpsf[3][kMaxN];
  float2 Lmsf[3][kMaxN];
  // the tables (unscaled and dt-scaled) and the trace weights in fixed point
  FixedSweep fx, fxs;
  FixedTrace ft;
  // FP32 sweep tables of the packed FP32 operator: Qf and Qsf in FP32, each value twice
  float2 qp[3][kMaxN * kMaxN];
  float2 qps[3][kMaxN * kMaxN];
};

struct MeshArgs {
  int n[3];
  int64_t ne;
  int64_t es[3];  // element index stride per direction
  // Division by n[0] and n[1] as a 32-bit multiply-high and a shift (division by invariant
  // integers, Granlund & Montgomery, PLDI 1994): with 2^(l-1) < n <= 2^l and
  // M = floor(2^(31+l) / n) + 1 < 2^32, floor(e / n) = (e M) >> (31 + l) for 0 <= e < 2^31
  // (e (M n - 2^(31+l)) <= e 2^l < 2^(31+l)); n = 1 is special-cased.
  uint32_t divm[2], divs[2];
};

// Fills es[], divm[] and divs[] from n[] (host side), n[0], n[1] <= 2^20.
inline void mesh_finish(MeshArgs& m) {
  m.es[0] = 1;
  m.es[1] = m.n[0];
  m.es[2] = (int64_t)m.n[0] * m.n[1];
  for (int i = 0; i < 2; ++i) {
    uint32_t l = 0;
    while (((uint32_t)1 << l) < (uint32_t)m.n[i]) ++l;
    m.divm[i] = l > 0 ? (uint32_t)(((uint64_t)1 << (31 + l)) / (uint64_t)m.n[i] + 1) : 0;
    m.divs[i] = l > 0 ? l - 1 : 0;
  }
}

enum UpdateMode { kModeRHS = 0, kMode2R = 1, kMode2N = 2 };

struct __align__(16) VolArgs {
  MeshArgs m;
  const OpTables* tab;
  double gamma;
  float2 gammaf;   // gamma as an FP32 pair
  double gm1;      // gamma - 1 (every node's pressure needs it)
  float2 gm1f;     // gamma - 1 as an FP32 pair
  int mode;        // UpdateMode
  int stage, last; // stage index; last = 1 on the final stage of a step
  double ca, cb;   // 2R: dt*a_m, dt*b_m ; 2N: A_m, B_m
  double dt;
  float2 caf, cbf, dtf;  // the same coefficients as FP32 pairs
  const double* w_in;    // FP64 stage input when it is the solution (2N, and 2R stage 0)
  const void* r_in;      // 2R stages > 0: the stage register r (operator storage type)
  double* w;             // solution (read + write, FP64)
  void* x;               // 2R: r (written); 2N: q (read + written); operator storage type
  double* kout;          // RHS mode: k = M^-1 L(w_in), FP64
  const void* fl;        // face fluxes [d][v][e][j] (storage type of the arithmetic)
  void* tr;              // traces of the next stage input [d][side][v][e][j]
  int write_traces;
  int scaled;            // 1: use the dt-scaled tables (2N), the accumulator is dt * k
  int bulk;              // 1: n_elem * nodes is a multiple of 4, so the element path may
                         // stage whole tiles by TMA bulk copies (16-byte aligned rows)
  FixedTrace ft;         // trace weights (FP64 and FP32 operators)
  const OpTables* tab_host;  // the tables in host memory: launches of the FP32 operator pass
                             // its sweep rows as a kernel argument
};

struct __align__(16) FluxArgs {
  MeshArgs m;
  double gamma;
  float2 gammaf;
  double gm1;      // gamma - 1 (every face node's pressures need it)
  float2 gm1f;
  const void* tr;
  void* fl;
  // subdomain-face handling
  int pe_mode;          // 0: all faces fresh; 1: apply ring rules on PE faces
  int flux_kind;        // adg_flux
  const int32_t* pe_slot;   // [d][e] -> PE face slot or -1
  const int32_t* pe_iface;  // [slot] -> interface id
  int64_t npe;              // PE faces
  void* ring;               // [level][v][slot][j] (AT_TRACE: [level][2][v][slot][j])
  int depth, head;          // ring depth, level written last (after this stage's store)
  int store;                // write fresh value to ring[head] (stage 0 of a storing step)
  int random;               // per-interface delays (random mode)
  int uniform_delay;        // CAA: 0 on communication steps, k otherwise
  int nterms;               // 1 (standard) or np+1 (AT)
  uint64_t seed;
  int64_t step;
  int n_iface, dmax, np;
  double ctab[kMaxCoefDelay][kMaxN];  // AT weights per delay for this stage
  float2 ctabf[kMaxCoefDelay][kMaxN]; // the same as FP32 pairs
};

// Arguments of the fused per-stage kernel (fused.cuh): one launch per RK stage does the
// face fluxes and the volume/update work of a tile of elements.
struct __align__(16) FusedArgs {
  VolArgs v;           // RK stage: coefficients, tables, w, x (mode 2R or 2N)
  FluxArgs f;          // face rules: gamma, ring, subdomain slots, AT weights of the stage
  const void* tr_in;   // traces of this stage's input, [d][side][v][e][j] (tile-boundary faces)
  void* tr_out;        // traces of the next stage's input on tile-boundary faces
  int ntile[3];        // tiles per direction
  int tma;             // 1: stage the tile by TMA tensor copies; 0: plain loads
  int* err;            // nonzero after a wait gave up (1: the tile's copies never completed)
};

struct TraceArgs {
  MeshArgs m;
  const OpTables* tab;
  const double* u;
  void* tr;
  FixedTrace ft;  // trace weights (FP64 trace arithmetic)
};

// Learned correction of subdomain traces (learned.cu).
struct LearnArgs {
  MeshArgs m;
  double gamma;
  float2 gammaf;
  double gm1;               // gamma - 1, as in the face-flux arguments
  float2 gm1f;
  const void* ring;         // trace ring [level][2][v][slot][j]
  void* fl;                 // face fluxes to overwrite on subdomain faces
  const int32_t* face_d;    // [slot] direction
  const int32_t* face_e;    // [slot] low-side element
  const int32_t* pe_iface;  // [slot] interface (random mode)
  const uint16_t* mlp;      // BF16 parameters
  float trust;              // largest accepted |correction| in units of the level spread
  int64_t npe;
  int depth, head, random, uniform_delay, n_iface, dmax;
  uint64_t seed;
  int64_t step;
  double ctab[kMaxCoefDelay][kMaxN];
  float2 ctabf[kMaxCoefDelay][kMaxN];
  double km[kMaxCoefDelay];  // stage delay k_m = k + c_m of each delay k
  // per-channel work buffers (channel = ((slot * NF + j) * 2 + side) * (dim+2) + var)
  void* E;                  // AT extrapolation (operator storage type)
  double* s;                // AT error estimate E3 - E2 (0: no correction)
  float* x;                 // network inputs [4]
  float* y;                 // network outputs
};
cudaError_t launch_learned(int prec, int dim, int N, const LearnArgs& a, cudaStream_t s);
cudaError_t launch_samples(const double* log, int64_t rec_len, int stages, const int32_t* picks,
                           int n, const double* ctab, const double* kmtab, int kmax, float* x,
                           float* target, int* ok, cudaStream_t s);
cudaError_t launch_log_traces(int prec, int dim, int N, const void* tr, const int32_t* face_d,
                              const int32_t* face_e, const MeshArgs& m, int64_t npe, double* out,
                              cudaStream_t s);

// ADG_PATH_AUTO: whether the element path is the faster one; GB300, us per stage element / split.
// FP32: one launch instead of two up to about 10^6 nodes (35^2 p=4 3.8 / 5.4, 100^2 8.5 / 9.6, 141^2
// 14.2 / 15.3; 20^3 p=1 6.6 / 7.1, 12^3 p=4 11.2 / 12.2); above, the second evaluation of every
// interior face costs more than the launch and the flux array (256^2 p=4 48.0 / 45.6, 640^2 p=1
// 59.9 / 55.7, 64^3 p=2 399 / 358, 40^3 p=4 349 / 332, 32^3 p=5 328 / 307), except with four nodes
// per direction, whose tiles fill their warps in every phase (200^2 p=3 16.5 / 17.8, 320^2 42.7 /
// 45.3, 1024^2 378 / 416, 96^3 2162 / 2203; but 24^3 43.2 / 39.7, 48^3 290 / 285).  FP64 and pairs
// would evaluate every interior face twice on the pipe that bounds them, or in the latency that
// bounds small meshes: FP64 16^2 p=2 12.7 / 10.4, 64^2 16.5 / 12.8, 256^2 p=4 241 / 177, 8^3 p=3 15.2 /
// 13.4; pairs 10.1 / 9.7, 11.1 / 11.0, 173 / 131, 12.5 / 13.1 (only 16^2 p=4 gains more: FP64 9.5 / 10.6,
// pairs 8.7 / 10.1).
inline bool element_path_faster(int prec, int N, int64_t nodes) {
  return prec == 1 && (N == 4 || nodes < ((int64_t)1 << 20));
}

// Launchers (one per arithmetic), implemented in the kernel translation units.
// prec: 0 = FP64, 1 = FP32, 2 = FP32 pair.
cudaError_t launch_trace(int prec, int dim, int N, const TraceArgs& a, cudaStream_t s);
cudaError_t launch_flux(int prec, int dim, int N, const FluxArgs& a, cudaStream_t s);
cudaError_t launch_vol(int prec, int dim, int N, const VolArgs& a, cudaStream_t s);
// Volume kernel with element-local face fluxes (kv_*.cu): a.v the stage (a.v.tr receives
// the next stage's traces), a.f the face rules, a.tr_in the current traces.
cudaError_t launch_vol_faces(int prec, int dim, int N, const FusedArgs& a, cudaStream_t s);
bool kernels_available(int prec, int dim, int N);
// Fused per-stage kernel (kf_*.cu): tile shape of (dim, N) in elements per direction, and
// the launch with the TMA tensor maps of w and of the RK register.
bool fused_tile(int dim, int N, int* tile);
cudaError_t launch_fused(int prec, int dim, int N, const FusedArgs& a, const CUtensorMap& tw,
                         const CUtensorMap& tx, cudaStream_t s);
size_t storage_bytes(int prec);  // bytes per stored trace/flux value

// Auxiliary kernels (FP64), in aux.cu.
cudaError_t launch_init_vortex(int dim, int N, const MeshArgs& m, const double* lo,
                               const double* h, const OpTables* tab, double gamma, double t,
                               double beta, double x0, double y0, double Lx, double Ly,
                               double* u, cudaStream_t s);
cudaError_t launch_init_tgv(int N, const MeshArgs& m, const double* lo, const double* h,
                            const OpTables* tab, double gamma, double mach, double* u,
                            cudaStream_t s);
cudaError_t launch_conservation(int dim, int N, const MeshArgs& m, const OpTables* tab,
                                double J, const double* u, double* partial, double* out,
                                int nblocks, cudaStream_t s);
cudaError_t launch_max_speed(int dim, int N, const MeshArgs& m, double gamma, const double* u,
                             double* partial, double* out, int nblocks, cudaStream_t s);
cudaError_t launch_l2_vortex(int dim, int N, const MeshArgs& m, const double* lo,
                             const double* h, const OpTables* tab, double gamma, double t,
                             double beta, double x0, double y0, double Lx, double Ly,
                             const double* u, double* partial, double* out, int nblocks,
                             cudaStream_t s);
cudaError_t launch_trace_order(const float* src, float* dst, int64_t rows, int NV, int planes,
                               bool by_variable, cudaStream_t s);
cudaError_t launch_check_finite(int64_t n, const double* u, double largest, int* flag, cudaStream_t s);

}  // namespace adg
