// kernels.cuh -- sm_103a kernels of the reactive multi-component LBM step.
//
// Storage: tiles of kTile slots (see Rec).  A tile holds one row of kTile elements per population of
// every lattice, the flow components first, so all populations of a warp's 32 slots lie in one
// contiguous record.  Node n = x + nx*(y + ny*z) sits at slot[n]; the slot map puts the fluid nodes
// first, in list order, so a warp's lanes touch consecutive elements of every row and no cache
// line carries solid-node bytes.  The cells named (n, i) below are row i at slot[n].
// Every lattice keeps ONE copy of its populations and streams in place with the A-A pattern:
//   even steps (parity 0) read f_i(n) from slot (n, i) and write the post-collision f*_i to
//   slot (n, opp i); odd steps (parity 1) read f_i(n) from (n - c_i, opp i) and write f*_i to
//   (n + c_i, i).  A population that meets a wall is written to (n, opp i) at either parity
//   (halfway bounce-back), and read back from (n, i).  Each slot is read and then written by
//   the same thread within a step, so one pass reads and writes every population exactly once.
// After an even number of steps the layout is natural (f_i(n) at (n, i)); after an odd number
// it is swapped.  Every reader of the state (moments, monitors, flips, checkpoints) follows
// the same rule.
//
// The reactive wet-node closure of scalar 0 (Eq. wetnode9) is applied when a node gathers its
// populations: the stored value of a reactive link is the bounce-back value, and the closure
// computes the unknown population from the gathered one moving toward the wall.
//
// Populations are stored as deviations from w_i * ref (ref = 0 in FP64 mode, the configured
// reference density / concentration otherwise), and the collision works on deviations, so
// the large w_i * ref part never enters a difference in reduced precision.  All parameter
// arithmetic is done on the host (Coef<T>): the kernels see only compute-type constants.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cstdint>
#include <type_traits>

#include "lattice.cuh"

namespace lbm {

// ------------------------------------------------------------------ storage

// Populations are loaded with ordinary loads.  The read-only path (__ldg) wants data that does not change while the
// kernel lives, and a step kernel lives from before its predecessor, which writes them, has ended (see pdl_wait).
template <class S>
struct Store;
template <>
struct Store<double> {
  using T = double;
  __device__ static T ld(const double* p) { return *p; }
  __device__ static void st(double* p, T v) { *p = v; }
};
template <>
struct Store<float> {
  using T = float;
  __device__ static T ld(const float* p) { return *p; }
  __device__ static void st(float* p, T v) { *p = v; }
};
template <>
struct Store<__half> {
  using T = float;
  __device__ static T ld(const __half* p) { return __half2float(*p); }
  __device__ static void st(__half* p, T v) { *p = __float2half_rn(v); }
};
template <>
struct Store<__nv_bfloat16> {
  using T = float;
  __device__ static T ld(const __nv_bfloat16* p) { return __bfloat162float(*p); }
  __device__ static void st(__nv_bfloat16* p, T v) { *p = __float2bfloat16_rn(v); }
};

// Mixed storage: 16-bit flow populations with the scalar lattices in FP32.  The tag types are
// the flow's storage element (2 bytes, loaded and stored like the plain 16-bit types); the scalar
// lattices of every storage type S are stored as ScalarOf<S>.
struct half_s32 {
  __half v;
};
struct bf16_s32 {
  __nv_bfloat16 v;
};
template <>
struct Store<half_s32> {
  using T = float;
  __device__ static T ld(const half_s32* p) { return __half2float(p->v); }
  __device__ static void st(half_s32* p, T v) { p->v = __float2half_rn(v); }
};
template <>
struct Store<bf16_s32> {
  using T = float;
  __device__ static T ld(const bf16_s32* p) { return __bfloat162float(p->v); }
  __device__ static void st(bf16_s32* p, T v) { p->v = __float2bfloat16_rn(v); }
};
template <class S>
struct ScalarOf {
  using type = S;
};
template <>
struct ScalarOf<half_s32> {
  using type = float;
};
template <>
struct ScalarOf<bf16_s32> {
  using type = float;
};

// ------------------------------------------------------------- arguments

enum : int { ERR_CAPACITY = 1, ERR_NONFINITE = 2, ERR_CAS = 4, ERR_BOUNDS = 8 };
enum : int { GEO_NONE = 0, GEO_DISSOLVE = 1, GEO_DEPOSIT = 2 };
enum : uint8_t { FL_FLUID = 0, FL_SOLID = 1, FL_REACTIVE = 2, FL_FLIPPING = 3 };

// Floor division by a fixed divisor d through a rounded-up reciprocal (Granlund and Montgomery,
// "Division by invariant integers using multiplication", 1994): with l = ceil(log2 d) and
// M = ceil(2^(31 + l) / d), floor(n / d) = (n * M) >> (31 + l) for every n < 2^31 and
// 1 <= d < 2^31.  The host builds M and the shift and checks them at every quotient boundary.
struct FastDiv {
  uint32_t M;
  int sh;
};
__host__ __device__ __forceinline__ unsigned int fast_div(unsigned int n, FastDiv d) {
  return (unsigned int)(((unsigned long long)n * d.M) >> d.sh);
}

// Everything a kernel needs, in double; kernels convert to their compute type.
struct Args {
  unsigned char* pop;        // every population, in tiles of kTile slots (see Rec): the flow components,
                             // the given scalars, then the reaction product (if any)
  long long pop_bytes;
  void* psi[2];              // compute-type psi per component (Shan-Chen only)
  uint8_t* flags;
  uint32_t* mask;
  double* acc;               // consumed (reactive solid) / deposited (fluid) per node
  uint32_t* fluid_list;       // fluid nodes (sorted at each rebuild, appended by flips): the node index,
                              // with kEdgeBit set where a neighbour may lie across a domain face
  unsigned int* fluid_count;  // [0] list length, [1] length at the last rebuild (see slot)
  // Storage slot of every node.  Each
  // rebuild renumbers the fluid nodes to slots 0 .. F-1 in list order (so list entry e < F has
  // slot e) and the solid nodes to F .. N-1; nodes that become fluid later keep their slot.
  uint32_t* slot;
  uint32_t* slot_new;         // rebuild scratch
  // Byte offset of every node's first cell in pop, plus kOffBias rows (see wall_offsets), for the odd step of the plain
  // kernels: in 32 bits while they hold it (off_ok), else in 64
  uint32_t* off;
  unsigned long long* off64;
  unsigned int* block_counts; // ordered-compaction scratch [chunks + 1]
  unsigned int* block_counts_v;   // the same for the in-domain positions of the fluid-list order
  double* wallx_slot;        // [NBANKS][WALLX_SLOTS] wall-exchange accumulators
  uint32_t* iface_list;       // reactive solids with a fluid scalar-lattice neighbour
  unsigned int* iface_count;
  uint8_t* listed;           // 1 once a node is in iface_list
  uint32_t* flip_list;
  unsigned int* flip_count;
  unsigned int flip_cap;
  double* flip_scratch;      // [flip_cap][5]: new node's mean density (2) and scalars (3)
  double* flip_mon;          // [11] inj_mass[2], inj_spec[3], rem_mass[2], rem_spec[3], solid_rem
  int* err;
  double* inflow_row;        // [3][rows]
  double* outflow_row;       // [3][rows]
  double* partials;          // monitor partial sums [blocks][NMON]
  double* mon_out;           // [NMON]
  double* d_rho;             // FP64 staging [n_comp][N]
  double* d_u;               // [3][N]
  double* d_C;               // [n_scal][N]
  void* snap;                // compute-type residual snapshots [4][pitch] by slot: u_x, u_y, u_z, C
  long long pitch;           // slots (>= N, multiple of 32)
  long long N;
  int nx, ny, nz;
  int n_comp, n_scal;        // n_scal: scalar lattices, the product included
  int product;               // the last scalar lattice is the reaction product (Eq. reactCO2)
  int per[3];                // flow periodicity
  int open_x;                // scalar inlet / outlet on the x faces
  int sc_on, ads_on, shift_forcing, psi_identity;
  int geo_mode, deposit_conservative;
  double tau[2], G[2][2], G_ads[2], psi_wall, rho0, g[3];
  double s_grp[5];           // MRT rates: e, eps, q, pi, m
  double tau_c[3], J0, k_react, C_in[3];
  double V_m, m_s0, DP;
  double rho_ref[2], C_ref[3];
  int bx, by;                // step-kernel block shape
  FastDiv div_x, div_y;      // node index / nx, (node index / nx) / ny
  double u_wall[3];          // velocity of the top plate beyond y = ny - 1
  int moving_wall;           // the top plate moves (closed y axis)
  int flow_open_x;           // flow velocity inlet at x = 0, zero-gradient outlet at x = nx - 1
  double* u_in_row;          // [ny] inlet velocity u_x(y)
  int off_ok;                // 32-bit byte offsets reach all of pop
  int arrhenius;             // scalar 1 is the temperature: rate k(T_b), reaction heat into T
  int n_it;                  // fixed-point iterations of the C_b - T_b coupling per link
  double arr_A, arr_Ta, heat_release;
  // conduction in the solid (with arrhenius): the solid thermal lattice in two compute-type
  // buffers [QC][N] by node (full values); step t reads gs[t & 1] and writes gs[(t + 1) & 1]
  int conjugate;
  unsigned int solid_blocks;   // blocks at the end of a step launch that advance the solid lattice
  double tau_s, c_fs;
  void* gs[2];
  void* kb;                  // compute-type [QC - 1][N]: k(T_b) of the link arriving in
                             // direction j at node n from the last exchange; NaN before one
};

// Fused multiply-add of the compute types.
__device__ __forceinline__ float fmad(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fmad(double a, double b, double c) { return fma(a, b, c); }

// Index guard of the bounds-checked build (-DLBM_BOUNDS_CHECK): an index outside [0, bound)
// sets ERR_BOUNDS and is replaced by 0, so the access stays inside its buffer.  In normal
// builds LBM_CHK is the bare index expression and the generated code is unchanged.
#ifdef LBM_BOUNDS_CHECK
__device__ __forceinline__ long long chk_index(int* err, long long i, long long bound) {
  if (i < 0 || i >= bound) {
    atomicOr(err, ERR_BOUNDS);
    return 0;
  }
  return i;
}
#define LBM_CHK(err, i, bound) chk_index((err), (long long)(i), (long long)(bound))
#else
#define LBM_CHK(err, i, bound) (i)
#endif

// Compute-type constants derived on the host from Args (see make_coef).
template <class T>
struct Coef {
  T om[2];          // 1 / tau
  T hom;            // (1 - 1 / tau) / 2 of component 0 (MRT)
  T oq, omm;        // s_q / 8, s_m / 8: odd D3Q19 MRT groups
  T tau[2];
  T G[2][2], G_ads[2], psi_wall, rho0, g[3];
  T mrt_g[10];      // (s_k - 1/tau) / |R_k|^2 of the MRT rows (one component)
  T omc[3];         // 1 / tau_c
  T wc0, wca;       // scalar weights: rest, axis
  T ics2c;          // 1 / c_s^2 of the scalar lattice
  T icb;            // 1 / (2 w_a + K), K = k tau_c / (tau_c - 1/2): wet-node closure
  T cl1, cl2;       // 4 w_a icb - 1, 2 k icb: closed population and reaction rate per gathered one
  T kr;             // k
  T C_in[3];
  T DP, keep;       // deposition probability, 1 - DP
  T rref[2], cref[3];   // storage references (0 in FP64 mode)
  T fp;             // tau_P / (tau_P - 1/2) of the product lattice
  T uw6[3];         // 6 u_wall = 2 u_wall / c_s^2 of the moving top plate
  T arrA, arrTa;    // temperature-dependent rate A exp(-Ta / T)
  T fc, fT;         // tau / (tau - 1/2) of scalar 0 and of the temperature (scalar 1)
  T hr;             // reaction heat per unit rate
  T oms;            // 1 / tau_s of the solid thermal lattice
  T cfs;            // heat-capacity ratio (rho c_p)_f / (rho c_p)_s
};

constexpr int NMON = 25;
constexpr int WALLX_SLOTS = 4096;
// partial-sum slots
enum : int {
  M_MASS = 0, M_MOM = 2, M_SPEC = 5, M_REACT = 7, M_DEPO = 8, M_IN = 9, M_OUT = 11,
  M_WALLX = 13, M_NSOLID = 14, M_NFLUID = 15, M_NONFIN = 16, M_HEAT = 17,
  M_SPEC2 = 18, M_IN2 = 19, M_OUT2 = 20, M_PROD = 21,  // the third scalar lattice; product gained
  M_TSOLID = 22, M_HEAT_S = 23, M_HEAT_SRC = 24         // conduction in the solid
};
// banks of the wall-exchange accumulators (WALLX_SLOTS doubles each)
enum : int { BANK_WALLX = 0, BANK_HEAT = 1, BANK_PROD = 2, BANK_HEAT_S = 3, BANK_HEAT_SRC = 4, NBANKS = 5 };
// monitor slots of scalar lattice s (0 .. 2)
__host__ __device__ constexpr int mon_spec(int s) { return s < 2 ? M_SPEC + s : M_SPEC2; }
__host__ __device__ constexpr int mon_in(int s) { return s < 2 ? M_IN + s : M_IN2; }
__host__ __device__ constexpr int mon_out(int s) { return s < 2 ? M_OUT + s : M_OUT2; }

// ------------------------------------------------------------- indexing

struct Nbr {
  int n;                              // linear node index
  int oxm, oxp, oym, oyp, ozm, ozp;   // linear offsets to the -/+ neighbours, periodic wrap
  __device__ __forceinline__ int at(int dx, int dy, int dz) const {
    return n + (dx < 0 ? oxm : (dx > 0 ? oxp : 0)) + (dy < 0 ? oym : (dy > 0 ? oyp : 0)) +
           (dz < 0 ? ozm : (dz > 0 ? ozp : 0));
  }
};

__device__ __forceinline__ Nbr make_nbr(const Args& a, int x, int y, int z) {
  Nbr b;
  const int sy = a.nx, sz = a.nx * a.ny;
  b.n = x + sy * y + sz * z;
  // always wrap: walls on closed axes are excluded by the link masks before any access
  b.oxm = x == 0 ? a.nx - 1 : -1;
  b.oxp = x == a.nx - 1 ? 1 - a.nx : 1;
  b.oym = y == 0 ? (a.ny - 1) * sy : -sy;
  b.oyp = y == a.ny - 1 ? (1 - a.ny) * sy : sy;
  b.ozm = z == 0 ? (a.nz - 1) * sz : -sz;
  b.ozp = z == a.nz - 1 ? (1 - a.nz) * sz : sz;
  return b;
}

template <class L>
__device__ __forceinline__ bool flow_wall(uint32_t m, int i) { return (m >> i) & 1u; }

// Fluid-list entries: node index, and a bit for nodes on the faces of the box.  Away from the faces a
// neighbour's index is a constant away, so the coordinates (two divisions) and the periodic wrap
// are worked out for edge nodes only.
constexpr uint32_t kEdgeBit = 0x80000000u;

template <class L>
__device__ __forceinline__ uint32_t list_entry(const Args& a, int n, int x, int y, int z) {
  const bool edge = x == 0 || x == a.nx - 1 || y == 0 || y == a.ny - 1 || (L::D == 3 && (z == 0 || z == a.nz - 1));
  return uint32_t(n) | (edge ? kEdgeBit : 0u);
}
__device__ __forceinline__ int list_node(const Args& a, uint32_t entry) {
  return int(LBM_CHK(a.err, entry & ~kEdgeBit, a.N));
}

// Neighbour offsets of fluid node n from its coordinates (fast divisions by nx and ny).
__device__ __forceinline__ Nbr nbr_of(const Args& a, int n) {
  const unsigned int q = fast_div(unsigned(n), a.div_x);
  const unsigned int z = fast_div(q, a.div_y);
  return make_nbr(a, n - int(q) * a.nx, int(q - z * unsigned(a.ny)), int(z));
}
// the same for a fluid-list entry of node n
__device__ __forceinline__ Nbr nbr_entry(const Args& a, int n, uint32_t entry) {
  if (entry & kEdgeBit) return nbr_of(a, n);
  const int sy = a.nx, sz = a.nx * a.ny;
  return Nbr{n, -1, 1, -sy, sy, -sz, sz};
}

// ------------------------------------------------------------- population tiles

// Record of one tile of kTile slots: NC * Q rows of kTile flow elements, then NS * QC rows of kTile scalar
// elements.  One record is a contiguous stretch (3.3 KB for D3Q19 + D3Q7 in FP32), so an even step
// reads and writes each of a warp's rows from one base address with constant offsets and within
// a few DRAM pages, where planes of the whole domain put every population in a page of its own.
// kTile is 64 for 16-bit flow elements and 32 otherwise: a row is then at least one 128-byte line.  An unaligned run
// of 32 neighbour cells (odd steps) in rows of 32 16-bit elements always crosses into another line, in rows of
// 64 half of the time: 232 x 203 x 181 with FP16 flow and FP32 scalars, odd step 200 us with 32, 188 us with 64.
// FP32 rows of 64 are no faster (256^3, both parities together 638 us each way).
__host__ __device__ constexpr int tile_slots(int elem) { return elem == 2 ? 64 : 32; }
template <class L, class S, int NC, int NS>
struct Rec {
  using SC = typename ScalarOf<S>::type;
  static constexpr int kTile = tile_slots((int)sizeof(S)), kElem = (int)sizeof(S);
  static constexpr int FROW = kTile * (int)sizeof(S), HROW = kTile * (int)sizeof(SC);
  static constexpr int H0 = NC * L::Q * FROW;
  static constexpr int BYTES = H0 + NS * L::QC * HROW;
  static constexpr bool kSameElem = sizeof(S) == sizeof(SC);
  __host__ __device__ static constexpr int frow(int s, int i) { return (s * L::Q + i) * FROW; }
  __host__ __device__ static constexpr int hrow(int s, int j) { return H0 + (s * L::QC + j) * HROW; }
  // byte offset of the first flow cell of a slot, and of its first scalar cell less H0
  __device__ __forceinline__ static long long cell(long long sn) {
    const uint32_t n = uint32_t(sn);   // slots are below 2^31
    return (long long)(n / kTile) * (BYTES - FROW) + (long long)n * (int)sizeof(S);
  }
  template <class O>
  __device__ __forceinline__ static O scell(O c) {
    if (kSameElem) return c;
    return c + ((c / O(sizeof(S))) % O(kTile)) * O(sizeof(SC) - sizeof(S));
  }
  __device__ __forceinline__ static S* f(const Args& a, long long c, int s, int i) {
    return reinterpret_cast<S*>(a.pop + LBM_CHK(a.err, c + frow(s, i), a.pop_bytes));
  }
  __device__ __forceinline__ static SC* h(const Args& a, long long c, int s, int j) {
    return reinterpret_cast<SC*>(a.pop + LBM_CHK(a.err, scell(c) + hrow(s, j), a.pop_bytes));
  }
};

// ------------------------------------------------------------- gathers

// cell offset of node n
template <class R>
__device__ __forceinline__ long long cell_of(const Args& a, long long n) {
  return R::cell((long long)LBM_CHK(a.err, __ldg(a.slot + LBM_CHK(a.err, n, a.N)), a.pitch));
}

// Stored (deviation) values of the pre-collision flow populations of the node whose cells start at
// offset c; neighbour cells come from the slot map.
template <class L, class S, int NC, int NS>
__device__ __forceinline__ void gather_flow(const Args& a, int s, long long c, uint32_t m, const Nbr& nb, int parity,
                                            typename Store<S>::T* out) {
  using R = Rec<L, S, NC, NS>;
  // one branch for all populations, so that their loads are in flight together (the read-back of the 256^3 packing
  // took 448 us with a branch per population, 311 us so)
  if (parity == 0) {
#pragma unroll
    for (int i = 0; i < L::Q; ++i) out[i] = Store<S>::ld(R::f(a, c, s, i));
  } else {
    long long cell[L::Q];
#pragma unroll
    for (int i = 0; i < L::Q; ++i)
      cell[i] = (i == 0 || flow_wall<L>(m, L::opp(i))) ? c + R::frow(s, i)
                                                       : cell_of<R>(a, nb.at(-L::cx(i), -L::cy(i), -L::cz(i))) + R::frow(s, L::opp(i));
#pragma unroll
    for (int i = 0; i < L::Q; ++i) out[i] = Store<S>::ld(reinterpret_cast<const S*>(a.pop + LBM_CHK(a.err, cell[i], a.pop_bytes)));
  }
}

template <class L, class S, int NC, int NS>
__device__ __forceinline__ void gather_scal(const Args& a, int s, long long c, uint32_t m, const Nbr& nb, int parity,
                                            typename Store<S>::T* out) {
  using R = Rec<L, S, NC, NS>;
  using SC = typename R::SC;
  if (parity == 0) {
#pragma unroll
    for (int j = 0; j < L::QC; ++j) out[j] = Store<SC>::ld(R::h(a, c, s, j));
  } else {
    const SC* p[L::QC];
#pragma unroll
    for (int j = 0; j < L::QC; ++j)
      p[j] = (j == 0 || MaskBits<L>::code(m, L::opp(j)) != 0) ? R::h(a, c, s, j)
                                                              : R::h(a, cell_of<R>(a, nb.at(-L::cx(j), -L::cy(j), -L::cz(j))), s, L::opp(j));
#pragma unroll
    for (int j = 0; j < L::QC; ++j) out[j] = Store<SC>::ld(p[j]);
  }
}

template <class T>
__device__ __forceinline__ T scal_w(int j, const Coef<T>& k) { return j == 0 ? k.wc0 : k.wca; }

// Wet-node closure (Eq. wetnode9 per link).  For direction j whose source n - c_j is a
// reactive solid: C_b = 2 hb / (2 w + K), h_j = 2 w C_b - hb, hb = gathered h_{opp j}.
// All closures use the values before closure.  Returns, through the callbacks' arguments,
// the reaction rate k C_b per link and the stored-minus-closed exchange.
// h holds deviations from w_j * cref; the closure works on full values at reactive links.
template <class L, class T, class OnLink>
__device__ __forceinline__ void close_scalar(T* h, uint32_t m, const Coef<T>& k, OnLink on_link) {
  T old[L::QC];
#pragma unroll
  for (int j = 0; j < L::QC; ++j) old[j] = h[j];
  const T sh = k.wca * k.cref[0];
#pragma unroll
  for (int j = 1; j < L::QC; ++j) {
    if (MaskBits<L>::code(m, L::opp(j)) == 2u) {
      const T hb = old[L::opp(j)] + sh;
      const T Cb = T(2) * hb * k.icb;
      const T hn = T(2) * k.wca * Cb - hb - sh;
      h[j] = hn;
      on_link(j, Cb, old[j] - hn);
    }
  }
}

// The same closure with its constants folded (h_j = cl1 hb, rate = cl2 hb), for the step kernels:
// on_link(j, rate, exchange).
template <class L, class T, class OnLink>
__device__ __forceinline__ void close_rate(T* h, uint32_t m, const Coef<T>& k, OnLink on_link) {
  T old[L::QC];
#pragma unroll
  for (int j = 0; j < L::QC; ++j) old[j] = h[j];
  const T sh = k.wca * k.cref[0];
#pragma unroll
  for (int j = 1; j < L::QC; ++j) {
    if (MaskBits<L>::code(m, L::opp(j)) == 2u) {
      const T hb = old[L::opp(j)] + sh;
      h[j] = fmad(k.cl1, hb, -sh);
      on_link(j, k.cl2 * hb, old[j] - h[j]);
    }
  }
}

// Reactive link with a temperature-dependent rate and reaction heat (Sec. 2.1.5, Eq. reactO2,
// reacRate, fluxCon with an adiabatic solid): scalar 0 is the reacting species, scalar 1 the
// temperature.  With hb, gb the gathered species and temperature populations moving toward the
// wall (full values), per link
//   C_b = 2 hb / (2 w + k(T_b) fc),  k(T) = A exp(-Ta / T),  Q = h_r k(T_b) C_b,
//   T_b = (2 gb + Q fT) / (2 w),     fc, fT = tau / (tau - 1/2) of the two scalars,
// solved by n_it fixed-point iterations from the zero-flux value T_b = gb / w; then
//   h_C = 2 w C_b - hb and h_T = gb + Q fT.  All closures of a node read the values before
// any closure.  on_link(j, rate k C_b, species exchange, heat exchange) does the bookkeeping.
template <class L, class T, class OnLink>
__device__ __forceinline__ void close_thermal(T* h0, T* h1, uint32_t m, const Coef<T>& k, int n_it,
                                              OnLink on_link) {
  T old0[L::QC], old1[L::QC];
#pragma unroll
  for (int j = 0; j < L::QC; ++j) {
    old0[j] = h0[j];
    old1[j] = h1[j];
  }
  const T sh0 = k.wca * k.cref[0], sh1 = k.wca * k.cref[1];
  const T w2 = T(2) * k.wca;
#pragma unroll
  for (int j = 1; j < L::QC; ++j) {
    if (MaskBits<L>::code(m, L::opp(j)) == 2u) {
      const T hb = old0[L::opp(j)] + sh0;
      const T gb = old1[L::opp(j)] + sh1;
      T Tb = gb / k.wca;
      for (int it = 0; it < n_it; ++it) {
        const T kt = k.arrA * exp(-k.arrTa / Tb);
        const T Cb = T(2) * hb / (w2 + kt * k.fc);
        const T Q = k.hr * kt * Cb;
        const T was = Tb;
        Tb = (T(2) * gb + Q * k.fT) / w2;
        if (Tb == was) break;   // every further iteration would repeat this one
      }
      const T kt = k.arrA * exp(-k.arrTa / Tb);
      const T Cb = T(2) * hb / (w2 + kt * k.fc);
      const T Q = k.hr * kt * Cb;
      const T hn0 = w2 * Cb - hb - sh0;
      const T hn1 = gb + Q * k.fT - sh1;
      h0[j] = hn0;
      h1[j] = hn1;
      on_link(j, kt * Cb, old0[j] - hn0, hn1 - old1[j]);
    }
  }
}

// Species closure with conduction in the solid (Sec. 2.1.5, Eq. reactO2, reacRate): the wet-node
// closure at each reactive link with the rate constant k(T_b) that the link's last exchange
// (k_exchange) found together with C_b, kept in kb[(j - 1) N + n] for the link arriving in direction
// j.  Before a link's first exchange (NaN entry) k is taken at the heat-capacity-weighted mean
// c_fs T_f + T_s over c_fs + 1 of the node's own temperature T_f and the solid's T_s.  The
// reaction heat entered the temperature through that exchange, so the temperature is not closed
// here.  h0 and h1 hold deviations from w cref; gsrc is the solid lattice the step reads.
template <class L, class T, class OnLink>
__device__ __forceinline__ void close_conjugate(T* h0, const T* h1, uint32_t m, const Coef<T>& k, const Args& a,
                                                const Nbr& nb, const T* gsrc, OnLink on_link) {
  T old[L::QC];
#pragma unroll
  for (int j = 0; j < L::QC; ++j) old[j] = h0[j];
  const T sh0 = k.wca * k.cref[0];
  const T w2 = T(2) * k.wca;
  const T* kb = reinterpret_cast<const T*>(a.kb);
#pragma unroll
  for (int j = 1; j < L::QC; ++j) {
    if (MaskBits<L>::code(m, L::opp(j)) == 2u) {
      T kt = kb[(long long)(j - 1) * a.N + nb.n];
      if (!(kt >= T(0))) {
        const int src = nb.at(-L::cx(j), -L::cy(j), -L::cz(j));
        T Tf = k.cref[1], Ts = T(0);
#pragma unroll
        for (int q = 0; q < L::QC; ++q) {
          Tf += h1[q];
          Ts += gsrc[(long long)q * a.N + src];
        }
        kt = k.arrA * exp(-k.arrTa / ((k.cfs * Tf + Ts) / (k.cfs + T(1))));
      }
      const T hb = old[L::opp(j)] + sh0;
      const T Cb = T(2) * hb / (w2 + kt * k.fc);
      const T hn = w2 * Cb - hb - sh0;
      h0[j] = hn;
      on_link(j, kt * Cb, old[j] - hn);
    }
  }
}

// The reaction product (Sec. 2.1.5, Eq. react, reactCO2): at each reactive link the product lattice
// gains what the reaction takes from scalar 0 there, r = k C_b of that link's closure.  The per-link
// wet-node ansatz of the species closure with the flux reversed, (1 - 1/(2 tau_P)) (h_P,j -
// h_P,opp j) = r, gives h_P,j = h_P,opp j + r tau_P / (tau_P - 1/2).  All closures of a node use the
// values before any closure; hp holds deviations from w C_ref,P on both sides of the link, so the
// shift cancels.  gain accumulates what the closure adds to the populations.
template <class L, class T>
__device__ __forceinline__ void close_product(T* hp, uint32_t m, const Coef<T>& k, const T* rl, T& gain) {
  T old[L::QC];
#pragma unroll
  for (int j = 0; j < L::QC; ++j) old[j] = hp[j];
#pragma unroll
  for (int j = 1; j < L::QC; ++j) {
    if (MaskBits<L>::code(m, L::opp(j)) == 2u) {
      hp[j] = old[L::opp(j)] + rl[j] * k.fp;
      gain += hp[j] - old[j];
    }
  }
}

// ---------------------------------------------------------- equilibria

// f_i^eq - w_i rref, given drho = rho - rref (Eq. 6 written as a deviation)
template <class L, class T>
__device__ __forceinline__ T feq_dev(int i, T rho, T drho, T ux, T uy, T uz) {
  const T cu = T(L::cx(i)) * ux + T(L::cy(i)) * uy + T(L::cz(i)) * uz;
  const T uu = ux * ux + uy * uy + uz * uz;
  return T(L::w(i)) * (drho + rho * (T(3) * cu + T(4.5) * cu * cu - T(1.5) * uu));
}

// -------------------------------------------------------- flip list append

__device__ __forceinline__ void push_flip(const Args& a, int n) {
  const unsigned int k = atomicAdd(a.flip_count, 1u);
  if (k < a.flip_cap)
    a.flip_list[k] = (uint32_t)n;
  else
    atomicOr(a.err, ERR_CAPACITY);
}

// A reactive solid node has consumed its solid mass once V_m acc >= m_s0, i.e. its remaining
// mass m_s0 - V_m acc has reached zero (solid consumption, Sec. 2.1.5).  The product is formed
// in FP64 exactly as written; a node whose V_m acc lies within rounding of m_s0 may flip one
// geometry update earlier or later than in a run that summed its links in another order.
__device__ __forceinline__ bool consumed(const Args& a, double acc) { return a.V_m * acc >= a.m_s0; }

// Exact float -> double widening by re-biasing the IEEE-754 fields with integer operations; the
// conversion instruction itself runs on the FP64 unit, which is narrow on this GPU.  Zero keeps
// its sign; subnormal, infinite and NaN inputs (never produced on the hot path) take the
// conversion instruction.
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ double widen(float v) {
  const unsigned int b = __float_as_uint(v);
  const unsigned int ex = (b >> 23) & 0xffu;
  const unsigned long long sign = (unsigned long long)(b & 0x80000000u) << 32;
  if ((b << 1) == 0u) return __longlong_as_double((long long)sign);
  if (ex == 0u || ex == 0xffu) return double(v);
  return __longlong_as_double((long long)(sign | ((unsigned long long)(ex + (1023u - 127u)) << 52) |
                                          ((unsigned long long)(b & 0x7fffffu) << 29)));
}

// Programmatic dependent launch: the kernels of a time step are launched so that each may start while its
// predecessor still runs.  A kernel lets its successor start at once, reads what no step changes (without
// geometry updates: lists, masks, maps), and waits for the completion of its predecessor before it touches
// anything else.  Every thread waits, so completion still runs in launch order.  What a step changes (populations, psi,
// totals, the solid lattice) is read after the wait and with ordinary loads: the wait makes the predecessor's writes
// visible to those, while the read-only path (__ldg) may only be used for data that is constant from this kernel's
// start to its end, which includes the end of its predecessor: slots, lists, masks.  On a small domain this hides the launch
// and the first dependent loads, which are most of a 4 us kernel.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

template <class T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ================================================================ step

#ifndef LBM_STEP_MIN_BLOCKS
#define LBM_STEP_MIN_BLOCKS 3   // resident 256-thread blocks per SM, one component in FP32 math (80 registers)
#endif
#ifndef LBM_STEP_MIN_BLOCKS_ODD
#define LBM_STEP_MIN_BLOCKS_ODD 3   // k_step's odd parity: the slot prefetch hides the lookups, registers pay
#endif
#ifndef LBM_TILES_MIN_BLOCKS_2D
#define LBM_TILES_MIN_BLOCKS_2D 4   // k_step_tiles in 2D (64 registers; 3 / 4 / 5 blocks: 22.6 / 18.5 / 20.6 us, spills at 5)
#endif
#ifndef LBM_TILES_MIN_BLOCKS_ODD
#define LBM_TILES_MIN_BLOCKS_ODD 3  // k_step_tiles: odd parity, slots prefetched a tile ahead (as k_step)
#endif

// Neighbour cache of the odd step.  An odd step reads cell (n - c_i, opp i) and writes cell
// (n + c_i, i): every neighbour it needs on the way in, it needs again on the way out, and the
// scalar lattices' axis links use the flow lattice's neighbours.  One shared-memory entry per
// direction k (entry k - 1, for the neighbour n + c_k) serves all of them.  The entries are copied
// in asynchronously (cp.async) while the previous node of the thread computes: the offset of the
// neighbour's cells (Args::off) for the plain kernels, its slot for the full ones.
//
// k_step keeps the cache as rows of LBM_STEP_CACHE_STRIDE threads per direction (consecutive
// threads in consecutive words; its blocks have at most that many threads); the ensemble's
// tile kernel gives each thread Q consecutive words of dynamic shared memory instead, sized
// to its block (Q - 1 used; the odd stride puts the threads of a warp on distinct banks).
#define LBM_STEP_CACHE_STRIDE 256
// Asynchronous copies (cp.async, sm_80 and later) of one 4- or 8-byte word from global to shared
// memory; a thread waits for its own groups with cp_async_wait.
template <class E>
__device__ __forceinline__ void cp_async_word(E* smem, const E* gmem) {
  const unsigned int s = (unsigned int)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(s), "l"(gmem), "n"((int)sizeof(E)) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Start copying the map's values of all Q - 1 neighbours n + c_i of a list entry's node into the
// cache.  Links into walls copy a value that is never read (the periodic image is a valid node).
template <class L, int CS, class E>
__device__ __forceinline__ void prefetch_nbrs(const Args& a, const E* map, uint32_t entry, E* cache) {
  const int n = list_node(a, entry);
  const Nbr nb = nbr_entry(a, n, entry);
#pragma unroll
  for (int i = 1; i < L::Q; ++i)
    cp_async_word(cache + (i - 1) * CS, map + LBM_CHK(a.err, nb.at(L::cx(i), L::cy(i), L::cz(i)), a.N));
}

// Offsets in the cache are biased by kOffBias rows.  Flow links into walls read and write the
// node's own cell: (n, i) for the population arriving in direction i, which sits in row i while
// a fluid link's cell sits in row opp(i).  Writing into a wall link's cache entry the own offset moved
// by opp(k) - k rows (at most two rows down, so the biased offset stays positive) lets every flow
// access take row + entry without testing the link.
// The entries are 32-bit byte offsets up to 4 GB of populations (41 M nodes of D3Q19 + D3Q7 in FP32) and 64-bit ones
// beyond (kWide), which cost registers and shared memory: 384^3 FP32, 22.6 M fluid nodes, 1053 us per step, 1050 us
// with 32-bit offsets in flow elements (whose multiply slows the 16-bit ensemble's odd step, 253 -> 266 us) and 1286
// us with slots and tests per link; 448^3 FP16 1439 us and 1704 us; 576^3 FP32 3726 us.
constexpr int kOffBias = 4;

// Variants of the step: plain; full with the boundary rules of a moving plate, a velocity inlet or the
// temperature-dependent reaction; plain with wide offsets (odd steps).  A cache entry is an offset, in the
// full variant a slot.
enum : int { kPlain = 0, kFull = 1, kWide = 2 };
template <int VAR>
struct Entries {
  using type = uint32_t;
  __device__ __forceinline__ static const uint32_t* map(const Args& a) { return VAR == kPlain ? a.off : a.slot; }
};
template <>
struct Entries<kWide> {
  using type = unsigned long long;
  __device__ __forceinline__ static const unsigned long long* map(const Args& a) { return a.off64; }
};

template <class L, class R, int CS, class E>
__device__ __forceinline__ void wall_offsets(long long slot, uint32_t m, E* cache) {
  const uint32_t n = uint32_t(slot);
  const E own = E(n / R::kTile) * E(R::BYTES - R::FROW) + E(n) * E(R::kElem) + E(kOffBias * R::FROW);
#pragma unroll
  for (int k = 1; k < L::Q; ++k)
    if (flow_wall<L>(m, k)) cache[(k - 1) * CS] = own + E((L::opp(k) - k) * R::FROW);
}

// The cells an odd step reads and writes through cache entry k: flow row (s, k) and scalar row (s, k)
// of the neighbour n + c_k, or of the own node behind a wall (rows opp(k)).
template <class L, class S, int NC, int NS, int CS, int VAR>
struct OddCells {
  using R = Rec<L, S, NC, NS>;
  using SC = typename R::SC;
  using E = typename Entries<VAR>::type;
  static constexpr long long kBias = (long long)kOffBias * R::FROW;
  const Args& a;
  long long c;      // the node's own cells
  uint32_t m;
  const E* cache;
  // row at byte `row` of the cells at an entry's offset, and the cells of the slot that an entry names
  __device__ __forceinline__ unsigned char* at(E e, long long row) const {
    return a.pop + LBM_CHK(a.err, (long long)e + (row - kBias), a.pop_bytes);
  }
  __device__ __forceinline__ long long cell(E e) const { return R::cell((long long)LBM_CHK(a.err, e, a.pitch)); }
  __device__ __forceinline__ S* flow(int s, int k) const {
    const E e = cache[(k - 1) * CS];
    if (VAR != kFull) return reinterpret_cast<S*>(at(e, R::frow(s, k)));
    if (flow_wall<L>(m, k)) return R::f(a, c, s, L::opp(k));
    return R::f(a, cell(e), s, k);
  }
  // A scalar link to a fluid neighbour is a fluid flow link and a wall or reactive link a flow wall,
  // so the entry serves both; only an open face (x links) may be a fluid link of a periodic flow.
  __device__ __forceinline__ SC* scal(int s, int k) const {
    const E e = cache[(k - 1) * CS];
    if (VAR != kFull && R::kSameElem) {
      if (L::cx(k) != 0 && MaskBits<L>::code(m, k) == 3u) return R::h(a, c, s, L::opp(k));
      return reinterpret_cast<SC*>(at(e, R::hrow(s, k)));
    }
    if (MaskBits<L>::code(m, k) != 0u) return R::h(a, c, s, L::opp(k));
    if (VAR != kFull) {
      const uint32_t lane = uint32_t(e) / R::kElem % R::kTile;
      return reinterpret_cast<SC*>(at(e, R::hrow(s, k) + lane * (uint32_t)(sizeof(SC) - sizeof(S))));
    }
    return R::h(a, cell(e), s, k);
  }
};

template <class L, class S, int NC, int NS, int CS, int VAR>
__device__ __forceinline__ void gather_odd(const OddCells<L, S, NC, NS, CS, VAR>& o, typename Store<S>::T (&f)[NC][L::Q],
                                           typename Store<S>::T (&h)[NS > 0 ? NS : 1][L::QC]) {
  using R = Rec<L, S, NC, NS>;
#pragma unroll
  for (int s = 0; s < NC; ++s) {
    f[s][0] = Store<S>::ld(R::f(o.a, o.c, s, 0));
#pragma unroll
    for (int i = 1; i < L::Q; ++i) f[s][i] = Store<S>::ld(o.flow(s, L::opp(i)));
  }
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    h[s][0] = Store<typename R::SC>::ld(R::h(o.a, o.c, s, 0));
#pragma unroll
    for (int j = 1; j < L::QC; ++j) h[s][j] = Store<typename R::SC>::ld(o.scal(s, L::opp(j)));
  }
}

template <class L, class S, int NC, int NS>
__device__ __forceinline__ void gather_even(const Args& a, long long c, typename Store<S>::T (&f)[NC][L::Q],
                                            typename Store<S>::T (&h)[NS > 0 ? NS : 1][L::QC]) {
  using R = Rec<L, S, NC, NS>;
#pragma unroll
  for (int s = 0; s < NC; ++s)
#pragma unroll
    for (int i = 0; i < L::Q; ++i) f[s][i] = Store<S>::ld(R::f(a, c, s, i));
#pragma unroll
  for (int s = 0; s < NS; ++s)
#pragma unroll
    for (int j = 0; j < L::QC; ++j) h[s][j] = Store<typename R::SC>::ld(R::h(a, c, s, j));
}

// ------------------------------------------------------------- collision helpers

// MRT correction on top of the BGK update: with n = f - f_eq + F_i / 2 split into pair sums sp
// and differences dp (indexed by the first member of each opposite pair, sp[0] = n_0),
// f_i -= sum_k R_k(c_i) g_k m_k, m_k = sum_i R_k(c_i) n_i, g_k = (s_k - 1/tau) / |R_k|^2.
// Generic form, row by row.
template <class L, class T, class G>
__device__ __forceinline__ void mrt_correct_rows(T* f, const T* sp, const T* dp, const G* g) {
  T coef[L::NMRT];
#pragma unroll
  for (int kk = 0; kk < L::NMRT; ++kk) {
    T mk = T(0);
    if (!mrt_odd<L>(kk)) {
      const int r0 = Mrt<L>::row(kk, 0);
      if (r0 != 0) mk += T(r0) * sp[0];
    }
#pragma unroll
    for (int i = 1; i < L::Q; ++i) {
      if (i > L::opp(i)) continue;
      const int r = Mrt<L>::row(kk, i);
      if (r != 0) mk += T(r) * (mrt_odd<L>(kk) ? dp[i] : sp[i]);
    }
    coef[kk] = T(g[kk]) * mk;
  }
  {
    T c = T(0);
#pragma unroll
    for (int kk = 0; kk < L::NMRT; ++kk) {
      const int r = Mrt<L>::row(kk, 0);
      if (r != 0 && !mrt_odd<L>(kk)) c += T(r) * coef[kk];
    }
    f[0] -= c;
  }
#pragma unroll
  for (int i = 1; i < L::Q; ++i) {
    if (i > L::opp(i)) continue;
    T ce = T(0), co = T(0);
#pragma unroll
    for (int kk = 0; kk < L::NMRT; ++kk) {
      const int r = Mrt<L>::row(kk, i);
      if (r == 0) continue;
      if (mrt_odd<L>(kk)) co += T(r) * coef[kk];
      else ce += T(r) * coef[kk];
    }
    f[i] -= ce + co;
    f[L::opp(i)] -= ce - co;
  }
}

// The collision works on opposite pairs: for the first member i of a pair (i < opp i) f[i] holds
// the sum f_i + f_opp and f[opp i] the difference f_i - f_opp (to_pairs).  Even moments, the
// equilibrium's and the force's even parts touch only sums, odd ones only differences, and the
// post-collision pair is E + O, E - O.
template <class L, class T>
__device__ __forceinline__ void to_pairs(T* f) {
#pragma unroll
  for (int i = 1; i < L::Q; ++i) {
    const int o = L::opp(i);
    if (i > o) continue;
    const T x = f[i], y = f[o];
    f[i] = x + y;
    f[o] = x - y;
  }
}
template <class L, class T>
__device__ __forceinline__ T cdot(int i, T x, T y, T z) {
  T r = T(0);
  bool first = true;
  const int c[3] = {L::cx(i), L::cy(i), L::cz(i)};
  const T v[3] = {x, y, z};
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    if (c[q] == 0) continue;
    if (first) r = c[q] > 0 ? v[q] : -v[q];
    else r = c[q] > 0 ? r + v[q] : r - v[q];
    first = false;
  }
  return r;
}

// BGK of one component on pairs (Eq. 1.16, 1.21), f* = f + om (f_eq - f) + (1 - om/2) F, from its drho, velocity u,
// momentum m = rho u and b = (1 - om/2) F.  The odd part of the equilibrium is 3 w c.m and of the force 3 w c.b, the
// even part of both, the density's share w drho aside, w (4.5 (c.u)(c.e) - 1.5 u.e), e = om m + 2 b.  Velocity-shift
// forcing (Eq. 1.17, 1.18) is the same with b = 0 and its own u.
// Mass and momentum: om multiplies the differences w drho - f and 3 w c.m - f, whose products are not rounded, and
// each pair takes an increment that is zero at equilibrium.  So no factor that is rounded once, the same way at every
// node, acts on mass or momentum: (1 - om) f + om f_eq, two operations less per pair, has two factors that add up to 1
// for some relaxation times only and else changes both by up to 6e-8 of themselves per step in FP32 (32 x 32 box, 2000
// steps, tau 0.9: 1.3e-4 of the mass deviation, 2e-5 this way), and rounded products that drift once a flow is
// uniform (momentum 5e-5, 2e-5 this way).  What is left is the weights' own rounding: 1/18, 1/36 and 1/9 round to
// FP32 within 7e-9 (1/6, 1/12 and 1/3 only within 3e-8, which is why the factor 3 goes to the vector).
template <class L, class T>
__device__ __forceinline__ void bgk_pairs(T* f, T om, T drho, T ux, T uy, T uz, T mx, T my, T mz, T bx, T by, T bz) {
  const T wa = T(L::w(1)), wd = T(L::w(L::Q - 1)), omh = T(0.5) * om;
  const T ex = fmad(om, mx, T(2) * bx), ey = fmad(om, my, T(2) * by), ez = fmad(om, mz, T(2) * bz);
  const T K = T(-1.5) * fmad(ux, ex, fmad(uy, ey, uz * ez));
  f[0] += fmad(om, fmad(T(L::w(0)), drho, -f[0]), T(L::w(0)) * K);
  const T Ka = wa * K, Kd = wd * K;
  const T a45 = T(4.5 * L::w(1)), d45 = T(4.5 * L::w(L::Q - 1));
  const T m3x = T(3) * mx, m3y = T(3) * my, m3z = T(3) * mz, b3x = T(3) * bx, b3y = T(3) * by, b3z = T(3) * bz;
#pragma unroll
  for (int i = 1; i < L::Q; ++i) {
    const int o = L::opp(i);
    if (i > o) continue;
    const bool axis = L::cx(i) * L::cx(i) + L::cy(i) * L::cy(i) + L::cz(i) * L::cz(i) == 1;
    const T w2 = T(2) * (axis ? wa : wd);
    const T cu = axis ? cdot<L>(i, a45 * ux, a45 * uy, a45 * uz) : cdot<L>(i, d45 * ux, d45 * uy, d45 * uz);
    const T Ee = fmad(cu, cdot<L>(i, ex, ey, ez), axis ? Ka : Kd);
    const T Oe = axis ? cdot<L>(i, wa * b3x, wa * b3y, wa * b3z) : cdot<L>(i, wd * b3x, wd * b3y, wd * b3z);
    const T E = fmad(T(0.5), f[i], fmad(omh, fmad(w2, drho, -f[i]), Ee));
    const T O = fmad(T(0.5), f[o], fmad(omh, fmad(w2, cdot<L>(i, m3x, m3y, m3z), -f[o]), Oe));
    f[i] = E + O;
    f[o] = E - O;
  }
}

// MRT with Guo forcing on pairs, generic rows: with G = f_eq - F/2 and H = f_eq + F/2, n = f - G
// relaxes to f* = H + (1 - om) n - sum_k R_k g_k (R_k.n).  rho u = j + F/2 (one component).
template <class L, class T, class K>
__device__ __forceinline__ void mrt_pairs_rows(T* f, const K& k, T drho, T jx, T jy, T jz, T ux, T uy, T uz, T Fx, T Fy,
                                               T Fz) {
  const T ax = fmad(T(-0.5), Fx, jx), ay = fmad(T(-0.5), Fy, jy), az = fmad(T(-0.5), Fz, jz);   // rho u - F
  const T bx = fmad(T(1.5), Fx, jx), by = fmad(T(1.5), Fy, jy), bz = fmad(T(1.5), Fz, jz);      // rho u + F
  const T KG = fmad(T(-1.5), fmad(ux, ax, fmad(uy, ay, uz * az)), drho);
  const T KH = fmad(T(-1.5), fmad(ux, bx, fmad(uy, by, uz * bz)), drho);
  const T hom = k.hom;
  T sp[L::Q], dp[L::Q];
  sp[0] = f[0] - T(L::w(0)) * KG;
  f[0] = fmad(T(2) * hom, sp[0], T(L::w(0)) * KH);
#pragma unroll
  for (int i = 1; i < L::Q; ++i) {
    const int o = L::opp(i);
    if (i > o) continue;
    const T w = T(L::w(i));
    const T cu = T(4.5) * cdot<L>(i, ux, uy, uz);
    const T Ge = w * fmad(cu, cdot<L>(i, ax, ay, az), KG), He = w * fmad(cu, cdot<L>(i, bx, by, bz), KH);
    const T Go = w * cdot<L>(i, T(3) * jx, T(3) * jy, T(3) * jz);
    const T Ho = w * cdot<L>(i, T(3) * (jx + Fx), T(3) * (jy + Fy), T(3) * (jz + Fz));
    sp[i] = fmad(T(-2), Ge, f[i]);
    dp[i] = fmad(T(-2), Go, f[o]);
    const T E = fmad(hom, sp[i], He), O = fmad(hom, dp[i], Ho);
    f[i] = E + O;
    f[o] = E - O;
  }
  mrt_correct_rows<L, T>(f, sp, dp, k.mrt_g);
}

// D3Q19 MRT (rows of d'Humieres et al. 2002) on pairs.  n has no momentum, and the nine odd moments are
// j, q, m, so its odd part is the q and m projections alone: f*_o = f_o + 3 w c.F - s_q, s_m times
// them, with q_x(n) = 5 (j_x / 3 - d_x), m_x(n) = P - R and the row norms 40 and 8.  The momentum stays in
// f_o and is not rebuilt from j with rounded weights.  The even rows are
// evaluated through the sums their polynomials share: axis pairs x, y, z and the diagonal classes.
// About 240 operations in place of 460 for the BGK update of single populations with a correction.
template <class T, class K>
__device__ __forceinline__ void mrt_pairs_d3q19(T* f, const K& k, T drho, T jx, T jy, T jz, T ux, T uy, T uz, T Fx, T Fy,
                                                T Fz) {
  // odd part: row classes of the differences (directions 7 +x+y, 9 +x+z, 11 +y+z, 13 +x-y, 15 +x-z, 17 +y-z)
  const T P = f[8] + f[14], Mxy = f[8] - f[14], R = f[10] + f[16], Mxz = f[10] - f[16], S = f[12] + f[18],
          Myz = f[12] - f[18];
  const T third = T(1.0 / 3.0), sixth = T(1.0 / 6.0), half6 = T(1.0 / 12.0), half = T(0.5);
  const T cqx = k.oq * fmad(third, jx, -f[2]), cqy = k.oq * fmad(third, jy, -f[4]), cqz = k.oq * fmad(third, jz, -f[6]);
  const T cmx = k.omm * (P - R), cmy = k.omm * (S - Mxy), cmz = k.omm * (Mxz - Myz);
  const T Ox = fmad(half, f[2], fmad(T(4), cqx, sixth * Fx)), Oy = fmad(half, f[4], fmad(T(4), cqy, sixth * Fy)),
          Oz = fmad(half, f[6], fmad(T(4), cqz, sixth * Fz));
  const T qx = fmad(half6, Fx, -cqx), qy = fmad(half6, Fy, -cqy), qz = fmad(half6, Fz, -cqz);
  const T u1 = qx - cmx, v1 = qy + cmy;   // pairs 7: u1 + v1, 13: u1 - v1
  const T u2 = qx + cmx, v2 = qz - cmz;   // pairs 9: u2 + v2, 15: u2 - v2
  const T u3 = qy - cmy, v3 = qz + cmz;   // pairs 11: u3 + v3, 17: u3 - v3
  // even part: G and H share u, with a = rho u - F and b = rho u + F
  const T ax = fmad(T(-0.5), Fx, jx), ay = fmad(T(-0.5), Fy, jy), az = fmad(T(-0.5), Fz, jz);
  const T bx = fmad(T(1.5), Fx, jx), by = fmad(T(1.5), Fy, jy), bz = fmad(T(1.5), Fz, jz);
  const T KG = fmad(T(-1.5), fmad(ux, ax, fmad(uy, ay, uz * az)), drho);
  const T KH = fmad(T(-1.5), fmad(ux, bx, fmad(uy, by, uz * bz)), drho);
  const T hom = k.hom;
  const T n0 = fmad(T(-1.0 / 3.0), KG, f[0]);
  // n sums: S - 2 w (KG + 4.5 (c.u)(c.a)), w = 1/18 and 1/36
  const T g9 = T(-1.0 / 9.0) * KG, g18 = T(-1.0 / 18.0) * KG;
  const T px = T(-0.5) * ux, py = T(-0.5) * uy, pz = T(-0.5) * uz;
  const T sx = fmad(px, ax, f[1] + g9), sy = fmad(py, ay, f[3] + g9), sz = fmad(pz, az, f[5] + g9);
  const T rx = T(-0.25) * ux, ry = T(-0.25) * uy, rz = T(-0.25) * uz;
  const T c7 = rx + ry, c13 = rx - ry, c9 = rx + rz, c15 = rx - rz, c11 = ry + rz, c17 = ry - rz;
  const T s7 = fmad(c7, ax + ay, f[7] + g18), s13 = fmad(c13, ax - ay, f[13] + g18);
  const T s9 = fmad(c9, ax + az, f[9] + g18), s15 = fmad(c15, ax - az, f[15] + g18);
  const T s11 = fmad(c11, ay + az, f[11] + g18), s17 = fmad(c17, ay - az, f[17] + g18);
  const T A = sx + sy + sz;
  const T Dxy = s7 + s13, Dxz = s9 + s15, Dyz = s11 + s17, Dx = Dxy + Dxz;
  const T D = Dx + Dyz;
  const T m_e = fmad(T(-30), n0, fmad(T(-11), A, T(8) * D));
  const T m_eps = fmad(T(12), n0, fmad(T(-4), A, D));
  const T m_pxx = fmad(T(-4), sx, fmad(T(2), sy + sz, fmad(T(-2), Dyz, Dx)));
  const T m_pww = fmad(T(2), sz - sy, Dxy - Dxz);
  const T ce = k.mrt_g[0] * m_e, cs = k.mrt_g[1] * m_eps, cpx = k.mrt_g[5] * m_pxx, cpw = k.mrt_g[6] * m_pww;
  f[0] = fmad(T(30), ce, fmad(T(-12), cs, fmad(T(2) * hom, n0, third * KH)));
  // E of a pair = H_e + (1 - om) n_e - (projections)
  const T h18 = T(1.0 / 18.0) * KH, h36 = T(1.0 / 36.0) * KH;
  const T a0 = fmad(T(11), ce, fmad(T(4), cs, h18));
  const T t = fmad(T(-2), cpx, a0);
  const T Ex = fmad(px, T(-0.5) * bx, fmad(hom, sx, fmad(T(4), cpx, a0)));
  const T Ey = fmad(py, T(-0.5) * by, fmad(hom, sy, fmad(T(2), cpw, t)));
  const T Ez = fmad(pz, T(-0.5) * bz, fmad(hom, sz, fmad(T(-2), cpw, t)));
  f[1] = Ex + Ox;
  f[2] = Ex - Ox;
  f[3] = Ey + Oy;
  f[4] = Ey - Oy;
  f[5] = Ez + Oz;
  f[6] = Ez - Oz;
  const T d0 = fmad(T(-8), ce, h36 - cs);
  const T dxy = d0 - (cpx + cpw), dxz = d0 - (cpx - cpw), dyz = fmad(T(2), cpx, d0);
  const T qbx = T(-0.5) * bx, qby = T(-0.5) * by, qbz = T(-0.5) * bz;
  auto pair = [&](int i, T base, T s, T cu, T cb, T uv) {
    const T E = fmad(cu, cb, fmad(hom, s, base)), O = fmad(half, f[i + 1], uv);
    f[i] = E + O;
    f[i + 1] = E - O;
  };
  pair(7, dxy, s7, c7, qbx + qby, u1 + v1);
  pair(13, dxy, s13, c13, qbx - qby, u1 - v1);
  pair(9, dxz, s9, c9, qbx + qbz, u2 + v2);
  pair(15, dxz, s15, c15, qbx - qbz, u2 - v2);
  pair(11, dyz, s11, c11, qby + qbz, u3 + v3);
  pair(17, dyz, s17, c17, qby - qbz, u3 - v3);
}

// Everything after the gather for one fluid node: wet-node closure and its bookkeeping,
// deposition, moments, forces, velocity, flow and scalar collision, in-place scatter.  entry: the
// node's fluid-list entry; c: its cells; o: its odd cells (parity 1).
template <class L, class S, int NC, int NS, int COLL, int parity, int VAR, int CS, class Pre>
__device__ __forceinline__ void collide_scatter(const Args& a, const Coef<typename Store<S>::T>& k, uint32_t entry, int n,
                                                uint32_t m, long long c, const OddCells<L, S, NC, NS, CS, VAR>& o,
                                                typename Store<S>::T (&f)[NC][L::Q],
                                                typename Store<S>::T (&h)[NS > 0 ? NS : 1][L::QC],
                                                typename Store<S>::T& wallx, typename Store<S>::T& heatx,
                                                typename Store<S>::T& prodx, Pre pre) {
  using T = typename Store<S>::T;
  using R = Rec<L, S, NC, NS>;
  using SC = typename R::SC;
  constexpr int Q = L::Q, QC = L::QC;
  constexpr bool BND = VAR == kFull;
  const Nbr nb = nbr_entry(a, n, entry);
  // ---- wet-node closure of scalar 0 and reaction bookkeeping (Eq. wetnode9, reactO2)
  if (NS > 0) {
    // the consumed totals are reductions (no value returned): the threshold test runs in
    // k_detect over the interface list before the geometry update; rl keeps each link's rate
    // for the product lattice's closure
    T rl[QC];
#pragma unroll
    for (int j = 0; j < QC; ++j) rl[j] = T(0);
    const auto solid_of = [&](int j) { return LBM_CHK(a.err, nb.at(-L::cx(j), -L::cy(j), -L::cz(j)), a.N); };
    if (BND && NS > 1 && a.conjugate) {
      // conduction in the solid: the rate constant of the link's last exchange
      close_conjugate<L, T>(h[0], h[NS > 1 ? 1 : 0], m, k, a, nb,
                            reinterpret_cast<const T*>(a.gs[parity]), [&](int j, T r, T exch) {
        atomicAdd(a.acc + solid_of(j), widen(r));
        wallx += exch;
        rl[j] = r;
      });
    } else if (BND && NS > 1 && a.arrhenius) {
      // temperature-dependent rate and reaction heat (the full kernel variant only)
      close_thermal<L, T>(h[0], h[NS > 1 ? 1 : 0], m, k, a.n_it, [&](int j, T r, T exch, T heat) {
        atomicAdd(a.acc + solid_of(j), widen(r));
        wallx += exch;
        heatx += heat;
        rl[j] = r;
      });
    } else if (MaskBits<L>::reactive(m) != 0u) {
      close_rate<L, T>(h[0], m, k, [&](int j, T r, T exch) {
        atomicAdd(a.acc + solid_of(j), widen(r));
        wallx += exch;
        rl[j] = r;
      });
    }
    if (NS > 1 && a.product) close_product<L, T>(h[NS - 1], m, k, rl, prodx);
    // ---- deposition at near-substrate nodes (Eq. surface_deposition)
    if (a.geo_mode == GEO_DEPOSIT) {
      bool near = false;
#pragma unroll
      for (int j = 1; j < QC; ++j) {
        const uint32_t c = MaskBits<L>::code(m, j);
        near |= (c == 1u || c == 2u);
      }
      if (near) {
        T sum = k.cref[0];
#pragma unroll
        for (int j = 0; j < QC; ++j) sum += h[0][j];
        const double dep = double(k.DP * sum);
        const double old = a.acc[n];
        a.acc[n] = old + dep;
        if (old <= 1.0 && old + dep > 1.0) push_flip(a, n);
        if (a.deposit_conservative) {
#pragma unroll
          for (int j = 0; j < QC; ++j) h[0][j] = h[0][j] * k.keep - scal_w<T>(j, k) * k.cref[0] * k.DP;
        }
      }
    }
  }
  // ---- moments (Eq. 1.7, 1.8): rho = rref + sum of deviations, from pair sums and differences
  T drho[NC], rho[NC], jx[NC], jy[NC], jz[NC];
#pragma unroll
  for (int s = 0; s < NC; ++s) {
    to_pairs<L, T>(f[s]);
    T r = f[s][0], ax = T(0), ay = T(0), az = T(0);
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      if (i > L::opp(i)) continue;
      const T d = f[s][L::opp(i)];
      r += f[s][i];
      if (L::cx(i)) ax += T(L::cx(i)) * d;
      if (L::cy(i)) ay += T(L::cy(i)) * d;
      if (L::cz(i)) az += T(L::cz(i)) * d;
    }
    drho[s] = r;
    rho[s] = k.rref[s] + r;
    jx[s] = ax; jy[s] = ay; jz[s] = az;
  }
  // ---- forces: Shan-Chen cohesion / solid psi (Eq. 1.13, 1.14), adhesion (1.15), body
  T Fx[NC], Fy[NC], Fz[NC];
#pragma unroll
  for (int s = 0; s < NC; ++s) {
    Fx[s] = rho[s] * k.g[0];
    Fy[s] = rho[s] * k.g[1];
    Fz[s] = rho[s] * k.g[2];
  }
  if (a.sc_on) {
    T sx[NC], sy[NC], sz[NC];
#pragma unroll
    for (int s2 = 0; s2 < NC; ++s2) {
      const T* ps = reinterpret_cast<const T*>(a.psi[s2]);
      T ax = T(0), ay = T(0), az = T(0);
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        const T pv = flow_wall<L>(m, i) ? k.psi_wall : ps[nb.at(L::cx(i), L::cy(i), L::cz(i))];
        const T wp = T(L::w(i)) * pv;
        if (L::cx(i)) ax += T(L::cx(i)) * wp;
        if (L::cy(i)) ay += T(L::cy(i)) * wp;
        if (L::cz(i)) az += T(L::cz(i)) * wp;
      }
      sx[s2] = ax; sy[s2] = ay; sz[s2] = az;
    }
#pragma unroll
    for (int s = 0; s < NC; ++s) {
      const T pself = reinterpret_cast<const T*>(a.psi[s])[n];
#pragma unroll
      for (int s2 = 0; s2 < NC; ++s2) {
        const T Gss = k.G[s][s2];
        Fx[s] -= pself * Gss * sx[s2];
        Fy[s] -= pself * Gss * sy[s2];
        Fz[s] -= pself * Gss * sz[s2];
      }
    }
  }
  if (a.ads_on) {
    T ax = T(0), ay = T(0), az = T(0);
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      if (flow_wall<L>(m, i)) {
        ax += T(L::w(i)) * T(L::cx(i));
        ay += T(L::w(i)) * T(L::cy(i));
        az += T(L::w(i)) * T(L::cz(i));
      }
    }
#pragma unroll
    for (int s = 0; s < NC; ++s) {
      const T ga = k.G_ads[s] * rho[s];
      Fx[s] -= ga * ax; Fy[s] -= ga * ay; Fz[s] -= ga * az;
    }
  }
  // ---- physical / barycentric velocity (Eq. 1.19, 1.20)
  T rt = T(0), mx = T(0), my = T(0), mz = T(0);
#pragma unroll
  for (int s = 0; s < NC; ++s) {
    rt += rho[s];
    mx += jx[s] + T(0.5) * Fx[s];
    my += jy[s] + T(0.5) * Fy[s];
    mz += jz[s] + T(0.5) * Fz[s];
  }
  const T irt = T(1) / rt;
  const T ux = mx * irt, uy = my * irt, uz = mz * irt;
  // ---- flow collision
  if (a.shift_forcing) {
    // Shan-Chen velocity shift (Eq. 1.17, 1.18), BGK, F_i = 0
    T nxs = T(0), nys = T(0), nzs = T(0), den = T(0);
#pragma unroll
    for (int s = 0; s < NC; ++s) {
      nxs += jx[s] * k.om[s]; nys += jy[s] * k.om[s]; nzs += jz[s] * k.om[s];
      den += rho[s] * k.om[s];
    }
    const T iden = T(1) / den;
#pragma unroll
    for (int s = 0; s < NC; ++s) {
      const T ir = T(1) / rho[s];
      const T ex = nxs * iden + k.tau[s] * Fx[s] * ir;
      const T ey = nys * iden + k.tau[s] * Fy[s] * ir;
      const T ez = nzs * iden + k.tau[s] * Fz[s] * ir;
      // rho u: of a single component its own momentum and the shift
      const T tx = NC == 1 ? fmad(k.tau[s], Fx[s], jx[s]) : rho[s] * ex, ty = NC == 1 ? fmad(k.tau[s], Fy[s], jy[s]) : rho[s] * ey,
              tz = NC == 1 ? fmad(k.tau[s], Fz[s], jz[s]) : rho[s] * ez;
      bgk_pairs<L, T>(f[s], k.om[s], drho[s], ex, ey, ez, tx, ty, tz, T(0), T(0), T(0));
    }
  } else if (COLL == 1) {
    if constexpr (Q == 19) mrt_pairs_d3q19<T>(f[0], k, drho[0], jx[0], jy[0], jz[0], ux, uy, uz, Fx[0], Fy[0], Fz[0]);
    else mrt_pairs_rows<L, T>(f[0], k, drho[0], jx[0], jy[0], jz[0], ux, uy, uz, Fx[0], Fy[0], Fz[0]);
  } else {
#pragma unroll
    for (int s = 0; s < NC; ++s) {
      const T b = T(1) - T(0.5) * k.om[s];
      // rho u: of a single component mx, which carries no rounding of the velocity's division
      const T tx = NC == 1 ? mx : rho[s] * ux, ty = NC == 1 ? my : rho[s] * uy, tz = NC == 1 ? mz : rho[s] * uz;
      bgk_pairs<L, T>(f[s], k.om[s], drho[s], ux, uy, uz, tx, ty, tz, b * Fx[s], b * Fy[s], b * Fz[s]);
    }
  }
  // ---- scalar collision (Eq. therpop_species, therpopeq_species), u = physical velocity
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    T dC = T(0);
#pragma unroll
    for (int j = 0; j < QC; ++j) dC += h[s][j];
    const T C = k.cref[s] + dC;
#pragma unroll
    for (int j = 0; j < QC; ++j) {
      const T cu = T(L::cx(j)) * ux + T(L::cy(j)) * uy + T(L::cz(j)) * uz;
      const T he = scal_w<T>(j, k) * (dC + C * cu * k.ics2c);
      h[s][j] -= k.omc[s] * (h[s][j] - he);
    }
  }
  // ---- scatter flow
  // a node under a moving top plate (Sec. 3.1.1): links through the face beyond y = ny - 1
  // reflect with Ladd's momentum exchange 2 w_i rho (c_i . u_wall) / c_s^2
  // a node on the inlet face (Sec. 3.4): links leaving through x = 0 reflect off a face moving
  // with the inlet profile (the same momentum exchange); on the outlet face the population
  // entering through x = nx - 1 repeats the node's own post-collision value (zero gradient)
  // (BND: the kernel variant for contexts with a moving plate or a velocity inlet)
  bool top = false, xin = false, xout = false;
  T uin = T(0);
  if (BND && (a.moving_wall || a.flow_open_x)) {
    const unsigned int q = fast_div(unsigned(n), a.div_x);
    const int yy = int(q - fast_div(q, a.div_y) * unsigned(a.ny));
    top = a.moving_wall && yy == a.ny - 1;
    if (a.flow_open_x) {
      const int xx = n - int(q) * a.nx;
      xin = xx == 0;
      xout = xx == a.nx - 1;
      if (xin) uin = T(a.u_in_row[yy]);
    }
  }
  // the cache entries move to registers, and the cache takes the next node's while this one is stored
  typename Entries<VAR>::type ent[parity ? Q - 1 : 1];
  if (parity) {
#pragma unroll
    for (int i = 0; i < Q - 1; ++i) ent[i] = o.cache[i * CS];
  }
  pre();
  const OddCells<L, S, NC, NS, 1, VAR> to{a, c, m, ent};
#pragma unroll
  for (int s = 0; s < NC; ++s) {
    Store<S>::st(R::f(a, c, s, 0), f[s][0]);
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      T v = f[s][i];
      bool keep = true;
      if (BND && (parity == 0 || flow_wall<L>(m, i))) {
        if (L::cx(i) < 0 && xin && flow_wall<L>(m, i))
          v += T(6.0 * L::w(i)) * rho[s] * uin;
        else if (L::cx(i) > 0 && xout)
          keep = false;   // leaves through the outlet; the cell is written below with opp(i)
        else if (L::cy(i) > 0 && top && flow_wall<L>(m, i))
          v -= T(L::w(i)) * rho[s] * (T(L::cx(i)) * k.uw6[0] + T(L::cz(i)) * k.uw6[2] + k.uw6[1]);
      }
      if (keep) Store<S>::st(parity ? to.flow(s, i) : R::f(a, c, s, L::opp(i)), v);
      // zero-gradient outlet: the population entering through x = nx - 1 with direction i
      // repeats the node's own post-collision f_i, in the cell where link opp(i) reflects
      if (BND && L::cx(i) < 0 && xout) Store<S>::st(R::f(a, c, s, i), f[s][i]);
    }
  }
  // ---- scatter scalars: bounce-back at walls, inlet ghost / zero-gradient outlet at open faces
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    Store<SC>::st(R::h(a, c, s, 0), h[s][0]);
#pragma unroll
    for (int j = 1; j < QC; ++j) {
      T v = h[s][j];
      if (L::cx(j) != 0 && MaskBits<L>::code(m, j) == 3u) {   // only the x faces are open
        // open face: the population arriving from outside replaces the one leaving, in the own
        // cell (row opp(j))
        const int jb = L::opp(j);
        const long long row = LBM_CHK(a.err, s * (a.ny * a.nz) + int(fast_div(unsigned(n), a.div_x)), 3ll * a.ny * a.nz);
        T b;
        if (L::cx(j) < 0) {
          const T cu = T(L::cx(jb)) * ux;
          b = k.wca * k.C_in[s] * (T(1) + cu * k.ics2c) - k.wca * k.cref[s];
          a.inflow_row[row] += widen(b) - widen(v);
        } else {
          b = h[s][jb];
          a.outflow_row[row] += widen(v) - widen(b);
        }
        v = b;
      }
      Store<SC>::st(parity ? to.scal(s, j) : R::h(a, c, s, L::opp(j)), v);
    }
  }
}

template <class L, class S>
__device__ __forceinline__ void solid_nodes(const Args& a, const Coef<typename Store<S>::T>& k, int parity, unsigned int block, unsigned int blocks);

// Blocks per SM of the odd step with 64-bit offsets: two leave the registers it needs (576^3 FP32 3726 us, 3929 us with
// three and spills), but mixed storage with its two address forms does better with three (3546 us, 3617 us with two).
template <class S>
constexpr int wide_min_blocks() { return std::is_same<S, typename ScalarOf<S>::type>::value ? 2 : 3; }

// One fused time step for every fluid node: gather (A-A parity), wet-node closure and its
// bookkeeping, deposition, moments, forces, velocity, flow collision (BGK / MRT, Guo or
// velocity shift), scalar collision, in-place scatter with bounce-back / inlet / outlet.
// Registers hold deviations from w_i * ref throughout.
//
// What bounds it (256^3 packing, D3Q19 MRT + D3Q7, 6.7 M fluid nodes): the even step in FP32 DRAM traffic, 1.1 times
// the 208 bytes per node (273 us with planes over the domain and a collision per population, 248 us now); the odd step
// the latency of its scattered neighbour cells (390 -> 362 us); with 16-bit storage instruction issue (232 x 203 x
// 181, FP16 flow and FP32 scalars: 140 / 190 -> 117 / 180 us); FP64 the FP64 units (64^3: 163 -> 88 us per
// step).  128^3 FP32, where half of the 0.17 GB of populations fit into L2: 49 -> 39 us per step, of which the walk
// back and forth gives 5.
template <class L, class S, int NC, int NS, int COLL, int parity, int VAR>
__global__ void __launch_bounds__(256, (NC == 1 && sizeof(typename Store<S>::T) == 4 ? (VAR == kWide ? wide_min_blocks<S>() : parity ? LBM_STEP_MIN_BLOCKS_ODD : LBM_STEP_MIN_BLOCKS) : 2)) k_step(const Args a, const Coef<typename Store<S>::T> k) {
  using T = typename Store<S>::T;
  constexpr int Q = L::Q, QC = L::QC, NSD = NS > 0 ? NS : 1;
  constexpr bool BND = VAR == kFull;
  using R = Rec<L, S, NC, NS>;
  using O = OddCells<L, S, NC, NS, LBM_STEP_CACHE_STRIDE, VAR>;
  T wallx = T(0), heatx = T(0), prodx = T(0);
  pdl_trigger();
  unsigned int blocks = gridDim.x;
  if constexpr (BND && NS > 1) {
    // conduction in the solid: the last blocks advance the solid lattice, of which the fluid's step reads the old state
    // only.  A launch of its own adds its latency to every step (420 x 80: 4.8 us beside a step of 8).
    blocks -= a.solid_blocks;
    if (blockIdx.x >= blocks) {
      pdl_wait();
      solid_nodes<L, S>(a, k, parity, blockIdx.x - blocks, a.solid_blocks);
      return;
    }
  }
  if (a.geo_mode != GEO_NONE) pdl_wait();
  const unsigned int count = a.fluid_count[0];
  const unsigned int base = a.fluid_count[1];   // entries below it have slot == entry
  // Block rounds over the list, forwards or backwards.  Each kernel that reads the populations starts where its
  // predecessor ended, so that the populations L2 still holds are read there: odd steps go backwards, and
  // after a psi pass (always forwards) so does every step.
  const bool back = parity == 1 || a.sc_on;
  unsigned int stride = blocks * blockDim.x;
  unsigned int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (back) {
    // whole blocks from the list's end; below its start e and e + stride wrap past count
    e = ((count + blockDim.x - 1) / blockDim.x - 1 - blockIdx.x) * blockDim.x + threadIdx.x;
    stride = 0u - stride;
    if (e >= count) e += stride;   // the last block's threads past the end
  }
  const auto slot = [&](unsigned int en, int n) { return en < base ? (long long)en : (long long)__ldg(a.slot + n); };
  // the list entry is fetched two iterations and the link mask one iteration ahead
  uint32_t w_cur = e < count ? a.fluid_list[e] : 0u;
  uint32_t w_nx = e + stride < count ? a.fluid_list[e + stride] : 0u;
  uint32_t m_cur = e < count ? a.mask[list_node(a, w_cur)] : 0u;
  if constexpr (parity == 1) {
    // the neighbours of the next entry are copied in (asynchronously) while this entry is stored
    using E = typename Entries<VAR>::type;
    __shared__ E slot_buf[(L::Q - 1) * LBM_STEP_CACHE_STRIDE];
    E* cb = slot_buf + threadIdx.x;
    const E* map = Entries<VAR>::map(a);
    if (e < count) prefetch_nbrs<L, LBM_STEP_CACHE_STRIDE>(a, map, w_cur, cb);
    cp_async_commit();
    if (a.geo_mode == GEO_NONE) pdl_wait();
    for (; e < count; e += stride) {
      const uint32_t w = w_cur, m = m_cur;
      const bool more = e + stride < count;
      if (more) {
        w_cur = w_nx;
        m_cur = a.mask[list_node(a, w_cur)];
      }
      if (e + 2 * stride < count) w_nx = a.fluid_list[e + 2 * stride];
      cp_async_wait<0>();   // this entry's neighbours have arrived
      const auto pre = [&]() {
        if (more) prefetch_nbrs<L, LBM_STEP_CACHE_STRIDE>(a, map, w_cur, cb);
        cp_async_commit();
      };
      if (m & 1u) {
        T f[NC][Q], h[NSD][QC];
        const int n = list_node(a, w);
        const long long sn = slot(e, n), c = R::cell(sn);
        // the plain variant addresses every flow link through its cache entry (wall_offsets);
        // the full variant keeps the per-link tests its boundary rules need
        if (VAR != kFull) wall_offsets<L, R, LBM_STEP_CACHE_STRIDE>(sn, m, cb);
        const O o{a, c, m, cb};
        gather_odd<L, S, NC, NS, LBM_STEP_CACHE_STRIDE, VAR>(o, f, h);
        collide_scatter<L, S, NC, NS, COLL, parity, VAR>(a, k, w, n, m, c, o, f, h, wallx, heatx, prodx, pre);
      } else {
        pre();
      }
    }
    cp_async_wait<0>();
  } else {
    if (a.geo_mode == GEO_NONE) pdl_wait();
    for (; e < count; e += stride) {
      const uint32_t w = w_cur, m = m_cur;
      w_cur = w_nx;
      if (e + stride < count) m_cur = a.mask[list_node(a, w_cur)];
      if (e + 2 * stride < count) w_nx = a.fluid_list[e + 2 * stride];
      if (!(m & 1u)) continue;   // a node removed by deposition since the last list rebuild
      T f[NC][Q], h[NSD][QC];
      const int n = list_node(a, w);
      const long long c = R::cell(slot(e, n));
      gather_even<L, S, NC, NS>(a, c, f, h);
      collide_scatter<L, S, NC, NS, COLL, parity, VAR>(a, k, w, n, m, c, O{a, c, m, nullptr}, f, h, wallx, heatx, prodx, []() {});
    }
  }
  // ---- wall-exchange monitor: one reduction per warp that saw a reactive link
  if (NS > 0) {
    const unsigned int any = __ballot_sync(0xffffffffu, wallx != T(0));
    if (any) {
      const T w = warp_sum(wallx);
      if ((threadIdx.x & 31) == 0)
        atomicAdd(a.wallx_slot + ((blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) % WALLX_SLOTS),
                  widen(w));
    }
  }
  // ---- reaction heat monitor (second bank of the slots)
  if (BND && NS > 1) {
    const unsigned int any = __ballot_sync(0xffffffffu, heatx != T(0));
    if (any) {
      const T w = warp_sum(heatx);
      if ((threadIdx.x & 31) == 0)
        atomicAdd(a.wallx_slot + WALLX_SLOTS +
                      ((blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) % WALLX_SLOTS),
                  widen(w));
    }
  }
  // ---- reaction product monitor (third bank)
  if (NS > 1) {
    const unsigned int any = __ballot_sync(0xffffffffu, prodx != T(0));
    if (any) {
      const T w = warp_sum(prodx);
      if ((threadIdx.x & 31) == 0)
        atomicAdd(a.wallx_slot + 2 * WALLX_SLOTS +
                      ((blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) % WALLX_SLOTS),
                  widen(w));
    }
  }
}

// ================================================================ ensembles

#ifndef LBM_TILE_CHUNK
#define LBM_TILE_CHUNK 8
#endif
// Work tile of an ensemble step: blockDim consecutive fluid-list entries of one member.
struct Tile {
  unsigned int member, first;
};

// One time step of every member of an ensemble in one launch.  Blocks take chunks of the work
// list of tiles in turn; whenever a block enters another member it stages that member's
// arguments and constants in shared memory, and for each tile it updates entries first ..
// first + blockDim - 1 exactly as k_step updates them.
template <class L, class S, int NC, int NS, int COLL, int parity, bool BND>
__global__ void __launch_bounds__(256, (NC == 1 && sizeof(typename Store<S>::T) == 4 ? (L::D == 2 ? LBM_TILES_MIN_BLOCKS_2D : (parity ? LBM_TILES_MIN_BLOCKS_ODD : LBM_STEP_MIN_BLOCKS)) : 2)) k_step_tiles(
    const Args* __restrict__ args, const Coef<typename Store<S>::T>* __restrict__ coefs,
    const Tile* __restrict__ tiles, unsigned int ntiles, unsigned int chunk) {
  using T = typename Store<S>::T;
  constexpr int Q = L::Q, QC = L::QC, NSD = NS > 0 ? NS : 1;
  static_assert(sizeof(Args) % 4 == 0 && sizeof(Coef<T>) % 4 == 0, "word copies");
  __shared__ Args sa;
  __shared__ Coef<T> sk;
  using R = Rec<L, S, NC, NS>;
  constexpr int VAR = BND ? kFull : kPlain;
  using O = OddCells<L, S, NC, NS, 1, VAR>;
  extern __shared__ uint32_t slot_smem[];   // blockDim.x * Q words at odd parity (launcher)
  uint32_t* cache = slot_smem + threadIdx.x * L::Q;
  // blocks take chunks of consecutive tiles in turn (at most LBM_TILE_CHUNK, fewer where that would leave
  // blocks idle): the work list holds each member's tiles together, so a chunk mostly stays within
  // one member and its arguments are staged again only when the chunk crosses into another; taking
  // chunks in turn keeps a mix of uneven members on every block
  auto next_tile = [&](unsigned int t) {
    return t + ((t % chunk == chunk - 1) ? (gridDim.x - 1) * chunk + 1 : 1);
  };
  // odd parity: the next tile's neighbours are copied in (cp.async) while this tile is stored, as in
  // k_step; the next tile's list entry and link mask are loaded one tile ahead at both parities
  // whenever it belongs to the member already staged
  bool have_next = false, waited = false;
  uint32_t w_pf = 0u, m_pf = 0u;
  unsigned int staged = 0xffffffffu;
  // odd steps take the tiles backwards, from those whose populations L2 still holds (see k_step)
  const auto tile_at = [&](unsigned int t) { return tiles[parity ? ntiles - 1 - t : t]; };
  pdl_trigger();
  for (unsigned int t = blockIdx.x * chunk; t < ntiles; t = next_tile(t)) {
    const Tile tile = tile_at(t);
    if (tile.member != staged) {   // block-uniform
      __syncthreads();   // the previous member's tiles are done with sa / sk
      const uint32_t* src = reinterpret_cast<const uint32_t*>(args + tile.member);
      uint32_t* dst = reinterpret_cast<uint32_t*>(&sa);
      for (unsigned int i = threadIdx.x; i < sizeof(Args) / 4; i += blockDim.x) dst[i] = src[i];
      const uint32_t* ksrc = reinterpret_cast<const uint32_t*>(coefs + tile.member);
      uint32_t* kdst = reinterpret_cast<uint32_t*>(&sk);
      for (unsigned int i = threadIdx.x; i < sizeof(Coef<T>) / 4; i += blockDim.x) kdst[i] = ksrc[i];
      __syncthreads();
      staged = tile.member;
      have_next = false;
    }
    const Args& a = sa;
    const uint32_t* map = Entries<VAR>::map(a);
    T wallx = T(0), heatx = T(0), prodx = T(0);
    const unsigned int e = tile.first + threadIdx.x;
    const unsigned int count = a.fluid_count[0];
    uint32_t w = 0u, m = 0u;
    if (have_next) {
      w = w_pf;
      m = m_pf;
    } else if (e < count) {
      w = a.fluid_list[e];
      m = a.mask[list_node(a, w)];
      if (parity) prefetch_nbrs<L, 1>(a, map, w, cache);
    }
    if (parity) {
      cp_async_commit();
      cp_async_wait<0>();   // this tile's neighbours have arrived
    }
    // the next tile of this block, if it belongs to the staged member
    have_next = false;
    bool next_in = false;
    const unsigned int tn = next_tile(t);
    if (tn < ntiles) {
      const Tile tile2 = tile_at(tn);
      if (tile2.member == staged) {
        const unsigned int e2 = tile2.first + threadIdx.x;
        w_pf = 0u;
        m_pf = 0u;
        if (e2 < count) {
          w_pf = a.fluid_list[e2];
          m_pf = a.mask[list_node(a, w_pf)];
          next_in = true;
        }
        have_next = true;
      }
    }
    const auto pre = [&]() {
      if (parity && next_in) prefetch_nbrs<L, 1>(a, map, w_pf, cache);
    };
    if (!waited) pdl_wait();   // ensembles keep their geometry: everything read so far is static
    waited = true;
    if (e < count && (m & 1u)) {
      const unsigned int base = a.fluid_count[1];
      T f[NC][Q], h[NSD][QC];
      const int n = list_node(a, w);
      const long long sn = e < base ? (long long)e : (long long)__ldg(a.slot + n), c = R::cell(sn);
      const O o{a, c, m, cache};
      if (parity) {
        // the plain variant addresses every flow link through its cache entry (wall_offsets)
        if (!BND) wall_offsets<L, R, 1>(sn, m, cache);
        gather_odd<L, S, NC, NS, 1, VAR>(o, f, h);
      } else {
        gather_even<L, S, NC, NS>(a, c, f, h);
      }
      collide_scatter<L, S, NC, NS, COLL, parity, VAR>(a, sk, w, n, m, c, o, f, h, wallx, heatx, prodx, pre);
    } else {
      pre();
    }
    if (NS > 0) {
      const unsigned int any = __ballot_sync(0xffffffffu, wallx != T(0));
      if (any) {
        const T w = warp_sum(wallx);
        if ((threadIdx.x & 31) == 0)
          atomicAdd(a.wallx_slot + ((t * (blockDim.x >> 5) + (threadIdx.x >> 5)) % WALLX_SLOTS), widen(w));
      }
    }
    if (BND && NS > 1) {
      const unsigned int any = __ballot_sync(0xffffffffu, heatx != T(0));
      if (any) {
        const T w = warp_sum(heatx);
        if ((threadIdx.x & 31) == 0)
          atomicAdd(a.wallx_slot + WALLX_SLOTS + ((t * (blockDim.x >> 5) + (threadIdx.x >> 5)) % WALLX_SLOTS),
                    widen(w));
      }
    }
    if (NS > 1) {
      const unsigned int any = __ballot_sync(0xffffffffu, prodx != T(0));
      if (any) {
        const T w = warp_sum(prodx);
        if ((threadIdx.x & 31) == 0)
          atomicAdd(a.wallx_slot + 2 * WALLX_SLOTS + ((t * (blockDim.x >> 5) + (threadIdx.x >> 5)) % WALLX_SLOTS),
                    widen(w));
      }
    }
  }
  if (parity) cp_async_wait<0>();
  if (!waited) pdl_wait();
}

// ================================================================ psi

template <class L, class S, int NC, int NS, int parity>
__global__ void __launch_bounds__(256) k_psi(const Args a, const Coef<typename Store<S>::T> k) {
  // Walks the fluid list in slot order, as k_step does: at parity 0 every population of the
  // node sits in its own cell (coalesced); at parity 1 population i sits in cell (n - c_i, opp i),
  // whose slot is looked up once for all components.  Sums in population order 0 .. Q-1 from
  // rho_ref, the order the gather of the step uses.  Bound by DRAM (parity 0: 128^3 with two components, 0.32 GB in
  // 57 us) and by the scattered cells (parity 1: 70 us; 62 and 94 us with planes over the domain).
  using T = typename Store<S>::T;
  using R = Rec<L, S, NC, NS>;
  pdl_trigger();
  if (a.geo_mode != GEO_NONE) pdl_wait();
  const unsigned int count = a.fluid_count[0];
  const unsigned int base = a.fluid_count[1];   // entries below it have slot == entry
  const unsigned int stride = gridDim.x * blockDim.x;
  unsigned int e = blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t w = e < count ? a.fluid_list[e] : 0u;
  uint32_t m = e < count ? a.mask[list_node(a, w)] : 0u;
  bool waited = a.geo_mode != GEO_NONE;
  for (; e < count; e += stride) {
    const int n = list_node(a, w);
    const long long c = R::cell(e < base ? (long long)e : (long long)__ldg(a.slot + n));
    long long cell[L::Q];   // offset of the row holding population i of component 0
    const Nbr nb = parity ? nbr_entry(a, n, w) : Nbr{};
    const uint32_t mn = m;
#pragma unroll
    for (int i = 0; i < L::Q; ++i)
      cell[i] = (parity == 0 || i == 0 || flow_wall<L>(mn, L::opp(i)))
                    ? c + R::frow(0, i)
                    : cell_of<R>(a, nb.at(-L::cx(i), -L::cy(i), -L::cz(i))) + R::frow(0, L::opp(i));
    if (e + stride < count) {   // the next entry and its mask, one iteration ahead
      w = a.fluid_list[e + stride];
      m = a.mask[list_node(a, w)];
    }
    if (!waited) pdl_wait();
    waited = true;
    if (!(mn & 1u)) continue;   // a node removed by deposition since the last list rebuild
#pragma unroll
    for (int s = 0; s < NC; ++s) {
      T r = k.rref[s];
#pragma unroll
      for (int i = 0; i < L::Q; ++i)
        r += Store<S>::ld(reinterpret_cast<const S*>(a.pop + LBM_CHK(a.err, cell[i] + s * L::Q * R::FROW, a.pop_bytes)));
      T p;
      if (a.psi_identity) p = r;
      else p = k.rho0 * (T(1) - exp(-r / k.rho0));   // Eq. 1.11
      reinterpret_cast<T*>(a.psi[s])[n] = p;
    }
  }
  if (!waited) pdl_wait();
}

// ================================================================ monitors

// Sums of K values over a block of 256 threads into out[0 .. K), in a fixed order; only the values with their bit in
// used (block-uniform) are added up, the others are 0 in every thread.  A warp takes every eighth value: 8 values per
// lane from shared memory, then 5 shuffle stages, a third of the FP64 additions of reducing every value in every warp
// (the FP64 unit is narrow: with 25 values per warp it was 56 % busy and most of the kernel's time).
template <int K>
__device__ __forceinline__ void block_reduce_store(double (&v)[K], unsigned int used, double* out) {
  constexpr int KB = K < 8 ? K : 8;   // values held at once
  __shared__ double sh[KB][256];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
#pragma unroll
  for (int q0 = 0; q0 < K; q0 += KB) {
    if ((used >> q0 & ((1u << KB) - 1u)) == 0u) {
      if (tid < KB && q0 + tid < K) out[q0 + tid] = 0.0;
      continue;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < KB; ++q)
      if (q0 + q < K && (used >> (q0 + q) & 1u)) sh[q][tid] = v[q0 + q];
    __syncthreads();
    if (wid < KB && q0 + wid < K) {
      double s = 0.0;
      if (used >> (q0 + wid) & 1u) {
#pragma unroll
        for (int i = 0; i < 8; ++i) s += sh[wid][lane + 32 * i];
        s = warp_sum(s);
      }
      if (lane == 0) out[q0 + wid] = s;
    }
  }
}

// Running sum of a thread over its nodes.  In FP32 the rounding error of every addition is kept (the two-sum of
// Knuth, The Art of Computer Programming 2, 4.2.2), so that the number of nodes per thread costs no accuracy and no
// FP64 operations; a sum that has left the finite numbers is its own result.
template <class T>
struct NodeSum {
  T s = T(0), c = T(0);
  __device__ __forceinline__ void add(T x) {
    const T t = s + x, b = t - s;
    c += (s - (t - b)) + (x - b);
    s = t;
  }
  __device__ __forceinline__ double value() const { return isfinite(s) ? double(s) + double(c) : double(s); }
};
template <>
struct NodeSum<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double x) { s += x; }
  __device__ __forceinline__ double value() const { return s; }
};

// Monitors, one wave of blocks: population sums over the fluid list, a node's in the compute type
// (deviations from the reference, so they stay accurate), bookkeeping sums over all nodes
// in FP64, per-block partials in FP64 (summed in fixed order by k_reduce_partials).  Bound by latency on small
// domains (15 us at any size up to 512 x 512, 38 to 44 us when every warp reduced every value), else by DRAM.
template <class L, class S, int NC, int NS>
__device__ __forceinline__ void monitor_block(const Args& a, const Coef<typename Store<S>::T>& k, const int parity,
                                              const unsigned int block, const unsigned int blocks) {
  using T = typename Store<S>::T;
  constexpr int Q = L::Q, QC = L::QC;
  const unsigned int tid = block * blockDim.x + threadIdx.x;
  const unsigned int nthr = blocks * blockDim.x;
  NodeSum<T> dm[NC > 0 ? NC : 1], mom[3], dsp[NS > 0 ? NS : 1];
  unsigned int nfluid = 0, nonfin = 0;
  const unsigned int count = a.fluid_count[0], base = a.fluid_count[1];
  for (unsigned int e = tid; e < count; e += nthr) {
    const uint32_t w = a.fluid_list[e];
    const int n = list_node(a, w);
    const uint32_t m = a.mask[n];
    if (!(m & 1u)) continue;
    ++nfluid;
    const Nbr nb = parity ? nbr_entry(a, n, w) : Nbr{};
    const long long cell = Rec<L, S, NC, NS>::cell(e < base ? (long long)e : (long long)a.slot[n]);
    bool bad = false;
    T jn[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int s = 0; s < NC; ++s) {
      T f[Q];
      gather_flow<L, S, NC, NS>(a, s, cell, m, nb, parity, f);
      T r = T(0);
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        r += f[i];
        if (L::cx(i)) jn[0] += T(L::cx(i)) * f[i];
        if (L::cy(i)) jn[1] += T(L::cy(i)) * f[i];
        if (L::cz(i)) jn[2] += T(L::cz(i)) * f[i];
      }
      bad |= !isfinite(r);
      dm[s].add(r);
    }
#pragma unroll
    for (int q = 0; q < L::D; ++q) mom[q].add(jn[q]);
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      T h[QC];
      gather_scal<L, S, NC, NS>(a, s, cell, m, nb, parity, h);
      T c = T(0);
#pragma unroll
      for (int j = 0; j < QC; ++j) c += h[j];
      bad |= !isfinite(c);
      dsp[s].add(c);
    }
    nonfin += bad ? 1u : 0u;
  }
  double v[NMON];
#pragma unroll
  for (int q = 0; q < NMON; ++q) v[q] = 0.0;
  for (int s = 0; s < NC; ++s) v[M_MASS + s] = dm[s].value() + double(k.rref[s]) * double(nfluid);
  for (int c = 0; c < 3; ++c) v[M_MOM + c] = mom[c].value();
  for (int s = 0; s < NS; ++s) v[mon_spec(s)] = dsp[s].value() + double(k.cref[s]) * double(nfluid);
  v[M_NFLUID] = double(nfluid);
  v[M_NONFIN] = double(nonfin);
  // bookkeeping over every node
  const bool dep = a.geo_mode == GEO_DEPOSIT;
  double react = 0.0, depo = 0.0, tsolid = 0.0;
  unsigned int nsolid = 0;
  const T* gcur = a.conjugate ? reinterpret_cast<const T*>(a.gs[parity]) : nullptr;
  for (long long n = tid; n < a.N; n += nthr) {
    const uint8_t fl = a.flags[n];
    nsolid += fl != FL_FLUID ? 1u : 0u;
    const double acc = a.acc[n];
    if (acc != 0.0) {
      if (dep && fl != FL_REACTIVE) depo += acc; else react += acc;
    }
    if (gcur && fl != FL_FLUID) {
      T t = T(0);
#pragma unroll
      for (int q = 0; q < QC; ++q) t += gcur[(long long)q * a.N + n];
      tsolid += double(t);
    }
  }
  v[M_REACT] = react;
  v[M_DEPO] = depo;
  v[M_NSOLID] = double(nsolid);
  v[M_TSOLID] = tsolid;
  const int rows = a.ny * a.nz;
  for (int r = tid; r < rows; r += nthr)
    for (int s = 0; s < NS; ++s) {
      v[mon_in(s)] += a.inflow_row[s * rows + r];
      v[mon_out(s)] += a.outflow_row[s * rows + r];
    }
  for (int q = tid; q < WALLX_SLOTS; q += nthr) {
    v[M_WALLX] += a.wallx_slot[BANK_WALLX * WALLX_SLOTS + q];
    v[M_HEAT] += a.wallx_slot[BANK_HEAT * WALLX_SLOTS + q];
    v[M_PROD] += a.wallx_slot[BANK_PROD * WALLX_SLOTS + q];
    v[M_HEAT_S] += a.wallx_slot[BANK_HEAT_S * WALLX_SLOTS + q];
    v[M_HEAT_SRC] += a.wallx_slot[BANK_HEAT_SRC * WALLX_SLOTS + q];
  }
  // what this kind of context can have in its sums
  unsigned int used = 1u << M_MASS | (NC > 1 ? 1u << (M_MASS + 1) : 0u) | 7u << M_MOM | 1u << M_NFLUID | 1u << M_NSOLID | 1u << M_NONFIN;
  if (NS > 0) used |= 1u << M_REACT | 1u << M_DEPO | 1u << M_WALLX;
  for (int s = 0; s < NS; ++s) {
    used |= 1u << mon_spec(s);
    if (a.open_x) used |= 1u << mon_in(s) | 1u << mon_out(s);
  }
  if (NS > 1) used |= 1u << M_HEAT | 1u << M_PROD;
  if (a.conjugate) used |= 1u << M_TSOLID | 1u << M_HEAT_S | 1u << M_HEAT_SRC;
  block_reduce_store<NMON>(v, used, a.partials + (long long)block * NMON);
}

template <class L, class S, int NC, int NS>
__global__ void __launch_bounds__(256) k_monitor(const Args a, const Coef<typename Store<S>::T> k, const int parity) {
  monitor_block<L, S, NC, NS>(a, k, parity, blockIdx.x, gridDim.x);
}

// ================================================================ node macroscopics

// rho^sigma, physical velocity (Eq. 1.19) and closed scalars of fluid node n; psi arrays must be
// current when Shan-Chen forces are on.
template <class L, class S, int NC, int NS>
__device__ __forceinline__ void node_macros(const Args& a, const Coef<typename Store<S>::T>& k, int n, const Nbr& nb,
                                            uint32_t m, long long cell, int parity, typename Store<S>::T* rho_out,
                                            typename Store<S>::T* u_out, typename Store<S>::T* C_out) {
  using T = typename Store<S>::T;
  constexpr int Q = L::Q, QC = L::QC;
  T rho[NC], jx[NC], jy[NC], jz[NC], Fx[NC], Fy[NC], Fz[NC];
#pragma unroll
  for (int s = 0; s < NC; ++s) {
    T f[Q];
    gather_flow<L, S, NC, NS>(a, s, cell, m, nb, parity, f);
    T r = T(0), ax = T(0), ay = T(0), az = T(0);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      r += f[i];
      ax += T(L::cx(i)) * f[i];
      ay += T(L::cy(i)) * f[i];
      az += T(L::cz(i)) * f[i];
    }
    r += k.rref[s];
    rho[s] = r; jx[s] = ax; jy[s] = ay; jz[s] = az;
    Fx[s] = r * k.g[0]; Fy[s] = r * k.g[1]; Fz[s] = r * k.g[2];
  }
  if (a.sc_on) {
    for (int s = 0; s < NC; ++s) {
      const T pself = reinterpret_cast<const T*>(a.psi[s])[n];
      for (int s2 = 0; s2 < NC; ++s2) {
        const T* ps = reinterpret_cast<const T*>(a.psi[s2]);
        T ax = T(0), ay = T(0), az = T(0);
#pragma unroll
        for (int i = 1; i < Q; ++i) {
          const T pv = flow_wall<L>(m, i) ? k.psi_wall : ps[nb.at(L::cx(i), L::cy(i), L::cz(i))];
          ax += T(L::w(i)) * pv * T(L::cx(i));
          ay += T(L::w(i)) * pv * T(L::cy(i));
          az += T(L::w(i)) * pv * T(L::cz(i));
        }
        const T Gss = k.G[s][s2];
        Fx[s] -= pself * Gss * ax; Fy[s] -= pself * Gss * ay; Fz[s] -= pself * Gss * az;
      }
    }
  }
  if (a.ads_on) {
    T ax = T(0), ay = T(0), az = T(0);
#pragma unroll
    for (int i = 1; i < Q; ++i)
      if (flow_wall<L>(m, i)) {
        ax += T(L::w(i)) * T(L::cx(i));
        ay += T(L::w(i)) * T(L::cy(i));
        az += T(L::w(i)) * T(L::cz(i));
      }
    for (int s = 0; s < NC; ++s) {
      const T ga = k.G_ads[s] * rho[s];
      Fx[s] -= ga * ax; Fy[s] -= ga * ay; Fz[s] -= ga * az;
    }
  }
  T rt = T(0), mx = T(0), my = T(0), mz = T(0);
  for (int s = 0; s < NC; ++s) {
    rt += rho[s];
    mx += jx[s] + T(0.5) * Fx[s];
    my += jy[s] + T(0.5) * Fy[s];
    mz += jz[s] + T(0.5) * Fz[s];
  }
  for (int s = 0; s < NC; ++s) rho_out[s] = rho[s];
  u_out[0] = mx / rt;
  u_out[1] = my / rt;
  u_out[2] = mz / rt;
  T hh[NS > 0 ? NS : 1][QC];
#pragma unroll
  for (int s = 0; s < NS; ++s)
    gather_scal<L, S, NC, NS>(a, s, cell, m, nb, parity, hh[s]);
  T rl[QC], gain = T(0);
#pragma unroll
  for (int j = 0; j < QC; ++j) rl[j] = T(0);
  if (NS > 1 && a.conjugate)
    close_conjugate<L, T>(hh[0], hh[NS > 1 ? 1 : 0], m, k, a, nb, reinterpret_cast<const T*>(a.gs[parity]),
                          [&](int j, T r, T) { rl[j] = r; });
  else if (NS > 1 && a.arrhenius)
    close_thermal<L, T>(hh[0], hh[NS > 1 ? 1 : 0], m, k, a.n_it, [&](int j, T r, T, T) { rl[j] = r; });
  else if (NS > 0)
    close_scalar<L, T>(hh[0], m, k, [&](int j, T Cb, T) { rl[j] = k.kr * Cb; });
  if (NS > 1 && a.product) close_product<L, T>(hh[NS - 1], m, k, rl, gain);
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    T C = k.cref[s];
#pragma unroll
    for (int j = 0; j < QC; ++j) C += hh[s][j];
    C_out[s] = C;
  }
}

// Macroscopic fields of every node into FP64 staging (solid nodes read 0).
template <class L, class S, int NC, int NS>
__global__ void __launch_bounds__(256) k_moments(const Args a, const Coef<typename Store<S>::T> k,
                                                 const int parity) {
  using T = typename Store<S>::T;
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (n >= a.N) return;
  const long long N = a.N;
  const uint32_t m = a.mask[n];
  T rho[NC], u[3], C[NS > 0 ? NS : 1];
  if (m & 1u) {
    node_macros<L, S, NC, NS>(a, k, int(n), nbr_of(a, int(n)), m, Rec<L, S, NC, NS>::cell(a.slot[n]), parity, rho, u, C);
  } else {
    for (int s = 0; s < NC; ++s) rho[s] = T(0);
    u[0] = u[1] = u[2] = T(0);
    for (int s = 0; s < NS; ++s) C[s] = T(0);
    if (NS > 1 && a.conjugate) {
      // the solid temperature (Eq. macroreacb_solid)
      const T* g = reinterpret_cast<const T*>(a.gs[parity]);
      T t = T(0);
#pragma unroll
      for (int q = 0; q < L::QC; ++q) t += g[(long long)q * N + n];
      C[NS > 1 ? 1 : 0] = t;
    }
  }
  for (int s = 0; s < NC; ++s) a.d_rho[s * N + n] = double(rho[s]);
  for (int c = 0; c < 3; ++c) a.d_u[c * N + n] = double(u[c]);
  for (int s = 0; s < NS; ++s) a.d_C[s * N + n] = double(C[s]);
}

// Residual partials over the fluid list against compute-type snapshots [4][pitch] (u, C) held
// at the nodes' storage slots, which are replaced: sum (u - u_s)^2, sum u^2, sum (C - C_s)^2,
// sum C^2.  (A re-slotting invalidates the snapshots; the runtime then skips one evaluation.)
template <class L, class S, int NC, int NS>
__device__ __forceinline__ void resid_block(const Args& a, const Coef<typename Store<S>::T>& k, const int parity,
                                            const unsigned int block, const unsigned int blocks) {
  using T = typename Store<S>::T;
  T* snap = reinterpret_cast<T*>(a.snap);
  const long long P = a.pitch;
  NodeSum<T> du, uu, dc, cc;
  const unsigned int count = a.fluid_count[0], base = a.fluid_count[1];
  for (unsigned int e = block * blockDim.x + threadIdx.x; e < count; e += blocks * blockDim.x) {
    const uint32_t w = a.fluid_list[e];
    const int n = list_node(a, w);
    const uint32_t m = a.mask[n];
    if (!(m & 1u)) continue;
    const long long sn = e < base ? (long long)e : (long long)a.slot[n];
    T rho[NC], u[3], C[NS > 0 ? NS : 1];
    node_macros<L, S, NC, NS>(a, k, n, nbr_entry(a, n, w), m, Rec<L, S, NC, NS>::cell(sn), parity, rho, u, C);
    T dn = T(0), un = T(0);
    for (int c = 0; c < 3; ++c) {
      const T d = u[c] - snap[c * P + sn];
      dn += d * d;
      un += u[c] * u[c];
      snap[c * P + sn] = u[c];
    }
    du.add(dn);
    uu.add(un);
    if (NS > 0) {
      const T d = C[0] - snap[3 * P + sn];
      dc.add(d * d);
      cc.add(C[0] * C[0]);
      snap[3 * P + sn] = C[0];
    }
  }
  double v[4] = {du.value(), uu.value(), dc.value(), cc.value()};
  block_reduce_store<4>(v, 15u, a.partials + (long long)block * 4);
}

template <class L, class S, int NC, int NS>
__global__ void __launch_bounds__(256) k_resid(const Args a, const Coef<typename Store<S>::T> k, const int parity) {
  resid_block<L, S, NC, NS>(a, k, parity, blockIdx.x, gridDim.x);
}

// One block of an evaluation of every member of an ensemble: `block` of `blocks` of its member.
struct EvalBlock {
  unsigned int member, block, blocks;
};

// Monitors or residual partials of all members in one launch, each block as k_monitor's or k_resid's of its
// member.  Launched member by member they are bound by latency: 15 us for the monitors of any small member.
template <class L, class S, int NC, int NS>
__global__ void __launch_bounds__(256) k_eval_members(const Args* __restrict__ args,
                                                      const Coef<typename Store<S>::T>* __restrict__ coefs,
                                                      const EvalBlock* __restrict__ list, const int resid,
                                                      const int parity) {
  __shared__ Args sa;
  __shared__ Coef<typename Store<S>::T> sk;
  const EvalBlock b = list[blockIdx.x];
  const uint32_t* src = reinterpret_cast<const uint32_t*>(args + b.member);
  for (unsigned int i = threadIdx.x; i < sizeof(Args) / 4; i += blockDim.x) reinterpret_cast<uint32_t*>(&sa)[i] = src[i];
  const uint32_t* ksrc = reinterpret_cast<const uint32_t*>(coefs + b.member);
  for (unsigned int i = threadIdx.x; i < sizeof(sk) / 4; i += blockDim.x) reinterpret_cast<uint32_t*>(&sk)[i] = ksrc[i];
  __syncthreads();
  if (resid) resid_block<L, S, NC, NS>(sa, sk, parity, b.block, b.blocks);
  else monitor_block<L, S, NC, NS>(sa, sk, parity, b.block, b.blocks);
}

// ================================================================ init / pop I/O

// Equilibrium populations from FP64 staging fields (Eq. 6, Eq. therpopeq_species), natural
// layout, computed in the compute type.
template <class L, class S, int NC, int NS>
__global__ void __launch_bounds__(256) k_init(const Args a, const Coef<typename Store<S>::T> k) {
  using T = typename Store<S>::T;
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (n >= a.N) return;
  const bool fluid = a.flags[n] == FL_FLUID;
  using R = Rec<L, S, NC, NS>;
  const long long c = R::cell(a.slot[n]);
  const T ux = T(a.d_u[n]), uy = T(a.d_u[a.N + n]), uz = (L::D == 3) ? T(a.d_u[2 * a.N + n]) : T(0);
  for (int s = 0; s < NC; ++s) {
    const T r = T(a.d_rho[s * a.N + n]);
    const T dr = T(a.d_rho[s * a.N + n] - double(k.rref[s]));
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      const T v = fluid ? feq_dev<L, T>(i, r, dr, ux, uy, uz) : T(0);
      Store<S>::st(R::f(a, c, s, i), v);
    }
  }
  for (int s = 0; s < NS; ++s) {
    using SC = typename R::SC;
    const T C = T(a.d_C[s * a.N + n]);
    const T dC = T(a.d_C[s * a.N + n] - double(k.cref[s]));
#pragma unroll
    for (int j = 0; j < L::QC; ++j) {
      const T cu = T(L::cx(j)) * ux + T(L::cy(j)) * uy + T(L::cz(j)) * uz;
      const T wj = scal_w<T>(j, k);
      const T v = fluid ? wj * (dC + C * cu * k.ics2c) : T(0);
      Store<SC>::st(R::h(a, c, s, j), v);
    }
  }
}

// Natural-order FP64 copy of the pre-collision populations (dir = 0: device state -> out,
// dir = 1: in -> device state at the current layout parity).  Full values (reference added
// back).  Solid nodes read as 0.
template <class L, class S, int NC, int NS>
__global__ void __launch_bounds__(256) k_pops_io(const Args a, const Coef<typename Store<S>::T> k,
                                                 const int parity, const int dir, double* fio,
                                                 double* hio) {
  using T = typename Store<S>::T;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  if (x >= a.nx || y >= a.ny) return;
  const int n = x + a.nx * (y + a.ny * z);
  const uint32_t m = a.mask[n];
  const bool fluid = (m & 1u) != 0u;
  const Nbr nb = make_nbr(a, x, y, z);
  using R = Rec<L, S, NC, NS>;
  const long long N = a.N;
  const long long c = R::cell(a.slot[n]);
  if (fio) {
    for (int s = 0; s < NC; ++s) {
#pragma unroll
      for (int i = 0; i < L::Q; ++i) {
        double* io = fio + ((long long)s * L::Q + i) * N + n;
        if (!fluid) {
          if (dir == 0) *io = 0.0;
          continue;
        }
        S* p;
        if (parity == 0 || i == 0 || flow_wall<L>(m, L::opp(i)))
          p = R::f(a, c, s, i);
        else
          p = R::f(a, cell_of<R>(a, nb.at(-L::cx(i), -L::cy(i), -L::cz(i))), s, L::opp(i));
        const double sh = L::w(i) * double(k.rref[s]);
        if (dir == 0) *io = double(Store<S>::ld(p)) + sh;
        else Store<S>::st(p, T(*io - sh));
      }
    }
  }
  if (hio) {
    using SC = typename R::SC;
    for (int s = 0; s < NS; ++s) {
#pragma unroll
      for (int j = 0; j < L::QC; ++j) {
        double* io = hio + ((long long)s * L::QC + j) * N + n;
        if (!fluid) {
          if (dir == 0) *io = 0.0;
          continue;
        }
        SC* p;
        if (parity == 0 || j == 0 || MaskBits<L>::code(m, L::opp(j)) != 0u)
          p = R::h(a, c, s, j);
        else
          p = R::h(a, cell_of<R>(a, nb.at(-L::cx(j), -L::cy(j), -L::cz(j))), s, L::opp(j));
        const double sh = double(scal_w<T>(j, k)) * double(k.cref[s]);
        if (dir == 0) *io = double(Store<SC>::ld(p)) + sh;
        else Store<SC>::st(p, T(*io - sh));
      }
    }
  }
}

// ================================================================ link masks

// Neighbour of (x, y, z) in direction (dx, dy, dz) under per-axis periodicity: -1 if outside.
// *axis_out receives the first axis that left the box (0, 1, 2) or -1.
__device__ __forceinline__ long long nbr_checked(const Args& a, int x, int y, int z, int dx, int dy,
                                                 int dz, const int* per, int* axis_out) {
  int v[3] = {x + dx, y + dy, z + dz};
  const int n3[3] = {a.nx, a.ny, a.nz};
  *axis_out = -1;
  for (int c = 0; c < 3; ++c) {
    if (v[c] < 0 || v[c] >= n3[c]) {
      if (!per[c]) {
        *axis_out = c;
        return -1;
      }
      v[c] = v[c] < 0 ? v[c] + n3[c] : v[c] - n3[c];
    }
  }
  return v[0] + (long long)a.nx * (v[1] + (long long)a.ny * v[2]);
}

template <class L>
__device__ uint32_t compute_mask(const Args& a, int x, int y, int z) {
  const long long n = x + (long long)a.nx * (y + (long long)a.ny * z);
  if (a.flags[n] != FL_FLUID) return 0u;
  uint32_t m = 1u;
  int ax;
  for (int i = 1; i < L::Q; ++i) {
    const long long q = nbr_checked(a, x, y, z, L::cx(i), L::cy(i), L::cz(i), a.per, &ax);
    if (q < 0 || a.flags[q] != FL_FLUID) m |= 1u << i;
  }
  const int perc[3] = {a.open_x ? 0 : a.per[0], a.per[1], a.per[2]};
  for (int j = 1; j < L::QC; ++j) {
    const long long q = nbr_checked(a, x, y, z, L::cx(j), L::cy(j), L::cz(j), perc, &ax);
    uint32_t code;
    if (q < 0) code = (ax == 0 && a.open_x) ? 3u : 1u;
    else {
      const uint8_t fl = a.flags[q];
      code = fl == FL_FLUID ? 0u : (fl == FL_REACTIVE ? 2u : 1u);
    }
    m |= code << (MaskBits<L>::SC_BASE + 2 * (j - 1));
  }
  return m;
}

template <class L>
__global__ void __launch_bounds__(256) k_masks(const Args a) {
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (n >= a.N) return;
  const int x = int(n % a.nx);
  const int y = int((n / a.nx) % a.ny);
  const int z = int(n / ((long long)a.nx * a.ny));
  a.mask[n] = compute_mask<L>(a, x, y, z);
}

// ================================================================ node lists

// Ordered stream compaction of the nodes that satisfy a predicate, in chunks of 1024 positions:
// count, scan, write.  PRED 0: fluid nodes (the step kernel's work list), in brick order (below);
// also assigns the storage slots.  PRED 1: reactive solids touching the fluid through a scalar
// link (the dissolution interface list, node order; also marks listed[]).
//
// Brick order: the domain is cut into bricks of BX x BY x BZ nodes, visited x-fastest, with the
// nodes x-fastest inside a brick.  A warp's 32 consecutive list entries then lie in a compact
// block, so the neighbour cells an odd step reads and writes fall in a few nearby slot ranges
// instead of nine distant rows.
#ifndef LBM_BRICK_X
#define LBM_BRICK_X 32
#endif
#ifndef LBM_BRICK_Y
#define LBM_BRICK_Y 8
#endif
#ifndef LBM_BRICK_Z
#define LBM_BRICK_Z 4
#endif
template <class L>
struct Brick {
  static constexpr int X = LBM_BRICK_X, Y = LBM_BRICK_Y, Z = L::D == 3 ? LBM_BRICK_Z : 1;
  static constexpr long long V = (long long)X * Y * Z;
};

// node at position t of the brick order, or -1 for a position outside the domain
template <class L>
__device__ __forceinline__ long long brick_node(const Args& a, long long t) {
  using B = Brick<L>;
  const long long b = t / B::V;
  const int l = int(t - b * B::V);
  const long long nbx = (a.nx + B::X - 1) / B::X, nby = (a.ny + B::Y - 1) / B::Y;
  const long long x = (b % nbx) * B::X + l % B::X;
  const long long y = ((b / nbx) % nby) * B::Y + (l / B::X) % B::Y;
  const long long z = (b / (nbx * nby)) * B::Z + l / (B::X * B::Y);
  if (x >= a.nx || y >= a.ny || z >= a.nz) return -1;
  return x + a.nx * (y + a.ny * z);
}

template <class L>
__device__ __forceinline__ bool has_fluid_scalar_neighbour(const Args& a, int x, int y, int z);

// node of position t in the order of list PRED (-1: no node), and whether it enters the list
template <class L, int PRED>
__device__ __forceinline__ bool list_pred(const Args& a, long long t, long long* node) {
  const long long n = PRED == 0 ? brick_node<L>(a, t) : (t < a.N ? t : -1);
  *node = n;
  if (n < 0) return false;
  if (PRED == 0) return a.flags[n] == FL_FLUID;
  if (a.flags[n] != FL_REACTIVE) return false;
  return has_fluid_scalar_neighbour<L>(a, int(n % a.nx), int((n / a.nx) % a.ny),
                                       int(n / ((long long)a.nx * a.ny)));
}

__device__ __forceinline__ unsigned int block_count(unsigned int b, unsigned int* wsum) {
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = __popc(b);
  __syncthreads();
  unsigned int v = 0;
  if (threadIdx.x < 32) {
    v = wsum[threadIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  }
  __syncthreads();
  return v;
}

template <class L, int PRED>
__global__ void __launch_bounds__(1024) k_list_count(const Args a) {
  __shared__ unsigned int wsum[32];
  const long long t = blockIdx.x * 1024ll + threadIdx.x;
  long long n;
  const bool f = list_pred<L, PRED>(a, t, &n);
  const unsigned int cf = block_count(__ballot_sync(0xffffffffu, f), wsum);
  if (threadIdx.x == 0) a.block_counts[blockIdx.x] = cf;
  if (PRED == 0) {
    const unsigned int cv = block_count(__ballot_sync(0xffffffffu, n >= 0), wsum);
    if (threadIdx.x == 0) a.block_counts_v[blockIdx.x] = cv;
  }
}

// exclusive scan of the chunk counts by one block; the total goes to count[0] and count[1]
template <int DUMMY = 0>
__global__ void __launch_bounds__(1024) k_list_scan(unsigned int* counts, unsigned int nchunks,
                                                    unsigned int* count) {
  __shared__ unsigned int part[1024];
  __shared__ unsigned int carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (unsigned int base = 0; base < nchunks; base += 1024) {
    const unsigned int i = base + threadIdx.x;
    const unsigned int v = i < nchunks ? counts[i] : 0u;
    part[threadIdx.x] = v;
    __syncthreads();
    for (unsigned int o = 1; o < 1024; o <<= 1) {
      const unsigned int t = threadIdx.x >= o ? part[threadIdx.x - o] : 0u;
      __syncthreads();
      part[threadIdx.x] += t;
      __syncthreads();
    }
    if (i < nchunks) counts[i] = carry + part[threadIdx.x] - v;
    __syncthreads();
    if (threadIdx.x == 1023) carry += part[1023];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    count[0] = carry;
    count[1] = carry;
  }
}

// exclusive prefix of ballot b over the block (chunk offset off added)
__device__ __forceinline__ unsigned int block_prefix(unsigned int b, unsigned int off, unsigned int* wsum) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) wsum[wid] = __popc(b);
  __syncthreads();
  if (threadIdx.x < 32) {
    unsigned int v = wsum[threadIdx.x], incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (threadIdx.x >= o) incl += t;
    }
    wsum[threadIdx.x] = incl - v;
  }
  __syncthreads();
  const unsigned int pos = off + wsum[wid] + __popc(b & ((1u << lane) - 1u));
  __syncthreads();
  return pos;
}

// PRED 0 also assigns the new storage slots: fluid nodes take their list position, solid nodes
// follow the fluid total in brick order (slot_new), and the offsets that go with them (off; rec
// bytes per tile of `tile` slots, elem per flow element).
template <class L, int PRED>
__global__ void __launch_bounds__(1024) k_list_write(const Args a, uint32_t* list, const uint32_t rec, const uint32_t tile, const uint32_t elem) {
  __shared__ unsigned int wsum[32];
  const long long t = blockIdx.x * 1024ll + threadIdx.x;
  long long n;
  const bool f = list_pred<L, PRED>(a, t, &n);
  const unsigned int pos = block_prefix(__ballot_sync(0xffffffffu, f), a.block_counts[blockIdx.x], wsum);
  if (PRED == 0) {
    const unsigned int vpos = block_prefix(__ballot_sync(0xffffffffu, n >= 0), a.block_counts_v[blockIdx.x], wsum);
    if (n >= 0) {
      const unsigned int sl = f ? pos : a.fluid_count[0] + (vpos - pos);
      a.slot_new[n] = sl;
      const unsigned long long o = (unsigned long long)(sl / tile) * rec + (sl % tile + kOffBias * tile) * elem;
      if (a.off_ok) a.off[n] = (uint32_t)o;
      else a.off64[n] = o;
    }
  }
  if (f) {
    list[pos] = PRED == 0 ? list_entry<L>(a, int(n), int(n % a.nx), int((n / a.nx) % a.ny), int(n / ((long long)a.nx * a.ny)))
                          : (uint32_t)n;
    if (PRED == 1) a.listed[n] = 1;
  }
}

// ================================================================ interface list

template <class L>
__device__ __forceinline__ bool has_fluid_scalar_neighbour(const Args& a, int x, int y, int z) {
  const int perc[3] = {a.open_x ? 0 : a.per[0], a.per[1], a.per[2]};
  int ax;
  for (int j = 1; j < L::QC; ++j) {
    const long long q = nbr_checked(a, x, y, z, L::cx(j), L::cy(j), L::cz(j), perc, &ax);
    if (q >= 0 && a.flags[q] == FL_FLUID) return true;
  }
  return false;
}

__device__ __forceinline__ void push_iface(const Args& a, long long n) {
  const unsigned int e = atomicAdd(a.iface_count, 1u);
  if (e < a.N) a.iface_list[e] = (uint32_t)n;
  else atomicOr(a.err, ERR_CAPACITY);
}

// ================================================================ geometry flips

__device__ __forceinline__ bool cas_flag(uint8_t* flags, long long n, uint8_t expect, uint8_t desired,
                                         int* err) {
  unsigned int* w = reinterpret_cast<unsigned int*>(flags + (n & ~3ll));
  const int sh = int(n & 3) * 8;
  unsigned int old = atomicAdd(w, 0u);
  for (int it = 0; it < 64; ++it) {
    if (((old >> sh) & 0xffu) != expect) return false;
    const unsigned int nw = (old & ~(0xffu << sh)) | (unsigned(desired) << sh);
    const unsigned int prev = atomicCAS(w, old, nw);
    if (prev == old) return true;
    old = prev;
  }
  atomicOr(err, ERR_CAS);
  return false;
}

// FLIPPING (0b11) -> v in {FLUID 0b00, SOLID 0b01, REACTIVE 0b10} with one atomic operation,
// so a concurrent reader never sees an intermediate value.
__device__ __forceinline__ void leave_flipping(uint8_t* flags, long long n, uint8_t v) {
  unsigned int* w = reinterpret_cast<unsigned int*>(flags + (n & ~3ll));
  const int sh = int(n & 3) * 8;
  atomicAnd(w, ~((3u ^ unsigned(v)) << sh));
}

__device__ __forceinline__ void coords_of(const Args& a, long long n, int* x, int* y, int* z) {
  *x = int(n % a.nx);
  *y = int((n / a.nx) % a.ny);
  *z = int(n / ((long long)a.nx * a.ny));
}

// The flip list in phases separated by barriers of one cluster of kFlipBlocks blocks, a warp per entry with
// its lanes over the neighbours or directions (a warp keeps its entries through all phases):
//   0 claim entries (validate, mark FLIPPING, drop duplicates)
//   1 dissolution: neighbour means (flags before the flip);  deposition: removed sums
//   2 write populations of the new fluid nodes / hand populations to remaining neighbours
//   3 final flags;  4 link masks of every node around a flipped one;  5 clear the list
// parity_next is the layout parity of the state the flips act on (steps completed & 1).
// What bounds it is the chain of dependent loads of an entry: flag, slot and mask of 18 neighbours, their
// populations, then the 18 flags around each of them.  One block with a thread per entry took longer than the step
// once a few hundred nodes flipped together (64^3 FP64 dissolution: 2.4 ms for ten steps, 1.3 ms with the cluster
// and all); an update without flips takes 2 us.
constexpr int kFlipBlocks = 8, kFlipThreads = 512;
__device__ __forceinline__ void cluster_barrier() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
template <class L, class S, int NC, int NS>
__global__ void __cluster_dims__(kFlipBlocks, 1, 1) __launch_bounds__(kFlipThreads)
    k_flip(const Args a, const Coef<typename Store<S>::T> k, const int parity_next) {
  using T = typename Store<S>::T;
  using R = Rec<L, S, NC, NS>;
  using SC = typename R::SC;   // scalar lattices' storage
  constexpr int Q = L::Q, QC = L::QC;
  pdl_trigger();
  pdl_wait();
  const unsigned int cnt_raw = *a.flip_count;
  const unsigned int cnt = cnt_raw < a.flip_cap ? cnt_raw : a.flip_cap;
  if (cnt == 0) return;   // the same in every block: nothing writes the count before the last barrier
  const int lane = threadIdx.x & 31;
  const unsigned int first = (blockIdx.x * kFlipThreads + threadIdx.x) >> 5, step = kFlipBlocks * kFlipThreads / 32;
  const int percf[3] = {a.per[0], a.per[1], a.per[2]};
  const int percs[3] = {a.open_x ? 0 : a.per[0], a.per[1], a.per[2]};
  const bool dissolve = a.geo_mode == GEO_DISSOLVE;
  // flip monitors: injected mass [0, 2), injected scalars [2, 5), removed mass [5, 7), removed
  // scalars [7, 10), solid temperature taken from the solid lattice [10]
  __shared__ double sred[11];
  if (threadIdx.x < 11) sred[threadIdx.x] = 0.0;
  // ---- phase 0: claim
  for (unsigned int e = first; e < cnt; e += step) {
    const long long s = a.flip_list[e];
    bool ok = false;
    if (lane == 0) {
      if (dissolve)
        ok = a.flags[s] == FL_REACTIVE && consumed(a, a.acc[s]) &&
             cas_flag(a.flags, s, FL_REACTIVE, FL_FLIPPING, a.err);
      else
        ok = a.flags[s] == FL_FLUID && a.acc[s] > 1.0 && cas_flag(a.flags, s, FL_FLUID, FL_FLIPPING, a.err);
      if (!ok) a.flip_list[e] = 0xffffffffu;
    }
    __syncwarp();
  }
  __syncthreads();
  cluster_barrier();
  // ---- phase 1
  for (unsigned int e = first; e < cnt; e += step) {
    if (a.flip_list[e] == 0xffffffffu) continue;
    const long long s = a.flip_list[e];
    int x, y, z;
    coords_of(a, s, &x, &y, &z);
    if (dissolve) {
      // lane i - 1: neighbour i
      double sr[NC] = {}, sc[NS > 0 ? NS : 1] = {};
      bool fluid = false;
      int ax;
      const int i = lane + 1;
      if (i < Q) {
        const long long q = nbr_checked(a, x, y, z, L::cx(i), L::cy(i), L::cz(i), percf, &ax);
        fluid = q >= 0 && a.flags[q] == FL_FLUID;
        if (fluid) {
          const Nbr nq = nbr_of(a, int(q));
          const uint32_t mq = a.mask[q];
          const long long cq = R::cell(a.slot[q]);
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            T f[Q];
            gather_flow<L, S, NC, NS>(a, c, cq, mq, nq, parity_next, f);
            double r = double(k.rref[c]);
#pragma unroll
            for (int j = 0; j < Q; ++j) r += double(f[j]);
            sr[c] = r;
          }
          T hh[NS > 0 ? NS : 1][QC];
#pragma unroll
          for (int c = 0; c < NS; ++c) gather_scal<L, S, NC, NS>(a, c, cq, mq, nq, parity_next, hh[c]);
          T rl[QC], gain = T(0);
#pragma unroll
          for (int j = 0; j < QC; ++j) rl[j] = T(0);
          if (NS > 1 && a.conjugate)
            close_conjugate<L, T>(hh[0], hh[NS > 1 ? 1 : 0], mq, k, a, nq,
                                  reinterpret_cast<const T*>(a.gs[parity_next]), [&](int j, T r, T) { rl[j] = r; });
          else if (NS > 1 && a.arrhenius)
            close_thermal<L, T>(hh[0], hh[NS > 1 ? 1 : 0], mq, k, a.n_it, [&](int j, T r, T, T) { rl[j] = r; });
          else if (NS > 0)
            close_scalar<L, T>(hh[0], mq, k, [&](int j, T Cb, T) { rl[j] = k.kr * Cb; });
          if (NS > 1 && a.product) close_product<L, T>(hh[NS - 1], mq, k, rl, gain);
#pragma unroll
          for (int c = 0; c < NS; ++c) {
            double C = double(k.cref[c]);
#pragma unroll
            for (int j = 0; j < QC; ++j) C += double(hh[c][j]);
            sc[c] = C;
          }
        }
      }
      const int count = __popc(__ballot_sync(0xffffffffu, fluid));
      if (count == 0) {   // nothing to average: stays solid
        if (lane == 0) {
          leave_flipping(a.flags, s, FL_REACTIVE);
          a.flip_list[e] = 0xffffffffu;
        }
        __syncwarp();
        continue;
      }
      double* sc4 = a.flip_scratch + 5ll * e;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const double r = warp_sum(sr[c]);
        if (lane == 0) sc4[c] = r / count;
      }
#pragma unroll
      for (int c = 0; c < NS; ++c) {
        const double r = warp_sum(sc[c]);
        if (lane == 0) sc4[2 + c] = r / count;
      }
      __syncwarp();
    } else if (lane == 0) {
      const Nbr ns = nbr_of(a, int(s));
      const uint32_t ms = a.mask[s];
      const long long cs = R::cell(a.slot[s]);
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        T f[Q];
        gather_flow<L, S, NC, NS>(a, c, cs, ms, ns, parity_next, f);
        double r = double(k.rref[c]);
#pragma unroll
        for (int j = 0; j < Q; ++j) r += double(f[j]);
        atomicAdd(&sred[5 + c], r);
      }
#pragma unroll
      for (int c = 0; c < NS; ++c) {
        T h[QC];
        gather_scal<L, S, NC, NS>(a, c, cs, ms, ns, parity_next, h);
        double C = double(k.cref[c]);
#pragma unroll
        for (int j = 0; j < QC; ++j) C += double(h[j]);
        atomicAdd(&sred[7 + c], C);
      }
    }
  }
  cluster_barrier();
  // ---- phase 2: lane j moves or sets the population of direction j
  for (unsigned int e = first; e < cnt; e += step) {
    if (a.flip_list[e] == 0xffffffffu) continue;
    const long long s = a.flip_list[e];
    const long long ss = R::cell(a.slot[s]);   // cells of the flipping node
    int x, y, z, ax;
    coords_of(a, s, &x, &y, &z);
    const int j = lane;
    // where direction j of the node comes from: a node (flow and scalar periodicity) or a face
    long long srcf = -1, srcs = -1;
    if (j < Q) {
      const int d = dissolve ? -1 : 1;
      srcf = nbr_checked(a, x, y, z, d * L::cx(j), d * L::cy(j), d * L::cz(j), percf, &ax);
      if (j < QC) srcs = nbr_checked(a, x, y, z, d * L::cx(j), d * L::cy(j), d * L::cz(j), percs, &ax);
    }
    const uint8_t flf = srcf < 0 ? FL_SOLID : a.flags[srcf], fls = srcs < 0 ? FL_SOLID : a.flags[srcs];
    const int o = j < Q ? L::opp(j) : 0;
    if (dissolve) {
      const double* sc4 = a.flip_scratch + 5ll * e;
      for (int c = 0; c < NC; ++c) {
        const double r = sc4[c];
        if (lane == 0) atomicAdd(&sred[c], r);
        if (j >= Q) continue;
        const T tv = T(L::w(j) * (r - double(k.rref[c])));   // f_eq(rho_bar, u = 0) - w rref
        if (parity_next == 0 || j == 0) {
          Store<S>::st(R::f(a, ss, c, j), tv);
        } else if (flf == FL_FLUID) {
          S* from = R::f(a, R::cell(a.slot[srcf]), c, o);
          *R::f(a, ss, c, j) = *from;     // neighbour's bounced value moves
          Store<S>::st(from, tv);
        } else if (flf == FL_FLIPPING) {
          Store<S>::st(R::f(a, R::cell(a.slot[srcf]), c, o), tv);
        } else {
          Store<S>::st(R::f(a, ss, c, j), tv);
        }
      }
      for (int c = 0; c < NS; ++c) {
        double C = sc4[2 + c];
        if (c == 1 && a.conjugate) {
          // with conduction in the solid the new fluid node keeps its own temperature: its solid
          // populations leave the solid lattice
          T* g = reinterpret_cast<T*>(a.gs[parity_next]);
          double own = 0.0;
          if (j < QC) {
            own = double(g[(long long)j * a.N + s]);
            g[(long long)j * a.N + s] = T(0);
          }
          C = warp_sum(own);
          if (lane == 0) atomicAdd(&sred[10], C);
        }
        if (lane == 0) atomicAdd(&sred[2 + c], C);
        if (j >= QC) continue;
        const double wj = double(scal_w<T>(j, k));
        const T tv = T(wj * (C - double(k.cref[c])));       // h_eq(C_bar, u = 0) - w cref
        if (parity_next == 0 || j == 0) {
          Store<SC>::st(R::h(a, ss, c, j), tv);
        } else if (fls == FL_FLUID) {
          SC* from = R::h(a, R::cell(a.slot[srcs]), c, o);
          *R::h(a, ss, c, j) = *from;
          Store<SC>::st(from, tv);
        } else if (fls == FL_FLIPPING) {
          Store<SC>::st(R::h(a, R::cell(a.slot[srcs]), c, o), tv);
        } else {
          Store<SC>::st(R::h(a, ss, c, j), tv);
        }
      }
    } else if (parity_next == 1 && j > 0) {
      // deposition in the swapped layout: a remaining fluid neighbour y = s + c_d now reads its
      // population from the new wall at (y, d); give it what s streamed toward it, (s, opp d)
      if (j < Q && srcf >= 0 && flf == FL_FLUID)
        for (int c = 0; c < NC; ++c) *R::f(a, R::cell(a.slot[srcf]), c, j) = *R::f(a, ss, c, o);
      if (j < QC && srcs >= 0 && fls == FL_FLUID)
        for (int c = 0; c < NS; ++c) *R::h(a, R::cell(a.slot[srcs]), c, j) = *R::h(a, ss, c, o);
    }
    __syncwarp();
  }
  cluster_barrier();
  // ---- phase 3: final flags; new fluid nodes join the fluid list (removed ones are skipped by
  // their mask until the next rebuild)
  for (unsigned int e = first; e < cnt; e += step) {
    if (a.flip_list[e] == 0xffffffffu || lane != 0) continue;
    leave_flipping(a.flags, a.flip_list[e], dissolve ? FL_FLUID : FL_SOLID);
    if (dissolve) {
      const unsigned int pos = atomicAdd(a.fluid_count, 1u);
      int x, y, z;
      coords_of(a, a.flip_list[e], &x, &y, &z);
      if (pos < a.N) a.fluid_list[pos] = list_entry<L>(a, int(a.flip_list[e]), x, y, z);
      else atomicOr(a.err, ERR_CAPACITY);
    }
  }
  __syncwarp();
  cluster_barrier();
  // ---- phase 4: masks around every flipped node, lane i: neighbour i (lane 0: the node itself)
  for (unsigned int e = first; e < cnt; e += step) {
    if (a.flip_list[e] == 0xffffffffu) continue;
    const long long s = a.flip_list[e];
    int x, y, z, ax;
    coords_of(a, s, &x, &y, &z);
    if (lane < Q) {
      const long long q = lane == 0 ? s : nbr_checked(a, x, y, z, L::cx(lane), L::cy(lane), L::cz(lane), percf, &ax);
      if (q >= 0) {
        int qx, qy, qz;
        coords_of(a, q, &qx, &qy, &qz);
        a.mask[q] = compute_mask<L>(a, qx, qy, qz);
      }
    }
    if (dissolve && lane > 0 && lane < QC) {
      // reactive solids that now touch the new fluid node join the interface list
      const long long q = nbr_checked(a, x, y, z, L::cx(lane), L::cy(lane), L::cz(lane), percs, &ax);
      if (q >= 0 && a.flags[q] == FL_REACTIVE && cas_flag(a.listed, q, 0, 1, a.err)) push_iface(a, q);
    }
    __syncwarp();
  }
  __syncthreads();
  if (threadIdx.x < 11 && sred[threadIdx.x] != 0.0) atomicAdd(a.flip_mon + threadIdx.x, sred[threadIdx.x]);
  if (blockIdx.x == 0 && threadIdx.x == 0) *a.flip_count = 0u;
}

// ================================================================ conduction in the solid

// Solid thermal lattice (Sec. 2.1.5, Eq. therpop_solid with g_s^eq = w T_s, Eq. macroreacb_solid):
// collision and streaming of every solid node, from gs[parity] into gs[parity ^ 1] (node-indexed
// planes, full values).  A population leaving toward another solid node streams there; one
// leaving toward a fluid node or through a face that is not periodic for the scalars is kept at
// the node as the arriving population of the opposite direction: at a closed face that is the
// reflection, at a fluid neighbour it is the solid side of the link that k_exchange replaces.
template <class L, class S>
__device__ __forceinline__ void solid_nodes(const Args& a, const Coef<typename Store<S>::T>& k, const int parity, const unsigned int block,
                            const unsigned int blocks) {
  using T = typename Store<S>::T;
  constexpr int QC = L::QC;
  const T* gin = reinterpret_cast<const T*>(a.gs[parity]);
  T* gout = reinterpret_cast<T*>(a.gs[parity ^ 1]);
  const int perc[3] = {a.open_x ? 0 : a.per[0], a.per[1], a.per[2]};
  const long long N = a.N;
  for (long long n = block * (long long)blockDim.x + threadIdx.x; n < N; n += (long long)blocks * blockDim.x) {
    if (a.flags[n] == FL_FLUID) continue;
    T g[QC];
    T Ts = T(0);
#pragma unroll
    for (int q = 0; q < QC; ++q) {
      g[q] = gin[(long long)q * N + n];
      Ts += g[q];
    }
    int x, y, z, ax;
    coords_of(a, n, &x, &y, &z);
#pragma unroll
    for (int q = 0; q < QC; ++q) {
      const T v = g[q] - (g[q] - scal_w<T>(q, k) * Ts) * k.oms;
      if (q == 0) {
        gout[n] = v;
        continue;
      }
      const long long d = nbr_checked(a, x, y, z, L::cx(q), L::cy(q), L::cz(q), perc, &ax);
      if (d >= 0 && a.flags[d] != FL_FLUID) gout[(long long)q * N + d] = v;
      else gout[(long long)L::opp(q) * N + n] = v;
    }
  }
}

// The exchange across every solid link of the temperature (Sec. 2.1.5, Eq. tempCon, fluxCon,
// reacRate), after the fluid step and the solid lattice's streaming.  For fluid node n and a
// direction j toward a solid node s = n + c_j (arriving direction i = opp(j)): the fluid
// population ho = h*_T,j that left n toward s (kept at n by the bounce-back of the step, in plane
// i) and the solid population go = g*_s,i that left s toward n (kept at s in plane j by solid_nodes)
// meet at one interface temperature T_b.  Each side receives 2 w T_b minus what it sent, and the
// link's energy in units of the fluid's rho c_p grows by the reaction heat Qp:
//     T_b = (c_fs ho + go + c_fs Qp / 2) / (w (c_fs + 1)).
// Qp = h_r k(T_b) C_b at a reactive link, where C_b = 2 hb / (2 w + k tau_c / (tau_c - 1/2)) closes
// the species population hb = h_C,j that has just streamed into n (read as the next step's
// gather reads it); T_b and C_b come from n_it + 1 fixed-point updates starting at the value
// without reaction, and k is kept for the next step's species closure.  The updates end early once T_b repeats: a
// fixed point of the rounded arithmetic, so the result is that of all of them.  Monitors: heat gained by
// the fluid side (bank HEAT), by the solid side (HEAT_S), reaction heat (HEAT_SRC).
template <class L, class S, int NC, int NS>
__global__ void __launch_bounds__(256) k_exchange(const Args a, const Coef<typename Store<S>::T> k,
                                                  const int parity_next) {
  using T = typename Store<S>::T;
  using R = Rec<L, S, NC, NS>;
  using SC = typename R::SC;
  constexpr int QC = L::QC;
  pdl_trigger();
  pdl_wait();
  T* g = reinterpret_cast<T*>(a.gs[parity_next]);
  T* kb = reinterpret_cast<T*>(a.kb);
  const int perc[3] = {a.open_x ? 0 : a.per[0], a.per[1], a.per[2]};
  const T sh0 = k.wca * k.cref[0], sh1 = k.wca * k.cref[1];
  const T w = k.wca, cf = k.cfs;
  const T den = w * (cf + T(1));
  T heat = T(0), heat_s = T(0), src_q = T(0);
  const unsigned int count = a.fluid_count[0], base = a.fluid_count[1];
  // one thread per link: the links of a node are independent, and the chain of a link (its iterations) is long
  constexpr unsigned int LN = QC <= 5 ? 4 : 8;   // threads per node (two of eight idle in 3D)
  const unsigned int j1 = threadIdx.x % LN;
  const int j = int(j1) + 1;
  for (unsigned int e = (blockIdx.x * blockDim.x + threadIdx.x) / LN; e < count; e += gridDim.x * blockDim.x / LN) {
    if (j >= QC) continue;
    const uint32_t wd = a.fluid_list[e];
    const int n = list_node(a, wd);
    const uint32_t m = a.mask[n];
    if (!(m & 1u)) continue;
    const uint32_t c = MaskBits<L>::code(m, j);
    if (c != 1u && c != 2u) continue;
    const int i = L::opp(j);
    int x, y, z, ax;
    coords_of(a, n, &x, &y, &z);
    const long long s = nbr_checked(a, x, y, z, L::cx(j), L::cy(j), L::cz(j), perc, &ax);
    if (s < 0) continue;   // a closed face: plain bounce-back
    const long long cell = R::cell(e < base ? (long long)e : (long long)a.slot[n]);
    SC* hp = R::h(a, cell, 1, i);
    T* gp = g + (long long)j * a.N + s;
    const T ho = Store<SC>::ld(hp) + sh1;
    const T go = *gp;
    T Tb = (cf * ho + go) / den;
    T Qp = T(0);
    if (c == 2u) {
      // the species population moving toward the wall, where the next step gathers it
      const SC* bp;
      if (parity_next == 0 || MaskBits<L>::code(m, i) != 0u)
        bp = R::h(a, cell, 0, j);
      else
        bp = R::h(a, cell_of<R>(a, nbr_entry(a, n, wd).at(-L::cx(j), -L::cy(j), -L::cz(j))), 0, i);
      const T hb = Store<SC>::ld(bp) + sh0;
      T kt = T(0);
      for (int it = 0; it <= a.n_it; ++it) {
        const T was = Tb;
        kt = k.arrA * exp(-k.arrTa / Tb);
        const T Cb = T(2) * hb / (T(2) * w + kt * k.fc);
        Qp = k.hr * kt * Cb;
        Tb = (cf * ho + go + T(0.5) * cf * Qp) / den;
        if (Tb == was) break;   // every further iteration would repeat this one
      }
      kb[(long long)(i - 1) * a.N + n] = kt;
    }
    const T hn = T(2) * w * Tb - ho;
    const T gn = T(2) * w * Tb - go;
    Store<SC>::st(hp, hn - sh1);
    *gp = gn;
    heat += hn - ho;
    heat_s += gn - go;
    src_q += Qp;
  }
  __syncwarp();
  const int lane_slot = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) % WALLX_SLOTS;
  const T vals[3] = {heat, heat_s, src_q};
  const int banks[3] = {BANK_HEAT, BANK_HEAT_S, BANK_HEAT_SRC};
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    if (__ballot_sync(0xffffffffu, vals[b] != T(0))) {
      const T v = warp_sum(vals[b]);
      if ((threadIdx.x & 31) == 0) atomicAdd(a.wallx_slot + banks[b] * WALLX_SLOTS + lane_slot, widen(v));
    }
  }
}

// The solid thermal lattice at rest equilibrium with the temperature given for each solid node
// (row 1 of the staged scalar fields): g_q = w_q T into gs[0]; gs[1] and the exchange's rate
// constants cleared (NaN: no exchange yet).
template <class L, class S>
__global__ void __launch_bounds__(256) k_solid_init(const Args a, const Coef<typename Store<S>::T> k) {
  using T = typename Store<S>::T;
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (n >= a.N) return;
  T* g0 = reinterpret_cast<T*>(a.gs[0]);
  T* g1 = reinterpret_cast<T*>(a.gs[1]);
  T* kb = reinterpret_cast<T*>(a.kb);
  const bool solid = a.flags[n] != FL_FLUID;
  const double Tn = a.d_C[a.N + n];
#pragma unroll
  for (int q = 0; q < L::QC; ++q) {
    g0[(long long)q * a.N + n] = solid ? T(double(scal_w<T>(q, k)) * Tn) : T(0);
    g1[(long long)q * a.N + n] = T(0);
    if (q > 0) kb[(long long)(q - 1) * a.N + n] = T(NAN);
  }
}

}  // namespace lbm
