// bl_internal.cuh -- device-side definitions shared by the library's kernels.
//
// The method is the coupled step of arXiv:1005.2594 (Sec. II, III); this file
// holds only lattice constants, the views passed to kernels and small device
// helpers.  Nothing here is shared with the CPU oracle.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>
#include <utility>

namespace bl {

constexpr int Q = 19;
constexpr int FLUID = -1;
constexpr int NWALL = 8;

// D3Q19 in the interface order (Sec. II): rest, 6 axis vectors, 12 diagonals,
// each followed by its opposite.  m = 36 alpha (alpha = 1/3, 1/18, 1/36).
struct D3Q19 {
  static __host__ __device__ constexpr int cx(int r) {
    return (r == 1 || r == 7 || r == 9 || r == 11 || r == 13) ? 1 : ((r == 2 || r == 8 || r == 10 || r == 12 || r == 14) ? -1 : 0);
  }
  static __host__ __device__ constexpr int cy(int r) {
    return (r == 3 || r == 7 || r == 10 || r == 15 || r == 17) ? 1 : ((r == 4 || r == 8 || r == 9 || r == 16 || r == 18) ? -1 : 0);
  }
  static __host__ __device__ constexpr int cz(int r) {
    return (r == 5 || r == 11 || r == 14 || r == 15 || r == 18) ? 1 : ((r == 6 || r == 12 || r == 13 || r == 16 || r == 17) ? -1 : 0);
  }
  static __host__ __device__ constexpr int opp(int r) { return r == 0 ? 0 : ((r & 1) ? r + 1 : r - 1); }
  static __host__ __device__ constexpr int m(int r) { return r == 0 ? 12 : (r <= 6 ? 2 : 1); }
};

// compile-time loop: f(std::integral_constant<int, I>) for I in [B, E)
template <int B, int E, class F>
__device__ __forceinline__ void sfor(F &&f) {
  if constexpr (B < E) {
    f(std::integral_constant<int, B>{});
    sfor<B + 1, E>(f);
  }
}

// storage of the shifted populations f~ = f - alpha rho_bar
template <class S>
struct Store;
template <>
struct Store<float> {
  static __device__ __forceinline__ float ld(const float *p) { return *p; }
  static __device__ __forceinline__ void st(float *p, float v) { *p = v; }
};
template <>
struct Store<__nv_bfloat16> {
  static __device__ __forceinline__ float ld(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
  static __device__ __forceinline__ void st(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }
};
// FP16 stores f~ scaled by 2^10 so that small deviations stay in the normal range
template <>
struct Store<__half> {
  static __device__ __forceinline__ float ld(const __half *p) { return __half2float(*p) * (1.0f / 1024.0f); }
  static __device__ __forceinline__ void st(__half *p, float v) { *p = __float2half_rn(v * 1024.0f); }
};

// division by a lattice extent through a multiply-high: with
// m = floor((2^64 - 1) / d) + 1, floor(n / d) is the high 64 bits of n m for
// every 32-bit n and 2 <= d < 2^32 (m = floor(2^64 / d) + 1, or 2^64 / d when
// d divides 2^64; the error of n m / 2^64 against n / d is below n / 2^64 <
// 2^-32 <= 1 / d, and frac(n / d) <= 1 - 1 / d); d = 1 is passed through
struct FastDiv {
  unsigned long long m;
  unsigned d;
};
inline FastDiv make_fastdiv(unsigned d) {
  FastDiv f;
  f.d = d;
  f.m = d > 1u ? ~0ull / d + 1ull : 0ull;
  return f;
}
__device__ __forceinline__ unsigned fdiv(unsigned n, const FastDiv &f) {
  return f.d == 1u ? n : (unsigned)__umul64hi((unsigned long long)n, f.m);
}

struct LatticeView {
  int nx, ny, nz;
  int per[3];
  unsigned N;  // nodes; 19 N < 2^32 is checked on the host
  FastDiv dnx, dnxy;  // division by nx and by nx ny (node index -> coordinates)
  float wall_vel[NWALL][3];
  float omega;  // 1 / tau
  float rho0;
  float g[3];
  int has_force;
  int sweep;  // sweep variant (0 one node per thread, 1 / 2 FP32 pipeline over 4 / 8 planes,
             // 3 / 4 bulk-copy pipeline over 8 / 4 planes, 5 persistent bulk-copy rows)
  int rows_grid[8];  // grid of the persistent row sweep per (parity, force, tau = 1)
  void *pop;       // 19 x N storage elements, slot r of node n at r * N + n
  int32_t *owner;  // N
  uint32_t *nbm;   // N neighbour words of the current owner map (NB_* bits), written by the geometry pass
  uint32_t *nbc;   // N neighbour-cell words (NBC_*), written with the neighbour words
  uint4 *nbx;      // N mixed words (NBX_*): read for nodes between a cell and another cell or a wall (null without cells)
  // Cell links of the sweep.  A fluid node next to a cell writes one link
  // record per cell into that cell's bucket, for the link-momentum sums.
  // The moving-boundary term C of its bounced populations needs the cell's
  // velocity of the half step, solved after the sweep: after the solve, the
  // node's record of its first cell becomes pu[n] = (rho (V + W x d), mask of
  // the bounced directions as the bits of .w), which the next sweep reads
  // with the populations and adds as C = -(m_r / 6) c_r . u; the links to a
  // second or third cell of one node get C in place right after the solve.
  float4 *pu;              // N
  float4 *rec;             // ncells x 2 x rec_cap: the first, then the second float4 of a cell's records
  int *rec_count;          // ncells
  int rec_cap;
  int *status;
  // Lees-Edwards shear (null when off): the sweep leaves (drho, u) of the
  // nodes at x = 0 (first ny nz) and x = nx - 1 (next ny nz), y + ny z
  float4 *le_mom;
  int dep;  // host: launch programmatic dependents
};

// Lees-Edwards shear across the plane between x = nx - 1 and x = 0 (Sec. IV,
// reading Q25): the image above moves with velocity offset U along z and is
// displaced by U t
struct LeView {
  double U;
  float4 *D;     // offset of the pass in flight, written by the gather, read by the scatter: floor(D), D - floor(D)
                 // and the same of -D (whole parts as the bits of .x, .z)
  long long *t;  // steps since the shear was set
  double *P;     // z-momentum moved along +x across the plane, summed over the steps
  long long *n;  // steps summed
  float *T;      // 2 x 5 x ny nz crossing populations of the two planes, shifted to the other frame
};

// A link record (two float4): node n (bits of .x), direction mask (bits of
// .y: bit r = the neighbour n + c_r belongs to the cell; bit 31 marks the
// links of a node's second or third cell, whose C is given in place right
// after the solve), the density deviation drho = rho - rho_bar (.z), then
// at tau = 1 the node's velocity u (.w, second .x, .y), uu (second .z) and
// u . F (second .w), from which the link sums rebuild the bounced
// populations; at any other tau the sum over the mask of 2 f~*_r c_r (.w,
// second .x, .y).
constexpr uint32_t REC_DIRECT = 1u << 31;

// neighbour word of a node: bit 0 the node is fluid; bit r (1..18) the
// neighbour x + c_r is solid; NB_WALL some solid neighbour is a wall node;
// NB_CELL some solid neighbour is a cell node.  For a cell node (bit 0
// clear) bit r marks a contact link: the neighbour x + c_r is a wall node or
// a node of another cell.  Zero for wall nodes.
constexpr uint32_t NB_FLUID = 1u;
constexpr uint32_t NB_SOLID = 0x7FFFEu;
constexpr uint32_t NB_WALL = 1u << 19;
constexpr uint32_t NB_CELL = 1u << 20;
// neighbour-cell word of a fluid node next to a cell: the index of the cell
// owning its first solid neighbour in direction order (low bits), and
// NBC_MIXED when not every solid neighbour belongs to that cell (a wall or a
// second cell among them: the sweep then reads the neighbours' owners)
constexpr uint32_t NBC_MIXED = 1u << 31;
constexpr uint32_t NBC_CELL = 0x7FFFFFFFu;
// mixed word of a fluid node with NB_CELL and NBC_MIXED: .x the first cell in
// direction order and, shifted by 16, the second one (NBX_NONE: none; a
// context holds at most 65535 cells), .y and .z the neighbours (bits 1..18)
// each of them owns, .w those that are walls; what is left of the solid
// neighbours belongs to a third cell
constexpr uint32_t NBX_NONE = 0xFFFFu;

// momentum given to each wall id by its bounce-back links: variable part in
// FP64, constant part 2 alpha_r rho_bar c_r as exact integer sums of m_r c_r.
// WALL_COPIES sets of sums, a block adding to one of them: every warp beside a
// wall adds to its wall's six words, and on one set those additions stood in
// line at one L2 slice (about 85 us of the even step of a 2.2 M node vessel
// loop, 223 -> 61 us with these sets and the row index).  The read-out adds the
// sets up (launch_wall_read).
constexpr int WALL_COPIES = 128;
constexpr int WALL_SUMS = NWALL * 3;
struct WallAcc {
  double *F;     // WALL_COPIES x 8 x 3
  long long *K;  // WALL_COPIES x 8 x 3
};

// the set of sums this block adds to
__device__ __forceinline__ WallAcc wall_copy(const WallAcc &wa) {
  const unsigned c = (blockIdx.x + 31u * blockIdx.y + 57u * blockIdx.z) % (unsigned)WALL_COPIES;
  return WallAcc{wa.F + c * WALL_SUMS, wa.K + c * WALL_SUMS};
}

// Cells.  Their bounce links come from the sweep's link records
// (LatticeView::rec); contact links enter as exact integer sums cK, cIT.
struct PartView {
  int n;
  double *X, *q, *V, *L, *Om;
  double *o;         // exact FP64 symmetry axis of the current q, n x 3
  float4 *axis;      // n: the current axis in FP32
  float4 *qf;        // n: the current quaternion in FP32
  float *oprev;      // n x 3 axis before the last move (FP32): the claims' old ellipsoid
  float4 *kin;       // kinematics of the current step, 3 float4 per cell:
                     //   (f.x, f.y, f.z, Xi.x), (V, Xi.y), (W, Xi.z); X = Xi + f, Xi = rint(X)
  float4 *kin_next;  // kinematics written for the next step
  int *rec_last;     // n: records of the last sweep (for the link read-out)
  int *cK, *cIT;     // n x 3 each: contact links, sum m_r c_r and sum m_r dI x c_r
  unsigned long long *touched;  // n x touched_cap nodes claimed or left in one re-discretisation (pack_xyzr)
  double *lsum;      // n x 6 link sums of one step: F, T (variable part)
  float *lsum_f;     // n x 21: Zff 6, Zft 9, Ztt 6
  int *lsum_i;       // n x 6 integer link sums: K, IT
  float *vw;         // n x 6 velocities of the half step the bounced populations are given
  int *touched_count;
  int touched_cap;
  double *Fpot, *Tpot;                 // potentials of the current step
  double *PF, *PT;                     // pending fill/drain impulses
  double *Flink, *Tlink, *Ftot, *Ttot; // read-out of the last step
  int *box;                            // n x 6 inclusive node box lo[3], hi[3]
  double *stage;                       // n x 13 staged state for particles_set
  int *status;                         // device status word (ST_* bits)
  double m, Iperp, Ipar, rho0;
  double g[3];
  int bfc, move;
  double le_dr;  // Lees-Edwards: reflect a cell within le_dr of the sheared plane (0: no shear)
  double inv_rpar2, inv_rperp2, R_par, R_perp;
  float Rpar2_f, Rperp2_f, Rmax_f;  // R^2 and the larger half-axis in FP32
  float inv_rpar2_f, inv_rperp2_f, kk_f;  // 1 / R^2 in FP32, kk = 1 / R_par^2 - 1 / R_perp^2
  int near_image;  // some period is shorter than two contact distances and two nodes
  int near_reach;  // some period is shorter than twice the owner search's reach and two nodes
  float sig_par, sig_perp, eps, eps_w, mu, nu, chi_prime, r_cut;
  float chi, sigbar, sigbar_w, chi_w, sigw_max;
  double chi_d, sigbar_d, sigbar_w_d, chi_w_d;  // the same in FP64 (contact geometry)
};

struct CellListView {
  int nb[3];
  int nbins;
  int *bin_of, *count, *start, *cursor, *ids;
};

// surface wall nodes (Sec. III: walls linked to the lumen) as one bit per
// node, rows of nxw 32-bit words along x
struct SurfBits {
  uint32_t *bits;  // ny nz nxw words, or null when there is no surface wall node
  int nxw;
  uint32_t *rows;  // one bit per lattice row (y, z): the row holds a surface wall node
};

// close pairs of the learned correction: pairs (i, j), their features
// (14 floats) and the network's outputs (6 floats)
struct PairBuf {
  int2 *pairs;
  float *feat, *out;
  int *count;
  int cap;
};

struct ChangeList {
  int *count;
  int32_t *items;  // triples (node, old, new)
  int cap;
};

// Programmatic dependent launch.  A kernel that calls pdl_trigger lets the next
// kernel of its stream, if that was launched by launch_dependent, start its
// blocks; that kernel calls pdl_wait before it reads anything the first one
// writes (the wait ends when the first has finished and its writes are
// visible).  It hides a launch of 2 to 3 us and what the second kernel can do
// with older data.  Both calls do nothing in a kernel launched otherwise.  For
// kernels of few blocks: the sweep launched so filled the SMs before the
// side streams' kernels, which then waited for its first wave (sheared box 81
// -> 84 us a step).
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... KArgs, class... Args>
inline void launch_dependent(bool dep, void (*kernel)(KArgs...), dim3 grid, dim3 block, cudaStream_t st,
                             Args &&...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.stream = st;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = dep ? 1 : 0;  // (else an ordinary launch)
  cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// ---------------------------------------------------------------------------
// launchers (each adds the number of kernels it launched to *nl where given)

void launch_lb_step(int dtype, const LatticeView &lv, int par, const WallAcc &wa, int *status, cudaStream_t st);
// the walls' momentum of all sets (WALL_SUMS values) to pinned host memory; the sums start anew
void launch_wall_read(const WallAcc &wa, double rho0, double *out, cudaStream_t st);
// the persistent row sweep's grid per instantiation (LatticeView::rows_grid)
void lb_rows_grids(int dtype, int out[8]);
// pend: add the pending moving-boundary terms (there are cells)
void launch_fields(int dtype, const LatticeView &lv, int par, int pend, double *rho, double *u, int32_t *owner,
                   cudaStream_t st);
void launch_pop_io(int dtype, const LatticeView &lv, int par, double *buf, int to_storage, cudaStream_t st);
void launch_init(int dtype, const LatticeView &lv, cudaStream_t st);
void launch_fill_int(int *a, unsigned n, int v, cudaStream_t st);
void launch_apply_wall_mask(const LatticeView &lv, const uint8_t *mask, cudaStream_t st);
void launch_surface_bits(const LatticeView &lv, const SurfBits &sb, int *count, cudaStream_t st);
void launch_surface_rows(const LatticeView &lv, const SurfBits &sb, cudaStream_t st);
unsigned links_blocks(const LatticeView &lv);
void launch_links(const LatticeView &lv, int contact, int pass, int *block_count, const int *block_off, int32_t *out,
                  long long cap, cudaStream_t st);
void launch_cell_list(const LatticeView &lv, const PartView &pv, const CellListView &cl, cudaStream_t st, int64_t *nl);
void launch_forces(const LatticeView &lv, const PartView &pv, const CellListView &cl, const SurfBits &sb,
                   cudaStream_t st, int64_t *nl);
// link sums from the sweep's records and the implicit solve + leap-frog;
// then the pending C of the records (independent of the claims, which need
// only the solve)
void launch_sums_solve(const LatticeView &lv, const PartView &pv, cudaStream_t st, int64_t *nl);
void launch_link_pending(int dtype, const LatticeView &lv, const PartView &pv, int par, cudaStream_t st,
                         int64_t *nl);
void launch_set_state(const LatticeView &lv, const PartView &pv, int mode, cudaStream_t st, int64_t *nl);
void launch_claims(const LatticeView &lv, const PartView &pv, int *claim, const ChangeList &chg, int mode,
                   cudaStream_t st, int64_t *nl);
void launch_geometry(const LatticeView &lv, const PartView &pv, cudaStream_t st, int64_t *nl);
// the geometry after a step's resolve, in two independent parts (together
// the same result as launch_geometry): neighbour words around the changed
// nodes (after resolve); contact sums cell by cell from the current owner
// map and kinematics (at the start of the next step)
void launch_nbm_update(const LatticeView &lv, const PartView &pv, const ChangeList &chg, cudaStream_t st,
                       int64_t *nl);
void launch_contacts(const LatticeView &lv, const PartView &pv, cudaStream_t st, int64_t *nl);
// the pending C of the last step into the stored populations (layout par),
// before read-outs and state changes between steps
void launch_flush_pending(int dtype, const LatticeView &lv, int par, cudaStream_t st, int64_t *nl);
// replaced: the cells were set anew (bl_particles_set), not moved by a step
void launch_resolve_fill(int dtype, const LatticeView &lv, const PartView &pv, const CellListView &cl, int *claim,
                         const ChangeList &chg, int par_next, int impulses, int replaced, cudaStream_t st,
                         int64_t *nl);
void launch_clear_cells(int dtype, const LatticeView &lv, int par, cudaStream_t st, int64_t *nl);

void launch_pair_features(const LatticeView &lv, const PartView &pv, const int2 *pairs, int n, float *out,
                          cudaStream_t st);
// the learned correction: the close pairs with their features and the network
// over them (after the cell list), then its forces (after the potentials)
void launch_mlp_pairs(const LatticeView &lv, const PartView &pv, const CellListView &cl, const PairBuf &pb,
                      float gap_lo, float gap_cut, float speed_lo, float speed_hi, const void *mlp, cudaStream_t st,
                      int64_t *nl);
void launch_mlp_apply(const PartView &pv, const PairBuf &pb, cudaStream_t st, int64_t *nl);
// forward pass of a bl_mlp over *count rows of x (at most cap), raw units
void launch_mlp_forward_dev(const void *mlp, const float *x, const int *count, int cap, float *y, cudaStream_t st);
// the Lees-Edwards passes after a sweep of parity par
void launch_lees_edwards(int dtype, const LatticeView &lv, const LeView &le, int par, cudaStream_t st, int64_t *nl);

// bit flags of the device status word
constexpr int ST_UNSTABLE = 1;
constexpr int ST_OVERFLOW = 2;
constexpr int ST_BARRIER = 4;  // a bounded wait on an mbarrier gave up
constexpr int ST_LEPLANE = 8;  // a node beside the Lees-Edwards plane is not fluid

// ---------------------------------------------------------------------------
// exact FP64 geometry (no contraction), matching the operation order of the
// plain reference so that inside decisions agree bit for bit

__device__ __forceinline__ void axis_exact(const double *q, double *o) {
  o[0] = __dmul_rn(2.0, __dadd_rn(__dmul_rn(q[1], q[3]), __dmul_rn(q[0], q[2])));
  o[1] = __dmul_rn(2.0, __dsub_rn(__dmul_rn(q[2], q[3]), __dmul_rn(q[0], q[1])));
  o[2] = __dsub_rn(1.0, __dmul_rn(2.0, __dadd_rn(__dmul_rn(q[1], q[1]), __dmul_rn(q[2], q[2]))));
}

__device__ __forceinline__ double min_image_exact(double d, int n, int per) {
  if (!per) return d;
  double half = __dmul_rn(0.5, (double)n);
  if (d > half) return __dsub_rn(d, (double)n);
  if (d < -half) return __dadd_rn(d, (double)n);
  return d;
}

__device__ __forceinline__ bool inside_exact(int x, int y, int z, const double *X, const double *o,
                                             double inv_rpar2, double inv_rperp2, const LatticeView &lv) {
  double d0 = min_image_exact(__dsub_rn((double)x, X[0]), lv.nx, lv.per[0]);
  double d1 = min_image_exact(__dsub_rn((double)y, X[1]), lv.ny, lv.per[1]);
  double d2 = min_image_exact(__dsub_rn((double)z, X[2]), lv.nz, lv.per[2]);
  double dpar = __dadd_rn(__dadd_rn(__dmul_rn(d0, o[0]), __dmul_rn(d1, o[1])), __dmul_rn(d2, o[2]));
  double dd = __dadd_rn(__dadd_rn(__dmul_rn(d0, d0), __dmul_rn(d1, d1)), __dmul_rn(d2, d2));
  double pp = __dmul_rn(dpar, dpar);
  double s = __dadd_rn(__dmul_rn(pp, inv_rpar2), __dmul_rn(__dsub_rn(dd, pp), inv_rperp2));
  return s <= 1.0;
}

// integer minimum image of a lattice displacement
__device__ __forceinline__ int imin_image(int d, int n, int per) {
  if (!per) return d;
  if (2 * d > n) return d - n;
  if (2 * d < -n) return d + n;
  return d;
}

// periodic image of a separation of two points, each given as its nearest node
// and the rest: d between the nodes, f between the rests (|f| <= 1).  The nearer
// image of the separation itself: of the nodes alone it would be the farther one
// for separations within a node of half a period, which two cells in contact
// have where a period is short (2 max(R) + 4 at least).
__device__ __forceinline__ float image_f(int d, float f, int n, int per) {
  int m = imin_image(d, n, per);
  if (per) {
    const float r = (float)m + f, h = 0.5f * (float)n;
    m -= r > h ? n : (r < -h ? -n : 0);
  }
  return (float)m + f;
}

// periodic wrap for coordinates at most a few periods out (no division)
__device__ __forceinline__ int wrapi(int v, int n) {
  while (v < 0) v += n;
  while (v >= n) v -= n;
  return v;
}

// packed node coordinates of the per-cell lists: r | x << 5 | y << 25 | z << 45
__host__ __device__ __forceinline__ unsigned long long pack_xyzr(int x, int y, int z, int r) {
  return (unsigned long long)r | ((unsigned long long)x << 5) | ((unsigned long long)y << 25) |
         ((unsigned long long)z << 45);
}
__device__ __forceinline__ void unpack_xyzr(unsigned long long e, int xyz[3], int &r) {
  r = (int)(e & 31ull);
  xyz[0] = (int)((e >> 5) & 0xFFFFFull);
  xyz[1] = (int)((e >> 25) & 0xFFFFFull);
  xyz[2] = (int)(e >> 45);
}

// the mixed word from the owners of a node and its 18 neighbours (on[r]: x + c_r)
__device__ __forceinline__ uint4 mixed_word(const int (&on)[Q]) {
  uint4 w = make_uint4(0u, 0u, 0u, 0u);
  int p1 = -1, p2 = -1;
  sfor<1, Q>([&](auto R) {
    constexpr int r = decltype(R)::value;
    if (on[r] <= -2) {
      w.w |= 1u << r;
    } else if (on[r] >= 0) {
      if (p1 < 0) p1 = on[r];
      else if (p2 < 0 && on[r] != p1) p2 = on[r];
      w.y |= (on[r] == p1 ? 1u : 0u) << r;
      w.z |= (on[r] == p2 ? 1u : 0u) << r;
    }
  });
  w.x = ((uint32_t)p1 & NBX_NONE) | ((uint32_t)p2 << 16);
  return w;
}

// direction masks of the lattice (bit r), for the record sums by popcount
template <class P>
__host__ __device__ constexpr uint32_t dir_mask(P pred) {
  uint32_t m = 0;
  for (int r = 1; r < Q; ++r)
    if (pred(r)) m |= 1u << r;
  return m;
}
using D3 = D3Q19;
constexpr int cxyz(int r, int a) { return a == 0 ? D3::cx(r) : (a == 1 ? D3::cy(r) : D3::cz(r)); }
template <int A, int SGN>
struct AxisDirs {  // axis vectors along A with sign SGN (m = 2)
  static constexpr uint32_t v = dir_mask([](int r) { return r <= 6 && cxyz(r, A) == SGN; });
};
template <int A, int SGN>
struct DiagDirs {  // diagonal vectors with c_A = SGN (m = 1)
  static constexpr uint32_t v = dir_mask([](int r) { return r > 6 && cxyz(r, A) == SGN; });
};
template <int A, int B, int SGN>
struct PairDirs {  // diagonal vectors with c_A c_B = SGN
  static constexpr uint32_t v = dir_mask([](int r) { return r > 6 && cxyz(r, A) * cxyz(r, B) == SGN; });
};

__device__ __forceinline__ int popm(uint32_t m, uint32_t sel) { return __popc(m & sel); }

// the components of c_r for a direction r known only at run time: c + 1
// packed two bits per direction in a 64-bit constant
template <int A>
__host__ __device__ constexpr unsigned long long packed_dirs() {
  unsigned long long v = 0;
  for (int r = 0; r < Q; ++r) v |= (unsigned long long)(cxyz(r, A) + 1) << (2 * r);
  return v;
}
template <int A>
__device__ __forceinline__ int rt_c(int r) {
  return (int)((packed_dirs<A>() >> (2 * r)) & 3ull) - 1;
}
__device__ __forceinline__ int rt_m(int r) { return r == 0 ? 12 : (r <= 6 ? 2 : 1); }
__device__ __forceinline__ int rt_opp(int r) { return r == 0 ? 0 : ((r & 1) ? r + 1 : r - 1); }

// node index -> coordinates
__device__ __forceinline__ void node_xyz(const LatticeView &lv, unsigned n, int xyz[3]) {
  const unsigned z = fdiv(n, lv.dnxy), rem = n - z * lv.dnxy.d, y = fdiv(rem, lv.dnx);
  xyz[0] = (int)(rem - y * lv.dnx.d);
  xyz[1] = (int)y;
  xyz[2] = (int)z;
}

// sums over the directions of a mask (bit r) by popcount: component A of
// K = sum m_r c_r, and the entries A A and A B of M = sum m_r c_r c_r^T
template <int A>
__device__ __forceinline__ int mask_K(uint32_t m) {
  return 2 * (popm(m, AxisDirs<A, 1>::v) - popm(m, AxisDirs<A, -1>::v)) + popm(m, DiagDirs<A, 1>::v) -
         popm(m, DiagDirs<A, -1>::v);
}
template <int A>
__device__ __forceinline__ int mask_Maa(uint32_t m) {
  return 2 * popm(m, AxisDirs<A, 1>::v | AxisDirs<A, -1>::v) + popm(m, DiagDirs<A, 1>::v | DiagDirs<A, -1>::v);
}
template <int A, int B>
__device__ __forceinline__ int mask_Mab(uint32_t m) {
  return popm(m, PairDirs<A, B, 1>::v) - popm(m, PairDirs<A, B, -1>::v);
}

// The populations an opposite pair r, rbar relaxes toward: the third-order
// equilibrium w (drho + rho t), t = 4.5 cu^2 - 1.5 uu +- cu (3 - 4.5 uu + 4.5
// cu^2), plus the Guo source over omega, src w (3 (cF - uF) + 9 cu cF) / omega
// with src = 1 - omega / 2 (so that f - omega (f - this) is the collision).
// The even and the odd part of t and of the source are shared by the pair, and
// rho t + drho is one fused multiply-add: 9 operations a pair, 13 with a
// force, where each direction by itself took 16 and 27.  Folding rho and the
// weight into the node's coefficients would save two more, but rounds each
// population twice more and raised the density error at tau = 0.8 by half.
// The sweeps of the dense and the indexed lattice and the link sums evaluate
// this same function, so the bounced populations the fluid keeps and those
// the cell's momentum counts agree.
struct Collide {
  float ux, uy, uz, rho;
  float a, b;        // 3 - 4.5 uu, 1.5 uu
  float drho;        // with a force drho - u . H
  float Hx, Hy, Hz;  // 3 src F / omega
};

template <bool FORCE>
__device__ __forceinline__ Collide collide_coeffs(float drho, float rho, float ux, float uy, float uz, float uu,
                                                  float omega, float Fx, float Fy, float Fz, float uF) {
  Collide k;
  k.ux = ux;
  k.uy = uy;
  k.uz = uz;
  k.rho = rho;
  k.a = fmaf(-4.5f, uu, 3.0f);
  k.b = 1.5f * uu;
  k.drho = drho;
  k.Hx = k.Hy = k.Hz = 0.f;
  if constexpr (FORCE) {
    const float h = 3.0f * (1.0f / omega - 0.5f);
    k.drho = fmaf(-h, uF, drho);
    k.Hx = h * Fx;
    k.Hy = h * Fy;
    k.Hz = h * Fz;
  }
  return k;
}

// component of c_R for odd R along u: at most two additions
template <int R>
__device__ __forceinline__ float dir_dot(float x, float y, float z) {
  using D = D3Q19;
  float v = 0.f;
  if constexpr (D::cx(R) != 0) v = D::cx(R) > 0 ? x : -x;
  if constexpr (D::cy(R) != 0) v = D::cy(R) > 0 ? v + y : v - y;
  if constexpr (D::cz(R) != 0) v = D::cz(R) > 0 ? v + z : v - z;
  return v;
}

// targets of populations R and R + 1 (odd R, opposite directions) over their
// weight
template <int R, bool FORCE>
__device__ __forceinline__ void collide_pair(const Collide &k, float &xr, float &xb) {
  const float cu = dir_dot<R>(k.ux, k.uy, k.uz);
  const float s = cu * cu;
  const float E = fmaf(4.5f, s, -k.b), q = fmaf(4.5f, s, k.a);
  const float tr = fmaf(cu, q, E), tb = fmaf(-cu, q, E);
  if constexpr (FORCE) {
    const float cH = dir_dot<R>(k.Hx, k.Hy, k.Hz), e = fmaf(3.0f * cu, cH, k.drho);
    xr = fmaf(k.rho, tr, e + cH);
    xb = fmaf(k.rho, tb, e - cH);
  } else {
    xr = fmaf(k.rho, tr, k.drho);
    xb = fmaf(k.rho, tb, k.drho);
  }
}

// the target of population 0 over its weight
__device__ __forceinline__ float collide_rest(const Collide &k) { return fmaf(-k.rho, k.b, k.drho); }

// relaxation of population R toward w x: f - omega (f - w x), at tau = 1 w x
template <int R, bool TAU1>
__device__ __forceinline__ float relax_to(float f, float x, float omega) {
  constexpr float w = (float)D3Q19::m(R) / 36.0f;
  return TAU1 ? __fmul_rn(w, x) : fmaf(-omega, fmaf(-w, x, f), f);
}

// velocity (j + F / 2) / rho of a node, its square and u . F, F = rho g, with
// every contraction written out: the two lattices' sweeps agree bit for bit
template <bool FORCE>
__device__ __forceinline__ void node_velocity(float rho, float jx, float jy, float jz, const float (&g)[3], float (&u)[3],
                                              float (&F)[3], float &uu, float &uF) {
  const float inv = 1.0f / rho;
  F[0] = F[1] = F[2] = uF = 0.f;
  if constexpr (FORCE) {
    for (int k = 0; k < 3; ++k) F[k] = __fmul_rn(rho, g[k]);
    jx = fmaf(0.5f, F[0], jx);
    jy = fmaf(0.5f, F[1], jy);
    jz = fmaf(0.5f, F[2], jz);
  }
  u[0] = __fmul_rn(jx, inv);
  u[1] = __fmul_rn(jy, inv);
  u[2] = __fmul_rn(jz, inv);
  uu = fmaf(u[2], u[2], fmaf(u[1], u[1], __fmul_rn(u[0], u[0])));
  if constexpr (FORCE) uF = fmaf(u[2], F[2], fmaf(u[1], F[1], __fmul_rn(u[0], F[0])));
}

// moving-wall term of a link along c_R into a wall of velocity v (Eq. c):
// 6 alpha rho c_rbar . v, added to the population that returns along rbar
template <int R>
__device__ __forceinline__ float wall_term(float rho, const float (&v)[3]) {
  using D = D3Q19;
  const float cv = fmaf((float)D::cz(R), v[2], fmaf((float)D::cy(R), v[1], __fmul_rn((float)D::cx(R), v[0])));
  return __fmul_rn(__fmul_rn(-(D::m(R) / 6.0f), rho), cv);
}

// a population with the pending moving-boundary term of its bounce along r
// added, f + C with C = -(m_r / 6) c_r . u, cu = c_r . u.  One function with the
// contraction written out: the field read-out and the flush of the pending
// terms form the same number, which FP16 storage then rounds alike
__device__ __forceinline__ float add_pending(float f, int m, float cu) { return fmaf(-((float)m / 6.0f), cu, f); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

}  // namespace bl
