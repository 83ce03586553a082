// lb_indexed.cu -- the indexed lattice of vessel networks: only the fluid
// nodes of a sparse geometry are stored and swept.
//
// The paper closes by pointing out that the method, joined to an indexed LB
// scheme, can take flow through digitised vessel networks, whose lumen fills
// a few per cent of its bounding box.  Here the fluid nodes of a lattice with
// walls (face walls and a wall mask, as for the dense lattice) get compact
// indices in dense node order (x fastest, so that runs along x stay
// contiguous and a warp's reads coalesce).  Memory and traffic scale with the
// lumen, not the box.
//
// Neighbours.  A node's neighbours along x are the indices beside its own, and
// in each of the eight other lattice rows (dy, dz) around it they are b - 1, b
// and b + 1 where they are fluid, with b the number of fluid nodes before the
// node's x in that row's order; along a run of nodes b grows by one with each
// node whose (dy, dz) neighbour is fluid.  So a node stores one word, with a
// bit per open direction, and each segment (a run of nodes consecutive in x
// within one warp's 32 nodes) stores the eight b of its first node, from which
// the lanes count their own with a warp vote per row.  That is 5 to 6 bytes per
// node where a table of 18 neighbours took 72, and the even step reads the
// word alone.  Nodes for which this does not hold, the ends of a periodic row
// and nodes between walls of different ids, are segments of their own that
// point to an explicit table; the builder checks every node against the
// neighbour table.
//
// The sweep is the dense lattice's plasma update (Sec. II: moments, Guo
// forcing, BGK toward the third-order equilibrium, mid-link bounce-back with
// the moving-wall term C of Eq. c, the walls' momentum) on one single AA
// buffer of 19 x Nf slots.  The AA pairing cannot use a wall node's slot for
// a bounce (walls have none), so bounced populations stay in their node's
// own slots:
//   even step: read slot r of i; write f*_r to slot rbar of i (open or wall)
//   odd step:  read direction r from slot rbar of i - c_r, or where i - c_r
//              is a wall from slot r of i; write f*_r to slot r of i + c_r,
//              or where i + c_r is a wall to slot rbar of i
// so that every slot is read and written by one thread per step.  Cells are
// not coupled to the indexed lattice (their owner map, claims and fill work
// on the dense node grid).
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <type_traits>
#include <vector>

#include "../../include/bloodlb.h"
#include "lb_moments.cuh"
#include "lb_sweep.cuh"

namespace bl {
namespace {

inline unsigned nblk(unsigned n, unsigned b) { return (n + b - 1) / b; }

// word of a node: bit 0 starts a segment, bits 1..18 open directions, bits
// 20..22 the wall id of its closed ones, SP_TABLE neighbours in the table
constexpr uint32_t SP_START = 1u;
constexpr int SP_WALL = 20;
constexpr uint32_t SP_TABLE = 1u << 24;

// the rows (dy, dz) in the order of a segment's eight b, by their dx = 0
// direction
__host__ __device__ constexpr int row_dir(int j) {
  return j < 4 ? 3 + j : 11 + j;  // +y, -y, +z, -z, (y,z) diagonals 15..18
}
__host__ __device__ constexpr int row_of(int r) {  // row of direction r (r = 1, 2: the node's own)
  for (int j = 0; j < 8; ++j)
    if (D3Q19::cy(row_dir(j)) == D3Q19::cy(r) && D3Q19::cz(row_dir(j)) == D3Q19::cz(r)) return j;
  return -1;
}

struct SparseView {
  unsigned Nf;            // fluid nodes
  void *pop;              // 19 x Nf storage elements, slot r of node i at r Nf + i
  const uint32_t *word;   // Nf
  const int32_t *seg0;    // first segment of each 32 nodes
  const int4 *seg;        // 2 per segment: its eight b, or the table entry of an SP_TABLE node
  const int32_t *table;   // ntable x 18: neighbour index or -1 - wall id
  const int32_t *dense;   // Nf: dense node index of each fluid node
  float wall_vel[NWALL][3];
  float omega, rho0, g[3];
  int *status;
};

// what a lane knows of its node's neighbours (all 32 lanes call rows_of)
struct SparseRows {
  uint32_t w;
  int b[8];           // b of each row; b[0] the table entry of an SP_TABLE node
};

__device__ __forceinline__ void rows_of(const SparseView &sv, unsigned i, uint32_t w, SparseRows &q) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  q.w = w;
  const unsigned le = FULL >> (31 - lane);
  const unsigned starts = __ballot_sync(FULL, w & SP_START) & le;
  const int first = 31 - __clz(starts | 1u);
  // (a warp past the last node has no start of its own: any segment will do)
  const int s = max(sv.seg0[i >> 5] + __popc(starts) - 1, 0);
  const int4 lo = sv.seg[2 * s], hi = sv.seg[2 * s + 1];
  q.b[0] = lo.x;
  q.b[1] = lo.y;
  q.b[2] = lo.z;
  q.b[3] = lo.w;
  q.b[4] = hi.x;
  q.b[5] = hi.y;
  q.b[6] = hi.z;
  q.b[7] = hi.w;
  const unsigned before = (le >> 1) & (FULL << first);  // the lanes of this segment before this one
  sfor<0, 8>([&](auto J) {
    constexpr int j = decltype(J)::value;
    const unsigned m = __ballot_sync(FULL, (w >> row_dir(j)) & 1u);
    q.b[j] += __popc(m & before);
  });
}

// indices of the open neighbours i + c_r (what stands at a closed direction is
// not used).  One branch for the table nodes: a choice per direction cost the
// odd step 36 branches, more than half its instructions.
__device__ __forceinline__ void open_nbrs(const SparseView &sv, const SparseRows &q, unsigned i, unsigned (&nb)[Q]) {
  sfor<1, Q>([&](auto R) {
    constexpr int r = decltype(R)::value, j = row_of(r), dx = D3Q19::cx(r);
    if constexpr (j < 0) nb[r] = i + (unsigned)dx;
    else nb[r] = (unsigned)(q.b[j] + (dx < 0 ? -1 : (dx > 0 ? (int)((q.w >> row_dir(j)) & 1u) : 0)));
  });
  if (q.w & SP_TABLE) {
    const int32_t *t = sv.table + 18 * (size_t)q.b[0];
    sfor<1, Q>([&](auto R) { nb[decltype(R)::value] = (unsigned)t[decltype(R)::value - 1]; });
  }
}

// wall id behind the closed direction R
template <int R>
__device__ __forceinline__ int wall_of(const SparseView &sv, const SparseRows &q) {
  if (q.w & SP_TABLE) return -1 - sv.table[18 * (size_t)q.b[0] + (R - 1)];
  return (int)(q.w >> SP_WALL) & 7;
}

// slot from which node i reads direction R in a step of parity par (nb: its
// open neighbours where par = 1)
template <int R>
__device__ __forceinline__ unsigned sparse_src(const SparseView &sv, uint32_t w, int par, unsigned i,
                                               const unsigned (&nb)[Q]) {
  constexpr int rb = D3Q19::opp(R);
  if (par == 0 || R == 0) return (unsigned)R * sv.Nf + i;
  return (w >> rb) & 1u ? (unsigned)rb * sv.Nf + nb[rb] : (unsigned)R * sv.Nf + i;
}

// One fluid node per thread.  Bound: HBM, 2 x 19 populations and about 5 bytes
// of words and segments per node; BL_SPARSE_MINB blocks of 128 threads keep
// enough loads in flight.
#ifndef BL_SPARSE_MINB
#define BL_SPARSE_MINB 8
#endif

template <class S, int PAR, bool FORCE, bool TAU1>
__global__ void __launch_bounds__(128, BL_SPARSE_MINB) k_sparse_step(SparseView sv, WallAcc wa0) {
  const WallAcc wa = wall_copy(wa0);
  using D = D3Q19;
  const unsigned Nf = sv.Nf;
  const unsigned i0 = blockIdx.x * 128u + threadIdx.x;
  const bool valid = i0 < Nf;
  const unsigned i = valid ? i0 : Nf - 1u;
  S *pop = reinterpret_cast<S *>(sv.pop);
  int wkey = -1;
  float wF[3] = {0.f, 0.f, 0.f};
  int wK[3] = {0, 0, 0};
  SparseRows q;
  q.w = valid ? sv.word[i] : 0u;
  if constexpr (PAR == 1) {
    rows_of(sv, i, q.w, q);
  } else {
    // in place: the segments are needed for a table node's walls alone
    const unsigned starts = __ballot_sync(0xffffffffu, q.w & SP_START) & (0xffffffffu >> (31 - (threadIdx.x & 31)));
    if (q.w & SP_TABLE) q.b[0] = sv.seg[2 * (sv.seg0[i >> 5] + __popc(starts) - 1)].x;
  }
  if (valid) {
    float f[Q];
    {
      unsigned nb[Q];
      if constexpr (PAR == 1) open_nbrs(sv, q, i, nb);
      sfor<0, Q>([&](auto R) {
        constexpr int r = decltype(R)::value;
        f[r] = Store<S>::ld(pop + sparse_src<r>(sv, q.w, PAR, i, nb));
      });
    }
    // moments of the shifted populations: rho = rho_bar + sum f~, j = sum f~ c
    float drho = f[0], jx = 0.f, jy = 0.f, jz = 0.f;
    sfor<0, 9>([&](auto P) {
      constexpr int r = 2 * decltype(P)::value + 1;
      const float s = f[r] + f[r + 1], d = f[r] - f[r + 1];
      drho += s;
      if constexpr (D::cx(r) != 0) jx += D::cx(r) > 0 ? d : -d;
      if constexpr (D::cy(r) != 0) jy += D::cy(r) > 0 ? d : -d;
      if constexpr (D::cz(r) != 0) jz += D::cz(r) > 0 ? d : -d;
    });
    const float rho = sv.rho0 + drho;
    float u[3], F[3], uu, uF;
    node_velocity<FORCE>(rho, jx, jy, jz, sv.g, u, F, uu, uF);
    if (!(rho > 0.f) || !(uu < 0.09f)) atomicOr(sv.status, ST_UNSTABLE);
    // the dense lattice's collision
    const float om = TAU1 ? 1.0f : sv.omega;
    const Collide k = collide_coeffs<FORCE>(drho, rho, u[0], u[1], u[2], uu, om, F[0], F[1], F[2], uF);
    f[0] = relax_to<0, TAU1>(f[0], collide_rest(k), om);
    sfor<0, 9>([&](auto P) {
      constexpr int r = 2 * decltype(P)::value + 1, rb = r + 1;
      float xr, xb;
      collide_pair<r, FORCE>(k, xr, xb);
      f[r] = relax_to<r, TAU1>(f[r], xr, om);
      f[rb] = relax_to<rb, TAU1>(f[rb], xb, om);
    });
    Store<S>::st(pop + i, f[0]);
    const uint32_t closed = ~q.w & NB_SOLID;
    if (closed) {
      // links into walls: the population returns along rbar with the
      // moving-wall term C (Eq. c), the wall receives (2 f*_r + C) c_r
      sfor<1, Q>([&](auto R) {
        constexpr int r = decltype(R)::value;
        if ((closed >> r) & 1u) {
          const int w = wall_of<r>(sv, q);
          const float C = wall_term<r>(rho, sv.wall_vel[w]);
          const float dp = 2.0f * f[r] + C;
          if (wkey != w && wkey >= 0) {
            for (int kk = 0; kk < 3; ++kk) {
              atomicAdd(&wa.F[3 * wkey + kk], (double)wF[kk]);
              atomicAdd((unsigned long long *)&wa.K[3 * wkey + kk], (unsigned long long)(long long)wK[kk]);
              wF[kk] = 0.f;
              wK[kk] = 0;
            }
          }
          wkey = w;
          wF[0] += dp * D::cx(r);
          wF[1] += dp * D::cy(r);
          wF[2] += dp * D::cz(r);
          wK[0] += D::m(r) * D::cx(r);
          wK[1] += D::m(r) * D::cy(r);
          wK[2] += D::m(r) * D::cz(r);
          f[r] += C;
        }
      });
    }
    unsigned nb[Q];  // (again: they do not stay live through the collision)
    if constexpr (PAR == 1) open_nbrs(sv, q, i, nb);
    sfor<1, Q>([&](auto R) {
      constexpr int r = decltype(R)::value;
      constexpr int rb = D::opp(r);
      unsigned dst = (unsigned)rb * Nf + i;
      if constexpr (PAR == 1)
        if ((q.w >> r) & 1u) dst = (unsigned)r * Nf + nb[r];
      Store<S>::st(pop + dst, f[r]);
    });
  }
  flush_wall_momentum(wa, wkey, wF, wK);
}

// moments on the dense grid (zero at walls): rho and u = j / rho + g / 2
template <class S>
__global__ void __launch_bounds__(256) k_sparse_fields(SparseView sv, int par, double rho0, double hg0, double hg1,
                                                       double hg2, double *rho, double *u) {
  const unsigned i0 = blockIdx.x * blockDim.x + threadIdx.x;
  const bool valid = i0 < sv.Nf;
  const unsigned i = valid ? i0 : sv.Nf - 1u;
  const S *pop = reinterpret_cast<const S *>(sv.pop);
  SparseRows q;
  rows_of(sv, i, valid ? sv.word[i] : 0u, q);
  if (!valid) return;
  float f[Q];
  unsigned nb[Q];
  open_nbrs(sv, q, i, nb);
  sfor<0, Q>([&](auto R) {
    constexpr int r = decltype(R)::value;
    f[r] = Store<S>::ld(pop + sparse_src<r>(sv, q.w, par, i, nb));
  });
  const double hg[3] = {hg0, hg1, hg2};
  double rh, uu[3];
  node_fields(f, rho0, hg, rh, uu);
  const unsigned n = (unsigned)sv.dense[i];
  if (rho) rho[n] = rh;
  if (u)
    for (int k = 0; k < 3; ++k) u[3 * (size_t)n + k] = uu[k];
}

// populations n_r (unshifted) on the dense grid, N x 19, to (0) or from (1) storage
template <class S>
__global__ void k_sparse_pop_io(SparseView sv, int par, double *buf, int to_storage) {
  const unsigned i0 = blockIdx.x * blockDim.x + threadIdx.x;
  const bool valid = i0 < sv.Nf;
  const unsigned i = valid ? i0 : sv.Nf - 1u;
  S *pop = reinterpret_cast<S *>(sv.pop);
  SparseRows q;
  rows_of(sv, i, valid ? sv.word[i] : 0u, q);
  if (!valid) return;
  const size_t n = (size_t)sv.dense[i];
  unsigned nb[Q];
  open_nbrs(sv, q, i, nb);
  sfor<0, Q>([&](auto R) {
    constexpr int r = decltype(R)::value;
    const double shift = (double)sv.rho0 * D3Q19::m(r) / 36.0;
    const unsigned s = sparse_src<r>(sv, q.w, par, i, nb);
    if (to_storage) Store<S>::st(pop + s, (float)(buf[n * Q + r] - shift));
    else buf[n * Q + r] = (double)Store<S>::ld(pop + s) + shift;
  });
}

template <class S>
__global__ void k_sparse_rest(SparseView sv) {
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= sv.Nf) return;
  S *pop = reinterpret_cast<S *>(sv.pop);
  for (int r = 0; r < Q; ++r) Store<S>::st(pop + (size_t)r * sv.Nf + i, 0.0f);
}

template <class S>
void launch_sparse_typed(const SparseView &sv, int par, bool force, bool tau1, const WallAcc &wa, cudaStream_t st) {
  const unsigned b = 128, g = nblk(sv.Nf, b);
#define BL_SP(P_, F_, T_) k_sparse_step<S, P_, F_, T_><<<g, b, 0, st>>>(sv, wa)
  if (par == 0) {
    if (force) { if (tau1) BL_SP(0, true, true); else BL_SP(0, true, false); }
    else { if (tau1) BL_SP(0, false, true); else BL_SP(0, false, false); }
  } else {
    if (force) { if (tau1) BL_SP(1, true, true); else BL_SP(1, true, false); }
    else { if (tau1) BL_SP(1, false, true); else BL_SP(1, false, false); }
  }
#undef BL_SP
}

}  // namespace
}  // namespace bl

using namespace bl;

struct bl_sparse {
  bl_lb_params lp;
  cudaStream_t stream, gstream;
  cudaEvent_t ev_fork, ev_join;
  cudaGraphExec_t gexec;
  int g_parity;
  SparseView sv;
  WallAcc wa;
  int parity;
  int64_t n_dense;
  int sticky;
  char err[256];
  int64_t launches;
  double *scratch;
  size_t scratch_bytes;
  double *pin;  // pinned: the walls' momentum, written by its kernel
};

static int sp_fail(bl_sparse *s, int code, const char *fmt, ...) {
  if (s && s->sticky == BL_OK) {
    s->sticky = code;
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(s->err, sizeof(s->err), fmt, ap);
    va_end(ap);
  }
  return code;
}

#define SPCU(call)                                                                  \
  do {                                                                              \
    cudaError_t e_ = (call);                                                        \
    if (e_ != cudaSuccess) return sp_fail(s, BL_ECUDA, "%s: %s", #call, cudaGetErrorString(e_)); \
  } while (0)

// wall id of node (x, y, z): the first walled axis (x, y, z order) whose
// layer holds it, a nonzero mask value k overriding with id k - 1; -1 fluid
static int node_wall(const bl_lb_params *p, const uint8_t *mask, int x, int y, int z) {
  const long long n = (long long)x + (long long)p->nx * ((long long)y + (long long)p->ny * z);
  if (mask && mask[n]) return (int)mask[n] - 1;
  const int c[3] = {x, y, z}, d[3] = {p->nx, p->ny, p->nz};
  for (int k = 0; k < 3; ++k) {
    if (p->periodic[k]) continue;
    if (c[k] == 0) return 2 * k;
    if (c[k] == d[k] - 1) return 2 * k + 1;
  }
  return -1;
}

// the number of each node among the fluid nodes, -1 - wall id at walls; their number
static long long index_ids(const bl_lb_params *p, const uint8_t *mask, std::vector<int32_t> &id) {
  long long nf = 0, n = 0;
  for (int z = 0; z < p->nz; ++z)
    for (int y = 0; y < p->ny; ++y)
      for (int x = 0; x < p->nx; ++x, ++n) {
        const int w = node_wall(p, mask, x, y, z);
        id[(size_t)n] = w >= 0 ? -1 - w : (int32_t)nf++;
      }
  return nf;
}

// dense index and neighbours of every fluid node (either array may be null)
static void index_fill(const bl_lb_params *p, const std::vector<int32_t> &id, long long nf, int32_t *dense_of,
                       int32_t *nbr) {
  const long long nx = p->nx, ny = p->ny, nz = p->nz;
  long long n = 0;
  for (long long z = 0; z < nz; ++z)
    for (long long y = 0; y < ny; ++y) {
      // a fluid node's neighbours lie in the box: a walled axis has wall
      // layers at its ends, a periodic one wraps
      long long row[3][3];
      for (int dz = -1; dz <= 1; ++dz)
        for (int dy = -1; dy <= 1; ++dy)
          row[dz + 1][dy + 1] = nx * ((y + dy + ny) % ny + ny * ((z + dz + nz) % nz));
      for (long long x = 0; x < nx; ++x, ++n) {
        const int32_t i = id[(size_t)n];
        if (i < 0) continue;
        if (dense_of) dense_of[i] = (int32_t)n;
        if (!nbr) continue;
        const long long xs[3] = {x == 0 ? nx - 1 : x - 1, x, x == nx - 1 ? 0 : x + 1};
        for (int r = 1; r < Q; ++r)
          nbr[(size_t)(r - 1) * nf + i] =
              id[(size_t)(row[1 + D3Q19::cz(r)][1 + D3Q19::cy(r)] + xs[1 + D3Q19::cx(r)])];
      }
    }
}

// what an index needs of its parameters
static bool index_ok(const bl_lb_params *p, const uint8_t *mask) {
  if (p->nx < 1 || p->ny < 1 || p->nz < 1) return false;
  const long long N = (long long)p->nx * p->ny * p->nz;
  if (N >= (1ll << 31)) return false;
  for (int k = 0; k < 3; ++k) {
    const int n = k == 0 ? p->nx : (k == 1 ? p->ny : p->nz);
    if (!p->periodic[k] && n < 3) return false;
  }
  if (mask)
    for (long long n = 0; n < N; ++n)
      if (mask[n] > NWALL) return false;
  return true;
}

extern "C" int bl_sparse_index_build(const bl_lb_params *p, const uint8_t *mask, int64_t *n_fluid, int32_t *dense_of,
                                     int32_t *nbr) {
  if (!p || !n_fluid || !index_ok(p, mask)) return BL_EINVAL;
  const long long N = (long long)p->nx * p->ny * p->nz;
  std::vector<int32_t> id((size_t)N);
  const long long nf = index_ids(p, mask, id);
  const long long prev = *n_fluid;
  *n_fluid = nf;
  if (!dense_of && !nbr) return BL_OK;
  if (prev < nf) return BL_EINVAL;  // the arrays hold fewer nodes than the lattice has
  index_fill(p, id, nf, dense_of, nbr);
  return BL_OK;
}

// words, segments and the explicit table of an index (see the head of this
// file).  A node is a table node where its row wraps (an end of a periodic row)
// or where its walls have different ids; the segments of the others are then
// checked against the neighbour table, and a node they do not reproduce becomes
// a table node too.
struct RowIndex {
  std::vector<uint32_t> word;
  std::vector<int32_t> seg0, seg, table;
};

static void build_rows(int nx, bool per_x, const std::vector<int32_t> &dense, const std::vector<int32_t> &nbr,
                       RowIndex &out) {
  const size_t nf = dense.size();
  out.word.assign(nf, 0u);
  for (int r = 1; r < Q; ++r) {
    const int32_t *nb = nbr.data() + (size_t)(r - 1) * nf;
    for (size_t i = 0; i < nf; ++i) {
      uint32_t &w = out.word[i];
      if (nb[i] >= 0) {
        w |= 1u << r;
      } else {
        const uint32_t id = (uint32_t)(-1 - nb[i]);
        if (!(w & (1u << 19))) w |= (1u << 19) | (id << SP_WALL);  // bit 19: a wall id is noted (cleared below)
        else if (((w >> SP_WALL) & 7u) != id) w |= SP_TABLE;
      }
    }
  }
  for (size_t i = 0; i < nf; ++i) {
    const int x = dense[i] % nx;
    if (per_x && (x == 0 || x == nx - 1)) out.word[i] |= SP_TABLE;
    out.word[i] &= ~(1u << 19);
  }
  for (bool again = true; again;) {
    again = false;
    out.seg0.assign((nf + 31) / 32, 0);
    out.seg.clear();
    out.table.clear();
    for (size_t i = 0; i < nf;) {
      if (i % 32 == 0) out.seg0[i / 32] = (int32_t)(out.seg.size() / 8);
      size_t e = i + 1;  // end of the segment
      const bool tab = out.word[i] & SP_TABLE;
      while (!tab && e < nf && e % 32 != 0 && dense[e] == dense[e - 1] + 1 && dense[e] % nx != 0 &&
             !(out.word[e] & SP_TABLE))
        ++e;
      int32_t b[8] = {0, 0, 0, 0, 0, 0, 0, 0};
      if (tab) {
        b[0] = (int32_t)(out.table.size() / 18);
        for (int r = 1; r < Q; ++r) out.table.push_back(nbr[(size_t)(r - 1) * nf + i]);
      } else {
        auto at = [&](int r, size_t k) { return nbr[(size_t)(r - 1) * nf + k]; };
        for (int j = 0; j < 8; ++j) {
          // the first node of the segment with a fluid neighbour in row j gives b
          const int r0 = row_dir(j);
          int rp = 0, rm = 0;
          for (int r = 7; r < 15; ++r)
            if (row_of(r) == j) (D3Q19::cx(r) > 0 ? rp : rm) = r;
          for (size_t k = i; k < e; ++k) {
            if (at(r0, k) >= 0) b[j] = at(r0, k);
            else if (rp && at(rp, k) >= 0) b[j] = at(rp, k);
            else if (rm && at(rm, k) >= 0) b[j] = at(rm, k) + 1;
            else continue;
            break;
          }
          int32_t bb = b[j];
          for (size_t k = i; k < e; ++k) {
            const bool mid = at(r0, k) >= 0;
            if ((mid && at(r0, k) != bb) || (rp && at(rp, k) >= 0 && at(rp, k) != bb + (mid ? 1 : 0)) ||
                (rm && at(rm, k) >= 0 && at(rm, k) != bb - 1)) {
              out.word[k] |= SP_TABLE;
              again = true;
            }
            bb += mid ? 1 : 0;
          }
        }
        for (size_t k = i; k < e; ++k)
          if ((at(1, k) >= 0 && at(1, k) != (int32_t)k + 1) || (at(2, k) >= 0 && at(2, k) != (int32_t)k - 1)) {
            out.word[k] |= SP_TABLE;
            again = true;
          }
      }
      out.word[i] |= SP_START;
      for (size_t k = i + 1; k < e; ++k) out.word[k] &= ~SP_START;
      out.seg.insert(out.seg.end(), b, b + 8);
      i = e;
    }
  }
}

extern "C" void bl_sparse_destroy(bl_sparse *s) {
  if (!s) return;
  if (s->stream) cudaStreamSynchronize(s->stream);
  if (s->gexec) cudaGraphExecDestroy(s->gexec);
  if (s->gstream) cudaStreamDestroy(s->gstream);
  if (s->ev_fork) cudaEventDestroy(s->ev_fork);
  if (s->ev_join) cudaEventDestroy(s->ev_join);
  void *ptrs[] = {s->sv.pop, (void *)s->sv.word, (void *)s->sv.seg0, (void *)s->sv.seg, (void *)s->sv.table,
                  (void *)s->sv.dense, s->sv.status, s->wa.F, s->wa.K, s->scratch};
  for (void *q : ptrs)
    if (q) cudaFree(q);
  if (s->pin) cudaFreeHost(s->pin);
  delete s;
}

static size_t sp_elem(int dtype) { return dtype == BL_STORE_F32 ? 4 : 2; }

static int sp_check(bl_sparse *s, const char *what) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return sp_fail(s, BL_ECUDA, "%s: %s", what, cudaGetErrorString(e));
  return BL_OK;
}

static void sp_launch_step(bl_sparse *s, cudaStream_t st, int par) {
  const bool force = s->lp.g[0] != 0.0 || s->lp.g[1] != 0.0 || s->lp.g[2] != 0.0;
  const bool tau1 = s->sv.omega == 1.0f;
  if (s->lp.store_dtype == BL_STORE_F32) launch_sparse_typed<float>(s->sv, par, force, tau1, s->wa, st);
  else if (s->lp.store_dtype == BL_STORE_BF16) launch_sparse_typed<__nv_bfloat16>(s->sv, par, force, tau1, s->wa, st);
  else launch_sparse_typed<__half>(s->sv, par, force, tau1, s->wa, st);
}

extern "C" int bl_sparse_init(bl_sparse **out, const bl_lb_params *p, const uint8_t *mask, void *cuda_stream) {
  if (!out) return BL_EINVAL;
  *out = nullptr;
  if (!p || !(p->tau > 0.5) || !(p->rho0 > 0) || p->store_dtype < 0 || p->store_dtype > 2) return BL_EINVAL;
  if (!index_ok(p, mask)) return BL_EINVAL;
  int rc = BL_OK;
  std::vector<int32_t> id((size_t)p->nx * p->ny * p->nz);
  const int64_t nf = index_ids(p, mask, id);
  if (nf < 1 || (unsigned long long)nf * Q >= (1ull << 32)) return BL_EINVAL;
  std::vector<int32_t> dense((size_t)nf), nbr((size_t)nf * 18);
  index_fill(p, id, nf, dense.data(), nbr.data());
  RowIndex rows;
  build_rows(p->nx, p->periodic[0] != 0, dense, nbr, rows);
  bl_sparse *s = new bl_sparse();
  s->lp = *p;
  s->stream = (cudaStream_t)cuda_stream;
  s->sticky = BL_OK;
  s->n_dense = (int64_t)p->nx * p->ny * p->nz;
  SparseView &sv = s->sv;
  sv.Nf = (unsigned)nf;
  for (int w = 0; w < NWALL; ++w)
    for (int k = 0; k < 3; ++k) sv.wall_vel[w][k] = (float)p->wall_vel[w][k];
  sv.omega = (float)(1.0 / p->tau);
  sv.rho0 = (float)p->rho0;
  for (int k = 0; k < 3; ++k) sv.g[k] = (float)p->g[k];
  do {
    // every array is handed to the context as it is made, so that destroy frees it
    auto put = [&](auto *&dst, const void *src, size_t bytes) {
      void *q = nullptr;
      if (cudaMalloc(&q, bytes > 0 ? bytes : 1) != cudaSuccess) return false;
      dst = static_cast<std::remove_reference_t<decltype(dst)>>(q);
      return !src || bytes == 0 ||
             cudaMemcpyAsync(q, src, bytes, cudaMemcpyHostToDevice, s->stream) == cudaSuccess;
    };
    if (!put(sv.pop, nullptr, sp_elem(p->store_dtype) * Q * (size_t)nf) ||
        !put(sv.word, rows.word.data(), sizeof(uint32_t) * rows.word.size()) ||
        !put(sv.seg0, rows.seg0.data(), sizeof(int32_t) * rows.seg0.size()) ||
        !put(sv.seg, rows.seg.data(), sizeof(int32_t) * rows.seg.size()) ||
        !put(sv.table, rows.table.data(), sizeof(int32_t) * rows.table.size()) ||
        !put(sv.dense, dense.data(), sizeof(int32_t) * (size_t)nf) || !put(sv.status, nullptr, sizeof(int)) ||
        !put(s->wa.F, nullptr, sizeof(double) * WALL_COPIES * WALL_SUMS) ||
        !put(s->wa.K, nullptr, sizeof(long long) * WALL_COPIES * WALL_SUMS)) {
      rc = sp_fail(s, BL_ENOMEM, "indexed lattice");
      break;
    }
    if (cudaMallocHost(&s->pin, sizeof(double) * WALL_SUMS) != cudaSuccess) {
      rc = sp_fail(s, BL_ENOMEM, "pinned memory");
      break;
    }
    if (cudaStreamCreateWithFlags(&s->gstream, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&s->ev_fork, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&s->ev_join, cudaEventDisableTiming) != cudaSuccess) {
      rc = sp_fail(s, BL_ECUDA, "streams");
      break;
    }
    if (cudaMemsetAsync(sv.status, 0, sizeof(int), s->stream) != cudaSuccess ||
        cudaMemsetAsync(s->wa.F, 0, sizeof(double) * WALL_COPIES * WALL_SUMS, s->stream) != cudaSuccess ||
        cudaMemsetAsync(s->wa.K, 0, sizeof(long long) * WALL_COPIES * WALL_SUMS, s->stream) != cudaSuccess) {
      rc = sp_fail(s, BL_ECUDA, "upload");
      break;
    }
    const unsigned b = 256, g = nblk(sv.Nf, b);
    if (p->store_dtype == BL_STORE_F32) k_sparse_rest<float><<<g, b, 0, s->stream>>>(sv);
    else if (p->store_dtype == BL_STORE_BF16) k_sparse_rest<__nv_bfloat16><<<g, b, 0, s->stream>>>(sv);
    else k_sparse_rest<__half><<<g, b, 0, s->stream>>>(sv);
    s->launches++;
    rc = sp_check(s, "init");
    // the host tables go out of scope: wait for their copies
    if (rc == BL_OK && cudaStreamSynchronize(s->stream) != cudaSuccess) rc = sp_fail(s, BL_ECUDA, "init");
  } while (0);
  if (rc != BL_OK) {
    bl_sparse_destroy(s);
    return rc;
  }
  *out = s;
  return BL_OK;
}

extern "C" int bl_sparse_step(bl_sparse *s, int nsteps) {
  if (!s || nsteps < 0) return BL_EINVAL;
  if (s->sticky) return s->sticky;
  int k = 0;
  if (nsteps >= 2) {
    // pairs of steps as one graph launch (the graph starts at its parity)
    if (!s->gexec || s->g_parity != s->parity) {
      if (s->gexec) cudaGraphExecDestroy(s->gexec);
      s->gexec = nullptr;
      cudaGraph_t g = nullptr;
      SPCU(cudaStreamBeginCapture(s->gstream, cudaStreamCaptureModeThreadLocal));
      sp_launch_step(s, s->gstream, s->parity);
      sp_launch_step(s, s->gstream, s->parity ^ 1);
      SPCU(cudaStreamEndCapture(s->gstream, &g));
      const cudaError_t e = cudaGraphInstantiate(&s->gexec, g, 0);
      cudaGraphDestroy(g);
      if (e != cudaSuccess) {
        s->gexec = nullptr;
        return sp_fail(s, BL_ECUDA, "graph instantiate: %s", cudaGetErrorString(e));
      }
      s->g_parity = s->parity;
    }
    SPCU(cudaEventRecord(s->ev_fork, s->stream));
    SPCU(cudaStreamWaitEvent(s->gstream, s->ev_fork, 0));
    for (; k + 2 <= nsteps; k += 2) {
      SPCU(cudaGraphLaunch(s->gexec, s->gstream));
      s->launches += 2;
    }
    SPCU(cudaEventRecord(s->ev_join, s->gstream));
    SPCU(cudaStreamWaitEvent(s->stream, s->ev_join, 0));
  }
  for (; k < nsteps; ++k) {
    sp_launch_step(s, s->stream, s->parity);
    s->parity ^= 1;
    s->launches++;
  }
  return sp_check(s, "step");
}

extern "C" int bl_sparse_sync(bl_sparse *s) {
  if (!s) return BL_EINVAL;
  const cudaError_t e = cudaStreamSynchronize(s->stream);
  if (e != cudaSuccess) return sp_fail(s, BL_ECUDA, "stream: %s", cudaGetErrorString(e));
  if (s->sticky) return s->sticky;
  int st = 0;
  SPCU(cudaMemcpy(&st, s->sv.status, sizeof(int), cudaMemcpyDeviceToHost));
  if (st & ST_UNSTABLE) return sp_fail(s, BL_EUNSTABLE, "unstable: rho <= 0, NaN or |u| >= 0.3 at some node");
  return BL_OK;
}

static int sp_scratch(bl_sparse *s, size_t bytes) {
  if (s->scratch_bytes >= bytes) return BL_OK;
  if (s->scratch) cudaFree(s->scratch);
  s->scratch = nullptr;
  s->scratch_bytes = 0;
  if (cudaMalloc(&s->scratch, bytes) != cudaSuccess) return sp_fail(s, BL_ENOMEM, "scratch");
  s->scratch_bytes = bytes;
  return BL_OK;
}

extern "C" int bl_sparse_fields_get(bl_sparse *s, double *rho, double *u, int on_device) {
  if (!s || (!rho && !u)) return BL_EINVAL;
  if (s->sticky) return s->sticky;
  const size_t N = (size_t)s->n_dense;
  double *dr = rho, *du = u;
  if (!on_device) {
    if (sp_scratch(s, sizeof(double) * 4 * N)) return s->sticky;
    dr = rho ? s->scratch : nullptr;
    du = u ? s->scratch + N : nullptr;
  }
  if (dr) SPCU(cudaMemsetAsync(dr, 0, sizeof(double) * N, s->stream));
  if (du) SPCU(cudaMemsetAsync(du, 0, sizeof(double) * 3 * N, s->stream));
  const unsigned b = 256, g = nblk(s->sv.Nf, b);
  const double r0 = (double)s->sv.rho0, h0 = 0.5 * (double)s->sv.g[0], h1 = 0.5 * (double)s->sv.g[1],
               h2 = 0.5 * (double)s->sv.g[2];
#define BL_SPF(S_) k_sparse_fields<S_><<<g, b, 0, s->stream>>>(s->sv, s->parity, r0, h0, h1, h2, dr, du)
  if (s->lp.store_dtype == BL_STORE_F32) BL_SPF(float);
  else if (s->lp.store_dtype == BL_STORE_BF16) BL_SPF(__nv_bfloat16);
  else BL_SPF(__half);
#undef BL_SPF
  s->launches++;
  if (sp_check(s, "fields")) return s->sticky;
  if (!on_device) {
    if (rho) SPCU(cudaMemcpyAsync(rho, dr, sizeof(double) * N, cudaMemcpyDeviceToHost, s->stream));
    if (u) SPCU(cudaMemcpyAsync(u, du, sizeof(double) * 3 * N, cudaMemcpyDeviceToHost, s->stream));
  }
  return bl_sparse_sync(s);
}

static int sp_pop_io(bl_sparse *s, double *pop, int to_storage) {
  if (!s || !pop) return BL_EINVAL;
  if (s->sticky) return s->sticky;
  const size_t bytes = sizeof(double) * Q * (size_t)s->n_dense;
  if (sp_scratch(s, bytes)) return s->sticky;
  if (to_storage) SPCU(cudaMemcpyAsync(s->scratch, pop, bytes, cudaMemcpyHostToDevice, s->stream));
  else SPCU(cudaMemsetAsync(s->scratch, 0, bytes, s->stream));
  const unsigned b = 256, g = nblk(s->sv.Nf, b);
  if (s->lp.store_dtype == BL_STORE_F32) k_sparse_pop_io<float><<<g, b, 0, s->stream>>>(s->sv, s->parity, s->scratch, to_storage);
  else if (s->lp.store_dtype == BL_STORE_BF16)
    k_sparse_pop_io<__nv_bfloat16><<<g, b, 0, s->stream>>>(s->sv, s->parity, s->scratch, to_storage);
  else k_sparse_pop_io<__half><<<g, b, 0, s->stream>>>(s->sv, s->parity, s->scratch, to_storage);
  s->launches++;
  if (sp_check(s, "populations")) return s->sticky;
  if (!to_storage) SPCU(cudaMemcpyAsync(pop, s->scratch, bytes, cudaMemcpyDeviceToHost, s->stream));
  return bl_sparse_sync(s);
}

extern "C" int bl_sparse_populations_get(bl_sparse *s, double *pop) { return sp_pop_io(s, pop, 0); }

extern "C" int bl_sparse_populations_set(bl_sparse *s, const double *pop) {
  return sp_pop_io(s, const_cast<double *>(pop), 1);
}

extern "C" int bl_sparse_wall_momentum_get(bl_sparse *s, double *wallmom) {
  if (!s || !wallmom) return BL_EINVAL;
  if (s->sticky) return s->sticky;
  launch_wall_read(s->wa, s->lp.rho0, s->pin, s->stream);
  s->launches++;
  if (sp_check(s, "wall momentum")) return s->sticky;
  SPCU(cudaStreamSynchronize(s->stream));
  memcpy(wallmom, s->pin, sizeof(double) * WALL_SUMS);
  return BL_OK;
}

extern "C" int64_t bl_sparse_nodes(const bl_sparse *s) { return s ? (int64_t)s->sv.Nf : -1; }

extern "C" int64_t bl_sparse_launch_count(const bl_sparse *s) { return s ? s->launches : -1; }

extern "C" const char *bl_sparse_last_error(const bl_sparse *s) { return s ? s->err : "null context"; }
