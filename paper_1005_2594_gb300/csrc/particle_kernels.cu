// particle_kernels.cu -- the cell side of the coupled step (arXiv:1005.2594):
//
//   cell list      count -> scan -> scatter -> per-bin sort, canonical (bin, id);
//                  in one block for up to 4096 cells
//   potentials     Berne-Pechukas-scaled Hookean cell-cell pairs (Sec. III,
//                  Eqs. phi, epsilon, sigma) and cell-wall spheres (Eq. sigmaw),
//                  one block per cell, FP64 contact geometry, FP32 forces,
//                  FP64 result
//   link sums      per cell over the link records the sweep wrote (Eq.
//                  deltap): link momentum at the predictor and the drag
//                  matrices
//   solve          four lanes per cell: velocities of the half step (reading
//                  Q3), leap-frog on unit quaternions (reading Q4)
//   second links   the moving-boundary term C (Eq. c) on the rare links to a
//                  node's second cell; the first cell's C is added by the
//                  next sweep as it reads the bounced populations
//   claims         one block per cell, one thread per lattice row: the nodes
//                  the cell's new ellipsoid enters or leaves
//   resolve        first-arrival owner rule (Sec. II single occupancy), then
//                  fill/drain of every changed node with the momentum balance
//                  given to the cells (Sec. II)
//   contacts       contact links of each cell as exact integer sums (Eqs.
//                  deltapppp, deltapppm)
//
// Ownership.  claim[] holds INT_MAX ("free") on every node between steps.
// A cell marks each fluid node its new ellipsoid enters with its index
// (atomicMin: the lowest index among the newcomers) and each node it owns
// but leaves with TOUCHED; both go to the cell's touched list.  Resolve takes
// each claim once (atomicExch back to free): a newcomer index -> that cell;
// TOUCHED -> the lowest-index cell now covering the node, else fluid.  This
// is the first-arrival rule: an owner keeps a node while it covers it.
//
// FP64 is used only where the state needs it (positions, velocities, angular
// momenta, the exact inside test near a surface, the contact geometry of the
// potentials); on this GPU an FP64 instruction holds the SM's FP64 pipe for 16
// cycles whatever number of lanes it has, so sums, the 6 x 6 solve and the
// rotation increment are FP32 around FP64 reference values, and the kernels
// that test nodes against ellipsoids read each cell's position (node + FP32
// fraction) and axis in the FP32 form the solve leaves them.
#include <climits>

#include "bl_internal.cuh"

namespace bl {

constexpr int CLAIM_FREE = INT_MAX;
constexpr int CLAIM_TOUCHED = INT_MAX - 1;
// the FP32 inside test decides when |s - 1| >= this; its error is below
// 1e-5 for cells with half-axis ratios up to 100 (positions carried as an
// integer node plus an FP32 fraction)
constexpr float INSIDE_MARGIN = 1e-4f;

// ---------------------------------------------------------------------------
// cell list

// bin of a coordinate, floor((X / N) nb) with X / N and the product rounded to
// FP64 as the plain reference does: from FP32, whose error is below 4e-7 nb,
// unless the bin's border is that near
__device__ __forceinline__ int axis_bin(double X, int dim, int nb) {
  const float t = (float)X * ((float)nb / (float)dim);
  int b;
  if (fabsf(t - rintf(t)) > 1e-6f * (float)nb + 1e-5f) b = (int)floorf(t);
  else b = (int)floor(__dmul_rn(__ddiv_rn(X, (double)dim), (double)nb));
  return min(max(b, 0), nb - 1);
}

__device__ __forceinline__ int cell_bin(const LatticeView &lv, const PartView &pv, const CellListView &cl, int i) {
  const int b0 = axis_bin(pv.X[3 * i], lv.nx, cl.nb[0]), b1 = axis_bin(pv.X[3 * i + 1], lv.ny, cl.nb[1]),
            b2 = axis_bin(pv.X[3 * i + 2], lv.nz, cl.nb[2]);
  return b0 + cl.nb[0] * (b1 + cl.nb[1] * b2);
}

// The whole list in one block, counts, starts and ids in shared memory: for up
// to CL_ONE cells (and CL_SMEM bytes of bins and cells) the four kernels below were
// four launches of 3 to 4 us each on the way to the potentials, the longest way
// through the step of a small lattice.  Larger lists, which the sweep hides,
// take the four kernels.  256 threads: a block of 1024 needs a whole SM's
// registers, and among the kernels of an ensemble none falls free (16-member
// sweep 368 -> 379 us a step).
constexpr int CL_T = 256, CL_ONE = 4096, CL_PER = CL_ONE / CL_T;
constexpr int CL_WSUM = 32;  // warp sums of the scan
// dynamic shared memory: a block has 48 KB without an opt-in, its static part included
constexpr size_t CL_SMEM = 48 * 1024 - sizeof(int) * CL_WSUM;

__global__ void __launch_bounds__(CL_T) k_cl_one(LatticeView lv, PartView pv, CellListView cl) {
  extern __shared__ int cl_smem[];
  int *cnt = cl_smem, *ids = cl_smem + cl.nbins;
  __shared__ int wsum[CL_WSUM];
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  pdl_trigger();  // the potentials' wall spheres need no list
  for (int b = t; b < cl.nbins; b += CL_T) cnt[b] = 0;
  __syncthreads();
  int bin[CL_PER], slot[CL_PER];
#pragma unroll
  for (int u = 0; u < CL_PER; ++u) {
    const int i = t + CL_T * u;
    if (i < pv.n) {
      bin[u] = cell_bin(lv, pv, cl, i);
      cl.bin_of[i] = bin[u];
      slot[u] = atomicAdd(&cnt[bin[u]], 1);
    }
  }
  __syncthreads();
  // exclusive scan: a run of bins per thread, the runs' sums over the block
  const int per = (cl.nbins + CL_T - 1) / CL_T, b0 = min(t * per, cl.nbins), b1 = min(b0 + per, cl.nbins);
  int sum = 0;
  for (int b = b0; b < b1; ++b) sum += cnt[b];
  int inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += v;
  }
  if (lane == 31) wsum[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    int w = lane < CL_T / 32 ? wsum[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += v;
    }
    wsum[lane] = w;
  }
  __syncthreads();
  int off = (wid > 0 ? wsum[wid - 1] : 0) + inc - sum;
  for (int b = b0; b < b1; ++b) {
    const int c = cnt[b];
    cnt[b] = off;
    cl.start[b] = off;
    off += c;
  }
  if (t == 0) cl.start[cl.nbins] = pv.n;
  __syncthreads();
#pragma unroll
  for (int u = 0; u < CL_PER; ++u)
    if (t + CL_T * u < pv.n) ids[cnt[bin[u]] + slot[u]] = t + CL_T * u;
  __syncthreads();
  for (int b = t; b < cl.nbins; b += CL_T) {
    const int s = cnt[b], e = b + 1 < cl.nbins ? cnt[b + 1] : pv.n;
    for (int i = s + 1; i < e; ++i) {
      const int v = ids[i];
      int j = i - 1;
      while (j >= s && ids[j] > v) {
        ids[j + 1] = ids[j];
        --j;
      }
      ids[j + 1] = v;
    }
  }
  __syncthreads();
  for (int i = t; i < pv.n; i += CL_T) cl.ids[i] = ids[i];
}

__global__ void k_cl_bin(LatticeView lv, PartView pv, CellListView cl) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= pv.n) return;
  const int bin = cell_bin(lv, pv, cl, i);
  cl.bin_of[i] = bin;
  atomicAdd(&cl.count[bin], 1);
}

// one block: exclusive scan of the bin counts into start, clears count/cursor
__global__ void __launch_bounds__(1024) k_cl_scan(CellListView cl) {
  __shared__ int wsum[32];
  __shared__ int carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int base = 0; base < cl.nbins; base += blockDim.x) {
    const int b = base + threadIdx.x;
    const int v = b < cl.nbins ? cl.count[b] : 0;
    int inc = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    if (lane == 31) wsum[wid] = inc;
    __syncthreads();
    if (wid == 0) {
      int w = lane < (int)(blockDim.x >> 5) ? wsum[lane] : 0;
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, w, o);
        if (lane >= o) w += t;
      }
      wsum[lane] = w;
    }
    __syncthreads();
    const int excl = carry + (wid > 0 ? wsum[wid - 1] : 0) + inc - v;
    if (b < cl.nbins) {
      cl.start[b] = excl;
      cl.count[b] = 0;
      cl.cursor[b] = 0;
    }
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry = excl + v;
    __syncthreads();
  }
  if (threadIdx.x == 0) cl.start[cl.nbins] = carry;
}

__global__ void k_cl_scatter(PartView pv, CellListView cl) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= pv.n) return;
  const int bin = cl.bin_of[i];
  const int slot = atomicAdd(&cl.cursor[bin], 1);
  cl.ids[cl.start[bin] + slot] = i;
}

__global__ void k_cl_sort(CellListView cl) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= cl.nbins) return;
  const int s = cl.start[b], e = cl.start[b + 1];
  for (int i = s + 1; i < e; ++i) {
    const int v = cl.ids[i];
    int j = i - 1;
    while (j >= s && cl.ids[j] > v) {
      cl.ids[j + 1] = cl.ids[j];
      --j;
    }
    cl.ids[j + 1] = v;
  }
}

// ---------------------------------------------------------------------------
// potentials (FP32)

// Contact geometry in FP64.  In contact the overlap h = 1 - r / sigma is a
// small difference of O(1) numbers (h ~ 1e-2), and the force is
// proportional to it: rounding r and sigma to FP32 (~1e-7) would put ~1e-5
// into the force.  With sigma = sigma_bar / sqrt(S) and P = r^2 S,
//   h = (sigma_bar^2 - P) / (sigma_bar (sigma_bar + sqrt(P))),
//   sigma = sigma_bar r / sqrt(P),
// so the one difference is formed from products of the positions and axes
// without a root or a normalised vector.  h, sigma and S are formed in FP64 and
// rounded to FP32 once (their quotients in FP32 raised the force's error from
// 8.6e-8 to 1.0e-7 rms).  FP64 reciprocals (Newton from the FP32 one) replace
// roots and divisions of some 20 FP64 instructions each: two steps where the
// result enters the difference, one where it is rounded to FP32 next.  The
// contact geometry was 170 FP64 instructions per warp, each holding the SM's
// FP64 pipe for 16 cycles, and bound the kernel (104 us on 256^3 with 8446
// cells).  The strength, its derivatives and the force and torque, which
// multiply h without cancelling it, are FP32.

// 1 / x in FP64 to about an ulp, or (STEPS = 1) to 2^-43, for x within FP32's range
template <int STEPS>
__device__ __forceinline__ double rcp64(double x) {
  double y = (double)(1.0f / (float)x);
#pragma unroll
  for (int k = 0; k < STEPS; ++k) y = fma(y, fma(-x, y, 1.0), y);
  return y;
}
// 1 / sqrt(x) to 2^-43 (below FP32's range the root and quotient themselves)
__device__ __forceinline__ double rsqrt64(double x) {
  if (!(x > 1e-30)) return 1.0 / sqrt(x);
  const double y = (double)rsqrtf((float)x);
  return fma(0.5 * y, fma(-x * y, y, 1.0), y);
}
__device__ __forceinline__ double dot64(const double a[3], const double b[3]) {
  return fma(a[2], b[2], fma(a[1], b[1], a[0] * b[0]));
}

// h and sigma from sigma_bar^2 - P (> 0), P and r
__device__ __forceinline__ void overlap(double D, double P, double r, double sigbar, float &h, float &sigma) {
  const double y = rsqrt64(P);
  h = (float)(D * rcp64<1>(sigbar * fma(P, y, sigbar)));
  sigma = (float)(sigbar * (r * y));
}

// FP32 test of a pair against its contact distance (Eq. sigma) with a
// relative margin of 1e-4: false only for pairs certainly out of contact
__device__ __forceinline__ bool near_contact(const float r[3], float r2, const float oi[3], const float oj[3],
                                             const PartView &pv) {
  if (!(r2 > 0.f)) return false;
  const float ir = rsqrtf(r2);
  const float a = (r[0] * oi[0] + r[1] * oi[1] + r[2] * oi[2]) * ir;
  const float b = (r[0] * oj[0] + r[1] * oj[1] + r[2] * oj[2]) * ir;
  const float c = oi[0] * oj[0] + oi[1] * oj[1] + oi[2] * oj[2];
  const float chi = pv.chi, ap = a + b, am = a - b;
  const float S = 1.0f - 0.5f * chi * (ap * ap / (1.0f + chi * c) + am * am / (1.0f - chi * c));
  return r2 * S < pv.sigbar * pv.sigbar * 1.0002f;  // r < sigma_bar / sqrt(S) (1 + 1e-4)
}

// cell-cell pair, force and torque on i; r = X_j - X_i (Eqs. phi, epsilon,
// sigma; the Gay-Berne factor eps2^mu of the variant)
__device__ __forceinline__ void bp_pair(const double rd[3], const double oid[3], const double ojd[3],
                                        const float oi[3], const float oj[3], const PartView &pv, float F[3],
                                        float T[3]) {
  const double r2 = dot64(rd, rd);
  if (!(r2 > 0.0)) return;
  const double A = dot64(rd, oid), B = dot64(rd, ojd), cd = dot64(oid, ojd);
  const double Ap = A + B, Am = A - B, qp = fma(pv.chi_d, cd, 1.0), qm = fma(-pv.chi_d, cd, 1.0);
  // (A + B)^2 / (1 + chi c) + (A - B)^2 / (1 - chi c)
  const double X = fma(Ap * Ap, qm, Am * Am * qp) * rcp64<2>(qp * qm);
  const double P = fma(-0.5 * pv.chi_d, X, r2), D = pv.sigbar_d * pv.sigbar_d - P;
  if (!(D > 0.0)) return;
  const double ird = rsqrt64(r2), rld = r2 * ird;
  float h, sigma;
  overlap(D, P, rld, pv.sigbar_d, h, sigma);
  const float rl = (float)rld, ir = (float)ird, S = (float)(P * (ird * ird));
  const float rh[3] = {(float)(rd[0] * ird), (float)(rd[1] * ird), (float)(rd[2] * ird)};
  const float a = (float)(A * ird), b = (float)(B * ird), c = (float)cd;
  const float chi = pv.chi;
  const float ap = (float)(Ap * ird), am = (float)(Am * ird);
  const float dp = 1.0f + chi * c, dm = 1.0f - chi * c;
  const float e1 = 1.0f - chi * chi * c * c;
  float eps = pv.eps * (pv.nu == 1.0f ? rsqrtf(e1) : powf(e1, -0.5f * pv.nu));
  float e2 = 1.0f, de2a = 0.f, de2b = 0.f, de2c = 0.f;
  if (pv.mu != 0.0f) {
    const float cp = pv.chi_prime;
    const float qp = 1.0f + cp * c, qm = 1.0f - cp * c;
    e2 = 1.0f - 0.5f * cp * (ap * ap / qp + am * am / qm);
    de2a = -cp * (ap / qp + am / qm);
    de2b = -cp * (ap / qp - am / qm);
    de2c = 0.5f * cp * cp * (ap * ap / (qp * qp) - am * am / (qm * qm));
    eps *= powf(e2, pv.mu);
  }
  const float dSa = -chi * (ap / dp + am / dm);
  const float dSb = -chi * (ap / dp - am / dm);
  const float dSc = 0.5f * chi * chi * (ap * ap / (dp * dp) - am * am / (dm * dm));
  const float eps_a = pv.mu != 0.0f ? eps * pv.mu * de2a / e2 : 0.f;
  const float eps_b = pv.mu != 0.0f ? eps * pv.mu * de2b / e2 : 0.f;
  const float eps_c = eps * (pv.nu * chi * chi * c / e1 + (pv.mu != 0.0f ? pv.mu * de2c / e2 : 0.f));
  const float k = eps * h * rl / (sigma * S);
  const float phi_r = -2.0f * eps * h / sigma;
  const float phi_a = h * h * eps_a - k * dSa;
  const float phi_b = h * h * eps_b - k * dSb;
  const float phi_c = h * h * eps_c - k * dSc;
  float dpi[3];
  for (int m = 0; m < 3; ++m) {
    F[m] += phi_r * rh[m] + (phi_a * (oi[m] - a * rh[m]) + phi_b * (oj[m] - b * rh[m])) * ir;
    dpi[m] = phi_a * rh[m] + phi_c * oj[m];
  }
  T[0] -= oi[1] * dpi[2] - oi[2] * dpi[1];
  T[1] -= oi[2] * dpi[0] - oi[0] * dpi[2];
  T[2] -= oi[0] * dpi[1] - oi[1] * dpi[0];
}

// cell-wall sphere (Eq. sigmaw), force and torque on the cell; r = x_wall - X
__device__ __forceinline__ void bp_wall(const double rd[3], const double oid[3], const float oi[3],
                                        const PartView &pv, float F[3], float T[3]) {
  const double r2 = dot64(rd, rd);
  if (!(r2 > 0.0)) return;
  const double A = dot64(rd, oid);
  const double P = fma(-pv.chi_w_d * A, A, r2), D = pv.sigbar_w_d * pv.sigbar_w_d - P;
  if (!(D > 0.0)) return;
  const double ird = rsqrt64(r2), rld = r2 * ird;
  float h, sigma;
  overlap(D, P, rld, pv.sigbar_w_d, h, sigma);
  const float rl = (float)rld, ir = (float)ird, S = (float)(P * (ird * ird)), a = (float)(A * ird);
  const float rh[3] = {(float)(rd[0] * ird), (float)(rd[1] * ird), (float)(rd[2] * ird)};
  const float eps = pv.eps_w;
  const float dsig_a = sigma * pv.chi_w * a / S;
  const float phi_r = -2.0f * eps * h / sigma;
  const float phi_a = 2.0f * eps * h * rl / (sigma * sigma) * dsig_a;
  for (int m = 0; m < 3; ++m) F[m] += phi_r * rh[m] + phi_a * (oi[m] - a * rh[m]) * ir;
  const float dpo[3] = {phi_a * rh[0], phi_a * rh[1], phi_a * rh[2]};
  T[0] -= oi[1] * dpo[2] - oi[2] * dpo[1];
  T[1] -= oi[2] * dpo[0] - oi[0] * dpo[2];
  T[2] -= oi[0] * dpo[1] - oi[1] * dpo[0];
}

// neighbour-bin offsets along one axis without duplicates
__device__ __forceinline__ int bin_offsets(int nb, int per, int b, int out[3]) {
  if (nb == 1) {
    out[0] = 0;
    return 1;
  }
  if (nb == 2 && per) {
    out[0] = 0;
    out[1] = 1;
    return 2;
  }
  int k = 0;
  for (int d = -1; d <= 1; ++d) {
    const int v = b + d;
    if (!per && (v < 0 || v >= nb)) continue;
    out[k++] = d;
  }
  return k;
}

// the cells of the bins around bin bc, numbered through: off[b] is the number
// of the first cell of neighbouring bin b, start[b] its place in the cell list.
// A thread per bin that walks its cells alone takes as many dependent reads as
// the fullest bin holds; numbered through, the cells are read one per thread.
struct NearBins {
  int off[28], start[27];
};

// (one whole warp)
__device__ __forceinline__ void near_bins(const LatticeView &lv, const CellListView &cl, int bin, NearBins &nbs) {
  const int lane = threadIdx.x & 31;
  const int bc[3] = {bin % cl.nb[0], (bin / cl.nb[0]) % cl.nb[1], bin / (cl.nb[0] * cl.nb[1])};
  int off[3][3], noff[3];
  for (int k = 0; k < 3; ++k) noff[k] = bin_offsets(cl.nb[k], lv.per[k], bc[k], off[k]);
  const int ix = lane % 3, iy = (lane / 3) % 3, iz = lane / 9;
  int s = 0, n = 0;
  if (lane < 27 && ix < noff[0] && iy < noff[1] && iz < noff[2]) {
    const int b = wrapi(bc[0] + off[0][ix], cl.nb[0]) +
                  cl.nb[0] * (wrapi(bc[1] + off[1][iy], cl.nb[1]) + cl.nb[1] * wrapi(bc[2] + off[2][iz], cl.nb[2]));
    s = cl.start[b];
    n = cl.start[b + 1] - s;
  }
  int inc = n;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane < 27) {
    nbs.off[lane] = inc - n;
    nbs.start[lane] = s;
    if (lane == 26) nbs.off[27] = inc;
  }
}

// cell number t (0 <= t < off[27])
__device__ __forceinline__ int near_cell(const CellListView &cl, const NearBins &nbs, int t) {
  int b = 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    if (b + o < 27 && nbs.off[b + o] <= t) b += o;
  return cl.ids[nbs.start[b] + t - nbs.off[b]];
}

// ---------------------------------------------------------------------------
// block-wide helpers (blockDim.x == 256)

constexpr int CB = 256;

// sums v over a block of NT threads; the result is valid in thread 0
template <int K, int NT = CB>
__device__ __forceinline__ void block_sum(float (&v)[K], float (*sh)[K]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < K; ++k) v[k] = warp_sum(v[k]);
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) sh[wid][k] = v[k];
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < NT / 32; ++w)
#pragma unroll
      for (int k = 0; k < K; ++k) v[k] += sh[w][k];
  __syncthreads();
}

template <int K, int NT = CB>
__device__ __forceinline__ void block_sum_i(int (&v)[K], int (*sh)[K]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < K; ++k) v[k] = __reduce_add_sync(0xffffffffu, v[k]);
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) sh[wid][k] = v[k];
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < NT / 32; ++w)
#pragma unroll
      for (int k = 0; k < K; ++k) v[k] += sh[w][k];
  __syncthreads();
}

// block-wide exclusive scan of one int per thread; returns the thread's
// offset, writes the total to *total (all threads)
template <int NT = CB>
__device__ __forceinline__ int block_scan(int v, int *sh_w, int *total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) sh_w[wid] = inc;
  __syncthreads();
  if (threadIdx.x == 0) {
    int s = 0;
    for (int w = 0; w < NT / 32; ++w) {
      const int t = sh_w[w];
      sh_w[w] = s;
      s += t;
    }
    sh_w[NT / 32] = s;
  }
  __syncthreads();
  const int off = sh_w[wid] + inc - v;
  *total = sh_w[NT / 32];
  __syncthreads();
  return off;
}

// per-warp append to a list whose length lives in shared memory: returns the
// first slot of this lane's cnt entries (one shared atomic per warp)
__device__ __forceinline__ int warp_append(int cnt, int *sh_len) {
  const int lane = threadIdx.x & 31;
  int inc = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  const int tot = __shfl_sync(0xffffffffu, inc, 31);
  int base = 0;
  if (lane == 31 && tot) base = atomicAdd(sh_len, tot);
  base = __shfl_sync(0xffffffffu, base, 31);
  return base + inc - cnt;
}

__device__ __forceinline__ unsigned node_of(const LatticeView &lv, int x, int y, int z) {
  return (unsigned)x + (unsigned)lv.nx * ((unsigned)y + (unsigned)lv.ny * z);
}

// slot where the sweep of parity par bounced direction r of fluid node y
__device__ __forceinline__ unsigned bounce_slot(const LatticeView &lv, int par, unsigned y, const int yc[3], int r) {
  if (par == 0) {
    const unsigned nb = node_of(lv, wrapi(yc[0] + rt_c<0>(r), lv.nx), wrapi(yc[1] + rt_c<1>(r), lv.ny),
                                wrapi(yc[2] + rt_c<2>(r), lv.nz));
    return (unsigned)r * lv.N + nb;
  }
  return (unsigned)rt_opp(r) * lv.N + y;
}

// ---------------------------------------------------------------------------
// potentials: one block per cell; all threads take the rows (y, z) of the
// wall-sphere range around the cell, then the cells around it.

constexpr int FB = 128;        // threads of a potentials block
constexpr int FQ_PAIR = 128;   // per-cell queue of pairs within contact reach
constexpr int FQ_WALL = 1024;  // per-cell queue of surface wall nodes within reach

// One block per cell.  The search runs in FP32 and queues what can be in
// contact: the cells j of the 27 bins around cell i within the largest
// contact distance (one thread per cell), and the surface wall nodes within
// the wall sphere's radius (rows without a surface wall node skipped by
// their row bit).  The queued pairs and wall nodes then get the FP64 contact
// geometry with one queue entry per thread, so that the few contacts of a
// cell share the FP64 instructions instead of each taking a pass of its own.
// A full queue evaluates the rest where they are found.
__global__ void __launch_bounds__(FB, 7) k_forces(LatticeView lv, PartView pv, CellListView cl, SurfBits sb) {
  __shared__ float sh[FB / 32][6];
  __shared__ int s_np, s_nw;
  __shared__ int s_pair[FQ_PAIR];
  __shared__ unsigned s_wall[FQ_WALL];
  __shared__ NearBins s_nb;
  const int i = blockIdx.x;
  if (threadIdx.x == 0) {
    s_np = 0;
    s_nw = 0;
  }
  __syncthreads();
  const float4 a0 = pv.kin[3 * i], a1 = pv.kin[3 * i + 1], a2 = pv.kin[3 * i + 2];
  const int Xi[3] = {(int)a0.w, (int)a1.w, (int)a2.w};
  const float fi[3] = {a0.x, a0.y, a0.z};
  const float4 ax = pv.axis[i];
  const float oif[3] = {ax.x, ax.y, ax.z};
  const int dims[3] = {lv.nx, lv.ny, lv.nz};
  float F[3] = {0.f, 0.f, 0.f}, T[3] = {0.f, 0.f, 0.f};
  // the FP64 state (of the step's start: the solve rewrites it only after the
  // join) is read where a contact is evaluated; the periodic image comes from
  // the nearest nodes, in integers, but in a box so short that a contact can
  // reach half a period (near_image)
  auto pair_force = [&](int j) {
    const int Xj[3] = {(int)pv.kin[3 * j].w, (int)pv.kin[3 * j + 1].w, (int)pv.kin[3 * j + 2].w};
    double rd[3];
    for (int m = 0; m < 3; ++m) {
      const double d = __dsub_rn(pv.X[3 * j + m], pv.X[3 * i + m]);
      const int dn = Xj[m] - Xi[m];
      rd[m] = pv.near_image ? min_image_exact(d, dims[m], lv.per[m]) : d + (double)(imin_image(dn, dims[m], lv.per[m]) - dn);
    }
    const double oid[3] = {pv.o[3 * i], pv.o[3 * i + 1], pv.o[3 * i + 2]};
    const double ojd[3] = {pv.o[3 * j], pv.o[3 * j + 1], pv.o[3 * j + 2]};
    const float4 aj = pv.axis[j];
    const float oj[3] = {aj.x, aj.y, aj.z};
    bp_pair(rd, oid, ojd, oif, oj, pv, F, T);
  };
  // the wall node at offsets (dx, oy, oz) from rint(X); queued packed in
  // 3 x 10 bits (offsets within +-511, else evaluated where found)
  auto wall_force = [&](int dx, int oy, int oz) {
    const double oid[3] = {pv.o[3 * i], pv.o[3 * i + 1], pv.o[3 * i + 2]};
    const double rd[3] = {(double)(dx + Xi[0]) - pv.X[3 * i], (double)(oy + Xi[1]) - pv.X[3 * i + 1],
                          (double)(oz + Xi[2]) - pv.X[3 * i + 2]};
    bp_wall(rd, oid, oif, pv, F, T);
  };
  if (sb.bits) {
    const int R = (int)ceilf(pv.sigw_max) + 1;
    const int side = 2 * R + 1;
    const float rw2 = pv.sigw_max * pv.sigw_max;
    const bool packable = R <= 511;
    for (int t = threadIdx.x; t < side * side; t += FB) {
      const int oy = t % side - R, oz = t / side - R;  // node offsets from rint(X)
      int y = Xi[1] + oy, z = Xi[2] + oz;
      const float ry = (float)oy - fi[1], rz = (float)oz - fi[2];
      if (ry * ry + rz * rz >= rw2) continue;
      if (lv.per[1]) y = wrapi(y, lv.ny);
      else if (y < 0 || y >= lv.ny) continue;
      if (lv.per[2]) z = wrapi(z, lv.nz);
      else if (z < 0 || z >= lv.nz) continue;
      const unsigned ri = (unsigned)y + (unsigned)lv.ny * (unsigned)z;
      if (!((sb.rows[ri >> 5] >> (ri & 31)) & 1u)) continue;  // no surface wall node in the row
      const uint32_t *row = sb.bits + (size_t)ri * sb.nxw;
      for (int dx = -R; dx <= R; ++dx) {
        int x = Xi[0] + dx;
        if (lv.per[0]) x = wrapi(x, lv.nx);
        else if (x < 0 || x >= lv.nx) continue;
        if (!((row[x >> 5] >> (x & 31)) & 1u)) continue;
        // FP32 test against the wall sphere's radius first (margin 1e-4)
        const float rx = (float)dx - fi[0];
        const float r2 = rx * rx + ry * ry + rz * rz;
        const float af = rx * oif[0] + ry * oif[1] + rz * oif[2];
        if (!(r2 > 0.f) || (r2 - pv.chi_w * af * af) >= pv.sigbar_w * pv.sigbar_w * 1.0002f) continue;
        const int q = packable ? atomicAdd(&s_nw, 1) : FQ_WALL;
        if (q < FQ_WALL) s_wall[q] = (unsigned)(dx + 512) | ((unsigned)(oy + 512) << 10) | ((unsigned)(oz + 512) << 20);
        else wall_force(dx, oy, oz);
      }
    }
  }
  pdl_wait();  // the cell list
  if (threadIdx.x < 32) near_bins(lv, cl, cl.bin_of[i], s_nb);
  __syncthreads();
  const float rc2 = pv.r_cut * pv.r_cut;
  const float smax = 2.0f * fmaxf(pv.sig_par, pv.sig_perp);
  const float smax2 = smax * smax * 1.0001f;
  for (int t = threadIdx.x; t < s_nb.off[27]; t += FB) {
    const int j = near_cell(cl, s_nb, t);
    if (j == i) continue;
    const float4 b0 = pv.kin[3 * j], b1 = pv.kin[3 * j + 1], b2 = pv.kin[3 * j + 2], aj = pv.axis[j];
    const int Xj[3] = {(int)b0.w, (int)b1.w, (int)b2.w};
    const float fj[3] = {b0.x, b0.y, b0.z};
    float r[3];
    if (pv.near_image)
      for (int m = 0; m < 3; ++m) r[m] = image_f(Xj[m] - Xi[m], fj[m] - fi[m], dims[m], lv.per[m]);
    else
      for (int m = 0; m < 3; ++m) r[m] = (float)imin_image(Xj[m] - Xi[m], dims[m], lv.per[m]) + (fj[m] - fi[m]);
    const float r2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2];
    // no contact distance exceeds 2 max(sigma_perp, sigma_par); nearer
    // pairs first get the contact distance in FP32 (its error is ~1e-6
    // relative, far inside the margin): only pairs at or within contact
    // take the FP64 geometry
    if (r2 >= rc2 || r2 > smax2) continue;
    const float oj[3] = {aj.x, aj.y, aj.z};
    if (!near_contact(r, r2, oif, oj, pv)) continue;
    const int q = atomicAdd(&s_np, 1);
    if (q < FQ_PAIR) s_pair[q] = j;
    else pair_force(j);
  }
  __syncthreads();
  // the queued contacts, one per thread
  const int np = min(s_np, FQ_PAIR), nw = min(s_nw, FQ_WALL);
  for (int k = threadIdx.x; k < np; k += FB) pair_force(s_pair[k]);
  for (int k = threadIdx.x; k < nw; k += FB) {
    const unsigned w = s_wall[k];
    wall_force((int)(w & 1023u) - 512, (int)((w >> 10) & 1023u) - 512, (int)(w >> 20) - 512);
  }
  float v[6] = {F[0], F[1], F[2], T[0], T[1], T[2]};
  block_sum<6, FB>(v, sh);
  if (threadIdx.x == 0)
    for (int m = 0; m < 3; ++m) {
      pv.Fpot[3 * i + m] = (double)v[m];
      pv.Tpot[3 * i + m] = (double)v[3 + m];
    }
}

// ---------------------------------------------------------------------------
// rigid-body helpers

__device__ void rotmat_f(const float4 &q, float R[3][3]) {
  const float w = q.x, x = q.y, y = q.z, z = q.w;
  R[0][0] = 1 - 2 * (y * y + z * z); R[0][1] = 2 * (x * y - w * z);     R[0][2] = 2 * (x * z + w * y);
  R[1][0] = 2 * (x * y + w * z);     R[1][1] = 1 - 2 * (x * x + z * z); R[1][2] = 2 * (y * z - w * x);
  R[2][0] = 2 * (x * z - w * y);     R[2][1] = 2 * (y * z + w * x);     R[2][2] = 1 - 2 * (x * x + y * y);
}

// I_lab = R diag(I_perp, I_perp, I_par) R^T and its inverse (FP32)
__device__ void inertia_f(const PartView &pv, const double q[4], float I[3][3], float Iinv[3][3]) {
  float R[3][3];
  rotmat_f(make_float4((float)q[0], (float)q[1], (float)q[2], (float)q[3]), R);
  const float d[3] = {(float)pv.Iperp, (float)pv.Iperp, (float)pv.Ipar};
  const float di[3] = {1.0f / d[0], 1.0f / d[1], 1.0f / d[2]};
  for (int a = 0; a < 3; ++a)
    for (int b = 0; b < 3; ++b) {
      I[a][b] = R[a][0] * d[0] * R[b][0] + R[a][1] * d[1] * R[b][1] + R[a][2] * d[2] * R[b][2];
      Iinv[a][b] = R[a][0] * di[0] * R[b][0] + R[a][1] * di[1] * R[b][1] + R[a][2] * di[2] * R[b][2];
    }
}

__device__ void write_kin(const PartView &pv, int p, const double X[3], const double V[3], const double Om[3]) {
  double Xi[3], f[3];
  for (int k = 0; k < 3; ++k) {
    Xi[k] = rint(X[k]);
    f[k] = X[k] - Xi[k];
  }
  pv.kin_next[3 * p + 0] = make_float4((float)f[0], (float)f[1], (float)f[2], (float)Xi[0]);
  pv.kin_next[3 * p + 1] = make_float4((float)V[0], (float)V[1], (float)V[2], (float)Xi[1]);
  pv.kin_next[3 * p + 2] = make_float4((float)Om[0], (float)Om[1], (float)Om[2], (float)Xi[2]);
}

// node range of an ellipsoid along one axis (centre x, axis component o)
__device__ __forceinline__ void aabb1(const PartView &pv, float x, float o, int &lo, int &hi) {
  const float h2 = pv.Rperp2_f * (1.0f - o * o) + pv.Rpar2_f * o * o;
  const float h = h2 * rsqrtf(h2) + 0.01f;  // the root to 2 ulp
  lo = (int)floorf(x - h);
  hi = (int)ceilf(x + h);
}

__device__ void aabb(const PartView &pv, const double X[3], const double o[3], int lo[3], int hi[3]) {
  for (int k = 0; k < 3; ++k) {
    const float ok = (float)o[k];
    aabb1(pv, (float)X[k], ok, lo[k], hi[k]);
  }
}

// position (nearest node + fraction) and axis of a cell in FP32, as the solve
// leaves them (kin: the kinematics that belong to the position, axis).  Formed
// from the FP64 state by every thread, they took 68 % of the FP64 pipe in the
// claims and most of the owner search.
struct CellGeo {
  float Xf[3], of[3];
  int Xi[3];
};

__device__ __forceinline__ void cell_geo(const PartView &pv, const float4 *kin, int p, CellGeo &g) {
  const float4 a = kin[3 * p], o = pv.axis[p];
  g.Xf[0] = a.x;
  g.Xf[1] = a.y;
  g.Xf[2] = a.z;
  g.Xi[0] = (int)a.w;
  g.Xi[1] = (int)kin[3 * p + 1].w;
  g.Xi[2] = (int)kin[3 * p + 2].w;
  g.of[0] = o.x;
  g.of[1] = o.y;
  g.of[2] = o.z;
}

// inside test of cell p: FP32 filter, exact FP64 re-evaluation near the surface
__device__ __forceinline__ bool inside_cell(int x, int y, int z, int p, const CellGeo &g, const PartView &pv,
                                            const LatticeView &lv) {
  const float d0 = (float)imin_image(x - g.Xi[0], lv.nx, lv.per[0]) - g.Xf[0];
  const float d1 = (float)imin_image(y - g.Xi[1], lv.ny, lv.per[1]) - g.Xf[1];
  const float d2 = (float)imin_image(z - g.Xi[2], lv.nz, lv.per[2]) - g.Xf[2];
  const float dpar = d0 * g.of[0] + d1 * g.of[1] + d2 * g.of[2];
  const float dd = d0 * d0 + d1 * d1 + d2 * d2;
  const float s = dpar * dpar * pv.inv_rpar2_f + (dd - dpar * dpar) * pv.inv_rperp2_f;
  if (fabsf(s - 1.0f) >= INSIDE_MARGIN) return s < 1.0f;
  return inside_exact(x, y, z, pv.X + 3 * p, pv.o + 3 * p, pv.inv_rpar2, pv.inv_rperp2, lv);
}

// lever arm of a node from the centre of cell p in FP64: the image of the node
// nearest the cell chosen in integers, one conversion and one subtraction per
// axis, but within half a node of half a period by the exact position (SET: a node
// left by a cell that was set elsewhere; in a step a node is within max(R) + 1 of
// the cell's nearest node, and a period is 2 max(R) + 4 at least)
template <bool SET>
__device__ __forceinline__ void arm64(const LatticeView &lv, const PartView &pv, const float4 *kin, int p,
                                      const int xyz[3], double a[3]) {
  const int Xi[3] = {(int)kin[3 * p].w, (int)kin[3 * p + 1].w, (int)kin[3 * p + 2].w};
  const int dims[3] = {lv.nx, lv.ny, lv.nz};
  for (int k = 0; k < 3; ++k) {
    const int m = imin_image(xyz[k] - Xi[k], dims[k], lv.per[k]);
    if (SET && lv.per[k] && 2 * abs(m) >= dims[k] - 1)
      a[k] = min_image_exact(__dsub_rn((double)xyz[k], pv.X[3 * p + k]), dims[k], 1);
    else
      a[k] = __dsub_rn((double)(Xi[k] + m), pv.X[3 * p + k]);
  }
}

// ---------------------------------------------------------------------------
// implicit coupling (reading Q3).  The sweep bounced each cell's links
// without C and wrote one record per (fluid node, cell) into the cell's
// bucket.  With the predictor (Vp, Wp) = velocities of t-1/2 the link
// momentum is (2 f*_r + C(Vp, Wp)) c_r; the reduction sums it (variable part
// in FP32, 2 alpha_r rho_bar c_r as exact integers) with the drag matrices
// Z = sum (m_r / 6) rho [c; a x c][c; a x c]^T.  The half-step velocities
// V = Vp + dV, W = Wp + dW solve
//   (m + Zff) dV + Zft dW = F_tot(Vp, Wp) - m (Vp - V(t-1/2))
//   Ztf dV + (I + Ztt) dW = T_tot(Vp, Wp) + L(t-1/2) - I Wp,
// and the bounced populations get C(V, W) (the next sweep adds it as it
// reads them), so the fluid and the cell exchange the same momentum.
//
// All links of one node into a cell share d = y - X: the arm of link r is
// a_r = d + c_r / 2 and a_r x c_r = d x c_r.  So a record (rho, mask, F_raw =
// sum over the mask of 2 f~*_r c_r) gives
//   F0 = F_raw - rho M v_p,  T0 = d x F0,  v_p = Vp + Wp x d,
//   Zff = rho M,  Zft = rho M [d]x^T,  Ztt = [d]x rho M [d]x^T,
// with M = sum over the mask of (m_r / 6) c_r c_r^T, and the constant parts
// K = sum m_r c_r, IT = d_int x K with d_int = y - rint(X) exactly.  At
// tau = 1 the record holds the node's moments instead of F_raw, and the
// bounced populations f~*_r are evaluated again here by the function the
// sweep collides with.

// One block per cell over its bucket.  Bound by issue: about 480 warp
// instructions per 32 records, 62 % of the issue slots busy (14.7 us for 628k
// records of 1022 cells; 83 us, half of that HBM, for 5.2 M of 8446).  The pair
// terms replaced a loop over each record's directions (18.6 us at 1022 cells,
// 123 at 8446).
constexpr int LT = 128;  // threads of a link-reduction block
// blocks of the link reduction and of the claims resident per SM: enough
// that one wave holds a thousand cells (the register cap this sets)
#ifndef BL_REDUCE_MINB
#define BL_REDUCE_MINB 7
#endif
#ifndef BL_CLAIMS_MINB
#define BL_CLAIMS_MINB 7
#endif
template <bool FORCE>
__global__ void __launch_bounds__(LT, BL_REDUCE_MINB) k_link_reduce(LatticeView lv, PartView pv) {
  __shared__ float shf[LT / 32][27];
  __shared__ int shi[LT / 32][6];
  const int p = blockIdx.x;
  pdl_trigger();  // the solve's blocks read the cells' state meanwhile
  const int nrec = min(lv.rec_count[p], lv.rec_cap);
  const float4 k0 = pv.kin[3 * p], k1 = pv.kin[3 * p + 1], k2 = pv.kin[3 * p + 2];
  const int Xi[3] = {(int)k0.w, (int)k1.w, (int)k2.w};
  float v[27];
  int iv[6];
#pragma unroll
  for (int k = 0; k < 27; ++k) v[k] = 0.f;
#pragma unroll
  for (int k = 0; k < 6; ++k) iv[k] = 0;
  const float4 *rec = lv.rec + 2 * (size_t)p * lv.rec_cap;
  const bool tau1 = lv.omega == 1.0f;  // the sweep's records hold moments (tau = 1) or link sums
  for (int i = threadIdx.x; i < nrec; i += LT) {
    const float4 r0 = rec[i], r1 = rec[lv.rec_cap + i];
    const unsigned n = __float_as_uint(r0.x);
    const uint32_t m = __float_as_uint(r0.y) & NB_SOLID;
    const float rho = lv.rho0 + r0.z;
    int yc[3];
    node_xyz(lv, n, yc);
    const int di[3] = {imin_image(yc[0] - Xi[0], lv.nx, lv.per[0]), imin_image(yc[1] - Xi[1], lv.ny, lv.per[1]),
                       imin_image(yc[2] - Xi[2], lv.nz, lv.per[2])};
    const float d[3] = {(float)di[0] - k0.x, (float)di[1] - k0.y, (float)di[2] - k0.z};
    // rho M and K from the mask
    const float w6 = rho * (1.0f / 6.0f);
    const float Axx = w6 * (float)mask_Maa<0>(m), Ayy = w6 * (float)mask_Maa<1>(m), Azz = w6 * (float)mask_Maa<2>(m);
    const float Axy = w6 * (float)mask_Mab<0, 1>(m), Axz = w6 * (float)mask_Mab<0, 2>(m),
                Ayz = w6 * (float)mask_Mab<1, 2>(m);
    const int K[3] = {mask_K<0>(m), mask_K<1>(m), mask_K<2>(m)};
    // the sum of 2 f~*_r c_r over the mask: at tau = 1 the bounced populations
    // again from the node's moments (drho, u, uu, uF), else the sweep's sums
    float Fr[3];
    if (tau1) {
      const float Fx = FORCE ? rho * lv.g[0] : 0.f, Fy = FORCE ? rho * lv.g[1] : 0.f, Fz = FORCE ? rho * lv.g[2] : 0.f;
      const Collide ck = collide_coeffs<FORCE>(r0.z, rho, r0.w, r1.x, r1.y, r1.z, 1.0f, Fx, Fy, Fz, r1.w);
      Fr[0] = Fr[1] = Fr[2] = 0.f;
      sfor<0, 9>([&](auto P) {
        constexpr int r = 2 * decltype(P)::value + 1;
        float fr, fb;
        collide_pair<r, FORCE>(ck, fr, fb);
        // 2 f~*_r c_r of r and of rbar (c_rbar = -c_r)
        float v = (m >> r) & 1u ? fr : 0.f;
        if ((m >> (r + 1)) & 1u) v -= fb;
        v *= 2.0f * (float)D3::m(r) / 36.0f;
        if constexpr (D3::cx(r) != 0) Fr[0] += D3::cx(r) > 0 ? v : -v;
        if constexpr (D3::cy(r) != 0) Fr[1] += D3::cy(r) > 0 ? v : -v;
        if constexpr (D3::cz(r) != 0) Fr[2] += D3::cz(r) > 0 ? v : -v;
      });
    } else {
      Fr[0] = r0.w;
      Fr[1] = r1.x;
      Fr[2] = r1.y;
    }
    const float A[3][3] = {{Axx, Axy, Axz}, {Axy, Ayy, Ayz}, {Axz, Ayz, Azz}};
    // predictor velocity at the node and the link momentum
    const float vp[3] = {k1.x + (k2.y * d[2] - k2.z * d[1]), k1.y + (k2.z * d[0] - k2.x * d[2]),
                         k1.z + (k2.x * d[1] - k2.y * d[0])};
    float F[3];
    F[0] = Fr[0] - (A[0][0] * vp[0] + A[0][1] * vp[1] + A[0][2] * vp[2]);
    F[1] = Fr[1] - (A[1][0] * vp[0] + A[1][1] * vp[1] + A[1][2] * vp[2]);
    F[2] = Fr[2] - (A[2][0] * vp[0] + A[2][1] * vp[1] + A[2][2] * vp[2]);
    v[0] += F[0];
    v[1] += F[1];
    v[2] += F[2];
    v[3] += d[1] * F[2] - d[2] * F[1];
    v[4] += d[2] * F[0] - d[0] * F[2];
    v[5] += d[0] * F[1] - d[1] * F[0];
    v[6] += Axx;
    v[7] += Axy;
    v[8] += Axz;
    v[9] += Ayy;
    v[10] += Ayz;
    v[11] += Azz;
    // G = A [d]x^T (the Zft block), then Ztt = [d]x G
    float G[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      G[a][0] = A[a][2] * d[1] - A[a][1] * d[2];
      G[a][1] = A[a][0] * d[2] - A[a][2] * d[0];
      G[a][2] = A[a][1] * d[0] - A[a][0] * d[1];
    }
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) v[12 + 3 * a + b] += G[a][b];
    v[21] += G[2][0] * d[1] - G[1][0] * d[2];
    v[22] += G[2][1] * d[1] - G[1][1] * d[2];
    v[23] += G[2][2] * d[1] - G[1][2] * d[2];
    v[24] += G[0][1] * d[2] - G[2][1] * d[0];
    v[25] += G[0][2] * d[2] - G[2][2] * d[0];
    v[26] += G[1][2] * d[0] - G[0][2] * d[1];
    iv[0] += K[0];
    iv[1] += K[1];
    iv[2] += K[2];
    iv[3] += di[1] * K[2] - di[2] * K[1];
    iv[4] += di[2] * K[0] - di[0] * K[2];
    iv[5] += di[0] * K[1] - di[1] * K[0];
  }
  // warp sums, then one thread per value adds the warps (FP64) and writes
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < 27; ++k) {
    const float t = warp_sum(v[k]);
    if (lane == 0) shf[wid][k] = t;
  }
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const int t = __reduce_add_sync(0xffffffffu, iv[k]);
    if (lane == 0) shi[wid][k] = t;
  }
  __syncthreads();
  if (threadIdx.x < 27) {
    double t = 0.0;
    for (int w2 = 0; w2 < LT / 32; ++w2) t += (double)shf[w2][threadIdx.x];
    if (threadIdx.x < 6) pv.lsum[6 * p + threadIdx.x] = t;
    else pv.lsum_f[21 * p + threadIdx.x - 6] = (float)t;
  } else if (threadIdx.x >= 32 && threadIdx.x < 38) {
    int t = 0;
    for (int w2 = 0; w2 < LT / 32; ++w2) t += shi[w2][threadIdx.x - 32];
    pv.lsum_i[6 * p + threadIdx.x - 32] = t;
  } else if (threadIdx.x == 64) {
    // the bucket is read: keep its size for the link read-out, empty it for the next sweep
    pv.rec_last[p] = nrec;
    lv.rec_count[p] = 0;
  }
}

// Link force at the predictor, 6 x 6 solve, leap-frog, kinematics and claim
// box of the next step.  Four lanes per cell, lane k holding component k of
// its vectors (lane 3 component 0 again) and of its quaternion: every FP64
// instruction holds the SM's FP64 pipe for 16 cycles, so a warp of 32 cells
// with three components in a row took 14.4 us at any number of cells.  The
// 6 x 6 system (FP32) is solved by all four lanes alike.
constexpr int SOLVE_CELLS = 8;  // per block of one warp

__device__ __forceinline__ float pick3f(int k, float a, float b, float c) { return k == 0 ? a : (k == 1 ? b : c); }

__global__ void __launch_bounds__(32) k_solve(LatticeView lv, PartView pv) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x, k4 = lane & 3, k = k4 < 3 ? k4 : 0, g0 = lane & ~3;
  const int pr = blockIdx.x * SOLVE_CELLS + (lane >> 2);
  const bool valid = pr < pv.n, wr = valid && k4 < 3;
  const int p = valid ? pr : pv.n - 1, c = 3 * p + k;
  // component j of the cell's vector
  auto at = [&](auto v, int j) { return __shfl_sync(FULL, v, g0 + j); };
  double X = pv.X[c], V = pv.V[c], L = pv.L[c], W = pv.Om[c], q = pv.q[4 * p + k4];
  const double Xold = X, o_old = pv.o[c];
  const float *kf = reinterpret_cast<const float *>(pv.kin + 3 * p);
  const float Vpf = kf[4 + k], Wpf = kf[8 + k];
  // beside the link sums that this kernel waits for: all that needs the state,
  // the potentials and the contact sums alone, with f = X - rint(X) the
  // fraction the sweep's lever arms used
  const int cK = pv.cK[c], cIT = pv.cIT[c];
  const double f = X - rint(X);
  const int k1 = k == 2 ? 0 : k + 1, k2 = k == 0 ? 2 : k - 1;
  const double f1 = at(f, k1), f2 = at(f, k2);
  const double cst = pv.rho0 / 18.0;
  const double Fo = pv.Fpot[c] + pv.PF[c] + (pv.bfc ? pv.m * pv.g[k] : 0.0), To = pv.Tpot[c] + pv.PT[c];
  const float oldf = (float)o_old;
  float I[3][3];
  double dP = 0.0, dL = 0.0;  // m (Vp - V(t-1/2)) and L(t-1/2) - I Wp (small differences, in FP64)
  if (pv.move == 1) {
    const float qf = (float)q;
    const float w = at(qf, 0), x = at(qf, 1), y = at(qf, 2), z = at(qf, 3);
    const float R[3][3] = {{1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)},
                           {2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)},
                           {2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)}};
    const float d0 = (float)pv.Iperp, d2 = (float)pv.Ipar;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b)
        I[a][b] = R[a][0] * d0 * R[b][0] + R[a][1] * d0 * R[b][1] + R[a][2] * d2 * R[b][2];
    double IW = 0.0;
#pragma unroll
    for (int t = 0; t < 3; ++t) IW += (double)pick3f(k, I[0][t], I[1][t], I[2][t]) * (double)at(Wpf, t);
    dL = L - IW;
    dP = pv.m * ((double)Vpf - V);
  }
  pdl_wait();
  float Zs[21];
#pragma unroll
  for (int i = 0; i < 21; ++i) Zs[i] = pv.lsum_f[21 * p + i];
  // (the link reduction and the contact kernel rewrite these every step)
  const double K = (double)(pv.lsum_i[6 * p + k] + cK), IT = (double)(pv.lsum_i[6 * p + 3 + k] + cIT);
  // link force at the predictor: variable part + exact constant part
  const double fxK = f1 * at(K, k2) - f2 * at(K, k1);
  double Fl = pv.lsum[6 * p + k] + cst * K, Tl = pv.lsum[6 * p + 3 + k] + cst * (IT - fxK);
  double Ft = Fl + Fo, Tt = Tl + To;
  if (wr) {
    pv.PF[c] = 0.0;
    pv.PT[c] = 0.0;
    pv.oprev[c] = oldf;  // the claims' old ellipsoid
  }
  const bool move = pv.move != 0;
  if (pv.move == 1) {  // free cells; 2: prescribed, V and W stay as set
    float Z[6][6], A[6][6], rhs[6], d[6], inv[6];
    {
      int i = 0;
#pragma unroll
      for (int s = 0; s < 3; ++s)
#pragma unroll
        for (int t = s; t < 3; ++t, ++i) Z[s][t] = Z[t][s] = Zs[i];
#pragma unroll
      for (int s = 0; s < 3; ++s)
#pragma unroll
        for (int t = 0; t < 3; ++t, ++i) Z[s][3 + t] = Z[3 + t][s] = Zs[i];
#pragma unroll
      for (int s = 0; s < 3; ++s)
#pragma unroll
        for (int t = s; t < 3; ++t, ++i) Z[3 + s][3 + t] = Z[3 + t][3 + s] = Zs[i];
    }
    {
      const float r0 = (float)(Ft - dP), r1 = (float)(Tt + dL);
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        rhs[s] = at(r0, s);
        rhs[3 + s] = at(r1, s);
      }
    }
    // Cholesky with the reciprocals of the diagonal (a Newton step on rsqrt)
    const float m = (float)pv.m;
#pragma unroll
    for (int s = 0; s < 6; ++s)
#pragma unroll
      for (int t = 0; t <= s; ++t) {
        A[s][t] = Z[s][t];
        if (s < 3 && s == t) A[s][t] += m;
        if (s >= 3 && t >= 3) A[s][t] += I[s >= 3 ? s - 3 : 0][t >= 3 ? t - 3 : 0];
      }
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      float dj = A[j][j];
#pragma unroll
      for (int t = 0; t < j; ++t) dj -= A[j][t] * A[j][t];
      const float y = rsqrtf(dj);
      inv[j] = fmaf(0.5f * y, fmaf(-dj * y, y, 1.0f), y);
#pragma unroll
      for (int i = j + 1; i < 6; ++i) {
        float v = A[i][j];
#pragma unroll
        for (int t = 0; t < j; ++t) v -= A[i][t] * A[j][t];
        A[i][j] = v * inv[j];
      }
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      float v = rhs[i];
#pragma unroll
      for (int t = 0; t < i; ++t) v -= A[i][t] * d[t];
      d[i] = v * inv[i];
    }
#pragma unroll
    for (int i = 5; i >= 0; --i) {
      float v = d[i];
#pragma unroll
      for (int t = i + 1; t < 6; ++t) v -= A[t][i] * d[t];
      d[i] = v * inv[i];
    }
    float dF[3], dT[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      dF[s] = dT[s] = 0.f;
#pragma unroll
      for (int t = 0; t < 6; ++t) {
        dF[s] += Z[s][t] * d[t];
        dT[s] += Z[3 + s][t] * d[t];
      }
    }
    const double dFk = pick3f(k, dF[0], dF[1], dF[2]), dTk = pick3f(k, dT[0], dT[1], dT[2]);
    Fl -= dFk;
    Tl -= dTk;
    Ft -= dFk;
    Tt -= dTk;
    V = (double)Vpf + (double)pick3f(k, d[0], d[1], d[2]);
    W = (double)Wpf + (double)pick3f(k, d[3], d[4], d[5]);
    L += Tt;
  }
  const float Wf = (float)W;
  float Vf = (float)V;
  if (wr) {
    pv.Flink[c] = Fl;
    pv.Tlink[c] = Tl;
    pv.Ftot[c] = Ft;
    pv.Ttot[c] = Tt;
    pv.vw[6 * p + k] = Vf;
    pv.vw[6 * p + 3 + k] = Wf;
  }
  if (move) {
    const int dim = k == 0 ? lv.nx : (k == 1 ? lv.ny : lv.nz);
    // Sec. IV: a free cell closer than le_dr to the sheared plane (x = -1/2)
    // and moving toward it has its normal velocity negated; the step's
    // coupling above used the solve's velocity, the cell moves with the
    // reflected one (reading Q25)
    if (pv.le_dr > 0.0 && pv.move == 1 && k == 0) {
      const double dlo = X + 0.5, dhi = (double)lv.nx - 0.5 - X;
      if ((dlo < pv.le_dr && V < 0.0) || (dhi < pv.le_dr && V > 0.0)) {
        V = -V;
        Vf = -Vf;
      }
    }
    // X += V (wrapped), q <- exp(W / 2) (x) q with the rotation increment in
    // FP32 and a first-order renormalisation (|q|^2 - 1 is O(1e-7))
    X += V;
    if (lv.per[k]) {
      if (X < 0.0) X += (double)dim;
      else if (X >= (double)dim) X -= (double)dim;
    }
    const float wx = at(Wf, 0), wy = at(Wf, 1), wz = at(Wf, 2);
    const float t2 = wx * wx + wy * wy + wz * wz;
    // cos(|W| / 2) and sin(|W| / 2) / |W| as their Taylor series in |W|^2 (for
    // |W| <= 1, a fast cell, the first term left out is below 3e-9 of each)
    float cs, sh;
    if (t2 <= 1.0f) {
      const float h2 = 0.25f * t2;
      cs = fmaf(h2, fmaf(h2, fmaf(h2, fmaf(h2, 1.0f / 40320.0f, -1.0f / 720.0f), 1.0f / 24.0f), -0.5f), 1.0f);
      sh = 0.5f * fmaf(h2, fmaf(h2, fmaf(h2, fmaf(h2, 1.0f / 362880.0f, -1.0f / 5040.0f), 1.0f / 120.0f), -1.0f / 6.0f), 1.0f);
    } else {
      const float th = sqrtf(t2);
      float sn;
      sincosf(0.5f * th, &sn, &cs);
      sh = sn / th;
    }
    // component l = k4 of the product: sum over m of +- dq[m] q[l xor m]
    const float dx = (k4 & 1) ? wx * sh : -(wx * sh);
    const float dy = (k4 == 1 || k4 == 2) ? wy * sh : -(wy * sh);
    const float dz = (k4 & 2) ? wz * sh : -(wz * sh);
    double nq = (double)cs * q;
    nq += (double)dx * __shfl_xor_sync(FULL, q, 1);
    nq += (double)dy * __shfl_xor_sync(FULL, q, 2);
    nq += (double)dz * __shfl_xor_sync(FULL, q, 3);
    double nn = nq * nq;
    nn += __shfl_xor_sync(FULL, nn, 1);
    nn += __shfl_xor_sync(FULL, nn, 2);
    if (t2 > 0.f) q = nq * (1.5 - 0.5 * nn);  // 1 / sqrt(nn) to second order in (nn - 1)
    // the exact axis (axis_exact), component by component
    const double a1 = at(q, k == 1 ? 2 : 1), b1 = at(q, k == 2 ? 1 : 3), a2 = at(q, k == 2 ? 2 : 0),
                 b2 = at(q, k == 1 ? 1 : 2);
    const double pa = __dmul_rn(a1, b1), pb = __dmul_rn(a2, b2);
    const double o2 = __dmul_rn(2.0, __dadd_rn(pa, k == 1 ? -pb : pb));
    const double o = k == 2 ? __dsub_rn(1.0, o2) : o2;
    const float of = (float)o, Xf = (float)X;
    // a cell faster than half a node per step is far outside the method's
    // low-Mach range (and would outrun the cell list of the step's start)
    const double vv = V * V, v2 = at(vv, 0) + at(vv, 1) + at(vv, 2);
    const bool ok = isfinite(X) && isfinite(o) && v2 < 0.25;
    const bool finite = ((__ballot_sync(FULL, ok) >> g0) & 7u) == 7u;
    int lo = 0, hi = -1;
    if (finite) {
      int lo2, hi2;
      aabb1(pv, Xf, of, lo, hi);
      aabb1(pv, (float)Xold, oldf, lo2, hi2);
      lo = min(lo, lo2);
      hi = max(hi, hi2);
      if (!lv.per[k]) {
        lo = max(lo, 0);
        hi = min(hi, dim - 1);
      } else if (hi - lo + 1 > dim) {
        lo = 0;
        hi = dim - 1;
      }
    } else if (valid) {
      atomicOr(pv.status, ST_UNSTABLE);
    }
    if (valid) {
      pv.q[4 * p + k4] = q;
      reinterpret_cast<float *>(pv.qf + p)[k4] = (float)q;
    }
    if (wr) {
      pv.X[c] = X;
      pv.V[c] = V;
      pv.L[c] = L;
      pv.Om[c] = W;
      pv.o[c] = o;
      reinterpret_cast<float *>(pv.axis + p)[k] = of;
      pv.box[6 * p + k] = lo;  // fixed cells keep the box of their last set: the geometry pass still needs it
      pv.box[6 * p + 3 + k] = hi;
    }
  }
  if (wr) {
    const double Xi = rint(X);
    float *kn = reinterpret_cast<float *>(pv.kin_next + 3 * p);
    kn[k] = (float)(X - Xi);
    kn[4 + k] = Vf;
    kn[8 + k] = Wf;
    kn[4 * k + 3] = (float)Xi;
  }
}

// The pending moving-boundary term of each record, right after the solve
// (one block per cell, beside the claims).  A record of a node's first cell
// becomes the node's pending velocity pu = rho (V + W x d) with its bounced
// directions, which the next sweep adds as C = -(m_r / 6) c_r . pu to the
// populations it reads; the records of a second or third cell of one node
// (marked REC_DIRECT) get their C in place.  V, W: the cell's half-step
// velocities of the solve; d: node minus the cell's position of this step.
// Every link is one cell's, so no two blocks touch the same slot.  Bound by
// scattered 16- and 4-byte accesses: 12.2 us for 1022 cells, 119 us (0.4 GB in
// 32-byte sectors) for 8446.  The second-cell records hold 18 populations and
// slots at once: 72 registers and 72 to 104 spilled bytes, on their rare path.
template <class S>
__global__ void __launch_bounds__(LT, 7) k_link_pending(LatticeView lv, PartView pv, int par) {
  constexpr int PQ = 512;  // queue of a block's second- and third-cell records
  __shared__ int s_nq;
  __shared__ int s_q[PQ];
  const int p = blockIdx.x;
  if (threadIdx.x == 0) s_nq = 0;
  __syncthreads();
  const int nrec = min(pv.rec_last[p], lv.rec_cap);
  const float4 k0 = pv.kin[3 * p], k1 = pv.kin[3 * p + 1], k2 = pv.kin[3 * p + 2];
  const int Xi[3] = {(int)k0.w, (int)k1.w, (int)k2.w};
  const float *vw = pv.vw + 6 * p;
  const float V[3] = {vw[0], vw[1], vw[2]}, W[3] = {vw[3], vw[4], vw[5]};
  S *pop = reinterpret_cast<S *>(lv.pop);
  const float4 *rec = lv.rec + 2 * (size_t)p * lv.rec_cap;
  // rho (V + W x d) of a record's node and its coordinates
  auto node_u = [&](const float4 &r0, int yc[3], float u[3]) {
    node_xyz(lv, __float_as_uint(r0.x), yc);
    const float d[3] = {(float)imin_image(yc[0] - Xi[0], lv.nx, lv.per[0]) - k0.x,
                        (float)imin_image(yc[1] - Xi[1], lv.ny, lv.per[1]) - k0.y,
                        (float)imin_image(yc[2] - Xi[2], lv.nz, lv.per[2]) - k0.z};
    const float rho = lv.rho0 + r0.z;
    u[0] = rho * (V[0] + (W[1] * d[2] - W[2] * d[1]));
    u[1] = rho * (V[1] + (W[2] * d[0] - W[0] * d[2]));
    u[2] = rho * (V[2] + (W[0] * d[1] - W[1] * d[0]));
  };
  // C in place for the directions of a second- or third-cell record: all its
  // populations requested together, then written
  auto direct = [&](int i) {
    const float4 r0 = rec[i];
    const unsigned n = __float_as_uint(r0.x);
    const uint32_t m = __float_as_uint(r0.y) & NB_SOLID;
    int yc[3];
    float u[3], v[Q];
    node_u(r0, yc, u);
    unsigned slot[Q];
    const unsigned nx = (unsigned)lv.nx, nxy = nx * (unsigned)lv.ny;
    const unsigned xo[3] = {(unsigned)(yc[0] == 0 ? lv.nx - 1 : yc[0] - 1), (unsigned)yc[0],
                            (unsigned)(yc[0] == lv.nx - 1 ? 0 : yc[0] + 1)};
    const unsigned yo[3] = {(unsigned)(yc[1] == 0 ? lv.ny - 1 : yc[1] - 1) * nx, (unsigned)yc[1] * nx,
                            (unsigned)(yc[1] == lv.ny - 1 ? 0 : yc[1] + 1) * nx};
    const unsigned zo[3] = {(unsigned)(yc[2] == 0 ? lv.nz - 1 : yc[2] - 1) * nxy, (unsigned)yc[2] * nxy,
                            (unsigned)(yc[2] == lv.nz - 1 ? 0 : yc[2] + 1) * nxy};
    sfor<1, Q>([&](auto R) {
      constexpr int r = decltype(R)::value;
      // the slot the sweep of parity par bounced direction r into
      slot[r] = par == 0 ? (unsigned)r * lv.N + xo[1 + D3::cx(r)] + yo[1 + D3::cy(r)] + zo[1 + D3::cz(r)]
                         : (unsigned)D3::opp(r) * lv.N + n;
      if ((m >> r) & 1u) v[r] = Store<S>::ld(pop + slot[r]);
    });
    sfor<1, Q>([&](auto R) {
      constexpr int r = decltype(R)::value;
      const float C = -(D3::m(r) / 6.0f) * (D3::cx(r) * u[0] + D3::cy(r) * u[1] + D3::cz(r) * u[2]);
      if ((m >> r) & 1u) Store<S>::st(pop + slot[r], v[r] + C);
    });
  };
  // four records per thread requested together: one memory round trip each
  // took most of the kernel's time
  constexpr int PU = 4;
  for (int i0 = threadIdx.x; i0 < nrec; i0 += PU * LT) {
    float4 r0[PU];
#pragma unroll
    for (int j = 0; j < PU; ++j)
      if (i0 + j * LT < nrec) r0[j] = rec[i0 + j * LT];
#pragma unroll
    for (int j = 0; j < PU; ++j) {
      const int i = i0 + j * LT;
      if (i >= nrec) break;
      const uint32_t mb = __float_as_uint(r0[j].y);
      if (mb & REC_DIRECT) {
        const int k = atomicAdd(&s_nq, 1);
        if (k < PQ) s_q[k] = i;
        continue;
      }
      int yc[3];
      float u[3];
      node_u(r0[j], yc, u);
      lv.pu[__float_as_uint(r0[j].x)] = make_float4(u[0], u[1], u[2], __uint_as_float(mb & NB_SOLID));
    }
  }
  // the records of a node's second or third cell, gathered so that the
  // warps take their per-direction loops with full lanes
  __syncthreads();
  const bool full = s_nq > PQ;  // more than the queue holds: found again among all records
  const int nq = full ? nrec : s_nq;
  for (int k = threadIdx.x; k < nq; k += LT) {
    const int i = full ? k : s_q[k];
    if (!full || (__float_as_uint(rec[i].y) & REC_DIRECT)) direct(i);
  }
}

// The pending C of the last step given to the stored populations, for
// read-outs and state changes between steps (the sweep's arithmetic); par is
// the layout of the stored populations (the next step's parity).
template <class S>
__global__ void k_flush_pending(LatticeView lv, int par) {
  using D = D3Q19;
  S *pop = reinterpret_cast<S *>(lv.pop);
  for (unsigned n = blockIdx.x * blockDim.x + threadIdx.x; n < lv.N; n += gridDim.x * blockDim.x) {
    const float4 pu = lv.pu[n];
    const uint32_t pm = __float_as_uint(pu.w);
    if (!pm) continue;
    int yc[3];
    node_xyz(lv, n, yc);
    for (uint32_t m = pm; m; m &= m - 1u) {
      const int r = __ffs(m) - 1;
      // the slot from which node n reads direction rbar in layout par
      const unsigned slot = bounce_slot(lv, par ^ 1, n, yc, r);
      Store<S>::st(pop + slot, add_pending(Store<S>::ld(pop + slot), D::m(r),
                                           D::cx(r) * pu.x + D::cy(r) * pu.y + D::cz(r) * pu.z));
    }
    reinterpret_cast<float *>(lv.pu + n)[3] = 0.f;
  }
}

// particles_set: the state comes from the stage.  mode 1: first set (the
// box holds the new ellipsoid); mode 2: later set (old and new ellipsoid)
__global__ void k_set_state(LatticeView lv, PartView pv, int mode) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= pv.n) return;
  double Xold[3], o_old[3];
  for (int k = 0; k < 3; ++k) {
    Xold[k] = pv.X[3 * p + k];
    o_old[k] = pv.o[3 * p + k];
  }
  const double *st = pv.stage + 13 * p;
  double X[3], q[4], V[3], L[3], W[3];
  for (int k = 0; k < 3; ++k) {
    X[k] = st[k];
    V[k] = st[7 + k];
    L[k] = st[10 + k];
  }
  for (int k = 0; k < 4; ++k) q[k] = st[3 + k];
  float I[3][3], Iinv[3][3];
  inertia_f(pv, q, I, Iinv);
  for (int k = 0; k < 3; ++k)
    W[k] = (double)(Iinv[k][0] * (float)L[0] + Iinv[k][1] * (float)L[1] + Iinv[k][2] * (float)L[2]);
  for (int k = 0; k < 3; ++k) {
    pv.X[3 * p + k] = X[k];
    pv.V[3 * p + k] = V[k];
    pv.L[3 * p + k] = L[k];
    pv.Om[3 * p + k] = W[k];
    pv.vw[6 * p + k] = (float)V[k];
    pv.vw[6 * p + 3 + k] = (float)W[k];
  }
  for (int k = 0; k < 4; ++k) pv.q[4 * p + k] = q[k];
  pv.qf[p] = make_float4((float)q[0], (float)q[1], (float)q[2], (float)q[3]);
  double o_new[3];
  axis_exact(q, o_new);
  for (int k = 0; k < 3; ++k) {
    pv.oprev[3 * p + k] = (float)(mode == 2 ? o_old[k] : o_new[k]);
    pv.o[3 * p + k] = o_new[k];
  }
  pv.axis[p] = make_float4((float)o_new[0], (float)o_new[1], (float)o_new[2], 0.f);
  write_kin(pv, p, X, V, W);
  int lo[3], hi[3], lo2[3], hi2[3];
  aabb(pv, X, o_new, lo, hi);
  bool finite = isfinite(X[0]) && isfinite(X[1]) && isfinite(X[2]);
  if (mode == 2) {
    finite = finite && isfinite(Xold[0]) && isfinite(Xold[1]) && isfinite(Xold[2]);
    aabb(pv, Xold, o_old, lo2, hi2);
    for (int k = 0; k < 3; ++k) {
      lo[k] = min(lo[k], lo2[k]);
      hi[k] = max(hi[k], hi2[k]);
    }
  }
  const int dims[3] = {lv.nx, lv.ny, lv.nz};
  for (int k = 0; k < 3; ++k) {
    if (!finite) {
      lo[k] = 0;
      hi[k] = -1;
    } else if (!lv.per[k]) {
      lo[k] = max(lo[k], 0);
      hi[k] = min(hi[k], dims[k] - 1);
    } else if (hi[k] - lo[k] + 1 > dims[k]) {
      lo[k] = 0;
      hi[k] = dims[k] - 1;
    }
    pv.box[6 * p + k] = lo[k];
    pv.box[6 * p + 3 + k] = hi[k];
  }
  if (!finite) atomicOr(pv.status, ST_UNSTABLE);
}

// Row intervals of an ellipsoid.  Along the lattice row (y, z) the inside
// function is a quadratic in t = x - X_x:
//   s(t) = A t^2 + B t + C0,  A = ip + kk o_x^2,  B = 2 kk o_x e,
//   C0 = (dy^2 + dz^2) ip + kk e^2,  e = o_y dy + o_z dz,
// ip = 1 / R_perp^2, kk = 1 / R_par^2 - 1 / R_perp^2 (A > 0 for any axis).
struct RowQuad {
  float A, B, C0;
};

__device__ __forceinline__ RowQuad row_quad(float dy, float dz, const float o[3], float ip, float kk) {
  const float e = o[1] * dy + o[2] * dz;
  return RowQuad{ip + kk * o[0] * o[0], 2.0f * kk * o[0] * e, (dy * dy + dz * dz) * ip + kk * e * e};
}

// node offsets i = x - rint(X_x) of the row with s <= L, as [lo, hi] (empty:
// lo > hi); xf = X_x - rint(X_x)
__device__ __forceinline__ void row_range(const RowQuad &q, float L, float xf, int &lo, int &hi) {
  const float disc = q.B * q.B - 4.0f * q.A * (q.C0 - L);
  if (!(disc >= 0.0f)) {
    lo = 1;
    hi = 0;
    return;
  }
  const float sq = sqrtf(disc), h = 0.5f / q.A;
  lo = (int)ceilf((-q.B - sq) * h + xf);
  hi = (int)floorf((-q.B + sq) * h + xf);
}

// Margin in s between the FP32 row intervals and the exact inside test: the
// FP32 interval ends are off by less than 1e-4 in s for half-axis ratios up
// to 100, so nodes with s <= 1 - ROW_EPS on a row's FP32 estimate are inside
// and nodes with s > 1 + ROW_EPS are outside.
constexpr float ROW_EPS = 2e-3f;

constexpr int PB = 128;  // threads of the claims and resolve blocks (8 blocks fit an SM)

// Claims (one block per cell, one thread per lattice row of the cell's box).
// A node's cover by cell p can change only where the old and the new
// ellipsoid differ: on each row, the nodes of the hull of the two outer
// intervals (s <= 1 + ROW_EPS) that are not in both inner ones (s <= 1 -
// ROW_EPS).  Those candidates get the exact inside test:
//   owned by p and no longer inside -> TOUCHED (resolve finds the new owner)
//   fluid and now inside            -> claim with p (atomicMin: lowest newcomer)
// Every node inside some cell is owned by a cell after each resolve, so a
// fluid node inside p is one that p's ellipsoid has just entered, and nodes
// owned by another cell need no claim: their owner keeps them while it
// covers them (first arrival), and hands them on through TOUCHED.
// mode 1: no old ellipsoid (first particles_set, all owners fluid).
// Bound by latency and issue (10.3 us for 1022 cells, 47 us for 8446); with
// each thread forming the cell's geometry from its FP64 state it was bound by
// FP64 issue (19.2 and 112 us).
// In particles_set (modes 1, 2) also clears the cell's link count and
// contact sums for the lattice-wide geometry pass, which adds to them; in a
// step (mode 0) the contact sums of this step are in use, and the next
// step's contact kernel rewrites them.
__global__ void __launch_bounds__(PB, BL_CLAIMS_MINB) k_claims(LatticeView lv, PartView pv, int *claim, ChangeList chg, int mode) {
  __shared__ int sh_len;
  const int p = blockIdx.x;
  if (threadIdx.x == 0) {
    sh_len = 0;
    if (mode != 0) {
      for (int k = 0; k < 3; ++k) {
        pv.cK[3 * p + k] = 0;
        pv.cIT[3 * p + k] = 0;
      }
    }
    if (p == 0) *chg.count = 0;
  }
  __syncthreads();
  const int lo1 = pv.box[6 * p + 1], lo2 = pv.box[6 * p + 2];
  const int by = pv.box[6 * p + 4] - lo1 + 1, bz = pv.box[6 * p + 5] - lo2 + 1;
  const int rows = (by > 0 && bz > 0) ? by * bz : 0;
  CellGeo g;
  cell_geo(pv, pv.kin_next, p, g);
  const bool has_old = mode != 1;
  int Xo[3] = {0, 0, 0};
  float xfo[3] = {0.f, 0.f, 0.f}, oo[3] = {0.f, 0.f, 0.f};
  if (has_old) {
    const float4 k0 = pv.kin[3 * p], k1 = pv.kin[3 * p + 1], k2 = pv.kin[3 * p + 2];
    Xo[0] = (int)k0.w;
    Xo[1] = (int)k1.w;
    Xo[2] = (int)k2.w;
    xfo[0] = k0.x;
    xfo[1] = k0.y;
    xfo[2] = k0.z;
    for (int k = 0; k < 3; ++k) oo[k] = pv.oprev[3 * p + k];
  }
  const float ip = pv.inv_rperp2_f, kk = pv.kk_f;
  const int shift = imin_image(Xo[0] - g.Xi[0], lv.nx, lv.per[0]);  // old rint(X_x) from the new one
  // offsets of one period (periodic x) or of the lattice (walled x)
  const int imin = lv.per[0] ? -(lv.nx / 2) : -g.Xi[0];
  const int imax = lv.per[0] ? imin + lv.nx - 1 : lv.nx - 1 - g.Xi[0];
  unsigned long long *touched = pv.touched + (size_t)p * pv.touched_cap;
  for (int t = threadIdx.x; t < rows; t += PB) {
    int y = lo1 + t % by, z = lo2 + t / by;
    if (lv.per[1]) y = wrapi(y, lv.ny);
    if (lv.per[2]) z = wrapi(z, lv.nz);
    const RowQuad qn = row_quad((float)imin_image(y - g.Xi[1], lv.ny, lv.per[1]) - g.Xf[1],
                                (float)imin_image(z - g.Xi[2], lv.nz, lv.per[2]) - g.Xf[2], g.of, ip, kk);
    int ao, bo, ai, bi;
    row_range(qn, 1.0f + ROW_EPS, g.Xf[0], ao, bo);
    row_range(qn, 1.0f - ROW_EPS, g.Xf[0], ai, bi);
    if (has_old) {
      const RowQuad qo = row_quad((float)imin_image(y - Xo[1], lv.ny, lv.per[1]) - xfo[1],
                                  (float)imin_image(z - Xo[2], lv.nz, lv.per[2]) - xfo[2], oo, ip, kk);
      int ao2, bo2, ai2, bi2;
      row_range(qo, 1.0f + ROW_EPS, xfo[0], ao2, bo2);
      row_range(qo, 1.0f - ROW_EPS, xfo[0], ai2, bi2);
      const int oa = ao2 + shift, ob = bo2 + shift;
      if (mode == 2 && ao2 <= bo2 && lv.per[0] && (oa < imin || ob > imax)) {
        // set far away (a step moves less than half a node): the old interval reaches over the end of the period
        // counted from the new centre, so every node of the row is looked at
        ao = imin;
        bo = imax;
        ai2 = 1;
        bi2 = 0;
      } else if (ao2 <= bo2) {
        if (ao > bo) {
          ao = oa;
          bo = ob;
        } else {
          ao = min(ao, oa);
          bo = max(bo, ob);
        }
      }
      if (ai2 <= bi2) {
        ai = max(ai, ai2 + shift);
        bi = min(bi, bi2 + shift);
      } else {
        ai = 1;
        bi = 0;
      }
    } else {
      ai = 1;  // nothing was covered: every node of the new interval
      bi = 0;
    }
    ao = max(ao, imin);
    bo = min(bo, imax);
    if (ao > bo) continue;
    // candidates: [ao, bo] without the common core [ai, bi]
    const bool core = ai <= bi;
    const int e1 = core ? min(bo, ai - 1) : bo;
    const int s2 = core ? max(ao, bi + 1) : bo + 1;
    for (int i = ao; i <= bo; ++i) {
      if (i > e1 && i < s2) {
        i = s2 - 1;
        continue;
      }
      int x = g.Xi[0] + i;
      if (lv.per[0]) x = wrapi(x, lv.nx);
      const unsigned idx = node_of(lv, x, y, z);
      const int ow = lv.owner[idx];
      int mark = 0;
      if (ow == p) {
        if (!inside_cell(x, y, z, p, g, pv, lv)) {
          atomicMin(&claim[idx], CLAIM_TOUCHED);
          mark = 1;
        }
      } else if (ow == FLUID) {
        if (inside_cell(x, y, z, p, g, pv, lv)) {
          atomicMin(&claim[idx], p);
          mark = 1;
        }
      }
      if (mark) {
        const int pos = atomicAdd(&sh_len, 1);
        if (pos < pv.touched_cap) touched[pos] = pack_xyzr(x, y, z, 0);
        else atomicOr(pv.status, ST_OVERFLOW);
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) pv.touched_count[p] = min(sh_len, pv.touched_cap);
}

// lowest-index cell whose ellipsoid covers node (x, y, z), FLUID if none.
// Cells are searched in the node's bin and its neighbours: a bin is at least
// r_cut wide, r_cut exceeds the largest half-axis by one node, and a cell
// moves less than half a node per step, so the cell list of the step's start
// holds every cover of the node.  Bins list their cells in index order.
// (one warp per node: lane b < 27 scans neighbouring bin b, the lowest
// covering index over the lanes wins; all 32 lanes call it)
__device__ int lowest_cover(const LatticeView &lv, const PartView &pv, const CellListView &cl, int x, int y,
                                 int z) {
  const int lane = threadIdx.x & 31;
  const int c[3] = {x, y, z};
  const int dims[3] = {lv.nx, lv.ny, lv.nz};
  int bc[3], off[3][3], noff[3];
  for (int k = 0; k < 3; ++k) {
    bc[k] = (int)(((long long)c[k] * cl.nb[k]) / dims[k]);
    noff[k] = bin_offsets(cl.nb[k], lv.per[k], bc[k], off[k]);
  }
  int best = INT_MAX;
  const int ix = lane % 3, iy = (lane / 3) % 3, iz = lane / 9;
  if (lane < 27 && ix < noff[0] && iy < noff[1] && iz < noff[2]) {
    const int b = wrapi(bc[0] + off[0][ix], cl.nb[0]) +
                  cl.nb[0] * (wrapi(bc[1] + off[1][iy], cl.nb[1]) + cl.nb[1] * wrapi(bc[2] + off[2][iz], cl.nb[2]));
    const int e = cl.start[b + 1];
    for (int k = cl.start[b]; k < e; ++k) {
      const int j = cl.ids[k];
      CellGeo g;
      cell_geo(pv, pv.kin_next, j, g);
      if (inside_cell(x, y, z, j, g, pv, lv)) {
        best = j;
        break;
      }
    }
  }
  best = __reduce_min_sync(0xffffffffu, best);
  return best == INT_MAX ? FLUID : best;
}

// ---------------------------------------------------------------------------
// resolve + fill/drain over each cell's touched nodes

__device__ __forceinline__ void atomic_add3(double *a, const double v[3]) {
  atomicAdd(a, v[0]);
  atomicAdd(a + 1, v[1]);
  atomicAdd(a + 2, v[2]);
}

// cells that can cover a node cell p leaves: within 2 max(R) + 2 of it after
// the move (the node is within max(R) + 1 of p's centre, a cell covers it
// within max(R)).  Gathered once per block into shared memory from the bins
// within reach (the list is of the step's start; a cell moves less than half a
// node), so that a node's search reads no memory: a search of its own per
// node, three dependent loads deep, was the longest chain of the kernel.
constexpr int NCAND = 64;

struct Cands {
  int n;
  int id[NCAND];
  CellGeo g[NCAND];
};

__device__ __forceinline__ void gather_cands(const LatticeView &lv, const PartView &pv, const CellListView &cl, int p,
                                             Cands &cd) {
  CellGeo g;
  cell_geo(pv, pv.kin_next, p, g);
  const float reach = 2.0f * pv.Rmax_f + 2.0f;
  const int dims[3] = {lv.nx, lv.ny, lv.nz};
  int b0[3], cnt[3];
  for (int k = 0; k < 3; ++k) {
    const float x = (float)g.Xi[k] + g.Xf[k], s = (float)cl.nb[k] / (float)dims[k];
    int lo = (int)floorf((x - reach - 0.6f) * s - 1e-3f), hi = (int)floorf((x + reach + 0.6f) * s + 1e-3f);
    if (!lv.per[k]) {
      lo = max(lo, 0);
      hi = min(hi, cl.nb[k] - 1);
    } else if (hi - lo + 1 >= cl.nb[k]) {
      lo = 0;
      hi = cl.nb[k] - 1;
    }
    b0[k] = lo;
    cnt[k] = hi - lo + 1;
  }
  const int total = cnt[0] * cnt[1] * cnt[2];
  for (int t = threadIdx.x; t < total; t += PB) {
    const int bx = wrapi(b0[0] + t % cnt[0], cl.nb[0]), by = wrapi(b0[1] + (t / cnt[0]) % cnt[1], cl.nb[1]),
              bz = wrapi(b0[2] + t / (cnt[0] * cnt[1]), cl.nb[2]);
    const int b = bx + cl.nb[0] * (by + cl.nb[1] * bz);
    const int e = cl.start[b + 1];
    for (int k = cl.start[b]; k < e; ++k) {
      const int j = cl.ids[k];
      CellGeo h;
      cell_geo(pv, pv.kin_next, j, h);
      float d2 = 0.f;
      for (int m = 0; m < 3; ++m) {
        const int dn = h.Xi[m] - g.Xi[m];
        const float df = h.Xf[m] - g.Xf[m];
        const float d = pv.near_reach ? image_f(dn, df, dims[m], lv.per[m]) : (float)imin_image(dn, dims[m], lv.per[m]) + df;
        d2 += d * d;
      }
      if (d2 > reach * reach) continue;
      const int i = atomicAdd(&cd.n, 1);
      if (i < NCAND) {
        cd.id[i] = j;
        cd.g[i] = h;
      }
    }
  }
}

// One block per cell over its touched nodes.  The new owners are decided first
// and the changed nodes queued, covered ones (fluid to cell) from the front,
// uncovered ones (a cell leaves) from the back; then each kind is worked off
// by warps of its own, so that the FP64 of the momentum balance is issued once
// for up to 32 nodes instead of for the few of one warp's nodes that take a
// branch.  Bound by latency: a chain of dependent reads per block (17 us for
// 1022 cells, 84 us for 8446; 23.5 and 128 before).
// SET: the cells were set anew (bl_particles_set), not moved by a step.
template <class S, bool SET>
__global__ void __launch_bounds__(PB) k_resolve_fill(LatticeView lv, PartView pv, CellListView cl, int *claim,
                                                      ChangeList chg, int par_next, int impulses) {
  using D = D3Q19;
  const int p = blockIdx.x;
  pdl_trigger();
  const unsigned long long *touched = pv.touched + (size_t)p * pv.touched_cap;
  // the first touched node of this thread is requested with the count (the
  // list holds touched_cap entries)
  unsigned long long tv0 = 0ull;
  if ((int)threadIdx.x < pv.touched_cap) tv0 = touched[threadIdx.x];
  const int nt = pv.touched_count[p];
  const int lane = threadIdx.x & 31;
  S *pop = reinterpret_cast<S *>(lv.pop);
  __shared__ int s_need[PB], s_res[PB];
  __shared__ unsigned long long s_xyz[PB];
  __shared__ int s_old[PB], s_new[PB];
  __shared__ int s_ns, s_nc, s_nu, s_base;
  __shared__ Cands s_cd;
  if (nt == 0) return;
  // (a re-placement can put cells anywhere: its nodes are searched one by one)
  if (threadIdx.x == 0) s_cd.n = SET ? NCAND + 1 : 0;
  __syncthreads();
  if constexpr (!SET) gather_cands(lv, pv, cl, p, s_cd);
  for (int t0 = 0; t0 < nt; t0 += PB) {
    const int t = t0 + threadIdx.x;
    int old = 0, nw = 0, xyz[3] = {0, 0, 0};
    bool changed = false, act = false, need = false;
    unsigned idx = 0;
    unsigned long long tv = 0ull;
    if (threadIdx.x == 0) s_ns = s_nc = s_nu = 0;
    __syncthreads();
    if (t < nt) {
      int r_unused;
      tv = t0 == 0 ? tv0 : touched[t];
      unpack_xyzr(tv, xyz, r_unused);
      idx = node_of(lv, xyz[0], xyz[1], xyz[2]);
      const int own = lv.owner[idx];  // requested beside the claim's exchange
      const int c = atomicExch(&claim[idx], CLAIM_FREE);
      if (c != CLAIM_FREE) {
        act = true;
        old = own;
        // TOUCHED: the old owner left the node -> the lowest-index cell now
        // covering it (searched below by a warp), else fluid; a claim: a
        // fluid node entered by the claimants, the lowest of which takes it
        // (reading Q5)
        if (c == CLAIM_TOUCHED) {
          need = true;
          s_need[atomicAdd(&s_ns, 1)] = threadIdx.x;
        } else {
          nw = c;
        }
      }
    }
    __syncthreads();
    for (int k = threadIdx.x >> 5; k < s_ns; k += PB / 32) {
      const int tt = s_need[k];
      int cc[3], r_unused;
      unpack_xyzr(touched[t0 + tt], cc, r_unused);
      const int ncd = s_cd.n;
      int best;
      if (ncd <= NCAND) {
        best = INT_MAX;
        for (int i = lane; i < ncd; i += 32)
          if (s_cd.id[i] < best && inside_cell(cc[0], cc[1], cc[2], s_cd.id[i], s_cd.g[i], pv, lv)) best = s_cd.id[i];
        best = __reduce_min_sync(0xffffffffu, best);
        if (best == INT_MAX) best = FLUID;
      } else {
        best = lowest_cover(lv, pv, cl, cc[0], cc[1], cc[2]);
      }
      if (lane == 0) s_res[tt] = best;
    }
    __syncthreads();
    if (act) {
      if (need) nw = s_res[threadIdx.x];
      changed = nw != old;
      if (changed) {
        lv.owner[idx] = nw;
        const int k = old == FLUID ? atomicAdd(&s_nc, 1) : PB - 1 - atomicAdd(&s_nu, 1);
        s_xyz[k] = tv;
        s_old[k] = old;
        s_new[k] = nw;
      }
    }
    __syncthreads();
    // room in the change list, asked for before the momentum balance and used
    // after it
    if (threadIdx.x == PB - 1) s_base = s_nc + s_nu ? atomicAdd(chg.count, s_nc + s_nu) : 0;
    // covered nodes first, then from a warp boundary on the uncovered ones
    const int nc = s_nc, nc32 = (nc + 31) & ~31, ntot = nc32 + s_nu;
    for (int k = threadIdx.x; k < ntot; k += PB) {
      if (k >= nc && k < nc32) continue;
      const bool cover = k < nc;
      const int e = cover ? k : PB - 1 - (k - nc32);
      int r_unused;
      unpack_xyzr(s_xyz[e], xyz, r_unused);
      idx = node_of(lv, xyz[0], xyz[1], xyz[2]);
      old = s_old[e];
      nw = s_new[e];
      unsigned slot[Q];
      for (int r = 0; r < Q; ++r) {
        if (par_next == 0 || r == 0) {
          slot[r] = (unsigned)r * lv.N + idx;
        } else {
          slot[r] = (unsigned)D::opp(r) * lv.N +
                    node_of(lv, wrapi(xyz[0] - D::cx(r), lv.nx), wrapi(xyz[1] - D::cy(r), lv.ny),
                            wrapi(xyz[2] - D::cz(r), lv.nz));
        }
      }
      if (cover) {
        // covered: the fluid is deleted, its momentum goes to the new owner;
        // its populations bounced off a cell in this step still owe their C
        // (the next sweep would have added it): C_r enters direction rbar,
        // momentum -C_r c_r, with the velocity of this step's half step at
        // the link's cell at its position of this step
        const float4 pu = lv.pu[idx];
        const uint32_t pm = __float_as_uint(pu.w);
        if (impulses) {
          float mf[3] = {0.f, 0.f, 0.f};
          for (int r = 0; r < Q; ++r) {
            const float v = Store<S>::ld(pop + slot[r]);
            mf[0] += v * D::cx(r);
            mf[1] += v * D::cy(r);
            mf[2] += v * D::cz(r);
          }
          // C_r owed to direction rbar: momentum -C_r c_r (the links to a second
          // or third cell got theirs in place)
          for (uint32_t m = pm; m; m &= m - 1u) {
            const int r = __ffs(m) - 1;
            const float cx = (float)rt_c<0>(r), cy = (float)rt_c<1>(r), cz = (float)rt_c<2>(r);
            const float C = -((float)rt_m(r) / 6.0f) * (cx * pu.x + cy * pu.y + cz * pu.z);
            mf[0] -= C * cx;
            mf[1] -= C * cy;
            mf[2] -= C * cz;
          }
          double arm[3];
          arm64<SET>(lv, pv, pv.kin_next, nw, xyz, arm);
          const double mom[3] = {mf[0], mf[1], mf[2]};
          const double tq[3] = {arm[1] * mom[2] - arm[2] * mom[1], arm[2] * mom[0] - arm[0] * mom[2],
                                arm[0] * mom[1] - arm[1] * mom[0]};
          atomic_add3(pv.PF + 3 * nw, mom);
          atomic_add3(pv.PT + 3 * nw, tq);
        }
        if (pm) reinterpret_cast<float *>(lv.pu + idx)[3] = 0.f;
      } else {
        double arm[3];
        arm64<SET>(lv, pv, pv.kin_next, old, xyz, arm);
        const double *W = pv.Om + 3 * old, *V = pv.V + 3 * old;
        const float u[3] = {(float)(V[0] + (W[1] * arm[2] - W[2] * arm[1])),
                            (float)(V[1] + (W[2] * arm[0] - W[0] * arm[2])),
                            (float)(V[2] + (W[0] * arm[1] - W[1] * arm[0]))};
        const double mom[3] = {pv.rho0 * u[0], pv.rho0 * u[1], pv.rho0 * u[2]};
        const double mneg[3] = {-mom[0], -mom[1], -mom[2]};
        const double tneg[3] = {arm[2] * mom[1] - arm[1] * mom[2], arm[0] * mom[2] - arm[2] * mom[0],
                                arm[1] * mom[0] - arm[0] * mom[1]};
        atomic_add3(pv.PF + 3 * old, mneg);
        atomic_add3(pv.PT + 3 * old, tneg);
        if (nw == FLUID) {
          // uncovered: new fluid at n^eq(rho_bar, u_rigid), stored shifted
          const float rho0 = lv.rho0;
          const float uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
          for (int r = 0; r < Q; ++r) {
            const float cu = D::cx(r) * u[0] + D::cy(r) * u[1] + D::cz(r) * u[2];
            const float w = D::m(r) / 36.0f;
            Store<S>::st(pop + slot[r], rho0 * w * (cu * (3.0f + cu * (4.5f + 4.5f * cu)) - uu * (1.5f + 4.5f * cu)));
          }
        } else {
          // direct change of owner: uncover by the old, cover by the new (reading Q6)
          double an[3];
          arm64<SET>(lv, pv, pv.kin_next, nw, xyz, an);
          const double tq2[3] = {an[1] * mom[2] - an[2] * mom[1], an[2] * mom[0] - an[0] * mom[2],
                                 an[0] * mom[1] - an[1] * mom[0]};
          atomic_add3(pv.PF + 3 * nw, mom);
          atomic_add3(pv.PT + 3 * nw, tq2);
        }
      }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < nc + s_nu; k += PB) {
      const int e = k < nc ? k : PB - 1 - (k - nc), pos = s_base + k;
      if (pos >= chg.cap) break;
      int r_unused;
      unpack_xyzr(s_xyz[e], xyz, r_unused);
      chg.items[3 * pos] = (int32_t)node_of(lv, xyz[0], xyz[1], xyz[2]);
      chg.items[3 * pos + 1] = s_old[e];
      chg.items[3 * pos + 2] = s_new[e];
    }
    __syncthreads();  // the queues are refilled by the next chunk
  }
}

// ---------------------------------------------------------------------------
// geometry of the step, incrementally.  After resolve, a node's neighbour
// word can differ from the last one only if its own owner or a neighbour's
// changed, and every change is in the change list.  The contact sums of a
// cell come from the nodes it owns, which lie inside its ellipsoid at its
// current position (a cell owns only nodes it covers); they are summed at
// the start of the next step, beside its sweep (the sweep needs only the
// neighbour words).

// neighbour word of node (x, y, z) from the owner map: for a fluid node bit 0,
// bit r neighbour x + c_r solid, NB_WALL / NB_CELL some solid neighbour is a
// wall / a cell; for a cell node its contact links (bit r: the neighbour is a
// wall node or another cell's); zero for wall nodes
// (the mixed word of a fluid node is written here, to node on_node)
__device__ __forceinline__ uint32_t node_word(const LatticeView &lv, int x, int y, int z, unsigned on_node,
                                              uint32_t &cellw) {
  using D = D3Q19;
  const unsigned nx = (unsigned)lv.nx, nxy = (unsigned)lv.nx * (unsigned)lv.ny;
  cellw = NBC_MIXED;
  const int xs[3] = {x == 0 ? lv.nx - 1 : x - 1, x, x == lv.nx - 1 ? 0 : x + 1};
  const int ys[3] = {y == 0 ? lv.ny - 1 : y - 1, y, y == lv.ny - 1 ? 0 : y + 1};
  const int zs[3] = {z == 0 ? lv.nz - 1 : z - 1, z, z == lv.nz - 1 ? 0 : z + 1};
  // the node's owner and its 18 neighbours' are requested together (one
  // memory round trip; a wall node's neighbour owners go unused)
  int on[Q];
  sfor<0, Q>([&](auto R) {
    constexpr int r = decltype(R)::value;
    on[r] = lv.owner[(unsigned)xs[1 + D::cx(r)] + nx * (unsigned)ys[1 + D::cy(r)] + nxy * (unsigned)zs[1 + D::cz(r)]];
  });
  const int own = on[0];
  if (own <= -2) return 0u;  // wall node
  if (own != FLUID) {
    // cell node: its contact links (neighbours owned by a wall or another cell)
    unsigned cmask = 0;
    sfor<1, Q>([&](auto R) {
      constexpr int r = decltype(R)::value;
      cmask |= (on[r] != FLUID && on[r] != own ? 1u : 0u) << r;
    });
    return cmask;
  }
  unsigned solid = 0, wall = 0;
  int first = -1;
  bool mixed = false;
  sfor<1, Q>([&](auto R) {
    constexpr int r = decltype(R)::value;
    solid |= (on[r] != FLUID ? 1u : 0u) << r;
    wall |= (on[r] <= -2 ? 1u : 0u) << r;
    if (on[r] != FLUID) {
      if (first == -1) first = on[r];
      else if (on[r] != first) mixed = true;
    }
  });
  if (first >= 0 && !mixed) cellw = (uint32_t)first;
  if (mixed && (solid & ~wall)) lv.nbx[on_node] = mixed_word(on);
  return NB_FLUID | solid | (wall ? NB_WALL : 0u) | ((solid & ~wall) ? NB_CELL : 0u);
}

// neighbour words of every changed node x and of the nodes x - c_r that see
// it; the whole lattice if the change list overflowed (grid-stride)
__global__ void k_nbm_update(LatticeView lv, ChangeList chg) {
  using D = D3Q19;
  pdl_wait();
  const int cnt = *chg.count;
  const bool all = cnt > chg.cap;
  const long long total = all ? (long long)lv.N : (long long)cnt * Q;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += stride) {
    int xyz[3];
    if (all) {
      node_xyz(lv, (unsigned)t, xyz);
    } else {
      const int c = (int)(t / Q), r = (int)(t - (long long)c * Q);
      node_xyz(lv, (unsigned)chg.items[3 * c], xyz);
      xyz[0] = wrapi(xyz[0] - D::cx(r), lv.nx);
      xyz[1] = wrapi(xyz[1] - D::cy(r), lv.ny);
      xyz[2] = wrapi(xyz[2] - D::cz(r), lv.nz);
    }
    uint32_t cw;
    const unsigned nn = node_of(lv, xyz[0], xyz[1], xyz[2]);
    lv.nbm[nn] = node_word(lv, xyz[0], xyz[1], xyz[2], nn, cw);
    lv.nbc[nn] = cw;
  }
}

// contact sums of one cell (one block per cell, Eqs. deltapppp,
// deltapppm): the rows of the cell's box, each cut to the outer interval of
// its ellipsoid at its current position, flattened over the block; every
// node the cell owns adds its links into another cell or a wall to exact
// integer sums (the cell's bounce links come from the sweep's records).  Each
// row writes its nodes into a list in shared memory, so that a node costs one
// shared read instead of a search of the row table (67 -> 48 us on 256^3
// beside the sweep, whose issue slots it shares), and only a node with
// contact links has its owner read.
constexpr int LB = 128;       // threads of a contact block (8 blocks fit an SM)
constexpr int CLIST = 4096;   // nodes listed at once: row (7 bits), place in the row (9 bits)

__global__ void __launch_bounds__(LB) k_contacts(LatticeView lv, PartView pv) {
  using D = D3Q19;
  __shared__ int sh_w[LB / 32 + 1];
  __shared__ int s_off[LB + 1], s_x0[LB], s_y[LB], s_z[LB];
  __shared__ uint16_t s_node[CLIST];
  __shared__ int s_ci[LB / 32][6];
  const int p = blockIdx.x;
  const int lo1 = pv.box[6 * p + 1], lo2 = pv.box[6 * p + 2];
  const int by = pv.box[6 * p + 4] - lo1 + 1, bz = pv.box[6 * p + 5] - lo2 + 1;
  const int rows = (by > 0 && bz > 0) ? by * bz : 0;
  CellGeo g;
  cell_geo(pv, pv.kin, p, g);
  const float ip = pv.inv_rperp2_f, kk = pv.kk_f;
  const int imin = lv.per[0] ? -(lv.nx / 2) : -g.Xi[0];
  const int imax = lv.per[0] ? imin + lv.nx - 1 : lv.nx - 1 - g.Xi[0];
  const unsigned nx = (unsigned)lv.nx, nxy = (unsigned)lv.nx * (unsigned)lv.ny;
  int ci[6] = {0, 0, 0, 0, 0, 0};
  for (int r0 = 0; r0 < rows; r0 += LB) {
    const int t = r0 + threadIdx.x;
    int len = 0, ao = 0, y = 0, z = 0;
    if (t < rows) {
      y = lo1 + t % by;
      z = lo2 + t / by;
      if (lv.per[1]) y = wrapi(y, lv.ny);
      if (lv.per[2]) z = wrapi(z, lv.nz);
      const RowQuad qn = row_quad((float)imin_image(y - g.Xi[1], lv.ny, lv.per[1]) - g.Xf[1],
                                  (float)imin_image(z - g.Xi[2], lv.nz, lv.per[2]) - g.Xf[2], g.of, ip, kk);
      int bo;
      row_range(qn, 1.0f + ROW_EPS, g.Xf[0], ao, bo);
      ao = max(ao, imin);
      bo = min(bo, imax);
      len = bo >= ao ? bo - ao + 1 : 0;
    }
    int tot;
    const int off = block_scan<LB>(len, sh_w, &tot);
    const bool listed = !__syncthreads_or(len > 511) && tot <= CLIST;
    s_off[threadIdx.x] = off;
    s_x0[threadIdx.x] = ao;
    s_y[threadIdx.x] = y;
    s_z[threadIdx.x] = z;
    if (listed)
      for (int j = 0; j < len; ++j) s_node[off + j] = (uint16_t)(threadIdx.x | (j << 7));
    __syncthreads();
    for (int k = threadIdx.x; k < tot; k += LB) {
      int lo = 0, j;
      if (listed) {
        lo = s_node[k] & 127;
        j = s_node[k] >> 7;
      } else {
        // the row holding flattened node k: the last row starting at or before k
        int hi = LB - 1;
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (s_off[mid] <= k) lo = mid;
          else hi = mid - 1;
        }
        j = k - s_off[lo];
      }
      int x = g.Xi[0] + s_x0[lo] + j;
      if (lv.per[0]) x = wrapi(x, lv.nx);
      const int yy = s_y[lo], zz = s_z[lo];
      const unsigned nn = (unsigned)x + nx * (unsigned)yy + nxy * (unsigned)zz;
      // the node's contact links, kept in its neighbour word by the geometry passes
      const uint32_t w = lv.nbm[nn];
      const unsigned cmask = (w & NB_FLUID) ? 0u : w & NB_SOLID;
      if (cmask && lv.owner[nn] == p) {
        const int di[3] = {imin_image(x - g.Xi[0], lv.nx, lv.per[0]), imin_image(yy - g.Xi[1], lv.ny, lv.per[1]),
                           imin_image(zz - g.Xi[2], lv.nz, lv.per[2])};
        sfor<1, Q>([&](auto R) {
          constexpr int r = decltype(R)::value;
          constexpr int m = D::m(r);
          if ((cmask >> r) & 1u) {
            ci[0] -= m * D::cx(r);
            ci[1] -= m * D::cy(r);
            ci[2] -= m * D::cz(r);
            ci[3] -= m * (di[1] * D::cz(r) - di[2] * D::cy(r));
            ci[4] -= m * (di[2] * D::cx(r) - di[0] * D::cz(r));
            ci[5] -= m * (di[0] * D::cy(r) - di[1] * D::cx(r));
          }
        });
      }
    }
    __syncthreads();  // the row tables are rewritten by the next chunk
  }
  block_sum_i<6, LB>(ci, s_ci);
  if (threadIdx.x == 0)
    for (int k = 0; k < 3; ++k) {
      pv.cK[3 * p + k] = ci[k];
      pv.cIT[3 * p + k] = ci[3 + k];
    }
}

// owners >= 0 become resting fluid (first particles_set), layout of parity par
template <class S>
__global__ void k_clear_cells(LatticeView lv, int par) {
  using D = D3Q19;
  const unsigned n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= lv.N) return;
  if (lv.owner[n] < 0) return;
  lv.owner[n] = FLUID;
  int xyz[3];
  node_xyz(lv, n, xyz);
  S *pop = reinterpret_cast<S *>(lv.pop);
  for (int r = 0; r < Q; ++r) {
    unsigned slot;
    if (par == 0 || r == 0) slot = (unsigned)r * lv.N + n;
    else
      slot = (unsigned)D::opp(r) * lv.N +
             node_of(lv, wrapi(xyz[0] - D::cx(r), lv.nx), wrapi(xyz[1] - D::cy(r), lv.ny), wrapi(xyz[2] - D::cz(r), lv.nz));
    Store<S>::st(pop + slot, 0.0f);
  }
}

// ---------------------------------------------------------------------------
// learned near-contact correction: pair features, close pairs, application

// features of the ordered pair (i, j) in the body frame of i (R the rotation
// of i): R^T r, q_i^* q_j with w >= 0, the gap |r| - sigma_R (Eq. sigma with
// the fluid-coupling half-axes), R^T (V_j - V_i), R^T (W_j - W_i); velocities
// of the current kinematics
__device__ void pair_features(const LatticeView &lv, const PartView &pv, int i, int j, float f[14], float R[3][3]) {
  const float4 a0 = pv.kin[3 * i], a1 = pv.kin[3 * i + 1], a2 = pv.kin[3 * i + 2];
  const float4 b0 = pv.kin[3 * j], b1 = pv.kin[3 * j + 1], b2 = pv.kin[3 * j + 2];
  const int dims[3] = {lv.nx, lv.ny, lv.nz};
  const int ai[3] = {(int)a0.w, (int)a1.w, (int)a2.w}, bi[3] = {(int)b0.w, (int)b1.w, (int)b2.w};
  const float af[3] = {a0.x, a0.y, a0.z}, bf[3] = {b0.x, b0.y, b0.z};
  float r[3];
  for (int k = 0; k < 3; ++k) r[k] = (float)imin_image(bi[k] - ai[k], dims[k], lv.per[k]) + (bf[k] - af[k]);
  const float4 qi = pv.qf[i], qj = pv.qf[j];
  rotmat_f(qi, R);
  float Rj[3][3];
  rotmat_f(qj, Rj);
  const float oi[3] = {R[0][2], R[1][2], R[2][2]}, oj[3] = {Rj[0][2], Rj[1][2], Rj[2][2]};
  const float rl = sqrtf(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]), ir = 1.0f / rl;
  const float a = (r[0] * oi[0] + r[1] * oi[1] + r[2] * oi[2]) * ir, b = (r[0] * oj[0] + r[1] * oj[1] + r[2] * oj[2]) * ir;
  const float c = oi[0] * oj[0] + oi[1] * oj[1] + oi[2] * oj[2];
  const float Rp2 = (float)(pv.R_par * pv.R_par), Rq2 = (float)(pv.R_perp * pv.R_perp);
  const float chi = (Rp2 - Rq2) / (Rp2 + Rq2);
  const float S = 1.0f - 0.5f * chi * ((a + b) * (a + b) / (1.0f + chi * c) + (a - b) * (a - b) / (1.0f - chi * c));
  const float gap = rl - 2.0f * (float)pv.R_perp * rsqrtf(S);
  const float dv[3] = {b1.x - a1.x, b1.y - a1.y, b1.z - a1.z}, dw[3] = {b2.x - a2.x, b2.y - a2.y, b2.z - a2.z};
  for (int k = 0; k < 3; ++k) {
    f[k] = R[0][k] * r[0] + R[1][k] * r[1] + R[2][k] * r[2];
    f[8 + k] = R[0][k] * dv[0] + R[1][k] * dv[1] + R[2][k] * dv[2];
    f[11 + k] = R[0][k] * dw[0] + R[1][k] * dw[1] + R[2][k] * dw[2];
  }
  const float w1 = qi.x, x1 = -qi.y, y1 = -qi.z, z1 = -qi.w;
  const float w2 = qj.x, x2 = qj.y, y2 = qj.z, z2 = qj.w;
  float qr[4] = {w1 * w2 - x1 * x2 - y1 * y2 - z1 * z2, w1 * x2 + x1 * w2 + y1 * z2 - z1 * y2,
                 w1 * y2 - x1 * z2 + y1 * w2 + z1 * x2, w1 * z2 + x1 * y2 - y1 * x2 + z1 * w2};
  const float sgn = qr[0] < 0.f ? -1.f : 1.f;
  for (int k = 0; k < 4; ++k) f[3 + k] = sgn * qr[k];
  f[7] = gap;
}

__global__ void k_pair_features(LatticeView lv, PartView pv, const int2 *pairs, int n, float *out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int2 pr = pairs[t];
  if (pr.x < 0 || pr.x >= pv.n || pr.y < 0 || pr.y >= pv.n || pr.x == pr.y) {
    for (int k = 0; k < 14; ++k) out[14 * t + k] = 0.f;
    return;
  }
  float f[14], R[3][3];
  pair_features(lv, pv, pr.x, pr.y, f, R);
  for (int k = 0; k < 14; ++k) out[14 * t + k] = f[k];
}

// close pairs (gap_lo <= gap < gap_cut, relative speed |V_j - V_i| in
// [speed_lo, speed_hi]) from the cell list, one warp per cell, with their
// features; a pair whose centres are farther apart than the largest contact
// distance and the cut-off is left before its features are formed
__global__ void __launch_bounds__(32) k_mlp_pairs(LatticeView lv, PartView pv, CellListView cl, PairBuf pb,
                                                  float gap_lo, float gap_cut, float speed_lo, float speed_hi) {
  __shared__ NearBins s_nb;
  const int i = blockIdx.x;
  near_bins(lv, cl, cl.bin_of[i], s_nb);
  __syncwarp();
  CellGeo g;
  cell_geo(pv, pv.kin, i, g);
  const int dims[3] = {lv.nx, lv.ny, lv.nz};
  const float far = (2.0f * pv.Rmax_f + gap_cut) * 1.0001f + 1e-3f;
  for (int t = threadIdx.x; t < s_nb.off[27]; t += 32) {
    const int j = near_cell(cl, s_nb, t);
    if (j == i) continue;
    CellGeo h;
    cell_geo(pv, pv.kin, j, h);
    float r2 = 0.f;
    for (int m = 0; m < 3; ++m) {
      const float d = (float)imin_image(h.Xi[m] - g.Xi[m], dims[m], lv.per[m]) + (h.Xf[m] - g.Xf[m]);
      r2 += d * d;
    }
    if (!(far > 0.f) || r2 > far * far) continue;
    float f[14], R[3][3];
    pair_features(lv, pv, i, j, f, R);
    if (!(f[7] >= gap_lo && f[7] < gap_cut)) continue;  // outside the range: the plain method
    const float sp = sqrtf(f[8] * f[8] + f[9] * f[9] + f[10] * f[10]);
    if (!(sp >= speed_lo && sp <= speed_hi)) continue;
    const int s = atomicAdd(pb.count, 1);
    if (s >= pb.cap) {
      atomicOr(pv.status, ST_OVERFLOW);
      continue;
    }
    pb.pairs[s] = make_int2(i, j);
    for (int q = 0; q < 14; ++q) pb.feat[14 * s + q] = f[q];
  }
}

// the network's force and torque on i, back from its body frame to the lab
// frame, added to the potentials of the step
__global__ void k_mlp_apply(PartView pv, PairBuf pb) {
  const int n = min(*pb.count, pb.cap);
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x) {
    const int i = pb.pairs[s].x;
    float R[3][3];
    rotmat_f(pv.qf[i], R);
    const float *y = pb.out + 6 * s;
    for (int k = 0; k < 3; ++k) {
      atomicAdd(&pv.Fpot[3 * i + k], (double)(R[k][0] * y[0] + R[k][1] * y[1] + R[k][2] * y[2]));
      atomicAdd(&pv.Tpot[3 * i + k], (double)(R[k][0] * y[3] + R[k][1] * y[4] + R[k][2] * y[5]));
    }
  }
}

// ---------------------------------------------------------------------------
// host-side launchers

static inline unsigned nblk(unsigned n, unsigned b) { return (n + b - 1) / b; }

// whether this context's cell kernels are launched as programmatic dependents:
// not in an ensemble, whose members' kernels would wait for SM slots that the
// waiting blocks hold (16 members: 368 -> 388 us a step), and not for
// thousands of cells, whose kernels fill the GPU by themselves (8446: 1081 ->
// 1084 us); 20 cells 44 -> 41 us, 1022 cells 160 -> 157 us
static inline bool dependents(const LatticeView &lv, const PartView &pv) { return lv.dep && pv.n <= 4096; }

void launch_cell_list(const LatticeView &lv, const PartView &pv, const CellListView &cl, cudaStream_t st, int64_t *nl) {
  if (pv.n == 0) return;
  const size_t smem = sizeof(int) * ((size_t)cl.nbins + (size_t)pv.n);
  if (pv.n <= CL_ONE && smem <= CL_SMEM) {
    k_cl_one<<<1, CL_T, smem, st>>>(lv, pv, cl);
    *nl += 1;
    return;
  }
  k_cl_bin<<<nblk(pv.n, 128), 128, 0, st>>>(lv, pv, cl);
  k_cl_scan<<<1, 1024, 0, st>>>(cl);
  k_cl_scatter<<<nblk(pv.n, 128), 128, 0, st>>>(pv, cl);
  k_cl_sort<<<nblk(cl.nbins, 128), 128, 0, st>>>(cl);
  *nl += 4;
}

void launch_forces(const LatticeView &lv, const PartView &pv, const CellListView &cl, const SurfBits &sb,
                   cudaStream_t st, int64_t *nl) {
  if (pv.n == 0) return;
  // few blocks may wait for the list on the SMs; a thousand would keep the sweep
  // beside them from its slots
  launch_dependent(dependents(lv, pv) && pv.n <= 2 * 152, k_forces, pv.n, FB, st, lv, pv, cl, sb);
  *nl += 1;
}

void launch_sums_solve(const LatticeView &lv, const PartView &pv, cudaStream_t st, int64_t *nl) {
  if (pv.n == 0) return;
  if (lv.has_force) k_link_reduce<true><<<pv.n, LT, 0, st>>>(lv, pv);
  else k_link_reduce<false><<<pv.n, LT, 0, st>>>(lv, pv);
  launch_dependent(dependents(lv, pv), k_solve, nblk(pv.n, SOLVE_CELLS), 32, st, lv, pv);
  *nl += 2;
}

void launch_link_pending(int dtype, const LatticeView &lv, const PartView &pv, int par, cudaStream_t st,
                         int64_t *nl) {
  if (pv.n == 0) return;
  if (dtype == 0) k_link_pending<float><<<pv.n, LT, 0, st>>>(lv, pv, par);
  else if (dtype == 1) k_link_pending<__nv_bfloat16><<<pv.n, LT, 0, st>>>(lv, pv, par);
  else k_link_pending<__half><<<pv.n, LT, 0, st>>>(lv, pv, par);
  *nl += 1;
}

void launch_flush_pending(int dtype, const LatticeView &lv, int par, cudaStream_t st, int64_t *nl) {
  // one node per thread: 608 blocks walking the lattice kept too few loads in
  // flight (1113 us on 256^3, whose 268 MB of pending velocities take 40 us)
  const unsigned b = 256, g = nblk(lv.N, b);
  if (dtype == 0) k_flush_pending<float><<<g, b, 0, st>>>(lv, par);
  else if (dtype == 1) k_flush_pending<__nv_bfloat16><<<g, b, 0, st>>>(lv, par);
  else k_flush_pending<__half><<<g, b, 0, st>>>(lv, par);
  *nl += 1;
}

void launch_pair_features(const LatticeView &lv, const PartView &pv, const int2 *pairs, int n, float *out,
                          cudaStream_t st) {
  if (n > 0) k_pair_features<<<nblk(n, 128), 128, 0, st>>>(lv, pv, pairs, n, out);
}

void launch_mlp_pairs(const LatticeView &lv, const PartView &pv, const CellListView &cl, const PairBuf &pb,
                      float gap_lo, float gap_cut, float speed_lo, float speed_hi, const void *mlp, cudaStream_t st,
                      int64_t *nl) {
  if (pv.n == 0) return;
  cudaMemsetAsync(pb.count, 0, sizeof(int), st);
  k_mlp_pairs<<<pv.n, 32, 0, st>>>(lv, pv, cl, pb, gap_lo, gap_cut, speed_lo, speed_hi);
  launch_mlp_forward_dev(mlp, pb.feat, pb.count, pb.cap, pb.out, st);
  *nl += 2;
}

void launch_mlp_apply(const PartView &pv, const PairBuf &pb, cudaStream_t st, int64_t *nl) {
  if (pv.n == 0) return;
  k_mlp_apply<<<nblk((unsigned)pb.cap, 128) < 152u ? nblk((unsigned)pb.cap, 128) : 152u, 128, 0, st>>>(pv, pb);
  *nl += 1;
}

void launch_set_state(const LatticeView &lv, const PartView &pv, int mode, cudaStream_t st, int64_t *nl) {
  if (pv.n == 0) return;
  k_set_state<<<nblk(pv.n, 64), 64, 0, st>>>(lv, pv, mode);
  *nl += 1;
}

void launch_claims(const LatticeView &lv, const PartView &pv, int *claim, const ChangeList &chg, int mode,
                   cudaStream_t st, int64_t *nl) {
  if (pv.n == 0) return;
  k_claims<<<pv.n, PB, 0, st>>>(lv, pv, claim, chg, mode);
  *nl += 1;
}

void launch_nbm_update(const LatticeView &lv, const PartView &pv, const ChangeList &chg, cudaStream_t st,
                       int64_t *nl) {
  if (pv.n == 0) return;
  launch_dependent(dependents(lv, pv), k_nbm_update, 4 * 152, 256, st, lv, chg);
  *nl += 1;
}

void launch_contacts(const LatticeView &lv, const PartView &pv, cudaStream_t st, int64_t *nl) {
  if (pv.n == 0) return;
  k_contacts<<<pv.n, LB, 0, st>>>(lv, pv);
  *nl += 1;
}

void launch_resolve_fill(int dtype, const LatticeView &lv, const PartView &pv, const CellListView &cl, int *claim,
                         const ChangeList &chg, int par_next, int impulses, int replaced, cudaStream_t st,
                         int64_t *nl) {
  if (pv.n == 0) return;
#define BL_RESOLVE(S_)                                                                              \
  if (replaced) k_resolve_fill<S_, true><<<pv.n, PB, 0, st>>>(lv, pv, cl, claim, chg, par_next, impulses); \
  else k_resolve_fill<S_, false><<<pv.n, PB, 0, st>>>(lv, pv, cl, claim, chg, par_next, impulses)
  if (dtype == 0) {
    BL_RESOLVE(float);
  } else if (dtype == 1) {
    BL_RESOLVE(__nv_bfloat16);
  } else {
    BL_RESOLVE(__half);
  }
#undef BL_RESOLVE
  *nl += 1;
}


void launch_clear_cells(int dtype, const LatticeView &lv, int par, cudaStream_t st, int64_t *nl) {
  const unsigned b = 256, g = nblk(lv.N, b);
  if (dtype == 0) k_clear_cells<float><<<g, b, 0, st>>>(lv, par);
  else if (dtype == 1) k_clear_cells<__nv_bfloat16><<<g, b, 0, st>>>(lv, par);
  else k_clear_cells<__half><<<g, b, 0, st>>>(lv, par);
  *nl += 1;
}

}  // namespace bl
