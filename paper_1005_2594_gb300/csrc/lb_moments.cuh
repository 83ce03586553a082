// lb_moments.cuh -- density deviation and momentum of a node's 19 shifted
// populations in FP64, for the field read-outs of the dense and the indexed
// lattice.
//
// FP64 arithmetic issues at 2 lanes per cycle and SM on this GPU: summed
// directly (19 conversions, 45 additions, three divisions), it took k_fields
// 5171 us on 256^3 with cells (FP32 storage), twenty times what its 1.9 GB
// need.  Here the sums are taken in FP32 without rounding: each population is
// split against a power of two above the node's largest one into a part q on
// a coarse grid, a second part on a grid 19 bits finer and a rest (error-free
// extraction, as in Rump, Ogita & Oishi, "Accurate floating-point summation",
// 2008).  Nineteen parts on one grid add exactly in 24 bits, and the rest is
// below 2^-37 of the largest population, so its FP32 sum is good to 2^-56 of
// it: no worse than FP64 additions.  The three sums go into one 64-bit integer
// whose conversion to FP64 rounds once.  What stays in FP64 is 13 instructions
// per node.
#pragma once

#include "bl_internal.cuh"

namespace bl {

// the sums in plain FP64, where a population is not within 2^-60..2^60, is
// infinite or NaN
static __device__ __noinline__ void moments_plain(const float *f, double *m) {
  double d = 0.0, j0 = 0.0, j1 = 0.0, j2 = 0.0;
  for (int r = 0; r < Q; ++r) {
    const double v = (double)f[r];
    d += v;
    j0 += v * rt_c<0>(r);
    j1 += v * rt_c<1>(r);
    j2 += v * rt_c<2>(r);
  }
  m[0] = d;
  m[1] = j0;
  m[2] = j1;
  m[3] = j2;
}

// power of two with biased exponent b
__device__ __forceinline__ float exp2_biased(unsigned b) { return __uint_as_float(b << 23); }

// sum of the populations (m[0]) and of the populations times c_r (m[1..3])
__device__ __forceinline__ void moments64(const float (&f)[Q], double (&m)[4]) {
  using D = D3Q19;
  float M = 0.f;
  bool ok = true;
  sfor<0, Q>([&](auto R) {
    constexpr int r = decltype(R)::value;
    M = fmaxf(M, fabsf(f[r]));
    ok = ok && (f[r] == f[r]);
  });
  if (ok && M == 0.f) {
    m[0] = m[1] = m[2] = m[3] = 0.0;
    return;
  }
  const unsigned be = __float_as_uint(M) >> 23;  // 2^(be - 127) <= M < 2^(be - 126)
  if (!ok || be < 67u || be > 187u) {
    float g[Q];
    for (int r = 0; r < Q; ++r) g[r] = f[r];
    moments_plain(g, m);
    return;
  }
  // E = be - 127.  Grid 1: |f| < 2^(E + 1), parts are multiples of 2^(E - 18),
  // a sum of 19 stays below 2^24 of them.  Grid 2: rests |p| <= 2^(E - 18),
  // parts multiples of 2^(E - 37).  The last rest is at most 2^(E - 37).
  const float s1 = exp2_biased(be + 6u), s2 = exp2_biased(be - 13u);
  float S[3][4];
#pragma unroll
  for (int l = 0; l < 3; ++l)
#pragma unroll
    for (int k = 0; k < 4; ++k) S[l][k] = 0.f;
  sfor<0, Q>([&](auto R) {
    constexpr int r = decltype(R)::value;
    const float q1 = __fsub_rn(__fadd_rn(s1, f[r]), s1), p1 = __fsub_rn(f[r], q1);
    const float q2 = __fsub_rn(__fadd_rn(s2, p1), s2), p2 = __fsub_rn(p1, q2);
    const float v[3] = {q1, q2, p2};
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      S[l][0] = __fadd_rn(S[l][0], v[l]);
      if constexpr (D::cx(r) != 0) S[l][1] = __fadd_rn(S[l][1], D::cx(r) > 0 ? v[l] : -v[l]);
      if constexpr (D::cy(r) != 0) S[l][2] = __fadd_rn(S[l][2], D::cy(r) > 0 ? v[l] : -v[l]);
      if constexpr (D::cz(r) != 0) S[l][3] = __fadd_rn(S[l][3], D::cz(r) > 0 ? v[l] : -v[l]);
    }
  });
  const float c1 = exp2_biased(272u - be), c2 = exp2_biased(291u - be), c3 = exp2_biased(311u - be);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    // units of 2^(E - 57): the first two are exact integers
    const long long K = ((long long)__float2int_rn(S[0][k] * c1) << 39) +
                        ((long long)__float2int_rn(S[1][k] * c2) << 20) + (long long)__float2int_rn(S[2][k] * c3);
    const long long bits = __double_as_longlong(__ll2double_rn(K)) + ((long long)((int)be - 184) << 52);
    m[k] = K != 0 ? __longlong_as_double(bits) : 0.0;
  }
}

// rho and u = j / rho + g / 2 (= (j + rho g / 2) / rho) of one fluid node;
// hg = g / 2.  1 / rho by two Newton steps in FP64 from the FP32 reciprocal.
__device__ __forceinline__ void node_fields(const float (&f)[Q], double rho0, const double (&hg)[3], double &rho,
                                            double (&u)[3]) {
  double m[4];
  moments64(f, m);
  rho = rho0 + m[0];
  const float rf = (float)rho;
  if (rf > 1e-30f && rf < 1e30f) {
    double x = (double)(1.0f / rf);
    x = fma(x, fma(-rho, x, 1.0), x);
    x = fma(x, fma(-rho, x, 1.0), x);
    for (int k = 0; k < 3; ++k) u[k] = fma(m[k + 1], x, hg[k]);
  } else {
    for (int k = 0; k < 3; ++k) u[k] = (m[k + 1] + rho * hg[k]) / rho;
  }
}

// u (n x 3 doubles) of a warp's 32 consecutive rows from row0, through shared
// memory so that the lanes write consecutive words (three strided 8-byte
// stores per lane touch every sector of the rows three times)
__device__ __forceinline__ void store_u_rows(double *out, size_t row0, size_t rows, double *stage, const double (&u)[3]) {
  const int lane = threadIdx.x & 31;
  for (int k = 0; k < 3; ++k) stage[3 * lane + k] = u[k];
  __syncwarp();
  for (int k = 0; k < 3; ++k) {
    const int e = lane + 32 * k;
    if (row0 + e / 3 < rows) out[3 * row0 + e] = stage[e];
  }
  __syncwarp();
}

}  // namespace bl
