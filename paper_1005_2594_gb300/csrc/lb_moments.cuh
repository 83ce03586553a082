// lb_moments.cuh -- density deviation and momentum of a node's 19 shifted
// populations in FP64, for the field read-outs of the dense and the indexed
// lattice.
//
// FP64 arithmetic issues at 2 lanes per cycle and SM on this GPU: summed
// directly (19 conversions, 45 additions, three divisions), it took k_fields
// 5171 us on 256^3 with cells (FP32 storage), twenty times what its 1.9 GB
// need.  Here the sums are taken in FP32 without rounding: each population is
// split against a power of two above the sum of their sizes into a part q on
// a coarse grid, a second part on a grid 19 bits finer and a rest (error-free
// extraction, as in Rump, Ogita & Oishi, "Accurate floating-point summation",
// 2008).  Nineteen parts on one grid add exactly in 24 bits, and the rest is
// below 2^-40 of their sum, so its FP32 sum is good to 2^-57 of it: no worse
// than FP64 additions.  The three sums go into one 64-bit integer that is
// rounded once to FP64 by its bits.  What stays in FP64 is 8 instructions per
// node (each holds the SM's FP64 pipe for 16 cycles: 13 took 472 us on 256^3).
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

// K 2^e in FP64, rounded once to nearest even; |K| < 2^63, the result normal
// (integer instructions: a conversion from 64-bit integers is an FP64 one)
__device__ __forceinline__ double scaled_int(long long K, int e) {
  if (K == 0) return 0.0;
  const unsigned long long s = (unsigned long long)K & (1ull << 63);
  unsigned long long a = (unsigned long long)(K < 0 ? -K : K);
  const int z = __clzll((long long)a);
  a <<= z;  // leading bit at 63
  // 53 bits kept; half an ulp, and the lowest kept bit where the rest is a tie
  a = (a >> 11) + (((a >> 10) & 1ull) & (((a & 0x3FFull) != 0ull || ((a >> 11) & 1ull)) ? 1ull : 0ull));
  // a is the significand with its leading one at bit 52 (or 53 after a carry,
  // which adds one to the exponent by itself)
  return __longlong_as_double((long long)(s | (a + ((unsigned long long)(63 - z + e + 1022) << 52))));
}

// a normal positive float as FP64 (exact; by its bits for the same reason)
__device__ __forceinline__ double widen(float x) {
  const unsigned b = __float_as_uint(x);
  return __hiloint2double((int)((b >> 3) + (896u << 20)), (int)(b << 29));
}

// sum of the populations (m[0]) and of the populations times c_r (m[1..3]);
// false if they are not finite or not within 2^-60..2^60
__device__ __forceinline__ bool moments64(const float (&f)[Q], double (&m)[4]) {
  using D = D3Q19;
  float A = 0.f;  // bounds each population and every partial sum
  sfor<0, Q>([&](auto R) { A += fabsf(f[decltype(R)::value]); });
  if (A == 0.f) {
    m[0] = m[1] = m[2] = m[3] = 0.0;
    return true;
  }
  const unsigned be = __float_as_uint(A) >> 23;  // 2^(be - 127) <= A < 2^(be - 126)
  if (be < 67u || be > 187u) return false;       // (NaN and infinity are above)
  // E = be - 127, sum |f| < 2^(E + 1) (1 + 2^-19).  Grid 1: parts are multiples
  // of 2^(E - 22), their sums below 2^24 of them.  Grid 2: rests |p| <= 2^(E - 22),
  // parts multiples of 2^(E - 41), their sums below 2^24 of them.  The last rest
  // is at most 2^(E - 41), its FP32 sum good to 2^(E - 57).
  const float s1 = exp2_biased(be + 2u), s2 = exp2_biased(be - 17u);
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
  const float c1 = exp2_biased(276u - be), c2 = exp2_biased(295u - be), c3 = exp2_biased(311u - be);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    // units of 2^(E - 57): the first two are exact integers
    const long long K = ((long long)__float2int_rn(S[0][k] * c1) << 35) +
                        ((long long)__float2int_rn(S[1][k] * c2) << 16) + (long long)__float2int_rn(S[2][k] * c3);
    m[k] = scaled_int(K, (int)be - 184);
  }
  return true;
}

// rho and u = j / rho + g / 2 (= (j + rho g / 2) / rho) of one fluid node;
// hg = g / 2.  1 / rho by two Newton steps in FP64 from the FP32 reciprocal.
__device__ __forceinline__ void node_fields(const float (&f)[Q], double rho0, const double (&hg)[3], double &rho,
                                            double (&u)[3]) {
  double m[4];
  if (!moments64(f, m)) {
    float g[Q];
    for (int r = 0; r < Q; ++r) g[r] = f[r];
    moments_plain(g, m);
  }
  rho = rho0 + m[0];
  // rho to FP32 from its bits, where it is a normal number above 0
  const unsigned hi = (unsigned)__double2hiint(rho), lo = (unsigned)__double2loint(rho);
  const unsigned ex = hi >> 20;  // sign and exponent
  if (ex > 1023u - 100u && ex < 1023u + 100u) {
    double x = widen(1.0f / __uint_as_float(((hi - (896u << 20)) << 3) | (lo >> 29)));
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
