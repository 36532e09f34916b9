// mt_pair.cuh -- per-pair arithmetic shared by the transfer kernels: the
// exact cutoff test, the co-location weight (Eq. 3), the normalisation
// (Sec. 1.1), and mass access / accumulation / update / reaction in each
// precision (Eq. 4, Eq. 7; Sec. 3 reaction).
#pragma once

#include "mt_internal.cuh"

namespace mt {

// ---------------------------------------------------------- pair weights --

__device__ __forceinline__ bool in_range2(long long dx, long long dy, long long S) {
  const unsigned long long ax = (unsigned long long)(dx < 0 ? -dx : dx);
  const unsigned long long ay = (unsigned long long)(dy < 0 ? -dy : dy);
  if (ax > (unsigned long long)S || ay > (unsigned long long)S) return false;
  return ax * ax + ay * ay <= (unsigned long long)S * (unsigned long long)S;
}

// nu_ij without its prefactor (it cancels in the normalisation):
// exp(-s^2 / (8 D_mt dt)) with s = |dX| 2^-k (Eq. 3).
template <bool MIX, int DIM>
struct Weight;

// ------------------------------------------------- binary64 exponential --
// exp(-t) for t >= 0 in binary64 (the weights of Eq. 3 in MT_FP64), by
// Tang's table-driven method (P. T. P. Tang, ACM TOMS 15(2), 1989): with
// k = rint(-t 32/ln2) = 32 m + j (0 <= j < 32) and r = -t - k ln2/32
// (|r| <= ln2/64; ln2/32 split into a 37-bit head, so that k times it is
// exact for |k| < 2^16, and a tail), exp(-t) = 2^m 2^(j/32) e^r, where
// 2^(j/32) comes from a table of its correctly rounded values and e^r - 1
// = r + r^2 q(r) from the Taylor polynomial of degree 6 (truncation below
// 2^-57 relative for |r| <= ln2/64).  The result is 2^(j/32) + 2^(j/32)
// (e^r - 1) with one rounding, then scaled by 2^m in its exponent field.
// Error about 1 ulp; 11 binary64 operations.
__constant__ double kExp2j32[32] = {
    0x1.0000000000000p+0, 0x1.059b0d3158574p+0, 0x1.0b5586cf9890fp+0, 0x1.11301d0125b51p+0,
    0x1.172b83c7d517bp+0, 0x1.1d4873168b9aap+0, 0x1.2387a6e756238p+0, 0x1.29e9df51fdee1p+0,
    0x1.306fe0a31b715p+0, 0x1.371a7373aa9cbp+0, 0x1.3dea64c123422p+0, 0x1.44e086061892dp+0,
    0x1.4bfdad5362a27p+0, 0x1.5342b569d4f82p+0, 0x1.5ab07dd485429p+0, 0x1.6247eb03a5585p+0,
    0x1.6a09e667f3bcdp+0, 0x1.71f75e8ec5f74p+0, 0x1.7a11473eb0187p+0, 0x1.82589994cce13p+0,
    0x1.8ace5422aa0dbp+0, 0x1.93737b0cdc5e5p+0, 0x1.9c49182a3f090p+0, 0x1.a5503b23e255dp+0,
    0x1.ae89f995ad3adp+0, 0x1.b7f76f2fb5e47p+0, 0x1.c199bdd85529cp+0, 0x1.cb720dcef9069p+0,
    0x1.d5818dcfba487p+0, 0x1.dfc97337b9b5fp+0, 0x1.ea4afa2a490dap+0, 0x1.f50765b6e4540p+0,
};
__device__ __forceinline__ double exp_neg(double t) {
  if (!(t <= 745.5)) return t > 745.5 ? 0.0 : t + t;  // underflow; a NaN stays one
  const double x = -t;
  const double kMagic = 0x1.8p52;  // rint by addition: ulp 1 at 1.5 * 2^52
  const double kd = __fma_rn(x, 0x1.71547652b82fep+5, kMagic);  // x 32 / ln2
  const int k = (int)(unsigned int)(unsigned long long)__double_as_longlong(kd);
  const double kf = kd - kMagic;
  double r = __fma_rn(-kf, 0x1.62e42fefa0000p-6, x);  // head of ln2 / 32
  r = __fma_rn(-kf, 0x1.cf79abc9e3b3ap-45, r);        // tail
  double q = __fma_rn(r, 0x1.6c16c16c16c17p-10, 0x1.1111111111111p-7);  // 1/720, 1/120
  q = __fma_rn(r, q, 0x1.5555555555555p-5);                               // 1/24
  q = __fma_rn(r, q, 0x1.5555555555555p-3);                               // 1/6
  q = __fma_rn(r, q, 0.5);
  const double em1 = __fma_rn(__dmul_rn(r, r), q, r);
  const double T = kExp2j32[k & 31];
  const double res = __fma_rn(T, em1, T);
  const int m = k >> 5;
  if (m >= -1021)
    return __longlong_as_double(__double_as_longlong(res) + ((long long)m << 52));
  return scalbn(res, m);  // a subnormal result
}

// ------------------------------------- binary64 weights within the cutoff --
// exp(-s^2 / (8 D_mt dt)) for a pair within the cutoff, from its squared
// separation R2 in ticks (an exact integer below 2^60), in 64-bit integer
// arithmetic: the binary64 pipe issues a warp instruction every ~19 cycles
// per multiprocessor, so the 13 binary64 operations of the table method
// above hold it for ~250 cycles per 32 weights, while the ~60 integer
// instructions here take ~20 issue cycles of the four schedulers.
//   v = R2 c (c = log2(e) / (8 D_mt dt) 2^-2k) in fixed point with d.eib
//   integer bits = m + F, and exp(-s^2/(8 D_mt dt)) = 2^-m 2^-F;
//   2^-F = T_j (1 - p(x)): T_j = 2^(-j/256) from a table (63 fraction bits,
//   the first 8 bits of F) and 1 - 2^(-x/256) ~ p(x) = x (b1 - x (b2 - x
//   (b3 - x b4))), x in [0, 1) the rest of F, the polynomial through the
//   Chebyshev points (truncation 2^-56.5); the 63-bit result is rounded once
//   to binary64 and 2^-m goes into its exponent field.
// Relative error below 1.11 2^-53 for the cutoffs in use (the table method
// over binary64 squares: up to 7 2^-53, since the exponent itself is rounded).
// Measured (75 dense realisations of 5000 particles, 10^8 ordered pairs per
// step): 8.58 -> 1.79 ms per step; N = 10^5 at one per unit length: 42 -> 36 us.
__device__ const unsigned long long kExp2Neg[256] = {
    0x8000000000000000ull, 0x7fa765aca88f6453ull, 0x7f4f08ae3dc7c426ull, 0x7ef6e8da4b544f9aull,
    0x7e9f06067a4360baull, 0x7e47600890f223deull, 0x7deff6b672f84e24ull, 0x7d98c9e62113e1faull,
    0x7d41d96db915019dull, 0x7ceb252375c9cf9bull, 0x7c94acddaeea5d3aull, 0x7c3e7072d904a6ceull,
    0x7be86fb985689ddcull, 0x7b92aa886214411cull, 0x7b3d20b6399fc237ull, 0x7ae7d219f329b948ull,
    0x7a92be8a92436616ull, 0x7a3de5df36dcfeefull, 0x79e947ef1d320d2dull, 0x7994e4919db5d74eull,
    0x7940bb9e2cffd89dull, 0x78ecccec5bb84661ull, 0x78991853d684a285ull, 0x78459dac65f45bb5ull,
    0x77f25ccdee6d7ae6ull, 0x779f559070195e36ull, 0x774c87cc06d1812eull, 0x76f9f358ea0c5249ull,
    0x76a7980f6cca15c2ull, 0x765575c7fd81d5a0ull, 0x76038c5b260e5eeeull, 0x75b1dba18b9b4c20ull,
    0x75606373ee921c97ull, 0x750f23ab2a87593eull, 0x74be1c203627c62bull, 0x746d4cac2325a155ull,
    0x741cb5281e25ee34ull, 0x73cc556d6eadce5full, 0x737c2d55770fe711ull, 0x732c3cb9b459d38bull,
    0x72dc8373be41a454ull, 0x728d015d47136b40ull, 0x723db6501b9ed447ull, 0x71eea2262324cb0cull,
    0x719fc4b95f452d29ull, 0x71511de3ebec8913ull, 0x7102ad7fff41e9b4ull, 0x70b47367e994ae92ull,
    0x70666f76154a7089ull, 0x7018a18506ccf314ull, 0x6fcb096f5c782210ull, 0x6f7da70fce881bf9ull,
    0x6f307a412f074892ull, 0x6ee382de69bc7bf8ull, 0x6e96c0c284192610ull, 0x6e4a33c89d278e49ull,
    0x6dfddbcbed791babull, 0x6db1b8a7c714a92bull, 0x6d65ca379564e639ull, 0x6d1a1056dd26c382ull,
    0x6cce8ae13c57ebdbull, 0x6c8339b26a25494eull, 0x6c381ca636d99642ull, 0x6bed33988bcbfab5ull,
    0x6ba27e656b4eb57aull, 0x6b57fce8f09dd17full, 0x6b0daeff4fcde703ull, 0x6ac39484d5bae8c5ull,
    0x6a79ad55e7f6fd10ull, 0x6a2ff94f04b962b0ull, 0x69e6784cc2cd61bdull, 0x699d2a2bd181482aull,
    0x69540ec8f895722dull, 0x690b2601182b5e56ull, 0x68c26fb128b4cd63ull, 0x6879ebb63ae2edc6ull,
    0x683199ed779592caull, 0x67e97a341fca775bull, 0x67a18c678c8c8c61ull, 0x6759d0652ee352afull,
    0x6712460a8fc24072ull, 0x66caed354ff83222ull, 0x6683c5c3281ee6e9ull, 0x663ccf91e88a8873ull,
    0x65f60a7f79393e2eull, 0x65af7669d9c2cbe4ull, 0x6569132f21483ba7ull, 0x6522e0ad7e639312ull,
    0x64dcdec3371793d1ull, 0x64970d4ea8bf8766ull, 0x64516c2e47ff1623ull, 0x640bfb40a0b22959ull,
    0x63c6ba6455dcd8aeull, 0x6381a978219b628full, 0x633cc85ad5122fbdull, 0x62f816eb585de1edull,
    0x62b39508aa836d6full, 0x626f4291e1603dd5ull, 0x622b1f66299a6599ull, 0x61e72b64c690d8afull,
    0x61a3666d124bb204ull, 0x615fd05e7d6c83e4ull, 0x611c69188f1eb339ull, 0x60d9307ae507dd9aull,
    0x6096266533384a2bull, 0x60534ab7441b6546ull, 0x60109d50f86846d8ull, 0x5fce1e124712437cull,
    0x5f8bccdb3d398841ull, 0x5f49a98bfe1bc11cull, 0x5f07b404c304c9f1ull, 0x5ec5ec25db3f6a41ull,
    0x5e8451cfac061b5full, 0x5e42e4e2b073d935ull, 0x5e01a53f7974fd86ull, 0x5dc092c6adb825b8ull,
    0x5d7fad59099f22feull, 0x5d3ef4d75f2ff504ull, 0x5cfe69229605cef5ull, 0x5cbe0a1bab4226dfull,
    0x5c7dd7a3b17dcf75ull, 0x5c3dd19bd0ba1c1aull, 0x5bfdf7e546520f3eull, 0x5bbe4a6164eb92f4ull,
    0x5b7ec8f19468bbc9ull, 0x5b3f737751d915c8ull, 0x5b0049d42f6afbb6ull, 0x5ac14be9d45cf869ull,
    0x5a827999fcef3242ull, 0x5a43d2c67a54e0c0ull, 0x5a05575132a5cc20ull, 0x59c7071c20cfd70cull,
    0x5988e20954889245ull, 0x594ae7faf23eda52ull, 0x590d18d3330c7f1eull, 0x58cf747464a7f584ull,
    0x5891fac0e95612c8ull, 0x5854ab9b37dbd1e5ull, 0x581786e5db7022c2ull, 0x57da8c8373adc331ull,
    0x579dbc56b48521baull, 0x57611642662e4a33ull, 0x57249a29651adc07ull, 0x56e847eea1e80a49ull,
    0x56ac1f752150a563ull, 0x5670209ffc1f2e82ull, 0x56344b525f1ff495ull, 0x55f89f6f8b133af4ull,
    0x55bd1cdad49f699cull, 0x5581c377a44346f0ull, 0x5546932976483b15ull, 0x550b8bd3dab49cbdull,
    0x54d0ad5a753e077cull, 0x5495f7a0fd3bbb8eull, 0x545b6a8b3d990704ull, 0x542105fd14c7b869ull,
    0x53e6c9da74b29ab5ull, 0x53acb60762affaaeull, 0x5372ca67f774358full, 0x533906e05f045106ull,
    0x52ff6b54d8a89c75ull, 0x52c5f7a9b6df5b77ull, 0x528cabc35f4f799dull, 0x525387864abb4762ull,
    0x521a8ad704f3404full, 0x51e1b59a2cc8da3eull, 0x51a907b474015dc9ull, 0x5170810a9f48c7cfull,
    0x513821818624b40cull, 0x50ffe8fe12e750c4ull, 0x50c7d76542a25b72ull, 0x508fec9c251a267cull,
    0x50582887dcb8a7e1ull, 0x50208b0d9e8090dfull, 0x4fe91412b2006e83ull, 0x4fb1c37c7145d328ull,
    0x4f7a993048d088d7ull, 0x4f439513b785cc80ull, 0x4f0cb70c4ea39210ull, 0x4ed5feffb1b3d155ull,
    0x4e9f6cd3967fdba8ull, 0x4e69006dc503ba65ull, 0x4e32b9b417619617ull, 0x4dfc988c79d52661ull,
    0x4dc69cdceaa72a9cull, 0x4d90c68b7a20eb1eull, 0x4d5b157e4a7fc325ull, 0x4d25899b8fe8b365ull,
    0x4cf022c9905bfd32ull, 0x4cbae0eea3a8c63cull, 0x4c85c3f13360c4d5ull, 0x4c50cbb7bacbf4cbull,
    0x4c1bf828c6dc54b8ull, 0x4be7492af621abd6ull, 0x4bb2bea4f8bd5847ull, 0x4b7e587d905625d1ull,
    0x4b4a169b900c2d00ull, 0x4b15f8e5dc6cbab0ull, 0x4ae1ff436b663ff7ull, 0x4aae299b443c4a6bull,
    0x4a7a77d47f7b84b1ull, 0x4a46e9d646edbf6aull, 0x4a137f87d58e025bull, 0x49e038d0777ca5e0ull,
    0x49ad159789f37496ull, 0x497a15c47b39d53eull, 0x4947393eca98fcd6ull, 0x49147fee085028d6ull,
    0x48e1e9b9d588e19bull, 0x48af7689e44b44eaull, 0x487d2645f7725895ull, 0x484af8d5e2a06536ull,
    0x4818ee218a3358eeull, 0x47e70610e3393241ull, 0x47b5408bf36472e2ull, 0x47839d7ad1009a90ull,
    0x47521cc5a2e6a9e0ull, 0x4720be54a071ad01ull, 0x46ef821011734e6bull, 0x46be67e04e28717cull,
    0x468d6fadbf2dd4f3ull, 0x465c9960dd74bd4bull, 0x462be4e23237a6efull, 0x45fb521a56ef0042ull,
    0x45cae0f1f545eb73ull, 0x459a9151c70f0819ull, 0x456a632296394492ull, 0x453a564d3cc4b723ull,
    0x450a6abaa4b77ecdull, 0x44daa053c812abd2ull, 0x44aaf701b0c72feeull, 0x447b6ead78aad636ull,
    0x444c0740496d4294ull, 0x441cc0a35c8cf8eaull, 0x43ed9abffb4c6bc9ull, 0x43be957f7ea712b6ull,
    0x438fb0cb4f468808ull, 0x4360ec8ce577ae44ull, 0x433248adc91fdd02ull, 0x4303c51791b21550ull,
    0x42d561b3e6243d8aull, 0x42a71e6c7ce464afull, 0x4278fb2b1bce0d15ull, 0x424af7d9981f7e98ull,
    0x421d1461d66f2023ull, 0x41ef50adcaa0d899ull, 0x41c1aca777db771bull, 0x41942838f07e22a3ull,
    0x4166c34c5615d0ecull, 0x41397dcbd952c4a6ull, 0x410c57a1b9fe12f6ull, 0x40df50b846ef302bull,
    0x40b268f9de0183baull, 0x4085a050ec0a036aull, 0x4058f6a7ecccd5b6ull, 0x402c6be96af2fb58ull,
};
constexpr unsigned long long kExpB1 = 0xb17217f7d1cecbull;  // b1 2^64
constexpr unsigned long long kExpB2 = 0x3d7f7bfeefbull;     // b2 2^60
constexpr unsigned int kExpB3 = 0xe3583fe6u;                // b3 2^60
constexpr unsigned int kExpB4 = 0x275a6cu;                  // b4 2^60

// The CTA's copy of the table in shared memory (its 32 lanes read 32
// different entries; the constant cache would serialise them).  Called by
// every thread; visible after the next barrier.
template <int NT>
__device__ __forceinline__ void exp_table(unsigned long long* s_tab) {
  for (int i = threadIdx.x; i < 256; i += NT) s_tab[i] = kExp2Neg[i];
}

__device__ __forceinline__ double exp_fix(const Dev& d, unsigned long long R2,
                                          const unsigned long long* s_tab) {
  if (R2 > d.emax) return 0.0;  // underflows (cutoffs far beyond the kernel's width)
  const unsigned long long V = __umul64hi(R2 << d.eq, d.ec);
  const int m = (int)(V >> (64 - d.eib));
  const unsigned long long F = V << d.eib;
  const unsigned long long T = s_tab[F >> 56];
  const unsigned long long X = F << 8;
  const unsigned int xh = (unsigned int)(X >> 32);
  const unsigned int t3 = kExpB3 - __umulhi(xh, kExpB4);
  const unsigned long long t2 = kExpB2 - __umulhi(xh, t3);
  const unsigned long long t1 = kExpB1 - (__umul64hi(X, t2) << 4);
  const unsigned long long r = T - __umul64hi(T, __umul64hi(X, t1));
  const unsigned long long q = (r + 512) >> 10;  // 2^-F 2^53, rounded
  if (m <= 1021)
    return __longlong_as_double((long long)(((unsigned long long)(1021 - m) << 52) + q));
  return scalbn(__longlong_as_double((long long)((1021ULL << 52) + q)), -m);  // subnormal
}

template <int DIM>
struct Weight<false, DIM> {
  using T = double;
  static __device__ __forceinline__ double eval(const Dev& d, long long dx, long long dy) {
    const double sx = __dmul_rn((double)dx, d.scale);
    double s2 = __dmul_rn(sx, sx);
    if (DIM == 2) {
      const double sy = __dmul_rn((double)dy, d.scale);
      s2 = __dadd_rn(s2, __dmul_rn(sy, sy));
    }
    return exp_neg(__dmul_rn(s2, d.inv8));
  }
  // within the cutoff, |D| <= Smax < 2^30 per axis (s_tab: exp_table)
  static __device__ __forceinline__ double near(const Dev& d, long long D,
                                                const unsigned long long* s_tab) {
    const int D32 = (int)D;
    return exp_fix(d, (unsigned long long)((long long)D32 * D32), s_tab);
  }
  static __device__ __forceinline__ double near2(const Dev& d, long long dx, long long dy,
                                                 const unsigned long long* s_tab) {
    const int x32 = (int)dx, y32 = (int)dy;
    return exp_fix(d, (unsigned long long)((long long)x32 * x32 + (long long)y32 * y32), s_tab);
  }
};

template <int DIM>
struct Weight<true, DIM> {
  using T = float;
  static __device__ __forceinline__ float eval(const Dev& d, long long dx, long long dy) {
    const float fx = ll_to_float(dx);
    float s2 = __fmul_rn(fx, fx);
    if (DIM == 2) {
      const float fy = ll_to_float(dy);
      s2 = __fadd_rn(s2, __fmul_rn(fy, fy));
    }
    return __expf(-__fmul_rn(s2, d.inv8f));
  }
  // within the cutoff, |D| <= Smax < 2^30 per axis (the same values as
  // eval; no table)
  static __device__ __forceinline__ float near(const Dev& d, long long D,
                                               const unsigned long long*) {
    const float f = __int2float_rn((int)D);
    return __expf(-__fmul_rn(__fmul_rn(f, f), d.inv8f));
  }
  static __device__ __forceinline__ float near2(const Dev& d, long long dx, long long dy,
                                                const unsigned long long*) {
    const float fx = __int2float_rn((int)dx), fy = __int2float_rn((int)dy);
    return __expf(-__fmul_rn(__fadd_rn(__fmul_rn(fx, fx), __fmul_rn(fy, fy)), d.inv8f));
  }
};

// Binary32 weights, normalised weights and 1 / r_i: both mixed precisions.
constexpr bool mixw(int precision) { return precision != MT_FP64; }
constexpr int exp_tab_words(int precision) { return mixw(precision) ? 1 : 256; }

// ------------------------------------------------------------ mass access --

template <int PR>
struct Mass;

// Per-particle accumulation of sum_j P_ij (M_j - M_i): binary64 in MT_FP64
// and MT_MIXED; in MT_MIXED_DF32 the binary32 terms are summed by cascaded
// compensated summation (Ogita, Rump & Oishi's Sum2): each addition's exact rounding error, from
// Knuth's two-sum, is added into a second sum, and the pair (s, c) is used
// unrounded.  The flux P_ij (M_j - M_i) is bitwise antisymmetric between i
// and j, so the transfer conserves mass to the pair's precision.
struct kahan {
  float s, c;
};
template <>
struct Mass<MT_FP64> {
  using V = double;
  using Acc = double;
  // the product and the accumulation as one fused multiply-add
  static __device__ __forceinline__ void acc(double& a, double P, double d) {
    a = __fma_rn(P, d, a);
  }
  static __device__ __forceinline__ double load(const unsigned long long* M, long long i) {
    return f64_load(M, i);
  }
  static __device__ __forceinline__ void store(unsigned long long* M, long long i, double v) {
    f64_store(M, i, v);
  }
  static __device__ __forceinline__ double diff(double a, double b) { return a - b; }
  // M + dM/2 (Eq. 7 with the 1/2 of Eq. 4), then the reaction.
  static __device__ __forceinline__ void update(double& A, double& B, double dA, double dB,
                                                int react) {
    A = __fma_rn(0.5, dA, A);  // 0.5 dA is exact: the same as A + 0.5 dA
    B = __fma_rn(0.5, dB, B);
    if (react) Mass::react(A, B);
  }
  // min(A, B) off both: the smaller becomes exactly 0.  Finite masses of no
  // sign compare by their bits, and a zero is not subtracted (after a
  // particle's first reaction one of its masses often is): the binary64 pipe
  // sees one subtraction, or nothing.
  static __device__ __forceinline__ void react(double& A, double& B) {
    const unsigned long long a = (unsigned long long)__double_as_longlong(A);
    const unsigned long long b = (unsigned long long)__double_as_longlong(B);
    if ((a | b) < 0x7ff0000000000000ULL) {
      const bool less = a < b;
      double rest = less ? B : A;
      if ((less ? a : b) != 0) rest = rest - (less ? A : B);
      A = less ? 0.0 : rest;
      B = less ? rest : 0.0;
    } else if (A < B) {
      B = B - A;
      A = 0.0;
    } else {
      A = A - B;
      B = 0.0;
    }
  }
  static __device__ __forceinline__ double to_double(double v) { return v; }
};

// MT_MIXED: the normalised weight P is binary32; the masses, the
// difference M_j - M_i, the flux term P (M_j - M_i) (P widened exactly), its
// sum, the update and the reaction are binary64.
template <>
struct Mass<MT_MIXED> {
  using V = double;
  using Acc = double;
  static __device__ __forceinline__ void acc(double& a, float P, double d) {
    a = __fma_rn(widen_exact(P), d, a);
  }
  static __device__ __forceinline__ double load(const unsigned long long* M, long long i) {
    return f64_load(M, i);
  }
  static __device__ __forceinline__ void store(unsigned long long* M, long long i, double v) {
    f64_store(M, i, v);
  }
  static __device__ __forceinline__ double diff(double a, double b) { return a - b; }
  static __device__ __forceinline__ void update(double& A, double& B, double dA, double dB,
                                                int react) {
    // the reaction as in MT_FP64, compared in binary64: the one-kernel step
    // is bound by its integer instructions in this precision (N = 10^6: 3 us
    // less per step than by the bits)
    Mass<MT_FP64>::update(A, B, dA, dB, 0);
    if (react) {
      if (A < B) {
        B = B - A;
        A = 0.0;
      } else {
        A = A - B;
        B = 0.0;
      }
    }
  }
  static __device__ __forceinline__ void react(double& A, double& B) {
    Mass<MT_FP64>::react(A, B);
  }
  static __device__ __forceinline__ double to_double(double v) { return v; }
};

// MT_MIXED_DF32: masses as unevaluated sums of two binary32 numbers, flux
// terms in binary32 summed with compensation, compensated update and
// reaction (binary32 arithmetic only).
template <>
struct Mass<MT_MIXED_DF32> {
  using V = df;
  using Acc = kahan;
  static __device__ __forceinline__ void acc(kahan& a, float P, float d) {
    const df e = two_sum(a.s, __fmul_rn(P, d));
    a.s = e.hi;
    a.c = __fadd_rn(a.c, e.lo);
  }
  static __device__ __forceinline__ df load(const unsigned long long* M, long long i) {
    return df_load(M, i);
  }
  static __device__ __forceinline__ void store(unsigned long long* M, long long i, df v) {
    df_store(M, i, v);
  }
  static __device__ __forceinline__ float diff(df a, df b) {
    return __fadd_rn(__fsub_rn(a.hi, b.hi), __fsub_rn(a.lo, b.lo));
  }
  static __device__ __forceinline__ void update(df& A, df& B, kahan dA, kahan dB, int react) {
    A = df_add(A, {0.5f * dA.s, 0.5f * dA.c});
    B = df_add(B, {0.5f * dB.s, 0.5f * dB.c});
    if (react) Mass::react(A, B);
  }
  static __device__ __forceinline__ void react(df& A, df& B) {
    if (df_le(A, B)) {
      B = df_sub(B, A);
      A = {0.0f, 0.0f};
    } else {
      A = df_sub(A, B);
      B = {0.0f, 0.0f};
    }
  }
  static __device__ __forceinline__ double to_double(df v) { return (double)v.hi + (double)v.lo; }
};

// The two mass arrays one exchange pass works on (word offsets into a mass
// buffer of nspec * n words): A and B, or the extra species sp and sp + 1;
// when sp is the last species the second array repeats it and is not
// stored.
struct SpeciesPair {
  long long oa, ob;
  bool store_b;
};
template <bool TR>
__device__ __forceinline__ SpeciesPair species_pair(const Dev& d, int sp) {
  if (!TR) return {0, d.n, true};
  const bool two = sp + 1 < d.nspec;
  return {(long long)sp * d.n, (long long)(two ? sp + 1 : sp) * d.n, two};
}

// Row sum r_i over a dense neighbourhood (hundreds to thousands of terms):
// binary64, or with binary32 weights a binary32 sum with each addition's rounding error
// (Knuth's two-sum) collected in a second term, so the sum keeps about twice
// binary32's precision however many weights it adds.
template <bool MIX>
struct RowSum;
template <>
struct RowSum<false> {
  double r;
  __device__ __forceinline__ explicit RowSum(double v) : r(v) {}
  __device__ __forceinline__ void add(double w) { r += w; }
  __device__ __forceinline__ double value() const { return r; }
};
template <>
struct RowSum<true> {
  float s, c;
  __device__ __forceinline__ explicit RowSum(float v) : s(v), c(0.0f) {}
  __device__ __forceinline__ void add(float w) {
    const df e = two_sum(s, w);
    s = e.hi;
    c = __fadd_rn(c, e.lo);
  }
  __device__ __forceinline__ float value() const { return __fadd_rn(s, c); }
};

template <bool MIX>
__device__ __forceinline__ void store_rinv(const Dev& d, long long p, typename Weight<MIX, 1>::T r) {
  if (MIX)
    static_cast<float*>(d.rinv)[p] = __frcp_rn((float)r);
  else
    static_cast<double*>(d.rinv)[p] = rcp_ge1((double)r);
}

template <bool MIX>
__device__ __forceinline__ typename Weight<MIX, 1>::T load_rinv(const Dev& d, long long p) {
  if (MIX)
    return static_cast<const float*>(d.rinv)[p];
  else
    return static_cast<const double*>(d.rinv)[p];
}

// Normalised weight of the ordered pair (p, q) (Sec. 1.1): ROW w / r_p, or
// SYM (w / r_p + w / r_q) / 2.
template <typename T>
__device__ __forceinline__ T normalised(int norm, T w, T ip, T iq) {
  return norm == MT_NORM_ROW ? w * ip : T(0.5) * w * (ip + iq);
}

// Combining per-lane partial sums in a fixed shuffle tree (warp-cooperative
// sums over a dense neighbourhood): row sums in T, flux accumulators in Acc.
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = __fadd_rn(v, __shfl_down_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double acc_warp_sum(double v) { return warp_sum(v); }
__device__ __forceinline__ double acc_merge(double a, double b) { return a + b; }
__device__ __forceinline__ kahan acc_merge(kahan a, kahan b) {
  const df e = two_sum(a.s, b.s);
  return {e.hi, __fadd_rn(__fadd_rn(a.c, b.c), e.lo)};
}
__device__ __forceinline__ double acc_shfl_xor(double v, int o) {
  return __shfl_xor_sync(0xffffffffu, v, o);
}
__device__ __forceinline__ kahan acc_shfl_xor(kahan v, int o) {
  return {__shfl_xor_sync(0xffffffffu, v.s, o), __shfl_xor_sync(0xffffffffu, v.c, o)};
}
__device__ __forceinline__ kahan acc_warp_sum(kahan v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float s2 = __shfl_down_sync(0xffffffffu, v.s, o);
    const float c2 = __shfl_down_sync(0xffffffffu, v.c, o);
    const df e = two_sum(v.s, s2);
    v.s = e.hi;
    v.c = __fadd_rn(__fadd_rn(v.c, c2), e.lo);
  }
  return v;
}

// Observables arithmetic: sums in the precision's own format (binary64 or
// double-binary32), converted to binary64 per CTA.
__device__ __forceinline__ double obs_add(double a, double b) { return a + b; }
__device__ __forceinline__ df obs_add(df a, df b) { return df_add(a, b); }
__device__ __forceinline__ double obs_shfl(double v, int o) {
  return __shfl_down_sync(0xffffffffu, v, o);
}
__device__ __forceinline__ df obs_shfl(df v, int o) {
  return {__shfl_down_sync(0xffffffffu, v.hi, o), __shfl_down_sync(0xffffffffu, v.lo, o)};
}
__device__ __forceinline__ double obs_double(double v) { return v; }
__device__ __forceinline__ double obs_double(df v) { return (double)v.hi + (double)v.lo; }
__device__ __forceinline__ double obs_diff(double a, double b) { return a - b; }
__device__ __forceinline__ df obs_diff(df a, df b) { return df_sub(a, b); }

// Fixed-order reductions of the observables sums (three values).
template <typename MV>
struct Obs3 {
  MV a, b, d;
};
template <typename MV>
__device__ __forceinline__ Obs3<MV> obs3_add(Obs3<MV> x, Obs3<MV> y) {
  return {obs_add(x.a, y.a), obs_add(x.b, y.b), obs_add(x.d, y.d)};
}
template <typename MV>
__device__ __forceinline__ Obs3<MV> obs3_warp(Obs3<MV> v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = obs3_add(v, Obs3<MV>{obs_shfl(v.a, o), obs_shfl(v.b, o), obs_shfl(v.d, o)});
  return v;
}
// Block-wide (NT threads): warp trees, then warp 0 over the warp totals;
// the result is valid in thread 0.  Called by every thread.
template <typename MV, int NT>
__device__ __forceinline__ Obs3<MV> obs3_block(Obs3<MV> v, Obs3<MV>* s_w) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  v = obs3_warp(v);
  if (lane == 0) s_w[warp] = v;
  __syncthreads();
  Obs3<MV> t{};
  if (warp == 0) {
    if (lane < NT / 32) t = s_w[lane];
    t = obs3_warp(t);
  }
  __syncthreads();
  return t;
}

__device__ __forceinline__ double ldcg_obs(const double* p) { return __ldcg(p); }
__device__ __forceinline__ df ldcg_obs(const df* p) {
  const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
  return {v.x, v.y};
}

template <typename MV>
__device__ __forceinline__ void obs_row(const Dev& d, long long row, int r, long long n,
                                        Obs3<MV> t) {
  double* o = d.obs + 4 * (row * d.nreal + r);
  const double a = obs_double(t.a);
  o[0] = a;
  o[1] = obs_double(t.b);
  o[2] = obs_double(t.d);
  o[3] = a / (double)n;
}

// The last CTA of a step's final pass advances the step counter and flips
// the buffer selectors.  Called by every thread.
__device__ __forceinline__ void finish_step(const Dev& d, int flip_x, int flip_m) {
  __shared__ bool s_last;
  Ctrl* c = d.ctrl;
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(&c->done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last || threadIdx.x != 0) return;
  __threadfence();
  c->step += 1;
  c->xcur ^= flip_x;
  c->mcur ^= flip_m;
  c->done = 0;
}

}  // namespace mt
