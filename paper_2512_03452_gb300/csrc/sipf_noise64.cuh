// Double-precision Box-Muller pieces from the 32-bit words of the generator:
// ln((w + 1/2) 2^-32) and the sine and cosine of 2 pi (w + 1/2) 2^-32.  The
// uniforms are known as integers, so no general range reduction is needed, and
// on the FP64 pipe (about one warp instruction per 19 clocks and SM, the bound
// of the FP64 form) they take some 12 and 20 instructions where the general
// log and sincos take about 30 and 45.
//   ln: u = m 2^e with m in [3/4, 3/2), a table of 128 pairs (c, -ln c) with c
//       near 1 / m (c = 1 next to m = 1, so that values near 0 keep their
//       relative precision), r = m c - 1, |r| < 2^-7, and the series of ln(1 + r);
//   sine and cosine: the nearest quarter turn taken off in integers, then the
//       Taylor series to theta^15 and theta^16 on |theta| <= pi / 4 (the next
//       terms are below 7e-17).
// Errors against long double over 2e7 words, in units of 2^-52 (rms, max):
// ln, relative, 0.26, 1.34 (general log 0.21, 0.50); sine and cosine, absolute,
// 0.25, 0.88 (general sine and cosine of the rounded angle 0.92, 3.11), so a
// normal is three times closer than with the general functions.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

namespace sipf {

#ifdef __CUDA_ARCH__
#define SIPF_LOG_TABLE static __device__ const double2
#else
#define SIPF_LOG_TABLE static const double2
#endif
// (c_i, -ln c_i): c_i the double nearest 1 / m at the middle of interval i of
// the leading seven fraction bits of the normalised u in [1, 2) (m is half of it
// for i >= 64), 1 for the intervals next to m = 1.
SIPF_LOG_TABLE kLogTable[128] = {
  {0x1.0000000000000p+0, 0x0.0p+0}, {0x1.fa11caa01fa12p-1, 0x1.7dc475f810a69p-7},
  {0x1.f6310aca0dbb5p-1, 0x1.3cea44346a584p-6}, {0x1.f25f644230ab5p-1, 0x1.b9fc027af919ap-6},
  {0x1.ee9c7f8458e02p-1, 0x1.1b0d98923d97fp-5}, {0x1.eae807aba01ebp-1, 0x1.58a5bafc8e4d3p-5},
  {0x1.e741aa59750e4p-1, 0x1.95c830ec8e3f2p-5}, {0x1.e3a9179dc1a73p-1, 0x1.d276b8adb0b56p-5},
  {0x1.e01e01e01e01ep-1, 0x1.075983598e471p-4}, {0x1.dca01dca01dcap-1, 0x1.253f62f0a1417p-4},
  {0x1.d92f2231e7f8ap-1, 0x1.42edcbea646eep-4}, {0x1.d5cac807572b2p-1, 0x1.60658a93750c4p-4},
  {0x1.d272ca3fc5b1ap-1, 0x1.7da766d7b12d0p-4}, {0x1.cf26e5c44bfc6p-1, 0x1.9ab42462033aep-4},
  {0x1.cbe6d9601cbe7p-1, 0x1.b78c82bb0eda0p-4}, {0x1.c8b265afb8a42p-1, 0x1.d4313d66cb35dp-4},
  {0x1.c5894d10d4986p-1, 0x1.f0a30c01162a4p-4}, {0x1.c26b5392ea01cp-1, 0x1.0671512ca596fp-3},
  {0x1.bf583ee868d8bp-1, 0x1.14785846742acp-3}, {0x1.bc4fd65883e7bp-1, 0x1.2266f190a5acdp-3},
  {0x1.b951e2b18ff23p-1, 0x1.303d718e47fd5p-3}, {0x1.b65e2e3beee05p-1, 0x1.3dfc2b0ecc62ap-3},
  {0x1.b37484ad806cep-1, 0x1.4ba36f39a55e5p-3}, {0x1.b094b31d922a4p-1, 0x1.59338d9982085p-3},
  {0x1.adbe87f94905ep-1, 0x1.66acd4272ad51p-3}, {0x1.aaf1d2f87ebfdp-1, 0x1.740f8f54037a3p-3},
  {0x1.a82e65130e159p-1, 0x1.815c0a14357e9p-3}, {0x1.a574107688a4ap-1, 0x1.8e928de886d41p-3},
  {0x1.a2c2a87c51ca0p-1, 0x1.9bb362e7dfb85p-3}, {0x1.a01a01a01a01ap-1, 0x1.a8becfc882f19p-3},
  {0x1.9d79f176b682dp-1, 0x1.b5b519e8fb5a6p-3}, {0x1.9ae24ea5510dap-1, 0x1.c2968558c18c2p-3},
  {0x1.9852f0d8ec0ffp-1, 0x1.cf6354e09c5ddp-3}, {0x1.95cbb0be377aep-1, 0x1.dc1bca0abec7bp-3},
  {0x1.934c67f9b2ce6p-1, 0x1.e8c0252aa5a60p-3}, {0x1.90d4f120190d5p-1, 0x1.f550a564b7b37p-3},
  {0x1.8e6527af1373fp-1, 0x1.00e6c45ad501dp-2}, {0x1.8bfce8062ff3ap-1, 0x1.071b85fcd590dp-2},
  {0x1.899c0f601899cp-1, 0x1.0d46b579ab74bp-2}, {0x1.87427bcc092b9p-1, 0x1.136870293a8b0p-2},
  {0x1.84f00c2780614p-1, 0x1.1980d2dd4236fp-2}, {0x1.82a4a0182a4a0p-1, 0x1.1f8ff9e48a2f3p-2},
  {0x1.8060180601806p-1, 0x1.2596010df763ap-2}, {0x1.7e225515a4f1dp-1, 0x1.2b9303ab89d25p-2},
  {0x1.7beb3922e017cp-1, 0x1.31871c9544185p-2}, {0x1.79baa6bb6398bp-1, 0x1.3772662bfd85cp-2},
  {0x1.77908119ac60dp-1, 0x1.3d54fa5c1f710p-2}, {0x1.756cac201756dp-1, 0x1.432ef2a04e813p-2},
  {0x1.734f0c541fe8dp-1, 0x1.49006804009d0p-2}, {0x1.713786d9c7c09p-1, 0x1.4ec9732600269p-2},
  {0x1.6f26016f26017p-1, 0x1.548a2c3add263p-2}, {0x1.6d1a62681c861p-1, 0x1.5a42ab0f4cfe2p-2},
  {0x1.6b1490aa31a3dp-1, 0x1.5ff3070a793d4p-2}, {0x1.691473a88d0c0p-1, 0x1.659b57303e1f2p-2},
  {0x1.6719f3601671ap-1, 0x1.6b3bb2235943dp-2}, {0x1.6524f853b4aa3p-1, 0x1.70d42e2789236p-2},
  {0x1.63356b88ac0dep-1, 0x1.7664e1239dbcfp-2}, {0x1.614b36831ae94p-1, 0x1.7bede0a37afbfp-2},
  {0x1.5f66434292dfcp-1, 0x1.816f41da0d495p-2}, {0x1.5d867c3ece2a5p-1, 0x1.86e919a330ba1p-2},
  {0x1.5babcc647fa91p-1, 0x1.8c5b7c858b48bp-2}, {0x1.59d61f123ccaap-1, 0x1.91c67eb45a83ep-2},
  {0x1.5805601580560p-1, 0x1.972a341135159p-2}, {0x1.56397ba7c52e2p-1, 0x1.9c86b02dc0862p-2},
  {0x1.54725e6bb82fep+0, -0x1.23ec5991eba49p-2}, {0x1.52aff56a8054bp+0, -0x1.1e9e1678899f5p-2},
  {0x1.50f22e111c4c5p+0, -0x1.1956d3b9bc2f9p-2}, {0x1.4f38f62dd4c9bp+0, -0x1.14167ef367784p-2},
  {0x1.4d843bedc2c4cp+0, -0x1.0edd060b78082p-2}, {0x1.4bd3edda68fe1p+0, -0x1.09aa572e6c6d4p-2},
  {0x1.4a27fad76014ap+0, -0x1.047e60cde83b7p-2}, {0x1.4880522014880p+0, -0x1.feb2233ea07cbp-3},
  {0x1.46dce34596066p+0, -0x1.f474b134df228p-3}, {0x1.453d9e2c776cap+0, -0x1.ea4449f04aaf5p-3},
  {0x1.43a2730abee4dp+0, -0x1.e020cc6235ab5p-3}, {0x1.420b5265e5951p+0, -0x1.d60a17f903514p-3},
  {0x1.40782d10e6566p+0, -0x1.cc000c9db3c52p-3}, {0x1.3ee8f42a5af07p+0, -0x1.c2028ab17f9b5p-3},
  {0x1.3d5d991aa75c6p+0, -0x1.b811730b823d4p-3}, {0x1.3bd60d9232955p+0, -0x1.ae2ca6f672bd8p-3},
  {0x1.3a524387ac822p+0, -0x1.a454082e6ab03p-3}, {0x1.38d22d366088ep+0, -0x1.9a8778debaa3ap-3},
  {0x1.3755bd1c945eep+0, -0x1.90c6db9fcbcdbp-3}, {0x1.35dce5f9f2af8p+0, -0x1.871213750e994p-3},
  {0x1.34679ace01346p+0, -0x1.7d6903caf5acdp-3}, {0x1.32f5ced6a1dfap+0, -0x1.73cb9074fd14dp-3},
  {0x1.3187758e9ebb6p+0, -0x1.6a399dabbd383p-3}, {0x1.301c82ac40260p+0, -0x1.60b3100b09474p-3},
  {0x1.2eb4ea1fed14bp+0, -0x1.5737cc9018cddp-3}, {0x1.2d50a012d50a0p+0, -0x1.4dc7b897bc1c7p-3},
  {0x1.2bef98e5a3711p+0, -0x1.4462b9dc9b3dcp-3}, {0x1.2a91c92f3c105p+0, -0x1.3b08b6757f2a7p-3},
  {0x1.293725bb804a5p+0, -0x1.31b994d3a4f86p-3}, {0x1.27dfa38a1ce4dp+0, -0x1.28753bc11aba2p-3},
  {0x1.268b37cd60127p+0, -0x1.1f3b925f25d44p-3}, {0x1.2539d7e9177b2p+0, -0x1.160c8024b27b0p-3},
  {0x1.23eb79717605bp+0, -0x1.0ce7ecdccc28bp-3}, {0x1.22a0122a0122ap+0, -0x1.03cdc0a51ec0dp-3},
  {0x1.21579804855e6p+0, -0x1.f57bc7d9005dbp-4}, {0x1.2012012012012p+0, -0x1.e3707ee30487bp-4},
  {0x1.1ecf43c7fb84cp+0, -0x1.d179788219362p-4}, {0x1.1d8f5672e4abdp+0, -0x1.bf968769fca18p-4},
  {0x1.1c522fc1ce059p+0, -0x1.adc77ee5aea8ep-4}, {0x1.1b17c67f2bae3p+0, -0x1.9c0c32d4d254dp-4},
  {0x1.19e0119e0119ep+0, -0x1.8a6477a91dc29p-4}, {0x1.18ab083902bdbp+0, -0x1.78d02263d82d7p-4},
  {0x1.1778a191bd684p+0, -0x1.674f089365a78p-4}, {0x1.1648d50fc3201p+0, -0x1.55e10050e0382p-4},
  {0x1.151b9a3fdd5c9p+0, -0x1.4485e03dbdfb0p-4}, {0x1.13f0e8d344724p+0, -0x1.333d7f8183f4ap-4},
  {0x1.12c8b89edc0acp+0, -0x1.2207b5c7854a1p-4}, {0x1.11a3019a74826p+0, -0x1.10e45b3cae829p-4},
  {0x1.107fbbe011080p+0, -0x1.ffa6911ab9309p-5}, {0x1.0f5edfab325a2p+0, -0x1.dda8adc67ee59p-5},
  {0x1.0e40655826011p+0, -0x1.bbcebfc68f424p-5}, {0x1.0d24456359e3ap+0, -0x1.9a187b573de81p-5},
  {0x1.0c0a7868b4171p+0, -0x1.788595a3577c8p-5}, {0x1.0af2f722eecb5p+0, -0x1.5715c4c03cee1p-5},
  {0x1.09ddba6af8360p+0, -0x1.35c8bfaa13069p-5}, {0x1.08cabb37565e2p+0, -0x1.149e3e4005a8dp-5},
  {0x1.07b9f29b8eae2p+0, -0x1.e72bf2813ce6ap-6}, {0x1.06ab59c7912fbp+0, -0x1.a55f548c5c427p-6},
  {0x1.059eea0727586p+0, -0x1.63d6178690bbep-6}, {0x1.04949cc1664c5p+0, -0x1.228fb1fea2e0ap-6},
  {0x1.038c6b78247fcp+0, -0x1.c317384c75f0dp-7}, {0x1.02864fc7729e9p+0, -0x1.41929f968330cp-7},
  {0x1.0182436517a37p+0, -0x1.8121214586b02p-8}, {0x1.0000000000000p+0, 0x0.0p+0},
};

__host__ __device__ __forceinline__ double bits_double(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double d;
  memcpy(&d, &b, 8);
  return d;
#endif
}

__host__ __device__ __forceinline__ double ln_uniform32(uint32_t w) {
  const uint64_t x = 2ull * w + 1ull;   // u = x 2^-33
#ifdef __CUDA_ARCH__
  const int s = __clzll((long long)x) - 11;
#else
  const int s = __builtin_clzll(x) - 11;
#endif
  const uint64_t f = (x << s) & 0x000FFFFFFFFFFFFFull;   // fraction of u normalised to [1, 2)
  const int i = (int)(f >> 45), up = i >= 64;
  const double m = bits_double(f | ((uint64_t)(0x3FF - up) << 52));
  const double e = (double)(52 - s - 33 + up);
#ifdef __CUDA_ARCH__
  const double2 t = __ldg(&kLogTable[i]);
#else
  const double2 t = kLogTable[i];
#endif
  const double r = fma(m, t.x, -1.0);
  double p = fma(r, 1.0 / 7.0, -1.0 / 6.0);
  p = fma(r, p, 1.0 / 5.0);
  p = fma(r, p, -1.0 / 4.0);
  p = fma(r, p, 1.0 / 3.0);
  p = fma(r, p, -0.5);
  p = fma(r * r, p, r);                                       // ln(1 + r)
  const double ln2_hi = 0x1.62e42fefap-1, ln2_lo = 0x1.cf79abc9e3b3ap-40;   // ln 2 to 36 bits and the rest
  return fma(e, ln2_hi, t.y + fma(e, ln2_lo, p));
}

__host__ __device__ __forceinline__ void sincos_turn32(uint32_t w, double* sn, double* cs) {
  const uint32_t k = (w + 0x20000000u) >> 30;               // nearest quarter turn
  const int32_t f = (int32_t)(w - (k << 30));               // in [-2^29, 2^29)
  // f + 1/2 exactly, through the bits of 2^51 + 2^32 + f + 1/2
  const double d = bits_double(0x4320000000000000ull + (uint64_t)((2ll * f + 1ll) + (1ll << 33))) -
                   (2251799813685248.0 + 4294967296.0);
  const double th = d * 1.4629180792671596e-09;             // 2 pi 2^-32
  const double z = th * th;
  double s = fma(z, -1.0 / 1307674368000.0, 1.0 / 6227020800.0);
  s = fma(z, s, -1.0 / 39916800.0);
  s = fma(z, s, 1.0 / 362880.0);
  s = fma(z, s, -1.0 / 5040.0);
  s = fma(z, s, 1.0 / 120.0);
  s = fma(z, s, -1.0 / 6.0);
  s = fma(th * z, s, th);
  double c = fma(z, 1.0 / 20922789888000.0, -1.0 / 87178291200.0);
  c = fma(z, c, 1.0 / 479001600.0);
  c = fma(z, c, -1.0 / 3628800.0);
  c = fma(z, c, 1.0 / 40320.0);
  c = fma(z, c, -1.0 / 720.0);
  c = fma(z, c, 1.0 / 24.0);
  c = fma(z * z, c, fma(z, -0.5, 1.0));
  const double a = (k & 1u) ? c : s, b = (k & 1u) ? s : c;
  *sn = (k & 2u) ? -a : a;
  *cs = ((k + 1u) & 2u) ? -b : b;
}

}  // namespace sipf
