// fixexp.h -- exp and reciprocal of a double in 64-bit integer arithmetic.
//
// GB300's FP64 pipe takes two lanes a clock on an SM, its integer pipe 64: a
// membrane evaluation of about 50 exponentials spends most of a quarter of its
// FP64 instructions inside exp().  This one takes none of them.  The method
// is Tang's table-driven exponential (P. T. P. Tang, ACM Trans. Math. Softw.
// 15, 1989) in fixed point:
//   |x| as a fixed-point number with 57 fraction bits, t = |x| log2(e) as a
//   128-bit product, k + j/256 + u/256 = +-t with integers k, 0 <= j < 256 and
//   0 <= u < 1, exp(x) = 2^k 2^(j/256) 2^(u/256), the table 2^(j/256) with 63
//   fraction bits and 2^(u/256) - 1 by the exponential series to degree 5 in
//   u (remainder below 2^-60).
// The result is rounded once: at most 0.56 units in the last place over the
// fast range (tests/test_exp_cpu.py, against long double; the library's exp is
// specified to 1).  |x| >= 64, infinities and NaN take the library's exp.
// Measured on GB300, FP64 steps with the library's / this exp: TP06 257^2 9.53 /
// 7.77 ms, LR91 65^2 2.02 / 1.84 ms.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define BD_FIX_FN __host__ __device__ __forceinline__
#else
#define BD_FIX_FN inline
#endif

namespace bd {

#define BD_EXP2_TABLE \
    0x8000000000000000ull, 0x8058d7d2d5e5f6b1ull, 0x80b1ed4fd999ab6cull, 0x810b40a1d81406d4ull, \
    0x8164d1f3bc030773ull, 0x81bea1708dde6056ull, 0x8218af4373fc25ecull, 0x8272fb97b2a5894cull, \
    0x82cd8698ac2ba1d7ull, 0x83285071e0fc4547ull, 0x8383594eefb6ee37ull, 0x83dea15b9541b132ull, \
    0x843a28c3acde4046ull, 0x8495efb3303efd30ull, 0x84f1f656379c1a29ull, 0x854e3cd8f9c8c95dull, \
    0x85aac367cc487b15ull, 0x86078a2f23642a9full, 0x8664915b923fba04ull, 0x86c1d919caef5c88ull, \
    0x871f61969e8d1010ull, 0x877d2afefd4e256cull, 0x87db357ff698d792ull, 0x88398146b919f1d4ull, \
    0x88980e8092da8527ull, 0x88f6dd5af155ac6bull, 0x8955ee03618e5fddull, 0x89b540a7902557a4ull, \
    0x8a14d575496efd9aull, 0x8a74ac9a79896e47ull, 0x8ad4c6452c728924ull, 0x8b3522a38e1e1032ull, \
    0x8b95c1e3ea8bd6e7ull, 0x8bf6a434adde0085ull, 0x8c57c9c4646f4ddeull, 0x8cb932c1bae97a95ull, \
    0x8d1adf5b7e5ba9e6ull, 0x8d7ccfc09c50e2f8ull, 0x8ddf042022e69cd6ull, 0x8e417ca940e35a01ull, \
    0x8ea4398b45cd53c0ull, 0x8f073af5a2013520ull, 0x8f6a8117e6c8e5c4ull, 0x8fce0c21c6726481ull, \
    0x9031dc431466b1dcull, 0x9095f1abc540ca6bull, 0x90fa4c8beee4b12bull, 0x915eed13c89689d3ull, \
    0x91c3d373ab11c336ull, 0x9228ffdc10a051adull, 0x928e727d9531f9acull, 0x92f42b88f673aa7cull, \
    0x935a2b2f13e6e92cull, 0x93c071a0eef94bc1ull, 0x9426ff0fab1c04b6ull, 0x948dd3ac8ddb7ed3ull, \
    0x94f4efa8fef70961ull, 0x955c5336887894d5ull, 0x95c3fe86d6cc7fefull, 0x962bf1cbb8d97560ull, \
    0x96942d3720185a00ull, 0x96fcb0fb20ac4ba3ull, 0x97657d49f17ab08eull, 0x97ce9255ec4357abull, \
    0x9837f0518db8a96full, 0x98a1976f7597e996ull, 0x990b87e266c189aaull, 0x9975c1dd47518c77ull, \
    0x99e0459320b7fa65ull, 0x9a4b13371fd166caull, 0x9ab62afc94ff864aull, 0x9b218d16f441d63dull, \
    0x9b8d39b9d54e5539ull, 0x9bf93118f3aa4cc1ull, 0x9c6573682ec32c2dull, 0x9cd200db8a0774cbull, \
    0x9d3ed9a72cffb751ull, 0x9dabfdff6367a2aaull, 0x9e196e189d472420ull, 0x9e872a276f0b98ffull, \
    0x9ef5326091a111aeull, 0x9f6386f8e28ba651ull, 0x9fd228256400dd06ull, 0xa041161b3d0121beull, \
    0xa0b0510fb9714fc2ull, 0xa11fd9384a344cf7ull, 0xa18faeca8544b6e4ull, 0xa1ffd1fc25cea188ull, \
    0xa27043030c496819ull, 0xa2e102153e918f9eull, 0xa3520f68e802bb93ull, 0xa3c36b345991b47cull, \
    0xa43515ae09e6809eull, 0xa4a70f0c95768ec5ull, 0xa5195786be9ef339ull, 0xa58bef536dbeb6eeull, \
    0xa5fed6a9b15138eaull, 0xa6720dc0be08a20cull, 0xa6e594cfeee86b1eull, 0xa7596c0ec55ff55bull, \
    0xa7cd93b4e965356aull, 0xa8420bfa298f70d1ull, 0xa8b6d5167b320e09ull, 0xa92bef41fa77771bull, \
    0xa9a15ab4ea7c0ef8ull, 0xaa1717a7b5693979ull, 0xaa8d2652ec907629ull, 0xab0386ef48868de1ull, \
    0xab7a39b5a93ed337ull, 0xabf13edf162675e9ull, 0xac6896a4be3fe929ull, 0xace0413ff83e5d04ull, \
    0xad583eea42a14ac6ull, 0xadd08fdd43d01491ull, 0xae493452ca35b80eull, 0xaec22c84cc5c9465ull, \
    0xaf3b78ad690a4375ull, 0xafb51906e75b8661ull, 0xb02f0dcbb6e04584ull, 0xb0a957366fb7a3c9ull, \
    0xb123f581d2ac2590ull, 0xb19ee8e8c94feb09ull, 0xb21a31a66618fe3bull, 0xb295cff5e47db4a4ull, \
    0xb311c412a9112489ull, 0xb38e0e38419fae18ull, 0xb40aaea2654b9841ull, 0xb487a58cf4a9c180ull, \
    0xb504f333f9de6484ull, 0xb58297d3a8b9f0d2ull, 0xb60093a85ed5f76cull, 0xb67ee6eea3b22b8full, \
    0xb6fd91e328d17791ull, 0xb77c94c2c9d725e9ull, 0xb7fbefca8ca41e7cull, 0xb87ba337a1743834ull, \
    0xb8fbaf4762fb9ee9ull, 0xb97c143756844dbfull, 0xb9fcd2452c0b9debull, 0xba7de9aebe5fea09ull, \
    0xbaff5ab2133e45fbull, 0xbb81258d5b704b6full, 0xbc034a7ef2e9fb0dull, 0xbc85c9c560e7b269ull, \
    0xbd08a39f580c36bfull, 0xbd8bd84bb67ed483ull, 0xbe0f6809860993e2ull, 0xbe935317fc378238ull, \
    0xbf1799b67a731083ull, 0xbf9c3c248e2486f8ull, 0xc0213aa1f0d08db0ull, 0xc0a6956e8836ca8dull, \
    0xc12c4cca66709456ull, 0xc1b260f5ca0fbb33ull, 0xc238d2311e3d6673ull, 0xc2bfa0bcfad907c9ull, \
    0xc346ccda24976407ull, 0xc3ce56c98d21b15dull, 0xc4563ecc5334cb33ull, 0xc4de8523c2c07baaull, \
    0xc5672a115506daddull, 0xc5f02dd6b0bbc3d9ull, 0xc67990b5aa245f79ull, 0xc70352f04336c51eull, \
    0xc78d74c8abb9b15dull, 0xc817f681416452b2ull, 0xc8a2d85c8ffe2c45ull, 0xc92e1a9d517f0eccull, \
    0xc9b9bd866e2f27a3ull, 0xca45c15afcc72624ull, 0xcad2265e4290774eull, 0xcb5eecd3b38597c9ull, \
    0xcbec14fef2727c5dull, 0xcc799f23d11510e5ull, 0xcd078b86503dcdd2ull, 0xcd95da6a9ff06445ull, \
    0xce248c151f8480e4ull, 0xceb3a0ca5dc6a55dull, 0xcf4318cf191918c1ull, 0xcfd2f4683f94eeb5ull, \
    0xd06333daef2b2595ull, 0xd0f3d76c75c5db8dull, 0xd184df6251699ac6ull, 0xd2164c023056bcabull, \
    0xd2a81d91f12ae45aull, 0xd33a5457a3029054ull, 0xd3ccf099859ac379ull, 0xd45ff29e0972c561ull, \
    0xd4f35aabcfedfa1full, 0xd5872909ab75d18aull, 0xd61b5dfe9f9bce07ull, 0xd6aff9d1e13ba2feull, \
    0xd744fccad69d6af4ull, 0xd7da67311797f56aull, 0xd870394c6db32c84ull, 0xd9067364d44a929cull, \
    0xd99d15c278afd7b6ull, 0xda3420adba4d8704ull, 0xdacb946f2ac9cc72ull, 0xdb63714f8e295255ull, \
    0xdbfbb797daf23755ull, 0xdc9467913a4f1c92ull, 0xdd2d818508324c20ull, 0xddc705bcd378f7f0ull, \
    0xde60f4825e0e9124ull, 0xdefb4e1f9d1037f2ull, 0xdf9612deb8f04420ull, 0xe031430a0d99e627ull, \
    0xe0ccdeec2a94e111ull, 0xe168e6cfd3295d23ull, 0xe2055afffe83d369ull, 0xe2a23bc7d7d91226ull, \
    0xe33f8972be8a5a51ull, 0xe3dd444c46499619ull, 0xe47b6ca0373da88dull, 0xe51a02ba8e26d681ull, \
    0xe5b906e77c8348a8ull, 0xe658797368b3a717ull, 0xe6f85aaaee1fce22ull, 0xe798aadadd5b9cbfull, \
    0xe8396a503c4bdc68ull, 0xe8da9958464b42abull, 0xe97c38406c4f8c57ull, 0xea1e4756550eb27bull, \
    0xeac0c6e7dd24392full, 0xeb63b74317369840ull, 0xec0718b64c1cbddcull, 0xecaaeb8ffb03ab41ull, \
    0xed4f301ed9942b84ull, 0xedf3e6b1d418a491ull, 0xee990f980da3025bull, 0xef3eab20e032bc6bull, \
    0xefe4b99bdcdaf5cbull, 0xf08b3b58cbe8b76aull, 0xf13230a7ad094509ull, 0xf1d999d8b7708cc1ull, \
    0xf281773c59ffb13aull, 0xf329c9233b6bae9cull, 0xf3d28fde3a641a5bull, 0xf47bcbbe6db9fddfull, \
    0xf5257d152486cc2cull, 0xf5cfa433e6537290ull, 0xf67a416c733f846eull, 0xf7255510c4288239ull, \
    0xf7d0df730ad13bb9ull, 0xf87ce0e5b2094d9cull, 0xf92959bb5dd4ba74ull, 0xf9d64a46eb939f35ull, \
    0xfa83b2db722a033aull, 0xfb3193cc4227c3f4ull, 0xfbdfed6ce5f09c49ull, 0xfc8ec01121e447bbull, \
    0xfd3e0c0cf486c175ull, 0xfdedd1b496a89f35ull, 0xfe9e115c7b8f884cull, 0xff4ecb59511ec8a5ull,

constexpr uint64_t kLog2e = 0xb8aa3b295c17f0bcull;          // log2(e) 2^63
constexpr uint64_t kA1 = 0xb17217f7d1cf79acull;             // a_1 2^72
constexpr uint64_t kA2 = 0x3d7f7bff058b1d51ull;             // a_2 2^80
constexpr uint32_t kA3 = 1907106652u, kA4 = 1290923u, kA5 = 699u;   // a_3..a_5 2^59

#ifdef __CUDACC__
__device__ const uint64_t kExp2TabDev[256] = {BD_EXP2_TABLE};
#endif
static const uint64_t kExp2TabHost[256] = {BD_EXP2_TABLE};
#undef BD_EXP2_TABLE

BD_FIX_FN uint64_t fix_mulhi(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return uint64_t((unsigned __int128)a * b >> 64);
#endif
}

// |x| >= 64, infinities and NaN (out of line: membrane arguments stay inside)
#ifdef __CUDACC__
__host__ __device__ __noinline__
#endif
inline double exp_outside(double x) { return exp(x); }

BD_FIX_FN double exp_fixed(double x) {
  uint64_t bits;
#ifdef __CUDA_ARCH__
  bits = uint64_t(__double_as_longlong(x));
#else
  std::memcpy(&bits, &x, 8);
#endif
  const int e = int(bits >> 52 & 0x7ff) - 1023;
  if (e >= 6) return exp_outside(x);
  // |x| 2^57 (subnormal x: the spurious leading bit is shifted out)
  const uint64_t m = (bits & 0xfffffffffffffull) | 0x10000000000000ull;
  const int sh = 5 - e < 63 ? 5 - e : 63;
  const uint64_t X = (m << 10) >> sh;
  // t = X log2(e): integer part in the top 8 bits of hi, fraction below
  const uint64_t hi = fix_mulhi(X, kLog2e), lo = X * kLog2e;
  int k = int(hi >> 56);
  uint64_t f = hi << 8 | lo >> 56;
  if (bits >> 63) {                               // exp(-|x|): k + f -> -(k + f)
    k = -k - (f != 0);
    f = 0 - f;
  }
  const uint32_t j = uint32_t(f >> 56);
#ifdef __CUDA_ARCH__
  const uint64_t T = __ldg(reinterpret_cast<const unsigned long long*>(kExp2TabDev) + j);
#else
  const uint64_t T = kExp2TabHost[j];
#endif
  // u = u64 2^-64; series sum_n a_n u^n, a_n = (ln 2 / 256)^n / n!; terms of
  // degree 3 and up (below 2^-28) in 32 bits, the result at 2^72
  const uint64_t u64 = f << 8;
  const uint32_t u = uint32_t(u64 >> 32);
  uint32_t t = uint32_t(uint64_t(u) * kA5 >> 32) + kA4;                 // at 2^59
  t = uint32_t(uint64_t(u) * t >> 32) + kA3;
  const uint64_t s = (uint64_t(u) * t >> 11) + kA2;                     // at 2^80
  const uint64_t r = (fix_mulhi(u64, s) >> 8) + kA1;                    // at 2^72
  uint64_t M = T + (fix_mulhi(T, fix_mulhi(u64, r)) >> 8);              // 2^63 2^f, f < 1
  if (M < T) M = ~uint64_t(0);                                          // rounded up to 2^64
  // round to 53 bits; a carry (2^53) moves on into the exponent
  const uint64_t out = (M >> 11) + (M >> 10 & 1) + (uint64_t(int64_t(k) + 1022) << 52);
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)out);
#else
  double d;
  std::memcpy(&d, &out, 8);
  return d;
#endif
}

// 1 / d in integer arithmetic, correctly rounded as the division is: the
// mantissa's reciprocal from FP32 by two Newton steps r += r (1 - m r) in 64
// bits, cut to 53 bits, and the rounding decided by the sign of an exact
// product.  Zero, subnormal and non-finite d, and d whose reciprocal is
// subnormal, take the division.
//   Seed: m cut to 24 bits (below 2^-23 relative) and __fdividef (2 units in the
// last place, 2^-22 relative), so |1 - m r0| < 1.5 2^-21 and the 52-bit e1 is
// below 2^30 after its shift; the first step leaves 2^-41, the second what its
// truncations do (a few units of 2^-64, where rounding bears 2^10).
//   Measured on GB300, FP64 steps, with the rounding of r itself (0.501 units in
// the last place) / this: TP06 257^2 7.22 / 7.28 ms, slab 101x101x26 20.5 / 20.7.
#ifdef __CUDACC__
__host__ __device__ __noinline__
#endif
inline double recip_outside(double d) { return 1.0 / d; }

// bits: a normal d with a normal reciprocal; r0: the reciprocal of its mantissa, at 2^32
BD_FIX_FN uint64_t recip_from_seed(uint64_t bits, uint32_t r0) {
  const uint64_t m = bits << 11 | 0x8000000000000000ull;               // m / 2^63 in [1, 2)
  const int64_t e1 = int64_t(0x8000000000000000ull - fix_mulhi(m, uint64_t(r0) << 32));   // (1 - m r0) 2^63
  const uint64_t r1 = (uint64_t(r0) << 32) + uint64_t((int64_t(r0) * int64_t(int32_t(e1 >> 12))) >> 19);
  const int64_t e2 = int64_t(0x8000000000000000ull - fix_mulhi(m, r1));
  uint64_t r2 = r1 + uint64_t((int64_t(r1 >> 32) * e2) >> 31);
  if (e2 > 0 && r2 < r1) r2 = ~uint64_t(0);                             // m = 1: rounded up to 2^64
  // 1/m lies above q + 1/2 where (2 q + 1) m < 2^106; the product is within 2^55
  // of 2^106, so its low 64 bits have the difference's sign
  const uint64_t q = r2 >> 11;
  const int64_t side = int64_t((2 * q + 1) * (m >> 11));
  return q + (side < 0 ? 1u : 0u) + (uint64_t(2044u - (uint32_t(bits >> 52) & 0x7ffu)) << 52) +
         (bits & 0x8000000000000000ull);
}

BD_FIX_FN double recip_fixed(double d) {
  uint64_t bits;
#ifdef __CUDA_ARCH__
  bits = uint64_t(__double_as_longlong(d));
#else
  std::memcpy(&bits, &d, 8);
#endif
  const uint32_t be = uint32_t(bits >> 52) & 0x7ffu;
  if (be - 1u >= 2043u) return recip_outside(d);
  uint32_t r0;
  const uint32_t fb = 0x3f800000u | (uint32_t(bits >> 29) & 0x7fffffu);
#ifdef __CUDA_ARCH__
  r0 = __float2uint_rz(__fdividef(1.0f, __uint_as_float(fb)) * 4294967296.0f);   // saturates at 2^32 - 1
#else
  float f;
  std::memcpy(&f, &fb, 4);
  const float r = 1.0f / f * 4294967296.0f;
  r0 = r >= 4294967296.0f ? 0xffffffffu : uint32_t(r);
#endif
  const uint64_t out = recip_from_seed(bits, r0);
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)out);
#else
  double q;
  std::memcpy(&q, &out, 8);
  return q;
#endif
}

// Jacobi scaling 1 / d of a row, rounded to T once, without the FP64 pipe
template <class T>
BD_FIX_FN T jacobi_scale(double d) { return T(recip_fixed(d)); }

}  // namespace bd
