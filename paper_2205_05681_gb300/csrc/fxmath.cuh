// Exponential, logarithm and reciprocal of doubles on the integer pipe.
//
// GB300 issues an FP64 instruction per 16 clocks and SM (64 clocks of latency); a 64-bit integer
// multiply (umul64hi, about six IMADs) takes 5 clocks of an SM and 41 of latency.  A CUDA exp()
// occupies an SM for 304 clocks, log() for 568 and a division for 86 (latencies 1087, 2088 and
// 380; measured with all warps busy and with one warp).  The functions below keep 58 or more
// correct bits in 64-bit fixed point, use no FP64 instruction, and round once to a double.
//
// Fixed-point formats are written Qn: an integer v stands for v 2^-n.
//   fx_exp2(lg)      2^lg of a Q52 logarithm (|lg| < 2048)
//   fx_log2(x)       log2 of a positive normal double, Q52
//   fx_rcp(x)        1/x of any double (denormal and extreme arguments by the division); fx_div(a, b) a/b
//   fx_exp, fx_log   drop-in forms of exp and log for doubles
// Methods: 2^(n + i/64 + s/64) = 2^n T_i (1 + p(s)) with T_i = 2^(i/64) tabulated to 64 bits and p the
// Taylor polynomial of 2^(s/64) - 1 to degree 6 (remainder below 2^-58); log2 m = -log2 c_i +
// log2(1 + z) with c_i a 10-bit reciprocal of the middle of m's 1/64 interval, z = m c_i - 1 exact
// and the series of log2(1 + z) to degree 8 (remainder below 2^-62); 1/m = x (1 + e + e^2) from a
// 24-bit x with e = 1 - m x exact.
#ifndef FX_HOST
#define FX_FN __device__ __forceinline__
#define FX_SLOW __device__ __noinline__
#define FX_TAB __device__ const
typedef unsigned long long fx_u64;
typedef long long fx_i64;
FX_FN fx_u64 fx_mulhi(fx_u64 a, fx_u64 b) { return __umul64hi(a, b); }
FX_FN fx_i64 fx_mulhi_s(fx_i64 a, fx_i64 b) { return __mul64hi(a, b); }
FX_FN unsigned fx_mulhi32(unsigned a, unsigned b) { return __umulhi(a, b); }
FX_FN int fx_mulhi32_s(int a, int b) { return __mulhi(a, b); }
FX_FN int fx_clz(fx_u64 a) { return __clzll((long long)a); }
FX_FN double fx_as_double(fx_u64 a) { return __longlong_as_double((long long)a); }
FX_FN fx_u64 fx_bits(double a) { return (fx_u64)__double_as_longlong(a); }
// any approximation of 1/f good to 2^-22 serves
FX_FN float fx_rcp_seed(float f) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(f));
  return r;
}
FX_FN unsigned fx_bits_f(float a) { return __float_as_uint(a); }
FX_FN float fx_as_float(unsigned a) { return __uint_as_float(a); }
#endif

FX_TAB fx_u64 fx_t_exp[64] = {  // 2^(i/64), Q63
    0x8000000000000000ULL, 0x8164d1f3bc030773ULL, 0x82cd8698ac2ba1d7ULL, 0x843a28c3acde4046ULL,
    0x85aac367cc487b15ULL, 0x871f61969e8d1010ULL, 0x88980e8092da8527ULL, 0x8a14d575496efd9aULL,
    0x8b95c1e3ea8bd6e7ULL, 0x8d1adf5b7e5ba9e6ULL, 0x8ea4398b45cd53c0ULL, 0x9031dc431466b1dcULL,
    0x91c3d373ab11c336ULL, 0x935a2b2f13e6e92cULL, 0x94f4efa8fef70961ULL, 0x96942d3720185a00ULL,
    0x9837f0518db8a96fULL, 0x99e0459320b7fa65ULL, 0x9b8d39b9d54e5539ULL, 0x9d3ed9a72cffb751ULL,
    0x9ef5326091a111aeULL, 0xa0b0510fb9714fc2ULL, 0xa27043030c496819ULL, 0xa43515ae09e6809eULL,
    0xa5fed6a9b15138eaULL, 0xa7cd93b4e965356aULL, 0xa9a15ab4ea7c0ef8ULL, 0xab7a39b5a93ed337ULL,
    0xad583eea42a14ac6ULL, 0xaf3b78ad690a4375ULL, 0xb123f581d2ac2590ULL, 0xb311c412a9112489ULL,
    0xb504f333f9de6484ULL, 0xb6fd91e328d17791ULL, 0xb8fbaf4762fb9ee9ULL, 0xbaff5ab2133e45fbULL,
    0xbd08a39f580c36bfULL, 0xbf1799b67a731083ULL, 0xc12c4cca66709456ULL, 0xc346ccda24976407ULL,
    0xc5672a115506daddULL, 0xc78d74c8abb9b15dULL, 0xc9b9bd866e2f27a3ULL, 0xcbec14fef2727c5dULL,
    0xce248c151f8480e4ULL, 0xd06333daef2b2595ULL, 0xd2a81d91f12ae45aULL, 0xd4f35aabcfedfa1fULL,
    0xd744fccad69d6af4ULL, 0xd99d15c278afd7b6ULL, 0xdbfbb797daf23755ULL, 0xde60f4825e0e9124ULL,
    0xe0ccdeec2a94e111ULL, 0xe33f8972be8a5a51ULL, 0xe5b906e77c8348a8ULL, 0xe8396a503c4bdc68ULL,
    0xeac0c6e7dd24392fULL, 0xed4f301ed9942b84ULL, 0xefe4b99bdcdaf5cbULL, 0xf281773c59ffb13aULL,
    0xf5257d152486cc2cULL, 0xf7d0df730ad13bb9ULL, 0xfa83b2db722a033aULL, 0xfd3e0c0cf486c175ULL};
FX_TAB unsigned short fx_t_rcp[64] = {  // round(1024 / (1 + (i + 1/2)/64))
    1016, 1001, 986, 971, 957, 943, 930, 917, 904, 892, 880, 868, 857, 846, 835, 824,
    814, 804, 794, 785, 776, 767, 758, 749, 741, 732, 724, 716, 708, 701, 694, 686,
    679, 672, 665, 659, 652, 646, 639, 633, 627, 621, 615, 610, 604, 599, 593, 588,
    583, 577, 572, 567, 563, 558, 553, 548, 544, 539, 535, 531, 526, 522, 518, 514};
FX_TAB fx_u64 fx_t_log[64] = {  // -log2(fx_t_rcp[i] / 1024), Q62
    0x00b963dd107b993bULL, 0x0218f7089de2f29bULL, 0x037dd922a35585caULL, 0x04e833d5a81b12a9ULL,
    0x063f7c72a3ba9a83ULL, 0x079bd430b67dd4f7ULL, 0x08e3f3beef19edc6ULL, 0x0a30b1cabd7816d6ULL,
    0x0b823018e3cfc25fULL, 0x0cbe0e589e3f6043ULL, 0x0dfe33d3fffa6603ULL, 0x0f42be9e9b09b3dfULL,
    0x1070352293d72469ULL, 0x11a190a5d674a069ULL, 0x12d6eb4152324f5dULL, 0x14106017c3eca28eULL,
    0x1530fd08f29fa70aULL, 0x16552b499862776bULL, 0x177d01b66fbd36a5ULL, 0x188a76b7e549c593ULL,
    0x199b072a96c6b26fULL, 0x1aaec59dadadbdffULL, 0x1bc5c5489254cb9dULL, 0x1ce01a12f5d8d11fULL,
    0x1dddecf870c4c16cULL, 0x1efec61b011f855bULL, 0x200286657c006546ULL, 0x2109298cd71ddf83ULL,
    0x2212c02bbdc9b3b1ULL, 0x22fd9d2aabfae415ULL, 0x23ead593db351a40ULL, 0x24fce4101f9bcb9aULL,
    0x25ef532ff6a54ba2ULL, 0x26e44576e0e8f74bULL, 0x27dbc85d118f0923ULL, 0x28b2048f599c783cULL,
    0x29ae701b9884591bULL, 0x2a88f6e4cc87354fULL, 0x2b8a7df1c5bdaf21ULL, 0x2c697c3b5631664eULL,
    0x2d4a9a34ccec4a08ULL, 0x2e2de252d6a9cd97ULL, 0x2f135f5816e1f4c2ULL, 0x2fd4545db2f99c45ULL,
    0x30bdfa0c58cad99cULL, 0x3182766f239dffedULL, 0x32706c142142c03aULL, 0x3338917c40c7907fULL,
    0x34026c7331074974ULL, 0x34f6f29c5bf61878ULL, 0x35c4ab033e045967ULL, 0x369431cb64081194ULL,
    0x373b89a17174a0dbULL, 0x380e657c3d3fd6dcULL, 0x38e32736bb10ac5aULL, 0x39b9d7a46e732954ULL,
    0x3a6702414dbb3a61ULL, 0x3b41442a8cd32368ULL, 0x3bf155c1c8deaceeULL, 0x3ca2b99d3ed411c9ULL,
    0x3d8259ed72f4bb3cULL, 0x3e36c9c457af079aULL, 0x3eec9cee85684f3bULL, 0x3fa3d8ee4a154e23ULL};

// out of line, one copy each: the division of exceptional arguments, and results outside the
// normal exponents (53-bit r in [2^52, 2^53], 2^(n - 52) r)
FX_SLOW double fx_rcp_slow(double x) { return 1.0 / x; }
FX_SLOW double fx_exp2_slow(int n, fx_u64 r) {
  if (n > 0) return fx_as_double(n > 1023 ? 0x7ff0000000000000ULL : (2045ULL << 52) + r);
  if (n < -1100) return 0.0;
  return fx_as_double(((fx_u64)(n + 1322) << 52) + r) * 4.909093465297727e-91;  // 2^-300
}

// 2^n 2^(F 2^-64) for a 64-bit fraction F
FX_FN double fx_exp2_nf(int n, fx_u64 F) {
  const int i = (int)(F >> 58);
  const fx_u64 s = F << 6;  // Q64 position within the 1/64 interval
  const unsigned sh = (unsigned)(s >> 32);
  // 64 (2^(s/64) - 1) = s (d1 + s (d2 + ...)), d_k = ln2^k / (k! 64^(k-1))
  unsigned v = 0xaec3ff3cu + (fx_mulhi32(sh, 0xa184897cu) >> 9);  // d5 Q65, d6 Q74
  v = 0x9d955b7eu + (fx_mulhi32(sh, v) >> 9);                     // d4 Q56
  fx_u64 w = 0xe35846b82505fc5aULL + (((fx_u64)sh * v) >> 8);     // d3 Q80
  w = 0xf5fdeffc162c7543ULL + (fx_mulhi(s, w) >> 8);              // d2 Q72
  w = 0xb17217f7d1cf79acULL + (fx_mulhi(s, w) >> 8);              // d1 Q64
  const fx_u64 t = fx_t_exp[i];
  const fx_u64 m = t + (fx_mulhi(t, fx_mulhi(s, w)) >> 6);        // Q63 in [1, 2)
  const fx_u64 r = ((m >> 1) + 0x200) >> 10;                      // 53 bits, rounded
  if ((unsigned)(n + 1021) < 2044u) return fx_as_double(((fx_u64)(n + 1022) << 52) + r);
  return fx_exp2_slow(n, r);
}
FX_FN double fx_exp2(fx_i64 lg) { return fx_exp2_nf((int)(lg >> 52), (fx_u64)lg << 12); }

// log2 of the 53-bit mantissa m in [2^52, 2^53): Q62, in [0, 1], off by 2.2 2^-59 at most (the 32-bit tail of
// the series)
FX_FN fx_i64 fx_log2_mant(fx_u64 m) {
  const int i = (int)(m >> 46) & 63;
  const fx_i64 z = (fx_i64)(m * fx_t_rcp[i] - (1ULL << 62)) << 7;  // 2^7 z, Q62
  const int zh = (int)(z >> 32);                                   // Q30
  // 2^7 log2(1 + z) = s (E1 - s (E2 - ...)), s = 2^7 z, E_k = 1 / (k ln2 2^(7(k-1)))
  int u = 0x6985d8aa - (fx_mulhi32_s(zh, 0x5c551d95) >> 5);   // E7 Q75, E8 Q82
  u = 0x7b1c2771 - (fx_mulhi32_s(zh, u) >> 5);                // E6 Q68
  u = 0x49ddb143 - (fx_mulhi32_s(zh, u) >> 6);                // E5 Q60
  u = 0x5c551d95 - (fx_mulhi32_s(zh, u) >> 5);                // E4 Q53
  fx_i64 w = 0x3d8e13b87407fae9LL - (((fx_i64)zh * u) >> 6);  // E3 Q77
  w = 0x2e2a8eca5705fc2fLL - (fx_mulhi_s(z, w) >> 6);         // E2 Q69
  w = 0x5c551d94ae0bf85eLL - (fx_mulhi_s(z, w) >> 5);         // E1 Q62
  return (fx_i64)fx_t_log[i] + (fx_mulhi_s(z, w) >> 5);
}
FX_FN bool fx_normal_pos(double x) {  // positive, finite and not denormal
  const unsigned hi = (unsigned)(fx_bits(x) >> 32);
  return hi - 0x00100000u < 0x7fe00000u;
}
FX_FN int fx_exponent(double x) { return (int)((fx_bits(x) >> 52) & 2047) - 1023; }
FX_FN fx_u64 fx_mant(double x) { return (fx_bits(x) & 0xfffffffffffffULL) | 0x10000000000000ULL; }
// log2 of a positive normal double, Q52
FX_FN fx_i64 fx_log2(double x) {
  return ((fx_i64)fx_exponent(x) << 52) + ((fx_log2_mant(fx_mant(x)) + 512) >> 10);
}

// v 2^-n as a double, rounded once
FX_FN double fx_to_double(fx_i64 v, int n) {
  const fx_u64 sg = (fx_u64)v & 0x8000000000000000ULL;
  fx_u64 a = sg ? 0 - (fx_u64)v : (fx_u64)v;
  if (!a) return 0.0;
  const int c = fx_clz(a);
  a <<= c;
  const fx_u64 r = ((a >> 1) + 0x200) >> 10;
  return fx_as_double(sg | (((fx_u64)(1023 + 62 - c - n) << 52) + r));
}
// x 2^n rounded to an integer; magnitudes of 2^63 and more saturate, NaN gives a finite value
FX_FN fx_i64 fx_from_double(double x, int n) {
  const fx_u64 b = fx_bits(x);
  const int sh = (int)((b >> 52) & 2047) - 1075 + n;
  const fx_u64 m = fx_mant(x);
  const fx_u64 q = sh >= 0 ? (sh > 10 ? 0x7ff0000000000000ULL : m << sh)
                           : (sh < -54 ? 0 : ((m >> (-sh - 1)) + 1) >> 1);
  return (fx_i64)b < 0 ? -(fx_i64)q : (fx_i64)q;
}

// log2 of a positive normal double as Q62 (arguments in [1/2, 2)) or Q52; *n says which
FX_FN fx_i64 fx_log2_n(double x, int* n) {
  const int e = fx_exponent(x);
  const fx_i64 f = fx_log2_mant(fx_mant(x));
  const bool near = e == 0 || e == -1;
  *n = near ? 62 : 52;
  return near ? f + ((fx_i64)e << 62) : ((fx_i64)e << 52) + ((f + 512) >> 10);
}
FX_FN double fx_log2_d(double x) {
  int n;
  const fx_i64 v = fx_log2_n(x, &n);
  return fx_to_double(v, n);
}

// 1/m of a 53-bit mantissa m in [2^52, 2^53) standing for [1, 2): Q63, in (1/2, 1]
FX_FN fx_u64 fx_rcp_mant(fx_u64 m) {
  const float f = fx_rcp_seed(fx_as_float(0x3f800000u | ((unsigned)(m >> 29) & 0x7fffffu)));
  const unsigned fb = fx_bits_f(f);
  // x0 = 2^24 f, f in [1/2, 1]
  const unsigned x0 = fb >= 0x3f800000u ? 0x1000000u : ((fb & 0x7fffffu) | 0x800000u);
  const fx_i64 e = -(fx_i64)(m * x0);  // 1 - m x0, Q76 exact: |e| < 2^54 (the product mod 2^64)
  const fx_i64 eh = e >> 24;
  const fx_i64 t = e + ((eh * eh) >> 28);
  return ((fx_u64)x0 << 39) + (fx_u64)(((t >> 16) * (fx_i64)x0) >> 21);
}
// 1/x; fx_rcp_normal gives a meaningless value unless fx_rcp_ok (zero, denormal, huge, infinite, NaN)
FX_FN bool fx_rcp_ok(double x) { return ((unsigned)(fx_bits(x) >> 52) & 2047) - 1u < 2040u; }
FX_FN double fx_rcp_normal(double x) {
  const fx_u64 b = fx_bits(x);
  const unsigned be = (unsigned)(b >> 52) & 2047;
  const fx_u64 r = (fx_rcp_mant(fx_mant(x)) + 0x200) >> 10;
  return fx_as_double((b & 0x8000000000000000ULL) | (((fx_u64)(2044 - be) << 52) + r));
}
FX_FN double fx_rcp(double x) { return fx_rcp_ok(x) ? fx_rcp_normal(x) : fx_rcp_slow(x); }
// a/b; a divisor without a normal reciprocal takes the division (1/b overflows where a/b need not)
FX_SLOW double fx_div_slow(double a, double b) { return a / b; }
FX_FN double fx_div(double a, double b) { return fx_rcp_ok(b) ? a * fx_rcp_normal(b) : fx_div_slow(a, b); }

// exp(x): x in Q53 (exact; Q62 below 1) times log2(e), the product's integer part and 64 bits of its
// fraction
FX_FN double fx_exp(double x) {
  const unsigned be = (unsigned)(fx_bits(x) >> 52) & 2047;
  if (be >= 1032u) return exp(x);  // |x| >= 512, NaN
  const int k = be < 1023u ? 60 : 51;
  const fx_i64 q = fx_from_double(x, k + 2);
  fx_i64 hi = fx_mulhi_s(q, 0x5c551d94ae0bf85eLL);
  fx_u64 lo = (fx_u64)q * 0x5c551d94ae0bf85eULL;
  const fx_i64 c = (q >> 32) * -549191832LL;  // the next 32 bits of log2(e)
  lo += (fx_u64)c;
  hi += (c >> 63) + (lo < (fx_u64)c ? 1 : 0);
  return fx_exp2_nf((int)(hi >> k), ((fx_u64)hi << (64 - k)) | (lo >> k));
}
// ln x; arguments that are not positive normal numbers take log()
FX_FN double fx_log(double x) {
  if (!fx_normal_pos(x)) return log(x);
  int n;
  const fx_i64 v = fx_log2_n(x, &n);
  const fx_u64 sg = (fx_u64)v & 0x8000000000000000ULL;
  fx_u64 a = sg ? 0 - (fx_u64)v : (fx_u64)v;
  if (!a) return 0.0;
  const int c = fx_clz(a);
  a = fx_mulhi(a << c, 0xb17217f7d1cf79acULL);  // times ln2 (Q64): in [2^62, 2^64)
  const int c2 = (int)(a >> 63) ^ 1;
  a <<= c2;
  const fx_u64 r = ((a >> 1) + 0x200) >> 10;
  return fx_as_double(sg | (((fx_u64)(1023 + 62 - c - c2 - n) << 52) + r));
}
