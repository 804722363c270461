// Double-precision exp, sin, cos, division and square root on the integer pipe.
//
// One source for the generated kernels (embedded as text and compiled with
// them) and the interpreter kernel.  On GB300 a double add, multiply or fma
// occupies a scheduler's FP64 unit for 64 clocks per warp (2 per clock and SM,
// measured), while a 32x32->64-bit multiply-add costs 4, a shift or logic op 2
// and an add 1, and straight-line programs leave those units idle.  The library
// functions are built from FP64 ops (in FMA-equivalents, measured: exp 15, sin
// and cos 18, division 7.7, square root 8.2: 490 to 1,180 clocks per warp); here
// the arithmetic is fixed point and leaves the FP64 unit to the adds and
// multiplies.  Arguments outside the stated ranges (special values, subnormals,
// far ends) go to the library function.
//
//   division, square root: exact remainders, results rounded to nearest as IEEE
//     754 asks, bit for bit the hardware library's.
//   exp, sin, cos: one rounding of a result known to about 2^-57: at most 0.58,
//     0.52 and 0.52 ulp over 4 million arguments each (the library: 1 ulp and more).
//
// Measured, clocks per warp and call with one / four warps per scheduler, library
// -> here: exp 1062 / 1144 -> 408 / 133, sin 1394 / 1350 -> 551 / 209, division
// 722 / 628 -> 344 / 120, square root 679 / 572 -> 298 / 103.
//
// Notation: "lsb 2^-k" is the weight of an integer's lowest bit.
typedef unsigned int cs_u32;
typedef unsigned long long cs_u64;

static __device__ __forceinline__ cs_u64 cs_wide(cs_u32 a, cs_u32 b) { return (cs_u64)a * b; }
static __device__ __forceinline__ cs_u32 cs_hi32(cs_u64 a) { return (cs_u32)(a >> 32); }
static __device__ __forceinline__ cs_u64 cs_pack(cs_u32 hi, cs_u32 lo) { return (cs_u64)hi << 32 | lo; }
#ifndef CS_MATH_HOST   // a host build (tests) brings its own
// shifts by any amount (64 and more give 0), one funnel shift per word
static __device__ __forceinline__ cs_u64 cs_shr64(cs_u64 a, cs_u32 s) {
  cs_u64 r;
  asm("shr.b64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(s));
  return r;
}
static __device__ __forceinline__ cs_u64 cs_shl64(cs_u64 a, cs_u32 s) {
  cs_u64 r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(s));
  return r;
}
// single-precision reciprocal and reciprocal square root, 1 ulp
static __device__ __forceinline__ float cs_rcpf(float a) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
static __device__ __forceinline__ float cs_rsqrtf(float a) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
#endif
// top 64 bits of a 64x64-bit product without the low partial product (at most 3
// units low); the sum of the cross products' high words must fit 32 bits or be
// allowed to carry: it is added as 64 bits
static __device__ __forceinline__ cs_u64 cs_mul_top(cs_u64 a, cs_u64 b) {
  const cs_u32 ah = cs_hi32(a), al = (cs_u32)a, bh = cs_hi32(b), bl = (cs_u32)b;
  return cs_wide(ah, bh) + __umulhi(ah, bl) + __umulhi(al, bh);
}
// low 64 bits of a 64x64-bit product
static __device__ __forceinline__ cs_u64 cs_mul_low(cs_u64 a, cs_u64 b) { return a * b; }

static __device__ __noinline__ double cs_exp_lib(double x) { return exp(x); }
static __device__ __noinline__ double cs_sin_lib(double x) { return sin(x); }
static __device__ __noinline__ double cs_cos_lib(double x) { return cos(x); }
static __device__ __noinline__ double cs_div_lib(double a, double b) { return a / b; }
static __device__ __noinline__ double cs_sqrt_lib(double a) { return sqrt(a); }

// 2^((j - 1/16) / 256), lsb 2^-61
static __device__ const cs_u64 cs_exp_table[256] = {
  0x1ffe9d237fe37188ull, 0x2014d221e76df99full, 0x202b168a2f771056ull, 0x20416a670ac64738ull,
  0x2057cdc3339022f2ull, 0x206e40a96b7b42b9ull, 0x2084c3247ba58b4full, 0x209b553f34a95595ull,
  0x20b1f7046ea2a0c0ull, 0x20c8a87f0934481eull, 0x20df69b9eb8d3c80ull, 0x20f63ac0046dc145ull,
  0x210d1b9c4a2cad00ull, 0x21240c59babcadd0ull, 0x213b0d035bb19151ull, 0x21521da43a459044ull,
  0x21693e476b5e9ddcull, 0x21806ef80b93babeull, 0x2197afc13f324bb4ull, 0x21af00ae32437410ull,
  0x21c661ca189173ccull, 0x21ddd3202dad095dull, 0x21f554bbb4f2d74bull, 0x220ce6a7f990cd80ull,
  0x222488f04e8b965cull, 0x223c3ba00ec4078dull, 0x2253fec29cfc96aeull, 0x226bd26363ded1aeull,
  0x2283b68dd600db04ull, 0x229bab4d6deae9b5ull, 0x22b3b0adae1ccd21ull, 0x22cbc6ba211374b0ull,
  0x22e3ed7e594e7b50ull, 0x22fc2505f155b6cbull, 0x23146d5c8bbecaf9ull, 0x232cc68dd332c0d8ull,
  0x234530a57a73a178ull, 0x235dabaf3c6214d8ull, 0x237637b6dc0304a2ull, 0x238ed4c8248542d1ull,
  0x23a782eee9473448ull, 0x23c0423705dc7f51ull, 0x23d912ac5e13be14ull, 0x23f1f45addfc34fbull,
  0x240ae74e79eb8d16ull, 0x2423eb932e839272ull, 0x243d013500b7f66dull, 0x2456283ffdd4160eull,
  0x246f60c03b80c45aull, 0x2488aac1d7ca18b0ull, 0x24a20650f925412eull, 0x24bb7379ce76591cull,
  0x24d4f2488f16436bull, 0x24ee82c97ad8893eull, 0x25082508da113c88ull, 0x2521d912fd9adec2ull,
  0x253b9ef43edc4bb6ull, 0x255576b8ffcea866ull, 0x256f606dab035614ull, 0x25895c1eb3a9e96aull,
  0x25a369d8959625c3ull, 0x25bd89a7d545fc9cull, 0x25d7bb98ffe79135ull, 0x25f1ffb8ab5f4055ull,
  0x260c5613764dac42ull, 0x2626beb60815ccf0ull, 0x264139ad10e3045aull, 0x265bc70549af371full,
  0x267666cb7448e954ull, 0x2691190c5b595f95ull, 0x26abddd4d26ac456ull, 0x26c6b531b5ee517cull,
  0x26e19f2feb427e3aull, 0x26fc9bdc60b93134ull, 0x2717ab440d9df6faull, 0x2732cd73f23c3cc9ull,
  0x274e027917e58f9full, 0x27694a6090f7dfafull, 0x2784a53778e3c81full, 0x27a0130af432db31ull,
  0x27bb93e8308df2bfull, 0x27d727dc64c3851eull, 0x27f2cef4d0cdfe6aull, 0x280e893ebdda1e31ull,
  0x282a56c77e4d5990ull, 0x2846379c6dcc41bfull, 0x28622bcaf140ef06ull, 0x287e336076e1702full,
  0x289a4e6a76363e6full, 0x28b67cf67020b5c1ull, 0x28d2bf11eee191c9ull, 0x28ef14ca861f6f34ull,
  0x290b7e2dd2ed5195ull, 0x2927fb497bd12dd8ull, 0x29448c2b30ca7932ull, 0x296130e0ab58bca1ull,
  0x297de977ae822d02ull, 0x299ab5fe06da47b6ull, 0x29b796818a8873deull, 0x29d48b10194ea833ull,
  0x29f193b79c90157aull, 0x2a0eb0860757d598ull, 0x2a2be189565f9f49ull, 0x2a4926cf90167e84ull,
  0x2a668066c4a7917dull, 0x2a83ee5d0e00ca61ull, 0x2aa170c08fd9b5bcull, 0x2abf079f77ba4592ull,
  0x2adcb307fd01a132ull, 0x2afa730860ecf9c4ull, 0x2b1847aeee9e638full, 0x2b363109fb23b408ull,
  0x2b542f27e57d64a0ull, 0x2b72421716a57a59ull, 0x2b9069e601967228ull, 0x2baea6a323523228ull,
  0x2bccf85d02e8ff96ull, 0x2beb5f22318079abull, 0x2c09db014a5a994aull, 0x2c286c08f2dcb587ull,
  0x2c471247da968d14ull, 0x2c65cdccbb495488ull, 0x2c849ea658eec995ull, 0x2ca384e381c04b1bull,
  0x2cc280930e3df637ull, 0x2ce191c3e135c832ull, 0x2d00b884e7cac56full, 0x2d1ff4e5197c254dull,
  0x2d3f46f3782c82fcull, 0x2d5eaebf1029135cull, 0x2d7e2c56f830dfd4ull, 0x2d9dbfca517c0630ull,
  0x2dbd692847c2fd8aull, 0x2ddd28801145e03aull, 0x2dfcfde0eed3bad8ull, 0x2e1ce95a2bd1e050ull,
  0x2e3ceafb1e43430dull, 0x2e5d02d326cfd33dull, 0x2e7d30f1b0cbe230ull, 0x2e9d7566323f8addull,
  0x2ebdd0402bee1f85ull, 0x2ede418f295d9c83ull, 0x2efec962c0de2047ull, 0x2f1f67ca9391687cull,
  0x2f401cd64d725464ull, 0x2f60e895a55c6c6cull, 0x2f81cb185d136ef4ull, 0x2fa2c46e414ae25aull,
  0x2fc3d4a729adac46ull, 0x2fe4fbd2f8e5ae36ull, 0x30063a019ca36755ull, 0x30278f430da59ba4ull,
  0x3048fba74fc10068ull, 0x306a7f3e71e7edf3ull, 0x308c1a188e3216c2ull, 0x30adcc45c9e443f7ull,
  0x30cf95d65578172full, 0x30f176da6ca3d1beull, 0x31136f625662214dull, 0x31357f7e64f9f1e7ull,
  0x3157a73ef606456cull, 0x3179e6b4727e107eull, 0x319c3def4ebc1cdfull, 0x31bead000a86f143ull,
  0x31e133f73118beacull, 0x3203d2e559275335ull, 0x322689db24ec1272ull, 0x324958e9422bf34cull,
  0x326c40206a3f8371ull, 0x328f3f91621af04full, 0x32b2574cfa5615a3ull, 0x32d587640f3491a4ull,
  0x32f8cfe788addec5ull, 0x331c30e85a757316ull, 0x333faa778402e54eull, 0x33633ca6109a1774ull,
  0x3386e7851753673aull, 0x33aaab25bb23e406ull, 0x33ce87992ae58aa6ull, 0x33f27cf0a15f86c9ull,
  0x34168b3d654e7a27ull, 0x343ab290c96cc96bull, 0x345ef2fc2c7aeee6ull, 0x34834c90f947d2ffull,
  0x34a7bf60a6b92a74ull, 0x34cc4b7cb7d3da6cull, 0x34f0f0f6bbc46254ull, 0x3515afe04de74b99ull,
  0x353a884b15d19f3full, 0x355f7a48c759614dull, 0x358485eb229e122aull, 0x35a9ab43f41135d6ull,
  0x35ceea65147ee114ull, 0x35f4436069164c81ull, 0x3619b647e3726da0ull, 0x363f432d81a295dfull,
  0x3664ea234e331792ull, 0x368aab3b6035f0f7ull, 0x36b08687db4b7d36ull, 0x36d67c1aefab2b6eull,
  0x36fc8c06da2c3bcdull, 0x3722b65de44e82baull, 0x3748fb326443320full, 0x376f5a96bcf5a877ull,
  0x3795d49d5e1446dbull, 0x37bc6958c4194bfdull, 0x37e318db7853b632ull, 0x3809e33810f02b4bull,
  0x3830c8813101e6a4ull, 0x3857c8c9888bad71ull, 0x387ee423d488c93aull, 0x38a61aa2def60894ull,
  0x38cd6c597edac61dull, 0x38f4d95a9851f5b7ull, 0x391c61b91c93380eull, 0x3944058809fbf46dull,
  0x396bc4da6c1878dfull, 0x39939fc35bad20a8ull, 0x39bb9655febf811cull, 0x39e3a8a5889f9ccbull,
  0x3a0bd6c539f11d17ull, 0x3a3420c860b49233ull, 0x3a5c86c25850b982ull, 0x3a8508c6899bca74ull,
  0x3aada6e86ae4c9d2ull, 0x3ad6613b7ffce37aull, 0x3aff37d35a40caabull, 0x3b282ac398a220c3ull,
  0x3b513a1fe7b0e289ull, 0x3b7a65fc01a4dc05ull, 0x3ba3ae6bae6722e3ull, 0x3bcd1382c39b976cull,
  0x3bf6955524aa6c1aull, 0x3c2033f6c2c9b3c2ull, 0x3c49ef7b9d06f66bull, 0x3c73c7f7c050ccbfull,
  0x3c9dbd7f47808233ull, 0x3cc7d0265b63bdd5ull, 0x3cf2000132c631d5ull, 0x3d1c4d24127b51c3ull,
  0x3d46b7a34d680f8bull, 0x3d713f93448c9f38ull, 0x3d9be508670e4178ull, 0x3dc6a817324114ecull,
  0x3df188d431b1ee50ull, 0x3e1c8753ff303770ull, 0x3e47a3ab42d7d4f8ull, 0x3e72ddeeb31b1328ull,
  0x3e9e363314cc9966ull, 0x3ec9ac8d3b2964baull, 0x3ef5411207e2c938ull, 0x3f20f3d66b287a5aull,
  0x3f4cc4ef63b29a56ull, 0x3f78b471fecbd063ull, 0x3fa4c273585b660full, 0x3fd0ef089aef6b8cull
};

// exp(x), 2^-126 <= |x| < 708: k = floor(256 x / ln 2) from a single-precision
// estimate (off by at most 0.04), r = x - (k - 1/16) ln2/256 in [0, 1.11 ln2/256)
// exactly in fixed point, exp = 2^(k/256 - 1/4096) (1 + r + r^2/2 + r^3/6 + r^4/24
// + r^5/120): the dropped term is below 2^-61.
static __device__ __forceinline__ double cs_exp64(double x) {
  const cs_u32 hi = (cs_u32)__double2hiint(x), lo = (cs_u32)__double2loint(x);
  const cs_u32 ahi = hi & 0x7fffffffu;
  if (ahi - 0x38100000u >= 0x40862000u - 0x38100000u) return cs_exp_lib(x);
  const cs_u32 f3 = __funnelshift_l(lo, hi, 3);
  const float xf = __uint_as_float((f3 + 0x40000000u) | (hi & 0x80000000u));   // x to 24 bits
  const cs_u32 k = __float_as_uint(__fmaf_rd(xf, 0x1.715476p+8f, 12582912.0f)); // 0x4B400000 + k
  // |x| with lsb 2^-58, modulo 2^64 (the bits above cancel against k ln2/256)
  const cs_u64 m = cs_pack(__funnelshift_l(lo, hi, 11) | 0x80000000u, lo << 11);
  const cs_u32 sh = 1028u - (ahi >> 20);
  const cs_u64 ax = cs_shr64(m, sh) | cs_shl64(m, 0u - sh);
  const cs_u32 s = (cs_u32)((int)hi >> 31);
  const cs_u64 sx = ax ^ cs_pack(s, s);
  cs_u64 r = sx + 0x262e8e0d780cf0d5ull + (hi >> 31) + cs_wide(k, 0xa020b8c2u) + __umulhi(k, 0x1950d871u);
  r += (cs_u64)(k * 0xfffd3a37u) << 32;
  r <<= 13;                                             // lsb 2^-71
  const cs_u32 rh = cs_hi32(r), rl = (cs_u32)r;         // rh: lsb 2^-39
  const cs_u64 q = cs_wide(rh, rh) + 2 * (cs_u64)__umulhi(rh, rl);     // r^2, lsb 2^-78
  const cs_u32 qn = __funnelshift_r((cs_u32)q, cs_hi32(q), 30);        // lsb 2^-48
  const cs_u64 c3 = cs_wide(qn, rh);                                   // r^3, lsb 2^-87
  const cs_u32 c = __funnelshift_r((cs_u32)c3, cs_hi32(c3), 30);       // lsb 2^-57
  // 1/6 + r/24 + r^2/120, lsb 2^-34
  const cs_u32 a = 0xaaaaaaabu + __umulhi(rh, 5592405u) + __umulhi(qn, 2185u);
  const cs_u64 p = r + (q >> 8) + (cs_wide(c, a) >> 20);               // exp(r) - 1, lsb 2^-71
  const cs_u64 t = cs_exp_table[k & 255u];
  const cs_u32 th = cs_hi32(t), tl = (cs_u32)t, ph = cs_hi32(p), pl = (cs_u32)p;
  const cs_u64 y = t + ((cs_wide(th, ph) + (cs_u64)(__umulhi(th, pl) + __umulhi(tl, ph))) >> 7);   // lsb 2^-61
  // [0.999, 2.01): the leading bit to bit 62, round, exponent
  const cs_u32 z = (cs_u32)__clz((int)cs_hi32(y));                     // 1, 2 or 3
  const cs_u64 n = (y << (z - 1u)) + 0x200u;
  const cs_u32 e = (k >> 8) + (1024u - 0x4b4000u) - z;                 // exponent field - 1
  return __hiloint2double((int)((cs_hi32(n) >> 10) + (e << 20)), (int)__funnelshift_r((cs_u32)n, cs_hi32(n), 10));
}

// sin and cos of x, 2^-27 <= |x| < 2^18: |x| = k pi/2 + r, |r| <= 0.82, r with
// lsb 2^-95 (a remainder below 2^-20 would keep too few bits: library);
// 1 - sin(r)/r and 1 - cos r are polynomials in z = r^2 of degree 7 with
// coefficients by interpolation at Chebyshev nodes (gen_math64_tables.py),
// evaluated as c1 - y (c2 - y (c3 - ...)), y = z/64, lsb 2^-61.
struct cs_trig {
  cs_u32 nh, nl, lz;      // |r| = (nh:nl) 2^(-63 - lz), leading bit set
  cs_u32 neg;             // bit 31: r negative
  cs_u32 k;               // quadrant
  cs_u64 z;               // r^2, lsb 2^-64
  bool rare;
};
static __device__ __forceinline__ cs_trig cs_trig_reduce(cs_u32 hi, cs_u32 lo) {
  cs_trig t;
  const cs_u32 e = (hi & 0x7fffffffu) >> 20;
  const cs_u32 f3 = __funnelshift_l(lo, hi, 3);
  const cs_u32 k = __float_as_uint(fmaf(__uint_as_float(f3 + 0x40000000u), 0x1.45f306p-1f, 12582912.0f)) - 0x4b400000u;
  // |x| with lsb 2^-63 (words 1 and 2 of 96 bits) minus k pi/2
  const cs_u32 mh = (hi & 0xfffffu) | 0x100000u;
  const cs_u64 xw = cs_pack(__funnelshift_l(lo, mh, e - 1012u), lo << ((e - 1012u) & 31u));
  const cs_u64 p0 = cs_wide(k, 0xc4c6628cu);
  const cs_u64 p1 = cs_wide(k, 0x2168c234u) + cs_hi32(p0) + ((cs_u64)(k * 0xc90fdaa2u) << 32);
  const cs_u64 d = xw - p1 - (cs_u64)((cs_u32)p0 != 0u);
  const cs_u32 s = (cs_u32)((int)cs_hi32(d) >> 31);                    // remainder negative: negate
  const cs_u32 r2 = cs_hi32(d) ^ s, r1 = (cs_u32)d ^ s, r0 = (0u - (cs_u32)p0) ^ s;
  t.lz = (cs_u32)__clz((int)r2);
  t.nh = __funnelshift_l(r1, r2, t.lz);
  t.nl = __funnelshift_l(r0, r1, t.lz);
  t.neg = s;
  t.k = k;
  t.rare = t.lz > 20u;
  if (e < 1022u) {                                                     // |x| < 1/2: r = x
    t.nh = __funnelshift_l(lo, hi, 11) | 0x80000000u;
    t.nl = lo << 11;
    t.lz = 1023u - e;
    t.neg = t.k = 0u;
    t.rare = false;
  }
  const cs_u64 rr = cs_shr64(cs_pack(t.nh, t.nl), t.lz - 1u);          // lsb 2^-64
  const cs_u32 rh = cs_hi32(rr);
  t.z = cs_wide(rh, rh) + 2 * (cs_u64)__umulhi(rh, (cs_u32)rr);
  return t;
}
// sin(r)/r (c false) or cos r (c true), lsb 2^-61
static __device__ __forceinline__ cs_u64 cs_trig_poly(cs_u64 z, bool c) {
  const cs_u64 y = z >> 6;
  const cs_u32 yh = cs_hi32(y), yl = (cs_u32)y;
  const cs_u32 v6 = (c ? 0x47ba723fu : 0x0584834eu) - __umulhi(yh, c ? 0x18f9411cu : 0x01aab7f7u);   // lsb 2^-29
  cs_u64 v = (c ? 0x93f27bf8eedb71c8ull : 0x0d7322997086c494ull) - (cs_wide(yh, v6) + __umulhi(yl, v6));
  v = (c ? 0xd00d00ce5cd425faull : 0x171de3a53d560bf6ull) - cs_mul_top(y, v);
  v = (c ? 0xb60b60b60a9b65c4ull : 0x1a01a01a01947c49ull) - cs_mul_top(y, v);
  v = (c ? 0x555555555555338cull : 0x1111111111110f14ull) - cs_mul_top(y, v);
  v = (c ? 0x0fffffffffffffffull : 0x0555555555555555ull) - cs_mul_top(y, v);
  return 0x2000000000000000ull - cs_mul_top(z, v);
}
// (nh:nl) 2^(-63 - lz) w with the sign bit of sg, rounded
static __device__ __forceinline__ double cs_trig_round(cs_u32 nh, cs_u32 nl, cs_u32 lz, cs_u64 w, cs_u32 sg) {
  const cs_u64 g = cs_mul_top(cs_pack(nh, nl), w << 2);                // lsb 2^-62, [0.66, 2)
  const cs_u32 h = 1u - (cs_hi32(g) >> 30);                            // leading bit to bit 62
  const cs_u64 n = (g << h) + 0x200u;
  return __hiloint2double((int)(((cs_hi32(n) >> 10) + ((1022u - lz - h) << 20)) | (sg & 0x80000000u)),
                          (int)__funnelshift_r((cs_u32)n, cs_hi32(n), 10));
}
// |x| outside the range: too small (true) or for the library
static __device__ __forceinline__ bool cs_trig_far(cs_u32 ahi) { return ahi - 0x3e400000u >= 0x41100000u - 0x3e400000u; }

// sin (quad 0) or cos (quad 1)
static __device__ __forceinline__ double cs_trig64(double x, cs_u32 quad) {
  const cs_u32 hi = (cs_u32)__double2hiint(x), lo = (cs_u32)__double2loint(x);
  cs_trig t = cs_trig_reduce(hi, lo);
  if (t.rare) return quad ? cs_cos_lib(x) : cs_sin_lib(x);
  const cs_u32 kq = t.k + quad;
  const bool c = (kq & 1u) != 0u;
  const cs_u64 w = cs_trig_poly(t.z, c);
  if (c) { t.nh = 0x80000000u; t.nl = 0u; t.lz = 0u; t.neg = 0u; }
  return cs_trig_round(t.nh, t.nl, t.lz, w, (kq << 30) ^ t.neg ^ (quad ? 0u : hi));
}
static __device__ __forceinline__ double cs_sin64(double x) {
  const cs_u32 ahi = (cs_u32)__double2hiint(x) & 0x7fffffffu;
  if (cs_trig_far(ahi)) return ahi < 0x3e400000u ? x : cs_sin_lib(x);
  return cs_trig64(x, 0u);
}
static __device__ __forceinline__ double cs_cos64(double x) {
  const cs_u32 ahi = (cs_u32)__double2hiint(x) & 0x7fffffffu;
  if (cs_trig_far(ahi)) return ahi < 0x3e400000u ? 1.0 : cs_cos_lib(x);
  return cs_trig64(x, 1u);
}
// both at once: one reduction, and the two polynomials overlap; the same bits
static __device__ __forceinline__ void cs_sincos64(double x, double& sn, double& cs) {
  const cs_u32 hi = (cs_u32)__double2hiint(x), lo = (cs_u32)__double2loint(x), ahi = hi & 0x7fffffffu;
  if (cs_trig_far(ahi)) {
    sn = ahi < 0x3e400000u ? x : cs_sin_lib(x);
    cs = ahi < 0x3e400000u ? 1.0 : cs_cos_lib(x);
    return;
  }
  const cs_trig t = cs_trig_reduce(hi, lo);
  if (t.rare) { sn = cs_sin_lib(x); cs = cs_cos_lib(x); return; }
  const bool odd = (t.k & 1u) != 0u;
  // sin x: +-sin r (k even) or +-cos r; cos x the other, by quadrant k + 1
  const cs_u32 ss = (t.k << 30) ^ hi, sc = (t.k + 1u) << 30;
  const double a = cs_trig_round(t.nh, t.nl, t.lz, cs_trig_poly(t.z, false), t.neg ^ (odd ? sc : ss));
  const double b = cs_trig_round(0x80000000u, 0u, 0u, cs_trig_poly(t.z, true), odd ? ss : sc);
  sn = odd ? b : a;
  cs = odd ? a : b;
}

// a / b, both magnitudes in [2^-509, 2^513): Y = 2^32/b from the single-precision
// reciprocal, low by at most 2^-21.2 and never high (b is rounded up first and Y
// lowered by 512; checked for all 2^23 mantissas), so that each quotient digit is
// low and each remainder positive and exact modulo 2^64; the last remainder
// decides the rounding.
static __device__ __forceinline__ bool cs_div_far(cs_u32 ha, cs_u32 hb) {   // outside the range
  return (ha << 1) - 0x40400000u >= 0x7fc00000u || (hb << 1) - 0x40400000u >= 0x7fc00000u;
}
static __device__ __forceinline__ double cs_div_rare(double a, double b) {
  const cs_u32 ha = (cs_u32)__double2hiint(a), la = (cs_u32)__double2loint(a), hb = (cs_u32)__double2hiint(b);
  const bool zero = ((ha & 0x7fffffffu) | la) == 0u;                   // 0 / normal
  if (zero && (hb & 0x7fffffffu) - 0x00100000u < 0x7fe00000u) return __hiloint2double((int)((ha ^ hb) & 0x80000000u), 0);
  return cs_div_lib(a, b);
}
// 2^32/b for the mantissa of b as a number in [1, 2)
static __device__ __forceinline__ cs_u32 cs_div_seed(cs_u32 hb, cs_u32 lb) {
  const float bf = __uint_as_float(((__funnelshift_l(lb, hb, 3) & 0x7fffffu) | 0x3f800000u) + 1u);
  return __float_as_uint(cs_rcpf(bf)) * 256u + (0x80000000u - 512u);
}
// rounds v, the quotient of the mantissas with lsb 2^-54 or up to one unit less
static __device__ __forceinline__ double cs_div_round(cs_u64 v, cs_u32 ha, cs_u32 la, cs_u32 hb, cs_u64 mb) {
  const cs_u32 h = cs_hi32(v) >> 22;                                   // quotient >= 1
  cs_u64 t = v >> h;                                                   // 53 bits and the rounding bit, or one less
  const cs_u64 rem = cs_pack(la << (22u - h), 0u) - cs_mul_low(t, mb);
  t = (t + (rem >= mb ? 2u : 1u)) >> 1;
  const cs_u32 e = (ha & 0x7ff00000u) - (hb & 0x7ff00000u) + ((1021u + h) << 20);
  return __hiloint2double((int)((cs_hi32(t) + e) | ((ha ^ hb) & 0x80000000u)), (int)(cs_u32)t);
}
static __device__ __forceinline__ double cs_div64(double a, double b) {
  const cs_u32 ha = (cs_u32)__double2hiint(a), la = (cs_u32)__double2loint(a);
  const cs_u32 hb = (cs_u32)__double2hiint(b), lb = (cs_u32)__double2loint(b);
  if (cs_div_far(ha, hb)) return cs_div_rare(a, b);
  const cs_u32 ah = (ha & 0xfffffu) | 0x100000u, bh = (hb & 0xfffffu) | 0x100000u;
  const cs_u64 ma = cs_pack(ah, la), mb = cs_pack(bh, lb);
  const cs_u32 Y = cs_div_seed(hb, lb);
  const cs_u32 q1 = __umulhi(__funnelshift_l(la, ah, 11), Y);          // lsb 2^-31
  cs_u64 r = (ma << 31) - cs_mul_low(mb, q1);
  const cs_u32 q2 = __umulhi(cs_hi32(r), Y);                           // lsb 2^-51
  r = (r << 20) - cs_mul_low(mb, q2);
  const cs_u32 q3 = __umulhi(cs_hi32(r), Y);                           // lsb 2^-71
  return cs_div_round(((cs_wide(q1, 1u << 20) + q2) << 3) + (q3 >> 17), ha, la, hb, mb);
}

// Division by a divisor used several times: cs_recip64(b) is 2^64/b of its
// mantissa, low by at most 4 units; the quotient of cs_divr64 then comes from one
// product (low by less than 2^-60) and the same exact rounding: 38 instructions
// in place of 75.  For constant divisors the compiler of the program provides r.
static __device__ __forceinline__ cs_u64 cs_recip64(double b) {
  const cs_u32 hb = (cs_u32)__double2hiint(b), lb = (cs_u32)__double2loint(b);
  const cs_u64 mb = cs_pack((hb & 0xfffffu) | 0x100000u, lb);
  const cs_u32 Y = cs_div_seed(hb, lb);
  const cs_u32 q1 = __umulhi(0x80000000u, Y);                          // a = 1: lsb 2^-31
  cs_u64 r = 0ull - cs_mul_low(mb, q1);                                // 2^83 modulo 2^64 is 0
  const cs_u32 q2 = __umulhi(cs_hi32(r), Y);
  r = (r << 20) - cs_mul_low(mb, q2);
  const cs_u32 q3 = __umulhi(cs_hi32(r), Y);
  return (cs_wide(q1, 1u << 20) << 13) + ((cs_u64)q2 << 13) + (q3 >> 7);
}
static __device__ __forceinline__ double cs_divr64(double a, double b, cs_u64 r) {
  const cs_u32 ha = (cs_u32)__double2hiint(a), la = (cs_u32)__double2loint(a);
  const cs_u32 hb = (cs_u32)__double2hiint(b), lb = (cs_u32)__double2loint(b);
  if (cs_div_far(ha, hb)) return cs_div_rare(a, b);
  const cs_u64 m = cs_pack(__funnelshift_l(la, ha, 11) | 0x80000000u, la << 11);
  return cs_div_round(cs_mul_top(m, r) >> 9, ha, la, hb, cs_pack((hb & 0xfffffu) | 0x100000u, lb));
}

// two quotients by one divisor: their products and roundings overlap
static __device__ __forceinline__ void cs_divr64x2(double a0, double a1, double b, cs_u64 r, double& q0, double& q1) {
  const cs_u32 h0 = (cs_u32)__double2hiint(a0), l0 = (cs_u32)__double2loint(a0);
  const cs_u32 h1 = (cs_u32)__double2hiint(a1), l1 = (cs_u32)__double2loint(a1);
  const cs_u32 hb = (cs_u32)__double2hiint(b), lb = (cs_u32)__double2loint(b);
  if (cs_div_far(h0, hb) || cs_div_far(h1, hb)) {
    q0 = cs_div_far(h0, hb) ? cs_div_rare(a0, b) : cs_divr64(a0, b, r);
    q1 = cs_div_far(h1, hb) ? cs_div_rare(a1, b) : cs_divr64(a1, b, r);
    return;
  }
  const cs_u64 mb = cs_pack((hb & 0xfffffu) | 0x100000u, lb);
  const cs_u64 v0 = cs_mul_top(cs_pack(__funnelshift_l(l0, h0, 11) | 0x80000000u, l0 << 11), r) >> 9;
  const cs_u64 v1 = cs_mul_top(cs_pack(__funnelshift_l(l1, h1, 11) | 0x80000000u, l1 << 11), r) >> 9;
  q0 = cs_div_round(v0, h0, l0, hb, mb);
  q1 = cs_div_round(v1, h1, l1, hb, mb);
}

// sqrt(a) for normal a > 0: m = a 4^-h in [1, 4), Y = 2^32/sqrt(m) from the
// single-precision reciprocal square root, low by at most 2^-20.4 and never high,
// digits and exact remainders as for the division.
static __device__ __forceinline__ double cs_sqrt64(double a) {
  const cs_u32 hi = (cs_u32)__double2hiint(a), lo = (cs_u32)__double2loint(a);
  if (hi - 0x00100000u >= 0x7fe00000u) return cs_sqrt_lib(a);
  const cs_u32 odd = ~(hi >> 20) & 1u;                                 // unbiased exponent odd: m in [2, 4)
  const cs_u32 mh = (hi & 0xfffffu) | 0x100000u;
  const cs_u64 m = cs_pack(mh, lo) << (8u + odd);                      // lsb 2^-60
  const float mf = __uint_as_float(((__funnelshift_l(lo, hi, 3) & 0x7fffffu) | 0x3f800000u) + (odd << 23) + 1u);
  const cs_u32 Y = __float_as_uint(cs_rsqrtf(mf)) * 256u + (0x80000000u - 1024u);
  const cs_u32 s1 = __umulhi(cs_hi32(m << 2), Y);                      // lsb 2^-30
  cs_u64 r = m - cs_wide(s1, s1);                                      // lsb 2^-60
  const cs_u32 q2 = __umulhi(cs_hi32(r << 20), Y);                     // lsb 2^-49
  r = (r << 38) - (cs_wide(s1, q2) << 20) - cs_wide(q2, q2);           // lsb 2^-98
  const cs_u32 q3 = __umulhi(cs_hi32(r), Y);                           // lsb 2^-67
  cs_u64 t = cs_wide(s1, 1u << 23) + ((cs_u64)q2 << 4) + (q3 >> 14);   // lsb 2^-53: 54 bits or one less
  const cs_u64 rem = (m << 46) - cs_mul_low(t, t);                     // lsb 2^-106
  t = (t + (rem > 2 * t ? 2u : 1u)) >> 1;
  const cs_u32 e = ((hi >> 20) + 1021u) >> 1;                           // exponent field - 1
  return __hiloint2double((int)(cs_hi32(t) + (e << 20)), (int)(cs_u32)t);
}
