// Device arithmetic of the libtami kernels: the counter-based momentum sampler, the lattice
// dispersion with its fixed-point cos/sin, the table-driven exponential, the reciprocal and the
// Fermi/Bose values and derivatives of one table segment.  Self-contained (no host headers, plain
// integer types), so that the same text also serves the kernels the library generates and
// compiles at run time for one diagram's table (tami_jit.cpp).  Internal to the library.
#pragma once

namespace tami {
namespace dev {

constexpr int kBlock = 128;                 // threads per block = samples per tile

__device__ __forceinline__ void philox4x32_10(unsigned int c[4], unsigned int k0, unsigned int k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    unsigned int hi0 = __umulhi(0xD2511F53u, c[0]), lo0 = 0xD2511F53u * c[0];
    unsigned int hi1 = __umulhi(0xCD9E8D57u, c[2]), lo1 = 0xCD9E8D57u * c[2];
    unsigned int n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
    k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
  }
}

// [0,1) from 53 bits of two words, u = m 2^-53, then k = 2 pi u - pi with one rounding.  m is
// exact in a double and the powers of two scale exactly, so fma(m, 2 pi 2^-53, -pi) is that
// rounding of the same real number: one FP64 multiply fewer.
__device__ __forceinline__ double to_momentum(unsigned int hi, unsigned int lo) {
  unsigned long long m = ((unsigned long long)hi << 21) | (unsigned long long)(lo >> 11);
  const double pi = 0x1.921fb54442d18p+1;
  return fma(__ull2double_rn(m), 2.0 * pi * 0x1.0p-53, -pi);
}

// ---------------------------------------------------------------------------------------------
// Fixed-point arithmetic.  A warp's FP64 instruction holds this GPU's FP64 unit for 16 clocks of an
// SM (2 lanes a clock), while the integer pipes take a warp instruction every half to one clock, so
// an elementary function in 64-bit fixed point costs a fraction of its FP64 polynomial: the
// reciprocal, the exponential and cos/sin below issue no FP64 instruction.

// (a b) 2^-64 of a, b < 2^63 from three 32-bit products; between 0 and 3 below the exact value.
__device__ __forceinline__ unsigned long long mulhi_trunc(unsigned long long a, unsigned long long b) {
  const unsigned int al = (unsigned int)a, ah = (unsigned int)(a >> 32), bl = (unsigned int)b, bh = (unsigned int)(b >> 32);
  return (unsigned long long)ah * bh + (__umulhi(al, bh) + __umulhi(ah, bl));
}

__device__ __forceinline__ float rcp_estimate(float x) {   // 1/x to about 2^-23, x normal
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// 1/m of m = M 2^-52 in [1, 2): Q 2^-63, Q in [2^62, 2^63), within 2^-61 of 1/m.  From the
// single-precision estimate y0 = Y 2^-24 of 1/m (its argument truncated to 24 bits) the residual
// F = m y0 - 1 is exact in 64-bit integers (|F| < 2^-21, so the product's low 64 bits hold it), and
// 1/m = y0 / (1 + F) = y0 (1 - F + F^2) to F^3 < 2^-63 (Newton's iteration, third order).
__device__ __forceinline__ unsigned long long recip_sig(unsigned long long M) {
  const float x0 = __uint_as_float(((unsigned int)(M >> 29) & 0x7FFFFFu) | 0x3F800001u);
  const float y0 = fmaxf(rcp_estimate(x0), 0.5f);                            // in [1/2, 1)
  const unsigned int Y = (__float_as_uint(y0) & 0x7FFFFFu) | 0x800000u;
  const long long F = (long long)(M * Y);                                     // F 2^76
  const int Fh = (int)(F >> 32);
  const long long G = F - (((long long)Fh * Fh) >> 12);                       // (F - F^2) 2^76
  const long long T = (long long)(int)(G >> 32) * (int)Y + __umulhi((unsigned int)G, Y);   // y0 (F - F^2) 2^68
  return ((unsigned long long)Y << 39) - (unsigned long long)(T >> 5);
}

// sign, 53 significant bits rounded from Q in [2^62, 2^63], and the biased exponent e of Q's
// leading bit 2^62 (1 <= e <= 2046)
__device__ __forceinline__ double pack62(unsigned long long Q, int e, unsigned int sign) {
  const unsigned long long m = (Q + 0x200ull) >> 10;
  return __hiloint2double((int)(((unsigned int)(m >> 32) + ((unsigned int)(e - 1) << 20)) | sign), (int)(unsigned int)m);
}

// ---------------------------------------------------------------------------------------------
// Double-precision multiplication on the integer pipes.  On this GPU the FP64 unit is the
// bottleneck of the evaluation kernels while the integer units sit mostly idle, and the two run
// concurrently.  imul computes the IEEE round-to-nearest-even product of two doubles with 64-bit
// integer arithmetic, bit for bit what DMUL gives, so a kernel can move part of its FP64 work to
// the integer pipes.  The integer fast path covers normal operands with a normal result; zeros,
// subnormals, infinities, NaNs and results that would underflow or overflow take the FP64
// instruction instead, out of line, so that the fast path issues no FP64 instruction at all.
// (Textbook IEEE 754 multiplication: the exact 106-bit product of the significands from four
// 32-bit products, its low half folded into a sticky bit, normalised and rounded.)
static __device__ __noinline__ double dmul_fp64(double a, double b) { return __dmul_rn(a, b); }

// The normal path shared by imul and imul_ftz: the rounded product's bits for normal operands
// whose result is normal (e in [1, 0x7FE]); e, the biased exponent before rounding, says whether
// it is.
__device__ __forceinline__ unsigned long long imul_bits(unsigned long long ua, unsigned long long ub, int ea, int eb,
                                                        int& e) {
  // significands at 2^63 and 2^62: the product's high word h lies in [2^61, 2^63)
  const unsigned long long ma = (ua << 11) | 0x8000000000000000ull, mb = ((ub << 10) & 0x3FFFFFFFFFFFFFFFull) | 0x4000000000000000ull;
  const unsigned int al = (unsigned int)ma, ah = (unsigned int)(ma >> 32), bl = (unsigned int)mb, bh = (unsigned int)(mb >> 32);
  const unsigned long long t0 = (unsigned long long)al * bl;
  const unsigned long long t1 = (unsigned long long)ah * bl + (unsigned int)(t0 >> 32);
  const unsigned long long t2 = (unsigned long long)al * bh + (unsigned int)t1;
  unsigned long long h = (unsigned long long)ah * bh + (unsigned int)(t1 >> 32) + (unsigned int)(t2 >> 32);
  const unsigned int top = (unsigned int)(h >> 62);                 // 1: the product is 2^105 or more
  h <<= 1u - top;                                                   // leading one at bit 62
  h |= (((unsigned int)t2 | (unsigned int)t0) != 0u);               // sticky: ten bits lie under the 53
  h += 0x1FFull + ((unsigned int)(h >> 10) & 1u);                   // half up, ties to even
  e = ea + eb - 1023 + (int)top;
  const unsigned long long m = h >> 10;                             // may carry into bit 53
  const unsigned int sign = (unsigned int)((ua ^ ub) >> 32) & 0x80000000u;
  const unsigned int hi = ((unsigned int)(m >> 32) + ((unsigned int)(e - 1) << 20)) | sign;
  return ((unsigned long long)hi << 32) | (unsigned int)m;
}

__device__ __forceinline__ double imul(double a, double b) {
  const unsigned long long ua = __double_as_longlong(a), ub = __double_as_longlong(b);
  const int ea = (int)(ua >> 52) & 0x7FF, eb = (int)(ub >> 52) & 0x7FF;
  int e;
  const unsigned long long r = imul_bits(ua, ub, ea, eb, e);
  if (ea == 0 || eb == 0 || ea == 0x7FF || eb == 0x7FF || e <= 0 || e >= 0x7FE) return dmul_fp64(a, b);
  return __longlong_as_double(r);
}

// The same product without the FP64 instruction anywhere (no call, no branch: the compiler cannot
// turn it into a predicated DMUL that would take an FP64 issue slot), for code whose products all
// move to the integer pipes.  Normal operands with a normal result: the IEEE product, bit for bit.
// Otherwise flush to zero: a zero or subnormal operand, or a result below the normal range, gives
// a signed zero; a result above the range a signed infinity; an infinite operand a signed
// infinity (a NaN against a zero or subnormal one); a NaN operand a quiet NaN (its payload kept).
__device__ __forceinline__ double imul_ftz(double a, double b) {
  const unsigned long long ua = __double_as_longlong(a), ub = __double_as_longlong(b);
  const int ea = (int)(ua >> 52) & 0x7FF, eb = (int)(ub >> 52) & 0x7FF;
  int e;
  unsigned long long r = imul_bits(ua, ub, ea, eb, e);
  const unsigned long long sign = (ua ^ ub) & 0x8000000000000000ull;
  const bool zero_in = ea == 0 || eb == 0;
  r = (e <= 0 || zero_in) ? sign : r;
  r = (e >= 0x7FF && !zero_in) ? (sign | 0x7FF0000000000000ull) : r;
  const bool a_nan = (ua << 1) > 0xFFE0000000000000ull, b_nan = (ub << 1) > 0xFFE0000000000000ull;
  const bool inf_in = ea == 0x7FF || eb == 0x7FF;
  const unsigned long long special = a_nan ? (ua | 0x0008000000000000ull)
                                   : b_nan ? (ub | 0x0008000000000000ull)
                                   : zero_in ? 0x7FF8000000000000ull : (sign | 0x7FF0000000000000ull);
  r = inf_in ? special : r;
  return __longlong_as_double(r);
}


// 1/d, within 0.502 ulp, in integer arithmetic (recip_sig): 60 clocks of an SM quarter per warp on
// the integer pipes, 215 on the FP64 unit for the hardware's FP64 estimate and a third-order Newton
// step (order 3 on the real axis, 2^21 samples x 256 frequencies: 45.4 -> 39.9 ms).  A zero, subnormal
// or infinite d and a NaN give a NaN (as the Newton step on the hardware's FP64 estimate did); |d| >=
// 2^1022, whose reciprocal is 2^-1022 or subnormal, a signed zero.
__device__ __forceinline__ double rcp(double d) {
  const unsigned int hi = (unsigned int)__double2hiint(d);
  const int ed = (int)(hi >> 20) & 0x7FF;
  const unsigned long long M = ((unsigned long long)((hi & 0xFFFFFu) | 0x100000u) << 32) | (unsigned int)__double2loint(d);
  const double r = pack62(recip_sig(M), 2045 - ed, hi & 0x80000000u);
  const unsigned int odd = ((hi + 0x100000u) & 0x7FE00000u) == 0u ? 0x7FF80000u : (hi & 0x80000000u);
  const bool normal = (unsigned int)(ed - 1) < 2044u;
  return normal ? r : __hiloint2double((int)odd, 0);
}

// cos and sin in fixed point.  |k| is put at 2^-58 (exact for |k| >= 2^-6) and multiplied by
// 2^70/(2 pi) modulo 2^64 turns: the turn fraction to 2^-62.  Its top two bits give the quadrant, the
// angle phi in [0, pi/2] (taken from the other end in odd quadrants) lies within d of a table
// point a = j pi/512, |d| <= pi/1024, and
//   cos phi = C - C (1 - cos d) - S sin d,   sin phi = S - S (1 - cos d) + C sin d
// with 1 - cos d = d^2/2 - d^4/24 and sin d = d - d^3/6 + d^5/120 (W. J. Cody and W. Waite 1980,
// reduction and series; truncation below 2e-18).  Values at 2^-61, a cosine within 1e-17 of the true
// one, a sine within 6e-18 beside the last rounding (3.2 ulp at most); the sine within 3 pi/1024 of a
// multiple of pi comes from sin_near, relatively accurate down to 0.  245 clocks of an SM quarter per
// warp for a cosine, 1200 with an FP64 Taylor series to r^20; a line energy 355 against 1520, with its
// gradients 676 against 2580 (order-5 forward, 2^23 samples, one frequency: 9.6 -> 5.6 ms; order-4
// forward + adjoint, 2^24 samples x 16 frequencies: 78.6 -> 71.9 ms).
__device__ const __align__(16) unsigned long long kTrigTab[514] = {
  0x2000000000000000ull, 0x0000000000000000ull, 0x1fffd8858e8a924dull, 0x003243e1fcce00e2ull,
  0x1fff62169b92db57ull, 0x00648747f37b1e12ull, 0x1ffe9cb44b51a12bull, 0x0096c9b5df1877eaull,
  0x1ffd886084cd0cbbull, 0x00c90aafbd1b33f0ull, 0x1ffc251df1d3f82full, 0x00fb49b98e8e7808ull,
  0x1ffa72effef75c9dull, 0x012d865759455cd1ull, 0x1ff871dadb81df31ull, 0x015fc00d290cd437ull,
  0x1ff621e3796d7de4ull, 0x0191f65f10dd813eull, 0x1ff3830f8d575bcdull, 0x01c428d12c0d7e2dull,
  0x1ff095658e71ad40ull, 0x01f656e79f820dffull, 0x1fed58ecb673c3c3ull, 0x022880269ae13650ull,
  0x1fe9cdad01883a15ull, 0x025aa41259c33ebaull, 0x1fe5f3af2e39406dull, 0x028cc22f24e412b6ull,
  0x1fe1cafcbd5b091aull, 0x02beda0153548318ull, 0x1fdd539ff1f455cbull, 0x02f0eb0d4bab642bull,
  0x1fd88da3d125259eull, 0x0322f4d78536857cull, 0x1fd37914220b8455ull, 0x0354f6e4892b806full,
  0x1fce15fd6da67ad4ull, 0x0386f0b8f3d85a9full, 0x1fc8646cfeb7214cull, 0x03b8e1d975d3f922ull,
  0x1fc26470e19fd348ull, 0x03eac9cad52e61c7ull, 0x1fbc1617e44185fbull, 0x041ca811eea0c749ull,
  0x1fb5797195d74123ull, 0x044e7c33b6bd5dabull, 0x1fae8e8e46cfbad9ull, 0x048045b53b1ef3aeull,
  0x1fa7557f08a516a1ull, 0x04b2041ba3984e89ull, 0x1f9fce55adb2c83eull, 0x04e3b6ec336344eeull,
  0x1f97f924c9099a87ull, 0x05155dac4a4f9677ull, 0x1f8fd5ffae41daceull, 0x0546f7e165f17c7eull,
  0x1f8764fa714ba935ull, 0x0578851122cff195ull, 0x1f7ea629e63d6e6full, 0x05aa04c13d92ac90ull,
  0x1f7599a3a1207761ull, 0x05db7677942fcc52ull, 0x1f6c3f7df5bbb731ull, 0x060cd9ba2719316eull,
  0x1f6297cff75cb02bull, 0x063e2e0f1a6982aeull, 0x1f58a2b1789e8424ull, 0x066f72fcb710d999ull,
  0x1f4e603b0b2f2cceull, 0x06a0a8096c011428ull, 0x1f43d085ff92dc9cull, 0x06d1ccbbcf59c89cull,
  0x1f38f3ac64e588c5ull, 0x0702e09a9f93d8bfull, 0x1f2dc9c9089a9d05ull, 0x0733e32cc4aca189ull,
  0x1f2252f7763ad9b8ull, 0x0764d3f95150c457ull, 0x1f168f53f7205ceeull, 0x0795b287840686d4ull,
  0x1f0a7efb9230d72aull, 0x07c67e5ec857c6acull, 0x1efe220c0b95ec72ull, 0x07f73706b7fb7e2dull,
  0x1ef178a3e473c259ull, 0x0827dc071bfed700ull, 0x1ee482e25a9dbbc9ull, 0x08586ce7ededc80aull,
  0x1ed740e76849633dull, 0x0888e93158fb3bb0ull, 0x1ec9b2d3c3bf8423ull, 0x08b9506bbb28bb92ull,
  0x1ebbd8c8df0b7439ull, 0x08e9a21fa66d9ee9ull, 0x1eadb2e8e7a88d9bull, 0x0919ddd5e1ddb8b3ull,
  0x1e9f4156c62dda5eull, 0x094a03176acf82d4ull, 0x1e9084361df7f273ull, 0x097a116d7601c351ull,
  0x1e817bab4cd10cc6ull, 0x09aa086170c0a8d8ull, 0x1e7227db6a974448ull, 0x09d9e77d020a5bbeull,
  0x1e6288ec48e111efull, 0x0a09ae4a0bb300a2ull, 0x1e529f04729ffc64ull, 0x0a395c52ab8829e0ull,
  0x1e426a4b2bc17e6aull, 0x0a68f1213c73b512ull, 0x1e31eae870ce24c8ull, 0x0a986c40579e11c1ull,
  0x1e212104f686e4c0ull, 0x0ac7cd3ad58fee7full, 0x1e100cca2980abf0ull, 0x0af7139bcf5349acull,
  0x1dfeae622dbe2aacull, 0x0b263eee9f93e309ull, 0x1ded05f7de47d9b5ull, 0x0b554ebee3bf0b59ull,
  0x1ddb13b6ccc23c61ull, 0x0b8442987d22cf57ull, 0x1dc8d7cb4102602dull, 0x0bb31a07920c7b25ull,
  0x1db6526238a09acaull, 0x0be1d4988ee67381ull, 0x1da383a9668987aaull, 0x0c1071d8275561faull,
  0x1d906bcf328d4629ull, 0x0c3ef1535754b169ull, 0x1d7d0b02b8ecf960ull, 0x0c6d5297645257e9ull,
  0x1d696173c9e68ac3ull, 0x0c9b9531de49eb97ull, 0x1d556f52e93eb0a0ull, 0x0cc9b8b0a0deff5dull,
  0x1d4134d14dc939acull, 0x0cf7bca1d476c517ull, 0x1d2cb220e0ef9ec2ull, 0x0d25a093ef50f248ull,
  0x1d17e7743e35dbf7ull, 0x0d536415b69fe4c5ull, 0x1d02d4feb2bd9246ull, 0x0d8106b63fa0048aull,
  0x1ced7af43cc772f1ull, 0x0dae8804f0ae6016ull, 0x1cd7d9898b32f5e1ull, 0x0ddbe791825e809aull,
  0x1cc1f0f3fcfc5c3dull, 0x0e0924ec008f7350ull, 0x1cabc169a0b90071ull, 0x0e363fa4cb800548ull,
  0x1c954b213411f4f7ull, 0x0e63374c98e22f0bull, 0x1c7e8e52233cf31bull, 0x0e900b7474edad63ull,
  0x1c678b3488739b1eull, 0x0ebcbbadc371c4abull, 0x1c5042012b6906eaull, 0x0ee9478a40e62bf8ull,
  0x1c38b2f180bdb0d2ull, 0x0f15ae9c037b1d8full, 0x1c20de3fa971af93ull, 0x0f41f0757c2889e8ull,
  0x1c08c4267255490eull, 0x0f6e0ca977bc6ac4ull, 0x1bf064e15377dd12ull, 0x0f9a02cb1fe833a1ull,
  0x1bd7c0ac6f95299full, 0x0fc5d26dfc4d5cfeull, 0x1bbed7c49380ea07ull, 0x0ff17b25f38907dbull,
  0x1ba5aa673590d260ull, 0x101cfc874c3eb6d9ull, 0x1b8c38d27504e8bbull, 0x10485626ae221a6eull,
  0x1b728345196e3d91ull, 0x1073879922ffed97ull, 0x1b5889fe921404e2ull, 0x109e907417c5e080ull,
  0x1b3e4d3ef5571185ull, 0x10c9704d5d898e9dull, 0x1b23cd470013b42bull, 0x10f426bb2a8e7d91ull,
  0x1b090a581501ff9bull, 0x111eb3541b4b2284ull, 0x1aee04b43c1473b1ull, 0x114915af336ceb3eull,
  0x1ad2bc9e21d510aeull, 0x11734d63dedb48a0ull, 0x1ab7325916c0d46aull, 0x119d5a09f2b9b7edull,
  0x1a9b66290ea1a303ull, 0x11c73b39ae68c86dull, 0x1a7f58529fe69c9aull, 0x11f0f08bbc861aefull,
  0x1a63091b02fae1c3ull, 0x121a799933eb58b1ull, 0x1a4678c8119ac847ull, 0x1243d5fb98ac1f39ull,
  0x1a29a7a0462781deull, 0x126d054cdd12dea9ull, 0x1a0c95eabaf93688ull, 0x12960727629ca82bull,
  0x19ef43ef29af9436ull, 0x12bedb25faf3e9f7ull, 0x19d1b1f5ea80d571ull, 0x12e780e3e8ea1694ull,
  0x19b3e047f38740b4ull, 0x130ff7fce17034e1ull, 0x1995cf2ed80d222full, 0x1338400d0c8e5695ull,
  0x19777ef4c7d741bbull, 0x136058b10659f2b8ull, 0x1958efe48e6dd6aaull, 0x13884185dfeb21ccull,
  0x193a22499263fb4full, 0x13affa292050b93cull, 0x191b166fd49da1ecull, 0x13d78238c58343bfull,
  0x18fbcca3ef940ce9ull, 0x13fed9534556d44eull, 0x18dc45331698cc12ull, 0x1425ff178e6bb15full,
  0x18bc806b151740b5ull, 0x144cf325091dd618ull, 0x189c7e9a4dd4aa77ull, 0x1473b51b9873471dull,
  0x187c400fba2ebeb5ull, 0x149a449b9b0938b6ull, 0x185bc51ae958cc51ull, 0x14c0a145ec000409ull,
  0x183b0e0bff976dd2ull, 0x14e6cabbe3e5e914ull, 0x181a1b33b57acba9ull, 0x150cc09f59a09b2dull,
  0x17f8ece357177099ull, 0x15328292a35595ccull, 0x17d7836cc33db223ull, 0x1558103897513751ull,
  0x17b5df226aafaedeull, 0x157d69348cec9fa3ull, 0x179400574f55e4bdull, 0x15a28d2a5d725056ull,
  0x1771e75f0372612cull, 0x15c77bbe65018c42ull, 0x174f948da8d28d00ull, 0x15ec34958370743cull,
  0x172d0837efff9643ull, 0x1610b7551d2cdedbull, 0x170a42b3176d79c5ull, 0x163503a31c1be911ull,
  0x16e74454eaa8ae89ull, 0x16591925f0783d71ull, 0x16c40d73c1827512ull, 0x167cf78491af1006ull,
  0x16a09e667f3bcc91ull, 0x16a09e667f3bcc91ull, 0x167cf78491af1006ull, 0x16c40d73c1827512ull,
  0x16591925f0783d71ull, 0x16e74454eaa8ae89ull, 0x163503a31c1be911ull, 0x170a42b3176d79c5ull,
  0x1610b7551d2cdedbull, 0x172d0837efff9643ull, 0x15ec34958370743cull, 0x174f948da8d28d00ull,
  0x15c77bbe65018c42ull, 0x1771e75f0372612cull, 0x15a28d2a5d725056ull, 0x179400574f55e4bdull,
  0x157d69348cec9fa3ull, 0x17b5df226aafaedeull, 0x1558103897513751ull, 0x17d7836cc33db223ull,
  0x15328292a35595ccull, 0x17f8ece357177099ull, 0x150cc09f59a09b2dull, 0x181a1b33b57acba9ull,
  0x14e6cabbe3e5e914ull, 0x183b0e0bff976dd2ull, 0x14c0a145ec000409ull, 0x185bc51ae958cc51ull,
  0x149a449b9b0938b6ull, 0x187c400fba2ebeb5ull, 0x1473b51b9873471dull, 0x189c7e9a4dd4aa77ull,
  0x144cf325091dd618ull, 0x18bc806b151740b5ull, 0x1425ff178e6bb15full, 0x18dc45331698cc12ull,
  0x13fed9534556d44eull, 0x18fbcca3ef940ce9ull, 0x13d78238c58343bfull, 0x191b166fd49da1ecull,
  0x13affa292050b93cull, 0x193a22499263fb4full, 0x13884185dfeb21ccull, 0x1958efe48e6dd6aaull,
  0x136058b10659f2b8ull, 0x19777ef4c7d741bbull, 0x1338400d0c8e5695ull, 0x1995cf2ed80d222full,
  0x130ff7fce17034e1ull, 0x19b3e047f38740b4ull, 0x12e780e3e8ea1694ull, 0x19d1b1f5ea80d571ull,
  0x12bedb25faf3e9f7ull, 0x19ef43ef29af9436ull, 0x12960727629ca82bull, 0x1a0c95eabaf93688ull,
  0x126d054cdd12dea9ull, 0x1a29a7a0462781deull, 0x1243d5fb98ac1f39ull, 0x1a4678c8119ac847ull,
  0x121a799933eb58b1ull, 0x1a63091b02fae1c3ull, 0x11f0f08bbc861aefull, 0x1a7f58529fe69c9aull,
  0x11c73b39ae68c86dull, 0x1a9b66290ea1a303ull, 0x119d5a09f2b9b7edull, 0x1ab7325916c0d46aull,
  0x11734d63dedb48a0ull, 0x1ad2bc9e21d510aeull, 0x114915af336ceb3eull, 0x1aee04b43c1473b1ull,
  0x111eb3541b4b2284ull, 0x1b090a581501ff9bull, 0x10f426bb2a8e7d91ull, 0x1b23cd470013b42bull,
  0x10c9704d5d898e9dull, 0x1b3e4d3ef5571185ull, 0x109e907417c5e080ull, 0x1b5889fe921404e2ull,
  0x1073879922ffed97ull, 0x1b728345196e3d91ull, 0x10485626ae221a6eull, 0x1b8c38d27504e8bbull,
  0x101cfc874c3eb6d9ull, 0x1ba5aa673590d260ull, 0x0ff17b25f38907dbull, 0x1bbed7c49380ea07ull,
  0x0fc5d26dfc4d5cfeull, 0x1bd7c0ac6f95299full, 0x0f9a02cb1fe833a1ull, 0x1bf064e15377dd12ull,
  0x0f6e0ca977bc6ac4ull, 0x1c08c4267255490eull, 0x0f41f0757c2889e8ull, 0x1c20de3fa971af93ull,
  0x0f15ae9c037b1d8full, 0x1c38b2f180bdb0d2ull, 0x0ee9478a40e62bf8ull, 0x1c5042012b6906eaull,
  0x0ebcbbadc371c4abull, 0x1c678b3488739b1eull, 0x0e900b7474edad63ull, 0x1c7e8e52233cf31bull,
  0x0e63374c98e22f0bull, 0x1c954b213411f4f7ull, 0x0e363fa4cb800548ull, 0x1cabc169a0b90071ull,
  0x0e0924ec008f7350ull, 0x1cc1f0f3fcfc5c3dull, 0x0ddbe791825e809aull, 0x1cd7d9898b32f5e1ull,
  0x0dae8804f0ae6016ull, 0x1ced7af43cc772f1ull, 0x0d8106b63fa0048aull, 0x1d02d4feb2bd9246ull,
  0x0d536415b69fe4c5ull, 0x1d17e7743e35dbf7ull, 0x0d25a093ef50f248ull, 0x1d2cb220e0ef9ec2ull,
  0x0cf7bca1d476c517ull, 0x1d4134d14dc939acull, 0x0cc9b8b0a0deff5dull, 0x1d556f52e93eb0a0ull,
  0x0c9b9531de49eb97ull, 0x1d696173c9e68ac3ull, 0x0c6d5297645257e9ull, 0x1d7d0b02b8ecf960ull,
  0x0c3ef1535754b169ull, 0x1d906bcf328d4629ull, 0x0c1071d8275561faull, 0x1da383a9668987aaull,
  0x0be1d4988ee67381ull, 0x1db6526238a09acaull, 0x0bb31a07920c7b25ull, 0x1dc8d7cb4102602dull,
  0x0b8442987d22cf57ull, 0x1ddb13b6ccc23c61ull, 0x0b554ebee3bf0b59ull, 0x1ded05f7de47d9b5ull,
  0x0b263eee9f93e309ull, 0x1dfeae622dbe2aacull, 0x0af7139bcf5349acull, 0x1e100cca2980abf0ull,
  0x0ac7cd3ad58fee7full, 0x1e212104f686e4c0ull, 0x0a986c40579e11c1ull, 0x1e31eae870ce24c8ull,
  0x0a68f1213c73b512ull, 0x1e426a4b2bc17e6aull, 0x0a395c52ab8829e0ull, 0x1e529f04729ffc64ull,
  0x0a09ae4a0bb300a2ull, 0x1e6288ec48e111efull, 0x09d9e77d020a5bbeull, 0x1e7227db6a974448ull,
  0x09aa086170c0a8d8ull, 0x1e817bab4cd10cc6ull, 0x097a116d7601c351ull, 0x1e9084361df7f273ull,
  0x094a03176acf82d4ull, 0x1e9f4156c62dda5eull, 0x0919ddd5e1ddb8b3ull, 0x1eadb2e8e7a88d9bull,
  0x08e9a21fa66d9ee9ull, 0x1ebbd8c8df0b7439ull, 0x08b9506bbb28bb92ull, 0x1ec9b2d3c3bf8423ull,
  0x0888e93158fb3bb0ull, 0x1ed740e76849633dull, 0x08586ce7ededc80aull, 0x1ee482e25a9dbbc9ull,
  0x0827dc071bfed700ull, 0x1ef178a3e473c259ull, 0x07f73706b7fb7e2dull, 0x1efe220c0b95ec72ull,
  0x07c67e5ec857c6acull, 0x1f0a7efb9230d72aull, 0x0795b287840686d4ull, 0x1f168f53f7205ceeull,
  0x0764d3f95150c457ull, 0x1f2252f7763ad9b8ull, 0x0733e32cc4aca189ull, 0x1f2dc9c9089a9d05ull,
  0x0702e09a9f93d8bfull, 0x1f38f3ac64e588c5ull, 0x06d1ccbbcf59c89cull, 0x1f43d085ff92dc9cull,
  0x06a0a8096c011428ull, 0x1f4e603b0b2f2cceull, 0x066f72fcb710d999ull, 0x1f58a2b1789e8424ull,
  0x063e2e0f1a6982aeull, 0x1f6297cff75cb02bull, 0x060cd9ba2719316eull, 0x1f6c3f7df5bbb731ull,
  0x05db7677942fcc52ull, 0x1f7599a3a1207761ull, 0x05aa04c13d92ac90ull, 0x1f7ea629e63d6e6full,
  0x0578851122cff195ull, 0x1f8764fa714ba935ull, 0x0546f7e165f17c7eull, 0x1f8fd5ffae41daceull,
  0x05155dac4a4f9677ull, 0x1f97f924c9099a87ull, 0x04e3b6ec336344eeull, 0x1f9fce55adb2c83eull,
  0x04b2041ba3984e89ull, 0x1fa7557f08a516a1ull, 0x048045b53b1ef3aeull, 0x1fae8e8e46cfbad9ull,
  0x044e7c33b6bd5dabull, 0x1fb5797195d74123ull, 0x041ca811eea0c749ull, 0x1fbc1617e44185fbull,
  0x03eac9cad52e61c7ull, 0x1fc26470e19fd348ull, 0x03b8e1d975d3f922ull, 0x1fc8646cfeb7214cull,
  0x0386f0b8f3d85a9full, 0x1fce15fd6da67ad4ull, 0x0354f6e4892b806full, 0x1fd37914220b8455ull,
  0x0322f4d78536857cull, 0x1fd88da3d125259eull, 0x02f0eb0d4bab642bull, 0x1fdd539ff1f455cbull,
  0x02beda0153548318ull, 0x1fe1cafcbd5b091aull, 0x028cc22f24e412b6ull, 0x1fe5f3af2e39406dull,
  0x025aa41259c33ebaull, 0x1fe9cdad01883a15ull, 0x022880269ae13650ull, 0x1fed58ecb673c3c3ull,
  0x01f656e79f820dffull, 0x1ff095658e71ad40ull, 0x01c428d12c0d7e2dull, 0x1ff3830f8d575bcdull,
  0x0191f65f10dd813eull, 0x1ff621e3796d7de4ull, 0x015fc00d290cd437ull, 0x1ff871dadb81df31ull,
  0x012d865759455cd1ull, 0x1ffa72effef75c9dull, 0x00fb49b98e8e7808ull, 0x1ffc251df1d3f82full,
  0x00c90aafbd1b33f0ull, 0x1ffd886084cd0cbbull, 0x0096c9b5df1877eaull, 0x1ffe9cb44b51a12bull,
  0x00648747f37b1e12ull, 0x1fff62169b92db57ull, 0x003243e1fcce00e2ull, 0x1fffd8858e8a924dull,
  0x0000000000000000ull, 0x2000000000000000ull};

// sin k next to a multiple of pi (|k - n pi| < 3 pi/1024, |k| < 32), where a fixed-point value keeps no
// relative accuracy, on the FP64 unit: r = k - n pi (n the integer nearest to k/pi, from one fma against
// 1.5 2^52; n times the first part of pi taken off exactly, the second with one rounding; a double below
// 32 is never closer than 1.2e-16 to a multiple of pi), r (1 - r^2/6 + r^4/120 - r^6/5040) and the sign
// (-1)^n: one rounding of r (none for n = 0) and one of the sum.  One argument in 170 comes here, a warp
// in six for one of its lanes, so that the size of the code counts: a reduction in 64-bit integers,
// called out of line within 5 pi/1024 (0.51 ulp), slowed the generic kernels by its instruction fetches
// (five bubbles, fused, 1.5 10^6 samples x 2 frequencies: 2.00 ms with fixed-point sines throughout,
// 2.44 with it, 2.07 with this; generated kernel, 2^22 x 16: 9.58, 9.81, 9.72 ms).
__device__ __forceinline__ double sin_near(double k) {
  const double nd = fma(k, 0x1.45f306dc9c883p-2, 0x1.8p52), n = nd - 0x1.8p52;
  const double r = fma(-n, 0x1.1a62633145c07p-53, fma(-n, 0x1.921fb54442d18p+1, k)), z = r * r;
  const double v = fma(r * z, fma(z, fma(z, -0x1.a01a01a01a01ap-13, 0x1.1111111111111p-7), -0x1.5555555555555p-3), r);
  return __hiloint2double((int)((unsigned int)__double2hiint(v) ^ ((unsigned int)__double2loint(nd) << 31)), __double2loint(v));
}

struct FixedTrig { long long c, s; bool near; };   // cos and sin times 2^61; near: the sine is sin_near's

// v 2^-S rounded to the nearest double
template <int S>
__device__ __forceinline__ double fixed_to_double(long long v) {
  const unsigned int sign = (unsigned int)(v >> 32) & 0x80000000u;
  const unsigned long long m = (unsigned long long)(v < 0 ? -v : v);
  const int z = __clzll((long long)m);
  const double r = pack62((m << (z & 63)) >> 1, 1086 - S - z, sign);
  return m == 0ull ? 0.0 : r;
}

// |k| < 32 (larger arguments, infinities and NaNs take the FP64 path); NEED_SIN = false leaves s out
template <bool NEED_SIN>
__device__ __forceinline__ FixedTrig trig_fixed(double k) {
  const unsigned int hi = (unsigned int)__double2hiint(k);
  const int ek = (int)(hi >> 20) & 0x7FF;
  const unsigned long long A =
      (((unsigned long long)((hi & 0xFFFFFu) | 0x100000u) << 32) | (unsigned int)__double2loint(k)) << 10;
  const unsigned long long K = A >> min(max(1027 - ek, 0), 63);                 // |k| 2^58, below 2^63
  const unsigned long long T = K * 10ull + mulhi_trunc(K, 0x2F9836E4E441529Full);   // turns 2^64
  const unsigned int q = (unsigned int)(T >> 62);
  unsigned long long phi = T & 0x3FFFFFFFFFFFFFFFull;
  if (q & 1u) phi = 0x4000000000000000ull - phi;
  const unsigned int j = (unsigned int)((phi + 0x20000000000000ull) >> 54);         // 0 .. 256
  const long long dt = (long long)(phi - ((unsigned long long)j << 54));
  const bool neg = dt < 0;
  const unsigned long long ad = (unsigned long long)(neg ? -dt : dt);
  const unsigned long long x = mulhi_trunc(ad << 9, 0x6487ED5110B4611Aull);         // |d| 2^69
  const unsigned long long x2 = mulhi_trunc(x << 2, x << 2);                        // d^2 2^78
  const unsigned int x2h = (unsigned int)(x2 >> 30);                                // d^2 2^48
  const unsigned int x4 = __umulhi(x2h, x2h);                                       // d^4 2^64
  const unsigned long long cm = x2 - ((unsigned long long)__umulhi(x4, 178956971u) << 15);   // (1 - cos d) 2^79
  const unsigned int x3 = __umulhi(x2h, (unsigned int)(x >> 29));                   // d^3 2^56
  const unsigned int w = 2863311531u - __umulhi(x2h, 2185u);                        // (1/6 - d^2/120) 2^34
  const unsigned long long sd = x - ((unsigned long long)__umulhi(x3, w) << 11);    // |sin d| 2^69
  const ulonglong2 cs = __ldg(reinterpret_cast<const ulonglong2*>(kTrigTab) + j);
  const unsigned long long sdn = sd << 2;                                           // 2^71
  const long long Ss = (long long)(mulhi_trunc(cs.y, sdn) >> 7);                    // S |sin d| 2^61
  long long c = (long long)(cs.x - (mulhi_trunc(cs.x, cm) >> 15));
  c = neg ? c + Ss : c - Ss;
  FixedTrig r;
  r.c = (q + 1u) & 2u ? -c : c;
  r.s = 0;
  r.near = NEED_SIN && j <= 1u;
  if (NEED_SIN) {
    const unsigned long long sds = x - (((2ull * x3 + min(x3, 1u)) * w) >> 22);       // sd to more bits, x3's middle
    const long long Cs = (long long)(mulhi_trunc(cs.x, sds << 2) >> 7);
    long long v = (long long)(cs.y - (mulhi_trunc(cs.y, cm) >> 15));
    v = neg ? v - Cs : v + Cs;
    r.s = ((q >> 1) ^ (hi >> 31)) & 1u ? -v : v;
  }
  return r;
}

// Arguments of 32 and above, infinities and NaNs: r = k - n pi on the FP64 unit with pi in three parts
// (a NaN for infinities and NaNs; from about 2^53 on the remainder of 2 pi's nearest double), and
// whether n is odd, which flips both signs.
__device__ __forceinline__ bool trig_far(double k) { return (__double2hiint(k) & 0x7FF00000) > 0x40300000; }
__device__ __forceinline__ double trig_reduce(double k, bool& odd) {
  const double n = rint(k * 0x1.45f306dc9c883p-2);
  double r = fma(-n, 0x1.921fb54442d18p+1, k);
  r = fma(-n, 0x1.1a62633145c07p-53, r);
  r = fma(-n, -0x1.f1976b7ed8fbcp-109, r);
  const bool good = fabs(r) <= 2.0;
  odd = good && ((long long)n & 1) != 0;
  return good ? r : fmod(k, 0x1.921fb54442d18p+2);
}

__device__ __forceinline__ double trig_sin(double k, const FixedTrig& t) {
  return t.near ? sin_near(k) : fixed_to_double<61>(t.s);
}

struct AnyTrig { long long c; double s; };   // cos times 2^61, sin
template <bool NEED_SIN>
__device__ __forceinline__ AnyTrig trig_any(double k, bool& finite) {
  bool odd = false;
  const double r = trig_far(k) ? trig_reduce(k, odd) : k;
  const FixedTrig t = trig_fixed<NEED_SIN>(r);
  AnyTrig a = {t.c, 0.0};
  if (NEED_SIN) a.s = trig_sin(r, t);
  if (odd) { a.c = -a.c; a.s = -a.s; }
  finite = r == r;
  return a;
}

__device__ __forceinline__ double cw_cos(double k) {
  bool finite;
  const double c = fixed_to_double<61>(trig_any<false>(k, finite).c);
  return finite ? c : k - k;
}

__device__ __forceinline__ void cw_sincos(double k, double& s_out, double& c_out) {
  bool finite;
  const AnyTrig t = trig_any<true>(k, finite);
  s_out = finite ? t.s : k - k;
  c_out = finite ? fixed_to_double<61>(t.c) : k - k;
}

// E = mu - eps(k),  eps(k) = -2t(cos kx + cos ky) - 4t' cos kx cos ky, from the fixed-point cosines:
// their sum and product are rounded to double once each
__device__ __forceinline__ double line_energy_of(long long cx, long long cy, double t, double tp, double mu) {
  const double sum = fixed_to_double<61>(cx + cy);
  const unsigned long long ax = (unsigned long long)(cx < 0 ? -cx : cx), ay = (unsigned long long)(cy < 0 ? -cy : cy);
  const long long ap = (long long)mulhi_trunc(ax << 1, ay << 1);
  const double prod = fixed_to_double<60>((cx ^ cy) < 0 ? -ap : ap);
  return fma(4.0 * tp, prod, fma(2.0 * t, sum, mu));
}

// Momenta of 32 and above (a large k_ext): out of line, so that the common path carries no FP64
// reduction.  A momentum that is not finite gives a NaN.
template <bool GRAD>
static __device__ __noinline__ double line_energy_far(double kx, double ky, double t, double tp, double mu, double& gx,
                                                      double& gy) {
  bool fx, fy;
  const AnyTrig x = trig_any<GRAD>(kx, fx), y = trig_any<GRAD>(ky, fy);
  const double bad = fx && fy ? 0.0 : (kx - kx) + (ky - ky);          // 0, or a NaN
  if (GRAD) {
    gx = fma(4.0 * tp, fixed_to_double<61>(y.c), 2.0 * t) * x.s + bad;
    gy = fma(4.0 * tp, fixed_to_double<61>(x.c), 2.0 * t) * y.s + bad;
  }
  return line_energy_of(x.c, y.c, t, tp, mu) + bad;
}

#ifndef TAMI_LINE_INLINE   // the generated kernels call one out-of-line copy
#define TAMI_LINE_INLINE __forceinline__
#endif
__device__ TAMI_LINE_INLINE double line_energy(double kx, double ky, double t, double tp, double mu) {
  double gx, gy;
  if (trig_far(kx) || trig_far(ky)) return line_energy_far<false>(kx, ky, t, tp, mu, gx, gy);
  return line_energy_of(trig_fixed<false>(kx).c, trig_fixed<false>(ky).c, t, tp, mu);
}

// Energy of a line that carries k_ext, with the factors G = (2t + 4t' cos K_perp) sin K of
// dE/dK = -G for both components (one sincos per component); E has line_energy's bits.
__device__ TAMI_LINE_INLINE double line_energy_grad(double kx, double ky, double t, double tp, double mu, double& gx,
                                                   double& gy) {
  if (trig_far(kx) || trig_far(ky)) return line_energy_far<true>(kx, ky, t, tp, mu, gx, gy);
  const FixedTrig x = trig_fixed<true>(kx), y = trig_fixed<true>(ky);
  gx = fma(4.0 * tp, fixed_to_double<61>(y.c), 2.0 * t) * trig_sin(kx, x);
  gy = fma(4.0 * tp, fixed_to_double<61>(x.c), 2.0 * t) * trig_sin(ky, y);
  return line_energy_of(x.c, y.c, t, tp, mu);
}

// e^t and e^t - 1 for t <= 0 in fixed point, after P. T. P. Tang, "Table-driven implementation of the
// exponential function in IEEE floating-point arithmetic", ACM TOMS 15 (1989) 144-157, with a
// 1024-entry table: |t| = (1024 I + j) ln2/1024 + z, 0 <= z < 1.3 ln2/1024, and
//   1 - e^t = 1 - 2^-I (1 - D0),   D0 = V_j + (1 - V_j) p,
// V_j = 1 - 2^(-j/1024) from the table at 2^64, p = 1 - e^-z = z (1 - s), s = z/2 - z^2/6 + z^3/24
// - z^4/120 (truncation below 2^-58 relative).  z is formed at 2^-72 modulo 2^-8, so its bits below
// the integer part of |t| are exact, with a 94-bit ln2/1024; |t| < ln2/1024 takes 1 - e^t = |t| (1 - s)
// on t's own significand, so the result is relatively exact down to t = 0.  180 clocks of an SM
// quarter per warp for e^t, 235 with e^t - 1; an FP64 polynomial after a 256-entry table took 859
// and 1102 (order-5 forward, 2^23 samples, one frequency: 13.3 -> 9.6 ms).  Within 0.51 ulp, e^t - 1
// within 0.75; e^t below 2^-1022 is rounded to a subnormal value with kExpSubnormal, else 0 (for code
// whose products flush those anyway).
constexpr int kExpMinusOne = 1, kExpSubnormal = 2, kFermiExp = kExpSubnormal, kBoseExp = kExpSubnormal | kExpMinusOne;
__device__ const __align__(16) unsigned long long kExpTab[1024] = {
  0x0000000000000000ull, 0x002c58ae3f081ef4ull, 0x0058a9ade372512eull, 0x0084f30041ea698bull,
  0x00b134a6aee1375bull, 0x00dd6ea27e8c909dull, 0x0109a0f504e75c36ull, 0x0135cb9f95b19c24ull,
  0x0161eea3847077b4ull, 0x018e0a02246e45b5ull, 0x01ba1dbcc8ba96a3ull, 0x01e629d4c42a3eddull,
  0x02122e4b695760cbull, 0x023e2b220aa1770dull, 0x026a2059fa2d5ea2ull, 0x02960df489e56110ull,
  0x02c1f3f30b793e8bull, 0x02edd256d05e3818ull, 0x0319a92129cf19acull, 0x0345785368cc4451ull,
  0x03713feede1bb845ull, 0x039cfff4da491f10ull, 0x03c8b866ada5d5a9ull, 0x03f46945a848f685ull,
  0x042012931a0f63b7ull, 0x044bb450529bd103ull, 0x04774e7ea156cdefull, 0x04a2e11f556ecfdbull,
  0x04ce6c33bdd83c0cull, 0x04f9efbd294d71bfull, 0x05256bbce64ed436ull, 0x0550e0344322d4c0ull,
  0x057c4d248dd5fcc6ull, 0x05a7b28f143af7d0ull, 0x05d3107523ea9d90ull, 0x05fe66d80a43fbe0ull,
  0x0629b5b9146c60cbull, 0x0654fd198f4f6488ull, 0x06803cfac79ef37full, 0x06ab755e09d35842ull,
  0x06d6a644a22b458cull, 0x0701cfafdcabe037ull, 0x072cf1a10520c93aull, 0x07580c19671c279bull,
  0x07831f1a4df6b264ull, 0x07ae2aa504cfba9bull, 0x07d92ebad68d352dull, 0x08042b5d0ddbc4e1ull,
  0x082f208cf52ec447ull, 0x085a0e4bd6c04fa2ull, 0x0884f49afc914ed2ull, 0x08afd37bb0697f42ull,
  0x08daaaef3bd77dc7ull, 0x09057af6e830d08dull, 0x09304393fe91f0f5ull, 0x095b04c7c7de557aull,
  0x0985be938cc07b92ull, 0x09b070f895a9f18bull, 0x09db1bf82ad36064ull, 0x0a05bf93943c95b2ull,
  0x0a305bcc19ac8d70ull, 0x0a5af0a302b17bd9ull, 0x0a857e1996a0d743ull, 0x0ab004311c9761edull,
  0x0ada82eadb7933d4ull, 0x0b04fa4819f1c484ull, 0x0b2f6a4a1e73f4e9ull, 0x0b59d2f22f3a1919ull,
  0x0b84344192460221ull, 0x0bae8e398d6107d1ull, 0x0bd8e0db661c1282ull, 0x0c032c2861cfa4dfull,
  0x0c2d7021c59be5a5ull, 0x0c57acc8d668a96full, 0x0c81e21ed8e57c70ull, 0x0cac10251189ac35ull,
  0x0cd636dcc4945164ull, 0x0d005647360c597aull, 0x0d2a6e65a9c09083ull, 0x0d547f396347aad5ull,
  0x0d7e88c3a6004ec6ull, 0x0da88b05b5111e64ull, 0x0dd28600d368c126ull, 0x0dfc79b643bdeda3ull,
  0x0e266627488f733full, 0x0e504b55242443d9ull, 0x0e7a2941188b7d80ull, 0x0ea3ffec679c7413ull,
  0x0ecdcf5852f6baf7ull, 0x0ef797861c022eb6ull, 0x0f21587703eefeacull, 0x0f4b122c4bb5b6aaull,
  0x0f74c4a734174896ull, 0x0f9e6fe8fd9d1612ull, 0x0fc813f2e898fa1bull, 0x0ff1b0c6352552a4ull,
  0x101b466423250a35ull, 0x1044d4cdf243a187ull, 0x106e5c04e1f5391dull, 0x1097dc0a31769ad9ull,
  0x10c154df1fcd4395ull, 0x10eac684ebc76cb7ull, 0x111430fcd3fc15c3ull, 0x113d944816cb0decull,
  0x1166f067f25cfda5ull, 0x1190455da4a3702bull, 0x11b9932a6b58dd16ull, 0x11e2d9cf8400b1e0ull,
  0x120c194e2be75b6full, 0x123551a7a0224f9cull, 0x125e82dd1d9016baull, 0x1287acefe0d85515ull,
  0x12b0cfe1266bd47cull, 0x12d9ebb22a848db9ull, 0x130300642925b216ull, 0x132c0df85e1bb4daull,
  0x1355147004fc54bfull, 0x137e13cc5926a574ull, 0x13a70c0e95c3190full, 0x13cffd37f5c38986ull,
  0x13f8e749b3e34224ull, 0x1421ca450aa708feull, 0x144aa62b345d2861ull, 0x14737afd6b1d7847ull,
  0x149c48bce8c967c0ull, 0x14c50f6ae70c0664ull, 0x14edcf089f5a0dbcull, 0x151687974af1eaa9ull,
  0x153f391822dbc6d1ull, 0x1567e38c5fe99204ull, 0x159086f53ab70b9cull, 0x15b92353eba9cbe7ull,
  0x15e1b8a9aaf14d85ull, 0x160a46f7b086f6c5ull, 0x1632ce3f342e230bull, 0x165b4e816d742c25ull,
  0x1683c7bf93b073a9ull, 0x16ac39fade046c4full, 0x16d4a534835ba348ull, 0x16fd096dba6bc993ull,
  0x172566a7b9b4bd55ull, 0x174dbce3b7809328ull, 0x17760c22e9e39f6cull, 0x179e546686bc7f9dull,
  0x17c695afc3b42398ull, 0x17eecfffd63dd6eeull, 0x18170357f3974a2dull, 0x183f2fb950c89c28ull,
  0x1867552522a46341ull, 0x188f739c9dc7b6acull, 0x18b78b20f69a37b5ull, 0x18df9bb3614e1b05ull,
  0x1907a55511e031deull, 0x192fa8073c17f35eull, 0x1957a3cb138785bfull, 0x197f98a1cb8bc78dull,
  0x19a7868c974c58e9ull, 0x19cf6d8ca9bba4baull, 0x19f74da33596e9eaull, 0x1a1f26d16d66449aull,
  0x1a46f918837cb758ull, 0x1a6ec479a9f8344eull, 0x1a9688f612c1a678ull, 0x1abe468eef8cfad1ull,
  0x1ae5fd4571d9297full, 0x1b0dad1acaf03f06ull, 0x1b3556102be7656aull, 0x1b5cf826c59eed60ull,
  0x1b84935fc8c25773ull, 0x1bac27bc65c85d26ull, 0x1bd3b53dccf2fa1eull, 0x1bfb3be52e4f7546ull,
  0x1c22bbb3b9b669e7ull, 0x1c4a34aa9ecbd0d4ull, 0x1c71a6cb0cff097full, 0x1c991216338ae31aull,
  0x1cc0768d4175a5afull, 0x1ce7d43165911b3dull, 0x1d0f2b03ce7a98ceull, 0x1d367b05aa9b078dull,
  0x1d5dc4382826eddaull, 0x1d85069c751e7860ull, 0x1dac4233bf4d8323ull, 0x1dd376ff344ba292ull,
  0x1dfaa500017c2c97ull, 0x1e21cc37540e41a0ull, 0x1e48eca658fcd5acull, 0x1e70064e3d0eb956ull,
  0x1e9719302cd6a2ddull, 0x1ebe254d54b33726ull, 0x1ee52aa6e0cf12c9ull, 0x1f0c293dfd20d30dull,
  0x1f332113d56b1eefull, 0x1f5a1229953cb01full, 0x1f80fc8067f05c02ull, 0x1fa7e01978ad1caaull,
  0x1fcebcf5f26619d9ull, 0x1ff59316ffdab1f4ull, 0x201c627dcb968300ull, 0x20432b2b7ff17397ull,
  0x2069ed21470fbbe0ull, 0x2090a8604ae1ee7eull, 0x20b75ce9b5250188ull, 0x20de0abeaf625775ull,
  0x2104b1e062efc80eull, 0x212b524ff8efa95cull, 0x2151ec0e9a50d893ull, 0x21787f1d6fcec2fbull,
  0x219f0b7da1f16edcull, 0x21c59130590d8465ull, 0x21ec1036bd445691ull, 0x22128891f683ec0aull,
  0x2238fa432c870810ull, 0x225f654b86d53356ull, 0x2285c9ac2cc2c4e6ull, 0x22ac27664570eafaull,
  0x22d27e7af7cdb3e0ull, 0x22f8ceeb6a9416ccull, 0x231f18b8c44bfcbaull, 0x23455be42b4a4941ull,
  0x236b986ec5b0e36eull, 0x2391ce59b96ebe94ull, 0x23b7fda62c3fe322ull, 0x23de265543ad7775ull,
  0x24044868250dc8abull, 0x242a63dff584536cull, 0x245078bdda01ccbdull, 0x24768702f7442ac8ull,
  0x249c8eb071d6adabull, 0x24c28fc76e11e83bull, 0x24e88a49101bc8d0ull, 0x250e7e367be7a208ull,
  0x25346b90d536338eull, 0x255a52593f95b2daull, 0x25803290de61d3f4ull, 0x25a60c38d4c3d233ull,
  0x25cbdf5245b278fcull, 0x25f1abde53f22c7cull, 0x261771de2214f269ull, 0x263d3152d27a7ab5ull,
  0x2662ea3d8750284aull, 0x26889c9f629119c1ull, 0x26ae487986063215ull, 0x26d3edcd13462158ull,
  0x26f98c9b2bb56d64ull, 0x271f24e4f0867a8full, 0x2744b6ab82b99454ull, 0x276a41f0031cf606ull,
  0x278fc6b3924cd37cull, 0x27b544f750b361b7ull, 0x27dabcbc5e88df90ull, 0x28002e03dbd39e5cull,
  0x282598cee8680a96ull, 0x284afd1ea3e8b481ull, 0x28705af42dc658c9ull, 0x2895b250a53fe92aull,
  0x28bb03352962950cull, 0x28e04da2d909d223ull, 0x2905919ad2df650eull, 0x292acf1e355b69edull,
  0x2950062e1ec45d02ull, 0x297536cbad2f2346ull, 0x299a60f7fe7f12ffull, 0x29bf84b43065fc59ull,
  0x29e4a201606431f9ull, 0x2a09b8e0abc8918full, 0x2a2ec9532fb08c66ull, 0x2a53d35a09082ff7ull,
  0x2a78d6f6548a2e76ull, 0x2a9dd4292ebfe75dull, 0x2ac2caf3b4016ffaull, 0x2ae7bb5700759bf6ull,
  0x2b0ca554301205e1ull, 0x2b3188ec5e9b17b4ull, 0x2b566620a7a4135bull, 0x2b7b3cf2268f1b36ull,
  0x2ba00d61f68d3a9full, 0x2bc4d771329e6e65ull, 0x2be99b20f591ad51ull, 0x2c0e58725a04f0a1ull,
  0x2c330f667a653c87ull, 0x2c57bffe70eea8a0ull, 0x2c7c6a3b57ac6872ull, 0x2ca10e1e4878d3e2ull,
  0x2cc5aba85cfd6facull, 0x2cea42daaeb2f5d5ull, 0x2d0ed3b656e15e22ull, 0x2d335e3c6e9fe68aull,
  0x2d57e26e0ed51ba6ull, 0x2d7c604c5036e11eull, 0x2da0d7d84b4a7a1dull, 0x2dc54913186491b6ull,
  0x2de9b3fdcfa94355ull, 0x2e0e1899890c2326ull, 0x2e3276e75c50467dull, 0x2e56cee861084c3cull,
  0x2e7b209dae96653aull, 0x2e9f6c085c2c5ca6ull, 0x2ec3b12980cba068ull, 0x2ee7f00233454982ull,
  0x2f0c28938a3a2473ull, 0x2f305ade9c1ab98full, 0x2f5486e47f275560ull, 0x2f78aca6497010feull,
  0x2f9ccc2510d4da6bull, 0x2fc0e561eb057ceaull, 0x2fe4f85ded81a955ull, 0x3009051a2d98fe72ull,
  0x302d0b97c06b114bull, 0x30510bd7bae77578ull, 0x307505db31cdc57aull, 0x3098f9a339adab00ull,
  0x30bce730e6e6e73full, 0x30e0ce854da95b36ull, 0x3104afa181f50fffull, 0x31288a86979a3f17ull,
  0x314c5f35a2395aa3ull, 0x31702dafb54315bcull, 0x3193f5f5e3f86cb3ull, 0x31b7b809416aad50ull,
  0x31db73eae07b7f1cull, 0x31ff299bd3dceb9eull, 0x3222d91d2e116699ull, 0x32468270016bd650ull,
  0x326a2595600f9bbbull, 0x328dc28e5bf09acaull, 0x32b1595c06d3429bull, 0x32d4e9ff724c95b1ull,
  0x32f87479afc2322eull, 0x331bf8cbd06a5a0aull, 0x333f76f6e54bfb43ull, 0x3362eefbff3eb811ull,
  0x338660dc2eeaef1bull, 0x33a9cc9884c9c3a1ull, 0x33cd3232112525b1ull, 0x33f091a9e417da4full,
  0x3413eb010d8d83a3ull, 0x34373e389d42a924ull, 0x345a8b51a2c4bfbfull, 0x347dd24d2d723200ull,
  0x34a1132c4c7a6837ull, 0x34c44df00eddd09eull, 0x34e78299836de77aull, 0x350ab129b8cd3f40ull,
  0x352dd9a1bd6f88b2ull, 0x3550fc029f999b02ull, 0x3574184d6d617becull, 0x35972e8334ae67d2ull,
  0x35ba3ea50338d9dcull, 0x35dd48b3e68a940cull, 0x36004cb0ebfea756ull, 0x36234a9d20c17bbcull,
  0x3646427991d0d85dull, 0x366934474bfbeb8eull, 0x368c20075be352e6ull, 0x36af05bacdf92356ull,
  0x36d1e562ae80f134ull, 0x36f4bf00098fd84dull, 0x37179293eb0c83ecull, 0x373a601f5eaf36ebull,
  0x375d27a37001d3bbull, 0x377fe9212a5fe46cull, 0x37a2a49998f6a2b4ull, 0x37c55a0dc6c4fff9ull,
  0x37e8097ebe9bad4eull, 0x380ab2ed8b1d237cull, 0x382d565b36bdab03ull, 0x384ff3c8cbc36417ull,
  0x38728b3754464ea3ull, 0x38951ca7da305244ull, 0x38b7a81b673d4646ull, 0x38da2d9304faf99dull,
  0x38fcad0fbcc93ae2ull, 0x391f269297d9e048ull, 0x39419a1c9f30cf95ull, 0x396407aedba40612ull,
  0x39866f4a55dba087ull, 0x39a8d0f01651e326ull, 0x39cb2ca125534181ull, 0x39ed825e8afe6678ull,
  0x3a0fd2294f443c27ull, 0x3a321c0279e7f3d1ull, 0x3a545feb127f0dd2ull, 0x3a769de420716182ull,
  0x3a98d5eeaaf92523ull, 0x3abb080bb922f5c4ull, 0x3add343c51cddf2dull, 0x3aff5a817bab63beull,
  0x3b217adc3d3f8456ull, 0x3b43954d9ce0c831ull, 0x3b65a9d6a0b844d0ull, 0x3b87b8784ec1a5d0ull,
  0x3ba9c133accb34cdull, 0x3bcbc409c075e13full, 0x3bedc0fb8f35484full, 0x3c0fb80a1e4fbcbaull,
  0x3c31a93672de4ea3ull, 0x3c53948191ccd36aull, 0x3c7579ec7fd9ed87ull, 0x3c97597841971458ull,
  0x3cb93325db689bf9ull, 0x3cdb06f65185bd14ull, 0x3cfcd4eaa7f89cafull, 0x3d1e9d03e29e5401ull,
  0x3d405f430526f837ull, 0x3d621ba91315a249ull, 0x3d83d2370fc076c0ull, 0x3da582edfe50ad7eull,
  0x3dc72dcee1c2998dull, 0x3de8d2dabce5b0dfull, 0x3e0a7212925c9417ull, 0x3e2c0b77649d164cull,
  0x3e4d9f0a35f044cdull, 0x3e6f2ccc08726ee1ull, 0x3e90b4bdde132d88ull, 0x3eb236e0b8956b3cull,
  0x3ed3b335998f6baaull, 0x3ef529bd826ad36full, 0x3f169a797464afd8ull, 0x3f38056a708d7e94ull,
  0x3f596a9177c93573ull, 0x3f7ac9ef8acf4a18ull, 0x3f9c2385aa2ab9aeull, 0x3fbd7754d63a10a2ull,
  0x3fdec55e0f2f7250ull, 0x40000da25510a0b4ull, 0x40215022a7b70421ull, 0x40428ce006cfb2e7ull,
  0x4063c3db71db7908ull, 0x4084f515e82edfdeull, 0x40a6209068f235cbull, 0x40c7464bf32195deull,
  0x40e86649858cef7dull, 0x4109808a1ed80e0eull, 0x412a950ebd7aa09aull, 0x414ba3d85fc0416full,
  0x416cace803c87dc8ull, 0x418db03ea786dd6cull, 0x41aeaddd48c2ea4cull, 0x41cfa5c4e5183825ull,
  0x41f097f679f66c1eull, 0x4211847304a14460ull, 0x42326b3b82309fb7ull, 0x42534c50ef908524ull,
  0x427427b449812b7dull, 0x4294fd668c970100ull, 0x42b5cd68b53ab2e8ull, 0x42d697bbbfa93502ull,
  0x42f75c60a7f3c941ull, 0x43181b586a000751ull, 0x4338d4a40187e424ull, 0x435988446a19b981ull,
  0x437a363a9f184d97ull, 0x439ade879bbada82ull, 0x43bb812c5b0d15deull, 0x43dc1e29d7ef3849ull,
  0x43fcb5810d1604f3ull, 0x441d4732f50ad11full, 0x443dd3408a2b8badull, 0x445e59aac6aac49cull,
  0x447eda72a48fb491ull, 0x449f55991db64454ull, 0x44bfcb1f2bcf1454ull, 0x44e03b05c85f8426ull,
  0x4500a54decc1ba05ull, 0x452109f89224aa48ull, 0x45416906b18c1ee7ull, 0x4561c27943d0beedull,
  0x4582165141a015f7ull, 0x45a2648fa37c9ba8ull, 0x45c2ad3561bdbb1full, 0x45e2f043748fda71ull,
  0x46032dbad3f46215ull, 0x4623659c77c1c45full, 0x464397e957a384e9ull, 0x4663c4a26b1a400bull,
  0x4683ebc8a97bb241ull, 0x46a40d5d09f2bfa1ull, 0x46c42960837f7b3full, 0x46e43fd40cf72e9eull,
  0x470450b89d046117ull, 0x47245c0f2a26df40ull, 0x474461d8aab3c255ull, 0x4764621614d5779dull,
  0x47845cc85e8bc7ccull, 0x47a451f07dabde6cull, 0x47c4418f67e05137ull, 0x47e42ba612a9277eull,
  0x48041035735be184ull, 0x4823ef3e7f237fdeull, 0x4843c8c22b008ad1ull, 0x48639cc16bc919a9ull,
  0x48836b3d3628da17ull, 0x48a334367ea11789ull, 0x48c2f7ae3988c280ull, 0x48e2b5a55b0c77e9ull,
  0x49026e1cd72e886full, 0x49222115a1c6ffd1ull, 0x4941ce90ae83ac34ull, 0x4961768ef0e82573ull,
  0x498119115c4dd471ull, 0x49a0b618e3e3fa66ull, 0x49c04da67aafb82dull, 0x49dfdfbb138c1590ull,
  0x49ff6c57a12a0894ull, 0x4a1ef37d16107cc2ull, 0x4a3e752c649c5a6cull, 0x4a5df1667f008dfbull,
  0x4a7d682c57460f2eull, 0x4a9cd97edf4be864ull, 0x4abc455f08c73ddcull, 0x4adbabcdc54354f7ull,
  0x4afb0ccc06219b7cull, 0x4b1a685abc99aed2ull, 0x4b39be7ad9b96345ull, 0x4b590f2d4e64cb3dull,
  0x4b785a730b563e80ull, 0x4b97a04d011e6165ull, 0x4bb6e0bc20242c13ull, 0x4bd61bc158a4f1b8ull,
  0x4bf5515d9ab467bfull, 0x4c148191d63cad05ull, 0x4c33ac5efafe510dull, 0x4c52d1c5f8905b35ull,
  0x4c71f1c7be6051e8ull, 0x4c910c653bb241ccull, 0x4cb0219f5fa0c4f2ull, 0x4ccf3177191d0a05ull,
  0x4cee3bed56eedb77ull, 0x4d0d410307b4a6abull, 0x4d2c40b919e38323ull, 0x4d4b3b107bc739a2ull,
  0x4d6a300a1b824b5cull, 0x4d891fa6e70df918ull, 0x4da809e7cc3a4a54ull, 0x4dc6eecdb8ae146full,
  0x4de5ce5999e701c5ull, 0x4e04a88c5d3998d5ull, 0x4e237d66efd14361ull, 0x4e424cea3eb0558bull,
  0x4e61171736b014f7ull, 0x4e7fdbeec480bfe2ull, 0x4e9e9b71d4a99443ull, 0x4ebd55a15388d6e2ull,
  0x4edc0a7e2d53da70ull, 0x4efaba094e1706a5ull, 0x4f196443a1b5df4eull, 0x4f38092e13eb0b69ull,
  0x4f56a8c990485c37ull, 0x4f7543170236d44bull, 0x4f93d81754f6aea4ull, 0x4fb267cb739f65b6ull,
  0x4fd0f234491fba7cull, 0x4fef7752c03dbb87ull, 0x500df727c396cc07ull, 0x502c71b43d9faaddull,
  0x504ae6f918a4799full, 0x506956f73ec8c3a3ull, 0x5087c1af9a078509ull, 0x50a62723143331c0ull,
  0x50c4875296f5bc8bull, 0x50e2e23f0bd09e06ull, 0x510137e95c1cdba9ull, 0x511f8852710b0ec9ull,
  0x513dd37b33a36b9bull, 0x515c19648cc5c82full, 0x517a5a0f6529a372ull, 0x5198957ca55e2c2aull,
  0x51b6cbad35ca47f2ull, 0x51d4fca1feac9a32ull, 0x51f3285be81b8b1dull, 0x52114edbda054ea3ull,
  0x522f7022bc2feb6full, 0x524d8c31763941d6ull, 0x526ba308ef9712d1ull, 0x5289b4aa0f9706ecull,
  0x52a7c115bd5eb53aull, 0x52c5c84cdfebaa47ull, 0x52e3ca505e136f05ull, 0x5301c7211e838fbeull,
  0x531fbec007c1a2fcull, 0x533db12e002b507cull, 0x535b9e6bedf65813ull, 0x5379867ab730989aull,
  0x5397695b41c016d7ull, 0x53b5470e73630462ull, 0x53d31f9531afc68full, 0x53f0f2f06214fd4full,
  0x540ec120e9d98a17ull, 0x542c8a27ae1c96bfull, 0x544a4e0593d59c65ull, 0x54680cbb7fd46a50ull,
  0x5485c64a56c12cc9ull, 0x54a37ab2fd1c73fdull, 0x54c129f6573f3adaull, 0x54ded415495aede6ull,
  0x54fc7910b779721full, 0x551a18e9857d2bd0ull, 0x5537b3a097210568ull, 0x55554936cff87656ull,
  0x5572d9ad136f89d7ull, 0x5590650444cae5d0ull, 0x55adeb3d4727d1a1ull, 0x55cb6c58fd7c3cf1ull,
  0x55e8e8584a96c687ull, 0x56065f3c111ec312ull, 0x5623d105339443fdull, 0x56413db494501e38ull,
  0x565ea54b1583f108ull, 0x567c07c9993a2cccull, 0x56996531015619cfull, 0x56b6bd822f93df07ull,
  0x56d410be058888e5ull, 0x56f15ee564a21014ull, 0x570ea7f92e276042ull, 0x572bebfa43385ee5ull,
  0x57492ae984cdf1f7ull, 0x576664c7d3ba06c0ull, 0x5783999610a79890ull, 0x57a0c9551c1ab77full,
  0x57bdf405d6708f2full, 0x57db19a91fdf6d83ull, 0x57f83a3fd876c95full, 0x581555cae01f4960ull,
  0x58326c4b169aca96ull, 0x584f7dc15b84673dull, 0x586c8a2e8e507d72ull, 0x588991938e4cb5e9ull,
  0x58a693f13aa00aa5ull, 0x58c39148724acda5ull, 0x58e0899a1426af9eull, 0x58fd7ce6fee6c6a4ull,
  0x591a6b30111794e2ull, 0x59375476291f0f43ull, 0x595438ba253ca421ull, 0x597117fce38941f2ull,
  0x598df23f41f75df4ull, 0x59aac7821e52fad7ull, 0x59c797c65641af64ull, 0x59e4630cc742ad28ull,
  0x5a0129564eaec716ull, 0x5a1deaa3c9b87833ull, 0x5a3aa6f6156bea35ull, 0x5a575e4e0eaefc28ull,
  0x5a7410ac92414912ull, 0x5a90be127cbc2e91ull, 0x5aad6680aa92d37cull, 0x5aca09f7f8122e82ull,
  0x5ae6a87941610cc7ull, 0x5b03420562801880ull, 0x5b1fd69d3749df90ull, 0x5b3c66419b72da21ull,
  0x5b58f0f36a89713bull, 0x5b7576b37ff6055full, 0x5b91f782b6faf51cull, 0x5bae7361eab4a3a4ull,
  0x5bcaea51f6197f62ull, 0x5be75c53b3fa088bull, 0x5c03c967ff00d7b4ull, 0x5c20318fb1b2a45cull,
  0x5c3c94cba66e4b84ull, 0x5c58f31cb76cd638ull, 0x5c754c83bec18020ull, 0x5c91a1019659be07ull,
  0x5cadf09717fd446dull, 0x5cca3b451d4e0e0full, 0x5ce6810c7fc8626cull, 0x5d02c1ee18c2dc52ull,
  0x5d1efdeac16e7062ull, 0x5d3b350352d67396ull, 0x5d576738a5e0a1c7ull, 0x5d73948b934d242eull,
  0x5d8fbcfcf3b697e7ull, 0x5dabe08d9f921475ull, 0x5dc7ff3e6f2f323bull, 0x5de419103ab81104ull,
  0x5e002e03da315e78ull, 0x5e1c3e1a257a5c9full, 0x5e384953f44ce858ull, 0x5e544fb21e3d7fd7ull,
  0x5e7051357abb491cull, 0x5e8c4ddee110186cull, 0x5ea845af286076c7ull, 0x5ec438a727aba85eull,
  0x5ee026c7b5cbb309ull, 0x5efc1011a97564b9ull, 0x5f17f485d93859eeull, 0x5f33d4251b7f0421ull,
  0x5f4faef0468eb03eull, 0x5f6b84e830878d0aull, 0x5f87560daf64b197ull, 0x5fa3226198fc23b0ull,
  0x5fbee9e4c2fede42ull, 0x5fdaac9802f8d7caull, 0x5ff66a7c2e5108bbull, 0x601223921a4971ecull,
  0x602dd7da9bff22faull, 0x60498756886a40b0ull, 0x60653206b45e0b6dull, 0x6080d7ebf488e587ull,
  0x609c79071d7459afull, 0x60b8155903852153ull, 0x60d3ace27afb2afcull, 0x60ef3fa457f1a0b1ull,
  0x610acd9f6e5eee52ull, 0x612656d49214c7fbull, 0x6141db4496c0305bull, 0x615d5af04fe97f0full,
  0x6178d5d890f46701ull, 0x61944bfe2d1ffcbdull, 0x61afbd61f786bcc9ull, 0x61cb2a04c31e9200ull,
  0x61e691e762b8dbe0ull, 0x6201f50aa90274e7ull, 0x621d536f6883b8e0ull, 0x6238ad1673a08b3aull,
  0x625402009c985d56ull, 0x626f522eb58634daull, 0x628a9da19060b1fdull, 0x62a5e459fefa15d7ull,
  0x62c12658d30048afull, 0x62dc639eddfce045ull, 0x62f79c2cf155261eull, 0x6312d003de4a1dcbull,
  0x632dff2475f88b35ull, 0x6349298f8958f8e4ull, 0x63644f45e93fbe42ull, 0x637f7048665d05e6ull,
  0x639a8c97d13cd3d3ull, 0x63b5a434fa470bbcull, 0x63d0b720b1bf774cull, 0x63ebc55bc7c5cc5cull,
  0x6406cee70c55b33full, 0x6421d3c34f46ccf7ull, 0x643cd3f1604cb978ull, 0x6457cf720ef71de5ull,
  0x6472c6462ab1aac7ull, 0x648db86e82c4224dull, 0x64a8a5ebe6525e82ull, 0x64c38ebf245c5785ull,
  0x64de72e90bbe29c3ull, 0x64f9526a6b301c2cull, 0x65142d441146a665ull, 0x652f0376cc727703ull,
  0x6549d5036b0079b6ull, 0x6564a1eabb19dd80ull, 0x657f6a2d8ac41ae6ull, 0x659a2dcca7e0fa1cull,
  0x65b4ecc8e02e9936ull, 0x65cfa72301477256ull, 0x65ea5cdbd8a261d9ull, 0x66050df43392ac7full,
  0x661fba6cdf48059bull, 0x663a6246a8ce9536ull, 0x665505825d0efe3cull, 0x666fa420c8ce64a1ull,
  0x668a3e22b8ae7389ull, 0x66a4d388f92d6369ull, 0x66bf645456a60031ull, 0x66d9f0859d4faf69ull,
  0x66f4781d993e7656ull, 0x670efb1d1663001dull, 0x67297984e08aa3dbull, 0x6743f355c35f6aceull,
  0x675e68908a68166aull, 0x6778d9360108267aull, 0x67934546f27fdf3aull, 0x67adacc429ec4f73ull,
  0x67c80fae72475691ull, 0x67e26e069667aabfull, 0x67fcc7cd6100defdull, 0x68171d039ca36936ull,
  0x68316daa13bca855ull, 0x684bb9c19096ea58ull, 0x6866014add597267ull, 0x68804446c4087ee2ull,
  0x689a82b60e854f72ull, 0x68b4bc99868e2b1cull, 0x68cef1f1f5be664dull, 0x68e922c0258e68ebull,
  0x69034f04df53b45dull, 0x691d76c0ec40e99bull, 0x693799f51565cf35ull, 0x6951b8a223af5761ull,
  0x696bd2c8dfe7a600ull, 0x6985e86a12b616a6ull, 0x699ff986849f42a4ull, 0x69ba061efe050706ull,
  0x69d40e3447268aa0ull, 0x69ee11c72820440cull, 0x6a0810d868ebffacull, 0x6a220b68d160e5b0ull,
  0x6a3c017929338011ull, 0x6a55f30a37f5c092ull, 0x6a6fe01cc51706c0ull, 0x6a89c8b197e425edull,
  0x6aa3acc977876b2bull, 0x6abd8c652b08a34bull, 0x6ad76785794d20d4ull, 0x6af13e2b2917c1fbull,
  0x6b0b10570108f69full, 0x6b24de09c79ec63cull, 0x6b3ea7444334d5e1ull, 0x6b586c073a046e2aull,
  0x6b722c537224812dull, 0x6b8be829b189b06full, 0x6ba59f8abe0652d8ull, 0x6bbf52775d4a7aa3ull,
  0x6bd900f054e3fb4aull, 0x6bf2aaf66a3e6f79ull, 0x6c0c508a62a33efbull, 0x6c25f1ad0339a4a4ull,
  0x6c3f8e5f1106b43full, 0x6c5926a150ed6078ull, 0x6c72ba7487ae80c4ull, 0x6c8c49d979e8d74dull,
  0x6ca5d4d0ec1916d4ull, 0x6cbf5b5ba299e89eull, 0x6cd8dd7a61a3f254ull, 0x6cf25b2ded4ddbebull,
  0x6d0bd477098c5584ull, 0x6d2549567a321d51ull, 0x6d3eb9cd02f00577ull, 0x6d5825db6754f9ebull,
  0x6d718d826ace0654ull, 0x6d8af0c2d0a65be8ull, 0x6da44f9d5c07574cull, 0x6dbdaa12cff8866aull,
  0x6dd70023ef5fae53ull, 0x6df051d17d00d117ull, 0x6e099f1c3b7e339cull, 0x6e22e804ed586378ull,
  0x6e3c2c8c54ee3ccaull, 0x6e556cb3347cf00cull, 0x6e6ea87a4e2007ebull, 0x6e87dfe263d16f1dull,
  0x6ea112ec3769762dull, 0x6eba41988a9ed956ull, 0x6ed36be81f06c64dull, 0x6eec91dbb614e218ull,
  0x6f05b374111b4ed5ull, 0x6f1ed0b1f14ab18full, 0x6f37e99617b23807ull, 0x6f50fe21453f9e83ull,
  0x6f6a0e543abf3595ull, 0x6f831a2fb8dbe7eaull, 0x6f9c21b4801f4011ull, 0x6fb524e350f16e41ull,
  0x6fce23bceb994e24ull, 0x6fe71e42103c6c98ull, 0x700014737edf0d7bull, 0x70190651f7643168ull,
  0x7031f3de398d9b7full, 0x704add1904fbd724ull, 0x7063c203192e3dc3ull, 0x707ca29d3582fc8eull,
  0x70957ee819371a3cull, 0x70ae56e483667cc8ull, 0x70c72a93330bef2dull, 0x70dff9f4e7012725ull,
  0x70f8c50a5dfecae0ull, 0x71118bd4569c76c1ull, 0x712a4e538f50c317ull, 0x71430c88c67149d2ull,
  0x715bc674ba32ac40ull, 0x71747c1828a898bdull, 0x718d2d73cfc5d06bull, 0x71a5da886d5c2ce9ull,
  0x71be8356bf1ca5ffull, 0x71d727df82975757ull, 0x71efc823753b862dull, 0x720864235457a6faull,
  0x7220fbdfdd19632aull, 0x72398f59cc8d9ec8ull, 0x72521e91dfa07e28ull, 0x726aa988d31d6b98ull,
  0x7283303f63af1d08ull, 0x729bb2b64ddf99b8ull, 0x72b430ee4e183fdcull, 0x72ccaae820a1ca49ull,
  0x72e520a481a4561aull, 0x72fd92242d276859ull, 0x7315ff67df11f3a0ull, 0x732e6870532a5dc2ull,
  0x7346cd3e4516856bull, 0x735f2dd2705bc7c4ull, 0x73778a2d905f0617ull, 0x738fe2506064ab69ull,
  0x73a8363b9b90b222ull, 0x73c085effce6a9a4ull, 0x73d8d16e3f49bbecull, 0x73f118b71d7cb331ull,
  0x74095bcb5221ff7bull, 0x74219aab97bbbc40ull, 0x7439d558a8abb5ffull, 0x74520bd33f336fd5ull,
  0x746a3e1c15742919ull, 0x74826c33e56ee2f1ull, 0x749a961b690465e8ull, 0x74b2bbd359f54781ull,
  0x74cadd5c71e1efceull, 0x74e2fab76a4a9f02ull, 0x74fb13e4fc8f7302ull, 0x751328e5e1f06cf7ull,
  0x752b39bad38d76dcull, 0x754346648a666912ull, 0x755b4ee3bf5b0fe8ull, 0x757353392b2b312dull,
  0x758b5365867691b9ull, 0x75a34f6989bcfafbull, 0x75bb4745ed5e4081ull, 0x75d33afb699a4581ull,
  0x75eb2a8ab6910266ull, 0x760315f48c428a50ull, 0x761afd39a28f10a2ull, 0x7632e05ab136ee80ull,
  0x764abf586fdaa85cull, 0x76629a3395faf372ull, 0x767a70ecdaf8bb4eull, 0x76924384f615274full,
  0x76aa11fc9e71a023ull, 0x76c1dc548b0fd54eull, 0x76d9a28d72d1c2a2ull, 0x76f164a80c79b5c0ull,
  0x770922a50eaa5395ull, 0x7720dc852fe69dd4ull, 0x773892492691f874ull, 0x775043f1a8f02f28ull,
  0x7767f17f6d257ad9ull, 0x777f9af32936871dull, 0x7797404d930877afull, 0x77aee18f6060ede7ull,
  0x77c67eb946e60e2cull, 0x77de17cbfc1e8569ull, 0x77f5acc835718e84ull, 0x780d3daea826f7cdull,
  0x7824ca800967286eull, 0x783c533d0e3b25e3ull, 0x7853d7e66b8c9960ull, 0x786b587cd625d548ull,
  0x7882d50102b1da94ull, 0x789a4d73a5bc5e45ull, 0x78b1c1d573b1cecfull, 0x78c9322720df5980ull,
  0x78e09e696172eff0ull, 0x78f8069ce97b4d64ull, 0x790f6ac26ce7fc3dull, 0x7926cada9f895b58ull,
  0x793e26e63510a378ull, 0x79557ee5e10fecaeull, 0x796cd2da56fa33b6ull, 0x798422c44a235f64ull,
  0x799b6ea46dc045fcull, 0x79b2b67b74e6b29dull, 0x79c9fa4a128d6a9dull, 0x79e13a10f98c32e8ull,
  0x79f875d0dc9bd561ull, 0x7a0fad8a6e56263full, 0x7a26e13e6136096cull, 0x7a3e10ed679777dbull,
  0x7a553c9833b784ebull, 0x7a6c643f77b463bcull, 0x7a8387e3e58d6c8aull, 0x7a9aa7862f232203ull,
  0x7ab1c327063736a3ull, 0x7ac8dac71c6c9206ull, 0x7adfee6723475640ull, 0x7af6fe07cc2ce530ull,
  0x7b0e09a9c863e5d7ull, 0x7b25114dc91449a5ull, 0x7b3c14f47f4751d0ull, 0x7b53149e9be794a4ull,
  0x7b6a104ccfc102d0ull, 0x7b8107ffcb80ecb9ull, 0x7b97fbb83fb607c4ull, 0x7baeeb76dcd073a9ull,
  0x7bc5d73c5321bfbaull, 0x7bdcbf0952dcf02full, 0x7bf3a2de8c168375ull, 0x7c0a82bcaec47771ull,
  0x7c215ea46abe4eceull, 0x7c3836966fbd1643ull, 0x7c4f0a936d5b69d8ull, 0x7c65da9c13157a30ull,
  0x7c7ca6b1104911c9ull, 0x7c936ed314359a44ull, 0x7caa3302cdfc21a6ull, 0x7cc0f340ec9f5f9bull,
  0x7cd7af8e1f03bab9ull, 0x7cee67eb13ef4dbdull, 0x7d051c587a09eccdull, 0x7d1bccd6ffdd2ab6ull,
  0x7d32796753d45e29ull, 0x7d49220a243ca6f9ull, 0x7d5fc6c01f44f358ull, 0x7d766789f2fe050dull,
  0x7d8d04684d5a76b4ull, 0x7da39d5bdc2ec0f4ull, 0x7dba32654d313fb8ull, 0x7dd0c3854dfa3765ull,
  0x7de750bc8c03da14ull, 0x7dfdda0bb4aa4cc4ull, 0x7e145f73752bac90ull, 0x7e2ae0f47aa813e3ull,
  0x7e415e8f72219faaull, 0x7e57d845087c7488ull, 0x7e6e4e15ea7ec403ull, 0x7e84c002c4d0d1b9ull,
  0x7e9b2e0c43fcf88dull, 0x7eb19833146fafd3ull, 0x7ec7fe77e2779084ull, 0x7ede60db5a455a63ull,
  0x7ef4bf5e27ebf92cull, 0x7f0b1a00f76089c1ull, 0x7f2170c4747a5f51ull, 0x7f37c3a94af30880ull,
  0x7f4e12b026665494ull, 0x7f645dd9b2525896ull, 0x7f7aa5269a17747cull, 0x7f90e89788f85850ull,
  0x7fa7282d2a1a094full, 0x7fbd63e82883e713ull, 0x7fd39bc92f1fb0afull, 0x7fe9cfd0e8b989d8ull};

template <int FORM>
__device__ __forceinline__ double exp_neg(double t, double& em) {
  constexpr bool NEED_EM = (FORM & kExpMinusOne) != 0;
  const unsigned int hi = (unsigned int)__double2hiint(t) & 0x7FFFFFFFu, lo = (unsigned int)__double2loint(t);
  const int et = (int)(hi >> 20);
  const unsigned long long M = ((unsigned long long)((hi & 0xFFFFFu) | 0x100000u) << 32) | lo;
  // k = 1024 I + j from |t| in single precision, clamped to [2^-15, 1024]: below the true quotient
  // by 0.1 to 1.3 (0 where |t| is small)
  const unsigned int hc = min(max(hi, 0x3F000000u), 0x40900000u);
  const float tf = __uint_as_float(__funnelshift_l(lo, hc - 0x38000000u, 3));
  const int k = max(__float_as_int(fmaf(tf, 1477.3197f, -0.7f) + 12582912.0f) - 0x4B400000, 0);
  const int sh = et - 1003;
  const unsigned long long tfix = (M << min(max(sh, 0), 63)) >> min(max(-sh, 0), 63);
  const unsigned long long z = tfix - ((unsigned long long)(unsigned int)k * 0x2C5C85FDF473DE6Aull +
                                       __umulhi((unsigned int)k, 0xF278ECE6u));               // z 2^72
  const unsigned int zh = (unsigned int)(z >> 30);                                            // z 2^42
  const unsigned long long z2 = mulhi_trunc(z << 1, z << 1);                                  // z^2 2^82
  const unsigned int z2h = (unsigned int)(z2 >> 30);                                          // z^2 2^52
  const unsigned int v = __umulhi(zh, 2863311531u) - __umulhi(z2h, 559241u);                  // (z/24 - z^2/120) 2^46
  const unsigned long long corr = mulhi_trunc(z2, 0x2AAAAAAAAAAAAAABull) -
                                  ((unsigned long long)__umulhi(z2h, v) << 16);               // (z^2/6 - z^2 v) 2^82
  const unsigned long long s = z - (corr >> 9);                                               // s 2^73
  const unsigned long long p = z - (mulhi_trunc(z, s) >> 9);                                  // p 2^72
  const unsigned int j = (unsigned int)k & 1023u;
  const int I = k >> 10;
  const unsigned long long V = __ldg(&kExpTab[j]);
  const unsigned long long D0 = V + ((p - mulhi_trunc(V, p) + 0x80ull) >> 8);                 // (1 - e^-(|t| mod ln2)) 2^64
  unsigned long long y = 0x8000000000000000ull - (D0 >> 1);                                   // in (2^62 (1 - 2^-10), 2^63]
  const bool low = y < 0x4000000000000000ull;
  y = low ? y << 1 : y;
  const int ey = 1022 - I - (low ? 1 : 0);
  double r = pack62(y, ey, 0u);
  const bool big = hi >= 0x40900000u;                                                         // |t| >= 1024, NaN: ey < 1
  const bool nan = hi > 0x7FF00000u || (hi == 0x7FF00000u && lo != 0u);
  if (!(FORM & kExpSubnormal)) {
    r = ey < 1 ? (nan ? t : 0.0) : r;
  } else if (ey < 1) {                                                                        // y 2^(ey - 11) of 2^-1074
    r = nan ? t : 0.0;
    if (ey > -53 && !big) r = __longlong_as_double((long long)((y + (1ull << (10 - ey))) >> (11 - ey)));
  }
  if (NEED_EM) {
    // 1 - e^t: leading bit at 2^63 after the shift, exponent e1 of that bit
    const unsigned long long D1 = 0ull - (((0ull - D0) >> min(I, 63)) | 1ull);
    const unsigned long long Mt = M << 10;
    unsigned long long D = I > 0 ? D1 : D0;
    D = k == 0 ? (Mt << 1) - (mulhi_trunc(Mt, s) >> 8) : D;
    const int c = __clz((int)(D >> 32));
    const double d = pack62((D << c) >> 1, (k == 0 ? et : 1022) - c, 0x80000000u);
    em = big ? (nan ? t : -1.0) : (et == 0 ? t : d);
  }
  return r;
}

// d^k/dx^k g at (g, h = 1 - g): (-beta)^k sum_i (-1)^i A(k,i) g^(i+1) h^(k-i), A = Eulerian
// Out of line: derivative values are few per sample, and one copy keeps the kernels' code small
// (instruction-fetch stalls are measurable in the adjoint).
static __device__ __noinline__ double fermi_poly(int k, double g, double h, double beta) {
  if (k == 0) return g;
  double gh = g * h;
  if (k == 1) return -beta * gh;
  double d = h - g;
  if (k == 2) return beta * beta * gh * d;
  if (k == 3) return -beta * beta * beta * gh * fma(d, d, -2.0 * gh);
  double b4 = beta * beta * beta * beta;
  double h2 = h * h, g2 = g * g;
  if (k == 4) return b4 * gh * (h2 * h - 11.0 * g * h2 + 11.0 * g2 * h - g2 * g);
  return -b4 * beta * gh * (h2 * h2 - 26.0 * g * h2 * h + 66.0 * g2 * h2 - 26.0 * g2 * g * h + g2 * g2);
}

// -v by its sign bit (no FP64 instruction)
__device__ __forceinline__ double neg_bits(double v) {
  return __hiloint2double(__double2hiint(v) ^ (int)0x80000000u, __double2loint(v));
}

// c v for a table coefficient c (the same in every thread): the tables' +-1 are a copy or a sign flip
__device__ __forceinline__ double coef_mul(double c, double v) {
  const int hi = __double2hiint(c);
  if ((hi & 0x7FFFFFFF) == 0x3FF00000 && __double2loint(c) == 0) return hi < 0 ? neg_bits(v) : v;
  return __dmul_rn(c, v);
}

// One pole-DAG step F a + v, or F a for a node's first child (the same flag in every thread): a
// product, which the integer pipes take
__device__ __forceinline__ double dag_step(double F, double a, double v, int first) {
  if (first) return imul(F, a);
  return fma(F, a, v);
}

// Fermi values of one segment of the term table: one energy combination x and one sigma, every
// value g_sigma^(k)(+-x) that the terms use (k = 0 first).  y = e^{-beta|x|} keeps the tails exact;
// the Bose-type segments (sigma = -1) take 1 - y = -(e^t - 1) from the same exponential.  With
// DUAL, fvd holds each value's derivative with respect to its own argument (order k + 1).
// seg = {combo, sigma, v_begin, first v with k >= 1, v_end}; fvr[v] = {sign, k}.
// S: the stride of x and fv (1, or the samples of a tile where they lie in shared memory).
template <bool BOSE, bool DUAL, int S = 1>
__device__ __forceinline__ void fermi_segment(const int* seg, const int* fvr, const double* x, double beta,
                                              double* fv, double* fvd) {
  const double xv = x[seg[0] * S];
  double em = 0.0;
  const double y = exp_neg<BOSE ? kBoseExp : kFermiExp>(neg_bits(imul(beta, fabs(xv))), em);
  const double rD = rcp(BOSE ? neg_bits(em) : 1.0 + y);
  const double t2 = imul(BOSE ? neg_bits(y) : y, rD);
  const bool neg = __double_as_longlong(xv) <= 0;   // xv <= 0 (+0, -0 and negatives), on the ALU
  const double g = neg ? rD : t2, h = neg ? t2 : rD;   // g_sigma(x) and g_sigma(-x)
  double d1 = 0.0;
  if (DUAL) d1 = neg_bits(imul(beta, imul(g, h)));
  for (int v = seg[2]; v < seg[3]; ++v) {
    fv[v * S] = fvr[2 * v] > 0 ? g : h;
    if (DUAL) fvd[v] = d1;
  }
  for (int v = seg[3]; v < seg[4]; ++v) {
    const bool pos = fvr[2 * v] > 0;
    const int k = fvr[2 * v + 1];
    const double gg = pos ? g : h, hg = pos ? h : g;
    fv[v * S] = fermi_poly(k, gg, hg, beta);
    if (DUAL) fvd[v] = fermi_poly(k + 1, gg, hg, beta);
  }
}

}  // namespace dev
}  // namespace tami
