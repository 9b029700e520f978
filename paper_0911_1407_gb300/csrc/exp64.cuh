// exp64.cuh -- e^x of a double on the integer pipes.
//
// GB300 issues two FP64 operations per SM and clock, so the library exp costs
// about nine clocks per lane and bounded every FP64 pass that forms e^s; this
// one takes about 16 wide integer multiply-adds and 100 single-cycle
// operations (1.6 clocks).  Table-driven as in Tang (ACM TOMS 15, 1989): x =
// (64 m + j) ln2/64 + r with |r| <= ln2/128, e^x = 2^m 2^(j/64) (1 + p(r)), p
// the Taylor polynomial of e^r - 1 to degree 6 (remainder below 2^-64), all in
// 61-bit fixed point.  x is taken to 2^-57 absolute, so the result carries one
// rounding to 53 bits and less than 2^-56 relative before it.  |x| >= 32, NaN
// and infinities take the library function.
#pragma once

#include "fx.cuh"

namespace plc {

// 2^(j/64) 2^61
static __device__ const long long kExp2Tab[64] = {
    2305843009213693952ll, 2330951993331335645ll, 2356334396359501942ll, 2381993195634921490ll,
    2407931400915394245ll, 2434152054732833796ll, 2460658232750154058ll, 2487453044122042215ll,
    2514539631859660218ll, 2541921173199317625ll, 2569600879975159024ll, 2597581998995909751ll,
    2625867812425724110ll, 2654461638169180747ll, 2683366830260470360ll, 2712586779256821376ll,
    2742124912636209756ll, 2771984695199399577ll, 2802169629476361550ll, 2832683256137117140ll,
    2863529154407056491ll, 2894710942486778865ll, 2926232277976504838ll, 2958096858305110056ll,
    2990308421163830843ll, 3022870744944692570ll, 3055787649183712190ll, 3089062995008926926ll,
    3122700685593301682ll, 3156704666612568285ll, 3191078926708050276ll, 3225827497954527522ll,
    3260954456333195553ll, 3296463922209775076ll, 3332360060817827770ll, 3368647082747335039ll,
    3405329244438597040ll, 3442410848681509921ll, 3479896245120279830ll, 3517789830763632898ll,
    3556096050500581047ll, 3594819397621804119ll, 3633964414346709481ll, 3673535692356230935ll,
    3713537873331429433ll, 3753975649497958757ll, 3794853764176460055ll, 3836177012338949768ll,
    3877950241171266237ll, 3920178350641640941ll, 3962866294075461077ll, 4006019078736290889ll,
    4049641766413219908ll, 4093739474014606996ll, 4138317374168289834ll, 4183380695828330266ll,
    4228934724888366668ll, 4274984804801645281ll, 4321536337207803251ll, 4368594782566476878ll,
    4416165660797809419ll, 4464254551929933550ll, 4512867096753504463ll, 4562008997483360349ll,
};

// a b 2^-61 (see operator*(fx, fxk))
__device__ __forceinline__ long long mul61(long long a, long long b) {
  return (fx{a} * fxk{fx_hi(b), fx_lo(b)}).v;
}

// The rare argument, out of line: inlined at every cell of an unrolled loop
// it costs more instruction cache than the loop itself.
static __device__ __noinline__ double exp64_far(double x) { return exp(x); }

__device__ __forceinline__ double exp64(double x) {
  const unsigned top = (unsigned)__double2hiint(x) & 0x7fffffffu;
  if (top >= 0x40400000u) return exp64_far(x);               // |x| >= 32 or NaN
  const long long q = fx_from(x, -57).v;                     // x 2^57
  // n = round(x 64 / ln2)
  const int n = (int)(((long long)(int)(q >> 32) * 96817625 + (1ll << 44)) >> 45);
  // r 2^57 = q - n ln2/64 2^57, the constant to 31 bits below the point
  const long long r57 = q - (long long)n * 1560828692041339ll - (((long long)n * 1722754959) >> 31);
  const long long R = r57 << 11;                             // r 2^68 = (2^7 r) 2^61
  const int r31 = (int)(R >> 30);                            // 2^7 r 2^31
  // 1/120 + r/720 (2^37), 1/24 + r () (2^35), 1/6 + r () (2^61), 1/2 + r () (2^61)
  const int a = 1145324612 + __mulhi(r31, 2982616);
  const int k = 1431655765 + (__mulhi(r31, a) >> 8);
  const long long g = 384307168202282325ll + (((long long)r31 * k) >> 12);
  const long long i = (1ll << 60) + (mul61(R, g) >> 7);
  const long long P = R + (mul61(R, mul61(R, i)) >> 7);      // (e^r - 1) 2^68
  const long long t = __ldg(kExp2Tab + (n & 63));
  return fx_to_double(fx{t + (mul61(P, t) >> 7)}, (n >> 6) - 61);
}
__device__ __forceinline__ double expt(double x) { return exp64(x); }
__device__ __forceinline__ float expt(float x) { return exp(x); }

}  // namespace plc
