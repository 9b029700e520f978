// log64.cuh -- ln u of a double on the integer pipes (see exp64.cuh).
//
// Table-driven as in Tang (ACM TOMS 16, 1990), with a reciprocal in place of
// the quotient that reduces the argument: u = 2^e m, m in [1, 2); c an 11-bit
// reciprocal of m's 1/128 interval, r = m c / 1024 - 1 exactly (|r| <= 2^-7),
// ln u = e ln2 - ln(c / 1024) + ln(1 + r), the last by its series to degree 8
// (remainder below 2^-66), in fixed point.  The intervals next to u = 1 on both
// sides have c / 1024 a power of two, so that ln u = ln(1 + r) there and keeps
// its relative accuracy down to |r| = 2^-14.  Error below 2^-59 for |ln u| < 3
// and 2^-55 for |ln u| < 31 before the rounding to 53 bits.  Nearer to 1, and for
// u <= 0, subnormal, infinite, NaN or outside 2^+-44: the library function.
#pragma once

#include "exp64.cuh"

namespace plc {

static __device__ const short kLogC[128] = {
    1024, 1012, 1004, 997, 989, 982, 975, 967, 960, 953, 946, 940, 933, 926, 920, 913,
    907, 901, 895, 889, 883, 877, 871, 865, 859, 854, 848, 843, 838, 832, 827, 822,
    817, 812, 807, 802, 797, 792, 787, 783, 778, 773, 769, 764, 760, 755, 751, 747,
    743, 738, 734, 730, 726, 722, 718, 714, 710, 707, 703, 699, 695, 692, 688, 684,
    681, 677, 674, 670, 667, 664, 660, 657, 654, 650, 647, 644, 641, 638, 635, 632,
    629, 626, 623, 620, 617, 614, 611, 608, 605, 603, 600, 597, 594, 592, 589, 586,
    584, 581, 579, 576, 574, 571, 569, 566, 564, 561, 559, 557, 554, 552, 550, 547,
    545, 543, 541, 538, 536, 534, 532, 530, 527, 525, 523, 521, 519, 517, 515, 512,
};
// -ln(c / 1024) 2^60 (of 2c for the last, which counts towards the next e)
static __device__ const long long kLogTab[128] = {
    0ll, 13590587681883476ll, 22740806383186690ll, 30807256611971992ll,
    40095697623689676ll, 48284925897373559ll, 56532738826279073ll, 66031630907523962ll,
    74407848895029353ll, 82845367507105431ll, 91345090609281748ll, 98680777104497848ll,
    107298489979452553ll, 115981102863242372ll, 123475743586234814ll, 132281515288628772ll,
    139883223077957170ll, 147535385049260804ll, 155238675430709328ll, 162993782056176734ll,
    170801406733800115ll, 178662265627103213ll, 186577089649202316ll, 194546624870637104ll,
    202571632941395479ll, 209302075316251029ll, 217430815250085943ll, 224248821545547734ll,
    231107387307935504ll, 239391888855743598ll, 246341406610004817ll, 253333068452935312ll,
    260367388655169787ll, 267444890958374919ll, 274566108809250114ll, 281731585600800027ll,
    288941874921151705ll, 296197540810201245ll, 303499158024387491ll, 309373929994866378ll,
    316759743239601816ll, 324193176498858454ll, 330174624439841240ll, 337695339331245288ll,
    343747434617714924ll, 351357505182575729ll, 357481936607473308ll, 363639075431354468ll,
    369829272877128732ll, 377614052654187498ll, 383879945819548197ll, 390180079008213048ll,
    396514828486998778ll, 402884576759251625ll, 409289712703438644ll, 415730631715610343ll,
    422207735855865135ll, 427089556154519998ll, 433630972310444216ll, 440209714866103200ll,
    446826212248530799ll, 451813623795130981ll, 458497245438126964ll, 465219838856089283ll,
    470287633849251483ll, 477079532752816140ll, 482199843928021953ll, 489062492194130819ll,
    494236419372191358ll, 499433670117473987ll, 506399984391350116ll, 511652483246587407ll,
    516929021081915578ll, 524002181331921822ll, 529335675059130803ll, 534693956607640943ll,
    540077257460307795ll, 545485812357783430ll, 550919859359936584ll, 556379639908727104ll,
    561865398892576254ll, 567377384712275760ll, 572915849348479956ll, 578481048430826889ll,
    584073241308735777ll, 589692691123929858ll, 595339664884735323ll, 601014433542208802ll,
    606717272068147649ll, 610534896432505178ll, 616285140295701454ll, 622064207556806876ll,
    627872388629724475ll, 631760829093401393ll, 637618190572363589ll, 643505462111937038ll,
    647447077932706926ll, 653384884214386239ll, 657360479548938670ll, 663349695639046460ll,
    667359861437219269ll, 673401385329787218ll, 677446728092792758ll, 683541481517595853ll,
    687622623848514955ll, 693771553115018854ll, 697889134293870562ll, 702021473859745046ll,
    708247887757740183ll, 712417590330251922ll, 716602427972498987ll, 722908304246474682ll,
    727131464663064449ll, 731370151439628013ll, 735624479162236468ll, 742035551314892863ll,
    746329491118624697ll, 750639483071090934ll, 754965647639121053ll, 759308106650758045ll,
    765852617154495627ll, 770236354392613706ll, 774636823492798840ll, 779054152669022208ll,
    783488471614654211ll, 787939911525312489ll, 792408605122152711ll, 0ll,
};

static __device__ __noinline__ double log64_far(double u) { return log(u); }

// ln u = q 2^E; false where the library function has to serve.
__device__ __forceinline__ bool log64_fixed(double u, long long& q, int& E) {
  const int top = __double2hiint(u);
  const unsigned long long b = (unsigned long long)__double_as_longlong(u);
  const int j = (top >> 13) & 127, e = (top >> 20) - 1023 + (j == 127);
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const long long R = ((long long)(m * (unsigned)__ldg(kLogC + j)) - (1ll << 62)) << 6;   // r 2^68
  const int r31 = (int)(R >> 30);                                        // 2^7 r 2^31
  // 1/7 - r/8 (2^33), 1/6 - r () (2^33), 1/5 - r () (2^33), 1/4 - r () (2^32),
  // 1/3 - r () (2^61), 1/2 - r () (2^61)
  const int a7 = 1227133513 - (r31 >> 8);
  const int a6 = 1431655765 - (__mulhi(r31, a7) >> 6);
  const int a5 = 1717986918 - (__mulhi(r31, a6) >> 6);
  const int a4 = 1073741824 - (__mulhi(r31, a5) >> 7);
  const long long g = 768614336404564651ll - (((long long)r31 * a4) >> 9);
  const long long h = (1ll << 60) - (mul61(R, g) >> 7);
  const long long P = R - (mul61(R, mul61(R, h)) >> 7);                  // ln(1 + r) 2^68
  const bool one = e == 0 && (j == 0 || j == 127), low = abs(e) <= 4;
  const int sh = low ? 0 : 4;
  const long long ln2 = low ? 799144290325165978ll : 49946518145322873ll;
  const int ext = low ? 1582243229 : 1441067482;                 // 31 bits below the point
  const long long x = (long long)e * ln2 + (((long long)e * ext) >> 31) + (__ldg(kLogTab + j) >> sh) +
                      ((P + (128ll << sh)) >> (8 + sh));
  q = one ? P : x;
  E = one ? -68 : sh - 60;
  return top >= ((1023 - 44) << 20) && top < ((1023 + 44) << 20) &&
         !(one && (unsigned long long)(R + (1ll << 54)) < (1ull << 55));
}
__device__ __forceinline__ double log64(double u) {
  long long q;
  int E;
  return log64_fixed(u, q, E) ? fx_to_double(fx{q}, E) : log64_far(u);
}
__device__ __forceinline__ double logt(double u) { return log64(u); }
__device__ __forceinline__ float logt(float u) { return log(u); }

}  // namespace plc
