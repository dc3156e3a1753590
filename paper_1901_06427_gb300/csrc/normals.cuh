// Box-Muller on 64-bit integers.  FP64 runs at 2 operations per SM and clock
// on this GPU, 32-bit integers at 64, and the logarithm, sine and cosine of
// the library are some 70 FP64 operations a pair of normals.  Here the
// polynomials are fixed-point Horner sums (Taylor series; Brent and
// Zimmermann, Modern Computer Arithmetic, ch. 4), exact to about 2^-60 and
// rounded once; the square root, conversions and products are left in FP64.
// Against extended precision: mean 0.43, at most 2.3 units in the last place
// (the library: 0.46, 2.8).  Forcing of a 128 x 128 x 64 grid, 9.4 million
// normals: 698 -> 226 us.
#pragma once
#include <cmath>

#include "common.cuh"

namespace rbfib {

typedef unsigned long long u64;

__device__ inline u64 mul_hi(u64 a, u64 b) {
  return __umul64hi(a, b);
}
__device__ inline long long mul_hi_s(long long a, long long b) {
  return __mul64hi(a, b);
}
__device__ inline int lead_zeros(u64 a) {
  return __clzll((long long)a);
}

// v / 2^63 for v in [2^62, 2^63], from its bits (rounded to 53)
__device__ inline double unit_double(u64 v) {
  const u64 m = (v + 512) >> 10;   // 53 bits, 2^53 for 1
  const u64 bits = (0x3FEULL << 52) + (m - (1ULL << 52));
  return __longlong_as_double((long long)bits);
}

// v 2^e, v > 0 (one rounding), -200 < e < 0
__device__ inline double scaled_double(u64 v, int e) {
  const double d = __ull2double_rn(v);
  return __hiloint2double(__double2hiint(d) + (e << 20), __double2loint(d));
}

// cos and sin of 2 pi k / 2^53 (k odd): the nearest quarter turn q and the
// rest, at most an eighth of a turn, in units of 2^-64 of an eighth: t.  With
// z = t^2 the series of sin(x) / t and cos(x), x = (pi / 4) t, have terms
// (pi / 4)^(2n + 1) / (2n + 1)! and (pi / 4)^2n / (2n)! in 2^64 fixed point,
// falling, so the alternating Horner sums stay positive.
__device__ inline void fixed_cossin(u64 k, double& c, double& s) {
  const u64 K = k << 11;
  const u64 q = (K + (1ULL << 61)) >> 62;
  const long long rest = (long long)(K - (q << 62));
  const u64 t = (u64)(rest < 0 ? -rest : rest) << 3;
  const u64 z = mul_hi(t, t);
  const u64 fs[9] = {0xC90FDAA22168C235ULL, 0x14ABBCE625BE52BFULL, 0x00A335E33BAD570FULL, 0x000265A599CC57B1ULL,
      0x00000541E0D21FBAULL, 0x000000078C1D3F7AULL, 0x0000000007A3D0D3ULL, 0x000000000005BEB7ULL,
      0x0000000000000356ULL};
  const u64 fc[9] = {0x4EF4F326F9177969ULL, 0x040F07C206D6B0EDULL, 0x00155D3C7E3CBFFAULL, 0x00003C3EA0D12375ULL,
      0x00000069B47CA881ULL, 0x000000007E74E28EULL, 0x00000000006DB894ULL, 0x0000000000004832ULL,
      0x0000000000000025ULL};
  u64 as = fs[8], ac = fc[8];
#pragma unroll
  for (int n = 7; n >= 0; --n) as = fs[n] - mul_hi(z, as);
#pragma unroll
  for (int n = 7; n >= 0; --n) ac = fc[n] - mul_hi(z, ac);
  const double cx = unit_double((1ULL << 63) - (mul_hi(z, ac) >> 1));
  // sin x = t times the sum, from the normalised t: one rounding
  const int nz = lead_zeros(t);
  const double x = scaled_double(mul_hi(t << nz, as), -64 - nz);
  const double y = rest < 0 ? -x : x;
  const int h = (int)(q & 3);
  c = h == 0 ? cx : (h == 1 ? -y : (h == 2 ? -cx : y));
  s = h == 0 ? y : (h == 1 ? cx : (h == 2 ? -y : -cx));
}

// 1 / m to 16 bits and log of that (scale 2^62), for m in [1 + i / 128, 1 + (i + 1) / 128)
// (i < 53) or half of it (i >= 53, so that numbers near 1 from below meet the
// entry 1, log 0, and keep their relative accuracy).
struct LogEntry { int c; long long l; };
constexpr int kLogHalf = 53;
#define RBFIB_LOG_TABLE \
  {65281, -17979030617864065LL}, {64777, -53721566841893809LL}, {64281, -89169311688258771LL}, {63792, -124385562132551897LL}, \
  {63310, -159362876675174486LL}, {62836, -194020328528059026LL}, {62369, -228422586551868754LL}, {61909, -262561939555911652LL}, \
  {61455, -296505633089862732LL}, {61008, -330171847459276224LL}, {60568, -363552625038834140LL}, {60133, -396793312413045394LL}, \
  {59705, -429734616644506846LL}, {59283, -462446144856591826LL}, {58867, -494921291898391171LL}, {58457, -527153383619098516LL}, \
  {58053, -559135679021566025LL}, {57654, -590941360872044003LL}, {57260, -622565208468182596LL}, {56872, -653920850503099834LL}, \
  {56489, -685082933859715454LL}, {56111, -716046057544234220LL}, {55738, -746804763687088968LL}, {55370, -777353538942321773LL}, \
  {55007, -807686815984830748LL}, {54649, -837798975107428958LL}, {54295, -867769282719454645LL}, {53946, -897508180140171349LL}, \
  {53601, -927095934962885391LL}, {53261, -956441792932719713LL}, {52925, -985627027780727351LL}, {52593, -1014647380906639480LL}, \
  {52265, -1043498550060978821LL}, {51942, -1072087404060262024LL}, {51622, -1100586577950519378LL}, {51306, -1128903408364953640LL}, \
  {50995, -1156942992926259548LL}, {50686, -1184972130452083048LL}, {50382, -1212714972451425057LL}, {50081, -1240349457688350988LL}, \
  {49784, -1267779984612355943LL}, {49490, -1295095085307753489LL}, {49200, -1322197989243369968LL}, {48913, -1349178260205028570LL}, \
  {48630, -1375937962185196011LL}, {48349, -1402663075824565448LL}, {48072, -1429160219421642853LL}, {47798, -1455521029051160012LL}, \
  {47528, -1481645246047701701LL}, {47260, -1507723128190822638LL}, {46995, -1533654909316137680LL}, {46733, -1559437277101490695LL}, \
  {46474, -1585066891895395618LL}, {92436, 1586036773904542518LL}, {91930, 1560722789933351138LL}, {91429, 1535521295106433173LL}, \
  {90933, 1510434907529758482LL}, {90443, 1485517259697886905LL}, {89958, 1460720577776134287LL}, {89478, 1436047551527460204LL}, \
  {89004, 1411552708217459701LL}, {88534, 1387135428624744671LL}, {88069, 1362850009302924683LL}, {87609, 1338699228708205262LL}, \
  {87154, 1314685886302267538LL}, {86704, 1290812802030761044LL}, {86258, 1267029352221629009LL}, {85817, 1243391310823455490LL}, \
  {85380, 1219847543500308654LL}, {84948, 1196454412226024489LL}, {84520, 1173160270411970494LL}, {84096, 1149967228314314286LL}, \
  {83677, 1126932527151959153LL}, {83262, 1104003749093858010LL}, {82850, 1081127394156362155LL}, {82443, 1058416692520174060LL}, \
  {82040, 1035818452163242267LL}, {81641, 1013334885151117886LL}, {81246, 990968219327318465LL}, {80854, 968663661113952821LL}, \
  {80466, 946479956359864936LL}, {80082, 924419378737970222LL}, {79702, 902484216382770391LL}, {79325, 880618635242701374LL}, \
  {78952, 858882538787793076LL}, {78582, 837219571245418092LL}, {78215, 815631251832371324LL}, {77853, 794237585833260137LL}, \
  {77493, 772863235175720620LL}, {77137, 751628505520970878LL}, {76784, 730475732103458504LL}, {76434, 709406498541089960LL}, \
  {76087, 688422400490191449LL}, {75744, 667585931057156858LL}, {75403, 646777213710538854LL}, {75066, 626119925009397864LL}, \
  {74731, 605493111498964170LL}, {74400, 585021571997238950LL}, {74072, 564645535103809444LL}, {73746, 544304141234732753LL}, \
  {73423, 524061060481372357LL}, {73103, 503917988643322778LL}, {72786, 483876631603282682LL}, {72472, 463938705081979454LL}, \
  {72160, 444042025652128303LL}, {71851, 424251687878372571LL}, {71545, 404569436439140153LL}, {71241, 384932291790362880LL}, \
  {70940, 365406200887995488LL}, {70641, 345927652644096734LL}, {70345, 326563161600450499LL}, {70051, 307248684389221414LL}, \
  {69760, 288051302648406119LL}, {69471, 268906440176533972LL}, {69184, 249815087141782248LL}, {68900, 230845174972632855LL}, \
  {68618, 211931326892856672LL}, {68339, 193142040051111389LL}, {68062, 174411403425541569LL}, {67787, 155740446887414269LL}, \
  {67514, 137130207619826967LL}, {67243, 118581730052356888LL}, {66975, 100164923133719907LL}, {66709, 81812538408213418LL}, \
  {66444, 63456235382273711LL}, {66182, 45235625417602780LL}, {65922, 27082656347884782LL}, {65536, 0LL}
static __device__ const LogEntry kLogDev[128] = {RBFIB_LOG_TABLE};
#undef RBFIB_LOG_TABLE

// -log(k / 2^53), k odd: k = m 2^e, r = m c - 1 exactly (|r| < 2^-7, scale
// 2^70), log(1 + r) = r (1 - r / 2 + ... - r^7 / 8) with the sum in 2^62.
// Added up in fixed point (scale 2^57 where a multiple of log 2 makes the
// result at least 1 / 3, 2^62 below) and rounded once; next to 1 the
// normalised product keeps the relative accuracy.
__device__ inline double fixed_neglog(u64 k) {
  const u64 K = k << 11;
  const int n = lead_zeros(K);
  const u64 M = K << n;
  const int i = (int)(M >> 56) & 127;
  const LogEntry e = kLogDev[i];
  const bool half = i >= kLogHalf;
  const long long hi = (long long)mul_hi(M, (u64)e.c) - (half ? 65536 : 32768);
  const u64 lo = M * (u64)e.c;
  const long long R = half ? (long long)(((u64)hi << 54) | (lo >> 10)) : (long long)(((u64)hi << 55) | (lo >> 9));
  const long long one = 1LL << 62;
  long long a = one / 8;
#pragma unroll
  for (int j = 7; j >= 1; --j) a = one / j - (mul_hi_s(R, a) >> 6);
  const int n2 = half ? n : n + 1;
  const long long rp = mul_hi_s(R, a);              // r p, scale 2^68
  if (n2 > 0) return scaled_double((u64)((long long)n2 * 99893036290645747LL + ((e.l - (rp >> 6)) >> 5)), -57);
  if (i < 127) return scaled_double((u64)(e.l - (rp >> 6)), -62);
  const u64 d = (u64)-R;                             // log 0 entry: r < 0
  const int nz = lead_zeros(d);
  return scaled_double(mul_hi(d << nz, (u64)a), -68 - nz);
}

// Two standard normals of two 64-bit words: u = (2 (word >> 12) + 1) 2^-53.
__device__ inline void box_muller(u64 w0, u64 w1, double& z0, double& z1) {
  const double rad = sqrt(2.0 * fixed_neglog((w0 >> 12) * 2 + 1));
  double c, s;
  fixed_cossin((w1 >> 12) * 2 + 1, c, s);
  z0 = rad * c;
  z1 = rad * s;
}

}  // namespace rbfib
