// Fixed-point contractions of the element kernels.
//
// FP64 issues 2 DFMA per clock and SM on this part (measured 1.71), the
// 32 x 32 + 64 bit integer multiply-add 64 (measured 63).  A dot product of n
// doubles with table coefficients is therefore done on integers: the n values
// share one exponent (their largest), become 61-bit integers D = dh 2^31 + dl,
// the coefficients are 62-bit integers C = ch 2^31 + cl, and
//   sum C D / 2^62 = sum dh ch + (sum dh cl + dl ch) / 2^31
// takes three multiply-adds per term (the dl cl products lie below the last
// bit kept), and the result is rounded once, to nearest, when it becomes a
// double again.  Its error is at most 2^(g - 58) of the line's largest value,
// with 2^g above the row's sum of |c|: FP64's own for a row that counts that
// value.  A row that does not (the zero coefficients of the middle node, n odd;
// the ragged passes' near the degenerate edge) keeps less beside it than FP64.
// For infinities, NaNs and subnormals see fx_wild.
//
// A value keeps its scale as `eb`: |x| < 2^(eb - 1023), x = R 2^(eb - 1084).
// Between the passes of one transform the integers stay in shared memory,
// every line with its own exponent, taken from its results (the OR of their
// magnitudes): the collapsed bases grow towards the degenerate edge where the
// weighted data shrink, so one exponent per element would cost the bits that
// the next pass needs there (measured, residual at N = 6: FP64 passes 3.5e-12,
// one exponent 2.5e-11, an exponent per line 2.8e-12).  In the
// derivative sum and the lift every line keeps its own too, and what meets at a
// point (in the lift that goes on into a transform, on a line) meets on the
// largest there: an element with a front in it holds lines of values 1e4 (1e12)
// times below its largest, whose derivatives one exponent per variable left
// 1e-12 (2e-4) of their size off at n = 5.
//
// A lane owns one line of n points of one variable: it reads the n values
// once and forms all n results, so the coefficients are the same for every
// lane of a pass (constant memory operands), except in the ragged passes
// (prism and tetrahedron b, pyramid and tetrahedron c), which read theirs
// from the table pool.
#pragma once
#include "dg_kernels.cuh"
// Unrolling of the loops over a line's results.  A kernel that runs every pass
// once per element keeps them unrolled; the Navier-Stokes volume phase, whose
// code is long, is faster rolled (fewer instruction-cache misses: the viscous
// 20^3 step 21.09 -> 20.07 ms; the Euler step 5.52 unrolled, 5.57 rolled).
#ifndef DG_UNROLL
#define DG_UNROLL 8
#endif

namespace dgk {
namespace {
constexpr int kUnroll = DG_UNROLL;

// Tables per n: coefficient c is stored as round(c 2^(62 - g)) =
// x 2^31 + y with -2^30 <= y < 2^30; g bounds every row (and column) sum of
// |c| by 2^g, and 2^31 sum |x| + 2^30 sum |y| < 2^63 per row.
//   A(p, i) = sqrt((2p + 1)/2) P_p(x_i)   (Legendre basis at the Gauss points)
//   D(r, i) = l'_r(x_i)                   (collocation derivative, transposed)
//   E(end, m) = l_m(-1), l_m(+1)          (extrapolation, g = kFxGE)
// S(r) = 2^30 + sum_i y(D(r, i)) / 2: the half that makes a row's shift by 31
// round to nearest, and the mean of the dl cl products that are not formed (dl
// is uniform on [0, 2^31)): without it every derivative sum would lean the same
// way, and the transform behind it adds the leanings up.
constexpr int kFxGE = 3;
constexpr int kFxGR = 3;   // growth of the ragged passes (rows scaled to at most 1, at most 7 terms)
template <int n>
struct FxTab;

__constant__ int2 kFxA2[4] = {
    {759250125, -12858223}, {759250125, -12858223}, {-759250125, 12858223}, {759250125, -12858223}};
__constant__ int2 kFxD2[4] = {
    {-929887697, 666064268}, {-929887697, 666064268}, {929887697, -666064268}, {929887697, -666064268}};
__constant__ int2 kFxE2[4] = {
    {366689652, 370354845}, {-98254196, -370354845}, {-98254196, -370354845}, {366689652, 370354845}};
__constant__ long long kFxS2[2] = {1739806092, 407677556};
template <> struct FxTab<2> {
  static constexpr int gA = 1, gD = 1;
  static __device__ __forceinline__ int2 A(int p, int i) { return kFxA2[p * 2 + i]; }
  static __device__ __forceinline__ int2 D(int r, int i) { return kFxD2[r * 2 + i]; }
  static __device__ __forceinline__ long long S(int r) { return kFxS2[r]; }
  static __device__ __forceinline__ int2 E(int end, int m) { return kFxE2[end * 2 + m]; }
};

__constant__ int2 kFxA3[9] = {
    {379625062, 1067312712}, {379625062, 1067312712}, {379625062, 1067312712}, {-509320467, -909560612}, {0, 0},
    {509320467, 909560612}, {339546978, 606373742}, {-424433723, 315774647}, {339546978, 606373742}};
__constant__ int2 kFxD3[9] = {
    {-519823025, -665283801}, {-173274342, 494066616}, {173274342, -494066616}, {693097367, 171217185}, {0, 0},
    {-693097367, -171217185}, {-173274342, 494066616}, {173274342, -494066616}, {519823025, 665283801}};
__constant__ int2 kFxE3[6] = {
    {396970555, 221761267}, {-178956971, 715827883}, {50421872, -937589150}, {50421872, -937589150},
    {-178956971, 715827883}, {396970555, 221761267}};
__constant__ long long kFxS3[3] = {741099923, 1073741824, 1406383724};
template <> struct FxTab<3> {
  static constexpr int gA = 2, gD = 3;
  static __device__ __forceinline__ int2 A(int p, int i) { return kFxA3[p * 3 + i]; }
  static __device__ __forceinline__ int2 D(int r, int i) { return kFxD3[r * 3 + i]; }
  static __device__ __forceinline__ long long S(int r) { return kFxS3[r]; }
  static __device__ __forceinline__ int2 E(int end, int m) { return kFxE3[end * 3 + m]; }
};

__constant__ int2 kFxA4[16] = {
    {379625062, 1067312712}, {379625062, 1067312712}, {379625062, 1067312712}, {379625062, 1067312712},
    {-566222869, -1000043699}, {-223547700, -546687481}, {223547700, 546687481}, {566222869, 1000043699},
    {519790077, -989244199}, {-277256521, 808801544}, {-277256521, 808801544}, {519790077, -989244199},
    {-306085893, 192663021}, {413536929, 955962303}, {-413536929, -955962303}, {306085893, -192663021}};
__constant__ int2 kFxD4[16] = {
    {-447213501, -899078943}, {-101677662, 241694245}, {44117129, -305844501}, {-77930594, 692007722},
    {652318883, 864221711}, {-51595226, -718762622}, {-197390017, -171223876}, {283035976, -726864953},
    {-283035976, 726864953}, {197390017, 171223876}, {51595226, 718762622}, {-652318883, -864221711},
    {77930594, -692007722}, {-44117129, 305844501}, {101677662, -241694245}, {447213501, 899078943}};
__constant__ int2 kFxE4[8] = {
    {409844067, -703286682}, {-218407798, 870975805}, {107578601, 970901277}, {-30579415, 1008893247},
    {-30579415, 1008893247}, {107578601, 970901277}, {-218407798, 870975805}, {409844067, -703286682}};
__constant__ long long kFxS4[4] = {938131085, 697426954, 1450056694, 1209352562};
template <> struct FxTab<4> {
  static constexpr int gA = 2, gD = 4;
  static __device__ __forceinline__ int2 A(int p, int i) { return kFxA4[p * 4 + i]; }
  static __device__ __forceinline__ int2 D(int r, int i) { return kFxD4[r * 4 + i]; }
  static __device__ __forceinline__ long long S(int r) { return kFxS4[r]; }
  static __device__ __forceinline__ int2 E(int end, int m) { return kFxE4[end * 4 + m]; }
};

__constant__ int2 kFxA5[25] = {
    {189812531, 533656356}, {189812531, 533656356}, {189812531, 533656356}, {189812531, 533656356},
    {189812531, 533656356}, {-297920170, 83774255}, {-177029835, 524643203}, {0, 0}, {177029835, -524643203},
    {297920170, -83774255}, {310576350, 839747701}, {-27620535, -334436249}, {-212216861, -915854501},
    {-27620535, -334436249}, {310576350, 839747701}, {-251616227, -975912404}, {209607937, 905822449}, {0, 0},
    {-209607937, -905822449}, {251616227, 975912404}, {139931009, -1020151954}, {-196171759, 1021104415},
    {213539098, -741813879}, {-196171759, 1021104415}, {139931009, -1020151954}};
__constant__ int2 kFxD5[25] = {
    {-340043338, -464414026}, {-64441691, 225275681}, {20211053, 155274482}, {-16402521, -846373609},
    {37028447, -942733549}, {516869255, 39386024}, {-50892223, 182790769}, {-96327274, -734527880},
    {62314474, 700400628}, {-131560158, 751241848}, {-271357628, 233536301}, {161245867, -554039431}, {0, 0},
    {-161245867, 554039431}, {271357628, -233536301}, {131560158, -751241848}, {-62314474, -700400628},
    {96327274, 734527880}, {50892223, -182790769}, {-516869255, -39386024}, {-37028447, 942733549},
    {16402521, 846373609}, {-20211053, -155274482}, {64441691, -225275681}, {340043338, 464414026}};
__constant__ int2 kFxE5[10] = {
    {416452927, 216256544}, {-239755380, -508451132}, {143165577, -1002159036}, {-71925040, 867629694},
    {20497372, 426723931}, {20497372, 426723931}, {-71925040, 867629694}, {143165577, -1002159036},
    {-239755380, -508451132}, {416452927, 216256544}};
__constant__ long long kFxS5[5] = {137256313, 1543387518, 1073741824, 604096129, 2010227334};
template <> struct FxTab<5> {
  static constexpr int gA = 3, gD = 5;
  static __device__ __forceinline__ int2 A(int p, int i) { return kFxA5[p * 5 + i]; }
  static __device__ __forceinline__ int2 D(int r, int i) { return kFxD5[r * 5 + i]; }
  static __device__ __forceinline__ long long S(int r) { return kFxS5[r]; }
  static __device__ __forceinline__ int2 E(int end, int m) { return kFxE5[end * 5 + m]; }
};

__constant__ int2 kFxA6[36] = {
    {189812531, 533656356}, {189812531, 533656356}, {189812531, 533656356}, {189812531, 533656356},
    {189812531, 533656356}, {189812531, 533656356}, {-306563291, -819992555}, {-217382470, 897060234},
    {-78449624, -672064299}, {78449624, 672064299}, {217382470, -897060234}, {306563291, 819992555},
    {341350436, 813569934}, {66125407, -57509816}, {-175966540, 47828096}, {-175966540, 47828096},
    {66125407, -57509816}, {341350436, 813569934}, {-315505072, -1040216138}, {135149066, -308332591},
    {162692597, 18236024}, {-162692597, -18236024}, {-135149066, 308332591}, {315505072, 1040216138},
    {240305517, 59302192}, {-243859293, -524105452}, {100028740, 957889305}, {100028740, 957889305},
    {-243859293, -524105452}, {240305517, 59302192}, {-129503500, -417942196}, {185332979, 1038570682},
    {-210655037, 834718133}, {210655037, -834718133}, {-185332979, -1038570682}, {129503500, 417942196}};
__constant__ int2 kFxD6[36] = {
    {-479514787, 597921728}, {-82095983, 547488998}, {21770942, 296410655}, {-12898916, -1049652637},
    {13973559, 836191447}, {-35984482, 1034952997}, {745531409, -820203965}, {-78843002, 111654258},
    {-107719820, -12926339}, {50588903, -123531274}, {-50747059, -823783667}, {126896921, -571362468},
    {-429685754, 323554590}, {234112882, 664201462}, {-16980306, -271292391}, {-140619170, -962107812},
    {109947398, -836546710}, {-254581571, -362318177}, {254581571, 362318177}, {-109947398, 836546710},
    {140619170, 962107812}, {16980306, 271292391}, {-234112882, -664201462}, {429685754, -323554590},
    {-126896921, 571362468}, {50747059, 823783667}, {-50588903, 123531274}, {107719820, 12926339},
    {78843002, -111654258}, {-745531409, 820203965}, {35984482, -1034952997}, {-13973559, -836191447},
    {12898916, 1049652637}, {-21770942, -296410655}, {82095983, -547488998}, {479514787, -597921728}};
__constant__ int2 kFxE6[12] = {
    {420282199, 922413512}, {-252453572, -341664032}, {165605901, -537754574}, {-101798161, -311317499},
    {51485924, 492366964}, {-14686835, -224044369}, {-14686835, -224044369}, {51485924, 492366964},
    {-101798161, -311317499}, {165605901, -537754574}, {-252453572, -341664032}, {420282199, 922413512}};
__constant__ long long kFxS6[6] = {2205398418, -46334904, 351487305, 1795996343, 2193818551, -57914770};
template <> struct FxTab<6> {
  static constexpr int gA = 3, gD = 5;
  static __device__ __forceinline__ int2 A(int p, int i) { return kFxA6[p * 6 + i]; }
  static __device__ __forceinline__ int2 D(int r, int i) { return kFxD6[r * 6 + i]; }
  static __device__ __forceinline__ long long S(int r) { return kFxS6[r]; }
  static __device__ __forceinline__ int2 E(int end, int m) { return kFxE6[end * 6 + m]; }
};

__constant__ int2 kFxA7[49] = {
    {189812531, 533656356}, {189812531, 533656356}, {189812531, 533656356}, {189812531, 533656356},
    {189812531, 533656356}, {189812531, 533656356}, {189812531, 533656356}, {-312033413, -1034234961},
    {-243789462, 643368571}, {-133427660, -221439034}, {0, 0}, {133427660, 221439034}, {243789462, -643368571},
    {312033413, 1034234961}, {361281696, 218237818}, {137857240, -265157790}, {-107353961, -79373268},
    {-212216861, -915854501}, {-107353961, -79373268}, {137857240, -265157790}, {361281696, 218237818},
    {-358439408, -273523909}, {46671745, -678880659}, {221795472, -575145396}, {0, 0}, {-221795472, 575145396},
    {-46671745, 678880659}, {358439408, 273523909}, {311526146, -95167372}, {-207390392, -1020774108},
    {-70594378, -580867171}, {213539098, -741813879}, {-70594378, -580867171}, {-207390392, -1020774108},
    {311526146, -95167372}, {-228917650, 221160001}, {259226256, 462864617}, {-165414722, 379312394}, {0, 0},
    {165414722, -379312394}, {-259226256, -462864617}, {228917650, -221160001}, {121017149, -541844870},
    {-175401296, -1007889148}, {204501750, -43865357}, {-213868379, -900660478}, {204501750, -43865357},
    {-175401296, -1007889148}, {121017149, -541844870}};
__constant__ int2 kFxD7[49] = {
    {-321054924, 845902738}, {-51630206, -423505199}, {12394788, -1070654788}, {-6197551, -47878989},
    {4969638, 389777488}, {-6339158, -1067834623}, {17676827, -839016535}, {506102643, -669638213},
    {-55276420, 713080389}, {-62803395, -39058071}, {24835543, -306580161}, {-18374287, -929670968},
    {22625098, 740676974}, {-62139300, 169420688}, {-307780304, -679006439}, {159092650, -688963064},
    {-16303210, 177762420}, {-72223114, -1022541253}, {41338959, -387006813}, {-46545479, 1035353814},
    {123403225, 169384752}, {201673337, 2530819}, {-82445562, -1039899609}, {94646127, 5050145}, {0, 0},
    {-94646127, -5050145}, {82445562, 1039899609}, {-201673337, -2530819}, {-123403225, -169384752},
    {46545479, -1035353814}, {-41338959, 387006813}, {72223114, 1022541253}, {16303210, -177762420},
    {-159092650, 688963064}, {307780304, 679006439}, {62139300, -169420688}, {-22625098, -740676974},
    {18374287, 929670968}, {-24835543, 306580161}, {62803395, 39058071}, {55276420, -713080389},
    {-506102643, 669638213}, {-17676827, 839016535}, {6339158, 1067834623}, {-4969638, -389777488},
    {6197551, 47878989}, {-12394788, 1070654788}, {51630206, 423505199}, {321054924, -845902738}};
__constant__ int2 kFxE7[14] = {
    {422695246, 334795903}, {-260577463, -919111227}, {180417580, 851078313}, {-122713351, -674923432},
    {76250204, 892527342}, {-38673524, 87890175}, {11036764, -572257074}, {11036764, -572257074},
    {-38673524, 87890175}, {76250204, 892527342}, {-122713351, -674923432}, {180417580, 851078313},
    {-260577463, -919111227}, {422695246, 334795903}};
__constant__ long long kFxS7[7] = {-32863130, 912857143, 376233532, 1073741824, 1771250115, 1234626505, 2180346778};
template <> struct FxTab<7> {
  static constexpr int gA = 3, gD = 6;
  static __device__ __forceinline__ int2 A(int p, int i) { return kFxA7[p * 7 + i]; }
  static __device__ __forceinline__ int2 D(int r, int i) { return kFxD7[r * 7 + i]; }
  static __device__ __forceinline__ long long S(int r) { return kFxS7[r]; }
  static __device__ __forceinline__ int2 E(int end, int m) { return kFxE7[end * 7 + m]; }
};

struct FxD {
  int h, l;   // D = h 2^31 + l, 0 <= l < 2^31
};

// D 2^k as (h, l), 0 <= k <= 29
__device__ __forceinline__ FxD fx_split(long long D, int k) {
  const unsigned lo = (unsigned)D, hi = (unsigned)((unsigned long long)D >> 32);
  FxD f;
  f.h = (int)__funnelshift_r(lo, hi, 31 - k);
  f.l = (int)((lo << k) & 0x7fffffffu);
  asm("" : "+r"(f.l));   // see fx_madw
  return f;
}

// x 2^(1083 - em) as an integer, |x| < 2^(em + 1 - 1023), em > 0; neg: of -x.
__device__ __forceinline__ long long fx_from(double x, int em, unsigned neg = 0u) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x), e = (hi >> 20) & 0x7ffu;
  const unsigned b = min(e, 1u);   // a subnormal has no hidden bit and the exponent of field 1
  const int d = min(em - 1 + (int)b - (int)e, 63);
  const unsigned mh = (__funnelshift_l(lo, hi, 8) & 0x0fffffffu) | (b << 28), ml = lo << 8;
  const unsigned long long M = (((unsigned long long)mh << 32) | ml) >> d;
  const long long s = (long long)((int)(hi ^ neg) >> 31);
  return ((long long)M ^ s) - s;
}

constexpr int kFxBad = 1 << 19;   // added to the exponent of a block with an infinity or a NaN

// R 2^(eb - 1084) rounded to nearest (zero below the normal range, infinity
// above it, NaN for a block that held an infinity or a NaN)
__device__ __forceinline__ double fx_to(long long R, int eb) {
  const int s = (int)(R >> 32) >> 31;
  const unsigned long long a = (unsigned long long)((R ^ (long long)s) - (long long)s);
  const unsigned a1 = (unsigned)(a >> 32), a0 = (unsigned)a;
  const bool low = a1 == 0u;
  const unsigned ah = low ? a0 : a1, al = low ? 0u : a0;
  const int z = __clz((int)ah);
  const int e = (low ? eb - 31 : eb + 1) - z;
  const unsigned nh = __funnelshift_l(al, ah, z), nl = __funnelshift_l(0u, al, z);
  const unsigned long long t =
      (((unsigned long long)((nh >> 11) + ((unsigned)e << 20)) << 32) | __funnelshift_r(nl, nh, 11)) +
      (unsigned long long)((nl >> 10) & 1u);
  unsigned th = (unsigned)(t >> 32), tl = (unsigned)t;
  if (nh == 0u || (unsigned)e >= 2046u) {
    tl = 0u;
    th = eb >= kFxBad ? 0x7ff80000u : (e >= 2046 ? 0x7ff00000u : 0u);
  }
  return __hiloint2double((int)(th | ((unsigned)s & 0x80000000u)), (int)tl);
}

// exponent of a block from the largest high word (sign cleared) of its values
__device__ __forceinline__ int fx_em(unsigned hmax) {
  const int e = (int)(hmax >> 20);
  return e == 2047 ? kFxBad + 2047 : max(e, 1);
}

// Whether the largest high word of a line is outside [2^-963, 2^1006) and not
// zero: infinities, NaNs, subnormals and what comes near them.  The phases of a
// residual give NaN for what meets an infinity or a NaN and zero below the normal
// range; the one-shot maps, whose results are the caller's, compute such an
// element in FP64 (the fx_..._ieee functions): infinities by value, subnormals.
__device__ __forceinline__ bool fx_wild(unsigned hmax) { return hmax - 0x03c00000u > 0x7b000000u && hmax != 0u; }

// shift that brings integers with OR of high words (one's complement) m to 61 bits
__device__ __forceinline__ int fx_shift(unsigned m) { return max(__clz((int)m) - 3, 0); }

__device__ __forceinline__ unsigned fx_mag(long long R) {
  const int h = (int)(R >> 32);
  return (unsigned)(h ^ (h >> 31));
}

// a b + c, 32 x 32 + 64 bits.  The low words pass through an empty asm statement
// (fx_split), so that the compiler does not know their sign: two steps of the
// mixed 16^3 mesh at N = 4 take 5.33 ms, 5.67 without (viscous 20^3 18.1, 19.1).
__device__ __forceinline__ long long fx_madw(int a, int b, long long c) { return (long long)a * b + c; }

__device__ __forceinline__ unsigned fx_hi(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

// Exponents of the lines between two passes: two sets of [5][n^2] lines, the
// second also as [4][5][n] lines of face values
template <int n>
__device__ __forceinline__ int* fx_exps() {
  __shared__ int e[5 * n * n + (n < 4 ? 20 * n : 5 * n * n)];
  return e;
}

// One lane's results R[0..n) of scale eb, brought to 61 bits and stored with
// the given stride; returns their exponent.
template <int n>
__device__ __forceinline__ int fx_store_line(const long long* R, int eb, long long* o, int stride) {
  unsigned mg = 0u;
#pragma unroll
  for (int i = 0; i < n; ++i) mg |= fx_mag(R[i]);
  const int k = fx_shift(mg);
#pragma unroll
  for (int i = 0; i < n; ++i) o[i * stride] = R[i] << k;
  return eb - k;
}

// The integers x[i stride] of exponents e[i estride] on the largest of them;
// returns it.
template <int n>
__device__ __forceinline__ int fx_load_aligned(const long long* x, int stride, const int* e, int estride, FxD* d) {
  int ei[n], em = e[0];
#pragma unroll
  for (int i = 0; i < n; ++i) {
    ei[i] = e[i * estride];
    em = max(em, ei[i]);
  }
#pragma unroll
  for (int i = 0; i < n; ++i) d[i] = fx_split(x[i * stride] >> min(em - ei[i], 63), 0);
  return em;
}

constexpr long long kFxHalf = 1ll << 30;   // rounds a sum's shift by 31 to nearest

// sum_m C(m) D_m 2^-62 over n terms; C(m) yields the coefficient pair
template <int n, class Coef>
__device__ __forceinline__ long long fx_dot(const FxD* d, Coef C, long long mid = kFxHalf) {
#pragma unroll
  for (int m = 0; m < n; ++m) {
    const int2 k = C(m);
    mid = fx_madw(d[m].h, k.y, mid);
    mid = fx_madw(d[m].l, k.x, mid);
  }
  long long hh = mid >> 31;
#pragma unroll
  for (int m = 0; m < n; ++m) hh = fx_madw(d[m].h, C(m).x, hh);
  return hh;
}

template <int n>
__device__ __forceinline__ bool fx_wild_line(const double* x) {
  bool w = false;
#pragma unroll
  for (int i = 0; i < n; ++i) w |= fx_wild(fx_hi(x[i]));
  return w;
}

// a + b on the larger of their exponents (returned in e), the other rounded to
// nearest: floors would lean every sum the same way (see S above).
__device__ __forceinline__ long long fx_sum(long long a, int ea, long long b, int eb, int& e) {
  const bool up = ea >= eb;
  const int k = min(up ? ea - eb : eb - ea, 61);
  e = up ? ea : eb;
  return (up ? a : b) + (((up ? b : a) + ((1ll << k) >> 1)) >> k);
}

// Exponent of n doubles (their largest) and their integers
template <int n>
__device__ __forceinline__ int fx_line(const double* x, FxD* d) {
  unsigned m = 0u;
#pragma unroll
  for (int i = 0; i < n; ++i) m = max(m, (unsigned)__double2hiint(x[i]) & 0x7fffffffu);
  const int em = fx_em(m);
#pragma unroll
  for (int i = 0; i < n; ++i) d[i] = fx_split(fx_from(x[i], em), 0);
  return em;
}

// ragged pass: outputs o < n of sum_t tab[t n + o] D_t, t < len
template <int n, class Load>
__device__ __forceinline__ void fx_ragged_out(const int2* tab, int len, Load load, long long* R) {
  long long mid[n], hh[n];
#pragma unroll
  for (int o = 0; o < n; ++o) {
    mid[o] = kFxHalf;
    hh[o] = 0;
  }
#pragma unroll 1
  for (int t = 0; t < len; ++t) {
    const FxD d = load(t);
#pragma unroll
    for (int o = 0; o < n; ++o) {
      const int2 k = __ldg(tab + t * n + o);
      mid[o] = fx_madw(d.h, k.y, mid[o]);
      mid[o] = fx_madw(d.l, k.x, mid[o]);
      hh[o] = fx_madw(d.h, k.x, hh[o]);
    }
  }
#pragma unroll
  for (int o = 0; o < n; ++o) R[o] = hh[o] + (mid[o] >> 31);
}

// Line `id` of direction l: start index and stride in the nodal block, and
// the two other indices (x1 < x2 by coordinate; face point x1 + n x2)
template <int n>
__device__ __forceinline__ void fx_line_of(int l, int id, int& start, int& stride, int& fp) {
  const int x1 = id / n, x2 = id - x1 * n;
  start = l == 0 ? id : (l == 1 ? x1 * n * n + x2 : id * n);
  stride = l == 0 ? n * n : (l == 1 ? n : 1);
  fp = x1 + n * x2;
}

// The face values at both ends of one line of direction l
template <int n, class Out>
__device__ __forceinline__ void fx_line_ends(const TypeTab& T, int l, int v, int fp, const double* x, Out out) {
  using Tab = FxTab<n>;
  FxD d[n];
  const int eb = fx_line<n>(x, d) + 1 + kFxGE;
  const int lf0 = __ldg(&T.face_of[2 * l]), lf1 = __ldg(&T.face_of[2 * l + 1]);
  if (lf0 >= 0) out(lf0, v, fp, fx_to(fx_dot<n>(d, [&](int m) { return Tab::E(0, m); }), eb));
  if (lf1 >= 0) out(lf1, v, fp, fx_to(fx_dot<n>(d, [&](int m) { return Tab::E(1, m); }), eb));
}

// Values of the nodal field src [5][nQ] on the element's own face points:
// out(local face, variable, face point, value), directions l0..2.  The faces
// at both ends of a coordinate share the line's integers.
template <int n, class Out>
__device__ __forceinline__ void fx_traces(const TypeTab& T, const double* src, Out out, int l0 = 0) {
  constexpr int n2 = n * n, nQ = n2 * n;
#pragma unroll 1
  for (int t0 = l0 * 5 * n2 + threadIdx.x; t0 < 15 * n2; t0 += blockDim.x) {
    const int l = t0 / (5 * n2), r = t0 - l * 5 * n2, v = r / n2;
    int st, sd, fp;
    fx_line_of<n>(l, r - v * n2, st, sd, fp);
    const double* s = src + v * nQ + st;
    double x[n];
#pragma unroll
    for (int m = 0; m < n; ++m) x[m] = s[m * sd];
    fx_line_ends<n>(T, l, v, fp, x, out);
  }
}

// The transforms in FP64, for elements the integers do not hold (fx_wild): the
// sum-factorised passes, one output per lane at a time.
template <int n>
__device__ __forceinline__ void fx_nodal_ieee(const Ctx& c, const TypeTab& T, const double* sQ, double* bufA, double* bufB) {
  constexpr int n2 = n * n, nQ = n2 * n;
  const double* dp = c.dpool;
  const int* ip = c.ipool;
  const int nM = T.nM, cn = T.ncols * n;
  for (int o = threadIdx.x; o < 5 * cn; o += blockDim.x) {
    const int v = o / cn, r = o - v * cn, col = r / n;
    const double* C = dp + T.C + ip[T.col_coff + col] + r - col * n;
    const double* q = sQ + v * nM + ip[T.col_moff + col];
    double acc = 0.0;
#pragma unroll 1
    for (int t = 0; t < ip[T.col_len + col]; ++t) acc = fma(C[t * n], q[t], acc);
    bufA[v * nQ + r] = acc;
  }
  __syncthreads();
  for (int o = threadIdx.x; o < 5 * nQ; o += blockDim.x) {
    const int v = o / nQ, r = o - v * nQ, p = r / n2, j = r / n % n, k = r % n;
    const double* B = dp + T.B + ip[T.p_boff + p] + j;
    const double* X = bufA + v * nQ + ip[T.p_cbase + p] * n + k;
    double acc = 0.0;
#pragma unroll 1
    for (int t = 0; t < ip[T.p_blen + p]; ++t) acc = fma(B[t * n], X[t * n], acc);
    bufB[o] = acc;
  }
  __syncthreads();
  for (int o = threadIdx.x; o < 5 * nQ; o += blockDim.x) {
    const int v = o / nQ, r = o - v * nQ, i = r / n2;
    double acc = 0.0;
#pragma unroll 1
    for (int p = 0; p < n; ++p) acc = fma(dp[T.A + p * n + i], bufB[v * nQ + p * n2 + r % n2], acc);
    bufA[o] = acc;
  }
  __syncthreads();
}

// bufA [5][nQ] (destroyed) -> r [5][nM]; r may alias bufB, not bufA
template <int n>
__device__ __forceinline__ void fx_modal_ieee(const Ctx& c, const TypeTab& T, double* bufA, double* bufB, double* r) {
  constexpr int n2 = n * n, nQ = n2 * n;
  const double* dp = c.dpool;
  const int* ip = c.ipool;
  const int nM = T.nM, cn = T.ncols * n;
  for (int o = threadIdx.x; o < 5 * nQ; o += blockDim.x) {
    const int v = o / nQ, w = o - v * nQ, p = w / n2;
    double acc = 0.0;
#pragma unroll 1
    for (int i = 0; i < n; ++i) acc = fma(dp[T.A + p * n + i], bufA[v * nQ + i * n2 + w % n2], acc);
    bufB[o] = acc;
  }
  __syncthreads();
  for (int o = threadIdx.x; o < 5 * cn; o += blockDim.x) {
    const int v = o / cn, w = o - v * cn, col = w / n, p = ip[T.col_p + col];
    const double* B = dp + T.B + ip[T.p_boff + p] + (col - ip[T.p_cbase + p]) * n;
    double acc = 0.0;
#pragma unroll 1
    for (int j = 0; j < n; ++j) acc = fma(B[j], bufB[v * nQ + p * n2 + j * n + w % n], acc);
    bufA[v * nQ + w] = acc;
  }
  __syncthreads();
  for (int o = threadIdx.x; o < 5 * nM; o += blockDim.x) {
    const int v = o / nM, mode = o - v * nM, col = ip[T.mode_col + mode];
    const double* C = dp + T.C + ip[T.col_coff + col] + (mode - ip[T.col_moff + col]) * n;
    double acc = 0.0;
#pragma unroll 1
    for (int k = 0; k < n; ++k) acc = fma(C[k], bufA[v * nQ + col * n + k], acc);
    r[o] = acc;
  }
  __syncthreads();
}

// Modal -> nodal, U = V Q: sQ [5][nM] doubles -> bufA [5][nQ] doubles, bufB
// [5][nQ] scratch (sQ may alias bufB).  Passes c, b, a, one line per lane.
// TR: the values at the element's face points too, out(local face, variable,
// face point, value), bit for bit fx_traces of U (the a faces by the lane that
// forms the line).  IEEE: an element of fx_wild's range goes through FP64.
template <int n, bool TR, bool IEEE, class Out>
__device__ __forceinline__ void fx_to_nodal(const Ctx& c, const TypeTab& T, const double* sQ, double* bufA,
                                            double* bufB, Out out) {
  constexpr int n2 = n * n, nQ = n2 * n;
  using Tab = FxTab<n>;
  int* e0 = fx_exps<n>();
  int* e1 = e0 + 5 * n2;
  const int* ip = c.ipool;
  const int nM = T.nM, ncols = T.ncols, nt = blockDim.x;
  long long* X = reinterpret_cast<long long*>(bufA);
  long long* Y = reinterpret_cast<long long*>(bufB);
  const bool uc = T.type == HEX || T.type == PRISM, ub = T.type == HEX || T.type == PYR;
  unsigned wild = 0u;
  // c-pass: X[col][k] = sum_t C[col][t][k] Q[moff[col] + t]
  for (int t0 = threadIdx.x; t0 < 5 * ncols; t0 += nt) {
    const int v = t0 / ncols, col = t0 - v * ncols;
    long long R[n];
    int eb;
    if (uc) {
      const double* q = sQ + v * nM + col * n;
      double x[n];
#pragma unroll
      for (int t = 0; t < n; ++t) x[t] = q[t];
      if (IEEE) wild |= fx_wild_line<n>(x);
      FxD d[n];
      eb = fx_line<n>(x, d) + 1 + Tab::gA;
#pragma unroll
      for (int k = 0; k < n; ++k) R[k] = fx_dot<n>(d, [&](int t) { return Tab::A(t, k); });
    } else {
      const double* q = sQ + v * nM + __ldg(ip + T.col_moff + col);
      const int len = __ldg(ip + T.col_len + col);
      const int* ms = ip + T.mode_s + (q - sQ - v * nM);
      int em = fx_em(fx_hi(q[0])) + __ldg(ms);
      for (int t = 1; t < len; ++t) em = max(em, fx_em(fx_hi(q[t])) + __ldg(ms + t));
      if (IEEE)
        for (int t = 0; t < len; ++t) wild |= fx_wild(fx_hi(q[t]));
      eb = em + 1 + kFxGR;
      fx_ragged_out<n>(c.fpool + T.C + __ldg(ip + T.col_coff + col), len,
                       [&](int t) { return fx_split(fx_from(q[t], em - __ldg(ms + t)), 0); }, R);
    }
    e0[v * n2 + col] = fx_store_line<n>(R, eb, X + v * nQ + col * n, 1);
  }
  if (IEEE) {
    static_assert(!(TR && IEEE), "the one-shot maps take no traces");
    if (__syncthreads_or(wild)) {
      fx_nodal_ieee<n>(c, T, sQ, bufA, bufB);
      return;
    }
  } else {
    __syncthreads();
  }
  // b-pass: Y[p][j][k] = sum_t B[p][t][j] X[cbase[p] + t][k]
  for (int t0 = threadIdx.x; t0 < 5 * n2; t0 += nt) {
    const int v = t0 / n2, pk = t0 - v * n2, p = pk / n, k = pk - p * n;
    const int cb = __ldg(ip + T.p_cbase + p);
    long long R[n];
    int eb;
    const long long* x = X + v * nQ + cb * n + k;
    const int* e = e0 + v * n2 + cb;
    if (ub) {
      FxD d[n];
      eb = fx_load_aligned<n>(x, n, e, 1, d) + Tab::gA;
#pragma unroll
      for (int j = 0; j < n; ++j) R[j] = fx_dot<n>(d, [&](int t) { return Tab::A(t, j); });
    } else {
      const int len = __ldg(ip + T.p_blen + p);
      const int* cs = ip + T.col_s + cb;
      int em = e[0] + __ldg(cs);
      for (int t = 1; t < len; ++t) em = max(em, e[t] + __ldg(cs + t));
      eb = em + kFxGR;
      fx_ragged_out<n>(c.fpool + T.B + __ldg(ip + T.p_boff + p), len,
                       [&](int t) { return fx_split(x[t * n] >> min(em - e[t] - __ldg(cs + t), 63), 0); }, R);
    }
    e1[v * n2 + pk] = fx_store_line<n>(R, eb, Y + v * nQ + p * n2 + k, n);
  }
  __syncthreads();
  // a-pass: U[i][j][k] = sum_p A[p][i] Y[p][j][k]
  for (int t0 = threadIdx.x; t0 < 5 * n2; t0 += nt) {
    const int v = t0 / n2, jk = t0 - v * n2, j = jk / n, k = jk - j * n;
    FxD d[n];
    const int eb = fx_load_aligned<n>(Y + v * nQ + jk, n2, e1 + v * n2 + k, n, d) + Tab::gA;
    double* o = bufA + v * nQ + jk;
#pragma unroll kUnroll
    for (int i = 0; i < n; ++i) o[i * n2] = fx_to(fx_dot<n>(d, [&](int p) { return Tab::A(p, i); }), eb);
    if (TR) {
      double x[n];
#pragma unroll
      for (int i = 0; i < n; ++i) x[i] = o[i * n2];
      fx_line_ends<n>(T, 0, v, j + n * k, x, out);
    }
  }
  __syncthreads();
  if (TR) {
    fx_traces<n>(T, bufA, out, 1);
    __syncthreads();
  }
}

// The b and c passes of V^T: Y [5][nQ] (integers of the a-pass, their lines'
// exponents in fx_exps) -> r [5][nM] doubles.  X [5][nQ] scratch; r may alias Y.
template <int n>
__device__ __forceinline__ void fx_modal_tail(const Ctx& c, const TypeTab& T, const long long* Y, long long* X,
                                              double* r) {
  constexpr int n2 = n * n, nQ = n2 * n;
  using Tab = FxTab<n>;
  const int* e0 = fx_exps<n>();
  int* e1 = fx_exps<n>() + 5 * n2;
  const int* ip = c.ipool;
  const int nM = T.nM, ncols = T.ncols, nt = blockDim.x;
  const bool uc = T.type == HEX || T.type == PRISM, ub = T.type == HEX || T.type == PYR;
  // b-pass: X[cbase[p] + t][k] = sum_j B[p][t][j] Y[p][j][k]
  for (int t0 = threadIdx.x; t0 < 5 * n2; t0 += nt) {
    const int v = t0 / n2, pk = t0 - v * n2, p = pk / n, k = pk - p * n;
    FxD d[n];
    int eb = fx_load_aligned<n>(Y + v * nQ + p * n2 + k, n, e0 + v * n2 + k, n, d);
    long long* o = X + v * nQ + __ldg(ip + T.p_cbase + p) * n + k;
    if (ub) {
      long long R[n];
#pragma unroll
      for (int t = 0; t < n; ++t) R[t] = fx_dot<n>(d, [&](int j) { return Tab::A(t, j); });
      eb = fx_store_line<n>(R, eb + Tab::gA, o, n);
    } else {
      const int2* B = c.fpool + T.B + __ldg(ip + T.p_boff + p);
      const int len = __ldg(ip + T.p_blen + p);
      unsigned mg = 0u;
#pragma unroll 1
      for (int t = 0; t < len; ++t) {
        const long long R = fx_dot<n>(d, [&](int j) { return __ldg(B + t * n + j); });
        o[t * n] = R;
        mg |= fx_mag(R);
      }
      const int s = fx_shift(mg);
      for (int t = 0; t < len; ++t) o[t * n] <<= s;
      eb += kFxGR - s;
    }
    e1[v * n2 + pk] = eb;
  }
  __syncthreads();
  // c-pass: r[moff[col] + t] = sum_k C[col][t][k] X[col][k]
  for (int t0 = threadIdx.x; t0 < 5 * ncols; t0 += nt) {
    const int v = t0 / ncols, col = t0 - v * ncols;
    FxD d[n];
    // ub: the b-pass used the unscaled table
    const int em = fx_load_aligned<n>(X + v * nQ + col * n, 1, e1 + v * n2 + __ldg(ip + T.col_p + col) * n, 1, d) +
                   (ub ? 0 : __ldg(ip + T.col_s + col));
    if (uc) {
      double* o = r + v * nM + col * n;
#pragma unroll kUnroll
      for (int t = 0; t < n; ++t) o[t] = fx_to(fx_dot<n>(d, [&](int k) { return Tab::A(t, k); }), em + Tab::gA);
    } else {
      const int2* C = c.fpool + T.C + __ldg(ip + T.col_coff + col);
      const int len = __ldg(ip + T.col_len + col), mo = __ldg(ip + T.col_moff + col);
      const int* ms = ip + T.mode_s + mo;
      double* o = r + v * nM + mo;
#pragma unroll 1
      for (int t = 0; t < len; ++t)
        o[t] = fx_to(fx_dot<n>(d, [&](int k) { return __ldg(C + t * n + k); }), em + kFxGR + __ldg(ms + t));
    }
  }
  __syncthreads();
}

// Nodal -> modal transpose, r = V^T h: bufA [5][nQ] doubles (destroyed) ->
// r [5][nM] doubles; bufB [5][nQ] scratch (r may alias bufB, not bufA).
template <int n, bool IEEE>
__device__ __forceinline__ void fx_to_modal(const TypeTab& T, const Ctx& c, double* bufA, double* bufB, double* r) {
  constexpr int n2 = n * n, nQ = n2 * n;
  using Tab = FxTab<n>;
  int* e0 = fx_exps<n>();
  long long* Y = reinterpret_cast<long long*>(bufB);
  unsigned wild = 0u;
  // a-pass: Y[p][j][k] = sum_i A[p][i] h[i][j][k]
  for (int t0 = threadIdx.x; t0 < 5 * n2; t0 += blockDim.x) {
    const int v = t0 / n2, jk = t0 - v * n2;
    const double* h = bufA + v * nQ + jk;
    double x[n];
#pragma unroll
    for (int i = 0; i < n; ++i) x[i] = h[i * n2];
    if (IEEE) wild |= fx_wild_line<n>(x);
    FxD d[n];
    const int eb = fx_line<n>(x, d) + 1 + Tab::gA;
    long long R[n];
#pragma unroll
    for (int p = 0; p < n; ++p) R[p] = fx_dot<n>(d, [&](int i) { return Tab::A(p, i); });
    e0[v * n2 + jk] = fx_store_line<n>(R, eb, Y + v * nQ + jk, n2);
  }
  if (IEEE) {
    if (__syncthreads_or(wild)) {
      fx_modal_ieee<n>(c, T, bufA, bufB, r);
      return;
    }
  } else {
    __syncthreads();
  }
  fx_modal_tail<n>(c, T, Y, reinterpret_cast<long long*>(bufA), r);
}

// r = V^T (H +- sum_f E_f^T F_f) of a prism, pyramid or tetrahedron: H(o) the
// nodal value at v nQ + q, F(f, v, p) the face values (each read once); neg
// 0x80000000 subtracts.  The sum stays in integers between the lift and the
// transform: a lane owns the line (j, k), takes its n values of H, adds the b
// and c face values with the two end coefficients of its j and k and the a
// face values with the line's, and goes on with the a-pass.  A line of face
// values along i keeps its own exponent, and the lane works on the largest of
// what meets on its line.  bufA [5][nQ], bufG [30 n^2] scratch (STAGE: H lies in
// global memory and is staged in bufA with the face values); r [5][nM] may be
// bufA or lie behind bufG's first 5 nQ.
template <int n, bool STAGE, class LoadH, class LoadF>
__device__ __forceinline__ void fx_lift_to_modal(const Ctx& c, const TypeTab& T, LoadH H, LoadF F, unsigned neg,
                                                 double* bufA, double* bufG, double* r) {
  constexpr int n2 = n * n, nQ = n2 * n;
  using Tab = FxTab<n>;
  int* e0 = fx_exps<n>();
  int* ef = e0 + 5 * n2;                 // [end][5][n] exponents of the b and c face lines
  const int nt = blockDim.x;
  long long* Y = reinterpret_cast<long long*>(bufA);
  long long* FI = reinterpret_cast<long long*>(bufG);   // [end][5][n^2], ends -b, +b, -c, +c
  double* FA = bufG + 20 * n2;                          // [2][5][n^2], ends -a, +a
  const int fa0 = __ldg(&T.face_of[0]), fa1 = __ldg(&T.face_of[1]);
  for (int t0 = threadIdx.x; t0 < 5 * n2; t0 += nt) {
    const int v = t0 / n2, jk = t0 - v * n2, j = jk / n, k = jk - j * n;
    if (STAGE) {
#pragma unroll
      for (int i = 0; i < n; ++i) bufA[v * nQ + jk + i * n2] = H(v * nQ + jk + i * n2);
    }
    FA[t0] = F(fa0, v, j + n * k);
    FA[5 * n2 + t0] = F(fa1, v, j + n * k);
  }
  for (int t0 = threadIdx.x; t0 < 20 * n; t0 += nt) {
    const int e = t0 / (5 * n), w = t0 - e * 5 * n, v = w / n, y = w - v * n;
    const int lf = __ldg(&T.face_of[2 + e]);
    if (lf < 0) continue;
    double x[n];
    unsigned m = 0u;
#pragma unroll
    for (int i = 0; i < n; ++i) {
      x[i] = F(lf, v, n * y + i);
      m = max(m, fx_hi(x[i]));
    }
    const int em = fx_em(m);
#pragma unroll
    for (int i = 0; i < n; ++i) FI[(e * 5 + v) * n2 + n * y + i] = fx_from(x[i], em, neg);
    ef[t0] = em;
  }
  __syncthreads();
  const int2* E = c.fpool + T.ext;
  for (int t0 = threadIdx.x; t0 < 5 * n2; t0 += nt) {
    const int v = t0 / n2, jk = t0 - v * n2, j = jk / n, k = jk - j * n;
    const double a0 = FA[t0], a1 = FA[5 * n2 + t0];
    double h[n];
    unsigned m = max(fx_hi(a0), fx_hi(a1));
#pragma unroll
    for (int i = 0; i < n; ++i) {
      h[i] = STAGE ? bufA[v * nQ + jk + i * n2] : H(v * nQ + jk + i * n2);
      m = max(m, fx_hi(h[i]));
    }
    int em = fx_em(m);
#pragma unroll 1
    for (int e = 0; e < 4; ++e)
      if (__ldg(&T.face_of[2 + e]) >= 0) em = max(em, ef[(e * 5 + v) * n + (e < 2 ? k : j)]);
    long long mid[n], hh[n], half = kFxHalf;
#pragma unroll
    for (int i = 0; i < n; ++i) {
      hh[i] = fx_from(h[i], em + kFxGE);
      mid[i] = 0;
    }
    // b faces (line value at (i, k), coefficient of j), then c faces ((i, j), of k)
#pragma unroll 1
    for (int e = 0; e < 4; ++e) {
      if (__ldg(&T.face_of[2 + e]) < 0) continue;
      const int2 co = __ldg(E + (e & 1) * n + (e < 2 ? j : k));
      const int fl = e * 5 + v, y = e < 2 ? k : j, sh = min(em - ef[fl * n + y], 63);
      const long long* f = FI + fl * n2 + n * y;
      half += co.y >> 1;   // the mean of the dl cl products (S above)
#pragma unroll
      for (int i = 0; i < n; ++i) {
        const FxD d = fx_split(f[i] >> sh, 0);
        mid[i] = fx_madw(d.h, co.y, mid[i]);
        mid[i] = fx_madw(d.l, co.x, mid[i]);
        hh[i] = fx_madw(d.h, co.x, hh[i]);
      }
    }
    unsigned mg = 0u;
    {
      const FxD d0 = fx_split(fx_from(a0, em, neg), 0), d1 = fx_split(fx_from(a1, em, neg), 0);
#pragma unroll
      for (int i = 0; i < n; ++i) {
        const int2 c0 = Tab::E(0, i), c1 = Tab::E(1, i);
        mid[i] = fx_madw(d0.h, c0.y, mid[i]);
        mid[i] = fx_madw(d0.l, c0.x, mid[i]);
        mid[i] = fx_madw(d1.h, c1.y, mid[i]);
        mid[i] = fx_madw(d1.l, c1.x, mid[i]);
        hh[i] = fx_madw(d0.h, c0.x, hh[i]);
        hh[i] = fx_madw(d1.h, c1.x, hh[i]);
        hh[i] += (mid[i] + half + ((c0.y + c1.y) >> 1)) >> 31;
        mg |= fx_mag(hh[i]);
      }
    }
    const int ks = fx_shift(mg);
    FxD d[n];
#pragma unroll
    for (int i = 0; i < n; ++i) d[i] = fx_split(hh[i], ks);
    long long R[n];
#pragma unroll
    for (int p = 0; p < n; ++p) R[p] = fx_dot<n>(d, [&](int i) { return Tab::A(p, i); });
    e0[v * n2 + jk] = fx_store_line<n>(R, em + 1 + kFxGE + Tab::gA - ks, Y + v * nQ + jk, n2);
  }
  __syncthreads();
  fx_modal_tail<n>(c, T, Y, FI, r);
}

// out = sum over the directions l in `dirs` of D_l^T G_l (collocation
// derivative): load(l, v, q) gives G_l at point q, read once.  out [5][nQ]
// (shared or global); tmp [5][nQ] scratch, which may be G_2 itself.  Every line
// keeps the exponent of its own values: a hexahedron's results are its nodal
// rates, and those of a line of small values are not to depend on a large value
// elsewhere in the element.  The directions' sums meet at a point on the largest
// of the exponents of the lines through it.
template <int n, class Load>
__device__ __forceinline__ void fx_dsum(Load load, unsigned dirs, double* tmp, double* out) {
  constexpr int n2 = n * n, nQ = n2 * n;
  using Tab = FxTab<n>;
  long long* A = reinterpret_cast<long long*>(tmp);
  int* es = fx_exps<n>();   // the lines' exponents: direction 2, direction 1
  bool first = true;
#pragma unroll 1
  for (int l = 2; l >= 0; --l) {
    if (!((dirs >> l) & 1u)) continue;
    const bool last = (dirs & ((1u << l) - 1u)) == 0u;
    // exponent of the sum so far at point m of a line: the largest of its lines';
    // a line's results are below 2^61, three of them below 2^63
    const bool two = l == 0 && (dirs & 6u) == 6u;
    const bool by1 = l == 0 && !(dirs & 4u);
    for (int t0 = threadIdx.x; t0 < 5 * n2; t0 += blockDim.x) {
      const int v = t0 / n2, id = t0 - v * n2, x1 = id / n, x2 = id - x1 * n;
      int st, sd, fp;
      fx_line_of<n>(l, id, st, sd, fp);
      double x[n];
#pragma unroll
      for (int m = 0; m < n; ++m) x[m] = load(l, v, st + m * sd);
      FxD d[n];
      const int eb = fx_line<n>(x, d) + 1 + Tab::gD;
      const int o = v * nQ + st;
      if (first) {
#pragma unroll kUnroll
        for (int i = 0; i < n; ++i) {
          const long long R = fx_dot<n>(d, [&](int m) { return Tab::D(i, m); }, Tab::S(i));
          if (last) out[o + i * sd] = fx_to(R, eb);
          else A[o + i * sd] = R;
        }
      } else {
        // the lines through a point of this one: direction 2 (x_0, x_1), direction 1 (x_0, x_2)
        const int* e2 = es + v * n2 + (l == 1 ? x1 * n : x1);
        const int* e1 = es + (5 + v) * n2 + x2;
        const int* p = by1 ? e1 : e2;
        const int* q = two ? e1 : p;
        const int se = l == 1 ? 1 : n;
#pragma unroll kUnroll
        for (int i = 0; i < n; ++i) {
          const long long R = fx_dot<n>(d, [&](int m) { return Tab::D(i, m); }, Tab::S(i));
          int e;
          const long long r = fx_sum(A[o + i * sd], max(p[i * se], q[i * se]), R, eb, e);
          if (last) out[o + i * sd] = fx_to(r, e);
          else A[o + i * sd] = r;
        }
      }
      if (!last) es[(l == 2 ? 0 : 5 * n2) + v * n2 + id] = eb;
    }
    first = false;
    __syncthreads();
  }
}

// dst_l = D_l src (the transposed derivative tables), l = 0..2: dst [3][5][nQ]
template <int n>
__device__ __forceinline__ void fx_grad(const double* src, double* dst) {
  constexpr int n2 = n * n, nQ = n2 * n;
  using Tab = FxTab<n>;
  for (int t0 = threadIdx.x; t0 < 15 * n2; t0 += blockDim.x) {
    const int l = t0 / (5 * n2), r = t0 - l * 5 * n2, v = r / n2;
    int st, sd, fp;
    fx_line_of<n>(l, r - v * n2, st, sd, fp);
    const double* s = src + v * nQ + st;
    double x[n];
#pragma unroll
    for (int m = 0; m < n; ++m) x[m] = s[m * sd];
    FxD d[n];
    const int eb = fx_line<n>(x, d) + 1 + Tab::gD;
    double* o = dst + (5 * l + v) * nQ + st;
#pragma unroll
    for (int i = 0; i < n; ++i) o[i * sd] = fx_to(fx_dot<n>(d, [&](int m) { return Tab::D(m, i); }), eb);
  }
  __syncthreads();
}

// dst = D_l src along one direction
template <int n>
__device__ __forceinline__ void fx_grad1(int l, const double* src, double* dst) {
  constexpr int n2 = n * n, nQ = n2 * n;
  using Tab = FxTab<n>;
  for (int t0 = threadIdx.x; t0 < 5 * n2; t0 += blockDim.x) {
    const int v = t0 / n2;
    int st, sd, fp;
    fx_line_of<n>(l, t0 - v * n2, st, sd, fp);
    const double* s = src + v * nQ + st;
    double x[n];
#pragma unroll
    for (int m = 0; m < n; ++m) x[m] = s[m * sd];
    FxD d[n];
    const int eb = fx_line<n>(x, d) + 1 + Tab::gD;
    double* o = dst + v * nQ + st;
#pragma unroll
    for (int i = 0; i < n; ++i) o[i * sd] = fx_to(fx_dot<n>(d, [&](int m) { return Tab::D(m, i); }), eb);
  }
  __syncthreads();
}

// out(o, h) with h = H(o) + sum_f E_f^T (+-F_f) at every node o = v nQ + q: F
// [nf][5][n^2] doubles (shared); neg 0x80000000 subtracts; A [5][nQ] scratch.
// The lane that puts out(o) reads H(o) just before, so out may write where H
// reads, or to A.  The two face values at the ends of a line share an exponent,
// and the sums meet H at each node on the largest of that node's own.
template <int n, class LoadH, class Out>
__device__ __forceinline__ void fx_lift(const TypeTab& T, LoadH H, const double* F, unsigned neg, double* scratch,
                                        Out out) {
  constexpr int n2 = n * n, nQ = n2 * n;
  using Tab = FxTab<n>;
  long long* A = reinterpret_cast<long long*>(scratch);
  int* es = fx_exps<n>();   // the lines' exponents: direction 2, direction 1
#pragma unroll 1
  for (int l = 2; l >= 0; --l) {
    const int lf0 = T.face_of[2 * l], lf1 = T.face_of[2 * l + 1];
    for (int t0 = threadIdx.x; t0 < 5 * n2; t0 += blockDim.x) {
      const int v = t0 / n2, id = t0 - v * n2, x1 = id / n, x2 = id - x1 * n;
      int st, sd, fp;
      fx_line_of<n>(l, id, st, sd, fp);
      double f[2];
      f[0] = lf0 >= 0 ? F[(lf0 * 5 + v) * n2 + fp] : 0.0;
      f[1] = lf1 >= 0 ? F[(lf1 * 5 + v) * n2 + fp] : 0.0;
      // 62 bits of each value: two end coefficients sum to less than 2, so a
      // line's results stay below 2^60, and three of them with H below 2^63
      FxD d[2];
      const int em = fx_em(max(fx_hi(f[0]), fx_hi(f[1]))), eb = em + kFxGE;
      d[0] = fx_split(fx_from(f[0], em, neg), 1);
      d[1] = fx_split(fx_from(f[1], em, neg), 1);
      const int o = v * nQ + st;
      // the lines through a point of this one: direction 2 (x_0, x_1), direction 1 (x_0, x_2)
      const int* e2 = es + v * n2 + (l == 1 ? x1 * n : x1);
      const int* e1 = es + (5 + v) * n2 + x2;
#pragma unroll kUnroll
      for (int i = 0; i < n; ++i) {
        const long long R = fx_dot<2>(d, [&](int e) { return Tab::E(e, i); });
        long long& a = A[o + i * sd];
        if (l == 2) {
          a = R;
        } else if (l == 1) {
          int e;
          a = fx_sum(a, e2[i], R, eb, e);
        } else {
          const double h = H(o + i * sd);
          const int eh = fx_em(fx_hi(h)) + 1;
          int e;
          long long r = fx_sum(a, max(e2[i * n], e1[i * n]), R, eb, e);
          r = fx_sum(r, e, fx_from(h, eh - 1), eh, e);
          out(o + i * sd, fx_to(r, e));
        }
      }
      if (l > 0) es[(l == 2 ? 0 : 5 * n2) + v * n2 + id] = eb;
    }
    __syncthreads();
  }
}

// out(mode, acc[5]) = Md r: the dense inverse mass matrix of a curved element
// (Algorithm 1 with a pointwise J), Md [nM][nM] in global memory, symmetric, r
// [5][nM] in shared memory.  Lanes run over output modes, so the column reads of
// Md are coalesced and every load feeds 5 sums.  In FP64: the modes of r and the
// entries of a row of Md span many orders, and the small ones count in theirs.
// What bounds it is the latency of Md's loads (two curved 12^3 steps at N = 4:
// 3.95 ms; 4.02 on integers with one exponent for all of r and one for Md, which
// left modes that decay over twelve orders 1e-8 of themselves off).
template <class Out>
__device__ __forceinline__ void dense_product(const double* Md, const double* r, int nM, Out out) {
  for (int a = threadIdx.x; a < nM; a += blockDim.x) {
    const double* Mc = Md + a;
    double acc[5] = {0, 0, 0, 0, 0};
#pragma unroll 4
    for (int j = 0; j < nM; ++j) {
      const double m = Mc[(size_t)j * nM];
#pragma unroll
      for (int v = 0; v < 5; ++v) acc[v] = fma(m, r[v * nM + j], acc[v]);
    }
    out(a, acc);
  }
}

}  // namespace
}  // namespace dgk
