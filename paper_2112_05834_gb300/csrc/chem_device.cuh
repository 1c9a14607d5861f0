// Device code of the batched stiff-chemistry integrator (sm_103a), shared by the
// translation units that instantiate the integration kernel (chem_kernels.cu: the
// RODAS4 stepper, diagnostics and launchers; chem_kernels_w.cu: the W-method).
//
// One CTA integrates one cell at a time; its warps share the cell's work:
// species and 32-reaction chunks are dealt over threads and warps for the rates,
// Jacobian rows over warps (columns over lanes) for the assembly; the FP64 form
// factorises in shared memory (rows over warps) and solves on one warp, the mixed
// form inverts in FP32 with the matrix in registers (columns over warps, rows over
// lanes) and solves by matrix-vector products over all threads. All per-cell data
// (state, stage vectors, per-reaction derivative data, the iteration matrix) lives
// in shared memory, except that the mixed form may keep its assembled matrix (float-
// float pairs) in a global-memory slot of the CTA when that lets more CTAs share an SM; the
// mechanism tables are read through the L1 cache.
//
// Paper mapping: rates and RHS = pyJac's reaction-rate evaluation; analytic
// Jacobian = pyJac's Jacobian (Methodology, "Analytical Jacobian and improved ODE
// solution"); LU + substitution = the LAPACK replacement of OpenFOAM's linear
// algebra (same section); the per-cell loop = the implicit ODE solver of the
// Introduction; the work queue = DLBFoam's redistribution of cell problems
// (Methodology, "DLBFoam: Dynamic load balancing"), reinterpreted inside one GPU.
#pragma once

#include <cuda_runtime.h>

#include <cfloat>
#include <cmath>
#include <cstdint>
#include <type_traits>

#include "chem.h"
#include "chem_fixed.cuh"
#include "chem_internal.h"
#include "chem_kernels.h"
#include "rodas4.h"

namespace chem {

#define FULLMASK 0xffffffffu

// ---------------------------------------------------------------------------
// Float-float arithmetic (a value is hi + lo with two FP32 numbers, |lo| below ulp(hi)):
// error-free products with FMA (Dekker's TwoProduct) and sums by Knuth's TwoSum
// give about 44-48 significant bits on the FP32 pipe. On GB300 an SM's FP32 pipe
// completes 64 times the operations per clock of its FP64 pipe, which the
// integration keeps busy, so the mixed form runs its long sums of products here:
// third-body concentrations, the Jacobian assembly and the refinement residuals.
// The _rn intrinsics keep the compiler from contracting a product and a sum into
// one FMA, which would break the error-free transformations.
// ---------------------------------------------------------------------------
struct __align__(8) ff2 {
  float hi, lo;
};
// Conversions between FP64 and FP32 run on the FP64 pipe on this part, at its rate,
// so the splits and widenings below use integer operations on the bit patterns.
// Double to float-float: hi = x truncated to 24 significant bits, lo = x - hi (the
// 29 remaining mantissa bits, rounded to 24 by the integer-to-float conversion and
// scaled by an exact power of two). In FP32's subnormal range (2^-149 <= |x| <
// 2^-126) hi = x truncated to a multiple of 2^-149 and lo = 0; below it (0, 0);
// |x| >= 2^128 gives +-inf (NaN stays NaN) with lo = 0.
__device__ __forceinline__ ff2 ff_split(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned hw = (unsigned)(b >> 32), lw = (unsigned)b;
  const unsigned sgn = hw & 0x80000000u;
  const int e = (int)((hw >> 20) & 0x7FFu);
  const float m = __uint2float_rn(lw & 0x1FFFFFFFu);
  // m 2^(e - 1075) as one power-of-two factor for e >= 949, else as 2^(e - 1011) 2^-64
  const bool big = e >= 949;
  const float s1 = __uint_as_float((unsigned)(big ? e - 948 : e - 884) << 23);
  const float s2 = big ? 1.0f : __uint_as_float(0x1F800000u);  // 2^-64
  ff2 r = {__uint_as_float(sgn | ((unsigned)(e - 896) << 23) | ((hw & 0xFFFFFu) << 3) | (lw >> 29)),
           __uint_as_float(__float_as_uint(__fmul_rn(__fmul_rn(m, s1), s2)) | sgn)};
  if (e < 897) {
    const int sh = 926 - e;  // the 53-bit significand times 2^(e - 1075) in units of 2^-149
    const unsigned frac = sh <= 52 ? (unsigned)(((1ull << 52) | (b & 0xFFFFFFFFFFFFFull)) >> sh) : 0u;
    r = {__uint_as_float(sgn | frac), 0.0f};
  }
  if (e > 1150) {
    const bool nan = e == 2047 && ((hw & 0xFFFFFu) | lw) != 0u;
    r = {__uint_as_float(sgn | 0x7F800000u | (nan ? 0x400000u : 0u)), 0.0f};
  }
  return r;
}
// float to double, exactly
__device__ __forceinline__ double f32_to_f64(float f) {
  const unsigned u = __float_as_uint(f);
  const unsigned e = (u >> 23) & 0xFFu, mant = u & 0x7FFFFFu, sgn = u & 0x80000000u;
  unsigned hw = sgn | ((e + 896u) << 20) | (mant >> 3), lw = mant << 29;
  if (e == 0u) {
    // zero or subnormal mant 2^-149 = 2^(p - 149) (1 + f), p = position of the leading bit
    const int p = 31 - __clz(mant);
    const unsigned long long fr = (unsigned long long)mant << (52 - p);
    hw = mant ? sgn | ((unsigned)(p + 874) << 20) | ((unsigned)(fr >> 32) & 0xFFFFFu) : sgn;
    lw = mant ? (unsigned)fr : 0u;
  } else if (e == 255u) {
    hw = sgn | 0x7FF00000u | (mant >> 3) | (mant ? 0x80000u : 0u);
    lw = 0u;
  }
  return __hiloint2double((int)hw, (int)lw);
}
__device__ __forceinline__ double ff_value(ff2 a) { return f32_to_f64(a.hi) + f32_to_f64(a.lo); }
__device__ __forceinline__ ff2 ff_neg(ff2 a) { return {-a.hi, -a.lo}; }
// s + e renormalised, |s| >= |e| (or s == 0)
__device__ __forceinline__ ff2 fast_two_sum(float s, float e) {
  const float h = __fadd_rn(s, e);
  return {h, __fsub_rn(e, __fsub_rn(h, s))};
}
// a + b = s + e exactly (Knuth)
__device__ __forceinline__ ff2 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ ff2 ff_add(ff2 a, ff2 b) {
  const ff2 s = two_sum(a.hi, b.hi);
  return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ ff2 ff_sub(ff2 a, ff2 b) { return ff_add(a, ff_neg(b)); }
// hi * hi exactly, plus the cross terms (the lo * lo term is below the precision kept)
__device__ __forceinline__ ff2 ff_prod(ff2 a, ff2 b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  return {p, e};  // not renormalised
}
__device__ __forceinline__ ff2 ff_mul(ff2 a, ff2 b) {
  const ff2 p = ff_prod(a, b);
  return fast_two_sum(p.hi, p.lo);
}
// a * b + c
__device__ __forceinline__ ff2 ff_fma(ff2 a, ff2 b, ff2 c) {
  const ff2 p = ff_prod(a, b);
  const ff2 s = two_sum(p.hi, c.hi);
  return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(p.lo, c.lo)));
}
// Running float-float sum s + c in the manner of Ogita, Rump and Oishi's Sum2/Dot2:
// each term's hi part enters s through TwoSum, its rounding error, its lo part and the
// cross terms of a product gather in c; renormalised once at the end. Each term waits
// on one FP32 add of the previous one (s and c are separate chains), where a chain of
// renormalised float-float sums waits on about eight.
struct ff_sum {
  float s = 0.0f, c = 0.0f;
  __device__ __forceinline__ ff_sum() = default;
  __device__ __forceinline__ explicit ff_sum(ff2 v) : s(v.hi), c(v.lo) {}
  __device__ __forceinline__ void add(ff2 v) {
    const ff2 t = two_sum(s, v.hi);
    s = t.hi;
    c = __fadd_rn(c, __fadd_rn(t.lo, v.lo));
  }
  __device__ __forceinline__ void add_prod(ff2 a, ff2 b) {
    const ff2 p = ff_prod(a, b);
    const ff2 t = two_sum(s, p.hi);
    s = t.hi;
    c = __fadd_rn(c, __fadd_rn(t.lo, p.lo));
  }
  __device__ __forceinline__ ff2 value() const { return fast_two_sum(s, c); }
};

// conversions between the matrix element types (double, float, float-float)
__device__ __forceinline__ float to_float(float a) { return a; }
__device__ __forceinline__ float to_float(double a) { return (float)a; }
__device__ __forceinline__ float to_float(ff2 a) { return a.hi; }
__device__ __forceinline__ double to_double(float a) { return (double)a; }
__device__ __forceinline__ double to_double(double a) { return a; }
__device__ __forceinline__ double to_double(ff2 a) { return ff_value(a); }
// A pair's hi part is what the FP32 inverse is formed from: a rounded to nearest, where
// ff_split truncates.
template <class R>
__device__ __forceinline__ R from_double(double a) {
  if constexpr (std::is_same<R, ff2>::value) {
    const ff2 s = ff_split(a);
    return fast_two_sum(s.hi, s.lo);
  } else {
    return (R)a;
  }
}

// ---------------------------------------------------------------------------
// Exponential by Tang's table-driven method (P. T. P. Tang, "Table-driven
// implementation of the exponential function in IEEE floating-point arithmetic",
// ACM TOMS 15(2), 1989), with a 256-entry table: x = (256 m + j) ln2/256 + r with
// |r| <= ln2/512, so exp(x) = 2^m 2^(j/256) exp(r). 2^(j/256) comes from a table of
// (lead, trail) pairs (lead = 2^(j/256) rounded to double, trail = the remainder
// rounded to double), exp(r) - 1 from its Taylor polynomial of degree 4 (truncation
// r^5/120 < 3.8e-17 relative), ln2/256 as a two-term split for the reduction, and
// 2^m is added to the exponent field. |x| >= 672, infinities and NaN take the
// library exp. Ten FP64 instructions; the table (4 KB) is read through the L1 cache.
// ---------------------------------------------------------------------------
static __device__ const double2 g_exp2_tab[256] = {
    {1.0, 0.0},
    {1.0027112750502025, -3.636615928692264e-17},
    {1.0054299011128027, 9.499186535455032e-17},
    {1.0081558981184175, -3.252058756084308e-17},
    {1.0108892860517005, -1.5234778603368577e-17},
    {1.0136300849514894, 9.283599768183568e-18},
    {1.016378314910953, -5.77217007319966e-17},
    {1.019133996077738, 3.601904982259662e-17},
    {1.0218971486541166, 5.109225028973444e-17},
    {1.0246677928971357, -7.56160786848778e-17},
    {1.0274459491187637, -4.9560741746453704e-17},
    {1.030231637686041, 3.319830041080813e-17},
    {1.0330248790212284, 7.600838874027088e-18},
    {1.0358256936019572, -7.806782391337636e-17},
    {1.0386341019613787, 5.996273788852511e-17},
    {1.041450124688316, 3.784830480287576e-17},
    {1.0442737824274138, 8.551889705537965e-17},
    {1.0471050958792898, 7.277077243104315e-17},
    {1.0499440858006872, 5.592937848127003e-17},
    {1.0527907730046264, -9.629482899026936e-17},
    {1.0556451783605572, 1.759325738772092e-18},
    {1.0585073227945128, -7.152651856637781e-17},
    {1.061377227289262, -1.1973537085365658e-17},
    {1.0642549128844645, 5.0787541986112304e-17},
    {1.0671404006768237, -7.899853966841582e-17},
    {1.0700337118202419, -9.937162711288919e-17},
    {1.0729348675259756, -3.839668843358824e-18},
    {1.075843889062791, -1.0002716151144136e-17},
    {1.0787607977571199, -6.656660436056593e-17},
    {1.0816856149932152, -4.782623902997086e-17},
    {1.0846183622133092, 3.166152845816346e-17},
    {1.0875590609177697, 5.409349307820291e-18},
    {1.0905077326652577, -3.046782079812471e-17},
    {1.0934643990728858, 1.441395814726921e-17},
    {1.0964290818163769, -5.919933484449316e-17},
    {1.099401802630222, 7.170459599701923e-17},
    {1.102382583307841, 5.2660368715706944e-17},
    {1.1053714457017412, 8.239288760500214e-17},
    {1.1083684117236787, -8.786813845180527e-17},
    {1.1113735033448175, 5.563945026669698e-17},
    {1.1143867425958924, 1.0410278456845571e-16},
    {1.1174081515673693, -7.97680590262822e-17},
    {1.1204377524096067, -6.201085906554179e-17},
    {1.12347556733302, -9.699737588987043e-17},
    {1.1265216186082418, 5.165856758795457e-17},
    {1.129575928566288, 6.712805858726257e-17},
    {1.1326385195987192, 3.237356166738e-17},
    {1.1357094141578055, 5.066599926126156e-17},
    {1.1387886347566916, 8.912812676025408e-17},
    {1.1418762039695616, 4.6510911775314124e-17},
    {1.1449721444318042, 4.6412898921700107e-17},
    {1.148076478840179, 6.897740236627192e-17},
    {1.1511892299529827, 3.250710218863827e-17},
    {1.154310420590216, 1.0417128946273266e-16},
    {1.1574400736337511, -9.1238712311344e-17},
    {1.1605782120274988, -3.261040205417394e-17},
    {1.1637248587775775, 3.8292048369240935e-17},
    {1.1668800369524817, -8.79187957999917e-17},
    {1.1700437696832502, -1.8477442017900047e-18},
    {1.1732160801636373, -7.287562586584994e-17},
    {1.1763969916502812, 5.554203254218079e-17},
    {1.1795865274628758, 1.009231277510039e-16},
    {1.182784710984341, 1.542975430079076e-17},
    {1.1859915656609938, -9.209506835293106e-18},
    {1.189207115002721, 3.982015231465646e-17},
    {1.1924313825831512, 4.3975514156097214e-17},
    {1.1956643920398273, 4.6166036704814814e-17},
    {1.1989061670743806, -9.809193356008423e-17},
    {1.202156731452703, 6.644981499252301e-17},
    {1.2054161090051239, -3.3572721932675296e-17},
    {1.2086843236265816, -4.746725945228984e-17},
    {1.2119613992768012, -4.8906110775211184e-17},
    {1.215247359980469, -7.712630692681488e-17},
    {1.2185422298274085, -9.006726958363838e-17},
    {1.2218460329727576, -1.0611021211402691e-16},
    {1.2251587936371455, -8.903533814269983e-17},
    {1.22848053610687, -1.89878163130253e-17},
    {1.2318112847340759, 7.38938247161005e-17},
    {1.2351510639369334, -1.0755244344307841e-16},
    {1.2384998981998165, 2.7677020555739674e-17},
    {1.241857812073484, 4.658027591836937e-17},
    {1.245224830175258, -4.6772404498467275e-17},
    {1.2486009771892048, -8.261810999021964e-17},
    {1.2519862778663162, 4.8341671524698976e-17},
    {1.255380757024691, -6.7113898212968784e-18},
    {1.2587844395497165, -8.421782587730599e-17},
    {1.2621973503942507, -3.0844648874738465e-17},
    {1.2656195145788063, 4.2505770034508686e-17},
    {1.2690509571917332, 2.667932131342186e-18},
    {1.2724917033894028, -1.0577916267212421e-17},
    {1.275941778396392, 9.91543024421429e-17},
    {1.2794012075056693, -9.759095008356062e-17},
    {1.2828700160787783, 1.713594918243561e-17},
    {1.2863482295460256, -3.416955706936182e-17},
    {1.2898358734066657, 8.949257530897592e-17},
    {1.2933329732290895, -2.9745904431327516e-17},
    {1.2968395546510096, 2.5382502794888315e-17},
    {1.3003556433796506, 5.678728102802217e-17},
    {1.3038812651919358, 8.647675598267871e-17},
    {1.3074164459346773, -7.336645652878869e-17},
    {1.3109612115247644, -7.181536135519454e-17},
    {1.3145155879493546, 2.2675433151045856e-17},
    {1.318079601266064, -5.4579558271491535e-17},
    {1.3216532776031575, -2.4806382459130217e-17},
    {1.3252366431597413, -2.8587312100388614e-17},
    {1.3288297242059544, 4.08908622391016e-17},
    {1.3324325470831615, -5.101586630916744e-17},
    {1.3360451382041458, -5.891866356388801e-17},
    {1.339667524053303, 8.927282594831732e-17},
    {1.3432997311868353, -5.802580890201438e-17},
    {1.3469417862329458, 3.224065101254679e-17},
    {1.3505937158920345, -8.287110381462417e-17},
    {1.3542555469368927, 7.70094837980299e-17},
    {1.3579273062129011, -9.529635744825189e-17},
    {1.3616090206382248, 1.533787661270668e-18},
    {1.365300717204012, -1.0005363125974765e-16},
    {1.3690024229745905, 9.593797919118849e-17},
    {1.3727141650876684, -4.495960595234841e-17},
    {1.3764359707545302, -6.898588935871801e-17},
    {1.380167867260238, 1.0510314579969984e-16},
    {1.383909881963832, -6.770511658794786e-17},
    {1.387662042298529, 8.422984274875415e-17},
    {1.3914243757719262, -4.9061748652889893e-17},
    {1.3951969099662003, -9.329336224225497e-17},
    {1.3989796725383112, -9.614213209051323e-17},
    {1.4027726912202048, -5.295783249407989e-17},
    {1.4065759938190154, 7.034914812136422e-18},
    {1.4103896082172707, 4.166548728435062e-17},
    {1.4142135623730951, -9.667293313452913e-17},
    {1.4180478843204152, 2.2744385421855295e-17},
    {1.4218926021691656, -1.6077828915890244e-17},
    {1.4257477441054942, 9.880690758500607e-17},
    {1.42961333839197, -1.2031642489053655e-17},
    {1.433489413367789, -5.802454243926826e-17},
    {1.4373759974489824, -4.2040340164675566e-17},
    {1.4412731191286257, 5.602503650878986e-18},
    {1.4451808069770467, -3.0237581349939873e-17},
    {1.449099089642035, -6.259405000819309e-17},
    {1.4530279958490526, -5.779948609396106e-17},
    {1.4569675544014438, 5.648679453876998e-17},
    {1.460917794180647, -5.600377186075216e-17},
    {1.4648787441464057, 9.530767543587157e-17},
    {1.4688504333369818, 8.465882756533628e-17},
    {1.4728328908693675, 6.691774081940589e-17},
    {1.4768261459394993, -3.483994556892796e-17},
    {1.4808302278224719, -9.686952102630619e-17},
    {1.4848451658727524, 1.0780086764407481e-16},
    {1.488870989524397, 6.155367157742871e-17},
    {1.4929077282912648, 1.4192920154284036e-17},
    {1.4969554117672355, -2.861663253899158e-17},
    {1.5010140696264256, -6.413767275790235e-17},
    {1.5050837316234065, 7.074710613582846e-17},
    {1.5091644275934228, -1.016455327754295e-16},
    {1.5132561874526098, 8.884497851338712e-17},
    {1.5173590411982147, -4.308699472043341e-17},
    {1.5214730189088146, -5.9963876759456834e-18},
    {1.5255981507445384, -1.1024941712342561e-16},
    {1.529734466947287, 3.7857921151572197e-17},
    {1.533881997840956, 8.875226844438446e-17},
    {1.5380407738316568, 1.0174672351161359e-16},
    {1.5422108254079407, 7.949834809697621e-17},
    {1.5463921831410214, 1.068396000565722e-16},
    {1.550584877685, -1.4600706590689385e-17},
    {1.5547889397770887, -8.003161350116036e-17},
    {1.559004400237837, 3.7812070533575275e-17},
    {1.5632312899713576, 7.484777645590734e-17},
    {1.567469639965553, -1.0352061768849722e-16},
    {1.5717194812923414, -3.3429840046872e-17},
    {1.5759808451078865, -1.0136916471278304e-17},
    {1.5802537626528246, -5.163402929554468e-17},
    {1.5845382652524937, -1.9337717034585703e-17},
    {1.588834384317164, -5.9949501188244794e-18},
    {1.593142151342267, -1.0094406542311964e-16},
    {1.597461597908627, 2.4868392796221e-17},
    {1.6017927556826934, -6.054917453527784e-17},
    {1.606135656416771, -1.0354545288059995e-16},
    {1.6104903319492543, 2.4707192569797888e-17},
    {1.6148568142048607, -7.316663399125123e-17},
    {1.6192351351948637, 2.0941334154229092e-17},
    {1.6236253270173289, -3.584512851414475e-17},
    {1.6280274218573478, -6.712955084707084e-17},
    {1.632441451987275, 9.852819230429993e-17},
    {1.6368674497669644, 7.698325071319876e-17},
    {1.6413054476440063, -9.247568737640706e-17},
    {1.645755478153965, -1.0125679913674773e-16},
    {1.6502175739206177, 9.133279588729904e-18},
    {1.6546917676561943, 9.643294303196029e-17},
    {1.6591780921616162, -7.275545550823051e-17},
    {1.6636765803267364, 5.8909926967131e-17},
    {1.6681872651305825, 4.269178019570615e-17},
    {1.6727101796415966, -5.476715964599563e-17},
    {1.6772453570178785, 8.303949509950733e-17},
    {1.681792830507429, 8.199010020581497e-17},
    {1.6863526334483934, -7.181463278358011e-17},
    {1.6909247992693053, -9.66967147439488e-17},
    {1.6955093614893326, 7.238416872845167e-17},
    {1.7001063537185235, -8.0237193703977e-18},
    {1.7047158096580513, -2.7288832847972816e-17},
    {1.709337763100463, -9.868779456632931e-17},
    {1.713972247929926, 6.473975107753367e-17},
    {1.718619298122478, -1.851380418263111e-17},
    {1.723278947746274, -9.5221238003938e-17},
    {1.7279512309618377, -1.0750981861204642e-16},
    {1.732636182022311, -1.6980510743154155e-18},
    {1.7373338352737062, 3.164389299292957e-17},
    {1.7420442251551564, -1.5259591189507888e-18},
    {1.746767386199169, -1.0752290483507515e-16},
    {1.7515033530318782, -5.1244504205967247e-17},
    {1.7562521603732995, 2.960140695448873e-17},
    {1.761013843037584, -7.943253125039228e-17},
    {1.7657884359332727, 9.461315018083268e-17},
    {1.7705759740635547, 5.961794510040556e-17},
    {1.7753764925265212, 6.429731796556572e-17},
    {1.7801900265154245, -5.2846272890916174e-17},
    {1.785016611318935, 1.5330400121031314e-17},
    {1.789856282321401, -4.1543546606833504e-17},
    {1.7947090750031072, 1.8227458427912087e-17},
    {1.7995750249405351, -2.526889233358898e-17},
    {1.804454167806624, -5.177222408793318e-17},
    {1.809346539371032, -9.03264140245003e-17},
    {1.8142521755003989, -9.969531538920349e-17},
    {1.8191711121586085, 7.402676901145839e-17},
    {1.8241033854070534, -1.0159627862277083e-16},
    {1.8290490314048973, 6.889192908835696e-17},
    {1.8340080864093424, 3.283107224245627e-17},
    {1.8389805867758937, 6.918969740272512e-18},
    {1.843966568958626, -5.939742026949965e-17},
    {1.8489660695104508, 9.027580446261089e-17},
    {1.8539791250833855, 9.761887490727594e-17},
    {1.8590057724288205, -9.528705461989941e-17},
    {1.864046048397789, 6.540912680620572e-17},
    {1.8690999899412386, -9.938505214255067e-17},
    {1.8741676341103, -6.122763413004143e-17},
    {1.8792490180565602, -1.6226315557835845e-17},
    {1.8843441790323345, -8.226593125533711e-17},
    {1.8894531543909392, -9.005168285059127e-17},
    {1.8945759815869656, 3.4034035352165297e-17},
    {1.8997126981765553, -3.8597397693785143e-17},
    {1.9048633418176741, 6.533857514718279e-17},
    {1.9100279502703899, -5.90968800674406e-17},
    {1.9152065613971474, -1.0619946056195963e-16},
    {1.9203992131630474, 7.116681540630314e-17},
    {1.925605943636125, -9.914963769693741e-17},
    {1.930826790987627, 6.16714970616911e-17},
    {1.9360617934922943, 1.0332385960676326e-16},
    {1.9413109895286405, -6.638029891621488e-17},
    {1.9465744175792332, 6.811022349533877e-17},
    {1.9518521162309783, -2.199016969979351e-17},
    {1.9571441241754002, 8.960767791036668e-17},
    {1.9624504802089273, 1.0976844000913547e-16},
    {1.9677712232331759, -1.0314928011531132e-16},
    {1.9731063922552343, -7.451617863956037e-18},
    {1.978456026387951, 4.0388753109278167e-17},
    {1.9838201648502194, -2.2034544123910627e-17},
    {1.9891988469672663, 8.2051326383692e-18},
    {1.9945921121709402, 1.7909710352002645e-17},
};

static __device__ __noinline__ double exp_outside(double x) { return exp(x); }

constexpr double kInvLn10 = 0.43429448190325176;  // 1 / ln 10
constexpr double kLnRcP0 = 4.407418589020958;  // ln(Rc / P0), cgs
constexpr long long kLnRcP0_Q52 = 19849248715180584ll;

__device__ __forceinline__ double xexp(double x) {
  if ((__double2hiint(x) & 0x7fffffff) >= 0x40850000) return exp_outside(x);  // |x| >= 672, inf, NaN
  constexpr double kInvL = 369.3299304675746;      // 256 / ln 2
  constexpr double kL1 = 0.0027076061740622863;    // ln2/256 rounded to double
  constexpr double kL2 = 9.058776616587108e-20;    // ln2/256 - kL1
  constexpr double kShift = 6755399441055744.0;    // 1.5 * 2^52: rounds to an integer in the low word
  const double t = fma(x, kInvL, kShift);
  const int N = __double2loint(t);
  const double2 sj = __ldg(&g_exp2_tab[N & 255]);
  const double Nd = t - kShift;
  double r = fma(-Nd, kL1, x);
  r = fma(-Nd, kL2, r);
  double q = fma(r, 1.0 / 24.0, 1.0 / 6.0);
  q = fma(r, q, 0.5);
  const double em1 = fma(r * r, q, r);  // exp(r) - 1
  const double y = sj.x + fma(sj.x, em1, sj.y);
  return __hiloint2double(__double2hiint(y) + (N >> 8) * (1 << 20), __double2loint(y));
}

// ---------------------------------------------------------------------------
// Natural logarithm, table-driven in the manner of Tang (P. T. P. Tang, "Table-
// driven implementation of the logarithm function in IEEE floating-point
// arithmetic", ACM TOMS 16(4), 1990): x = 2^m y with y in [1, 2), F = 1 + j/128 the
// nearest of 129 points, c = 1/F rounded to double, r = y c - 1 (one FMA rounding,
// |r| <= 1/256 + 2^-30), and ln x = m ln 2 - ln c + ln(1 + r), with ln(1 + r) from
// its Taylor series to degree 7 (truncation below 2e-18 relative). The table holds
// (c, -ln c as lead + trail) for the rounded c; ln 2 is split so m ln2_hi is exact.
// Zero, negative, subnormal, infinite and NaN arguments take the library log.
// ---------------------------------------------------------------------------
static __device__ const double g_log_tab[129][3] = {
    {1.0, 0.0, 0.0},
    {0.9922480620155039, 0.007782140442054963, -1.2819179123343749e-20},
    {0.9846153846153847, 0.015504186535965199, -3.2783210228924137e-19},
    {0.9770992366412213, 0.023167059281534418, -3.095927552179262e-19},
    {0.9696969696969697, 0.03077165866675366, 1.0431732029005972e-18},
    {0.9624060150375939, 0.03831886430213666, -2.3579961573512846e-18},
    {0.9552238805970149, 0.04580953603129422, 1.6823639049745016e-19},
    {0.9481481481481482, 0.05324451451881224, 1.803871134979952e-18},
    {0.9411764705882353, 0.060624621816434854, 2.6424025938726934e-18},
    {0.9343065693430657, 0.06795066190850778, 3.9239563038692484e-18},
    {0.927536231884058, 0.07522342123758752, -4.195880720316434e-18},
    {0.920863309352518, 0.08244366921107454, -4.707903082046854e-18},
    {0.9142857142857143, 0.08961215868968717, -1.9573659817110993e-18},
    {0.9078014184397163, 0.09672962645855114, -4.0291867005826106e-18},
    {0.9014084507042254, 0.10379679368164355, -3.195893222617445e-18},
    {0.8951048951048951, 0.11081436634029011, 2.0511100808140527e-18},
    {0.8888888888888888, 0.11778303565638351, -1.1971685747593662e-18},
    {0.8827586206896552, 0.12470347850095725, -4.6522609636496624e-18},
    {0.8767123287671232, 0.13157635778871932, 1.112300087972959e-17},
    {0.8707482993197279, 0.1384023228591192, -1.3766819196398948e-17},
    {0.8648648648648649, 0.14518200984449783, 8.242418783022477e-18},
    {0.8590604026845637, 0.151916042025842, 4.1233095848339465e-19},
    {0.8533333333333334, 0.15860503017663852, 2.583386492298558e-18},
    {0.847682119205298, 0.16524957289530717, -9.227573884334224e-18},
    {0.8421052631578947, 0.17185025692665928, -6.022453821011369e-18},
    {0.8366013071895425, 0.17840765747281825, 1.2720936612962572e-17},
    {0.8311688311688312, 0.18492233849401193, -7.384679440503435e-18},
    {0.8258064516129032, 0.19139485299962947, -1.126213516780448e-17},
    {0.8205128205128205, 0.19782574332991992, -7.995487338741543e-18},
    {0.8152866242038217, 0.20421554142869083, 7.9379985298027e-18},
    {0.810126582278481, 0.21056476910734964, 1.136310596906137e-17},
    {0.8050314465408805, 0.2168739383006143, 6.285749669211092e-18},
    {0.8, 0.2231435513142097, -9.091270597324798e-18},
    {0.7950310559006211, 0.2293741010648459, -5.684839459813236e-18},
    {0.7901234567901234, 0.23556607131276697, -2.394337149518734e-18},
    {0.7852760736196319, 0.24171993688714513, 1.323779871210866e-17},
    {0.7804878048780488, 0.2478361639045812, 8.384472133019162e-18},
    {0.7757575757575758, 0.25391520998096345, -7.180735656435798e-18},
    {0.7710843373493976, 0.259957524436926, 2.4167516341742964e-17},
    {0.7664670658682635, 0.2659635484971379, 1.35209848201012e-19},
    {0.7619047619047619, 0.2719337154836418, 7.833196376974436e-19},
    {0.757396449704142, 0.2778684510034563, 2.2502748630777633e-17},
    {0.7529411764705882, 0.2837681731306446, -6.448868003452105e-18},
    {0.7485380116959064, 0.2896332925830427, 2.0535953219858177e-17},
    {0.7441860465116279, 0.2954642128938359, -7.768320796245443e-18},
    {0.7398843930635838, 0.30126133057816185, -1.5120043309967385e-17},
    {0.735632183908046, 0.3070250352949119, 1.5578716077124932e-18},
    {0.7314285714285714, 0.3127557100038969, -1.3650721793001109e-17},
    {0.7272727272727273, 0.3184537311185346, -6.407962483026777e-19},
    {0.7231638418079096, 0.324119468654212, -4.488767429940198e-18},
    {0.7191011235955056, 0.32975328637246804, -2.5633554999431966e-17},
    {0.7150837988826816, 0.3353555419211378, -1.3746739934976202e-17},
    {0.7111111111111111, 0.3409265869705932, -2.069678002794501e-17},
    {0.7071823204419889, 0.3464667673462086, -3.591951952851805e-18},
    {0.7032967032967034, 0.3519764231571781, 2.0005853013367377e-17},
    {0.6994535519125683, 0.3574558889218038, -2.4269548334425144e-17},
    {0.6956521739130435, 0.3629054936893685, 6.2632141603179415e-18},
    {0.6918918918918919, 0.36832556115870757, 2.690672380132659e-17},
    {0.6881720430107527, 0.373716409793584, -2.449917382477111e-18},
    {0.6844919786096256, 0.3790783529349695, 1.8481479367349684e-17},
    {0.6808510638297872, 0.38441169891033206, 8.164631656028572e-18},
    {0.6772486772486772, 0.38971675114002524, 2.734172667856699e-17},
    {0.6736842105263158, 0.394993808240869, 7.437680769362324e-18},
    {0.6701570680628273, 0.40024316412701266, -1.655340963311913e-17},
    {0.6666666666666666, 0.40546510810816444, -2.881138025962641e-18},
    {0.6632124352331606, 0.4106599249852683, 2.7752739097728695e-17},
    {0.6597938144329897, 0.415827895143711, -5.793440801214822e-18},
    {0.6564102564102564, 0.42096929464412963, 4.5972855136437464e-18},
    {0.6530612244897959, 0.42608439531090014, -7.056391017993593e-19},
    {0.649746192893401, 0.43117346481837143, -1.3539234990021841e-17},
    {0.6464646464646465, 0.43623676677491796, 2.4182887316590065e-17},
    {0.6432160804020101, 0.4412745608048752, 1.0343758877897315e-17},
    {0.64, 0.4462871026284195, 1.6511928324886544e-17},
    {0.6368159203980099, 0.4512746441394586, -9.65179553937242e-18},
    {0.6336633663366337, 0.4562374334815876, 9.07916350878553e-18},
    {0.6305418719211823, 0.46117571512217015, 6.140445034134513e-18},
    {0.6274509803921569, 0.46608972992459924, -2.387354320899491e-19},
    {0.624390243902439, 0.470979715218791, 7.099457177589995e-18},
    {0.6213592233009708, 0.475845904869964, 2.5043069845040313e-17},
    {0.6183574879227053, 0.48068852934575196, -2.7402100563370574e-18},
    {0.6153846153846154, 0.48550781578170077, -1.6618350693852045e-17},
    {0.6124401913875598, 0.4903039880451939, 4.612452524535198e-18},
    {0.6095238095238096, 0.4950772667978514, 1.2508730752094332e-17},
    {0.6066350710900474, 0.49982786955644926, -2.25665388836583e-18},
    {0.6037735849056604, 0.5045560107523953, 1.3275397597891851e-17},
    {0.6009389671361502, 0.5092619017898079, 2.1678544367048826e-17},
    {0.5981308411214953, 0.5139457511022344, -2.4537074021915265e-18},
    {0.5953488372093023, 0.5186077642080457, -1.6859591393570242e-17},
    {0.5925925925925926, 0.5232481437645479, 2.3677269014906905e-17},
    {0.5898617511520737, 0.5278670896208424, -3.071514383985515e-18},
    {0.5871559633027523, 0.5324647988694717, 5.4596227307139745e-17},
    {0.5844748858447488, 0.5370414658968837, -1.9513712761861967e-17},
    {0.5818181818181818, 0.5415972824327444, 1.108461486609421e-17},
    {0.579185520361991, 0.5461324375981356, -6.169692458083718e-18},
    {0.5765765765765766, 0.5506471179526623, -1.3720677478685045e-17},
    {0.5739910313901345, 0.5551415075405016, -1.449278054403172e-17},
    {0.5714285714285714, 0.5596157879354228, -2.8656225429134744e-17},
    {0.5688888888888889, 0.564070138284803, -4.6267923647049475e-17},
    {0.5663716814159292, 0.5685047353526688, -4.0389558221668317e-17},
    {0.5638766519823789, 0.5729197535617854, 4.4242614369063874e-17},
    {0.5614035087719298, 0.5773153650348236, 4.660755938428382e-17},
    {0.5589519650655022, 0.5816917396346225, 2.7912851075301e-17},
    {0.5565217391304348, 0.5860490450035782, -4.272669638447342e-17},
    {0.5541125541125541, 0.5903874466021763, 2.876546074301208e-17},
    {0.5517241379310345, 0.5947071077466928, 2.7629477772138132e-17},
    {0.5493562231759657, 0.5990081896460834, 2.5162534548420983e-17},
    {0.5470085470085471, 0.6032908514380841, 2.0348397202878346e-17},
    {0.5446808510638298, 0.6075552502245418, -4.1692640626751196e-17},
    {0.5423728813559322, 0.6118015411059929, -3.392831249677239e-17},
    {0.540084388185654, 0.616029877215514, 4.9247969628553695e-17},
    {0.5378151260504201, 0.6202404097518576, 3.4764762563436685e-18},
    {0.5355648535564853, 0.6244332880118936, 1.4444646832738594e-17},
    {0.5333333333333333, 0.6286086594223742, -5.360577204673081e-17},
    {0.5311203319502075, 0.6327666695710378, 5.223564575344447e-17},
    {0.5289256198347108, 0.6369074622370692, 2.6473983119023558e-17},
    {0.5267489711934157, 0.6410311794209312, -3.4765774267087093e-17},
    {0.5245901639344263, 0.6451379613735847, -5.110700818729212e-17},
    {0.5224489795918368, 0.6492279466251097, -1.3266356651077771e-17},
    {0.5203252032520326, 0.6533012720127456, -3.7864752792363655e-17},
    {0.5182186234817814, 0.65735807270836, 2.2462005860533567e-17},
    {0.5161290322580645, 0.661398482245365, 2.015224182999491e-17},
    {0.5140562248995983, 0.6654226325450905, 5.424612435933966e-17},
    {0.512, 0.6694306539426292, 7.420657727561746e-18},
    {0.5099601593625498, 0.6734226752121667, 3.84128539325942e-17},
    {0.5079365079365079, 0.6773988235918061, 5.341333284299263e-17},
    {0.5059288537549407, 0.6813592248079031, 1.7765482243852914e-17},
    {0.5039370078740157, 0.6853040030989195, -4.8209665191998585e-17},
    {0.5019607843137255, 0.689233281238809, -9.330006029414747e-18},
    {0.5, 0.6931471805599453, 2.3190468138462996e-17}
};

static __device__ __noinline__ double log_outside(double x) { return log(x); }

__device__ __forceinline__ double xlog(double x) {
  const int hx = __double2hiint(x);
  if (hx < 0x00100000 || hx >= 0x7ff00000) return log_outside(x);
  constexpr double kLn2Hi = 0.6931467056274414;      // ln 2 with the low 32 mantissa bits cleared
  constexpr double kLn2Lo = 4.7493250390316726e-07;  // ln 2 - kLn2Hi
  const int mb = hx & 0x000fffff;
  const int j = (mb + 0x1000) >> 13;
  const double y = __hiloint2double(mb | 0x3ff00000, __double2loint(x));
  const double* e = g_log_tab[j];
  const double r = fma(y, __ldg(e), -1.0);
  double q = fma(r, 1.0 / 7.0, -1.0 / 6.0);
  q = fma(r, q, 1.0 / 5.0);
  q = fma(r, q, -0.25);
  q = fma(r, q, 1.0 / 3.0);
  q = fma(r, q, -0.5);
  const double l1p = fma(r * r, q, r);  // ln(1 + r)
  const double md = (double)((hx >> 20) - 1023);
  const double t = fma(md, kLn2Hi, __ldg(e + 1));
  return t + fma(md, kLn2Lo, __ldg(e + 2) + l1p);
}

// 1/x from the hardware's approximate reciprocal r (relative error below 2^-20) by one
// cubic step r <- r + r (e + e^2), e = 1 - x r, whose truncation e^3 is below 2^-60: three
// dependent FP64 instructions, where two Newton steps take four; magnitudes outside
// [2^-1000, 2^1000], zero, infinities and NaN take the IEEE division.
static __device__ __noinline__ double rcp_outside(double x) { return 1.0 / x; }

__device__ __forceinline__ double xrcp(double x) {
  const int ex = (__double2hiint(x) >> 20) & 0x7ff;
  if (ex < 23 || ex > 2023) return rcp_outside(x);
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}


// RODAS4 coefficients in constant memory (stages are indexed at run time).
static __constant__ double c_rodasA[6][6] = CHEM_RODAS_A;
static __constant__ double c_rodasC[6][6] = CHEM_RODAS_C;
static __constant__ double c_rodasM[6] = CHEM_RODAS_M;

// Method traits: stage count, step-size exponent 1/Q and the transformed coefficients.
// RODAS4 reads its published table from constant memory; the W-method reads the table
// the host converted from its published original form (kernel arguments).
template <int MTH>
struct Meth;
template <>
struct Meth<METHOD_RODAS4> {
  static constexpr int S = 6, Q = 4;
  static constexpr bool E_LAST = true;  // error estimate = last stage
  __device__ static double gamma(const IntegrateArgs&) { return kRodasGamma; }
  __device__ static double a(const IntegrateArgs&, int i, int j) { return c_rodasA[i][j]; }
  __device__ static double c(const IntegrateArgs&, int i, int j) { return c_rodasC[i][j]; }
  __device__ static double m(const IntegrateArgs&, int j) { return c_rodasM[j]; }
  __device__ static double e(const IntegrateArgs&, int) { return 0.0; }
};
template <>
struct Meth<METHOD_ROS34PW2> {
  static constexpr int S = 4, Q = 3;
  static constexpr bool E_LAST = false;
  __device__ static double gamma(const IntegrateArgs& g) { return g.tab.gamma; }
  __device__ static double a(const IntegrateArgs& g, int i, int j) { return g.tab.a[i][j]; }
  __device__ static double c(const IntegrateArgs& g, int i, int j) { return g.tab.c[i][j]; }
  __device__ static double m(const IntegrateArgs& g, int j) { return g.tab.m[j]; }
  __device__ static double e(const IntegrateArgs& g, int j) { return g.tab.e[j]; }
};

// Loads of tables that stream through once per step: they do not displace the rate
// evaluation's tables, which every right-hand side reads, from the L1 cache.
__device__ __forceinline__ uint2 ld_stream(const uint2* p) {
  uint2 v;
  asm("ld.global.nc.L1::no_allocate.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ ff2 ld_stream(const ff2* p) {
  ff2 v;
  asm("ld.global.nc.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(v.hi), "=f"(v.lo) : "l"(p));
  return v;
}

// Precision policy: LU = type of the factorised matrix, ASM = type the Jacobian is
// assembled in; IR = refine each solve against the assembled matrix.
template <int PREC>
struct Policy {
  using LU = double;
  using ASM = double;
  static constexpr bool IR = false;
};
template <>
struct Policy<PREC_MIXED> {
  using LU = float;
  using ASM = ff2;  // float-float: about 48 significant bits, on the FP32 pipe
  static constexpr bool IR = true;
};
template <>
struct Policy<PREC_FP32ASM> {
  using LU = float;
  using ASM = float;
  static constexpr bool IR = true;
};

// ---------------------------------------------------------------------------
// shared-memory carve-up
// ---------------------------------------------------------------------------
struct Layout {
  int nmax, ld;            // matrix dimension bound and leading dimension (odd)
  int Kmax, Imax;
  size_t off_vec, off_M, off_M0, off_piv, total;
  bool x_tab;
};

__host__ __device__ inline int odd_ld(int n) { return n | 1; }
// 8-byte entries of a CTA's global-memory slot: the matrix by columns and the mass-action sums
__host__ __device__ inline int slot_ld(int n) { return (n + 7) & ~3; }
__host__ __device__ inline size_t slot_entries(int K) {
  return ((size_t)(K + 1) * slot_ld(K + 1) + (size_t)K * K + 3) & ~(size_t)3;
}

// vectors (double): y, yn, ys, f0, fv, rr, u[6], sc  -> 13 n
// species (8 bytes): C, hRT, cpR, g, dcp, dk, akT, ek, 1/W -> 9 K
// reactions (double): q, D, dTc, P, dqs[4] -> 8 I
// m0_global: the mixed form's assembled matrix lives in a global-memory slot of
// the CTA instead of shared memory (large mechanisms, persistent schedulers).
// want_xt: the exponential's table (2 KB) in shared memory, where that still fits.
// n_sp: 9, or 0 for a kernel without a mechanism.
constexpr size_t kMaxSmem = 227 * 1024 - 16;  // k_integrate has 16 bytes of static shared memory
__host__ __device__ inline Layout make_layout(int Kmax, int Imax, int prec, bool m0_global = false,
                                              bool want_xt = false, int n_sp = 9) {
  Layout L;
  L.nmax = Kmax + 1;
  L.ld = odd_ld(L.nmax);
  L.Kmax = Kmax;
  L.Imax = Imax;
  size_t o = 0;
  o += 64 * sizeof(double);
  L.x_tab = want_xt;
  if (want_xt) o += 256 * sizeof(double);
  L.off_vec = o;
  o += (size_t)13 * L.nmax * sizeof(double);
  o += (size_t)n_sp * Kmax * sizeof(double);
  if (prec == PREC_FP64) {
    o += (size_t)8 * Imax * sizeof(double);
    L.off_M = o;
    o += (size_t)L.nmax * L.ld * sizeof(double);
  } else {
    // The FP32 factor matrix is written only after the assembly has consumed the
    // per-reaction Jacobian data (everything after q), so it shares their space.
    L.off_M = o + (size_t)Imax * sizeof(double);
    const size_t jac = (size_t)7 * Imax * sizeof(double);
    const size_t mat = (size_t)L.nmax * L.ld * sizeof(float);
    o += (size_t)Imax * sizeof(double) + (jac > mat ? jac : mat);
  }
  o = (o + 15) & ~(size_t)15;
  L.off_M0 = o;
  if (prec == PREC_MIXED && !m0_global) o += (size_t)L.nmax * L.ld * sizeof(double);
  if (prec == PREC_FP32ASM) o += (size_t)L.nmax * L.ld * sizeof(float);
  o = (o + 15) & ~(size_t)15;
  L.off_piv = o;
  o += (size_t)2 * L.nmax * sizeof(int);  // pivots, permutation
  o += (size_t)L.nmax * sizeof(double);   // inverse diagonal of U
  o = (o + 15) & ~(size_t)15;
  L.total = o;
  return want_xt && o > kMaxSmem ? make_layout(Kmax, Imax, prec, m0_global, false, n_sp) : L;
}


// Scalars kept in the reduction area (its first 32 slots are unused).
// SC_OUT: 8 broadcast results of Cta::reduce; SC_PIV: pivot search slots (12 NW bytes)
// (SC_INVT during the rate evaluation, SC_INVP during the LU: never live together)
enum { SC_OUT = 32, SC_LOGT = 48, SC_INVT = 49, SC_INVP = 49, SC_ICPM = 50, SC_DCPM = 51, SC_PIV = 52 };

// A CTA's view of its shared memory. Arrays are functions of a few 32-bit sizes, so that
// an address is one or two integer instructions and a shared-memory access: as stored
// pointers they would take 60 registers, or local memory.
extern __shared__ __align__(16) unsigned char smem[];

template <int NW>
struct Cta {
  static constexpr int NT = NW * 32;
  static constexpr int SW = NW - 1;  // the warp that computes CTA scalars (ln T, 1/T, the FP64 solve)
  int tid, lane, warp;
  unsigned vec, n8, k8, i8, off_M, off_piv;  // byte offsets; bytes of n, K and I 8-byte entries
  bool x_tab;
  void* M0;     // mixed forms: the assembled matrix by columns, entry (i, j) at j ld0 + i0 + i
  int ld0, i0;
  int Km;       // species of the mechanism the matrix geometry is set for
  double p_rc, rc_p;  // p/Rc and Rc/p of the cell

  __device__ __forceinline__ static double* at(unsigned off) { return reinterpret_cast<double*>(smem + off); }
  __device__ __forceinline__ double* red() const { return at(0); }
  // vectors of n
  __device__ __forceinline__ double* y() const { return at(vec); }
  __device__ __forceinline__ double* yn() const { return at(vec + n8); }
  __device__ __forceinline__ double* ys() const { return at(vec + 2 * n8); }
  __device__ __forceinline__ double* f0() const { return at(vec + 3 * n8); }
  __device__ __forceinline__ double* fv() const { return at(vec + 4 * n8); }
  __device__ __forceinline__ double* rr() const { return at(vec + 5 * n8); }
  __device__ __forceinline__ double* u() const { return at(vec + 6 * n8); }  // 6 n
  __device__ __forceinline__ double* sc() const { return at(vec + 12 * n8); }
  // species
  __device__ __forceinline__ unsigned sp(int a) const { return vec + 13 * n8 + a * k8; }
  __device__ __forceinline__ double* C() const { return at(sp(0)); }
  __device__ __forceinline__ double* hRT() const { return at(sp(1)); }
  __device__ __forceinline__ double* cpR() const { return at(sp(2)); }
  __device__ __forceinline__ double* g() const { return at(sp(3)); }
  __device__ __forceinline__ double* dcp() const { return at(sp(4)); }
  __device__ __forceinline__ double* dk() const { return at(sp(5)); }
  __device__ __forceinline__ double* akT() const { return at(sp(6)); }
  __device__ __forceinline__ double* ek() const { return at(sp(7)); }
  __device__ __forceinline__ double* iW() const { return at(sp(8)); }
  // reactions
  __device__ __forceinline__ double* q() const { return at(sp(9)); }
  __device__ __forceinline__ double* D() const { return at(sp(9) + i8); }
  __device__ __forceinline__ double* dTc() const { return at(sp(9) + 2 * i8); }
  __device__ __forceinline__ double* P() const { return at(sp(9) + 3 * i8); }
  __device__ __forceinline__ double* dqs() const { return at(sp(9) + 4 * i8); }
  __device__ __forceinline__ void* M() const { return smem + off_M; }
  __device__ __forceinline__ int* piv() const { return reinterpret_cast<int*>(smem + off_piv); }
  __device__ __forceinline__ int* perm() const { return reinterpret_cast<int*>(smem + off_piv + n8 / 2); }
  __device__ __forceinline__ double* invd() const { return at(off_piv + n8); }
  // the exponential's table
  __device__ __forceinline__ const unsigned long long* xt() const {
    return x_tab ? reinterpret_cast<const unsigned long long*>(smem + 64 * sizeof(double)) : g_fx_exp_tab;
  }
  // float-float assembly: mass-action sum (k, j), see set_matrix
  __device__ __forceinline__ ff2& pair(int k, int j) const {
    ff2* a = reinterpret_cast<ff2*>(M0);
    return i0 ? a[(size_t)(Km + 1) * ld0 + k * Km + j] : a[(1 + j) * ld0 + 1 + k];
  }

  __device__ void bind(const Layout& L) {
    tid = threadIdx.x;
    lane = tid & 31;
    warp = tid >> 5;
    vec = (unsigned)L.off_vec;
    n8 = 8 * L.nmax;
    k8 = 8 * L.Kmax;
    i8 = 8 * L.Imax;
    off_M = (unsigned)L.off_M;
    off_piv = (unsigned)L.off_piv;
    M0 = smem + L.off_M0;
    ld0 = L.ld;
    i0 = 0;
    Km = L.Kmax;
    x_tab = L.x_tab;
    if (x_tab) {
      unsigned long long* t = reinterpret_cast<unsigned long long*>(smem + 64 * sizeof(double));
#pragma unroll 1
      for (int i = tid; i < 256; i += NT) t[i] = g_fx_exp_tab[i];
      __syncthreads();
    }
  }

  // The mechanism's matrix geometry. In the CTA's global-memory slot (slot != null) a
  // column starts at a 32-byte boundary for row 1, so that four rows of a column are one
  // sector, and the mass-action sums have rows of their own behind the matrix; in shared
  // memory the odd leading dimension avoids bank conflicts and the sums take the places of
  // the finished entries.
  __device__ void set_matrix(int K, double* slot) {
    Km = K;
    if (slot) {
      ld0 = slot_ld(K + 1);
      i0 = 3;
      M0 = slot;
    } else {
      ld0 = odd_ld(K + 1);
      i0 = 0;
    }
  }

  // A cell's pressure and the mechanism's 1/W, which every rate evaluation reads (from
  // shared memory: the tables' L1 lines are evicted between evaluations).
  __device__ void set_cell(const DevMech& m, double p) {
    p_rc = p / kRc;
    rc_p = kRc / p;
#pragma unroll 1
    for (int k = tid; k < m.K; k += NT) iW()[k] = m.invW[k];
  }

  // Sum of NV (1, 2 or 4) values over the CTA; every thread receives the same
  // totals (fixed summation order: deterministic). Only the first nw warps may hold
  // non-zero values, nw = warps_for(count) of a loop over count <= n entries.
  // The FP64 pipe, shared by the SM's four schedulers, bounds the integration, so
  // the sum is arranged to issue few FP64 instructions:
  //  1. each data warp folds its NV values into one value per lane by log2(NV)
  //     transposing butterfly levels (a lane keeps one of two values and adds the
  //     partner's half of it), so that lane groups of 32/NV lanes carry one value each;
  //  2. warps 1..nw-1 leave their lane values in the scratch vector sc (free outside
  //     the solves; 32 (nw-1) <= count <= n entries), warp 0 adds them lane by lane;
  //  3. warp 0 finishes the butterfly inside each lane group and passes the totals to
  //     fin(tot, out), which derives NO scalars from them; lane 0's out[] reaches
  //     every thread through shared memory, so scalar follow-up work (reciprocals,
  //     roots) runs on one warp, not all.
  // With two data warps: 6, 7 and 10 FP64 warp instructions for 1, 2 and 4 values,
  // against 11, 22 and 44 for one shuffle tree per value and warp.
  template <int NV, int NO, class F>
  __device__ void reduce(const double (&v)[NV], int nw, F fin, double (&out)[NO]) {
    static_assert(NV == 1 || NV == 2 || NV == 4, "reduce: 1, 2 or 4 values");
    static_assert(NO <= 8, "reduction slots");
    constexpr int LV = NV == 1 ? 0 : (NV == 2 ? 1 : 2);  // transposing levels
    double x = 0.0;
    if (warp < nw) {
      if constexpr (NV == 1) {
        x = v[0];
      } else {
        // level 16: lanes 0-15 keep value 0 (and 2), lanes 16-31 value 1 (and 3)
        const bool h16 = lane & 16;
        x = (h16 ? v[1] : v[0]) + __shfl_xor_sync(FULLMASK, h16 ? v[0] : v[1], 16);
        if constexpr (NV == 4) {
          const double x2 = (h16 ? v[3] : v[2]) + __shfl_xor_sync(FULLMASK, h16 ? v[2] : v[3], 16);
          // level 8: lanes with bit 3 clear keep values 0/1, set keep 2/3
          const bool h8 = lane & 8;
          x = (h8 ? x2 : x) + __shfl_xor_sync(FULLMASK, h8 ? x : x2, 8);
        }
      }
      if (warp > 0) sc()[(warp - 1) * 32 + lane] = x;
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll 1
      for (int w = 1; w < nw; ++w) x += sc()[(w - 1) * 32 + lane];
#pragma unroll
      for (int o = 16 >> LV; o; o >>= 1) x += __shfl_xor_sync(FULLMASK, x, o);
      double tot[NV];
#pragma unroll
      for (int a = 0; a < NV; ++a) {
        // value a's lane group: bit 4 = a & 1, bit 3 = a >> 1
        const int src = NV == 1 ? 0 : (((a & 1) << 4) | ((a >> 1) << 3));
        tot[a] = NV == 1 ? x : __shfl_sync(FULLMASK, x, src);
      }
      double o[NO];
      fin(tot, o);
      if (lane == 0) {
#pragma unroll
        for (int b = 0; b < NO; ++b) red()[SC_OUT + b] = o[b];
      }
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < NO; ++b) out[b] = red()[SC_OUT + b];
  }

  // Plain CTA sum of NV values (nw as in reduce).
  template <int NV>
  __device__ void sum(double (&v)[NV], int nw) {
    reduce(v, nw, [](const double (&t)[NV], double (&o)[NV]) {
#pragma unroll
      for (int a = 0; a < NV; ++a) o[a] = t[a];
    }, v);
  }
};

// number of warps that hold data in a loop `for (i = tid; i < count; i += NT)`
template <int NW>
__device__ __forceinline__ int warps_for(int count) {
  const int w = (count + 31) >> 5;
  return w < NW ? w : NW;
}

// Cell-level scalars shared by all threads of the CTA (identical in every thread).
struct Scal {
  double T, invT, rho, irho, Wbar, icpm, fT, dcpm, Scpw;
};

// ---------------------------------------------------------------------------
// thermo, rates, RHS and the per-reaction Jacobian data
// ---------------------------------------------------------------------------
// RHS of y = [T, Y] at constant p into f[0..K]. With JAC, also the data the
// Jacobian assembly needs: per reaction the slot derivatives dq/dC, dq/dT at
// fixed C, sum_k C_k dq/dC_k (D), and the third-body/falloff coefficient P of
// eff_j in dq/dC_j; per species d_k = sum_i nu_ki D_i and a_kT = sum nu dTc.
// Rate constants come from one exponential each: kf from ln A + b ln T - Theta/T
// (+ the falloff terms), kr from that argument + dG/RT + dnu ln(Rc T/P0).
// FX: arguments, logarithms and exponentials in 64-bit fixed point (chem_fixed.cuh),
// for T in the range m.T_fx, where every argument fits; otherwise (FX = false, out of
// line) the same formulas in FP64. One RHS of the 54-species mechanism issues 196 FP64
// warp instructions with FX, 546 with FP64 exponentials and species factors
// exp(+-G/RT) (counted in the source); the FP64 pipe bounded the rate evaluation.
// FF (the forms with FP32 factors): the third-body sums [M] in float-float, and the
// slot derivatives and P stored as float-float pairs for the assembly.
template <bool FX>
__device__ __forceinline__ double rate_exp(typename std::conditional<FX, long long, double>::type a,
                                           const unsigned long long* tab) {
  if constexpr (FX) return fx_exp(a, tab);
  else return xexp(a);
}
template <bool FX>
__device__ __forceinline__ double rate_log(double x) {
  if constexpr (FX) {
    const int hx = __double2hiint(x);
    if (hx < 0x00100000 || hx >= 0x7ff00000) return log_outside(x);
    return fx_to_double(fx_log(x, 52));
  } else {
    return xlog(x);
  }
}

// One reaction's record: Arrhenius parameters in fixed point (Q52, Q56, Q45), species
// slots (reactants, products; 255 = empty), rev (DevMech::rx).
struct RxRec {
  long long lnA, b, th;
  unsigned slots;
  int rev;
};
__device__ __forceinline__ RxRec load_rec(const longlong2* rx, int i) {
  const longlong2 a = __ldg(rx + 2 * i), b = __ldg(rx + 2 * i + 1);
  return {a.x, a.y, b.x, (unsigned)b.y, (int)(b.y >> 32)};
}
// x with its sign bit flipped when sg = 2^31
__device__ __forceinline__ double flip_sign(double x, unsigned sg) {
  return __hiloint2double(__double2hiint(x) ^ (int)sg, __double2loint(x));
}

template <int NW, bool JAC, bool FF, bool FX>
__device__ Scal eval_rhs_t(const DevMech& m, Cta<NW>& c, const double* y, double p, double* f) {
  constexpr int NT = NW * 32;
  using Arg = typename std::conditional<FX, long long, double>::type;
  auto sum = [](Arg a, Arg b) -> Arg {
    if constexpr (FX) return fx_add(a, b);
    else return a + b;
  };
  auto difference = [](Arg a, Arg b) -> Arg {
    if constexpr (FX) return fx_sub(a, b);
    else return a - b;
  };
  const int K = m.K;
  Scal s;
  s.T = y[0];
  // Phase A: Y/W of every species and its sum; ln T and 1/T on the scalar warp.
  if (c.warp == Cta<NW>::SW) {
    const double lg = FX ? __longlong_as_double(fx_log(s.T, 58)) : xlog(s.T);
    const double iT = xrcp(s.T);
    if (c.lane == 0) {
      c.red()[SC_LOGT] = lg;
      c.red()[SC_INVT] = iT;
    }
  }
  const int nsw = warps_for<NW>(K);  // warps that hold species
  ff2* const yWf = reinterpret_cast<ff2*>(c.dk());
  double part = 0.0;
#pragma unroll 1
  for (int k = c.tid; k < K; k += NT) {
    const double yW = y[1 + k] * c.iW()[k];
    c.C()[k] = yW;
    // copy for the third-body sums, in the slot of d_k (written after the reaction loop)
    if (FF) yWf[k] = ff_split(yW);
    else c.dk()[k] = yW;
    part += yW;
  }
  if (c.warp > 0 && c.warp < nsw) c.sc()[(c.warp - 1) * 32 + c.lane] = part;
  __syncthreads();
  // Phase B: the species warps finish the sum (warp 0) and evaluate the species; the other
  // warps meanwhile take the third-body sums, which need Y/W only: [M] = rho sum eff Y/W.
  // The species warps wait for warp 0's scalars on a barrier of their own.
  if (c.warp < nsw) {
    if (c.warp == 0) {
#pragma unroll 1
      for (int w = 1; w < nsw; ++w) part += c.sc()[(w - 1) * 32 + c.lane];
#pragma unroll
      for (int o = 16; o; o >>= 1) part += __shfl_xor_sync(FULLMASK, part, o);
      const double Wbar = xrcp(part);
      const double rho = c.p_rc * c.red()[SC_INVT] * Wbar;  // p Wbar / (Rc T)
      const double irho = c.rc_p * s.T * part;
      if (c.lane == 0) {
        c.red()[SC_OUT] = Wbar;
        c.red()[SC_OUT + 1] = rho;
        c.red()[SC_OUT + 2] = irho;
      }
    }
    if (nsw == NW) __syncthreads();
    else if (nsw > 1) asm volatile("bar.sync 1, %0;" ::"r"(nsw * 32) : "memory");
    else __syncwarp();
  }
  const double lgT = c.red()[SC_LOGT];
  s.invT = c.red()[SC_INVT];
  const double T = s.T, invT = s.invT;
  // ln T (Q60), 1/T (Q71) and ln(Rc T/P0) (Q52), or their FP64 forms
  const unsigned long long LT = (unsigned long long)__double_as_longlong(lgT) << 2;
  const unsigned long long IT = fx_scale(invT, 19);
  const Arg lc = FX ? (Arg)((long long)(LT >> 8) + kLnRcP0_Q52) : (Arg)(lgT + kLnRcP0);
  Arg* const g_RT = reinterpret_cast<Arg*>(c.g());
  // species: thermo, G/RT, concentrations
  if (c.warp < nsw) s.rho = c.red()[SC_OUT + 1];
#pragma unroll 1
  for (int k = c.tid; k < K; k += NT) {
    const bool low = T < m.T_mid[k];
    double cp, h;
    const double2* a = m.hcp + 10 * k + (low ? 0 : 5);
    const double2 a0 = a[0], a1 = a[1], a2 = a[2], a3 = a[3], a4 = a[4];
    cp = a0.x + T * (a0.y + T * (a1.x + T * (a1.y + T * a2.x)));
    h = a0.x + T * (a2.y + T * (a3.x + T * (a3.y + T * a4.x))) + a4.y * invT;
    c.cpR()[k] = cp;
    c.hRT()[k] = h;
    if constexpr (FX) {
      // T 2^(fx_low - 12) below T_mid, T / 8192 above (Q64)
      const unsigned long long t = fx_scale(T, low ? m.fx_low : -1);
      const longlong2* q = reinterpret_cast<const longlong2*>(m.gfx + 16 * k + (low ? 0 : 8));
      const longlong2 q0 = q[0], q1 = q[1], q2 = q[2], q3 = q[3];
      const long long poly = fx_mul(q1.y + fx_mul(q2.x + fx_mul(q2.y + fx_mul(q3.x, t), t), t), t);
      g_RT[k] = fx_add(fx_add(q0.x, fx_mul(q0.y, LT)), fx_add(fx_mul(q1.x, IT), poly));
    } else {
      const double* b = m.nasa + 36 * k + (low ? 0 : 17);
      const double sr = b[11] * lgT + T * (b[12] + T * (b[13] + T * (b[14] + T * b[15]))) + b[16];
      g_RT[k] = h - sr;
    }
    c.C()[k] *= s.rho;
    if (JAC) c.dcp()[k] = a0.y + T * (2.0 * a1.x + T * (3.0 * a1.y + T * 4.0 * a2.x));
  }
  // third-body sums of 32 reactions at a time into their q slots, efficiencies species-
  // major: the warp's 32 reactions read one row per species
  constexpr int v = NW == 2 ? 0 : NW == 4 ? 1 : 2;
#pragma unroll 1
  for (int pos = m.tb_sched[v][c.warp]; pos < m.tb_sched[v][c.warp + 1]; ++pos) {
    const int r = m.tb_sched[v][NW + 1 + pos] * 32 + c.lane, ntb = m.n_tb;
    double S;
    if (FF) {
      // eight terms at a time, the next eight efficiencies loaded while these are summed
      // (the loads past the last species reach the table's padding, eff_rows)
      constexpr int B = kEffBatch;
      const ff2* ef = m.effT_ff + r;
      ff_sum acc;
      ff2 e[B];
#pragma unroll
      for (int u = 0; u < B; ++u) e[u] = ef[u * ntb];
#pragma unroll 1
      for (int k = 0; k < K; k += B) {
        ff2 y4[B], en[B];
        ef += B * ntb;
#pragma unroll
        for (int u = 0; u < B; ++u) {
          en[u] = ef[u * ntb];
          y4[u] = k + u < K ? yWf[k + u] : ff2{0.0f, 0.0f};
        }
#pragma unroll
        for (int u = 0; u < B; ++u) acc.add_prod(e[u], y4[u]);
#pragma unroll
        for (int u = 0; u < B; ++u) e[u] = en[u];
      }
      S = ff_value(acc.value());
    } else {
      const double* e = m.effT + r;
      S = 0.0;
#pragma unroll 6
      for (int k = 0; k < K; ++k) S += e[(size_t)k * ntb] * c.dk()[k];
    }
    c.q()[m.i_tb0 + r] = S;
  }
  __syncthreads();
  s.Wbar = c.red()[SC_OUT];
  s.rho = c.red()[SC_OUT + 1];
  s.irho = c.red()[SC_OUT + 2];
  // 32-reaction chunks of one kind each, dealt to the warps by estimated time; the next
  // chunk's record is loaded while this one is evaluated
  const int* cs = m.chunk_sched[v];
  const int pos1 = cs[c.warp + 1];
  int pos = cs[c.warp];
  int i_next = pos < pos1 ? cs[NW + 1 + pos] * 32 + c.lane : 0;
  RxRec rec_next = {};
  if (pos < pos1) rec_next = load_rec(m.rx, i_next);
#pragma unroll 1
  for (; pos < pos1; ++pos) {
    const int i = i_next;
    const RxRec rec = rec_next;
    if (pos + 1 < pos1) {
      i_next = cs[NW + 2 + pos] * 32 + c.lane;
      rec_next = load_rec(m.rx, i_next);
    }
    const int4 sl = make_int4(rec.slots & 255u, (rec.slots >> 8) & 255u, (rec.slots >> 16) & 255u, rec.slots >> 24);
    if (sl.x == 255) {  // null padding reaction
      c.q()[i] = 0.0;
      if (JAC) {
        c.D()[i] = c.dTc()[i] = c.P()[i] = 0.0;
        c.dqs()[4 * i] = c.dqs()[4 * i + 1] = c.dqs()[4 * i + 2] = c.dqs()[4 * i + 3] = 0.0;
      }
      continue;
    }
    Arg ka;  // ln kf
    double b_rx = 0.0, th_rx = 0.0, dnu = 0.0;
    if (!FX || JAC) {
      const double2 a01 = reinterpret_cast<const double2*>(m.arr + 4 * i)[0];
      const double2 a23 = reinterpret_cast<const double2*>(m.arr + 4 * i)[1];
      b_rx = a01.y;
      th_rx = a23.x;
      dnu = a23.y;
      if (!FX) ka = (Arg)(a01.x + a01.y * lgT - a23.x * invT);
    }
    if constexpr (FX) ka = fx_sub(fx_add(rec.lnA, fx_mul(rec.b, LT)), fx_mul(rec.th, IT));
    const bool two_f = sl.y != 255, two_r = sl.w != 255;
    const double Ca = c.C()[sl.x];
    const double Cb = two_f ? c.C()[sl.y] : 1.0;
    const double Cc = c.C()[sl.z];
    const double Cd = two_r ? c.C()[sl.w] : 1.0;
    const int rv = rec.rev;
    // factor of the mass-action rate: 1, [M], or [M] / (1 + Pr) (falloff)
    double Mc = 0.0, phi = 1.0, red1 = 1.0;
    double dlnk = (b_rx + th_rx * invT) * invT, gM = 1.0;  // d ln k/dT; d ln q/d ln[M]
    if (i >= m.i_tb0) {
      Mc = s.rho * c.q()[i];
      phi = Mc;
    }
    if (i >= m.i_fo0) {
      // k = k0 F / (1 + Pr) [M] with Pr = (k0/kinf) [M]; the tables hold the low-pressure
      // minus the high-pressure Arrhenius parameters, so ln k0 = ln kinf + fa
      const double* fo = m.fo + 8 * (i - m.i_fo0);
      Arg fa;
      if constexpr (FX) {
        const long long* x = m.fox + 4 * (i - m.i_fo0);
        fa = fx_sub(fx_add(x[0], fx_mul(x[1], LT)), fx_mul(x[2], IT));
      } else {
        fa = fo[0] + fo[1] * lgT - fo[2] * invT;
      }
      const double Pr = rate_exp<FX>(fa, c.xt()) * Mc;
      red1 = xrcp(1.0 + Pr);
      double dlgF_dL = 0.0, dlnF_dT = 0.0;
      ka = sum(ka, fa);
      if (i >= m.i_troe0) {
        const double alpha = fo[3];
        // fo[4] = 1/T***, fo[5] = 1/T*
        const double x3 = -T * fo[4], x1 = -T * fo[5];
        // (rolled loops: one copy of the exponential and of the logarithm in the code)
        double e3 = 0.0, e1 = 0.0, e2 = 0.0;
        const int ne = fo[6] > 0.0 ? 3 : 2;
#pragma unroll 1
        for (int u = 0; u < ne; ++u) {
          const double xa = u == 0 ? x3 : u == 1 ? x1 : -fo[6] * invT;
          double ex;
          if constexpr (FX) ex = fx_exp(fx_from_double(xa), c.xt());
          else ex = xexp(xa);
          if (u == 0) e3 = ex;
          else if (u == 1) e1 = ex;
          else e2 = ex;
        }
        const double Fc = (1.0 - alpha) * e3 + alpha * e1 + e2;
        double lF = 0.0, lP = 0.0;  // natural logarithms
#pragma unroll 1
        for (int u = 0; u < 2; ++u) {
          const double l = rate_log<FX>(u == 0 ? Fc : Pr);
          if (u == 0) lF = l;
          else lP = l;
        }
        const double cc = fma(lF, -0.67 * kInvLn10, -0.4), nn = fma(lF, -1.27 * kInvLn10, 0.75);
        const double x = fma(lP, kInvLn10, cc);
        const double den = fma(x, -0.14, nn);
        double lnF;
        if (JAC) {
          const double iden = xrcp(den);
          const double f1 = x * iden;
          const double ig = xrcp(fma(f1, f1, 1.0));
          lnF = lF * ig;
          const double lgF = lnF * kInvLn10;
          // partial derivatives of log10 F by log10 Pr and by log10 Fc
          const double df1_dL = nn * iden * iden;
          const double df1_dlF = (-0.67 - f1 * (-1.27 + 0.14 * 0.67)) * iden;
          dlgF_dL = -2.0 * lgF * ig * f1 * df1_dL;
          const double dlgF_dlF = ig - 2.0 * lgF * ig * f1 * df1_dlF;
          double dFc = -(1.0 - alpha) * fo[4] * e3 - alpha * fo[5] * e1;
          if (fo[6] > 0.0) dFc += fo[6] * invT * invT * e2;
          dlnF_dT = dlgF_dlF * dFc * xrcp(Fc);  // d ln F / dT at fixed Pr
        } else {
          const double den2 = den * den;
          lnF = lF * (den2 * xrcp(fma(x, x, den2)));
        }
        if constexpr (FX) {
          ka = fx_add(ka, fx_from_double(lnF));
          if ((__double2hiint(lnF) & 0x7ff00000) == 0x7ff00000) red1 = lnF;  // NaN: no valid [M] or Fc
        } else {
          ka += lnF;
        }
      }
      phi = Mc * red1;
      if (JAC) {
        gM = red1 + dlgF_dL;  // d ln k/d ln Pr
        dlnk += gM * (fo[1] + fo[2] * invT) * invT + dlnF_dT;
      }
    }
    const double kfP = rate_exp<FX>(ka, c.xt());
    double krP = 0.0;
    if (rv & 1) {
      Arg dg = difference(g_RT[sl.z], g_RT[sl.x]);
      if (two_r) dg = sum(dg, g_RT[sl.w]);
      if (two_f) dg = difference(dg, g_RT[sl.y]);
      dg = sum(dg, (rv >> 1) == 2 ? lc : (rv >> 1) == 0 ? -lc : Arg(0));
      krP = rate_exp<FX>(sum(ka, dg), c.xt());
    }
    const double Pf = Ca * Cb, Pb = Cc * Cd;
    if constexpr (!JAC) {
      const double net = fma(kfP, Pf, -krP * Pb);
      c.q()[i] = i >= m.i_tb0 ? phi * net : net;
    } else {
      const double qf = kfP * Pf, qr = krP * Pb;
      const double net = qf - qr;
      c.q()[i] = i >= m.i_tb0 ? phi * net : net;
      // d ln Kc / dT = dH/(R T^2) - dnu/T
      const double dH = c.hRT()[sl.z] + (two_r ? c.hRT()[sl.w] : 0.0) - c.hRT()[sl.x] -
                        (two_f ? c.hRT()[sl.y] : 0.0);
      const double dlnKc = (dH - dnu) * invT;
      const double kfp = phi * kfP, krp = -phi * krP;
      const double dq0 = kfp * Cb, dq1 = two_f ? kfp * Ca : 0.0;
      const double dq2 = krp * Cd, dq3 = two_r ? krp * Cc : 0.0;
      if (FF) {
        // the float-float assembly's copy (hi, lo), split once here
        ff2* dqf = reinterpret_cast<ff2*>(c.dqs()) + 4 * i;
        dqf[0] = ff_split(dq0);
        dqf[1] = ff_split(dq1);
        dqf[2] = ff_split(dq2);
        dqf[3] = ff_split(dq3);
      } else {
        c.dqs()[4 * i] = dq0;
        c.dqs()[4 * i + 1] = dq1;
        c.dqs()[4 * i + 2] = dq2;
        c.dqs()[4 * i + 3] = dq3;
      }
      c.dTc()[i] = phi * fma(dlnk, net, qr * dlnKc);
      const double Pc = i >= m.i_tb0 ? gM * red1 * net : 0.0;
      if (FF)
        reinterpret_cast<ff2*>(c.P())[i] = ff_split(Pc);
      else
        c.P()[i] = Pc;
      // sum_k C_k dq/dC_k: the mass-action orders, and [M]
      double Dsum = phi * ((two_f ? 2.0 * qf : qf) - (two_r ? 2.0 * qr : qr));
      if (i >= m.i_tb0) Dsum = fma(Mc, Pc, Dsum);
      c.D()[i] = Dsum;
    }
  }
  const uint2* ps = m.ps_ent[v] + c.tid;
  uint2 en = ps[0];  // (in flight across the barrier)
  // cp (and d cp/dT) of the mixture, on the scalar warp: mean over C, rho sum Y/W x = sum C x
  if (c.warp == Cta<NW>::SW) {
    double cs1 = 0.0, cs2 = 0.0;
#pragma unroll 1
    for (int k = c.lane; k < K; k += 32) {
      cs1 += c.C()[k] * c.cpR()[k];
      if (JAC) cs2 += c.C()[k] * c.dcp()[k];
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      cs1 += __shfl_xor_sync(FULLMASK, cs1, o);
      if (JAC) cs2 += __shfl_xor_sync(FULLMASK, cs2, o);
    }
    const double rr = kRc * s.irho;
    const double icpm = xrcp(cs1 * rr);
    if (c.lane == 0) {
      c.red()[SC_ICPM] = icpm;
      if (JAC) c.red()[SC_DCPM] = cs2 * rr;
    }
  }
  __syncthreads();
  // Production rates: each species' reactions over a group of ps_g adjacent lanes, from a
  // table of 16-bit entries (reaction << 1 | sign), four to a load and padded to the
  // longest list; the signed terms are added one FP64 instruction each.
#pragma unroll 1
  for (int pass = 0; pass < m.ps_passes[v]; ++pass) {
    const int g = m.ps_g[v];
    double w = 0.0, dd = 0.0, at = 0.0;
    auto add = [&](unsigned e) {
      if (e != 0xffffu) {
        const unsigned i = e >> 1, sg = e << 31;
        w += flip_sign(c.q()[i], sg);
        if (JAC) {
          dd += flip_sign(c.D()[i], sg);
          at += flip_sign(c.dTc()[i], sg);
        }
      }
    };
#pragma unroll 1
    for (int r = 0; r < m.ps_quads[v]; ++r) {
      const uint2 e = en;
      const int nx = pass * m.ps_quads[v] + r + 1;
      if (nx < m.ps_passes[v] * m.ps_quads[v]) en = ps[(size_t)nx * NT];
      add(e.x & 0xffffu);
      add(e.x >> 16);
      add(e.y & 0xffffu);
      add(e.y >> 16);
    }
#pragma unroll 1
    for (int o = 1; o < g; o <<= 1) {
      w += __shfl_xor_sync(FULLMASK, w, o);
      if (JAC) {
        dd += __shfl_xor_sync(FULLMASK, dd, o);
        at += __shfl_xor_sync(FULLMASK, at, o);
      }
    }
    const int k = (pass * NT + c.tid) / g;
    if ((c.tid & (g - 1)) == 0 && k < K) {
      c.ek()[k] = w;
      if (JAC) {
        c.dk()[k] = dd;
        c.akT()[k] = at;
      }
    }
  }
  __syncthreads();
  // species: f_k and the enthalpy sums
  s.icpm = c.red()[SC_ICPM];
  if (JAC) s.dcpm = c.red()[SC_DCPM];
  {
    double part2[JAC ? 2 : 1] = {};
#pragma unroll 1
    for (int k = c.tid; k < K; k += NT) {
      const double w = c.ek()[k];
      f[1 + k] = m.W[k] * w * s.irho;
      part2[0] += c.hRT()[k] * w;  // Qh / (Rc T)
      if (JAC) part2[JAC ? 1 : 0] += c.cpR()[k] * w;  // sum cp_k omega_k / Rc
    }
    double o[2];
    const double T = s.T, irho = s.irho, icpm = s.icpm;
    c.reduce(part2, nsw, [&](const double (&t)[JAC ? 2 : 1], double (&r)[2]) {
      const double fT = -kRc * T * t[0] * irho * icpm;  // -Qh / (rho cp), Qh = Rc T sum hRT_k w_k
      r[0] = fT;
      r[1] = JAC ? kRc * t[JAC ? 1 : 0] : 0.0;
      if (c.lane == 0) f[0] = fT;  // visible after the reduction's last barrier
    }, o);
    s.fT = o[0];
    s.Scpw = o[1];
  }
  return s;
}

// (The CTA's pointers are passed by value: a reference to them that leaves the caller
// would keep them in local memory there, to be read again after every store.)
template <int NW, bool JAC, bool FF>
__device__ __noinline__ Scal eval_rhs_fp64(const DevMech& m, Cta<NW> c, const double* y, double p, double* f) {
  return eval_rhs_t<NW, JAC, FF, false>(m, c, y, p, f);
}

// RHS (and with JAC the Jacobian data) of the state y; T = y[0] selects the path.
template <int NW, bool JAC, bool FF = false>
__device__ __forceinline__ Scal eval_rhs(const DevMech& m, Cta<NW>& c, const double* y, double p, double* f) {
  const int2 range = m.T_fx;
  const int hT = __double2hiint(y[0]);  // (NaN is above every range)
  if (hT < range.x || hT >= range.y) return eval_rhs_fp64<NW, JAC, FF>(m, c, y, p, f);
  return eval_rhs_t<NW, JAC, FF, true>(m, c, y, p, f);
}

// ---------------------------------------------------------------------------
// Jacobian assembly (precision R) from the data of eval_rhs<JAC=true>.
// With A_kj = sum_i nu_ki dq_i/dC_j (mass-action slot terms plus the third-body /
// falloff term nu_ki P_i eff_ij), the species rows of the Jacobian are
//   J_kj = (W_k / W_j) (A_kj - (Wbar/rho) d_k) + f_k Wbar / W_j,
// so with sg = -1 for the iteration matrix M = I/(h gamma) - J (rf = 1/(h gamma))
// and sg = +1, rf = 0 for the Jacobian itself (JO), the stored value is
//   S_kj = B_kj / W_j + rf delta_kj,  B_kj = sg W_k A_kj + beta_k,
//   beta_k = sg (f_k Wbar - W_k (Wbar/rho) d_k).
// (1) species pass: e_k = h_k / (W_k cp), beta_k, the temperature column
//     J_k0 = (W_k/rho)(a_kT - d_k/T) + f_k/T; and the mass-action pair sums
//     sum sg nu_ki W_k dq_i/dC_j on the thread-balanced schedule, stored in place;
// (2) one warp per row: beta + pair sum, the dense third-body part in registers
//     (lane l holds columns l + 32 u), scaled by 1/W_j;
// (3) temperature row from column sums of the stored rows:
//     J_0j = -sum_k e_k J_kj - f_T cp_j/(W_j cp),
//     J_00 = -sum_k e_k J_k0 - sum_k cp_k omega_k/(rho cp) - f_T cp'/cp.
// ---------------------------------------------------------------------------
template <class R>
__device__ __forceinline__ R fmaR(R a, R b, R c) {
  if constexpr (std::is_same<R, float>::value) return fmaf(a, b, c);
  else return fma(a, b, c);
}

// FFD: the per-reaction data (dq/dC, P) is stored as float-float pairs (the forms
// with FP32 factors); R = float then reads their hi parts.
template <bool FFD>
__device__ __forceinline__ double rx_data(const double* a, int i) {
  if constexpr (FFD) return (double)reinterpret_cast<const ff2*>(a)[i].hi;
  else return a[i];
}

// Entry (i, j) of the assembled matrix at i si + j sj.
template <int NW, class R, bool JO, int U, bool FFD>
__device__ void assemble_rows(const DevMech& m, Cta<NW>& c, R* A, int K, int si, int sj, R rf) {
  constexpr double SG = JO ? 1.0 : -1.0;
#pragma unroll 1
  for (int k = c.warp; k < K; k += NW) {
    R* row = A + (1 + k) * si + sj;
    const R beta = R(c.akT()[k]), Wk = R(SG * m.W[k]);
    R acc[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const unsigned msk = m.jmask[k * U + u];
      acc[u] = ((msk >> c.lane) & 1u) ? fmaR(Wk, row[(c.lane + 32 * u) * sj], beta) : beta;
    }
    // third-body / falloff part: 32 row coefficients sg nu_ki W_k P_i at a time,
    // broadcast from their lanes
    const int t1 = m.tr_ptr[k + 1];
#pragma unroll 1
    for (int tb = m.tr_ptr[k]; tb < t1; tb += 32) {
      const int t = tb + c.lane;
      R cl = R(0);
      int rl = 0;
      if (t < t1) {
        const int ri = m.tr_ent[t].x;
        cl = R(SG * m.tr_nu[t] * rx_data<FFD>(c.P(), ri));
        rl = ri - m.i_tb0;
      }
      const int cnt = min(32, t1 - tb);
#pragma unroll 1
      for (int q = 0; q < cnt; ++q) {
        const R coef = __shfl_sync(FULLMASK, cl, q);
        const double* e = m.eff + (size_t)__shfl_sync(FULLMASK, rl, q) * K;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int j = c.lane + 32 * u;
          if (u < U - 1 || j < K) acc[u] = fmaR(coef, R(e[j]), acc[u]);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = c.lane + 32 * u;
      if (u < U - 1 || j < K) row[j * sj] = fmaR(acc[u], R(c.iW()[j]), j == k ? rf : R(0));
    }
  }
}

// Mass-action sums sum_i nu_ki dq_i/dC_j, one per existing (k, j), on the thread-balanced
// schedule js: entry x = (dq index) << 1 | sign (~0: padding), y = k << 8 | j where the
// finished sum goes (~0: it continues); put(k, j, sum) stores it. The entries are loaded
// four rounds ahead: the table streams through once per step and misses the L1 cache.
template <int NW, class Acc, class Get, class Put>
__device__ void mass_action_sums(const DevMech& m, Cta<NW>& c, Get get, Put put) {
  constexpr int NT = NW * 32, v = NT == 64 ? 0 : NT == 128 ? 1 : 2, B = 4;
  const uint2* se = m.js_ent[v] + c.tid;
  const int rounds = m.js_rounds[v];  // a multiple of B
  uint2 e[B], en[B];
#pragma unroll
  for (int u = 0; u < B; ++u) en[u] = ld_stream(se + u * NT);
  Acc a{};
#pragma unroll 1
  for (int r = 0; r < rounds; r += B) {
#pragma unroll
    for (int u = 0; u < B; ++u) e[u] = en[u];
    if (r + B < rounds) {
#pragma unroll
      for (int u = 0; u < B; ++u) en[u] = ld_stream(se + (size_t)(r + B + u) * NT);
    }
#pragma unroll
    for (int u = 0; u < B; ++u) {
      if (e[u].x != 0xffffffffu) get(a, (int)(e[u].x >> 1), e[u].x << 31);
      if (e[u].y != 0xffffffffu) {
        put((int)(e[u].y >> 8), (int)(e[u].y & 255u), a);
        a = Acc{};
      }
    }
  }
}

// FP64 form: row-major in the LU matrix (BYCOL = false); FP32-assembled form: by columns.
template <int NW, class R, bool JO, bool FFD = false, bool BYCOL = false>
__device__ void assemble(const DevMech& m, Cta<NW>& c, const Scal& s, const double* f, double fac, void* target) {
  constexpr int NT = NW * 32;
  constexpr double SG = JO ? 1.0 : -1.0;
  const int K = m.K, n = K + 1, ld = odd_ld(n);
  const int si = BYCOL ? 1 : ld, sj = BYCOL ? ld : 1;
  R* A = reinterpret_cast<R*>(target);
  const R rf = JO ? R(0) : R(fac);
  // (1) species pass
  const double eT = kRc * s.T * s.icpm, wr = s.Wbar * s.irho;
#pragma unroll 1
  for (int k = c.tid; k < K; k += NT) {
    c.ek()[k] = c.hRT()[k] * eT * c.iW()[k];
    const double Wk = m.W[k], dk = c.dk()[k], fk = f[1 + k];
    A[(1 + k) * si] = R(SG * (Wk * s.irho * (c.akT()[k] - dk * s.invT) + fk * s.invT));
    c.akT()[k] = SG * (fk * s.Wbar - Wk * wr * dk);  // beta_k (a_kT is consumed)
  }
  mass_action_sums<NW, R>(
      m, c,
      [&](R& a, int i, unsigned sg) {
        if constexpr (FFD)
          a += __uint_as_float(__float_as_uint(reinterpret_cast<const ff2*>(c.dqs())[i].hi) ^ sg);
        else
          a += flip_sign(c.dqs()[i], sg);
      },
      [&](int k, int j, R a) { A[(1 + k) * si + (1 + j) * sj] = a; });
  __syncthreads();
  // (2) species rows
  switch ((K + 31) >> 5) {
    case 1: assemble_rows<NW, R, JO, 1, FFD>(m, c, A, K, si, sj, rf); break;
    case 2: assemble_rows<NW, R, JO, 2, FFD>(m, c, A, K, si, sj, rf); break;
    case 3: assemble_rows<NW, R, JO, 3, FFD>(m, c, A, K, si, sj, rf); break;
    case 4: assemble_rows<NW, R, JO, 4, FFD>(m, c, A, K, si, sj, rf); break;
    case 5: assemble_rows<NW, R, JO, 5, FFD>(m, c, A, K, si, sj, rf); break;
    case 6: assemble_rows<NW, R, JO, 6, FFD>(m, c, A, K, si, sj, rf); break;
    case 7: assemble_rows<NW, R, JO, 7, FFD>(m, c, A, K, si, sj, rf); break;
    default: assemble_rows<NW, R, JO, 8, FFD>(m, c, A, K, si, sj, rf); break;
  }
  __syncthreads();
  // (3) temperature row; with acc = sum_k e_k S_kj, sum_k e_k J_kj = sg (acc - rf e_(j-1)),
  //     so S_0j = rf e_(j-1) - acc - sg extra_j (j >= 1) and S_00 = rf - acc - sg extra_0
  const double ft = s.fT * s.icpm;
#pragma unroll 1
  for (int j = NT - 1 - c.tid; j < n; j += NT) {  // from the last warp down, as the residual rows
    R acc = R(0);
#pragma unroll 1
    for (int k = 0; k < K; ++k) acc = fmaR(R(c.ek()[k]), A[(1 + k) * si + j * sj], acc);
    R v;
    if (j == 0)
      v = rf - acc - R(SG * (s.Scpw * s.irho * s.icpm + ft * s.dcpm));
    else
      v = rf * R(c.ek()[j - 1]) - acc - R(SG * ft * c.cpR()[j - 1] * kRc * c.iW()[j - 1]);
    A[j * sj] = v;
  }
  __syncthreads();
}

// The same assembly in float-float arithmetic (the mixed form): the same terms in the
// same order, from float-float copies of the per-reaction data (dq/dC and P, split
// once by eval_rhs) and of the mechanism's constants (1/W, nu W, efficiencies), so
// that every sum and product of the pass runs on the FP32 pipe; the species-level
// scalars are formed in FP64 and split once per species. A holds (hi, lo) per entry;
// its error is a few units of 2^-48 relative to the sums' terms, far below the FP32
// factorisation's, so the refinement converges to the same solutions.
//
// A warp takes RG consecutive rows (lanes on the columns, all sums in registers), so that
// a lane finishes RG entries of a column side by side (one 32-byte sector for RG = 4), and
// adds e_k S_kj to its share of the temperature row; the warps' shares meet in shared
// memory (the vectors rr, u and sc). Third-body coefficients sg nu_ki W_k P_i come from
// shared memory (cf, in the place of dq once the mass-action sums have consumed it).
template <int NW, bool JO, int U, int RG>
__device__ void assemble_rows_ff(const DevMech& m, Cta<NW>& c, ff2* A, int K, ff2 rf) {
  const ff2* beta_ff = reinterpret_cast<const ff2*>(c.akT());
  const ff2* ek = reinterpret_cast<const ff2*>(c.ek());
  const ff2* cf = reinterpret_cast<const ff2*>(c.dqs());
  const ff2 zero = {0.0f, 0.0f};
  const int ld0 = c.ld0;
  ff2* A1 = A + c.i0 + 1;  // row of species 0
  ff_sum accT[U], accT0;
#pragma unroll 1
  for (int k0 = c.warp * RG; k0 < K; k0 += NW * RG) {
    ff2 S[RG][U];
#pragma unroll
    for (int rr = 0; rr < RG; ++rr) {
      const int k = k0 + rr;
#pragma unroll
      for (int u = 0; u < U; ++u) S[rr][u] = zero;
      if (k < K) {
        const ff2 beta = beta_ff[k], Wk = m.W_ff[k];
        ff_sum acc[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const unsigned msk = m.jmask[k * U + u];
          acc[u] = ff_sum(beta);
          if ((msk >> c.lane) & 1u) acc[u].add_prod(JO ? Wk : ff_neg(Wk), c.pair(k, c.lane + 32 * u));
        }
        const int t1 = m.tr_ptr[k + 1];
        // four entries at a time: their efficiencies' loads overlap (row: offset of the
        // entry's efficiencies; entries past the row's end have coefficient 0)
#pragma unroll 1
        for (int t = m.tr_ptr[k]; t < t1; t += 4) {
          ff2 e[4][U];
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const ff2* er = m.eff_ff + __ldg(m.tr_row + t + v);
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const int j = c.lane + 32 * u;
              if (u < U - 1 || j < K) {
                const float2 x = __ldg(reinterpret_cast<const float2*>(er + j));
                e[v][u] = {x.x, x.y};
              } else {
                e[v][u] = zero;
              }
            }
          }
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const ff2 coef = t + v < t1 ? cf[t + v] : zero;
#pragma unroll
            for (int u = 0; u < U; ++u) acc[u].add_prod(coef, e[v][u]);
          }
        }
        const ff2 ekk = ek[k];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int j = c.lane + 32 * u;
          S[rr][u] = u < U - 1 || j < K ? ff_fma(acc[u].value(), m.invW_ff[j], j == k ? rf : zero) : zero;
          accT[u].add_prod(ekk, S[rr][u]);
        }
        accT0.add_prod(ekk, A1[k]);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = c.lane + 32 * u;
      if (u < U - 1 || j < K) {
        ff2* o = A1 + (size_t)(1 + j) * ld0 + k0;
        if (RG % 2 == 0 && c.i0 != 0) {  // the slot: aligned and padded columns
#pragma unroll
          for (int rr = 0; rr < RG; rr += 2)
            if (k0 + rr < K)
              *reinterpret_cast<float4*>(o + rr) = make_float4(S[rr][u].hi, S[rr][u].lo, S[rr + 1 < RG ? rr + 1 : rr][u].hi,
                                                               S[rr + 1 < RG ? rr + 1 : rr][u].lo);
        } else {
#pragma unroll
          for (int rr = 0; rr < RG; ++rr)
            if (k0 + rr < K) o[rr] = S[rr][u];
        }
      }
    }
  }
  // the warp's share of the temperature row: entry j (0: temperature column) at warp n + j
  ff2* tp = reinterpret_cast<ff2*>(c.rr()) + c.warp * (K + 1);
  if (c.lane == 0) tp[0] = accT0.value();
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int j = c.lane + 32 * u;
    if (u < U - 1 || j < K) tp[1 + j] = accT[u].value();
  }
}

template <int NW, bool JO>
__device__ void assemble_ff(const DevMech& m, Cta<NW>& c, const Scal& s, const double* f, double fac, ff2* A) {
  constexpr int NT = NW * 32;
  constexpr double SG = JO ? 1.0 : -1.0;
  const int K = m.K, n = K + 1, ld0 = c.ld0;
  const ff2 zero = {0.0f, 0.0f};
  const ff2 rf = JO ? zero : ff_split(fac);
  ff2* ek = reinterpret_cast<ff2*>(c.ek());
  ff2* beta = reinterpret_cast<ff2*>(c.akT());
  const ff2* dq = reinterpret_cast<const ff2*>(c.dqs());
  // (1) species pass
  const double eT = kRc * s.T * s.icpm, wr = s.Wbar * s.irho;
#pragma unroll 1
  for (int k = c.tid; k < K; k += NT) {
    ek[k] = ff_split(c.hRT()[k] * eT * c.iW()[k]);
    const double Wk = m.W[k], dk = c.dk()[k], fk = f[1 + k];
    A[c.i0 + 1 + k] = ff_split(SG * (Wk * s.irho * (c.akT()[k] - dk * s.invT) + fk * s.invT));
    beta[k] = ff_split(SG * (fk * s.Wbar - Wk * wr * dk));  // beta_k (a_kT is consumed)
  }
  mass_action_sums<NW, ff_sum>(
      m, c,
      [&](ff_sum& a, int i, unsigned sg) {
        const ff2 d = dq[i];
        a.add({__uint_as_float(__float_as_uint(d.hi) ^ sg), __uint_as_float(__float_as_uint(d.lo) ^ sg)});
      },
      [&](int k, int j, const ff_sum& a) { c.pair(k, j) = a.value(); });
  __syncthreads();
  {
    // third-body coefficients (tr_ptr[K] <= 4 n_tb, dq holds 4 I pairs)
    const ff2* Pf = reinterpret_cast<const ff2*>(c.P());
    ff2* cf = reinterpret_cast<ff2*>(c.dqs());
    const int nt = m.tr_ptr[K];
#pragma unroll 1
    for (int t = c.tid; t < nt; t += NT) {
      const ff2 tn = m.tr_nu_ff[t];
      cf[t] = ff_mul(JO ? tn : ff_neg(tn), Pf[m.tr_ent[t].x]);
    }
  }
  __syncthreads();
  // (2) species rows
  switch ((K + 31) >> 5) {
    case 1: assemble_rows_ff<NW, JO, 1, 4>(m, c, A, K, rf); break;
    case 2: assemble_rows_ff<NW, JO, 2, 4>(m, c, A, K, rf); break;
    case 3: assemble_rows_ff<NW, JO, 3, 2>(m, c, A, K, rf); break;
    case 4: assemble_rows_ff<NW, JO, 4, 2>(m, c, A, K, rf); break;
    case 5: assemble_rows_ff<NW, JO, 5, 1>(m, c, A, K, rf); break;
    case 6: assemble_rows_ff<NW, JO, 6, 1>(m, c, A, K, rf); break;
    case 7: assemble_rows_ff<NW, JO, 7, 1>(m, c, A, K, rf); break;
    default: assemble_rows_ff<NW, JO, 8, 1>(m, c, A, K, rf); break;
  }
  __syncthreads();
  // (3) temperature row, as in assemble(), from the warps' shares
  const double ft = s.fT * s.icpm;
  const ff2* tp = reinterpret_cast<const ff2*>(c.rr());
#pragma unroll 1
  for (int j = c.tid; j < n; j += NT) {
    ff2 acc = tp[j];
#pragma unroll
    for (int w = 1; w < NW; ++w) acc = ff_add(acc, tp[w * n + j]);
    ff2 v;
    if (j == 0)
      v = ff_sub(ff_sub(rf, acc), ff_split(SG * (s.Scpw * s.irho * s.icpm + ft * s.dcpm)));
    else
      v = ff_sub(ff_sub(ff_mul(rf, ek[j - 1]), acc), ff_split(SG * ft * c.cpR()[j - 1] * kRc * c.iW()[j - 1]));
    A[j * ld0 + c.i0] = v;
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------
// Pivot candidates: every warp writes (max |value|, lowest row index) of its rows;
// every thread then reduces the NW partials in the same order (same result).
// ---------------------------------------------------------------------------
template <int NW>
__device__ __forceinline__ int pivot_reduce(Cta<NW>& c, float* pmax, int* pidx, int n) {
  float best = -1.0f;
  int bi = n;
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    const float v = pmax[w];
    const int i = pidx[w];
    if (v > best || (v == best && i < bi)) { best = v; bi = i; }
  }
  return bi;
}

// Warp-level (value, index) maximum with the lowest index on ties; lane 0 stores it.
__device__ __forceinline__ void warp_argmax_store(float v, int i, int lane, float* pmax, int* pidx, int warp) {
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const float ov = __shfl_xor_sync(FULLMASK, v, o);
    const int oi = __shfl_xor_sync(FULLMASK, i, o);
    if (ov > v || (ov == v && oi < i)) { v = ov; i = oi; }
  }
  if (lane == 0) {
    pmax[warp] = v;
    pidx[warp] = i;
  }
}

// ---------------------------------------------------------------------------
// dense LU with partial pivoting (row interchange to the largest |a_ik|, lowest
// row index on ties; the pivot choice compares magnitudes rounded to FP32), in
// place; the search for the next pivot is fused into the elimination, so each
// column costs two CTA barriers. Then the composed row permutation and the
// inverse diagonal of U for the solves. Returns 0 or 1 + k for a zero pivot.
// ---------------------------------------------------------------------------
template <int NW, class R>
__device__ int lu_factor(Cta<NW>& c, R* a, int n, bool pivot = true) {
  constexpr int NT = NW * 32;
  const int ld = odd_ld(n);
  float* pmax = reinterpret_cast<float*>(c.red() + SC_PIV);
  int* pidx = reinterpret_cast<int*>(c.red() + SC_PIV + NW);
  double* spinv = c.red() + SC_INVP;
  int info = 0;
  // candidates for column 0
  {
    float v = -1.0f;
    int bi = n;
#pragma unroll 1
    for (int i = c.tid; i < n; i += NT) {
      const float x = fabsf((float)a[i * ld]);
      if (x > v || (x == v && i < bi)) { v = x; bi = i; }
    }
    warp_argmax_store(v, bi, c.lane, pmax, pidx, c.warp);
  }
  __syncthreads();
#pragma unroll 1
  for (int k = 0; k < n; ++k) {
    int p = pivot ? pivot_reduce<NW>(c, pmax, pidx, n) : k;  // no pivoting: the diagonal
    if (p >= n) p = k;  // a column of NaN: the zero-pivot path below
    // the reciprocal on the thread that also interchanges column k: it reads the pivot
    // before its own store to that place, which no barrier separates from other threads
    if (c.tid == (k & (NT - 1))) {
      c.piv()[k] = p;
      const double pv = (double)a[p * ld + k];
      spinv[0] = pv != 0.0 && isfinite(pv) ? 1.0 / pv : 0.0;
    }
    if (p != k)
#pragma unroll 1
      for (int j = c.tid; j < n; j += NT) {
        const R t = a[k * ld + j];
        a[k * ld + j] = a[p * ld + j];
        a[p * ld + j] = t;
      }
    __syncthreads();
    const R invp = R(spinv[0]);
    if (invp == R(0) && info == 0) info = k + 1;
    float v = -1.0f;
    int bi = n;
#pragma unroll 1
    for (int i = k + 1 + c.warp; i < n; i += NW) {
      const R l = a[i * ld + k] * invp;
      __syncwarp();
      if (c.lane == 0) a[i * ld + k] = l;
#pragma unroll 1
      for (int j = k + 1 + c.lane; j < n; j += 32) {
        const R nv = a[i * ld + j] - l * a[k * ld + j];
        a[i * ld + j] = nv;
        if (j == k + 1) {
          const float x = fabsf((float)nv);
          if (x > v || (x == v && i < bi)) { v = x; bi = i; }
        }
      }
    }
    warp_argmax_store(v, bi, c.lane, pmax, pidx, c.warp);
    __syncthreads();
  }
  // composed permutation: position i of the pivoted system holds original row perm[i]
  if (c.tid == 0) {
    for (int i = 0; i < n; ++i) c.perm()[i] = i;
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
      const int p = c.piv()[k];
      const int t = c.perm()[k];
      c.perm()[k] = c.perm()[p];
      c.perm()[p] = t;
    }
  }
#pragma unroll 1
  for (int i = c.tid; i < n; i += NT) c.invd()[i] = 1.0 / (double)a[i * ld + i];
  __syncthreads();
  return info;
}

// Forward/back substitution by one warp, in place on x (already permuted).
template <class R>
__device__ void lu_solve_warp(const R* a, int n, const double* invd, R* x, int lane) {
  const int ld = odd_ld(n);
#pragma unroll 1
  for (int i0 = 0; i0 < n; i0 += 32) {
    const int i = i0 + lane;
    const int jend = min(i0 + 32, n);
    R xi = i < n ? x[i] : R(0);
#pragma unroll 1
    for (int j = i0; j < jend; ++j) {
      const R xj = __shfl_sync(FULLMASK, xi, j - i0);
      if (i > j && i < n) xi -= a[i * ld + j] * xj;
    }
    if (i < n) x[i] = xi;
    __syncwarp();
#pragma unroll 1
    for (int r = i0 + 32 + lane; r < n; r += 32) {
      R sacc = R(0);
#pragma unroll 1
      for (int j = i0; j < jend; ++j) sacc += a[r * ld + j] * x[j];
      x[r] -= sacc;
    }
    __syncwarp();
  }
  for (int i1 = n; i1 > 0; i1 -= 32) {
    const int i0 = max(0, i1 - 32);
    const int i = i0 + lane;
    R xi = i < i1 ? x[i] : R(0);
    for (int j = i1 - 1; j >= i0; --j) {
      if (i == j) xi *= R(invd[j]);
      const R xj = __shfl_sync(FULLMASK, xi, j - i0);
      if (i < j) xi -= a[i * ld + j] * xj;
    }
    if (i < i1) x[i] = xi;
    __syncwarp();
#pragma unroll 1
    for (int r = lane; r < i0; r += 32) {
      R sacc = R(0);
      for (int j = i0; j < i1; ++j) sacc += a[r * ld + j] * x[j];
      x[r] -= sacc;
    }
    __syncwarp();
  }
}

// In-place Gauss-Jordan inverse (FP32) with partial pivoting: row interchange to
// the largest |a_ik| (lowest row index on ties), the normalised pivot row kept in a
// copy while every other row is eliminated (the next pivot search is fused into
// that elimination: three CTA barriers per column); the inverse is completed by the
// column interchanges in reverse order. Returns 0 or 1 + k for a zero pivot.
template <int NW>
__device__ int gj_invert(Cta<NW>& c, float* a, int n) {
  constexpr int NT = NW * 32;
  const int ld = odd_ld(n);
  float* pmax = reinterpret_cast<float*>(c.red() + SC_PIV);
  int* pidx = reinterpret_cast<int*>(c.red() + SC_PIV + NW);
  float* pr = reinterpret_cast<float*>(c.rr());  // normalised pivot row
  int info = 0;
  {
    float v = -1.0f;
    int bi = n;
#pragma unroll 1
    for (int i = c.tid; i < n; i += NT) {
      const float x = fabsf(a[i * ld]);
      if (x > v || (x == v && i < bi)) { v = x; bi = i; }
    }
    warp_argmax_store(v, bi, c.lane, pmax, pidx, c.warp);
  }
  __syncthreads();
#pragma unroll 1
  for (int k = 0; k < n; ++k) {
    int p = pivot_reduce<NW>(c, pmax, pidx, n);
    if (p >= n) p = k;
    const float pv = a[p * ld + k];
    const float pinv = (pv != 0.0f && isfinite(pv)) ? 1.0f / pv : 0.0f;
    if (pinv == 0.0f && info == 0) info = k + 1;
    if (c.tid == 0) c.piv()[k] = p;
    __syncthreads();  // every thread has read the pivot: the interchange overwrites it
    // interchange rows k and p; the new row k, normalised, goes to the copy
#pragma unroll 1
    for (int j = c.tid; j < n; j += NT) {
      const float rk = a[k * ld + j], rp = a[p * ld + j];
      if (p != k) a[p * ld + j] = rk;
      pr[j] = (j == k ? 1.0f : rp) * pinv;
    }
    __syncthreads();
    const int cn = k + 1;              // next pivot column
    const int own = cn & 31;           // lane owning column cn in the loops below
    float v = -1.0f;
    int bi = n;
#pragma unroll 1
    for (int i = c.warp; i < n; i += NW) {
      if (i == k) {
#pragma unroll 1
        for (int j = c.lane; j < n; j += 32) a[k * ld + j] = pr[j];
        continue;
      }
      const float fct = a[i * ld + k];
      __syncwarp();
#pragma unroll 1
      for (int j = c.lane; j < n; j += 32) {
        const float nv = (j == k ? 0.0f : a[i * ld + j]) - fct * pr[j];
        a[i * ld + j] = nv;
        if (j == cn && i > k) {
          const float x = fabsf(nv);
          if (x > v || (x == v && i < bi)) { v = x; bi = i; }
        }
      }
    }
    (void)own;
    warp_argmax_store(v, bi, c.lane, pmax, pidx, c.warp);
    __syncthreads();
  }
  // column interchanges in reverse order; each thread owns whole rows
#pragma unroll 1
  for (int i = c.tid; i < n; i += NT)
#pragma unroll 1
    for (int k = n - 1; k >= 0; --k) {
      const int p = c.piv()[k];
      if (p != k) {
        const float t = a[i * ld + k];
        a[i * ld + k] = a[i * ld + p];
        a[i * ld + p] = t;
      }
    }
  __syncthreads();
  return info;
}

// Gauss-Jordan inverse (FP32) with the matrix in registers, by columns: warp w owns
// the columns j = w + NW c (c < CC), lane l the rows l + 32 s (s < RS). Partial
// pivoting by index (the unused row with the largest |a_ik|, lowest row index on
// ties; rows are not moved, the k-th pivot row is recorded instead). The warp owning
// column k publishes it through shared memory (double-buffered); every warp searches the
// pivot in it, broadcasts the pivot row's values of its own columns by warp shuffles and
// updates them. Column k ends up holding column k of the inverse (in-place Gauss-Jordan).
// A pivot row keeps its values and takes its factor 1/a_pk at the end: later steps
// subtract multiples of other rows from it, which commutes with the factor, so it is just
// a row whose multiplier is zero in its own step. The columns rotate through the registers
// once per NW pivots, so that the current one is always c = 0 and no register is selected
// by a run-time index.
// The chain from one pivot to the next (search column k, update column k + 1, publish it)
// is all that the warps wait for: the owner of column k + 1 updates it ahead of its other
// columns and only arrives at the barrier the others wait on; and as every warp searches
// for itself, the chain holds one pass through shared memory and one barrier. (n = 55 on
// four warps, alone on an SM, cycles a pivot: 908 with a search by the owner after all
// updates; 811 with the owner ahead; 692 with the rotation and the deferred factor; the
// search by the owner alone took 540 of these.) The inverse is written as
// inv[Pinv[i]][P[j]] = W[i][j] (P = pivot rows in step order). Requires n <= 32 RS
// and n <= NW CC. src: the matrix by columns, leading dimension ld0. Returns 0 or 1 + k
// for a zero pivot, or kRowRange.
// A row that waits for its factor is larger or smaller than the normalised row by its pivot,
// and so are its multipliers. Pivots within 2^80 of each other and of 1 leave FP32 2^48 on
// either side of that (the integrator's lie between 1 and about 2^60). Beyond, or where no
// pivot is left, the result is kRowRange and nothing is written: gj_invert, whose pivot rows
// are normalised, takes the matrix. (Row sizes 40 decades apart gave infinities. 8,192 solves
// of n = 55 take 520 us without the test of the range, 525 with it, 531 with it on the
// factors in registers; scaling pivot rows once a step finds the range exceeded takes 563 us.)
constexpr int kRowRange = -1;
template <int NW, int RS, int CC, class A>
__device__ int gj_invert_wc(Cta<NW>& c, const A* src, int ld0, float* inv, int n) {
  const int ld = odd_ld(n);
  const int lane = c.lane, wp = c.warp;
  float* pcol = reinterpret_cast<float*>(c.u());  // [2][n] the published columns (u: 6 n doubles)
  float a[RS][CC];
#pragma unroll
  for (int cc = 0; cc < CC; ++cc)
#pragma unroll
    for (int s = 0; s < RS; ++s) {
      const int i = lane + 32 * s, j = wp + NW * cc;
      a[s][cc] = (i < n && j < n) ? to_float(src[(size_t)j * ld0 + i]) : 0.0f;
    }
  unsigned used = 0u;  // bit s: row lane + 32 s is a pivot row already
  float scale[RS];     // 1/a_pk of the pivot rows
#pragma unroll
  for (int s = 0; s < RS; ++s) scale[s] = 0.0f;
  if (wp == 0) {
#pragma unroll
    for (int s = 0; s < RS; ++s)
      if (lane + 32 * s < n) pcol[lane + 32 * s] = a[s][0];
  }
#pragma unroll 1
  for (int i = c.tid; i < n; i += NW * 32) c.perm()[i] = i;  // (a zero pivot leaves entries unset below)
  __syncthreads();
  int info = 0;
#pragma unroll 1
  for (int k = 0; k < n; ++k) {
    const int buf = k & 1, k1 = k + 1;
    const bool own_next = k1 < n && wp == k1 % NW;
    // pivot of column k: argmax of |v| over the unused rows, lowest row on ties, NaN never
    // chosen: the bit pattern of a non-negative float orders like its value, so key =
    // bits + 1 (0: no candidate) goes through one warp max-reduction; every lane forms the
    // reciprocal of its own candidate (one Newton step on the approximate reciprocal)
    float v[RS], best = 0.0f;
    unsigned kmax = 0u;
    int bs = 0;
#pragma unroll
    for (int s = 0; s < RS; ++s) {
      const int i = lane + 32 * s;
      v[s] = pcol[buf * n + min(i, n - 1)];
      const float x = fabsf(v[s]);
      const unsigned key = (i < n && !((used >> s) & 1u) && !isnan(x)) ? __float_as_uint(x) + 1u : 0u;
      best = key > kmax ? v[s] : best;
      bs = key > kmax ? s : bs;
      kmax = max(key, kmax);
    }
    const unsigned km = __reduce_max_sync(FULLMASK, kmax);
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(best));
    r = fmaf(r, fmaf(-best, r, 1.0f), r);
    r = fabsf(r) < 3.4e38f ? r : 0.0f;  // zero pivot (or none): no finite reciprocal
    unsigned win = __ballot_sync(FULLMASK, kmax == km);
    if (RS > 1 && (win & (win - 1u))) {  // a tie: the lowest row, i.e. the lowest slot first
#pragma unroll
      for (int s = RS - 1; s >= 0; --s) {
        const unsigned w = __ballot_sync(FULLMASK, kmax == km && bs == s);
        if (w) win = w;
      }
    }
    const int pl = __ffs(win) - 1;
    const float pinv = __shfl_sync(FULLMASK, r, pl);
    const int ps = RS > 1 ? __shfl_sync(FULLMASK, bs, pl) : 0;
    const int p = pl + 32 * ps;  // (a column of NaN: some row in range, zero pivot)
    if (pinv == 0.0f && info == 0) info = k + 1;
    if (c.tid == 0) {
      c.piv()[k] = p;
      reinterpret_cast<unsigned*>(c.invd())[k] = __float_as_uint(fabsf(pinv));
    }
    float fp[RS];  // multipliers over the pivot: a_ij -= (a_ik / a_pk) a_pj
    bool isp[RS];
#pragma unroll
    for (int s = 0; s < RS; ++s) {
      isp[s] = lane == pl && s == ps;
      fp[s] = isp[s] || lane + 32 * s >= n ? 0.0f : v[s] * pinv;
      used |= isp[s] ? 1u << s : 0u;
      scale[s] = isp[s] ? pinv : scale[s];
    }
    auto pivot_row = [&](const float (&x)[RS]) {  // the pivot row's entry of a column
      float r = x[0];
#pragma unroll
      for (int s = 1; s < RS; ++s) r = ps == s ? x[s] : r;
      return __shfl_sync(FULLMASK, r, pl);
    };
    // barrier 2 + (k1 & 1): column k + 1 is published
    if (own_next) {
      const bool next_group = k1 % NW == 0;  // the columns rotate after this step
      float w[RS];
#pragma unroll
      for (int s = 0; s < RS; ++s) w[s] = next_group ? a[s][CC > 1 ? 1 : 0] : a[s][0];
      const float pr = pivot_row(w);
#pragma unroll
      for (int s = 0; s < RS; ++s)
        if (lane + 32 * s < n) pcol[(k1 & 1) * n + lane + 32 * s] = fmaf(-fp[s], pr, w[s]);
      __syncwarp();
      if (k1 & 1) asm volatile("bar.arrive 3, %0;" ::"n"(NW * 32) : "memory");
      else asm volatile("bar.arrive 2, %0;" ::"n"(NW * 32) : "memory");
    }
    // all broadcasts first (their latencies overlap), then the updates
    float pr[CC];
#pragma unroll
    for (int cc = 0; cc < CC; ++cc) {
      float x[RS];
#pragma unroll
      for (int s = 0; s < RS; ++s) x[s] = a[s][cc];
      pr[cc] = pivot_row(x);
    }
#pragma unroll
    for (int cc = 0; cc < CC; ++cc)
#pragma unroll
      for (int s = 0; s < RS; ++s) a[s][cc] = fmaf(-fp[s], pr[cc], a[s][cc]);
    // column k, as from the unit vector e_p, becomes column k of the inverse
    if (wp == k % NW) {
#pragma unroll
      for (int s = 0; s < RS; ++s) a[s][0] = isp[s] ? 1.0f : -fp[s];
    }
    if (k1 % NW == 0) {
#pragma unroll
      for (int s = 0; s < RS; ++s) {
        const float t = a[s][0];
#pragma unroll
        for (int cc = 0; cc + 1 < CC; ++cc) a[s][cc] = a[s][cc + 1];
        a[s][CC - 1] = t;
      }
    }
    if (k1 < n && !own_next) {
      if (k1 & 1) asm volatile("bar.sync 3, %0;" ::"n"(NW * 32) : "memory");
      else asm volatile("bar.sync 2, %0;" ::"n"(NW * 32) : "memory");
    }
  }
  __syncthreads();
  {
    // smallest and largest of the pivots' factors and 1 (0: no pivot)
    unsigned lo = 0x3f800000u, hi = lo;
#pragma unroll
    for (int s = 0; s < RS; ++s) {
      const unsigned e = lane + 32 * s < n ? reinterpret_cast<unsigned*>(c.invd())[lane + 32 * s] : 0x3f800000u;
      lo = min(lo, e);
      hi = max(hi, e);
    }
    if (__reduce_max_sync(FULLMASK, hi) - __reduce_min_sync(FULLMASK, lo) > 80u << 23) return kRowRange;
  }
  // inverse permutation of the pivot rows, then the scatter into the true inverse
#pragma unroll 1
  for (int k = c.tid; k < n; k += NW * 32) c.perm()[c.piv()[k]] = k;
  __syncthreads();
  const int rot = n / NW % CC;  // rotations made
#pragma unroll
  for (int s = 0; s < RS; ++s) {
    const int i = lane + 32 * s;
    float* row = inv + (i < n ? c.perm()[i] * ld : 0);
#pragma unroll
    for (int cc = 0; cc < CC; ++cc) {
      const int j = wp + NW * (cc + rot < CC ? cc + rot : cc + rot - CC);
      if (i < n && j < n) row[c.piv()[j]] = a[s][cc] * scale[s];
    }
  }
  __syncthreads();
  return info;
}

// One row of the FP32 inverse times xf (16-byte aligned).
__device__ __forceinline__ float inv_row(const float* row, const float* xf, int n) {
  float a0 = 0.0f, a1 = 0.0f, a2 = 0.0f, a3 = 0.0f;
  int j = 0;
#pragma unroll 2
  for (; j + 4 <= n; j += 4) {
    const float4 x = *reinterpret_cast<const float4*>(xf + j);
    a0 = fmaf(row[j], x.x, a0);
    a1 = fmaf(row[j + 1], x.y, a1);
    a2 = fmaf(row[j + 2], x.z, a2);
    a3 = fmaf(row[j + 3], x.w, a3);
  }
  for (; j < n; ++j) a0 = fmaf(row[j], xf[j], a0);
  return (a0 + a1) + (a2 + a3);
}

// Solve M x = b for the FP64 right-hand side b; x written as double. b's entry i was
// written by the thread i (mod the CTA) that reads it here.
// FP64: LU forward/back substitution. Otherwise: x = M32^-1 b with the FP32
// inverse, then `ir` sweeps of r = b - M0 x (about 48 bits, against the assembled matrix
// M0) and x += M32^-1 r. One thread per row of the inverse; a residual row is shared by
// up to three threads (each a range of columns), since a row costs 14 FP32 instructions
// per entry and n rows leave half of the CTA's warps without one.
template <int NW, int PREC>
__device__ void solve(Cta<NW>& c, int n, const double* b, double* x, int ir) {
  constexpr int NT = NW * 32;
  using P = Policy<PREC>;
  if constexpr (!P::IR) {
    __syncthreads();
#pragma unroll 1
    for (int i = c.tid; i < n; i += NT) x[i] = b[c.perm()[i]];
    __syncthreads();
    if (c.warp == Cta<NW>::SW) lu_solve_warp<double>(reinterpret_cast<double*>(c.M()), n, c.invd(), x, c.lane);
    __syncthreads();
  } else {
    using A = typename P::ASM;
    const float* Ai = reinterpret_cast<const float*>(c.M());
    const A* M0 = reinterpret_cast<const A*>(c.M0) + c.i0;
    float* xf = reinterpret_cast<float*>(c.sc());  // scratch vector reused as float
    ff2* xq = reinterpret_cast<ff2*>(c.rr());      // x as float-float pairs (rr is free in the solves)
    ff2* part = reinterpret_cast<ff2*>(c.yn());    // partial residuals (yn and ys are free in the solves)
    const int ld = odd_ld(n), ld0 = c.ld0;
    const int nwr = (n + 31) >> 5;                    // warps that hold a row each lane
    const int np = nwr >= NW ? 1 : min(3, NW / nwr);  // threads per row
    const int cols = (n + np - 1) / np;
    const int q = np > 1 ? c.warp / nwr : 0;          // this thread's range of columns
#pragma unroll 1
    for (int i = c.tid; i < n; i += NT) xf[i] = ff_split(b[i]).hi;
    __syncthreads();
#pragma unroll 1
    for (int sweep = 0;; ++sweep) {
#pragma unroll 1
      for (int i = c.tid; i < n; i += NT) {
        const float acc = inv_row(Ai + i * ld, xf, n);
        if (sweep == 0) {
          x[i] = f32_to_f64(acc);
          xq[i] = {acc, 0.0f};
        } else {
          x[i] += f32_to_f64(acc);
          if (sweep < ir) xq[i] = ff_split(x[i]);
        }
      }
      __syncthreads();
      if (sweep == ir) break;
      // Residual rows r = b - M0 x as a compensated dot product on the FP32 pipe (Ogita,
      // Rump and Oishi's Dot2: exact products of the hi parts, TwoSum of the running sum, the
      // rounding errors and cross terms gathered in a second accumulator): as accurate as
      // a sum in about 48-bit arithmetic, then rounded to FP32 for the correction solve.
      // M0 lies by columns: a warp reads 32 consecutive rows.
      float sh = 0.0f, sl = 0.0f;
#pragma unroll 1
      for (int i = np > 1 ? c.tid - q * nwr * 32 : c.tid; i < n && q < np; i += np > 1 ? n : NT) {
        if (q == 0) {
          const ff2 bi = ff_split(b[i]);
          sh = bi.hi;
          sl = bi.lo;
        }
        const int j1 = min(n, (q + 1) * cols);
#pragma unroll 4
        for (int j = q * cols; j < j1; ++j) {
          const ff2 xj = xq[j];
          float mh, ml = 0.0f;
          if constexpr (std::is_same<A, ff2>::value) {
            const ff2 mj = M0[j * ld0 + i];
            mh = mj.hi;
            ml = mj.lo;
          } else {
            mh = M0[j * ld0 + i];
          }
          const float p = __fmul_rn(mh, xj.hi);
          float pe = fmaf(mh, xj.hi, -p);
          pe = fmaf(mh, xj.lo, pe);
          if constexpr (std::is_same<A, ff2>::value) pe = fmaf(ml, xj.hi, pe);
          const ff2 t = two_sum(sh, -p);
          sh = t.hi;
          sl = __fadd_rn(sl, __fsub_rn(t.lo, pe));
        }
        if (q > 0) part[(q - 1) * n + i] = {sh, sl};
        else if (np == 1) xf[i] = __fadd_rn(sh, sl);
      }
      __syncthreads();
      if (np > 1) {
        if (c.tid < n) {  // its first range's sum is still in sh + sl
          ff_sum r(ff2{sh, sl});
          for (int w = 0; w + 1 < np; ++w) r.add(part[w * n + c.tid]);
          xf[c.tid] = __fadd_rn(r.s, r.c);
        }
        __syncthreads();
      }
    }
  }
}

// Factorisation of the iteration matrix: LU (FP64 form) or the FP32 inverse.
// NMAX: the largest n the caller may pass.
template <int NW, int PREC, int NMAX = 256>
__device__ int factor(Cta<NW>& c, int n, bool pivot = true) {
  if constexpr (!Policy<PREC>::IR) {
    return lu_factor<NW, double>(c, reinterpret_cast<double*>(c.M()), n, pivot);
  } else {
    using A = typename Policy<PREC>::ASM;
    float* inv = reinterpret_cast<float*>(c.M());
    const A* src = reinterpret_cast<const A*>(c.M0) + c.i0;
    int info = kRowRange;
    if constexpr (NW == 4) {
      if (n <= 32) info = gj_invert_wc<4, 1, 8>(c, src, c.ld0, inv, n);
      else if (n <= 56) info = gj_invert_wc<4, 2, 14>(c, src, c.ld0, inv, n);
      else if (n <= 64) info = gj_invert_wc<4, 2, 16>(c, src, c.ld0, inv, n);
    } else if constexpr (NW == 8) {
      if (n <= 64) info = gj_invert_wc<8, 2, 8>(c, src, c.ld0, inv, n);
      else if (n <= 128) info = gj_invert_wc<8, 4, 16>(c, src, c.ld0, inv, n);
    } else if constexpr (NW == 2) {
      if (NMAX <= 32 || n <= 32) info = gj_invert_wc<2, 1, 16>(c, src, c.ld0, inv, n);
      else if (n <= 64) info = gj_invert_wc<2, 2, 32>(c, src, c.ld0, inv, n);
    }
    if (info != kRowRange) return info;
    const int ld = odd_ld(n);
#pragma unroll 1
    for (int j = c.warp; j < n; j += NW)
#pragma unroll 1
      for (int i = c.lane; i < n; i += 32) inv[i * ld + j] = to_float(src[(size_t)j * c.ld0 + i]);
    __syncthreads();
    return gj_invert<NW>(c, inv, n);
  }
}

// Assemble the iteration matrix (fac = 1/(h gamma)) or the Jacobian (JO) in the
// policy's assembly precision.
template <int NW, int PREC, bool JO>
__device__ void build_matrix(const DevMech& m, Cta<NW>& c, const Scal& s, const double* f, double fac) {
  using P = Policy<PREC>;
  if constexpr (!P::IR)
    assemble<NW, double, JO>(m, c, s, f, fac, c.M());
  else if constexpr (std::is_same<typename P::ASM, ff2>::value)
    assemble_ff<NW, JO>(m, c, s, f, fac, reinterpret_cast<ff2*>(c.M0));
  else
    assemble<NW, typename P::ASM, JO, true, true>(m, c, s, f, fac, c.M0);
}

// Iteration matrix (FP64 form) from a forward-difference Jacobian, column by column:
// J_.j = (f(y + d_j e_j) - f(y)) / d_j with d_j = sqrt(eps) max(|y_j|, floor_j)
// (floor 1 K for T, 1e-6 for mass fractions: a smaller floor lets rounding in f
// dominate the columns of trace species); S = sg J + fac I as in assemble.
// Costs n RHS evaluations: the classical alternative to the analytical Jacobian.
template <int NW, bool JO>
__device__ void fd_matrix(const DevMech& m, Cta<NW>& c, double p, const double* y, const double* f0, double fac) {
  constexpr int NT = NW * 32;
  const int n = m.K + 1, ld = odd_ld(n);
  double* A = reinterpret_cast<double*>(c.M());
  for (int j = 0; j < n; ++j) {
    const double d = 1.4901161193847656e-8 * fmax(fabs(y[j]), j == 0 ? 1.0 : 1e-6);
#pragma unroll 1
    for (int i = c.tid; i < n; i += NT) c.ys()[i] = y[i] + (i == j ? d : 0.0);
    __syncthreads();
    eval_rhs<NW, false, false>(m, c, c.ys(), p, c.fv());
    const double id = 1.0 / d;
#pragma unroll 1
    for (int i = c.tid; i < n; i += NT) {
      const double J = (c.fv()[i] - f0[i]) * id;
      A[i * ld + j] = JO ? J : -J + (i == j ? fac : 0.0);
    }
    __syncthreads();
  }
}

// Sum over the CTA of (e_i / (atol + rtol max(|ya_i|, |yb_i|)))^2, finished by fin on warp 0.
template <int NW, int NO, class F>
__device__ void scaled_square_sum(Cta<NW>& c, int n, const double* e, const double* ya, const double* yb, double rtol,
                                  double atol, F fin, double (&out)[NO]) {
  constexpr int NT = NW * 32;
  double part[1] = {0.0};
#pragma unroll 1
  for (int i = c.tid; i < n; i += NT) {
    const double sc = atol + rtol * fmax(fabs(ya[i]), fabs(yb[i]));
    const double r = e[i] * xrcp(sc);
    part[0] += r * r;
  }
  c.reduce(part, warps_for<NW>(n), fin, out);
}

// WRMS norm of e with scale atol + rtol max(|ya|, |yb|).
template <int NW>
__device__ double wrms(Cta<NW>& c, int n, const double* e, const double* ya, const double* yb, double rtol,
                       double atol) {
  double o[1];
  scaled_square_sum(c, n, e, ya, yb, rtol, atol,
                    [&](const double (&t)[1], double (&r)[1]) { r[0] = sqrt(t[0] / n); }, o);
  return o[0];
}

// The error test of a step: the square of the WRMS norm of e, and the step-size factor
// 0.9 err^(-1/q) (q = 4: RODAS4, 3: ROS34PW2; kFacMax for err = 0) by the fixed-point
// logarithm and exponential (about 300 cycles on warp 0, where the FP64 roots and
// division took 2,500).
template <int NW>
__device__ double error_test(Cta<NW>& c, int n, const double* e, const double* ya, const double* yb, double rtol,
                             double atol, double* step_fac, int q) {
  double o[2];
  const double inv_n = xrcp((double)n);
  scaled_square_sum(c, n, e, ya, yb, rtol, atol, [&](const double (&t)[1], double (&r)[2]) {
    const double err2 = t[0] * inv_n;
    r[0] = err2;
    const int hx = __double2hiint(err2);
    if (hx >= 0x00100000 && hx < 0x7ff00000) {
      const long long l = fx_log(err2, 52);
      r[1] = kSafety * fx_exp(q == 4 ? -(l >> 3) : -(l / 6), c.xt());
    } else {
      r[1] = kFacMax;  // zero or subnormal (a non-finite norm's factor is not used)
    }
  }, o);
  *step_fac = o[1];
  return o[0];
}

// Hairer-Wanner starting step (Solving ODEs I, Sec. II.4) in the WRMS norm with
// scale atol + rtol |y0|, exponent 1/q (the method's embedded order + 1), clamped
// to dt; a vanishing derivative selects the whole interval. Uses f0 = f(y0)
// (already in c.f0()) and c.ys(), c.fv().
template <int NW, bool FF = false>
__device__ double starting_step(const DevMech& m, Cta<NW>& c, double p, double dt, double rtol,
                                double atol, int q = 4) {
  constexpr int NT = NW * 32;
  const int n = m.K + 1;
  const double d0 = wrms(c, n, c.y(), c.y(), c.y(), rtol, atol);
  const double d1 = wrms(c, n, c.f0(), c.y(), c.y(), rtol, atol);
  double ha = (d1 > 1e-300) ? 0.01 * d0 / d1 : dt;
  ha = fmin(ha, dt);
#pragma unroll 1
  for (int i = c.tid; i < n; i += NT) c.ys()[i] = c.y()[i] + ha * c.f0()[i];
  __syncthreads();
  eval_rhs<NW, false, FF>(m, c, c.ys(), p, c.fv());
#pragma unroll 1
  for (int i = c.tid; i < n; i += NT) c.rr()[i] = c.fv()[i] - c.f0()[i];
  __syncthreads();
  const double d2 = wrms(c, n, c.rr(), c.y(), c.y(), rtol, atol) / ha;
  const double mx = fmax(d1, d2);
  const double hb = (mx > 1e-300) ? (q == 4 ? pow(0.01 / mx, 0.25) : cbrt(0.01 / mx)) : dt;
  return fmin(fmin(100.0 * ha, hb), dt);
}

// Mass enthalpy and heat capacity at T for mass fractions Y (CTA sums).
template <int NW>
__device__ void h_cp_mass(const DevMech& m, Cta<NW>& c, double T, const double* Y, double& h,
                          double& cp) {
  constexpr int NT = NW * 32;
  const double invT = 1.0 / T;
  double part[2] = {0.0, 0.0};
#pragma unroll 1
  for (int k = c.tid; k < m.K; k += NT) {
    const double* a = m.nasa + 36 * k;
    a += (T < a[34]) ? 0 : 17;
    const double cpr = a[0] + T * (a[1] + T * (a[2] + T * (a[3] + T * a[4])));
    const double hr = a[5] + T * (a[6] + T * (a[7] + T * (a[8] + T * a[9]))) + a[10] * invT;
    part[0] += Y[k] * hr * m.invW[k];
    part[1] += Y[k] * cpr * m.invW[k];
  }
  c.sum(part, warps_for<NW>(m.K));
  h = part[0] * kRc * T;
  cp = part[1] * kRc;
}

// ---------------------------------------------------------------------------
// one cell
// ---------------------------------------------------------------------------
// Per-phase cycle counters (diagnostic; thread 0 reads the clock right after the
// CTA barriers that close each phase): 0 load + starting step, 1 RHS and Jacobian
// data at the step point, 2 iteration-matrix assembly, 3 factorisation, 4 stage RHS,
// 5 stage solves, 6 stage combination + error norm + control, 7 T recovery + store.
#define PHASE(k)                                                              \
  do {                                                                        \
    if (prof) {                                                               \
      const long long now_ = clock64();                                       \
      atomicAdd(args.phase + cur_, (unsigned long long)(now_ - last_));       \
      last_ = now_;                                                           \
      cur_ = (k);                                                             \
    }                                                                         \
  } while (0)

template <int NW, int PREC, int MTH>
__device__ void integrate_cell(const Job& job, int64_t cell, const IntegrateArgs& args, Cta<NW>& c, double* slot) {
  using MT = Meth<MTH>;
  const bool prof = args.phase != nullptr && c.tid == 0;
  long long last_ = prof ? clock64() : 0;
  int cur_ = 0;
  constexpr int NT = NW * 32;
  const DevMech& m = job.m;
  const int K = m.K, n = K + 1;
  const double p = job.p[cell];
  const double dt = args.dt, rtol = args.rtol, atol = args.atol;
  // load (coalesced over species)
  if (c.tid == 0) c.y()[0] = job.T[cell];
#pragma unroll 1
  for (int k = c.tid; k < K; k += NT) c.y()[1 + k] = job.Y[(size_t)cell * K + k];
  c.set_cell(m, p);
  c.set_matrix(K, slot);
  __syncthreads();
  int status = CHEM_CELL_OK;
  {
    double part[1] = {0.0};
#pragma unroll 1
    for (int i = c.tid; i < n; i += NT) part[0] += isfinite(c.y()[i]) ? 0.0 : 1.0;
    c.sum(part, warps_for<NW>(n));
    if (part[0] > 0.0 || !(c.y()[0] > 0.0) || !(p > 0.0)) status = CHEM_CELL_NONFINITE;
  }
  int steps = 0, rejects = 0;
  double h_first = 0.0, h_next = 0.0;
  if (status == CHEM_CELL_OK) {
    double h_target, cp_dummy;
    h_cp_mass(m, c, c.y()[0], c.y() + 1, h_target, cp_dummy);
    // initial step
    double h = -1.0;
    bool guard = false;  // a supplied initial step, checked against f(y0) at the first step
    if (args.use_h0 && job.h0) {
      const double g = job.h0[cell];
      if (isfinite(g) && g > 0.0) {
        h = fmin(g, dt);
        guard = args.h0_guard != 0;
      }
    }
    if (h <= 0.0) {
      eval_rhs<NW, false, Policy<PREC>::IR>(m, c, c.y(), p, c.f0());
      h = starting_step<NW, Policy<PREC>::IR>(m, c, p, dt, rtol, atol, MT::Q);
    }
    double t = 0.0, h_unclipped = h;
    bool after_reject = false;
    while (true) {
      if (dt - t <= 1e-12 * dt) break;
      if (steps >= args.max_steps) { status = CHEM_CELL_MAX_STEPS; break; }
      if (!(h >= kHmin)) { status = CHEM_CELL_H_UNDERFLOW; break; }  // also catches NaN
      h_unclipped = h;
      if (t + h > dt) h = dt - t;
      ++steps;
      // Jacobian and f0 at y; iteration matrix; factorisation
      PHASE(1);
      // A supplied initial step (learned or carried over) is kept inside the starting
      // step heuristic's envelope [h_a, 100 h_a], h_a = 0.01 |y0| / |f(y0)| in the WRMS
      // norm: f(y0) is the first step's first-stage RHS, so the check costs no RHS
      // evaluation, and a prediction far from the states it was trained on cannot cost
      // more than the heuristic's own range of answers.
      auto apply_guard = [&]() {
        if (!guard) return;
        guard = false;
        const double d0 = wrms(c, n, c.y(), c.y(), c.y(), rtol, atol);
        const double d1 = wrms(c, n, c.f0(), c.y(), c.y(), rtol, atol);
        const double ha = d1 > 1e-300 ? 0.01 * d0 / d1 : dt;
        h = fmin(fmin(fmax(h, ha), 100.0 * ha), dt - t);
        h_unclipped = h;
      };
      if (PREC == PREC_FP64 && args.jac_fd) {
        eval_rhs<NW, false, false>(m, c, c.y(), p, c.f0());
        apply_guard();
        PHASE(2);
        fd_matrix<NW, false>(m, c, p, c.y(), c.f0(), 1.0 / (h * MT::gamma(args)));
      } else {
        const Scal s = eval_rhs<NW, true, Policy<PREC>::IR>(m, c, c.y(), p, c.f0());
        apply_guard();
        PHASE(2);
        build_matrix<NW, PREC, false>(m, c, s, c.f0(), 1.0 / (h * MT::gamma(args)));
      }
      PHASE(3);
      const int info = factor<NW, PREC>(c, n, !(PREC == PREC_FP64 && args.no_pivot));
      PHASE(6);
      double err, step_fac = kFacMin;  // err: square of the norm
      if (info != 0) {
        err = NAN;
      } else {
        const double invh = 1.0 / h;
        constexpr int S = MT::S;
#pragma unroll 1
        for (int st = 0; st < S; ++st) {
          if (st > 0) {
            PHASE(6);
            // stage point y_s = y + sum_j a_sj u_j and sum_j c_sj u_j (kept in yn); with
            // half the CTA's threads enough for n entries, each half takes one of the two
            auto stage_sum = [&](int i, double v, auto coef) {
#pragma unroll
              for (int j = 0; j < S - 1; ++j)
                if (j < st) v = fma(coef(j), c.u()[j * n + i], v);
              return v;
            };
            auto ca = [&](int j) { return MT::a(args, st, j); };
            auto cc = [&](int j) { return MT::c(args, st, j); };
            if (n <= NT / 2) {
              const int i = c.tid & (NT / 2 - 1);
              if (i < n) {
                if (c.tid < NT / 2) c.ys()[i] = stage_sum(i, c.y()[i], ca);
                else c.yn()[i] = stage_sum(i, 0.0, cc);
              }
            } else {
#pragma unroll 1
              for (int i = c.tid; i < n; i += NT) {
                c.ys()[i] = stage_sum(i, c.y()[i], ca);
                c.yn()[i] = stage_sum(i, 0.0, cc);
              }
            }
            __syncthreads();
            PHASE(4);
            eval_rhs<NW, false, Policy<PREC>::IR>(m, c, c.ys(), p, c.fv());
          }
          PHASE(6);
          // stage right-hand side f(y_s) + sum_j (c_sj / h) u_j, in place in fv
#pragma unroll 1
          for (int i = c.tid; i < n; i += NT) c.fv()[i] = st > 0 ? fma(invh, c.yn()[i], c.fv()[i]) : c.f0()[i];
          PHASE(5);
          solve<NW, PREC>(c, n, c.fv(), c.u() + st * n, args.ir_sweeps);
        }
        PHASE(6);
#pragma unroll 1
        for (int i = c.tid; i < n; i += NT) {
          double v = c.y()[i], e = 0.0;
#pragma unroll
          for (int j = 0; j < S; ++j) {
            v += MT::m(args, j) * c.u()[j * n + i];
            if (!MT::E_LAST) e += MT::e(args, j) * c.u()[j * n + i];
          }
          c.yn()[i] = v;
          if (!MT::E_LAST) c.rr()[i] = e;
        }
        __syncthreads();
        err = error_test(c, n, MT::E_LAST ? c.u() + (S - 1) * n : c.rr(), c.y(), c.yn(), rtol, atol, &step_fac, MT::Q);
      }
      if (!(err <= 1.0)) {
        ++rejects;
        after_reject = true;
        h *= isfinite(err) ? fmax(step_fac, kFacMin) : kFacMin;
        continue;
      }
      t += h;
#pragma unroll 1
      for (int i = c.tid; i < n; i += NT) c.y()[i] = c.yn()[i];
      __syncthreads();
      if (h_first == 0.0) h_first = h;
      const double fac = fmin(fmax(step_fac, kFacMin), after_reject ? 1.0 : kFacMax);
      after_reject = false;
      h *= fac;
    }
    // step size to carry to the next call: the controller's proposal, or the step
    // before the final clipping to dt when that was longer
    h_next = fmax(h, h_unclipped);
    // temperature from the conserved mass enthalpy (Newton, |dT| < 1e-10 T)
    PHASE(7);
    if (status == CHEM_CELL_OK) {
      double T = c.y()[0];
#pragma unroll 1
      for (int it = 0; it < 50; ++it) {
        double hm, cpm;
        h_cp_mass(m, c, T, c.y() + 1, hm, cpm);
        const double dT = (hm - h_target) / cpm;
        T -= dT;
        if (fabs(dT) < 1e-10 * T) break;
      }
      if (!(T >= kTmin && T <= kTmax)) status = CHEM_CELL_T_RANGE;
      else if (c.tid == 0) c.y()[0] = T;
      __syncthreads();
    }
  }
  // store (the last accepted state for failed cells)
  if (status != CHEM_CELL_NONFINITE) {
    if (c.tid == 0) job.T[cell] = c.y()[0];
#pragma unroll 1
    for (int k = c.tid; k < K; k += NT) job.Y[(size_t)cell * K + k] = c.y()[1 + k];
  }
  PHASE(7);
  if (c.tid == 0) {
    if (job.st.substeps) job.st.substeps[cell] = steps;
    if (job.st.rejects) job.st.rejects[cell] = rejects;
    if (job.st.h_first) job.st.h_first[cell] = h_first;
    if (job.st.status) job.st.status[cell] = status;
    if (job.st.h_last) job.st.h_last[cell] = status == CHEM_CELL_OK ? h_next : 0.0;
    if (job.cost_out) job.cost_out[cell] = (float)steps;
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------
// kernels
// ---------------------------------------------------------------------------
// Launch bounds: 128 registers a thread for four CTAs of 128 threads (FP64 form: its
// shared-memory footprint allows no more up to ~60 species), eight of 64 or two of 256;
// the mixed form with 128 threads takes 168 registers for three CTAs per SM: it is bound by
// the latency of its phases, which spills lengthen (16,384 cells of 54 species: 415 ms;
// four CTAs with 128 registers 487 ms, five with 96 registers 531 ms).
template <int NW, int PREC, int MTH>
__global__ void __launch_bounds__(NW * 32, NW == 4 ? (PREC == PREC_MIXED ? 3 : 4) : NW == 2 ? 8 : 2) k_integrate(const __grid_constant__ IntegrateArgs args) {
  __shared__ long long s_work;
  const bool m0g = PREC == PREC_MIXED && args.m0_scratch != nullptr;
  const Layout L = make_layout(args.smem_K, args.smem_I, PREC, m0g, true);
  Cta<NW> c;
  c.bind(L);
  double* const slot = m0g ? args.m0_scratch + (size_t)blockIdx.x * args.m0_stride : nullptr;
  for (long long it = 0;; ++it) {
    long long w;
    if (args.sched == SCHED_PLAIN) {
      if (it > 0) break;
      w = blockIdx.x;
    } else if (args.sched == SCHED_STATIC) {
      w = blockIdx.x + it * (long long)gridDim.x;
    } else {
      if (threadIdx.x == 0) s_work = atomicAdd(args.queue, 1);
      __syncthreads();
      w = s_work;
      __syncthreads();
    }
    if (w >= args.n_total) break;
    const long long g = args.perm ? args.perm[w] : w;
    int j = 0;
    while (j + 1 < args.n_jobs && g >= args.jobs[j + 1].offset) ++j;
    integrate_cell<NW, PREC, MTH>(args.jobs[j], g - args.jobs[j].offset, args, c, slot);
  }
}

// ---------------------------------------------------------------------------
// launch helper
// ---------------------------------------------------------------------------
template <class KernelT>
static cudaError_t prep(KernelT k, size_t smem) {
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

template <int NW, int PREC, int MTH>
static cudaError_t launch_integrate_m(const IntegrateArgs& a, int grid, cudaStream_t st) {
  const size_t smem = smem_bytes(a.smem_K, a.smem_I, PREC, a.m0_scratch != nullptr);
  cudaError_t e = prep(k_integrate<NW, PREC, MTH>, smem);
  if (e != cudaSuccess) return e;
  k_integrate<NW, PREC, MTH><<<grid, NW * 32, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace chem
