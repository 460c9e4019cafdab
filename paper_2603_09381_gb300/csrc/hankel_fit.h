// Generated by gen_hankel_fit.py (do not edit): polynomials in 60-bit fixed
// point (value 2^60) for P_nu and z Q_nu (nu = 0, 1; Hankel's modulus-phase
// functions) in x = (1/z^2 - vm) ivh on [za, zb), and for sin(pi/4 g) / g and
// cos(pi/4 g) in x = g^2; x31 is x 2^31.  The worst errors are those of the
// integer evaluation against 40-digit values.
#pragma once
#include "fx.cuh"

// [8, 12): degree 9; worst errors P0 3.1e-18, zQ0 4.0e-18, P1 1.7e-18, zQ1 4.6e-18
constexpr double HK_IVH0 = 230.39880192553878, HK_SH0 = 0.4000115199400963;   // 3 + x = v ivh + sh
__device__ __forceinline__ void hankel_fit0(Fx x, int x31, long long& P0, long long& zQ0, long long& P1, long long& zQ1) {
  P0 = (((long long)(__mulhi(__mulhi(__mulhi(__mulhi(__mulhi(-75497, x31) + 369009, x31) + -2011947, x31) + 13271949, x31) + -107727473, x31) + 1153656588) * x31) >> 31) + -36506640537ll;
  P0 = fx_mul(fx(P0), x) + 2091616869006ll;
  P0 = fx_mul(fx(P0), x) + -340132312063272ll;
  P0 = fx_mul(fx(P0), x) + 1152022323267156046ll;
  zQ0 = (((long long)(__mulhi(__mulhi(__mulhi(__mulhi(1846158, x31) + -8360641, x31) + 41507879, x31) + -245893239, x31) + 1746187918) * x31) >> 34) + -3932516902ll;
  zQ0 = fx_mul(fx(zQ0), x) + 98227679808ll;
  zQ0 = fx_mul(fx(zQ0), x) + -3952975497315ll;
  zQ0 = fx_mul(fx(zQ0), x) + 343617037986412ll;
  zQ0 = fx_mul(fx(zQ0), x) + -143193127628803991ll;
  P1 = (((long long)(__mulhi(__mulhi(__mulhi(__mulhi(__mulhi(81744, x31) + -402068, x31) + 2210662, x31) + -14740625, x31) + 121479208, x31) + -1331313680) * x31) >> 31) + 43816075326ll;
  P1 = fx_mul(fx(P1), x) + -2721800739440ll;
  P1 = fx_mul(fx(P1), x) + 571256442247997ll;
  P1 = fx_mul(fx(P1), x) + 1154426003570932652ll;
  zQ1 = (((long long)(__mulhi(__mulhi(__mulhi(__mulhi(-995790, x31) + 4534715, x31) + -22679061, x31) + 135586513, x31) + -975028249) * x31) >> 33) + 4473115236ll;
  zQ1 = fx_mul(fx(zQ1), x) + -115069537238ll;
  zQ1 = fx_mul(fx(zQ1), x) + 4889799343820ll;
  zQ1 = fx_mul(fx(zQ1), x) + -484961023115042ll;
  zQ1 = fx_mul(fx(zQ1), x) + 431049353818652747ll;
}

// [12, 20): degree 8; worst errors P0 1.2e-18, zQ0 1.8e-18, P1 1.5e-18, zQ1 2.5e-18
constexpr double HK_IVH1 = 449.9980875067781, HK_SH1 = 0.8750070312201174;   // 3 + x = v ivh + sh
__device__ __forceinline__ void hankel_fit1(Fx x, int x31, long long& P0, long long& zQ0, long long& P1, long long& zQ1) {
  P0 = (((long long)(__mulhi(__mulhi(__mulhi(__mulhi(148362, x31) + -1096284, x31) + 9852092, x31) + -115574610, x31) + 1887269839) * x31) >> 35) + -6040276433ll;
  P0 = fx_mul(fx(P0), x) + 596430936214ll;
  P0 = fx_mul(fx(P0), x) + -177523159095511ll;
  P0 = fx_mul(fx(P0), x) + 1152541515363450942ll;
  zQ0 = (((long long)(__mulhi(__mulhi(__mulhi(__mulhi(-241604, x31) + 1611835, x31) + -12790680, x31) + 129123574, x31) + -1740746727) * x31) >> 33) + 17230318826ll;
  zQ0 = fx_mul(fx(zQ0), x) + -1169551860577ll;
  zQ0 = fx_mul(fx(zQ0), x) + 182428191255145ll;
  zQ0 = fx_mul(fx(zQ0), x) + -143722073235753236ll;
  P1 = (((long long)(__mulhi(__mulhi(__mulhi(__mulhi(-79992, x31) + 595935, x31) + -5415613, x31) + 64527295, x31) + -1079001320) * x31) >> 34) + 7190808990ll;
  P1 = fx_mul(fx(P1), x) + -771030987004ll;
  P1 = fx_mul(fx(P1), x) + 296861328839925ll;
  P1 = fx_mul(fx(P1), x) + 1153555886449906696ll;
  zQ1 = (((long long)(__mulhi(__mulhi(__mulhi(__mulhi(129749, x31) + -871789, x31) + 6984415, x31) + -71425934, x31) + 981350571) * x31) >> 32) + -20026260650ll;
  zQ1 = fx_mul(fx(zQ1), x) + 1437374082965ll;
  zQ1 = fx_mul(fx(zQ1), x) + -256310060300338ll;
  zQ1 = fx_mul(fx(zQ1), x) + 431794213516225119ll;
}

// [20, 30): degree 6; worst errors P0 1.2e-18, zQ0 1.8e-18, P1 1.6e-18, zQ1 1.9e-18
constexpr double HK_IVH2 = 1439.9925120346174, HK_SH2 = 0.4000115199400963;   // 3 + x = v ivh + sh
__device__ __forceinline__ void hankel_fit2(Fx x, int x31, long long& P0, long long& zQ0, long long& P1, long long& zQ1) {
  P0 = (((long long)(__mulhi(__mulhi(__mulhi(16192, x31) + -498559, x31) + 22346600, x31) + -1643007791) * x31) >> 34) + 60695711973ll;
  P0 = fx_mul(fx(P0), x) + -55975404844096ll;
  P0 = fx_mul(fx(P0), x) + 1152775555224312600ll;
  zQ0 = (((long long)(__mulhi(__mulhi(__mulhi(-22727, x31) + 593247, x31) + -21616667, x31) + 1210658654) * x31) >> 32) + -121318518304ll;
  zQ0 = fx_mul(fx(zQ0), x) + 57997397654245ll;
  zQ0 = fx_mul(fx(zQ0), x) + -143963564508812217ll;
  P1 = (((long long)(__mulhi(__mulhi(__mulhi(-17689, x31) + 553487, x31) + -25421313, x31) + 1947550461) * x31) >> 34) + -78207016989ll;
  P1 = fx_mul(fx(P1), x) + 93413752583658ll;
  P1 = fx_mul(fx(P1), x) + 1153164912315653951ll;
  zQ1 = (((long long)(__mulhi(__mulhi(__mulhi(24669, x31) + -652618, x31) + 24250550, x31) + -1401128031) * x31) >> 32) + 148608334503ll;
  zQ1 = fx_mul(fx(zQ1), x) + -81309881848326ll;
  zQ1 = fx_mul(fx(zQ1), x) + 432133142287821409ll;
}

// [30, 60): degree 6; worst errors P0 8.1e-19, zQ0 1.1e-18, P1 2.1e-18, zQ1 1.7e-18
constexpr double HK_IVH3 = 2399.9920000194666, HK_SH3 = 1.3333368888770372;   // 3 + x = v ivh + sh
__device__ __forceinline__ void hankel_fit3(Fx x, int x31, long long& P0, long long& zQ0, long long& P1, long long& zQ1) {
  P0 = (((long long)(__mulhi(__mulhi(__mulhi(3917, x31) + -182525, x31) + 12705247, x31) + -1484241651) * x31) >> 36) + 22213223316ll;
  P0 = fx_mul(fx(P0), x) + -33702675623519ll;
  P0 = fx_mul(fx(P0), x) + 1152865271681221178ll;
  zQ0 = (((long long)(__mulhi(__mulhi(__mulhi(-5716, x31) + 223813, x31) + -12559773, x31) + 1109262107) * x31) >> 34) + -44751532086ll;
  zQ0 = fx_mul(fx(zQ0), x) + 35034147624808ll;
  zQ0 = fx_mul(fx(zQ0), x) + -144056672997020199ll;
  P1 = (((long long)(__mulhi(__mulhi(__mulhi(-4266, x31) + 202105, x31) + -14421031, x31) + 1756183503) * x31) >> 36) + -28584139020ll;
  P1 = fx_mul(fx(P1), x) + 56199441159698ll;
  P1 = fx_mul(fx(P1), x) + 1153015249798176109ll;
  zQ1 = (((long long)(__mulhi(__mulhi(__mulhi(6186, x31) + -245574, x31) + 14058722, x31) + -1281455197) * x31) >> 34) + 54744148306ll;
  zQ1 = fx_mul(fx(zQ1), x) + -49074453594471ll;
  zQ1 = fx_mul(fx(zQ1), x) + 432263620831174666ll;
}

// [60, inf): degree 5; worst errors P0 3.8e-18, zQ0 1.5e-18, P1 2.3e-18, zQ1 1.6e-18
constexpr double HK_IVH4 = 7199.9784000288, HK_SH4 = 2.000001999998;   // 3 + x = v ivh + sh
__device__ __forceinline__ void hankel_fit4(Fx x, int x31, long long& P0, long long& zQ0, long long& P1, long long& zQ1) {
  P0 = (((long long)(__mulhi(__mulhi(__mulhi(-26, x31) + 5147, x31) + -1758051, x31) + 1244493904) * x31) >> 30) + -11254049595363ll;
  P0 = fx_mul(fx(P0), x) + 1152910248089021218ll;
  zQ0 = (((long long)(__mulhi(__mulhi(32734, x31) + -5272507, x31) + 1355594956) * x31) >> 39) + -5034963891ll;
  zQ0 = fx_mul(fx(zQ0), x) + 11718073379233ll;
  zQ0 = fx_mul(fx(zQ0), x) + -144103464985663420ll;
  P1 = (((long long)(__mulhi(__mulhi(__mulhi(28, x31) + -5835, x31) + 2078197, x31) + -1600338001) * x31) >> 30) + 18758647156994ll;
  P1 = fx_mul(fx(P1), x) + 1152940266419231021ll;
  zQ1 = (((long long)(__mulhi(__mulhi(-35865, x31) + 5894639, x31) + -1564530870) * x31) >> 39) + 6154932962ll;
  zQ1 = fx_mul(fx(zQ1), x) + -16407094677854ll;
  zQ1 = fx_mul(fx(zQ1), x) + 432329151004672616ll;
}

// sin(pi/4 g) / g and cos(pi/4 g), x = g^2 in [0, 1]: degree 7; worst errors 2.7e-18, 1.9e-18
__device__ __forceinline__ void hankel_sincos_fit(Fx x, int x31, long long& s, long long& c) {
  s = (((long long)(__mulhi(__mulhi(-46638, x31) + 8010676, x31) + -1012984170) * x31) >> 30) + 361281429875ll;
  s = fx_mul(fx(s), x) + -42169492358488ll;
  s = fx_mul(fx(s), x) + 2871229454931309ll;
  s = fx_mul(fx(s), x) + -93093237402363180ll;
  s = fx_mul(fx(s), x) + 905502432259640355ll;
  c = (((long long)(__mulhi(-7117105, x31) + 1060735015) * x31) >> 34) + -28374970853ll;
  c = fx_mul(fx(c), x) + 4139980228268ll;
  c = fx_mul(fx(c), x) + -375843056765200ll;
  c = fx_mul(fx(c), x) + 18278814420134577ll;
  c = fx_mul(fx(c), x) + -355589973624321938ll;
  c = fx_mul(fx(c), x) + 1152921504606846976ll;
}
