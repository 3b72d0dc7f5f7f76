// Generated by gen_os.py -- do not edit.
// Straight-line 3c-CP integral code of one shell-pair class: the Obara-Saika VRR
// (App. A, Eq. vrr) with the primitive pairs contracted into scalars first (the
// derivation is in gen_os.py), and the HRR (Eq. hrr), with the operation counts.
#pragma once

namespace snk {

// sigma^i kappa^j of one primitive pair, c<i><j>; a class reads those with i + 2j <= L.
// FP64: times the primitive pair's prefactor, c00 the prefactor itself; elsewhere the
// seeds carry the prefactor and c00 is not read (acc_lead)
template <typename R> struct OsCoef {
  R c00, c10, c20, c30, c40, c01, c11, c21, c02;
};

template <int LA, int LB> struct OsClass;

// class (0,0): 1 operations (1 flops) per primitive pair,
// 0 (0 flops) per contracted pair
template <> struct OsClass<0, 0> {
  static constexpr int L = 0;
  static constexpr int NM = 1;
  static constexpr int NACC = 1;
  static constexpr int NA = 1;
  static constexpr int NB = 1;
  static constexpr int PRIM_FLOPS = 1;
  static constexpr int PAIR_FLOPS = 0;
  static constexpr int VRR_FLOPS = 1;
  static constexpr int HRR_FLOPS = 0;
  template <typename R, typename A>
  __device__ static __forceinline__ void prim(const R* S, const OsCoef<R>& c, A* M) {
    (void)c;
    const R w0_0 = S[0];
    acc_lead(M[0], c.c00, w0_0);
  }
  template <typename R, typename A>
  __device__ static __forceinline__ void build(const A* M, R nABx, R nABy, R nABz, R nACx, R nACy, R nACz,
                                               R* acc) {
    (void)nABx; (void)nABy; (void)nABz; (void)nACx; (void)nACy; (void)nACz;
    const R v000_000 = acc_get(M[0]);
    acc[0] = v000_000;
  }
  template <typename R, typename A>
  __device__ static __forceinline__ void vrr(const R* S, R PAx, R PAy, R PAz, R PCx, R PCy, R PCz,
                                             R k1, R k2, R k3, A* acc) {
    (void)PAx; (void)PAy; (void)PAz; (void)PCx; (void)PCy; (void)PCz; (void)k1; (void)k2; (void)k3;
    const R t000_0 = S[0];
    acc[0] += t000_0;
  }
  template <typename R>
  __device__ static __forceinline__ void hrr(const R* acc, R ABx, R ABy, R ABz, R* xi) {
    (void)ABx; (void)ABy; (void)ABz;
    const R x000_000 = acc[0];
    xi[0] = x000_000;
  }
};

// class (1,0): 3 operations (4 flops) per primitive pair,
// 6 (9 flops) per contracted pair
template <> struct OsClass<1, 0> {
  static constexpr int L = 1;
  static constexpr int NM = 2;
  static constexpr int NACC = 3;
  static constexpr int NA = 3;
  static constexpr int NB = 1;
  static constexpr int PRIM_FLOPS = 4;
  static constexpr int PAIR_FLOPS = 9;
  static constexpr int VRR_FLOPS = 12;
  static constexpr int HRR_FLOPS = 0;
  template <typename R, typename A>
  __device__ static __forceinline__ void prim(const R* S, const OsCoef<R>& c, A* M) {
    (void)c;
    const R w0_0 = S[0];
    const R w0_1 = S[1];
    const R w1_0 = w0_0 - w0_1;
    acc_lead(M[0], c.c00, w0_1);
    acc_mac(M[1], c.c10, w1_0);
  }
  template <typename R, typename A>
  __device__ static __forceinline__ void build(const A* M, R nABx, R nABy, R nABz, R nACx, R nACy, R nACz,
                                               R* acc) {
    (void)nABx; (void)nABy; (void)nABz; (void)nACx; (void)nACy; (void)nACz;
    const R v000_001 = acc_get(M[0]);
    const R v000_100 = acc_get(M[1]);
    const R v100_000 = dot2(nABx, v000_100, nACx, v000_001);
    const R v010_000 = dot2(nABy, v000_100, nACy, v000_001);
    const R v001_000 = dot2(nABz, v000_100, nACz, v000_001);
    acc[0] = v100_000;
    acc[1] = v010_000;
    acc[2] = v001_000;
  }
  template <typename R, typename A>
  __device__ static __forceinline__ void vrr(const R* S, R PAx, R PAy, R PAz, R PCx, R PCy, R PCz,
                                             R k1, R k2, R k3, A* acc) {
    (void)PAx; (void)PAy; (void)PAz; (void)PCx; (void)PCy; (void)PCz; (void)k1; (void)k2; (void)k3;
    const R t000_0 = S[0];
    const R t000_1 = S[1];
    const R t100_0 = fma(PAx, t000_0, -PCx * t000_1);
    const R t010_0 = fma(PAy, t000_0, -PCy * t000_1);
    const R t001_0 = fma(PAz, t000_0, -PCz * t000_1);
    acc[0] += t100_0;
    acc[1] += t010_0;
    acc[2] += t001_0;
  }
  template <typename R>
  __device__ static __forceinline__ void hrr(const R* acc, R ABx, R ABy, R ABz, R* xi) {
    (void)ABx; (void)ABy; (void)ABz;
    const R x001_000 = acc[2];
    const R x010_000 = acc[1];
    const R x100_000 = acc[0];
    xi[0] = x100_000;
    xi[1] = x010_000;
    xi[2] = x001_000;
  }
};

// class (1,1): 9 operations (13 flops) per primitive pair,
// 42 (66 flops) per contracted pair
template <> struct OsClass<1, 1> {
  static constexpr int L = 2;
  static constexpr int NM = 6;
  static constexpr int NACC = 9;
  static constexpr int NA = 3;
  static constexpr int NB = 3;
  static constexpr int PRIM_FLOPS = 13;
  static constexpr int PAIR_FLOPS = 66;
  static constexpr int VRR_FLOPS = 54;
  static constexpr int HRR_FLOPS = 18;
  template <typename R, typename A>
  __device__ static __forceinline__ void prim(const R* S, const OsCoef<R>& c, A* M) {
    (void)c;
    const R w0_0 = S[0];
    const R w0_1 = S[1];
    const R w0_2 = S[2];
    const R w1_0 = w0_0 - w0_1;
    const R w1_1 = w0_1 - w0_2;
    const R w2_0 = w1_0 - w1_1;
    acc_lead(M[0], c.c00, w0_1);
    acc_mac(M[1], c.c10, w1_0);
    acc_lead(M[2], c.c00, w0_2);
    acc_mac(M[3], c.c10, w1_1);
    acc_mac(M[4], c.c20, w2_0);
    acc_mac(M[5], c.c01, w1_0);
  }
  template <typename R, typename A>
  __device__ static __forceinline__ void build(const A* M, R nABx, R nABy, R nABz, R nACx, R nACy, R nACz,
                                               R* acc) {
    (void)nABx; (void)nABy; (void)nABz; (void)nACx; (void)nACy; (void)nACz;
    const R v000_001 = acc_get(M[0]);
    const R v000_002 = acc_get(M[2]);
    const R v000_010 = acc_get(M[5]);
    const R v000_100 = acc_get(M[1]);
    const R v000_101 = acc_get(M[3]);
    const R v000_200 = acc_get(M[4]);
    const R v100_000 = dot2(nABx, v000_100, nACx, v000_001);
    const R v100_001 = dot2(nABx, v000_101, nACx, v000_002);
    const R v100_100 = dot2(nABx, v000_200, nACx, v000_101);
    const R v010_000 = dot2(nABy, v000_100, nACy, v000_001);
    const R v010_001 = dot2(nABy, v000_101, nACy, v000_002);
    const R v010_100 = dot2(nABy, v000_200, nACy, v000_101);
    const R v001_000 = dot2(nABz, v000_100, nACz, v000_001);
    const R v001_001 = dot2(nABz, v000_101, nACz, v000_002);
    const R v001_100 = dot2(nABz, v000_200, nACz, v000_101);
    const R v200_000 = dot2_add<1>(nABx, v100_100, nACx, v100_001, v000_010);
    const R v110_000 = dot2(nABy, v100_100, nACy, v100_001);
    const R v101_000 = dot2(nABz, v100_100, nACz, v100_001);
    const R v020_000 = dot2_add<1>(nABy, v010_100, nACy, v010_001, v000_010);
    const R v011_000 = dot2(nABy, v001_100, nACy, v001_001);
    const R v002_000 = dot2_add<1>(nABz, v001_100, nACz, v001_001, v000_010);
    acc[0] = v100_000;
    acc[1] = v010_000;
    acc[2] = v001_000;
    acc[3] = v200_000;
    acc[4] = v110_000;
    acc[5] = v101_000;
    acc[6] = v020_000;
    acc[7] = v011_000;
    acc[8] = v002_000;
  }
  template <typename R, typename A>
  __device__ static __forceinline__ void vrr(const R* S, R PAx, R PAy, R PAz, R PCx, R PCy, R PCz,
                                             R k1, R k2, R k3, A* acc) {
    (void)PAx; (void)PAy; (void)PAz; (void)PCx; (void)PCy; (void)PCz; (void)k1; (void)k2; (void)k3;
    const R t000_0 = S[0];
    const R t000_1 = S[1];
    const R t000_2 = S[2];
    const R t100_0 = fma(PAx, t000_0, -PCx * t000_1);
    const R t100_1 = fma(PAx, t000_1, -PCx * t000_2);
    const R t010_0 = fma(PAy, t000_0, -PCy * t000_1);
    const R t010_1 = fma(PAy, t000_1, -PCy * t000_2);
    const R t001_0 = fma(PAz, t000_0, -PCz * t000_1);
    const R t001_1 = fma(PAz, t000_1, -PCz * t000_2);
    const R t200_0 = fma(k1, t000_0 - t000_1, fma(PAx, t100_0, -PCx * t100_1));
    const R t110_0 = fma(PAx, t010_0, -PCx * t010_1);
    const R t101_0 = fma(PAx, t001_0, -PCx * t001_1);
    const R t020_0 = fma(k1, t000_0 - t000_1, fma(PAy, t010_0, -PCy * t010_1));
    const R t011_0 = fma(PAy, t001_0, -PCy * t001_1);
    const R t002_0 = fma(k1, t000_0 - t000_1, fma(PAz, t001_0, -PCz * t001_1));
    acc[0] += t100_0;
    acc[1] += t010_0;
    acc[2] += t001_0;
    acc[3] += t200_0;
    acc[4] += t110_0;
    acc[5] += t101_0;
    acc[6] += t020_0;
    acc[7] += t011_0;
    acc[8] += t002_0;
  }
  template <typename R>
  __device__ static __forceinline__ void hrr(const R* acc, R ABx, R ABy, R ABz, R* xi) {
    (void)ABx; (void)ABy; (void)ABz;
    const R x002_000 = acc[8];
    const R x011_000 = acc[7];
    const R x020_000 = acc[6];
    const R x101_000 = acc[5];
    const R x110_000 = acc[4];
    const R x200_000 = acc[3];
    const R x001_000 = acc[2];
    const R x010_000 = acc[1];
    const R x100_000 = acc[0];
    const R x001_001 = fma(ABz, x001_000, x002_000);
    const R x001_010 = fma(ABy, x001_000, x011_000);
    const R x001_100 = fma(ABx, x001_000, x101_000);
    const R x010_001 = fma(ABz, x010_000, x011_000);
    const R x010_010 = fma(ABy, x010_000, x020_000);
    const R x010_100 = fma(ABx, x010_000, x110_000);
    const R x100_001 = fma(ABz, x100_000, x101_000);
    const R x100_010 = fma(ABy, x100_000, x110_000);
    const R x100_100 = fma(ABx, x100_000, x200_000);
    xi[0] = x100_100;
    xi[1] = x100_010;
    xi[2] = x100_001;
    xi[3] = x010_100;
    xi[4] = x010_010;
    xi[5] = x010_001;
    xi[6] = x001_100;
    xi[7] = x001_010;
    xi[8] = x001_001;
  }
};

// class (2,0): 7 operations (10 flops) per primitive pair,
// 27 (39 flops) per contracted pair
template <> struct OsClass<2, 0> {
  static constexpr int L = 2;
  static constexpr int NM = 4;
  static constexpr int NACC = 6;
  static constexpr int NA = 6;
  static constexpr int NB = 1;
  static constexpr int PRIM_FLOPS = 10;
  static constexpr int PAIR_FLOPS = 39;
  static constexpr int VRR_FLOPS = 51;
  static constexpr int HRR_FLOPS = 0;
  template <typename R, typename A>
  __device__ static __forceinline__ void prim(const R* S, const OsCoef<R>& c, A* M) {
    (void)c;
    const R w0_0 = S[0];
    const R w0_1 = S[1];
    const R w0_2 = S[2];
    const R w1_0 = w0_0 - w0_1;
    const R w1_1 = w0_1 - w0_2;
    const R w2_0 = w1_0 - w1_1;
    acc_lead(M[0], c.c00, w0_2);
    acc_mac(M[1], c.c10, w1_1);
    acc_mac(M[2], c.c20, w2_0);
    acc_mac(M[3], c.c01, w1_0);
  }
  template <typename R, typename A>
  __device__ static __forceinline__ void build(const A* M, R nABx, R nABy, R nABz, R nACx, R nACy, R nACz,
                                               R* acc) {
    (void)nABx; (void)nABy; (void)nABz; (void)nACx; (void)nACy; (void)nACz;
    const R v000_002 = acc_get(M[0]);
    const R v000_010 = acc_get(M[3]);
    const R v000_101 = acc_get(M[1]);
    const R v000_200 = acc_get(M[2]);
    const R v100_001 = dot2(nABx, v000_101, nACx, v000_002);
    const R v100_100 = dot2(nABx, v000_200, nACx, v000_101);
    const R v010_001 = dot2(nABy, v000_101, nACy, v000_002);
    const R v010_100 = dot2(nABy, v000_200, nACy, v000_101);
    const R v001_001 = dot2(nABz, v000_101, nACz, v000_002);
    const R v001_100 = dot2(nABz, v000_200, nACz, v000_101);
    const R v200_000 = dot2_add<1>(nABx, v100_100, nACx, v100_001, v000_010);
    const R v110_000 = dot2(nABy, v100_100, nACy, v100_001);
    const R v101_000 = dot2(nABz, v100_100, nACz, v100_001);
    const R v020_000 = dot2_add<1>(nABy, v010_100, nACy, v010_001, v000_010);
    const R v011_000 = dot2(nABy, v001_100, nACy, v001_001);
    const R v002_000 = dot2_add<1>(nABz, v001_100, nACz, v001_001, v000_010);
    acc[0] = v200_000;
    acc[1] = v110_000;
    acc[2] = v101_000;
    acc[3] = v020_000;
    acc[4] = v011_000;
    acc[5] = v002_000;
  }
  template <typename R, typename A>
  __device__ static __forceinline__ void vrr(const R* S, R PAx, R PAy, R PAz, R PCx, R PCy, R PCz,
                                             R k1, R k2, R k3, A* acc) {
    (void)PAx; (void)PAy; (void)PAz; (void)PCx; (void)PCy; (void)PCz; (void)k1; (void)k2; (void)k3;
    const R t000_0 = S[0];
    const R t000_1 = S[1];
    const R t000_2 = S[2];
    const R t100_0 = fma(PAx, t000_0, -PCx * t000_1);
    const R t100_1 = fma(PAx, t000_1, -PCx * t000_2);
    const R t010_0 = fma(PAy, t000_0, -PCy * t000_1);
    const R t010_1 = fma(PAy, t000_1, -PCy * t000_2);
    const R t001_0 = fma(PAz, t000_0, -PCz * t000_1);
    const R t001_1 = fma(PAz, t000_1, -PCz * t000_2);
    const R t200_0 = fma(k1, t000_0 - t000_1, fma(PAx, t100_0, -PCx * t100_1));
    const R t110_0 = fma(PAx, t010_0, -PCx * t010_1);
    const R t101_0 = fma(PAx, t001_0, -PCx * t001_1);
    const R t020_0 = fma(k1, t000_0 - t000_1, fma(PAy, t010_0, -PCy * t010_1));
    const R t011_0 = fma(PAy, t001_0, -PCy * t001_1);
    const R t002_0 = fma(k1, t000_0 - t000_1, fma(PAz, t001_0, -PCz * t001_1));
    acc[0] += t200_0;
    acc[1] += t110_0;
    acc[2] += t101_0;
    acc[3] += t020_0;
    acc[4] += t011_0;
    acc[5] += t002_0;
  }
  template <typename R>
  __device__ static __forceinline__ void hrr(const R* acc, R ABx, R ABy, R ABz, R* xi) {
    (void)ABx; (void)ABy; (void)ABz;
    const R x002_000 = acc[5];
    const R x011_000 = acc[4];
    const R x020_000 = acc[3];
    const R x101_000 = acc[2];
    const R x110_000 = acc[1];
    const R x200_000 = acc[0];
    xi[0] = x200_000;
    xi[1] = x110_000;
    xi[2] = x101_000;
    xi[3] = x020_000;
    xi[4] = x011_000;
    xi[5] = x002_000;
  }
};

// class (2,1): 16 operations (24 flops) per primitive pair,
// 114 (177 flops) per contracted pair
template <> struct OsClass<2, 1> {
  static constexpr int L = 3;
  static constexpr int NM = 10;
  static constexpr int NACC = 16;
  static constexpr int NA = 6;
  static constexpr int NB = 3;
  static constexpr int PRIM_FLOPS = 24;
  static constexpr int PAIR_FLOPS = 177;
  static constexpr int VRR_FLOPS = 130;
  static constexpr int HRR_FLOPS = 36;
  template <typename R, typename A>
  __device__ static __forceinline__ void prim(const R* S, const OsCoef<R>& c, A* M) {
    (void)c;
    const R w0_0 = S[0];
    const R w0_1 = S[1];
    const R w0_2 = S[2];
    const R w0_3 = S[3];
    const R w1_0 = w0_0 - w0_1;
    const R w1_1 = w0_1 - w0_2;
    const R w1_2 = w0_2 - w0_3;
    const R w2_0 = w1_0 - w1_1;
    const R w2_1 = w1_1 - w1_2;
    const R w3_0 = w2_0 - w2_1;
    acc_lead(M[0], c.c00, w0_2);
    acc_mac(M[1], c.c10, w1_1);
    acc_mac(M[2], c.c20, w2_0);
    acc_mac(M[3], c.c01, w1_0);
    acc_lead(M[4], c.c00, w0_3);
    acc_mac(M[5], c.c10, w1_2);
    acc_mac(M[6], c.c20, w2_1);
    acc_mac(M[7], c.c30, w3_0);
    acc_mac(M[8], c.c01, w1_1);
    acc_mac(M[9], c.c11, w2_0);
  }
  template <typename R, typename A>
  __device__ static __forceinline__ void build(const A* M, R nABx, R nABy, R nABz, R nACx, R nACy, R nACz,
                                               R* acc) {
    (void)nABx; (void)nABy; (void)nABz; (void)nACx; (void)nACy; (void)nACz;
    const R v000_002 = acc_get(M[0]);
    const R v000_003 = acc_get(M[4]);
    const R v000_010 = acc_get(M[3]);
    const R v000_011 = acc_get(M[8]);
    const R v000_101 = acc_get(M[1]);
    const R v000_102 = acc_get(M[5]);
    const R v000_110 = acc_get(M[9]);
    const R v000_200 = acc_get(M[2]);
    const R v000_201 = acc_get(M[6]);
    const R v000_300 = acc_get(M[7]);
    const R v100_001 = dot2(nABx, v000_101, nACx, v000_002);
    const R v100_002 = dot2(nABx, v000_102, nACx, v000_003);
    const R v100_010 = dot2(nABx, v000_110, nACx, v000_011);
    const R v100_100 = dot2(nABx, v000_200, nACx, v000_101);
    const R v100_101 = dot2(nABx, v000_201, nACx, v000_102);
    const R v100_200 = dot2(nABx, v000_300, nACx, v000_201);
    const R v010_001 = dot2(nABy, v000_101, nACy, v000_002);
    const R v010_002 = dot2(nABy, v000_102, nACy, v000_003);
    const R v010_010 = dot2(nABy, v000_110, nACy, v000_011);
    const R v010_100 = dot2(nABy, v000_200, nACy, v000_101);
    const R v010_101 = dot2(nABy, v000_201, nACy, v000_102);
    const R v010_200 = dot2(nABy, v000_300, nACy, v000_201);
    const R v001_001 = dot2(nABz, v000_101, nACz, v000_002);
    const R v001_002 = dot2(nABz, v000_102, nACz, v000_003);
    const R v001_010 = dot2(nABz, v000_110, nACz, v000_011);
    const R v001_100 = dot2(nABz, v000_200, nACz, v000_101);
    const R v001_101 = dot2(nABz, v000_201, nACz, v000_102);
    const R v001_200 = dot2(nABz, v000_300, nACz, v000_201);
    const R v200_000 = dot2_add<1>(nABx, v100_100, nACx, v100_001, v000_010);
    const R v200_001 = dot2_add<1>(nABx, v100_101, nACx, v100_002, v000_011);
    const R v200_100 = dot2_add<1>(nABx, v100_200, nACx, v100_101, v000_110);
    const R v110_000 = dot2(nABx, v010_100, nACx, v010_001);
    const R v110_001 = dot2(nABx, v010_101, nACx, v010_002);
    const R v110_100 = dot2(nABx, v010_200, nACx, v010_101);
    const R v101_000 = dot2(nABz, v100_100, nACz, v100_001);
    const R v020_000 = dot2_add<1>(nABy, v010_100, nACy, v010_001, v000_010);
    const R v020_001 = dot2_add<1>(nABy, v010_101, nACy, v010_002, v000_011);
    const R v020_100 = dot2_add<1>(nABy, v010_200, nACy, v010_101, v000_110);
    const R v011_000 = dot2(nABz, v010_100, nACz, v010_001);
    const R v002_000 = dot2_add<1>(nABz, v001_100, nACz, v001_001, v000_010);
    const R v002_001 = dot2_add<1>(nABz, v001_101, nACz, v001_002, v000_011);
    const R v002_100 = dot2_add<1>(nABz, v001_200, nACz, v001_101, v000_110);
    const R v300_000 = dot2_add<2>(nABx, v200_100, nACx, v200_001, v100_010);
    const R v210_000 = dot2(nABy, v200_100, nACy, v200_001);
    const R v201_000 = dot2(nABz, v200_100, nACz, v200_001);
    const R v120_000 = dot2(nABx, v020_100, nACx, v020_001);
    const R v111_000 = dot2(nABz, v110_100, nACz, v110_001);
    const R v102_000 = dot2(nABx, v002_100, nACx, v002_001);
    const R v030_000 = dot2_add<2>(nABy, v020_100, nACy, v020_001, v010_010);
    const R v021_000 = dot2(nABz, v020_100, nACz, v020_001);
    const R v012_000 = dot2(nABy, v002_100, nACy, v002_001);
    const R v003_000 = dot2_add<2>(nABz, v002_100, nACz, v002_001, v001_010);
    acc[0] = v200_000;
    acc[1] = v110_000;
    acc[2] = v101_000;
    acc[3] = v020_000;
    acc[4] = v011_000;
    acc[5] = v002_000;
    acc[6] = v300_000;
    acc[7] = v210_000;
    acc[8] = v201_000;
    acc[9] = v120_000;
    acc[10] = v111_000;
    acc[11] = v102_000;
    acc[12] = v030_000;
    acc[13] = v021_000;
    acc[14] = v012_000;
    acc[15] = v003_000;
  }
  template <typename R, typename A>
  __device__ static __forceinline__ void vrr(const R* S, R PAx, R PAy, R PAz, R PCx, R PCy, R PCz,
                                             R k1, R k2, R k3, A* acc) {
    (void)PAx; (void)PAy; (void)PAz; (void)PCx; (void)PCy; (void)PCz; (void)k1; (void)k2; (void)k3;
    const R t000_0 = S[0];
    const R t000_1 = S[1];
    const R t000_2 = S[2];
    const R t000_3 = S[3];
    const R t100_0 = fma(PAx, t000_0, -PCx * t000_1);
    const R t100_1 = fma(PAx, t000_1, -PCx * t000_2);
    const R t100_2 = fma(PAx, t000_2, -PCx * t000_3);
    const R t010_0 = fma(PAy, t000_0, -PCy * t000_1);
    const R t010_1 = fma(PAy, t000_1, -PCy * t000_2);
    const R t010_2 = fma(PAy, t000_2, -PCy * t000_3);
    const R t001_0 = fma(PAz, t000_0, -PCz * t000_1);
    const R t001_1 = fma(PAz, t000_1, -PCz * t000_2);
    const R t001_2 = fma(PAz, t000_2, -PCz * t000_3);
    const R t200_0 = fma(k1, t000_0 - t000_1, fma(PAx, t100_0, -PCx * t100_1));
    const R t200_1 = fma(k1, t000_1 - t000_2, fma(PAx, t100_1, -PCx * t100_2));
    const R t110_0 = fma(PAx, t010_0, -PCx * t010_1);
    const R t101_0 = fma(PAx, t001_0, -PCx * t001_1);
    const R t020_0 = fma(k1, t000_0 - t000_1, fma(PAy, t010_0, -PCy * t010_1));
    const R t020_1 = fma(k1, t000_1 - t000_2, fma(PAy, t010_1, -PCy * t010_2));
    const R t011_0 = fma(PAy, t001_0, -PCy * t001_1);
    const R t011_1 = fma(PAy, t001_1, -PCy * t001_2);
    const R t002_0 = fma(k1, t000_0 - t000_1, fma(PAz, t001_0, -PCz * t001_1));
    const R t002_1 = fma(k1, t000_1 - t000_2, fma(PAz, t001_1, -PCz * t001_2));
    const R t300_0 = fma(k2, t100_0 - t100_1, fma(PAx, t200_0, -PCx * t200_1));
    const R t210_0 = fma(PAy, t200_0, -PCy * t200_1);
    const R t201_0 = fma(PAz, t200_0, -PCz * t200_1);
    const R t120_0 = fma(PAx, t020_0, -PCx * t020_1);
    const R t111_0 = fma(PAx, t011_0, -PCx * t011_1);
    const R t102_0 = fma(PAx, t002_0, -PCx * t002_1);
    const R t030_0 = fma(k2, t010_0 - t010_1, fma(PAy, t020_0, -PCy * t020_1));
    const R t021_0 = fma(PAz, t020_0, -PCz * t020_1);
    const R t012_0 = fma(PAy, t002_0, -PCy * t002_1);
    const R t003_0 = fma(k2, t001_0 - t001_1, fma(PAz, t002_0, -PCz * t002_1));
    acc[0] += t200_0;
    acc[1] += t110_0;
    acc[2] += t101_0;
    acc[3] += t020_0;
    acc[4] += t011_0;
    acc[5] += t002_0;
    acc[6] += t300_0;
    acc[7] += t210_0;
    acc[8] += t201_0;
    acc[9] += t120_0;
    acc[10] += t111_0;
    acc[11] += t102_0;
    acc[12] += t030_0;
    acc[13] += t021_0;
    acc[14] += t012_0;
    acc[15] += t003_0;
  }
  template <typename R>
  __device__ static __forceinline__ void hrr(const R* acc, R ABx, R ABy, R ABz, R* xi) {
    (void)ABx; (void)ABy; (void)ABz;
    const R x003_000 = acc[15];
    const R x012_000 = acc[14];
    const R x021_000 = acc[13];
    const R x030_000 = acc[12];
    const R x102_000 = acc[11];
    const R x111_000 = acc[10];
    const R x120_000 = acc[9];
    const R x201_000 = acc[8];
    const R x210_000 = acc[7];
    const R x300_000 = acc[6];
    const R x002_000 = acc[5];
    const R x011_000 = acc[4];
    const R x020_000 = acc[3];
    const R x101_000 = acc[2];
    const R x110_000 = acc[1];
    const R x200_000 = acc[0];
    const R x002_001 = fma(ABz, x002_000, x003_000);
    const R x002_010 = fma(ABy, x002_000, x012_000);
    const R x002_100 = fma(ABx, x002_000, x102_000);
    const R x011_001 = fma(ABz, x011_000, x012_000);
    const R x011_010 = fma(ABy, x011_000, x021_000);
    const R x011_100 = fma(ABx, x011_000, x111_000);
    const R x020_001 = fma(ABz, x020_000, x021_000);
    const R x020_010 = fma(ABy, x020_000, x030_000);
    const R x020_100 = fma(ABx, x020_000, x120_000);
    const R x101_001 = fma(ABz, x101_000, x102_000);
    const R x101_010 = fma(ABy, x101_000, x111_000);
    const R x101_100 = fma(ABx, x101_000, x201_000);
    const R x110_001 = fma(ABz, x110_000, x111_000);
    const R x110_010 = fma(ABy, x110_000, x120_000);
    const R x110_100 = fma(ABx, x110_000, x210_000);
    const R x200_001 = fma(ABz, x200_000, x201_000);
    const R x200_010 = fma(ABy, x200_000, x210_000);
    const R x200_100 = fma(ABx, x200_000, x300_000);
    xi[0] = x200_100;
    xi[1] = x200_010;
    xi[2] = x200_001;
    xi[3] = x110_100;
    xi[4] = x110_010;
    xi[5] = x110_001;
    xi[6] = x101_100;
    xi[7] = x101_010;
    xi[8] = x101_001;
    xi[9] = x020_100;
    xi[10] = x020_010;
    xi[11] = x020_001;
    xi[12] = x011_100;
    xi[13] = x011_010;
    xi[14] = x011_001;
    xi[15] = x002_100;
    xi[16] = x002_010;
    xi[17] = x002_001;
  }
};

// class (2,2): 29 operations (45 flops) per primitive pair,
// 313 (503 flops) per contracted pair
template <> struct OsClass<2, 2> {
  static constexpr int L = 4;
  static constexpr int NM = 19;
  static constexpr int NACC = 31;
  static constexpr int NA = 6;
  static constexpr int NB = 6;
  static constexpr int PRIM_FLOPS = 45;
  static constexpr int PAIR_FLOPS = 503;
  static constexpr int VRR_FLOPS = 268;
  static constexpr int HRR_FLOPS = 158;
  template <typename R, typename A>
  __device__ static __forceinline__ void prim(const R* S, const OsCoef<R>& c, A* M) {
    (void)c;
    const R w0_0 = S[0];
    const R w0_1 = S[1];
    const R w0_2 = S[2];
    const R w0_3 = S[3];
    const R w0_4 = S[4];
    const R w1_0 = w0_0 - w0_1;
    const R w1_1 = w0_1 - w0_2;
    const R w1_2 = w0_2 - w0_3;
    const R w1_3 = w0_3 - w0_4;
    const R w2_0 = w1_0 - w1_1;
    const R w2_1 = w1_1 - w1_2;
    const R w2_2 = w1_2 - w1_3;
    const R w3_0 = w2_0 - w2_1;
    const R w3_1 = w2_1 - w2_2;
    const R w4_0 = w3_0 - w3_1;
    acc_lead(M[0], c.c00, w0_2);
    acc_mac(M[1], c.c10, w1_1);
    acc_mac(M[2], c.c20, w2_0);
    acc_mac(M[3], c.c01, w1_0);
    acc_lead(M[4], c.c00, w0_3);
    acc_mac(M[5], c.c10, w1_2);
    acc_mac(M[6], c.c20, w2_1);
    acc_mac(M[7], c.c30, w3_0);
    acc_mac(M[8], c.c01, w1_1);
    acc_mac(M[9], c.c11, w2_0);
    acc_lead(M[10], c.c00, w0_4);
    acc_mac(M[11], c.c10, w1_3);
    acc_mac(M[12], c.c20, w2_2);
    acc_mac(M[13], c.c30, w3_1);
    acc_mac(M[14], c.c40, w4_0);
    acc_mac(M[15], c.c01, w1_2);
    acc_mac(M[16], c.c11, w2_1);
    acc_mac(M[17], c.c21, w3_0);
    acc_mac(M[18], c.c02, w2_0);
  }
  template <typename R, typename A>
  __device__ static __forceinline__ void build(const A* M, R nABx, R nABy, R nABz, R nACx, R nACy, R nACz,
                                               R* acc) {
    (void)nABx; (void)nABy; (void)nABz; (void)nACx; (void)nACy; (void)nACz;
    const R v000_002 = acc_get(M[0]);
    const R v000_003 = acc_get(M[4]);
    const R v000_004 = acc_get(M[10]);
    const R v000_010 = acc_get(M[3]);
    const R v000_011 = acc_get(M[8]);
    const R v000_012 = acc_get(M[15]);
    const R v000_020 = acc_get(M[18]);
    const R v000_101 = acc_get(M[1]);
    const R v000_102 = acc_get(M[5]);
    const R v000_103 = acc_get(M[11]);
    const R v000_110 = acc_get(M[9]);
    const R v000_111 = acc_get(M[16]);
    const R v000_200 = acc_get(M[2]);
    const R v000_201 = acc_get(M[6]);
    const R v000_202 = acc_get(M[12]);
    const R v000_210 = acc_get(M[17]);
    const R v000_300 = acc_get(M[7]);
    const R v000_301 = acc_get(M[13]);
    const R v000_400 = acc_get(M[14]);
    const R v100_001 = dot2(nABx, v000_101, nACx, v000_002);
    const R v100_002 = dot2(nABx, v000_102, nACx, v000_003);
    const R v100_003 = dot2(nABx, v000_103, nACx, v000_004);
    const R v100_010 = dot2(nABx, v000_110, nACx, v000_011);
    const R v100_011 = dot2(nABx, v000_111, nACx, v000_012);
    const R v100_100 = dot2(nABx, v000_200, nACx, v000_101);
    const R v100_101 = dot2(nABx, v000_201, nACx, v000_102);
    const R v100_102 = dot2(nABx, v000_202, nACx, v000_103);
    const R v100_110 = dot2(nABx, v000_210, nACx, v000_111);
    const R v100_200 = dot2(nABx, v000_300, nACx, v000_201);
    const R v100_201 = dot2(nABx, v000_301, nACx, v000_202);
    const R v100_300 = dot2(nABx, v000_400, nACx, v000_301);
    const R v010_001 = dot2(nABy, v000_101, nACy, v000_002);
    const R v010_002 = dot2(nABy, v000_102, nACy, v000_003);
    const R v010_003 = dot2(nABy, v000_103, nACy, v000_004);
    const R v010_010 = dot2(nABy, v000_110, nACy, v000_011);
    const R v010_011 = dot2(nABy, v000_111, nACy, v000_012);
    const R v010_100 = dot2(nABy, v000_200, nACy, v000_101);
    const R v010_101 = dot2(nABy, v000_201, nACy, v000_102);
    const R v010_102 = dot2(nABy, v000_202, nACy, v000_103);
    const R v010_110 = dot2(nABy, v000_210, nACy, v000_111);
    const R v010_200 = dot2(nABy, v000_300, nACy, v000_201);
    const R v010_201 = dot2(nABy, v000_301, nACy, v000_202);
    const R v010_300 = dot2(nABy, v000_400, nACy, v000_301);
    const R v001_001 = dot2(nABz, v000_101, nACz, v000_002);
    const R v001_002 = dot2(nABz, v000_102, nACz, v000_003);
    const R v001_003 = dot2(nABz, v000_103, nACz, v000_004);
    const R v001_010 = dot2(nABz, v000_110, nACz, v000_011);
    const R v001_011 = dot2(nABz, v000_111, nACz, v000_012);
    const R v001_100 = dot2(nABz, v000_200, nACz, v000_101);
    const R v001_101 = dot2(nABz, v000_201, nACz, v000_102);
    const R v001_102 = dot2(nABz, v000_202, nACz, v000_103);
    const R v001_110 = dot2(nABz, v000_210, nACz, v000_111);
    const R v001_200 = dot2(nABz, v000_300, nACz, v000_201);
    const R v001_201 = dot2(nABz, v000_301, nACz, v000_202);
    const R v001_300 = dot2(nABz, v000_400, nACz, v000_301);
    const R v200_000 = dot2_add<1>(nABx, v100_100, nACx, v100_001, v000_010);
    const R v200_001 = dot2_add<1>(nABx, v100_101, nACx, v100_002, v000_011);
    const R v200_002 = dot2_add<1>(nABx, v100_102, nACx, v100_003, v000_012);
    const R v200_010 = dot2_add<1>(nABx, v100_110, nACx, v100_011, v000_020);
    const R v200_100 = dot2_add<1>(nABx, v100_200, nACx, v100_101, v000_110);
    const R v200_101 = dot2_add<1>(nABx, v100_201, nACx, v100_102, v000_111);
    const R v200_200 = dot2_add<1>(nABx, v100_300, nACx, v100_201, v000_210);
    const R v110_000 = dot2(nABx, v010_100, nACx, v010_001);
    const R v101_000 = dot2(nABx, v001_100, nACx, v001_001);
    const R v101_001 = dot2(nABx, v001_101, nACx, v001_002);
    const R v101_100 = dot2(nABx, v001_200, nACx, v001_101);
    const R v020_000 = dot2_add<1>(nABy, v010_100, nACy, v010_001, v000_010);
    const R v020_001 = dot2_add<1>(nABy, v010_101, nACy, v010_002, v000_011);
    const R v020_002 = dot2_add<1>(nABy, v010_102, nACy, v010_003, v000_012);
    const R v020_010 = dot2_add<1>(nABy, v010_110, nACy, v010_011, v000_020);
    const R v020_100 = dot2_add<1>(nABy, v010_200, nACy, v010_101, v000_110);
    const R v020_101 = dot2_add<1>(nABy, v010_201, nACy, v010_102, v000_111);
    const R v020_200 = dot2_add<1>(nABy, v010_300, nACy, v010_201, v000_210);
    const R v011_000 = dot2(nABy, v001_100, nACy, v001_001);
    const R v002_000 = dot2_add<1>(nABz, v001_100, nACz, v001_001, v000_010);
    const R v002_001 = dot2_add<1>(nABz, v001_101, nACz, v001_002, v000_011);
    const R v002_002 = dot2_add<1>(nABz, v001_102, nACz, v001_003, v000_012);
    const R v002_010 = dot2_add<1>(nABz, v001_110, nACz, v001_011, v000_020);
    const R v002_100 = dot2_add<1>(nABz, v001_200, nACz, v001_101, v000_110);
    const R v002_101 = dot2_add<1>(nABz, v001_201, nACz, v001_102, v000_111);
    const R v002_200 = dot2_add<1>(nABz, v001_300, nACz, v001_201, v000_210);
    const R v300_000 = dot2_add<2>(nABx, v200_100, nACx, v200_001, v100_010);
    const R v300_001 = dot2_add<2>(nABx, v200_101, nACx, v200_002, v100_011);
    const R v300_100 = dot2_add<2>(nABx, v200_200, nACx, v200_101, v100_110);
    const R v210_000 = dot2(nABy, v200_100, nACy, v200_001);
    const R v201_000 = dot2(nABz, v200_100, nACz, v200_001);
    const R v201_001 = dot2(nABz, v200_101, nACz, v200_002);
    const R v201_100 = dot2(nABz, v200_200, nACz, v200_101);
    const R v120_000 = dot2(nABx, v020_100, nACx, v020_001);
    const R v120_001 = dot2(nABx, v020_101, nACx, v020_002);
    const R v120_100 = dot2(nABx, v020_200, nACx, v020_101);
    const R v111_000 = dot2(nABy, v101_100, nACy, v101_001);
    const R v102_000 = dot2(nABx, v002_100, nACx, v002_001);
    const R v030_000 = dot2_add<2>(nABy, v020_100, nACy, v020_001, v010_010);
    const R v030_001 = dot2_add<2>(nABy, v020_101, nACy, v020_002, v010_011);
    const R v030_100 = dot2_add<2>(nABy, v020_200, nACy, v020_101, v010_110);
    const R v021_000 = dot2(nABz, v020_100, nACz, v020_001);
    const R v012_000 = dot2(nABy, v002_100, nACy, v002_001);
    const R v012_001 = dot2(nABy, v002_101, nACy, v002_002);
    const R v012_100 = dot2(nABy, v002_200, nACy, v002_101);
    const R v003_000 = dot2_add<2>(nABz, v002_100, nACz, v002_001, v001_010);
    const R v003_001 = dot2_add<2>(nABz, v002_101, nACz, v002_002, v001_011);
    const R v003_100 = dot2_add<2>(nABz, v002_200, nACz, v002_101, v001_110);
    const R v400_000 = dot2_add<3>(nABx, v300_100, nACx, v300_001, v200_010);
    const R v310_000 = dot2(nABy, v300_100, nACy, v300_001);
    const R v301_000 = dot2(nABz, v300_100, nACz, v300_001);
    const R v220_000 = dot2_add<1>(nABx, v120_100, nACx, v120_001, v020_010);
    const R v211_000 = dot2(nABy, v201_100, nACy, v201_001);
    const R v202_000 = dot2_add<1>(nABz, v201_100, nACz, v201_001, v200_010);
    const R v130_000 = dot2(nABx, v030_100, nACx, v030_001);
    const R v121_000 = dot2(nABz, v120_100, nACz, v120_001);
    const R v112_000 = dot2(nABx, v012_100, nACx, v012_001);
    const R v103_000 = dot2(nABx, v003_100, nACx, v003_001);
    const R v040_000 = dot2_add<3>(nABy, v030_100, nACy, v030_001, v020_010);
    const R v031_000 = dot2(nABz, v030_100, nACz, v030_001);
    const R v022_000 = dot2_add<1>(nABy, v012_100, nACy, v012_001, v002_010);
    const R v013_000 = dot2(nABy, v003_100, nACy, v003_001);
    const R v004_000 = dot2_add<3>(nABz, v003_100, nACz, v003_001, v002_010);
    acc[0] = v200_000;
    acc[1] = v110_000;
    acc[2] = v101_000;
    acc[3] = v020_000;
    acc[4] = v011_000;
    acc[5] = v002_000;
    acc[6] = v300_000;
    acc[7] = v210_000;
    acc[8] = v201_000;
    acc[9] = v120_000;
    acc[10] = v111_000;
    acc[11] = v102_000;
    acc[12] = v030_000;
    acc[13] = v021_000;
    acc[14] = v012_000;
    acc[15] = v003_000;
    acc[16] = v400_000;
    acc[17] = v310_000;
    acc[18] = v301_000;
    acc[19] = v220_000;
    acc[20] = v211_000;
    acc[21] = v202_000;
    acc[22] = v130_000;
    acc[23] = v121_000;
    acc[24] = v112_000;
    acc[25] = v103_000;
    acc[26] = v040_000;
    acc[27] = v031_000;
    acc[28] = v022_000;
    acc[29] = v013_000;
    acc[30] = v004_000;
  }
  template <typename R, typename A>
  __device__ static __forceinline__ void vrr(const R* S, R PAx, R PAy, R PAz, R PCx, R PCy, R PCz,
                                             R k1, R k2, R k3, A* acc) {
    (void)PAx; (void)PAy; (void)PAz; (void)PCx; (void)PCy; (void)PCz; (void)k1; (void)k2; (void)k3;
    const R t000_0 = S[0];
    const R t000_1 = S[1];
    const R t000_2 = S[2];
    const R t000_3 = S[3];
    const R t000_4 = S[4];
    const R t100_0 = fma(PAx, t000_0, -PCx * t000_1);
    const R t100_1 = fma(PAx, t000_1, -PCx * t000_2);
    const R t100_2 = fma(PAx, t000_2, -PCx * t000_3);
    const R t100_3 = fma(PAx, t000_3, -PCx * t000_4);
    const R t010_0 = fma(PAy, t000_0, -PCy * t000_1);
    const R t010_1 = fma(PAy, t000_1, -PCy * t000_2);
    const R t010_2 = fma(PAy, t000_2, -PCy * t000_3);
    const R t010_3 = fma(PAy, t000_3, -PCy * t000_4);
    const R t001_0 = fma(PAz, t000_0, -PCz * t000_1);
    const R t001_1 = fma(PAz, t000_1, -PCz * t000_2);
    const R t001_2 = fma(PAz, t000_2, -PCz * t000_3);
    const R t001_3 = fma(PAz, t000_3, -PCz * t000_4);
    const R t200_0 = fma(k1, t000_0 - t000_1, fma(PAx, t100_0, -PCx * t100_1));
    const R t200_1 = fma(k1, t000_1 - t000_2, fma(PAx, t100_1, -PCx * t100_2));
    const R t200_2 = fma(k1, t000_2 - t000_3, fma(PAx, t100_2, -PCx * t100_3));
    const R t110_0 = fma(PAx, t010_0, -PCx * t010_1);
    const R t101_0 = fma(PAx, t001_0, -PCx * t001_1);
    const R t020_0 = fma(k1, t000_0 - t000_1, fma(PAy, t010_0, -PCy * t010_1));
    const R t020_1 = fma(k1, t000_1 - t000_2, fma(PAy, t010_1, -PCy * t010_2));
    const R t020_2 = fma(k1, t000_2 - t000_3, fma(PAy, t010_2, -PCy * t010_3));
    const R t011_0 = fma(PAy, t001_0, -PCy * t001_1);
    const R t011_1 = fma(PAy, t001_1, -PCy * t001_2);
    const R t002_0 = fma(k1, t000_0 - t000_1, fma(PAz, t001_0, -PCz * t001_1));
    const R t002_1 = fma(k1, t000_1 - t000_2, fma(PAz, t001_1, -PCz * t001_2));
    const R t002_2 = fma(k1, t000_2 - t000_3, fma(PAz, t001_2, -PCz * t001_3));
    const R t300_0 = fma(k2, t100_0 - t100_1, fma(PAx, t200_0, -PCx * t200_1));
    const R t300_1 = fma(k2, t100_1 - t100_2, fma(PAx, t200_1, -PCx * t200_2));
    const R t210_0 = fma(PAy, t200_0, -PCy * t200_1);
    const R t201_0 = fma(PAz, t200_0, -PCz * t200_1);
    const R t201_1 = fma(PAz, t200_1, -PCz * t200_2);
    const R t120_0 = fma(PAx, t020_0, -PCx * t020_1);
    const R t120_1 = fma(PAx, t020_1, -PCx * t020_2);
    const R t111_0 = fma(PAx, t011_0, -PCx * t011_1);
    const R t102_0 = fma(PAx, t002_0, -PCx * t002_1);
    const R t102_1 = fma(PAx, t002_1, -PCx * t002_2);
    const R t030_0 = fma(k2, t010_0 - t010_1, fma(PAy, t020_0, -PCy * t020_1));
    const R t030_1 = fma(k2, t010_1 - t010_2, fma(PAy, t020_1, -PCy * t020_2));
    const R t021_0 = fma(PAz, t020_0, -PCz * t020_1);
    const R t021_1 = fma(PAz, t020_1, -PCz * t020_2);
    const R t012_0 = fma(PAy, t002_0, -PCy * t002_1);
    const R t012_1 = fma(PAy, t002_1, -PCy * t002_2);
    const R t003_0 = fma(k2, t001_0 - t001_1, fma(PAz, t002_0, -PCz * t002_1));
    const R t003_1 = fma(k2, t001_1 - t001_2, fma(PAz, t002_1, -PCz * t002_2));
    const R t400_0 = fma(k3, t200_0 - t200_1, fma(PAx, t300_0, -PCx * t300_1));
    const R t310_0 = fma(PAy, t300_0, -PCy * t300_1);
    const R t301_0 = fma(PAz, t300_0, -PCz * t300_1);
    const R t220_0 = fma(k1, t020_0 - t020_1, fma(PAx, t120_0, -PCx * t120_1));
    const R t211_0 = fma(PAy, t201_0, -PCy * t201_1);
    const R t202_0 = fma(k1, t002_0 - t002_1, fma(PAx, t102_0, -PCx * t102_1));
    const R t130_0 = fma(PAx, t030_0, -PCx * t030_1);
    const R t121_0 = fma(PAx, t021_0, -PCx * t021_1);
    const R t112_0 = fma(PAx, t012_0, -PCx * t012_1);
    const R t103_0 = fma(PAx, t003_0, -PCx * t003_1);
    const R t040_0 = fma(k3, t020_0 - t020_1, fma(PAy, t030_0, -PCy * t030_1));
    const R t031_0 = fma(PAz, t030_0, -PCz * t030_1);
    const R t022_0 = fma(k1, t002_0 - t002_1, fma(PAy, t012_0, -PCy * t012_1));
    const R t013_0 = fma(PAy, t003_0, -PCy * t003_1);
    const R t004_0 = fma(k3, t002_0 - t002_1, fma(PAz, t003_0, -PCz * t003_1));
    acc[0] += t200_0;
    acc[1] += t110_0;
    acc[2] += t101_0;
    acc[3] += t020_0;
    acc[4] += t011_0;
    acc[5] += t002_0;
    acc[6] += t300_0;
    acc[7] += t210_0;
    acc[8] += t201_0;
    acc[9] += t120_0;
    acc[10] += t111_0;
    acc[11] += t102_0;
    acc[12] += t030_0;
    acc[13] += t021_0;
    acc[14] += t012_0;
    acc[15] += t003_0;
    acc[16] += t400_0;
    acc[17] += t310_0;
    acc[18] += t301_0;
    acc[19] += t220_0;
    acc[20] += t211_0;
    acc[21] += t202_0;
    acc[22] += t130_0;
    acc[23] += t121_0;
    acc[24] += t112_0;
    acc[25] += t103_0;
    acc[26] += t040_0;
    acc[27] += t031_0;
    acc[28] += t022_0;
    acc[29] += t013_0;
    acc[30] += t004_0;
  }
  template <typename R>
  __device__ static __forceinline__ void hrr(const R* acc, R ABx, R ABy, R ABz, R* xi) {
    (void)ABx; (void)ABy; (void)ABz;
    const R x004_000 = acc[30];
    const R x013_000 = acc[29];
    const R x022_000 = acc[28];
    const R x031_000 = acc[27];
    const R x040_000 = acc[26];
    const R x103_000 = acc[25];
    const R x112_000 = acc[24];
    const R x121_000 = acc[23];
    const R x130_000 = acc[22];
    const R x202_000 = acc[21];
    const R x211_000 = acc[20];
    const R x220_000 = acc[19];
    const R x301_000 = acc[18];
    const R x310_000 = acc[17];
    const R x400_000 = acc[16];
    const R x003_000 = acc[15];
    const R x012_000 = acc[14];
    const R x021_000 = acc[13];
    const R x030_000 = acc[12];
    const R x102_000 = acc[11];
    const R x111_000 = acc[10];
    const R x120_000 = acc[9];
    const R x201_000 = acc[8];
    const R x210_000 = acc[7];
    const R x300_000 = acc[6];
    const R x002_000 = acc[5];
    const R x011_000 = acc[4];
    const R x020_000 = acc[3];
    const R x101_000 = acc[2];
    const R x110_000 = acc[1];
    const R x200_000 = acc[0];
    const R x003_001 = fma(ABz, x003_000, x004_000);
    const R x012_001 = fma(ABz, x012_000, x013_000);
    const R x012_010 = fma(ABy, x012_000, x022_000);
    const R x021_001 = fma(ABz, x021_000, x022_000);
    const R x021_010 = fma(ABy, x021_000, x031_000);
    const R x030_001 = fma(ABz, x030_000, x031_000);
    const R x030_010 = fma(ABy, x030_000, x040_000);
    const R x102_001 = fma(ABz, x102_000, x103_000);
    const R x102_010 = fma(ABy, x102_000, x112_000);
    const R x102_100 = fma(ABx, x102_000, x202_000);
    const R x111_001 = fma(ABz, x111_000, x112_000);
    const R x111_010 = fma(ABy, x111_000, x121_000);
    const R x111_100 = fma(ABx, x111_000, x211_000);
    const R x120_001 = fma(ABz, x120_000, x121_000);
    const R x120_010 = fma(ABy, x120_000, x130_000);
    const R x120_100 = fma(ABx, x120_000, x220_000);
    const R x201_001 = fma(ABz, x201_000, x202_000);
    const R x201_010 = fma(ABy, x201_000, x211_000);
    const R x201_100 = fma(ABx, x201_000, x301_000);
    const R x210_001 = fma(ABz, x210_000, x211_000);
    const R x210_010 = fma(ABy, x210_000, x220_000);
    const R x210_100 = fma(ABx, x210_000, x310_000);
    const R x300_001 = fma(ABz, x300_000, x301_000);
    const R x300_010 = fma(ABy, x300_000, x310_000);
    const R x300_100 = fma(ABx, x300_000, x400_000);
    const R x002_001 = fma(ABz, x002_000, x003_000);
    const R x002_010 = fma(ABy, x002_000, x012_000);
    const R x002_100 = fma(ABx, x002_000, x102_000);
    const R x011_001 = fma(ABz, x011_000, x012_000);
    const R x011_010 = fma(ABy, x011_000, x021_000);
    const R x011_100 = fma(ABx, x011_000, x111_000);
    const R x020_001 = fma(ABz, x020_000, x021_000);
    const R x020_010 = fma(ABy, x020_000, x030_000);
    const R x020_100 = fma(ABx, x020_000, x120_000);
    const R x101_001 = fma(ABz, x101_000, x102_000);
    const R x101_010 = fma(ABy, x101_000, x111_000);
    const R x101_100 = fma(ABx, x101_000, x201_000);
    const R x110_001 = fma(ABz, x110_000, x111_000);
    const R x110_010 = fma(ABy, x110_000, x120_000);
    const R x110_100 = fma(ABx, x110_000, x210_000);
    const R x200_001 = fma(ABz, x200_000, x201_000);
    const R x200_010 = fma(ABy, x200_000, x210_000);
    const R x200_100 = fma(ABx, x200_000, x300_000);
    const R x002_002 = fma(ABz, x002_001, x003_001);
    const R x002_011 = fma(ABy, x002_001, x012_001);
    const R x002_020 = fma(ABy, x002_010, x012_010);
    const R x002_101 = fma(ABx, x002_001, x102_001);
    const R x002_110 = fma(ABx, x002_010, x102_010);
    const R x002_200 = fma(ABx, x002_100, x102_100);
    const R x011_002 = fma(ABz, x011_001, x012_001);
    const R x011_011 = fma(ABy, x011_001, x021_001);
    const R x011_020 = fma(ABy, x011_010, x021_010);
    const R x011_101 = fma(ABx, x011_001, x111_001);
    const R x011_110 = fma(ABx, x011_010, x111_010);
    const R x011_200 = fma(ABx, x011_100, x111_100);
    const R x020_002 = fma(ABz, x020_001, x021_001);
    const R x020_011 = fma(ABy, x020_001, x030_001);
    const R x020_020 = fma(ABy, x020_010, x030_010);
    const R x020_101 = fma(ABx, x020_001, x120_001);
    const R x020_110 = fma(ABx, x020_010, x120_010);
    const R x020_200 = fma(ABx, x020_100, x120_100);
    const R x101_002 = fma(ABz, x101_001, x102_001);
    const R x101_011 = fma(ABy, x101_001, x111_001);
    const R x101_020 = fma(ABy, x101_010, x111_010);
    const R x101_101 = fma(ABx, x101_001, x201_001);
    const R x101_110 = fma(ABx, x101_010, x201_010);
    const R x101_200 = fma(ABx, x101_100, x201_100);
    const R x110_002 = fma(ABz, x110_001, x111_001);
    const R x110_011 = fma(ABy, x110_001, x120_001);
    const R x110_020 = fma(ABy, x110_010, x120_010);
    const R x110_101 = fma(ABx, x110_001, x210_001);
    const R x110_110 = fma(ABx, x110_010, x210_010);
    const R x110_200 = fma(ABx, x110_100, x210_100);
    const R x200_002 = fma(ABz, x200_001, x201_001);
    const R x200_011 = fma(ABy, x200_001, x210_001);
    const R x200_020 = fma(ABy, x200_010, x210_010);
    const R x200_101 = fma(ABx, x200_001, x300_001);
    const R x200_110 = fma(ABx, x200_010, x300_010);
    const R x200_200 = fma(ABx, x200_100, x300_100);
    xi[0] = x200_200;
    xi[1] = x200_110;
    xi[2] = x200_101;
    xi[3] = x200_020;
    xi[4] = x200_011;
    xi[5] = x200_002;
    xi[6] = x110_200;
    xi[7] = x110_110;
    xi[8] = x110_101;
    xi[9] = x110_020;
    xi[10] = x110_011;
    xi[11] = x110_002;
    xi[12] = x101_200;
    xi[13] = x101_110;
    xi[14] = x101_101;
    xi[15] = x101_020;
    xi[16] = x101_011;
    xi[17] = x101_002;
    xi[18] = x020_200;
    xi[19] = x020_110;
    xi[20] = x020_101;
    xi[21] = x020_020;
    xi[22] = x020_011;
    xi[23] = x020_002;
    xi[24] = x011_200;
    xi[25] = x011_110;
    xi[26] = x011_101;
    xi[27] = x011_020;
    xi[28] = x011_011;
    xi[29] = x011_002;
    xi[30] = x002_200;
    xi[31] = x002_110;
    xi[32] = x002_101;
    xi[33] = x002_020;
    xi[34] = x002_011;
    xi[35] = x002_002;
  }
};

}  // namespace snk
