// Integral-contraction kernel of libsnk (sm_103a): for every shell pair (a, b)
// of a batch's pair list V_j and every grid point r_i of the batch,
//
//   Theta^n_0 = pref * F_n(zeta |P - r_i|^2)              (App. A, seed)
//   the primitive pairs contracted into scalars, one VRR   (App. A, Eq. vrr)
//   HRR to the target block Xi_ab                          (App. A, Eq. hrr)
//   G_{i a} += Xi_ab F_{i b},  G_{i b} += Xi_ab^T F_{i a}  (Eq. gmat, a != b)
//
// with F already scaled by w_i and the component factor of its column, so the
// 3c-CP block is never stored (the merged HRR + contraction of App. A).
//
// Parallel decomposition (Sec. II.F, batching levels (1)-(3)): one thread per
// grid point, a 128-point tile of one batch per CTA iteration, the batch's
// whole pair list of one class per tile; persistent CTAs take tiles from an
// atomic ticket (largest batches first).  Each G entry of a launch therefore
// has a single writer, its point's thread, whose reductions land in list
// order: G, and with it K, is the same bit for bit from run to run.  The Boys
// interpolation table of the class's L lives in shared memory.
//
// GB300 issues FP64 at 2 DFMA per SM per clock (1/64 of FP32), so the kernel
// is FP64-pipe bound by construction: table lookups, index arithmetic, F loads
// and the G atomics (L2 reductions, ~600 G/s) all hide under the DFMA stream,
// and what counts is the number of FP64 instructions.  The primitive pairs are
// therefore contracted before the recursion (gen_os.py): a dd primitive pair
// costs 29 operations after its Boys functions instead of 180, and the
// recursion's 313 run once per contracted pair.  Measured with 9 primitive
// pairs per shell pair, against the recursion per primitive pair: FP64, 24
// atoms and 72,000 points, 260 -> 172 ms a build (dd 33 -> 15, dp 65 -> 34, pp
// 40 -> 27, ps 57 -> 48, ss 20); double-FP32, 96 atoms and 768,000 points, 491
// -> 333 ms (dp 143 -> 74, dd 160 -> 122).  The mixed
// form adds an FP32 kernel for its low-estimate pairs and a double-FP32 one
// (ds_arith.cuh) for the rest; all three take the number of densities sharing
// each 3c-CP block as a template parameter.
#include <cuda_runtime.h>

#include <cstdint>

#include "async_copy.cuh"
#include "ds_arith.cuh"
#include "f2_arith.cuh"
#include "os_generated.cuh"
#include "snk_internal.h"

namespace snk {

namespace {

constexpr int kIntThreads = kPointTile;
constexpr int kMaxRun = kMaxPairsPerStep;
constexpr int kPrimF4 = kPrimF32Words / 4;  // float4 per FP32 primitive record
constexpr unsigned long long kCopyWaitNs = 2000000000ull;  // 2 s per wait on a bulk copy, then give up
constexpr long long kBoysTMaxBits = 0x4049000000000000LL;  // bit pattern of 50.0
static_assert(kBoysTMax == 50.0, "kBoysTMaxBits encodes 50.0");

// S_n = F_n(T), n = 0..L (Eq. boys).  Below T = 50: F_L by a polynomial of
// degree 6 about the nearest table node (the Taylor series, dF_n/dT = -F_{n+1},
// economised) and the downward recursion F_n = (2T F_{n+1} + e^{-T}) / (2n+1);
// above: F_0 = sqrt(pi/T)/2 and F_{n+1} = (2n+1) F_n / (2T) (e^{-T} < 2e-22 is
// dropped).  Every FP64 operation costs the whole SM 16 clocks per warp, so: the
// primitive pair's prefactor is in its contraction coefficients, where it rides
// on a multiply-add; 2T is one integer addition to T's exponent.  Against eight
// Taylor terms on |x| <= 0.05 and seeds with the prefactor: 24 atoms 176.0 ->
// 168.8 ms per build, 4 atoms 0.780 -> 0.743 ms; largest error of a seed times its
// prefactor 1.4e-15 -> 6.8e-16 relative, rms at most 2.0e-16 -> 1.5e-16.
// With a prefactor (the recursion of a single primitive pair) every seed has it.
template <int L>
__device__ __forceinline__ void boys_seeds(double T, const double* tab, double* S, double pref = 1.0) {
  if (__double_as_longlong(T) < kBoysTMaxBits) {
    // T in FP32 by integer operations: the conversion runs on the FP64 pipe (24
    // atoms, FP64 integrals 156.7 -> 155.6 ms)
    const int hi = max(__double2hiint(T), 0x38000000) - 0x38000000;  // 0 below 2^-127
    const float tf = __int_as_float((int)__funnelshift_l((unsigned)__double2loint(T), (unsigned)hi, 3));
    const int k = __float2int_rn(tf * (float)(1.0 / kBoysH));
    const double* row = tab + k * kBoysCols;
    const double x = row[kBoysCols - 1] - T;  // T_k - T, |x| <= 1/24
    double f = row[kBoysTerms - 1];
#pragma unroll
    for (int m = kBoysTerms - 2; m >= 0; --m) f = fma(f, x, row[m]);
    S[L] = pref * f;
    if (L > 0) {
      // e^{-T} = e^{-T_k} e^{x}, e^{x} by its 8-term Taylor polynomial
      double e = 1.0 / 5040.0;
      e = fma(e, x, 1.0 / 720.0);
      e = fma(e, x, 1.0 / 120.0);
      e = fma(e, x, 1.0 / 24.0);
      e = fma(e, x, 1.0 / 6.0);
      e = fma(e, x, 0.5);
      e = fma(e, x, 1.0);
      e = fma(e, x, 1.0);
      const double pe = pref * (row[kBoysTerms] * e);
      // below 2^-1022 the sum is not 2T but as small, and e^{-T} = 1 beside it
      const double T2 = __hiloint2double(__double2hiint(T) + 0x00100000, __double2loint(T));
#pragma unroll
      for (int n = L - 1; n >= 0; --n) S[n] = fma(T2, S[n + 1], pe) * (1.0 / (2 * n + 1));
    }
  } else {
    const double r = rsqrt(T);
    S[0] = pref * (0.88622692545275801365 * r);  // sqrt(pi)/2
    if (L > 0) {
      const double o = 0.5 * (r * r);
#pragma unroll
      for (int n = 0; n < L; ++n) S[n + 1] = S[n] * ((2 * n + 1) * o);
    }
  }
}

// Classes where a pair of uncontracted shells runs the recursion for its one
// primitive pair (the pair is the same for the whole block): contracting one pair
// first costs dd 342 operations instead of 259, dp 134 instead of 110, pp 51 instead
// of 46; from two primitive pairs on it is the cheaper form.  Uncontracted shells,
// 36 atoms, 288,000 points, ms per build without / with: d alone 246.2 / 200.4, p
// alone 50.5 / 47.1, p and d 312.8 / 272.5, s, p and d 349.8 / 324.2; contracted s
// and p with one d primitive 221.6 / 218.2.
template <int LA, int LB>
constexpr bool kOneByRecursion = LA + LB >= 2 && LB > 0;

// The sum of one term (0 + x is an addition to the compiler).
struct OnlyTerm {
  double v;
  __device__ __forceinline__ void operator+=(double x) { v = x; }
};

// Contracted Xi_ab (no component factors) of one pair at the point (cx, cy, cz);
// A is the centre of shell a.
template <int LA, int LB>
__device__ __forceinline__ void pair_xi(const PairHdr& h, const PrimPair* __restrict__ prims,
                                        const double* __restrict__ A, const double* tab, double cx, double cy,
                                        double cz, double* xi) {
  using C = OsClass<LA, LB>;
  if (kOneByRecursion<LA, LB> && h.pp_n == 1) {
    const PrimPair pp = prims[h.pp_off];
    const double PCx = pp.Px - cx, PCy = pp.Py - cy, PCz = pp.Pz - cz;
    const double T = pp.zeta * fma(PCx, PCx, fma(PCy, PCy, PCz * PCz));
    double S[C::L + 1], acc[C::NACC];
    boys_seeds<C::L>(T, tab, S, pp.pref);
    OnlyTerm one[C::NACC];
    const double kappa = pp.pref_far;
    C::vrr(S, pp.Px - A[0], pp.Py - A[1], pp.Pz - A[2], PCx, PCy, PCz, kappa, 2.0 * kappa, 3.0 * kappa, one);
#pragma unroll
    for (int k = 0; k < C::NACC; ++k) acc[k] = one[k].v;
    C::hrr(acc, h.ABx, h.ABy, h.ABz, xi);
    return;
  }
  double M[C::NM];
#pragma unroll
  for (int k = 0; k < C::NM; ++k) M[k] = 0.0;
  for (int q = 0; q < h.pp_n; ++q) {
    const PrimPair pp = prims[h.pp_off + q];
    const double PCx = pp.Px - cx, PCy = pp.Py - cy, PCz = pp.Pz - cz;
    const double T = pp.zeta * fma(PCx, PCx, fma(PCy, PCy, PCz * PCz));
    double S[C::L + 1];
    boys_seeds<C::L>(T, tab, S);
    C::prim(S, OsCoef<double>{pp.pref, pp.c10, pp.c20, pp.c30, pp.c40, pp.c01, pp.c11, pp.c21, pp.c02}, M);
  }
  double acc[C::NACC];
  C::build(M, -h.ABx, -h.ABy, -h.ABz, cx - A[0], cy - A[1], cz - A[2], acc);
  C::hrr(acc, h.ABx, h.ABy, h.ABz, xi);
}

// Work item t of the FP64 / ds lists: tile t mod n_tiles, the launch's range t /
// n_tiles of its list.
__device__ __forceinline__ Tile tile_part(const IntegralArgs& a, int t) {
  Tile tile = a.tiles[t % a.n_tiles];
  if (a.parts > 1) {
    const int64_t n = tile.k1 - tile.k0, part = a.part0 + t / a.n_tiles;
    tile.k1 = tile.k0 + (int)(n * (part + 1) / a.parts);
    tile.k0 += (int)(n * part / a.parts);
  }
  return tile;
}

// ND densities share every Xi block: F and G of density d sit d ldq nS
// doubles after the batch's first block.
template <int LA, int LB, int ND>
__global__ void __launch_bounds__(kIntThreads) integral_kernel(IntegralArgs a) {
  using C = OsClass<LA, LB>;
  constexpr int NA = C::NA, NB = C::NB;
  extern __shared__ double s_tab[];
  const double* gtab = a.boys + (size_t)C::L * kBoysRows * kBoysCols;
  for (int e = threadIdx.x; e < kBoysRows * kBoysCols; e += blockDim.x) s_tab[e] = gtab[e];
  __shared__ int s_tile;
  __syncthreads();
  for (;;) {
    if (threadIdx.x == 0) s_tile = atomicAdd(a.ticket, 1);
    __syncthreads();
    const int t = s_tile;
    __syncthreads();
    if (t >= a.n_tiles * a.part_n) break;
    const Tile tile = tile_part(a, t);
    const BatchDesc bd = a.batches[tile.batch];
    const int i = tile.i0 + threadIdx.x;
    if (i >= bd.q) continue;
    const int64_t ldq = bd.ldq, dstr = (int64_t)bd.ldq * bd.nS;
    const double cx = a.xyz[3 * (bd.p0 + i)], cy = a.xyz[3 * (bd.p0 + i) + 1], cz = a.xyz[3 * (bd.p0 + i) + 2];
    const double* F = a.ws + bd.foff + i;
    double* G = a.ws + bd.goff + a.gshift + (t / a.n_tiles) * a.gpart + i;
    const int* cmap = a.colmap + bd.cm_off - bd.ms0;  // indexed by global shell id
    double ga[ND][NA], fa[ND][NA];
    int cur = -1, cola = 0;
    for (int k = tile.k0; k < tile.k1; ++k) {
      const PairHdr h = a.pairs[a.pairlist[k]];
      if (h.sa != cur) {
        if (cur >= 0) {
#pragma unroll
          for (int d = 0; d < ND; ++d)
#pragma unroll
            for (int u = 0; u < NA; ++u) atomicAdd(G + d * dstr + (cola + u) * ldq, ga[d][u]);
        }
        cur = h.sa;
        cola = cmap[cur];
#pragma unroll
        for (int d = 0; d < ND; ++d)
#pragma unroll
          for (int u = 0; u < NA; ++u) {
            ga[d][u] = 0.0;
            fa[d][u] = F[d * dstr + (cola + u) * ldq];
          }
      }
      const int colb = cmap[h.sb];
      if (cola < 0 || colb < 0) continue;  // cannot happen: the screen marks both shells of a kept pair
      double fb[ND][NB];
#pragma unroll
      for (int d = 0; d < ND; ++d)
#pragma unroll
        for (int v = 0; v < NB; ++v) fb[d][v] = F[d * dstr + (colb + v) * ldq];
      double xi[NA * NB];
      pair_xi<LA, LB>(h, a.prims, a.shell_xyz + 3 * h.sa, s_tab, cx, cy, cz, xi);
#pragma unroll
      for (int d = 0; d < ND; ++d)
#pragma unroll
        for (int u = 0; u < NA; ++u)
#pragma unroll
          for (int v = 0; v < NB; ++v) ga[d][u] = fma(xi[u * NB + v], fb[d][v], ga[d][u]);
      if (h.sa != h.sb) {
#pragma unroll
        for (int d = 0; d < ND; ++d)
#pragma unroll
          for (int v = 0; v < NB; ++v) {
            double g = 0.0;
#pragma unroll
            for (int u = 0; u < NA; ++u) g = fma(xi[u * NB + v], fa[d][u], g);
            atomicAdd(G + d * dstr + (colb + v) * ldq, g);
          }
      }
    }
    if (cur >= 0) {
#pragma unroll
      for (int d = 0; d < ND; ++d)
#pragma unroll
        for (int u = 0; u < NA; ++u) atomicAdd(G + d * dstr + (cola + u) * ldq, ga[d][u]);
    }
  }
}

// ---------------------------------------------------------------- FP32 pairs (mixed form)

// FP32 seeds S_n = pref F_n(T) at two points: 4-term Taylor about the nearest
// node of a 0.05-spaced float table below T = 30 (|T - T_k| <= 0.025:
// truncation below 2e-8 relative; one 16-byte row per lookup, the distance to the
// node k 0.05f formed by one multiply-add), the asymptotic form above (e^{-T} < 1e-13 is
// below FP32 resolution).  e^{-T} of the downward recursion comes from the
// hardware exponential (__expf, ~2^-21 relative).  The lookups and the
// polynomial run per point (the two rows' coefficients sit in different
// registers, and pairing them up costs more moves than it saves), everything
// else on both points at once.
// The argument is -T (the records hold -zeta): the expansion, the exponential
// and the row index then need no negation, which has no packed form.  Both
// forms are chosen by warp votes: the points of a warp are close together, so
// most primitive pairs are near or far for all of them, and the branches stay
// uniform.  Every lane of the warp must call it.
__device__ __forceinline__ float ex2_ftz(float x) {  // 2^x, |x| < 126 here
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rsqrt_ftz(float x) {  // normal x only
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float4 lds_f4(uint32_t addr) {
  float4 v;
  asm("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}
// k = round(20 T) is formed by adding 1.5 2^23: the sum's bit pattern is
// kRowMagic + k, so that row k of the table at the shared address tab is at
// (tab - 16 kRowMagic) + 16 pattern (mod 2^32)
constexpr float kRowMagicF = 12582912.0f;
constexpr uint32_t kRowMagic = 0x4B400000u;

template <int L>
__device__ __forceinline__ void boys_seeds_f32(f2 nT, f2 pref, f2 pref_far, uint32_t tab_adj, f2* S) {
  static_assert(kBoysColsF == 4 && kBoysTermsF == 4, "an FP32 table row is one float4");
  const bool near0 = nT.v.x > -kBoysTMaxF, near1 = nT.v.y > -kBoysTMaxF;
  const bool any_far = __any_sync(0xffffffffu, !(near0 && near1));
  if (__any_sync(0xffffffffu, near0 || near1)) {
    // a far point reads the last row and is replaced below
    const f2 Tc(fmaxf(nT.v.x, -kBoysTMaxF), fmaxf(nT.v.y, -kBoysTMaxF));
    const f2 u = fma(Tc, f2(-1.0f / kBoysHF), f2(kRowMagicF));
    const float4 r0 = lds_f4(tab_adj + 16u * __float_as_uint(u.v.x));
    const float4 r1 = lds_f4(tab_adj + 16u * __float_as_uint(u.v.y));
    const f2 x = fma(u + f2(-kRowMagicF), f2(kBoysHF), Tc);  // T_k - T
    const f2 F(fmaf(fmaf(fmaf(r0.w, x.v.x, r0.z), x.v.x, r0.y), x.v.x, r0.x),
               fmaf(fmaf(fmaf(r1.w, x.v.y, r1.z), x.v.y, r1.y), x.v.y, r1.x));
    S[L] = pref * F;
    if (L > 0) {
      const f2 y = Tc * f2(1.44269504088896341f);
      const f2 pe = pref * f2(ex2_ftz(y.v.x), ex2_ftz(y.v.y));
      const f2 T2 = Tc * f2(-2.0f);
#pragma unroll
      for (int n = L - 1; n >= 0; --n) S[n] = n ? fma(T2, S[n + 1], pe) * f2(1.0f / (2 * n + 1)) : fma(T2, S[n + 1], pe);
    }
  }
  if (any_far) {
    const f2 r(rsqrt_ftz(-nT.v.x), rsqrt_ftz(-nT.v.y));
    f2 F = pref_far * r;
    const f2 o = f2(0.5f) * (r * r);
#pragma unroll
    for (int n = 0; n <= L; ++n) {
      S[n] = f2(near0 ? S[n].v.x : F.v.x, near1 ? S[n].v.y : F.v.y);
      if (n < L) F = F * (f2((float)(2 * n + 1)) * o);
    }
  }
}

// The FP64 value of v by integer operations: the conversion instruction runs on
// the FP64 pipe (2 lanes per clock and SM), which the G updates kept 20-35 %
// busy.  Magnitudes below 2^-126 give zero: such a term of G cannot reach K, whose
// accumulator resolves 2^-76.  Infinities and NaN stay what they are.
__device__ __forceinline__ double f32_to_f64_bits(float v) {
  const uint32_t b = __float_as_uint(v), m = b & 0x7fffffffu;
  uint32_t hi = (b & 0x80000000u) | ((m >> 3) + 0x38000000u);
  if (m >= 0x7f800000u) hi |= 0x7ff00000u;
  return m < 0x00800000u ? 0.0 : __hiloint2double((int)hi, (int)(b << 29));
}

// The FP32 lists of the mixed form, two points per thread in packed FP32
// arithmetic (f2).  One thread per point was bound by instruction issue (71-82
// % of the slots, the FMA pipe 26-58 % busy): a packed instruction does both
// points' operation in one slot, and the records, loop control and staging are
// paid once for the two.  The FMA pipe's lane rate is the same either way.
//
// A tile is a batch's whole list on 128 points, a CTA of two warps per tile;
// a lane holds the points l and l + 32 of its warp's 64, so that every F load
// and G reduction of a warp is a full row.  The list is taken in steps of
// a.run pairs: each step's pair headers, columns, R_a - R_b and R_a are staged
// in shared memory (after the tile screen), and the tile's batch descriptor
// sits in shared memory too, so that nothing of the tile stays in registers
// across the pair loop.
//
// A primitive pair is a 64-byte record of scalars stored twice, {-zeta, PAx,
// pref, pref_far, PAy, PAz, kappa, -sigma}, so that a 16-byte load gives two
// packed operands.  Per (pair, point) the kernel forms A - r_i once from the
// (hi, lo) float splits of A and r_i, and P - r_i = (P - A) + (A - r_i) per
// primitive: accurate to FP32 relative to the larger of |P - A| and |A - r_i|
// wherever the molecule sits, which is what the VRR terms PA_x Theta and PC_x
// Theta need.  In ps and ds (f32_early) the primitive pairs are contracted
// before the recursion as in the other kernels; the other classes keep the
// recursion per primitive pair and with it their rounding.
//
// Per pair each warp needs the pair's primitive records and the F columns of
// shell b at its 64 points:
//   - heavy classes (L >= 2): a ring of three slots per warp, filled by TMA
//     bulk copies that lane 0 issues two pairs ahead, each slot completing
//     on its own mbarrier (bounded waits);
//   - light classes: the next pair's F from global memory into registers and
//     its records into a second shared buffer while the current pair
//     computes (fewer instructions per pair than the ring, whose serial
//     issue does not pay for a pair of a few primitives).
//
// 96 atoms and 768,000 points, ms per build before / now: ss 37.3 / 28.2, ps 87.5
// / 70.3, pp 68.5 / 61.4, ds 66.8 / 47.1, dp 105.9 / 94.5, dd 43.3 / 39.7.  What
// bounds it now is latency (IPC 0.5 per scheduler, fixed-latency and shared-
// memory waits): two points double the registers, so half as many warps fit.
constexpr int kF32Threads = kPointTile / 2;
// CTAs per SM asked of the compiler, chosen with one density (with two, dp spills 152
// bytes, ps 64, pp 32 and ss 12 under it).  96 atoms and 768,000 points, ms per build
// without / with: ss 30.5 / 29.1, ps 75.9 / 72.5, pp 65.8 / 60.1, dp 107 / 95; ds
// and dd lose (47.3 / 48.8 in ds).
constexpr int f32_min_ctas(int la, int lb) {
  return la == 0 ? 11 : la == 1 ? (lb == 0 ? 10 : 8) : lb == 1 ? 5 : 1;
}

template <int LA, int LB, int ND>
__global__ void __launch_bounds__(kF32Threads, f32_min_ctas(LA, LB)) integral_kernel_f32(IntegralArgs a) {
  using C = OsClass<LA, LB>;
  constexpr int NA = C::NA, NB = C::NB;
  constexpr bool kEarly = f32_early(LA, LB);  // contraction before the recursion
  constexpr int kStage = 16;                      // primitive records of a pair staged
  constexpr bool RING = C::L >= 2;
  constexpr int kRing = 3;
  constexpr int kRF4 = C::L == 0 ? 3 : kPrimF4;  // float4 of a record that the class reads
  constexpr int kRecF4 = kRF4 * kStage;  // float4 of records per slot
  constexpr int kFbF4 = ND * NB * 64 / 4;   // float4 of F_b per ring slot
  constexpr int kW = kF32Threads / 32;
  constexpr int kHalves = kMaxRun / kF32Threads;  // pairs a thread stages per step
  extern __shared__ __align__(16) float s_tabf[];
  const uint32_t tab = smem_u32(s_tabf) - 16u * kRowMagic;  // see kRowMagic
  const float* gtab = a.boys_f + (size_t)C::L * kBoysRowsF * kBoysColsF;
  for (int e = threadIdx.x; e < kBoysRowsF * kBoysColsF; e += blockDim.x) s_tabf[e] = gtab[e];
  __shared__ int s_ppo[kMaxRun], s_ppn[kMaxRun], s_sa[kMaxRun], s_sb[kMaxRun], s_ca[kMaxRun], s_cb[kMaxRun];
  __shared__ float2 s_ab[kMaxRun][3];  // R_a - R_b (FP32), stored twice
  __shared__ float2 s_A[kMaxRun][3];   // R_a as (hi, lo)
  __shared__ __align__(128) float4 s_ring[RING ? kW : 1][RING ? kRing : 1][RING ? kRecF4 + kFbF4 : 1];
  __shared__ __align__(8) uint64_t s_full[kW][kRing];
  __shared__ float4 s_pr[RING ? 1 : kW][2][RING ? 1 : kRecF4];
  __shared__ Tile s_t;
  __shared__ BatchDesc s_bd;
  __shared__ int s_tid, s_wcnt[kHalves][kW];
  __shared__ volatile int s_abort;  // a wait ran out: the CTA stops taking work
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_abort = 0;
  if (RING && lane == 0) {
#pragma unroll
    for (int s = 0; s < kRing; ++s) mbar_init(&s_full[wid][s], 1);
    mbar_init_fence();
  }
  uint32_t prod = 0, cons = 0;  // ring: this warp's pairs issued into / taken from its slots
  for (;;) {
    __syncthreads();  // every thread is done with the previous tile's descriptors and pairs
    if (threadIdx.x == 0) {
      const int t = atomicAdd(a.ticket, 1);
      s_tid = t;
      if (t < a.n_tiles) {
        s_t = a.tiles[t];
        s_bd = a.batches[s_t.batch];
      }
    }
    __syncthreads();
    if (s_tid >= a.n_tiles || s_abort) break;
    // the tile's list in steps of a.run pairs (block-uniform loop: every
    // thread passes the same barriers)
    for (int kb = s_t.k0; kb < s_t.k1; kb += a.run) {
      // stage the step's pairs (kHalves per thread, order kept); with the tile
      // screen only those whose bound on this tile's points reaches eps_tile
      const int n = min(a.run, s_t.k1 - kb);  // n <= kMaxRun
      int pp_[kHalves], keep_n[kHalves];      // pair, primitive pairs kept (0: pair left out)
      unsigned bal[kHalves];
      unsigned npp_sum = 0;
#pragma unroll
      for (int hf = 0; hf < kHalves; ++hf) {
        const int r = threadIdx.x + hf * kF32Threads;
        keep_n[hf] = 0;
        pp_[hf] = 0;
        if (r < n) {
          const int p = a.pairlist[kb + r];
          const PairHdr h = a.pairs[p];
          pp_[hf] = p;
          int npp = h.pp_n32;  // the leading primitive pairs the FP32 tier keeps
          if (a.eps_tile > 0.f) {
            const int* cmap = a.colmap + s_bd.cm_off - s_bd.ms0;  // indexed by global shell id
            const int ca = cmap[h.sa], cb = cmap[h.sb];
            const float* ts = a.tsum + s_bd.ssoff + (int64_t)(s_t.i0 / kPointTile) * (s_bd.nS + 4);
            float sa = 0.f, sb = 0.f;
#pragma unroll
            for (int u = 0; u < NA; ++u) sa += ts[ca + u];
#pragma unroll
            for (int v = 0; v < NB; ++v) sb += ts[cb + v];
            // |A_ab| <= min(global bound, total charge / distance) on the tile's sphere
            const double* A = a.shell_xyz + 3 * h.sa;
            const float vx = (float)-h.ABx, vy = (float)-h.ABy, vz = (float)-h.ABz;  // B - A
            const float wx = ts[s_bd.nS] - (float)A[0], wy = ts[s_bd.nS + 1] - (float)A[1],
                        wz = ts[s_bd.nS + 2] - (float)A[2];
            const float vv = vx * vx + vy * vy + vz * vz;
            float tt = vv > 0.f ? (wx * vx + wy * vy + wz * vz) / vv : 0.f;
            tt = fminf(fmaxf(tt, 0.f), 1.f);
            const float dx = wx - tt * vx, dy = wy - tt * vy, dz = wz - tt * vz;
            const float d = sqrtf(dx * dx + dy * dy + dz * dz) - ts[s_bd.nS + 3] - 1e-4f;
            const float glob = (float)a.pbound[p], smax = fmaxf(sa, sb);
            float bnd = glob;
            if (d > 0.f) bnd = fminf(bnd, (float)a.qbound[p] / d);
            if (bnd * smax >= a.eps_tile) {
              // primitive pairs come largest bound first: leave out the tail whose
              // bounds on this tile add up to less than eps_tile
              const float* share = a.prim_share + h.pp_off;
              float tail = 0.f;
              while (npp > 1) {
                const float t2 = tail + share[npp - 1] * glob * smax;
                if (t2 >= a.eps_tile) break;
                tail = t2;
                --npp;
              }
            } else {
              npp = 0;
            }
          }
          keep_n[hf] = npp;
          npp_sum += (unsigned)npp;
        }
        bal[hf] = __ballot_sync(0xffffffffu, keep_n[hf] > 0);
        if (lane == 0) s_wcnt[hf][wid] = __popc(bal[hf]);
      }
      npp_sum = __reduce_add_sync(0xffffffffu, npp_sum);
      __syncthreads();
      int nrun = 0;
#pragma unroll
      for (int hf = 0; hf < kHalves; ++hf) {
        int q = nrun + __popc(bal[hf] & ((1u << lane) - 1u));
#pragma unroll
        for (int w = 0; w < kW; ++w) {
          q += w < wid ? s_wcnt[hf][w] : 0;
          nrun += s_wcnt[hf][w];
        }
        if (keep_n[hf] > 0) {
          const int p = pp_[hf];
          const PairHdr h = a.pairs[p];
          const int* cmap = a.colmap + s_bd.cm_off - s_bd.ms0;
          s_ppo[q] = h.pp_off;
          s_ppn[q] = keep_n[hf];
          s_sa[q] = h.sa;
          s_sb[q] = h.sb;
          s_ca[q] = cmap[h.sa];
          s_cb[q] = cmap[h.sb];
          const float2* ab = a.pair_ab + 4 * (size_t)p;
          const float2* pa = a.pair_a + 4 * (size_t)p;
#pragma unroll
          for (int m = 0; m < 3; ++m) {
            s_ab[q][m] = make_float2(ab[m].x, ab[m].x);
            s_A[q][m] = pa[m];
          }
        }
      }
      if (lane == 0 && npp_sum > 0) {  // the work this step computes, for the flop counts
        unsigned kept = 0;
#pragma unroll
        for (int hf = 0; hf < kHalves; ++hf) kept += __popc(bal[hf]);
        const unsigned long long pts = (unsigned long long)min(kPointTile, s_bd.q - s_t.i0);
        atomicAdd(&a.exec[0], (unsigned long long)npp_sum * pts);
        atomicAdd(&a.exec[1], (unsigned long long)kept * pts);
      }
      __syncthreads();
      // this lane's points i and i + 32 (rows up to ldq exist, and F is zero
      // beyond the batch's points, so a point past the end adds zero to G)
      const int iw = s_t.i0 + 64 * wid, i = iw + lane;
      if (nrun <= 0 || s_abort || iw >= s_bd.q) continue;
      ds cx[2], cy[2], cz[2];
#pragma unroll
      for (int w = 0; w < 2; ++w) {
        cx[w] = cy[w] = cz[w] = ds_make(0.f, 0.f);
        if (i + 32 * w < s_bd.q) {
          const double* c = a.xyz + 3 * (s_bd.p0 + i + 32 * w);
          cx[w] = ds_from(c[0]);
          cy[w] = ds_from(c[1]);
          cz[w] = ds_from(c[2]);
        }
      }
      const int ldq = s_bd.ldq;
      const int64_t dstr = (int64_t)s_bd.ldq * s_bd.nS;  // density d's F / G: + d dstr
      const float* F = a.ws32 + s_bd.foff32 + i;
      double* G64 = a.ws + s_bd.goff + a.gshift + i;
      // the FP32 contributions are added to the FP64 G with FP64 reductions;
      // each G entry of the launch has one writer (its point's thread), so
      // they land in list order and G is the same from run to run
      auto gadd = [&](int d, int col, f2 v) {
        double* g = G64 + d * dstr + (int64_t)col * ldq;
        atomicAdd(g, f32_to_f64_bits(v.v.x));
        atomicAdd(g + 32, f32_to_f64_bits(v.v.y));
      };
      auto fload = [&](int d, int col) {
        const float* f = F + d * dstr + (int64_t)col * ldq;
        return f2(f[0], f[32]);
      };
      f2 ga[ND][NA], fa[ND][NA];
      int cur = -1, cola = 0;
      // pair r at this thread's points, from its records (shared memory, or
      // global memory for more than kStage primitive pairs) and F_b
      auto compute = [&](int r, const float4* rec, const f2 (&fb)[ND][NB]) {
        const int sa = s_sa[r];
        if (sa != cur) {
          if (cur >= 0) {
#pragma unroll
            for (int d = 0; d < ND; ++d)
#pragma unroll
              for (int u = 0; u < NA; ++u) gadd(d, cola + u, ga[d][u]);
          }
          cur = sa;
          cola = s_ca[r];
#pragma unroll
          for (int d = 0; d < ND; ++d)
#pragma unroll
            for (int u = 0; u < NA; ++u) {
              ga[d][u] = f2(0.f);
              fa[d][u] = fload(d, cola + u);
            }
        }
        // A - r_i, once per pair and point
        auto ac = [&](int m, const ds* c) {
          const float2 A = s_A[r][m];
          return f2((A.x - c[0].hi) + (A.y - c[0].lo), (A.x - c[1].hi) + (A.y - c[1].lo));
        };
        const f2 ACx = ac(0, cx), ACy = ac(1, cy), ACz = ac(2, cz);
        const f2 ABx(s_ab[r][0]), ABy(s_ab[r][1]), ABz(s_ab[r][2]);
        f2 acc[C::NACC], M[C::NM];
        if (kEarly) {
#pragma unroll
          for (int u = 0; u < C::NM; ++u) M[u] = f2(0.f);
        } else {
#pragma unroll
          for (int u = 0; u < C::NACC; ++u) acc[u] = f2(0.f);
        }
        auto prim = [&](const float4* q) {
          const float4 r0 = q[0], r1 = q[1], r2 = q[2];
          const f2 nz(r0.x, r0.y), PAx(r0.z, r0.w), PAy(r2.x, r2.y), PAz(r2.z, r2.w);
          const f2 PCx = PAx + ACx, PCy = PAy + ACy, PCz = PAz + ACz;
          f2 S[C::L + 1];
          boys_seeds_f32<C::L>(nz * fma(PCx, PCx, fma(PCy, PCy, PCz * PCz)), f2(r1.x, r1.y), f2(r1.z, r1.w), tab, S);
          f2 kp(0.f), nsg(0.f);
          if (C::L > 0) {
            const float4 r3 = q[3];
            kp = f2(r3.x, r3.y);
            nsg = f2(r3.z, r3.w);
          }
          if (kEarly) {
            OsCoef<f2> c;
            c.c10 = nsg;
            c.c20 = nsg * nsg;
            c.c01 = kp;
            C::prim(S, c, M);
          } else {
            C::vrr(S, PAx, PAy, PAz, PCx, PCy, PCz, kp, f2(2.0f) * kp, f2(3.0f) * kp, acc);
          }
        };
        const int ppn = s_ppn[r];
        if (ppn <= kStage) {
#pragma unroll 1
          for (int q = 0; q < ppn; ++q) prim(rec + kRF4 * q);
        } else {  // more primitive pairs than staged: global memory
          const float4* pp = a.prims_f32 + (size_t)s_ppo[r] * kPrimF4;
          for (int q = 0; q < ppn; ++q) prim(pp + kPrimF4 * q);
        }
        if (kEarly) C::build(M, ABx, ABy, ABz, -ACx, -ACy, -ACz, acc);  // powers of -sigma in M
        f2 xi[NA * NB];
        C::hrr(acc, ABx, ABy, ABz, xi);
#pragma unroll
        for (int d = 0; d < ND; ++d)
#pragma unroll
          for (int u = 0; u < NA; ++u)
#pragma unroll
            for (int v = 0; v < NB; ++v) ga[d][u] = fma(xi[u * NB + v], fb[d][v], ga[d][u]);
        if (sa != s_sb[r]) {
          const int colb = s_cb[r];
#pragma unroll
          for (int d = 0; d < ND; ++d)
#pragma unroll
            for (int v = 0; v < NB; ++v) {
              f2 g(0.f);
#pragma unroll
              for (int u = 0; u < NA; ++u) g = fma(xi[u * NB + v], fa[d][u], g);
              gadd(d, colb + v, g);
            }
        }
      };
      if constexpr (RING) {
        // the warp's 64 points of every F column: 256 contiguous, 16-byte
        // aligned bytes (foff32, ldq and i0 are multiples of 128 floats, and
        // the columns are ldq >= i0 + 128 long)
        const float* Fw = a.ws32 + s_bd.foff32 + iw;
        // pair r into the next slot: its records (at most kStage primitive
        // pairs; longer contractions are read from global memory) and its
        // F_b columns, one bulk copy each, all on the slot's barrier.  The
        // slot was last read by this warp's lanes before the __syncwarp that
        // precedes every call.
        auto issue = [&](int r) {
          if (lane == 0) {
            const int sl = prod % kRing;
            uint64_t* bar = &s_full[wid][sl];
            const int ppn = s_ppn[r];
            const uint32_t rec_bytes = ppn <= kStage ? 16u * kPrimF4 * (uint32_t)ppn : 0u;
            fence_proxy_async_smem();
            mbar_expect_tx(bar, rec_bytes + ND * NB * 256);
            if (rec_bytes) bulk_copy(s_ring[wid][sl], a.prims_f32 + (size_t)s_ppo[r] * kPrimF4, rec_bytes, bar);
            float* fdst = reinterpret_cast<float*>(s_ring[wid][sl] + kRecF4);
            const int cb = s_cb[r];
#pragma unroll
            for (int d = 0; d < ND; ++d)
#pragma unroll
              for (int v = 0; v < NB; ++v)
                bulk_copy(fdst + (d * NB + v) * 64, Fw + d * dstr + (int64_t)(cb + v) * ldq, 256, bar);
          }
          ++prod;
        };
        for (int r = 0; r < min(nrun, kRing); ++r) issue(r);
        for (int r = 0; r < nrun; ++r) {
          const int sl = cons % kRing;
          const bool ok = __all_sync(0xffffffffu, mbar_wait(&s_full[wid][sl], (cons / kRing) & 1u, a.err,
                                                            kCopyWaitNs));
          ++cons;
          if (!ok) {
            // give up: no further work in this CTA; wait (bounded again) for
            // the copies still in flight into this warp's ring, then leave
            s_abort = 1;
            for (uint32_t q = cons - 1; q < prod; ++q)
              mbar_wait(&s_full[wid][q % kRing], (q / kRing) & 1u, nullptr, kCopyWaitNs);
            cons = prod;
            break;
          }
          const float* fsl = reinterpret_cast<const float*>(s_ring[wid][sl] + kRecF4);
          f2 fb[ND][NB];
#pragma unroll
          for (int d = 0; d < ND; ++d)
#pragma unroll
            for (int v = 0; v < NB; ++v) fb[d][v] = f2(fsl[(d * NB + v) * 64 + lane], fsl[(d * NB + v) * 64 + 32 + lane]);
          compute(r, s_ring[wid][sl], fb);
          __syncwarp();  // every lane is done with slot sl: it takes pair r + kRing
          if (r + kRing < nrun) issue(r + kRing);
        }
      } else {
        constexpr int kRecL = (kRecF4 + 31) / 32;  // float4 of a pair's records per lane
        auto rec_load = [&](int r, float4 (&pre)[kRecL]) {
          const int n4 = min(s_ppn[r], kStage) * kRF4;
          const float4* src = a.prims_f32 + (size_t)s_ppo[r] * kPrimF4;
#pragma unroll
          for (int m = 0; m < kRecL; ++m) {
            const int e = lane + 32 * m;
            if (e < n4) pre[m] = src[(e / kRF4) * kPrimF4 + e % kRF4];
          }
          return n4;
        };
        auto rec_store = [&](int buf, int n4, const float4 (&pre)[kRecL]) {
#pragma unroll
          for (int m = 0; m < kRecL; ++m)
            if (lane + 32 * m < n4) s_pr[RING ? 0 : wid][buf][lane + 32 * m] = pre[m];
          __syncwarp();
        };
        float4 pre[kRecL];
        rec_store(0, rec_load(0, pre), pre);
        f2 fn[ND][NB];
#pragma unroll
        for (int d = 0; d < ND; ++d)
#pragma unroll
          for (int v = 0; v < NB; ++v) fn[d][v] = fload(d, s_cb[0] + v);
        for (int r = 0; r < nrun; ++r) {
          // the next pair's records and F are in flight while this pair computes
          const int n4 = r + 1 < nrun ? rec_load(r + 1, pre) : 0;
          f2 fb[ND][NB];
#pragma unroll
          for (int d = 0; d < ND; ++d)
#pragma unroll
            for (int v = 0; v < NB; ++v) {
              fb[d][v] = fn[d][v];
              if (r + 1 < nrun) fn[d][v] = fload(d, s_cb[r + 1] + v);
            }
          compute(r, s_pr[RING ? 0 : wid][r & 1], fb);
          // every lane is past its reads of the other buffer (the previous
          // iteration's closing __syncwarp), so it can take the next records
          rec_store((r + 1) & 1, n4, pre);
        }
      }
      if (cur >= 0) {
#pragma unroll
        for (int d = 0; d < ND; ++d)
#pragma unroll
          for (int u = 0; u < NA; ++u) gadd(d, cola + u, ga[d][u]);
      }
    }  // steps of the tile's list
  }
}

// ---------------------------------------------------------------- double-FP32 pairs (mixed form)

// Constants of the ds Boys evaluation as (hi, lo) float pairs, rounded at
// compile time: 1/m! for the e^x Taylor series, then 1/(2n+1).
struct DsConst {
  float hi, lo;
};
#define SNK_DS_C(v) {(float)(v), (float)((v) - (double)(float)(v))}
__constant__ DsConst c_ds_invfact[8] = {SNK_DS_C(1.0),         SNK_DS_C(1.0),         SNK_DS_C(1.0 / 2.0),
                                        SNK_DS_C(1.0 / 6.0),   SNK_DS_C(1.0 / 24.0),  SNK_DS_C(1.0 / 120.0),
                                        SNK_DS_C(1.0 / 720.0), SNK_DS_C(1.0 / 5040.0)};
__constant__ DsConst c_ds_inv_odd[kBoysLMax + 1] = {SNK_DS_C(1.0), SNK_DS_C(1.0 / 3.0), SNK_DS_C(1.0 / 5.0),
                                                    SNK_DS_C(1.0 / 7.0), SNK_DS_C(1.0 / 9.0)};
#undef SNK_DS_C

__device__ __forceinline__ ds ds_ld(const float2* p) {
  const float2 v = *p;
  return ds_make(v.x, v.y);
}

__device__ __forceinline__ ds ds_c(const DsConst& c) { return ds_make(c.hi, c.lo); }

// S_n = pref F_n(T), n = 0..L, in ds arithmetic: an 8-term
// Taylor expansion about the nearest node of the 0.1-spaced table (nodes
// rounded to ds-representable values, so T_k - T is exact to ds precision),
// the downward recursion with e^{-T} = e^{-T_k} e^{x}, and the asymptotic
// form above T = 50 with a ds reciprocal square root.
//
// Taylor sums c_0 + c_1 x + ... + c_7 x^7 with |x| <= 0.05 and c_m >= 0 falling
// like 1/m!: the terms from x^5 on are below 0.05^5/5! = 2.6e-9 of the sum, so
// plain FP32 leaves them at 2^-52 of it; in the other steps the coefficient is
// at least five times the product, so the leading parts add error-free in
// three operations (Dekker) instead of six, and only the end renormalises.  49
// operations instead of 105, with fewer roundings.  With the squares of P - r summed
// unnormalised and no product with 1/(2n+1) = 1, the tier went from 333 to 275
// ms per build (96 atoms, 768,000 points; dd 122 -> 89, ps 39.5 -> 34.3).
struct DsRow {
  const float2* p;
  __device__ __forceinline__ float2 operator()(int m) const { return p[m]; }
};
struct DsInvFact {
  __device__ __forceinline__ float2 operator()(int m) const { return make_float2(c_ds_invfact[m].hi, c_ds_invfact[m].lo); }
};
template <class Coef>
__device__ __forceinline__ ds ds_taylor(const Coef& c, ds x) {
  const float g = fmaf(fmaf(c(7).x, x.hi, c(6).x), x.hi, c(5).x);
  ds f = ds_make(g, 0.f);
#pragma unroll
  for (int m = 4; m >= 0; --m) {
    const float2 cm = c(m);
    const float p = __fmul_rn(f.hi, x.hi);
    float e = __fmaf_rn(f.hi, x.hi, -p);
    e = __fmaf_rn(f.hi, x.lo, e);
    if (m < 4) e = __fmaf_rn(f.lo, x.hi, e);
    const float sum = __fadd_rn(cm.x, p);
    f = ds_make(sum, __fadd_rn(__fsub_rn(p, __fsub_rn(sum, cm.x)), __fadd_rn(e, cm.y)));
  }
  return ds_fast_two_sum(f.hi, f.lo);
}

template <int L>
__device__ __forceinline__ void boys_seeds_ds(ds T, ds pref, ds pref_far, const float2* tab, ds* S) {
  if (T.hi < (float)kBoysTMax) {
    const int k = __float2int_rn(T.hi * (float)(1.0 / kBoysHDs));
    const float2* row = tab + k * kBoysColsDs;
    const ds x = ds_ld(row + kBoysColsDs - 1) - T;  // T_k - T, |x| <= 0.05
    S[L] = pref * ds_taylor(DsRow{row}, x);
    if (L > 0) {
      const ds pe = (pref * ds_ld(row + kBoysTermsDs)) * ds_taylor(DsInvFact{}, x);
      const ds T2 = ds_make(2.0f * T.hi, 2.0f * T.lo);
#pragma unroll
      for (int n = L - 1; n >= 0; --n) {
        S[n] = fma(T2, S[n + 1], pe);
        if (n > 0) S[n] = S[n] * ds_c(c_ds_inv_odd[n]);
      }
    }
  } else {
    const ds r = ds_rsqrt(T);
    S[0] = pref_far * r;
    if (L > 0) {
      const ds o = (r * r) * 0.5f;
#pragma unroll
      for (int n = 0; n < L; ++n) S[n + 1] = S[n] * (o * (float)(2 * n + 1));
    }
  }
}

// Contracted Xi_ab of one pair at the point c in ds arithmetic; the primitive
// pair data are the host-split (hi, lo) copies of PrimPair; A is the centre of
// shell a.
template <int LA, int LB>
__device__ __forceinline__ void pair_xi_ds(const PairHdr& h, const float2* __restrict__ prims,
                                           const float2* __restrict__ ab, const float2* __restrict__ A,
                                           const float2* tab, ds cx, ds cy, ds cz, ds* xi) {
  using C = OsClass<LA, LB>;
  ds M[C::NM];
#pragma unroll
  for (int k = 0; k < C::NM; ++k) M[k] = ds_make(0.f, 0.f);
  // in blocks of 16 primitive pairs, the sums of a longer contraction renormalised in
  // between (a test of q in the inner loop costs the tier 1.3 %, also where it never holds)
  for (int q = 0;;) {
    const int q1 = min(q + 16, h.pp_n);
#pragma unroll 1
    for (; q < q1; ++q) {
      // two (hi, lo) pairs per load; the class reads what its L needs
      const float4* pp = reinterpret_cast<const float4*>(prims + (size_t)(h.pp_off + q) * kPrimWords);
      auto first = [](float4 v) { return ds_make(v.x, v.y); };
      auto second = [](float4 v) { return ds_make(v.z, v.w); };
      const float4 r0 = pp[0], r1 = pp[1], r2 = pp[2];
      const ds PCx = second(r0) - cx, PCy = first(r1) - cy, PCz = second(r1) - cz;
      const ds T = first(r0) * ds_norm2_raw(PCx, PCy, PCz);
      ds S[C::L + 1];
      boys_seeds_ds<C::L>(T, first(r2), second(r2), tab, S);
      OsCoef<ds> c;
      if (C::L >= 1) {
        const float4 r3 = pp[3];
        c.c10 = first(r3);
        c.c20 = second(r3);
      }
      if (C::L >= 3) {
        const float4 r4 = pp[4];
        c.c30 = first(r4);
        c.c40 = second(r4);
      }
      if (C::L >= 2) {
        const float4 r5 = pp[5];
        c.c01 = first(r5);
        c.c11 = second(r5);
      }
      if (C::L >= 4) {
        const float4 r6 = pp[6];
        c.c21 = first(r6);
        c.c02 = second(r6);
      }
      C::prim(S, c, M);
    }
    if (q >= h.pp_n) break;
#pragma unroll
    for (int k = 0; k < C::NM; ++k) acc_renorm(M[k]);
  }
  const ds ABx = ds_ld(ab), ABy = ds_ld(ab + 1), ABz = ds_ld(ab + 2);
  ds acc[C::NACC];
  C::build(M, -ABx, -ABy, -ABz, cx - ds_ld(A), cy - ds_ld(A + 1), cz - ds_ld(A + 2), acc);
  C::hrr(acc, ABx, ABy, ABz, xi);
}

// The FP64 lists of the mixed form in ds arithmetic: same tiles, tickets,
// contraction and FP64 G atomics as integral_kernel; F is read in FP64 and
// split, each G update is rounded to FP64 once.  Bound by the FP32 FMA pipe
// (70-80 % busy), dd by instruction fetch: its recursion, HRR and contraction
// are about 5,000 straight-line instructions (80 KB), and warps in different
// places of it evict each other's lines.  There the CTA's warps start every
// pair together (a barrier per pair, block-uniform; threads past the batch's
// points compute the last point and add nothing): 96 atoms, 768,000 points, dd
// 89.6 -> 66.1 ms.  dp gains nothing from it (66.4 / 66.6).
template <int LA, int LB, int ND>
__global__ void __launch_bounds__(kIntThreads) integral_kernel_ds(IntegralArgs a) {
  using C = OsClass<LA, LB>;
  constexpr int NA = C::NA, NB = C::NB;
  constexpr bool kLockstep = C::L == 4;
  extern __shared__ float2 s_tab2[];
  const float2* gtab = a.boys_ds + (size_t)C::L * kBoysRowsDs * kBoysColsDs;
  for (int e = threadIdx.x; e < kBoysRowsDs * kBoysColsDs; e += blockDim.x) s_tab2[e] = gtab[e];
  __shared__ int s_tile;
  __syncthreads();
  for (;;) {
    if (threadIdx.x == 0) s_tile = atomicAdd(a.ticket, 1);
    __syncthreads();
    const int t = s_tile;
    __syncthreads();
    if (t >= a.n_tiles * a.part_n) break;
    const Tile tile = tile_part(a, t);
    const BatchDesc bd = a.batches[tile.batch];
    int i = tile.i0 + threadIdx.x;
    const bool act = i < bd.q;
    if (!kLockstep && !act) continue;
    if (!act) i = bd.q - 1;
    const int64_t ldq = bd.ldq, dstr = (int64_t)bd.ldq * bd.nS;
    const ds cx = ds_from(a.xyz[3 * (bd.p0 + i)]), cy = ds_from(a.xyz[3 * (bd.p0 + i) + 1]),
             cz = ds_from(a.xyz[3 * (bd.p0 + i) + 2]);
    const double* F = a.ws + bd.foff + i;
    double* G = a.ws + bd.goff + a.gshift + (t / a.n_tiles) * a.gpart + i;
    const int* cmap = a.colmap + bd.cm_off - bd.ms0;
    ds ga[ND][NA], fa[ND][NA];
    int cur = -1, cola = 0;
    // act holds for every thread here but in lockstep
    auto gadd = [&](int d, int col, ds v) {
      if (act) atomicAdd(G + d * dstr + col * ldq, ds_to(v));
    };
    for (int k = tile.k0; k < tile.k1; ++k) {
      if (kLockstep) __syncthreads();
      const int p = a.pairlist[k];
      const PairHdr h = a.pairs[p];
      if (h.sa != cur) {
        if (cur >= 0) {
#pragma unroll
          for (int d = 0; d < ND; ++d)
#pragma unroll
            for (int u = 0; u < NA; ++u) gadd(d, cola + u, ga[d][u]);
        }
        cur = h.sa;
        cola = cmap[cur];
#pragma unroll
        for (int d = 0; d < ND; ++d)
#pragma unroll
          for (int u = 0; u < NA; ++u) {
            ga[d][u] = ds_make(0.f, 0.f);
            fa[d][u] = ds_from(F[d * dstr + (cola + u) * ldq]);
          }
      }
      const int colb = cmap[h.sb];
      if (cola < 0 || colb < 0) continue;  // cannot happen: the screen marks both shells of a kept pair
      ds fb[ND][NB];
#pragma unroll
      for (int d = 0; d < ND; ++d)
#pragma unroll
        for (int v = 0; v < NB; ++v) fb[d][v] = ds_from(F[d * dstr + (colb + v) * ldq]);
      ds xi[NA * NB];
      pair_xi_ds<LA, LB>(h, a.prims_ds, a.pair_ab + 4 * (size_t)p, a.pair_a + 4 * (size_t)p, s_tab2, cx, cy, cz, xi);
#pragma unroll
      for (int d = 0; d < ND; ++d)
#pragma unroll
        for (int u = 0; u < NA; ++u) {
#pragma unroll
          for (int v = 0; v < NB; ++v) acc_mac(ga[d][u], xi[u * NB + v], fb[d][v]);
          acc_renorm(ga[d][u]);  // a run of pairs of one shell a can have thousands of terms
        }
      if (h.sa != h.sb) {
#pragma unroll
        for (int d = 0; d < ND; ++d)
#pragma unroll
          for (int v = 0; v < NB; ++v) {
            ds g = ds_make(0.f, 0.f);
#pragma unroll
            for (int u = 0; u < NA; ++u) acc_mac(g, xi[u * NB + v], fa[d][u]);
            gadd(d, colb + v, g);
          }
      }
    }
    if (cur >= 0) {
#pragma unroll
      for (int d = 0; d < ND; ++d)
#pragma unroll
        for (int u = 0; u < NA; ++u) gadd(d, cola + u, ga[d][u]);
    }
  }
}

// Training labels of the learned screen, from the plain FP64 integrals: for
// every list entry (batch j, pair ab) of the sampled batches, the sums over
// the batch's points of |dG_u(i)| max_nu |Phi_{nu i}|, dG_u the block's
// contribution to G row u of shell a (slots 0..5) or b (slots 6..11): an
// upper bound of the block's contribution to K-tilde row u.  Same tiles as
// integral_kernel.
template <int LA, int LB>
__global__ void __launch_bounds__(kIntThreads) label_kernel(IntegralArgs a, const int64_t* __restrict__ slot_base,
                                                            const int64_t* __restrict__ list_off,
                                                            const double* __restrict__ xm,
                                                            float* __restrict__ lab) {
  using C = OsClass<LA, LB>;
  constexpr int NA = C::NA, NB = C::NB;
  extern __shared__ double s_tab[];
  const double* gtab = a.boys + (size_t)C::L * kBoysRows * kBoysCols;
  for (int e = threadIdx.x; e < kBoysRows * kBoysCols; e += blockDim.x) s_tab[e] = gtab[e];
  __shared__ int s_tile;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  for (;;) {
    if (threadIdx.x == 0) s_tile = atomicAdd(a.ticket, 1);
    __syncthreads();
    const int t = s_tile;
    __syncthreads();
    if (t >= a.n_tiles) break;
    const Tile tile = a.tiles[t];
    const BatchDesc bd = a.batches[tile.batch];
    const int i = tile.i0 + threadIdx.x;
    const bool active = i < bd.q;
    const int64_t ldq = bd.ldq;
    const double cx = active ? a.xyz[3 * (bd.p0 + i)] : 0.0, cy = active ? a.xyz[3 * (bd.p0 + i) + 1] : 0.0,
                 cz = active ? a.xyz[3 * (bd.p0 + i) + 2] : 0.0;
    const double* F = a.ws + bd.foff + (active ? i : 0);
    const int* cmap = a.colmap + bd.cm_off - bd.ms0;
    const int64_t s0 = slot_base[tile.batch] - list_off[(int64_t)tile.batch * kNumLists];
    for (int k = tile.k0; k < tile.k1; ++k) {
      const PairHdr h = a.pairs[a.pairlist[k]];
      const int cola = cmap[h.sa], colb = cmap[h.sb];
      float part[NA + NB];
#pragma unroll
      for (int u = 0; u < NA + NB; ++u) part[u] = 0.f;
      if (active && cola >= 0 && colb >= 0) {
        double xi[NA * NB], fa[NA], fb[NB];
#pragma unroll
        for (int u = 0; u < NA; ++u) fa[u] = F[(cola + u) * ldq];
#pragma unroll
        for (int v = 0; v < NB; ++v) fb[v] = F[(colb + v) * ldq];
        pair_xi<LA, LB>(h, a.prims, a.shell_xyz + 3 * h.sa, s_tab, cx, cy, cz, xi);
#pragma unroll
        for (int u = 0; u < NA; ++u) {
          double g = 0.0;
#pragma unroll
          for (int v = 0; v < NB; ++v) g = fma(xi[u * NB + v], fb[v], g);
          part[u] = (float)(fabs(g) * xm[bd.p0 + i]);
        }
        if (h.sa != h.sb) {
#pragma unroll
          for (int v = 0; v < NB; ++v) {
            double g = 0.0;
#pragma unroll
            for (int u = 0; u < NA; ++u) g = fma(xi[u * NB + v], fa[u], g);
            part[NA + v] = (float)(fabs(g) * xm[bd.p0 + i]);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < NA + NB; ++u) {
        float s = part[u];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0 && s > 0.f) atomicAdd(&lab[(s0 + k) * 12 + (u < NA ? u : 6 + (u - NA))], s);
      }
    }
  }
}

// One shell pair's block at n points, by the recursion for every primitive pair
// about its own centre P.  The contracted form of the builds takes P - A as
// -sigma AB; the two differ by the rounding of P, about 1e-16 |R_p|, which only
// shows in blocks that vanish by symmetry.  A few launches of latency, so the
// operation count does not matter here.
template <int LA, int LB>
__global__ void debug_xi_kernel(const PairHdr* pair, const PrimPair* prims, const double* shell_xyz,
                                const double* boys, int64_t n, const double* xyz, double* out) {
  using C = OsClass<LA, LB>;
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double* tab = boys + (size_t)C::L * kBoysRows * kBoysCols;
  const PairHdr h = *pair;
  const double* A = shell_xyz + 3 * h.sa;
  const double cx = xyz[3 * i], cy = xyz[3 * i + 1], cz = xyz[3 * i + 2];
  double acc[C::NACC];
#pragma unroll
  for (int k = 0; k < C::NACC; ++k) acc[k] = 0.0;
  for (int q = 0; q < h.pp_n; ++q) {
    const PrimPair pp = prims[h.pp_off + q];
    const double PCx = pp.Px - cx, PCy = pp.Py - cy, PCz = pp.Pz - cz;
    const double T = pp.zeta * fma(PCx, PCx, fma(PCy, PCy, PCz * PCz));
    double S[C::L + 1];
    boys_seeds<C::L>(T, tab, S);
    for (int m = 0; m <= C::L; ++m) S[m] *= pp.pref;
    const double kappa = 0.5 / pp.zeta;
    C::vrr(S, pp.Px - A[0], pp.Py - A[1], pp.Pz - A[2], PCx, PCy, PCz, kappa, 2.0 * kappa, 3.0 * kappa, acc);
  }
  double xi[C::NA * C::NB];
  C::hrr(acc, h.ABx, h.ABy, h.ABz, xi);
  for (int k = 0; k < C::NA * C::NB; ++k) out[i * C::NA * C::NB + k] = xi[k];
}

template <int L>
__device__ void boys_row(double T, const double* boys, double* out) {
  double S[L + 1];
  boys_seeds<L>(T, boys + (size_t)L * kBoysRows * kBoysCols, S);
  for (int n = 0; n <= L; ++n) out[n] = S[n];
}

__global__ void debug_boys_kernel(const double* boys, int64_t n, const double* T, int nmax, double* out) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  double* o = out + i * (nmax + 1);
  switch (nmax) {
    case 0: boys_row<0>(T[i], boys, o); break;
    case 1: boys_row<1>(T[i], boys, o); break;
    case 2: boys_row<2>(T[i], boys, o); break;
    case 3: boys_row<3>(T[i], boys, o); break;
    default: boys_row<4>(T[i], boys, o); break;
  }
}

constexpr size_t kSmem64 = sizeof(double) * kBoysRows * kBoysCols;
constexpr size_t kSmemDs = sizeof(float2) * kBoysRowsDs * kBoysColsDs;
constexpr size_t kSmem32 = sizeof(float) * kBoysRowsF * kBoysColsF;

// list < kNumClasses: FP64 kernel of that class; otherwise the FP32 kernel of
// class list - kNumClasses.
template <class K>
cudaError_t launch_kernel(K kernel, size_t smem, cudaStream_t st, const IntegralArgs& a, int grid,
                          int threads = kIntThreads) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kernel<<<grid, threads, smem, st>>>(a);
  return cudaGetLastError();
}

template <int LA, int LB, int ND>
cudaError_t launch_class_nd(cudaStream_t st, bool f32, const IntegralArgs& a, int grid) {
  if (f32) return launch_kernel(integral_kernel_f32<LA, LB, ND>, kSmem32, st, a, grid, kF32Threads);
  if (a.hi_ds) return launch_kernel(integral_kernel_ds<LA, LB, ND>, kSmemDs, st, a, grid);
  return launch_kernel(integral_kernel<LA, LB, ND>, kSmem64, st, a, grid);
}

template <int LA, int LB>
cudaError_t launch_class(cudaStream_t st, bool f32, const IntegralArgs& a, int grid) {
  return a.n_dens == 2 ? launch_class_nd<LA, LB, 2>(st, f32, a, grid) : launch_class_nd<LA, LB, 1>(st, f32, a, grid);
}

template <class K>
int ctas_for(K kernel, size_t smem, int num_sms, int threads = kIntThreads) {
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess || per_sm < 1)
    per_sm = 1;
  return per_sm * num_sms;
}

template <int LA, int LB, int ND>
int max_ctas_nd(bool f32, bool ds, int num_sms) {
  return f32  ? ctas_for(integral_kernel_f32<LA, LB, ND>, kSmem32, num_sms, kF32Threads)
         : ds ? ctas_for(integral_kernel_ds<LA, LB, ND>, kSmemDs, num_sms)
              : ctas_for(integral_kernel<LA, LB, ND>, kSmem64, num_sms);
}

template <int LA, int LB>
int max_ctas(bool f32, bool ds, int nd, int num_sms) {
  return nd == 2 ? max_ctas_nd<LA, LB, 2>(f32, ds, num_sms) : max_ctas_nd<LA, LB, 1>(f32, ds, num_sms);
}

}  // namespace

cudaError_t launch_integrals(cudaStream_t st, int list, const IntegralArgs& a, int grid_ctas) {
  if (a.n_tiles == 0) return cudaSuccess;
  const bool f32 = list >= kNumClasses;
  switch (list % kNumClasses) {
    case 0: return launch_class<0, 0>(st, f32, a, grid_ctas);
    case 1: return launch_class<1, 0>(st, f32, a, grid_ctas);
    case 2: return launch_class<1, 1>(st, f32, a, grid_ctas);
    case 3: return launch_class<2, 0>(st, f32, a, grid_ctas);
    case 4: return launch_class<2, 1>(st, f32, a, grid_ctas);
    case 5: return launch_class<2, 2>(st, f32, a, grid_ctas);
  }
  return cudaErrorInvalidValue;
}

int integral_max_ctas(int list, int num_sms, bool ds, int n_dens) {
  const bool f32 = list >= kNumClasses;
  switch (list % kNumClasses) {
    case 0: return max_ctas<0, 0>(f32, ds, n_dens, num_sms);
    case 1: return max_ctas<1, 0>(f32, ds, n_dens, num_sms);
    case 2: return max_ctas<1, 1>(f32, ds, n_dens, num_sms);
    case 3: return max_ctas<2, 0>(f32, ds, n_dens, num_sms);
    case 4: return max_ctas<2, 1>(f32, ds, n_dens, num_sms);
    case 5: return max_ctas<2, 2>(f32, ds, n_dens, num_sms);
  }
  return num_sms;
}

cudaError_t launch_labels(cudaStream_t st, int cls, const IntegralArgs& a, int grid, const int64_t* slot_base,
                          const int64_t* list_off, const double* xm, float* lab) {
  if (a.n_tiles == 0) return cudaSuccess;
#define SNK_LAB(A, B)                                                                                       \
  {                                                                                                         \
    cudaError_t e =                                                                                         \
        cudaFuncSetAttribute(label_kernel<A, B>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem64); \
    if (e != cudaSuccess) return e;                                                                         \
    label_kernel<A, B><<<grid, kIntThreads, kSmem64, st>>>(a, slot_base, list_off, xm, lab);              \
    break;                                                                                                  \
  }
  switch (cls) {
    case 0: SNK_LAB(0, 0)
    case 1: SNK_LAB(1, 0)
    case 2: SNK_LAB(1, 1)
    case 3: SNK_LAB(2, 0)
    case 4: SNK_LAB(2, 1)
    case 5: SNK_LAB(2, 2)
    default: return cudaErrorInvalidValue;
  }
#undef SNK_LAB
  return cudaGetLastError();
}

cudaError_t launch_debug_A(cudaStream_t st, int cls, const PairHdr* pair, const PrimPair* prims,
                           const double* shell_xyz, const double* boys, int64_t n, const double* xyz, double* xi) {
  if (n == 0) return cudaSuccess;
  const int th = 128;
  const unsigned blocks = (unsigned)((n + th - 1) / th);
  switch (cls) {
    case 0: debug_xi_kernel<0, 0><<<blocks, th, 0, st>>>(pair, prims, shell_xyz, boys, n, xyz, xi); break;
    case 1: debug_xi_kernel<1, 0><<<blocks, th, 0, st>>>(pair, prims, shell_xyz, boys, n, xyz, xi); break;
    case 2: debug_xi_kernel<1, 1><<<blocks, th, 0, st>>>(pair, prims, shell_xyz, boys, n, xyz, xi); break;
    case 3: debug_xi_kernel<2, 0><<<blocks, th, 0, st>>>(pair, prims, shell_xyz, boys, n, xyz, xi); break;
    case 4: debug_xi_kernel<2, 1><<<blocks, th, 0, st>>>(pair, prims, shell_xyz, boys, n, xyz, xi); break;
    case 5: debug_xi_kernel<2, 2><<<blocks, th, 0, st>>>(pair, prims, shell_xyz, boys, n, xyz, xi); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_debug_boys(cudaStream_t st, const double* boys, int64_t n, const double* T, int nmax,
                              double* out) {
  if (n == 0) return cudaSuccess;
  const int th = 128;
  debug_boys_kernel<<<(unsigned)((n + th - 1) / th), th, 0, st>>>(boys, n, T, nmax, out);
  return cudaGetLastError();
}

// Algorithmic flops per (grid point, contracted shell pair), FMA = 2: per primitive
// pair the T evaluation (8), the Boys seeds counted at the cheaper large-T form (1
// for L = 0, else 3 + 2L; the library rsqrt is not counted) and what the tier's form
// does for it, the contraction into the scalars or (FP32 tier but for ps and ds) the
// whole recursion; per contracted pair the rest, VRR and HRR or HRR alone, and the G_a
// contraction (2 NA NB).  FP64 pairs of uncontracted shells count like the others.
// The G_b half of off-diagonal pairs is not counted.
void class_flops(int cls, bool f32, double* per_prim, double* per_pair) {
  int prim = 0, pair = 0, L = 0, na = 1, nb = 1;
  switch (cls) {
#define SNK_CASE(c, A, B)                                                                   \
  case c: {                                                                                 \
    const bool first = !f32 || f32_early(A, B);                                             \
    prim = first ? OsClass<A, B>::PRIM_FLOPS : OsClass<A, B>::VRR_FLOPS;                    \
    pair = first ? OsClass<A, B>::PAIR_FLOPS : OsClass<A, B>::HRR_FLOPS;                    \
    L = OsClass<A, B>::L;                                                                   \
    na = OsClass<A, B>::NA;                                                                 \
    nb = OsClass<A, B>::NB;                                                                 \
    break;                                                                                  \
  }
    SNK_CASE(0, 0, 0)
    SNK_CASE(1, 1, 0)
    SNK_CASE(2, 1, 1)
    SNK_CASE(3, 2, 0)
    SNK_CASE(4, 2, 1)
    SNK_CASE(5, 2, 2)
#undef SNK_CASE
  }
  const double boys = L == 0 ? 1.0 : 3.0 + 2.0 * L;
  *per_prim = 8.0 + boys + prim;
  *per_pair = pair + 2.0 * na * nb;
}

}  // namespace snk
