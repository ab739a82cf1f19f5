// Nuclear gradient of E = 1/2 tr(DJ) - 1/4 tr(DK) with D fixed (SI Sec. 1.4).
//
// Only bra derivatives are needed when the sum runs over every ordered pair
// of shell pairs (SI Eq. si_dE_J, si_dE_K).  Folding the four orderings inside
// the bra and ket pairs into one term gives, per ordered (bra pair, ket pair)
// item with shells (a b | c d),
//   dE/dR += w sum_{mu nu lam sig} G_{mu nu lam sig} d(mu nu|lam sig)/dR_bra,
//   G = 4 D_mn D_ls - D_ml D_ns - D_ms D_nl,  w = 1/2^[a=b] 1/2^[c=d].
// The bra derivative follows SI Eq. si_pair_derivative: in direction tau,
//   d/dA_tau: coefficient of Lambda_t is (a/p) E_{t-1} + E^{(1)}_t,
//   d/dB_tau: coefficient of Lambda_t is (b/p) E_{t-1} - E^{(1)}_t,
// with E^{(1)} = dE/dDelta_tau from the recurrence SI Eq. si_dE_recursion and
// base E^{00,(1)}_0 = 2a (P-A)_tau (the exp(-ab/p |AB|^2) factor of E^{00}_0
// lives in the pair prefactor).  Hermite indices run one higher than for the
// energy, so R goes to L+1 (the paper raises one bra angular momentum, SI Sec. 2).
// E^{(1)} needs no recurrence of its own: P and p held fixed, E^{ij}_t depends on
// Delta through P-A = -(b/p) Delta, P-B = (a/p) Delta and the exponential, and
// dE^{ij}_t/d(P-A) = i E^{i-1,j}_t, dE^{ij}_t/d(P-B) = j E^{i,j-1}_t, so
//   E^{(1)ij}_t = 2a (P-A) E^{ij}_t - (b/p) i E^{i-1,j}_t + (a/p) j E^{i,j-1}_t.
// With gP_tau = sum E_P W_{P+1_tau} (the pair moves as a whole) and gR_tau =
// sum E^{(1)}_P W_P, dE/dA = (a/p) gP + gR and dE/dB = (b/p) gP - gR per
// primitive pair.  The density factor is summed over the ket components first,
//   V^{ab}_P = sum_cd G_{ab,cd} W_P[cd],
// for the Hermite indices that ab needs (at most one direction raised), so the
// derivative sums run once per ab and not once per (ab, cd): about half the
// FP64 operations of differentiating every (ab|cd).
//
// Two kernels, in FP64 or (mixed precision: items below tau, split on the
// device as for the energy) in FP32 with each item's sums added in FP64: one
// item per thread with everything in registers for the small classes, one item
// per block for the others (see kernels_c.cuh for the cost model).  Both are bound
// by the FP64 pipe (FP32: shared memory).  Measured on GB300, mixed gradient of
// 135 functions: 634 ms with one item per warp, 32 ms now; one (ff|ff) item 22 ms
// with one warp.
#pragma once
#include "kernels_c.cuh"

namespace eri {

struct GradArgs {
  PairData pd;
  ShellPairInfo sp;
  WorkList wl;  // ordered (J-engine) list
  BoysTabs bt;
  const RStep* rsteps;
  const double* Dp;
  const float* Dpf;    // D' in FP32 for the FP32 tier
  const double* ea;    // exponent of the s1 primitive of each primitive pair
  const int* sh_atom;
  double* grad;        // natom * 3 (all molecules' atoms)
  double cj, ck;       // weights of the Coulomb and exchange parts (1 or 0)
  double omega2;       // erf(omega r)/r: omega^2 (0 = Coulomb)
  float omega2f;
  int det;             // 1: fixed-point gradient accumulator (deterministic builds)
  unsigned long long* counter;  // items, primitive quartets, bra primitives of this launch (may be null)
  // mixed precision: this tier's compacted list (bra position, ket position) written
  // by the tier split, *nitems of them; null: items are positions in wl
  const int2* items;
  const unsigned int* nitems;
};

template <> __device__ __forceinline__ double om2<double, GradArgs>(const GradArgs& a) { return a.omega2; }
template <> __device__ __forceinline__ float om2<float, GradArgs>(const GradArgs& a) { return a.omega2f; }
template <typename T> __device__ __forceinline__ const T* gdens(const GradArgs& a);
template <> __device__ __forceinline__ const double* gdens<double>(const GradArgs& a) { return a.Dp; }
template <> __device__ __forceinline__ const float* gdens<float>(const GradArgs& a) { return a.Dpf; }

// dE/dA and dE/dB of direction d.  Of two shells on one atom the sum: the parts that
// move the shells against each other cancel in it and not in the gradient's rounding.
__device__ __forceinline__ void add_pair(const GradArgs& a, int d, int atA, int atB, double x, double y) {
  acc_add(a.grad + 3 * atA + d, atA == atB ? x + y : x, a.det);
  if (atA != atB) acc_add(a.grad + 3 * atB + d, y, a.det);
}

// ---------------------------------------------------------------------------
// one item per thread
// ---------------------------------------------------------------------------

// Values per thread that the register form keeps at once (W, G and R); beyond
// the register file they are lane-interleaved local memory, which costs little
// beside the FP64 pipe.
__host__ __device__ constexpr int grad_footprint(int la, int lb, int lc, int ld) {
  const int ncd = ncart(lc) * ncart(ld);
  return ncd * nherm(la + lb + 1) + ncart(la) * ncart(lb) * ncd + nherm(la + lb + lc + ld + 1);
}
// (235 and 330: the classes above were faster by item and block)
#ifndef ERI_GRAD_THREAD64
#define ERI_GRAD_THREAD64 235
#endif
#ifndef ERI_GRAD_THREAD32
#define ERI_GRAD_THREAD32 330
#endif
__host__ __device__ constexpr bool use_grad_thread(int la, int lb, int lc, int ld, bool fp32) {
  // (a large bra against (ss|: little work per thread and long code; a block is faster)
  return grad_footprint(la, lb, lc, ld) <= (fp32 ? ERI_GRAD_THREAD32 : ERI_GRAD_THREAD64) &&
         !(lc + ld == 0 && ncart(la) * ncart(lb) > 18);
}

// FP64 thread classes with long code run a block per item while the list is short
// (see block_when_short)
template <int LA, int LB, int LC, int LD, typename T>
__host__ __device__ constexpr bool grad_block_when_short() {
  return sizeof(T) == 8 && grad_footprint(LA, LB, LC, LD) >= 100;
}

// dE/dA and dE/dB of one item, bra primitives [pb0, pb1) and ket primitives [pk0, pk1)
template <int LA, int LB, int LC, int LD, typename T>
__device__ __forceinline__ void grad_item(const GradArgs& a, int pb_id, int pk_id, int mol, int pb0, int pb1, int pk0,
                                          int pk1, T* gA, T* gB) {
  constexpr int LAB = LA + LB, LCD = LC + LD, L = LAB + LCD + 1, NA = ncart(LA), NB = ncart(LB), NC = ncart(LC),
                ND = ncart(LD), NCD = NC * ND, HAB = nherm(LAB + 1);
  constexpr int NEB = (LA + 1) * (LB + 1) * (LAB + 1), NEK = (LC + 1) * (LD + 1) * (LCD + 1);
  const int offb = __ldg(a.sp.poff + pb_id), eb0 = __ldg(a.sp.eoff + pb_id);
  const int offk = __ldg(a.sp.poff + pk_id), ek0 = __ldg(a.sp.eoff + pk_id);
  T G[NA * NB * NCD];
  {
    const int ao1 = __ldg(a.sp.ao1 + pb_id), ao2 = __ldg(a.sp.ao2 + pb_id);
    const int ao3 = __ldg(a.sp.ao1 + pk_id), ao4 = __ldg(a.sp.ao2 + pk_id);
    const int n = __ldg(a.sp.mat_n + mol);
    const T* Dp = gdens<T>(a) + __ldg(a.sp.mat_off + mol);
    T w = T(1);
    if (__ldg(a.sp.s1 + pb_id) == __ldg(a.sp.s2 + pb_id)) w *= T(0.5);
    if (__ldg(a.sp.s1 + pk_id) == __ldg(a.sp.s2 + pk_id)) w *= T(0.5);
    const T cj = T(4.0 * a.cj) * w, ck = T(a.ck) * w;
#pragma unroll
    for (int x = 0; x < NA; ++x)
#pragma unroll
      for (int y = 0; y < NB; ++y) {
        const T dab = cj * __ldg(Dp + (size_t)(ao1 + x) * n + ao2 + y);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const T dac = ck * __ldg(Dp + (size_t)(ao1 + x) * n + ao3 + c);
          const T dbc = ck * __ldg(Dp + (size_t)(ao2 + y) * n + ao3 + c);
#pragma unroll
          for (int d = 0; d < ND; ++d)
            G[(x * NB + y) * NCD + c * ND + d] =
                dab * __ldg(Dp + (size_t)(ao3 + c) * n + ao4 + d) -
                (dac * __ldg(Dp + (size_t)(ao2 + y) * n + ao4 + d) + __ldg(Dp + (size_t)(ao1 + x) * n + ao4 + d) * dbc);
        }
      }
  }
  for (int pb = pb0; pb < pb1; ++pb) {
    Prim<T> bp;
    bp.load(a.pd, offb + pb);
    T W[NCD * HAB];
#pragma unroll
    for (int x = 0; x < NCD * HAB; ++x) W[x] = T(0);
    for (int pk = pk0; pk < pk1; ++pk) {
      Prim<T> kp;
      kp.load(a.pd, offk + pk);
      T ek[3 * NEK];
      load_or_build_e<LC, LD, T>(a.pd, ek0 + pk * 3 * NEK, kp, ek);
      T rho, rs;
      quartet_rho(bp.p, kp.p, rho, rs);
      T pref = bp.pref * kp.pref * rs;
      attenuate(om2<T>(a), rho, pref);  // s depends on exponents only: the derivative rules hold as they are
      const T PQx = bp.P[0] - kp.P[0], PQy = bp.P[1] - kp.P[1], PQz = bp.P[2] - kp.P[2];
      T F[L + 1];
      Boys<T>::template eval<L>(rho * (PQx * PQx + PQy * PQy + PQz * PQz), a.bt, F);
      T R[nherm(L)];
      r_build_reg<L, T>(F, pref, PQx, PQy, PQz, T(-2) * rho, R);
      for_cart<LC>([&](auto kx, auto ky, auto kz) {
        for_cart<LD>([&](auto lx, auto ly, auto lz) {
          constexpr int KX = ERI_CI(kx), KY = ERI_CI(ky), KZ = ERI_CI(kz);
          constexpr int LX = ERI_CI(lx), LY = ERI_CI(ly), LZ = ERI_CI(lz);
          constexpr int icd = cidx(LC, KY, KZ) * ND + cidx(LD, LY, LZ);
          const T* ex = ek + 0 * NEK + (KX * (LD + 1) + LX) * (LCD + 1);
          const T* ey = ek + 1 * NEK + (KY * (LD + 1) + LY) * (LCD + 1);
          const T* ez = ek + 2 * NEK + (KZ * (LD + 1) + LZ) * (LCD + 1);
          for_herm<LAB + 1>([&](auto t, auto u, auto v) {
            T& w = W[icd * HAB + herm_index(ERI_CI(t), ERI_CI(u), ERI_CI(v))];
            w = ket_term<L, KX + LX, KY + LY, KZ + LZ, ERI_CI(t), ERI_CI(u), ERI_CI(v)>(ex, ey, ez, R, w);
          });
        });
      });
    }
    T e[3 * NEB], e1[3 * NEB];
    load_or_build_e<LA, LB, T>(a.pd, eb0 + pb * 3 * NEB, bp, e);
    const T ea = (T)__ldg(a.ea + offb + pb), aop = ea / bp.p, bop = T(1) - aop;
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int i = 0; i <= LA; ++i)
#pragma unroll
        for (int j = 0; j <= LB; ++j)
#pragma unroll
          for (int t = 0; t <= i + j; ++t) {
            const int r = d * NEB + (i * (LB + 1) + j) * (LAB + 1) + t;
            T v = T(2) * ea * bp.PA[d] * e[r];
            if (i > 0 && t < i + j) v = fma(-bop * T(i), e[r - (LB + 1) * (LAB + 1)], v);
            if (j > 0 && t < i + j) v = fma(aop * T(j), e[r - (LAB + 1)], v);
            e1[r] = v;
          }
    T gP[3] = {T(0), T(0), T(0)}, gR[3] = {T(0), T(0), T(0)};
    for_cart<LA>([&](auto ix, auto iy, auto iz) {
      for_cart<LB>([&](auto jx, auto jy, auto jz) {
        constexpr int IX = ERI_CI(ix), IY = ERI_CI(iy), IZ = ERI_CI(iz);
        constexpr int JX = ERI_CI(jx), JY = ERI_CI(jy), JZ = ERI_CI(jz);
        constexpr int iab = cidx(LA, IY, IZ) * NB + cidx(LB, JY, JZ);
        constexpr int NX = IX + JX, NY = IY + JY, NZ = IZ + JZ;
        const T* ex = e + 0 * NEB + (IX * (LB + 1) + JX) * (LAB + 1);
        const T* ey = e + 1 * NEB + (IY * (LB + 1) + JY) * (LAB + 1);
        const T* ez = e + 2 * NEB + (IZ * (LB + 1) + JZ) * (LAB + 1);
        const T *fx = e1 + (ex - e), *fy = e1 + (ey - e), *fz = e1 + (ez - e);
        T V[HAB];
        sfor<NX + 2>([&](auto tx) {
          sfor<NY + 2>([&](auto ty) {
            sfor<NZ + 2>([&](auto tz) {
              constexpr int t = ERI_CI(tx), u = ERI_CI(ty), v = ERI_CI(tz);
              if constexpr ((t > NX) + (u > NY) + (v > NZ) <= 1) {
                constexpr int P = herm_index(t, u, v);
                T s = T(0);
#pragma unroll
                for (int cd = 0; cd < NCD; ++cd) s = fma(G[iab * NCD + cd], W[cd * HAB + P], s);
                V[P] = s;
              }
            });
          });
        });
        auto at = [&](auto t, auto u, auto v) { return V[herm_index(ERI_CI(t), ERI_CI(u), ERI_CI(v))]; };
        sfor<NX + 2>([&](auto t) {
          const T s = tsum<0, NY, NZ, false>(ex, ey, ez, [&](auto, auto u, auto v) { return at(t, u, v); });
          constexpr int x = ERI_CI(t);
          if constexpr (x > 0) gP[0] = NX == 0 ? gP[0] + s : fma(ex[x - 1], s, gP[0]);
          if constexpr (x <= NX) gR[0] = fma(fx[x], s, gR[0]);
        });
        sfor<NY + 2>([&](auto u) {
          const T s = tsum<NX, 0, NZ, false>(ex, ey, ez, [&](auto t, auto, auto v) { return at(t, u, v); });
          constexpr int x = ERI_CI(u);
          if constexpr (x > 0) gP[1] = NY == 0 ? gP[1] + s : fma(ey[x - 1], s, gP[1]);
          if constexpr (x <= NY) gR[1] = fma(fy[x], s, gR[1]);
        });
        sfor<NZ + 2>([&](auto v) {
          const T s = tsum<NX, NY, 0, false>(ex, ey, ez, [&](auto t, auto u, auto) { return at(t, u, v); });
          constexpr int x = ERI_CI(v);
          if constexpr (x > 0) gP[2] = NZ == 0 ? gP[2] + s : fma(ez[x - 1], s, gP[2]);
          if constexpr (x <= NZ) gR[2] = fma(fz[x], s, gR[2]);
        });
      });
    });
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      gA[d] += fma(aop, gP[d], gR[d]);
      gB[d] += fma(bop, gP[d], -gR[d]);
    }
  }
}

// SHORT: the form for short lists, a group of lanes per item (see prim_split)
template <int LA, int LB, int LC, int LD, typename T, bool SHORT>
__global__ void __launch_bounds__(128) grad_thread_kernel(GradArgs a) {
  const bool compact = a.items != nullptr;
  const int64_t total = compact ? (int64_t)__ldg(a.nitems) : a.wl.total;
  const int64_t first = compact ? 0 : a.wl.first;
  const int nshard = compact ? 1 : a.wl.nshard, shard = compact ? 0 : a.wl.shard;
  const int lane = threadIdx.x & 31;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const PrimSplit sp = prim_split<T>(a.wl, total - first, 32 * nwarps, SHORT ? SplitBy::lanes : SplitBy::parts);
  // items a warp takes at a time; this lane's of them, and its place in the item's group
  const int per = SHORT ? 32 / sp.g : 32, li = SHORT ? lane / sp.g : lane, sub = SHORT ? lane % sp.g : 0;
  const unsigned lanes = SHORT ? group_lanes(sp.g, li) : 0u;
  const int64_t span = SHORT ? per : 32 * thread_tile(a.wl, total - first, nwarps),
                ntiles = (total - first + span - 1) / span;
  unsigned long long done = 0, doneq = 0, doneb = 0;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  for (int64_t turn = 0; turn * nwarps * nshard < ntiles * sp.n; ++turn) {
    const int64_t tl = warp_tile(turn, warp, nwarps) * nshard + shard;
    if (tl >= ntiles * sp.n) continue;
    const int part = (int)(tl / ntiles);
    const int64_t t0 = first + (tl - part * ntiles) * span, i1 = t0 + span < total ? t0 + span : total;
    BraCursor cur;
    if (!compact) cur.seek(a.wl, t0 + li < i1 ? t0 + li : t0);
    for (int64_t base = t0; base < i1; base += per) {  // uniform over the warp
      const int64_t item = base + li;
      const bool ok = item < i1;
      T gA[3] = {T(0), T(0), T(0)}, gB[3] = {T(0), T(0), T(0)};
      int atA = -1, atB = -1;
      if (ok) {
        int ib, ik;
        if (compact) {
          const int2 v = __ldg(a.items + item);
          ib = v.x;
          ik = v.y;
        } else {
          ik = cur.at(a.wl, item);
          ib = cur.ib;
        }
        const int pb_id = __ldg(a.wl.bra + ib), mol = __ldg(a.sp.pmol + pb_id);
        const int seg = __ldg(a.wl.kseg + mol * NPAIRCLASS);
        if (!compact) ik = ket_pos(a.wl, seg, ik, cur.be - cur.bs);
        const int pk_id = __ldg(a.wl.ket + seg + ik);
        const int npb = __ldg(a.sp.np + pb_id), npk = __ldg(a.sp.np + pk_id);
        if (part == 0 && sub == 0) {
          ++done;
          doneq += (unsigned long long)npb * npk;
          doneb += npb;
        }
        atA = __ldg(a.sh_atom + __ldg(a.sp.s1 + pb_id));
        atB = __ldg(a.sh_atom + __ldg(a.sp.s2 + pb_id));
        int pb0, pb1, pk0, pk1;
        sp.range(part, sub, npb, npk, pb0, pb1, pk0, pk1);
        if (pb0 < pb1 && pk0 < pk1) grad_item<LA, LB, LC, LD, T>(a, pb_id, pk_id, mol, pb0, pb1, pk0, pk1, gA, gB);
      }
      if constexpr (SHORT)
        if (ok) {  // the item's sums, in the first lane of its group
          group_sum<3>(gA, sp.g, sub, lanes);
          group_sum<3>(gB, sp.g, sub, lanes);
          if (sub != 0)
#pragma unroll
            for (int d = 0; d < 3; ++d) gA[d] = gB[d] = T(0);
        }
      // the lists are bra-major: a warp's items usually share the two atoms, and
      // their sums go out as one atomic each (deterministic builds keep one
      // fixed-point add per item, whose sum does not depend on the grouping)
      const int a0 = __shfl_sync(0xffffffffu, atA, 0), b0 = __shfl_sync(0xffffffffu, atB, 0);
      if (!a.det && __all_sync(0xffffffffu, !ok || (atA == a0 && atB == b0))) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          double x = (double)gA[d], y = (double)gB[d];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            x += __shfl_xor_sync(0xffffffffu, x, o);
            y += __shfl_xor_sync(0xffffffffu, y, o);
          }
          if (lane == 0) {
            atomicAdd(a.grad + 3 * a0 + d, a0 == b0 ? x + y : x);  // (see add_pair)
            if (a0 != b0) atomicAdd(a.grad + 3 * b0 + d, y);
          }
        }
      } else if (ok && sub == 0) {
#pragma unroll
        for (int d = 0; d < 3; ++d) add_pair(a, d, atA, atB, (double)gA[d], (double)gB[d]);
      }
    }
  }
  if (a.counter && done) {
    atomicAdd(a.counter, done);
    atomicAdd(a.counter + 1, doneq);
    atomicAdd(a.counter + 2, doneb);
  }
}

// ---------------------------------------------------------------------------
// one item per block
// ---------------------------------------------------------------------------

// V tasks of a bra pair class: the Hermite indices each ab needs, rounded up to
// pairs per ab
__host__ __device__ constexpr int grad_needed(int nx, int ny, int nz) {
  return (nx + 1) * (ny + 1) * (nz + 1) + (ny + 1) * (nz + 1) + (nx + 1) * (nz + 1) + (nx + 1) * (ny + 1);
}
__host__ __device__ constexpr int grad_tasks(int la, int lb) {
  int s = 0;
  for (int c = 0; c < ncart(la) * ncart(lb); ++c) {
    int ix = 0, iy = 0, iz = 0, jx = 0, jy = 0, jz = 0;
    cart_xyz(la, c / ncart(lb), ix, iy, iz);
    cart_xyz(lb, c % ncart(lb), jx, jy, jz);
    s += (grad_needed(ix + jx, iy + jy, iz + jz) + 1) / 2 * 2;
  }
  return s;
}

template <int LA, int LB, int LC, int LD, typename T>
struct GShape {
  static constexpr int LAB = LA + LB, LCD = LC + LD, L = LAB + LCD + 1;
  static constexpr int NA = ncart(LA), NB = ncart(LB), NC = ncart(LC), ND = ncart(LD);
  static constexpr int NAB = NA * NB, NCD = NC * ND, HAB = nherm(LAB + 1), HABP = HAB | 1;
  static constexpr int B = L + 1, BOX = B * B * B, NP = nherm(L - 1), NSC = L + 5;
  static constexpr int TK = pair_terms(LC, LD), NV = grad_tasks(LA, LB);
  static constexpr int RL = LAB + 3;  // E rows: t = -1 .. LAB + 1, zero outside 0 .. i + j
  static constexpr int NEB = (LA + 1) * (LB + 1) * (LAB + 1), NER = (LA + 1) * (LB + 1) * RL,
                       NEK = (LC + 1) * (LD + 1) * (LCD + 1);
  static constexpr int NDB = (NA + NB) * (NC + ND) + NAB + NCD;
  static constexpr int PER_G = BOX + 2 * NP + TK;
  // G is held whole, or (where that would not fit) in NH parts of the bra pairs
  static constexpr int REST = NCD * HABP + 6 * NER + kWin * NSC + NDB + 48;
  static constexpr size_t TABLES = 4 * (size_t)(TK + NV + NCD + 1 + 2 * NAB + 1) + 2 * (TK + HAB + 2) + NCD;
  static constexpr int NH = sizeof(T) * (size_t)(REST + PER_G + NAB * NCD + 4) + TABLES <= 226 * 1024 ? 1 : 2;
  static constexpr int NABH = (NAB + NH - 1) / NH;
  static constexpr int FIXED = REST + NABH * NCD;
  static constexpr int GT = (LC <= 1 && LD <= 1) ? 9 : (LC <= 1 || LD <= 1) ? 3 : 1;
  static constexpr int ROOM = (48 * 1024 / (int)sizeof(T) - FIXED) / PER_G;
  static constexpr int G = ROOM < 1 ? 1 : (ROOM > GT ? GT : ROOM);
  static constexpr int NT = NAB * NCD >= 1500 ? 256 : 128;
  static constexpr int TOTAL = (FIXED + G * PER_G + 3) / 4 * 4;
  static constexpr size_t smem() { return sizeof(T) * TOTAL + TABLES; }
};

template <int LA, int LB, int LC, int LD, typename T>
__global__ void __launch_bounds__(GShape<LA, LB, LC, LD, T>::NT) grad_block_kernel(GradArgs a) {
  using S = GShape<LA, LB, LC, LD, T>;
  constexpr int LAB = S::LAB, LCD = S::LCD, L = S::L, B = S::B, NA = S::NA, NB = S::NB, NC = S::NC, ND = S::ND,
                NAB = S::NAB, NCD = S::NCD, HAB = S::HAB, HABP = S::HABP, G = S::G, NT = S::NT, RL = S::RL;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  T* Ws = reinterpret_cast<T*>(smraw);  // [NCD][HABP]
  T* Gs = Ws + NCD * HABP;              // [NABH][NCD]
  T* box = Gs + S::NABH * NCD;          // [G][BOX]
  T* ping = box + G * S::BOX;           // [G][2][NP]
  T* ek = ping + G * 2 * S::NP;         // [G][TK]
  T* er = ek + G * S::TK;               // E [3][NER], then E1 [3][NER]
  T* scal = er + 6 * S::NER;            // [kWin][NSC]
  T* db = scal + kWin * S::NSC;         // D' blocks: [a+b][c+d], [ab], [cd]
  T* red = db + S::NDB;                 // [6][8]
  int* ks = reinterpret_cast<int*>(Ws + S::TOTAL);         // [NCD + 1]
  unsigned* kt = reinterpret_cast<unsigned*>(ks + NCD + 1);  // [TK]
  unsigned* vt = kt + S::TK;            // [NV]: ab | P << 8 | t << 16 | u << 20 | v << 24, ~0: none
  unsigned* abr = vt + S::NV;           // [NAB]: E row offsets x | y << 10 | z << 20
  int* vs = reinterpret_cast<int*>(abr + NAB);             // [NAB + 1]: first task of ab
  uint16_t* ko = reinterpret_cast<uint16_t*>(vs + NAB + 1);  // [TK]
  uint16_t* pbox = ko + S::TK;          // [HAB]
  build_terms<LC, LD, LCD + 1>(ks, kt, ko, [](int t, int u, int v) { return (t * B + u) * B + v; });
  for (int i = tid; i < HAB; i += NT) pbox[i] = (uint16_t)((herm_t(i) * B + herm_u(i)) * B + herm_v(i));
  uint8_t* cdo = reinterpret_cast<uint8_t*>(pbox + HAB);  // [NCD]: order of the tasks
  order_by_terms<NCD>(ks, cdo);
  auto powers = [](int m, int* x, int* y) {
    cart_xyz(LA, m / NB, x[0], x[1], x[2]);
    cart_xyz(LB, m % NB, y[0], y[1], y[2]);
  };
  block_starts<NAB>(vs, [&](int m) {
    int x[3], y[3];
    powers(m, x, y);
    return (grad_needed(x[0] + y[0], x[1] + y[1], x[2] + y[2]) + 1) / 2 * 2;
  });
  if (tid < NAB) {
    int x[3], y[3];
    powers(tid, x, y);
    abr[tid] = (unsigned)((x[0] * (LB + 1) + y[0]) * RL) | (unsigned)((x[1] * (LB + 1) + y[1]) * RL) << 10 |
               (unsigned)((x[2] * (LB + 1) + y[2]) * RL) << 20;
    const int nx = x[0] + y[0], ny = x[1] + y[1], nz = x[2] + y[2];
    int k = vs[tid];
    for (int t = 0; t <= nx + 1; ++t)
      for (int u = 0; u <= ny + 1; ++u)
        for (int v = 0; v <= nz + 1; ++v)
          if ((t > nx) + (u > ny) + (v > nz) <= 1)
            vt[k++] = (unsigned)tid | (unsigned)herm_index(t, u, v) << 8 | (unsigned)t << 16 | (unsigned)u << 20 |
                      (unsigned)v << 24;
    if (k < vs[tid + 1]) vt[k] = 0xffffffffu;
  }
  const bool compact = a.items != nullptr;
  const int64_t total = compact ? (int64_t)__ldg(a.nitems) : a.wl.total;
  const int64_t first = compact ? 0 : a.wl.first;
  const int nshard = compact ? 1 : a.wl.nshard, shard = compact ? 0 : a.wl.shard;
  unsigned long long done = 0, doneq = 0, doneb = 0;
  const int64_t tile = item_tile(a.wl, total - first, gridDim.x), ntiles = (total - first + tile - 1) / tile;
  T gA[3] = {T(0), T(0), T(0)}, gB[3] = {T(0), T(0), T(0)};
  int atA = -1, atB = -1;
  // sum the threads' gA, gB and add them to the two atoms (whole block)
  auto flush = [&]() {
    __syncthreads();
#pragma unroll
    for (int d = 0; d < 6; ++d) {
      T v = d < 3 ? gA[d % 3] : gB[d % 3];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) red[d * 8 + wp] = v;
    }
    __syncthreads();
    if (tid < 3) {
      double v = 0.0, u = 0.0;
      for (int x = 0; x < NT / 32; ++x) {
        v += (double)red[tid * 8 + x];
        u += (double)red[(tid + 3) * 8 + x];
      }
      add_pair(a, tid, atA, atB, v, u);
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) gA[d] = gB[d] = T(0);
  };
  const PrimSplit sp = prim_split<T>(a.wl, total - first, gridDim.x, SplitBy::blocks);
  for (int64_t tl = (int64_t)blockIdx.x * nshard + shard; tl < ntiles * sp.n; tl += (int64_t)gridDim.x * nshard) {
    const int part = (int)(tl / ntiles);
    const int64_t t0 = first + (tl - part * ntiles) * tile, t1 = t0 + tile < total ? t0 + tile : total;
    BraCursor cur;
    if (!compact) cur.seek(a.wl, t0);
    for (int64_t item = t0; item < t1; ++item) {
      int ib, ik;
      if (compact) {
        const int2 v = __ldg(a.items + item);
        ib = v.x;
        ik = v.y;
      } else {
        ik = cur.at(a.wl, item);
        ib = cur.ib;
      }
      const int pb_id = __ldg(a.wl.bra + ib);
      const int mol = __ldg(a.sp.pmol + pb_id);
      const int pk_id = __ldg(a.wl.ket + __ldg(a.wl.kseg + mol * NPAIRCLASS) + ik);
      const int s1 = __ldg(a.sp.s1 + pb_id), s2 = __ldg(a.sp.s2 + pb_id);
      const int npb = __ldg(a.sp.np + pb_id), offb = __ldg(a.sp.poff + pb_id), eb0 = __ldg(a.sp.eoff + pb_id);
      const int npk = __ldg(a.sp.np + pk_id), offk = __ldg(a.sp.poff + pk_id), ek0 = __ldg(a.sp.eoff + pk_id);
      const int ao1 = __ldg(a.sp.ao1 + pb_id), ao2 = __ldg(a.sp.ao2 + pb_id);
      const int ao3 = __ldg(a.sp.ao1 + pk_id), ao4 = __ldg(a.sp.ao2 + pk_id);
      if (part == 0) {
        ++done;
        doneq += (unsigned long long)npb * npk;
        doneb += npb;
      }
      int pb0, pb1, pk0, pk1;
      sp.range(part, 0, npb, npk, pb0, pb1, pk0, pk1);
      if (pb0 >= pb1 || npk == 0) continue;  // uniform over the block; W has no value without a ket primitive
      // items of a tile usually share the bra atoms: their sums go out together
      // (FP32 sums and deterministic builds: once per item)
      const int nA = __ldg(a.sh_atom + s1), nB = __ldg(a.sh_atom + s2);
      if (atA >= 0 && (sizeof(T) == 4 || a.det || nA != atA || nB != atB)) flush();
      atA = nA;
      atB = nB;
      T w = T(1);
      if (s1 == s2) w *= T(0.5);
      if (__ldg(a.sp.s1 + pk_id) == __ldg(a.sp.s2 + pk_id)) w *= T(0.5);
      const T cj = T(4.0 * a.cj) * w, ck = T(a.ck) * w;
      const int n = __ldg(a.sp.mat_n + mol);
      const T* Dp = gdens<T>(a) + __ldg(a.sp.mat_off + mol);
      __syncthreads();  // the previous item's shared memory (first item: the tables) is done with
      for (int x = tid; x < S::NDB; x += NT) {
        int r, c;
        if (x < (NA + NB) * (NC + ND)) {
          const int i = x / (NC + ND), j = x - i * (NC + ND);
          r = i < NA ? ao1 + i : ao2 + i - NA;
          c = j < NC ? ao3 + j : ao4 + j - NC;
        } else if (x < (NA + NB) * (NC + ND) + NAB) {
          const int i = x - (NA + NB) * (NC + ND);
          r = ao1 + i / NB;
          c = ao2 + i % NB;
        } else {
          const int i = x - (NA + NB) * (NC + ND) - NAB;
          r = ao3 + i / ND;
          c = ao4 + i % ND;
        }
        db[x] = __ldg(Dp + (size_t)r * n + c);
      }
      // G of the bra pairs [m0, m0 + NABH)
      auto density = [&](int m0) {
        const T* dab = db + (NA + NB) * (NC + ND);
        const T* dcd = dab + NAB;
        const int nm = min(S::NABH, NAB - m0);
        for (int x = tid; x < nm * NCD; x += NT) {
          const int ab = m0 + x / NCD, cd = x % NCD;
          const T* ra = db + (ab / NB) * (NC + ND);
          const T* rb = db + (NA + ab % NB) * (NC + ND);
          const int c = cd / ND, d = NC + cd % ND;
          Gs[x] = cj * dab[ab] * dcd[cd] - ck * (ra[c] * rb[d] + ra[d] * rb[c]);
        }
      };
      if constexpr (S::NH == 1) {
        __syncthreads();
        density(0);
      }
      const int nq = pb1 * npk;
      int win = 0, wend = 0;
      for (int pb = pb0; pb < pb1; ++pb) {
        const int ipb = offb + pb;
        const T ea = (T)__ldg(a.ea + ipb), aop = ea / pdv<T>(a.pd.p, a.pd.pf, ipb), bop = T(1) - aop;
        for (int x = tid; x < 3 * S::NER; x += NT) {  // E and E1 rows, zero-padded
          const int d = x / S::NER, r = x - d * S::NER, row = r / RL, t = r - row * RL - 1;
          const int i = row / (LB + 1), j = row - i * (LB + 1);
          T v = T(0), v1 = T(0);
          if (t >= 0 && t <= i + j) {
            const int e = eb0 + pb * 3 * S::NEB + d * S::NEB + row * (LAB + 1) + t;
            v = ldE<T>(a.pd, e);
            v1 = T(2) * ea * pdv<T>(a.pd.PA, a.pd.PAf, d * a.pd.n + ipb) * v;
            if (t < i + j) {
              if (i > 0) v1 = fma(-bop * T(i), ldE<T>(a.pd, e - (LB + 1) * (LAB + 1)), v1);
              if (j > 0) v1 = fma(aop * T(j), ldE<T>(a.pd, e - (LAB + 1)), v1);
            }
          }
          er[x] = v;
          er[3 * S::NER + x] = v1;
        }
        for (int k0 = 0; k0 < npk;) {
          const int q = pb * npk + k0;
          if (q >= wend) {  // uniform over the block
            win = q;
            quartet_scalars<L, T>(a, q, nq, npk, offb, offk, scal);
            wend = min(nq, q + kWin);
          }
          const int ng = min(min(G, npk - k0), wend - q);
          for (int x = tid; x < ng * S::TK; x += NT) {
            const int g = x / S::TK, k = x - g * S::TK;
            const unsigned wd = kt[k];
            const int e = ek0 + (k0 + g) * 3 * S::NEK, ox = wd & 1023, oy = (wd >> 10) & 1023, oz = wd >> 20;
            const T v = ldE<T>(a.pd, e + ox) * ldE<T>(a.pd, e + oy) * ldE<T>(a.pd, e + oz);
            ek[x] = (ox % (LCD + 1) + oy % (LCD + 1) + oz % (LCD + 1)) & 1 ? -v : v;
          }
          __syncthreads();
          r_build_block<L, T>(scal + (q - win) * S::NSC, ng, a.rsteps, ping, box);
          __syncthreads();
          constexpr int HH = (HAB + 1) / 2;
          for (int it = tid; it < NCD * HH; it += NT) {
            const int row = it / HH, cd = cdo[row], P = it - row * HH, P2 = P + HH < HAB ? P + HH : P;
            const int s0 = ks[cd], s1k = ks[cd + 1];
            T x0 = T(0), x1 = T(0);
            for (int g = 0; g < ng; ++g) {
              const T* e = ek + g * S::TK;
              const T* r0 = box + g * S::BOX + pbox[P];
              const T* r1 = box + g * S::BOX + pbox[P2];
#pragma unroll 4
              for (int k = s0; k < s1k; ++k) {
                const T c = e[k];
                const int o = ko[k];
                x0 = fma(c, r0[o], x0);
                x1 = fma(c, r1[o], x1);
              }
            }
            T* wr = Ws + cd * HABP;
            if (k0 == 0) {
              wr[P] = x0;
              if (P2 != P) wr[P2] = x1;
            } else {
              wr[P] += x0;
              if (P2 != P) wr[P2] += x1;
            }
          }
          __syncthreads();
          k0 += ng;
        }
        T gP[3] = {T(0), T(0), T(0)}, gR[3] = {T(0), T(0), T(0)};
#pragma unroll 1
        for (int h = 0; h < S::NH; ++h) {
          const int m0 = h * S::NABH;
          if constexpr (S::NH > 1) {
            if (h > 0) __syncthreads();
            density(m0);
            __syncthreads();
          }
          const int v0 = vs[m0], v1 = vs[min(NAB, m0 + S::NABH)];
          for (int it = v0 / 2 + tid; it < v1 / 2; it += NT) {
            const unsigned e0 = vt[2 * it], e1 = vt[2 * it + 1];
            const int ab = e0 & 255;
            const bool two = e1 != 0xffffffffu;
            const T* g = Gs + (ab - m0) * NCD;
            const T* w0 = Ws + ((e0 >> 8) & 255);
            const T* w1 = two ? Ws + ((e1 >> 8) & 255) : w0;
            T x[2] = {T(0), T(0)};
#pragma unroll 4
            for (int cd = 0; cd < NCD; ++cd) {
              const T c = g[cd];
              x[0] = fma(c, w0[cd * HABP], x[0]);
              x[1] = fma(c, w1[cd * HABP], x[1]);
            }
            const unsigned ar = abr[ab];
            const T* bx = er + (ar & 1023) + 1;
            const T* by = er + S::NER + ((ar >> 10) & 1023) + 1;
            const T* bz = er + 2 * S::NER + (ar >> 20) + 1;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              const unsigned e = k ? e1 : e0;
              if (k && !two) break;
              const int t = (e >> 16) & 15, u = (e >> 20) & 15, v = e >> 24;
              const T ex = bx[t], ey = by[u], ez = bz[v];
              const T vx = x[k] * ey * ez, vy = x[k] * ex * ez, vz = x[k] * ex * ey;
              gP[0] = fma(bx[t - 1], vx, gP[0]);
              gP[1] = fma(by[u - 1], vy, gP[1]);
              gP[2] = fma(bz[v - 1], vz, gP[2]);
              gR[0] = fma(bx[3 * S::NER + t], vx, gR[0]);
              gR[1] = fma(by[3 * S::NER + u], vy, gR[1]);
              gR[2] = fma(bz[3 * S::NER + v], vz, gR[2]);
            }
          }
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          gA[d] += fma(aop, gP[d], gR[d]);
          gB[d] += fma(bop, gP[d], -gR[d]);
        }
        __syncthreads();
      }
    }
  }
  if (atA >= 0) flush();
  if (a.counter && tid == 0 && done) {
    atomicAdd(a.counter, done);
    atomicAdd(a.counter + 1, doneq);
    atomicAdd(a.counter + 2, doneb);
  }
}

}  // namespace eri
