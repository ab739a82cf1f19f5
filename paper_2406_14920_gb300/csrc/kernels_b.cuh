// FP32 J+K kernel of the middle classes: one warp per canonical shell quartet,
// contracted ERI block staged in shared memory, both transforms written out at
// compile time.  Used for the FP32 classes that do not fit the register kernel
// (kernels_a.cuh) and whose transforms do (use_block_kernel); the larger ones
// and FP64 run a block per quartet (kernels_c.cuh).
//
// Per quartet, per bra primitive pair, the ket primitive pairs are taken G at a
// time:
//   step A  (lane g): quartet scalars for ket primitive g -- rho, P-Q, prefactor,
//           Boys F_0..F_L (Eq. boys_function); all lanes: ket E tables to smem
//           with (-1)^|Q| folded in;
//   step B  R^0 of the G primitive quartets (Eq. R_recursion), a lane per quartet
//           in registers up to L = 6, level by level over the warp above;
//   step C  lane-owned bra Hermite index P: W[cd][P] += sum_g sum_Q E'_Q^{cd}(g) R_{P+Q}(g);
// then for the bra primitive:
//   step D  lane-owned ket pair cd: X[ab][cd] += sum_P E_P^{ab} W[cd][P]   (Eq. eri_formula)
// and the contraction, one lane per output element:
//   Kh_ac, Kh_ad, Kh_bc, Kh_bd (Eq. k_definition), Jh_ab, Jh_cd (Eq. j_definition),
//   one atomic per element.
#pragma once
#include "kernels_a.cuh"

// base shared memory per warp (KB), about 16-20 warps per SM, and the upper limit
// when a larger ket-primitive batch saves a batch
#ifndef ERI_WARP_SMEM32_KB
#define ERI_WARP_SMEM32_KB 12
#endif
#ifndef ERI_WARP_SMEM32_MAX_KB
#define ERI_WARP_SMEM32_MAX_KB 16
#endif
// compile-time bra transform: largest X slice per lane, and the shared memory per
// warp a class may take to get there (measured on GB300: (fd|fp) 58 -> 9.9 ms with
// the 24 KB budget, (ff|dp) 35 -> 4.8 ms with 100-value slices)
#ifndef ERI_REGD32_MAX
#define ERI_REGD32_MAX 100
#endif
#ifndef ERI_WARP_SMEM32_FULL_KB
#define ERI_WARP_SMEM32_FULL_KB 24
#endif

namespace eri {

template <int LA, int LB, int LC, int LD, typename T>
struct BShape {
  static constexpr int LAB = LA + LB, LCD = LC + LD, L = LAB + LCD;
  static constexpr int NA = ncart(LA), NB = ncart(LB), NC = ncart(LC), ND = ncart(LD);
  static constexpr int NAB = NA * NB, NCD = NC * ND, HAB = nherm(LAB), HABP = HAB | 1;
  static constexpr int B = L + 1, BOX = B * B * B, NPING = L > 0 ? nherm(L - 1) : 1;
  static constexpr int NEB = (LA + 1) * (LB + 1) * (LAB + 1), NEK = (LC + 1) * (LD + 1) * (LCD + 1);
  static constexpr int NSC = L + 5;  // F'_0..F'_L, PQx, PQy, PQz, c
  // Shared memory per warp (elements of T).  Steps A and B cost the same per
  // batch of G ket primitives whatever G, so G should cover a ket pair's
  // primitives in as few batches as the memory allows: contracted s/p pairs
  // commonly have 9 (3 x 3), pairs with a d or f shell 3.  The budget starts at
  // BASE (occupancy) and grows up to MAX until that batch count is reached.
  static constexpr int FIXED = 3 * NEB;
  static constexpr int PER_G = BOX + 2 * NPING + NSC + 3 * NEK;
  static constexpr int PER_C = HABP + NAB;
  static constexpr int BASE = (ERI_WARP_SMEM32_KB * 1024) / 4;
  static constexpr int MAXB = (ERI_WARP_SMEM32_MAX_KB * 1024) / 4;
  static constexpr int GTARGET = (LC <= 1 && LD <= 1) ? 9 : 3;
  static constexpr int fit_g(int budget) { return (budget - FIXED - NCD * PER_C) / PER_G; }
  static constexpr int GMAXB = fit_g(MAXB) < 1 ? 1 : fit_g(MAXB);
  static constexpr int NBATCH = (GTARGET + GMAXB - 1) / GMAXB;
  static constexpr int GWANT = (GTARGET + NBATCH - 1) / NBATCH;
  static constexpr int NEED = FIXED + NCD * PER_C + GWANT * PER_G;
  static constexpr int BUDGET0 = NEED <= BASE ? BASE : (NEED <= MAXB ? NEED : MAXB);
  // classes with many ket components take a larger budget when that is
  // what lets the whole ket range sit in one pass (one ket primitive per
  // batch), the condition of the compile-time bra transform below
  static constexpr int NEED_FULL = FIXED + NCD * PER_C + PER_G;
  static constexpr bool WANT_FULL = NCD >= 8 && NAB * ((NCD + 31) / 32) <= ERI_REGD32_MAX &&
                                    NEED_FULL <= (ERI_WARP_SMEM32_FULL_KB * 1024) / 4;
  static constexpr int BUDGET = (WANT_FULL && BUDGET0 < NEED_FULL) ? NEED_FULL : BUDGET0;
  static constexpr int G0 = (BUDGET - FIXED - NCD * PER_C) / PER_G;
  static constexpr int G = G0 >= 1 ? (G0 > 16 ? 16 : G0) : 1;
  static constexpr int CHMAX = (BUDGET - FIXED - G * PER_G) / PER_C;
  static constexpr bool FITS = CHMAX >= NCD;  // the whole ket range in one pass
  // step C: lane j-slot P = lane + 32 j holds W[cd][P]
  // for every ket pair cd in registers, the cd loop unrolled at compile time
  static constexpr int NPS = (HAB + 31) / 32;
  static constexpr bool REGW = FITS && NCD * NPS <= 64;
  // step D with compile-time indices: lane owns ket pair cd = lane + 32 j, the
  // bra pairs ab are a compile-time loop (E broadcast, W row at a per-lane
  // base), X[ab][cd] stays in registers over the bra primitives.  Worth it
  // from 8 ket components up, when the X slice fits in registers (measured on
  // workload 1, FP32: (ff|pp) 17.9 -> 9.6 ms, (fd|fs) 15.8 -> 9.4 ms, against
  // the (ab, cd) item loop).
  static constexpr int NCS = (NCD + 31) / 32;
  static constexpr bool REGD = FITS && NCD >= 8 && NAB * NCS <= ERI_REGD32_MAX;
  static constexpr int SM_BOX = 0, SM_PING = SM_BOX + G * BOX, SM_SC = SM_PING + G * 2 * NPING,
                       SM_EK = SM_SC + G * NSC, SM_EB = SM_EK + G * 3 * NEK, SM_W = SM_EB + 3 * NEB,
                       SM_X = SM_W + NCD * HABP, SM_TOTAL = SM_X + NAB * NCD;
  __host__ __device__ static constexpr size_t smem_per_warp() { return sizeof(T) * SM_TOTAL; }
  // block-shared index table (ints): per bra Hermite index P its box offset and W slot
  static constexpr int TABLE_BYTES = ((4 * HAB + 15) / 16) * 16;
  __host__ __device__ static constexpr size_t table_bytes() { return TABLE_BYTES; }
};

// W is stored per cd with a "lexicographic" Hermite index (t, then u, then v)
// so that for fixed (t, u) consecutive v are consecutive: lex(t,u,v) = base(t,u) + v.
__host__ __device__ constexpr int lex_base(int lmax, int t, int u) {
  int b = 0;
  for (int x = 0; x < t; ++x) b += (lmax - x + 1) * (lmax - x + 2) / 2;
  for (int y = 0; y < u; ++y) b += lmax - t - y + 1;
  return b;
}

template <int LA, int LB, int LC, int LD, typename T>
__global__ void __launch_bounds__(128) jk_warp_kernel(JKArgs A) {
  using S = BShape<LA, LB, LC, LD, T>;
  static_assert(sizeof(T) == 4 && S::REGW && S::REGD);
  constexpr int LAB = S::LAB, LCD = S::LCD, L = S::L, B = S::B, BOX = S::BOX, NSC = S::NSC;
  constexpr int NA = S::NA, NB = S::NB, NC = S::NC, ND = S::ND, NAB = S::NAB, NCD = S::NCD, HAB = S::HAB, HABP = S::HABP,
                G = S::G, NEB = S::NEB, NEK = S::NEK, NPING = S::NPING;
  const KArgs& a = A.k;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  int* tab_p = reinterpret_cast<int*>(smraw);
  for (int i = threadIdx.x; i < HAB; i += blockDim.x) {
    const int t = herm_t(i), u = herm_u(i), v = herm_v(i);
    tab_p[i] = ((t * B + u) * B + v) | ((lex_base(LAB, t, u) + v) << 16);
  }
  __syncthreads();
  int pslot[S::NPS];  // box offset of this lane's bra Hermite indices P = lane + 32 j
#pragma unroll
  for (int j = 0; j < S::NPS; ++j) pslot[j] = lane + 32 * j < HAB ? (tab_p[lane + 32 * j] & 0xffff) : 0;
  T* sm = reinterpret_cast<T*>(smraw + S::table_bytes()) + (size_t)wib * S::SM_TOTAL;
  T* boxes = sm + S::SM_BOX;
  T* pings = sm + S::SM_PING;
  T* scal = sm + S::SM_SC;
  T* Ek = sm + S::SM_EK;
  T* Eb = sm + S::SM_EB;
  T* Ws = sm + S::SM_W;
  T* Xs = sm + S::SM_X;
  const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
  // items: positions in the work list, or (mixed precision) this tier's compacted list
  const bool compact = a.items != nullptr;
  const int64_t total = compact ? (int64_t)__ldg(a.nitems) : a.wl.total;
  const int64_t first = compact ? 0 : a.wl.first;
  const int nshard = compact ? 1 : a.wl.nshard, shard = compact ? 0 : a.wl.shard;
  unsigned long long done = 0, doneq = 0, doneb = 0;
  const int64_t tile = item_tile(a.wl, total - first, nwarps), ntiles = (total - first + tile - 1) / tile;
  for (int64_t tl = ((int64_t)blockIdx.x * (blockDim.x >> 5) + wib) * nshard + shard; tl < ntiles;
       tl += nwarps * nshard) {
  const int64_t t0 = first + tl * tile, i1 = t0 + tile < total ? t0 + tile : total;
  // the lanes locate 32 items at a time; the warp then runs them one by one
  BraCursor cur;
  if (!compact) cur.seek(a.wl, t0 + lane < i1 ? t0 + lane : t0);
  for (int64_t cq = t0; cq < i1; cq += 32) {
  int my_ib = 0, my_ik = 0;
  const bool ok = cq + lane < i1;
  if (ok) {
    if (compact) {
      const int2 v = __ldg(a.items + cq + lane);
      my_ib = v.x;
      my_ik = v.y;
    } else {
      my_ik = cur.at(a.wl, cq + lane);
      my_ib = cur.ib;
    }
  }
  unsigned pend = __ballot_sync(0xffffffffu, ok);
  while (pend) {
    const int src = __ffs(pend) - 1;
    pend &= pend - 1;
    const int ib = __shfl_sync(0xffffffffu, my_ib, src), ik = __shfl_sync(0xffffffffu, my_ik, src);
    const int pb_id = __ldg(a.wl.bra + ib);
    const int mol = __ldg(a.sp.pmol + pb_id);
    const int pk_id = __ldg(a.wl.ket + __ldg(a.wl.kseg + mol * NPAIRCLASS) + ik);
    const int s1 = __ldg(a.sp.s1 + pb_id), s2 = __ldg(a.sp.s2 + pb_id);
    const int s3 = __ldg(a.sp.s1 + pk_id), s4 = __ldg(a.sp.s2 + pk_id);
    const int npb = __ldg(a.sp.np + pb_id), offb = __ldg(a.sp.poff + pb_id), eb0 = __ldg(a.sp.eoff + pb_id);
    const int npk = __ldg(a.sp.np + pk_id), offk = __ldg(a.sp.poff + pk_id), ek0 = __ldg(a.sp.eoff + pk_id);
    ++done;
    doneq += (unsigned long long)npb * npk;
    doneb += npb;
    const int ao1 = __ldg(a.sp.ao1 + pb_id), ao2 = __ldg(a.sp.ao2 + pb_id);
    const int ao3 = __ldg(a.sp.ao1 + pk_id), ao4 = __ldg(a.sp.ao2 + pk_id);
    T w = T(1);
    if (s1 == s2) w *= T(0.5);
    if (s3 == s4) w *= T(0.5);
    if (pb_id == pk_id) w *= T(0.5);
    const int64_t mbase = __ldg(a.sp.mat_off + mol);
    const int n = __ldg(a.sp.mat_n + mol);
    const T* Dp = dens<T>(a) + mbase;
    double* Kh = a.Kh ? a.Kh + mbase : nullptr;
    double* Jh = A.Jh ? A.Jh + mbase : nullptr;

    {
      T xreg[S::NCS * NAB];
#pragma unroll
      for (int x = 0; x < S::NCS * NAB; ++x) xreg[x] = T(0);
      for (int pb = 0; pb < npb; ++pb) {
        for (int x = lane; x < 3 * NEB; x += 32) Eb[x] = ldE<T>(a.pd, eb0 + pb * 3 * NEB + x);
        T wreg[S::NPS * NCD];
#pragma unroll
        for (int x = 0; x < S::NPS * NCD; ++x) wreg[x] = T(0);
        const int ipb = offb + pb;
        const T bp_p = pdv<T>(a.pd.p, a.pd.pf, ipb), bp_pref = pdv<T>(a.pd.pref, a.pd.preff, ipb);
        const T bPx = pdv<T>(a.pd.P, a.pd.Pf, ipb), bPy = pdv<T>(a.pd.P, a.pd.Pf, a.pd.n + ipb),
                bPz = pdv<T>(a.pd.P, a.pd.Pf, 2 * a.pd.n + ipb);
        for (int k0 = 0; k0 < npk; k0 += G) {
          const int ng = npk - k0 < G ? npk - k0 : G;
          // step A: ket E tables (sign folded) and per-primitive-quartet scalars
          for (int x = lane; x < ng * 3 * NEK; x += 32) {
            const int g = x / (3 * NEK), r = x - g * 3 * NEK;
            const T v = ldE<T>(a.pd, ek0 + (k0 + g) * 3 * NEK + r);
            Ek[x] = ((r % (LCD + 1)) & 1) ? -v : v;
          }
          if (lane < ng) {
            const int ipk = offk + k0 + lane;
            const T kp = pdv<T>(a.pd.p, a.pd.pf, ipk);
            const T ps = bp_p + kp;
            T rho = bp_p * kp / ps;
            T pref = bp_pref * pdv<T>(a.pd.pref, a.pd.preff, ipk) * rsqrt_t(ps);
            attenuate(om2<T>(a), rho, pref);
            const T X = bPx - pdv<T>(a.pd.P, a.pd.Pf, ipk);
            const T Y = bPy - pdv<T>(a.pd.P, a.pd.Pf, a.pd.n + ipk);
            const T Z = bPz - pdv<T>(a.pd.P, a.pd.Pf, 2 * a.pd.n + ipk);
            T F[L + 1];
            Boys<T>::template eval<L>(rho * (X * X + Y * Y + Z * Z), a.bt, F);
            T* sc = scal + lane * NSC;
#pragma unroll
            for (int m = 0; m <= L; ++m) sc[m] = pref * F[m];
            sc[L + 1] = X;
            sc[L + 2] = Y;
            sc[L + 3] = Z;
            sc[L + 4] = T(-2) * rho;
          }
          __syncwarp();
          // step B: R^0 for the ng primitive quartets.  L <= 6: each lane
          // builds its own quartet's table in registers (compile-time indices) and
          // stores it in its box.  Otherwise the warp builds all of them level by
          // level (scaled form, see r_build_warp).
          if constexpr (L <= 6) {
            if (lane < ng) {
              const T* sc = scal + lane * NSC;
              T Fl[L + 1];
#pragma unroll
              for (int m = 0; m <= L; ++m) Fl[m] = sc[m];
              T R[nherm(L)];
              r_build_reg<L, T>(Fl, T(1), sc[L + 1], sc[L + 2], sc[L + 3], sc[L + 4], R);
              T* bx = boxes + lane * BOX;
#pragma unroll
              for (int t = 0; t <= L; ++t)
#pragma unroll
                for (int u = 0; u <= L - t; ++u)
#pragma unroll
                  for (int v = 0; v <= L - t - u; ++v) bx[(t * B + u) * B + v] = R[herm_index(t, u, v)];
            }
          } else {
            if (lane < ng) pings[lane * 2 * NPING] = scal[lane * NSC + L];
            __syncwarp();
            int cur = 0;
#pragma unroll
            for (int m = L - 1; m >= 0; --m) {
              const int ne = nherm(L - m);
              for (int it = lane; it < ng * ne; it += 32) {
                const int g = it / ne, e = it - g * ne;
                const T* sc = scal + g * NSC;
                const T* src = pings + g * 2 * NPING + cur * NPING;
                const RStep st = a.rsteps[e];
                T val;
                if (e == 0) {
                  val = sc[m];
                } else {
                  const T pq = sc[L + 1 + st.dir];
                  val = pq * src[st.dep1];
                  if (st.dep2 >= 0) val = fma((T)st.k, src[st.dep2], val);
                  val *= sc[L + 4];
                }
                if (m == 0) boxes[g * BOX + (st.t * B + st.u) * B + st.v] = val;
                else pings[g * 2 * NPING + (1 - cur) * NPING + e] = val;
              }
              __syncwarp();
              cur = 1 - cur;
            }
          }
          __syncwarp();
          // step C: ket transform; lane-owned P, every cd unrolled: R read at a
          // per-lane base plus compile-time offsets, E' broadcast, W in registers
          {
            for (int g = 0; g < ng; ++g) {
              const T* ek = Ek + g * 3 * NEK;
              const T* rbox = boxes + g * BOX;
              for_cart<LC>([&](auto kx, auto ky, auto kz) {
                for_cart<LD>([&](auto lx, auto ly, auto lz) {
                  constexpr int KX = ERI_CI(kx), KY = ERI_CI(ky), KZ = ERI_CI(kz);
                  constexpr int LX = ERI_CI(lx), LY = ERI_CI(ly), LZ = ERI_CI(lz);
                  constexpr int icd = cidx(LC, KY, KZ) * ND + cidx(LD, LY, LZ);
                  const T* ex = ek + (KX * (LD + 1) + LX) * (LCD + 1);
                  const T* ey = ek + NEK + (KY * (LD + 1) + LY) * (LCD + 1);
                  const T* ez = ek + 2 * NEK + (KZ * (LD + 1) + LZ) * (LCD + 1);
                  sfor<S::NPS>([&](auto j_) {
                    constexpr int j = ERI_CI(j_);
                    if (j * 32 + 32 <= HAB || lane + 32 * j < HAB) {
                      const T* r = rbox + pslot[j];
                      wreg[j * NCD + icd] = tsum<KX + LX, KY + LY, KZ + LZ, false>(
                          ex, ey, ez, [&](auto sx, auto sy, auto sz) {
                            return r[(ERI_CI(sx) * B + ERI_CI(sy)) * B + ERI_CI(sz)];
                          }, wreg[j * NCD + icd]);
                    }
                  });
                });
              });
            }
          }
          __syncwarp();
        }
#pragma unroll
        for (int j = 0; j < S::NPS; ++j)
          if (lane + 32 * j < HAB) {
            const int slot = tab_p[lane + 32 * j] >> 16;
#pragma unroll
            for (int icd = 0; icd < NCD; ++icd) Ws[icd * HABP + slot] = wreg[j * NCD + icd];
          }
        __syncwarp();
        // step D: bra transform
        {
          sfor<S::NCS>([&](auto j_) {
            constexpr int j = ERI_CI(j_);
            const int cd = lane + 32 * j;
            if (j * 32 + 32 <= NCD || cd < NCD) {
              const T* wc = Ws + cd * HABP;
              for_cart<LA>([&](auto ix, auto iy, auto iz) {
                for_cart<LB>([&](auto jx, auto jy, auto jz) {
                  constexpr int IX = ERI_CI(ix), IY = ERI_CI(iy), IZ = ERI_CI(iz);
                  constexpr int JX = ERI_CI(jx), JY = ERI_CI(jy), JZ = ERI_CI(jz);
                  constexpr int iab = cidx(LA, IY, IZ) * NB + cidx(LB, JY, JZ);
                  const T* fx = Eb + (IX * (LB + 1) + JX) * (LAB + 1);
                  const T* fy = Eb + NEB + (IY * (LB + 1) + JY) * (LAB + 1);
                  const T* fz = Eb + 2 * NEB + (IZ * (LB + 1) + JZ) * (LAB + 1);
                  xreg[j * NAB + iab] = tsum<IX + JX, IY + JY, IZ + JZ, false>(
                      fx, fy, fz, [&](auto tx, auto ty, auto tz) {
                        return wc[lex_base(LAB, ERI_CI(tx), ERI_CI(ty)) + ERI_CI(tz)];
                      }, xreg[j * NAB + iab]);
                });
              });
            }
          });
        }
        __syncwarp();
      }
      {  // X to shared memory for the contraction
        sfor<S::NCS>([&](auto j_) {
          constexpr int j = ERI_CI(j_);
          const int cd = lane + 32 * j;
          if (j * 32 + 32 <= NCD || cd < NCD) {
#pragma unroll
            for (int iab = 0; iab < NAB; ++iab) Xs[iab * NCD + cd] = xreg[j * NAB + iab];
          }
        });
        __syncwarp();
      }
      // contraction; one lane per output element
      if (Kh) {
        // Kh_ac[a][c] += w sum_{b, d} X D_bd ; Kh_bc[b][c] += w sum_{a, d} X D_ad
        for (int o = lane; o < (NA + NB) * NC; o += 32) {
          const bool isA = o < NA * NC;
          const int oo = isA ? o : o - NA * NC;
          const int r = oo / NC, c = oo % NC;
          T s = T(0);
          for (int d = 0; d < ND; ++d) {
            const int ci = c * ND + d;
            if (isA) {
              for (int b = 0; b < NB; ++b) s = fma(Xs[(r * NB + b) * NCD + ci], __ldg(Dp + (size_t)(ao2 + b) * n + ao4 + d), s);
            } else {
              for (int x = 0; x < NA; ++x) s = fma(Xs[(x * NB + r) * NCD + ci], __ldg(Dp + (size_t)(ao1 + x) * n + ao4 + d), s);
            }
          }
          const int row = isA ? ao1 + r : ao2 + r;
          acc_add(Kh + (size_t)row * n + ao3 + c, (double)(w * s), a.det);
        }
        // Kh_ad[a][d] += w sum_{b, c} X D_bc ; Kh_bd[b][d] += w sum_{a, c} X D_ac
        for (int o = lane; o < (NA + NB) * ND; o += 32) {
          const bool isA = o < NA * ND;
          const int oo = isA ? o : o - NA * ND;
          const int r = oo / ND, d = oo % ND;
          T s = T(0);
          for (int c = 0; c < NC; ++c) {
            const int ci = c * ND + d;
            if (isA) {
              for (int b = 0; b < NB; ++b) s = fma(Xs[(r * NB + b) * NCD + ci], __ldg(Dp + (size_t)(ao2 + b) * n + ao3 + c), s);
            } else {
              for (int x = 0; x < NA; ++x) s = fma(Xs[(x * NB + r) * NCD + ci], __ldg(Dp + (size_t)(ao1 + x) * n + ao3 + c), s);
            }
          }
          const int row = isA ? ao1 + r : ao2 + r;
          acc_add(Kh + (size_t)row * n + ao4 + d, (double)(w * s), a.det);
        }
      }
      if (Jh) {
        const T w2 = T(2) * w;
        for (int iab = lane; iab < NAB; iab += 32) {  // Jh_ab += 2w sum_cd X D_cd
          T s = T(0);
          for (int cd = 0; cd < NCD; ++cd)
            s = fma(Xs[iab * NCD + cd], __ldg(Dp + (size_t)(ao3 + cd / ND) * n + ao4 + cd % ND), s);
          acc_add(Jh + (size_t)(ao1 + iab / NB) * n + ao2 + iab % NB, (double)(w2 * s), a.det);
        }
        for (int cd = lane; cd < NCD; cd += 32) {  // Jh_cd += 2w sum_ab X D_ab
          T s = T(0);
          for (int iab = 0; iab < NAB; ++iab)
            s = fma(Xs[iab * NCD + cd], __ldg(Dp + (size_t)(ao1 + iab / NB) * n + ao2 + iab % NB), s);
          acc_add(Jh + (size_t)(ao3 + cd / ND) * n + ao4 + cd % ND, (double)(w2 * s), a.det);
        }
      }
      __syncwarp();
    }
  }
  }
  }
  if (a.counter && lane == 0 && done) {
    atomicAdd(a.counter, done);
    atomicAdd(a.counter + 1, doneq);
    atomicAdd(a.counter + 2, doneb);
  }
}

}  // namespace eri
