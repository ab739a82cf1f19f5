// J+K kernel of the large classes: one block per canonical shell quartet.
//
// What bounds it: GB300 issues 1.8 FP64 FMAs per clock and SM, one warp
// instruction every 17 clocks however many lanes are active, so FP64 time is
// the number of FP64 warp instructions; loads, address arithmetic and loop
// control beside them are nearly free as long as enough warps are resident.
// FP32 time is shared-memory bandwidth.  Hence:
//   - the whole ket range of a quartet sits in shared memory at once (W, X), so
//     R is built once per primitive quartet and not once per chunk of ket
//     components (one warp per quartet had 27 KB: (ff|ff) rebuilt R 100 times);
//   - a block's warps share that memory, so 4 to 8 times more warps fit an SM;
//   - every step is a flat list of tasks over all threads: (cd, P) and (ab, cd)
//     keep nearly every lane busy, where a lane-owned index kept 35 of 64;
//   - E_x E_y E_z is multiplied out once per primitive pair into one coefficient
//     per term, so a task is a plain dot product of prod (n_t + 1) terms (the
//     nested sums also multiplied by E^{00}_0 = 1 and closed every direction).
// Steps per quartet (Eq. eri_formula):
//   A  thread per primitive quartet, up to kWin at a time: rho, P-Q, prefactor,
//      Boys F_0..F_L;  E' products of G ket primitives
//   B  R^0 of G primitive quartets, level by level (Eq. R_recursion)
//   C  W[cd][P] += sum_g sum_Q E'_Q^{cd}(g) R_{P+Q}(g)
//   D  X[ab][cd] += sum_P E_P^{ab} W[cd][P], once per bra primitive
//   contraction: a thread per output element of Kh and Jh, D' blocks staged in
//   shared memory, one atomic per element.
// Measured on GB300: one (ff|ff) quartet 5.4 ms with a warp per quartet; FP64 J/K
// of 225 functions 184 ms then, 104 ms with this kernel, 53 ms now.  Component
// pairs ordered by their number of terms (lanes of a warp then run equally long
// sums; 22 of 32 lanes were active): (dp|pp) of it 4.05 -> 3.31 ms.
#pragma once
#include "kernels_b.cuh"

namespace eri {

// sum over the component pairs of prod_t (i_t + j_t + 1): terms of one transform
__host__ __device__ constexpr int pair_terms(int la, int lb) {
  int s = 0;
  for (int x = 0; x < ncart(la); ++x)
    for (int y = 0; y < ncart(lb); ++y) {
      int ix = 0, iy = 0, iz = 0, jx = 0, jy = 0, jz = 0;
      cart_xyz(la, x, ix, iy, iz);
      cart_xyz(lb, y, jx, jy, jz);
      s += (ix + jx + 1) * (iy + jy + 1) * (iz + jz + 1);
    }
  return s;
}

constexpr int kWin = 32;  // primitive quartets per Boys pass (one warp)

// start[m] = count(0) + .. + count(m - 1), m <= N <= 100 < blockDim.x (whole block; syncs)
template <int N, typename F>
__device__ __forceinline__ void block_starts(int* start, F&& count) {
  const int m = threadIdx.x;
  if (m < N) start[m] = count(m);
  __syncthreads();
  int s = 0;
  if (m <= N)
    for (int c = 0; c < m; ++c) s += start[c];
  __syncthreads();
  if (m <= N) start[m] = s;
  __syncthreads();
}

// order[0 .. N) = the component pairs by decreasing number of terms: the lanes of
// a warp take neighbours of this order and run loops of the same length
template <int N>
__device__ __forceinline__ void order_by_terms(const int* start, uint8_t* order) {
  const int m = threadIdx.x;
  if (m < N) {
    const int k = start[m + 1] - start[m];
    int r = 0;
    for (int c = 0; c < N; ++c) {
      const int kc = start[c + 1] - start[c];
      r += kc > k || (kc == k && c < m);
    }
    order[r] = (uint8_t)m;
  }
}

// Term table of a shell pair (la, lb), built once per block: component pair m
// owns terms [start[m], start[m+1]); term k is the product of the 1D
// coefficients at element offsets te[k] & 1023, (te[k] >> 10) & 1023, te[k] >> 20
// of the pair's x|y|z table (row length RL), and to[k] = its target offset
// off(tx, ty, tz).
template <int LI, int LJ, int RL, typename Off>
__device__ __forceinline__ void build_terms(int* start, unsigned* te, uint16_t* to, Off&& off) {
  constexpr int NJ = ncart(LJ), N = ncart(LI) * NJ, NE = (LI + 1) * (LJ + 1) * RL;
  block_starts<N>(start, [](int m) {
    int x[3], y[3];
    cart_xyz(LI, m / NJ, x[0], x[1], x[2]);
    cart_xyz(LJ, m % NJ, y[0], y[1], y[2]);
    return (x[0] + y[0] + 1) * (x[1] + y[1] + 1) * (x[2] + y[2] + 1);
  });
  const int m = threadIdx.x;
  if (m < N) {
    int k = start[m], x[3], y[3];
    cart_xyz(LI, m / NJ, x[0], x[1], x[2]);
    cart_xyz(LJ, m % NJ, y[0], y[1], y[2]);
    for (int a = 0; a <= x[0] + y[0]; ++a)
      for (int b = 0; b <= x[1] + y[1]; ++b)
        for (int c = 0; c <= x[2] + y[2]; ++c, ++k) {
          te[k] = (unsigned)((x[0] * (LJ + 1) + y[0]) * RL + a) |
                  ((unsigned)(NE + (x[1] * (LJ + 1) + y[1]) * RL + b) << 10) |
                  ((unsigned)(2 * NE + (x[2] * (LJ + 1) + y[2]) * RL + c) << 20);
          to[k] = (uint16_t)off(a, b, c);
        }
  }
}

// Scalars of the primitive quartets q0 .. q0 + kWin - 1 of one item (q = pb npk
// + pk), one thread each: pref F_0 .. pref F_L, c X, c Y, c Z, c  (c = -2 rho)
template <int L, typename T, typename A>
__device__ __forceinline__ void quartet_scalars(const A& a, int q0, int nq, int npk, int offb, int offk, T* scal) {
  const int t = threadIdx.x;
  if (t < kWin && q0 + t < nq) {
    const int pb = (q0 + t) / npk, pk = q0 + t - pb * npk;
    const int ib = offb + pb, ik = offk + pk;
    const T bp = pdv<T>(a.pd.p, a.pd.pf, ib), kp = pdv<T>(a.pd.p, a.pd.pf, ik);
    T rho, rs;
    quartet_rho(bp, kp, rho, rs);
    T pref = pdv<T>(a.pd.pref, a.pd.preff, ib) * pdv<T>(a.pd.pref, a.pd.preff, ik) * rs;
    attenuate(om2<T>(a), rho, pref);
    const T X = pdv<T>(a.pd.P, a.pd.Pf, ib) - pdv<T>(a.pd.P, a.pd.Pf, ik);
    const T Y = pdv<T>(a.pd.P, a.pd.Pf, a.pd.n + ib) - pdv<T>(a.pd.P, a.pd.Pf, a.pd.n + ik);
    const T Z = pdv<T>(a.pd.P, a.pd.Pf, 2 * a.pd.n + ib) - pdv<T>(a.pd.P, a.pd.Pf, 2 * a.pd.n + ik);
    T F[L + 1];
    Boys<T>::template eval<L>(rho * (X * X + Y * Y + Z * Z), a.bt, F);
    T* sc = scal + t * (L + 5);
#pragma unroll
    for (int m = 0; m <= L; ++m) sc[m] = pref * F[m];
    const T c = T(-2) * rho;
    sc[L + 1] = c * X;
    sc[L + 2] = c * Y;
    sc[L + 3] = c * Z;
    sc[L + 4] = c;
  }
}

// R^0 of ng primitive quartets into boxes of B^3 (B = L + 1), level by level
// over the block (Eq. R_recursion in the scaled form of r_build_warp); syncs
// before each level, not after the last
template <int L, typename T>
__device__ __forceinline__ void r_build_block(const T* scal, int ng, const RStep* __restrict__ steps, T* ping, T* box) {
  constexpr int NSC = L + 5, B = L + 1, BOX = B * B * B, NP = L > 0 ? nherm(L - 1) : 1;
  if constexpr (L == 0) {
    for (int g = threadIdx.x; g < ng; g += blockDim.x) box[g] = scal[g * NSC];
  } else {
    // level L holds one entry per quartet, pref F_L; the first pass reads it from the scalars
#pragma unroll
    for (int m = L - 1; m >= 0; --m) {
      const int ne = nherm(L - m);
      T* dst = ping + ((L - 1 - m) & 1) * NP;
      const T* src = ping + ((L - m) & 1) * NP;
      for (int it = threadIdx.x; it < ng * ne; it += blockDim.x) {
        const int g = it / ne, e = it - g * ne;
        const T* sc = scal + g * NSC;
        const RStep st = steps[e];
        T val;
        if (e == 0) {
          val = sc[m];
        } else {
          const T* s = m == L - 1 ? sc + L : src + g * 2 * NP;
          val = sc[L + 1 + st.dir] * s[st.dep1];
          if (st.dep2 >= 0) val = fma(sc[L + 4] * (T)st.k, s[st.dep2], val);
        }
        if (m == 0) box[g * BOX + (st.t * B + st.u) * B + st.v] = val;
        else dst[g * 2 * NP + e] = val;
      }
      if (m > 0) __syncthreads();
    }
  }
}

template <int LA, int LB, int LC, int LD, typename T>
struct CShape {
  static constexpr int LAB = LA + LB, LCD = LC + LD, L = LAB + LCD;
  static constexpr int NA = ncart(LA), NB = ncart(LB), NC = ncart(LC), ND = ncart(LD);
  static constexpr int NAB = NA * NB, NCD = NC * ND, HAB = nherm(LAB), HABP = HAB | 1, NCDP = NCD | 1;
  static constexpr int B = L + 1, BOX = B * B * B, NP = L > 0 ? nherm(L - 1) : 1, NSC = L + 5;
  static constexpr int TB = pair_terms(LA, LB), TK = pair_terms(LC, LD);
  static constexpr int NEB = (LA + 1) * (LB + 1) * (LAB + 1), NEK = (LC + 1) * (LD + 1) * (LCD + 1);
  static constexpr int NDB = (NA + NB) * (NC + ND) + NAB + NCD;  // the six D' blocks
  static constexpr int PER_G = BOX + 2 * NP + TK;
  // the bra coefficients have their own room, or (where that would not fit) share the ket's
  static constexpr bool SHARED_E = sizeof(T) * (size_t)(NCD * HABP + NAB * NCDP + 2 * TB + TK) > 180 * 1024;
  static constexpr int FIXED = NCD * HABP + NAB * NCDP + (SHARED_E ? (TB > TK ? TB - TK : 0) : TB) + kWin * NSC + NDB;
  // ket primitives per batch: those of a contracted s/p pair commonly 9, 3 with
  // a d or f shell; as many as keep the block near 48 KB (four blocks per SM)
  static constexpr int GT = (LC <= 1 && LD <= 1) ? 9 : (LC <= 1 || LD <= 1) ? 3 : 1;
  static constexpr int ROOM = (48 * 1024 / (int)sizeof(T) - FIXED) / PER_G;
  static constexpr int G = ROOM < 1 ? 1 : (ROOM > GT ? GT : ROOM);
  static constexpr int NT = NAB * NCD >= 1500 ? 256 : 128;
  static constexpr int TOTAL = FIXED + G * PER_G;
  static constexpr size_t smem() {
    return sizeof(T) * ((TOTAL + 3) / 4 * 4) + 4 * (TB + TK + NAB + NCD + 2) + 2 * (TB + TK + HAB + 3) + NAB + NCD;
  }
};

template <int LA, int LB, int LC, int LD, typename T>
__global__ void __launch_bounds__(CShape<LA, LB, LC, LD, T>::NT) jk_block_kernel(JKArgs A) {
  using S = CShape<LA, LB, LC, LD, T>;
  constexpr int LAB = S::LAB, LCD = S::LCD, L = S::L, B = S::B, NA = S::NA, NB = S::NB, NC = S::NC, ND = S::ND,
                NAB = S::NAB, NCD = S::NCD, HAB = S::HAB, HABP = S::HABP, NCDP = S::NCDP, G = S::G, NT = S::NT;
  const KArgs& a = A.k;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int tid = threadIdx.x;
  T* Ws = reinterpret_cast<T*>(smraw);       // [NCD][HABP]
  T* Xs = Ws + NCD * HABP;                   // [NAB][NCDP]
  T* box = Xs + NAB * NCDP;                  // [G][BOX]
  T* ping = box + G * S::BOX;                // [G][2][NP]
  T* ek = ping + G * 2 * S::NP;              // [G][TK]
  T* eb = S::SHARED_E ? ek : ek + G * S::TK;  // [TB]
  T* scal = Ws + S::TOTAL - kWin * S::NSC - S::NDB;  // [kWin][NSC]
  T* db = scal + kWin * S::NSC;              // D' blocks: [a+b][c+d], [ab], [cd]
  int* ks = reinterpret_cast<int*>(Ws + (S::TOTAL + 3) / 4 * 4);  // [NCD + 1]
  int* bs = ks + NCD + 1;                    // [NAB + 1]
  unsigned* kt = reinterpret_cast<unsigned*>(bs + NAB + 1);  // [TK]
  unsigned* btm = kt + S::TK;                // [TB]
  uint16_t* ko = reinterpret_cast<uint16_t*>(btm + S::TB);   // [TK] box offsets
  uint16_t* bo = ko + S::TK;                 // [TB] W columns
  uint16_t* pbox = bo + S::TB;               // [HAB] box offset of bra Hermite index P
  build_terms<LC, LD, LCD + 1>(ks, kt, ko, [](int t, int u, int v) { return (t * B + u) * B + v; });
  build_terms<LA, LB, LAB + 1>(bs, btm, bo, [](int t, int u, int v) { return herm_index(t, u, v); });
  for (int i = tid; i < HAB; i += NT) pbox[i] = (uint16_t)((herm_t(i) * B + herm_u(i)) * B + herm_v(i));
  uint8_t* cdo = reinterpret_cast<uint8_t*>(pbox + HAB);  // [NCD], [NAB]: order of the tasks
  uint8_t* abo = cdo + NCD;
  order_by_terms<NCD>(ks, cdo);
  order_by_terms<NAB>(bs, abo);

  const bool compact = a.items != nullptr;
  const int64_t total = compact ? (int64_t)__ldg(a.nitems) : a.wl.total;
  const int64_t first = compact ? 0 : a.wl.first;
  const int nshard = compact ? 1 : a.wl.nshard, shard = compact ? 0 : a.wl.shard;
  unsigned long long done = 0, doneq = 0, doneb = 0;
  const int64_t tile = item_tile(a.wl, total - first, gridDim.x), ntiles = (total - first + tile - 1) / tile;
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
      const int npb = __ldg(a.sp.np + pb_id), offb = __ldg(a.sp.poff + pb_id), eb0 = __ldg(a.sp.eoff + pb_id);
      const int npk = __ldg(a.sp.np + pk_id), offk = __ldg(a.sp.poff + pk_id), ek0 = __ldg(a.sp.eoff + pk_id);
      const int ao1 = __ldg(a.sp.ao1 + pb_id), ao2 = __ldg(a.sp.ao2 + pb_id);
      const int ao3 = __ldg(a.sp.ao1 + pk_id), ao4 = __ldg(a.sp.ao2 + pk_id);
      const int64_t mbase = __ldg(a.sp.mat_off + mol);
      const int n = __ldg(a.sp.mat_n + mol);
      if (part == 0) {
        ++done;
        doneq += (unsigned long long)npb * npk;
        doneb += npb;
      }
      int pb0, pb1, pk0, pk1;
      sp.range(part, 0, npb, npk, pb0, pb1, pk0, pk1);
      if (pb0 >= pb1 || npk == 0) continue;  // uniform over the block; W has no value without a ket primitive
      __syncthreads();  // the previous item's shared memory (first item: the tables) is done with
      const T* Dp = dens<T>(a) + mbase;
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
      const int nq = pb1 * npk;
      int win = 0, wend = 0;  // primitive quartets whose scalars are in `scal`
      for (int pb = pb0; pb < pb1; ++pb) {
        auto bra_terms = [&]() {
          for (int x = tid; x < S::TB; x += NT) {
            const unsigned w = btm[x];
            const int e = eb0 + pb * 3 * S::NEB;
            eb[x] = ldE<T>(a.pd, e + (w & 1023)) * ldE<T>(a.pd, e + ((w >> 10) & 1023)) * ldE<T>(a.pd, e + (w >> 20));
          }
        };
        if constexpr (!S::SHARED_E) bra_terms();
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
            const unsigned w = kt[k];
            const int e = ek0 + (k0 + g) * 3 * S::NEK, ox = w & 1023, oy = (w >> 10) & 1023, oz = w >> 20;
            const T v = ldE<T>(a.pd, e + ox) * ldE<T>(a.pd, e + oy) * ldE<T>(a.pd, e + oz);
            ek[x] = (ox % (LCD + 1) + oy % (LCD + 1) + oz % (LCD + 1)) & 1 ? -v : v;
          }
          __syncthreads();
          r_build_block<L, T>(scal + (q - win) * S::NSC, ng, a.rsteps, ping, box);
          __syncthreads();
          // C: two Hermite indices per task share the coefficients
          constexpr int HH = (HAB + 1) / 2;
          for (int it = tid; it < NCD * HH; it += NT) {
            const int row = it / HH, cd = cdo[row], P = it - row * HH, P2 = P + HH < HAB ? P + HH : P;
            const int s0 = ks[cd], s1 = ks[cd + 1];
            T x0 = T(0), x1 = T(0);
            for (int g = 0; g < ng; ++g) {
              const T* e = ek + g * S::TK;
              const T* r0 = box + g * S::BOX + pbox[P];
              const T* r1 = box + g * S::BOX + pbox[P2];
#pragma unroll 4
              for (int k = s0; k < s1; ++k) {
                const T c = e[k];
                const int o = ko[k];
                x0 = fma(c, r0[o], x0);
                x1 = fma(c, r1[o], x1);
              }
            }
            T* w = Ws + cd * HABP;
            if (k0 == 0) {
              w[P] = x0;
              if (P2 != P) w[P2] = x1;
            } else {
              w[P] += x0;
              if (P2 != P) w[P2] += x1;
            }
          }
          __syncthreads();
          k0 += ng;
        }
        if constexpr (S::SHARED_E) {
          bra_terms();
          __syncthreads();
        }
        // D: two ket pairs per task
        constexpr int CH = (NCD + 1) / 2;
        for (int it = tid; it < NAB * CH; it += NT) {
          const int row = it / CH, iab = abo[row], c0 = it - row * CH, c1 = c0 + CH < NCD ? c0 + CH : c0;
          const int s0 = bs[iab], s1 = bs[iab + 1];
          const T* w0 = Ws + c0 * HABP;
          const T* w1 = Ws + c1 * HABP;
          T x0 = T(0), x1 = T(0);
#pragma unroll 4
          for (int k = s0; k < s1; ++k) {
            const T c = eb[k];
            const int o = bo[k];
            x0 = fma(c, w0[o], x0);
            x1 = fma(c, w1[o], x1);
          }
          T* x = Xs + iab * NCDP;
          if (pb == pb0) {
            x[c0] = x0;
            if (c1 != c0) x[c1] = x1;
          } else {
            x[c0] += x0;
            if (c1 != c0) x[c1] += x1;
          }
        }
        __syncthreads();
      }
      // contraction (Eq. j_definition, Eq. k_definition with the canonical-quartet weights)
      T w = T(1);
      if (__ldg(a.sp.s1 + pb_id) == __ldg(a.sp.s2 + pb_id)) w *= T(0.5);
      if (__ldg(a.sp.s1 + pk_id) == __ldg(a.sp.s2 + pk_id)) w *= T(0.5);
      if (pb_id == pk_id) w *= T(0.5);
      if (a.Kh) {
        double* Kh = a.Kh + mbase;
        // output (row r of a|b, column c of c|d): row a takes D_b*, row b takes D_a*, likewise the columns
        for (int o = tid; o < (NA + NB) * (NC + ND); o += NT) {
          const int i = o / (NC + ND), j = o - i * (NC + ND);
          const bool isa = i < NA, isc = j < NC;
          const int nr = isa ? NB : NA, nc = isc ? ND : NC;
          const int xr = isa ? i * NB : i - NA, sr = isa ? 1 : NB;        // X row = xr + sr * (summed bra index)
          const int xc = isc ? j * ND : j - NC, sc = isc ? 1 : ND;        // X column likewise
          const T* d0 = db + (isa ? NA : 0) * (NC + ND) + (isc ? NC : 0);
          T s = T(0);
          for (int p = 0; p < nr; ++p) {
            const T* x = Xs + (xr + sr * p) * NCDP + xc;
            const T* d = d0 + p * (NC + ND);
            for (int q = 0; q < nc; ++q) s = fma(x[sc * q], d[q], s);
          }
          acc_add(Kh + (size_t)(isa ? ao1 + i : ao2 + i - NA) * n + (isc ? ao3 + j : ao4 + j - NC), (double)(w * s),
                  a.det);
        }
      }
      if (A.Jh) {
        double* Jh = A.Jh + mbase;
        const T* dab = db + (NA + NB) * (NC + ND);
        const T* dcd = dab + NAB;
        const T w2 = T(2) * w;
        for (int o = tid; o < NAB + NCD; o += NT) {
          T s = T(0);
          if (o < NAB) {
            for (int c = 0; c < NCD; ++c) s = fma(Xs[o * NCDP + c], dcd[c], s);
            acc_add(Jh + (size_t)(ao1 + o / NB) * n + ao2 + o % NB, (double)(w2 * s), a.det);
          } else {
            const int cd = o - NAB;
            for (int x = 0; x < NAB; ++x) s = fma(Xs[x * NCDP + cd], dab[x], s);
            acc_add(Jh + (size_t)(ao3 + cd / ND) * n + ao4 + cd % ND, (double)(w2 * s), a.det);
          }
        }
      }
    }
  }
  if (a.counter && tid == 0 && done) {
    atomicAdd(a.counter, done);
    atomicAdd(a.counter + 1, doneq);
    atomicAdd(a.counter + 2, doneb);
  }
}

// FP64 classes of the register kernel whose unrolled code is long run a block per
// quartet while the list is short (at most kShortList quartets per SM): a warp
// that passes once through some hundred kilobytes of straight-line code waits on
// instruction fetches (6 (pp|pp) quartets: 0.36 ms).  The line lies above the lists
// of a small molecule and below those of a medium one: 75 functions 1.64 ms at 8 per
// SM, 1.54 ms at 256; 225 functions 52.9 ms at 8, 55.2 ms at 256 ((pp|pp) 3.0 against
// 4.0 ms).
constexpr int kShortList = 16;
template <int LA, int LB, int LC, int LD, typename T>
__host__ __device__ constexpr bool block_when_short() {
  return sizeof(T) == 8 && ncart(LA) * ncart(LB) * ncart(LC) * ncart(LD) >= 36;
}

// Which J+K classes outside the register kernel run a block per quartet: every
// FP64 one, and the FP32 ones whose transforms do not fit the warp kernel's
// compile-time form.
template <int LA, int LB, int LC, int LD, typename T>
__host__ __device__ constexpr bool use_block_kernel() {
  return sizeof(T) == 8 || !(BShape<LA, LB, LC, LD, T>::REGW && BShape<LA, LB, LC, LD, T>::REGD);
}

}  // namespace eri
