// Plan construction, preparation kernels and the C ABI (include/eri.h).
//
// Every numerical step of the path runs in a kernel of this library:
//   normalisation (Sec. 2.1)            k_normalize, k_compfac
//   Boys table (Eq. boys_function)      k_boys_table
//   primitive pair data (Eq. pair_definition)   k_pairs
//   Schwarz bounds (Eq. cauchy_schwarz_bound)   k_schwarz
//   class-sorted lists (Sec. 3.2, Eq. kernel_upperbound)   k_sig, k_rank, k_counts, k_prefix
//   Hermite density (Eq. j_formula, first sub-step)        k_hermite_density
//   J-engine / exchange kernels (kernels.cuh)
//   Hermite J -> Cartesian J (Eq. j_formula, last sub-step) k_post_j
//   K symmetrisation (Eq. 8_fold_symmetry)                 k_post_k
//   energies (SI Eq. si_E_J_K)                             k_energy
// Host code only validates arguments, does integer bookkeeping (offsets,
// launch sizes) and launches.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "../../include/eri.h"
#include "dispatch.cuh"
#include "plan.cuh"

using namespace eri;

// ---------------------------------------------------------------------------
// device kernels
// ---------------------------------------------------------------------------

// Per-primitive normalised coefficient of the (l,0,0) component:
// c_k N_l(a_k) s, N_l(a) = (2a/pi)^(3/4) (4a)^(l/2) / sqrt((2l-1)!!),
// s chosen so the contracted (l,0,0) function has unit norm; for two
// normalised (l,0,0) primitives on one centre <g_a|g_b> = (2 sqrt(ab)/(a+b))^(l+3/2).
__global__ void k_normalize(int nshell, const int* __restrict__ l, const int* __restrict__ nprim,
                            const int* __restrict__ poff, const double* __restrict__ ex,
                            const double* __restrict__ co, double* __restrict__ cn) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= nshell) return;
  const int L = l[s], n = nprim[s], o = poff[s];
  double df = 1.0;
  for (int k = 2 * L - 1; k > 1; k -= 2) df *= k;
  double S = 0.0;
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < n; ++j) {
      double ai = ex[o + i], aj = ex[o + j];
      S += co[o + i] * co[o + j] * pow(2.0 * sqrt(ai * aj) / (ai + aj), L + 1.5);
    }
  const double sc = 1.0 / sqrt(S);
  for (int i = 0; i < n; ++i) {
    double a = ex[o + i];
    cn[o + i] = co[o + i] * sc * pow(2.0 * a / 3.14159265358979323846, 0.75) * pow(4.0 * a, 0.5 * L) / sqrt(df);
  }
}

// Component factor f(x,y,z) = sqrt((2l-1)!! / ((2x-1)!! (2y-1)!! (2z-1)!!)) per AO.
__global__ void k_compfac(int nshell, const int* __restrict__ l, const int* __restrict__ ao, double* __restrict__ f) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= nshell) return;
  const int L = l[s];
  auto df = [](int n) {
    double r = 1.0;
    for (int k = n; k > 1; k -= 2) r *= k;
    return r;
  };
  for (int k = 0; k < ncart(L); ++k) {
    int x, y, z;
    cart_xyz(L, k, x, y, z);
    f[ao[s] + k] = sqrt(df(2 * L - 1) / (df(2 * x - 1) * df(2 * y - 1) * df(2 * z - 1)));
  }
}

// Boys tables: F_m(T_k), T_k = k h, from the series for a high order m_top,
// F_m(T) = exp(-T) sum_i (2T)^i / ((2m+1)(2m+3)...(2m+2i+1)), then the stable
// downward recursion F_m = (2T F_{m+1} + exp(-T)) / (2m+1).  Stored as Taylor
// coefficients c[k][m][j] = F_{m+j}(T_k) / j!  and exp(-T_k).
__global__ void k_boys_table(double* __restrict__ c64, double* __restrict__ e64, float* __restrict__ c32,
                             float* __restrict__ e32) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= BOYS_NT) return;
  const double T = k * BOYS_H;
  const int mtop = BOYS_MMAX + BOYS_J64 + 24;
  double term = 1.0 / (2 * mtop + 1), sum = term;
  for (int i = 1; i < 2000; ++i) {
    term *= 2.0 * T / (2 * mtop + 2 * i + 1);
    sum += term;
    if (term < 1e-18 * sum) break;
  }
  const double e = exp(-T);
  double F[BOYS_MMAX + BOYS_J64 + 1];
  double f = e * sum;
  for (int m = mtop - 1; m >= 0; --m) {
    f = (2.0 * T * f + e) / (2 * m + 1);
    if (m <= BOYS_MMAX + BOYS_J64) F[m] = f;
  }
  double fact = 1.0;
  for (int j = 0; j < BOYS_J64; ++j) {
    if (j > 0) fact *= j;
    for (int m = 0; m <= BOYS_MMAX; ++m) {
      c64[((size_t)k * (BOYS_MMAX + 1) + m) * BOYS_J64 + j] = F[m + j] / fact;
      if (j < BOYS_J32) c32[((size_t)k * (BOYS_MMAX + 1) + m) * BOYS_J32 + j] = (float)(F[m + j] / fact);
    }
  }
  e64[k] = e;
  e32[k] = (float)e;
}

// Primitive-pair data for every shell pair (Eq. pair_definition):
// p = a+b, P = (aA+bB)/p, PA = P-A, PB = P-B,
// pref = c_a c_b exp(-ab/p |AB|^2) sqrt(2 pi^(5/2)) / p  (so that a quartet's
// prefactor 2 pi^(5/2)/(pq sqrt(p+q)) K_AB K_CD c c c c = pref_ab pref_cd / sqrt(p+q)).
__global__ void k_pairs(int npair, const int* __restrict__ s1, const int* __restrict__ s2,
                        const int* __restrict__ poff, const int* __restrict__ sh_atom, const int* __restrict__ sh_np,
                        const int* __restrict__ sh_po, const double* __restrict__ ex, const double* __restrict__ cn,
                        const double* __restrict__ coords, int nprimpair, double* p_, double* P_, double* PA_,
                        double* PB_, double* pref_, float* pf, float* Pf, float* PAf, float* PBf, float* preff,
                        float* pmaxp, float* prefmaxp, double* ea_, float4* q4) {
  const int ip = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;  // one warp per pair
  if (ip >= npair) return;
  const int a = s1[ip], b = s2[ip];
  const double* A = coords + 3 * sh_atom[a];
  const double* Bc = coords + 3 * sh_atom[b];
  double AB2 = 0.0;
  for (int d = 0; d < 3; ++d) AB2 += (A[d] - Bc[d]) * (A[d] - Bc[d]);
  const int nb = sh_np[b];
  double pmx = 0.0, prmx = 0.0;
  const double s2pi52 = 5.9149671727956129;  // sqrt(2 pi^(5/2))
  for (int k = lane; k < sh_np[a] * nb; k += 32) {
      const int i = k / nb, j = k - i * nb, o = poff[ip] + k;
      const double ea = ex[sh_po[a] + i], eb = ex[sh_po[b] + j];
      const double p = ea + eb;
      const double pr = cn[sh_po[a] + i] * cn[sh_po[b] + j] * exp(-ea * eb / p * AB2) * s2pi52 / p;
      p_[o] = p;
      ea_[o] = ea;
      pmx = fmax(pmx, p);
      prmx = fmax(prmx, fabs(pr));
      pref_[o] = pr;
      pf[o] = (float)p;
      preff[o] = (float)pr;
      float fP[3], fA[3], fB[3];
      for (int d = 0; d < 3; ++d) {
        const double P = (ea * A[d] + eb * Bc[d]) / p;
        P_[d * nprimpair + o] = P;
        PA_[d * nprimpair + o] = P - A[d];
        PB_[d * nprimpair + o] = P - Bc[d];
        fP[d] = (float)P;
        fA[d] = (float)(P - A[d]);
        fB[d] = (float)(P - Bc[d]);
        Pf[d * nprimpair + o] = fP[d];
        PAf[d * nprimpair + o] = fA[d];
        PBf[d * nprimpair + o] = fB[d];
      }
      q4[3 * (size_t)o] = make_float4(fP[0], fP[1], fP[2], (float)p);
      q4[3 * (size_t)o + 1] = make_float4(fA[0], fA[1], fA[2], (float)pr);
      q4[3 * (size_t)o + 2] = make_float4(fB[0], fB[1], fB[2], 0.0f);
    }
  for (int o = 16; o > 0; o >>= 1) {
    pmx = fmax(pmx, __shfl_xor_sync(0xffffffffu, pmx, o));
    prmx = fmax(prmx, __shfl_xor_sync(0xffffffffu, prmx, o));
  }
  if (lane != 0) return;
  pmaxp[ip] = (float)pmx;
  prefmaxp[ip] = (float)fmin(prmx, 1.0e30);
}

// Mixed-precision tier split of the items [wl.first, wl.total) of one class
// pair: one warp per run of `rounds` x 32 items (runs t with t % nshard == shard;
// the host takes one round per run where the work is shared over GPUs or the list
// is short), each lane locates and tests one item per round; the FP64-tier and
// FP32-tier quartets are appended to out0 / out1 (one atomic per run on cnt[0],
// cnt[1]).  Inside a run the items of a tier are written by increasing number of
// primitive quartets, so that the 32 lanes of a thread kernel's warp have about as
// many (runs of 32 in list order: the FP32 (fp|pp) kernel of 900 functions took
// 38.6 ms, its lanes waiting for the longest).
constexpr int kSplitRounds = 8;
__global__ void __launch_bounds__(256) k_tier_split(KArgs a, int rounds, int2* __restrict__ out0,
                                                    int2* __restrict__ out1, unsigned int* __restrict__ cnt) {
  __shared__ unsigned slots[8][32];  // per warp: [tier][work bucket] counts, then positions
  const int lane = threadIdx.x & 31;
  unsigned* slot = slots[threadIdx.x >> 5];
  const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
  const int64_t nrun = (a.wl.total - a.wl.first + 32 * rounds - 1) / (32 * rounds);
  for (int64_t run = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * a.wl.nshard + a.wl.shard;
       run < nrun; run += nwarps * a.wl.nshard) {
    int ib[kSplitRounds], ik[kSplitRounds], key[kSplitRounds];
    int guard = 0, dropped = 0;
    __syncwarp();
    slot[lane] = 0;
    __syncwarp();
#pragma unroll
    for (int r = 0; r < kSplitRounds; ++r) {
      key[r] = -1;
      const int64_t item = a.wl.first + (run * rounds + r) * 32 + lane;
      if (r >= rounds || item >= a.wl.total) continue;
      ib[r] = find_bra(a.wl.prefix, a.wl.nbra, item);
      ik[r] = (int)(item - __ldg(a.wl.prefix + ib[r]));
      const int pb_id = __ldg(a.wl.bra + ib[r]);
      const int mol = __ldg(a.sp.pmol + pb_id);
      const int seg = __ldg(a.wl.kseg + mol * NPAIRCLASS);
      ik[r] = ket_pos(a.wl, seg, ik[r], __ldg(a.wl.prefix + ib[r] + 1) - __ldg(a.wl.prefix + ib[r]));
      const int pk_id = __ldg(a.wl.ket + seg + ik[r]);
      const int tier = a.mixed || a.screen > 0.0f
                           ? quartet_tier(a, mol, pb_id, pk_id, __ldg(a.sp.s1 + pb_id), __ldg(a.sp.s2 + pb_id),
                                          __ldg(a.sp.s1 + pk_id), __ldg(a.sp.s2 + pk_id))
                           : 0;  // plain FP64 builds: the order only
      guard += tier == 2;
      dropped += tier == 3;
      if (tier == 3) continue;
      key[r] = (tier == 1 ? 16 : 0) + work_bucket(a.wl, __ldg(a.sp.np + pb_id), __ldg(a.sp.np + pk_id));
      atomicAdd(slot + key[r], 1u);
    }
    guard = __reduce_add_sync(0xffffffffu, guard);
    dropped = __reduce_add_sync(0xffffffffu, dropped);
    if (lane == 0 && guard && a.guard) atomicAdd(a.guard, (unsigned long long)guard);
    if (lane == 0 && dropped && a.screened) atomicAdd(a.screened, (unsigned long long)dropped);
    __syncwarp();
    const unsigned v = slot[lane];
    unsigned x = v;  // inclusive sum over the buckets of the lane's tier
#pragma unroll
    for (int d = 1; d < 16; d <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, x, d, 16);
      if ((lane & 15) >= d) x += y;
    }
    unsigned base = 0;
    if ((lane & 15) == 15 && x) base = atomicAdd(cnt + (lane >> 4), x);
    base = __shfl_sync(0xffffffffu, base, 15, 16);
    slot[lane] = base + x - v;
    __syncwarp();
#pragma unroll
    for (int r = 0; r < kSplitRounds; ++r)
      if (key[r] >= 0) (key[r] < 16 ? out0 : out1)[atomicAdd(slot + key[r], 1u)] = make_int2(ib[r], ik[r]);
  }
}

// max |D'| over the blocks (s1, s2) and (s2, s1) of every shell pair (used by
// the mixed-precision tier test)
__global__ void k_dmax(int npair, const int* __restrict__ s1, const int* __restrict__ s2, const int* __restrict__ l,
                       const int* __restrict__ pao1, const int* __restrict__ pao2, const int* __restrict__ pmol,
                       const int64_t* __restrict__ mat_off, const int* __restrict__ mat_n,
                       const double* __restrict__ Dp, float* __restrict__ dmax) {
  int ip = blockIdx.x * blockDim.x + threadIdx.x;
  if (ip >= npair) return;
  const int m = pmol[ip], n = mat_n[m];
  const double* D = Dp + mat_off[m];
  const int a = pao1[ip], b = pao2[ip], na = ncart(l[s1[ip]]), nb = ncart(l[s2[ip]]);
  double mx = 0.0;
  for (int i = 0; i < na; ++i)
    for (int j = 0; j < nb; ++j)
      mx = fmax(mx, fmax(fabs(D[(size_t)(a + i) * n + b + j]), fabs(D[(size_t)(b + j) * n + a + i])));
  dmax[ip] = __double2float_ru(mx);
}


// Hermite coefficients E^{ij}_t (Eq. E_recursion) of every primitive pair, per
// direction, stored as (i*(l2+1)+j)*(l1+l2+1)+t, i <= l1, j <= l2 (x, then y, then z).
__global__ void k_etab(int npair, const int* __restrict__ s1, const int* __restrict__ s2, const int* __restrict__ np,
                       const int* __restrict__ poff, const int* __restrict__ eoff, const int* __restrict__ sh_l,
                       PairData pd, double* __restrict__ E, float* __restrict__ Ef) {
  const int ip = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (ip >= npair) return;
  const int l1 = sh_l[s1[ip]], l2 = sh_l[s2[ip]];
  const int ne = (l1 + 1) * (l2 + 1) * (l1 + l2 + 1);
  double tmp[225];
  for (int x = lane; x < 3 * np[ip]; x += 32) {  // one warp per pair, a lane per (primitive pair, direction)
    const int k = x / 3, d = x - 3 * k, pi = poff[ip] + k;
    md_e_rt(l1, l2, pd.PA[d * pd.n + pi], pd.PB[d * pd.n + pi], 0.5 / pd.p[pi], tmp);
    const size_t o = (size_t)eoff[ip] + (size_t)x * ne;
    for (int i = 0; i <= l1; ++i)
      for (int j = 0; j <= l2; ++j)
        for (int t = 0; t <= l1 + l2; ++t) {
          const double v = t <= i + j ? tmp[(i * 5 + j) * 9 + t] : 0.0;
          E[o + (i * (l2 + 1) + j) * (l1 + l2 + 1) + t] = v;
          Ef[o + (i * (l2 + 1) + j) * (l1 + l2 + 1) + t] = (float)v;
        }
  }
}

// Schwarz bound per shell pair: Q = sqrt(max_{mu,nu} |(mu nu|mu nu)|) in FP64, rounded up to float32.
// One block per pair.  Contracted pairs: a warp per primitive quartet; single
// primitive pairs: the warps share the component pairs.  R goes level by level
// over the lanes; then component pair by component pair (uniform loops) a lane
// per bra Hermite index, summed over the warp in a fixed order.  (A lane per
// component pair ran the union of the lanes' nested loops: 1.2 ms for the (ff|ff)
// diagonal; a thread per pair with local arrays 2 ms; now 0.1 ms.)  The E tables
// are those of k_etab; primitive quartets (i, j) and (j, i) are equal, so j <= i
// with weight 2.
constexpr int kSchwarzWarps = 6;  // 44 KB of shared memory
constexpr int kSchwarzR = nherm(4 * LMAX);
__global__ void __launch_bounds__(32 * kSchwarzWarps)
    k_schwarz(int npair, const int* __restrict__ s1, const int* __restrict__ s2, const int* __restrict__ np,
              const int* __restrict__ poff, const int* __restrict__ eoff, const int* __restrict__ sh_l,
              const int* __restrict__ ao, const double* __restrict__ f, PairData pd, BoysTabs bt,
              const RStep* __restrict__ st, float* __restrict__ Q) {
  __shared__ double Rs[kSchwarzWarps][2][kSchwarzR], Fs[kSchwarzWarps][4 * LMAX + 1], dsum[kSchwarzWarps][100];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, ip = blockIdx.x;
  const int l1 = sh_l[s1[ip]], l2 = sh_l[s2[ip]], lp = l1 + l2, L = 2 * lp;
  const int n2 = ncart(l2), nc = ncart(l1) * n2, ne = (l1 + 1) * (l2 + 1) * (lp + 1);
  const bool shared_quartet = np[ip] == 1;
  double* F = Fs[w];
  for (int c = lane; c < nc; c += 32) dsum[w][c] = 0.0;
  __syncwarp();
  int turn = 0;
  for (int i = 0; i < np[ip]; ++i) {
    const int pi = poff[ip] + i;
    for (int j = 0; j <= i; ++j) {
      if (!shared_quartet && turn++ % kSchwarzWarps != w) continue;
      const int pj = poff[ip] + j;
      const double p = pd.p[pi], q = pd.p[pj], rho = p * q / (p + q);
      const double X = pd.P[pi] - pd.P[pj], Y = pd.P[pd.n + pi] - pd.P[pd.n + pj],
                   Z = pd.P[2 * pd.n + pi] - pd.P[2 * pd.n + pj];
      const double T = rho * (X * X + Y * Y + Z * Z);
      // generic Boys (runtime order): Taylor at the top order then downward
      double fm;
      if (T < boys_tmax(4 * LMAX)) {
        const int k = __double2int_rn(T * BOYS_INV_H);
        const double* c = bt.c64 + ((size_t)k * (BOYS_MMAX + 1) + L) * BOYS_J64;
        const double dd = k * BOYS_H - T;
        fm = c[BOYS_J64 - 1];
        for (int jj = BOYS_J64 - 2; jj >= 0; --jj) fm = fm * dd + c[jj];
        if (lane == 0) F[L] = fm;
        const double e = exp(-T);
        for (int m = L - 1; m >= 0; --m) {
          fm = (2 * T * fm + e) / (2 * m + 1);
          if (lane == 0) F[m] = fm;
        }
      } else {
        const double e = exp(-T);
        fm = 0.5 * sqrt(3.14159265358979323846 / T);
        if (lane == 0) F[0] = fm;
        for (int m = 0; m < L; ++m) {
          fm = ((2 * m + 1) * fm - e) / (2 * T);
          if (lane == 0) F[m + 1] = fm;
        }
      }
      __syncwarp();
      const double pref = (i == j ? 1.0 : 2.0) * pd.pref[pi] * pd.pref[pj] / sqrt(p + q);
      double* cur = Rs[w][0];
      double* nxt = Rs[w][1];
      if (lane == 0) cur[0] = pref * F[L];
      __syncwarp();
      for (int m = L - 1; m >= 0; --m) {
        const int nr = nherm(L - m);
        for (int e = lane; e < nr; e += 32) {
          double v;
          if (e == 0) {
            v = pref * F[m];
          } else {
            const RStep s = st[e];
            v = (s.dir == 0 ? X : (s.dir == 1 ? Y : Z)) * cur[s.dep1];
            if (s.dep2 >= 0) v += s.k * cur[s.dep2];
            v *= -2.0 * rho;
          }
          nxt[e] = v;
        }
        __syncwarp();
        double* t = cur; cur = nxt; nxt = t;
      }
      const double* E1 = pd.E + eoff[ip] + (size_t)i * 3 * ne;
      const double* E2 = pd.E + eoff[ip] + (size_t)j * 3 * ne;
      for (int c = shared_quartet ? w : 0; c < nc; c += shared_quartet ? kSchwarzWarps : 1) {  // uniform over the warp
        int ix, iy, iz, jx, jy, jz;
        cart_xyz(l1, c / n2, ix, iy, iz);
        cart_xyz(l2, c % n2, jx, jy, jz);
        const int mx = ix + jx + 1, my = iy + jy + 1, mz = iz + jz + 1;
        const int ox = (ix * (l2 + 1) + jx) * (lp + 1), oy = ne + (iy * (l2 + 1) + jy) * (lp + 1),
                  oz = 2 * ne + (iz * (l2 + 1) + jz) * (lp + 1);
        double v = 0.0;
        for (int t = lane; t < mx * my * mz; t += 32) {
          const int tx = t / (my * mz), ty = t / mz % my, tz = t % mz;
          double u = 0.0;
          for (int sx = 0; sx < mx; ++sx)
            for (int sy = 0; sy < my; ++sy) {
              double uz = 0.0;
              for (int sz = 0; sz < mz; ++sz)
                uz = fma((sx + sy + sz) & 1 ? -E2[oz + sz] : E2[oz + sz], cur[herm_index(tx + sx, ty + sy, tz + sz)], uz);
              u = fma(E2[ox + sx] * E2[oy + sy], uz, u);
            }
          v = fma(E1[ox + tx] * E1[oy + ty] * E1[oz + tz], u, v);
        }
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) dsum[w][c] += v;
      }
      __syncwarp();
    }
  }
  __syncthreads();
  if (w != 0) return;
  double mx = 0.0;
  for (int c = lane; c < nc; c += 32) {
    double v = 0.0;
    for (int x = 0; x < kSchwarzWarps; ++x) v += dsum[x][c];
    const double fn = f[ao[s1[ip]] + c / n2] * f[ao[s2[ip]] + c % n2];
    mx = fmax(mx, fabs(v * fn * fn));
  }
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) Q[ip] = __double2float_ru(sqrt(mx));
}

// Primitive screening.  A contracted pair holds primitive pairs whose prefactor
// exp(-ab/p |AB|^2) is far below anything a quartet of the lists contributes
// (tight exponents on two centres).  In the Coulomb metric ||x|| = (x|x)^(1/2)
// the triangle inequality bounds a primitive pair by its Hermite functions,
//   q = |pref| (2p)^(-1/4) max_{mu nu} prod_d sum_t |E_t| ((2t-1)!! p^t)^(1/2)
// (||Lambda_tuv||^2 = (2p)^(-1/2) p^n (2t-1)!! (2u-1)!! (2v-1)!! / (2n+1) in the
// units of pref), and |(ab|cd)| <= q_ab q_cd for every primitive quartet.
// k_primpack moves the primitive pairs with q qmax >= kPrimEps thresh to the
// front of their shell pair and counts them; the J/K, J-engine and gradient
// kernels run over those (a pair keeps at least one).  Each dropped primitive
// quartet is below 1e-8 of the quartet threshold (thresh = 0 drops none).  That
// bounds the integral; the gradient's derivatives raise a Hermite index or bring
// down an exponent, up to about sqrt((2l + 1) p) + 2 (ab/p) |AB| times it, 1e2 to 1e3
// for the tightest pairs, which leaves 1e-5 of the threshold and less.
constexpr double kPrimEps = 1e-8;
__global__ void __launch_bounds__(128)
    k_primq(int npair, const int* __restrict__ s1, const int* __restrict__ s2, const int* __restrict__ np,
            const int* __restrict__ poff, const int* __restrict__ eoff, const int* __restrict__ sh_l,
            const int* __restrict__ ao, const double* __restrict__ f, const int* __restrict__ pmol, PairData pd,
            double* __restrict__ pq, unsigned int* __restrict__ pqmax) {
  __shared__ double Ss[4][3 * (LMAX + 1) * (LMAX + 1)];
  const int ip = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;  // one warp per pair
  if (ip >= npair) return;
  double* S = Ss[threadIdx.x >> 5];
  const int a = s1[ip], b = s2[ip], l1 = sh_l[a], l2 = sh_l[b], lp = l1 + l2;
  const int rows = (l1 + 1) * (l2 + 1), n2 = ncart(l2), nc = ncart(l1) * n2;
  double fm = 0.0, fn = 0.0;
  for (int c = 0; c < ncart(l1); ++c) fm = fmax(fm, f[ao[a] + c]);
  for (int c = 0; c < n2; ++c) fn = fmax(fn, f[ao[b] + c]);
  const double df[2 * LMAX + 1] = {1.0, 1.0, 3.0, 15.0, 105.0, 945.0, 10395.0};  // (2t-1)!!
  double top = 0.0;
  for (int k = 0; k < np[ip]; ++k) {
    const int pi = poff[ip] + k;
    const double p = pd.p[pi];
    for (int r = lane; r < 3 * rows; r += 32) {
      const double* E = pd.E + eoff[ip] + ((size_t)k * 3 * rows + r) * (lp + 1);
      double v = 0.0, pt = 1.0;
      for (int t = 0; t <= lp; ++t) {
        v += fabs(E[t]) * sqrt(pt * df[t]);
        pt *= p;
      }
      S[r] = v;
    }
    __syncwarp();
    double mx = 0.0;
    for (int c = lane; c < nc; c += 32) {
      int ix, iy, iz, jx, jy, jz;
      cart_xyz(l1, c / n2, ix, iy, iz);
      cart_xyz(l2, c % n2, jx, jy, jz);
      mx = fmax(mx, S[ix * (l2 + 1) + jx] * S[rows + iy * (l2 + 1) + jy] * S[2 * rows + iz * (l2 + 1) + jz]);
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const double q = fabs(pd.pref[pi]) * rsqrt(sqrt(2.0 * p)) * mx * fm * fn;
    if (lane == 0) pq[pi] = q;
    top = fmax(top, q);
    __syncwarp();
  }
  if (lane == 0) atomicMax(pqmax + pmol[ip], __float_as_uint(__double2float_ru(fmin(top, 1e38))));
}

template <typename T>
__device__ __forceinline__ void dswap(T& x, T& y) {
  const T t = x;
  x = y;
  y = t;
}
__global__ void k_primpack(int npair, const int* __restrict__ s1, const int* __restrict__ s2,
                           const int* __restrict__ np, const int* __restrict__ poff, const int* __restrict__ eoff,
                           const int* __restrict__ sh_l, const int* __restrict__ pmol,
                           const unsigned int* __restrict__ pqmax, double limit, int n, double* pq, double* p,
                           double* P, double* PA, double* PB, double* pref, double* ea, float* pf, float* Pf,
                           float* PAf, float* PBf, float* preff, float4* q4, double* E, float* Ef,
                           int* __restrict__ nkeep) {
  const int ip = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;  // one warp per pair
  if (ip >= npair) return;
  const int l1 = sh_l[s1[ip]], l2 = sh_l[s2[ip]], ne3 = 3 * (l1 + 1) * (l2 + 1) * (l1 + l2 + 1);
  const int o = poff[ip];
  const double qmax = (double)__uint_as_float(pqmax[pmol[ip]]);
  int m = 0;
  for (int k = 0; k < np[ip]; ++k) {
    if (pq[o + k] * qmax < limit) continue;  // (a NaN bound is kept)
    if (k != m) {
      const int x = o + k, y = o + m;
      __syncwarp();  // every lane has read pq[o + k]
      if (lane == 0) {
        dswap(pq[x], pq[y]);
        dswap(p[x], p[y]);
        dswap(pref[x], pref[y]);
        dswap(ea[x], ea[y]);
        dswap(pf[x], pf[y]);
        dswap(preff[x], preff[y]);
      } else if (lane <= 3) {
        const int d = lane - 1;
        dswap(P[d * n + x], P[d * n + y]);
        dswap(PA[d * n + x], PA[d * n + y]);
        dswap(PB[d * n + x], PB[d * n + y]);
        dswap(Pf[d * n + x], Pf[d * n + y]);
        dswap(PAf[d * n + x], PAf[d * n + y]);
        dswap(PBf[d * n + x], PBf[d * n + y]);
        dswap(q4[3 * (size_t)x + d], q4[3 * (size_t)y + d]);
      }
      const size_t ex = (size_t)eoff[ip] + (size_t)k * ne3, ey = (size_t)eoff[ip] + (size_t)m * ne3;
      for (int e = lane; e < ne3; e += 32) {
        dswap(E[ex + e], E[ey + e]);
        dswap(Ef[ex + e], Ef[ey + e]);
      }
      __syncwarp();
    }
    ++m;
  }
  // Never none: a pair of frozen lists that the atoms have pulled apart stays listed,
  // and the kernels count on a first primitive pair (whose integrals are as small as
  // its bound; it is in place already).
  if (lane == 0) nkeep[ip] = max(m, 1);
}

// Per-molecule Schwarz maximum (pairs never cross molecules).  Q >= 0, so
// the unsigned order of the float bits is the float order.
__global__ void k_qmax(int n, const float* __restrict__ Q, const int* __restrict__ pmol, unsigned int* __restrict__ out) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int m = i < n ? pmol[i] : -1;
  unsigned int v = i < n ? __float_as_uint(Q[i]) : 0u;
  const int m0 = __shfl_sync(0xffffffffu, m, 0);
  if (__all_sync(0xffffffffu, m == m0 || m < 0)) {
    v = __reduce_max_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0 && m0 >= 0) atomicMax(out + m0, v);
  } else if (m >= 0) {
    atomicMax(out + m, v);
  }
}

// significance of each pair: (double)Q * (double)Qmax(molecule) >= thresh;
// counts per (molecule, class)
__global__ void k_sig(int npair, const float* __restrict__ Q, const int* __restrict__ pmol,
                      const unsigned int* __restrict__ qmax_bits, double thresh, const int* __restrict__ cls,
                      int* __restrict__ sig, int* __restrict__ ccm) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= npair) return;
  const int m = pmol[i];
  const double qmax = (double)__uint_as_float(qmax_bits[m]);
  const int s = ((double)Q[i] * qmax >= thresh) ? 1 : 0;
  sig[i] = s;
  if (s) atomicAdd(ccm + m * NPAIRCLASS + cls[i], 1);
}

// rank of each significant pair inside its (molecule, class) segment: Q
// descending, pair index ascending.  The sorted array is class-major, molecule
// by molecule inside a class: segment (X, m) starts at coff[X] + segloc[m][X].
__global__ void k_rank(int npair, const float* __restrict__ Q, const int* __restrict__ cls, const int* __restrict__ sig,
                       const int* __restrict__ pmol, const int* __restrict__ pbase, const int* __restrict__ coff,
                       const int* __restrict__ segloc, int* __restrict__ sorted, int* __restrict__ pos) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= npair || !sig[i]) return;
  const float qi = Q[i];
  const int ci = cls[i], m = pmol[i];
  int r = 0;
  for (int j = pbase[m]; j < pbase[m + 1]; ++j) {
    if (!sig[j] || cls[j] != ci) continue;
    const float qj = Q[j];
    if (qj > qi || (qj == qi && j < i)) ++r;
  }
  sorted[coff[ci] + segloc[m * NPAIRCLASS + ci] + r] = i;
  pos[i] = r;
}

// counts[pair][Y] = number of kets of class Y (same molecule) with Q_i Q_k >= thresh
// (binary search on the Q-sorted segment)
__global__ void k_counts(int npair, const float* __restrict__ Q, const int* __restrict__ sig,
                         const int* __restrict__ pmol, const int* __restrict__ sorted, const int* __restrict__ coff,
                         const int* __restrict__ segloc, const int* __restrict__ ccm, double thresh,
                         int* __restrict__ counts) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= npair * NPAIRCLASS) return;
  const int i = t / NPAIRCLASS, Y = t % NPAIRCLASS;
  if (!sig[i]) { counts[t] = 0; return; }
  const int m = pmol[i];
  const double qi = (double)Q[i];
  const int* lst = sorted + coff[Y] + segloc[m * NPAIRCLASS + Y];
  int lo = 0, hi = ccm[m * NPAIRCLASS + Y];  // first position with Q_i Q_k < thresh
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (qi * (double)Q[lst[mid]] >= thresh) lo = mid + 1; else hi = mid;
  }
  counts[t] = lo;
}

// Visiting order of the kets of one (molecule, class) segment: inside each full
// group of kKetGroup positions by decreasing number of primitive pairs (ties by
// position).  One block of kKetGroup threads per group; grid (segment, group).
__global__ void __launch_bounds__(kKetGroup)
    k_ketorder(const int* __restrict__ sorted, const int* __restrict__ coff, const int* __restrict__ segloc,
               const int* __restrict__ ccm, const int* __restrict__ np, int* __restrict__ korder) {
  __shared__ int key[kKetGroup];
  const int s = blockIdx.x, X = s % NPAIRCLASS, n = ccm[s], t = threadIdx.x;
  const int64_t base = (int64_t)coff[X] + segloc[s];
  for (int g = blockIdx.y * kKetGroup; g < n; g += gridDim.y * kKetGroup) {
    const int i = g + t;
    if (g + kKetGroup > n) {  // a partial group keeps the order of the list
      if (i < n) korder[base + i] = i;
      return;
    }
    const int k = np[sorted[base + i]];
    key[t] = k;
    __syncthreads();
    int r = 0;
    for (int j = 0; j < kKetGroup; ++j) r += key[j] > k || (key[j] == k && j < t);
    korder[base + g + r] = i;
    __syncthreads();
  }
}

// Exclusive scan of one int64 per thread over the block (blockDim.x a multiple
// of 32); *total receives the block sum.  Every thread of the block must call it.
__device__ __forceinline__ int64_t block_exscan(int64_t v, int64_t* wsum, int64_t* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int64_t x = v;
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[w] = x;
  __syncthreads();
  if (w == 0) {
    int64_t t = lane < nw ? wsum[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    if (lane < nw) wsum[lane] = t;
  }
  __syncthreads();
  const int64_t before = w > 0 ? wsum[w - 1] : 0;
  *total = wsum[nw - 1];
  __syncthreads();
  return before + x - v;
}

// cumnp[coff[Y] + Y + k] = primitive pairs of the first k entries of class Y's
// sorted list (all molecules, in list order); one block per class
__global__ void k_cumnp(const int* __restrict__ sorted, const int* __restrict__ coff, const int* __restrict__ ccount,
                        const int* __restrict__ np, int64_t* __restrict__ cumnp) {
  __shared__ int64_t wsum[32];
  const int Y = blockIdx.x;
  const int n = ccount[Y];
  const int* kl = sorted + coff[Y];
  int64_t* out = cumnp + coff[Y] + Y;  // class Y occupies ccount[Y] + 1 slots
  int64_t carry = 0;
  for (int base = 0; base < n; base += blockDim.x) {
    const int k = base + threadIdx.x;
    const int64_t v = k < n ? np[kl[k]] : 0;
    int64_t tot;
    const int64_t ex = block_exscan(v, wsum, &tot);
    if (k < n) out[k] = carry + ex;
    carry += tot;
  }
  if (threadIdx.x == 0) out[n] = carry;
}

// Prefix arrays of the K (canonical) and J (ordered) work lists, one block per
// class pair (X, Y).  A bra of class X sees the kets of class Y of its own
// molecule; canonical lists (Y <= X) keep, for X == Y, only kets at or before
// the bra's own rank in the (molecule, class) segment.
__global__ void k_prefix(const int* __restrict__ sorted, const int* __restrict__ coff, const int* __restrict__ ccount,
                         const int* __restrict__ segloc, const int* __restrict__ pmol, const int* __restrict__ pos,
                         const int* __restrict__ counts, const int64_t* __restrict__ koff,
                         const int64_t* __restrict__ joff, int64_t* __restrict__ kpre, int64_t* __restrict__ jpre,
                         int64_t* __restrict__ ktot, int64_t* __restrict__ jtot, const int* __restrict__ np,
                         const int64_t* __restrict__ cumnp, int64_t* __restrict__ kprim) {
  __shared__ int64_t wsum[32];
  const int cp = blockIdx.x;
  const int X = cp / NPAIRCLASS, Y = cp % NPAIRCLASS;
  const bool canon = Y <= X;
  const int nb = ccount[X];
  const int* bl = sorted + coff[X];
  int64_t* jp = jpre + joff[cp];
  int64_t* kp = canon ? kpre + koff[cp] : nullptr;
  const int64_t* cy = cumnp + coff[Y] + Y;
  int64_t cj_carry = 0, ck_carry = 0, cp_carry = 0;
  for (int base = 0; base < nb; base += blockDim.x) {
    const int i = base + threadIdx.x;
    int64_t cj = 0, ck = 0, pp = 0;
    if (i < nb) {
      const int b = bl[i];
      cj = counts[b * NPAIRCLASS + Y];
      if (canon) {
        ck = cj;
        if (X == Y && ck > pos[b] + 1) ck = pos[b] + 1;
        const int s0 = segloc[pmol[b] * NPAIRCLASS + Y];
        pp = (cy[s0 + ck] - cy[s0]) * np[b];
      }
    }
    int64_t tot;
    const int64_t exj = block_exscan(cj, wsum, &tot);
    if (i < nb) jp[i] = cj_carry + exj;
    cj_carry += tot;
    if (canon) {
      const int64_t exk = block_exscan(ck, wsum, &tot);
      if (i < nb) kp[i] = ck_carry + exk;
      ck_carry += tot;
      block_exscan(pp, wsum, &tot);
      cp_carry += tot;
    }
  }
  if (threadIdx.x == 0) {
    jp[nb] = cj_carry;
    jtot[cp] = cj_carry;
    if (canon) {
      kp[nb] = ck_carry;
      ktot[cp] = ck_carry;
      kprim[cp] = cp_carry;
    }
  }
}

// Where each molecule's nbf_m x nbf_m block sits in packed D / J / K, and the
// global AO index of its first function (component factors f are global).

// D' = D f f (component norms folded in); grid (x, molecule)
__global__ void k_scale_d(MolMats mm, const double* __restrict__ D, const double* __restrict__ f,
                          double* __restrict__ Dp, float* __restrict__ Dpf) {
  const int m = blockIdx.y, n = mm.n[m];
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)n * n) return;
  const int64_t o = mm.off[m] + i;
  const int a0 = mm.aobase[m];
  const double v = D[o] * f[a0 + i / n] * f[a0 + i % n];
  Dp[o] = v;
  if (Dpf) Dpf[o] = (float)v;
}

// Hermite density per primitive pair (Eq. j_formula, first sub-step):
// D_Q = (-1)^|Q| s sum_{l in s1, s in s2} E_Q^{ls} D'_ls, s = 2 for s1 != s2
// (the pair stands for both orders), 1 for a diagonal pair.
// One warp per shell pair, a lane per Hermite index (E is zero outside t <= i + j).
__global__ void __launch_bounds__(128)
    k_hermite_density(int npair, const int* __restrict__ s1, const int* __restrict__ s2, const int* __restrict__ np,
                      const int* __restrict__ poff, const int* __restrict__ hoff, const int* __restrict__ eoff,
                      const int* __restrict__ sh_l, const int* __restrict__ pao1, const int* __restrict__ pao2,
                      const int* __restrict__ pmol, MolMats mm, const int* __restrict__ sig, PairData pd,
                      const double* __restrict__ Dp, double* __restrict__ Dh, float* __restrict__ Dhf) {
  const int ip = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (ip >= npair || !sig[ip]) return;
  const int a = s1[ip], b = s2[ip], la = sh_l[a], lb = sh_l[b], lp = la + lb, H = nherm(lp);
  const int ne = (la + 1) * (lb + 1) * (lp + 1);
  const int m = pmol[ip], nbf = mm.n[m];
  const double* Dm = Dp + mm.off[m];
  const double sc = a == b ? 1.0 : 2.0;
  for (int k = 0; k < np[ip]; ++k) {
    const double* E = pd.E + eoff[ip] + (size_t)k * 3 * ne;
    for (int q = lane; q < H; q += 32) {
      const int t = herm_t(q), u = herm_u(q), v = herm_v(q);
      double acc = 0.0;
      for (int mu = 0; mu < ncart(la); ++mu) {
        int ix, iy, iz;
        cart_xyz(la, mu, ix, iy, iz);
        for (int nu = 0; nu < ncart(lb); ++nu) {
          int jx, jy, jz;
          cart_xyz(lb, nu, jx, jy, jz);
          const double e = E[(ix * (lb + 1) + jx) * (lp + 1) + t] * E[ne + (iy * (lb + 1) + jy) * (lp + 1) + u] *
                           E[2 * ne + (iz * (lb + 1) + jz) * (lp + 1) + v];
          acc = fma(Dm[(size_t)(pao1[ip] + mu) * nbf + pao2[ip] + nu], e, acc);
        }
      }
      acc *= (t + u + v) & 1 ? -sc : sc;
      const size_t o = hoff[ip] + (size_t)k * H + q;
      Dh[o] = acc;
      if (Dhf) Dhf[o] = (float)acc;  // FP32 copy for the FP32 tier of a mixed J-engine build
    }
  }
}

// Cartesian J from Hermite J (Eq. j_formula, last sub-step): thread per (pair, mu, nu)
__global__ void k_post_j(int npair, const int* __restrict__ s1, const int* __restrict__ s2, const int* __restrict__ np,
                         const int* __restrict__ hoff, const int* __restrict__ eoff, const int* __restrict__ sh_l,
                         const int* __restrict__ pao1, const int* __restrict__ pao2, const int* __restrict__ pmol,
                         MolMats mm, const int* __restrict__ sig, const double* __restrict__ E,
                         const double* __restrict__ Jh, const double* __restrict__ f, double* __restrict__ J, int det,
                         int* __restrict__ status) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= npair * 100) return;
  const int ip = t / 100, c = t % 100;
  if (sig && !sig[ip]) return;
  const int a = s1[ip], b = s2[ip], la = sh_l[a], lb = sh_l[b], lp = la + lb;
  const int mu = c / 10, nu = c % 10;
  if (mu >= ncart(la) || nu >= ncart(lb)) return;
  int ix, iy, iz, jx, jy, jz;
  cart_xyz(la, mu, ix, iy, iz);
  cart_xyz(lb, nu, jx, jy, jz);
  const int H = nherm(lp), ne = (la + 1) * (lb + 1) * (lp + 1);
  double v = 0.0;
  for (int k = 0; k < np[ip]; ++k) {
    const double* e = E + eoff[ip] + (size_t)k * 3 * ne;  // the tables of k_etab
    const double *ex = e + (ix * (lb + 1) + jx) * (lp + 1), *ey = e + ne + (iy * (lb + 1) + jy) * (lp + 1),
                 *ez = e + 2 * ne + (iz * (lb + 1) + jz) * (lp + 1);
    const double* jh = Jh + hoff[ip] + (size_t)k * H;
    for (int tx = 0; tx <= ix + jx; ++tx)
      for (int ty = 0; ty <= iy + jy; ++ty)
        for (int tz = 0; tz <= iz + jz; ++tz) {
          const double hv = acc_value(jh + herm_index(tx, ty, tz), det);
          if (det && fabs(hv) > kFixLimit) atomicOr(status, DEV_RANGE);
          v += ex[tx] * ey[ty] * ez[tz] * hv;
        }
  }
  const int m = pmol[ip], nbf = mm.n[m], a0 = mm.aobase[m];
  const int r = pao1[ip] + mu, cc = pao2[ip] + nu;
  v *= f[a0 + r] * f[a0 + cc];
  double* Jm = J + mm.off[m];
  Jm[(size_t)r * nbf + cc] = v;
  if (a != b) Jm[(size_t)cc * nbf + r] = v;
}

// K = (Kh + Kh^T) f f  (Eq. 8_fold_symmetry: the transposes carry permutations 5-8); grid (x, molecule)
// (deterministic builds: Kh holds fixed point, see acc_add; an element above the
// reporting limit sets DEV_RANGE in the plan's status word)
__global__ void k_post_k(MolMats mm, const double* __restrict__ Kh, const double* __restrict__ f,
                         double* __restrict__ K, int det, int* __restrict__ status) {
  const int m = blockIdx.y, n = mm.n[m];
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)n * n) return;
  const int r = (int)(i / n), c = (int)(i % n), a0 = mm.aobase[m];
  const int64_t o = mm.off[m];
  const double x = acc_value(Kh + o + i, det), y = acc_value(Kh + o + (int64_t)c * n + r, det);
  if (det && (fabs(x) > kFixLimit || fabs(y) > kFixLimit)) atomicOr(status, DEV_RANGE);
  K[o + i] = (x + y) * f[a0 + r] * f[a0 + c];
}

// deterministic gradient: fixed-point accumulators -> doubles, in place
__global__ void k_fix_to_double(int n, double* __restrict__ x, int* __restrict__ status) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = acc_value(x + i, 1);
  if (fabs(v) > kFixLimit) atomicOr(status, DEV_RANGE);
  x[i] = v;
}

// E_J = 1/2 sum D J, E_K = -1/4 sum D K per molecule (one block each, fixed
// order: deterministic); E[2m], E[2m+1]
__global__ void k_energy(MolMats mm, const double* __restrict__ D, const double* __restrict__ J,
                         const double* __restrict__ K, double* __restrict__ E) {
  __shared__ double sj[32], sk[32];
  const int m = blockIdx.x;
  const int64_t nn = (int64_t)mm.n[m] * mm.n[m], o = mm.off[m];
  double aj = 0.0, ak = 0.0;
  for (int64_t i = threadIdx.x; i < nn; i += blockDim.x) {
    if (J) aj += D[o + i] * J[o + i];
    if (K) ak += D[o + i] * K[o + i];
  }
  for (int w = 16; w > 0; w >>= 1) {
    aj += __shfl_xor_sync(0xffffffffu, aj, w);
    ak += __shfl_xor_sync(0xffffffffu, ak, w);
  }
  if ((threadIdx.x & 31) == 0) { sj[threadIdx.x >> 5] = aj; sk[threadIdx.x >> 5] = ak; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double tj = 0.0, tk = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { tj += sj[w]; tk += sk[w]; }
    E[2 * m] = 0.5 * tj;
    E[2 * m + 1] = -0.25 * tk;
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

#define CK(x)                                   \
  do {                                          \
    cudaError_t e_ = (x);                       \
    if (e_ != cudaSuccess) return eri_fail(e_); \
  } while (0)

static int eri_fail(cudaError_t e) {
  if (e == cudaErrorMemoryAllocation) return ERI_ENOMEM;
  return ERI_ECUDA;
}

template <typename T>
static cudaError_t dalloc(T** p, size_t n) {
  *p = nullptr;
  if (n == 0) n = 1;
  return cudaMalloc((void**)p, n * sizeof(T));
}

static int grid1(int64_t n, int b) { return (int)((n + b - 1) / b); }

static std::vector<RStep> make_rsteps() {
  std::vector<RStep> st(nherm(LMAX_QUARTET));
  for (int n = 0; n <= LMAX_QUARTET; ++n)
    for (int r = 0; r <= n; ++r)
      for (int v = 0; v <= r; ++v) {
        int u = r - v, t = n - r;
        int e = herm_index(t, u, v);
        RStep s{};
        s.t = (uint8_t)t; s.u = (uint8_t)u; s.v = (uint8_t)v;
        s.dep1 = -1; s.dep2 = -1; s.k = 0; s.dir = 0;
        int c[3] = {t, u, v};
        if (n > 0) {
          int d = t > 0 ? 0 : (u > 0 ? 1 : 2);
          s.dir = (uint8_t)d;
          int c1[3] = {c[0], c[1], c[2]};
          c1[d] -= 1;
          s.dep1 = (int16_t)herm_index(c1[0], c1[1], c1[2]);
          if (c1[d] > 0) {
            int c2[3] = {c1[0], c1[1], c1[2]};
            c2[d] -= 1;
            s.dep2 = (int16_t)herm_index(c2[0], c2[1], c2[2]);
            s.k = (int16_t)c1[d];
          }
        }
        st[e] = s;
      }
  return st;
}

int eri_plan_impl::alloc_pairs() {
  CK(dalloc(&d_p, nprimpair)); CK(dalloc(&d_P, 3 * (size_t)nprimpair)); CK(dalloc(&d_PA, 3 * (size_t)nprimpair));
  CK(dalloc(&d_PB, 3 * (size_t)nprimpair)); CK(dalloc(&d_pref, nprimpair));
  CK(dalloc(&d_pf, nprimpair)); CK(dalloc(&d_Pf, 3 * (size_t)nprimpair)); CK(dalloc(&d_PAf, 3 * (size_t)nprimpair));
  CK(dalloc(&d_PBf, 3 * (size_t)nprimpair)); CK(dalloc(&d_preff, nprimpair));
  CK(dalloc(&d_q4, 3 * (size_t)nprimpair));
  return ERI_OK;
}

PairData eri_plan_impl::pairdata() const {
  PairData pd;
  pd.p = d_p; pd.P = d_P; pd.PA = d_PA; pd.PB = d_PB; pd.pref = d_pref;
  pd.pf = d_pf; pd.Pf = d_Pf; pd.PAf = d_PAf; pd.PBf = d_PBf; pd.preff = d_preff;
  pd.E = d_E; pd.Ef = d_Ef; pd.ea = d_ea; pd.q4 = d_q4;
  pd.n = nprimpair;
  return pd;
}

BoysTabs eri_plan_impl::boystabs() const {
  BoysTabs b;
  b.c64 = d_boys64; b.e64 = d_bexp64; b.c32 = d_boys32; b.e32 = d_bexp32;
  return b;
}

ShellPairInfo eri_plan_impl::spinfo() const {
  ShellPairInfo sp;
  sp.s1 = d_ps1; sp.s2 = d_ps2; sp.np = d_pnk; sp.poff = d_ppoff; sp.ao1 = d_pao1; sp.ao2 = d_pao2; sp.hoff = d_phoff; sp.eoff = d_peoff;
  sp.pmol = d_pmol; sp.mat_off = d_mat_off; sp.mat_n = d_mat_n;
  return sp;
}

dim3 eri_plan_impl::mat_grid(int block) const {
  return dim3((unsigned)std::max<int64_t>(1, ((int64_t)max_nbf * max_nbf + block - 1) / block), (unsigned)nmol);
}

// D' = D f f into the plan's FP64 workspace (also used by nuclear.cu)
void k_scale_d_launch(const eri_plan_impl* P, const double* D, cudaStream_t s) {
  k_scale_d<<<P->mat_grid(256), 256, 0, s>>>(molmats(P), D, P->d_f, P->d_Dp, nullptr);
}

MolMats molmats(const eri_plan_impl* P) {
  MolMats m;
  m.off = P->d_mat_off; m.n = P->d_mat_n; m.aobase = P->d_aobase;
  return m;
}

// pair data + Schwarz + lists for the current device coordinates
int eri_plan_impl::geometry(cudaStream_t s, bool rebuild_q) {
  k_pairs<<<grid1(npair, 4), 128, 0, s>>>(npair, d_ps1, d_ps2, d_ppoff, d_sh_atom, d_sh_np, d_sh_po, d_exps, d_cn,
                                        d_coords, nprimpair, d_p, d_P, d_PA, d_PB, d_pref, d_pf, d_Pf, d_PAf, d_PBf,
                                        d_preff, d_pmaxp, d_prefmaxp, d_ea, d_q4);
  CK(cudaGetLastError());
  k_etab<<<grid1(npair, 4), 128, 0, s>>>(npair, d_ps1, d_ps2, d_pnp, d_ppoff, d_peoff, d_sh_l, pairdata(), d_E, d_Ef);
  CK(cudaGetLastError());
  if (rebuild_q) {
    k_schwarz<<<npair, 32 * kSchwarzWarps, 0, s>>>(npair, d_ps1, d_ps2, d_pnp, d_ppoff, d_peoff,
                                                                         d_sh_l, d_sh_ao, d_f, pairdata(), boystabs(),
                                                                         d_rsteps, d_Q);
    CK(cudaGetLastError());
  }
  CK(cudaMemsetAsync(d_pqmax, 0, sizeof(unsigned int) * nmol, s));
  k_primq<<<grid1(npair, 4), 128, 0, s>>>(npair, d_ps1, d_ps2, d_pnp, d_ppoff, d_peoff, d_sh_l, d_sh_ao, d_f, d_pmol,
                                          pairdata(), d_pq, d_pqmax);
  CK(cudaGetLastError());
  return rebuild_q ? build_lists(thresh, s) : pack_primitives(s);
}

int eri_plan_impl::pack_primitives(cudaStream_t s) {
  k_primpack<<<grid1(npair, 4), 128, 0, s>>>(npair, d_ps1, d_ps2, d_pnp, d_ppoff, d_peoff, d_sh_l, d_pmol, d_pqmax,
                                             kPrimEps * thresh, nprimpair, d_pq, d_p, d_P, d_PA, d_PB, d_pref, d_ea,
                                             d_pf, d_Pf, d_PAf, d_PBf, d_preff, d_q4, d_E, d_Ef, d_pnk);
  CK(cudaGetLastError());
  return ERI_OK;
}

int eri_plan_impl::build_lists(double th, cudaStream_t s) {
  thresh = th;
  if (gexec) {  // a captured build holds the old list sizes and offsets
    CK(cudaDeviceSynchronize());
    CK(cudaGraphExecDestroy(gexec));
    gexec = nullptr;
  }
  int rc = pack_primitives(s);
  if (rc != ERI_OK) return rc;
  const int nm10 = nmol * NPAIRCLASS;
  CK(cudaMemsetAsync(d_qmax, 0, sizeof(unsigned int) * nmol, s));
  CK(cudaMemsetAsync(d_ccm, 0, sizeof(int) * nm10, s));
  k_qmax<<<grid1(npair, 256), 256, 0, s>>>(npair, d_Q, d_pmol, d_qmax);
  k_sig<<<grid1(npair, 256), 256, 0, s>>>(npair, d_Q, d_pmol, d_qmax, th, d_pcls, d_sig, d_ccm);
  CK(cudaGetLastError());
  h_ccm.assign(nm10, 0);
  CK(cudaMemcpyAsync(h_ccm.data(), d_ccm, sizeof(int) * nm10, cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  // class-major layout, molecule by molecule inside a class
  h_segloc.assign(nm10, 0);
  int acc = 0;
  for (int X = 0; X < NPAIRCLASS; ++X) {
    h_coff[X] = acc;
    int loc = 0;
    for (int m = 0; m < nmol; ++m) {
      h_segloc[m * NPAIRCLASS + X] = loc;
      loc += h_ccm[m * NPAIRCLASS + X];
    }
    h_ccount[X] = loc;
    acc += loc;
  }
  nsig = acc;
  CK(cudaMemcpyAsync(d_coff, h_coff, sizeof(int) * NPAIRCLASS, cudaMemcpyHostToDevice, s));
  CK(cudaMemcpyAsync(d_ccount, h_ccount, sizeof(int) * NPAIRCLASS, cudaMemcpyHostToDevice, s));
  CK(cudaMemcpyAsync(d_segloc, h_segloc.data(), sizeof(int) * nm10, cudaMemcpyHostToDevice, s));
  k_rank<<<grid1(npair, 256), 256, 0, s>>>(npair, d_Q, d_pcls, d_sig, d_pmol, d_pbase, d_coff, d_segloc, d_sorted,
                                           d_pos);
  k_counts<<<grid1((int64_t)npair * NPAIRCLASS, 256), 256, 0, s>>>(npair, d_Q, d_sig, d_pmol, d_sorted, d_coff,
                                                                   d_segloc, d_ccm, th, d_counts);
  k_ketorder<<<dim3(nm10, 16), kKetGroup, 0, s>>>(d_sorted, d_coff, d_segloc, d_ccm, d_pnk, d_korder);
  CK(cudaGetLastError());
  int64_t ko = 0, jo = 0;
  for (int X = 0; X < NPAIRCLASS; ++X)
    for (int Y = 0; Y < NPAIRCLASS; ++Y) {
      h_koff[X * NPAIRCLASS + Y] = ko;
      h_joff[X * NPAIRCLASS + Y] = jo;
      jo += h_ccount[X] + 1;
      if (Y <= X) ko += h_ccount[X] + 1;
    }
  if (ko > kpre_cap) {
    cudaFree(d_kpre);
    CK(dalloc(&d_kpre, ko));
    kpre_cap = ko;
  }
  if (jo > jpre_cap) {
    cudaFree(d_jpre);
    CK(dalloc(&d_jpre, jo));
    jpre_cap = jo;
  }
  CK(cudaMemcpyAsync(d_koff, h_koff, sizeof(h_koff), cudaMemcpyHostToDevice, s));
  CK(cudaMemcpyAsync(d_joff, h_joff, sizeof(h_joff), cudaMemcpyHostToDevice, s));
  k_cumnp<<<NPAIRCLASS, 1024, 0, s>>>(d_sorted, d_coff, d_ccount, d_pnp, d_cumnp);
  k_prefix<<<NPAIRCLASS * NPAIRCLASS, 1024, 0, s>>>(d_sorted, d_coff, d_ccount, d_segloc, d_pmol, d_pos, d_counts,
                                                     d_koff, d_joff, d_kpre, d_jpre, d_ktot, d_jtot, d_pnp, d_cumnp,
                                                     d_kprim);
  CK(cudaGetLastError());
  CK(cudaMemcpyAsync(h_ktot, d_ktot, sizeof(h_ktot), cudaMemcpyDeviceToHost, s));
  CK(cudaMemcpyAsync(h_jtot, d_jtot, sizeof(h_jtot), cudaMemcpyDeviceToHost, s));
  CK(cudaMemcpyAsync(h_kprim, d_kprim, sizeof(h_kprim), cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  // Tier lists that have become too short are replaced here and by no later call: a
  // build that the caller captures, in FP64 too, holds their addresses, and it is
  // good until the next list rebuild.  (Without room for them the plan has none.)
  if (tier_nb > 0 && tier_len() > tier_cap && ensure_tier_bufs(1) != ERI_OK) cudaGetLastError();
  return ERI_OK;
}

WorkList eri_plan_impl::klist(int X, int Y) const {
  WorkList w;
  w.first = 0;
  w.tile = 1;
  w.shard = shard;
  w.nshard = nshard;
  w.bra = d_sorted + h_coff[X];
  w.ket = d_sorted + h_coff[Y];
  w.kseg = d_segloc + Y;
  w.korder = d_korder + h_coff[Y];
  w.prefix = d_kpre + h_koff[X * NPAIRCLASS + Y];
  w.nbra = h_ccount[X];
  w.total = h_ktot[X * NPAIRCLASS + Y];
  w.mpb = h_maxnp[X];
  w.mpk = h_maxnp[Y];
  return w;
}

WorkList eri_plan_impl::jlist(int X, int Y) const {
  WorkList w;
  w.first = 0;
  w.tile = 4;
  w.shard = shard;
  w.nshard = nshard;
  w.bra = d_sorted + h_coff[X];
  w.ket = d_sorted + h_coff[Y];
  w.kseg = d_segloc + Y;
  w.korder = d_korder + h_coff[Y];
  w.prefix = d_jpre + h_joff[X * NPAIRCLASS + Y];
  w.nbra = h_ccount[X];
  w.total = h_jtot[X * NPAIRCLASS + Y];
  w.mpb = h_maxnp[X];
  w.mpk = h_maxnp[Y];
  return w;
}

void eri_plan_impl::release() {
  void* ptrs[] = {d_sh_l, d_sh_atom, d_sh_np, d_sh_po, d_sh_ao, d_exps, d_coefs, d_cn, d_f, d_coords, d_ps1, d_ps2,
                  d_pnp, d_ppoff, d_pao1, d_pao2, d_phoff, d_pcls, d_p, d_P, d_PA, d_PB, d_pref, d_pf, d_Pf, d_PAf,
                  d_PBf, d_preff, d_Q, d_qmax, d_sig, d_ccount, d_coff, d_sorted, d_pos, d_counts, d_koff, d_joff,
                  d_kpre, d_jpre, d_ktot, d_jtot, d_kprim, d_boys64, d_boys32, d_rsteps, d_Dp, d_Kh, d_Jh, d_Dherm,
                  d_Jherm, d_status, d_bexp64, d_bexp32, d_peoff, d_E, d_Ef, d_pmaxp, d_dmax, d_counters, d_cumnp, d_prefmaxp, d_ea,
                  d_mat_off, d_mat_n, d_aobase, d_pbase, d_pmol, d_shloc, d_ccm, d_segloc, d_Dpf,
                  d_nuc_list, d_nuc_goff, d_nuc_dens, d_counters2, d_q4, d_Dhermf, d_pq, d_pqmax, d_pnk, d_korder};
  xc_release();
  for (auto& e : prof_events) cudaEventDestroy(e);
  prof_events.clear();
  if (gexec) cudaGraphExecDestroy(gexec);
  gexec = nullptr;
  for (int b = 0; b < kStreams; ++b) {
    if (branch[b]) cudaStreamDestroy(branch[b]);
    if (join_ev[b]) cudaEventDestroy(join_ev[b]);
    branch[b] = nullptr;
    join_ev[b] = nullptr;
  }
  for (int b = 0; b < kStreams; ++b) {
    if (tbuf[b]) cudaFree(tbuf[b]);
    tbuf[b] = nullptr;
  }
  if (tcnt) cudaFree(tcnt);
  tcnt = nullptr;
  if (fork_ev) cudaEventDestroy(fork_ev);
  if (cap_stream) cudaStreamDestroy(cap_stream);
  fork_ev = nullptr;
  cap_stream = nullptr;
  for (void* p : ptrs)
    if (p) cudaFree(p);
}

// pairs with an exponent sum above this stay in FP64 in mixed mode (FP32 range)
static const double kPmax32 = 1.0e3;

static const int kClassL1[NPAIRCLASS] = {0, 1, 1, 2, 2, 2, 3, 3, 3, 3};
static const int kClassL2[NPAIRCLASS] = {0, 0, 1, 0, 1, 2, 0, 1, 2, 3};

static void ensure_order_bufs(eri_plan_impl* P);

int eri_plan_impl::ensure_streams() {
  if (cap_stream) return ERI_OK;
  CK(cudaStreamCreateWithFlags(&cap_stream, cudaStreamNonBlocking));
  CK(cudaEventCreateWithFlags(&fork_ev, cudaEventDisableTiming));
  for (int b = 0; b < kStreams; ++b) {
    CK(cudaStreamCreateWithFlags(&branch[b], cudaStreamNonBlocking));
    CK(cudaEventCreateWithFlags(&join_ev[b], cudaEventDisableTiming));
  }
  return ERI_OK;
}

// longest compacted tier list (items); longer class-pair lists are split in windows
static const int64_t kTierCap = 1 << 23;

// Eager calls overlap their class launches (independent sums into the same
// accumulators) on the plan's side streams: a small molecule's fifty launches
// hold a few blocks each, and one after another they leave most SMs idle.
// Profiled calls run in order on the caller's stream, so that an event pair
// times one launch.
// With tier lists the streams are as many (4 to kStreams) as keep the lists
// within 512 MB, at the length they have or would get.
int eri_plan_impl::eager_branches(bool lists) const {
  if (opts.profile) return 0;
  int n = kStreams;
  if (lists) {
    int64_t mx = 1;
    for (int64_t t : h_jtot) mx = std::max(mx, t);
    mx = std::max(tier_cap, std::min(mx, kTierCap));
    while (n > kBranches && n * mx > (int64_t)1 << 25) n /= 2;
  }
  return n;
}

// Compacted tier lists of mixed-precision builds: per branch, two lists of
// tier_cap items (int2 bra / ket positions) and two counters.  tier_cap is the
// longest class-pair list, at most kTierCap; longer lists are split in windows.
// The first call that needs lists takes those of every stream of an eager build, so
// that no later call allocates until the lists grow; builds run over no more
// streams than there are lists.  An error only if fewer than `need` could be had.
int64_t eri_plan_impl::tier_len() const {
  int64_t mx = 1;
  for (int X = 0; X < NPAIRCLASS; ++X)
    for (int Y = 0; Y <= X; ++Y) mx = std::max(mx, h_ktot[X * NPAIRCLASS + Y]);
  return std::min(mx, kTierCap);
}

int eri_plan_impl::ensure_tier_bufs(int need) {
  const int64_t cap = tier_len();
  if (tier_nb == 0) {
    tier_cap = cap;
  } else if (cap > tier_cap) {
    CK(cudaDeviceSynchronize());
    for (int b = 0; b < kStreams; ++b) {
      if (tbuf[b]) cudaFree(tbuf[b]);
      tbuf[b] = nullptr;
    }
    tier_nb = 0;
    // (lists that grow once, atoms moving closer, grow again: an eighth to spare)
    tier_cap = std::min(kTierCap, cap + cap / 8);
  }
  if (!tcnt) CK(dalloc(&tcnt, 2 * kStreams));
  const int want = tier_nb == 0 ? std::max(need, eager_branches(true)) : need;
  for (; tier_nb < want; ++tier_nb)
    if (const cudaError_t e = dalloc(&tbuf[tier_nb], 2 * (size_t)tier_cap)) {
      tbuf[tier_nb] = nullptr;
      if (tier_nb < need) return eri_fail(e);
      cudaGetLastError();  // fewer streams
      break;
    }
  return ERI_OK;
}

// tier split of the window ka.wl into buf (FP64 tier) and buf + tier_cap (FP32 tier)
static cudaError_t launch_tier_split(const eri_plan_impl* P, const KArgs& ka, int2* buf, unsigned int* cnt,
                                     cudaStream_t s) {
  const int64_t items = ka.wl.total - ka.wl.first, warps = (int64_t)P->nsm * 64;
  // long runs sort better; they may leave this kernel short of warps (8 per SM), not the tiers' kernels
  const int rounds =
      ka.wl.nshard > 1 ? 1 : (int)std::max<int64_t>(1, std::min<int64_t>(kSplitRounds, items / (4 * warps)));
  const int64_t runs = (items + 32 * rounds - 1) / (32 * rounds);
  k_tier_split<<<(int)std::max<int64_t>(1, std::min<int64_t>((runs + 7) / 8, warps / 8)), 256, 0, s>>>(
      ka, rounds, buf, buf + P->tier_cap, cnt);
  return cudaGetLastError();
}

cudaError_t eri_plan_impl::prof_event_pair(cudaEvent_t* a, cudaEvent_t* b) {
  while ((int)prof_events.size() < prof_ev_used + 2) {
    cudaEvent_t e;
    cudaError_t r = cudaEventCreate(&e);
    if (r != cudaSuccess) return r;
    prof_events.push_back(e);
  }
  *a = prof_events[prof_ev_used];
  *b = prof_events[prof_ev_used + 1];
  prof_ev_used += 2;
  return cudaSuccess;
}

// Algorithmic FLOPs of the McMurchie-Davidson J/K path as implemented (FMA = 2):
//   per primitive quartet: Boys 2(L+1)+20, R recursion 3 sum_{m<L} (nherm(L-m)-1),
//     ket transform 2 nherm(la+lb) sum_{cd} prod_t (k_t+l_t+1);
//   per bra primitive of a quartet: bra transform 2 ncd sum_{ab} prod_t (i_t+j_t+1);
//   per contracted quartet: K 8 nab ncd, J 4 nab ncd.
static double sum_terms(int la, int lb) {
  double s = 0.0;
  for (int x = 0; x < ncart(la); ++x)
    for (int y = 0; y < ncart(lb); ++y) {
      int ix, iy, iz, jx, jy, jz;
      cart_xyz(la, x, ix, iy, iz);
      cart_xyz(lb, y, jx, jy, jz);
      s += (double)(ix + jx + 1) * (iy + jy + 1) * (iz + jz + 1);
    }
  return s;
}
static double class_flops(int X, int Y, double nq, double npq, double nbp, bool dj, bool dk) {
  const int la = kClassL1[X], lb = kClassL2[X], lc = kClassL1[Y], ld = kClassL2[Y];
  const int L = la + lb + lc + ld;
  double rf = 0.0;
  for (int m = 0; m < L; ++m) rf += 3.0 * (nherm(L - m) - 1);
  const double nab = ncart(la) * ncart(lb), ncd = ncart(lc) * ncart(ld);
  const double per_pq = 2.0 * (L + 1) + 20.0 + rf + 2.0 * nherm(la + lb) * sum_terms(lc, ld);
  const double per_bp = 2.0 * ncd * sum_terms(la, lb);
  const double per_q = (dk ? 8.0 : 0.0) * nab * ncd + (dj ? 4.0 : 0.0) * nab * ncd;
  return npq * per_pq + nbp * per_bp + nq * per_q;
}

// J-engine (Eq. j_formula) per primitive quartet of an ordered (bra, ket) item:
// Boys 2(L+1)+20, R recursion, J_P += sum_Q R_{P+Q} D_Q: 2 nherm(lab) nherm(lcd).
static double jengine_flops(int X, int Y, double npq) {
  const int lab = kClassL1[X] + kClassL2[X], lcd = kClassL1[Y] + kClassL2[Y], L = lab + lcd;
  double rf = 0.0;
  for (int m = 0; m < L; ++m) rf += 3.0 * (nherm(L - m) - 1);
  return npq * (2.0 * (L + 1) + 20.0 + rf + 2.0 * nherm(lab) * nherm(lcd));
}

// Gradient (bra derivatives, SI Eq. si_dE_J / si_dE_K) per ordered item:
//   per primitive quartet: Boys 2(L+2)+20, R recursion to L+1, ket transform
//     2 nherm(lab+1) sum_{cd} prod_t (k_t+l_t+1);
//   per bra primitive: for every (ab, cd), direction t opened to n_t+1 (raised
//     Hermite index) and the other two closed: 2 sum_t (n_t+2) prod_{u!=t} (n_u+1)
//     plus 4 (n_t+2) for the A and B coefficients;
//   per item: the density factor, 8 FLOPs per (ab, cd).
static double grad_flops(int X, int Y, double nq, double npq, double nbp) {
  const int la = kClassL1[X], lb = kClassL2[X], lc = kClassL1[Y], ld = kClassL2[Y];
  const int L1 = la + lb + lc + ld + 1;
  double rf = 0.0;
  for (int m = 0; m < L1; ++m) rf += 3.0 * (nherm(L1 - m) - 1);
  double dab = 0.0;
  for (int x = 0; x < ncart(la); ++x)
    for (int y = 0; y < ncart(lb); ++y) {
      int ix, iy, iz, jx, jy, jz;
      cart_xyz(la, x, ix, iy, iz);
      cart_xyz(lb, y, jx, jy, jz);
      const int n[3] = {ix + jx, iy + jy, iz + jz};
      for (int t = 0; t < 3; ++t)
        dab += 2.0 * (n[t] + 2) * (n[(t + 1) % 3] + 1) * (n[(t + 2) % 3] + 1) + 4.0 * (n[t] + 2);
    }
  const double nab = ncart(la) * ncart(lb), ncd = ncart(lc) * ncart(ld);
  const double per_pq = 2.0 * (L1 + 1) + 20.0 + rf + 2.0 * nherm(la + lb + 1) * sum_terms(lc, ld);
  return npq * per_pq + nbp * ncd * dab + nq * 8.0 * nab * ncd;
}

// Default work-tile length: the thread kernel's lanes already take adjacent
// items; a warp or block takes 4 consecutive quartets (mostly one bra) per tile,
// fewer on short lists (item_tile).
static int default_tile(int X, int Y, int tier) {
  return use_thread_kernel(kClassL1[X], kClassL2[X], kClassL1[Y], kClassL2[Y], tier == 1) ? 1 : 4;
}

int eri_plan_impl::tile_for(int X, int Y, int tier) const {
  const int t = tile_k[(X * NPAIRCLASS + Y) * 2 + tier];
  return t > 0 ? t : default_tile(X, Y, tier);
}

static cudaError_t launch_jk_class(int X, int Y, int prec, const JKArgs& ja, cudaStream_t s, int nsm) {
#define ERI_JK_UNIT_CALL(UX, UP, YLO, YHI) \
  if (X == UX && prec == UP && Y >= YLO && Y <= YHI) return launch_jk_unit<UX, UP, YLO, YHI>(Y, ja, s, nsm);
  ERI_JK_UNITS(ERI_JK_UNIT_CALL)
#undef ERI_JK_UNIT_CALL
  return cudaErrorInvalidValue;
}

extern "C" int eri_default_opts(eri_opts_t* o) {
  if (!o) return ERI_EINVAL;
  o->thresh = 1e-12;
  o->precision = ERI_FP64;
  o->mixed_tau = 1e-5;
  o->device = -1;
  o->j_engine = 1;
  o->profile = 0;
  o->tune_cache = nullptr;
  o->deterministic = 0;
  o->density_screen = 0;
  return ERI_OK;
}

// Tile cache file (opts.tune_cache): one line per entry,
//   <key> t_0 ... t_199      key = <device name>|nbf=<n>|nmol=<m>|npair=<p>|prec=<0|1>
// with spaces in the device name replaced by '_', the tiles in eri_get_tiles order.
static std::string tune_key(const eri_plan_impl* P, int precision) {
  cudaDeviceProp prop;
  std::string name = cudaGetDeviceProperties(&prop, P->device) == cudaSuccess ? prop.name : "unknown";
  for (char& c : name)
    if (c == ' ') c = '_';
  char buf[160];
  snprintf(buf, sizeof(buf), "|nbf=%d|nmol=%d|npair=%d|prec=%d", P->nbf, P->nmol, P->npair, precision);
  return name + buf;
}

static std::vector<std::string> read_lines(const std::string& path) {
  std::vector<std::string> out;
  FILE* f = fopen(path.c_str(), "r");
  if (!f) return out;
  std::string cur;
  int ch;
  while ((ch = fgetc(f)) != EOF) {
    if (ch == '\n') {
      if (!cur.empty()) out.push_back(cur);
      cur.clear();
    } else {
      cur.push_back((char)ch);
    }
  }
  if (!cur.empty()) out.push_back(cur);
  fclose(f);
  return out;
}

// Load the entry for (this plan, precision) into tile_k; a missing file or
// entry leaves the tiles unchanged.  Malformed entries are ignored.
static void tune_cache_load(eri_plan_impl* P, int precision) {
  if (P->tune_cache.empty()) return;
  const std::string key = tune_key(P, precision) + " ";
  for (const std::string& ln : read_lines(P->tune_cache)) {
    if (ln.compare(0, key.size(), key) != 0) continue;
    int t[NPAIRCLASS * NPAIRCLASS * 2];
    const char* c = ln.c_str() + key.size();
    int k = 0;
    for (; k < NPAIRCLASS * NPAIRCLASS * 2; ++k) {
      char* e = nullptr;
      const long v = strtol(c, &e, 10);
      if (e == c || v < 0 || v > 1024) break;
      t[k] = (int)v;
      c = e;
    }
    if (k == NPAIRCLASS * NPAIRCLASS * 2) memcpy(P->tile_k, t, sizeof(t));
  }
}

// Store tile_k as the entry for (this plan, precision), replacing an older one
// (write to a temporary file, then rename).  Returns ERI_EINVAL if the file
// cannot be written.
static int tune_cache_store(const eri_plan_impl* P, int precision) {
  if (P->tune_cache.empty()) return ERI_OK;
  const std::string key = tune_key(P, precision);
  std::vector<std::string> lines;
  for (const std::string& ln : read_lines(P->tune_cache))
    if (ln.compare(0, key.size() + 1, key + " ") != 0) lines.push_back(ln);
  std::string mine = key;
  for (int X = 0; X < NPAIRCLASS; ++X)
    for (int Y = 0; Y < NPAIRCLASS; ++Y)
      for (int t = 0; t < 2; ++t) mine += " " + std::to_string(Y <= X ? P->tile_for(X, Y, t) : 0);
  lines.push_back(mine);
  const std::string tmp = P->tune_cache + ".tmp" + std::to_string((long long)(uintptr_t)P);
  FILE* f = fopen(tmp.c_str(), "w");
  if (!f) return ERI_EINVAL;
  for (const std::string& ln : lines) fprintf(f, "%s\n", ln.c_str());
  const bool ok = fclose(f) == 0;
  if (!ok || rename(tmp.c_str(), P->tune_cache.c_str()) != 0) {
    remove(tmp.c_str());
    return ERI_EINVAL;
  }
  return ERI_OK;
}

static int check_basis(const eri_basis_t* basis, const double* coords, int* nprim_out) {
  if (!basis || !coords || !basis->shells || !basis->exps || !basis->coefs) return ERI_EINVAL;
  const int ns = basis->nshell, na = basis->natom;
  if (ns <= 0 || na <= 0 || ns > 100000) return ERI_EINVAL;
  int nprim_tot = 0;
  for (int s = 0; s < ns; ++s) {
    const eri_shell_t& sh = basis->shells[s];
    if (sh.l < 0 || sh.l > LMAX || sh.nprim <= 0 || sh.nprim > 64 || sh.atom < 0 || sh.atom >= na ||
        sh.prim_offset < 0)
      return sh.l > LMAX ? ERI_EUNSUPPORTED : ERI_EINVAL;
    nprim_tot = std::max(nprim_tot, sh.prim_offset + sh.nprim);
  }
  for (int i = 0; i < nprim_tot; ++i)
    if (!(basis->exps[i] > 0.0) || !std::isfinite(basis->exps[i]) || !std::isfinite(basis->coefs[i])) return ERI_EINVAL;
  for (int i = 0; i < 3 * na; ++i)
    if (!std::isfinite(coords[i])) return ERI_EINVAL;
  *nprim_out = nprim_tot;
  return ERI_OK;
}

template <typename T>
static cudaError_t upload(T* d, const std::vector<T>& h) {
  return cudaMemcpy(d, h.data(), sizeof(T) * h.size(), cudaMemcpyHostToDevice);
}

// One plan over nmol independent molecules.  Shells, atoms and primitives are
// numbered globally (molecule after molecule); shell pairs are formed inside
// each molecule only, pair index pairbase[m] + a(a+1)/2 + b for local shells a >= b.
static int plan_create(int nmol, const eri_basis_t* const* bases, const double* const* coords, const eri_opts_t* opts,
                       eri_plan_t** out) {
  if (!out || nmol <= 0 || nmol > 65535 || !bases || !coords) return ERI_EINVAL;
  *out = nullptr;
  std::vector<int> nprim_m(nmol);
  for (int m = 0; m < nmol; ++m) {
    const int rc = check_basis(bases[m], coords[m], &nprim_m[m]);
    if (rc != ERI_OK) return rc;
  }
  eri_opts_t o;
  eri_default_opts(&o);
  if (opts) o = *opts;
  if (!(o.thresh >= 0.0) || !(o.mixed_tau >= 0.0) || (o.precision != ERI_FP64 && o.precision != ERI_MIXED))
    return ERI_EINVAL;

  eri_plan_impl* P = new (std::nothrow) eri_plan_impl();
  if (!P) return ERI_ENOMEM;
  P->opts = o;
  if (o.tune_cache) P->tune_cache = o.tune_cache;
  P->opts.tune_cache = nullptr;  // the caller's string is not kept
  if (o.device >= 0) {
    if (cudaSetDevice(o.device) != cudaSuccess) { delete P; return ERI_ECUDA; }
  }
  cudaGetDevice(&P->device);
  cudaDeviceGetAttribute(&P->nsm, cudaDevAttrMultiProcessorCount, P->device);
  P->nmol = nmol;
  // global numbering
  std::vector<int> l, atom, np, po, ao, aol, shloc;
  std::vector<double> ex, co, xyz;
  P->h_mat_off.assign(nmol + 1, 0);
  P->h_mat_n.assign(nmol, 0);
  P->h_aobase.assign(nmol + 1, 0);
  P->h_atombase.assign(nmol + 1, 0);
  P->h_pairbase.assign(nmol + 1, 0);
  std::vector<int> shellbase(nmol + 1, 0);
  int nbf = 0, nprim_tot = 0;
  int64_t npair64 = 0;
  for (int m = 0; m < nmol; ++m) {
    const eri_basis_t* B = bases[m];
    shellbase[m] = (int)l.size();
    P->h_atombase[m] = (int)(xyz.size() / 3);
    P->h_aobase[m] = nbf;
    P->h_pairbase[m] = (int)npair64;
    int nb = 0;
    for (int s = 0; s < B->nshell; ++s) {
      const eri_shell_t& sh = B->shells[s];
      l.push_back(sh.l);
      atom.push_back(P->h_atombase[m] + sh.atom);
      np.push_back(sh.nprim);
      po.push_back(nprim_tot + sh.prim_offset);
      ao.push_back(nbf + nb);
      aol.push_back(nb);
      shloc.push_back(s);
      nb += ncart(sh.l);
    }
    ex.insert(ex.end(), B->exps, B->exps + nprim_m[m]);
    co.insert(co.end(), B->coefs, B->coefs + nprim_m[m]);
    xyz.insert(xyz.end(), coords[m], coords[m] + 3 * B->natom);
    nprim_tot += nprim_m[m];
    nbf += nb;
    P->h_mat_n[m] = nb;
    P->h_mat_off[m + 1] = P->h_mat_off[m] + (int64_t)nb * nb;
    P->max_nbf = std::max(P->max_nbf, nb);
    npair64 += (int64_t)B->nshell * (B->nshell + 1) / 2;
  }
  const int ns = (int)l.size(), na = (int)(xyz.size() / 3);
  shellbase[nmol] = ns;
  P->h_atombase[nmol] = na;
  P->h_aobase[nmol] = nbf;
  P->h_pairbase[nmol] = (int)std::min<int64_t>(npair64, INT32_MAX);
  ao.push_back(nbf);
  if (npair64 > (1LL << 28)) { delete P; return ERI_EUNSUPPORTED; }
  P->nshell = ns;
  P->natom = na;
  P->nbf = nbf;
  P->nmat = P->h_mat_off[nmol];
  // shell pairs, molecule by molecule in pair-index order (a >= b), oriented so that s1 has the higher l
  const int npair = (int)npair64;
  P->npair = npair;
  std::vector<int> ps1(npair), ps2(npair), pnp(npair), ppoff(npair), pao1(npair), pao2(npair), phoff(npair), pcls(npair),
      peoff(npair), pmol(npair);
  int64_t nprimpair = 0, nherm_tot = 0, ne_tot = 0;
  for (int m = 0; m < nmol; ++m) {
    const int sb = shellbase[m], nsm = shellbase[m + 1] - sb;
    for (int a = 0; a < nsm; ++a)
      for (int b = 0; b <= a; ++b) {
        const int ip = P->h_pairbase[m] + a * (a + 1) / 2 + b;
        int x = sb + a, y = sb + b;
        if (l[y] > l[x]) std::swap(x, y);
        ps1[ip] = x; ps2[ip] = y;
        pnp[ip] = np[x] * np[y];
        ppoff[ip] = (int)std::min<int64_t>(nprimpair, INT32_MAX);
        pao1[ip] = aol[x]; pao2[ip] = aol[y];
        phoff[ip] = (int)std::min<int64_t>(nherm_tot, INT32_MAX);
        pcls[ip] = pair_class(l[x], l[y]);
        peoff[ip] = (int)std::min<int64_t>(ne_tot, INT32_MAX);
        pmol[ip] = m;
        P->h_maxnp[pcls[ip]] = std::max(P->h_maxnp[pcls[ip]], pnp[ip]);
        nprimpair += pnp[ip];
        nherm_tot += (int64_t)pnp[ip] * nherm(l[x] + l[y]);
        ne_tot += (int64_t)pnp[ip] * 3 * (l[x] + 1) * (l[y] + 1) * (l[x] + l[y] + 1);
      }
  }
  if (nprimpair > (1LL << 30) || nherm_tot > (1LL << 31) - 1 || ne_tot > (1LL << 31) - 1) {
    delete P;
    return ERI_EUNSUPPORTED;
  }
  P->nprimpair = (int)nprimpair;
  P->nherm_tot = nherm_tot;
  int rc = ERI_OK;
#define CKP(x)                                   \
  do {                                           \
    cudaError_t e_ = (x);                        \
    if (e_ != cudaSuccess) { rc = eri_fail(e_); goto fail; } \
  } while (0)
  {
    cudaStream_t s = 0;
    std::vector<RStep> st = make_rsteps();
    const size_t nm10 = (size_t)nmol * NPAIRCLASS;
    CKP(dalloc(&P->d_sh_l, ns)); CKP(dalloc(&P->d_sh_atom, ns)); CKP(dalloc(&P->d_sh_np, ns));
    CKP(dalloc(&P->d_sh_po, ns)); CKP(dalloc(&P->d_sh_ao, ns + 1)); CKP(dalloc(&P->d_shloc, ns));
    CKP(dalloc(&P->d_exps, nprim_tot)); CKP(dalloc(&P->d_coefs, nprim_tot)); CKP(dalloc(&P->d_cn, nprim_tot));
    CKP(dalloc(&P->d_f, nbf)); CKP(dalloc(&P->d_coords, 3 * (size_t)na));
    CKP(dalloc(&P->d_mat_off, nmol + 1)); CKP(dalloc(&P->d_mat_n, nmol)); CKP(dalloc(&P->d_aobase, nmol + 1));
    CKP(dalloc(&P->d_pbase, nmol + 1)); CKP(dalloc(&P->d_ccm, nm10)); CKP(dalloc(&P->d_segloc, nm10));
    CKP(dalloc(&P->d_ps1, npair)); CKP(dalloc(&P->d_ps2, npair)); CKP(dalloc(&P->d_pnp, npair));
    CKP(dalloc(&P->d_ppoff, npair)); CKP(dalloc(&P->d_pao1, npair)); CKP(dalloc(&P->d_pao2, npair));
    CKP(dalloc(&P->d_phoff, npair)); CKP(dalloc(&P->d_pcls, npair)); CKP(dalloc(&P->d_pmol, npair));
    CKP(dalloc(&P->d_Q, npair)); CKP(dalloc(&P->d_qmax, nmol)); CKP(dalloc(&P->d_sig, npair));
    CKP(dalloc(&P->d_ccount, NPAIRCLASS)); CKP(dalloc(&P->d_coff, NPAIRCLASS)); CKP(dalloc(&P->d_sorted, npair));
    CKP(dalloc(&P->d_pos, npair)); CKP(dalloc(&P->d_counts, (size_t)npair * NPAIRCLASS));
    CKP(dalloc(&P->d_cumnp, (size_t)npair + NPAIRCLASS));
    CKP(dalloc(&P->d_koff, NPAIRCLASS * NPAIRCLASS)); CKP(dalloc(&P->d_joff, NPAIRCLASS * NPAIRCLASS));
    CKP(dalloc(&P->d_ktot, NPAIRCLASS * NPAIRCLASS)); CKP(dalloc(&P->d_jtot, NPAIRCLASS * NPAIRCLASS));
    CKP(dalloc(&P->d_kprim, NPAIRCLASS * NPAIRCLASS));
    CKP(dalloc(&P->d_boys64, (size_t)BOYS_NT * (BOYS_MMAX + 1) * BOYS_J64));
    CKP(dalloc(&P->d_boys32, (size_t)BOYS_NT * (BOYS_MMAX + 1) * BOYS_J32));
    CKP(dalloc(&P->d_bexp64, BOYS_NT)); CKP(dalloc(&P->d_bexp32, BOYS_NT));
    CKP(dalloc(&P->d_pq, nprimpair)); CKP(dalloc(&P->d_pqmax, nmol)); CKP(dalloc(&P->d_pnk, npair)); CKP(dalloc(&P->d_korder, npair));
    CKP(dalloc(&P->d_peoff, npair)); CKP(dalloc(&P->d_E, ne_tot)); CKP(dalloc(&P->d_Ef, ne_tot));
    CKP(dalloc(&P->d_pmaxp, npair)); CKP(dalloc(&P->d_prefmaxp, npair)); CKP(dalloc(&P->d_ea, nprimpair));
    CKP(dalloc(&P->d_dmax, npair));
    CKP(dalloc(&P->d_counters, NPAIRCLASS * NPAIRCLASS * 2 * 3 + 2));  // + range-guard and screened counts
    CKP(dalloc(&P->d_counters2, 4 * NPAIRCLASS * NPAIRCLASS * 3));
    CKP(cudaMemset(P->d_counters2, 0, sizeof(unsigned long long) * 4 * NPAIRCLASS * NPAIRCLASS * 3));
    CKP(dalloc(&P->d_rsteps, st.size()));
    CKP(dalloc(&P->d_Dp, (size_t)P->nmat)); CKP(dalloc(&P->d_Dpf, (size_t)P->nmat));
    CKP(dalloc(&P->d_Kh, (size_t)P->nmat));
    CKP(dalloc(&P->d_Jh, (size_t)P->nmat));
    CKP(dalloc(&P->d_Dherm, nherm_tot)); CKP(dalloc(&P->d_Jherm, nherm_tot)); CKP(dalloc(&P->d_Dhermf, nherm_tot));
    CKP(dalloc(&P->d_status, 1));
    if (P->alloc_pairs() != ERI_OK) { rc = ERI_ENOMEM; goto fail; }
    if ((rc = P->ensure_streams()) != ERI_OK) goto fail;  // here: builds allocate and create nothing
    CKP(upload(P->d_sh_l, l)); CKP(upload(P->d_sh_atom, atom)); CKP(upload(P->d_sh_np, np));
    CKP(upload(P->d_sh_po, po)); CKP(upload(P->d_sh_ao, ao)); CKP(upload(P->d_shloc, shloc));
    CKP(upload(P->d_exps, ex)); CKP(upload(P->d_coefs, co)); CKP(upload(P->d_coords, xyz));
    CKP(upload(P->d_mat_off, P->h_mat_off)); CKP(upload(P->d_mat_n, P->h_mat_n));
    CKP(upload(P->d_aobase, P->h_aobase)); CKP(upload(P->d_pbase, P->h_pairbase));
    CKP(upload(P->d_ps1, ps1)); CKP(upload(P->d_ps2, ps2)); CKP(upload(P->d_pnp, pnp));
    CKP(upload(P->d_ppoff, ppoff)); CKP(upload(P->d_pao1, pao1)); CKP(upload(P->d_pao2, pao2));
    CKP(upload(P->d_phoff, phoff)); CKP(upload(P->d_peoff, peoff)); CKP(upload(P->d_pcls, pcls));
    CKP(upload(P->d_pmol, pmol)); CKP(upload(P->d_rsteps, st));
    CKP(cudaMemset(P->d_status, 0, sizeof(int)));
    k_normalize<<<grid1(ns, 64), 64>>>(ns, P->d_sh_l, P->d_sh_np, P->d_sh_po, P->d_exps, P->d_coefs, P->d_cn);
    k_compfac<<<grid1(ns, 64), 64>>>(ns, P->d_sh_l, P->d_sh_ao, P->d_f);
    k_boys_table<<<grid1(BOYS_NT, 128), 128>>>(P->d_boys64, P->d_bexp64, P->d_boys32, P->d_bexp32);
    CKP(cudaGetLastError());
    P->thresh = o.thresh;
    rc = P->geometry(s, true);
    if (rc != ERI_OK) goto fail;
    CKP(cudaDeviceSynchronize());
    ensure_order_bufs(P);
  }
#undef CKP
  tune_cache_load(P, o.precision);
  *out = reinterpret_cast<eri_plan_t*>(P);
  return ERI_OK;
fail:
  P->release();
  delete P;
  return rc;
}

extern "C" int eri_plan(const eri_basis_t* basis, const double* coords, const eri_opts_t* opts, eri_plan_t** out) {
  if (!basis || !coords || !out) return ERI_EINVAL;
  return plan_create(1, &basis, &coords, opts, out);
}

extern "C" int eri_plan_batch(int32_t nmol, const eri_basis_t* const* bases, const double* const* coords,
                              const eri_opts_t* opts, eri_plan_t** out) {
  return plan_create(nmol, bases, coords, opts, out);
}

extern "C" int eri_plan_layout(eri_plan_t* plan, int32_t* nmol, int64_t* mat_off, int32_t* nbf, int32_t* atom_off) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  if (!P) return ERI_EINVAL;
  if (nmol) *nmol = P->nmol;
  for (int m = 0; m <= P->nmol; ++m) {
    if (mat_off) mat_off[m] = P->h_mat_off[m];
    if (atom_off) atom_off[m] = P->h_atombase[m];
    if (nbf && m < P->nmol) nbf[m] = P->h_mat_n[m];
  }
  return ERI_OK;
}

extern "C" int eri_plan_set_coords(eri_plan_t* plan, const double* coords_dev, int32_t freeze_lists, void* stream) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  if (!P || !coords_dev) return ERI_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  CK(cudaSetDevice(P->device));
  CK(cudaMemcpyAsync(P->d_coords, coords_dev, sizeof(double) * 3 * P->natom, cudaMemcpyDeviceToDevice, s));
  ++P->geom_serial;  // an exchange-correlation grid follows the atoms at its next use
  return P->geometry(s, freeze_lists == 0);
}

// Class pairs of a build in launch order, and the side stream each goes to: by
// decreasing estimated work, to the least-loaded of nbranch streams (nbranch = 0:
// in class order, on the caller's stream).
struct ClassLaunch {
  int X, Y;
  double cost;
  int branch;
};
// Returns the number of streams used (no more than there are launches: a fork and
// join costs the host about 1 us per stream).
static int assign_branches(std::vector<ClassLaunch>& v, int nbranch) {
  nbranch = std::min(nbranch, (int)v.size());
  if (nbranch <= 0) return 0;
  std::stable_sort(v.begin(), v.end(), [](const ClassLaunch& a, const ClassLaunch& b) { return a.cost > b.cost; });
  double load[eri_plan_impl::kStreams] = {};
  for (ClassLaunch& l : v) {
    l.branch = (int)(std::min_element(load, load + nbranch) - load);
    load[l.branch] += l.cost;
  }
  return nbranch;
}

// Whether a plain FP64 build orders this class pair's list by work first: a thread
// kernel, contracted pairs, and some quartets per lane (225 functions: (pp|ps) 6.5
// ms in list order, of which a third is lanes waiting for the longest).
static bool order_first(const eri_plan_impl* P, int X, int Y) {
  return use_thread_kernel(kClassL1[X], kClassL2[X], kClassL1[Y], kClassL2[Y], false) &&
         P->h_maxnp[X] * P->h_maxnp[Y] > 1 && P->nshard == 1 &&
         P->h_ktot[X * NPAIRCLASS + Y] >= (int64_t)256 * P->nsm;
}

// The lists that order FP64 builds, taken when the plan is made (a build allocates
// nothing); a plan without room for them builds in list order.
static void ensure_order_bufs(eri_plan_impl* P) {
  bool any = false;
  for (int X = 0; X < NPAIRCLASS; ++X)
    for (int Y = 0; Y <= X; ++Y) any = any || order_first(P, X, Y);
  if (any && P->ensure_tier_bufs(1) != ERI_OK) cudaGetLastError();
}

// One J/K build on stream s, lists as they stand.  nbranch > 0: the class
// launches are spread over that many of the plan's side streams (fork / join by
// events); 0: they run in order on s (profiled builds).
static int build_impl(eri_plan_impl* P, const double* D, double* J, double* K, int precision, cudaStream_t s,
                      int nbranch) {
  const bool concurrent = nbranch > 0;
  const int64_t nn = P->nmat;
  const MolMats mm = molmats(P);
  k_scale_d<<<P->mat_grid(256), 256, 0, s>>>(mm, D, P->d_f, P->d_Dp, P->d_Dpf);
  CK(cudaGetLastError());
  const bool jengine = J && !K && P->opts.j_engine;
  if (jengine) {
    // J alone: Hermite density -> J-engine -> Hermite J to Cartesian (Eq. j_formula).
    // Mixed precision: each ordered list is split on the device by the energy's
    // tier test (reading 5) and each tier's kernel runs its own compacted list;
    // both add into the FP64 Hermite J.
    const bool jmixed = precision == ERI_MIXED;
    CK(cudaMemsetAsync(P->d_Jherm, 0, sizeof(double) * (size_t)P->nherm_tot, s));
    k_hermite_density<<<grid1(P->npair, 4), 128, 0, s>>>(P->npair, P->d_ps1, P->d_ps2, P->d_pnk, P->d_ppoff,
                                                         P->d_phoff, P->d_peoff, P->d_sh_l, P->d_pao1, P->d_pao2,
                                                         P->d_pmol, mm, P->d_sig, P->pairdata(), P->d_Dp, P->d_Dherm,
                                                         jmixed ? P->d_Dhermf : nullptr);
    CK(cudaGetLastError());
    if (jmixed) {
      k_dmax<<<grid1(P->npair, 128), 128, 0, s>>>(P->npair, P->d_ps1, P->d_ps2, P->d_sh_l, P->d_pao1, P->d_pao2,
                                                  P->d_pmol, P->d_mat_off, P->d_mat_n, P->d_Dp, P->d_dmax);
      CK(cudaGetLastError());
      const int rc = P->ensure_tier_bufs(1);  // (a graph capture has them already)
      if (rc != ERI_OK) return rc;
      nbranch = std::min(nbranch, P->tier_nb);
    }
    JArgs ja{};
    ja.pd = P->pairdata(); ja.sp = P->spinfo(); ja.bt = P->boystabs();
    ja.rsteps = P->d_rsteps; ja.Dherm = P->d_Dherm; ja.Dhermf = P->d_Dhermf; ja.Jherm = P->d_Jherm;
    ja.omega2 = P->omega * P->omega; ja.omega2f = (float)ja.omega2;
    ja.det = P->opts.deterministic ? 1 : 0;
    ja.items = nullptr;
    ja.nitems = nullptr;
    KArgs ka{};  // tier split of the ordered lists
    ka.pd = P->pairdata(); ka.sp = P->spinfo();
    ka.Q = P->d_Q; ka.dmax = P->d_dmax; ka.pmaxp = P->d_pmaxp; ka.prefmaxp = P->d_prefmaxp;
    ka.shloc = P->d_shloc; ka.pbase = P->d_pbase;
    ka.tau = (float)P->opts.mixed_tau; ka.pmax32 = (float)kPmax32; ka.mixed = 1;
    // counters2 kinds 0 (J-engine FP64) and 3 (J-engine FP32)
    CK(cudaMemsetAsync(P->d_counters2, 0, sizeof(unsigned long long) * NPAIRCLASS * NPAIRCLASS * 3, s));
    CK(cudaMemsetAsync(P->d_counters2 + 3 * NPAIRCLASS * NPAIRCLASS * 3, 0,
                       sizeof(unsigned long long) * NPAIRCLASS * NPAIRCLASS * 3, s));
    P->last_jmixed = jmixed;
    const bool prof = P->opts.profile && !concurrent;
    auto jlaunch = [&](int X, int Y, int tier, cudaStream_t ls) -> int {
      const int lab = kClassL1[X] + kClassL2[X], lcd = kClassL1[Y] + kClassL2[Y];
      ja.counter = P->d_counters2 + ((tier ? 3 : 0) * NPAIRCLASS * NPAIRCLASS + X * NPAIRCLASS + Y) * 3;
      cudaEvent_t e0 = nullptr, e1 = nullptr;
      if (prof) {
        CK(P->prof_event_pair(&e0, &e1));
        CK(cudaEventRecord(e0, ls));
      }
      cudaError_t e = cudaErrorInvalidValue;
      switch (lab) {
        case 0: e = launch_j_lab0(lcd, tier, ja, ls, P->nsm); break;
        case 1: e = launch_j_lab1(lcd, tier, ja, ls, P->nsm); break;
        case 2: e = launch_j_lab2(lcd, tier, ja, ls, P->nsm); break;
        case 3: e = launch_j_lab3(lcd, tier, ja, ls, P->nsm); break;
        case 4: e = launch_j_lab4(lcd, tier, ja, ls, P->nsm); break;
        case 5: e = launch_j_lab5(lcd, tier, ja, ls, P->nsm); break;
        case 6: e = launch_j_lab6(lcd, tier, ja, ls, P->nsm); break;
      }
      CK(e);
      if (prof) {
        CK(cudaEventRecord(e1, ls));
        P->prof_log.push_back({X, Y, tier ? 5 : 3, P->prof_ev_used - 2});
      }
      return ERI_OK;
    };
    std::vector<ClassLaunch> order;
    for (int X = 0; X < NPAIRCLASS; ++X)
      for (int Y = 0; Y < NPAIRCLASS; ++Y) {
        const int64_t tot = P->h_jtot[X * NPAIRCLASS + Y];
        if (tot > 0) order.push_back({X, Y, jengine_flops(X, Y, (double)tot * P->h_maxnp[X] * P->h_maxnp[Y]), 0});
      }
    nbranch = assign_branches(order, nbranch);
    Fork side(s, P->branch, P->fork_ev, P->join_ev);
    if (concurrent) CK(side.open(nbranch));
    for (const ClassLaunch& l : order) {
        const int X = l.X, Y = l.Y, b = l.branch;
        const WorkList full = P->jlist(X, Y);
        const cudaStream_t ls = concurrent ? P->branch[b] : s;
        if (!jmixed) {
          ja.wl = full;
          const int rc = jlaunch(X, Y, 0, ls);
          if (rc != ERI_OK) return rc;
          continue;
        }
        int2* buf = P->tbuf[b];
        unsigned int* cnt = P->tcnt + 2 * b;
        for (int64_t f = 0; f < full.total; f += P->tier_cap) {
          KArgs sa = ka;
          sa.wl = full;
          sa.wl.first = f;
          sa.wl.total = std::min<int64_t>(full.total, f + P->tier_cap);
          CK(cudaMemsetAsync(cnt, 0, 2 * sizeof(unsigned int), ls));
          CK(launch_tier_split(P, sa, buf, cnt, ls));
          for (int tier = 0; tier < 2; ++tier) {
            ja.wl = full;
            ja.wl.first = 0;
            ja.wl.total = sa.wl.total - f;  // upper bound of the tier's count (grid sizing)
            ja.items = buf + (tier ? P->tier_cap : 0);
            ja.nitems = cnt + tier;
            const int rc = jlaunch(X, Y, tier, ls);
            if (rc != ERI_OK) return rc;
          }
        }
        ja.items = nullptr;
        ja.nitems = nullptr;
    }
    CK(side.join());
    CK(cudaMemsetAsync(J, 0, sizeof(double) * nn, s));
    k_post_j<<<grid1((int64_t)P->npair * 100, 128), 128, 0, s>>>(P->npair, P->d_ps1, P->d_ps2, P->d_pnk, P->d_phoff,
                                                                 P->d_peoff, P->d_sh_l, P->d_pao1, P->d_pao2,
                                                                 P->d_pmol, mm, P->d_sig, P->d_E, P->d_Jherm, P->d_f,
                                                                 J, ja.det, P->d_status);
    CK(cudaGetLastError());
  } else {
    // J and/or K from contracted Cartesian ERIs over canonical quartets
    if (K) CK(cudaMemsetAsync(P->d_Kh, 0, sizeof(double) * nn, s));
    if (J) CK(cudaMemsetAsync(P->d_Jh, 0, sizeof(double) * nn, s));
    CK(cudaMemsetAsync(P->d_counters, 0, sizeof(unsigned long long) * (NPAIRCLASS * NPAIRCLASS * 6 + 2), s));
    const bool mixed = precision == ERI_MIXED;
    // the device split pass serves the precision tiers and the density screen
    const bool split = mixed || P->opts.density_screen;
    if (split) {
      k_dmax<<<grid1(P->npair, 128), 128, 0, s>>>(P->npair, P->d_ps1, P->d_ps2, P->d_sh_l, P->d_pao1, P->d_pao2,
                                                  P->d_pmol, P->d_mat_off, P->d_mat_n, P->d_Dp, P->d_dmax);
      CK(cudaGetLastError());
    }
    JKArgs ja{};
    KArgs& ka = ja.k;
    ka.pd = P->pairdata(); ka.sp = P->spinfo(); ka.bt = P->boystabs();
    ka.rsteps = P->d_rsteps; ka.Dp = P->d_Dp; ka.Dpf = P->d_Dpf; ka.Kh = K ? P->d_Kh : nullptr;
    ka.Q = P->d_Q; ka.dmax = P->d_dmax; ka.pmaxp = P->d_pmaxp; ka.prefmaxp = P->d_prefmaxp;
    ka.shloc = P->d_shloc; ka.pbase = P->d_pbase;
    ka.tau = mixed ? (float)P->opts.mixed_tau : 0.0f; ka.pmax32 = (float)kPmax32; ka.mixed = mixed ? 1 : 0;
    ka.items = nullptr; ka.nitems = nullptr;
    ka.guard = P->d_counters + NPAIRCLASS * NPAIRCLASS * 6;
    ka.screened = P->d_counters + NPAIRCLASS * NPAIRCLASS * 6 + 1;
    ka.screen = P->opts.density_screen ? (float)P->thresh : 0.0f;
    ka.omega2 = P->omega * P->omega; ka.omega2f = (float)ka.omega2;
    ka.det = P->opts.deterministic ? 1 : 0;
    ja.Jh = J ? P->d_Jh : nullptr;
    P->last_mixed = mixed;
    P->last_do_j = J != nullptr;
    P->last_do_k = K != nullptr;
    std::vector<ClassLaunch> order;  // cost: primitive quartets x class cost
    for (int X = 0; X < NPAIRCLASS; ++X)
      for (int Y = 0; Y <= X; ++Y) {
        const int64_t tot = P->h_ktot[X * NPAIRCLASS + Y];
        if (tot == 0) continue;
        order.push_back({X, Y, class_flops(X, Y, (double)tot, (double)P->h_kprim[X * NPAIRCLASS + Y], 0.0,
                                           J != nullptr, K != nullptr), 0});
      }
    if (split) {
      const int rc = P->ensure_tier_bufs(1);  // (a graph capture has them already)
      if (rc != ERI_OK) return rc;
      nbranch = std::min(nbranch, P->tier_nb);
    }
    // Plain FP64 builds order the long lists of the thread kernels the same way
    // (every quartet in one list, see k_tier_split) where the plan holds the lists
    // (see ensure_order_bufs); without them they run in list order.
    bool ordered = false;
    if (!split && P->tier_nb >= std::max(1, std::min(nbranch, eri_plan_impl::kBranches)))
      for (const ClassLaunch& l : order) ordered = ordered || order_first(P, l.X, l.Y);
    if (ordered) nbranch = std::min(nbranch, P->tier_nb);
    // (Deterministic builds order only lists that fit one window: the windows follow
    // the size of the plan's lists, which may change between two calls, and a short
    // last window takes other kernels and primitive splits than the list as a whole.)
    auto by_work = [&](int X, int Y) {
      return ordered && order_first(P, X, Y) &&
             !(P->opts.deterministic && P->h_ktot[X * NPAIRCLASS + Y] > P->tier_cap);
    };
    nbranch = assign_branches(order, nbranch);
    Fork side(s, P->branch, P->fork_ev, P->join_ev);
    if (concurrent) CK(side.open(nbranch));
    const bool prof = P->opts.profile && !concurrent;
    auto launch = [&](int X, int Y, int tier, cudaStream_t ls) -> int {
      ka.tier_want = tier;
      ka.wl.tile = P->tile_for(X, Y, tier);
      ka.counter = P->d_counters + ((X * NPAIRCLASS + Y) * 2 + tier) * 3;
      cudaEvent_t e0 = nullptr, e1 = nullptr;
      if (prof) {
        CK(P->prof_event_pair(&e0, &e1));
        CK(cudaEventRecord(e0, ls));
      }
      CK(launch_jk_class(X, Y, tier, ja, ls, P->nsm));
      if (prof) {
        CK(cudaEventRecord(e1, ls));
        P->prof_log.push_back({X, Y, tier, P->prof_ev_used - 2});
      }
      return ERI_OK;
    };
    for (const ClassLaunch& l : order) {
      const int b = l.branch;
      const cudaStream_t ls = concurrent ? P->branch[b] : s;
      ka.same_class = l.X == l.Y;
      if (!split && !by_work(l.X, l.Y)) {
        ka.wl = P->klist(l.X, l.Y);
        ka.items = nullptr;
        ka.nitems = nullptr;
        const int rc = launch(l.X, l.Y, 0, ls);
        if (rc != ERI_OK) return rc;
        continue;
      }
      // mixed precision and/or density screen: split each window of the list
      // into its two tiers, dropping screened quartets (compacted on the
      // device), then run each tier over its own list (FP64 builds: tier 0 only)
      const WorkList full = P->klist(l.X, l.Y);
      int2* buf = P->tbuf[b];
      unsigned int* cnt = P->tcnt + 2 * b;
      for (int64_t f = 0; f < full.total; f += P->tier_cap) {
        KArgs sa = ka;
        sa.wl = full;
        sa.wl.first = f;
        sa.wl.total = std::min<int64_t>(full.total, f + P->tier_cap);
        CK(cudaMemsetAsync(cnt, 0, 2 * sizeof(unsigned int), ls));
        CK(launch_tier_split(P, sa, buf, cnt, ls));
        for (int tier = 0; tier < (mixed ? 2 : 1); ++tier) {
          ka.wl = full;
          ka.wl.first = 0;
          ka.wl.total = sa.wl.total - f;  // upper bound of the tier's count (grid sizing)
          ka.items = buf + (tier ? P->tier_cap : 0);
          ka.nitems = cnt + tier;
          const int rc = launch(l.X, l.Y, tier, ls);
          if (rc != ERI_OK) return rc;
        }
      }
      ka.items = nullptr;
      ka.nitems = nullptr;
    }
    CK(side.join());
    P->prof_builds += P->opts.profile ? 1 : 0;
    if (K) {
      k_post_k<<<P->mat_grid(256), 256, 0, s>>>(mm, P->d_Kh, P->d_f, K, ka.det, P->d_status);
      CK(cudaGetLastError());
    }
    if (J) {
      k_post_k<<<P->mat_grid(256), 256, 0, s>>>(mm, P->d_Jh, P->d_f, J, ka.det, P->d_status);
      CK(cudaGetLastError());
    }
  }
  return ERI_OK;
}

extern "C" int eri_build_jk(eri_plan_t* plan, const double* D, double* J, double* K, double thresh, int32_t precision,
                            void* stream) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  if (!P || !D || (!J && !K)) return ERI_EINVAL;
  if (precision != ERI_FP64 && precision != ERI_MIXED) return ERI_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  CK(cudaSetDevice(P->device));
  if (thresh >= 0.0 && thresh != P->thresh) {
    int rc = P->build_lists(thresh, s);
    if (rc != ERI_OK) return rc;
  }
  return build_impl(P, D, J, K, precision, s, P->eager_branches(true));
}

extern "C" int eri_build_jk_graph(eri_plan_t* plan, const double* D, double* J, double* K, int32_t precision,
                                  void* stream) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  if (!P || !D || (!J && !K)) return ERI_EINVAL;
  if (precision != ERI_FP64 && precision != ERI_MIXED) return ERI_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  CK(cudaSetDevice(P->device));
  if (!P->gexec || P->gkey[0] != D || P->gkey[1] != J || P->gkey[2] != K || P->gprec != precision) {
    int rc = P->ensure_streams();
    if (rc != ERI_OK) return rc;
    rc = P->ensure_tier_bufs(eri_plan_impl::kBranches);
    if (rc != ERI_OK) {
      if (precision == ERI_MIXED || P->opts.density_screen) return rc;
      rc = ERI_OK;  // a plain FP64 build runs without them
      cudaGetLastError();
    }
    if (P->gexec) {
      CK(cudaStreamSynchronize(s));
      CK(cudaGraphExecDestroy(P->gexec));
      P->gexec = nullptr;
    }
    // Capture the build twice: class launches in one serial chain, and forked
    // over kBranches branches (least-loaded first).  Long launches that fill
    // the GPU by themselves run best in order; many short ones (batched
    // plans, small molecules) gain from overlapping.  Each graph is replayed
    // twice on `stream` (CUDA events) and the faster one is kept.
    const int cand[2] = {1, eri_plan_impl::kBranches};
    cudaGraphExec_t ex[2] = {nullptr, nullptr};
    for (int c = 0; c < 2 && rc == ERI_OK; ++c) {
      CK(cudaStreamBeginCapture(P->cap_stream, cudaStreamCaptureModeThreadLocal));
      rc = build_impl(P, D, J, K, precision, P->cap_stream, cand[c]);
      cudaGraph_t g = nullptr;
      const cudaError_t ce = cudaStreamEndCapture(P->cap_stream, &g);
      if (rc == ERI_OK && ce != cudaSuccess) rc = eri_fail(ce);
      if (rc == ERI_OK) {
        const cudaError_t ie = cudaGraphInstantiate(&ex[c], g, 0);
        if (ie != cudaSuccess) {
          ex[c] = nullptr;
          rc = eri_fail(ie);
        }
      }
      if (g) cudaGraphDestroy(g);
    }
    float best[2] = {0.0f, 0.0f};
    if (rc == ERI_OK) {
      cudaEvent_t e0 = nullptr, e1 = nullptr;
      cudaError_t te = cudaEventCreate(&e0);
      if (te == cudaSuccess) te = cudaEventCreate(&e1);
      for (int c = 0; c < 2 && te == cudaSuccess; ++c) {
        best[c] = 3.4e38f;
        for (int r = 0; r < 2 && te == cudaSuccess; ++r) {
          float ms = 0.0f;
          te = cudaEventRecord(e0, s);
          if (te == cudaSuccess) te = cudaGraphLaunch(ex[c], s);
          if (te == cudaSuccess) te = cudaEventRecord(e1, s);
          if (te == cudaSuccess) te = cudaEventSynchronize(e1);
          if (te == cudaSuccess) te = cudaEventElapsedTime(&ms, e0, e1);
          if (te == cudaSuccess && ms < best[c]) best[c] = ms;
        }
      }
      if (e0) cudaEventDestroy(e0);
      if (e1) cudaEventDestroy(e1);
      if (te != cudaSuccess) rc = eri_fail(te);
    }
    const int keep = best[1] < best[0] ? 1 : 0;
    for (int c = 0; c < 2; ++c)
      if (ex[c] && (rc != ERI_OK || c != keep)) cudaGraphExecDestroy(ex[c]);
    if (rc != ERI_OK) {
      cudaGetLastError();
      return rc;
    }
    P->gexec = ex[keep];
    P->gbranches = cand[keep];
    P->gkey[0] = D;
    P->gkey[1] = J;
    P->gkey[2] = K;
    P->gprec = precision;
  }
  CK(cudaGraphLaunch(P->gexec, s));
  return ERI_OK;
}

// Autotuner: for every (bra class, ket class, tier) launch of this plan, time
// each candidate work-tile length on three windows of the launch's own work
// list (at 1/6, 1/2 and 5/6 of it, so that a mixed-precision tier sees its
// share of quartets) and keep the fastest.  A window is sized so that the
// default tile takes about trial_ms; each candidate is timed twice (minimum).
// The trials write into the plan's scratch accumulators only.
extern "C" int eri_autotune(eri_plan_t* plan, const double* D, int32_t precision, double trial_ms, void* stream) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  if (!P || !D || !(trial_ms > 0.0)) return ERI_EINVAL;
  if (precision != ERI_FP64 && precision != ERI_MIXED) return ERI_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  CK(cudaSetDevice(P->device));
  const bool mixed = precision == ERI_MIXED;
  const MolMats mm = molmats(P);
  k_scale_d<<<P->mat_grid(256), 256, 0, s>>>(mm, D, P->d_f, P->d_Dp, P->d_Dpf);
  if (mixed)
    k_dmax<<<grid1(P->npair, 128), 128, 0, s>>>(P->npair, P->d_ps1, P->d_ps2, P->d_sh_l, P->d_pao1, P->d_pao2,
                                                P->d_pmol, P->d_mat_off, P->d_mat_n, P->d_Dp, P->d_dmax);
  CK(cudaGetLastError());
  JKArgs ja{};
  KArgs& ka = ja.k;
  ka.pd = P->pairdata(); ka.sp = P->spinfo(); ka.bt = P->boystabs();
  ka.rsteps = P->d_rsteps; ka.Dp = P->d_Dp; ka.Dpf = P->d_Dpf; ka.Kh = P->d_Kh;
  ka.Q = P->d_Q; ka.dmax = P->d_dmax; ka.pmaxp = P->d_pmaxp; ka.prefmaxp = P->d_prefmaxp;
  ka.shloc = P->d_shloc; ka.pbase = P->d_pbase;
  ka.tau = (float)P->opts.mixed_tau; ka.pmax32 = (float)kPmax32; ka.mixed = mixed ? 1 : 0;
  ka.counter = nullptr;
  ka.guard = nullptr;
  ka.omega2 = P->omega * P->omega; ka.omega2f = (float)ka.omega2;
  ja.Jh = P->d_Jh;
  cudaEvent_t e0, e1;
  CK(cudaEventCreate(&e0));
  CK(cudaEventCreate(&e1));
  int rc = ERI_OK;
  if (mixed) {
    rc = P->ensure_tier_bufs(1);
    if (rc != ERI_OK) {
      cudaEventDestroy(e0);
      cudaEventDestroy(e1);
      return rc;
    }
  }
  // time the three windows of `win` items each with tile t; returns ms (< 0 on
  // error).  Mixed precision: each window is first split into its tiers
  // (untimed) and the tier's compacted list is timed.
  auto trial = [&](int X, int Y, int tier, int t, int64_t win) -> double {
    const WorkList full = P->klist(X, Y);
    const int64_t tot = full.total;
    if (mixed) win = std::min<int64_t>(win, P->tier_cap);
    double best = 1e300;
    for (int rep = 0; rep < 2; ++rep) {
      double sum = 0.0;
      for (int w = 0; w < 3; ++w) {
        const int64_t c = tot * (2 * w + 1) / 6;
        const int64_t f = std::max<int64_t>(0, std::min<int64_t>(c - win / 2, tot - win));
        const int64_t last = std::min<int64_t>(tot, f + win);
        ka.wl = full;
        ka.wl.first = f;
        ka.wl.total = last;
        ka.wl.tile = t;
        ka.same_class = X == Y;
        ka.tier_want = tier;
        ka.items = nullptr;
        ka.nitems = nullptr;
        if (mixed) {
          if (cudaMemsetAsync(P->tcnt, 0, 2 * sizeof(unsigned int), s) != cudaSuccess) return -1.0;
          if (launch_tier_split(P, ka, P->tbuf[0], P->tcnt, s) != cudaSuccess) return -1.0;
          ka.wl.first = 0;
          ka.wl.total = last - f;
          ka.items = P->tbuf[0] + (tier ? P->tier_cap : 0);
          ka.nitems = P->tcnt + tier;
        }
        if (cudaEventRecord(e0, s) != cudaSuccess) return -1.0;
        if (launch_jk_class(X, Y, tier, ja, s, P->nsm) != cudaSuccess) return -1.0;
        if (cudaEventRecord(e1, s) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess) return -1.0;
        float ms = 0.0f;
        if (cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) return -1.0;
        sum += ms;
      }
      best = std::min(best, sum);
    }
    ka.items = nullptr;
    ka.nitems = nullptr;
    return best;
  };
  static const int kThreadTiles[] = {1, 2, 4, 8};
  static const int kWarpTiles[] = {1, 2, 4, 8, 16, 32};
  for (int X = 0; X < NPAIRCLASS && rc == ERI_OK; ++X)
    for (int Y = 0; Y <= X && rc == ERI_OK; ++Y) {
      const int64_t tot = P->h_ktot[X * NPAIRCLASS + Y];
      if (tot == 0) continue;
      for (int tier = 0; tier < (mixed ? 2 : 1) && rc == ERI_OK; ++tier) {
        const int def = default_tile(X, Y, tier);
        // windows long enough that every resident warp gets several tiles (a
        // short window measures the launch tail, not the tile length)
        int64_t win = std::min<int64_t>(tot, 3 * (int64_t)P->nsm * 2048);
        double t0 = trial(X, Y, tier, def, win / 3);
        if (t0 < 0.0) { rc = ERI_ECUDA; break; }
        for (int grow = 0; grow < 2 && t0 < 0.5 * trial_ms && win < tot; ++grow) {
          win = std::min<int64_t>(tot, (int64_t)((double)win * trial_ms / std::max(t0, 1e-3)));
          t0 = trial(X, Y, tier, def, win / 3 + 1);
          if (t0 < 0.0) { rc = ERI_ECUDA; break; }
        }
        if (rc != ERI_OK) break;
        const bool thr = use_thread_kernel(kClassL1[X], kClassL2[X], kClassL1[Y], kClassL2[Y], tier == 1);
        const int* cand = thr ? kThreadTiles : kWarpTiles;
        const int nc = thr ? 4 : 6;
        int best = def;
        double bt = t0;
        for (int i = 0; i < nc; ++i) {
          if (cand[i] == def) continue;
          const double t = trial(X, Y, tier, cand[i], win / 3 + 1);
          if (t < 0.0) { rc = ERI_ECUDA; break; }
          if (t < 0.95 * bt) { bt = t; best = cand[i]; }
        }
        if (rc == ERI_OK && best != def) {  // confirm against the default once more
          const double td = trial(X, Y, tier, def, win / 3 + 1), tb = trial(X, Y, tier, best, win / 3 + 1);
          if (td < 0.0 || tb < 0.0) { rc = ERI_ECUDA; break; }
          if (!(tb < 0.95 * td)) best = def;
        }
        P->tile_k[(X * NPAIRCLASS + Y) * 2 + tier] = best;
      }
    }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (P->gexec) {  // captured builds carry the old tiles
    cudaStreamSynchronize(s);
    cudaGraphExecDestroy(P->gexec);
    P->gexec = nullptr;
  }
  if (rc == ERI_OK) rc = tune_cache_store(P, precision);
  return rc;
}

extern "C" int eri_plan_set_shard(eri_plan_t* plan, int32_t shard, int32_t nshard) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  if (!P || nshard < 1 || shard < 0 || shard >= nshard) return ERI_EINVAL;
  if (P->gexec && (shard != P->shard || nshard != P->nshard)) {  // captured builds carry the old share
    CK(cudaSetDevice(P->device));
    CK(cudaDeviceSynchronize());
    CK(cudaGraphExecDestroy(P->gexec));
    P->gexec = nullptr;
  }
  P->shard = shard;
  P->nshard = nshard;
  return ERI_OK;
}

extern "C" int eri_plan_set_omega(eri_plan_t* plan, double omega) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  if (!P || !(omega >= 0.0) || !(omega < 1.0e30)) return ERI_EINVAL;
  if (P->gexec && omega != P->omega) {  // a captured graph carries the old operator
    CK(cudaSetDevice(P->device));
    CK(cudaDeviceSynchronize());
    CK(cudaGraphExecDestroy(P->gexec));
    P->gexec = nullptr;
  }
  P->omega = omega;
  return ERI_OK;
}

extern "C" int eri_plan_set_tau(eri_plan_t* plan, double mixed_tau) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  if (!P || !(mixed_tau >= 0.0)) return ERI_EINVAL;
  if (P->gexec && mixed_tau != P->opts.mixed_tau) {  // the graph's launches carry the old threshold
    CK(cudaSetDevice(P->device));
    CK(cudaDeviceSynchronize());
    CK(cudaGraphExecDestroy(P->gexec));
    P->gexec = nullptr;
  }
  P->opts.mixed_tau = mixed_tau;
  return ERI_OK;
}

extern "C" int eri_get_tiles(eri_plan_t* plan, int32_t* tiles) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  if (!P || !tiles) return ERI_EINVAL;
  for (int X = 0; X < NPAIRCLASS; ++X)
    for (int Y = 0; Y < NPAIRCLASS; ++Y)
      for (int t = 0; t < 2; ++t) {
        const int k = (X * NPAIRCLASS + Y) * 2 + t;
        tiles[k] = Y <= X ? P->tile_for(X, Y, t) : 0;
      }
  return ERI_OK;
}

extern "C" int eri_set_tiles(eri_plan_t* plan, const int32_t* tiles) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  if (!P || !tiles) return ERI_EINVAL;
  for (int k = 0; k < NPAIRCLASS * NPAIRCLASS * 2; ++k)
    if (tiles[k] < 0 || tiles[k] > 1024) return ERI_EINVAL;
  if (P->gexec) {  // a captured graph carries the old tiles: wait for it on the plan's device, then drop it
    CK(cudaSetDevice(P->device));
    CK(cudaDeviceSynchronize());
    CK(cudaGraphExecDestroy(P->gexec));
    P->gexec = nullptr;
  }
  for (int k = 0; k < NPAIRCLASS * NPAIRCLASS * 2; ++k) P->tile_k[k] = tiles[k];
  return ERI_OK;
}

// FP64 J/K over canonical quartets with caller-provided scratch (D', half-K,
// half-J, each nbf*nbf doubles).  Serves eri_build_jk_noalloc (noalloc.cu):
// launches kernels only, allocates nothing, uses the plan's current lists.
int eri_build_jk_scratch(eri_plan_t* plan, const double* D, double* J, double* K, double* Dp, double* Kh, double* Jh,
                         cudaStream_t s) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  const int64_t nn = P->nmat;
  const MolMats mm = molmats(P);
  k_scale_d<<<P->mat_grid(256), 256, 0, s>>>(mm, D, P->d_f, Dp, nullptr);
  CK(cudaGetLastError());
  if (K) CK(cudaMemsetAsync(Kh, 0, sizeof(double) * nn, s));
  if (J) CK(cudaMemsetAsync(Jh, 0, sizeof(double) * nn, s));
  JKArgs ja{};
  KArgs& ka = ja.k;
  ka.pd = P->pairdata(); ka.sp = P->spinfo(); ka.bt = P->boystabs();
  ka.rsteps = P->d_rsteps; ka.Dp = Dp; ka.Dpf = nullptr; ka.Kh = K ? Kh : nullptr;
  ka.Q = P->d_Q; ka.dmax = P->d_dmax; ka.pmaxp = P->d_pmaxp; ka.prefmaxp = P->d_prefmaxp;
  ka.shloc = P->d_shloc; ka.pbase = P->d_pbase;
  ka.tau = 0.0f; ka.pmax32 = 0.0f; ka.mixed = 0; ka.tier_want = 0; ka.counter = nullptr; ka.guard = nullptr;
  ka.items = nullptr; ka.nitems = nullptr;
  ka.omega2 = P->omega * P->omega; ka.omega2f = (float)ka.omega2;
  ka.det = P->opts.deterministic ? 1 : 0;
  ja.Jh = J ? Jh : nullptr;
  P->last_mixed = false;
  P->last_do_j = J != nullptr;
  P->last_do_k = K != nullptr;
  for (int X = 0; X < NPAIRCLASS; ++X)
    for (int Y = 0; Y <= X; ++Y) {
      ka.wl = P->klist(X, Y);
      ka.wl.tile = P->tile_for(X, Y, 0);
      ka.same_class = X == Y;
      if (ka.wl.total == 0) continue;
      CK(launch_jk_class(X, Y, 0, ja, s, P->nsm));
    }
  if (K) {
    k_post_k<<<P->mat_grid(256), 256, 0, s>>>(mm, Kh, P->d_f, K, ka.det, P->d_status);
    CK(cudaGetLastError());
  }
  if (J) {
    k_post_k<<<P->mat_grid(256), 256, 0, s>>>(mm, Jh, P->d_f, J, ka.det, P->d_status);
    CK(cudaGetLastError());
  }
  return ERI_OK;
}

int eri_plan_nbf_device(eri_plan_t* plan, int* nbf, int* device, int* nmol) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  *nbf = P->nbf;
  *nmol = P->nmol;
  *device = P->device;
  return ERI_OK;
}

extern "C" int eri_energy(eri_plan_t* plan, const double* D, const double* J, const double* K, double* E_out,
                          void* stream) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  if (!P || !D || !E_out) return ERI_EINVAL;
  CK(cudaSetDevice(P->device));
  k_energy<<<P->nmol, 1024, 0, (cudaStream_t)stream>>>(molmats(P), D, J, K, E_out);
  CK(cudaGetLastError());
  return ERI_OK;
}

static cudaError_t launch_grad_class(int X, int Y, int prec, const GradArgs& ga, cudaStream_t s, int nsm) {
#define ERI_GRAD_UNIT_CALL(UX, UP) \
  if (X == UX && prec == UP) return launch_grad_unit<UX, UP, 0>(Y, ga, s, nsm);
  ERI_GRAD_UNITS(ERI_GRAD_UNIT_CALL)
#undef ERI_GRAD_UNIT_CALL
  return cudaErrorInvalidValue;
}

extern "C" int eri_jk_grad_prec(eri_plan_t* plan, const double* D, double* dEdR, int32_t want_j, int32_t want_k,
                                int32_t precision, void* stream) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  if (!P || !D || !dEdR) return ERI_EINVAL;
  if (precision != ERI_FP64 && precision != ERI_MIXED) return ERI_EINVAL;
  const bool mixed = precision == ERI_MIXED;
  cudaStream_t s = (cudaStream_t)stream;
  CK(cudaSetDevice(P->device));
  const MolMats mm = molmats(P);
  k_scale_d<<<P->mat_grid(256), 256, 0, s>>>(mm, D, P->d_f, P->d_Dp, mixed ? P->d_Dpf : nullptr);
  CK(cudaGetLastError());
  CK(cudaMemsetAsync(dEdR, 0, sizeof(double) * 3 * P->natom, s));
  if (!want_j && !want_k) return ERI_OK;
  if (mixed) {
    k_dmax<<<grid1(P->npair, 128), 128, 0, s>>>(P->npair, P->d_ps1, P->d_ps2, P->d_sh_l, P->d_pao1, P->d_pao2,
                                                P->d_pmol, P->d_mat_off, P->d_mat_n, P->d_Dp, P->d_dmax);
    CK(cudaGetLastError());
    const int rc = P->ensure_tier_bufs(1);
    if (rc != ERI_OK) return rc;
  }
  GradArgs ga{};
  ga.pd = P->pairdata(); ga.sp = P->spinfo(); ga.bt = P->boystabs(); ga.rsteps = P->d_rsteps; ga.Dp = P->d_Dp;
  ga.Dpf = P->d_Dpf;
  ga.ea = P->d_ea; ga.sh_atom = P->d_sh_atom; ga.grad = dEdR;
  ga.cj = want_j ? 1.0 : 0.0;
  ga.ck = want_k ? 1.0 : 0.0;
  ga.omega2 = P->omega * P->omega;
  ga.omega2f = (float)ga.omega2;
  ga.det = P->opts.deterministic ? 1 : 0;
  // tier split of the ordered lists: the energy's test (reading 5) on each item
  KArgs ka{};
  ka.pd = P->pairdata(); ka.sp = P->spinfo();
  ka.Q = P->d_Q; ka.dmax = P->d_dmax; ka.pmaxp = P->d_pmaxp; ka.prefmaxp = P->d_prefmaxp;
  ka.shloc = P->d_shloc; ka.pbase = P->d_pbase;
  ka.tau = (float)P->opts.mixed_tau; ka.pmax32 = (float)kPmax32; ka.mixed = 1;
  unsigned long long* gcnt = P->d_counters2 + NPAIRCLASS * NPAIRCLASS * 3;  // kinds 1 (FP64) and 2 (FP32)
  CK(cudaMemsetAsync(gcnt, 0, sizeof(unsigned long long) * 2 * NPAIRCLASS * NPAIRCLASS * 3, s));
  auto launch = [&](int X, int Y, int tier, cudaStream_t ls) -> int {
    ga.counter = gcnt + ((tier * NPAIRCLASS + X) * NPAIRCLASS + Y) * 3;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (P->opts.profile) {
      CK(P->prof_event_pair(&e0, &e1));
      CK(cudaEventRecord(e0, ls));
    }
    CK(launch_grad_class(X, Y, tier, ga, ls, P->nsm));
    if (P->opts.profile) {
      CK(cudaEventRecord(e1, ls));
      P->prof_log.push_back({X, Y, tier ? 4 : 2, P->prof_ev_used - 2});
    }
    return ERI_OK;
  };
  int nbranch = P->eager_branches(mixed);
  if (mixed) nbranch = std::min(nbranch, P->tier_nb);
  std::vector<ClassLaunch> order;
  for (int X = 0; X < NPAIRCLASS; ++X)
    for (int Y = 0; Y < NPAIRCLASS; ++Y) {
      const double tot = (double)P->h_jtot[X * NPAIRCLASS + Y], mb = P->h_maxnp[X], mk = P->h_maxnp[Y];
      if (tot > 0.0) order.push_back({X, Y, grad_flops(X, Y, tot, tot * mb * mk, tot * mb), 0});
    }
  nbranch = assign_branches(order, nbranch);
  Fork side(s, P->branch, P->fork_ev, P->join_ev);
  CK(side.open(nbranch));
  for (const ClassLaunch& l : order) {
    const WorkList full = P->jlist(l.X, l.Y);
    const cudaStream_t ls = nbranch > 0 ? P->branch[l.branch] : s;
    if (!mixed) {
      ga.wl = full;
      ga.items = nullptr;
      ga.nitems = nullptr;
      const int rc = launch(l.X, l.Y, 0, ls);
      if (rc != ERI_OK) return rc;
      continue;
    }
    int2* buf = P->tbuf[l.branch];
    unsigned int* cnt = P->tcnt + 2 * l.branch;
    for (int64_t f = 0; f < full.total; f += P->tier_cap) {
      ka.wl = full;
      ka.wl.first = f;
      ka.wl.total = std::min<int64_t>(full.total, f + P->tier_cap);
      CK(cudaMemsetAsync(cnt, 0, 2 * sizeof(unsigned int), ls));
      CK(launch_tier_split(P, ka, buf, cnt, ls));
      for (int tier = 0; tier < 2; ++tier) {
        ga.wl = full;
        ga.wl.first = 0;
        ga.wl.total = ka.wl.total - f;  // upper bound of the tier's count (grid sizing)
        ga.items = buf + (tier ? P->tier_cap : 0);
        ga.nitems = cnt + tier;
        const int rc = launch(l.X, l.Y, tier, ls);
        if (rc != ERI_OK) return rc;
      }
    }
  }
  CK(side.join());
  if (ga.det) {
    k_fix_to_double<<<grid1(3 * P->natom, 128), 128, 0, s>>>(3 * P->natom, dEdR, P->d_status);
    CK(cudaGetLastError());
  }
  return ERI_OK;
}

extern "C" int eri_jk_grad(eri_plan_t* plan, const double* D, double* dEdR, int32_t want_j, int32_t want_k,
                           void* stream) {
  return eri_jk_grad_prec(plan, D, dEdR, want_j, want_k, ERI_FP64, stream);
}

extern "C" int eri_get_lists(eri_plan_t* plan, float* Q, int32_t* sig, int32_t* counts, int32_t* sorted,
                             int32_t* class_count) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  if (!P) return ERI_EINVAL;
  CK(cudaSetDevice(P->device));
  CK(cudaDeviceSynchronize());
  if (Q) CK(cudaMemcpy(Q, P->d_Q, sizeof(float) * P->npair, cudaMemcpyDeviceToHost));
  if (sig) CK(cudaMemcpy(sig, P->d_sig, sizeof(int) * P->npair, cudaMemcpyDeviceToHost));
  if (counts) CK(cudaMemcpy(counts, P->d_counts, sizeof(int) * P->npair * NPAIRCLASS, cudaMemcpyDeviceToHost));
  if (sorted) CK(cudaMemcpy(sorted, P->d_sorted, sizeof(int) * P->nsig, cudaMemcpyDeviceToHost));
  if (class_count) memcpy(class_count, P->h_ccount, sizeof(int) * NPAIRCLASS);
  return ERI_OK;
}

extern "C" int eri_check(eri_plan_t* plan) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  if (!P) return ERI_EINVAL;
  CK(cudaSetDevice(P->device));
  CK(cudaDeviceSynchronize());
  int status = 0;
  CK(cudaMemcpy(&status, P->d_status, sizeof(int), cudaMemcpyDeviceToHost));
  if (status == 0) return ERI_OK;
  CK(cudaMemset(P->d_status, 0, sizeof(int)));
  return ERI_EDEVICE;
}

extern "C" int eri_get_stats(eri_plan_t* plan, eri_stats_t* st) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  if (!P || !st) return ERI_EINVAL;
  CK(cudaSetDevice(P->device));
  memset(st, 0, sizeof(*st));
  st->nbf = P->nbf;
  st->nshell = P->nshell;
  st->npair = P->npair;
  st->nsig_pair = P->nsig;
  for (int i = 0; i < NPAIRCLASS * NPAIRCLASS; ++i) {
    st->quartets_j += P->h_jtot[i];
    int X = i / NPAIRCLASS, Y = i % NPAIRCLASS;
    if (Y <= X) {
      st->quartets_k += P->h_ktot[i];
      st->prim_quartets_k += P->h_kprim[i];
    }
  }
  {
    unsigned long long c[NPAIRCLASS * NPAIRCLASS * 6 + 2];
    CK(cudaMemcpy(c, P->d_counters, sizeof(c), cudaMemcpyDeviceToHost));
    st->quartets_k_guard = P->last_mixed ? (int64_t)c[NPAIRCLASS * NPAIRCLASS * 6] : 0;
    st->quartets_k_screened = (int64_t)c[NPAIRCLASS * NPAIRCLASS * 6 + 1];
    st->graph_branches = P->gexec ? P->gbranches : 0;
    double fl = 0.0;
    for (int X = 0; X < NPAIRCLASS; ++X)
      for (int Y = 0; Y <= X; ++Y)
        for (int t = 0; t < 2; ++t) {
          const unsigned long long* q = c + ((X * NPAIRCLASS + Y) * 2 + t) * 3;
          fl += class_flops(X, Y, (double)q[0], (double)q[1], (double)q[2], P->last_do_j, P->last_do_k);
          if (t == 1) st->quartets_k_fp32 += (int64_t)q[0];
        }
    st->flops_k = fl;
    st->flops_j = 0.0;
    unsigned long long c2[NPAIRCLASS * NPAIRCLASS * 3];
    CK(cudaMemcpy(c2, P->d_counters2 + 3 * NPAIRCLASS * NPAIRCLASS * 3, sizeof(c2), cudaMemcpyDeviceToHost));
    for (int i = 0; i < NPAIRCLASS * NPAIRCLASS; ++i) st->quartets_j_fp32 += P->last_jmixed ? (int64_t)c2[3 * i] : 0;
  }
  int status = 0;
  CK(cudaMemcpy(&status, P->d_status, sizeof(int), cudaMemcpyDeviceToHost));
  st->device_status = status;
  return ERI_OK;
}

extern "C" int eri_get_profile(eri_plan_t* plan, eri_launch_prof_t* out, int32_t cap, int32_t* count) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  if (!P || !count || (cap > 0 && !out)) return ERI_EINVAL;
  CK(cudaSetDevice(P->device));
  CK(cudaDeviceSynchronize());
  unsigned long long c[NPAIRCLASS * NPAIRCLASS * 6], c2[4 * NPAIRCLASS * NPAIRCLASS * 3];
  CK(cudaMemcpy(c, P->d_counters, sizeof(c), cudaMemcpyDeviceToHost));
  CK(cudaMemcpy(c2, P->d_counters2, sizeof(c2), cudaMemcpyDeviceToHost));
  constexpr int NT = 6;  // tiers: 0 FP64 J/K, 1 FP32 J/K, 2 gradient FP64, 3 J-engine, 4 gradient FP32, 5 J-engine FP32
  double ms[NPAIRCLASS * NPAIRCLASS * NT] = {};
  int nl[NPAIRCLASS * NPAIRCLASS * NT] = {};
  for (const auto& r : P->prof_log) {
    float t = 0.0f;
    CK(cudaEventElapsedTime(&t, P->prof_events[r.ev], P->prof_events[r.ev + 1]));
    const int k = (r.X * NPAIRCLASS + r.Y) * NT + r.tier;
    ms[k] += t;
    nl[k] += 1;
  }
  int n = 0;
  for (int k = 0; k < NPAIRCLASS * NPAIRCLASS * NT; ++k) {
    if (!nl[k]) continue;
    if (n < cap) {
      const int X = k / (NT * NPAIRCLASS), Y = (k / NT) % NPAIRCLASS, t = k % NT;
      // counters2 kinds: J-engine FP64, gradient FP64, gradient FP32, J-engine FP32
      const int kind = t == 3 ? 0 : (t == 2 ? 1 : (t == 4 ? 2 : 3));
      const unsigned long long* q = t < 2 ? c + ((X * NPAIRCLASS + Y) * 2 + t) * 3
                                          : c2 + (kind * NPAIRCLASS * NPAIRCLASS + X * NPAIRCLASS + Y) * 3;
      eri_launch_prof_t& o = out[n];
      o.bra_class = X;
      o.ket_class = Y;
      o.tier = t;
      o.launches = nl[k];
      o.ms = ms[k];
      o.quartets = (int64_t)q[0];
      o.prim_quartets = (int64_t)q[1];
      o.flops = t < 2 ? class_flops(X, Y, (double)q[0], (double)q[1], (double)q[2], P->last_do_j, P->last_do_k)
                      : (t == 2 || t == 4) ? grad_flops(X, Y, (double)q[0], (double)q[1], (double)q[2])
                               : jengine_flops(X, Y, (double)q[1]);
    }
    ++n;
  }
  *count = n;
  P->prof_log.clear();
  P->prof_ev_used = 0;
  P->prof_builds = 0;
  return ERI_OK;
}

extern "C" int eri_plan_destroy(eri_plan_t* plan) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  if (!P) return ERI_OK;
  cudaSetDevice(P->device);
  cudaDeviceSynchronize();
  P->release();
  delete P;
  return ERI_OK;
}

extern "C" const char* eri_strerror(int code) {
  switch (code) {
    case ERI_OK: return "success";
    case ERI_EINVAL: return "invalid argument";
    case ERI_ENOMEM: return "out of memory";
    case ERI_ECUDA: return "CUDA runtime error";
    case ERI_EUNSUPPORTED: return "unsupported request";
    case ERI_ETIMEOUT: return "bounded device wait timed out";
    case ERI_EDEVICE: return "device-side check failed";
  }
  return "unknown error";
}
