// Point-charge attraction matrix V and its gradient (Sec. 2.4 of Wang et al.).
//
//   V_mn = sum_C q_C (m| 1/|r - C| |n)                       Eq. v1e_definition
//        = sum_{prim pairs} (2 pi / p) C_m C_n K_AB sum_P E_P^{mn} sum_C q_C R^0_P(p, P - C)
//                                                            Eq. v1e_formula
// The sum over charges is taken in Hermite space first, exactly like the
// J-engine's ket sum (Eq. j_formula): per primitive pair of every shell pair,
//   h_P = sum_C q_C (2 pi / p) C C K R^0_P(p, P - C),
// then one Hermite-to-Cartesian pass (the J-engine's k_post_j) gives V.
//
// Gradient of E_V = sum_mn D_mn V_mn with D fixed (SI Sec. 1.3,
// Eq. si_v1e_derivative_A / _B / _C).  With the Hermite densities of each
// primitive pair (sign-free, the pair counted in both orders)
//   d_P      = s sum_mn D'_mn E_P^{mn},     dR_{t,P} = s sum_mn D'_mn E_P^{(1_t) mn}
// (E^{(1_t)}: the derivative of E with respect to (A-B)_t at fixed P, in closed
// form from E, see kernels_g.cuh), the pair moves as a whole with P:
//   dE/dP_t = sum_C q_C sum_P d_P R_{P+1_t},   dE/dA = (a/p) dE/dP + g_R,
//   dE/dB = (b/p) dE/dP - g_R,   g_{R,t} = sum_P dR_{t,P} sum_C q_C R_P,
//   dE/dC_t = -q_C sum_pairs sum_P d_P R_{P+1_t}.
// The sums over charges commute with the densities, so A and B need only
// h_P = sum_C q_C R_P to order l1 + l2 + 1, like V itself; per (pair, charge) the
// work is one R table, its addition to h and the 3 nherm(l1 + l2) products of
// dE/dC.  One kernel does all three (a kernel per pair and one per charge built R
// twice and contracted six densities per term); dE/dC is transposed through
// shared memory so that a lane sums one charge over the warp's 32 pairs (3
// additions per charge instead of 15 shuffles).
// Bound by the FP64 pipe.  12 atoms and 3001 charges on GB300, V plus gradient:
// 64.7 ms with a kernel per pair and one per charge, 37.7 ms with this one, 10.7 ms
// with chunks sized to the lists and the pair orders side by side.
#include <algorithm>
#include <vector>

#include "../../include/eri.h"
#include "dispatch.cuh"
#include "plan.cuh"

using namespace eri;

namespace {

static_assert(2 * LMAX + 1 <= eri_plan_impl::kStreams, "one stream per pair order");
constexpr double kVfac = 1.0622519320271968;  // (2 pi / p) / (sqrt(2 pi^(5/2)) / p): pair prefactor of V from the ERI one
constexpr int kChunk = 256;  // charges per warp at most
constexpr int kTr = 16;      // at least (and the charges whose gradients are transposed at a time)

// A warp takes 32 primitive pairs and a chunk of the charges.  The chunks are as
// long as leave 16 warps per SM: the lists of f pairs are short, and in fixed
// chunks of 256 charges ten (ff) pairs were 12 warps with 2 ms each.
struct NucGrid {
  int groups, chunk, blocks;
};
inline NucGrid nuc_grid(const eri_plan_impl* P, int n, int nc) {
  NucGrid g;
  g.groups = (n + 31) / 32;
  const int64_t c = (int64_t)nc * g.groups / (16 * (int64_t)P->nsm);
  g.chunk = (int)std::max<int64_t>(kTr, std::min<int64_t>(kChunk, c / kTr * kTr));
  const int64_t warps = (int64_t)g.groups * ((nc + g.chunk - 1) / g.chunk);
  g.blocks = (int)((warps + 3) / 4);
  return g;
}

#define NCK(x)                                                                   \
  do {                                                                           \
    cudaError_t e_ = (x);                                                        \
    if (e_ != cudaSuccess) return e_ == cudaErrorMemoryAllocation ? ERI_ENOMEM : ERI_ECUDA; \
  } while (0)

__device__ __forceinline__ double warp_add(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// h_P of one list entry (primitive pair) summed over one chunk of charges
template <int L>
__global__ void __launch_bounds__(128) k_nuc_herm(const int4* __restrict__ list, int n, NucGrid ng, PairData pd,
                                                  BoysTabs bt, int nc, const double* __restrict__ q,
                                                  const double* __restrict__ xyz, double* __restrict__ Vh) {
  constexpr int NH = nherm(L);
  const int64_t warp = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
  const int i = (int)(warp % ng.groups) * 32 + (threadIdx.x & 31);
  const int64_t c0 = warp / ng.groups * ng.chunk;
  if (i >= n || c0 >= nc) return;
  const int4 e = __ldg(list + i);
  const int pi = e.x;
  const double p = __ldg(pd.p + pi), pref = __ldg(pd.pref + pi) * kVfac;
  const double Px = __ldg(pd.P + pi), Py = __ldg(pd.P + pd.n + pi), Pz = __ldg(pd.P + 2 * pd.n + pi);
  double h[NH];
#pragma unroll
  for (int x = 0; x < NH; ++x) h[x] = 0.0;
  const int c1 = (int)min((int64_t)nc, c0 + ng.chunk);
  for (int c = (int)c0; c < c1; ++c) {
    const double X = Px - __ldg(xyz + 3 * c), Y = Py - __ldg(xyz + 3 * c + 1), Z = Pz - __ldg(xyz + 3 * c + 2);
    double F[L + 1];
    boys_f64<L>(p * (X * X + Y * Y + Z * Z), bt, F);
    double R[NH];
    r_build_reg<L, double>(F, pref * __ldg(q + c), X, Y, Z, -2.0 * p, R);
#pragma unroll
    for (int x = 0; x < NH; ++x) h[x] += R[x];
  }
#pragma unroll
  for (int x = 0; x < NH; ++x) atomicAdd(Vh + e.y + x, h[x]);
}

// Layout of a primitive pair's gradient block: d_P [H], dR_x, dR_y, dR_z [H each],
// h [H1], H = nherm(l1 + l2), H1 = nherm(l1 + l2 + 1)
__host__ __device__ constexpr int grad_block(int L) { return 4 * nherm(L) + nherm(L + 1); }

// d_P and dR_{t,P} of every primitive pair, h = 0 (one warp per shell pair, a
// lane per Hermite index; E is zero outside t <= i + j)
__global__ void __launch_bounds__(128)
    k_nuc_dens(int npair, const int* __restrict__ s1, const int* __restrict__ s2, const int* __restrict__ np,
               const int* __restrict__ poff, const int* __restrict__ goff, const int* __restrict__ eoff,
               const int* __restrict__ sh_l, const int* __restrict__ pao1, const int* __restrict__ pao2,
               const int* __restrict__ pmol, MolMats mm, PairData pd, const double* __restrict__ Dp,
               double* __restrict__ G) {
  const int ip = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (ip >= npair) return;
  const int a = s1[ip], b = s2[ip], la = sh_l[a], lb = sh_l[b], L = la + lb;
  const int H = nherm(L), H1 = nherm(L + 1), stride = grad_block(L), ne = (la + 1) * (lb + 1) * (L + 1);
  const int m = pmol[ip], nbf = mm.n[m];
  const double* Dm = Dp + mm.off[m];
  const double sc = a == b ? 1.0 : 2.0;
  for (int k = 0; k < np[ip]; ++k) {
    const int pi = poff[ip] + k;
    const double ea = pd.ea[pi], aop = ea / pd.p[pi], bop = 1.0 - aop;
    const double* E = pd.E + eoff[ip] + (size_t)k * 3 * ne;
    double* out = G + goff[ip] + (size_t)k * stride;
    for (int q = lane; q < H; q += 32) {
      const int t[3] = {herm_t(q), herm_u(q), herm_v(q)};
      double s0 = 0.0, sr[3] = {0.0, 0.0, 0.0};
      for (int mu = 0; mu < ncart(la); ++mu) {
        int i3[3];
        cart_xyz(la, mu, i3[0], i3[1], i3[2]);
        for (int nu = 0; nu < ncart(lb); ++nu) {
          int j3[3];
          cart_xyz(lb, nu, j3[0], j3[1], j3[2]);
          const double dv = sc * Dm[(size_t)(pao1[ip] + mu) * nbf + pao2[ip] + nu];
          double e[3], e1[3];
          for (int d = 0; d < 3; ++d) {
            const double* r = E + d * ne + (i3[d] * (lb + 1) + j3[d]) * (L + 1) + t[d];
            e[d] = *r;
            double v = 2.0 * ea * pd.PA[d * pd.n + pi] * e[d];
            if (i3[d] > 0) v = fma(-bop * i3[d], r[-(lb + 1) * (L + 1)], v);
            if (j3[d] > 0) v = fma(aop * j3[d], r[-(L + 1)], v);
            e1[d] = v;
          }
          s0 = fma(dv, e[0] * e[1] * e[2], s0);
          sr[0] = fma(dv, e1[0] * e[1] * e[2], sr[0]);
          sr[1] = fma(dv, e[0] * e1[1] * e[2], sr[1]);
          sr[2] = fma(dv, e[0] * e[1] * e1[2], sr[2]);
        }
      }
      out[q] = s0;
      for (int d = 0; d < 3; ++d) out[(1 + d) * H + q] = sr[d];
    }
    for (int q = lane; q < H1; q += 32) out[4 * H + q] = 0.0;
  }
}

// h_P of one primitive pair over one chunk of charges, and dE/dC of the chunk
// (dEdC may be null) over the block's pairs
template <int L>
__global__ void __launch_bounds__(128) k_nuc_grad(const int4* __restrict__ list, int n, NucGrid ng, PairData pd,
                                                  BoysTabs bt, double* __restrict__ G, int nc, const double* __restrict__ q,
                                                  const double* __restrict__ xyz, double* __restrict__ dEdC) {
  constexpr int H = nherm(L), H1 = nherm(L + 1);
  __shared__ double tr[4][3 * kTr][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t warp = (int64_t)blockIdx.x * 4 + w;
  const int i = (int)(warp % ng.groups) * 32 + lane;
  const int64_t c0 = warp / ng.groups * ng.chunk;
  if (c0 >= nc) return;   // whole warp; nothing syncs the block
  const bool ok = i < n;  // lanes past the list repeat its last entry with weight 0
  const int4 e = __ldg(list + (ok ? i : n - 1));
  const int pi = e.x;
  const double p = __ldg(pd.p + pi), pref = ok ? __ldg(pd.pref + pi) * kVfac : 0.0;
  const double Px = __ldg(pd.P + pi), Py = __ldg(pd.P + pd.n + pi), Pz = __ldg(pd.P + 2 * pd.n + pi);
  const double* g = G + e.z;
  double h[H1];
#pragma unroll
  for (int x = 0; x < H1; ++x) h[x] = 0.0;
  const int c1 = (int)min((int64_t)nc, c0 + ng.chunk);
  for (int cb = (int)c0; cb < c1; cb += kTr) {
    const int ce = min(c1, cb + kTr);
    for (int c = cb; c < ce; ++c) {
      const double X = Px - __ldg(xyz + 3 * c), Y = Py - __ldg(xyz + 3 * c + 1), Z = Pz - __ldg(xyz + 3 * c + 2);
      double F[L + 2];
      boys_f64<L + 1>(p * (X * X + Y * Y + Z * Z), bt, F);
      double R[H1];
      r_build_reg<L + 1, double>(F, pref * __ldg(q + c), X, Y, Z, -2.0 * p, R);
#pragma unroll
      for (int x = 0; x < H1; ++x) h[x] += R[x];
      if (dEdC) {
        double s[3] = {0.0, 0.0, 0.0};
        for_herm<L>([&](auto x, auto y, auto z) {
          const double d = __ldg(g + herm_index(ERI_CI(x), ERI_CI(y), ERI_CI(z)));
          s[0] = fma(d, R[herm_index(ERI_CI(x) + 1, ERI_CI(y), ERI_CI(z))], s[0]);
          s[1] = fma(d, R[herm_index(ERI_CI(x), ERI_CI(y) + 1, ERI_CI(z))], s[1]);
          s[2] = fma(d, R[herm_index(ERI_CI(x), ERI_CI(y), ERI_CI(z) + 1)], s[2]);
        });
#pragma unroll
        for (int t = 0; t < 3; ++t) tr[w][3 * (c - cb) + t][lane] = s[t];
      }
    }
    if (dEdC) {
      __syncwarp();
      for (int r = lane; r < 3 * (ce - cb); r += 32) {
        double s = 0.0;
#pragma unroll 8
        for (int x = 0; x < 32; ++x) s += tr[w][r][x];
        atomicAdd(dEdC + 3 * cb + r, -s);
      }
      __syncwarp();
    }
  }
  if (ok) {
    double* hg = G + e.z + 4 * H;
#pragma unroll
    for (int x = 0; x < H1; ++x) atomicAdd(hg + x, h[x]);
  }
}

// dE/dA and dE/dB of every primitive pair from its densities and h
__global__ void __launch_bounds__(128)
    k_nuc_atoms(const int4* __restrict__ list, int n, int L, PairData pd, const int* __restrict__ s1,
                const int* __restrict__ s2, const int* __restrict__ sh_atom, const double* __restrict__ G,
                double* __restrict__ dEdR) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
  const bool ok = i < n;
  double gA[3] = {0.0, 0.0, 0.0}, gB[3] = {0.0, 0.0, 0.0};
  int atA = -1, atB = -1;
  if (ok) {
    const int4 e = __ldg(list + i);
    const int H = nherm(L);
    const double* g = G + e.z;
    const double* h = g + 4 * H;
    double gP[3] = {0.0, 0.0, 0.0}, gR[3] = {0.0, 0.0, 0.0};
    for (int q = 0; q < H; ++q) {
      const int t = herm_t(q), u = herm_u(q), v = herm_v(q);
      gP[0] = fma(g[q], h[herm_index(t + 1, u, v)], gP[0]);
      gP[1] = fma(g[q], h[herm_index(t, u + 1, v)], gP[1]);
      gP[2] = fma(g[q], h[herm_index(t, u, v + 1)], gP[2]);
      for (int d = 0; d < 3; ++d) gR[d] = fma(g[(1 + d) * H + q], h[q], gR[d]);
    }
    const double aop = __ldg(pd.ea + e.x) / __ldg(pd.p + e.x), bop = 1.0 - aop;
    atA = __ldg(sh_atom + __ldg(s1 + e.w));
    atB = __ldg(sh_atom + __ldg(s2 + e.w));
    for (int d = 0; d < 3; ++d) {
      gA[d] = fma(aop, gP[d], gR[d]);
      gB[d] = fma(bop, gP[d], -gR[d]);
    }
  }
  const int a0 = __shfl_sync(0xffffffffu, atA, 0), b0 = __shfl_sync(0xffffffffu, atB, 0);
  if (__all_sync(0xffffffffu, !ok || (atA == a0 && atB == b0))) {  // the warp's pairs share their atoms
    if (a0 < 0) return;
    for (int d = 0; d < 3; ++d) {
      const double x = warp_add(gA[d]), y = warp_add(gB[d]);
      if (lane == 0) {
        atomicAdd(dEdR + 3 * a0 + d, x);
        atomicAdd(dEdR + 3 * b0 + d, y);
      }
    }
  } else if (ok) {
    for (int d = 0; d < 3; ++d) {
      atomicAdd(dEdR + 3 * atA + d, gA[d]);
      atomicAdd(dEdR + 3 * atB + d, gB[d]);
    }
  }
}

template <int L>
cudaError_t launch_herm(const eri_plan_impl* P, int nc, const double* q, const double* xyz, cudaStream_t s) {
  const int n = P->nuc_cnt[L];
  if (n == 0 || nc == 0) return cudaSuccess;
  const NucGrid ng = nuc_grid(P, n, nc);
  k_nuc_herm<L><<<ng.blocks, 128, 0, s>>>(P->d_nuc_list + P->nuc_first[L], n, ng, P->pairdata(), P->boystabs(), nc, q,
                                          xyz, P->d_Jherm);
  return cudaGetLastError();
}

template <int L>
cudaError_t launch_grad(const eri_plan_impl* P, int nc, const double* q, const double* xyz, double* dEdR,
                        double* dEdC, cudaStream_t s) {
  const int n = P->nuc_cnt[L];
  if (n == 0 || nc == 0) return cudaSuccess;
  const int4* list = P->d_nuc_list + P->nuc_first[L];
  const NucGrid ng = nuc_grid(P, n, nc);
  k_nuc_grad<L><<<ng.blocks, 128, 0, s>>>(list, n, ng, P->pairdata(), P->boystabs(), P->d_nuc_dens, nc, q, xyz, dEdC);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_nuc_atoms<<<(n + 127) / 128, 128, 0, s>>>(list, n, L, P->pairdata(), P->d_ps1, P->d_ps2, P->d_sh_atom,
                                              P->d_nuc_dens, dEdR);
  return cudaGetLastError();
}

// Per-l1+l2 lists of every primitive pair and the offsets of their Hermite
// densities (basis only: built once per plan; synchronises the device).
int ensure_nuc(eri_plan_impl* P) {
  if (P->nuc_built) return ERI_OK;
  const int npair = P->npair;
  std::vector<int> s1(npair), s2(npair), np(npair), poff(npair), hoff(npair), shl(P->nshell);
  NCK(cudaMemcpy(s1.data(), P->d_ps1, sizeof(int) * npair, cudaMemcpyDeviceToHost));
  NCK(cudaMemcpy(s2.data(), P->d_ps2, sizeof(int) * npair, cudaMemcpyDeviceToHost));
  NCK(cudaMemcpy(np.data(), P->d_pnp, sizeof(int) * npair, cudaMemcpyDeviceToHost));
  NCK(cudaMemcpy(poff.data(), P->d_ppoff, sizeof(int) * npair, cudaMemcpyDeviceToHost));
  NCK(cudaMemcpy(hoff.data(), P->d_phoff, sizeof(int) * npair, cudaMemcpyDeviceToHost));
  NCK(cudaMemcpy(shl.data(), P->d_sh_l, sizeof(int) * P->nshell, cudaMemcpyDeviceToHost));
  constexpr int NL = 2 * LMAX + 1;
  std::vector<int4> lists[NL];
  std::vector<int> goff(npair);
  int64_t g = 0;
  for (int ip = 0; ip < npair; ++ip) {
    const int L = shl[s1[ip]] + shl[s2[ip]], H = nherm(L), G = grad_block(L);
    goff[ip] = (int)g;
    for (int k = 0; k < np[ip]; ++k) lists[L].push_back(make_int4(poff[ip] + k, hoff[ip] + k * H, (int)(g + (int64_t)k * G), ip));
    g += (int64_t)np[ip] * G;
    if (g > INT32_MAX) return ERI_EUNSUPPORTED;
  }
  std::vector<int4> all;
  for (int L = 0; L < NL; ++L) {
    P->nuc_first[L] = (int)all.size();
    P->nuc_cnt[L] = (int)lists[L].size();
    all.insert(all.end(), lists[L].begin(), lists[L].end());
  }
  P->nuc_first[NL] = (int)all.size();
  NCK(cudaMalloc(&P->d_nuc_list, sizeof(int4) * std::max<size_t>(1, all.size())));
  NCK(cudaMalloc(&P->d_nuc_goff, sizeof(int) * std::max(1, npair)));
  NCK(cudaMalloc(&P->d_nuc_dens, sizeof(double) * std::max<int64_t>(1, g)));
  NCK(cudaMemcpy(P->d_nuc_list, all.data(), sizeof(int4) * all.size(), cudaMemcpyHostToDevice));
  NCK(cudaMemcpy(P->d_nuc_goff, goff.data(), sizeof(int) * npair, cudaMemcpyHostToDevice));
  P->nuc_built = 1;
  return ERI_OK;
}

int check_charges(eri_plan_impl* P, int32_t nc, const double* q, const double* xyz) {
  if (!P || nc < 0 || (nc > 0 && (!q || !xyz))) return ERI_EINVAL;
  return ERI_OK;
}

}  // namespace

extern "C" int eri_nuclear(eri_plan_t* plan, int32_t ncharge, const double* q, const double* xyz, double* V,
                           void* stream) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  int rc = check_charges(P, ncharge, q, xyz);
  if (rc != ERI_OK || !V) return rc != ERI_OK ? rc : ERI_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  NCK(cudaSetDevice(P->device));
  if ((rc = ensure_nuc(P)) != ERI_OK) return rc;
  NCK(cudaMemsetAsync(P->d_Jherm, 0, sizeof(double) * (size_t)P->nherm_tot, s));
  // independent sums (atomics), one of the plan's streams each
  Fork side(s, P->branch, P->fork_ev, P->join_ev);
  NCK(side.open(2 * LMAX + 1));
  NCK(launch_herm<6>(P, ncharge, q, xyz, P->branch[0]));
  NCK(launch_herm<5>(P, ncharge, q, xyz, P->branch[1]));
  NCK(launch_herm<4>(P, ncharge, q, xyz, P->branch[2]));
  NCK(launch_herm<3>(P, ncharge, q, xyz, P->branch[3]));
  NCK(launch_herm<2>(P, ncharge, q, xyz, P->branch[4]));
  NCK(launch_herm<1>(P, ncharge, q, xyz, P->branch[5]));
  NCK(launch_herm<0>(P, ncharge, q, xyz, P->branch[6]));
  NCK(side.join());
  const MolMats mm = molmats(P);
  k_post_j<<<(int)(((int64_t)P->npair * 100 + 127) / 128), 128, 0, s>>>(
      P->npair, P->d_ps1, P->d_ps2, P->d_pnp, P->d_phoff, P->d_peoff, P->d_sh_l, P->d_pao1, P->d_pao2, P->d_pmol, mm,
      nullptr, P->d_E, P->d_Jherm, P->d_f, V, 0, P->d_status);
  NCK(cudaGetLastError());
  return ERI_OK;
}

extern "C" int eri_nuclear_grad(eri_plan_t* plan, const double* D, int32_t ncharge, const double* q,
                                const double* xyz, double* dEdR, double* dEdC, void* stream) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  int rc = check_charges(P, ncharge, q, xyz);
  if (rc != ERI_OK || !D || !dEdR) return rc != ERI_OK ? rc : ERI_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  NCK(cudaSetDevice(P->device));
  if ((rc = ensure_nuc(P)) != ERI_OK) return rc;
  const MolMats mm = molmats(P);
  k_scale_d_launch(P, D, s);
  NCK(cudaGetLastError());
  k_nuc_dens<<<(P->npair + 3) / 4, 128, 0, s>>>(P->npair, P->d_ps1, P->d_ps2, P->d_pnp, P->d_ppoff, P->d_nuc_goff,
                                                P->d_peoff, P->d_sh_l, P->d_pao1, P->d_pao2, P->d_pmol, mm,
                                                P->pairdata(), P->d_Dp, P->d_nuc_dens);
  NCK(cudaGetLastError());
  NCK(cudaMemsetAsync(dEdR, 0, sizeof(double) * 3 * (size_t)P->natom, s));
  if (dEdC && ncharge > 0) NCK(cudaMemsetAsync(dEdC, 0, sizeof(double) * 3 * (size_t)ncharge, s));
  // independent sums (atomics), one of the plan's streams each
  Fork side(s, P->branch, P->fork_ev, P->join_ev);
  NCK(side.open(2 * LMAX + 1));
  NCK(launch_grad<6>(P, ncharge, q, xyz, dEdR, dEdC, P->branch[0]));
  NCK(launch_grad<5>(P, ncharge, q, xyz, dEdR, dEdC, P->branch[1]));
  NCK(launch_grad<4>(P, ncharge, q, xyz, dEdR, dEdC, P->branch[2]));
  NCK(launch_grad<3>(P, ncharge, q, xyz, dEdR, dEdC, P->branch[3]));
  NCK(launch_grad<2>(P, ncharge, q, xyz, dEdR, dEdC, P->branch[4]));
  NCK(launch_grad<1>(P, ncharge, q, xyz, dEdR, dEdC, P->branch[5]));
  NCK(launch_grad<0>(P, ncharge, q, xyz, dEdR, dEdC, P->branch[6]));
  NCK(side.join());
  return ERI_OK;
}
