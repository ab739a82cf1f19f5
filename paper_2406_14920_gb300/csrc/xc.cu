// Exchange-correlation quadrature on a molecular grid (Sec. 2.6 of Wang et al.).
//
// The paper's four steps, each a device kernel here:
//  (1) grid        k_xc_nodes, k_xc_points: atom-centred products of a radial
//                  rule (Gauss-Chebyshev nodes of the second kind mapped by
//                  Becke's r = R (1+x)/(1-x)) and an angular rule
//                  (Gauss-Legendre in cos(theta) x trapezoid in phi, 2 n_theta
//                  azimuths), weighted by Becke's fuzzy cells of equal size;
//  (2) density     rho = sum_mn D_mn phi_m phi_n and grad rho
//                  (Eq. xc_density_0, Eq. xc_density_1): k_xc_ao, k_xc_rho;
//  (3) functional  Slater or Becke-88 exchange per point (k_xc_func);
//  (4) matrix      V_mn = sum_g w_g [v_rho phi_m phi_n + v_grad . grad(phi_m phi_n)]
//                  (Eq. xc_grid_sum_0 + Eq. xc_grid_sum_1): k_xc_vmat.
//
// Layout.  Points are grouped into blocks of at most 32 that are close in
// space: one atom, a group of adjacent radial shells and one thirty-second of
// the sphere (a quarter of the theta nodes x an eighth of the azimuths).  A block keeps
// the shells whose extent (the radius beyond which every component and its
// gradient stays below 1e-15) reaches its bounding sphere: the paper's grid
// boxes with pair cutoffs (Sec. 3.5), per shell instead of per pair.  The
// values phi and grad phi of every block's significant functions are computed
// once per geometry and kept in HBM ([block][component c = phi, d/dx, d/dy,
// d/dz][function][point]); above the workspace cap they are recomputed per
// chunk of blocks instead.  The density is one dense product X = D_b Phi_b per
// block, then rho = sum_m phi_m X_m and grad rho = 2 sum_m grad phi_m X_m; the
// matrix is V = sum_b (Z_b Phi_b^T + Phi_b Z_b^T) with
// Z = w (v_rho phi / 2 + v_grad . grad phi), one product A_b = Z_b Phi_b^T per
// block added to a half matrix by atomics, V = Vh + Vh^T at the end.  Both
// products run on the tensor cores as exact digit sums (xc_mma.cuh); everything
// else is FP64.
// Measured on GB300: 60 atoms, 900 functions, 983,040 points, Becke-88: 450 ms with
// both products on the FP64 pipe (at its peak), 69.5 ms now; 7 atoms, Slater: 1.59 ->
// 0.53 ms.  Bound by the issue of mma.sync, digit splitting and sums around it (the
// tensor pipe about 40 % busy).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "../../include/eri.h"
#include "plan.cuh"
#include "xc_mma.cuh"

using namespace eri;

namespace {

constexpr int kBP = 32;           // points per block (at most) = threads of the per-block kernels
constexpr int kWarps = kBP / 32;
constexpr int kRhoWarps = 4;      // k_xc_rho: warps per block, 16 rows of D_b each at a time
constexpr int kKC = 128;          // k_xc_rho: functions of Phi_b staged at a time
constexpr int kVWarps = 8;        // k_xc_vmat: warps per block, 16 rows of Z_b each at a time
constexpr int kVC = 128;          // k_xc_vmat: functions of Phi_b staged at a time
// V is summed in up to kParts half matrices, 2^kPartShift consecutive blocks to
// one (two or three are in L2 at a time), and these are added at the end: one sum
// over the thousands of blocks of an element loses sqrt(blocks) roundings (60
// atoms: 5.7e-15 of V against 1.6e-15).  They take at most kPartBytes: where that is
// too little for all of them (from 2,900 functions on), V itself is the first and the
// others are as many as fit (none from 11,586 functions on).
constexpr int kParts = 16, kPartShift = 8;
constexpr size_t kPartBytes = size_t(1) << 30;
constexpr int kSlots = 5;         // workspace rows per function: phi, d/dx, d/dy, d/dz, Z
constexpr double kAoEps = 1e-15;  // shell extent: every |phi| and |grad phi| below this beyond it
constexpr double kRhoMin = 1e-14; // points with a smaller density contribute nothing
constexpr double kPi = 3.14159265358979323846;
constexpr size_t kDefaultCap = size_t(16) << 30;  // default workspace cap for resident basis values

#define XCK(x)                                                                             \
  do {                                                                                     \
    cudaError_t e_ = (x);                                                                  \
    if (e_ != cudaSuccess) return e_ == cudaErrorMemoryAllocation ? ERI_ENOMEM : ERI_ECUDA; \
  } while (0)

template <typename T>
cudaError_t xalloc(T** p, size_t n) {
  *p = nullptr;
  return cudaMalloc((void**)p, std::max<size_t>(n, 1) * sizeof(T));
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Radial nodes r_i, weights (pi/(n+1)) sin(theta_i) r^2 dr/dx for i = 1..nrad
// (Gauss-Chebyshev of the second kind, Becke's map); Gauss-Legendre nodes in
// cos(theta) (ascending) and weights, by Newton's method on P_n.
__global__ void k_xc_nodes(int nrad, int ntheta, double R, double* __restrict__ rad, double* __restrict__ ang) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < nrad) {
    const int i = t + 1;
    const double th = i * kPi / (nrad + 1), x = cos(th);
    const double r = R * (1.0 + x) / (1.0 - x);
    rad[2 * t] = r;
    rad[2 * t + 1] = kPi / (nrad + 1) * sin(th) * r * r * 2.0 * R / ((1.0 - x) * (1.0 - x));
  }
  if (t < ntheta) {
    const int n = ntheta;
    double x = cos(kPi * (t + 0.75) / (n + 0.5)), dp = 1.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = x;
      for (int k = 2; k <= n; ++k) {
        const double p2 = ((2 * k - 1) * x * p1 - (k - 1) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      dp = n * (x * p1 - p0) / (x * x - 1.0);
      const double dx = p1 / dp;
      x -= dx;
      if (fabs(dx) < 1e-16) break;
    }
    double p0 = 1.0, p1 = x;
    for (int k = 2; k <= n; ++k) {
      const double p2 = ((2 * k - 1) * x * p1 - (k - 1) * p0) / k;
      p0 = p1;
      p1 = p2;
    }
    dp = n * (x * p1 - p0) / (x * x - 1.0);
    ang[2 * (n - 1 - t)] = x;
    ang[2 * (n - 1 - t) + 1] = 2.0 / ((1.0 - x * x) * dp * dp);
  }
}

// 1/|A - B| for every atom pair (0 on the diagonal)
__global__ void k_xc_invab(int na, const double* __restrict__ xyz, double* __restrict__ inv) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= na * na) return;
  const int a = i / na, b = i % na;
  if (a == b) {
    inv[i] = 0.0;
    return;
  }
  const double dx = xyz[3 * a] - xyz[3 * b], dy = xyz[3 * a + 1] - xyz[3 * b + 1], dz = xyz[3 * a + 2] - xyz[3 * b + 2];
  inv[i] = 1.0 / sqrt(dx * dx + dy * dy + dz * dz);
}

// Step (1): point g = ((atom * nrad + i) * ntheta + j) * nphi + k, weight
// w_rad * w_ang * (Becke weight of its atom)
__global__ void k_xc_points(int64_t G, int na, int nrad, int ntheta, const double* __restrict__ xyz,
                            const double* __restrict__ rad, const double* __restrict__ ang,
                            const double* __restrict__ invab, double* __restrict__ pts, double* __restrict__ w) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= G) return;
  const int nphi = 2 * ntheta;
  int64_t q = g;
  const int k = (int)(q % nphi); q /= nphi;
  const int j = (int)(q % ntheta); q /= ntheta;
  const int i = (int)(q % nrad); q /= nrad;
  const int a = (int)q;
  const double r = rad[2 * i], wr = rad[2 * i + 1];
  const double ct = ang[2 * j], st = sqrt(1.0 - ct * ct), wa = ang[2 * j + 1] * 2.0 * kPi / nphi;
  const double ph = 2.0 * kPi * (k + 0.5) / nphi;
  const double px = xyz[3 * a] + r * st * cos(ph), py = xyz[3 * a + 1] + r * st * sin(ph), pz = xyz[3 * a + 2] + r * ct;
  pts[3 * g] = px;
  pts[3 * g + 1] = py;
  pts[3 * g + 2] = pz;
  // Becke cells: P_A = prod_{B != A} s(mu_AB), w = P_a / sum_A P_A
  double sumP = 0.0, Pown = 0.0;
  for (int A = 0; A < na; ++A) {
    const double ax = px - __ldg(xyz + 3 * A), ay = py - __ldg(xyz + 3 * A + 1), az = pz - __ldg(xyz + 3 * A + 2);
    const double dA = sqrt(ax * ax + ay * ay + az * az);
    double P = 1.0;
    for (int B = 0; B < na && P != 0.0; ++B) {
      if (B == A) continue;
      const double bx = px - __ldg(xyz + 3 * B), by = py - __ldg(xyz + 3 * B + 1), bz = pz - __ldg(xyz + 3 * B + 2);
      double mu = (dA - sqrt(bx * bx + by * by + bz * bz)) * __ldg(invab + A * na + B);
      mu = 1.5 * mu - 0.5 * mu * mu * mu;
      mu = 1.5 * mu - 0.5 * mu * mu * mu;
      mu = 1.5 * mu - 0.5 * mu * mu * mu;
      P *= 0.5 * (1.0 - mu);
    }
    sumP += P;
    if (A == a) Pown = P;
  }
  w[g] = wr * wa * (sumP > 0.0 ? Pown / sumP : 0.0);
}

// bounding sphere (centre, radius) of every block
__global__ void __launch_bounds__(kBP) k_xc_bsph(const int* __restrict__ perm, const double* __restrict__ pts,
                                                 XcSphere* __restrict__ bsph) {
  __shared__ double red[kWarps][4];
  const int b = blockIdx.x, t = threadIdx.x, lane = t & 31, wp = t >> 5;
  const int g = perm[(int64_t)b * kBP + t];
  double x = 0.0, y = 0.0, z = 0.0, c = 0.0;
  if (g >= 0) {
    x = pts[3 * (int64_t)g];
    y = pts[3 * (int64_t)g + 1];
    z = pts[3 * (int64_t)g + 2];
    c = 1.0;
  }
  double sx = warp_sum(x), sy = warp_sum(y), sz = warp_sum(z), sc = warp_sum(c);
  if (lane == 0) { red[wp][0] = sx; red[wp][1] = sy; red[wp][2] = sz; red[wp][3] = sc; }
  __syncthreads();
  double n = 0.0, cx = 0.0, cy = 0.0, cz = 0.0;
#pragma unroll
  for (int x = 0; x < kWarps; ++x) {
    n += red[x][3];
    cx += red[x][0];
    cy += red[x][1];
    cz += red[x][2];
  }
  cx /= n;
  cy /= n;
  cz /= n;
  __syncthreads();
  double d = g >= 0 ? sqrt((x - cx) * (x - cx) + (y - cy) * (y - cy) + (z - cz) * (z - cz)) : 0.0;
  d = warp_max(d);
  if (lane == 0) red[wp][0] = d;
  __syncthreads();
  if (t == 0) {
    double rmax = 0.0;
#pragma unroll
    for (int x = 0; x < kWarps; ++x) rmax = fmax(rmax, red[x][0]);
    bsph[b] = XcSphere{cx, cy, cz, rmax};
  }
}

// extent of every shell: largest r (step 0.02 bohr, up to 80) where
// sum_k |c_k| f_max (r^l + l r^(l-1) + 2 a_k r^(l+1)) exp(-a_k r^2) >= kAoEps,
// a bound on every component and its gradient; a shell above the bound at
// 80 bohr (exponents below about 0.005) gets an unlimited extent
__global__ void k_xc_extent(int nshell, const int* __restrict__ sh_l, const int* __restrict__ sh_np,
                            const int* __restrict__ sh_po, const int* __restrict__ sh_ao,
                            const double* __restrict__ ex, const double* __restrict__ cn, const double* __restrict__ f,
                            double* __restrict__ ext) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= nshell) return;
  const int L = sh_l[s], np = sh_np[s], o = sh_po[s];
  double fm = 0.0;
  for (int k = 0; k < ncart(L); ++k) fm = fmax(fm, f[sh_ao[s] + k]);
  double e = 0.0;
  for (int st = 4000; st >= 0; --st) {
    const double r = 0.02 * st;
    double b = 0.0;
    for (int k = 0; k < np; ++k) {
      const double a = ex[o + k];
      double rl = 1.0;
      for (int x = 0; x < L; ++x) rl *= r;
      const double rlm = L > 0 ? (r > 0.0 ? rl / r : (L == 1 ? 1.0 : 0.0)) : 0.0;
      b += fabs(cn[o + k]) * fm * (rl + L * rlm + 2.0 * a * rl * r) * exp(-a * r * r);
    }
    if (b >= kAoEps) {
      e = st == 4000 ? 1e300 : r + 0.02;  // still significant at 80 bohr: never screened
      break;
    }
  }
  ext[s] = e;
}

// significant shells of every block (in shell order), their local function
// offsets, and the block's function list (global AO indices, ascending)
__global__ void __launch_bounds__(kBP) k_xc_sig(int nshell, int nbf, const XcSphere* __restrict__ bsph,
                                                const int* __restrict__ sh_atom, const int* __restrict__ sh_l,
                                                const int* __restrict__ sh_ao, const double* __restrict__ xyz,
                                                const double* __restrict__ ext, int* __restrict__ nsh,
                                                int* __restrict__ shl, int* __restrict__ shoff,
                                                int* __restrict__ nbfb, int* __restrict__ bfl) {
  __shared__ int wcnt[kWarps];
  __shared__ int base;
  const int b = blockIdx.x, t = threadIdx.x, lane = t & 31, wp = t >> 5;
  const XcSphere sp = bsph[b];
  int* myshl = shl + (int64_t)b * nshell;
  int* myoff = shoff + (int64_t)b * nshell;
  if (t == 0) base = 0;
  __syncthreads();
  for (int s0 = 0; s0 < nshell; s0 += kBP) {
    const int s = s0 + t;
    bool sig = false;
    if (s < nshell) {
      const int a = sh_atom[s];
      const double dx = sp.x - xyz[3 * a], dy = sp.y - xyz[3 * a + 1], dz = sp.z - xyz[3 * a + 2];
      sig = sqrt(dx * dx + dy * dy + dz * dz) - sp.r < ext[s];
    }
    const unsigned m = __ballot_sync(0xffffffffu, sig);
    if (lane == 0) wcnt[wp] = __popc(m);
    __syncthreads();
    int pre = base;
    for (int x = 0; x < wp; ++x) pre += wcnt[x];
    if (sig) myshl[pre + __popc(m & ((1u << lane) - 1u))] = s;
    __syncthreads();
    if (t == 0)
      for (int x = 0; x < kWarps; ++x) base += wcnt[x];
    __syncthreads();
  }
  const int n = base;
  if (t == 0) {
    int off = 0;
    for (int i = 0; i < n; ++i) {
      myoff[i] = off;
      off += ncart(sh_l[myshl[i]]);
    }
    nsh[b] = n;
    nbfb[b] = off;
  }
  __syncthreads();
  for (int i = t; i < n; i += kBP) {
    const int s = myshl[i], o = myoff[i], L = sh_l[s], ao = sh_ao[s];
    for (int k = 0; k < ncart(L); ++k) bfl[(int64_t)b * nbf + o + k] = ao + k;
  }
}

// phi and grad phi of a block's significant functions at its points
// (Eq. contracted_basis with the component norms)
__global__ void __launch_bounds__(kBP) k_xc_ao(int b0, const int* __restrict__ perm, const double* __restrict__ pts,
                                               const int* __restrict__ nsh, const int* __restrict__ shl,
                                               const int* __restrict__ shoff, const int* __restrict__ nbfb,
                                               int nshell, const int64_t* __restrict__ woff,
                                               const int* __restrict__ sh_atom, const int* __restrict__ sh_l,
                                               const int* __restrict__ sh_np, const int* __restrict__ sh_po,
                                               const int* __restrict__ sh_ao, const double* __restrict__ ex,
                                               const double* __restrict__ cn, const double* __restrict__ f,
                                               const double* __restrict__ xyz, double* __restrict__ work,
                                               int* __restrict__ pexp) {
  const int b = b0 + blockIdx.x, t = threadIdx.x;
  const int g = perm[(int64_t)b * kBP + t];
  const int n = nbfb[b], ns = nsh[b];
  int emax = 0;  // largest exponent of phi at this point
  double* W = work + woff[b];
  double px = 0.0, py = 0.0, pz = 0.0;
  if (g >= 0) {
    px = pts[3 * (int64_t)g];
    py = pts[3 * (int64_t)g + 1];
    pz = pts[3 * (int64_t)g + 2];
  }
  for (int i = 0; i < ns; ++i) {
    const int s = shl[(int64_t)b * nshell + i], o = shoff[(int64_t)b * nshell + i];
    const int L = sh_l[s], a = sh_atom[s], np = sh_np[s], po = sh_po[s], ao = sh_ao[s];
    const double d[3] = {px - xyz[3 * a], py - xyz[3 * a + 1], pz - xyz[3 * a + 2]};
    const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    double e0 = 0.0, e1 = 0.0;  // sum c exp(-a r^2), sum c a exp(-a r^2)
    for (int k = 0; k < np; ++k) {
      const double al = ex[po + k], e = cn[po + k] * exp(-al * r2);
      e0 += e;
      e1 += al * e;
    }
    if (g < 0) e0 = e1 = 0.0;
    for (int k = 0; k < ncart(L); ++k) {
      int e[3];
      cart_xyz(L, k, e[0], e[1], e[2]);
      double pw[3], pl[3], pu[3];  // d^e, d^(e-1) (0 if e = 0), d^(e+1)
      for (int x = 0; x < 3; ++x) {
        double v = 1.0;
        for (int q = 0; q < e[x]; ++q) v *= d[x];
        pw[x] = v;
        pu[x] = v * d[x];
        double vl = 1.0;
        for (int q = 1; q < e[x]; ++q) vl *= d[x];
        pl[x] = e[x] > 0 ? e[x] * vl : 0.0;
      }
      const double fc = f[ao + k];
      const int row = o + k;
      const double phi = fc * pw[0] * pw[1] * pw[2] * e0;
      emax = max(emax, exponent_of(phi));
      W[(int64_t)row * kBP + t] = phi;
      W[((int64_t)n + row) * kBP + t] = fc * (pl[0] * e0 - 2.0 * pu[0] * e1) * pw[1] * pw[2];
      W[((int64_t)2 * n + row) * kBP + t] = fc * (pl[1] * e0 - 2.0 * pu[1] * e1) * pw[0] * pw[2];
      W[((int64_t)3 * n + row) * kBP + t] = fc * (pl[2] * e0 - 2.0 * pu[2] * e1) * pw[0] * pw[1];
    }
  }
  pexp[(int64_t)b * kBP + t] = emax;
}

// Digits of D, 8 f16 per element (16 bytes), row by row under the row's exponent,
// which is kept (2047: the row holds an infinity or NaN)
__global__ void __launch_bounds__(256) k_xc_ddigits(int nbf, const double* __restrict__ D, uint4* __restrict__ Dd,
                                                    int* __restrict__ dexp) {
  __shared__ int red[8];
  const int r = blockIdx.x, t = threadIdx.x;
  const double* row = D + (int64_t)r * nbf;
  int E = 0;
  for (int c = t; c < nbf; c += blockDim.x) E = max(E, exponent_of(row[c]));
  E = __reduce_max_sync(0xffffffffu, E);
  if ((t & 31) == 0) red[t >> 5] = E;
  __syncthreads();
#pragma unroll
  for (int x = 0; x < 8; ++x) E = max(E, red[x]);
  if (t == 0) dexp[r] = E;
  for (int c = t; c < nbf; c += blockDim.x) {
    const unsigned long long u = digits_of(row[c], E);
    Dd[(int64_t)r * nbf + c] = make_uint4(digit_two(u, 0), digit_two(u, 2), digit_two(u, 4), digit_two(u, 6));
  }
}

// Step (2): X_m = sum_n D_mn phi_n at every point of the block, then
// rho = sum_m phi_m X_m, grad rho = 2 sum_m grad phi_m X_m (D symmetric).
// A warp owns 16 rows of X x the 32 points (nine accumulators of 16 values per
// lane).  It gathers the digit rows of D at the block's functions (16 B per
// element, from L2) one step of 16 ahead with cp.async, so that the L2 latency
// runs under the 172 products of a step (read straight into registers, 2.7 of 8.5
// issue slots waited on it); the digits of kKC functions of Phi_b are staged in
// shared memory in operand order.  X goes through shared
// memory to a lane per point for the sums with phi and grad phi.  A block that
// holds a function with an infinity or NaN in its row of D takes the plain sums.
struct RhoSmem {
  uint2 B[kKC / 16][kBP / 8][kDigits][32];
  // two steps of a warp's operand A, 16 B per element of D, rows 17 elements apart
  // (no bank conflicts); X, the warp's 16 x 32 sums, takes their place at the end
  union {
    uint4 A[2][16][17];
    double X[16][kBP];
  } w[kRhoWarps];
  double sum[kRhoWarps][4][kBP];
  int pexp[kBP];
};
__global__ void __launch_bounds__(32 * kRhoWarps, 2)
    k_xc_rho(int b0, int nbf, const int* __restrict__ perm, const int* __restrict__ nbfb, const int* __restrict__ bfl,
             const int64_t* __restrict__ woff, const double* __restrict__ work, const int* __restrict__ pexp,
             const double* __restrict__ D, const uint4* __restrict__ Dd, const int* __restrict__ dexp,
             double* __restrict__ rho, double* __restrict__ grad) {
  extern __shared__ __align__(16) unsigned char smraw[];
  RhoSmem& S = *reinterpret_cast<RhoSmem*>(smraw);
  const int b = b0 + blockIdx.x, tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const int n = nbfb[b];
  const int* L = bfl + (int64_t)b * nbf;
  const double* W = work + woff[b];
  int isbad = 0;
  for (int i = tid; i < n; i += 32 * kRhoWarps) isbad |= dexp[L[i]] == 2047;
  isbad = __syncthreads_or(isbad);
  double sum[4] = {0.0, 0.0, 0.0, 0.0};  // rho, grad rho / 2 of point `lane` over this warp's rows
  auto add_row = [&](int row, double x) {
#pragma unroll
    for (int c = 0; c < 4; ++c) sum[c] = fma(W[((int64_t)c * n + row) * kBP + lane], x, sum[c]);
  };
  if (isbad) {
    for (int m = wp; m < n; m += kRhoWarps) {
      double x = 0.0;
      for (int c = 0; c < n; ++c) x = fma(D[(int64_t)L[m] * nbf + L[c]], W[(int64_t)c * kBP + lane], x);
      add_row(m, x);
    }
  } else {
    const int g = lane >> 2, t = lane & 3;  // operand row and column pair of this lane
    if (tid < kBP) S.pexp[tid] = pexp[(int64_t)b * kBP + tid];
    for (int mg = 0; mg < n; mg += 16 * kRhoWarps) {
      const int m0 = mg + 16 * wp;
      // step of 16 functions from k on: lane l copies column l % 16 of rows l / 16 + 2 i
      int arow[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) arow[i] = L[min(m0 + 2 * i + (lane >> 4), n - 1)];
      auto fetch = [&](int k, int stage) {
        if (m0 < n && k < n) {
          const uint4* col = Dd + __ldg(L + min(k + (lane & 15), n - 1));
#pragma unroll
          for (int i = 0; i < 8; ++i)
            copy16(&S.w[wp].A[stage][2 * i + (lane >> 4)][lane & 15], col + (int64_t)arow[i] * nbf);
        }
        copy_commit();
      };
      __syncwarp();  // X of the previous rows has been read
      fetch(0, 0);
      for (int seg = 0; seg < n; seg += kExactTerms) {
        const int send = min(n, seg + kExactTerms);
        float acc[kBP / 8][kWeights][4];
#pragma unroll
        for (int x = 0; x < kBP / 8; ++x)
#pragma unroll
          for (int k = 0; k < kWeights; ++k)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[x][k][c] = 0.0f;
        for (int kc = seg; kc < send; kc += kKC) {
          const int nks = (min(send - kc, kKC) + 15) / 16;
          __syncthreads();  // the previous chunk has been read
          // one pair of functions (k, k + 1) at one point per step, both halves of a 16-step
          // (four at a time: their loads are in flight together)
          const int ntask = nks * (kBP / 8) * 64;
#pragma unroll 1
          for (int e0 = tid; e0 < ntask; e0 += 4 * 32 * kRhoWarps) {
            double v[4][2];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int e = e0 + i * 32 * kRhoWarps, el = e & 31, h = (e >> 5) & 1, nt = (e >> 6) & (kBP / 8 - 1);
              const int k = kc + 16 * (e >> 8) + 2 * (el & 3) + 8 * h, p = 8 * nt + (el >> 2);
              v[i][0] = e < ntask && k < n ? W[(int64_t)k * kBP + p] : 0.0;
              v[i][1] = e < ntask && k + 1 < n ? W[(int64_t)(k + 1) * kBP + p] : 0.0;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int e = e0 + i * 32 * kRhoWarps, el = e & 31, h = (e >> 5) & 1, nt = (e >> 6) & (kBP / 8 - 1);
              if (e < ntask) {
                const int E = S.pexp[8 * nt + (el >> 2)];
                const unsigned long long u0 = digits_of(v[i][0], E), u1 = digits_of(v[i][1], E);
#pragma unroll
                for (int x = 0; x < kDigits; ++x) (&S.B[e >> 8][nt][x][el].x)[h] = digit_pair(u0, u1, x);
              }
            }
          }
          __syncthreads();
          if (m0 < n) {
            for (int ks = 0; ks < nks; ++ks) {
              const int k = kc + 16 * ks, stage = (k >> 4) & 1;
              if (k + 16 < send) fetch(k + 16, stage ^ 1);  // (X is in the way of the next segment's first step)
              else copy_commit();
              copy_wait<1>();
              __syncwarp();
              uint32_t a[kDigits][4];
#pragma unroll
              for (int h = 0; h < 2; ++h)  // columns 2t, 2t+1 and 2t+8, 2t+9 of rows g and g + 8
#pragma unroll
                for (int y = 0; y < 2; ++y) {
                  const uint4* e = &S.w[wp].A[stage][g + 8 * y][2 * t + 8 * h];
                  const uint4 u = e[0], v = e[1];
                  const uint32_t uu[4] = {u.x, u.y, u.z, u.w}, vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                  for (int x = 0; x < 4; ++x) {
                    a[2 * x][2 * h + y] = __byte_perm(uu[x], vv[x], 0x5410);
                    a[2 * x + 1][2 * h + y] = __byte_perm(uu[x], vv[x], 0x7632);
                  }
                }
              __syncwarp();  // the step has been read; its place may be refilled
#pragma unroll
              for (int nt = 0; nt < kBP / 8; ++nt)
#pragma unroll
                for (int y = 0; y < kDigits; ++y) {
                  const uint2 bb = S.B[ks][nt][y][lane];
#pragma unroll
                  for (int x = 0; x < kDigits; ++x)
                    if (x + y < kWeights) mma_f16(acc[nt][x + y], a[x], bb);
                }
            }
          }
        }
        if (m0 < n) {
          const int e0 = dexp[L[min(m0 + g, n - 1)]], e1 = dexp[L[min(m0 + g + 8, n - 1)]];
          __syncwarp();
#pragma unroll
          for (int nt = 0; nt < kBP / 8; ++nt)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const int p = 8 * nt + 2 * t + (c & 1);
              S.w[wp].X[g + 8 * (c >> 1)][p] = combine<false>(acc[nt], c, c < 2 ? e0 : e1, S.pexp[p]);
            }
          __syncwarp();
          // four rows at a time: their 16 values of phi and grad phi are in flight together
#pragma unroll 1
          for (int r = 0; r < 16; r += 4) {
            double v[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int c = 0; c < 4; ++c) v[i][c] = W[((int64_t)c * n + min(m0 + r + i, n - 1)) * kBP + lane];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const double x = m0 + r + i < n ? S.w[wp].X[r + i][lane] : 0.0;
#pragma unroll
              for (int c = 0; c < 4; ++c) sum[c] = fma(v[i][c], x, sum[c]);
            }
          }
          if (send < n) {
            __syncwarp();
            fetch(send, 0);
          }
        }
      }
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) S.sum[wp][c][lane] = sum[c];
  __syncthreads();
  if (wp == 0) {
    const int g = perm[(int64_t)b * kBP + lane];
    if (g < 0) return;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int x = 0; x < kRhoWarps; ++x)
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] += S.sum[x][c][lane];
    rho[g] = v[0];
    if (grad) {
#pragma unroll
      for (int c = 0; c < 3; ++c) grad[3 * (int64_t)g + c] = 2.0 * v[1 + c];
    }
  }
}

// Step (3): energy density eps, v_rho = d eps/d rho, v_grad = d eps/d(grad rho)
// of closed-shell Slater exchange (kind 1) or Becke-88 exchange (kind 2,
// beta = 0.0042, on the spin density rho/2); E_xc += sum w eps
__global__ void k_xc_func(int64_t G, int kind, const double* __restrict__ w, const double* __restrict__ rho,
                          const double* __restrict__ grad, double* __restrict__ vrho, double* __restrict__ vgrad,
                          double* __restrict__ exc) {
  __shared__ double red[8];
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double e = 0.0;
  if (g < G) {
    const double r = rho[g];
    double vr = 0.0, vg[3] = {0.0, 0.0, 0.0};
    if (r >= kRhoMin) {
      const double cx = 0.75 * cbrt(3.0 / kPi);
      if (kind == 1) {
        e = -cx * r * cbrt(r);
        vr = -4.0 / 3.0 * cx * cbrt(r);
      } else {
        const double cxs = 1.5 * cbrt(3.0 / (4.0 * kPi)), beta = 0.0042;
        const double rs = 0.5 * r, a = rs * cbrt(rs);
        const double g0 = grad[3 * g], g1 = grad[3 * g + 1], g2 = grad[3 * g + 2];
        const double x = 0.5 * sqrt(g0 * g0 + g1 * g1 + g2 * g2) / a, as = asinh(x);
        const double den = 1.0 + 6.0 * beta * x * as;
        const double F = beta * x * x / den;
        const double Fpx = (2.0 * beta * den - beta * x * (6.0 * beta * as + 6.0 * beta * x / sqrt(1.0 + x * x))) /
                           (den * den);  // F'(x) / x
        e = -2.0 * a * (cxs + F);
        vr = -4.0 / 3.0 * cbrt(rs) * (cxs + F - x * x * Fpx);
        const double sc = -Fpx / (2.0 * a);
        vg[0] = sc * g0;
        vg[1] = sc * g1;
        vg[2] = sc * g2;
      }
    }
    vrho[g] = vr;
    vgrad[3 * g] = vg[0];
    vgrad[3 * g + 1] = vg[1];
    vgrad[3 * g + 2] = vg[2];
    e *= w[g];
  }
  e = warp_sum(e);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = e;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
    atomicAdd(exc, s);
  }
}

// Step (4a): Z_m(g) = w_g (v_rho,g phi_m(g) / 2 + v_grad,g . grad phi_m(g)) for
// every significant function of the block (workspace slot 4)
__global__ void __launch_bounds__(kBP) k_xc_z(int b0, const int* __restrict__ perm, const int* __restrict__ nbfb,
                                              const int64_t* __restrict__ woff, const double* __restrict__ w,
                                              const double* __restrict__ vrho, const double* __restrict__ vgrad,
                                              double* __restrict__ work, int* __restrict__ bad) {
  const int b = b0 + blockIdx.x, t = threadIdx.x;
  const int g = perm[(int64_t)b * kBP + t];
  const int n = nbfb[b];
  double* W = work + woff[b];
  double pw = 0.0, pv = 0.0, g0 = 0.0, g1 = 0.0, g2 = 0.0;
  int inf = 0;
  if (g >= 0) {
    pw = w[g];
    pv = 0.5 * vrho[g];
    g0 = vgrad[3 * (int64_t)g];
    g1 = vgrad[3 * (int64_t)g + 1];
    g2 = vgrad[3 * (int64_t)g + 2];
  }
  for (int m = 0; m < n; ++m) {
    const double phi = W[(int64_t)m * kBP + t], dx = W[((int64_t)n + m) * kBP + t],
                 dy = W[((int64_t)2 * n + m) * kBP + t], dz = W[((int64_t)3 * n + m) * kBP + t];
    const double z = pw * (pv * phi + g0 * dx + g1 * dy + g2 * dz);
    W[((int64_t)4 * n + m) * kBP + t] = z;
    inf |= exponent_of(z) == 2047;
  }
  inf = __any_sync(0xffffffffu, inf);
  if (t == 0) bad[b] = inf;  // an infinity or NaN among the block's Z
}

// The digits of one function's 32 values that a lane holds as an operand (row or
// column `lane >> 2`, steps 16 s + 2t, +1, +8, +9): d[s][h][digit], h the half of
// the step; returns the function's exponent.  Whole warp; `row` may differ per lane.
__device__ __forceinline__ int operand_digits(const double* row, int t, uint32_t (&d)[2][2][kDigits]) {
  double2 v[2][2];
  int E = 0;
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      v[s][h] = *reinterpret_cast<const double2*>(row + 16 * s + 2 * t + 8 * h);
      E = max(E, max(exponent_of(v[s][h].x), exponent_of(v[s][h].y)));
    }
  E = max(E, __shfl_xor_sync(0xffffffffu, E, 1));  // the four lanes of the function
  E = max(E, __shfl_xor_sync(0xffffffffu, E, 2));
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const unsigned long long lo = digits_of(v[s][h].x, E), hi = digits_of(v[s][h].y, E);
#pragma unroll
      for (int x = 0; x < kDigits; ++x) d[s][h][x] = digit_pair(lo, hi, x);
    }
  return E;
}

// Step (4b): A_ij = sum_g Z_i(g) phi_j(g) of one block over its functions, added
// to the half matrix Vh.  A warp holds the digits of 16 functions of Z over the
// block's 32 points in registers and walks the staged functions of Phi, 8 at a
// time; the 32 points are one exact accumulation.  Half of the sums are put
// together in integers and half on the FP64 pipe (combine_fp64), so that neither
// pipe outlasts the tensor work of a tile.  (Tiles of V that walk every
// block waste products on functions a block does not hold, 2.8 times as many on
// workload 1 at 32 x 32.)
struct VmatSmem {
  uint2 B[kVC / 8][2][kDigits][32];
  int exp[kVC], ao[kVC];
};
__global__ void __launch_bounds__(32 * kVWarps, 2)
    k_xc_vmat(int b0, int nbf, const int* __restrict__ nbfb, const int* __restrict__ bfl,
              const int64_t* __restrict__ woff, const double* __restrict__ work, const int* __restrict__ bad, int parts,
              double* V, double* Vparts) {
  extern __shared__ __align__(16) unsigned char smraw[];
  VmatSmem& S = *reinterpret_cast<VmatSmem*>(smraw);
  const int b = b0 + blockIdx.x, tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const int n = nbfb[b];
  const int* L = bfl + (int64_t)b * nbf;
  const double* phi = work + woff[b];
  const double* Z = phi + (int64_t)4 * n * kBP;
  const int part = (b >> kPartShift) % parts;
  double* Vh = Vparts + (int64_t)part * nbf * nbf;
  if (V) Vh = part == 0 ? V : Vh - (int64_t)nbf * nbf;  // V is the first part
  if (bad[b]) {  // an infinity or NaN: plain sums
    for (int64_t o = tid; o < (int64_t)n * n; o += 32 * kVWarps) {
      const int i = (int)(o / n), j = (int)(o - (int64_t)i * n);
      double v = 0.0;
      for (int p = 0; p < kBP; ++p) v = fma(Z[(int64_t)i * kBP + p], phi[(int64_t)j * kBP + p], v);
      atomicAdd(Vh + (int64_t)L[i] * nbf + L[j], v);
    }
    return;
  }
  const int g = lane >> 2, t = lane & 3;
  for (int j0 = 0; j0 < n; j0 += kVC) {
    const int nj = min(kVC, n - j0), njt = (nj + 7) / 8;
    __syncthreads();  // the previous chunk has been read
    for (int nt = wp; nt < njt; nt += kVWarps) {
      const int j = min(j0 + 8 * nt + g, n - 1);
      uint32_t d[2][2][kDigits];
      const int E = operand_digits(phi + (int64_t)j * kBP, t, d);
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int x = 0; x < kDigits; ++x) S.B[nt][s][x][lane] = make_uint2(d[s][0][x], d[s][1][x]);
      if (t == 0) {
        S.exp[8 * nt + g] = E;
        S.ao[8 * nt + g] = L[j];
      }
    }
    __syncthreads();
    for (int m0 = 16 * wp; m0 < n; m0 += 16 * kVWarps) {
      const int i0 = min(m0 + g, n - 1), i1 = min(m0 + g + 8, n - 1);
      uint32_t a[2][kDigits][4];
      int e0, e1;
      {
        uint32_t d[2][2][kDigits];
        e0 = operand_digits(Z + (int64_t)i0 * kBP, t, d);
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
          for (int x = 0; x < kDigits; ++x) {
            a[s][x][0] = d[s][0][x];
            a[s][x][2] = d[s][1][x];
          }
        e1 = operand_digits(Z + (int64_t)i1 * kBP, t, d);
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
          for (int x = 0; x < kDigits; ++x) {
            a[s][x][1] = d[s][0][x];
            a[s][x][3] = d[s][1][x];
          }
      }
      double* v0 = Vh + (int64_t)L[i0] * nbf;
      double* v1 = Vh + (int64_t)L[i1] * nbf;
      const bool ok0 = m0 + g < n, ok1 = m0 + g + 8 < n;
      for (int nt = 0; nt < njt; ++nt) {
        float acc[kWeights][4];
#pragma unroll
        for (int k = 0; k < kWeights; ++k)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[k][c] = kMagic;
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
          for (int y = 0; y < kDigits; ++y) {
            const uint2 bb = S.B[nt][s][y][lane];
#pragma unroll
            for (int x = 0; x < kDigits; ++x)
              if (x + y < kWeights) mma_f16(acc[x + y], a[s][x], bb);
          }
        const int jl = 8 * nt + 2 * t, ej[2] = {S.exp[jl], S.exp[jl + 1]}, aj[2] = {S.ao[jl], S.ao[jl + 1]};
        double v[4];
#pragma unroll
        for (int c = 0; c < 4; ++c)
          v[c] = c & 1 ? combine_fp64(acc, c, c < 2 ? e0 : e1, ej[c & 1]) : combine<true>(acc, c, c < 2 ? e0 : e1, ej[c & 1]);
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (jl + (c & 1) < nj && (c < 2 ? ok0 : ok1) && v[c] != 0.0) atomicAdd((c < 2 ? v0 : v1) + aj[c & 1], v[c]);
      }
    }
  }
}

// V = Vh + Vh^T, Vh = sum of the parts: those of Vparts and (IN_V) V itself, whose
// elements (i, j) and (j, i) are read and written by one thread
template <bool IN_V>
__global__ void k_xc_symm(int nbf, int parts, const double* __restrict__ Vparts, double* V) {
  const int i = blockIdx.x;
  for (int j = threadIdx.x; j <= i; j += blockDim.x) {
    double v = IN_V ? V[(int64_t)i * nbf + j] + V[(int64_t)j * nbf + i] : 0.0;
    for (int p = 0; p < parts - IN_V; ++p) {
      const double* Vh = Vparts + (int64_t)p * nbf * nbf;
      v += Vh[(int64_t)i * nbf + j] + Vh[(int64_t)j * nbf + i];
    }
    V[(int64_t)i * nbf + j] = v;
    V[(int64_t)j * nbf + i] = v;
  }
}

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

void eri_plan_impl::xc_release() {
  void* ptrs[] = {xc.d_pts, xc.d_w, xc.d_rad, xc.d_ang, xc.d_invab, xc.d_perm, xc.d_bsph, xc.d_ext, xc.d_nsh,
                  xc.d_shl, xc.d_shoff, xc.d_nbfb, xc.d_bfl, xc.d_woff, xc.d_work, xc.d_rho, xc.d_grad,
                  xc.d_vrho, xc.d_vgrad, xc.d_pexp, xc.d_ddig, xc.d_dexp, xc.d_zbad, xc.d_vpart};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  xc = XcState{};
}

static int xc_build(eri_plan_impl* P, cudaStream_t s) {
  XcState& X = P->xc;
  const int na = P->natom, nrad = X.nrad, nth = X.ntheta, nphi = 2 * nth;
  // block table: (atom, group of nrb radial shells, one of kTP theta ranges, one
  // of kPP azimuth ranges), chunks of <= kBP points
  constexpr int kTP = 4, kPP = 8;
  const int patch = ((nth + kTP - 1) / kTP) * ((nphi + kPP - 1) / kPP);
  const int nrb = std::max(1, kBP / patch);
  std::vector<int> perm;
  perm.reserve((size_t)X.npts + kBP);
  std::vector<int> cur;
  auto flush = [&]() {
    for (size_t k = 0; k < cur.size(); k += kBP) {
      for (int t = 0; t < kBP; ++t) perm.push_back(k + t < cur.size() ? cur[k + t] : -1);
    }
    cur.clear();
  };
  for (int a = 0; a < na; ++a)
    for (int i0 = 0; i0 < nrad; i0 += nrb)
      for (int h = 0; h < kTP; ++h)
        for (int q = 0; q < kPP; ++q) {
          for (int i = i0; i < std::min(nrad, i0 + nrb); ++i)
            for (int j = h * nth / kTP; j < (h + 1) * nth / kTP; ++j)
              for (int k = q * nphi / kPP; k < (q + 1) * nphi / kPP; ++k)
                cur.push_back((int)(((int64_t)(a * nrad + i) * nth + j) * nphi + k));
          flush();
        }
  X.nblock = (int)(perm.size() / kBP);
  const int nb = X.nblock, ns = P->nshell, nbf = P->nbf;
  XCK(xalloc(&X.d_pts, 3 * (size_t)X.npts));
  XCK(xalloc(&X.d_w, (size_t)X.npts));
  XCK(xalloc(&X.d_rad, 2 * (size_t)nrad));
  XCK(xalloc(&X.d_ang, 2 * (size_t)nth));
  XCK(xalloc(&X.d_invab, (size_t)na * na));
  XCK(xalloc(&X.d_perm, perm.size()));
  XCK(xalloc(&X.d_bsph, (size_t)nb));
  XCK(xalloc(&X.d_ext, (size_t)ns));
  XCK(xalloc(&X.d_nsh, (size_t)nb));
  XCK(xalloc(&X.d_shl, (size_t)nb * ns));
  XCK(xalloc(&X.d_shoff, (size_t)nb * ns));
  XCK(xalloc(&X.d_nbfb, (size_t)nb));
  XCK(xalloc(&X.d_bfl, (size_t)nb * nbf));
  XCK(xalloc(&X.d_woff, (size_t)nb + 1));
  XCK(xalloc(&X.d_rho, (size_t)X.npts));
  XCK(xalloc(&X.d_grad, 3 * (size_t)X.npts));
  XCK(xalloc(&X.d_vrho, (size_t)X.npts));
  XCK(xalloc(&X.d_vgrad, 3 * (size_t)X.npts));
  XCK(xalloc(&X.d_pexp, (size_t)nb * kBP));
  XCK(xalloc(&X.d_ddig, (size_t)nbf * nbf));
  XCK(xalloc(&X.d_dexp, (size_t)nbf));
  XCK(xalloc(&X.d_zbad, (size_t)nb));
  const size_t nn8 = sizeof(double) * (size_t)nbf * nbf;
  X.parts = (int)std::min<size_t>(kParts, (size_t)(nb >> kPartShift) + 1);
  X.in_v = (size_t)X.parts * nn8 > kPartBytes;
  if (X.in_v) X.parts = (int)std::min<size_t>(X.parts, 1 + kPartBytes / nn8);
  XCK(xalloc(&X.d_vpart, (size_t)(X.parts - X.in_v) * nbf * nbf));
  XCK(cudaMemcpyAsync(X.d_perm, perm.data(), sizeof(int) * perm.size(), cudaMemcpyHostToDevice, s));
  const int nt = std::max(nrad, nth);
  k_xc_nodes<<<(nt + 127) / 128, 128, 0, s>>>(nrad, nth, X.radius, X.d_rad, X.d_ang);
  k_xc_invab<<<(na * na + 127) / 128, 128, 0, s>>>(na, P->d_coords, X.d_invab);
  k_xc_points<<<(int)((X.npts + 127) / 128), 128, 0, s>>>(X.npts, na, nrad, nth, P->d_coords, X.d_rad, X.d_ang,
                                                           X.d_invab, X.d_pts, X.d_w);
  k_xc_bsph<<<nb, kBP, 0, s>>>(X.d_perm, X.d_pts, X.d_bsph);
  k_xc_extent<<<(ns + 63) / 64, 64, 0, s>>>(ns, P->d_sh_l, P->d_sh_np, P->d_sh_po, P->d_sh_ao, P->d_exps, P->d_cn,
                                            P->d_f, X.d_ext);
  k_xc_sig<<<nb, kBP, 0, s>>>(ns, nbf, X.d_bsph, P->d_sh_atom, P->d_sh_l, P->d_sh_ao, P->d_coords, X.d_ext,
                              X.d_nsh, X.d_shl, X.d_shoff, X.d_nbfb, X.d_bfl);
  XCK(cudaGetLastError());
  // workspace plan: per block kSlots x n_b x kBP doubles; chunks under the cap
  std::vector<int> nbfb(nb);
  XCK(cudaMemcpyAsync(nbfb.data(), X.d_nbfb, sizeof(int) * nb, cudaMemcpyDeviceToHost, s));
  XCK(cudaStreamSynchronize(s));
  const size_t cap = std::max<size_t>(X.cap_bytes / sizeof(double), (size_t)kSlots * nbf * kBP);
  std::vector<int64_t> woff(nb + 1);
  X.chunk.assign(1, 0);
  X.sum_nb = X.sum_nb2 = X.sum_nbp = X.sum_nb2p = 0.0;
  size_t used = 0, peak = 0;
  for (int b = 0; b < nb; ++b) {
    const size_t need = (size_t)kSlots * nbfb[b] * kBP;
    if (used + need > cap) {
      X.chunk.push_back(b);
      used = 0;
    }
    woff[b] = (int64_t)used;
    used += need;
    peak = std::max(peak, used);
    int np = 0;
    for (int t = 0; t < kBP; ++t) np += perm[(size_t)b * kBP + t] >= 0;
    X.sum_nb += nbfb[b];
    X.sum_nb2 += (double)nbfb[b] * nbfb[b];
    X.sum_nbp += (double)nbfb[b] * np;
    X.sum_nb2p += (double)nbfb[b] * nbfb[b] * np;
  }
  X.chunk.push_back(nb);
  woff[nb] = 0;
  X.work_doubles = std::max<size_t>(peak, 1);
  X.resident = X.chunk.size() == 2;
  XCK(xalloc(&X.d_work, X.work_doubles));
  XCK(cudaMemcpyAsync(X.d_woff, woff.data(), sizeof(int64_t) * (nb + 1), cudaMemcpyHostToDevice, s));
  if (X.resident) {
    k_xc_ao<<<nb, kBP, 0, s>>>(0, X.d_perm, X.d_pts, X.d_nsh, X.d_shl, X.d_shoff, X.d_nbfb, ns, X.d_woff,
                               P->d_sh_atom, P->d_sh_l, P->d_sh_np, P->d_sh_po, P->d_sh_ao, P->d_exps, P->d_cn,
                               P->d_f, P->d_coords, X.d_work, X.d_pexp);
    XCK(cudaGetLastError());
  }
  X.built_serial = P->geom_serial;
  return ERI_OK;
}

// (re)build the grid after a change of coordinates
static int xc_ready(eri_plan_impl* P, cudaStream_t s) {
  if (P->xc.nrad == 0) return ERI_EINVAL;  // no grid requested
  if (P->xc.built_serial == P->geom_serial) return ERI_OK;
  // work queued on the old grid's buffers (any stream of this device) must end before they go
  XCK(cudaDeviceSynchronize());
  XcState keep;
  keep.nrad = P->xc.nrad;
  keep.ntheta = P->xc.ntheta;
  keep.radius = P->xc.radius;
  keep.cap_bytes = P->xc.cap_bytes;
  keep.npts = P->xc.npts;
  P->xc_release();
  P->xc.nrad = keep.nrad;
  P->xc.ntheta = keep.ntheta;
  P->xc.radius = keep.radius;
  P->xc.cap_bytes = keep.cap_bytes;
  P->xc.npts = keep.npts;
  const int rc = xc_build(P, s);
  if (rc != ERI_OK) {
    P->xc_release();
    return rc;
  }
  return ERI_OK;
}

static void xc_launch_ao(eri_plan_impl* P, int b0, int b1, cudaStream_t s) {
  XcState& X = P->xc;
  k_xc_ao<<<b1 - b0, kBP, 0, s>>>(b0, X.d_perm, X.d_pts, X.d_nsh, X.d_shl, X.d_shoff, X.d_nbfb, P->nshell, X.d_woff,
                                  P->d_sh_atom, P->d_sh_l, P->d_sh_np, P->d_sh_po, P->d_sh_ao, P->d_exps, P->d_cn,
                                  P->d_f, P->d_coords, X.d_work, X.d_pexp);
}

static int xc_density_impl(eri_plan_impl* P, const double* D, double* rho, double* grad, cudaStream_t s) {
  XcState& X = P->xc;
  const int nbf = P->nbf;
  XCK(cudaFuncSetAttribute(k_xc_rho, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RhoSmem)));
  k_xc_ddigits<<<nbf, 256, 0, s>>>(nbf, D, X.d_ddig, X.d_dexp);
  XCK(cudaGetLastError());
  for (size_t c = 0; c + 1 < X.chunk.size(); ++c) {
    const int b0 = X.chunk[c], b1 = X.chunk[c + 1];
    if (b1 <= b0) continue;
    if (!X.resident) xc_launch_ao(P, b0, b1, s);
    k_xc_rho<<<b1 - b0, 32 * kRhoWarps, sizeof(RhoSmem), s>>>(b0, nbf, X.d_perm, X.d_nbfb, X.d_bfl, X.d_woff, X.d_work,
                                                             X.d_pexp, D, X.d_ddig, X.d_dexp, rho, grad);
    XCK(cudaGetLastError());
  }
  return ERI_OK;
}

static int xc_matrix_impl(eri_plan_impl* P, const double* vrho, const double* vgrad, double* V, cudaStream_t s) {
  XcState& X = P->xc;
  const int nbf = P->nbf;
  double* first = X.in_v ? V : nullptr;
  if (first) XCK(cudaMemsetAsync(V, 0, sizeof(double) * (size_t)nbf * nbf, s));
  if (X.parts > X.in_v)
    XCK(cudaMemsetAsync(X.d_vpart, 0, sizeof(double) * (size_t)(X.parts - X.in_v) * nbf * nbf, s));
  XCK(cudaFuncSetAttribute(k_xc_vmat, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(VmatSmem)));
  for (size_t c = 0; c + 1 < X.chunk.size(); ++c) {
    const int b0 = X.chunk[c], b1 = X.chunk[c + 1];
    if (b1 <= b0) continue;
    if (!X.resident) xc_launch_ao(P, b0, b1, s);
    k_xc_z<<<b1 - b0, kBP, 0, s>>>(b0, X.d_perm, X.d_nbfb, X.d_woff, X.d_w, vrho, vgrad, X.d_work, X.d_zbad);
    k_xc_vmat<<<b1 - b0, 32 * kVWarps, sizeof(VmatSmem), s>>>(b0, nbf, X.d_nbfb, X.d_bfl, X.d_woff, X.d_work, X.d_zbad,
                                                             X.parts, first, X.d_vpart);
    XCK(cudaGetLastError());
  }
  if (first) k_xc_symm<true><<<nbf, 128, 0, s>>>(nbf, X.parts, X.d_vpart, V);
  else k_xc_symm<false><<<nbf, 128, 0, s>>>(nbf, X.parts, X.d_vpart, V);
  XCK(cudaGetLastError());
  return ERI_OK;
}

static int xc_check_plan(eri_plan_impl* P) {
  if (!P) return ERI_EINVAL;
  if (P->nmol != 1) return ERI_EUNSUPPORTED;
  return ERI_OK;
}

extern "C" int eri_xc_grid(eri_plan_t* plan, int32_t nrad, int32_t ntheta, double radius, double cap_bytes,
                           int64_t* npoints, void* stream) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  int rc = xc_check_plan(P);
  if (rc != ERI_OK) return rc;
  if (nrad < 2 || nrad > 1000 || ntheta < 2 || ntheta > 64 || (ntheta & 1) || !(radius > 0.0) ||
      !(radius < 1e6) || !(cap_bytes >= 0.0))
    return ERI_EINVAL;
  const int64_t G = (int64_t)P->natom * nrad * ntheta * 2 * ntheta;
  if (G >= (int64_t)1 << 31) return ERI_EUNSUPPORTED;  // point indices are int32
  cudaStream_t s = (cudaStream_t)stream;
  XCK(cudaSetDevice(P->device));
  XCK(cudaDeviceSynchronize());  // the old grid's buffers may still be read by queued work on any stream
  P->xc_release();
  P->xc.nrad = nrad;
  P->xc.ntheta = ntheta;
  P->xc.radius = radius;
  P->xc.cap_bytes = cap_bytes > 0.0 ? (size_t)std::min(cap_bytes, 1e18) : kDefaultCap;
  P->xc.npts = G;
  P->xc.built_serial = -1;
  rc = xc_ready(P, s);
  if (rc != ERI_OK) {
    P->xc_release();
    return rc;
  }
  if (npoints) *npoints = G;
  return ERI_OK;
}

extern "C" int eri_xc_get_grid(eri_plan_t* plan, double* points, double* weights, void* stream) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  int rc = xc_check_plan(P);
  if (rc != ERI_OK) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  XCK(cudaSetDevice(P->device));
  rc = xc_ready(P, s);
  if (rc != ERI_OK) return rc;
  if (points)
    XCK(cudaMemcpyAsync(points, P->xc.d_pts, sizeof(double) * 3 * P->xc.npts, cudaMemcpyDeviceToDevice, s));
  if (weights)
    XCK(cudaMemcpyAsync(weights, P->xc.d_w, sizeof(double) * P->xc.npts, cudaMemcpyDeviceToDevice, s));
  return ERI_OK;
}

extern "C" int eri_xc_density(eri_plan_t* plan, const double* D, double* rho, double* grad_rho, void* stream) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  int rc = xc_check_plan(P);
  if (rc != ERI_OK) return rc;
  if (!D || !rho) return ERI_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  XCK(cudaSetDevice(P->device));
  rc = xc_ready(P, s);
  if (rc != ERI_OK) return rc;
  return xc_density_impl(P, D, rho, grad_rho, s);
}

extern "C" int eri_xc_matrix(eri_plan_t* plan, const double* vrho, const double* vgrad, double* V, void* stream) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  int rc = xc_check_plan(P);
  if (rc != ERI_OK) return rc;
  if (!vrho || !vgrad || !V) return ERI_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  XCK(cudaSetDevice(P->device));
  rc = xc_ready(P, s);
  if (rc != ERI_OK) return rc;
  return xc_matrix_impl(P, vrho, vgrad, V, s);
}

extern "C" int eri_xc(eri_plan_t* plan, const double* D, int32_t functional, double* V, double* Exc, void* stream) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  int rc = xc_check_plan(P);
  if (rc != ERI_OK) return rc;
  if (!D || !V || !Exc || (functional != ERI_XC_SLATER && functional != ERI_XC_B88)) return ERI_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  XCK(cudaSetDevice(P->device));
  rc = xc_ready(P, s);
  if (rc != ERI_OK) return rc;
  XcState& X = P->xc;
  rc = xc_density_impl(P, D, X.d_rho, X.d_grad, s);
  if (rc != ERI_OK) return rc;
  XCK(cudaMemsetAsync(Exc, 0, sizeof(double), s));
  k_xc_func<<<(int)((X.npts + 255) / 256), 256, 0, s>>>(X.npts, functional, X.d_w, X.d_rho, X.d_grad, X.d_vrho,
                                                         X.d_vgrad, Exc);
  XCK(cudaGetLastError());
  return xc_matrix_impl(P, X.d_vrho, X.d_vgrad, V, s);
}

extern "C" int eri_xc_stats(eri_plan_t* plan, eri_xc_stats_t* st) {
  eri_plan_impl* P = reinterpret_cast<eri_plan_impl*>(plan);
  int rc = xc_check_plan(P);
  if (rc != ERI_OK) return rc;
  if (!st) return ERI_EINVAL;
  const XcState& X = P->xc;
  std::memset(st, 0, sizeof(*st));
  st->npoints = X.npts;
  st->nblock = X.nblock;
  st->block_points = kBP;
  st->sum_block_functions = X.sum_nb;
  st->sum_block_functions_sq = X.sum_nb2;
  st->workspace_bytes = (double)X.work_doubles * sizeof(double);
  st->resident = X.resident;
  st->nchunk = X.chunk.empty() ? 0 : (int32_t)X.chunk.size() - 1;
  // density X = D_b Phi_b (2 n_b^2 per point) and the rho / grad rho
  // epilogue (8 n_b); matrix Z_b Phi_b^T + Phi_b Z_b^T on the lower triangle
  // (2 n_b^2 per point) and Z (8 n_b); FMA = 2 FLOP
  st->flops_density = 2.0 * X.sum_nb2p + 8.0 * X.sum_nbp;
  st->flops_matrix = 2.0 * X.sum_nb2p + 8.0 * X.sum_nbp;
  return ERI_OK;
}
