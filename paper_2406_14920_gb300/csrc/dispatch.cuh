// Launch helpers for the class-specialised kernels.  Each bra class gets its own
// translation unit (k_bra<X>.cu, j_lab<N>.cu) so that the build compiles them
// in parallel.
#pragma once
#include <algorithm>
#include <atomic>
#include <type_traits>
#include "kernels_g.cuh"
#include "units.h"

namespace eri {

template <int X> struct ClassL;
template <> struct ClassL<0> { static constexpr int l1 = 0, l2 = 0; };
template <> struct ClassL<1> { static constexpr int l1 = 1, l2 = 0; };
template <> struct ClassL<2> { static constexpr int l1 = 1, l2 = 1; };
template <> struct ClassL<3> { static constexpr int l1 = 2, l2 = 0; };
template <> struct ClassL<4> { static constexpr int l1 = 2, l2 = 1; };
template <> struct ClassL<5> { static constexpr int l1 = 2, l2 = 2; };
template <> struct ClassL<6> { static constexpr int l1 = 3, l2 = 0; };
template <> struct ClassL<7> { static constexpr int l1 = 3, l2 = 1; };
template <> struct ClassL<8> { static constexpr int l1 = 3, l2 = 2; };
template <> struct ClassL<9> { static constexpr int l1 = 3, l2 = 3; };

// Resident blocks per SM of a kernel with `smem` bytes of dynamic shared memory
// (raising the kernel's limit first).  Both are constants of the kernel and the
// device, so they are asked for once per device and kept: the two runtime calls
// cost about 2 us, and a build of a small molecule is some fifty launches.
constexpr int kMaxDev = 64;
template <auto Kern>
cudaError_t blocks_per_sm(int threads, size_t smem, int* occ) {
  static std::atomic<int> known[kMaxDev] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  int n = dev < kMaxDev ? known[dev].load(std::memory_order_acquire) : 0;
  if (n == 0) {
    if (smem > 48 * 1024) {
      e = cudaFuncSetAttribute(Kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
    }
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, Kern, threads, smem);
    if (e != cudaSuccess) return e;
    if (n < 1) return cudaErrorInvalidConfiguration;
    if (dev < kMaxDev) known[dev].store(n, std::memory_order_release);
  }
  *occ = n;
  return cudaSuccess;
}

// Persistent launch of Kern over `workers` independent work items of `per_block`
// items per block: as many blocks as the items need, at most those the device holds.
template <auto Kern, typename Args>
cudaError_t launch_over(const Args& a, int64_t workers, int per_block, int threads, size_t smem, cudaStream_t s,
                        int nsm) {
  int occ = 0;
  const cudaError_t e = blocks_per_sm<Kern>(threads, smem, &occ);
  if (e != cudaSuccess) return e;
  const int64_t grid = std::min<int64_t>((workers + per_block - 1) / per_block, (int64_t)nsm * occ);
  Kern<<<(int)std::max<int64_t>(1, grid), threads, smem, s>>>(a);
  cudaError_t r = cudaGetLastError();
  if (r == cudaErrorInvalidValue && smem > 48 * 1024) {  // the limit was set in a context that cudaDeviceReset ended
    r = cudaFuncSetAttribute(Kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (r != cudaSuccess) return r;
    Kern<<<(int)std::max<int64_t>(1, grid), threads, smem, s>>>(a);
    r = cudaGetLastError();
  }
  return r;
}

// lanes that a list of n items can use: those of the largest split of a short list,
// see prim_split; longer lists fill the grid by themselves
template <typename T>
inline int64_t split_items(const WorkList& wl, int64_t n, SplitBy by) {
  const PrimSplit s = prim_split<T>(wl, 1, INT32_MAX, by);
  const int per = 32 / s.g;
  return (n * s.n * 32 + per - 1) / per;
}

// Thread kernel of a class in its form for short lists (where it has one: while the
// launch has two lanes and more for every item) or in the other one.
template <auto Short, auto Long, typename T, bool HAS_SHORT, typename Args>
cudaError_t launch_thread(const Args& a, const WorkList& wl, int64_t n, cudaStream_t s, int nsm) {
  if constexpr (HAS_SHORT) {
    int occ = 0;
    const cudaError_t e = blocks_per_sm<Short>(128, 0, &occ);
    if (e != cudaSuccess) return e;
    if (wl.nshard == 1 && 2 * n <= (int64_t)nsm * occ * 128)
      return launch_over<Short>(a, split_items<T>(wl, n, SplitBy::lanes), 128, 128, 0, s, nsm);
  }
  return launch_over<Long>(a, split_items<T>(wl, n, SplitBy::parts), 128, 128, 0, s, nsm);
}

// Blocks of a block kernel over a list of n items: short lists are split (by bra
// primitives, see prim_split) while that leaves SMs without a block.  More parts would
// be additions for nothing: other classes' launches run beside this one (split to
// every resident block, 75 functions took 1.53 ms, now 1.46).
template <typename T>
inline int64_t split_blocks(const WorkList& wl, int64_t n, int nsm) {
  return n * prim_split<T>(wl, n, nsm, SplitBy::blocks).n;
}

template <int LA, int LB, int LC, int LD, typename T>
cudaError_t launch_jk_t(const JKArgs& a, cudaStream_t s, int nsm) {
  const int64_t n = a.k.wl.total - a.k.wl.first;
  if (n <= 0) return cudaSuccess;
  if constexpr (use_thread_kernel(LA, LB, LC, LD, sizeof(T) == 4)) {
    constexpr bool blocks = block_when_short<LA, LB, LC, LD, T>();
    if constexpr (blocks) {
      using S = CShape<LA, LB, LC, LD, T>;
      if (n <= (int64_t)kShortList * nsm)
        return launch_over<jk_block_kernel<LA, LB, LC, LD, T>>(a, split_blocks<T>(a.k.wl, n, nsm), 1, S::NT, S::smem(), s, nsm);
    }
    // (the lane form of these larger classes would hold up to 108 sums through the
    // shuffles: ptxas spills all of it)
    return launch_thread<jk_thread_kernel<LA, LB, LC, LD, T, sizeof(T) == 8 && !blocks>,
                         jk_thread_kernel<LA, LB, LC, LD, T, false>, T, sizeof(T) == 8 && !blocks>(a, a.k.wl, n, s, nsm);
  } else if constexpr (use_block_kernel<LA, LB, LC, LD, T>()) {
    using S = CShape<LA, LB, LC, LD, T>;
    static_assert(S::smem() <= 227 * 1024, "block kernel exceeds 227 KB");
    return launch_over<jk_block_kernel<LA, LB, LC, LD, T>>(a, split_blocks<T>(a.k.wl, n, nsm), 1, S::NT, S::smem(), s, nsm);
  } else {
    using S = BShape<LA, LB, LC, LD, T>;
    constexpr int WPB = 4;
    constexpr size_t smem = S::table_bytes() + WPB * S::smem_per_warp();
    static_assert(smem <= 227 * 1024, "warp kernel block exceeds 227 KB");
    return launch_over<jk_warp_kernel<LA, LB, LC, LD, T>>(a, n, WPB, 32 * WPB, smem, s, nsm);
  }
}

// Launch of class pair (X, y) in precision P for y in YLO..YHI (compile-time
// chain of the ket classes of one compilation unit, see units.h)
template <int X, int P, int YLO, int YHI>
cudaError_t launch_jk_unit(int y, const JKArgs& a, cudaStream_t s, int nsm) {
  if constexpr (YLO > YHI || YLO > X) {
    return cudaErrorInvalidValue;
  } else {
    if (y == YLO) {
      constexpr int LA = ClassL<X>::l1, LB = ClassL<X>::l2, LC = ClassL<YLO>::l1, LD = ClassL<YLO>::l2;
      using T = std::conditional_t<P == 1, float, double>;
      return launch_jk_t<LA, LB, LC, LD, T>(a, s, nsm);
    }
    return launch_jk_unit<X, P, YLO + 1, YHI>(y, a, s, nsm);
  }
}

// Gradient launch of class pair (X, y) in precision P, y in 0..9 (compile-time
// chain; one compilation unit per (X, P), see units.h)
template <int X, int P, int Y = 0>
cudaError_t launch_grad_unit(int y, const GradArgs& a, cudaStream_t s, int nsm) {
  if constexpr (Y >= NPAIRCLASS) {
    return cudaErrorInvalidValue;
  } else {
    if (y == Y) {
      if (a.wl.total <= 0) return cudaSuccess;
      constexpr int LA = ClassL<X>::l1, LB = ClassL<X>::l2, LC = ClassL<Y>::l1, LD = ClassL<Y>::l2;
      using T = std::conditional_t<P == 1, float, double>;
      const int64_t n = a.wl.total - a.wl.first;
      if constexpr (use_grad_thread(LA, LB, LC, LD, P == 1)) {
        if constexpr (grad_block_when_short<LA, LB, LC, LD, T>()) {
          using S = GShape<LA, LB, LC, LD, T>;
          if (n <= (int64_t)kShortList * nsm)
            return launch_over<grad_block_kernel<LA, LB, LC, LD, T>>(a, split_blocks<T>(a.wl, n, nsm), 1, S::NT,
                                                                     S::smem(), s, nsm);
        }
        return launch_thread<grad_thread_kernel<LA, LB, LC, LD, T, P == 0>, grad_thread_kernel<LA, LB, LC, LD, T, false>, T,
                             P == 0>(a, a.wl, n, s, nsm);
      } else {
        using S = GShape<LA, LB, LC, LD, T>;
        static_assert(S::smem() <= 227 * 1024, "gradient block exceeds 227 KB");
        return launch_over<grad_block_kernel<LA, LB, LC, LD, T>>(a, split_blocks<T>(a.wl, n, nsm), 1, S::NT, S::smem(), s, nsm);
      }
    }
    return launch_grad_unit<X, P, Y + 1>(y, a, s, nsm);
  }
}

template <int LAB, int LCD, typename T>
cudaError_t launch_j_t(const JArgs& a, cudaStream_t s, int nsm) {
  const int64_t n = a.wl.total - a.wl.first;
  if (n <= 0) return cudaSuccess;
  constexpr bool small = j_footprint(LAB, LCD) <= kJAlways;
  if constexpr (use_j_thread(LAB, LCD)) {
    if (small || n > (int64_t)kJLong * nsm)
      return launch_over<j_thread_kernel<LAB, LCD, T>>(a, split_items<T>(a.wl, n, SplitBy::parts), 128, 128, 0, s, nsm);
  }
  if constexpr (small) {
    return cudaErrorInvalidValue;  // (not reached)
  } else {
    constexpr int WPB = 4;
    constexpr size_t smem = WPB * JShape<LAB, LCD, T>::smem_per_warp();
    static_assert(smem <= 227 * 1024, "J-engine block exceeds 227 KB");
    return launch_over<j_warp_kernel<LAB, LCD, T>>(a, n, WPB, 32 * WPB, smem, s, nsm);
  }
}

template <int LAB>
cudaError_t launch_j_lab(int LCD, int prec, const JArgs& a, cudaStream_t s, int nsm) {
#define ERI_JCASE(N) \
  case N: return prec ? launch_j_t<LAB, N, float>(a, s, nsm) : launch_j_t<LAB, N, double>(a, s, nsm);
  switch (LCD) {
    ERI_JCASE(0)
    ERI_JCASE(1)
    ERI_JCASE(2)
    ERI_JCASE(3)
    ERI_JCASE(4)
    ERI_JCASE(5)
    ERI_JCASE(6)
  }
#undef ERI_JCASE
  return cudaErrorInvalidValue;
}

// J/K entry points: explicitly instantiated once per entry of units.h in its own
// compilation unit (k_unit.cu), referenced from plan.cu
#define ERI_JK_UNIT_DECL(X, P, YLO, YHI) \
  extern template cudaError_t launch_jk_unit<X, P, YLO, YHI>(int, const JKArgs&, cudaStream_t, int);
ERI_JK_UNITS(ERI_JK_UNIT_DECL)
#undef ERI_JK_UNIT_DECL
#define ERI_GRAD_UNIT_DECL(X, P) extern template cudaError_t launch_grad_unit<X, P, 0>(int, const GradArgs&, cudaStream_t, int);
ERI_GRAD_UNITS(ERI_GRAD_UNIT_DECL)
#undef ERI_GRAD_UNIT_DECL
cudaError_t launch_j_lab0(int, int, const JArgs&, cudaStream_t, int);
cudaError_t launch_j_lab1(int, int, const JArgs&, cudaStream_t, int);
cudaError_t launch_j_lab2(int, int, const JArgs&, cudaStream_t, int);
cudaError_t launch_j_lab3(int, int, const JArgs&, cudaStream_t, int);
cudaError_t launch_j_lab4(int, int, const JArgs&, cudaStream_t, int);
cudaError_t launch_j_lab5(int, int, const JArgs&, cudaStream_t, int);
cudaError_t launch_j_lab6(int, int, const JArgs&, cudaStream_t, int);

}  // namespace eri
