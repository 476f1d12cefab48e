// Templated LBM kernels of the block forest.  Included once per velocity-set
// translation unit, which instantiates them through AMR_LBM_OPS.
//
// Population layout (every storage type): block-major, g[b * Q M + p * M + l],
// M = 4^D cells per block, l = i + 4 j + 16 k (collide_stream.cuh).  Two buffers A/B
// are used per level in ping-pong; a level's current buffer is bit L of `cur`.
// The stored values are the outgoing post-collision populations; every kernel
// reads a cell's pre-collision populations with gather_cell and writes them
// with scatter_cell (collide_stream.cuh).
#pragma once
#include "collide_stream.cuh"

#include <algorithm>

namespace amr {

// =========================================== coarse-to-fine linear interpolation
// Per parent block: every parent cell rescales its populations to the fine
// level (f_eq + (f - f_eq) r, Section 3.4.1) into shared memory; then, for
// each child c, fine cell (I,J,K) takes the multilinear interpolant of the
// 2^D parent cells of quadrant c at local coordinates -1/4 + I/2.  Writes the
// ghost cells of every child (mode_all = 0) or every cell (mode_all = 1).
// Neighbour rows of the blocks a CTA works on, copied to shared memory
// (the gathers and scatters read one entry per link).
template <int D>
__device__ __forceinline__ void stage_row(int32_t* dst, const int32_t* __restrict__ nbr, int b,
                                          int t, int nt) {
  constexpr int NK = Nbr<D>::K;
  for (int k = t; k < NK; k += nt) dst[k] = b >= 0 ? __ldg(nbr + (size_t)b * NBR_STRIDE + k) : NONE;
}

template <int D, int Q, class T, bool SOLID, bool COH = false>
__device__ __forceinline__ void interp_stage(typename Store<T>::R (*sF)[Block<D>::M],
                                             const T* __restrict__ fpar, int P,
                                             int l, double ratio, const int32_t* prow,
                                             const uint64_t* __restrict__ solidmask) {
  using S = Store<T>;
  using R = typename S::R;
  R f[Q];
  gather_cell<D, Q, T, SOLID, COH>(f, fpar, P, l, prow, solidmask);
  R rho, ux, uy, uz;
  moments<D, Q>(f, rho, ux, uy, uz);
  const R usq15 = R(1.5) * (ux * ux + uy * uy + uz * uz);
  const R r = R(ratio);
  static_for<0, Q>([&](auto Pp) {
    const R e = feq<D, Q, Pp>(rho, ux, uy, uz, usq15);
    sF[Pp][l] = e + (f[Pp] - e) * r;
  });
}

// Store the interpolated populations v of cell l of child ch.  mode_all (new
// children of an adaptation): values that old neighbours stored in the new
// block's place are moved first (scatter_cell MOVE); a solid cell takes the
// rest state.
template <int D, int Q, class T, bool SOLID>
__device__ __forceinline__ void store_child_cell(typename Store<T>::R (&v)[Q], T* __restrict__ fch,
                                                 int ch, int l, const int32_t* row,
                                                 const uint64_t* __restrict__ solidmask,
                                                 const int32_t* __restrict__ parent,
                                                 const int8_t* __restrict__ marks, int mode_all) {
  using S = Store<T>;
  using R = typename S::R;
  constexpr int M = Block<D>::M;
  if (mode_all & 4) {   // the level step: as they are, into the child's own slots
    const size_t own = (size_t)ch * (Q * M) + l;
    static_for<0, Q>([&](auto Pp) { fch[own + (size_t)Pp * M] = S::template save<D, Q, Pp>(v[Pp]); });
    return;
  }
  if (mode_all & 1) {
    auto is_new = [&](int blk) {
      const int pp = __ldg(parent + blk);
      return pp >= 0 && __ldg(marks + pp) > 0;
    };
    scatter_cell<D, Q, T, SOLID, true>(v, fch, ch, l, row, solidmask, is_new);
  } else {
    scatter_cell<D, Q, T, SOLID>(v, fch, ch, l, row, solidmask);
  }
}

template <int D, int Q, class T, bool SOLID>
__device__ __forceinline__ void interp_children(const typename Store<T>::R (*sF)[Block<D>::M],
                                                int l, T* __restrict__ fch, int c0, const uint64_t* __restrict__ cellmask,
                                                const int32_t (*crow)[Nbr<D>::K],
                                                const uint64_t* __restrict__ solidmask,
                                                const int32_t* __restrict__ parent,
                                                const int8_t* __restrict__ marks, int mode_all) {
  using S = Store<T>;
  using R = typename S::R;
  constexpr int NC = Block<D>::NC;
  const int i = Block<D>::ci(l), j = Block<D>::cj(l), k = Block<D>::ck(l);
  const R x = R(-0.25) + R(0.5) * R(i);
  const R y = R(-0.25) + R(0.5) * R(j);
  const R z = R(-0.25) + R(0.5) * R(k);
  R wgt[NC];
#pragma unroll
  for (int a = 0; a < NC; ++a) {
    R wv = ((a & 1) ? x : R(1) - x) * ((a & 2) ? y : R(1) - y);
    if (D == 3) wv *= (a & 4) ? z : R(1) - z;
    wgt[a] = wv;
  }
#pragma unroll 1
  for (int c = 0; c < NC; ++c) {
    const int ch = c0 + c;
    if (!(mode_all & 1)) {
      const uint64_t gm = __ldg(cellmask + 2 * (size_t)ch);   // ghost cells of the child
      if (gm == 0ull) continue;
      if (!((gm >> l) & 1ull)) continue;
    }
    R v[Q];
    if (SOLID && solidmask && ((__ldg(solidmask + ch) >> l) & 1ull)) {
      if (!(mode_all & 1)) continue;                 // solid cells keep the rest state
      static_for<0, Q>([&](auto Pp) { v[Pp] = R(VS<D, Q>::w[Pp]); });
    } else {
      const int qx = c & 1, qy = (c >> 1) & 1, qz = (c >> 2) & 1;
      int corner[NC];
#pragma unroll
      for (int a = 0; a < NC; ++a)
        corner[a] = Block<D>::cell(2 * qx + (a & 1), 2 * qy + ((a >> 1) & 1),
                                   2 * qz + ((a >> 2) & 1));
      static_for<0, Q>([&](auto Pp) {
        R acc = R(0);
#pragma unroll
        for (int a = 0; a < NC; ++a) acc += wgt[a] * sF[Pp][corner[a]];
        v[Pp] = acc;
      });
    }
    store_child_cell<D, Q, T, SOLID>(v, fch, ch, l, crow[c], solidmask, parent, marks,
                                     mode_all);
  }
}

template <int D, int Q, class T, bool SOLID>
__global__ void __launch_bounds__(128, 8)
    k_interp(const int32_t* __restrict__ list, int n, const T* __restrict__ fpar,
             T* __restrict__ fch, const int32_t* __restrict__ child0,
             const uint64_t* __restrict__ cellmask, const int32_t* __restrict__ nbr,
             const uint64_t* __restrict__ solidmask, const int32_t* __restrict__ parent,
             const int8_t* __restrict__ marks, double ratio, int mode_all) {
  using R = typename Store<T>::R;
  constexpr int M = Block<D>::M;
  constexpr int NC = Block<D>::NC;
  constexpr int NK = Nbr<D>::K;
  constexpr int BPC = 128 / M;
  __shared__ R sF[BPC][Q][M];
  __shared__ int32_t s_row[BPC][1 + NC][NK];   // the parent's row, then its children's
  const int slot = threadIdx.x / M;
  const int l = threadIdx.x - slot * M;
  const int bi = blockIdx.x * BPC + slot;
  const bool valid = bi < n;
  const int P = valid ? list[bi] : 0;
  const int c0 = valid ? child0[P] : 0;
  for (int r = 0; r <= NC; ++r)
    stage_row<D>(s_row[slot][r], nbr, valid ? (r == 0 ? P : c0 + r - 1) : NONE, l, M);
  __syncthreads();
  if (valid) interp_stage<D, Q, T, SOLID>(sF[slot], fpar, P, l, ratio, s_row[slot][0],
                                          solidmask);
  __syncthreads();
  if (!valid) return;
  interp_children<D, Q, T, SOLID>(sF[slot], l, fch, c0, cellmask, s_row[slot] + 1,
                                  solidmask, parent, marks, mode_all);
}

// ========================================== coarse-to-fine cubic interpolation
// Section 3.4.2: the interpolant is the polynomial with exponents 0..3 in
// each direction through all 4^D rescaled cells of the parent block, on the
// unit square / cube spanned by the corner cell centres (parent cell m at
// m/3).  That polynomial is the tensor product of 1D cubic Lagrange bases on
// the nodes 0, 1/3, 2/3, 1, so it is evaluated one direction at a time: child
// c's cell I sits at x = -1/12 + I/6 + c_x 2/3, i.e. at position q = I + 4 c_x
// of eight, and F(x, y, z) = sum_l w_K(l) sum_n w_J(n) sum_m w_I(m) F_mnl.
// A CTA of 64 threads handles 64/M parents: every thread rescales one parent
// cell into shared memory; then, child by child, the x, y (and z) sums run in
// three passes through shared memory, each thread producing one of the 4^D
// partial sums per pass (4 multiply-adds per population).
struct CubicW {
  double w[8][4];   // w[q][m]: weight of node m at position q = I + 4 c_d
};
constexpr CubicW make_cubic_w() {
  CubicW t{};
  for (int q = 0; q < 8; ++q)
    for (int m = 0; m < 4; ++m) {
      // in units of 1/12: position 2q - 1, nodes 0, 4, 8, 12
      double v = 1.0;
      for (int j = 0; j < 4; ++j)
        if (j != m) v *= double(2 * q - 1 - 4 * j) / double(4 * m - 4 * j);
      t.w[q][m] = v;
    }
  return t;
}
static __constant__ CubicW c_cubic_w = make_cubic_w();

template <int D, int Q, class T, bool SOLID>
// (ten CTAs per SM: what the shared memory of D3Q27 in FP32 leaves room for)
__global__ void __launch_bounds__(64, sizeof(typename Store<T>::R) == 8 ? 5 : 10)
    k_interp_cubic(const int32_t* __restrict__ list, int n, const T* __restrict__ fpar,
                   T* __restrict__ fch, const int32_t* __restrict__ child0,
                   const uint64_t* __restrict__ cellmask, const int32_t* __restrict__ nbr,
                   const uint64_t* __restrict__ solidmask, const int32_t* __restrict__ parent,
                   const int8_t* __restrict__ marks, double ratio, int mode_all) {
  using S = Store<T>;
  using R = typename S::R;
  constexpr int M = Block<D>::M;
  constexpr int NC = Block<D>::NC;
  constexpr int PPC = 64 / M;   // parents per CTA
  __shared__ R sF[PPC][Q][M];   // rescaled parent cells
  __shared__ R sA[PPC][Q][M];   // x sums
  __shared__ R sB[D == 3 ? PPC : 1][D == 3 ? Q : 1][M];   // x-y sums (3D)
  __shared__ R sw[8][4];
  const int slot = threadIdx.x / M;
  const int l = threadIdx.x - slot * M;
  const int i = Block<D>::ci(l), j = Block<D>::cj(l), k = Block<D>::ck(l);
  if (threadIdx.x < 32) sw[threadIdx.x >> 2][threadIdx.x & 3] = R(c_cubic_w.w[threadIdx.x >> 2][threadIdx.x & 3]);
  constexpr int NK = Nbr<D>::K;
  __shared__ int32_t s_row[PPC][1 + NC][NK];   // the parent's row, then its children's
  const int bi = blockIdx.x * PPC + slot;
  const bool valid = bi < n;
  const int P = valid ? list[bi] : 0;
  const int c0 = valid ? child0[P] : 0;
  chain_start();
  for (int r = 0; r <= NC; ++r)
    stage_row<D>(s_row[slot][r], nbr, valid ? (r == 0 ? P : c0 + r - 1) : NONE, l, M);
  __syncthreads();
  if (valid) interp_stage<D, Q, T, SOLID>(sF[slot], fpar, P, l, ratio, s_row[slot][0],
                                          solidmask);
  __syncthreads();
  for (int c = 0; c < NC; ++c) {
    const int cx = c & 1, cy = (c >> 1) & 1, cz = (c >> 2) & 1;
    const int ch = c0 + c;
    uint64_t gm = 0ull;
    if (valid) gm = (mode_all & 1) ? ~0ull : __ldg(cellmask + 2 * (size_t)ch);
    const bool need = gm != 0ull;   // uniform over the parent's threads
    // pass 1: thread (i, j, k) -> sum_m w_i(m) F(m, j, k)
    if (need) {
      const R w0 = sw[i + 4 * cx][0], w1 = sw[i + 4 * cx][1], w2 = sw[i + 4 * cx][2],
              w3 = sw[i + 4 * cx][3];
      const int r = 4 * j + 16 * k;
      static_for<0, Q>([&](auto Pp) {
        const R* f = sF[slot][Pp];
        sA[slot][Pp][l] = w0 * f[r] + w1 * f[r + 1] + w2 * f[r + 2] + w3 * f[r + 3];
      });
    }
    __syncthreads();
    // pass 2: thread (i, j, k) -> sum_n w_j(n) A(i, n, k)
    R out2[D == 2 ? Q : 1];
    if (need) {
      const R w0 = sw[j + 4 * cy][0], w1 = sw[j + 4 * cy][1], w2 = sw[j + 4 * cy][2],
              w3 = sw[j + 4 * cy][3];
      const int r = i + 16 * k;
      static_for<0, Q>([&](auto Pp) {
        const R* a = sA[slot][Pp];
        const R v = w0 * a[r] + w1 * a[r + 4] + w2 * a[r + 8] + w3 * a[r + 12];
        if constexpr (D == 3) sB[slot][Pp][l] = v;
        else out2[Pp] = v;
      });
    }
    if constexpr (D == 3) {
      __syncthreads();
    }
    // pass 3 (3D): thread (i, j, k) -> sum_l w_k(l) B(i, j, l); then the write
    if (need && ((gm >> l) & 1ull)) {
      R v[Q];
      const bool solid_cell = SOLID && solidmask && ((__ldg(solidmask + ch) >> l) & 1ull);
      if (solid_cell) {
        static_for<0, Q>([&](auto Pp) { v[Pp] = R(VS<D, Q>::w[Pp]); });
      } else if constexpr (D == 3) {
        const R w0 = sw[k + 4 * cz][0], w1 = sw[k + 4 * cz][1], w2 = sw[k + 4 * cz][2],
                w3 = sw[k + 4 * cz][3];
        const int r = i + 4 * j;
        static_for<0, Q>([&](auto Pp) {
          const R* b = sB[slot][Pp];
          v[Pp] = w0 * b[r] + w1 * b[r + 16] + w2 * b[r + 32] + w3 * b[r + 48];
        });
      } else {
        static_for<0, Q>([&](auto Pp) { v[Pp] = out2[Pp]; });
      }
      // solid cells: the rest state for new children, untouched otherwise
      if (!solid_cell || (mode_all & 1))
        store_child_cell<D, Q, T, SOLID>(v, fch, ch, l, s_row[slot][1 + c], solidmask,
                                         parent, marks, mode_all);
    }
    (void)cz;
    // 2D: pass 1 of the next child rewrites the x sums that pass 2 just read
    if constexpr (D == 2) __syncthreads();
  }
}

// ===================================================== fine-to-coarse averaging
// Section 3.4.3.  A child covers 2^D parent cells (g = gx + 2 gy [+ 4 gz]),
// each the mean of a 2^D group of the child's fine cells, which share one
// class.  The level step takes the groups of interface cells, the
// synchronisation (and the level step with cubic interpolation) every group
// that is not of ghosts; the parent cell must not be solid.

// The first cell of group g of a child.
template <int D>
__device__ __forceinline__ int group_cell(int g) {
  return Block<D>::cell(2 * (g & 1), 2 * ((g >> 1) & 1), 2 * ((g >> 2) & 1));
}

// The batched forms' averaging, by interface groups: one thread per fine cell
// gathers it and rescales it to the coarse level (f_eq + (f - f_eq) r) into
// shared memory; then one thread per taken group sums its 2^D cells and
// scatters the mean into the parent cell.

template <int D, int Q, class T, bool COH = false>
__device__ __forceinline__ void average_child(typename Store<T>::R (*sR)[Block<D>::M],
                                              bool valid, int P, int c, int ch,
                                              int l, T* __restrict__ fpar,
                                              const T* __restrict__ fch, const uint64_t* __restrict__ cellmask,
                                              const int32_t* crow, const int32_t* prow,
                                              double ratio) {
  using S = Store<T>;
  using R = typename S::R;
  constexpr int M = Block<D>::M;
  constexpr int NC = Block<D>::NC;
  const int i = Block<D>::ci(l), j = Block<D>::cj(l), k = Block<D>::ck(l);
  const int g = (i >> 1) + 2 * (j >> 1) + (D == 3 ? 4 * (k >> 1) : 0);
  auto parent_cell = [&](int gg) {
    return Block<D>::cell(2 * (c & 1) + (gg & 1), 2 * ((c >> 1) & 1) + ((gg >> 1) & 1),
                          2 * ((c >> 2) & 1) + ((gg >> 2) & 1));
  };
  auto taken = [&](int gg) {
    return (__ldg(cellmask + 2 * (size_t)ch + 1) >> group_cell<D>(gg)) & 1ull;
  };
  if (valid && taken(g)) {
    R f[Q];
    gather_cell<D, Q, T, false, COH>(f, fch, ch, l, crow, nullptr);
    R rho, ux, uy, uz;
    moments<D, Q>(f, rho, ux, uy, uz);
    const R usq15 = R(1.5) * (ux * ux + uy * uy + uz * uz);
    const R r = R(ratio);
    static_for<0, Q>([&](auto Pp) {
      const R e = feq<D, Q, Pp>(rho, ux, uy, uz, usq15);
      sR[Pp][l] = e + (f[Pp] - e) * r;
    });
  }
  __syncthreads();
  // one thread per taken group: the mean of its 2^D rescaled cells,
  // scattered into the parent cell
  if (valid && l < NC && taken(l)) {
    const int f0 = group_cell<D>(l);
    R acc[Q];
    const R inv = R(1) / R(NC);
    static_for<0, Q>([&](auto Pp) {
      R a = R(0);
#pragma unroll
      for (int s = 0; s < NC; ++s) a += sR[Pp][f0 + Block<D>::cell(s & 1, (s >> 1) & 1, (s >> 2) & 1)];
      acc[Pp] = a * inv;
    });
    scatter_cell<D, Q, T, false>(acc, fpar, P, parent_cell(l), prow, nullptr);
  }
}

// CTAs of THREADS threads per SM the register budget of the averaging (and of
// the summaries, which hold as much) is set for: 1024 threads for D3Q19 (64
// registers), 768 for D3Q27 (80).  Measured (marks and summaries of a cavity,
// D3Q19 / prism with cubic interpolation, D3Q27): 0.91 / 17.8 ms with 768 / 512
// threads, 0.88 / 16.9 with these, 0.94 / 17.1 with 1152 / 896 (spills).
template <int Q, class T, int THREADS>
constexpr int average_min_ctas() {
  return (Q == 9 ? 1024 : (sizeof(T) == 8 ? 384 : (Q == 27 ? 768 : 1024))) / THREADS;
}

// The averaging of a group's cells by x-pairs (3D; by cells in 2D): each of
// the four lanes of a group holds V of its 2^D cells, gathers and rescales
// them (f_eq + (f - f_eq) r = f + (f_eq - f)(1 - r), Section 3.4.3), sums them, and
// the lanes XA and XB apart sum theirs with a reduce-scatter: at each
// exchange a lane keeps half of the directions it carries, so that afterwards
// it holds the sums of a quarter of them, whose means it stores into the
// parent cell's slots.  Every lane of the warp takes part in the exchanges;
// `take` is the same for the lanes of a group.  Values stay as stored (the
// shift of the 16-bit types is the same on both sides of a mean).
template <int D, int Q, class T, int V, bool SOLID, int XA, int XB>
__device__ __forceinline__ void average_lanes(bool take, int ch, int P, int c, int g,
                                              const RowPos<D, V>& pos, const int32_t* nb,
                                              const uint64_t* sm, int flags,
                                              const T* fch, T* fpar,
                                              const int32_t* __restrict__ prow,
                                              const uint64_t* __restrict__ solidmask,
                                              typename Store<T>::R keep) {
  using S = Store<T>;
  using R = typename S::R;
  constexpr int PER = (Q + 3) / 4;      // directions a lane keeps
  constexpr int QP = 4 * PER;
  R v[QP];
#pragma unroll
  for (int p = Q; p < QP; ++p) v[p] = R(0);
  if (take) {
    Vec<T, V> in[Q];
    gather_row<D, Q, T, V, true, SOLID, false>(in, fch, ch, pos, nb, sm,
                                               SOLID && (flags & BF_SOLID));
    static_for<0, V>([&](auto I) {
      R f[Q];
      static_for<0, Q>([&](auto Pp) { f[Pp] = S::raw(in[Pp].v[I]); });
      const Relax<D, Q, S::kShifted, R> r(f);
      r.each([&](auto Pp, R w, R x) {
        const R y = relaxed(f[Pp], w, x, keep);
        if constexpr (I == 0) v[Pp] = y;
        else v[Pp] += y;
      });
    });
  } else {
#pragma unroll
    for (int p = 0; p < Q; ++p) v[p] = R(0);
  }
  int base = 0;
  auto halve = [&](auto K, int x) {     // K directions -> K / 2, with the lane x apart
    const bool hi = (threadIdx.x & x) != 0;
    if (hi) base += K / 2;
#pragma unroll
    for (int i = 0; i < K / 2; ++i) {
      const R send = hi ? v[i] : v[i + K / 2];
      const R recv = __shfl_xor_sync(0xffffffffu, send, x);
      v[i] = (hi ? v[i + K / 2] : v[i]) + recv;
    }
  };
  halve(std::integral_constant<int, QP>{}, XA);
  halve(std::integral_constant<int, QP / 2>{}, XB);
  if (!take) return;
  const int pc = Block<D>::cell(2 * (c & 1) + (g & 1), 2 * ((c >> 1) & 1) + ((g >> 1) & 1),
                                2 * ((c >> 2) & 1) + ((g >> 2) & 1));
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int p = base + j;
    if (p < Q)
      fpar[src_slot<D, Q>(p, P, pc, prow, SOLID ? solidmask : nullptr)] =
          S::from_raw(v[j] * (R(1) / R(Block<D>::NC)));
  }
}

// The weights as a device table (for a runtime p).
template <int D, int Q>
struct WeightTable {
  float w[Q];
};
template <int D, int Q>
constexpr WeightTable<D, Q> make_weight() {
  WeightTable<D, Q> t{};
  for (int p = 0; p < Q; ++p) t.w[p] = float(VS<D, Q>::w[p]);
  return t;
}
template <int D, int Q>
__device__ const WeightTable<D, Q> g_weight = make_weight<D, Q>();

// Two lanes of a group, x apart, hand one another half of the N directions
// they carry: NIN values of each before, 2 NIN of N / 2 after, in cell order
// (those of the lane without bit X first).  `base` becomes the first direction
// this lane keeps.
template <int N, int NIN, class R>
__device__ __forceinline__ void gather_half(R (&out)[N / 2][2 * NIN], const R (&in)[N][NIN], int x,
                                            int& base) {
  const bool hi = (threadIdx.x & x) != 0;
  if (hi) base += N / 2;
#pragma unroll
  for (int i = 0; i < N / 2; ++i)
#pragma unroll
    for (int c = 0; c < NIN; ++c) {
      const R keep = hi ? in[i + N / 2][c] : in[i][c];
      const R recv = __shfl_xor_sync(0xffffffffu, hi ? in[i][c] : in[i + N / 2][c], x);
      out[i][c] = hi ? recv : keep;
      out[i][NIN + c] = hi ? keep : recv;
    }
}

// Whole children: one warp per child in 3D, two children per warp in 2D.  Each
// of the four lanes of a group gathers V of its 2^D cells and rescales them
// (f_eq + (f - f_eq) r, Section 3.4.3); the group's lanes then exchange values
// until each holds all 2^D of a quarter of the directions, adds them in cell
// order and stores the means.  The order is part of the result: refinement
// marks are thresholds on values derived from this state, so its last bits
// must not follow the layout of the lanes (average_lanes, whose sums go by
// pairs, serves the level step only).  Synchronisation, criterion, summaries
// and inference of a 90,000-block cavity, D3Q19 FP32: 0.93 ms; 0.88 with sums
// by pairs here and in k_features, 1.40 with a thread per cell.
// by_parent: child item i is child i % N_c of list[i / N_c]; else it is the
// block list[i].  Every group of non-ghost cells is taken.
template <int D, int Q, class T, bool SOLID>
__global__ void __launch_bounds__(128, (average_min_ctas<Q, T, 128>()))
    k_average(const int32_t* __restrict__ list, int64_t n_items, bool by_parent,
              T* fpar, const T* fch, const int32_t* __restrict__ child0,
              const int32_t* __restrict__ parent, const uint64_t* __restrict__ cellmask,
              const int32_t* __restrict__ nbr, const uint64_t* __restrict__ solidmask,
              double ratio) {
  using S = Store<T>;
  using R = typename S::R;
  constexpr int V = D == 3 ? 2 : 1;
  constexpr int TPB = Block<D>::M / V;
  constexpr int NC = Block<D>::NC;
  constexpr int CPC = 128 / TPB;
  constexpr int NCODE = D == 2 ? 9 : 27;
  __shared__ int32_t s_nb[CPC][NCODE];
  __shared__ uint64_t s_sm[SOLID ? CPC : 1][SOLID ? NCODE : 1];
  const int slot = threadIdx.x / TPB, t = threadIdx.x % TPB;
  const int64_t item = (int64_t)blockIdx.x * CPC + slot;
  const bool valid = item < n_items;
  chain_start();
  int P = 0, c = 0, ch = 0, flags = 0;
  bool take = false;
  const RowPos<D, V> pos(t);
  const int g = (pos.i0 >> 1) + 2 * (Block<D>::cj(pos.l0) >> 1) +
                (D == 3 ? 4 * (Block<D>::ck(pos.l0) >> 1) : 0);
  if (valid) {
    if (by_parent) {
      P = __ldg(list + item / NC);
      c = (int)(item % NC);
      ch = __ldg(child0 + P) + c;
    } else {
      ch = __ldg(list + item);
      P = __ldg(parent + ch);
      c = ch - __ldg(child0 + P);
    }
    take = !((__ldg(cellmask + 2 * (size_t)ch) >> group_cell<D>(g)) & 1ull);
    if (SOLID && take) {
      const int pc = Block<D>::cell(2 * (c & 1) + (g & 1), 2 * ((c >> 1) & 1) + ((g >> 1) & 1),
                                    2 * ((c >> 2) & 1) + ((g >> 2) & 1));
      take = !((__ldg(solidmask + P) >> pc) & 1ull);
    }
    flags = stage_block<D, TPB, SOLID>(s_nb[slot], SOLID ? s_sm[slot] : nullptr, ch, t,
                                       block_lanes<TPB>(), nbr, solidmask, nullptr);
  }
  chain_wait();
  constexpr int QP = (Q + 3) / 4 * 4;   // directions, a quarter of them per lane
  R v[QP][V];
#pragma unroll
  for (int p = 0; p < QP; ++p)
#pragma unroll
    for (int i = 0; i < V; ++i) v[p][i] = R(0);
  if (take) {
    Vec<T, V> in[Q];
    gather_row<D, Q, T, V, true, SOLID, false>(in, fch, ch, pos, s_nb[slot],
                                               SOLID ? s_sm[slot] : nullptr,
                                               SOLID && (flags & BF_SOLID));
    const R r = R(ratio);
    static_for<0, V>([&](auto I) {
      R f[Q];
      static_for<0, Q>([&](auto Pp) { f[Pp] = S::template load<D, Q, Pp>(in[Pp].v[I]); });
      R rho, ux, uy, uz;
      moments<D, Q>(f, rho, ux, uy, uz);
      const R usq15 = R(1.5) * (ux * ux + uy * uy + uz * uz);
      static_for<0, Q>([&](auto Pp) {
        const R e = feq<D, Q, Pp>(rho, ux, uy, uz, usq15);
        v[Pp][I] = e + (f[Pp] - e) * r;
      });
    });
  }
  int base = 0;
  R v2[QP / 2][2 * V], v4[QP / 4][4 * V];
  gather_half<QP, V>(v2, v, D == 3 ? 2 : 1, base);          // the group's y (2D: x) neighbour
  gather_half<QP / 2, 2 * V>(v4, v2, D == 3 ? 8 : 4, base);   // its z (2D: y) neighbour
  if (!take) return;
  const int pc = Block<D>::cell(2 * (c & 1) + (g & 1), 2 * ((c >> 1) & 1) + ((g >> 1) & 1),
                                2 * ((c >> 2) & 1) + ((g >> 2) & 1));
  const R inv = R(1) / R(NC);
#pragma unroll
  for (int j = 0; j < QP / 4; ++j) {
    R sum = R(0);
#pragma unroll
    for (int i = 0; i < NC; ++i) sum += v4[j][i];
    const int p = base + j;
    if (p < Q) {
      sum *= inv;
      if constexpr (S::kShifted) sum -= __ldg(&g_weight<D, Q>.w[p]);
      fpar[src_slot<D, Q>(p, P, pc, nbr + (size_t)P * NBR_STRIDE, SOLID ? solidmask : nullptr)] =
          S::from_raw(sum);
    }
  }
}

// The level step's averaging (mode 0) over a list of (child block, group)
// items, the groups of 2^D interface cells of the fine level's boundary
// blocks whose parent cell is fluid: four lanes per group, so every lane is
// busy.  The kernel is bound by its chain of loads (item, neighbour row,
// populations, parent's row) and by the sectors its groups half use (64^3
// cavity with three extra levels: 41 us per launch against 44 with a lane per
// cell; the FP64 2D cavity, where the lanes' work counts, 1.66 -> 1.57 ms per
// 20 coarse steps).  Children are groups of N_c IDs from first_child on.
template <int D, int Q, class T, bool SOLID>
__global__ void __launch_bounds__(64, (average_min_ctas<Q, T, 64>()))
    k_average_groups(const int32_t* __restrict__ items, int n, T* fpar,
                     const T* fch, int first_child,
                     const int32_t* __restrict__ parent, const int32_t* __restrict__ nbr,
                     const uint64_t* __restrict__ solidmask, typename Store<T>::R keep) {
  constexpr int V = D == 3 ? 2 : 1;
  constexpr int NC = Block<D>::NC;
  constexpr int NCODE = D == 2 ? 9 : 27;
  constexpr int GPC = 64 / 4;
  __shared__ int32_t s_nb[GPC][NCODE];
  __shared__ uint64_t s_sm[SOLID ? GPC : 1][SOLID ? NCODE : 1];
  const int slot = threadIdx.x / 4, s = threadIdx.x & 3;
  const int64_t item = (int64_t)blockIdx.x * GPC + slot;
  const bool valid = item < n;
  chain_start();
  int ch = first_child, g = 0, P = 0, flags = 0;
  if (valid) {
    const int it = __ldg(items + item);
    ch = it >> 3;
    g = it & 7;
    P = __ldg(parent + ch);
    flags = stage_block<D, 4, SOLID>(s_nb[slot], SOLID ? s_sm[slot] : nullptr, ch, s,
                                     block_lanes<4>(), nbr, solidmask, nullptr);
  }
  const int l = D == 3 ? Block<D>::cell(2 * (g & 1), 2 * ((g >> 1) & 1) + (s & 1),
                                        2 * ((g >> 2) & 1) + (s >> 1))
                       : Block<D>::cell(2 * (g & 1) + (s & 1), 2 * ((g >> 1) & 1) + (s >> 1), 0);
  const RowPos<D, V> pos(l / V);
  chain_wait();
  average_lanes<D, Q, T, V, SOLID, 1, 2>(valid, ch, P, (ch - first_child) & (NC - 1), g, pos,
                                         s_nb[slot], SOLID ? s_sm[slot] : nullptr, flags, fch, fpar,
                                         nbr + (size_t)P * NBR_STRIDE, solidmask, keep);
}

// ================================================ batched instances (lock-step)
// Work items pack (instance, block) as inst << BATCH_SHIFT | block; each
// instance's buffers, tables and per-level factors come from its descriptor.
// The same step as k_collide_stream (no solid cells in a batch).
template <int D, int Q, class T, int THREADS>
__global__ void __launch_bounds__(THREADS, (row_min_ctas<Q, T, row_cells<D, Q, T>(), THREADS>()))
    k_collide_stream_batch(const uint32_t* __restrict__ items, int n,
                           const InstDesc* __restrict__ descs, int level, int which_in) {
  using R = typename Store<T>::R;
  constexpr int V = row_cells<D, Q, T>();
  constexpr int TPB = Block<D>::M / V, LPR = TPB < 32 ? TPB : 32;
  constexpr int BPC = THREADS / TPB;
  __shared__ int32_t s_nb[THREADS / LPR][D == 2 ? 9 : 27];
  const int row = threadIdx.x / LPR;
  const int t = threadIdx.x % TPB;
  const int bi = blockIdx.x * BPC + threadIdx.x / TPB;
  if (bi >= n) return;
  const uint32_t it = __ldg(items + bi);
  const InstDesc& d = descs[it >> BATCH_SHIFT];
  const int b = (int)(it & BATCH_MASK);
  const int flags = stage_block<D, LPR, false>(s_nb[row], nullptr, b, t % LPR, block_lanes<LPR>(),
                                               d.nbr, nullptr, &d.faces);
  step_row<D, Q, T, V, false, false, false, false>(
      (const T*)d.f[which_in], (T*)d.f[which_in ^ 1], b, t, s_nb[row], nullptr, flags, 0ull,
      R(d.omega[level]), d.faces, ParentOut<R>{nullptr, R(0)});
}

template <int D, int Q, class T>
__global__ void __launch_bounds__(128, 5)
    k_interp_batch(const uint32_t* __restrict__ items, int n, const InstDesc* __restrict__ descs,
                   int level, int which_par, int which_ch) {
  using R = typename Store<T>::R;
  constexpr int M = Block<D>::M;
  constexpr int NC = Block<D>::NC;
  constexpr int NK = Nbr<D>::K;
  constexpr int BPC = 128 / M;
  __shared__ R sF[BPC][Q][M];
  __shared__ int32_t s_row[BPC][1 + NC][NK];
  const int slot = threadIdx.x / M;
  const int l = threadIdx.x - slot * M;
  const int bi = blockIdx.x * BPC + slot;
  const bool valid = bi < n;
  int inst = 0, P = 0, c0 = 0;
  if (valid) {
    const uint32_t it = __ldg(items + bi);
    inst = (int)(it >> BATCH_SHIFT);
    P = (int)(it & BATCH_MASK);
    c0 = descs[inst].child0[P];
  }
  const InstDesc& d = descs[inst];
  for (int r = 0; r <= NC; ++r)
    stage_row<D>(s_row[slot][r], d.nbr, valid ? (r == 0 ? P : c0 + r - 1) : NONE, l, M);
  __syncthreads();
  if (valid)
    interp_stage<D, Q, T, false>(sF[slot], (const T*)d.f[which_par], P, l,
                                 d.r_cf[level], s_row[slot][0], nullptr);
  __syncthreads();
  if (!valid) return;
  interp_children<D, Q, T, false>(sF[slot], l, (T*)d.f[which_ch], c0, d.cellmask,
                                  s_row[slot] + 1, nullptr, nullptr, nullptr, 0);
}

// items are parents; child item i is child i % N_c of items[i / N_c]; one
// child per 4^D threads as in k_average
template <int D, int Q, class T>
__global__ void __launch_bounds__(128)
    k_average_batch(const uint32_t* __restrict__ items, int64_t n_items,
                    const InstDesc* __restrict__ descs, int level, int which_par, int which_ch) {
  using R = typename Store<T>::R;
  constexpr int M = Block<D>::M;
  constexpr int NC = Block<D>::NC;
  constexpr int NK = Nbr<D>::K;
  constexpr int CPC = 128 / M;
  __shared__ R sR[CPC][Q][M];
  __shared__ int32_t s_row[CPC][2][NK];
  const int slot = threadIdx.x / M;
  const int l = threadIdx.x - slot * M;
  const int64_t item = (int64_t)blockIdx.x * CPC + slot;
  const bool valid = item < n_items;
  int inst = 0, P = 0, c = 0, ch = 0;
  if (valid) {
    const uint32_t it = __ldg(items + item / NC);
    inst = (int)(it >> BATCH_SHIFT);
    P = (int)(it & BATCH_MASK);
    c = (int)(item % NC);
    ch = descs[inst].child0[P] + c;
  }
  const InstDesc& d = descs[inst];
  stage_row<D>(s_row[slot][0], d.nbr, valid ? ch : NONE, l, M);
  stage_row<D>(s_row[slot][1], d.nbr, valid ? P : NONE, l, M);
  __syncthreads();
  average_child<D, Q, T>(sR[slot], valid, P, c, ch, l, (T*)d.f[which_par],
                         (const T*)d.f[which_ch], d.cellmask, s_row[slot][0], s_row[slot][1],
                         d.r_fc[level]);
}

// ============================ batched instances: persistent form (PersistArgs)
__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Wait until *cnt >= target.  False when *abort is raised, or when `limit`
// clock64 cycles have passed (then this wait raises *abort itself).
__device__ __forceinline__ bool persist_wait(const uint32_t* cnt, uint32_t target, int32_t* abort,
                                             long long limit) {
  const long long t0 = clock64();
  for (;;) {
    if (ld_acquire_u32(cnt) >= target) return true;
    if (*(volatile int32_t*)abort) return false;
    if (clock64() - t0 > limit) {
      atomicExch(abort, 1);
      return false;
    }
    __nanosleep(64);
  }
}

// Collide-stream tile: `nblk` (<= PERSIST_MAX_TILE) active blocks of one
// member, their rows spread over the CTA's threads, V cells each.  The same step
// as k_collide_stream_batch, with every population read from L2.  `s_nb`: a row
// for each warp, which takes a block (half of one with V = 1 in 3D) at a time.
template <int D, int Q, class T, int THREADS, int V>
__device__ __forceinline__ void persist_collide(const InstDesc& d, const uint32_t* items, int nblk,
                                                int level, int which_in,
                                                int32_t (*s_nb)[D == 2 ? 9 : 27]) {
  using R = typename Store<T>::R;
  constexpr int TPB = Block<D>::M / V, LPR = TPB < 32 ? TPB : 32;
  constexpr int PARTS = TPB / LPR;      // of a block
  int32_t* nb = s_nb[threadIdx.x / LPR];
  for (int s = threadIdx.x / LPR; s < nblk * PARTS; s += THREADS / LPR) {
    const int b = (int)(__ldg(items + s / PARTS) & BATCH_MASK);
    const int t = s % PARTS * LPR + threadIdx.x % LPR;
    const int flags = stage_block<D, LPR, false>(nb, nullptr, b, t % LPR, block_lanes<LPR>(),
                                                 d.nbr, nullptr, &d.faces);
    step_row<D, Q, T, V, false, false, false, true>(
        (const T*)d.f[which_in], (T*)d.f[which_in ^ 1], b, t, nb, nullptr, flags, 0ull,
        R(d.omega[level]), d.faces, ParentOut<R>{nullptr, R(0)});
    __syncwarp(block_lanes<LPR>());     // the row is done with
  }
}

// Interpolation tile: THREADS / M parents of one member (as k_interp_batch).
// Out of line, like the averaging tile, so that their register needs do not
// weigh on the collide-stream tiles.
template <int D, int Q, class T, int THREADS>
__device__ __noinline__ void persist_interp(const InstDesc& d, const uint32_t* items, int ni,
                                            int tile, int level, int win, int wch,
                                            typename Store<T>::R (*sF)[Q][Block<D>::M],
                                            int32_t (*s_rows)[1 + Block<D>::NC][Nbr<D>::K]) {
  constexpr int M = Block<D>::M;
  constexpr int NC = Block<D>::NC;
  const int slot = threadIdx.x / M;
  const int l = threadIdx.x - slot * M;
  const int j = tile * (THREADS / M) + slot;
  const bool valid = j < ni;
  int P = 0, c0 = 0;
  if (valid) {
    P = (int)(__ldg(items + j) & BATCH_MASK);
    c0 = __ldg(d.child0 + P);
  }
  for (int rr = 0; rr <= NC; ++rr)
    stage_row<D>(s_rows[slot][rr], d.nbr, valid ? (rr == 0 ? P : c0 + rr - 1) : NONE, l, M);
  __syncthreads();
  if (valid)
    interp_stage<D, Q, T, false, true>(sF[slot], (const T*)d.f[win], P, l,
                                       d.r_cf[level], s_rows[slot][0], nullptr);
  __syncthreads();
  if (valid)
    interp_children<D, Q, T, false>(sF[slot], l, (T*)d.f[wch], c0, d.cellmask,
                                    s_rows[slot] + 1, nullptr, nullptr, nullptr, 0);
}

// Averaging tile: THREADS / M children of one member; child item j is child
// j % N_c of parent item j / N_c (as k_average_batch).
template <int D, int Q, class T, int THREADS>
__device__ __noinline__ void persist_average(const InstDesc& d, const uint32_t* items, int ni,
                                             int tile, int level, int win, int wch,
                                             typename Store<T>::R (*sF)[Q][Block<D>::M],
                                             int32_t (*s_rows)[1 + Block<D>::NC][Nbr<D>::K]) {
  constexpr int M = Block<D>::M;
  constexpr int NC = Block<D>::NC;
  const int slot = threadIdx.x / M;
  const int l = threadIdx.x - slot * M;
  const int j = tile * (THREADS / M) + slot;
  const bool valid = j < ni * NC;
  int P = 0, c = 0, ch = 0;
  if (valid) {
    P = (int)(__ldg(items + j / NC) & BATCH_MASK);
    c = j % NC;
    ch = __ldg(d.child0 + P) + c;
  }
  stage_row<D>(s_rows[slot][0], d.nbr, valid ? ch : NONE, l, M);
  stage_row<D>(s_rows[slot][1], d.nbr, valid ? P : NONE, l, M);
  __syncthreads();
  average_child<D, Q, T, true>(sF[slot], valid, P, c, ch, l, (T*)d.f[win],
                               (const T*)d.f[wch], d.cellmask, s_rows[slot][0], s_rows[slot][1],
                               d.r_fc[level]);
}

// CTAs per SM of the persistent kernel: the interpolation and averaging tiles
// and tiles smaller than the CTA leave threads idle, so larger CTAs are given
// more of them than the collide-stream's budget (threads per SM for CTAs of 64 /
// 128 / 256; three batches of 4 to 14 cavities, D3Q19 FP32, the largest tile of
// each, ms per two steps with 896 / 1024 / 1280 / 1536: CTAs of 64 1.19 / 1.21 /
// 1.39 / 2.04, of 128 1.24 / 1.16 / 1.19 / 1.38, of 256 1.47 / 1.31 / 1.28 / 1.39).
template <int Q, class T, int THREADS>
constexpr int persist_min_ctas() {
  constexpr int size = THREADS == 64 ? 0 : (THREADS == 128 ? 1 : 2);
  constexpr int f64[3][3] = {{1024, 1024, 1024}, {512, 512, 768}, {384, 384, 512}};
  constexpr int f32[3][3] = {{1152, 1280, 1536}, {896, 1024, 1280},
                             {704, sizeof(T) == 2 ? 768 : 896, sizeof(T) == 2 ? 768 : 1024}};
  constexpr int q = Q == 9 ? 0 : (Q == 19 ? 1 : 2);
  return (sizeof(T) == 8 ? f64 : f32)[q][size] / THREADS;
}

// The persistent kernel.  Dynamic shared memory: the rescaled populations of
// the THREADS / M parents (interpolation) or children (averaging) of a tile,
// then their neighbour rows.
template <int D, int Q, class T, int THREADS>
__global__ void __launch_bounds__(THREADS, (persist_min_ctas<Q, T, THREADS>()))
    k_batch_persistent(PersistArgs a) {
  using R = typename Store<T>::R;
  constexpr int M = Block<D>::M;
  constexpr int NC = Block<D>::NC;
  constexpr int NK = Nbr<D>::K;
  constexpr int U = THREADS / M;     // parents or children per interface tile
  extern __shared__ __align__(16) unsigned char s_dyn[];
  R (*sF)[Q][M] = reinterpret_cast<R (*)[Q][M]>(s_dyn);
  int32_t (*s_rows)[1 + NC][NK] =
      reinterpret_cast<int32_t (*)[1 + NC][NK]>(s_dyn + sizeof(R) * U * Q * M);
  __shared__ int32_t s_nb[THREADS / (D == 2 ? 16 : 32)][D == 2 ? 9 : 27];
  __shared__ long long s_take;
  __shared__ int32_t s_go;
  const long long total = (long long)a.tiles_per_step * a.n_steps;
  for (;;) {
    if (threadIdx.x == 0) {
      long long t = -1;
      if (!*(volatile int32_t*)a.abort) {
        const unsigned long long q = atomicAdd(a.head, 1ull);
        if ((long long)q < total) t = (long long)q;
      }
      s_take = t;
    }
    __syncthreads();
    const long long t = s_take;
    if (t < 0) return;
    const int step = (int)(t / a.tiles_per_step);
    const int r = (int)(t - (long long)step * a.tiles_per_step);
    const PersistPhase* list = a.phases + (size_t)((a.parity0 + step) & 1) * a.n_phase;
    // the phase: the last one starting at or before tile r (every listed
    // phase has tiles); the member: the last one whose tiles start at or
    // before the phase-local tile
    int lo = 0, hi = a.n_phase - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (__ldg(&list[mid].tile0) <= r) lo = mid;
      else hi = mid - 1;
    }
    const int k = lo;
    const int tt = r - __ldg(&list[k].tile0);
    const int32_t* toff = a.tile_off + (size_t)k * (a.n_inst + 1);
    int ilo = 0, ihi = a.n_inst - 1;
    while (ilo < ihi) {
      const int mid = (ilo + ihi + 1) >> 1;
      if (__ldg(toff + mid) <= tt) ilo = mid;
      else ihi = mid - 1;
    }
    const int inst = ilo;
    const int tile = tt - __ldg(toff + inst);
    if (threadIdx.x == 0) {
      int go = 1;
      const int dep = __ldg(a.dep + (size_t)k * a.n_inst + inst);
      const int dk = dep >> 1;
      const long long need = (long long)step + 1 - (dep & 1);   // coarse steps of phase dk
      if (need > 0) {
        const int32_t* doff = a.tile_off + (size_t)dk * (a.n_inst + 1);
        uint32_t target = (uint32_t)need * (uint32_t)(__ldg(doff + inst + 1) - __ldg(doff + inst));
        if (a.stall) target += 1u << 30;
        go = persist_wait(a.done + (size_t)dk * a.n_inst + inst, target, a.abort, a.wait_limit);
        if (!go)
          for (int i = 0; i < a.n_inst; ++i) atomicExch(a.descs[i].wait_flag, 1);
      }
      __threadfence();
      s_go = go;
    }
    __syncthreads();
    if (!s_go) return;
    const InstDesc& d = a.descs[inst];
    const int op = __ldg(&list[k].op), level = __ldg(&list[k].level);
    const int win = __ldg(&list[k].which_in), wch = __ldg(&list[k].which_ch);
    const int32_t i0 = __ldg(a.item_off + (size_t)k * (a.n_inst + 1) + inst);
    const int32_t ni = __ldg(a.item_off + (size_t)k * (a.n_inst + 1) + inst + 1) - i0;
    const uint32_t* items = list[k].items + i0;
    if (op == PH_COLLIDE) {
      const int first = tile * a.tile_blocks;
      const int nblk = min(a.tile_blocks, ni - first);
      // a cell per thread where two would leave half of the warps without work
      // (the batch above, CTAs of 256 with tiles of one block: 5.1 ms against
      // 3.3 with this and the budget)
      if (row_cells<D, Q, T>() == 1 || 2 * nblk * 32 <= THREADS)
        persist_collide<D, Q, T, THREADS, 1>(d, items + first, nblk, level, win, s_nb);
      else
        persist_collide<D, Q, T, THREADS, row_cells<D, Q, T>()>(d, items + first, nblk, level, win,
                                                             s_nb);
    } else if (op == PH_INTERP) {
      persist_interp<D, Q, T, THREADS>(d, items, ni, tile, level, win, wch, sF, s_rows);
    } else {
      persist_average<D, Q, T, THREADS>(d, items, ni, tile, level, win, wch, sF, s_rows);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      atomicAdd(a.done + (size_t)k * a.n_inst + inst, 1u);
    }
  }
}

template <int D, int Q, class T, int THREADS>
constexpr size_t persist_smem_bytes() {
  return sizeof(typename Store<T>::R) * THREADS * Q +
         sizeof(int32_t) * (THREADS / Block<D>::M) * (1 + Block<D>::NC) * Nbr<D>::K;
}

// ================================================ whole blocks, read only
// The kernels below read the pre-collision populations of whole blocks by
// x-rows (gather_row): a warp per block in 3D (FP64: two, a cell per thread, see
// row_cells), two blocks per warp in 2D.
template <int D, class T, int V_ = D == 2 || sizeof(T) == 8 ? 1 : 2>
struct BlockRows {
  static constexpr int V = V_;
  static constexpr int TPB = Block<D>::M / V;
  static constexpr int LPR = TPB < 32 ? TPB : 32;   // lanes that share a staged row
  static constexpr int NCODE = D == 2 ? 9 : 27;
  static constexpr int BPC = 128 / TPB;     // blocks of a CTA of 128 threads
  struct Shared {
    int32_t nb[128 / LPR][NCODE];
    uint64_t sm[128 / LPR][NCODE];
  };
};

// CTAs of 128 threads per SM the register budget of the criterion and of the
// export of moments is set for.  FP64, criterion and its synchronisation: 24^3
// cavity, one level, D3Q27 36.5 us (41.9 with two cells per thread), 96^3 box,
// D3Q19 167 us (173 with two), 170 with 768 threads for 640; 1024^2 box 108 us
// with 1536 threads, 109 with 1280, 114 with 1024.
template <int Q, class T>
constexpr int read_min_ctas() {
  return (Q == 9 ? 1536 : (sizeof(T) == 8 ? (Q == 27 ? 512 : 640) : (Q == 27 ? 768 : 1024))) / 128;
}

// Populations of the V cells of this thread of block b.
template <int D, int Q, class T, int V>
__device__ __forceinline__ void read_rows(Vec<T, V> (&g)[Q], const T* f, int b,
                                          const RowPos<D, V>& pos,
                                          typename BlockRows<D, T, V>::Shared& s,
                                          const int32_t* __restrict__ nbr,
                                          const uint64_t* __restrict__ solidmask) {
  using B = BlockRows<D, T, V>;
  const int row = threadIdx.x / B::LPR;
  const int flags = stage_block<D, B::LPR, true>(s.nb[row], s.sm[row], b, threadIdx.x % B::LPR,
                                                 block_lanes<B::LPR>(), nbr, solidmask, nullptr);
  gather_row<D, Q, T, V, true, true, false>(g, f, b, pos, s.nb[row], s.sm[row], flags & BF_SOLID);
}

// The TPB threads of a block meet (`slot`: of the CTA).
template <int TPB>
__device__ __forceinline__ void block_sync(int slot) {
  if constexpr (TPB > 32) asm volatile("bar.sync %0, %1;" ::"r"(slot + 1), "n"(TPB) : "memory");
  else __syncwarp(block_lanes<TPB>());
}

// Block-local first-order difference of a value along AXIS (forward, backward
// at the last cell) for the V cells of a thread; val: the thread's values.  The
// neighbour's value comes by a shuffle, or, in blocks of more than a warp, from
// `all`, the values of the block in shared memory.
template <int D, int V, int AXIS, class R>
__device__ __forceinline__ void block_diff(R (&out)[V], const R (&val)[V],
                                           const RowPos<D, V>& pos, unsigned lanes, const R* all) {
  const int lane = threadIdx.x & 31;
  // a - b or b - a, one subtraction (an FP64 one is a 64-cycle instruction)
  auto minus = [](bool plain, R a, R b) { return (plain ? a : b) - (plain ? b : a); };
  if constexpr (Block<D>::M / V > 32) {
    static_assert(V == 1, "a cell per thread");
    constexpr int STEP = AXIS == 0 ? 1 : (AXIS == 1 ? 4 : 16);
    const int at = AXIS == 0 ? pos.i0 : (AXIS == 1 ? Block<D>::cj(pos.l0) : Block<D>::ck(pos.l0));
    const R o = all[pos.l0 + (at == 3 ? -STEP : STEP)];
    out[0] = minus(at == 3, val[0], o);
  } else if constexpr (AXIS == 0) {
    if constexpr (V == 2) {
      const R next = __shfl_sync(lanes, val[0], pos.i0 == 0 ? lane + 1 : lane);
      out[0] = val[1] - val[0];
      out[1] = pos.i0 == 0 ? next - val[1] : out[0];
    } else {
      const bool last = pos.i0 == 3;
      const R o = __shfl_sync(lanes, val[0], last ? lane - 1 : lane + 1);
      out[0] = minus(last, val[0], o);
    }
  } else {
    constexpr int STEP = (AXIS == 1 ? 4 : 16) / V;    // lanes between cells along the axis
    const bool last = (AXIS == 1 ? Block<D>::cj(pos.l0) : Block<D>::ck(pos.l0)) == 3;
#pragma unroll
    for (int i = 0; i < V; ++i) {
      const R o = __shfl_sync(lanes, val[i], last ? lane - STEP : lane + STEP);
      out[i] = minus(last, val[i], o);
    }
  }
}

// ================================================================ criterion
// Vorticity magnitude from block-local first-order differences (forward, and
// backward at the last cell), block maximum of |w|^2, desired level of
// Algorithm 3 (eps < T evaluated as |w|^2 < 4^T), mark: +1 for a leaf with
// L_des > L, -1 for a REFINED block with L_des <= L.
template <int D, int Q, class T>
__global__ void __launch_bounds__(128, (read_min_ctas<Q, T>()))
    k_criterion(const int32_t* __restrict__ list, int n, const T* __restrict__ f, const int32_t* __restrict__ nbr, const uint64_t* __restrict__ solidmask,
                const int32_t* __restrict__ status, int level, int lmax, double inv_dx,
                int n_start, int n_inc, int8_t* __restrict__ marks, double* __restrict__ w2out) {
  using S = Store<T>;
  using R = typename S::R;
  using B = BlockRows<D, T>;
  constexpr int V = B::V;
  constexpr bool WIDE = B::TPB > 32;         // a block takes two warps
  __shared__ typename B::Shared sh;
  __shared__ R su[WIDE ? B::BPC : 1][D][WIDE ? Block<D>::M : 1];
  __shared__ R sw[128 / 32];
  const int slot = threadIdx.x / B::TPB, t = threadIdx.x % B::TPB;
  const int bi = blockIdx.x * B::BPC + slot;
  if (bi >= n) return;                       // (the same for the threads of a block)
  const unsigned lanes = block_lanes<B::LPR>();
  const int b = __ldg(list + bi);
  const RowPos<D, V> pos(t);
  Vec<T, V> g[Q];
  read_rows<D, Q, T, V>(g, f, b, pos, sh, nbr, solidmask);
  R u[3][V];
  static_for<0, V>([&](auto I) {
    R fl[Q];
    static_for<0, Q>([&](auto P) { fl[P] = S::template load<D, Q, P>(g[P].v[I]); });
    R rho;
    moments<D, Q>(fl, rho, u[0][I], u[1][I], u[2][I]);
  });
  const R* all[3] = {};
  if constexpr (WIDE) {
    static_for<0, D>([&](auto C) {
      su[slot][C][pos.l0] = u[C][0];
      all[C] = su[slot][C];
    });
    block_sync<B::TPB>(slot);
  }
  const R s = R(inv_dx);
  R a[V], c[V], w2[V];
  block_diff<D, V, 0>(a, u[1], pos, lanes, all[1]);
  block_diff<D, V, 1>(c, u[0], pos, lanes, all[0]);
#pragma unroll
  for (int i = 0; i < V; ++i) w2[i] = (a[i] - c[i]) * s;
  if constexpr (D == 2) {
#pragma unroll
    for (int i = 0; i < V; ++i) w2[i] = w2[i] * w2[i];
  } else {
    R wx[V], wy[V];
    block_diff<D, V, 1>(a, u[2], pos, lanes, all[2]);
    block_diff<D, V, 2>(c, u[1], pos, lanes, all[1]);
#pragma unroll
    for (int i = 0; i < V; ++i) wx[i] = (a[i] - c[i]) * s;
    block_diff<D, V, 2>(a, u[0], pos, lanes, all[0]);
    block_diff<D, V, 0>(c, u[2], pos, lanes, all[2]);
#pragma unroll
    for (int i = 0; i < V; ++i) {
      wy[i] = (a[i] - c[i]) * s;
      w2[i] = wx[i] * wx[i] + wy[i] * wy[i] + w2[i] * w2[i];
    }
  }
  R top = w2[0];
#pragma unroll
  for (int i = 1; i < V; ++i) top = max(top, w2[i]);
#pragma unroll
  for (int off = B::LPR / 2; off > 0; off >>= 1)
    top = max(top, __shfl_xor_sync(lanes, top, off));
  if constexpr (WIDE) {
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) sw[warp] = top;
    block_sync<B::TPB>(slot);
    if (t == 0) top = max(top, sw[warp + 1]);
  }
  if (t != 0) return;
  const double w2d = (double)top;
  int ldes = lmax - 1;
  for (int p = 1; p < lmax; ++p) {
    const int T_ = n_start - p * n_inc;
    if (T_ > 1 || w2d < ldexp(1.0, 2 * T_)) ldes = (lmax - 1) - p;
  }
  const int st = status[b];
  int8_t m = 0;
  if (st == ST_UNREFINED && ldes > level) m = 1;
  else if (st == ST_REFINED && ldes <= level) m = -1;
  marks[b] = m;
  if (w2out) w2out[b] = w2d;
}


// ============================================ block summaries (27 features)
// Inputs of the learned refinement proposal, per 4^3 block after the level
// synchronisation: for the 9 velocity-gradient components G_ab = du_a/dx_b
// (block-local first-order differences as in the criterion, physical units)
// their mean and max |.|; mean and max-min of rho; mean u_x, u_y, u_z and
// max |u|; mean and max |w|; level / L_max.  Gradient and vorticity entries
// are compressed as sign(x) log(1 + |x|); density entries are (rho - 1) * 100
// and (max - min) * 100; velocities are scaled by 20.
constexpr int N_FEATURES = 27;

__device__ __forceinline__ float squash(float x) { return copysignf(log1pf(fabsf(x)), x); }

// A warp per block: the cells' values go to shared memory, 16 rows of 64, and
// 16 lanes walk a row each.  The sums are taken in cell order: the proposal
// compares a function of them with a threshold, so that the marks hang on
// their last bits.
template <int Q, class T>
__global__ void __launch_bounds__(128, (average_min_ctas<Q, T, 128>()))
    k_features(const int32_t* __restrict__ list, int n, const T* __restrict__ f, const int32_t* __restrict__ nbr, const uint64_t* __restrict__ solidmask,
               int level, int lmax, double inv_dx, float* __restrict__ out) {
  using S = Store<T>;
  using R = typename S::R;
  using B = BlockRows<3, T, 2>;
  // (rows of 68 words: 16-byte reads of eight rows touch every bank once)
  __shared__ __align__(16) float s_row[B::BPC][16][68];
  __shared__ typename B::Shared sh;
  const int slot = threadIdx.x / 32, lane = threadIdx.x & 31;
  const int bi = blockIdx.x * B::BPC + slot;
  if (bi >= n) return;
  const int b = __ldg(list + bi);
  const RowPos<3, 2> pos(lane);
  Vec<T, 2> g[Q];
  read_rows<3, Q, T, 2>(g, f, b, pos, sh, nbr, solidmask);
  float u[3][2], rho[2];
  static_for<0, 2>([&](auto I) {
    R fl[Q];
    static_for<0, Q>([&](auto P) { fl[P] = S::template load<3, Q, P>(g[P].v[I]); });
    R r, ux, uy, uz;
    moments<3, Q>(fl, r, ux, uy, uz);
    rho[I] = (float)r;
    u[0][I] = (float)ux;
    u[1][I] = (float)uy;
    u[2][I] = (float)uz;
  });
  const float s = (float)inv_dx;
  float G[9][2];
  static_for<0, 3>([&](auto C) {
    block_diff<3, 2, 0>(G[3 * C], u[C], pos, 0xffffffffu, (const float*)nullptr);
    block_diff<3, 2, 1>(G[3 * C + 1], u[C], pos, 0xffffffffu, (const float*)nullptr);
    block_diff<3, 2, 2>(G[3 * C + 2], u[C], pos, 0xffffffffu, (const float*)nullptr);
  });
  // rows: 0..8 G, 9 rho, 10..12 u, 13 |u|, 14 |w|, 15 -rho
  float (*row)[68] = s_row[slot];
  auto put = [&](int q, float a, float c) {
    *reinterpret_cast<float2*>(&row[q][pos.l0]) = make_float2(a, c);
  };
  float speed[2], om[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
#pragma unroll
    for (int q = 0; q < 9; ++q) G[q][i] *= s;
    const float wx = G[7][i] - G[5][i], wy = G[2][i] - G[6][i], wz = G[3][i] - G[1][i];
    speed[i] = sqrtf(u[0][i] * u[0][i] + u[1][i] * u[1][i] + u[2][i] * u[2][i]);
    om[i] = sqrtf(wx * wx + wy * wy + wz * wz);
  }
#pragma unroll
  for (int q = 0; q < 9; ++q) put(q, G[q][0], G[q][1]);
  put(9, rho[0], rho[1]);
#pragma unroll
  for (int a = 0; a < 3; ++a) put(10 + a, u[a][0], u[a][1]);
  put(13, speed[0], speed[1]);
  put(14, om[0], om[1]);
  put(15, -rho[0], -rho[1]);
  __syncwarp();
  // largest magnitude, of rho and -rho the largest value
  const int q = lane & 15;
  const bool is_rho = q == 9 || q == 15;
  float sum = 0.f, top = is_rho ? row[q][0] : 0.f;
#pragma unroll 4
  for (int c = 0; c < 64; c += 4) {
    const float4 x = *reinterpret_cast<const float4*>(&row[q][c]);
    sum += x.x;
    sum += x.y;
    sum += x.z;
    sum += x.w;
    top = fmaxf(top, is_rho ? x.x : fabsf(x.x));
    top = fmaxf(top, is_rho ? x.y : fabsf(x.y));
    top = fmaxf(top, is_rho ? x.z : fabsf(x.z));
    top = fmaxf(top, is_rho ? x.w : fabsf(x.w));
  }
  const float minus_min = __shfl_sync(0xffffffffu, top, 15);
  const float mean = sum / 64.f;
  float* o = out + (size_t)b * N_FEATURES;
  if (lane < 9) {
    o[lane] = squash(mean);
    o[9 + lane] = squash(top);
  } else if (lane == 9) {
    o[18] = (mean - 1.f) * 100.f;
    o[19] = (top + minus_min) * 100.f;
  } else if (lane < 13) {
    o[20 + (lane - 10)] = mean * 20.f;
  } else if (lane == 13) {
    o[23] = top * 20.f;
  } else if (lane == 14) {
    o[24] = squash(mean);
    o[25] = squash(top);
  } else if (lane == 15) {
    o[26] = (float)level / (float)lmax;
  }
}

// ============================================================ exports/imports
// `wide`: the destination is aligned for vector stores (the caller's pointer
// need not be).
template <int V>
struct Doubles {
  double v[V];
};
template <int V>
__device__ __forceinline__ void store_doubles(double* at, const Doubles<V>& x, bool wide) {
  if constexpr (V == 2) {
    if (wide) {
      *reinterpret_cast<double2*>(at) = make_double2(x.v[0], x.v[1]);
      return;
    }
  }
#pragma unroll
  for (int c = 0; c < V; ++c) at[c] = x.v[c];
}

// Cells per thread of the export: one; a thread holds its Q values before it
// stores them, and with two the 126 to 178 registers of D3Q27 left too few
// threads to keep the stores going (130,000 blocks: 296 us with two, 224 with
// one in FP32, 338 / 253 in FP64).  D3Q19 in FP32 is faster with two (163 / 171).
template <int D, int Q, class T>
constexpr int export_cells() {
  return D == 3 && Q == 19 && sizeof(T) == 4 ? 2 : 1;
}
template <int D, int Q, class T>
__global__ void __launch_bounds__(128, D == 2 || export_cells<D, Q, T>() == 2 ? 0 : (sizeof(T) == 8 ? 6 : 8))
    k_export_f(int64_t cap, int64_t b0, int64_t nb, const T* __restrict__ fa,
               const T* __restrict__ fb, unsigned cur, const int32_t* __restrict__ level,
               const int32_t* __restrict__ nbr, const uint64_t* __restrict__ solidmask,
               double* __restrict__ out, bool wide) {
  using B = BlockRows<D, T, export_cells<D, Q, T>()>;
  constexpr int M = Block<D>::M, V = B::V;
  __shared__ typename B::Shared sh;
  const int slot = threadIdx.x / B::TPB, t = threadIdx.x % B::TPB;
  const int64_t i = (int64_t)blockIdx.x * B::BPC + slot;
  if (i >= nb) return;
  const int b = (int)(b0 + i);
  const int L = __ldg(level + b);
  const RowPos<D, V> pos(t);
  double* o = out + i * M + pos.l0;
  const size_t plane = (size_t)nb * M;
  if (L < 0) {
    for (int p = 0; p < Q; ++p) store_doubles<V>(o + p * plane, Doubles<V>{}, wide);
    return;
  }
  Vec<T, V> g[Q];
  read_rows<D, Q, T, V>(g, ((cur >> L) & 1u) ? fb : fa, b, pos, sh, nbr, solidmask);
  static_for<0, Q>([&](auto P) {
    Doubles<V> x;
#pragma unroll
    for (int c = 0; c < V; ++c) x.v[c] = (double)Store<T>::template load<D, Q, P>(g[P].v[c]);
    store_doubles<V>(o + P * plane, x, wide);
  });
}

template <int D, int Q, class T>
__global__ void k_import_f(int64_t cap, int64_t b0, int64_t nb, T* __restrict__ fa,
                           T* __restrict__ fb, unsigned cur, const int32_t* __restrict__ level,
                           const int32_t* __restrict__ nbr, const uint64_t* __restrict__ solidmask,
                           const double* __restrict__ in) {
  using R = typename Store<T>::R;
  constexpr int M = Block<D>::M;
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= nb * M) return;
  const int64_t b = b0 + g / M;
  const int l = (int)(g % M);
  const int L = level[b];
  if (L < 0) return;
  T* f = ((cur >> L) & 1u) ? fb : fa;
  R v[Q];
  static_for<0, Q>([&](auto P) { v[P] = (R)in[(size_t)P * nb * M + g]; });
  scatter_cell<D, Q, T, true>(v, f, (int)b, l, nbr + (size_t)b * NBR_STRIDE, solidmask);
}

template <int D, int Q, class T>
__global__ void __launch_bounds__(128, (read_min_ctas<Q, T>()))
    k_export_rho_u(int64_t cap, int64_t b0, int64_t nb, const T* __restrict__ fa,
                   const T* __restrict__ fb, unsigned cur, const int32_t* __restrict__ level,
                   const int32_t* __restrict__ nbr, const uint64_t* __restrict__ solidmask,
                   double* __restrict__ out, bool wide) {
  using S = Store<T>;
  using R = typename S::R;
  using B = BlockRows<D, T>;
  constexpr int M = Block<D>::M, V = B::V;
  __shared__ typename B::Shared sh;
  const int slot = threadIdx.x / B::TPB, t = threadIdx.x % B::TPB;
  const int64_t i = (int64_t)blockIdx.x * B::BPC + slot;
  if (i >= nb) return;
  const int b = (int)(b0 + i);
  const int L = __ldg(level + b);
  const RowPos<D, V> pos(t);
  double v[V][1 + D] = {};
  if (L >= 0) {
    Vec<T, V> g[Q];
    read_rows<D, Q, T, V>(g, ((cur >> L) & 1u) ? fb : fa, b, pos, sh, nbr, solidmask);
    static_for<0, V>([&](auto I) {
      R fl[Q];
      static_for<0, Q>([&](auto P) { fl[P] = S::template load<D, Q, P>(g[P].v[I]); });
      R rho, ux, uy, uz;
      moments<D, Q>(fl, rho, ux, uy, uz);
      v[I][0] = rho;
      v[I][1] = ux;
      v[I][2] = uy;
      if constexpr (D == 3) v[I][3] = uz;
    });
  }
  double* o = out + (size_t)(i * M + pos.l0) * (1 + D);
#pragma unroll
  for (int c = 0; c < V; ++c) {
    if (D == 3 && wide) {
      asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(o + 4 * c), "d"(v[c][0]),
                   "d"(v[c][1]), "d"(v[c][2]), "d"(v[c][D])
                   : "memory");
    } else {
#pragma unroll
      for (int a = 0; a <= D; ++a) o[(1 + D) * c + a] = v[c][a];
    }
  }
}

// The rest state (f = w_p in every slot; the gather of it is w_p everywhere).
template <int D, int Q, class T>
__global__ void k_init_rest(int64_t cap, T* __restrict__ f) {
  using R = typename Store<T>::R;
  constexpr int M = Block<D>::M;
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= cap * M) return;
  const size_t own = (size_t)(g / M) * (Q * M) + (size_t)(g % M);
  static_for<0, Q>([&](auto P) {
    constexpr double wp = VS<D, Q>::w[P];
    f[own + (size_t)P * M] = Store<T>::template save<D, Q, P>(R(wp));
  });
}

// The rest state in the own slots of the solid cells of the listed blocks.  No
// step writes these slots, and an ID may have belonged to a fluid block before,
// so they are set in both buffers when a block is made: here in the one that
// the interpolation of new children does not fill.
template <int D, int Q, class T>
__global__ void k_solid_rest(const int32_t* __restrict__ list, int n,
                             const uint64_t* __restrict__ solidmask, T* __restrict__ f) {
  using R = typename Store<T>::R;
  constexpr int M = Block<D>::M;
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= (int64_t)n * M) return;
  const int b = __ldg(list + g / M), l = (int)(g % M);
  if (!((__ldg(solidmask + b) >> l) & 1ull)) return;
  const size_t own = (size_t)b * (Q * M) + l;
  static_for<0, Q>([&](auto P) {
    constexpr double wp = VS<D, Q>::w[P];
    f[own + (size_t)P * M] = Store<T>::template save<D, Q, P>(R(wp));
  });
}

// Adaptation: for every cell x of a child about to be removed and every link
// p whose target y = x + c_p lies in a same-level block that stays, the value
// stored in x's slot p is y's pre-collision f_p; once the block is gone y
// reads it from its own opposite slot, so it is moved there.  One thread per
// (removed child, cell).
template <int D, int Q, class T>
__global__ void k_coarsen_fixup(const int32_t* __restrict__ list, int n,
                                const int32_t* __restrict__ child0,
                                const int32_t* __restrict__ parent,
                                const int8_t* __restrict__ marks,
                                const int32_t* __restrict__ nbr,
                                const uint64_t* __restrict__ solidmask,
                                const int32_t* __restrict__ level, T* __restrict__ fa,
                                T* __restrict__ fb, unsigned cur) {
  constexpr int M = Block<D>::M, NC = Block<D>::NC;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)n * NC * M) return;
  const int l = (int)(t % M);
  const int64_t it = t / M;
  const int x = child0[list[it / NC]] + (int)(it % NC);
  if (solidmask && ((solidmask[x] >> l) & 1ull)) return;
  T* g = ((cur >> level[x]) & 1u) ? fb : fa;
  const int32_t* row = nbr + (size_t)x * NBR_STRIDE;
  static_for<1, Q>([&](auto P) {
    constexpr int p = P;
    constexpr int pb = VS<D, Q>::opp[p];
    const int e = link_entry<D, Q, p>(g_tgt_k<D, Q>, l);
    const int k = e & 31, tl = e >> 5;
    if (k == 0) return;
    const int y = row[k];
    if (y < 0) return;
    const int py = parent[y];
    if (py >= 0 && marks[py] == -1) return;       // removed as well
    if (solidmask && ((solidmask[y] >> tl) & 1ull)) return;
    g[(size_t)y * (Q * M) + (size_t)pb * M + tl] = g[(size_t)x * (Q * M) + (size_t)p * M + l];
  });
}

// ------------------------------------------------------- block reductions
template <int NV>
__device__ __forceinline__ void block_sum_store(double (&v)[NV], double* out) {
  __shared__ double sred[NV][32];
#pragma unroll
  for (int a = 0; a < NV; ++a)
    for (int off = 16; off > 0; off >>= 1) v[a] += __shfl_xor_sync(0xffffffffu, v[a], off);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0)
    for (int a = 0; a < NV; ++a) sred[a][warp] = v[a];
  __syncthreads();
  if (warp == 0) {
    const int nw = blockDim.x >> 5;
    for (int a = 0; a < NV; ++a) {
      double x = lane < nw ? sred[a][lane] : 0.0;
      for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
      if (lane == 0) out[(size_t)blockIdx.x * NV + a] = x;
    }
  }
}

// FP64 audit of mass and momentum over leaf cells (grid-fixed grid).
template <int D, int Q, class T>
__global__ void __launch_bounds__(256)
    k_mass_partial(int64_t cap, const T* __restrict__ fa, const T* __restrict__ fb, unsigned cur,
                   const int32_t* __restrict__ level, const int32_t* __restrict__ status,
                   const int32_t* __restrict__ nbr, const uint64_t* __restrict__ solidmask,
                   double* __restrict__ partial) {
  using R = typename Store<T>::R;
  constexpr int M = Block<D>::M;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < cap * M;
       g += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = g / M;
    if (status[b] != ST_UNREFINED) continue;
    const int L = level[b];
    const T* f = ((cur >> L) & 1u) ? fb : fa;
    R fl[Q];
    gather_cell<D, Q, T, true>(fl, f, (int)b, (int)(g % M),
                               nbr + (size_t)b * NBR_STRIDE, solidmask);
    double r = 0, jx = 0, jy = 0, jz = 0;
    static_for<0, Q>([&](auto P) {
      const double v = (double)fl[P];
      constexpr int cx = VS<D, Q>::cx[P], cy = VS<D, Q>::cy[P], cz = VS<D, Q>::cz[P];
      r += v;
      jx += cx * v;
      jy += cy * v;
      jz += cz * v;
    });
    const double vol = ldexp(1.0, -D * L);
    acc[0] += r * vol;
    acc[1] += jx * vol;
    acc[2] += jy * vol;
    acc[3] += jz * vol;
  }
  block_sum_store<4>(acc, partial);
}

// Momentum-exchange force: F = 2 dx^(D-1) sum over fluid cells and links p
// whose target x + c_p is solid of f*_p c_p (Section 5.3, with dt = dx per
// link), f* recomputed by BGK from the stored state.  A warp per block: its
// lanes look at the solid cells of the block's neighbours first, and only
// the few blocks that touch the solid read populations (gathering every cell
// of every leaf took 350 us per level on 85,000 blocks).
template <int D, int Q, class T>
__global__ void __launch_bounds__(256)
    k_force_partial(const int32_t* __restrict__ list, int n, const T* __restrict__ f,
                    const int32_t* __restrict__ nbr,
                    const int32_t* __restrict__ status, const uint64_t* __restrict__ solidmask,
                    double omega, double dx, double* __restrict__ partial) {
  using V = VS<D, Q>;
  using S = Store<T>;
  using R = typename S::R;
  constexpr int M = Block<D>::M;
  constexpr int NCODE = D == 2 ? 9 : 27, CENTER = D == 2 ? 4 : 13;
  __shared__ uint64_t s_sm[8][NCODE];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double acc[3] = {0.0, 0.0, 0.0};
  for (int bi = blockIdx.x * 8 + warp; bi < n; bi += gridDim.x * 8) {
    const int b = __ldg(list + bi);
    uint64_t m = 0ull;
    if (lane < NCODE) {
      const int v = __ldg(nbr + (size_t)b * NBR_STRIDE + geo_to_k<D>(lane));
      if (v >= 0) m = __ldg(solidmask + v);
    }
    if (!__any_sync(0xffffffffu, m != 0ull) || __ldg(status + b) != ST_UNREFINED) continue;
    __syncwarp();
    if (lane < NCODE) s_sm[warp][lane] = m;
    __syncwarp();
    for (int l = lane; l < M; l += 32) {
      if ((s_sm[warp][CENTER] >> l) & 1ull) continue;
      uint32_t hit = 0u;               // links into the solid
      static_for<1, Q>([&](auto P) {
        const int e = link_entry<D, Q, P>(g_tgt_geo<D, Q>, l);
        if ((s_sm[warp][e & 31] >> (e >> 5)) & 1ull) hit |= 1u << P;
      });
      if (!hit) continue;
      R fl[Q];
      gather_cell<D, Q, T, true>(fl, f, b, l, nbr + (size_t)b * NBR_STRIDE, solidmask);
      R rho, ux, uy, uz;
      moments<D, Q>(fl, rho, ux, uy, uz);
      const R usq15 = R(1.5) * (ux * ux + uy * uy + uz * uz);
      static_for<1, Q>([&](auto P) {
        constexpr int p = P;
        if (!((hit >> p) & 1u)) return;
        const R fs = fl[p] + R(omega) * (feq<D, Q, p>(rho, ux, uy, uz, usq15) - fl[p]);
        constexpr int cx = V::cx[p], cy = V::cy[p], cz = V::cz[p];
        acc[0] += (double)fs * cx;
        acc[1] += (double)fs * cy;
        acc[2] += (double)fs * cz;
      });
    }
  }
  const double scale = 2.0 * pow(dx, (double)(D - 1));
  for (int a = 0; a < 3; ++a) acc[a] *= scale;
  block_sum_store<3>(acc, partial);
}

// =============================================================== launchers
inline int grid_for(int64_t n, int per) { return (int)((n + per - 1) / per); }

// Launch a kernel that calls chain_start / chain_wait (lattice.cuh).
template <class... P, class... A>
inline void launch_chained(void (*kernel)(P...), bool chained, int grid, int threads,
                           cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.stream = s;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = chained ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

template <int D, int Q, class T>
struct Launch {
  static constexpr int M = Block<D>::M;
  static inline int sm_count = 152;
  // cells per CTA.  2D meshes are small: CTAs of one or two warps spread them
  // over the SMs (an SM executes one FP64 warp instruction per 19 cycles; the
  // 64^2 FP64 cavity took 2.20 ms with 256 cells per CTA, 1.66 with 32)
  static constexpr int kAutoCells = D == 3 ? (row_cells<D, Q, T>() == 1 ? 64 : 256)
                                           : (sizeof(T) == 8 ? 32 : 64);
  // ... 2D FP32 launches above this many cells: CTAs of 128 (one level, us per
  // step with 64 / 128 cells: 512^2 8.3 / 8.3, 768^2 12.4 / 10.4, 1024^2 20.6 /
  // 16.6, 2048^2 71.8 / 63.6, 3072^2 153.8 / 134.9)
  static constexpr int64_t kWideCells = int64_t(1) << 18;
  // ... D3Q27 FP32 launches of more blocks than this without solid cells: two
  // cells per thread, 256 per CTA (192^3 box: 244 us per step, 261 with one; 64^3
  // cavity with an extra level, launches of up to 13,000 blocks: 102 and 97)
  static constexpr int kLargeQ27 = 1 << 14;

  static int setup() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return -1;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
    sm_count = sms;
    return 0;
  }

  // CELLS cells per CTA (at least the blocks of a warp); XCHG:
  // instantiated for launches with exchanging parents as well
  template <bool SOLID, int CELLS, bool XCHG, int V = row_cells<D, Q, T>(), bool DENSE = false>
  static void one_pass(cudaStream_t s, const int32_t* list, int n, const void* fin, void* fout,
                       const int32_t* nbr, const uint64_t* sm, const StepParams& prm,
                       const uint64_t* gm, const Exchange* xchg) {
    constexpr int THREADS = row_threads<V>(CELLS);
    constexpr int MIN = row_min_ctas<Q, T, V, THREADS, DENSE>();
    const T* in = (const T*)fin;
    T* out = (T*)fout;
    Exchange ex{};
    if (xchg) ex = *xchg;
    auto launch = [&](auto ghost, auto parents) {
      constexpr bool G = decltype(ghost)::value, X = decltype(parents)::value;
      const int grid = grid_for(n, THREADS * V / M);
      launch_chained(k_collide_stream<D, Q, T, SOLID, V, THREADS, MIN, G, X>, prm.chained, grid,
                     THREADS, s, list, n, in, out, nbr, sm, prm, gm, ex);
    };
    if constexpr (XCHG) {
      if (gm && xchg) return launch(std::true_type{}, std::true_type{});
      if (xchg) return launch(std::false_type{}, std::true_type{});
    }
    if (gm) launch(std::true_type{}, std::false_type{});
    else launch(std::false_type{}, std::false_type{});
  }

  template <bool SOLID>
  static void collide_stream_t(cudaStream_t s, const int32_t* list, int n, const void* fin,
                               void* fout, const int32_t* nbr, const uint64_t* sm,
                               const StepParams& prm, const uint64_t* gm, const Exchange* x) {
    // kernel_variant: 1 / 2 / 3 / 4: CTAs of 512 / 256 / 128 / 64 cells (8 /
    // 4 / 2 / 1 blocks of 4^3 cells; never less than a warp); 5: 128 cells
    // with 128 more resident threads per SM (tighter register budget); 0
    // (auto), every other value, and launches with exchanging parents: kAutoCells
    switch (x ? 0 : prm.variant) {
      case 1: one_pass<SOLID, 512, false>(s, list, n, fin, fout, nbr, sm, prm, gm, nullptr); break;
      case 2: one_pass<SOLID, 256, false>(s, list, n, fin, fout, nbr, sm, prm, gm, nullptr); break;
      case 3: one_pass<SOLID, 128, false>(s, list, n, fin, fout, nbr, sm, prm, gm, nullptr); break;
      case 4: one_pass<SOLID, 64, false>(s, list, n, fin, fout, nbr, sm, prm, gm, nullptr); break;
      case 5:
        one_pass<SOLID, 128, false, row_cells<D, Q, T>(), true>(s, list, n, fin, fout, nbr, sm, prm, gm, nullptr);
        break;
      default:
        if constexpr (D == 2 && sizeof(T) == 4) {
          if ((int64_t)n * M > kWideCells) {
            one_pass<SOLID, 128, true>(s, list, n, fin, fout, nbr, sm, prm, gm, x);
            break;
          }
        }
        if constexpr (Q == 27 && sizeof(T) == 4 && !SOLID) {
          if (n > kLargeQ27) {
            one_pass<SOLID, 256, true, 2>(s, list, n, fin, fout, nbr, sm, prm, gm, x);
            break;
          }
        }
        one_pass<SOLID, kAutoCells, true>(s, list, n, fin, fout, nbr, sm, prm, gm, x);
    }
  }

  static void collide_stream(cudaStream_t s, const int32_t* list, int n, const void* fin,
                             void* fout, const int32_t* nbr, const uint64_t* sm,
                             const StepParams& prm, bool solid, const uint64_t* gm,
                             const Exchange* x) {
    if (n <= 0) return;
    if (solid) collide_stream_t<true>(s, list, n, fin, fout, nbr, sm, prm, gm, x);
    else collide_stream_t<false>(s, list, n, fin, fout, nbr, nullptr, prm, gm, x);
  }

  static void interp(cudaStream_t s, const int32_t* list, int n, const void* fpar, void* fch,
                     const int32_t* child0, const uint64_t* nm,
                     const int32_t* nbr, const uint64_t* sm, const int32_t* parent,
                     const int8_t* marks, double ratio, int mode_all, bool solid) {
    if (n <= 0) return;
    // mode bit 0: every cell (new children), else ghost cells; bit 1: cubic;
    // bit 2: direct writes into the children's own slots
    const int all = mode_all & 5;
    if (mode_all & 2) {
      const int grid = grid_for(n, 64 / M);
      // never a dependent of the launch before: its CTAs would wait with their
      // shared memory in hand (2D FP64 prism, 4 levels, 8 coarse steps: 4.9 ms
      // chained, 3.15 not)
      if (solid)
        k_interp_cubic<D, Q, T, true><<<grid, 64, 0, s>>>(list, n, (const T*)fpar, (T*)fch,
                                                         child0, nm, nbr, sm, parent,
                                                         marks, ratio, all);
      else
        k_interp_cubic<D, Q, T, false><<<grid, 64, 0, s>>>(list, n, (const T*)fpar, (T*)fch,
                                                          child0, nm, nbr, nullptr,
                                                          parent, marks, ratio, all);
      return;
    }
    const int grid = grid_for(n, 128 / M);
    if (solid)
      k_interp<D, Q, T, true><<<grid, 128, 0, s>>>(list, n, (const T*)fpar, (T*)fch, child0, nm, nbr, sm, parent, marks, ratio, all);
    else
      k_interp<D, Q, T, false><<<grid, 128, 0, s>>>(list, n, (const T*)fpar, (T*)fch, child0, nm, nbr, nullptr, parent, marks, ratio,
                                                   all);
  }
  static void average(cudaStream_t s, const int32_t* list, int n, bool by_parent, void* fpar,
                      const void* fch, const int32_t* child0,
                      const int32_t* parent, const uint64_t* nm,
                      const int32_t* nbr, const uint64_t* sm, double ratio, bool solid,
                      bool chained) {
    if (n <= 0) return;
    constexpr int CPC = 128 / (M / (D == 3 ? 2 : 1));
    const int64_t items = by_parent ? (int64_t)n * Block<D>::NC : (int64_t)n;
    const int grid = (int)((items + CPC - 1) / CPC);
    launch_chained(solid ? k_average<D, Q, T, true> : k_average<D, Q, T, false>, chained, grid,
                   128, s, list, items, by_parent, (T*)fpar, (const T*)fch, child0, parent, nm,
                   nbr, solid ? sm : nullptr, ratio);
  }
  static void criterion(cudaStream_t s, const int32_t* list, int n, const void* f, const int32_t* nbr, const uint64_t* sm, const int32_t* status, int level,
                        int lmax, double inv_dx, int ns, int ni, int8_t* marks, double* w2out) {
    if (n <= 0) return;
    k_criterion<D, Q, T><<<grid_for(n, BlockRows<D, T>::BPC), 128, 0, s>>>(
        list, n, (const T*)f, nbr, sm, status, level, lmax, inv_dx, ns, ni, marks, w2out);
  }
  static void export_f(cudaStream_t s, int64_t cap, int64_t b0, int64_t nb, const void* fa,
                       const void* fb, unsigned cur, const int32_t* level, const int32_t* nbr,
                       const uint64_t* sm, double* out) {
    k_export_f<D, Q, T><<<grid_for(nb, BlockRows<D, T, export_cells<D, Q, T>()>::BPC), 128, 0, s>>>(
        cap, b0, nb, (const T*)fa, (const T*)fb, cur, level, nbr, sm, out, (uintptr_t)out % 16 == 0);
  }
  static void import_f(cudaStream_t s, int64_t cap, int64_t b0, int64_t nb, void* fa, void* fb,
                       unsigned cur, const int32_t* level, const int32_t* nbr,
                       const uint64_t* sm, const double* in) {
    k_import_f<D, Q, T><<<grid_for(nb * M, 256), 256, 0, s>>>(cap, b0, nb, (T*)fa, (T*)fb, cur,
                                                               level, nbr, sm, in);
  }
  static void export_rho_u(cudaStream_t s, int64_t cap, int64_t b0, int64_t nb, const void* fa,
                           const void* fb, unsigned cur, const int32_t* level,
                           const int32_t* nbr, const uint64_t* sm, double* out) {
    k_export_rho_u<D, Q, T><<<grid_for(nb, BlockRows<D, T>::BPC), 128, 0, s>>>(
        cap, b0, nb, (const T*)fa, (const T*)fb, cur, level, nbr, sm, out, (uintptr_t)out % 32 == 0);
  }
  static void init_rest(cudaStream_t s, int64_t cap, void* f) {
    k_init_rest<D, Q, T><<<grid_for(cap * M, 256), 256, 0, s>>>(cap, (T*)f);
  }
  static void solid_rest(cudaStream_t s, const int32_t* list, int n, const uint64_t* sm, void* f) {
    if (n > 0) k_solid_rest<D, Q, T><<<grid_for((int64_t)n * M, 256), 256, 0, s>>>(list, n, sm, (T*)f);
  }
  static int mass_partial(cudaStream_t s, int64_t cap, const void* fa, const void* fb,
                          unsigned cur, const int32_t* level, const int32_t* status,
                          const int32_t* nbr, const uint64_t* sm, double* partial) {
    const int grid = 152 * 4;
    k_mass_partial<D, Q, T><<<grid, 256, 0, s>>>(cap, (const T*)fa, (const T*)fb, cur, level,
                                                 status, nbr, sm, partial);
    return grid;
  }
  static int force_partial(cudaStream_t s, const int32_t* list, int n, const void* f,
                           const int32_t* nbr, const int32_t* status,
                           const uint64_t* sm, double omega, double dx, double* partial) {
    const int grid = std::min(152 * 8, grid_for(std::max(n, 1), 8));   // 3 grid doubles of scratch
    k_force_partial<D, Q, T><<<grid, 256, 0, s>>>(list, n, (const T*)f, nbr, status, sm,
                                                  omega, dx, partial);
    return grid;
  }
  static void features(cudaStream_t s, const int32_t* list, int n, const void* f, const int32_t* nbr, const uint64_t* sm, int level, int lmax,
                       double inv_dx, float* out) {
    if constexpr (D == 3) {
      if (n > 0)
        k_features<Q, T><<<grid_for(n, 4), 128, 0, s>>>(list, n, (const T*)f, nbr, sm,
                                                        level, lmax, inv_dx, out);
    }
  }
  static void coarsen_fixup(cudaStream_t s, const int32_t* list, int n, const int32_t* child0,
                            const int32_t* parent, const int8_t* marks, const int32_t* nbr,
                            const uint64_t* sm, const int32_t* level, void* fa, void* fb,
                            unsigned cur) {
    if (n <= 0) return;
    const int64_t threads = (int64_t)n * Block<D>::NC * M;
    k_coarsen_fixup<D, Q, T><<<(int)((threads + 255) / 256), 256, 0, s>>>(
        list, n, child0, parent, marks, nbr, sm, level, (T*)fa, (T*)fb, cur);
  }

  static void collide_stream_batch(cudaStream_t s, const uint32_t* items, int n,
                                   const InstDesc* descs, int level, int which_in, int variant) {
    if (n <= 0) return;
    // variant: 64 / 128 / 256 / 512 cells per CTA, i.e. M_L = 64/M .. 512/M
    // blocks (never less than a warp; anything else: 512)
    switch (variant) {
      case 64: batch_cells<64>(s, items, n, descs, level, which_in); break;
      case 128: batch_cells<128>(s, items, n, descs, level, which_in); break;
      case 256: batch_cells<256>(s, items, n, descs, level, which_in); break;
      default: batch_cells<512>(s, items, n, descs, level, which_in);
    }
  }
  template <int CELLS>
  static void batch_cells(cudaStream_t s, const uint32_t* items, int n, const InstDesc* descs,
                          int level, int which_in) {
    constexpr int V = row_cells<D, Q, T>(), THREADS = row_threads<V>(CELLS);
    k_collide_stream_batch<D, Q, T, THREADS>
        <<<grid_for(n, THREADS * V / M), THREADS, 0, s>>>(items, n, descs, level, which_in);
  }
  static void interp_batch(cudaStream_t s, const uint32_t* items, int n, const InstDesc* descs,
                           int level, int which_par, int which_ch) {
    if (n <= 0) return;
    k_interp_batch<D, Q, T><<<grid_for(n, 128 / M), 128, 0, s>>>(items, n, descs, level,
                                                                   which_par, which_ch);
  }
  static void average_batch(cudaStream_t s, const uint32_t* items, int n, const InstDesc* descs,
                            int level, int which_par, int which_ch) {
    if (n <= 0) return;
    const int64_t kids = (int64_t)n * Block<D>::NC;
    k_average_batch<D, Q, T><<<(int)((kids + 128 / M - 1) / (128 / M)), 128, 0, s>>>(
        items, kids, descs, level, which_par, which_ch);
  }

  static void average_groups(cudaStream_t s, const int32_t* items, int n, void* fpar,
                             const void* fch, int64_t first_child,
                             const int32_t* parent, const int32_t* nbr, const uint64_t* sm,
                             double ratio, bool solid, bool chained) {
    if (n <= 0) return;
    const int grid = grid_for((int64_t)n, 16);
    using R = typename Store<T>::R;
    const R keep = R(1.0 - ratio);
    launch_chained(solid ? k_average_groups<D, Q, T, true> : k_average_groups<D, Q, T, false>,
                   chained, grid, 64, s, items, n, (T*)fpar, (const T*)fch, (int)first_child,
                   parent, nbr, solid ? sm : nullptr, keep);
  }

  template <int THREADS>
  static int persistent_ctas_t() {
    constexpr size_t smem = persist_smem_bytes<D, Q, T, THREADS>();
    auto k = k_batch_persistent<D, Q, T, THREADS>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
        cudaSuccess)
      return 0;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, THREADS, smem) != cudaSuccess)
      return 0;
    return per_sm * sm_count;
  }
  static int persistent_ctas(int threads) {
    switch (threads) {
      case 64: return persistent_ctas_t<64>();
      case 128: return persistent_ctas_t<128>();
      case 256: return persistent_ctas_t<256>();
      default: return 0;
    }
  }
  static void batch_persistent(cudaStream_t s, const PersistArgs& a, int threads, int ctas) {
    switch (threads) {
      case 64:
        k_batch_persistent<D, Q, T, 64><<<ctas, 64, persist_smem_bytes<D, Q, T, 64>(), s>>>(a);
        break;
      case 128:
        k_batch_persistent<D, Q, T, 128><<<ctas, 128, persist_smem_bytes<D, Q, T, 128>(), s>>>(a);
        break;
      default:
        k_batch_persistent<D, Q, T, 256><<<ctas, 256, persist_smem_bytes<D, Q, T, 256>(), s>>>(a);
    }
  }

  static const LbmOps* ops() {
    static const LbmOps o = {setup,         collide_stream, interp,   average,
                             average_groups, criterion,     export_f,       import_f, export_rho_u,
                             init_rest,     mass_partial,   force_partial,
                             collide_stream_batch, interp_batch, average_batch,
                             persistent_ctas, batch_persistent, features,
                             coarsen_fixup, solid_rest};
    return &o;
  }
};

}  // namespace amr
