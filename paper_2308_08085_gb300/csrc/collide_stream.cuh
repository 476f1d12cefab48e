// Fused collide + stream of one level (Sections 4.2, 4.3) in pull form, and
// the link tables and the gather / scatter of a cell's populations that every
// other kernel uses to read or write the state.  Included by lbm_kernels.cuh.
//
// Population layout (every storage type): block-major, g[b * Q M + p * M + l],
// M = 4^D cells per block, l = i + 4 j + 16 k: the Q planes of a block are one
// contiguous run, so blocks with unrelated IDs still move whole DRAM pages.
//
// What is stored.  The paper stores the post-streaming (pre-collision)
// populations f(x, t) of every cell.  This library stores, for every cell y
// and direction p, the value that will stream out of y along c_p: the
// post-collision f*_p(y) of the last step.  The pre-collision state is
// therefore spread over the neighbours and is read by a gather:
//
//   f_p(x) = g_p(x - c_p)        when x - c_p is a fluid cell of the same level
//          = g_pbar(x)           otherwise (no same-level block there -- the
//                                coarse-fine interface --, a wall, or a solid
//                                cell), pbar the opposite of p.
//
// In the second case the slot g_pbar(x) holds the value that bounced back
// into x: the step that wrote it applied the boundary rule of the link (the
// moving-wall term or the anti-bounce-back outlet value, Section 2), so the
// gather needs no boundary arithmetic.  Writing a pre-collision value f_p(x)
// (interpolation, averaging, imports) is the scatter into the same slot.
// Each slot is the source of exactly one (cell, direction) pair, so gathers
// and scatters of different cells never collide, and the whole method
// (interpolation, averaging, criterion, exports) sees exactly the state of
// the paper's formulation.  The fused step reads its Q values through the
// gather (loads shifted across block edges, served by L1/L2) and writes all
// Q post-collision values of a cell to its own slots: every store is a whole
// row of the block, and no store crosses a block edge.
#pragma once
#include "lattice.cuh"
#include "lbm_ops.h"

#include <algorithm>

namespace amr {

constexpr int ST_UNREFINED = 1;
constexpr int ST_REFINED = 2;
constexpr int CLS_INTERIOR = 0, CLS_INTERFACE = 1, CLS_GHOST = 2;
constexpr int FACE_NOSLIP = 0, FACE_OUTLET = 2;

// geometric neighbour code (sx+1) + 3 (sy+1) [+ 9 (sz+1)] -> neighbour index k
struct GeoTable {
  int8_t k_of_code[27];
};
template <int D>
constexpr GeoTable make_geo() {
  GeoTable t{};
  for (int c = 0; c < 27; ++c) {
    int sx = c % 3 - 1, sy = (c / 3) % 3 - 1, sz = c / 9 - 1;
    if (D == 2) t.k_of_code[c] = (c < 9) ? (int8_t)Nbr<2>::dir_of(sx, sy, 0) : (int8_t)-1;
    else t.k_of_code[c] = (int8_t)Nbr<3>::dir_of(sx, sy, sz);
  }
  return t;
}
static __constant__ GeoTable c_geo2 = make_geo<2>();
static __constant__ GeoTable c_geo3 = make_geo<3>();

template <int D>
__device__ __forceinline__ int geo_to_k(int code) {
  return D == 2 ? c_geo2.k_of_code[code] : c_geo3.k_of_code[code];
}

// Link tables: for direction p and cell l, the block that holds the cell
// x + s c_p (s = +1: the target of the link leaving x, s = -1: the source of
// the link arriving at x) and the cell index inside it, packed as
// e = blk | (cell << 5).  blk is the geometric code of the neighbour block
// (0 .. 3^D - 1, centre = the block itself) or, in the _K tables, its index
// k in the block's neighbour row (0 = the block itself).
template <int D, int Q>
struct LinkTable {
  uint16_t e[Q * Block<D>::M];
};
template <int D, int Q, int SIGN, bool BY_K>
constexpr LinkTable<D, Q> make_link_table() {
  LinkTable<D, Q> t{};
  constexpr int M = Block<D>::M;
  for (int p = 0; p < Q; ++p)
    for (int l = 0; l < M; ++l) {
      const int ti = Block<D>::ci(l) + SIGN * VS<D, Q>::cx[p];
      const int tj = Block<D>::cj(l) + SIGN * VS<D, Q>::cy[p];
      const int tk = Block<D>::ck(l) + SIGN * VS<D, Q>::cz[p];
      const int sx = ti < 0 ? -1 : (ti > 3 ? 1 : 0);
      const int sy = tj < 0 ? -1 : (tj > 3 ? 1 : 0);
      const int sz = tk < 0 ? -1 : (tk > 3 ? 1 : 0);
      const int blk = BY_K ? Nbr<D>::dir_of(sx, sy, sz)
                           : (sx + 1) + 3 * (sy + 1) + (D == 3 ? 9 * (sz + 1) : 0);
      const int cell = (ti & 3) + 4 * (tj & 3) + (D == 3 ? 16 * (tk & 3) : 0);
      t.e[p * M + l] = (uint16_t)(blk | (cell << 5));
    }
  return t;
}
template <int D, int Q>
__device__ const LinkTable<D, Q> g_tgt_geo = make_link_table<D, Q, +1, false>();
template <int D, int Q>
__device__ const LinkTable<D, Q> g_src_k = make_link_table<D, Q, -1, true>();
template <int D, int Q>
__device__ const LinkTable<D, Q> g_tgt_k = make_link_table<D, Q, +1, true>();

template <int D, int Q, int P>
__device__ __forceinline__ int link_entry(const LinkTable<D, Q>& t, int l) {
  return __ldg(&t.e[P * Block<D>::M + l]);
}

// A population load.  COH: the value may have been stored by another CTA of
// the same launch (the persistent batched kernel), so it is read from L2
// (ld.global.cg), never through a path that may hold an older copy.
template <bool COH, class T>
__device__ __forceinline__ T ld_pop(const T* p) {
  if constexpr (COH) return __ldcg(p);
  else return *p;
}

// --------------------------------------------------------- gather / scatter
// Pre-collision populations of cell l of block b (see the file comment).
// `row` is the block's neighbour row (neighbour-index order), in global or
// shared memory.  A solid cell holds its own (rest) values.  With
// SOLID, `solidmask` (one bit per cell) may still be null: no solid cells.
template <int D, int Q, class T, bool SOLID, bool COH = false>
__device__ __forceinline__ void gather_cell(typename Store<T>::R (&f)[Q],
                                            const T* __restrict__ g, int b, int l,
                                            const int32_t* __restrict__ row,
                                            const uint64_t* __restrict__ solidmask) {
  using S = Store<T>;
  constexpr int M = Block<D>::M;
  const size_t own = (size_t)b * (Q * M) + l;
  const bool has_sm = SOLID && solidmask != nullptr;
  const bool solid_cell = has_sm && ((__ldg(solidmask + b) >> l) & 1ull);
  static_for<0, Q>([&](auto P) {
    constexpr int p = P;
    constexpr int pb = VS<D, Q>::opp[p];
    if constexpr (p == 0) {
      f[0] = S::template load<D, Q, 0>(ld_pop<COH>(g + own));
    } else {
      const int e = link_entry<D, Q, p>(g_src_k<D, Q>, l);
      const int k = e & 31, sl = e >> 5;
      const int src = k == 0 ? b : row[k];
      bool back = src < 0;
      if (has_sm && !back) back = (__ldg(solidmask + src) >> sl) & 1ull;
      const size_t at = solid_cell ? own + (size_t)p * M
                                   : (back ? own + (size_t)pb * M
                                           : (size_t)src * (Q * M) + (size_t)p * M + sl);
      f[p] = S::template load<D, Q, p>(ld_pop<COH>(g + at));
    }
  });
}

// Opposite directions as a device table (for loops over runtime p).
template <int D, int Q>
struct OppTable {
  int8_t o[Q];
};
template <int D, int Q>
constexpr OppTable<D, Q> make_opp() {
  OppTable<D, Q> t{};
  for (int p = 0; p < Q; ++p) t.o[p] = (int8_t)VS<D, Q>::opp[p];
  return t;
}
template <int D, int Q>
__device__ const OppTable<D, Q> g_opp = make_opp<D, Q>();

// The element of g that holds the pre-collision f_p of cell l of block b
// (the scatter rule of scatter_cell for one runtime direction p).
template <int D, int Q>
__device__ __forceinline__ size_t src_slot(int p, int b, int l, const int32_t* row,
                                           const uint64_t* __restrict__ solidmask) {
  constexpr int M = Block<D>::M;
  const size_t own = (size_t)b * (Q * M) + l;
  if (p == 0) return own;
  const int e = __ldg(&g_src_k<D, Q>.e[p * M + l]);
  const int k = e & 31, sl = e >> 5;
  const int src = k == 0 ? b : row[k];
  bool back = src < 0;
  if (solidmask && !back) back = (__ldg(solidmask + src) >> sl) & 1ull;
  if (solidmask && ((__ldg(solidmask + b) >> l) & 1ull)) return own + (size_t)p * M;
  return back ? own + (size_t)g_opp<D, Q>.o[p] * M : (size_t)src * (Q * M) + (size_t)p * M + sl;
}

// Store pre-collision populations f of cell l of block b so that gather_cell
// returns them.  MOVE (new blocks of an adaptation): where the source cell
// x - c_p lies in a block that existed before (is_new(block) false), its slot
// still holds the value that bounced back into that old cell, which now has
// to come from this cell: it is moved to this cell's opposite slot first.
template <int D, int Q, class T, bool SOLID, bool MOVE = false, class IsNew = int>
__device__ __forceinline__ void scatter_cell(const typename Store<T>::R (&f)[Q],
                                             T* __restrict__ g, int b, int l,
                                             const int32_t* __restrict__ row,
                                             const uint64_t* __restrict__ solidmask,
                                             IsNew is_new = 0) {
  using S = Store<T>;
  constexpr int M = Block<D>::M;
  const size_t own = (size_t)b * (Q * M) + l;
  const bool has_sm = SOLID && solidmask != nullptr;
  const bool solid_cell = has_sm && ((__ldg(solidmask + b) >> l) & 1ull);
  static_for<0, Q>([&](auto P) {
    constexpr int p = P;
    constexpr int pb = VS<D, Q>::opp[p];
    if constexpr (p == 0) {
      g[own] = S::template save<D, Q, 0>(f[0]);
    } else {
      const int e = link_entry<D, Q, p>(g_src_k<D, Q>, l);
      const int k = e & 31, sl = e >> 5;
      const int src = k == 0 ? b : row[k];
      bool back = src < 0;
      if (has_sm && !back) back = (__ldg(solidmask + src) >> sl) & 1ull;
      if (solid_cell) {
        g[own + (size_t)p * M] = S::template save<D, Q, p>(f[p]);
      } else if (back) {
        g[own + (size_t)pb * M] = S::template save<D, Q, p>(f[p]);
      } else {
        T* slot = g + (size_t)src * (Q * M) + (size_t)p * M + sl;
        if constexpr (MOVE) {
          if (k != 0 && !is_new(src)) g[own + (size_t)pb * M] = *slot;
        }
        *slot = S::template save<D, Q, p>(f[p]);
      }
    }
  });
}

// ------------------------------------------------------------ BGK collision
// The collision (Section 2) by pairs of opposite directions: with c3 = 3 c.u,
// f_eq,p = w_p rho (S + c3) and f_eq,pbar = w_p rho (S - c3),
// S = 1 - 1.5 u^2 + c3^2 / 2, so a pair shares c3 and S.  With SHIFTED the
// values are g_p = f_p - w_p, as the 16-bit storages hold them: rho = 1 +
// sum_p g_p, j = sum_p c_p g_p (the weights have no first moment), and
// f_eq,p - w_p = w_p rho (S' +- c3) with (rho - 1) / rho - 1.5 u^2 + c3^2 / 2
// for S': the shift is neither added on load nor removed on store.  One FP64
// instruction occupies a scheduler for 64 cycles here (32 lanes, measured), so
// the FP64 kernels are bound by the operations of this function: 4.5 per
// direction, 7 when each direction is evaluated on its own.  (-f is an operand
// modifier; 0 - f would be an operation.)
__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float rcp_(float a) { return 1.f / a; }
__device__ __forceinline__ double rcp_(double a) { return 1.0 / a; }

// Two FP32 values in a register pair: one instruction for both (the rate per
// value is that of FP32, the issue slots are half).
struct F2 {
  unsigned long long v;
  F2() = default;
  __device__ __forceinline__ explicit F2(float a) : F2(a, a) {}
  __device__ __forceinline__ F2(float a, float b) {
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
  }
  __device__ __forceinline__ float get(int c) const {
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
    return c ? b : a;
  }
  __device__ __forceinline__ void set(int c, float x) { *this = c ? F2(get(0), x) : F2(x, get(1)); }
};
__device__ __forceinline__ F2 operator+(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 operator-(F2 a, F2 b) {
  F2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 operator*(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 fma_(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ F2 rcp_(F2 a) { return F2(1.f / a.get(0), 1.f / a.get(1)); }

template <int D, int Q, bool SHIFTED, class R>
struct Relax {
  R rho, base, ux3, uy3, uz3;
  __device__ __forceinline__ Relax(R rho_, R base_, R x, R y, R z)
      : rho(rho_), base(base_), ux3(x), uy3(y), uz3(z) {}
  __device__ __forceinline__ explicit Relax(const R (&f)[Q]) {
    using V = VS<D, Q>;
    // sums of the values, and of the differences along each axis
    R s = f[0], j[3];
    bool any[3] = {false, false, false};
    static_for<1, Q>([&](auto P) {
      constexpr int p = P, pb = V::opp[p];
      if constexpr (pb > p) {
        constexpr int c[3] = {V::cx[p], V::cy[p], V::cz[p]};
        s = s + (f[p] + f[pb]);
        constexpr bool flip = c[0] < 0 || (c[0] == 0 && (c[1] < 0 || (c[1] == 0 && c[2] < 0)));
        const R d = flip ? f[pb] - f[p] : f[p] - f[pb];   // along the first non-zero axis
        static_for<0, D>([&](auto A) {
          constexpr int ca = flip ? -c[A] : c[A];
          if constexpr (ca != 0) {
            j[A] = !any[A] ? d : (ca > 0 ? j[A] + d : j[A] - d);
            any[A] = true;
          }
        });
      }
    });
    rho = SHIFTED ? R(1) + s : s;
    const R inv = rcp_(rho);
    const R inv3 = R(3) * inv;
    ux3 = j[0] * inv3;
    uy3 = j[1] * inv3;
    R usq9 = fma_(uy3, uy3, ux3 * ux3);
    if constexpr (D == 3) {
      uz3 = j[2] * inv3;
      usq9 = fma_(uz3, uz3, usq9);
    } else {
      uz3 = R(0);
    }
    base = fma_(R(-1.0 / 6.0), usq9, SHIFTED ? s * inv : R(1));
  }
  // 3 c_p . u, for the member of a pair whose first non-zero component is positive
  template <int P>
  __device__ __forceinline__ R c3() const {
    using V = VS<D, Q>;
    constexpr int cx = V::cx[P], cy = V::cy[P], cz = V::cz[P];
    if constexpr (cx > 0) {
      const R a = cy == 0 ? ux3 : (cy > 0 ? ux3 + uy3 : ux3 - uy3);
      return cz == 0 ? a : (cz > 0 ? a + uz3 : a - uz3);
    } else if constexpr (cy > 0) {
      return cz == 0 ? uy3 : (cz > 0 ? uy3 + uz3 : uy3 - uz3);
    } else {
      return uz3;
    }
  }
  // f_eq of every direction (shifted alike) as a product, handed to use(p, w, x):
  // f_eq,p = w x, w = w_p rho
  template <class Use>
  __device__ __forceinline__ void each(Use&& use) const {
    using V = VS<D, Q>;
    const R half = R(0.5);
    constexpr double w0 = V::w[0];
    use(std::integral_constant<int, 0>{}, R(w0) * rho, base);
    static_for<1, Q>([&](auto P) {
      constexpr int p = P, pb = V::opp[p];
      if constexpr (pb > p) {
        constexpr bool flip = V::cx[p] < 0 || (V::cx[p] == 0 && (V::cy[p] < 0 ||
                                               (V::cy[p] == 0 && V::cz[p] < 0)));
        constexpr int up = flip ? pb : p, dn = flip ? p : pb;
        constexpr double wp = V::w[p];
        const R c = c3<up>();
        const R wr = R(wp) * rho;
        const R S = fma_(half, c * c, base);
        use(std::integral_constant<int, up>{}, wr, S + c);
        use(std::integral_constant<int, dn>{}, wr, S - c);
      }
    });
  }
};

// f + rate (f_eq - f), f_eq = w x.  (Packed pairs have no negated operand; the
// product form (rate w) x + (1 - rate) f was no faster there: 12.8 against 12.4
// ms for five coarse steps of the 128x32x32 prism in FP16.)
__device__ __forceinline__ float relaxed(float f, float w, float x, float rate) {
  return fmaf(rate, fmaf(w, x, -f), f);
}
__device__ __forceinline__ double relaxed(double f, double w, double x, double rate) {
  return fma(rate, fma(w, x, -f), f);
}
__device__ __forceinline__ F2 relaxed(F2 f, F2 w, F2 x, F2 rate) {
  return fma_(rate, fma_(w, x, F2(0.f) - f), f);
}

// Value stored in the own slot p of a cell whose link p leaves through wall
// face `face` (Section 2 boundary equations): the moving-wall bounce-back
// f* + bb, or the anti-bounce-back outlet value with the cell's velocity.
// fs is the value as stored (SHIFTED: less w_p).
template <int D, int Q, int P, bool SHIFTED, class R>
__device__ __forceinline__ R wall_value(R fs, int face, const Relax<D, Q, SHIFTED, R>& r,
                                        const FaceParams& faces) {
  using V = VS<D, Q>;
  constexpr int cx = V::cx[P], cy = V::cy[P], cz = V::cz[P];
  if (faces.kind[face] == FACE_OUTLET) {
    R c3 = R(0);
    if constexpr (cx != 0) c3 += cx > 0 ? r.ux3 : -r.ux3;
    if constexpr (cy != 0) c3 += cy > 0 ? r.uy3 : -r.uy3;
    if constexpr (cz != 0) c3 += cz > 0 ? r.uz3 : -r.uz3;
    constexpr double wp = V::w[P];
    R usq9 = r.ux3 * r.ux3 + r.uy3 * r.uy3;
    if constexpr (D == 3) usq9 += r.uz3 * r.uz3;
    const R sym = R(0.5) * (c3 * c3) - R(1.0 / 6.0) * usq9;   // 4.5 (c.u)^2 - 1.5 u^2
    const R wall = R(2.0 * wp) * faces.rho<R>(face) * (R(1) + sym);
    return SHIFTED ? -fs + (wall - R(2.0 * wp)) : -fs + wall;
  }
  return fs + faces.link<R>(face, P);
}

// ======================================================= cells by x-rows
// A thread holds V cells that are consecutive in x (a row of a block has 4).
// The values of a direction with c_x = 0 that reach the V cells are V
// consecutive values of one row (a source block and a row in it, or the own
// opposite slots where that block is missing): one vector load.  With
// c_x = +-1 they are V - 1 values of such a row and one value beside it,
// which comes from the x neighbour when the thread holds that end of the row:
// one vector load and one scalar load.  The kernel is bound by how many loads
// its warps keep in flight and by the address arithmetic of the links; V cells
// per thread divide the latter and the load and store instructions by V.
template <class T, int V>
struct alignas(sizeof(T) * V) Vec {
  T v[V];
};
template <int BYTES> struct Raw;
template <> struct Raw<2> { using type = unsigned short; };
template <> struct Raw<4> { using type = unsigned; };
template <> struct Raw<8> { using type = uint2; };
template <> struct Raw<16> { using type = uint4; };

template <bool COH, class T, int V>
__device__ __forceinline__ Vec<T, V> ld_vec(const T* p) {
  if constexpr (COH) {
    using W = typename Raw<sizeof(T) * V>::type;
    union { W w; Vec<T, V> v; } u;
    u.w = __ldcg(reinterpret_cast<const W*>(p));
    return u.v;
  } else {
    return *reinterpret_cast<const Vec<T, V>*>(p);
  }
}

// Cells per thread.  3D: two, so that a warp is one block and takes one path.
// Four (two blocks per warp) were faster on the periodic 256^3 forest, where
// every block takes the same path (0.37 against 0.40 ms per step), and slower
// on the 64^3 cavity with three extra levels, where they differ (38.2 against
// 36.1 ms for ten coarse steps).  FP64: one.  An FP64 instruction occupies a
// scheduler for 64 cycles and an SM for 19, so an SM needs four warps to run at
// its rate: two warps per block reach it with half the blocks (coarse steps of
// cavities and prisms, one against two: 24^3 16.4 / 26.6 us, 24^3 with two extra
// levels 658 / 773, 64^3 with one 579 / 612, 128x32x16 prism with three 3461 /
// 3632; none slower).  D3Q27 in FP32: one; two leave room for 20 warps of 96
// registers, one for 32 of 64 (prism of 2.6 million finest blocks 24,830 / 24,050
// MLUPS, 128x32x32 prism, cubic, five coarse steps 14.1 / 14.7 ms, 48x24x16 prism
// with one level 40 / 53 us).  2D: one; the meshes are small and latency counts
// (128^2 cavity, FP32, 20 coarse steps: 1.9 / 2.2 / 3.0 ms with 1 / 2 / 4).
template <int D, int Q, class T>
constexpr int row_cells() {
  return D == 2 || sizeof(T) == 8 || (Q == 27 && sizeof(T) == 4) ? 1 : 2;
}

// Threads of a CTA that holds `cells` cells, V per thread (at least a warp), and
// the CTAs per SM its register budget is set for: 896 threads for D3Q19 in 32 bits and
// less (72 registers; the cavity above takes 37.0 / 36.1 / 36.3 ms with 768 /
// 896 / 1024), 1024 for D3Q27 with a cell per thread, 640 with two (96
// registers; 13.8 ms against 15.4 with 768 for five coarse steps of the
// 128x32x32 prism in FP16), fewer for FP64, whose arithmetic saturates with few
// warps.
template <int V>
constexpr int row_threads(int cells) {
  return cells / V < 32 ? 32 : cells / V;
}
template <int Q, class T, int V, int THREADS, bool DENSE = false>
constexpr int row_min_ctas() {
  const int threads = (Q == 9 ? 1024 : (sizeof(T) == 8 ? (Q == 19 ? 512 : 384)
                                                       : (Q == 19 ? 896 : (V == 1 ? 1024 : 640)))) +
                      (DENSE ? 128 : 0);
  return threads / THREADS > 0 ? threads / THREADS : 1;
}

// Where the sources of a thread's cells lie: t of the M / V threads of a block.
template <int D, int V>
struct RowPos {
  int l0, i0;          // first cell, its x
  int yp, ym, zp, zm;  // code steps of the source row for c_y = +1, -1, c_z = +1, -1
  int oyp, oym, oy0, ozp, ozm, oz0;   // cell offsets of the source row
  __device__ __forceinline__ explicit RowPos(int t) {
    l0 = V * t;
    i0 = l0 & 3;
    const int j = (l0 >> 2) & 3, k = D == 3 ? l0 >> 4 : 0;
    yp = j == 0 ? -3 : 0;
    ym = j == 3 ? 3 : 0;
    oyp = ((j - 1) & 3) * 4;
    oym = ((j + 1) & 3) * 4;
    oy0 = j * 4;
    zp = D == 3 && k == 0 ? -9 : 0;
    zm = D == 3 && k == 3 ? 9 : 0;
    ozp = ((k - 1) & 3) * 16;
    ozm = ((k + 1) & 3) * 16;
    oz0 = k * 16;
  }
  // neighbour code of the source row for links c = (., CY, CZ)
  template <int CY, int CZ>
  __device__ __forceinline__ int code() const {
    return (D == 2 ? 4 : 13) + (CY > 0 ? yp : (CY < 0 ? ym : 0)) +
           (CZ > 0 ? zp : (CZ < 0 ? zm : 0));
  }
  template <int CY, int CZ>
  __device__ __forceinline__ int row() const {   // first cell of the source row
    return (CY > 0 ? oyp : (CY < 0 ? oym : oy0)) +
           (D == 3 ? (CZ > 0 ? ozp : (CZ < 0 ? ozm : oz0)) : 0);
  }
  // the value beside the vector for c_x = CX: x of its cell, code step
  template <int CX>
  __device__ __forceinline__ int edge_x() const {
    return CX > 0 ? (i0 - 1) & 3 : (i0 + V) & 3;
  }
  template <int CX>
  __device__ __forceinline__ int edge_code() const {
    return CX > 0 ? (i0 == 0 ? -1 : 0) : (i0 + V == 4 ? 1 : 0);
  }
};

// Stored values that arrive at the V cells of thread t of block b: the gather
// of gather_cell (see the file comment) without conversion.  `nb` is the
// block's neighbour row in geometric order; `sm` (SOLID) the solid cells of
// those blocks, read when any_solid.
template <int D, int Q, class T, int V, bool CHECK, bool SOLID, bool COH>
__device__ __forceinline__ void gather_row(Vec<T, V> (&g)[Q], const T* gin, int b,
                                           const RowPos<D, V>& pos, const int32_t* nb,
                                           const uint64_t* sm, bool any_solid,
                                           const T* in_place = nullptr) {
  constexpr int M = Block<D>::M;
  using VS_ = VS<D, Q>;
  const T* own = gin + (size_t)b * (Q * M) + pos.l0;
  const bool stay = V == 1 && in_place != nullptr;
  static_for<0, Q>([&](auto P) {
    constexpr int p = P, pb = VS_::opp[p];
    constexpr int cx = VS_::cx[p], cy = VS_::cy[p], cz = VS_::cz[p];
    if constexpr (cy == 0 && cz == 0 && cx == 0) {
      g[p] = ld_vec<COH, T, V>(stay ? in_place : own);
    } else {
      bool has = true;
      const T* at = own;
      if constexpr (cy != 0 || cz != 0) {
        const int s = nb[pos.template code<cy, cz>()];
        has = !CHECK || s >= 0;
        at = has ? gin + ((int64_t)s * (Q * M) + (pos.template row<cy, cz>() + pos.i0))
                 : own + (pb - p) * M;
      }
      if constexpr (cx == 0) {
        g[p] = ld_vec<COH, T, V>((stay ? in_place : at) + p * M);
      } else {
        const int se = nb[pos.template code<cy, cz>() + pos.template edge_code<cx>()];
        const T* ae = !CHECK || se >= 0 ? gin + ((int64_t)se * (Q * M) + (pos.template row<cy, cz>() +
                                                                pos.template edge_x<cx>()))
                              : own + ((pb - p) * M + (cx > 0 ? 0 : V - 1));
        const T e = ld_pop<COH>((stay ? in_place : ae) + p * M);
        if constexpr (V == 1) {
          g[p].v[0] = e;
        } else {
          const Vec<T, V> v = ld_vec<COH, T, V>(at + p * M);
          if constexpr (cx > 0) {
            g[p].v[0] = e;
#pragma unroll
            for (int i = 1; i < V; ++i) g[p].v[i] = has ? v.v[i - 1] : v.v[i];
          } else {
            g[p].v[V - 1] = e;
#pragma unroll
            for (int i = 0; i + 1 < V; ++i) g[p].v[i] = has ? v.v[i + 1] : v.v[i];
          }
        }
      }
    }
  });
  if constexpr (CHECK && SOLID) {
    // a solid source: the value that bounced back into the cell's own slot
    if (any_solid && !stay) {
      static_for<1, Q>([&](auto P) {
        constexpr int p = P, pb = VS_::opp[p];
        constexpr int cx = VS_::cx[p], cy = VS_::cy[p], cz = VS_::cz[p];
        const int code = pos.template code<cy, cz>(), row = pos.template row<cy, cz>();
        const unsigned in_row = (unsigned)(sm[code] >> row) & 15u;
        unsigned hit;   // bit i: the source of cell i is solid
        if constexpr (cx == 0) {
          hit = in_row >> pos.i0;
        } else {
          const unsigned e = (unsigned)(sm[code + pos.template edge_code<cx>()] >>
                                        (row + pos.template edge_x<cx>())) & 1u;
          if constexpr (cx > 0) hit = ((in_row >> pos.i0) << 1) | e;
          else hit = (((in_row >> pos.i0) >> 1) & ((1u << (V - 1)) - 1u)) | (e << (V - 1));
        }
        hit &= (1u << V) - 1u;
        if (hit) {
          const Vec<T, V> v = ld_vec<COH, T, V>(own + pb * M);
#pragma unroll
          for (int i = 0; i < V; ++i)
            if ((hit >> i) & 1u) g[p].v[i] = v.v[i];
        }
      });
      // a solid cell holds its own (rest) values
      const unsigned self = (unsigned)(sm[D == 2 ? 4 : 13] >> pos.l0) & ((1u << V) - 1u);
      if (self) {
        static_for<1, Q>([&](auto P) {
          const Vec<T, V> v = ld_vec<COH, T, V>(own + P * M);
#pragma unroll
          for (int i = 0; i < V; ++i)
            if ((self >> i) & 1u) g[P].v[i] = v.v[i];
        });
      }
    }
  }
}

constexpr int BF_WALL = 1;      // a neighbour is a moving wall or an outlet (a no-slip wall
                                // bounces back with no added term, like a missing block)
constexpr int BF_SOLID = 2;     // the block or a neighbour has solid cells
constexpr int BF_OUTSIDE = 4;   // a neighbour block is missing or a wall

// The lanes of the TPB threads that share this thread's block.
template <int TPB>
__device__ __forceinline__ unsigned block_lanes() {
  if constexpr (TPB == 32) return 0xffffffffu;
  else return ((1u << TPB) - 1u) << ((threadIdx.x & 31) & ~(TPB - 1));
}

// The TPB threads of a block stage its neighbour row in geometric order (and
// the solid cells of those blocks) in shared memory and return the block's
// flags to every one of them.  `lanes`: their bits within the warp.
// (faces null: the walls are not looked at)
template <int D, int TPB, bool SOLID>
__device__ __forceinline__ int stage_block(int32_t* s_nb, uint64_t* s_sm, int b, int t,
                                           unsigned lanes, const int32_t* __restrict__ nbr,
                                           const uint64_t* __restrict__ solidmask,
                                           const FaceParams* faces) {
  constexpr int NCODE = D == 2 ? 9 : 27;
  int flags = 0;
  const int32_t* row = nbr + (size_t)b * NBR_STRIDE;
#pragma unroll
  for (int c0 = 0; c0 < NCODE; c0 += TPB) {
    const int code = c0 + t;
    if (NCODE % TPB == 0 || code < NCODE) {
      const int v = __ldg(row + geo_to_k<D>(code));
      s_nb[code] = v;
      if (v < 0) flags |= BF_OUTSIDE;
      if (v <= -2 && faces && faces->kind[-2 - v] != FACE_NOSLIP) flags |= BF_WALL;
      if constexpr (SOLID) {
        const uint64_t m = v >= 0 && solidmask ? __ldg(solidmask + v) : 0ull;
        s_sm[code] = m;
        if (m) flags |= BF_SOLID;
      }
    }
  }
  __syncwarp(lanes);
  return (int)__reduce_or_sync(lanes, (unsigned)flags);
}

// The links of cell l that leave through a moving wall or an outlet: their
// stored value takes the wall's rule.
template <int D, int Q, bool SHIFTED, class R>
__device__ __forceinline__ void wall_links_in(R* f, const Relax<D, Q, SHIFTED, R>& r, int l,
                                              const int32_t* nb, const FaceParams& faces) {
  static_for<1, Q>([&](auto P) {
    constexpr int p = P;
    const int to = nb[link_entry<D, Q, p>(g_tgt_geo<D, Q>, l) & 31];
    if (to <= -2) f[p] = wall_value<D, Q, p, SHIFTED>(f[p], -2 - to, r, faces);
  });
}

// 3D: out of line, few blocks have such a link.  The values go through an array
// of their own, which lives in local memory: handing f itself over makes every
// cell of every block store its f there (1.6x the write traffic of the level,
// measured).  2D: in line; a launch is as long as its slowest block (80x100
// FP32 cavity, one level: 7.7 us per launch out of line, 7.2 in
// line, of which 4.3 without walls).
template <int D, int Q, bool SHIFTED, class R>
__device__ __noinline__ void wall_links_of(R* f, const Relax<D, Q, SHIFTED, R> r, int l,
                                           const int32_t* nb, const FaceParams& faces) {
  wall_links_in<D, Q, SHIFTED, R>(f, r, l, nb, faces);
}

template <int D, int Q, bool SHIFTED, class R>
__device__ __forceinline__ void wall_links(R (&f)[Q], const Relax<D, Q, SHIFTED, R>& r, int l,
                                           const int32_t* nb, const FaceParams& faces) {
  if constexpr (D == 2) {
    wall_links_in<D, Q, SHIFTED, R>(f, r, l, nb, faces);
  } else {
    R w[Q];
    static_for<0, Q>([&](auto P) { w[P] = f[P]; });
    wall_links_of<D, Q, SHIFTED, R>(w, r, l, nb, faces);
    static_for<0, Q>([&](auto P) { f[P] = w[P]; });
  }
}
template <int D, int Q, bool SHIFTED>
__device__ __forceinline__ void wall_links(F2 (&f)[Q], const Relax<D, Q, SHIFTED, F2>& r, int l,
                                           const int32_t* nb, const FaceParams& faces) {
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    float w[Q];
    static_for<0, Q>([&](auto P) { w[P] = f[P].get(c); });
    wall_links_of<D, Q, SHIFTED, float>(
        w, {r.rho.get(c), r.base.get(c), r.ux3.get(c), r.uy3.get(c), r.uz3.get(c)}, l + c, nb,
        faces);
    static_for<0, Q>([&](auto P) { f[P].set(c, w[P]); });
  }
}

// The children of exchanging parents (see Exchange) and how the interpolation
// reaches them: `rc` [Q][M] takes the rescaled parent cells.
template <class R>
struct ParentOut {
  R* rc;        // null: not an exchanging parent
  R keep;       // 1 - r_cf
};

// Collide-stream of the V cells of thread t of block b.  ghost: the bits of
// cells that read the interpolated values in their own slots of gout (the
// first substep of a level below the coarsest).  par.rc: the block exchanges
// with its children, and its pre-collision values rescaled to the fine level
// (f_eq + (f - f_eq) r_cf = f + (f_eq - f)(1 - r_cf), Section 3.4.1) go there.
template <int D, int Q, class T, int V, bool SOLID, bool GHOST, bool XCHG, bool COH>
__device__ __forceinline__ void step_row(const T* gin, T* gout, int b,
                                         int t, const int32_t* nb, const uint64_t* sm, int flags,
                                         uint64_t ghost, typename Store<T>::R om,
                                         const FaceParams& faces,
                                         ParentOut<typename Store<T>::R> par) {
  using S = Store<T>;
  using R = typename S::R;
  constexpr int M = Block<D>::M;
  constexpr bool SH = S::kShifted;
  constexpr unsigned ALL = (1u << V) - 1u;
  const RowPos<D, V> pos(t);
  Vec<T, V> g[Q];
  T* own = gout + (size_t)b * (Q * M) + pos.l0;
  const unsigned gm = GHOST ? (unsigned)(ghost >> pos.l0) & ALL : 0u;
  // (blocks that share a warp take the checked gather together)
  if (M / V < 32 || (flags & (BF_OUTSIDE | BF_SOLID)))
    gather_row<D, Q, T, V, true, SOLID, COH>(g, gin, b, pos, nb, sm, SOLID && (flags & BF_SOLID),
                                             GHOST && V == 1 && gm ? own : nullptr);
  else
    gather_row<D, Q, T, V, false, SOLID, COH>(g, gin, b, pos, nb, sm, false);
  if constexpr (GHOST && V > 1) {
    if (gm) {
      static_for<0, Q>([&](auto P) {
        const Vec<T, V> v = ld_vec<COH, T, V>(own + P * M);
#pragma unroll
        for (int i = 0; i < V; ++i)
          if ((gm >> i) & 1u) g[P].v[i] = v.v[i];
      });
    }
  }
  // W cells at a time: a packed pair, or one
  constexpr int W = V >= 2 && sizeof(T) == 2 ? 2 : 1;
  using RW = std::conditional_t<W == 2, F2, R>;
  static_for<0, V / W>([&](auto I) {
    constexpr int i = I * W;
    RW f[Q];
    static_for<0, Q>([&](auto P) {
      if constexpr (W == 2) f[P] = F2(S::raw(g[P].v[i]), S::raw(g[P].v[i + 1]));
      else f[P] = S::raw(g[P].v[i]);
    });
    const Relax<D, Q, SH, RW> r(f);
    r.each([&](auto P, RW w, RW x) {
      if constexpr (XCHG) {
        if (par.rc)
          *reinterpret_cast<RW*>(par.rc + P * M + pos.l0 + i) = relaxed(f[P], w, x, RW(par.keep));
      }
      f[P] = relaxed(f[P], w, x, RW(om));
    });
    if (flags & BF_WALL) wall_links<D, Q, SH>(f, r, pos.l0 + i, nb, faces);
    static_for<0, Q>([&](auto P) {
      if constexpr (W == 2) {
        g[P].v[i] = S::from_raw(f[P].get(0));
        g[P].v[i + 1] = S::from_raw(f[P].get(1));
      } else {
        g[P].v[i] = S::from_raw(f[P]);
      }
    });
  });
  unsigned solid = 0u;   // solid cells are not advanced
  if constexpr (SOLID) {
    if (flags & BF_SOLID) solid = (unsigned)(sm[D == 2 ? 4 : 13] >> pos.l0) & ALL;
  }
  if constexpr (SOLID && XCHG) {
    // a solid cell is at rest; its slots, which no step writes, may hold what
    // an earlier block of the same ID left there
    if (par.rc && solid) {
      static_for<0, Q>([&](auto P) {
        constexpr double wp = VS<D, Q>::w[P];
#pragma unroll
        for (int i = 0; i < V; ++i)
          if ((solid >> i) & 1u) par.rc[P * M + pos.l0 + i] = SH ? R(0) : R(wp);
      });
    }
  }
  if (!SOLID || solid == 0u) {
    static_for<0, Q>([&](auto P) { *reinterpret_cast<Vec<T, V>*>(own + P * M) = g[P]; });
  } else if (solid != ALL) {
    static_for<0, Q>([&](auto P) {
#pragma unroll
      for (int i = 0; i < V; ++i)
        if (!((solid >> i) & 1u)) own[P * M + i] = g[P].v[i];
    });
  }
}

// The ghost cells of the children of an exchanging parent: the V cells of
// thread t of every child c with ghost cells take the multilinear interpolant
// of the 2^D rescaled parent cells of quadrant c (child cell I at -1/4 + I/2
// between the parent cell centres; Section 3.4.1), written as it is into
// their own slots of the fine output buffer: first the interpolants in y and z at
// the quadrant's two x, then the V cells between them.  Ghost cells come in
// pairs along x (two layers).  Solid cells are skipped.
// One cell per thread: the weights of the quadrant's 2^D parent cells come from
// a table (an FP64 product of weights is a 64-cycle instruction).
template <int D>
struct CornerWeights {
  double w[Block<D>::M][Block<D>::NC];
};
template <int D>
constexpr CornerWeights<D> make_corner_weights() {
  CornerWeights<D> t{};
  for (int l = 0; l < Block<D>::M; ++l)
    for (int a = 0; a < Block<D>::NC; ++a) {
      const double x = -0.25 + 0.5 * Block<D>::ci(l), y = -0.25 + 0.5 * Block<D>::cj(l),
                   z = -0.25 + 0.5 * Block<D>::ck(l);
      double w = ((a & 1) ? x : 1 - x) * ((a & 2) ? y : 1 - y);
      if (D == 3) w *= (a & 4) ? z : 1 - z;
      t.w[l][a] = w;
    }
  return t;
}
template <int D>
__device__ const CornerWeights<D> g_corner = make_corner_weights<D>();

template <int D, int Q, class T, int V>
__device__ __forceinline__ void interp_rows(const typename Store<T>::R* rc, int t, int c0,
                                            const uint64_t* __restrict__ cellmask,
                                            T* fout,
                                            const uint64_t* __restrict__ solidmask) {
  using S = Store<T>;
  using R = typename S::R;
  constexpr int M = Block<D>::M;
  constexpr int NC = Block<D>::NC;
  constexpr int NR = NC / 2;                 // parent rows of a quadrant
  constexpr unsigned ALL = (1u << V) - 1u;
  const int l0 = V * t, i0 = l0 & 3, J = Block<D>::cj(l0), K = Block<D>::ck(l0);
  const R x = R(-0.25) + R(0.5) * R(i0);     // of the thread's first cell
  const R y = R(-0.25) + R(0.5) * R(J);
  const R z = R(-0.25) + R(0.5) * R(K);
  R wr[NR], wc[V == 1 ? NC : 1];
  if constexpr (V == 1) {
#pragma unroll
    for (int a = 0; a < NC; ++a) wc[a] = R(__ldg(&g_corner<D>.w[l0][a]));
  } else {
#pragma unroll
    for (int a = 0; a < NR; ++a) {
      wr[a] = (a & 1) ? y : R(1) - y;
      if (D == 3) wr[a] *= (a & 2) ? z : R(1) - z;
    }
  }
#pragma unroll 1
  for (int c = 0; c < NC; ++c) {
    const int ch = c0 + c;
    unsigned gm = (unsigned)(__ldg(cellmask + 2 * (size_t)ch) >> l0) & ALL;
    if (gm && solidmask) gm &= ~((unsigned)(__ldg(solidmask + ch) >> l0));
    if (!gm) continue;
    const int qx = c & 1, qy = (c >> 1) & 1, qz = (c >> 2) & 1;
    const R* q = rc + Block<D>::cell(2 * qx, 2 * qy, 2 * qz);
    T* own = fout + (size_t)ch * (Q * M) + l0;
    static_for<0, Q>([&](auto P) {
      R a0 = R(0), a1 = R(0);
      Vec<T, V> o;
#pragma unroll
      for (int a = 0; a < NR; ++a) {
        const Vec<R, 2> v = *reinterpret_cast<const Vec<R, 2>*>(
            q + P * M + Block<D>::cell(0, a & 1, a >> 1));
        if constexpr (V == 1) {
          a0 += wc[2 * a] * v.v[0];
          a0 += wc[2 * a + 1] * v.v[1];
        } else {
          a0 += wr[a] * v.v[0];
          a1 += wr[a] * v.v[1];
        }
      }
      if constexpr (V == 1) {
        o.v[0] = S::from_raw(a0);
      } else {
        const R slope = a1 - a0;
#pragma unroll
        for (int i = 0; i < V; ++i)
          o.v[i] = S::from_raw(fma_(x + R(0.5) * R(i), slope, a0));
      }
      if (gm == ALL) {
        *reinterpret_cast<Vec<T, V>*>(own + P * M) = o;
      } else {
#pragma unroll
        for (int i = 0; i < V; ++i)
          if ((gm >> i) & 1u) own[P * M + i] = o.v[i];
      }
    });
  }
}

// ================================================= fused collide + stream
// The list's blocks in tree order.  GHOST_IN (the first of the two substeps of
// a level below the coarsest): the coarse-to-fine interpolation of the level
// step (Section 4.1) wrote the pre-collision values of this level's ghost
// cells into their own slots of the output buffer (a direct write, see
// LbmOps::interp); the ghost cells read them there instead of gathering, and
// overwrite them with their post-collision values.  `cellmask`: [2 b] the
// ghost cells of block b.
// XCHG: the level has exchanging parents (see Exchange): the coarse-to-fine
// interpolation of the level step fused into the parent level's
// collide-stream.  A refined block has every same-level neighbour, so a
// parent never holds ghost cells.

// One thread per V cells of an x-row (row_cells).  The threads of a block lie
// in one warp, so staging its neighbour row, and handing a parent's rescaled
// cells to its children's interpolation, need no CTA barrier.  With one cell
// per thread in 3D a block takes two warps: each stages the row for itself, and
// the CTA, which then holds one block, meets before the interpolation.
template <int D, int Q, class T, bool SOLID, int V, int THREADS, int MIN_CTAS, bool GHOST_IN,
          bool XCHG>
__global__ void __launch_bounds__(THREADS, MIN_CTAS)
    k_collide_stream(const int32_t* __restrict__ list, int n, const T* gin,
                     T* gout, const int32_t* __restrict__ nbr,
                     const uint64_t* __restrict__ solidmask,
                     const __grid_constant__ StepParams prm,
                     const uint64_t* __restrict__ cellmask, const __grid_constant__ Exchange ex) {
  using R = typename Store<T>::R;
  constexpr int M = Block<D>::M;
  constexpr int TPB = M / V;                // threads of a block
  constexpr int LPR = TPB < 32 ? TPB : 32;  // lanes that share a staged row
  constexpr int NCODE = D == 2 ? 9 : 27;
  constexpr int BPC = THREADS / TPB, RPC = THREADS / LPR;
  static_assert(THREADS % 32 == 0 && (32 % TPB == 0 || THREADS == TPB || !XCHG),
                "the threads of an exchanging parent lie in one warp or fill the CTA");
  __shared__ int32_t s_nb[RPC][NCODE];
  __shared__ uint64_t s_sm[SOLID ? RPC : 1][SOLID ? NCODE : 1];
  __shared__ __align__(16) R s_rc[XCHG ? BPC : 1][XCHG ? Q * M : 1];   // rescaled parent cells

  chain_start();
  const int slot = threadIdx.x / TPB, row = threadIdx.x / LPR;
  const int t = threadIdx.x % TPB;
  const int bi = blockIdx.x * BPC + slot;
  if (bi >= n) {                           // (the same for the threads of a block)
    chain_wait();
    return;
  }
  const unsigned lanes = block_lanes<LPR>();
  const int b = __ldg(list + bi);
  uint64_t ghost = 0ull;
  if constexpr (GHOST_IN) ghost = __ldg(cellmask + 2 * (size_t)b);
  int c0 = NONE;
  if constexpr (XCHG) c0 = __ldg(ex.child0 + b);
  const int flags = stage_block<D, LPR, SOLID>(s_nb[row], SOLID ? s_sm[row] : nullptr, b, t % LPR,
                                               lanes, nbr, solidmask, &prm.faces);
  chain_wait();
  ParentOut<R> par{nullptr, R(0)};
  if constexpr (XCHG) par = {c0 >= 0 ? s_rc[slot] : nullptr, ex.keep<R>()};
  step_row<D, Q, T, V, SOLID, GHOST_IN, XCHG, false>(gin, gout, b, t, s_nb[row],
                                                     SOLID ? s_sm[row] : nullptr, flags, ghost,
                                                     prm.rate<R>(), prm.faces, par);
  if constexpr (XCHG) {
    if (c0 >= 0) {
      if constexpr (TPB > 32) __syncthreads();   // (one block: the same for the CTA)
      else __syncwarp(lanes);
      interp_rows<D, Q, T, V>(s_rc[slot], t, c0, ex.cellmask, (T*)ex.fine_out, solidmask);
    }
  }
}

}  // namespace amr
