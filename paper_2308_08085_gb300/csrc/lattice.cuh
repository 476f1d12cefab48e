// Compile-time velocity sets, storage traits and block/cell geometry shared
// by the LBM kernels.  Numbering follows the paper's velocity-set figure
// (Section 2); weights are the standard Gauss-Hermite weights by speed shell.
#pragma once
#include <cstdint>
#include <type_traits>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

namespace amr {

constexpr int NONE = -1;
constexpr int NBR_STRIDE = 32;   // int32 slots per block row of the nbr table

// ------------------------------------------------- chained kernel launches
// The launches of a captured coarse step depend on one another in a chain.  A
// kernel launched as a programmatic dependent starts when every CTA of its
// predecessor has started; what it reads before chain_wait() is only what no
// kernel of the step writes (lists, neighbour rows, masks), and chain_wait()
// returns when the predecessor has finished (which waited for its own).  Both
// are no-ops in other launches.  A 2D coarse step is 10 to 22 launches of a few
// microseconds: the start of a launch and its first loads overlap the end of
// the one before (20 coarse steps of the 128^2 FP32 cavity 1.91 -> 1.61 ms, of
// the 64^2 FP64 cavity 1.57 -> 1.45).
//
// A dependent kernel is resident while its predecessor writes populations.
// `const __restrict__` would promise the compiler that nobody writes them
// during the kernel: it could read them through the read-only path or move the
// loads above the wait, which clobbers only memory that others may reach.  The
// population pointers of a kernel that calls chain_wait(), and of what it
// calls, are therefore plain; lists, rows, masks and tables keep the promise.
__device__ __forceinline__ void chain_start() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ----------------------------------------------------------- static loops
template <int B, int E, class F>
__host__ __device__ __forceinline__ void static_for(F&& f) {
  if constexpr (B < E) {
    f(std::integral_constant<int, B>{});
    static_for<B + 1, E>(f);
  }
}

// ----------------------------------------------------------- velocity sets
template <int D, int Q> struct VS;

template <> struct VS<2, 9> {
  static constexpr int cx[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
  static constexpr int cy[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
  static constexpr int cz[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
  static constexpr int opp[9] = {0, 3, 4, 1, 2, 7, 8, 5, 6};
  static constexpr double w[9] = {4.0 / 9, 1.0 / 9, 1.0 / 9, 1.0 / 9, 1.0 / 9,
                                  1.0 / 36, 1.0 / 36, 1.0 / 36, 1.0 / 36};
};

#define AMR_D3_CX 0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 0, 0, 1, -1, 1, -1, 0, 0
#define AMR_D3_CY 0, 0, 0, 1, -1, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 1, -1
#define AMR_D3_CZ 0, 0, 0, 0, 0, 1, -1, 0, 0, 1, -1, 1, -1, 0, 0, -1, 1, -1, 1
#define AMR_D3_OPP 0, 2, 1, 4, 3, 6, 5, 8, 7, 10, 9, 12, 11, 14, 13, 16, 15, 18, 17

template <> struct VS<3, 19> {
  static constexpr int cx[19] = {AMR_D3_CX};
  static constexpr int cy[19] = {AMR_D3_CY};
  static constexpr int cz[19] = {AMR_D3_CZ};
  static constexpr int opp[19] = {AMR_D3_OPP};
  static constexpr double w[19] = {1.0 / 3,  1.0 / 18, 1.0 / 18, 1.0 / 18, 1.0 / 18,
                                   1.0 / 18, 1.0 / 18, 1.0 / 36, 1.0 / 36, 1.0 / 36,
                                   1.0 / 36, 1.0 / 36, 1.0 / 36, 1.0 / 36, 1.0 / 36,
                                   1.0 / 36, 1.0 / 36, 1.0 / 36, 1.0 / 36};
};

template <> struct VS<3, 27> {
  static constexpr int cx[27] = {AMR_D3_CX, 1, -1, 1, -1, 1, -1, -1, 1};
  static constexpr int cy[27] = {AMR_D3_CY, 1, -1, 1, -1, -1, 1, 1, -1};
  static constexpr int cz[27] = {AMR_D3_CZ, 1, -1, -1, 1, 1, -1, 1, -1};
  static constexpr int opp[27] = {AMR_D3_OPP, 20, 19, 22, 21, 24, 23, 26, 25};
  static constexpr double w[27] = {
      8.0 / 27,  2.0 / 27,  2.0 / 27,  2.0 / 27,  2.0 / 27,  2.0 / 27,  2.0 / 27,
      1.0 / 54,  1.0 / 54,  1.0 / 54,  1.0 / 54,  1.0 / 54,  1.0 / 54,  1.0 / 54,
      1.0 / 54,  1.0 / 54,  1.0 / 54,  1.0 / 54,  1.0 / 54,  1.0 / 216, 1.0 / 216,
      1.0 / 216, 1.0 / 216, 1.0 / 216, 1.0 / 216, 1.0 / 216, 1.0 / 216};
};

// Block-neighbour numbering: D2Q9 in 2D, D3Q27 in 3D.  dir_of(sx,sy,sz)
// returns the index of the direction (sx,sy,sz) in {-1,0,1}^D.
template <int D> struct Nbr {
  static constexpr int K = D == 2 ? 9 : 27;
  using V = std::conditional_t<D == 2, VS<2, 9>, VS<3, 27>>;
  static constexpr int dir_of(int sx, int sy, int sz) {
    for (int k = 0; k < K; ++k)
      if (V::cx[k] == sx && V::cy[k] == sy && V::cz[k] == sz) return k;
    return -1;
  }
};

// ------------------------------------------------------------ block geometry
template <int D> struct Block {
  static constexpr int M = D == 2 ? 16 : 64;
  static constexpr int NC = D == 2 ? 4 : 8;
  __host__ __device__ static constexpr int ci(int l) { return l & 3; }
  __host__ __device__ static constexpr int cj(int l) { return (l >> 2) & 3; }
  __host__ __device__ static constexpr int ck(int l) { return D == 2 ? 0 : (l >> 4); }
  __host__ __device__ static constexpr int cell(int i, int j, int k) {
    return i + 4 * j + (D == 2 ? 0 : 16 * k);
  }
};

// ---------------------------------------------------------- storage traits
// Values are stored either as the population itself (FP64, FP32) or as the
// shifted value f - w_p in BF16 / FP16, rounded to nearest even.
template <class T> struct Store;
template <> struct Store<double> {
  using R = double;
  static constexpr bool kShifted = false;
  __device__ static R raw(double v) { return v; }
  __device__ static double from_raw(R v) { return v; }
  template <int D, int Q, int P> __device__ static R load(double v) { return v; }
  template <int D, int Q, int P> __device__ static double save(R v) { return v; }
};
template <> struct Store<float> {
  using R = float;
  static constexpr bool kShifted = false;
  __device__ static R raw(float v) { return v; }
  __device__ static float from_raw(R v) { return v; }
  template <int D, int Q, int P> __device__ static R load(float v) { return v; }
  template <int D, int Q, int P> __device__ static float save(R v) { return v; }
};
template <> struct Store<__nv_bfloat16> {
  using R = float;
  static constexpr bool kShifted = true;   // holds f - w_p
  __device__ static R raw(__nv_bfloat16 v) { return __bfloat162float(v); }
  __device__ static __nv_bfloat16 from_raw(R v) { return __float2bfloat16_rn(v); }
  template <int D, int Q, int P> __device__ static R load(__nv_bfloat16 v) {
    constexpr float wp = float(VS<D, Q>::w[P]);
    return __bfloat162float(v) + wp;
  }
  template <int D, int Q, int P> __device__ static __nv_bfloat16 save(R v) {
    constexpr float wp = float(VS<D, Q>::w[P]);
    return __float2bfloat16_rn(v - wp);
  }
};
template <> struct Store<__half> {
  using R = float;
  static constexpr bool kShifted = true;   // holds f - w_p
  __device__ static R raw(__half v) { return __half2float(v); }
  __device__ static __half from_raw(R v) { return __float2half_rn(v); }
  template <int D, int Q, int P> __device__ static R load(__half v) {
    constexpr float wp = float(VS<D, Q>::w[P]);
    return __half2float(v) + wp;
  }
  template <int D, int Q, int P> __device__ static __half save(R v) {
    constexpr float wp = float(VS<D, Q>::w[P]);
    return __float2half_rn(v - wp);
  }
};

// ------------------------------------------------------- BGK building blocks
template <int D, int Q, class R>
__device__ __forceinline__ void moments(const R* f, R& rho, R& ux, R& uy, R& uz) {
  using V = VS<D, Q>;
  R r = 0, jx = 0, jy = 0, jz = 0;
  static_for<0, Q>([&](auto P) {
    constexpr int p = P;
    constexpr int cx = V::cx[p], cy = V::cy[p], cz = V::cz[p];
    r += f[p];
    if constexpr (cx != 0) jx += cx > 0 ? f[p] : -f[p];
    if constexpr (cy != 0) jy += cy > 0 ? f[p] : -f[p];
    if constexpr (cz != 0) jz += cz > 0 ? f[p] : -f[p];
  });
  rho = r;
  R inv = R(1) / r;
  ux = jx * inv;
  uy = jy * inv;
  uz = D == 3 ? jz * inv : R(0);
}

template <int D, int Q, int P, class R>
__device__ __forceinline__ R feq(R rho, R ux, R uy, R uz, R usq15) {
  using V = VS<D, Q>;
  constexpr int cx = V::cx[P], cy = V::cy[P], cz = V::cz[P];
  R cu = R(0);
  if constexpr (cx != 0) cu += cx > 0 ? ux : -ux;
  if constexpr (cy != 0) cu += cy > 0 ? uy : -uy;
  if constexpr (cz != 0) cu += cz > 0 ? uz : -uz;
  constexpr double wp = V::w[P];
  return R(wp) * rho * (R(1) + R(3) * cu + R(4.5) * cu * cu - usq15);
}

}  // namespace amr
