// Yamamoto power-spectrum multipoles from the m >= 0 spherical-harmonic weighted transforms.
//
// Each S_l^m(k) = sum_x F(x) Y_l^m(xhat) e^{-ik.x} with m >= 0 (Eq. key1) is the transform of the
// complex field F Y_l^m = F ReY + i F ImY; we transform its two real parts, A = FFT[F ReY] and
// B = FFT[F ImY], so S_l^m = A + iB and, by the conjugation symmetry the paper exploits (Eq.
// F_lm_SIC), S_l^{-m}(k) = (-1)^m [A(k) - iB(k)].  Summing over m (Eq. hand) then gives, with
// real coefficients only,
//   F_l(k) = 4 pi/(2l+1) [ Y_l0(khat) A_l0 + 2 sum_{m>=1} (ReY_lm(khat) A_lm + ImY_lm(khat) B_lm) ],
// which is Hermitian for even l: F_l is the space-inverted 1/2[G_l(k) + G_l^*(-k)] of Eq.
// F_and_new_G obtained directly, and Re<F_0 G_l^*> = <F_0 F_l^*> (Eq. pk_final).  All fields are
// real, so only the half spectrum kz in [0, n/2) is computed and stored (Nyquist planes are
// excluded from every bin) and every stored mode also stands for -k.
//
// Passes (3D transform by axes, shared-memory Stockham stages):
//   k_fwd_z           reads the painted meshes and transforms, per (phase, l, m), the real signal
//                     F(z) Q_lm(uz) r^-m of each column along z (phase a at grid points origin + jH,
//                     phase b at origin + (j - 1/2)H), two signals per complex transform.
//   k_fft_cols_weighted  multiplies by the real and imaginary part of the column factor
//                     (px + i py)^m and transforms both along y (k_fft_cols: without factors).
//   k_fft_x_contract  transforms every field's x-row of one (ky, kz), one row per thread group, then per
//                     mode: interlacing 1/2[A_a + e^{iH(kx+ky+kz)/2} A_b], division by W(k) (Eq.
//                     compensation), F_l assembly, Re[F_0 F_l^*] and Re[F_l F_l'^*] (Eq. Pllp), binned
//                     in float64 with a warp-segmented reduction into per-warp partial sums (no atomics
//                     between warps, fixed order: reproducible run to run).
//   k_power_finalize  fixed-order sum of the partials, normalisation (2l+1)/I22, shot noise,
//                     the modified multipoles of Eq. Plnew.
#include <cmath>

#include "fft_core.cuh"

namespace {

// 1/sqrt(a) for the direction of a mode: the hardware approximation errs to one side, and P_4b and P_8b are
// small differences of sums that all scale with the length of khat (to the powers 2 and 4); one Newton step
// brought their errors from 1.7e-6 and 4.9e-6 to 1.0e-6 and 0.9e-6 (256^3, mean over eight catalogues).
__device__ __forceinline__ float rsqrt_unbiased(float a) {
  const float y = rsqrt(a);
  return fmaf(0.5f * y, fmaf(-a * y, y, 1.0f), y);
}
__device__ __forceinline__ double rsqrt_unbiased(double a) { return rsqrt(a); }

constexpr int CONTRACT_THREADS = 256;
constexpr int MAX_PRODS = 8;              // P_0 .. P_4 and P_22, P_42, P_44
constexpr int MAX_SUMS = MAX_PRODS + 2;   // and the modes and their |k|

template <int N> struct ColCfg {
  static constexpr int TX = N >= 1024 ? 4 : (N >= 512 ? 8 : 16);  // TX <= N
  static constexpr int THREADS = TX * N / 8;
};

// First pass for a single unweighted real field (global line of sight without interlacing, mesh
// gradients): two neighbouring x columns share one complex transform, c = F(x) + i F(x+1), and
// their half spectra follow from c(kz) and conj c(N - kz).  grid = (N / (2 TX), N).
template <int N> struct SingleCfg {   // column pairs per CTA: 2 TX divides N, TX <= the z-pass TX
  static constexpr int TX = (ColCfg<N>::TX >= 16 && N % 32 == 0) ? 16
                          : (ColCfg<N>::TX >= 8 && N % 16 == 0) ? 8 : 4;
  static constexpr int THREADS = TX * N / 8;
};

// The two columns' values are neighbours in memory: one 8-byte load when the mesh is aligned to it (VEC).
template <typename T, int N, bool VEC>
__global__ void __launch_bounds__(SingleCfg<N>::THREADS, 1)
k_fwd_z_single(const T* __restrict__ mesh, cplx<T>* __restrict__ half, const cplx<T>* __restrict__ tw_g, int KZ) {
  using C = cplx<T>;
  constexpr int TX = SingleCfg<N>::TX;
  constexpr int TPF = N / 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* work = tw + N;
  const int tid = threadIdx.x;
  const int c = tid % TX, t = tid / TX;
  const int x0 = blockIdx.x * 2 * TX, y = blockIdx.y;
  for (int i = tid; i < N; i += blockDim.x) tw[i] = tw_g[i];
  C v[8];
  const T* col = mesh + (size_t)y * N + x0 + 2 * c;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const size_t zoff = (size_t)(t + q * TPF) * N * N;
    if constexpr (VEC) v[q] = *reinterpret_cast<const C*>(col + zoff);
    else v[q] = cmk(col[zoff], col[zoff + 1]);
  }
  __syncthreads();
  fft_block<N, -1>(v, t, tw, ColPadView<C, TX, true>{work + c});
#pragma unroll
  for (int q = 0; q < 8; ++q) work[(t + q * TPF) * TX + c] = v[q];
  __syncthreads();
  for (int i = tid; i < KZ * TX; i += blockDim.x) {
    const int kz = i / TX, cc = i % TX;
    const C z1 = work[kz * TX + cc];
    const C z2 = cconj(work[((N - kz) % N) * TX + cc]);
    const C a = cscale(cadd(z1, z2), T(0.5));
    const C d = csub(z1, z2);
    const C b = cmk(T(0.5) * d.y, T(-0.5) * d.x);
    C* dst = half + ((size_t)kz * N + y) * N + x0 + 2 * cc;
    dst[0] = a;
    dst[1] = b;
  }
}

// Polynomial factor Q_lm(uz) of Y_lm = norm_lm Q_lm(uz) (ux + i uy)^m, l <= 4: the associated
// Legendre function with its (-1)^m phase, divided by sin^m(theta).
template <typename T, int L, int M>
__device__ __forceinline__ T ylm_q(T uz) {
  const T z2 = uz * uz;
  if constexpr (L == 0) return T(1);
  else if constexpr (L == 1 && M == 0) return uz;
  else if constexpr (L == 1 && M == 1) return T(-1);
  else if constexpr (L == 3 && M == 0) return T(0.5) * uz * (T(5) * z2 - T(3));
  else if constexpr (L == 3 && M == 1) return T(-1.5) * (T(5) * z2 - T(1));
  else if constexpr (L == 3 && M == 2) return T(15) * uz;
  else if constexpr (L == 3 && M == 3) return T(-15);
  else if constexpr (L == 2 && M == 0) return T(1.5) * z2 - T(0.5);
  else if constexpr (L == 2 && M == 1) return T(-3) * uz;
  else if constexpr (L == 2 && M == 2) return T(3);
  else if constexpr (L == 4 && M == 0) return (T(35) * z2 * z2 - T(30) * z2 + T(3)) * T(0.125);
  else if constexpr (L == 4 && M == 1) return T(-2.5) * uz * (T(7) * z2 - T(3));
  else if constexpr (L == 4 && M == 2) return T(7.5) * (T(7) * z2 - T(1));
  else if constexpr (L == 4 && M == 3) return T(-105) * uz;
  else return T(105);
}

// Keeps a value where it is computed: the per-pair factors below must not be hoisted out of the
// pair loop (every pair's factors would then stay live in registers).
__device__ __forceinline__ void keep_here(float& x) { asm volatile("" : "+f"(x)); }
__device__ __forceinline__ void keep_here(double& x) { asm volatile("" : "+d"(x)); }

// ---------------------------------------------------------------------------------------------
// Weighted first passes.  Y_lm(xhat) = norm Q_lm(uz) ((px + i py)/r)^m splits into a real signal along z,
// s(z) = mesh(z) Q_lm(uz) r^-m, and the column factor norm (px + i py)^m, constant along z.  So
//   k_fwd_z     transforms the signals of every (phase, l, m), two real signals per complex transform
//               (phases a and b of one harmonic where both exist), and stores one half spectrum S per
//               signal: 18 for l = 0, 2, 4 and two phases, where the parts of Y_lm make 30 real fields;
//   k_fft_cols_weighted  reads S once, multiplies it by the real and by the imaginary part of the column
//               factor and transforms both along y.  S lies in the slot of the imaginary part's field:
//               the CTA that overwrites a column of it has read that column before.
// (With the column factors applied in the first pass the 30 fields were written by it and read by the
// second: at 512^3 16.1 + 28.7 GB instead of 9.7 + 22.3 GB.)
// ---------------------------------------------------------------------------------------------
struct Signal {
  int8_t phase, l, m;
  int8_t re, im;     // fields of the real and of the imaginary part (-1: none; m = 0 has re only)
  __host__ __device__ int slot() const { return im >= 0 ? im : re; }
};
// Two signals that share a complex transform have to be of one magnitude, since each is rounded at the
// larger one's: phases a and b of a harmonic are, and without interlacing two harmonics of one m (r^-m)
// are once they carry their norm.
constexpr int MAX_SIGNALS = 32;   // 2 phases x 15 harmonics, and room to pair them
struct SignalList {
  int n;                          // pairs (2p, 2p + 1); one without a partner has a second with re = im = -1
  int norm_in_signal;             // the norm of Y_lm multiplies s(z), else the column factor
  Signal s[MAX_SIGNALS];
};

// A grid point can lie at the observer up to the rounding of its coordinates, and r^-m and (px + i py)^m can
// then leave the range of float32 while their product cannot.  The coordinates are in units of a power of two
// that makes the largest one about 1, whatever the user's unit of length.  Columns with |px|, |py| < near, a
// power of two of at most half a cell (`near` columns: the one or few at the observer's x and y) take out of
// r^-m a power of two f^m <= 1 that their column factor puts back.  f = 2^floor(log2(max(|px|, |py|))) / near
// comes from the bits of px and py, so both passes form the same one; it is at most r / near, which leaves
// the signal no larger than its neighbours'.  Every other column has r >= near.  Few meshes have near columns,
// and the code for them would cost all others (512^3: z pass 4.51 -> 4.78 ms, y pass 6.00 -> 6.23), so it is
// a variant (NEAR) of the passes that the host launches for meshes with near columns.
__device__ __forceinline__ float pow2_floor(float x) { return __uint_as_float(__float_as_uint(x) & 0x7f800000u); }
__device__ __forceinline__ double pow2_floor(double x) {
  return __longlong_as_double(__double_as_longlong(x) & 0x7ff0000000000000ll);
}
// 1 / pow2_floor(x), finite at x = 0
__device__ __forceinline__ float pow2_inv(float x) {
  return __uint_as_float(0x7f000000u - (__float_as_uint(x) & 0x7f800000u));
}
__device__ __forceinline__ double pow2_inv(double x) {
  return __longlong_as_double(0x7fe0000000000000ll - (__double_as_longlong(x) & 0x7ff0000000000000ll));
}
__device__ __forceinline__ float absmax(float x, float y) { return fmaxf(fabsf(x), fabsf(y)); }
__device__ __forceinline__ double absmax(double x, double y) { return fmax(fabs(x), fabs(y)); }

// s(z) times norm of one signal of a near column, pz from the table (near r = 0 the rounding of a sum would
// turn the direction).  A grid point exactly at the observer has the direction of the z axis.
template <typename T, int N, int TX>
__device__ __forceinline__ void near_signal(T (&sv)[8], int l, int m, const T* tile, int c, int t,
                                            const T* __restrict__ coords, int phase, int x, int y, T near, T norm) {
  constexpr int TPF = N / 8;
  const T px = coords[phase * N + x], py = coords[(2 + phase) * N + y];
  const T own = absmax(px, py);
  T near_sv[8];
#pragma unroll 1
  for (int q = 0; q < 8; ++q) {
    const int z = t + q * TPF;
    const T pz = coords[(4 + phase) * N + z];
    const T scale = pow2_inv(absmax(own, pz));   // the largest coordinate near 1: r^2 cannot underflow
    const T ux = px * scale, uy = py * scale, uz0 = pz * scale;
    const T r2 = ux * ux + uy * uy + uz0 * uz0;
    const T inv = r2 > T(0) ? rsqrt(r2) : T(0);
    const T uz = r2 > T(0) ? uz0 * inv : T(1);
    T v;
#define NPC_Q(L, M) case L * (L + 1) / 2 + M: v = ylm_q<T, L, M>(uz); break;
    switch (l * (l + 1) / 2 + m) {
      NPC_Q(1, 0) NPC_Q(1, 1) NPC_Q(2, 0) NPC_Q(2, 1) NPC_Q(2, 2) NPC_Q(3, 0) NPC_Q(3, 1) NPC_Q(3, 2) NPC_Q(3, 3)
      NPC_Q(4, 0) NPC_Q(4, 1) NPC_Q(4, 2) NPC_Q(4, 3) NPC_Q(4, 4)
      default: v = T(1);
    }
#undef NPC_Q
    v = tile[z * TX + c] * (norm * v);
    for (int j = 0; j < m; ++j) v *= pow2_floor(own) * scale * inv / near;
    near_sv[q] = v;
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) sv[q] = near_sv[q];
}

// s(z) times norm of one signal at the thread's elements z = t + q TPF of a column that is not near
template <typename T, int N, int TX, int L, int M>
__device__ __forceinline__ void column_signal(T (&sv)[8], const T* tile, int c, int t, T pxy2, T pz0, T dz, T norm) {
  constexpr int TPF = N / 8;
  keep_here(pxy2);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const T F = tile[(t + q * TPF) * TX + c];
    if constexpr (L == 0) {
      sv[q] = F;
    } else {
      const T pz = pz0 + T(q) * dz;
      const T r2 = pxy2 + pz * pz;
      const T inv = rsqrt(r2);
      if constexpr (M == 0) {
        sv[q] = F * (norm * ylm_q<T, L, 0>(pz * inv));
      } else {
        T v = F * (norm * ylm_q<T, L, M>(pz * inv));
#pragma unroll
        for (int j = 0; j < M; ++j) v *= inv;
        sv[q] = v;
      }
    }
  }
}

template <typename T, int N, int TX, bool NEAR>
__device__ __forceinline__ void any_signal(T (&sv)[8], const Signal& sg, const T* tileA, const T* tileB, int c, int t,
                                           const T (&pxy2)[2], const T (&pz0)[2], T dz, const YNorm& nrm,
                                           bool norm_in, int near_phases, const T* __restrict__ coords, int x, int y,
                                           T near) {
  const T* tile = sg.phase ? tileB : tileA;
  if (NEAR && (near_phases & (1 << sg.phase))) {
    const int lm = sg.l * (sg.l + 1) / 2 + sg.m;
    near_signal<T, N, TX>(sv, sg.l, sg.m, tile, c, t, coords, sg.phase, x, y, near,
                          sg.l > 0 && (sg.m == 0 || norm_in) ? ynorm<T>(nrm, lm) : T(1));
    return;
  }
  const T p2 = sg.phase ? pxy2[1] : pxy2[0], z0 = sg.phase ? pz0[1] : pz0[0];
#define NPC_S(L, M) \
  case L * (L + 1) / 2 + M: column_signal<T, N, TX, L, M>(sv, tile, c, t, p2, z0, dz, M == 0 || norm_in ? ynorm<T>(nrm, L * (L + 1) / 2 + M) : T(1)); break;
  switch (sg.l * (sg.l + 1) / 2 + sg.m) {
    NPC_S(1, 0) NPC_S(1, 1) NPC_S(2, 0) NPC_S(2, 1) NPC_S(2, 2) NPC_S(3, 0) NPC_S(3, 1) NPC_S(3, 2) NPC_S(3, 3)
    NPC_S(4, 0) NPC_S(4, 1) NPC_S(4, 2) NPC_S(4, 3) NPC_S(4, 4)
    default: column_signal<T, N, TX, 0, 0>(sv, tile, c, t, p2, z0, dz, T(1));
  }
#undef NPC_S
}

// float: occupancy of the register counts this kernel needs (64 at 512 threads, at most 80 otherwise)
template <typename T, int N> constexpr int zpass_min_blocks() {
  return sizeof(T) == 4 ? 65536 / (ColCfg<N>::THREADS * (ColCfg<N>::THREADS == 512 ? 64 : 80)) : 1;
}

// Coordinates of the grid points from the observer times `unit`, tab[axis][phase][n], formed in float64 step
// by step (no fused multiply-add: half a box plus minus half a box is 0) and rounded once; phase b lies half
// a cell lower.  The weighted passes look them up instead of forming them per thread, since float64
// arithmetic is scarce on this part (y pass at 512^3: 10.1 ms with, 6.0 without).
template <typename T>
__global__ void k_axis_coords(const Geom g, double unit, T* __restrict__ tab) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 6 * g.n; i += gridDim.x * blockDim.x) {
    const int a = i / (2 * g.n), ph = (i / g.n) % 2, j = i % g.n;
    const double o = a == 0 ? g.o[0] : (a == 1 ? g.o[1] : g.o[2]);
    const double obs = a == 0 ? g.obs[0] : (a == 1 ? g.obs[1] : g.obs[2]);
    tab[i] = (T)((__dadd_rn(o, __dmul_rn((double)j - (ph ? 0.5 : 0.0), g.h)) - obs) * unit);
  }
}

// First pass: the signals' half spectra along z, S[slot][kz][y][x].  Bound by instruction issue (256^3: 61 % of
// the slots, DRAM 32 %) with two CTAs of 512 threads per SM; 512^3, l = 0, 2, 4 and two phases: 4.51 ms for 10.7
// GB (6.2 ms when it formed and wrote the 30 fields).
template <typename T, int N, bool NEAR>
__global__ void __launch_bounds__(ColCfg<N>::THREADS, zpass_min_blocks<T, N>())
k_fwd_z(const T* __restrict__ mesh_a, const T* __restrict__ mesh_b, cplx<T>* __restrict__ half,
        const __grid_constant__ SignalList sl, const T* __restrict__ coords, const T dz, const T near, const YNorm nrm,
        const cplx<T>* __restrict__ tw_g, int KZ) {
  using C = cplx<T>;
  constexpr int TX = ColCfg<N>::TX;
  constexpr int TPF = N / 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* work = tw + N;
  T* tileA = reinterpret_cast<T*>(work + col_rows<N, TX>() * TX);
  T* tileB = mesh_b ? tileA + N * TX : tileA;
  const int tid = threadIdx.x;
  const int c = tid % TX, t = tid / TX;
  const int x0 = blockIdx.x * TX, y = blockIdx.y;
  for (int i = tid; i < N; i += blockDim.x) tw[i] = tw_g[i];
  for (int i = tid; i < N * TX; i += blockDim.x) {
    const int z = i / TX, cc = i % TX;
    const size_t gi = ((size_t)z * N + y) * N + x0 + cc;
    tileA[i] = mesh_a[gi];
    if (mesh_b) tileB[i] = mesh_b[gi];
  }
  T pxy2[2] = {T(0), T(0)}, pz0[2] = {T(0), T(0)};
  int near_phases = 0;
  if (coords) {
#pragma unroll
    for (int ph = 0; ph < 2; ++ph) {
      const T px = coords[ph * N + x0 + c], py = coords[(2 + ph) * N + y];
      pxy2[ph] = px * px + py * py;
      pz0[ph] = coords[(4 + ph) * N + t];
      if (NEAR) near_phases |= absmax(px, py) < near ? 1 << ph : 0;
    }
  }
  __syncthreads();
  const size_t fstride = (size_t)KZ * N * N;
#pragma unroll 1
  for (int p = 0; p < sl.n; p += 2) {
    const Signal s0 = sl.s[p], s1 = sl.s[p + 1];
    C v[8];
    {
      T a[8], b[8];
      any_signal<T, N, TX, NEAR>(a, s0, tileA, tileB, c, t, pxy2, pz0, dz, nrm, sl.norm_in_signal, near_phases, coords,
                                 x0 + c, y, near);
      if (s1.re >= 0) {
        any_signal<T, N, TX, NEAR>(b, s1, tileA, tileB, c, t, pxy2, pz0, dz, nrm, sl.norm_in_signal, near_phases,
                                   coords, x0 + c, y, near);
      } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) b[q] = T(0);
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = cmk(a[q], b[q]);
    }
    fft_block<N, -1>(v, t, tw, ColPadView<C, TX, true>{work + c});
#pragma unroll
    for (int q = 0; q < 8; ++q) work[(t + q * TPF) * TX + c] = v[q];
    __syncthreads();
    // split the packed pair, S_0 = (Z(k) + Z(N - k)^*) / 2 and S_1 = (Z(k) - Z(N - k)^*) / 2i; thread tid
    // owns (kz0 + j KZSTEP, c)
    {
      constexpr int KZSTEP = ColCfg<N>::THREADS / TX;
      const size_t row0 = ((size_t)t * N + y) * N + x0 + c;
      C* o0 = half + (size_t)s0.slot() * fstride + row0;
      C* o1 = half + (size_t)(s1.re >= 0 ? s1.slot() : 0) * fstride + row0;
      for (int kz = t; kz < KZ; kz += KZSTEP, o0 += (size_t)KZSTEP * N * N, o1 += (size_t)KZSTEP * N * N) {
        const C z1 = work[kz * TX + c];
        const C z2 = cconj(work[(kz == 0 ? 0 : N - kz) * TX + c]);
        *o0 = cscale(cadd(z1, z2), T(0.5));
        const C d = csub(z1, z2);
        if (s1.re >= 0) *o1 = cmk(T(0.5) * d.y, T(-0.5) * d.x);
      }
    }
    __syncthreads();
  }
}

// The signals of a field list: phases a and b of one harmonic paired, the others two of one m.
static SignalList make_signals(const FieldList& fl) {
  std::vector<Signal> all;
  for (int f = 0; f < fl.nf; ++f) {
    const Comp c = fl.f[f];
    const bool one = c.part == PART_ONE;
    Signal* s = nullptr;
    for (Signal& x : all)
      if (x.phase == c.phase && x.l == (one ? 0 : c.ell) && x.m == (one ? 0 : c.m)) s = &x;
    if (!s) {
      all.push_back(Signal{c.phase, (int8_t)(one ? 0 : c.ell), (int8_t)(one ? 0 : c.m), -1, -1});
      s = &all.back();
    }
    (c.part == PART_IM ? s->im : s->re) = (int8_t)f;
  }
  SignalList sl{};
  std::vector<Signal> rest;
  for (const Signal& a : all) {
    if (a.phase) continue;
    const Signal* b = nullptr;
    for (const Signal& x : all)
      if (x.phase && x.l == a.l && x.m == a.m) b = &x;
    if (b) {
      sl.s[sl.n++] = a;
      sl.s[sl.n++] = *b;
    } else {
      rest.push_back(a);
    }
  }
  sl.norm_in_signal = rest.empty() ? 0 : 1;
  for (int m = 0; m <= 4; ++m) {
    for (const Signal& x : rest)
      if (x.m == m) sl.s[sl.n++] = x;
    if (sl.n % 2) sl.s[sl.n++] = Signal{0, 0, 0, -1, -1};
  }
  return sl;
}

// v = S norm Re (px + i py)^M and keep = S norm Im (px + i py)^M at the thread's elements
template <typename T, int N, int TX, int M, bool NEAR>
__device__ __forceinline__ void column_factors(cplx<T> (&v)[8], cplx<T>* keep, const T* __restrict__ pys, T px, T near,
                                               T norm, int c, int t) {
  constexpr int TPF = N / 8;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    T fx = px, fy = pys[t + q * TPF];
    const T own = absmax(fx, fy);
    if (NEAR && own < near) {
      const T back = near * pow2_inv(own);
      fx *= back;
      fy *= back;
    }
    T cr = norm, ci = T(0);
#pragma unroll
    for (int j = 0; j < M; ++j) {
      const T nr = cr * fx - ci * fy;
      ci = cr * fy + ci * fx;
      cr = nr;
    }
    keep[(t + q * TPF) * TX + c] = cscale(v[q], ci);
    v[q] = cscale(v[q], cr);
  }
}

// y pass with the column factors: plane (signal, kz) = blockIdx.y; the transforms of S times the
// real and the imaginary part of norm (px + i py)^m go to the two parts' fields (m = 0: S itself, in place).
// Bound by HBM and the exchanges' barriers (256^3: DRAM and issue 57 % each, three CTAs of 512 threads per SM);
// 512^3: 6.0 ms for 22.3 GB (6.2 ms for the plain pass over 30 fields).
template <typename T, int N, int TX, bool NEAR>
__global__ void __launch_bounds__(TX * N / 8, (sizeof(T) == 4 && TX * N / 8 <= 512 ? 1536 / (TX * N / 8) : 1))
k_fft_cols_weighted(cplx<T>* __restrict__ half, const __grid_constant__ SignalList sl, const T* __restrict__ coords,
                    const T near, const YNorm nrm, const cplx<T>* __restrict__ tw_g, int KZ, int row_n2max) {
  using C = cplx<T>;
  constexpr int TPF = N / 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* work = tw + N;
  C* keep = work + col_rows<N, TX>() * TX;   // the imaginary part's elements, each thread its own
  const int tid = threadIdx.x;
  const int c = tid % TX, t = tid / TX;
  const int plane = blockIdx.y, kz = plane % KZ;
  const Signal sg = sl.s[plane / KZ];
  if (sg.re < 0) return;
  const int x = blockIdx.x * TX + c;
  const size_t fstride = (size_t)KZ * N * N, poff = (size_t)kz * N * N + x;
  for (int i = tid; i < N; i += blockDim.x) tw[i] = tw_g[i];
  C v[8];
  {
    const C* src = half + (size_t)sg.slot() * fstride + poff;
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = src[(size_t)(t + q * TPF) * N];
  }
  if (sg.m > 0) {
    const T px = coords[sg.phase * N + x];
    const T* __restrict__ pys = coords + (2 + sg.phase) * N;
    const T norm = sl.norm_in_signal ? T(1) : ynorm<T>(nrm, sg.l * (sg.l + 1) / 2 + sg.m);
    switch (sg.m) {
      case 1: column_factors<T, N, TX, 1, NEAR>(v, keep, pys, px, near, norm, c, t); break;
      case 2: column_factors<T, N, TX, 2, NEAR>(v, keep, pys, px, near, norm, c, t); break;
      case 3: column_factors<T, N, TX, 3, NEAR>(v, keep, pys, px, near, norm, c, t); break;
      default: column_factors<T, N, TX, 4, NEAR>(v, keep, pys, px, near, norm, c, t);
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int part = 0; part < 2; ++part) {
    const int f = part ? sg.im : sg.re;
    if (f < 0) continue;
    if (part) {
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = keep[(t + q * TPF) * TX + c];
    }
    fft_block<N, -1>(v, t, tw, ColPadView<C, TX, false>{work + c});
    // rows (ky, kz) outside every k-bin are never read again: not stored
    C* dst = half + (size_t)f * fstride + poff;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int yi = t + q * TPF;
      const int jy = yi < N / 2 ? yi : yi - N;
      if (jy * jy + kz * kz <= row_n2max) dst[(size_t)yi * N] = v[q];
    }
  }
}

// Column transform along a strided axis: element j of column (plane, x) at
// data[plane*plane_stride + j*row_stride + x].  grid = (N/TX, nplanes); TX columns per CTA is a
// tuning parameter (see tune_y_pass).
template <typename T, int N, int DIR, int TX>
__global__ void __launch_bounds__(TX * N / 8, (TX * N / 8 <= 512 ? 1536 / (TX * N / 8) : 1))
k_fft_cols(cplx<T>* __restrict__ data, size_t plane_stride, int row_stride, const cplx<T>* __restrict__ tw_g,
           int plane0, int kz_planes, int row_n2max) {
  using C = cplx<T>;
  constexpr int TPF = N / 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* work = tw + N;
  const int tid = threadIdx.x;
  const int c = tid % TX, t = tid / TX;
  for (int i = tid; i < N; i += blockDim.x) tw[i] = tw_g[i];
  C* base = data + (size_t)blockIdx.y * plane_stride + blockIdx.x * TX + c;
  C v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = base[(size_t)(t + q * TPF) * row_stride];
  __syncthreads();
  fft_block<N, DIR>(v, t, tw, ColView<C>{work + c, TX});
  // rows (ky, kz) outside every k-bin are never read again: not stored (plane p holds kz = p % kz_planes)
  const int kz = (plane0 + (int)blockIdx.y) % kz_planes;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int yi = t + q * TPF;
    const int jy = yi < N / 2 ? yi : yi - N;
    if (jy * jy + kz * kz <= row_n2max) base[(size_t)yi * row_stride] = v[q];
  }
}

// One step of the x pass: a stored real field, its k-space coefficient scale * part of Q_lm(uz)
// (ux + i uy)^m, and what follows it.  scale = 4 pi/(2l+1) * (m > 0 ? 2 : 1) * norm_lm^2 = 2 (l-m)!/(l+m)!
// (m > 0) over the norm that the first passes applied, in the value it had there.  A rounding of scale
// would be common to all modes, and P_4 is a small difference of large terms of different m, so the float
// coefficient is a product of two factors chosen to match it to about 2^-36; the products round per mode.
struct FieldStep {
  int8_t field;  // index into the half-spectrum buffer
  int8_t weight; // 2 (l(l+1)/2 + m) + (1 for the imaginary part); 0: no weight (F_0, global line of sight)
  int8_t acc;    // accumulator of the step's multipole
  int8_t flags;  // STEP_ROTATE, STEP_STORE
  float scale_f[2];
  double scale_d;
};
// the accumulator holds phase b only so far: apply the interlacing phase e^{i pi (i + j + l)/N}
constexpr int8_t STEP_ROTATE = 1;
// the accumulator's last field: apply the window factor and store F_l
constexpr int8_t STEP_STORE = 2;
__device__ __forceinline__ float scaled(const FieldStep& c, float w) { return c.scale_f[1] * (c.scale_f[0] * w); }
__device__ __forceinline__ double scaled(const FieldStep& c, double w) { return c.scale_d * w; }

// factors f[0] f[1] = w to about 2^-36
static void split_scale(double w, float (&f)[2]) {
  double best = 1e300;
  for (int k = 0; k < 4096; ++k) {
    const float a = 1.0f + (float)k * 1.1920929e-07f, b = (float)(w / (double)a);
    const double e = std::fabs((double)a * (double)b - w);
    if (e < best) {
      best = e;
      f[0] = a;
      f[1] = b;
    }
  }
}

// The scales of all harmonics, entry l(l+1)/2 + m, for both types.  They depend on (l, m) only and are formed
// once per process: searched for in every call, 8 us per weighted field, they delayed the x pass of small
// meshes (16^3, l = 0..4: 537 us a call, of which 20 more fields than l = 0, 2, 4 took 163).
struct HarmonicScales {
  float f[15][2];
  double d[15];
  HarmonicScales() {
    const YNorm nrm = ylm_norm_table();
    for (int l = 0; l <= 4; ++l)
      for (int m = 0; m <= l; ++m) {
        const int lm = l * (l + 1) / 2 + m;
        const double w = 4.0 * M_PI / (2 * l + 1) * (m > 0 ? 2.0 : 1.0) * nrm.v[lm] * nrm.v[lm];
        split_scale(w / (double)nrm.f[lm], f[lm]);   // over the norm as the first passes apply it
        d[lm] = w / nrm.v[lm];
      }
  }
};
static const HarmonicScales& harmonic_scales() {
  static const HarmonicScales scales;
  return scales;
}

// A binned sum: Re (Im, when one of the two l is odd) of F_lx F_ly^*, and the accumulators that hold them
// (F_0's for every l with a global line of sight).
struct SumDesc {
  int8_t lx, ly, acc_x, acc_y;
};

struct ContractParams {
  int nsteps;
  FieldStep step[NPC_MAX_FIELDS];   // grouped by accumulator, phase b before phase a
  int nacc;                     // F accumulators: of F_0, F_1, ... of tracer B, then F_0^A if cross
  int nphase;
  int pair_rows;                // rows ky and -ky are binned together
  int shared_part;              // the warps' partial sums are kept in shared memory
  int nbins, nsum;
  int row_n2max;                // rows (ky, kz) with ky^2 + kz^2 above this hold no binned mode
  int KZ;                       // planes kz < KZ stored per field by the forward passes
  int nprod;                    // product sums; then the modes and their |k| are summed
  SumDesc sum[MAX_PRODS];
  int global_los;
  double los[3];
  double kf;
};

// L_l(mu), l <= 4, as polynomials (uniform l, no division)
template <typename T> __device__ __forceinline__ T legendre_0to4(int l, T mu) {
  const T m2 = mu * mu;
  switch (l) {
    case 0: return T(1);
    case 1: return mu;
    case 2: return T(1.5) * m2 - T(0.5);
    case 3: return mu * (T(2.5) * m2 - T(1.5));
  }
  return (T(4.375) * m2 - T(3.75)) * m2 + T(0.375);
}

// Threads of a CTA that meet at one barrier in the x pass: the warps of one row where a row takes whole
// warps, one warp holding several rows where rows pack into a warp, else (lengths 3 * 2^k) the block.
template <int N> struct XTeam {
  static constexpr int TPF = N / 8;
  static constexpr bool BLOCK = !(TPF % 32 == 0 || 32 % TPF == 0);
  // exchange buffers per row: two where every exchange of the transform writes the other one, which
  // leaves one barrier per exchange
  static constexpr int XBUF = BLOCK ? 1 : 2;
  // slots per row: the buffers, and for rows of fewer than 16 threads an offset that puts the rows of one
  // 16-lane access on different banks
  static constexpr int ROW = XBUF * row_pad_len<N>() + (TPF < 16 ? TPF : 0);
  // threads per CTA: whole warps of whole rows for the lengths 3 * 2^k
  static constexpr int THREADS = BLOCK ? 96 : CONTRACT_THREADS;
  static_assert(THREADS % TPF == 0, "whole rows");
};

// v[q] (mode kx = t + q TPF) times the step's scale * the part of Q_LM(uz) (ux + i uy)^M, added to acc.
template <typename T, int N, int L, int M, int IM>
__device__ __forceinline__ void add_weighted(cplx<T> (&acc)[8], const cplx<T> (&v)[8], const T (&inv)[8],
                                             const FieldStep& st, int t, T fj, T fk) {
  constexpr int TPF = N / 8;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    T iv = inv[q];
    keep_here(iv);   // the weights of the other fields must not be formed beside this one's
    const T ux = T(t + (q < 4 ? q : q - 8) * TPF) * iv, uy = fj * iv;
    T pr = T(1), pi = T(0);
#pragma unroll
    for (int j = 0; j < M; ++j) {
      const T nr = pr * ux - pi * uy;
      pi = pr * uy + pi * ux;
      pr = nr;
    }
    const T w = scaled(st, ylm_q<T, L, M>(fk * iv) * (IM ? pi : pr));
    acc[q] = cmk(acc[q].x + w * v[q].x, acc[q].y + w * v[q].y);
  }
}

// Last pass.  A group of N/8 threads owns a row (ky, kz): it transforms the row of every field along x,
// one after the other, and adds it with its coefficient to one F_l accumulator in registers (F_l is
// linear in the fields, and they come grouped by multipole, so one accumulator is live at a time); the
// finished F_l go to the group's shared memory, from which the team's threads form the products
// Re[F_0 F_l^*], Re[F_l F_l'^*] per pair of mirror modes and bin them.  Groups of one or more warps never
// wait for each other.  The modes (kx, ky) with either sign of each have one |k|, hence one bin: all four
// (the two signs of kx where rows are not paired) are added before the warp-segmented scan.
// Bound by latency and issue: 16 warps per SM (127 registers, two CTAs), 256^3: issue 56 % of the slots, DRAM 28
// %, stalls led by fixed latencies and instruction fetch (the weights' 23 cases).  512^3, 30 fields: 5.6 ms for
// 12.5 GB (7.9 ms with a row shared by all groups of a CTA).
template <typename T, int N, int MINB>
__global__ void __launch_bounds__(XTeam<N>::THREADS, MINB)
k_fft_x_contract(const cplx<T>* __restrict__ half, const __grid_constant__ ContractParams P,
                 const int16_t* __restrict__ bintab, const cplx<T>* __restrict__ tw_g,
                 const cplx<T>* __restrict__ factors, double* __restrict__ part) {
  using C = cplx<T>;
  using Team = XTeam<N>;
  constexpr int TPF = Team::TPF;
  constexpr int NP = row_pad_len<N>();
  const int G = blockDim.x / TPF;             // rows in flight
  const int nw = blockDim.x >> 5;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* phs = tw + N;                            // e^{i pi m/N}, m = -N .. N-1
  C* rowbuf = phs + 2 * N;                    // [G][ROW]
  C* fsm = rowbuf + (size_t)G * Team::ROW;   // [G][1 or 2 rows][nacc][N]
  const int nslot = P.pair_rows ? 2 : 1;
  T* winv = reinterpret_cast<T*>(fsm + (size_t)G * nslot * P.nacc * N);   // 1/sinc^p, a = 0..N/2
  double* spart = reinterpret_cast<double*>(smem_raw + (((reinterpret_cast<unsigned char*>(winv + N / 2 + 2) - smem_raw) + 15) & ~(size_t)15));
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nent = P.nbins * P.nsum;
  for (int i = tid; i < N; i += blockDim.x) tw[i] = tw_g[i];
  for (int i = tid; i < 2 * N; i += blockDim.x) phs[i] = factors[i];
  for (int i = tid; i <= N / 2; i += blockDim.x) winv[i] = reinterpret_cast<const T*>(factors + 2 * N)[i];
  if (P.shared_part)
    for (int i = tid; i < nw * nent; i += blockDim.x) spart[i] = 0.0;
  __syncthreads();
  double* mypart = P.shared_part ? spart + (size_t)warp * nent : part + ((size_t)blockIdx.x * nw + warp) * nent;
  const int g = tid / TPF, t = tid % TPF;
  const size_t fstride = (size_t)P.KZ * N * N;
  const T half_or_one = P.nphase == 2 ? T(0.5) : T(1);
  // items (kz, |ky|), ky >= 0 before -ky
  const int nitems = P.KZ * (N / 2), istep = gridDim.x * G;
  auto in_bins = [&](int item) {
    const int kz = item / (N / 2), ay = item % (N / 2);
    return item < nitems && kz * kz + ay * ay <= P.row_n2max;
  };
  // first item at or after `item` (steps of istep) with modes in the bins
  auto seek = [&](int item) {
    while (item < nitems && !in_bins(item)) item += istep;
    return item;
  };
  auto row_of = [&](int item, int sgn) {
    const int kz = item / (N / 2), ay = item % (N / 2);
    return half + ((size_t)kz * N + (sgn && ay ? N - ay : ay)) * N;
  };
  // team-uniform loop: a team's groups (rows of one warp, or of the block) go on until none has an item
  int item = blockIdx.x * G + g;
  if (!Team::BLOCK) item = seek(item);
  int pass = 0, flip = 0;
  C* bufs = rowbuf + (size_t)g * Team::ROW;
  C v[8], vn[8];
  if (in_bins(item)) {
    const C* src = row_of(item, 0) + (size_t)P.step[0].field * fstride;
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = src[t + q * TPF];
  }
  auto team_sync = [&]() {
    if constexpr (Team::BLOCK) __syncthreads();
    else if constexpr (TPF <= 32) __syncwarp();
    else SyncNamed{1 + g, TPF}();
  };
  auto team_any = [&](bool p) -> bool {
    if constexpr (Team::BLOCK) return __syncthreads_or(p);
    else if constexpr (TPF < 32) return __any_sync(0xffffffffu, p);
    else return p;
  };
  while (team_any(item < nitems)) {
    const bool live0 = in_bins(item);
    const int next = Team::BLOCK ? item + istep : seek(item + istep);
    // (a group without an item transforms zeros with its team: its table look-ups stay in range)
    const int kz = live0 ? item / (N / 2) : 0, ay = live0 ? item % (N / 2) : 0;
    if (!Team::BLOCK || team_any(live0)) {
#pragma unroll 1
      for (int sgn = 0; sgn < 2; ++sgn) {
        const bool live = live0 && (sgn == 0 || ay > 0);
        const int jy = sgn ? -ay : ay;
        // |k| of the thread's modes, and the row's factor of the window
        T inv[8];
        C racc[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const T fi = T(t + (q < 4 ? q : q - 8) * TPF), fj = T(jy), fk = T(kz);
          const T r2 = fi * fi + fj * fj + fk * fk;
          inv[q] = r2 > T(0) ? rsqrt_unbiased(r2) : T(0);
          racc[q] = cmk(T(0), T(0));
        }
        if (team_any(live)) {
#pragma unroll 1
          for (int st = 0; st < P.nsteps; ++st) {
            const FieldStep c = P.step[st];
            {
              // the row that comes next: this row's next field, else the first field of the next row
              const bool more = st + 1 < P.nsteps;
              const int nsgn = more ? sgn : (sgn == 0 && ay > 0 ? 1 : 0);
              const int nitem = more || nsgn > sgn ? item : next;
              if (more ? live : in_bins(nitem)) {
                const C* src = row_of(nitem, nsgn) + (size_t)P.step[more ? st + 1 : 0].field * fstride;
#pragma unroll
                for (int q = 0; q < 8; ++q) vn[q] = src[t + q * TPF];
              }
            }
            if (!live) {
#pragma unroll
              for (int q = 0; q < 8; ++q) v[q] = cmk(T(0), T(0));
            }
            if constexpr (Team::BLOCK) {
              fft_block<N, -1>(v, t, tw, RowView<C>{bufs}, SyncBlock{});
            } else {
              const RowView<C> b0{bufs + flip * NP}, b1{bufs + (flip ^ 1) * NP};
              if constexpr (TPF <= 32) fft_block_alternate<N, -1>(v, t, tw, b0, b1, SyncWarp{});
              else fft_block_alternate<N, -1>(v, t, tw, b0, b1, SyncNamed{1 + g, TPF});
              flip ^= fft_exchanges<N>() & 1;
            }
            const T fj = T(jy), fk = T(kz);
#define NPC_W(L, M, IM) \
  case 2 * (L * (L + 1) / 2 + M) + IM: add_weighted<T, N, L, M, IM>(racc, v, inv, c, t, fj, fk); break;
            switch (c.weight) {
              NPC_W(1, 0, 0) NPC_W(1, 1, 0) NPC_W(1, 1, 1)
              NPC_W(2, 0, 0) NPC_W(2, 1, 0) NPC_W(2, 1, 1) NPC_W(2, 2, 0) NPC_W(2, 2, 1)
              NPC_W(3, 0, 0) NPC_W(3, 1, 0) NPC_W(3, 1, 1) NPC_W(3, 2, 0) NPC_W(3, 2, 1) NPC_W(3, 3, 0) NPC_W(3, 3, 1)
              NPC_W(4, 0, 0) NPC_W(4, 1, 0) NPC_W(4, 1, 1) NPC_W(4, 2, 0) NPC_W(4, 2, 1) NPC_W(4, 3, 0) NPC_W(4, 3, 1)
              NPC_W(4, 4, 0) NPC_W(4, 4, 1)
              default:
#pragma unroll
                for (int q = 0; q < 8; ++q) racc[q] = cadd(racc[q], v[q]);
            }
#undef NPC_W
            if (c.flags & STEP_ROTATE) {
#pragma unroll
              for (int q = 0; q < 8; ++q) {
                int m = t + (q < 4 ? q : q - 8) * TPF + jy + kz;   // in (-N, 3N/2)
                if (m >= N) m -= 2 * N;
                racc[q] = cmul(racc[q], phs[m + N]);
              }
            }
            if (c.flags & STEP_STORE) {
              C* f = fsm + (((size_t)g * nslot + (P.pair_rows ? sgn : 0)) * P.nacc + c.acc) * N;
              const T wr = half_or_one * winv[ay] * winv[kz];
#pragma unroll
              for (int q = 0; q < 8; ++q) {
                const int ai = q < 4 ? t + q * TPF : (8 - q) * TPF - t;
                f[t + q * TPF] = cscale(racc[q], wr * winv[ai]);
                racc[q] = cmk(T(0), T(0));
              }
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = vn[q];
          }
        }
        if (P.pair_rows && sgn == 0) continue;
        team_sync();
        // bin the team's rows: tasks (row, chunk of 32 modes kx = jp >= 0 with their mirror modes)
        constexpr int NJ = N / 2, CH = (NJ + 31) / 32;
        const int trows = Team::BLOCK ? G : (TPF < 32 ? 32 / TPF : 1);
        const int twarps = Team::BLOCK ? nw : (TPF > 32 ? TPF / 32 : 1);
        const int twarp = Team::BLOCK ? warp : warp % twarps;
        for (int task = twarp; task < trows * CH; task += twarps) {
          const int tr = task / CH, jp = (task % CH) * 32 + lane;
          const int gr = Team::BLOCK ? tr : (TPF < 32 ? warp * trows + tr : g);   // the task's group
          int titem = item;
          if constexpr (Team::BLOCK) titem = blockIdx.x * G + gr + pass * istep;
          else if constexpr (TPF < 32) titem = __shfl_sync(0xffffffffu, item, tr * TPF);
          if (!in_bins(titem)) continue;   // warp-uniform
          const int tkz = titem / (N / 2), tay = titem % (N / 2);
          int bin = -1;
          T vals[MAX_SUMS];
#pragma unroll
          for (int e = 0; e < MAX_SUMS; ++e) vals[e] = T(0);
          const int n2 = jp * jp + tay * tay + tkz * tkz;
          if (jp < NJ && n2 > 0) bin = bintab[n2];
          if (bin >= 0) {
            const T wgt = tkz > 0 ? T(2) : T(1), fkz = T(tkz);
            const T kk = sqrt(T(n2));
            T modes = T(0);
#pragma unroll 1
            for (int m = 0; m < 4; ++m) {   // kx = jp, -jp at ky of either sign
              const int ms = P.pair_rows ? m >> 1 : sgn;
              if ((m & 1) && jp == 0) continue;
              if ((m >> 1) && (!P.pair_rows || tay == 0)) continue;
              if (ms && tay == 0) continue;
              const int i = (m & 1) ? -jp : jp, j = (m & 1) ? N - jp : jp;
              const C* f = fsm + ((size_t)gr * nslot + (P.pair_rows ? ms : 0)) * P.nacc * N + j;
              T mu = T(0);
              if (P.global_los)
                mu = (T(i) * T(P.los[0]) + T(ms ? -tay : tay) * T(P.los[1]) + fkz * T(P.los[2])) / kk;
              modes += T(1);
#pragma unroll
              for (int e = 0; e < MAX_PRODS; ++e) {
                if (e >= P.nprod) break;
                const SumDesc sd = P.sum[e];
                const C x = f[(size_t)sd.acc_x * N], y = f[(size_t)sd.acc_y * N];
                // Re x y^*; with one odd l Im x y^* (Sec. 2.1, odd multipoles)
                T p = wgt * (((sd.lx + sd.ly) & 1) ? (x.y * y.x - x.x * y.y) : (x.x * y.x + x.y * y.y));
                if (P.global_los) p *= legendre_0to4<T>(sd.lx, mu) * legendre_0to4<T>(sd.ly, mu);
                vals[e] += p;
              }
            }
            modes *= wgt;
            vals[MAX_SUMS - 2] = modes;
            vals[MAX_SUMS - 1] = modes * (T(P.kf) * kk);
          }
          // warp-segmented inclusive scan over the runs of consecutive lanes with equal bin (bins rise
          // with kx, so a bin has one run)
          const int pb = __shfl_up_sync(0xffffffffu, bin, 1);
          const bool head = (lane == 0) || (pb != bin);
          const unsigned heads = __ballot_sync(0xffffffffu, head);
          const int first = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));   // lane of the run's head
          const bool last = (lane == 31) || ((heads >> (lane + 1)) & 1u);
          // run sums (of at most 32 lanes, 2 modes each, or 4 with ky and -ky) stay in T; only run ends convert to
          // float64.  Runs cut to 32 modes have the same errors against 64 bits to three digits (128^3, 96
          // catalogues; 256^3, 16) and cost 6 % of the pass at 128^3, 36 % with ky and -ky at 256^3.
#pragma unroll
          for (int e = 0; e < MAX_SUMS; ++e) {
            if (e < MAX_PRODS && e >= P.nprod) continue;
            T x = vals[e];
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
              const T y = __shfl_up_sync(0xffffffffu, x, off);
              if (lane - off >= first) x += y;
            }
            if (last && bin >= 0) {
              double* dst = mypart + (size_t)bin * P.nsum + (e < MAX_PRODS ? e : P.nprod + e - MAX_PRODS);
              if (P.shared_part) *dst += (double)x;
              else atomicAdd(dst, (double)x);
            }
          }
          if (P.shared_part) __syncwarp();
        }
        if constexpr (Team::BLOCK) __syncthreads();
      }
    }
    else if (in_bins(next)) {   // nothing to do in this pass of the block: the next pass's first row
      const C* src = row_of(next, 0) + (size_t)P.step[0].field * fstride;
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = src[t + q * TPF];
    }
    item = next;
    if constexpr (Team::BLOCK) ++pass;
  }
  if (P.shared_part) {   // the CTA's sums, warps in order
    __syncthreads();
    for (int i = tid; i < nent; i += blockDim.x) {
      double x = 0.0;
      for (int w = 0; w < nw; ++w) x += spart[(size_t)w * nent + i];
      part[(size_t)blockIdx.x * nent + i] = x;
    }
  }
}

struct FinalParams {
  int nbins, nsum, nparts;
  int nell, ell_list[5];
  int nll, lla[3], llb[3];
  int nmod, mod_list[3];
  int out_rows;          // 2 + requested P_l + requested P_lb + requested P_ll'
  int ll_req;            // output P_22 (bit 0), P_42 (bit 1), P_44 (bit 2)
  int req_mask;          // requested P_l (bits)
};

constexpr int FIN_THREADS = 256;

// one block per bin: the partials are summed with a fixed per-thread stride and a fixed tree
__global__ void __launch_bounds__(FIN_THREADS)
k_power_finalize(const double* __restrict__ part, const FinalParams F, const double* __restrict__ sc,
                 double* __restrict__ out) {
  const int nb = F.nbins;
  __shared__ double red[MAX_SUMS][FIN_THREADS];
  for (int b = blockIdx.x; b < nb; b += gridDim.x) {
    double S[MAX_SUMS];
    for (int s = 0; s < MAX_SUMS; ++s) S[s] = 0.0;
    for (int p = threadIdx.x; p < F.nparts; p += FIN_THREADS) {
#pragma unroll
      for (int s = 0; s < MAX_SUMS; ++s)
        if (s < F.nsum) S[s] += part[((size_t)p * nb + b) * F.nsum + s];
    }
    for (int s = 0; s < MAX_SUMS; ++s) red[s][threadIdx.x] = S[s];
    __syncthreads();
    for (int off = FIN_THREADS / 2; off > 0; off >>= 1) {
      if (threadIdx.x < off)
        for (int s = 0; s < MAX_SUMS; ++s) red[s][threadIdx.x] += red[s][threadIdx.x + off];
      __syncthreads();
    }
    for (int s = 0; s < MAX_SUMS; ++s) S[s] = red[s][0];
    __syncthreads();
    if (threadIdx.x != 0) continue;
    const double cnt = S[F.nsum - 2];
    const double i22 = sc[SC_I22], n0 = sc[SC_N0];
    const bool ok = cnt > 0;
    out[0 * nb + b] = ok ? S[F.nsum - 1] / cnt : 0.0;
    out[1 * nb + b] = cnt;
    double Pl[5] = {0, 0, 0, 0, 0};   // index l
    int row = 2;
    for (int e = 0; e < F.nell; ++e) {
      const int l = F.ell_list[e];
      const double v = ok ? (2 * l + 1) / i22 * S[e] / cnt - (l == 0 ? n0 : 0.0) : 0.0;
      Pl[l] = v;
      if (F.req_mask & (1 << l)) out[(row++) * nb + b] = v;
    }
    double P22 = 0, P42 = 0, P44 = 0;
    for (int e = 0; e < F.nll; ++e) {
      const int a = F.lla[e], c = F.llb[e];
      const double nsh = (a == c) ? (2 * (a + c) + 1) * n0 / (2 * a + 1) : 0.0;
      const double v = ok ? (2 * (a + c) + 1) / i22 * S[F.nell + e] / cnt - nsh : 0.0;
      if (a == 2 && c == 2) P22 = v;
      if (a == 4 && c == 2) P42 = v;
      if (a == 4 && c == 4) P44 = v;
    }
    for (int e = 0; e < F.nmod; ++e) {
      const int lb = F.mod_list[e];
      double v = 0.0;
      if (ok) {
        if (lb == 4) v = 35.0 / 18.0 * P22 - Pl[2] - 3.5 * Pl[0];
        if (lb == 6) v = 11.0 / 5.0 * P42 - 52.0 / 63.0 * Pl[4] - 286.0 / 175.0 * Pl[2];
        if (lb == 8)
          v = 1287.0 / 490.0 * P44 - 374.0 / 245.0 * P42 - 3553.0 / 15435.0 * Pl[4] - 1326.0 / 8575.0 * Pl[2] -
              2431.0 / 490.0 * Pl[0];
      }
      out[(row++) * nb + b] = v;
    }
    // the two-index spectra themselves (Eq. Pllp), when requested: P_22, P_42, P_44
    if (F.ll_req & 1) out[(row++) * nb + b] = P22;
    if (F.ll_req & 2) out[(row++) * nb + b] = P42;
    if (F.ll_req & 4) out[(row++) * nb + b] = P44;
  }
  if (blockIdx.x == 0 && threadIdx.x < 8) out[(size_t)F.out_rows * nb + threadIdx.x] = sc[threadIdx.x];
}

// ---------------------------------------------------------------------------------------------
// y pass with a selectable number of columns per CTA
// ---------------------------------------------------------------------------------------------
template <int N> constexpr bool ytx_ok(int tx) { return tx <= N && N % tx == 0 && tx * N / 8 <= 1024; }

// with column factors: a second copy of the columns has to fit an SM's shared memory as well
template <typename T, int N> constexpr size_t ytxw_smem(int tx) {
  return sizeof(cplx<T>) * (N + (size_t)(tx < 16 ? N + N / 8 : N) * tx + (size_t)N * tx);
}
template <typename T, int N> constexpr bool ytxw_ok(int tx) { return ytx_ok<N>(tx) && ytxw_smem<T, N>(tx) <= 227 * 1024; }

// Columns per CTA that are not tuned: the fastest of both forms or within 4 % of it in float32 (1024^3: 7 % with
// column factors), in float64 within 3 % plain and 12 % with column factors (192: 576 us with 4, 646 with 16).
constexpr int default_ytx(int n) { return n >= 1024 ? 4 : (n >= 512 ? 8 : 16); }
template <typename T, int N> constexpr int default_ytxw() { return default_ytx(N); }

// the tuned width of the plain y pass, else the default
int ytx_for(const npc_ctx* ctx, int n, bool fp64) {
  auto it = ctx->ytx.find(n * 2 + (fp64 ? 1 : 0));
  return it != ctx->ytx.end() ? it->second : default_ytx(n);
}
template <typename T, int N> int ytxw_for(const npc_ctx* ctx) {
  auto it = ctx->ytxw.find(N * 2 + (sizeof(T) == 8 ? 1 : 0));
  return it != ctx->ytxw.end() ? it->second : default_ytxw<T, N>();
}

template <typename T, int N, int TX>
npc_status y_pass_tx(npc_ctx* ctx, cplx<T>* data, int nplanes, const cplx<T>* tw, int kz_planes, int row_n2max) {
  using C = cplx<T>;
  if constexpr (!ytx_ok<N>(TX)) {
    return set_err(ctx, NPC_ERR_INVALID_ARG, "y pass: %d columns per CTA not valid at n = %d", TX, N);
  } else {
    const size_t smem = sizeof(C) * (N + N * TX);
    auto kern = k_fft_cols<T, N, -1, TX>;
    NPC_TRY(allow_smem(ctx, (const void*)kern, smem));
    for (int p0 = 0; p0 < nplanes; p0 += 65535) {
      const int np = std::min(65535, nplanes - p0);
      kern<<<dim3(N / TX, np), TX * N / 8, smem, ctx->stream>>>(data + (size_t)p0 * N * N, (size_t)N * N, N, tw, p0,
                                                                kz_planes, row_n2max);
      NPC_LAUNCH(ctx);
    }
    return NPC_OK;
  }
}

template <typename T, int N>
npc_status y_pass(npc_ctx* ctx, cplx<T>* data, int nplanes, const cplx<T>* tw, int tx, int kz_planes = 1,
                  int row_n2max = 1 << 30) {
  switch (tx) {
    case 4: return y_pass_tx<T, N, 4>(ctx, data, nplanes, tw, kz_planes, row_n2max);
    case 8: return y_pass_tx<T, N, 8>(ctx, data, nplanes, tw, kz_planes, row_n2max);
    case 16: return y_pass_tx<T, N, 16>(ctx, data, nplanes, tw, kz_planes, row_n2max);
    case 32: return y_pass_tx<T, N, 32>(ctx, data, nplanes, tw, kz_planes, row_n2max);
  }
  return set_err(ctx, NPC_ERR_INVALID_ARG, "y pass: unsupported columns per CTA %d", tx);
}

template <typename T, int N, int TX, bool NEAR = false>
npc_status y_pass_weighted_tx(npc_ctx* ctx, cplx<T>* half, const SignalList& sl, const T* coords, T near,
                              const YNorm& nrm, const cplx<T>* tw, int KZ, int row_n2max) {
  using C = cplx<T>;
  if constexpr (!ytxw_ok<T, N>(TX)) {
    return set_err(ctx, NPC_ERR_INVALID_ARG, "y pass: %d columns per CTA not valid at n = %d", TX, N);
  } else {
    constexpr size_t smem = ytxw_smem<T, N>(TX);
    static_assert(smem == sizeof(C) * (N + col_rows<N, TX>() * TX + N * TX), "shared memory of the kernel");
    auto kern = k_fft_cols_weighted<T, N, TX, NEAR>;
    NPC_TRY(allow_smem(ctx, (const void*)kern, smem));
    const int nplanes = sl.n * KZ;   // at most 32 x 512
    kern<<<dim3(N / TX, nplanes), TX * N / 8, smem, ctx->stream>>>(half, sl, coords, near, nrm, tw, KZ, row_n2max);
    NPC_LAUNCH(ctx);
    return NPC_OK;
  }
}

template <typename T, int N>
npc_status y_pass_weighted(npc_ctx* ctx, cplx<T>* half, const SignalList& sl, const T* coords, T near,
                           bool near_columns, const YNorm& nrm, const cplx<T>* tw, int tx, int KZ, int row_n2max) {
  if (near_columns)
    return y_pass_weighted_tx<T, N, default_ytxw<T, N>(), true>(ctx, half, sl, coords, near, nrm, tw, KZ, row_n2max);
  switch (tx) {
    case 4: return y_pass_weighted_tx<T, N, 4>(ctx, half, sl, coords, near, nrm, tw, KZ, row_n2max);
    case 8: return y_pass_weighted_tx<T, N, 8>(ctx, half, sl, coords, near, nrm, tw, KZ, row_n2max);
    case 16: return y_pass_weighted_tx<T, N, 16>(ctx, half, sl, coords, near, nrm, tw, KZ, row_n2max);
    case 32: return y_pass_weighted_tx<T, N, 32>(ctx, half, sl, coords, near, nrm, tw, KZ, row_n2max);
  }
  return set_err(ctx, NPC_ERR_INVALID_ARG, "y pass: unsupported columns per CTA %d", tx);
}

// Autotuner for the y pass: times every valid columns-per-CTA choice of both forms (plain and with column
// factors, which needs twice the shared memory per column) on a scratch buffer of `nplanes` planes (values
// irrelevant to the timing) and keeps the fastest of each for (n, precision).
template <typename Run>
npc_status fastest_width(npc_ctx* ctx, const std::vector<int>& widths, Run&& run, int* best_tx) {
  cudaEvent_t e0, e1;
  NPC_CUDA(ctx, cudaEventCreate(&e0));
  NPC_CUDA(ctx, cudaEventCreate(&e1));
  float best = 1e30f;
  npc_status st = NPC_OK;
  for (int tx : widths) {
    st = run(tx);  // warm-up
    if (st != NPC_OK) break;
    cudaEventRecord(e0, ctx->stream);
    for (int rep = 0; rep < 3 && st == NPC_OK; ++rep) st = run(tx);
    cudaEventRecord(e1, ctx->stream);
    if (st != NPC_OK) break;
    cudaEventSynchronize(e1);
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    if (ms < best) {
      best = ms;
      *best_tx = tx;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return st;
}

template <typename T, int N>
npc_status tune_y_impl(npc_ctx* ctx, int nplanes) {
  using C = cplx<T>;
  constexpr bool fp64 = sizeof(T) == 8;
  const void* twp;
  NPC_TRY(get_twiddles(ctx, N, fp64 ? NPC_PREC_FP64 : NPC_PREC_MIXED, &twp));
  const C* tw = (const C*)twp;
  C* buf;
  T* coords;
  NPC_TRY(ws_get(ctx, "tune.y", sizeof(C) * (size_t)nplanes * N * N, (void**)&buf));
  NPC_TRY(ws_get(ctx, "tune.coords", sizeof(T) * 6 * N, (void**)&coords));
  NPC_CUDA(ctx, cudaMemsetAsync(buf, 0, sizeof(C) * (size_t)nplanes * N * N, ctx->stream));
  NPC_CUDA(ctx, cudaMemsetAsync(coords, 0, sizeof(T) * 6 * N, ctx->stream));
  std::vector<int> plain, weighted;
  for (int tx : {4, 8, 16, 32}) {
    if (ytx_ok<N>(tx)) plain.push_back(tx);
    if (ytxw_ok<T, N>(tx)) weighted.push_back(tx);
  }
  int tx = default_ytx(N), txw = default_ytxw<T, N>();
  NPC_TRY(fastest_width(ctx, plain, [&](int w) { return y_pass<T, N>(ctx, buf, nplanes, tw, w); }, &tx));
  SignalList sl{};   // phases a and b of Y_21: two signals read, four fields written
  sl.n = 2;
  for (int8_t ph = 0; ph < 2; ++ph) sl.s[ph] = Signal{ph, 2, 1, (int8_t)(2 * ph), (int8_t)(2 * ph + 1)};
  const YNorm nrm = ylm_norm_table();
  const int kz = std::max(1, std::min(nplanes / 4, N / 2));
  if (nplanes >= 4)
    NPC_TRY(fastest_width(ctx, weighted, [&](int w) {
      return y_pass_weighted<T, N>(ctx, buf, sl, coords, T(0), false, nrm, tw, w, kz, 1 << 30);
    }, &txw));
  ctx->ytx[N * 2 + fp64] = tx;
  ctx->ytxw[N * 2 + fp64] = txw;
  return NPC_OK;
}

// ---------------------------------------------------------------------------------------------
template <typename T, int N>
npc_status fwd_impl(npc_ctx* ctx, const PowerPlan& plan, const Geom& g, const void* mesh_a, const void* mesh_b,
                    void* half) {
  const int KZ = plan.kz_keep > 0 ? std::min(plan.kz_keep, N / 2) : N / 2;
  using C = cplx<T>;
  constexpr int TX = ColCfg<N>::TX;
  const void* twp;
  NPC_TRY(get_twiddles(ctx, N, sizeof(T) == 8 ? NPC_PREC_FP64 : NPC_PREC_MIXED, &twp));
  const C* tw = (const C*)twp;
  const YNorm nrm = ylm_norm_table();
  const bool single = !mesh_b && plan.fl.nf == 1 && plan.fl.f[0].part == PART_ONE && plan.fl.f[0].phase == 0;
  const SignalList sl = make_signals(plan.fl);
  bool directions = false, weighted = false;   // harmonics of l > 0, of m > 0
  for (int i = 0; i < sl.n; ++i) {
    directions |= sl.s[i].l > 0;
    weighted |= sl.s[i].m > 0;
  }
  // unit of the coordinates: the power of two at or below the farthest grid point's distance along an axis
  double far = 0.0;
  for (int a = 0; a < 3; ++a) far = std::max(far, std::fabs(g.o[a] - g.obs[a]) + g.h * N);
  const double unit = std::ldexp(1.0, -std::ilogb(far));
  const T near = (T)std::ldexp(1.0, std::ilogb(0.5 * g.h * unit));
  bool near_columns = false;
  T* coords = nullptr;
  if (directions) {
    bool close[2] = {false, false};   // k_axis_coords has a value below `near` on the x, on the y axis
    for (int a = 0; a < 2; ++a)
      for (int j = 0; j < N; ++j)
        for (double shift : {0.0, 0.5})
          close[a] |= std::fabs((T)((g.o[a] + ((double)j - shift) * g.h - g.obs[a]) * unit)) < near;
    near_columns = close[0] && close[1];
    NPC_TRY(ws_get(ctx, "fwd.coords", sizeof(T) * 6 * N, (void**)&coords));
    k_axis_coords<T><<<(6 * N + 255) / 256, 256, 0, ctx->stream>>>(g, unit, coords);
    NPC_LAUNCH(ctx);
  }
  if (single) {
    constexpr int STX = SingleCfg<N>::TX;
    static_assert(N % (2 * STX) == 0, "column pairs must tile the mesh");
    const size_t ssmem = sizeof(C) * (N + col_rows<N, STX>() * STX);
    auto kern = (uintptr_t)mesh_a % sizeof(C) == 0 ? k_fwd_z_single<T, N, true> : k_fwd_z_single<T, N, false>;
    NPC_TRY(allow_smem(ctx, (const void*)kern, ssmem));
    kern<<<dim3(N / (2 * STX), N), SingleCfg<N>::THREADS, ssmem, ctx->stream>>>((const T*)mesh_a, (C*)half, tw, KZ);
  } else {
    const size_t smem = sizeof(C) * (N + col_rows<N, TX>() * TX) + sizeof(T) * (mesh_b ? 2 : 1) * N * TX;
    auto kern = near_columns ? k_fwd_z<T, N, true> : k_fwd_z<T, N, false>;
    NPC_TRY(allow_smem(ctx, (const void*)kern, smem));
    kern<<<dim3(N / TX, N), ColCfg<N>::THREADS, smem, ctx->stream>>>((const T*)mesh_a, (const T*)mesh_b, (C*)half, sl,
                                                                     coords, (T)(g.h * (N / 8) * unit), near, nrm, tw, KZ);
  }
  NPC_LAUNCH(ctx);
  NPC_TRY(stage_mark(ctx, "fft_z_weighted"));
  const int n2max = plan.row_n2max > 0 ? plan.row_n2max : (1 << 30);
  // planes (f, kz) are contiguous N*N blocks; y rows have stride N
  if (weighted)
    NPC_TRY((y_pass_weighted<T, N>(ctx, (C*)half, sl, coords, near, near_columns, nrm, tw,
                                   ytxw_for<T, N>(ctx), KZ, n2max)));
  else
    NPC_TRY((y_pass<T, N>(ctx, (C*)half, plan.fl.nf * KZ, tw, ytx_for(ctx, N, sizeof(T) == 8), KZ, n2max)));
  NPC_TRY(stage_mark(ctx, "fft_y"));
  return NPC_OK;
}

template <typename T, int N>
npc_status contract_impl(npc_ctx* ctx, const PowerPlan& plan, const npc_mesh_spec& m, const npc_kbins& kb,
                         const void* half, const double* sc, double* dev_out) {
  using C = cplx<T>;
  const void* twp;
  NPC_TRY(get_twiddles(ctx, N, sizeof(T) == 8 ? NPC_PREC_FP64 : NPC_PREC_MIXED, &twp));
  const void* factors;
  NPC_TRY(get_mode_factors(ctx, N, plan.assign, sizeof(T) == 8 ? NPC_PREC_FP64 : NPC_PREC_MIXED, &factors));
  const int16_t* bintab;
  NPC_TRY(get_bin_table(ctx, N, m.box, kb, &bintab));
  ContractParams P{};
  P.nphase = plan.nphase;
  int req_internal = plan.ells_mask;
  if (plan.mod_mask) req_internal |= 1 | 4 | 16;
  // accumulators: one per multipole with fields of tracer B (in l order), then F_0^A
  int acc_of[5] = {-1, -1, -1, -1, -1};
  int nacc_b = 0;
  if (plan.global_los) {
    acc_of[0] = 0;
    nacc_b = 1;
  } else {
    for (int l = 0; l <= 4; ++l) {
      bool has = false;
      for (int f = 0; f < plan.fl.nf; ++f) has |= !plan.fl.f[f].tracer && plan.fl.f[f].ell == l;
      if (has) acc_of[l] = nacc_b++;
    }
  }
  const int acc_a = plan.cross ? nacc_b : -1;
  P.nacc = nacc_b + (plan.cross ? 1 : 0);
  if (P.nacc > 6) return set_err(ctx, NPC_ERR_UNSUPPORTED, "x pass: at most 6 accumulators");
  if (plan.cross && plan.mod_mask)
    return set_err(ctx, NPC_ERR_UNSUPPORTED, "cross spectra: no modified multipoles");
  const HarmonicScales& scales = harmonic_scales();
  for (int f = 0; f < plan.fl.nf; ++f) {
    const Comp c = plan.fl.f[f];
    if (c.tracer && (!plan.cross || c.part != PART_ONE))
      return set_err(ctx, NPC_ERR_INVALID_ARG, "x pass: tracer-A field must be an unweighted F_0");
    if (c.phase && P.nphase == 1) return set_err(ctx, NPC_ERR_INVALID_ARG, "phase-b field without interlacing");
    if ((c.part == PART_RE || c.part == PART_IM) && (c.ell < 1 || c.ell > 4 || c.m < 0 || c.m > c.ell))
      return set_err(ctx, NPC_ERR_UNSUPPORTED, "Y_%d%d field in the x pass", c.ell, c.m);
  }
  // steps by accumulator, phase b first: its sum is rotated by the interlacing phase once
  for (int acc = 0; acc < P.nacc; ++acc) {
    for (int ph = P.nphase - 1; ph >= 0; --ph) {
      for (int f = 0; f < plan.fl.nf; ++f) {
        const Comp c = plan.fl.f[f];
        if ((c.phase ? 1 : 0) != ph || (c.tracer ? acc_a : (plan.global_los ? 0 : acc_of[c.ell])) != acc) continue;
        FieldStep& st = P.step[P.nsteps++];
        st.field = (int8_t)f;
        st.acc = (int8_t)acc;
        st.scale_d = 1.0;
        if (c.part == PART_RE || c.part == PART_IM) {
          const int lm = c.ell * (c.ell + 1) / 2 + c.m;
          st.weight = (int8_t)(2 * lm + (c.part == PART_IM ? 1 : 0));
          st.scale_d = scales.d[lm];
          st.scale_f[0] = scales.f[lm][0];
          st.scale_f[1] = scales.f[lm][1];
        }
      }
      if (ph == 1) P.step[P.nsteps - 1].flags |= STEP_ROTATE;
    }
    P.step[P.nsteps - 1].flags |= STEP_STORE;
  }
  P.nbins = kb.nbins;
  FinalParams F{};
  for (int l = 0; l <= 4; ++l)
    if (req_internal & (1 << l)) F.ell_list[F.nell++] = l;
  auto add_ll = [&](int a, int b) { F.lla[F.nll] = a; F.llb[F.nll++] = b; };
  if (plan.mod_mask & ((1 << 4) | (1 << 16))) add_ll(2, 2);
  if (plan.mod_mask & ((1 << 6) | (1 << 8) | (1 << 17))) add_ll(4, 2);
  if (plan.mod_mask & ((1 << 8) | (1 << 18))) add_ll(4, 4);
  auto add_sum = [&](int lx, int ly, int acc_x) {
    P.sum[P.nprod++] = SumDesc{(int8_t)lx, (int8_t)ly, (int8_t)acc_x, (int8_t)(plan.global_los ? 0 : acc_of[ly])};
  };
  // cross spectra take F_0 of tracer A against F_l of B
  for (int e = 0; e < F.nell; ++e) add_sum(0, F.ell_list[e], plan.cross ? acc_a : 0);
  for (int e = 0; e < F.nll; ++e) add_sum(F.lla[e], F.llb[e], plan.global_los ? 0 : acc_of[F.lla[e]]);
  P.nsum = P.nprod + 2;
  P.KZ = plan.kz_keep > 0 ? std::min(plan.kz_keep, N / 2) : N / 2;
  P.global_los = plan.global_los;
  for (int a = 0; a < 3; ++a) P.los[a] = plan.los[a];
  P.kf = 2.0 * M_PI / m.box;
  {
    // a mode is binned only if k_f |q| < kmin + nbins dk; its row has ky^2 + kz^2 <= |q|^2
    const double kmax = kb.kmin + kb.nbins * kb.dk;
    const double r2 = std::pow(kmax / P.kf, 2);
    P.row_n2max = r2 >= 3.0 * (N / 2) * (N / 2) ? 3 * (N / 2) * (N / 2) : (int)std::floor(r2) + 1;
  }

  // shared memory of a CTA: tables, two exchange buffers per row, the finished F_l of one row (or of
  // rows ky and -ky), the warps' partial sums where they are small
  auto smem_of = [&](int threads) {
    const int G = threads / XTeam<N>::TPF;
    size_t b = sizeof(C) * ((size_t)3 * N + (size_t)G * XTeam<N>::ROW +
                            (size_t)G * (P.pair_rows ? 2 : 1) * P.nacc * N) + sizeof(T) * (N / 2 + 2);
    b = (b + 15) & ~(size_t)15;
    if (P.shared_part) b += sizeof(double) * (threads / 32) * P.nbins * P.nsum;
    return b;
  };
  P.pair_rows = P.nacc == 1 ? 1 : 0;
  // Shared sums save the clearing of the partials and leave the finalize one set per CTA: 10 us of 128^3, 18 of
  // a 256^3 box (the pass itself is up to 3 % slower); at 512^3 14 us of 7 ms, not taken.  Above 32 KB they
  // would take the second CTA's shared memory.
  P.shared_part = N <= 256 && sizeof(double) * (CONTRACT_THREADS / 32) * P.nbins * P.nsum <= 32768 ? 1 : 0;
  // fewer threads per CTA where the rows would not fill the SMs four times over (a CTA of 256 threads
  // holds 32 rows at n = 64), or where the shared memory asks for it (FP64 at 256^3 with odd multipoles)
  const int nitems = P.KZ * (N / 2);
  int threads = XTeam<N>::THREADS;
  while (!XTeam<N>::BLOCK && threads > std::max(32, XTeam<N>::TPF) &&
         (smem_of(threads) > 227 * 1024 || nitems < 4 * ctx->num_sms * (threads / XTeam<N>::TPF)))
    threads /= 2;
  const size_t smem = smem_of(threads);
  // float32: as many CTAs as 128 registers a thread allow (five of 96 threads: up to 136 without a spill)
  auto kern = k_fft_x_contract<T, N, (sizeof(T) == 8 ? 1 : (XTeam<N>::BLOCK ? 5 : 2))>;
  NPC_TRY(allow_smem(ctx, (const void*)kern, smem));
  int per_sm = 0;
  NPC_TRY(ctas_per_sm(ctx, (const void*)kern, threads, smem, &per_sm));
  if (per_sm < 1) return set_err(ctx, NPC_ERR_UNSUPPORTED, "contraction does not fit on an SM (%zu B smem)", smem);
  const int G = threads / XTeam<N>::TPF;
  const int grid = std::min((nitems + G - 1) / G, per_sm * ctx->num_sms);
  const size_t nparts = (size_t)grid * (P.shared_part ? 1 : threads / 32);
  double* part;
  NPC_TRY(ws_get(ctx, "power.part", sizeof(double) * nparts * P.nbins * P.nsum, (void**)&part));
  if (!P.shared_part)
    NPC_CUDA(ctx, cudaMemsetAsync(part, 0, sizeof(double) * nparts * P.nbins * P.nsum, ctx->stream));
  NPC_TRY(stage_mark(ctx, "contract_setup"));
  kern<<<grid, threads, smem, ctx->stream>>>((const C*)half, P, bintab, (const C*)twp, (const C*)factors, part);
  NPC_LAUNCH(ctx);
  NPC_TRY(stage_mark(ctx, "fft_x_contract"));

  F.nbins = P.nbins;
  F.nsum = P.nsum;
  F.nparts = (int)nparts;
  F.nmod = 0;
  for (int lb = 4; lb <= 8; lb += 2)
    if (plan.mod_mask & (1 << lb)) F.mod_list[F.nmod++] = lb;
  int nreq = 0;
  for (int l = 0; l <= 4; ++l) nreq += (plan.ells_mask >> l) & 1;
  F.ll_req = (plan.mod_mask >> 16) & 7;
  F.out_rows = 2 + nreq + F.nmod + ((F.ll_req & 1) + ((F.ll_req >> 1) & 1) + ((F.ll_req >> 2) & 1));
  F.req_mask = plan.ells_mask;
  k_power_finalize<<<std::min(P.nbins, 1024), FIN_THREADS, 0, ctx->stream>>>(part, F, sc, dev_out);
  NPC_LAUNCH(ctx);
  NPC_TRY(stage_mark(ctx, "finalize"));
  return NPC_OK;
}

// float32 transforms for n = 2^k in [16, 1024] and n = 48, 96, 192; float64 transforms for n <= 256
template <typename T>
npc_status fwd_dispatch(npc_ctx* ctx, const PowerPlan& plan, const Geom& g, const void* a, const void* b, void* half) {
  switch (plan.n) {
    case 16: return fwd_impl<T, 16>(ctx, plan, g, a, b, half);
    case 32: return fwd_impl<T, 32>(ctx, plan, g, a, b, half);
    case 64: return fwd_impl<T, 64>(ctx, plan, g, a, b, half);
    case 128: return fwd_impl<T, 128>(ctx, plan, g, a, b, half);
    case 256: return fwd_impl<T, 256>(ctx, plan, g, a, b, half);
    case 48: return fwd_impl<T, 48>(ctx, plan, g, a, b, half);
    case 96: return fwd_impl<T, 96>(ctx, plan, g, a, b, half);
    case 192: return fwd_impl<T, 192>(ctx, plan, g, a, b, half);
  }
  if constexpr (sizeof(T) == 4) {
    if (plan.n == 512) return fwd_impl<T, 512>(ctx, plan, g, a, b, half);
    if (plan.n == 1024) return fwd_impl<T, 1024>(ctx, plan, g, a, b, half);
  }
  return set_err(ctx, NPC_ERR_UNSUPPORTED, "mesh size %d not supported at this precision", plan.n);
}

template <typename T>
npc_status contract_dispatch(npc_ctx* ctx, const PowerPlan& plan, const npc_mesh_spec& m, const npc_kbins& kb,
                             const void* half, const double* sc, double* out) {
  switch (plan.n) {
    case 16: return contract_impl<T, 16>(ctx, plan, m, kb, half, sc, out);
    case 32: return contract_impl<T, 32>(ctx, plan, m, kb, half, sc, out);
    case 64: return contract_impl<T, 64>(ctx, plan, m, kb, half, sc, out);
    case 128: return contract_impl<T, 128>(ctx, plan, m, kb, half, sc, out);
    case 256: return contract_impl<T, 256>(ctx, plan, m, kb, half, sc, out);
    case 48: return contract_impl<T, 48>(ctx, plan, m, kb, half, sc, out);
    case 96: return contract_impl<T, 96>(ctx, plan, m, kb, half, sc, out);
    case 192: return contract_impl<T, 192>(ctx, plan, m, kb, half, sc, out);
  }
  if constexpr (sizeof(T) == 4) {
    if (plan.n == 512) return contract_impl<T, 512>(ctx, plan, m, kb, half, sc, out);
    if (plan.n == 1024) return contract_impl<T, 1024>(ctx, plan, m, kb, half, sc, out);
  }
  return set_err(ctx, NPC_ERR_UNSUPPORTED, "mesh size %d not supported at this precision", plan.n);
}

}  // namespace

npc_status tune_y_pass(npc_ctx* ctx, int n, int prec, int nplanes) {
  const bool d = prec == NPC_PREC_FP64;
#define NPC_TY(NN)                                                              \
  case NN:                                                                      \
    return d ? tune_y_impl<double, NN>(ctx, nplanes) : tune_y_impl<float, NN>(ctx, nplanes);
  switch (n) {
    NPC_TY(16) NPC_TY(32) NPC_TY(48) NPC_TY(64) NPC_TY(96) NPC_TY(128) NPC_TY(192) NPC_TY(256)
    case 512: return d ? set_err(ctx, NPC_ERR_UNSUPPORTED, "FP64 n <= 256") : tune_y_impl<float, 512>(ctx, nplanes);
    case 1024: return d ? set_err(ctx, NPC_ERR_UNSUPPORTED, "FP64 n <= 256") : tune_y_impl<float, 1024>(ctx, nplanes);
  }
#undef NPC_TY
  return set_err(ctx, NPC_ERR_UNSUPPORTED, "mesh size %d", n);
}

npc_status run_forward_transforms(npc_ctx* ctx, int prec, const PowerPlan& plan, const Geom& g,
                                  const void* mesh_a, const void* mesh_b, void* half) {
  if (prec == NPC_PREC_FP64) {
    if (plan.n > 256) return set_err(ctx, NPC_ERR_UNSUPPORTED, "FP64 precision supports n <= 256");
    return fwd_dispatch<double>(ctx, plan, g, mesh_a, mesh_b, half);
  }
  return fwd_dispatch<float>(ctx, plan, g, mesh_a, mesh_b, half);
}

npc_status run_power_contract(npc_ctx* ctx, int prec, const PowerPlan& plan, const npc_mesh_spec& m,
                              const npc_kbins& kb, const void* half, const double* sc, double* dev_out) {
  if (prec == NPC_PREC_FP64) return contract_dispatch<double>(ctx, plan, m, kb, half, sc, dev_out);
  return contract_dispatch<float>(ctx, plan, m, kb, half, sc, dev_out);
}
