// kbc_aux.cuh -- kernels around the step: canonical-state transfer (init, get, set, moments),
// diagnostics, the stabilizer gap and the density pre-solve, with their Ops<S> launchers.
//
// Included at the end of kbc_kernels.cuh (it uses the step kernels' device code and host
// helpers); kept apart so that the step kernels' sources stay separate from these.
#pragma once

namespace kbc {
// ------------------------------------------------------------------ canonical addressing
// Address of canonical population i of node (x, y, z) at a time of the given parity.
template <typename S>
__device__ __forceinline__ S* canon_addr(S* b0, S* b1, const Geo& g, const Nbr& nb, int scheme,
                                         int parity, int i) {
  const uint32_t back = nb.ox[1 - cx(i)] + nb.oy[1 - cy(i)] + nb.oz[1 - cz(i)];
  const uint32_t here = nb.ox[1] + nb.oy[1] + nb.oz[1];
  if (scheme == 0) return (parity ? b1 : b0) + (uint64_t)i * g.P + back;
  if (parity == 0) return b0 + (uint64_t)i * g.P + here;
  return b0 + (uint64_t)(26 - i) * g.P + back;
}

// (32-bit arithmetic: a box holds fewer than 2^31 nodes; a 64-bit division would be a long
// software sequence)
__device__ __forceinline__ void node_coords(const Geo& g, uint64_t n, uint32_t& x, uint32_t& y,
                                            uint32_t& z) {
  const uint32_t m = (uint32_t)n;
  z = m / g.nxy;
  const uint32_t r = m - z * g.nxy;
  y = r / g.nx;
  x = r - y * g.nx;
}

// The same address for a compile-time layout: KIND 0 pull (buf = the buffer of parity t), 1 AA
// at even t, 2 AA at odd t (buf = the one AA buffer).
template <int KIND, int I, typename S>
__device__ __forceinline__ S* canon_ptr(S* buf, const Geo& g, const Nbr& nb) {
  if constexpr (KIND == 1) return buf + (uint64_t)I * g.P + nb.template at<I, 0>();
  else if constexpr (KIND == 0) return buf + (uint64_t)I * g.P + nb.template at<I, -1>();
  else return buf + (uint64_t)(26 - I) * g.P + nb.template at<I, -1>();
}

// ------------------------------------------------------------------ transfers
// The kernels between the stored shifts and the caller's FP64 fields. What they compute is a few
// operations per population, but GB300 converts to and from FP64 at the rate of its FP64 pipe (2
// lanes per SM and cycle): with a conversion and an addition there per population they ran at
// 2 to 15 times the time of their memory traffic. So the conversions are integer operations (a
// rebiased exponent), sums are integer sums and initial equilibria are computed in fixed point;
// the one FP64 operation left per population of get and set is the addition or subtraction of
// W. Values outside the normal ranges go to the compiler's conversions.

// 256^3, FP32 pull, one thread per node (before: a grid-stride loop with the layout picked at run
// time): get 1.83 -> 1.07 ms, set 1.65 -> 1.33, moments 4.05 -> 0.73, init 6.09 -> 0.77; their
// traffic alone takes 0.81, 0.81, 0.35, 0.33 ms. FP16: get 1.77 -> 1.06, set 2.52 -> 1.11, moments
// 4.06 -> 0.62, init 6.98 -> 0.87; FP64: get 1.29 -> 1.08, set 1.55 -> 1.11, moments 3.21 -> 0.76.
// Moments and init are bound by the integer pipe (moments: 400 instructions a node), get and set
// by DRAM and the FP64 addition together.

// FP32 to FP64 exactly for normal numbers; *odd is set for zero, subnormals, infinities and NaN
__device__ __forceinline__ double widen(float v, bool* odd) {
  const uint32_t b = __float_as_uint(v), a = b & 0x7fffffffu;
  *odd |= a - 0x00800000u >= 0x7f000000u;
  return __hiloint2double((int)((b & 0x80000000u) | ((a >> 3) + 0x38000000u)), (int)(b << 29));
}

// FP64 to FP32, rounded to nearest even, for results in the normal range below 2^64; *odd is set
// otherwise (zero too)
__device__ __forceinline__ float narrow(double v, bool* odd) {
  const uint32_t h = (uint32_t)__double2hiint(v), l = (uint32_t)__double2loint(v);
  const uint32_t a = h & 0x7fffffffu;
  *odd |= a - 0x38100000u >= 0x43f00000u - 0x38100000u;
  const uint32_t t = __funnelshift_l(l, a - 0x38000000u, 3);
  const uint32_t rest = l << 3;  // the 29 bits below the result's last
  const uint32_t r = t + (rest > 0x80000000u - (t & 1u) ? 1u : 0u);
  return __uint_as_float((h & 0x80000000u) | r);
}

// f_I = W_I + (stored value), and back, in FP64
template <typename S, int I> __device__ __forceinline__ double population_of(S v, bool* odd) {
  if constexpr (std::is_same<S, double>::value) return __dadd_rn(wgt(I), v);
  else if constexpr (std::is_same<S, float>::value) return __dadd_rn(wgt(I), widen(v, odd));
  else return __fma_rn(wgt(I), widen(__half2float(__ushort_as_half(v)), odd), wgt(I));
}
template <typename S, int I> __device__ __forceinline__ S stored_of(double f, bool* odd) {
  if constexpr (std::is_same<S, double>::value) {
    return __dadd_rn(f, -wgt(I));
  } else if constexpr (std::is_same<S, float>::value) {
    return narrow(__dadd_rn(f, -wgt(I)), odd);
  } else {
    // (f - W) / W in one rounding, to FP32 towards zero with the lost bits in the last one
    // (round to odd), so that the rounding to half is the only one
    const double d = __fma_rn(f, inv_wgt(I), -1.0);
    const uint32_t h = (uint32_t)__double2hiint(d), l = (uint32_t)__double2loint(d);
    const uint32_t a = h & 0x7fffffffu;
    *odd |= a - 0x38100000u >= 0x43f00000u - 0x38100000u;
    const uint32_t t = __funnelshift_l(l, a - 0x38000000u, 3) | ((l << 3) != 0 ? 1u : 0u);
    return __half_as_ushort(__float2half_rn(__uint_as_float((h & 0x80000000u) | t)));
  }
}

template <typename S, int KIND>
__global__ void __launch_bounds__(256) get_kernel(const S* buf, Geo g, double* out, uint64_t n0,
                                                  uint64_t cnt, uint64_t ld) {
  const uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (k >= cnt) return;
  uint32_t x, y, z;
  node_coords(g, n0 + k, x, y, z);
  Nbr nb;
  nb.init(g, x, y, z);
  S v[27];
  Unroll<0, 27>::run([&](auto ic) {
    constexpr int I = decltype(ic)::value;
    v[I] = *canon_ptr<KIND, I>(buf, g, nb);
  });
  bool odd = false;
  double f[27];
  Unroll<0, 27>::run([&](auto ic) {
    constexpr int I = decltype(ic)::value;
    f[I] = population_of<S, I>(v[I], &odd);
  });
  if (odd) {
    Unroll<0, 27>::run([&](auto ic) {
      constexpr int I = decltype(ic)::value;
      f[I] = wgt(I) + Codec<S>::to_delta(v[I], I);
    });
  }
#pragma unroll
  for (int i = 0; i < 27; ++i) out[i * ld + k] = f[i];
}

template <typename S, int KIND>
__global__ void __launch_bounds__(256) set_kernel(S* buf, Geo g, const double* in, uint64_t n0,
                                                  uint64_t cnt, uint64_t ld) {
  const uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (k >= cnt) return;
  uint32_t x, y, z;
  node_coords(g, n0 + k, x, y, z);
  Nbr nb;
  nb.init(g, x, y, z);
  double f[27];
#pragma unroll
  for (int i = 0; i < 27; ++i) f[i] = in[i * ld + k];
  bool odd = false;
  S v[27];
  Unroll<0, 27>::run([&](auto ic) {
    constexpr int I = decltype(ic)::value;
    v[I] = stored_of<S, I>(f[I], &odd);
  });
  if (odd) {
    Unroll<0, 27>::run([&](auto ic) {
      constexpr int I = decltype(ic)::value;
      v[I] = Codec<S>::from_delta(f[I] - wgt(I), I);
    });
  }
  Unroll<0, 27>::run([&](auto ic) {
    constexpr int I = decltype(ic)::value;
    *canon_ptr<KIND, I>(buf, g, nb) = v[I];
  });
}

// rho - 1 and rho u of 27 shifts in FP64 arithmetic
template <typename T>
__device__ __forceinline__ void moments_fp64(const T (&d)[27], double& drho, double (&m)[3]) {
  double s = 0.0, mx = 0.0, my = 0.0, mz = 0.0;
#pragma unroll
  for (int i = 0; i < 27; ++i) {
    const double dv = (double)d[i];
    s += dv;
    if (cx(i)) mx += cx(i) * dv;
    if (cy(i)) my += cy(i) * dv;
    if (cz(i)) mz += cz(i) * dv;
  }
  drho = s;
  m[0] = mx;
  m[1] = my;
  m[2] = mz;
}

// rho - 1 and u of 27 shifts (FP16: of shifts times 216, see load_shifts), in FP64. The shifts of a
// node are scaled to integers by the node's largest exponent (57 bits below it, so the sums are
// at least as exact as FP64 sums), summed, and the four sums converted; u is rho u times the
// reciprocal of rho. m, if given, receives rho u.
template <bool HALF, typename T>
__device__ __forceinline__ void velocity(const T (&d)[27], double& drho, double (&u)[3],
                                         double* m = nullptr) {
  constexpr int kMant = std::is_same<T, double>::value ? 52 : 23;
  constexpr int kBias = std::is_same<T, double>::value ? 1023 : 127;
  constexpr int kShift = sizeof(T) == 8 ? 20 : 23;
  uint32_t top = 0;  // the largest sign-free high word
#pragma unroll
  for (int i = 0; i < 27; ++i) {
    const uint32_t a = (uint32_t)(fix::bits_of(d[i]) >> (sizeof(T) == 8 ? 32 : 0)) & 0x7fffffffu;
    top = a > top ? a : top;
  }
  const int et = (int)(top >> kShift);  // biased exponent of the largest
  // the fast path: the largest value between 2^-100 and 1/4 (FP16: 54), rho within the range of
  // the fixed-point reciprocal
  bool fast = et > kBias - 100 && et < kBias - 2 + (HALF ? 8 : 0);
  if (fast) {
    fix::fx v[27];
#pragma unroll
    for (int i = 0; i < 27; ++i) {
      const auto b = fix::bits_of(d[i]);
      const uint32_t h = (uint32_t)(b >> (sizeof(T) == 8 ? 32 : 0));
      const uint32_t e = (h >> kShift) & (sizeof(T) == 8 ? 0x7ffu : 0xffu);
      // 1.mantissa with its leading bit at 63, shifted so that the largest has it at 57
      const uint64_t q = ((uint64_t)b << (63 - kMant)) | 0x8000000000000000ull;
      const fix::fx a = (fix::fx)fix::shr(e == 0 ? 0 : q, (uint32_t)et + 6u - e);
      v[i] = (int32_t)h < 0 ? -a : a;
    }
    // the four sums, x first
    fix::fx X0[9], X1[9];
#pragma unroll
    for (int r = 0; r < 9; ++r) {
      X0[r] = v[3 * r] + v[3 * r + 1] + v[3 * r + 2];
      X1[r] = v[3 * r + 2] - v[3 * r];
    }
    const fix::fx zm = X0[0] + X0[1] + X0[2], z0 = X0[3] + X0[4] + X0[5],
                  zp = X0[6] + X0[7] + X0[8];
    const fix::fx sum[4] = {zm + z0 + zp,
                            X1[0] + X1[1] + X1[2] + X1[3] + X1[4] + X1[5] + X1[6] + X1[7] + X1[8],
                            X0[2] + X0[5] + X0[8] - X0[0] - X0[3] - X0[6], zp - zm};
    // value = sum 2^(et - bias - 57)
    const int ex = et - kBias - 57;
    double val[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const double c = (double)sum[j];
      const int h = __double2hiint(c);
      val[j] = __hiloint2double(h == 0 ? 0 : h + ex * (1 << 20), __double2loint(c));
    }
    drho = val[0];
    if constexpr (HALF) drho *= 1.0 / 216.0;
    // rho in units of 2^-60 (FP16: 216 rho in units of 2^-52)
    const int sh = ex + (HALF ? 52 : 60);
    const fix::fx ds = sh >= 0 ? fix::shl(sum[0], sh) : (sh < -63 ? 0 : sum[0] >> -sh);
    const fix::fx r = HALF ? (216ll << 52) + ds : fix::kOne + ds;
    fast = r > fix::kOne / 2 && r < 2 * fix::kOne;
    if (fast) {
      // 1 / rho, or 1 / (216 rho) = 2^-8 / (r 2^-60)
      const double ir = fix::to_f64<HALF ? 8 : 0>(fix::reciprocal(r));
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        u[a] = __dmul_rn(val[a + 1], ir);
        if (m) m[a] = HALF ? val[a + 1] * (1.0 / 216.0) : val[a + 1];
      }
    }
  }
  if (!fast) {
    double j[3];
    moments_fp64(d, drho, j);
    if constexpr (HALF) drho /= 216.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if constexpr (HALF) j[a] /= 216.0;
      if (m) m[a] = j[a];
      u[a] = j[a] / (1.0 + drho);
    }
  }
}

// The shifts of a node for velocity(). FP16: times 216, which are exact FP32 numbers (the weights
// are 64 : 16 : 4 : 1).
template <typename S> struct ShiftType { using T = float; };
template <> struct ShiftType<double> { using T = double; };
template <typename S, int KIND>
__device__ __forceinline__ void load_shifts(const S* buf, const Geo& g, const Nbr& nb,
                                            typename ShiftType<S>::T (&d)[27]) {
  Unroll<0, 27>::run([&](auto ic) {
    constexpr int I = decltype(ic)::value;
    const S v = *canon_ptr<KIND, I>(buf, g, nb);
    if constexpr (std::is_same<S, uint16_t>::value)
      d[I] = __fmul_rn(__half2float(__ushort_as_half(v)), (float)(216.0 * wgt(I)));
    else
      d[I] = v;
  });
}

// rho and u of canonical f(t)
template <typename S, int KIND>
__global__ void __launch_bounds__(256) moments_kernel(const S* buf, Geo g, double* rho_out,
                                                      double* u_out, uint64_t n0, uint64_t cnt,
                                                      uint64_t ld) {
  const uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (k >= cnt) return;
  uint32_t x, y, z;
  node_coords(g, n0 + k, x, y, z);
  Nbr nb;
  nb.init(g, x, y, z);
  typename ShiftType<S>::T d[27];
  load_shifts<S, KIND>(buf, g, nb, d);
  double drho, u[3];
  velocity<std::is_same<S, uint16_t>::value>(d, drho, u);
  if (rho_out) rho_out[k] = 1.0 + drho;
#pragma unroll
  for (int a = 0; a < 3; ++a) u_out[a * ld + k] = u[a];
}

// f_eq(rho, u) in FP64 instructions, stored (FP64 storage, and nodes off the fixed-point range)
template <typename S, int KIND>
__device__ __noinline__ void init_node_fp64(S* buf, Geo g, uint32_t x, uint32_t y, uint32_t z,
                                            double rho, double ux, double uy, double uz) {
  Nbr nb;
  nb.init(g, x, y, z);
  double dq[27];
  equilibrium_shift<double>(rho, ux, uy, uz, dq);
  Unroll<0, 27>::run([&](auto ic) {
    constexpr int I = decltype(ic)::value;
    *canon_ptr<KIND, I>(buf, g, nb) = Codec<S>::from_delta(dq[I], I);
  });
}

// f_eq from its fixed-point populations; SHORT: FP32 by to_f32_short()
template <typename S, int KIND, bool SHORT>
__device__ __forceinline__ void init_store(S* buf, Geo g, uint32_t x, uint32_t y, uint32_t z,
                                           const fix::fx (&p)[27]) {
  Nbr nb;
  nb.init(g, x, y, z);
  Unroll<0, 27>::run([&](auto ic) {
    constexpr int I = decltype(ic)::value;
    constexpr int N = fix::nonzero(I);
    S* q = canon_ptr<KIND, I>(buf, g, nb);
    if constexpr (!std::is_same<S, float>::value)  // (f - W) / W = 27/8 4^N (f - W)
      *q = __half_as_ushort(__float2half_rn(fix::to_f32_odd<3 - N>(27 * p[I])));
    else if constexpr (SHORT)
      *q = fix::to_f32_short<N>(p[I]);
    else
      *q = fix::to_f32<N>(p[I]);
  });
}
// a node with populations (but for their weights) below 2^-22, out of line
template <typename S, int KIND>
__device__ __noinline__ void init_node_small(S* buf, Geo g, uint32_t x, uint32_t y, uint32_t z,
                                             fix::fx dr, fix::fx ux, fix::fx uy, fix::fx uz) {
  fix::fx p[27];
  fix::equilibrium(dr, ux, uy, uz, p);
  init_store<S, KIND, false>(buf, g, x, y, z, p);
}

// f = f_eq(rho, u). FP32 and FP16 storage: the equilibrium's moments and populations in fixed
// point (kbc_fix.cuh; 2^-59 absolute, far below the rounding of the stored values), for nodes
// whose velocity or density shift is at least 2^-18, so that this holds relative to the node too.
// The integer pipe bounds it (73 % busy); the writes are 0.32 of the FP32 kernel's 0.77 ms at 256^3.
template <typename S, int KIND>
__global__ void __launch_bounds__(256) init_kernel(S* buf, Geo g, const double* rho,
                                                   const double* u, uint64_t n0, uint64_t cnt,
                                                   uint64_t ld) {
  const uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (k >= cnt) return;
  uint32_t x, y, z;
  node_coords(g, n0 + k, x, y, z);
  const double r = rho ? rho[k] : 1.0, ux = u[k], uy = u[ld + k], uz = u[2 * ld + k];
  if constexpr (!std::is_same<S, double>::value) {
    const double dr = r - 1.0;
    uint32_t top = 0;
    const fix::fx v[4] = {fix::from_f64(dr, &top), fix::from_f64(ux, &top),
                          fix::from_f64(uy, &top), fix::from_f64(uz, &top)};
    if (top < fix::kTopF64 && top >= 0x3ed00000u) {
      fix::fx p[27];
      fix::equilibrium(v[0], v[1], v[2], v[3], p);
      if constexpr (std::is_same<S, float>::value) {
        bool all = true;
#pragma unroll
        for (int i = 0; i < 27; ++i) all = all && fix::short_way(p[i]);
        if (!all) return init_node_small<S, KIND>(buf, g, x, y, z, v[0], v[1], v[2], v[3]);
      }
      return init_store<S, KIND, true>(buf, g, x, y, z, p);
    }
  }
  init_node_fp64<S, KIND>(buf, g, x, y, z, r, ux, uy, uz);
}

// ------------------------------------------------------------------ diagnostics
// Sums (FP64) in partials[block * kDiagSums + j], over the nodes whose rho and u are finite
// (0-10) or whose velocity gradients are finite (11-19):
//  0 sum (rho - 1), 1-3 sum rho u, 4-6 sum u, 7 unused, 8 sum gamma, 9 sum gamma^2,
//  10 non-finite nodes, 11 sum |curl u|^2, 12 sum (d_b u_a + d_a u_b)^2,
//  13-17 sum (d u_x / d x)^n for n = 2..6, 18 sum |u - <u>|^2 (second pass, with <u> from the
//  first), 19 nodes with finite gradients
//
// Warp sums by halving: a lane gives half of its values away at each step and adds the other
// half's, so that N <= 16 values cost 16 FP64 additions a lane and not 5 N (on GB300's FP64 pipe
// the trees of 11 and 9 values took most of a 32^3 diagnostics' 40 us).
template <int O, int M>
__device__ __forceinline__ void halve(double (&v)[M > 0 ? 2 * M : 1], int lane, int& slot,
                                      double& sum) {
  if constexpr (M == 0) {
    sum = v[0];
#pragma unroll
    for (int o = O; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  } else {
    const bool up = lane & O;
    double w[M];
#pragma unroll
    for (int j = 0; j < M; ++j) {
      const double give = up ? v[j] : v[j + M], keep = up ? v[j + M] : v[j];
      w[j] = keep + __shfl_xor_sync(0xffffffffu, give, O);
    }
    if (up) slot += M;
    halve<O / 2, M / 2>(w, lane, slot, sum);
  }
}

template <int N>
__device__ __forceinline__ void block_reduce_store(const double (&in)[N], double* dst) {
  constexpr int M = N > 8 ? 16 : 8;
  __shared__ double sh[32][M];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double v[M], sum;
#pragma unroll
  for (int j = 0; j < M; ++j) v[j] = j < N ? in[j] : 0.0;
  int slot = 0;
  halve<16, M / 2>(v, lane, slot, sum);
  if ((lane & (32 / M - 1)) == 0) sh[warp][slot] = sum;
  __syncthreads();
  if (threadIdx.x < N) {
    double acc = 0.0;
    const int nw = (blockDim.x + 31) >> 5;
    for (int w = 0; w < nw; ++w) acc += sh[w][threadIdx.x];
    dst[threadIdx.x] = acc;
  }
}

// isfinite() without the FP64 pipe's compare
__device__ __forceinline__ bool finite_bits(double v) {
  return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000;
}
__device__ __forceinline__ bool finite_bits(float v) {
  return (__float_as_uint(v) & 0x7f800000u) != 0x7f800000u;
}

// rho - 1 and rho u of canonical f(t) at one node, in the arithmetic type of the storage
template <typename S, int KIND>
__device__ __forceinline__ void node_moments_r(const S* buf, const Geo& g, const Nbr& nb,
                                               typename Codec<S>::R& drho,
                                               typename Codec<S>::R (&m)[3]) {
  using R = typename Codec<S>::R;
  R s = R(0), mx = R(0), my = R(0), mz = R(0);
  Unroll<0, 27>::run([&](auto ic) {
    constexpr int I = decltype(ic)::value;
    const R dv = Codec<S>::template load<I>(canon_ptr<KIND, I>(buf, g, nb));
    s += dv;
    if constexpr (cx(I) != 0) mx += R(cx(I)) * dv;
    if constexpr (cy(I) != 0) my += R(cy(I)) * dv;
    if constexpr (cz(I) != 0) mz += R(cz(I)) * dv;
  });
  drho = s;
  m[0] = mx;
  m[1] = my;
  m[2] = mz;
}

// Per-node quantities in the storage's arithmetic type; block and global sums in FP64.
// 4 blocks of 256 threads per SM: the fixed grid of 608 blocks is then resident in one wave (FP64:
// 2 blocks, whose integer sums need 128 registers)
template <typename S, int KIND>
__global__ void __launch_bounds__(256, std::is_same<S, double>::value ? 2 : 4) diag_fields_kernel(const S* buf, Geo g,
                                                          const float* gamma, int with_gamma,
                                                          typename Codec<S>::R* uf,
                                                          double* partials) {
  using R = typename Codec<S>::R;
  // per-thread sums in R (FP64 arithmetic per node would saturate GB300's FP64 pipe); the
  // density enters as rho - 1 so that FP32 sums keep their relative accuracy
  R acc[11] = {R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0)};
  for (uint64_t n = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; n < g.P;
       n += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t x, y, z;
    node_coords(g, n, x, y, z);
    Nbr nb;
    nb.init(g, x, y, z);
    R drho, m[3], ux, uy, uz;
    if constexpr (std::is_same<S, double>::value) {
      // integer sums: the FP64 pipe would take 130 operations a node for the moments
      double d[27], uu[3];
      load_shifts<S, KIND>(buf, g, nb, d);
      velocity<false>(d, drho, uu, m);
      ux = uu[0], uy = uu[1], uz = uu[2];
    } else {
      node_moments_r<S, KIND>(buf, g, nb, drho, m);
      const R ir = R(1) / (R(1) + drho);
      ux = m[0] * ir, uy = m[1] * ir, uz = m[2] * ir;
    }
    const R rho = R(1) + drho;
    uf[n] = ux;
    uf[g.P + n] = uy;
    uf[2 * g.P + n] = uz;
    if (!finite_bits(rho) || !finite_bits(ux) || !finite_bits(uy) || !finite_bits(uz)) {
      acc[10] += R(1);
      continue;
    }
    acc[0] += drho;
    acc[1] += m[0];
    acc[2] += m[1];
    acc[3] += m[2];
    acc[4] += ux;
    acc[5] += uy;
    acc[6] += uz;
    if (with_gamma) {
      const R gm = (R)gamma[n];
      acc[8] += gm;
      acc[9] += gm * gm;
    }
  }
  double v[11];
#pragma unroll
  for (int j = 0; j < 11; ++j) v[j] = (double)acc[j];
  block_reduce_store<11>(v, partials + blockIdx.x * kDiagSums);
}

// central-difference coefficients c_k of d u / d x = sum_k c_k (u(x + k) - u(x - k)):
// second order (K = 1) and eighth order (K = 4)
template <int K> struct FdCoef;
template <> struct FdCoef<1> {
  static __device__ __forceinline__ double c(int) { return 0.5; }
};
template <> struct FdCoef<4> {
  static __device__ __forceinline__ double c(int k) {
    return k == 1 ? 4.0 / 5.0 : k == 2 ? -1.0 / 5.0 : k == 3 ? 4.0 / 105.0 : -1.0 / 280.0;
  }
};

// Per-thread sums in the arithmetic type R (a thread covers about P / 155,648 nodes, ~100 at
// 256^3; FP64 arithmetic per node would saturate GB300's FP64 pipe), then FP64 from the
// block reduction on.
template <typename R, int K>
__global__ void __launch_bounds__(256) diag_grad_kernel(Geo g, const R* uf, const double* sums,
                                                        double* partials) {
  R acc[9] = {R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0)};
  const uint32_t dims[3] = {g.nx, g.ny, g.nz};
  // <u> over the finite nodes, from the sums of the first pass
  const double nfin = (double)g.P - sums[10];
  const R mean[3] = {(R)(sums[4] / nfin), (R)(sums[5] / nfin), (R)(sums[6] / nfin)};
  for (uint64_t n = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; n < g.P;
       n += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t c[3];
    node_coords(g, n, c[0], c[1], c[2]);
    R gr[3][3];  // gr[a][b] = d u_a / d x_b
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) gr[a][b] = R(0);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int64_t stride = b == 0 ? 1 : b == 1 ? (int64_t)g.nx : (int64_t)g.nxy;
      const int64_t dim = dims[b];
      // periodic neighbours c_b + k and c_b - k, stepped one node at a time so that each
      // step wraps at most once (the stencil may go round a 3-node box more than once)
      int64_t cp = c[b], cm = c[b];
#pragma unroll
      for (int k = 1; k <= K; ++k) {
        ++cp;
        if (cp >= dim) cp -= dim;
        --cm;
        if (cm < 0) cm += dim;
        const uint64_t np = n + (cp - (int64_t)c[b]) * stride;
        const uint64_t nm = n + (cm - (int64_t)c[b]) * stride;
        const R ck = (R)FdCoef<K>::c(k);
#pragma unroll
        for (int a = 0; a < 3; ++a) gr[a][b] += ck * (uf[a * g.P + np] - uf[a * g.P + nm]);
      }
    }
    const R wx = gr[2][1] - gr[1][2], wy = gr[0][2] - gr[2][0], wz = gr[1][0] - gr[0][1];
    const R ww = wx * wx + wy * wy + wz * wz;
    R ss = R(0);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const R s = gr[a][b] + gr[b][a];
        ss += s * s;
      }
    if (finite_bits(ww) && finite_bits(ss)) {
      acc[0] += ww;
      acc[1] += ss;
      const R q = gr[0][0];
      R qn = q * q;
#pragma unroll
      for (int m = 2; m <= 6; ++m) {
        acc[m] += qn;
        qn *= q;
      }
      acc[8] += R(1);
    }
    const R d0 = uf[n] - mean[0], d1 = uf[g.P + n] - mean[1], d2 = uf[2 * g.P + n] - mean[2];
    const R dd = d0 * d0 + d1 * d1 + d2 * d2;
    if (finite_bits(dd)) acc[7] += dd;
  }
  double v[9];
#pragma unroll
  for (int j = 0; j < 9; ++j) v[j] = (double)acc[j];
  block_reduce_store<9>(v, partials + blockIdx.x * kDiagSums + 11);
}

// Fixed-order final reduction of the slots [first, first + blockDim.x / 32): sums[j] = sum over
// blocks of partials[block][j], a warp per slot (each lane every 32nd block, then the lanes). One
// thread per slot over 608 blocks took 54 us a call, as long as a 32^3 diagnostics otherwise.
// With counters given, slots 20 and 21 take the guard count and the timeout flag, so that one
// copy brings the host everything.
static __global__ void diag_final_kernel(const double* partials, int nblocks, int first,
                                         double* sums, const StepCounters* ctr) {
  const int j = first + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  double acc = 0.0;
  for (int b = lane; b < nblocks; b += 32) acc += partials[b * kDiagSums + j];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if (lane == 0) sums[j] = acc;
  if (ctr && threadIdx.x == 0) {
    sums[20] = (double)ctr->guarded;
    sums[21] = (double)ctr->timeout;
  }
}

// Stabilizer gap on canonical f(t): per node the estimate eq:result21 and the root of
// eq:result1 from the same collision inputs. Partial sums per block: [0] nodes evaluated,
// [1] sum |gamma_est - gamma*|, [2] sum gamma_est, [3] sum gamma*, [4] nodes where the Newton
// iteration did not converge, [5] nodes skipped (guarded or non-finite), [6] max |difference|.
constexpr int kGapSums = 7;
template <typename S, bool CENTRAL>
__global__ void __launch_bounds__(256) gap_kernel(const S* b0, const S* b1, Geo g, int scheme,
                                                  int parity, CollideParams cp,
                                                  double* partials) {
  using R = typename Codec<S>::R;
  double v[6] = {0, 0, 0, 0, 0, 0};
  double vmax = 0.0;
  for (uint64_t n = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; n < g.P;
       n += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t x, y, z;
    node_coords(g, n, x, y, z);
    Nbr nb;
    nb.init(g, x, y, z);
    R d[27];
    Unroll<0, 27>::run([&](auto ic) {
      constexpr int I = decltype(ic)::value;
      d[I] = Codec<S>::template load<I>(canon_addr<S>((S*)b0, (S*)b1, g, nb, scheme, parity, I));
    });
    int guarded, status = 1;
    R gest = R(0);
    const R gex = collide<R, CENTRAL, true>(d, cp, &guarded, &gest, &status);
    if (guarded || !(gex == gex) || !(gest == gest)) {
      v[5] += 1.0;
      continue;
    }
    const double diff = fabs((double)gex - (double)gest);
    v[0] += 1.0;
    v[1] += diff;
    v[2] += (double)gest;
    v[3] += (double)gex;
    if (status != 0) v[4] += 1.0;
    vmax = fmax(vmax, diff);
  }
  block_reduce_store<6>(v, partials + blockIdx.x * kDiagSums);
  // block maximum
  __shared__ double shm[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) vmax = fmax(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) shm[warp] = vmax;
  __syncthreads();
  if (threadIdx.x == 0) {
    double m = 0.0;
    for (int w = 0; w < (int)((blockDim.x + 31) >> 5); ++w) m = fmax(m, shm[w]);
    partials[blockIdx.x * kDiagSums + 6] = m;
  }
}

// fixed-order final reduction of the gap partials, a warp per slot (slot 6 by maximum)
static __global__ void gap_final_kernel(const double* partials, int nblocks, double* sums) {
  const int j = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double acc = 0.0;
  for (int b = lane; b < nblocks; b += 32) {
    const double p = partials[b * kDiagSums + j];
    acc = j == 6 ? fmax(acc, p) : acc + p;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double p = __shfl_down_sync(0xffffffffu, acc, o);
    acc = j == 6 ? fmax(acc, p) : acc + p;
  }
  if (lane == 0) sums[j] = acc;
}

// ------------------------------------------------------------------ density pre-solve
// rho - 1 of 27 stored shifts, for the density change of the pre-solve
__device__ __forceinline__ float presolve_drho(const float (&d)[27]) {
  float s = 0.0f;
#pragma unroll
  for (int i = 0; i < 27; ++i) s += d[i];
  return s;
}
__device__ __forceinline__ double presolve_drho(const double (&d)[27]) {
  fix::fx v[27], sum;
  uint32_t s, top;
  bool in_range;
  return fix::presolve_density(d, v, &sum, &s, &top, &in_range);
}

// One iteration of the consistent-initialisation loop (Sec. "Numerical Simulations", after
// Mei et al.): f' = f - 2 beta_pre (f - f_eq(rho(f), u0(x))) with the velocity held at u0,
// streamed by the pattern of MODE. u0 is [3][P] in the collision precision. With `store`
// set, rho - 1 of the loaded state is kept in rho_prev (FP32) for rho_change_kernel.
template <typename S, int MODE>
__global__ void __launch_bounds__(MaxThreads<S>::value) presolve_kernel(
    const S* src, S* dst, Geo g, typename Codec<S>::R beta2, const typename Codec<S>::R* u0,
    float* rho_prev, int store) {
  using C = Codec<S>;
  using R = typename C::R;
  using Pat = Pattern<MODE>;
  const uint32_t x = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t y = blockIdx.y * blockDim.y + threadIdx.y;
  const uint32_t z = blockIdx.z;
  if (x >= g.nx || y >= g.ny) return;
  Nbr nb;
  nb.init(g, x, y, z);
  R d[27];
  Unroll<0, 27>::run([&](auto ic) {
    constexpr int I = decltype(ic)::value;
    d[I] = C::template load<I>(src + (uint64_t)Pat::load_plane(I) * g.P +
                               nb.template at<I, Pat::load_shift>());
  });
  const R s = presolve_drho(d);
  const uint32_t n = nb.ox[1] + nb.oy[1] + nb.oz[1];
  R eq[27];
  equilibrium_shift<R>(R(1) + s, u0[n], u0[g.P + n], u0[2 * g.P + n], eq);
#pragma unroll
  for (int i = 0; i < 27; ++i) d[i] -= beta2 * (d[i] - eq[i]);
  Unroll<0, 27>::run([&](auto ic) {
    constexpr int I = decltype(ic)::value;
    C::template store<I>(dst + (uint64_t)Pat::store_plane(I) * g.P +
                             nb.template at<I, Pat::store_shift>(),
                         d[I]);
  });
  if (store) rho_prev[n] = (float)s;
}

// one node of the FP64 pre-solve in FP64 instructions
template <int MODE>
__device__ __noinline__ void presolve_node_fp64(const double* src, double* dst, Geo g,
                                                double beta2, double ux, double uy, double uz,
                                                uint32_t x, uint32_t y, uint32_t z) {
  using Pat = Pattern<MODE>;
  Nbr nb;
  nb.init(g, x, y, z);
  double d[27];
  Unroll<0, 27>::run([&](auto ic) {
    constexpr int I = decltype(ic)::value;
    d[I] = src[(uint64_t)Pat::load_plane(I) * g.P + nb.template at<I, Pat::load_shift>()];
  });
  double s = 0.0;
#pragma unroll
  for (int i = 0; i < 27; ++i) s += d[i];
  double eq[27];
  equilibrium_shift<double>(1.0 + s, ux, uy, uz, eq);
  Unroll<0, 27>::run([&](auto ic) {
    constexpr int I = decltype(ic)::value;
    dst[(uint64_t)Pat::store_plane(I) * g.P + nb.template at<I, Pat::store_shift>()] =
        d[I] - beta2 * (d[I] - eq[I]);
  });
}

// The FP64 pre-solve step in fixed point (kbc_fix.cuh), one node per thread over the node order;
// nodes outside the format's range are stepped in FP64. FULL: beta2 = 1, the default relaxation,
// sets f to f_eq, so that the populations are only summed. 100^3 AA: 564 -> 117 us an iteration
// (456 B a node: 68 us), 141 for a general beta2; bound by the integer pipe (FP64: by the FP64
// pipe, ~190 operations a node).
template <int MODE, bool FULL>
__global__ void __maxnreg__(128) presolve_fix_kernel(const double* src, double* dst, Geo g,
                                                     double beta2, const double* u0,
                                                     float* rho_prev, int store) {
  using Pat = Pattern<MODE>;
  wait_before();
  const uint32_t n = blockIdx.x * blockDim.x + threadIdx.x;  // P < 2^31
  if (n >= g.P) return;
  const uint32_t row = n / g.nx;
  const uint32_t x = n - row * g.nx;
  const uint32_t z = row / g.ny;
  const uint32_t y = row - z * g.ny;
  Nbr nb;
  nb.init(g, x, y, z);
  double d[27];
  Unroll<0, 27>::run([&](auto ic) {
    constexpr int I = decltype(ic)::value;
    d[I] = src[(uint64_t)Pat::load_plane(I) * g.P + nb.template at<I, Pat::load_shift>()];
  });
  const double ux = u0[n], uy = u0[g.P + n], uz = u0[2 * g.P + n];
  fix::fx p[27];
  uint32_t sc;
  double drho;
  const bool ok = fix::presolve<FULL>(d, ux, uy, uz, beta2, p, &sc, &drho);
  if (store) rho_prev[n] = (float)drho;
  if (!ok) {
    presolve_node_fp64<MODE>(src, dst, g, beta2, ux, uy, uz, x, y, z);
    return;
  }
  Unroll<0, 27>::run([&](auto ic) {
    constexpr int I = decltype(ic)::value;
    dst[(uint64_t)Pat::store_plane(I) * g.P + nb.template at<I, Pat::store_shift>()] =
        fix::to_f64<fix::nonzero(I)>(p[I], sc);
  });
}

// *resid = max over nodes of |(rho - 1) of canonical f(t) - rho_prev| in FP32 (as the bits of
// a non-negative float, so that atomicMax orders them); NaN is raised to +Inf.
template <typename S, int KIND>
__global__ void __launch_bounds__(256) rho_change_kernel(const S* buf, Geo g,
                                                         const float* rho_prev,
                                                         unsigned int* resid) {
  using R = typename Codec<S>::R;
  float m = 0.0f;
  for (uint64_t n = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; n < g.P;
       n += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t x, y, z;
    node_coords(g, n, x, y, z);
    Nbr nb;
    nb.init(g, x, y, z);
    R d[27];
    Unroll<0, 27>::run([&](auto ic) {
      constexpr int I = decltype(ic)::value;
      d[I] = Codec<S>::template load<I>(canon_ptr<KIND, I>(buf, g, nb));
    });
    float ch = fabsf((float)presolve_drho(d) - rho_prev[n]);
    if (!(ch == ch)) ch = INFINITY;
    m = fmaxf(m, ch);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(resid, __float_as_uint(m));
}

// ufield[a * P + n0 + k] = (R) u[a * ld + k]
template <typename R>
__global__ void convert_u_kernel(const double* u, R* ufield, uint64_t n0, uint64_t cnt,
                                 uint64_t ld, uint64_t P) {
  for (uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; k < cnt;
       k += (uint64_t)gridDim.x * blockDim.x) {
#pragma unroll
    for (int a = 0; a < 3; ++a) ufield[a * P + n0 + k] = (R)u[a * ld + k];
  }
}

// launch<KIND>(buffer) for the layout of a box at time t
template <typename S, typename F>
static cudaError_t with_layout(const BoxView& b, int64_t t, F&& launch) {
  const int parity = (int)(t & 1);
  if (b.scheme == 0) launch(std::integral_constant<int, 0>{}, (S*)b.pop[parity]);
  else if (parity == 0) launch(std::integral_constant<int, 1>{}, (S*)b.pop[0]);
  else launch(std::integral_constant<int, 2>{}, (S*)b.pop[0]);
  return cudaGetLastError();
}
inline unsigned node_blocks(uint64_t cnt) { return (unsigned)((cnt + 255) / 256); }

template <typename S>
cudaError_t Ops<S>::init(const BoxView& b, int64_t t, const double* rho, const double* u,
                         uint64_t n0, uint64_t cnt, uint64_t ld, cudaStream_t st) {
  return with_layout<S>(b, t, [&](auto kind, S* buf) {
    init_kernel<S, decltype(kind)::value><<<node_blocks(cnt), 256, 0, st>>>(
        buf, make_geo(b), rho, u, n0, cnt, ld);
  });
}

template <typename S>
cudaError_t Ops<S>::get(const BoxView& b, int64_t t, double* out, uint64_t n0, uint64_t cnt,
                        uint64_t ld, cudaStream_t st) {
  return with_layout<S>(b, t, [&](auto kind, S* buf) {
    get_kernel<S, decltype(kind)::value><<<node_blocks(cnt), 256, 0, st>>>(buf, make_geo(b), out,
                                                                           n0, cnt, ld);
  });
}

template <typename S>
cudaError_t Ops<S>::set(const BoxView& b, int64_t t, const double* in, uint64_t n0,
                        uint64_t cnt, uint64_t ld, cudaStream_t st) {
  return with_layout<S>(b, t, [&](auto kind, S* buf) {
    set_kernel<S, decltype(kind)::value><<<node_blocks(cnt), 256, 0, st>>>(buf, make_geo(b), in,
                                                                           n0, cnt, ld);
  });
}

template <typename S>
cudaError_t Ops<S>::moments(const BoxView& b, int64_t t, double* rho, double* u, uint64_t n0,
                            uint64_t cnt, uint64_t ld, cudaStream_t st) {
  return with_layout<S>(b, t, [&](auto kind, S* buf) {
    moments_kernel<S, decltype(kind)::value><<<node_blocks(cnt), 256, 0, st>>>(
        buf, make_geo(b), rho, u, n0, cnt, ld);
  });
}

template <typename S>
cudaError_t Ops<S>::presolve_step(const BoxView& b, int64_t t, double beta_pre, const void* u0,
                                  bool store, const StepOpts& o, cudaStream_t st) {
  using R = typename Codec<S>::R;
  const Geo g = make_geo(b);
  const R beta2 = (R)(2.0 * beta_pre);
  const int parity = (int)(t & 1);
  auto run = [&](auto mode, const void* from, void* to) {
    constexpr int M = decltype(mode)::value;
    const S* src = (const S*)from;
    S* dst = (S*)to;
    const R* u = (const R*)u0;
    const int keep = store ? 1 : 0;
    if constexpr (std::is_same<S, double>::value) {
      const unsigned blocks = (unsigned)((g.P + 127) / 128);
      return beta2 == 1.0 ? launch_following(presolve_fix_kernel<M, true>, blocks, 128, st, src,
                                             dst, g, beta2, u, b.gamma, keep)
                          : launch_following(presolve_fix_kernel<M, false>, blocks, 128, st, src,
                                             dst, g, beta2, u, b.gamma, keep);
    } else {
      const dim3 block(o.bx, o.by, 1);
      const dim3 grid((b.nx + o.bx - 1) / o.bx, (b.ny + o.by - 1) / o.by, b.nz);
      presolve_kernel<S, M><<<grid, block, 0, st>>>(src, dst, g, beta2, u, b.gamma, keep);
      return cudaGetLastError();
    }
  };
  if (b.scheme == 0)
    return run(std::integral_constant<int, MODE_PULL>{}, b.pop[parity], b.pop[parity ^ 1]);
  if (parity == 0) return run(std::integral_constant<int, MODE_AA_EVEN>{}, b.pop[0], b.pop[0]);
  return run(std::integral_constant<int, MODE_AA_ODD>{}, b.pop[0], b.pop[0]);
}

template <typename S>
cudaError_t Ops<S>::rho_change(const BoxView& b, int64_t t, unsigned int* resid, int nblocks,
                               cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(resid, 0, sizeof(unsigned int), st);
  if (e != cudaSuccess) return e;
  return with_layout<S>(b, t, [&](auto kind, S* buf) {
    rho_change_kernel<S, decltype(kind)::value><<<nblocks, 256, 0, st>>>(buf, make_geo(b), b.gamma,
                                                                         resid);
  });
}

template <typename S>
cudaError_t Ops<S>::convert_u(const double* u, void* ufield, uint64_t n0, uint64_t cnt,
                              uint64_t ld, uint64_t P, cudaStream_t st) {
  using R = typename Codec<S>::R;
  convert_u_kernel<R><<<grid_for(cnt, 256), 256, 0, st>>>(u, (R*)ufield, n0, cnt, ld, P);
  return cudaGetLastError();
}

template <typename S>
cudaError_t Ops<S>::gamma_gap(const BoxView& b, int64_t t, double* partials, int nblocks,
                              double* sums, cudaStream_t st) {
  const Geo g = make_geo(b);
  CollideParams cp = make_cp(b.beta, b.with_t, b.with_q, GAMMA_EXACT);
  if (b.central)
    gap_kernel<S, true><<<nblocks, 256, 0, st>>>((const S*)b.pop[0], (const S*)b.pop[1], g,
                                                 b.scheme, (int)(t & 1), cp, partials);
  else
    gap_kernel<S, false><<<nblocks, 256, 0, st>>>((const S*)b.pop[0], (const S*)b.pop[1], g,
                                                  b.scheme, (int)(t & 1), cp, partials);
  gap_final_kernel<<<1, 32 * kGapSums, 0, st>>>(partials, nblocks, sums);
  return cudaGetLastError();
}

template <typename S>
cudaError_t Ops<S>::diag(const BoxView& b, int64_t t, bool with_gamma, int order, void* ufield,
                         double* partials, int nblocks, double* sums, const StepCounters* ctr,
                         cudaStream_t st) {
  using R = typename Codec<S>::R;
  const Geo g = make_geo(b);
  // blocks without a node would only reduce zeros
  if ((uint64_t)nblocks * 256 > g.P) nblocks = (int)((g.P + 255) / 256);
  const int parity = (int)(t & 1);
  const int wg = with_gamma ? 1 : 0;
  if (b.scheme == 0)
    diag_fields_kernel<S, 0><<<nblocks, 256, 0, st>>>((const S*)b.pop[parity], g, b.gamma, wg,
                                                      (R*)ufield, partials);
  else if (parity == 0)
    diag_fields_kernel<S, 1><<<nblocks, 256, 0, st>>>((const S*)b.pop[0], g, b.gamma, wg,
                                                      (R*)ufield, partials);
  else
    diag_fields_kernel<S, 2><<<nblocks, 256, 0, st>>>((const S*)b.pop[0], g, b.gamma, wg,
                                                      (R*)ufield, partials);
  if (order == 0) return cudaGetLastError();
  // <u> for the second pass
  diag_final_kernel<<<1, 11 * 32, 0, st>>>(partials, nblocks, 0, sums, nullptr);
  if (order == 8)
    diag_grad_kernel<R, 4><<<nblocks, 256, 0, st>>>(g, (const R*)ufield, sums, partials);
  else
    diag_grad_kernel<R, 1><<<nblocks, 256, 0, st>>>(g, (const R*)ufield, sums, partials);
  diag_final_kernel<<<1, 9 * 32, 0, st>>>(partials, nblocks, 11, sums, ctr);
  return cudaGetLastError();
}

}  // namespace kbc
