// FP64 and FP64-accurate radiation integral through Chebyshev moments (sm_103a).
//
// The direct kernels (rad_fp64.cu, rad_df.cu) evaluate one sin/cos per (sample, photon energy,
// direction). Over a run of samples whose phase lengths a_k from the run's centre stay within
// a_lim, the factor e^{i w a_k} of every photon energy w <= w_hi is a short Chebyshev series in
// x_k = a_k / a_lim (Jacobi-Anger):
//   e^{i w a_k} = sum_m (2 - delta_m0) i^m J_m(w a_lim) T_m(x_k),
// so the run's amplitude is a combination of kM real moments that do not depend on the energy:
//   sum_k f_k e^{i w a_k} = sum_m (2 - delta_m0) i^m J_m(w a_lim) M_m,  M_m = sum_k f_k T_m(x_k).
// A sample then costs one recurrence step and one multiply-add per component and moment whatever
// the number of energies, and an energy costs kM multiply-adds per component, one sin/cos of the
// run's base phase and one rotation per run instead of per sample. Spin 1/2 has three components and keeps 24
// moments, the others 32; w_hi a_lim (Cheb::kPhi) keeps the first dropped term below the form's rounding;
// terms that are below 1e-18 at an energy's own w a_lim are left out for it.
//
// Work split: a block of 4 warps takes 32 directions (one per lane: x_k, the recurrence and the
// moments live in the lane's registers and need no exchange) and the energies of one tile. The warps
// take a quarter of a run's samples each, add their moments through shared memory and then take a
// quarter of the energies each. Amplitudes are kept in a block's own scratch, [energy][component]
// [lane], one coalesced read and write per run and energy.
//
// DF = false: everything FP64. DF = true: the phase lengths, f and the base phase are formed in
// FP64, the moments, the series and the rotations in the float-pair arithmetic of rad_df.cu
// (products by FMA, Ogita-Rump-Oishi Dot2 sums), because GB300 executes FP64 at 1/64 of its FP32
// rate: a float-pair multiply-add takes about a sixth of the time of an FP64 one.
//
// What bounds it: the FP64 pipe (86 % busy on the sections below) in FP64; latency at 8 warps an SM in float pairs
// (255 registers a thread hold the moments, with 60 to 76 bytes of spill stores; 48 % of the issue slots). Measured, all kernels
// of a call, before (direct kernel alone) and with it: one undulator, 4096 samples x 128 energies x 256 directions, FP64, 4.49
// -> 0.46 to 0.56 ms (from run to run); 64 sections of 500 samples x 192 log energies x 324 directions, spin 1/2, FP64, 80.9 ->
// 41.8 ms (the 64 highest energies stay direct: 25.7 ms of it); 20 undulator periods, 40960 samples x 500 energies x 225
// directions, float pairs, 21.6 -> 5.2 ms; 6 positrons x 12000 samples x 384 log energies x 576 directions, spin 1/2, float
// pairs, 108 -> 57 ms. Tried and slower: 28 moments for spin 1/2 (41.1 against 39.6 ms, and spills in float pairs), 24
// for the other models (5.6 -> 7.2 ms); 4 KB of base phases in shared memory instead of 1 (one block an SM in spin 1/2).
#include <type_traits>

#include "rad_df_reduce.cuh"
#include "rad_fp64_sincos.cuh"
#include "rad_internal.cuh"

namespace rad {
namespace {

constexpr int kW = 4;        // warps per block
constexpr int kWin = 256;    // samples of a window, the longest run
constexpr int kRecW = 10;    // doubles per prepared sample
// A particle's amplitudes are added up over kFlush runs at a time and these sums in FP64: the rounding of each
// addition grows with the sum that it is added to (in one float-pair sum over the 2000 runs of 12000
// samples the spectrum was off by 1.1e-12, in FP64 by 1.1e-15; 2e-14 and 8e-16 by the direct kernels).
template <bool DF>
constexpr int kFlush = DF ? 64 : 16;

template <int MODE>
struct Cheb {
  static constexpr bool kSpin = MODE == RAD_SPIN_HALF;
  static constexpr int NP = kSpin ? 3 : 2;   // summed components (f_x, f_y, j)
  static constexpr int kM = kSpin ? 24 : 32;
  // Phase range w_hi a_lim. The samples of a run end at x = +-1, and where they add up coherently the tile's
  // highest energies see the first dropped term, 2 J_kM(kPhi), at about a quarter: it is held to 1e-16
  // of |f| in FP64 (at 5 and 9 it was 9e-15 and 4e-15: 4e-15 of the spectrum at the top of a tile), and below the
  // float pairs' own 1e-14 in double-float.
  template <bool DF>
  static constexpr double kPhi = kSpin ? (DF ? 5.0 : 4.25) : (DF ? 9.0 : 8.25);
  static constexpr int kTile = kSpin ? 256 : 512;  // energies of a tile
};

// float pair
struct df2 {
  float h, l;
};

__device__ __forceinline__ df2 df_norm(float a, float b) {  // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

// 2 x t - u
__device__ __forceinline__ df2 df_rec(const df2 &x2, const df2 &t, const df2 &u) {
  const float p = __fmul_rn(x2.h, t.h);
  float e = __fmaf_rn(x2.h, t.h, -p);
  e = __fmaf_rn(x2.h, t.l, __fmaf_rn(x2.l, t.h, e));
  float s, r;
  dfr::two_sum(p, -u.h, s, r);
  return df_norm(s, __fadd_rn(r, __fsub_rn(e, u.l)));
}

__device__ __forceinline__ df2 to_df(double v) {
  df2 r;
  dfr::split_df(v, r.h, r.l);
  return r;
}

// s + v, its rounding error added to e (Knuth's TwoSum); s - a b the same
__device__ __forceinline__ void add_err(double &s, double &e, double v) {
  const double t = s + v, b = t - s;
  e += (s - (t - b)) + (v - b);
  s = t;
}
__device__ __forceinline__ void sub_prod(double &s, double &e, double a, double b) {
  const double p = __dmul_rn(a, b);
  e -= fma(a, b, -p);
  add_err(s, e, -p);
}

__device__ __forceinline__ void async16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// running sum of products and its value as a number of the arithmetic
template <bool DF>
struct Num;
template <>
struct Num<false> {
  using T = double;
  using A = double;
  static __device__ __forceinline__ A zero() { return 0.0; }
  static __device__ __forceinline__ T from(double v) { return v; }
  static __device__ __forceinline__ T rec(T x2, T t, T u) { return fma(x2, t, -u); }
  static __device__ __forceinline__ T neg(T v) { return -v; }
  static __device__ __forceinline__ void mac(A &a, T x, T y) { a = fma(x, y, a); }
  static __device__ __forceinline__ void add(A &a, T x) { a += x; }
  static __device__ __forceinline__ T value(A a) { return a; }
  static __device__ __forceinline__ A settle(A a) { return a; }
  static __device__ __forceinline__ double to_double(A a) { return a; }
};
template <>
struct Num<true> {
  using T = df2;
  using A = df2;  // h: leading sum, l: sum of the errors (not normalised)
  static __device__ __forceinline__ A zero() { return {0.f, 0.f}; }
  static __device__ __forceinline__ T from(double v) { return to_df(v); }
  static __device__ __forceinline__ T rec(const T &x2, const T &t, const T &u) { return df_rec(x2, t, u); }
  static __device__ __forceinline__ T neg(const T &v) { return {-v.h, -v.l}; }
  static __device__ __forceinline__ void mac(A &a, const T &x, const T &y) { dfr::dot2(a.h, a.l, x.h, x.l, y.h, y.l); }
  static __device__ __forceinline__ void add(A &a, const T &x) {
    float s, t;
    dfr::two_sum(a.h, x.h, s, t);
    a.h = s;
    a.l = __fadd_rn(a.l, __fadd_rn(t, x.l));
  }
  static __device__ __forceinline__ T value(const A &a) {
    float s, t;
    dfr::two_sum(a.h, a.l, s, t);
    return {s, t};
  }
  // the sum with its errors moved into the leading part: left beside it they are rounded at their own, growing size
  static __device__ __forceinline__ A settle(const A &a) { return value(a); }
  static __device__ __forceinline__ double to_double(const A &a) {
    return static_cast<double>(a.h) + static_cast<double>(a.l);
  }
};

// A block's scratch for n energies (the tile, or all of the call's if fewer): amplitudes of the last runs and
// of those before [n][2 NP][32] each,
// particle sums S [n][32], series coefficients [n][kM], w* [n], number of terms [n] and (DF) the
// float-pair sin/cos table; every part on 16 bytes.
template <int MODE>
struct Scratch {
  using C = Cheb<MODE>;
  size_t amp, sum, s, coef, ws, terms, tab, total;
  __host__ __device__ explicit Scratch(int64_t n_omega) {
    const size_t n = (static_cast<size_t>(n_omega < C::kTile ? n_omega : C::kTile) + 3) / 4 * 4;
    amp = 0;
    sum = amp + n * 2 * C::NP * 32 * 8;
    s = sum + n * 2 * C::NP * 32 * 8;
    coef = s + n * 32 * 8;
    ws = coef + n * C::kM * 8;
    terms = ws + n * 8;
    tab = terms + n * 4;
    total = tab + dfr::kTabN * 16;
  }
};

template <int MODE>
struct Smem {
  using C = Cheb<MODE>;
  static constexpr int kRecs = 0;                                    // double [256][10]
  static constexpr int kMom = kRecs + kWin * kRecW * 8;              // 8 bytes [4][NP kM][32]
  static constexpr int kStep = kMom + kW * C::NP * C::kM * 32 * 8;   // float4 [256]
  // per warp, two slots: series coefficients and amplitudes of the energy at hand and of the next one
  static constexpr int kSlot = C::kM * 8 + 2 * C::NP * 32 * 8;
  static constexpr int kRing = kStep + kWin * 16;
  static constexpr int kMisc = kRing + kW * 2 * kSlot;               // item, status; float [4]
  // double [4][32]: each lane's phase length and its error at the run's centre and at the window's reference, the same
  // in the four warps (which write the same values, behind the barriers that end the last run's reads); two blocks
  // fit an SM with 1 KB of it, not with 4
  static constexpr int kBase = kMisc + 64;
  static constexpr int kTotal = kBase + 4 * 32 * 8;
};

// (2 - delta_m0) (-1)^{m/2} J_m(z) for m < M into out (as T), and the number of terms above 1e-18,
// rounded up to even. Power series below z = 2^-8 (its dropped terms are below 1e-18), Miller's backward
// recurrence normalised by J_0 + 2 sum J_2k = 1 above (M. Abramowitz, I. A. Stegun, 9.12). All runs of an energy
// share its coefficients, so their errors do not average out: 2/z and the normalising sum carry their
// rounding errors (worst J_m over z 1.0 units of 2^-53, J_0 0.3 in the mean; 2.5 and 0.6 without). The unnormalised
// values wait in out. One thread per energy, once per energy tile and particle energy: an FP64 instruction
// costs the warp 64 clocks and the branches of a warp's lanes follow one another, so the recurrence has no division
// and the series is a few instructions.
template <bool DF, int M>
__device__ int bessel_row(double z, typename Num<DF>::T *out) {
  double *raw = reinterpret_cast<double *>(out);
  int terms = 2;
  auto put = [&](int m, double j) {
    const double v = (m ? 2.0 : 1.0) * ((m >> 1) & 1 ? -j : j);
    out[m] = Num<DF>::from(v);
    if (fabs(v) > 1e-18 && m + 1 > terms) terms = m + 1;
  };
  if (z < 0x1p-8) {
    const double h = 0.5 * z, q = h * h;
    put(0, fma(-q, fma(-q, fma(-q, 1.0 / 36.0, 0.25), 1.0), 1.0));
    put(1, fma(-q, fma(-q, 1.0 / 12.0, 0.5), 1.0) * h);
    put(2, fma(-q, fma(-q, 1.0 / 24.0, 1.0 / 3.0), 1.0) * (q * 0.5));
    put(3, fma(-q, 0.25, 1.0) * (q * h * (1.0 / 6.0)));
    put(4, q * q * (1.0 / 24.0));
    put(5, q * q * h * (1.0 / 120.0));
    for (int m = 6; m < M; ++m) out[m] = Num<DF>::from(0.0);  // below 1e-19
  } else {
    const double rz = 2.0 / z, rl = fma(-rz, z, 2.0) / z;
    double hi = 0.0, lo = 1e-200, sum = 0.0, err = 0.0;
    double dm = M + 8;
#pragma unroll 2
    for (int m = M + 8; m > 0; --m, dm -= 1.0) {  // J_{M+8} is below 1e-21 for z <= 9
      const double p = dm * rz, pe = fma(dm, rl, fma(dm, rz, -p));
      const double t = fma(p, lo, fma(pe, lo, -hi));  // J_{m-1}
      hi = lo;
      lo = t;
      if (m <= M) raw[m - 1] = t;
      if (m % 2 != 0 && m > 1) add_err(sum, err, t);
    }
    double norm = lo;
    err *= 2.0;
    add_err(norm, err, 2.0 * sum);
    const double scale = 1.0 / norm, scale_e = (fma(-scale, norm, 1.0) - scale * err) * scale;
    for (int m = 0; m < M; ++m) {
      const double t = raw[m];
      put(m, fma(t, scale, t * scale_e));
    }
  }
  return (terms + 1) & ~1;
}

template <int MODE, bool DF>
__global__ void __launch_bounds__(kW * 32, 2) k_cheb(const Params P, unsigned char *__restrict__ scratch_all) {
  using C = Cheb<MODE>;
  using N = Num<DF>;
  using T = typename N::T;
  using A = typename N::A;
  using SM = Smem<MODE>;
  constexpr int NP = C::NP, kM = C::kM, kTile = C::kTile;
  constexpr int NC = C::kSpin ? 8 : 6;
  static_assert(sizeof(T) == 8 && sizeof(A) == 8, "8-byte numbers");
  extern __shared__ __align__(128) unsigned char sm[];
  double *recs = reinterpret_cast<double *>(sm + SM::kRecs);
  A *s_mom = reinterpret_cast<A *>(sm + SM::kMom);
  float4 *s_step = reinterpret_cast<float4 *>(sm + SM::kStep);
  int *s_item = reinterpret_cast<int *>(sm + SM::kMisc);
  volatile double *s_base = reinterpret_cast<volatile double *>(sm + SM::kBase);
  float *s_max = reinterpret_cast<float *>(s_item + 2);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  if (tid == 0) s_item[1] = *reinterpret_cast<volatile int *>(P.status);
  __syncthreads();
  if (s_item[1] != 0) return;
  const int64_t cut = *P.node_cut;  // energies [0, cut) are summed here, the others by the direct kernel
  if (cut <= 0) return;
  const Scratch<MODE> sc(P.n_omega);
  unsigned char *scr = scratch_all + static_cast<size_t>(blockIdx.x) * sc.total;
  A *amp = reinterpret_cast<A *>(scr + sc.amp);
  double *Ssum = reinterpret_cast<double *>(scr + sc.s);
  T *coef = reinterpret_cast<T *>(scr + sc.coef);
  double *wsv = reinterpret_cast<double *>(scr + sc.ws);
  int *n_terms = reinterpret_cast<int *>(scr + sc.terms);
  float4 *tab = reinterpret_cast<float4 *>(scr + sc.tab);
  if (DF)
    for (int i = tid; i < dfr::kTabN; i += kW * 32) tab[i] = dfr::table_pair(P.table[2 * i]);

  const int64_t n_wt = (cut + kTile - 1) / kTile, n_dt = (P.n_angles + 31) / 32;
  const int64_t per_chunk = n_wt * n_dt, n_items = per_chunk * P.n_chunks;
  int64_t have_wt = -1;
  double have_E = -1.0, a_lim = 0.0;

  for (;;) {
    __syncthreads();
    if (tid == 0) s_item[0] = atomicAdd(P.counter2, 1);
    __syncthreads();
    const int64_t item = s_item[0];
    if (item >= n_items) break;
    const int64_t chunk = item / per_chunk, rem = item % per_chunk;
    const int64_t dt = rem / n_wt, wt = rem % n_wt;
    const int64_t jdir = dt * 32 + lane;
    const int64_t jread = jdir < P.n_angles ? jdir : P.n_angles - 1;
    const double nx = P.theta_x[jread], ny = P.theta_y[jread];
    const double th2h = (nx * nx + ny * ny) * 0.5;
    const int64_t e0 = wt * kTile;
    const int ne = static_cast<int>(cut - e0 < kTile ? cut - e0 : kTile);
    int64_t p0, p1;
    int q;
    chunk_range(P, chunk, p0, p1, q);
    // component c (I_x, I_y, I_z, J as re, im) of an energy from its summed ones
    auto comp = [&](const double *a, int c) {
      if (c < 4) return a[c];
      if (c < 6) return -fma(nx, a[c - 4], ny * a[c - 2]);
      return a[c - 2];
    };
    for (int64_t p = p0; p < p1; ++p) {
      const int64_t off = P.offsets[p], len = P.offsets[p + 1] - off;
      const int64_t kb = P.amp_mode ? (len * q) / P.n_q : 0, ke = P.amp_mode ? (len * (q + 1)) / P.n_q : len;
      const double *S = P.samples + off * kRec;
      const double gam = P.gamma[p], En = P.energy[p];
      const double inv2g2 = 1.0 / (2.0 * gam * gam), cn = inv2g2 + th2h;
      if (wt != have_wt || (MODE != RAD_CLASSICAL && En != have_E)) {  // series of the tile's energies
        have_wt = wt;
        have_E = En;
        auto ws_of = [&](double h) {
          const double w = __ddiv_rn(h, kHbarC);
          return MODE == RAD_CLASSICAL ? w : __ddiv_rn(w, __dsub_rn(1.0, __ddiv_rn(h, En)));
        };
        a_lim = C::template kPhi<DF> / ws_of(P.hw[e0 + ne - 1]);  // the energies ascend
        __syncthreads();  // the last particle's series is no longer read
        for (int e = tid; e < ne; e += kW * 32) {
          const double w = ws_of(P.hw[e0 + e]);
          wsv[e] = w;
          n_terms[e] = bessel_row<DF, kM>(w * a_lim, coef + static_cast<size_t>(e) * kM);
        }
        __syncthreads();
      }
      const double inv_a = 1.0 / a_lim;
      const double cns = cn * inv_a, nxs = nx * inv_a, nys = ny * inv_a;
      const float cnf = static_cast<float>(cn), nxf = static_cast<float>(nx), nyf = static_cast<float>(ny);
      // runs since the last flush, plus 256 once there was one (one register); the first run of a
      // particle's piece or after a flush writes its amplitudes, the others add to them
      int since = 0;
      for (int64_t w0 = kb; w0 < ke; w0 += kWin) {
        const int n = static_cast<int>(ke - w0 < kWin ? ke - w0 : kWin);
        const double *r0 = S + w0 * kRec;  // the window's reference
        __syncthreads();  // the last window's records are no longer read
        for (int k = tid; k < n; k += kW * 32) {
          const double *rc = r0 + k * kRec;
          const int64_t K = w0 + k;
          const double tm = K == 0 ? rc[F_T] : rc[F_T - kRec], tp = K == len - 1 ? rc[F_T] : rc[F_T + kRec];
          const double w = 0.5 * (tp - tm);
          double *o = recs + k * kRecW;
          o[0] = rc[F_T] - r0[F_T];
          o[1] = rc[F_DZ] - r0[F_DZ];
          o[2] = rc[F_X] - r0[F_X];
          o[3] = rc[F_Y] - r0[F_Y];
          o[4] = rc[F_VX];
          o[5] = rc[F_VY];
          o[6] = rc[F_AX] * w;
          o[7] = rc[F_AY] * w;
          o[8] = rc[F_AZ] * w;
          o[9] = rc[F_DVZ];
          // step to the next sample (none after the window's last)
          const double *rn = k + 1 < n ? rc + kRec : rc;
          s_step[k] = make_float4(static_cast<float>(rn[F_T] - rc[F_T]), static_cast<float>(rn[F_DZ] - rc[F_DZ]),
                                static_cast<float>(rn[F_X] - rc[F_X]), static_cast<float>(rn[F_Y] - rc[F_Y]));
        }
        __syncthreads();
        // widest step in phase length over the window and the block's directions, FP32 with a margin
        // for its rounding; runs of L samples span at most (L - 1) of it
        float st = 0.f;
        for (int k = warp; k < n; k += kW) {
          const float4 d = s_step[k];
          const float a = cnf * d.x, b = nxf * d.z, c = nyf * d.w;
          const float v = fabsf(a - d.y - b - c) + 4e-7f * (fabsf(a) + fabsf(d.y) + fabsf(b) + fabsf(c));
          st = v > st || v != v ? v : st;  // a NaN stays
          if (st != st) break;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const float v = __shfl_xor_sync(0xffffffffu, st, o);
          st = v > st || v != v ? v : st;
        }
        if (lane == 0) s_max[warp] = st;
        __syncthreads();
        int run = kWin;
        {
          float m = s_max[0];
#pragma unroll
          for (int i = 1; i < kW; ++i) m = s_max[i] > m || s_max[i] != s_max[i] ? s_max[i] : m;
          const float lim = static_cast<float>(2.0 * a_lim);
          // the fewest runs of about equal length; a NaN step gives runs of one sample
          const float most = m > 0.f ? fminf(lim / m, static_cast<float>(kWin)) + 1.f : m == 0.f ? kWin : 1.f;
          run = most < 2.f ? 1 : static_cast<int>(most);
          run = run > kWin ? kWin : run;
          const int runs = (n + run - 1) / run;
          run = (n + runs - 1) / runs;
        }
        // phase length of the window's reference, with its rounding error: all samples of a run share
        // the run's base phase, so its error does not average out as that of a phase per sample does
        double A0 = __dmul_rn(cn, r0[F_T]), A0e = fma(cn, r0[F_T], -A0);
        add_err(A0, A0e, -r0[F_DZ]);
        sub_prod(A0, A0e, nx, r0[F_X]);
        sub_prod(A0, A0e, ny, r0[F_Y]);
        s_base[64 + lane] = A0;  // registers are what is short here
        s_base[96 + lane] = A0e;
        for (int k0 = 0; k0 < n; k0 += run) {
          const int m = n - k0 < run ? n - k0 : run;  // samples of this run
          auto length = [&](int k) {  // phase length from the window's reference
            const double *o = recs + k * kRecW;
            return fma(-ny, o[3], fma(-nx, o[2], fma(cn, o[0], -o[1])));
          };
          const double ctr = 0.5 * (length(k0) + length(k0 + m - 1));
          const double off_x = -ctr * inv_a;
          A M[kM][NP];
#pragma unroll
          for (int i = 0; i < kM; ++i)
#pragma unroll
            for (int c = 0; c < NP; ++c) M[i][c] = N::zero();
          const int share = (m + kW - 1) / kW;
          const int ka = k0 + min(warp * share, m), kz = k0 + min((warp + 1) * share, m);
          for (int k = ka; k < kz; ++k) {
            const double *o = recs + k * kRecW;
            const double x = fma(-nys, o[3], fma(-nxs, o[2], fma(-inv_a, o[1], fma(cns, o[0], off_x))));
            const double vx = o[4], vy = o[5];
            const double D = cn - o[9] - nx * vx - ny * vy;  // 1 - n.beta (Sec. II, g)
            const double r = __drcp_rn(D), g = r * r;
            const double a = nx - vx, b = ny - vy;
            const double mm = fma(ny, o[7], fma(nx, o[6], o[8]));  // n.beta_dot, weighted
            T f[NP];
            f[0] = N::from(fma(a, mm, -o[6] * D) * g);
            f[1] = N::from(fma(b, mm, -o[7] * D) * g);
            if (C::kSpin) f[NP - 1] = N::from(mm * g);
            // T_{m+2} = 2 T_2 T_m - T_{m-2}: the even and the odd orders as two chains of half the
            // length, which quarters the growth of the recurrence's rounding near x = +-1
            const T x1 = N::from(x), t2x2 = N::from(fma(4.0 * x, x, -2.0));
            T ev0 = N::from(1.0), od0 = x1;          // T_0, T_1
            T ev1 = N::from(fma(2.0 * x, x, -1.0));  // T_2
            T od1 = N::rec(t2x2, x1, x1);            // T_3 = 2 T_2 T_1 - T_1
#pragma unroll
            for (int i = 0; i < kM; i += 2) {
#pragma unroll
              for (int c = 0; c < NP; ++c) {
                if (i == 0)
                  N::add(M[0][c], f[c]);
                else
                  N::mac(M[i][c], f[c], ev0);
                N::mac(M[i + 1][c], f[c], od0);
              }
              if (i + 4 < kM) {
                const T e2 = N::rec(t2x2, ev1, ev0), o2 = N::rec(t2x2, od1, od0);
                ev0 = ev1;
                ev1 = e2;
                od0 = od1;
                od1 = o2;
              } else {
                ev0 = ev1;
                od0 = od1;
              }
            }
          }
          // moments of the run: the warps' shares, added in a fixed order, a quarter of them per warp
          __syncthreads();  // the last run's moments are no longer read
#pragma unroll
          for (int i = 0; i < kM; ++i)
#pragma unroll
            for (int c = 0; c < NP; ++c) s_mom[((warp * kM + i) * NP + c) * 32 + lane] = M[i][c];
          __syncthreads();
          for (int i = warp; i < kM * NP; i += kW) {
            A v = s_mom[i * 32 + lane];
#pragma unroll
            for (int w = 1; w < kW; ++w) N::add(v, N::value(s_mom[(w * kM * NP + i) * 32 + lane]));
            reinterpret_cast<T *>(s_mom)[i * 32 + lane] = N::value(v);
          }
          __syncthreads();
          T Mv[kM][NP];
#pragma unroll
          for (int i = 0; i < kM; ++i)
#pragma unroll
            for (int c = 0; c < NP; ++c) Mv[i][c] = reinterpret_cast<const T *>(s_mom)[(i * NP + c) * 32 + lane];
          {
            double Ac = s_base[64 + lane], Ae = s_base[96 + lane];
            add_err(Ac, Ae, ctr);
            s_base[lane] = Ac;
            s_base[32 + lane] = Ae;
          }
          // the next energy's coefficients and amplitudes are on their way from L2 while this one's
          // series is summed: eight warps an SM are too few to hide those loads
          unsigned char *ring = sm + SM::kRing + warp * 2 * SM::kSlot;
          auto fetch = [&](int e, int slot) {
            if (e < ne) {
              unsigned char *d = ring + slot * SM::kSlot;
              const unsigned char *c = reinterpret_cast<const unsigned char *>(coef + static_cast<size_t>(e) * kM);
              if (lane < kM / 2) async16(d + lane * 16, c + lane * 16);
              if (since & 255) {
                const unsigned char *a = reinterpret_cast<const unsigned char *>(amp + static_cast<size_t>(e) * 2 * NP * 32);
#pragma unroll
                for (int i = 0; i < NP; ++i) async16(d + kM * 8 + (i * 32 + lane) * 16, a + (i * 32 + lane) * 16);
              }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
          };
          fetch(warp, 0);
          int slot = 0, terms_next = warp < ne ? n_terms[warp] : 0;
          double ws_next = warp < ne ? wsv[warp] : 0.0;
          for (int e = warp; e < ne; e += kW, slot ^= 1) {
            fetch(e + kW, slot ^ 1);
            const int terms = terms_next;
            const double Ac = s_base[lane], phi = __dmul_rn(ws_next, Ac);
            const double phi_e = fma(ws_next, s_base[32 + lane], fma(ws_next, Ac, -phi));
            if (e + kW < ne) {
              terms_next = n_terms[e + kW];
              ws_next = wsv[e + kW];
            }
            T sn, cs;
            float4 entry;
            float xh, xl;
            if constexpr (DF) {
              entry = tab[dfr::reduce_phase(phi, xh, xl) & (dfr::kTabN - 1)];
              xl = __fadd_rn(xl, __double2float_rn(phi_e));
            }
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            __syncwarp();
            const T *cf = reinterpret_cast<const T *>(ring + slot * SM::kSlot);
            const A *old = reinterpret_cast<const A *>(ring + slot * SM::kSlot + kM * 8) + lane;
            A re[NP], im[NP];
#pragma unroll
            for (int c = 0; c < NP; ++c) re[c] = im[c] = N::zero();
#pragma unroll
            for (int i = 0; i < kM; i += 2) {
              if (i < terms) {
                const T ce = cf[i], co = cf[i + 1];
#pragma unroll
                for (int c = 0; c < NP; ++c) {
                  N::mac(re[c], ce, Mv[i][c]);
                  N::mac(im[c], co, Mv[i + 1][c]);
                }
              }
            }
            if constexpr (DF) {
              dfr::sincos_from_entry(entry, xh, xl, sn.h, sn.l, cs.h, cs.l);
            } else {
              double r;
              const int j = reduce_table(phi, r);
              sincos_reduced(j, r + phi_e, P.table, sn, cs);
            }
            A *o = amp + static_cast<size_t>(e) * 2 * NP * 32 + lane;
#pragma unroll
            for (int c = 0; c < NP; ++c) {
              A zr = since & 255 ? old[(2 * c) * 32] : N::zero(), zi = since & 255 ? old[(2 * c + 1) * 32] : N::zero();
              const T vr = N::value(re[c]), vi = N::value(im[c]);
              N::mac(zr, cs, vr);
              N::mac(zr, N::neg(sn), vi);
              N::mac(zi, sn, vr);
              N::mac(zi, cs, vi);
              o[(2 * c) * 32] = N::settle(zr);
              o[(2 * c + 1) * 32] = N::settle(zi);
            }
            __syncwarp();  // the slot is read; the fetch after next refills it
          }
          if ((++since & 255) == kFlush<DF>) {  // each lane its own amplitudes
            double *total = reinterpret_cast<double *>(amp + sc.sum / 8);
            for (int e = warp; e < ne; e += kW) {
              const size_t at = static_cast<size_t>(e) * 2 * NP * 32 + lane;
#pragma unroll 1
              for (int c = 0; c < 2 * NP; ++c)
                total[at + c * 32] = N::to_double(amp[at + c * 32]) + (since & 256 ? total[at + c * 32] : 0.0);
            }
            since = 256;
          }
        }
      }
      // the particle's (piece's) amplitudes: each warp its own energies
      for (int e = warp; e < ne; e += kW) {
        double a[2 * NP];
#pragma unroll
        for (int c = 0; c < 2 * NP; ++c)
          a[c] = (since & 255 ? N::to_double(amp[(static_cast<size_t>(e) * 2 * NP + c) * 32 + lane]) : 0.0) +
                 (since & 256 ? reinterpret_cast<double *>(amp + sc.sum / 8)[(static_cast<size_t>(e) * 2 * NP + c) * 32 + lane] : 0.0);
        if (P.amp_mode) {
          if (jdir < P.n_angles) {
#pragma unroll
            for (int c = 0; c < NC; ++c) P.part[((chunk * NC + c) * P.n_angles + jdir) * P.n_omega + e0 + e] = comp(a, c);
          }
          continue;
        }
        double I2 = 0.0;
#pragma unroll
        for (int c = 0; c < 6; ++c) {
          const double v = comp(a, c);
          I2 = fma(v, v, I2);
        }
        double Sv = I2;
        if (MODE != RAD_CLASSICAL) {
          const double u = P.hw[e0 + e] / En;
          if (MODE == RAD_SPIN0) {
            Sv = (1.0 - u) * I2;
          } else {
            const double J2 = a[2 * NP - 2] * a[2 * NP - 2] + a[2 * NP - 1] * a[2 * NP - 1];
            Sv = 0.5 * (1.0 + (1.0 - u) * (1.0 - u)) * I2 + (u * u) / (2.0 * gam * gam) * J2;
          }
        }
        const double wp = P.weight ? P.weight[p] : 1.0;
        const double acc = fma(wp, Sv, p == p0 ? 0.0 : Ssum[e * 32 + lane]);
        if (p + 1 < p1)
          Ssum[e * 32 + lane] = acc;
        else if (jdir < P.n_angles)
          P.part[(chunk * P.n_angles + jdir) * P.n_omega + e0 + e] = acc;
      }
    }
    if (p0 >= p1 && !P.amp_mode && jdir < P.n_angles)  // no particles: an empty sum
      for (int e = warp; e < ne; e += kW) P.part[(chunk * P.n_angles + jdir) * P.n_omega + e0 + e] = 0.0;
  }
}

template <int MODE, bool DF>
cudaError_t occ_t(int *nb) {
  auto kern = k_cheb<MODE, DF>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem<MODE>::kTotal);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(nb, kern, kW * 32, Smem<MODE>::kTotal);
}

template <int MODE, bool DF>
cudaError_t launch_t(const Params &P, unsigned char *scratch, int grid, cudaStream_t st) {
  auto kern = k_cheb<MODE, DF>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem<MODE>::kTotal);
  if (e != cudaSuccess) return e;
  kern<<<grid, kW * 32, Smem<MODE>::kTotal, st>>>(P, scratch);
  return cudaGetLastError();
}

template <typename F>
cudaError_t by_mode(int mode, F f) {
  switch (mode) {
    case RAD_CLASSICAL: return f(std::integral_constant<int, RAD_CLASSICAL>{});
    case RAD_SPIN0: return f(std::integral_constant<int, RAD_SPIN0>{});
    case RAD_SPIN_HALF: return f(std::integral_constant<int, RAD_SPIN_HALF>{});
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

int64_t cheb_tiles(int mode, int64_t n_omega, int64_t n_angles) {
  const int64_t tile = cheb_tile(mode);
  return (n_omega + tile - 1) / tile * ((n_angles + 31) / 32);
}

int cheb_tile(int mode) { return mode == RAD_SPIN_HALF ? Cheb<RAD_SPIN_HALF>::kTile : Cheb<RAD_CLASSICAL>::kTile; }

int occupancy_cheb(int mode, bool df) {
  int nb = 0;
  const cudaError_t e = by_mode(mode, [&](auto m) {
    return df ? occ_t<decltype(m)::value, true>(&nb) : occ_t<decltype(m)::value, false>(&nb);
  });
  return e == cudaSuccess ? nb : 0;
}

size_t cheb_scratch_bytes(int mode, int64_t n_omega, int grid) {
  return static_cast<size_t>(grid) *
         (mode == RAD_SPIN_HALF ? Scratch<RAD_SPIN_HALF>(n_omega).total : Scratch<RAD_CLASSICAL>(n_omega).total);
}

// Cost per sample and direction in SM clocks, for the choice of the cut, from the measured rates of the
// kernels (direct: 1.3e8 and 4.6e9 terms; moments: the cases in the header).
NodeCost cheb_cost(int mode, bool df, int direct_gran) {
  NodeCost c;
  const bool spin = mode == RAD_SPIN_HALF;
  c.gran = direct_gran;
  c.tile = cheb_tile(mode);
  c.cap = kWin;
  c.tile_steps = 1;
  c.widen = 1.05f;  // the widest of a window's steps against the widest of the 32 looked at
  c.reach = 0.95f * 2.f * static_cast<float>(spin ? (df ? Cheb<RAD_SPIN_HALF>::kPhi<true> : Cheb<RAD_SPIN_HALF>::kPhi<false>)
                                                     : (df ? Cheb<RAD_CLASSICAL>::kPhi<true> : Cheb<RAD_CLASSICAL>::kPhi<false>));
  c.direct = df ? (spin ? 1.45f : 1.3f) : (spin ? 11.5f : 9.6f);
  c.fixed = df ? (spin ? 36.f : 32.f) : 85.f;
  c.per_run = df ? 20.f : 110.f;
  c.per_energy = df ? (spin ? 17.f : 14.f) : (spin ? 58.f : 50.f);
  c.setup = 11.f;  // once per piece, bessel_row: some 690 FP64 instructions per 32 energies, 16 clocks each, for 32 directions
  return c;
}

cudaError_t launch_cheb(const Params &P, bool df, unsigned char *scratch, int grid, cudaStream_t st) {
  return by_mode(P.mode, [&](auto m) {
    return df ? launch_t<decltype(m)::value, true>(P, scratch, grid, st)
              : launch_t<decltype(m)::value, false>(P, scratch, grid, st);
  });
}

}  // namespace rad
