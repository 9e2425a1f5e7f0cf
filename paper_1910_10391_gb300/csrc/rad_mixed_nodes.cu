// Mixed-precision radiation integral through equispaced frequency nodes (sm_103a).
//
// k_mixed_pp evaluates one sin/cos per (sample, photon energy, direction). Over a short run of
// samples the amplitude F(w) = sum_k f_k e^{i w a_k} (a_k: the phase length of sample k from the
// run's centre) is band limited in w: it varies no faster than max |a_k|. So it is summed directly
// at kNodes equispaced node frequencies only, and read off at the photon energies by the
// interpolation of a non-uniform Fourier transform (A. Dutt, V. Rokhlin, "Fast Fourier transforms
// for nonequispaced data", SIAM J. Sci. Comput. 14 (1993); the Kaiser-Bessel kernel of J. A.
// Fessler, B. P. Sutton, IEEE Trans. Signal Process. 51 (2003)):
//   F(w_j) = sum_{c < 8} K((w_j - w_m)/h) sum_k [psi(h a_k) f_k] e^{i w_m a_k},  m = m_j + c
// with node spacing h, twofold oversampling |h a_k| <= pi/2, K the Kaiser-Bessel window of 8 nodes
// and psi the reciprocal of its Fourier transform. The truncation error is below 2.6e-7 of |f_k|
// per sample. The phases that sin/cos see are those of the nodes about the band's centre, at most 50 rad, and of the
// centre about the run's, at most (w_c / h) pi / 2: 50 rad in a tile that starts near zero, up to 6400 in a band
// narrow against its energies (h is w_hi / 4096 at least), but never more than the window's range of phases, which the direct
// form sees. Errors in both: tests/test_run_precision_gpu.py.
//
// Work split: a block of 4 warps takes one direction and 128 R photon energies. Per window of 256
// samples (the pre-pass's time tiles) each warp prepares 64 samples, cuts them into the longest
// power-of-two runs that satisfy |h a_k| <= pi/2 (down to single samples, which always do), and
// sums one run at the 64 nodes, two nodes w_c +- (l + 1/2) h per lane from one sin/cos pair; then
// every warp interpolates its own energies (R per lane, the kernel values in registers) from the
// runs of all four warps. A run's node sums cost about as much as 30 photon energies summed
// directly and the interpolation of one energy about as much as 5 samples, so the form pays where
// runs are long against 5 samples and energies many against 30.
//
// What bounds it: shared-memory wavefronts (64 % of the peak on the ensemble below, 76 % on the labels) and issue slots
// (59 %), with 15 warps an SM to hide the latency of either. Measured, all kernels of
// a call, before (k_mixed_pp alone) and with it: 32 positrons x 20000 samples x 512 log energies x 4096
// directions 546 -> 158 ms; 64 electrons of 2000 to 200000 samples x 1024 energies x 576 directions,
// spin 1/2, 437 -> 187 ms; 64 particles x 8192 samples x 256 energies x 512 directions with 15 rad per
// sample at the top (where the upper energies stay direct) 30.7 -> 19.5 ms; one undulator of 4096
// samples x 128 energies x 256 directions 135 -> 96 us. Tried and slower: window values in registers
// (168 of them, spills), 3 blocks an SM, node sums per sample instead of per pair of samples.
#include "rad_mixed_common.cuh"

namespace rad {
namespace {

constexpr int kNodeWarps = 4;
constexpr int kNodeT = 256;                 // window: the pre-pass's time tile
constexpr int kSeg = kNodeT / kNodeWarps;   // samples of a window that one warp prepares
constexpr int kNodes = 64;                  // node frequencies
constexpr int kKbW = 8;                     // nodes that one interpolation reads
constexpr float kXiMax = 1.57079632679489662f;  // |h a_k| at twofold oversampling

// The Kaiser-Bessel window I0(beta sqrt(1 - (2u/8)^2)), beta = 18.661, over its Fourier transform at
// 0, on the four unit intervals u in [3,4], [2,3], [1,2], [0,1] as polynomials in z = 2 frac(u) - 1
// (Chebyshev fits, error below 1e-9); the other four intervals mirror them. All of it times 1 + 1.65e-7: the
// SFU's sin and cos are short of modulus 1 by 1.0e-7 in the mean, and this form multiplies three of them (node,
// centre frequency and run) where the direct kernel has two, so that its peaks came out 4.7e-7 too
// low (2.1e-7 directly; means over bins above 5 % of the peak).
__constant__ float kKbRow[4][9] = {
    {4.143404837e-05f, -1.647157762e-04f, 2.796030420e-04f, -2.649951861e-04f, 1.526980023e-04f, -5.340338511e-05f,
     9.562849793e-06f, 3.008195943e-07f, -4.480140505e-07f},
    {8.204614455e-03f, -1.478727492e-02f, 1.093403750e-02f, -3.991893522e-03f, 5.446628305e-04f, 1.068984968e-04f,
     -4.987233932e-05f, 3.268000771e-06f, 1.223625176e-06f},
    {1.155015073e-01f, -1.057883490e-01f, 2.801810855e-02f, 2.838174081e-03f, -2.546929604e-03f, 2.065807806e-04f,
     9.103261369e-05f, -1.478784568e-05f, -1.669980529e-06f},
    {3.762525465e-01f, -1.075457679e-01f, -3.923191071e-02f, 1.330029758e-02f, 1.849859684e-03f, -7.821835692e-04f,
     -5.083793540e-05f, 2.760262983e-05f, 8.255166342e-07f}};

__device__ __forceinline__ float kb_row(int row, float z) {
  float v = kKbRow[row][8];
#pragma unroll
  for (int i = 7; i >= 0; --i) v = fmaf(v, z, kKbRow[row][i]);
  return v;
}

// psi: the reciprocal of the window's Fourier transform, as a polynomial in (h a_k / (pi/2))^2
__device__ __forceinline__ float kb_psi(float y) {
  float v = 1.255510908e-03f;
  v = fmaf(v, y, 1.821370374e-03f);
  v = fmaf(v, y, 1.519394823e-02f);
  v = fmaf(v, y, 5.663918166e-02f);
  v = fmaf(v, y, 1.956056633e-01f);
  v = fmaf(v, y, 5.278406413e-01f);
  v = fmaf(v, y, 1.001092611e+00f);
  return fmaf(v, y, 9.999999932e-01f);
}

// Two FP32 values in one 64-bit register: fma.rn.f32x2 does two FMAs in one issue slot, and issue
// slots are what this kernel spends most.
using f2 = unsigned long long;
__device__ __forceinline__ f2 pack2(float lo, float hi) {
  f2 v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
  return v;
}
__device__ __forceinline__ float2 unpack2(f2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float halves(f2 v) {
  const float2 r = unpack2(v);
  return r.x + r.y;
}

template <int MODE, int R>
struct NodeLayout {
  static constexpr bool kSpin = MODE == RAD_SPIN_HALF;
  static constexpr int kStageBytes = kNodeT * kPP * 4;
  static constexpr int kStage = 0;
  static constexpr int kG = kStage + kStageBytes;               // per pair of samples and component (re, re', im, im') of g
  static constexpr int kX = kG + kNodeT * 8 * (kSpin ? 3 : 2);  // float [256]: h a
  static constexpr int kN = kX + kNodeT * 4;                    // float4 [2][4][64]: node sums (x re, im, y re, im)
  static constexpr int kNj = kN + 2 * kNodeWarps * kNodes * 16; // float2 [2][4][64]: node sums of j
  static constexpr int kC = kNj + (kSpin ? 2 * kNodeWarps * kNodes * 8 : 0);  // float2 [256]: phase lengths of run centres
  static constexpr int kRef = kC + kNodeT * 8;              // float2 [2][32]: phase length at the windows' references
  static constexpr int kKb = kRef + 2 * 32 * 8;                 // float4 [2][128 R]: window values of each energy
  static constexpr int kBar = kKb + 2 * 128 * R * 16;           // the stage's barrier
  static constexpr int kMisc = kBar + 16;                       // item, status, levels [4]
  static constexpr int kTotal = kMisc + 32;
};

template <int MODE, int R>
__global__ void __launch_bounds__(kNodeWarps * 32, 4) k_mixed_nodes(const Params P, const float *__restrict__ prep) {
  using L = NodeLayout<MODE, R>;
  constexpr bool kSpin = L::kSpin;
  constexpr int NC = kSpin ? 8 : 6;
  constexpr int NA = NC - 2;  // I_z = -(n_x I_x + n_y I_y) is formed from the sums, as in k_mixed_pp
  constexpr int NWN = kNodeWarps;
  constexpr int kTile = 128 * R;
  extern __shared__ __align__(128) unsigned char sm[];
  uint64_t *full = reinterpret_cast<uint64_t *>(sm + L::kBar);
  int *s_item = reinterpret_cast<int *>(sm + L::kMisc);
  int *s_lvl = s_item + 2;
  constexpr int NP = kSpin ? 3 : 2;  // complex components
  float *sx = reinterpret_cast<float *>(sm + L::kX);
  float *sg = reinterpret_cast<float *>(sm + L::kG);
  float2 *s_ctr = reinterpret_cast<float2 *>(sm + L::kC);
  float4 *sn = reinterpret_cast<float4 *>(sm + L::kN);
  float2 *snj = reinterpret_cast<float2 *>(sm + L::kNj);
  float2 *s_ref = reinterpret_cast<float2 *>(sm + L::kRef);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  if (tid == 0) s_item[1] = *reinterpret_cast<volatile int *>(P.status);
  __syncthreads();
  if (s_item[1] != 0) return;
  const int64_t cut = *P.node_cut;  // energies [0, cut) are summed here, the others by k_mixed_pp
  if (cut <= 0) return;
  if (tid == 0) {
    mbar_init(full, 1);
    fence_mbar_init();
  }
  __syncthreads();
  const int64_t n_wt = (cut + kTile - 1) / kTile;
  const int64_t per_chunk = n_wt * P.n_angles;
  const int64_t n_items = per_chunk * P.n_chunks;
  uint32_t full_par = 0u;
  int nb = 0, rb = 0;  // node buffer, reference buffer

  // thread 0, when no warp reads the stage any more: start the next window's copy. One stage is
  // enough: a window's records go to registers at once, and the copy has the rest of its time.
  auto produce = [&](const TileCursor &c) {
    const int64_t n = (c.ke - c.k0) < kNodeT ? (c.ke - c.k0) : kNodeT;
    const uint32_t bytes = static_cast<uint32_t>(n * kPP * 4);
    fence_proxy_async();
    mbar_arrive_expect_tx(full, bytes);
    bulk_g2s(sm + L::kStage, prep + (P.offsets[c.p] + c.k0) * kPP, bytes, full);
  };

  // state of the energies, kept from item to item while the energy tile and the particle energy stay
  float4 *s_kb = reinterpret_cast<float4 *>(sm + L::kKb);  // of energy 128 r + 32 warp + lane, own lanes only
  int kofs[R];
  float wt_hi[R], wt_lo[R];
  float hf = 0.f, wcf = 0.f;  // node spacing and centre
  int64_t have_wt = -1;
  double have_E = -1.0, have_g = -1.0, inv2g2 = 0.0;
  const float pf = static_cast<float>(lane) + 0.5f;

  for (;;) {
    if (tid == 0) s_item[0] = atomicAdd(P.counter2, 1);
    __syncthreads();
    const int64_t item = s_item[0];
    __syncthreads();
    if (item >= n_items) break;
    const int64_t chunk = item / per_chunk;
    const int64_t rem = item % per_chunk;
    const int64_t jdir = rem / n_wt, wt = rem % n_wt;
    const double nx = P.theta_x[jdir], ny = P.theta_y[jdir];
    const double th2h = (nx * nx + ny * ny) * 0.5;
    const float nxf = static_cast<float>(nx), nyf = static_cast<float>(ny);
    const int64_t e0 = wt * kTile + warp * 32 + lane;  // energy of r: e0 + 128 r
    auto live = [&](int r) { return wt * kTile + warp * 32 + 128 * r < cut; };  // the warp has energies at r
    auto hw_of = [&](int r) { return P.hw[e0 + 128 * r < cut ? e0 + 128 * r : cut - 1]; };

    double S_acc[R];
    float ks[R][NA], kc[R][NA];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      S_acc[r] = 0.0;
#pragma unroll
      for (int c = 0; c < NA; ++c) ks[r][c] = kc[r][c] = 0.f;
    }
    auto component = [&](int r, int c) -> double {
      auto v = [&](int i) { return static_cast<double>(ks[r][i]) - static_cast<double>(kc[r][i]); };
      if (c < 4) return v(c);
      if (c < 6) return -fma(nx, v(c - 4), ny * v(c - 2));
      return v(c - 2);
    };
    int64_t p0, p1;
    int q;
    chunk_range(P, chunk, p0, p1, q);
    TileCursor cur;
    cur.p = p0;
    cur.p_end = p1;
    cursor_settle(P, cur, q);
    if (cur.valid) {
      if (tid == 0) produce(cur);
      int64_t cur_p = -1;
      double cn = 0.0, wp = 1.0, gam = 2.0, En = 1.0;
      float cn_hi = 0.f, cn_lo = 0.f;
      int wi = 0;  // window of the current particle
      for (;;) {
        TileCursor nxt = cur;
        cursor_next<kNodeT>(P, nxt, q);
        if (cur.p != cur_p) {
          cur_p = cur.p;
          wi = 0;
          gam = P.gamma[cur_p];
          En = P.energy[cur_p];
          wp = P.weight ? P.weight[cur_p] : 1.0;
          if (gam != have_g) {
            have_g = gam;
            inv2g2 = 1.0 / (2.0 * gam * gam);
          }
          cn = inv2g2 + th2h;
          cn_hi = static_cast<float>(cn);
          cn_lo = static_cast<float>(cn - static_cast<double>(cn_hi));
          if (wt != have_wt || (MODE != RAD_CLASSICAL && En != have_E)) {
            have_wt = wt;
            have_E = En;
            auto ws_of = [&](double h) {
              const double w = h / kHbarC;
              return MODE == RAD_CLASSICAL ? w : w / (1.0 - h / En);
            };
            const double wlo = ws_of(P.hw[wt * kTile]);
            const double whi = ws_of(P.hw[((wt + 1) * kTile < cut ? (wt + 1) * kTile : cut) - 1]);
            // 56 spacings between the lowest and the highest energy, 3.5 nodes beyond on either side
            const double h = fmax((whi - wlo) * (1.0 / (kNodes - kKbW)), whi * (1.0 / 4096.0));
            const double wc = 0.5 * (wlo + whi), rh = 1.0 / h;
            hf = static_cast<float>(h);
            wcf = static_cast<float>(wc);
#pragma unroll
            for (int r = 0; r < R; ++r) {
              const double w = ws_of(hw_of(r));
              const double wtd = w * kInvTwoPi;
              wt_hi[r] = static_cast<float>(wtd);
              wt_lo[r] = static_cast<float>(wtd - static_cast<double>(wt_hi[r]));
              const double u = (w - wc) * rh + 0.5 * (kNodes - 1);
              int i = static_cast<int>(floor(u)) - (kKbW / 2 - 1);
              i = i < 0 ? 0 : i > kNodes - kKbW ? kNodes - kKbW : i;
              kofs[r] = i;
              const float z = 2.f * static_cast<float>(u - (i + kKbW / 2 - 1)) - 1.f;
              float4 *k = s_kb + r * 128 + tid;
              k[0] = make_float4(kb_row(0, z), kb_row(1, z), kb_row(2, z), kb_row(3, z));
              k[128 * R] = make_float4(kb_row(3, -z), kb_row(2, -z), kb_row(1, -z), kb_row(0, -z));
            }
          }
#pragma unroll
          for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < NA; ++c) ks[r][c] = kc[r][c] = 0.f;
        }
        // phase lengths at the references (middle samples) of the next 32 windows, FP64, one
        // window per lane of warp 0, kept as float pairs: the FP64 pipe is charged per warp
        if ((wi & 31) == 0) {
          rb ^= 1;
          if (warp == 0) {
            const int64_t k0 = cur.k0 + static_cast<int64_t>(lane) * kNodeT;
            if (k0 < cur.ke) {
              const int64_t m = (cur.ke - k0) < kNodeT ? (cur.ke - k0) : kNodeT;
              const double *r0 = P.samples + (P.offsets[cur.p] + k0 + ((m - 1) >> 1)) * kRec;
              const double A0 = ((cn * r0[F_T] - r0[F_DZ]) - nx * r0[F_X]) - ny * r0[F_Y];
              const float a = static_cast<float>(A0);
              s_ref[rb * 32 + lane] = make_float2(a, static_cast<float>(A0 - static_cast<double>(a)));
            }
          }
        }
        const bool ok = mbar_wait_bounded(full, full_par);
        full_par ^= 1u;
        const float *st = reinterpret_cast<const float *>(sm + L::kStage);
        const int n = static_cast<int>((cur.ke - cur.k0) < kNodeT ? (cur.ke - cur.k0) : kNodeT);

        // two samples per lane: phase length from the window's reference, weighted f_x, f_y, j
        float al[2], fx[2], fy[2], fj[2], mn[2], mx[2], ctr[7][2];
        uint32_t viol = 0;  // bit l: some run of 2^l samples is too wide
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int k = warp * kSeg + i * 32 + lane;
          al[i] = fx[i] = fy[i] = fj[i] = 0.f;
          mn[i] = INFINITY;
          mx[i] = -INFINITY;
          if (ok && k < n) {
            const float4 ra = reinterpret_cast<const float4 *>(st + k * kPP)[0];
            const float4 rbv = reinterpret_cast<const float4 *>(st + k * kPP)[1];
            const float2 rcz = reinterpret_cast<const float2 *>(st + k * kPP)[4];
            const float a = nxf - rbv.x, b = nyf - rbv.y;
            const float m = fmaf(nyf, rbv.w, fmaf(nxf, rbv.z, rcz.x));
            const float D = fmaf(0.5f, fmaf(a, a, b * b), rcz.y);
            const float rD = __frcp_rn(D);
            const float g = rD * rD;
            al[i] = fmaf(-nyf, ra.w, fmaf(-nxf, ra.z, fmaf(cn_hi, ra.x, fmaf(cn_lo, ra.x, -ra.y))));
            fx[i] = fmaf(a, m, -rbv.z * D) * g;
            fy[i] = fmaf(b, m, -rbv.w * D) * g;
            if (kSpin) fj[i] = m * g;
            mn[i] = mx[i] = al[i];
          }
          ctr[0][i] = al[i];
        }
        const float lim = 2.0f * kXiMax / hf;  // widest run
#pragma unroll
        for (int l = 1; l <= 6; ++l) {
          if (l < 6) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              mn[i] = fminf(mn[i], __shfl_xor_sync(0xffffffffu, mn[i], 1 << (l - 1)));
              mx[i] = fmaxf(mx[i], __shfl_xor_sync(0xffffffffu, mx[i], 1 << (l - 1)));
            }
          } else {
            mn[0] = mn[1] = fminf(mn[0], mn[1]);
            mx[0] = mx[1] = fmaxf(mx[0], mx[1]);
          }
          bool wide = false;
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            ctr[l][i] = 0.5f * mn[i] + 0.5f * mx[i];
            wide |= !(mx[i] - mn[i] <= lim) && mx[i] >= mn[i];
          }
          if (__any_sync(0xffffffffu, wide)) viol |= 1u << l;
        }
        if (lane == 0) s_lvl[warp] = viol ? __ffs(static_cast<int>(viol)) - 1 : 7;  // longest run: 2^(level - 1)
        if (__syncthreads_or(!ok)) {  // bounded wait ran out
          if (tid == 0) {
            set_status(P.status, RAD_ETIMEOUT);
            mbar_wait_bounded(full, full_par ^ 1u);  // the stalled copy, again
          }
          return;
        }
        if (tid == 0 && nxt.valid) produce(nxt);  // every warp has read the stage
        int lvl = s_lvl[0];
#pragma unroll
        for (int w = 1; w < NWN; ++w) lvl = min(lvl, s_lvl[w]);
        lvl -= 1;
        const int run = 1 << lvl, rounds = kSeg >> lvl;
        // samples about their run's centre: h a, psi f e^{i w_c a}
        const float2 ref = s_ref[rb * 32 + (wi & 31)];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          float c = ctr[0][i];
#pragma unroll
          for (int l = 1; l <= 6; ++l) c = lvl == l ? ctr[l][i] : c;
          const int kl = i * 32 + lane;
          const bool in = warp * kSeg + kl < n;
          const float a = in ? al[i] - c : 0.f;
          const float t = hf * a;
          const float xr = t * (1.f / kXiMax);
          const float ps = in ? kb_psi(xr * xr) : 0.f;
          float sn_, cs_;
          __sincosf(wcf * a, &sn_, &cs_);
          const float gr = ps * cs_, gi = ps * sn_;
          sx[warp * kSeg + kl] = t;
          float *g = sg + (warp * kSeg + kl) / 2 * (4 * NP) + (kl & 1);
          g[0] = fx[i] * gr;
          g[2] = fx[i] * gi;
          g[4] = fy[i] * gr;
          g[6] = fy[i] * gi;
          if (kSpin) {
            g[4 * NP - 4] = fj[i] * gr;
            g[4 * NP - 2] = fj[i] * gi;
          }
          if ((kl & (run - 1)) == 0) {
            // phase length at the run's centre, reference + centre as a float pair (Knuth's TwoSum:
            // either may be the larger)
            const float ah = __fadd_rn(ref.x, c);
            const float bb = __fsub_rn(ah, ref.x);
            s_ctr[warp * kSeg + (kl >> lvl)] =
                make_float2(ah, __fadd_rn(__fadd_rn(__fsub_rn(ref.x, __fsub_rn(ah, bb)), __fsub_rn(c, bb)), ref.y));
          }
        }
        __syncwarp();

        for (int rd = 0; rd < rounds; ++rd) {
          // node sums of this warp's run: lane l takes the nodes w_c +- (l + 1/2) h
          const int kb0 = warp * kSeg + rd * run;
          if (kb0 < n) {
            // sums of Re g cos, Re g sin, Im g cos, Im g sin over the even and the odd samples: the two
            // samples of a pair are the halves of one register pair, so that an operand needs no copy
            f2 rc[NP], rs[NP], ic[NP], is[NP];
#pragma unroll
            for (int c = 0; c < NP; ++c) rc[c] = rs[c] = ic[c] = is[c] = 0ull;
            auto two = [&](int kp, bool masked, f2 keep) {  // samples 2 kp and 2 kp + 1, or one of them
              const float2 t = reinterpret_cast<const float2 *>(sx)[kp];
              float s0, c0, s1, c1;
              __sincosf(pf * t.x, &s0, &c0);
              __sincosf(pf * t.y, &s1, &c1);
              f2 cs = pack2(c0, c1), sn2 = pack2(s0, s1);
              if (masked) {
                cs = mul2(cs, keep);
                sn2 = mul2(sn2, keep);
              }
#pragma unroll
              for (int c = 0; c < NP; ++c) {
                const ulonglong2 G = reinterpret_cast<const ulonglong2 *>(sg)[kp * NP + c];
                rc[c] = fma2(G.x, cs, rc[c]);
                rs[c] = fma2(G.x, sn2, rs[c]);
                ic[c] = fma2(G.y, cs, ic[c]);
                is[c] = fma2(G.y, sn2, is[c]);
              }
            };
            if (run >= 8) {
              for (int k = 0; k < run; k += 8)
#pragma unroll
                for (int u = 0; u < 4; ++u) two((kb0 + k) / 2 + u, false, 0ull);
            } else if (run >= 2) {
              for (int k = 0; k < run; k += 2) two((kb0 + k) / 2, false, 0ull);
            } else {  // single samples: the other half of the pair is another run's
              two(kb0 / 2, true, kb0 & 1 ? pack2(0.f, 1.f) : pack2(1.f, 0.f));
            }
            float4 *nd = sn + (nb * NWN + warp) * kNodes;
            float2 u[NP], v[NP];  // (Re g cos, Re g sin), (Im g cos, Im g sin)
#pragma unroll
            for (int c = 0; c < NP; ++c) {
              u[c] = make_float2(halves(rc[c]), halves(rs[c]));
              v[c] = make_float2(halves(ic[c]), halves(is[c]));
            }
            nd[kNodes / 2 + lane] = make_float4(u[0].x - v[0].y, u[0].y + v[0].x, u[1].x - v[1].y, u[1].y + v[1].x);
            nd[kNodes / 2 - 1 - lane] = make_float4(u[0].x + v[0].y, v[0].x - u[0].y, u[1].x + v[1].y, v[1].x - u[1].y);
            if (kSpin) {
              float2 *nj = snj + (nb * NWN + warp) * kNodes;
              nj[kNodes / 2 + lane] = make_float2(u[NP - 1].x - v[NP - 1].y, u[NP - 1].y + v[NP - 1].x);
              nj[kNodes / 2 - 1 - lane] = make_float2(u[NP - 1].x + v[NP - 1].y, v[NP - 1].x - u[NP - 1].y);
            }
          }
          __syncthreads();
          // this warp's energies from the runs of all warps
          const int runs = min(NWN, (n - rd * run + kSeg - 1) / kSeg);  // warps with samples in this round
#pragma unroll
          for (int r = 0; r < R; ++r) {
            if (!live(r)) continue;
            f2 kd[kKbW];
            {
              const float4 a = s_kb[r * 128 + tid], b = s_kb[r * 128 + tid + 128 * R];
              const float k[kKbW] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
              for (int c = 0; c < kKbW; ++c) kd[c] = pack2(k[c], k[c]);
            }
            // C = sum cos(w A_run) v, S = sum sin(w A_run) v over the runs, v = (re, im)
            f2 C[NP], S[NP];
#pragma unroll
            for (int c = 0; c < NP; ++c) C[c] = S[c] = 0ull;
            auto one_run = [&](int w) {
              const ulonglong2 *nd = reinterpret_cast<const ulonglong2 *>(sn) + (nb * NWN + w) * kNodes + kofs[r];
              f2 v[NP];
#pragma unroll
              for (int c = 0; c < NP; ++c) v[c] = 0ull;
#pragma unroll
              for (int c = 0; c < kKbW; ++c) {
                const ulonglong2 N = nd[c];
                v[0] = fma2(kd[c], N.x, v[0]);
                v[1] = fma2(kd[c], N.y, v[1]);
              }
              if (kSpin) {
                const f2 *nj = reinterpret_cast<const f2 *>(snj) + (nb * NWN + w) * kNodes + kofs[r];
#pragma unroll
                for (int c = 0; c < kKbW; ++c) v[NP - 1] = fma2(kd[c], nj[c], v[NP - 1]);
              }
              const float2 a = s_ctr[w * kSeg + rd];
              float c0, s0;
              tile_base_sincos(wt_hi[r], wt_lo[r], a.x, a.y, s0, c0);
              const f2 cc = pack2(c0, c0), ss = pack2(s0, s0);
#pragma unroll
              for (int c = 0; c < NP; ++c) {
                C[c] = fma2(cc, v[c], C[c]);
                S[c] = fma2(ss, v[c], S[c]);
              }
            };
            if (runs == NWN) {
#pragma unroll
              for (int w = 0; w < NWN; ++w) one_run(w);
            } else {
#pragma unroll 1
              for (int w = 0; w < runs; ++w) one_run(w);
            }
#pragma unroll
            for (int c = 0; c < NP; ++c) {
              const float2 x = unpack2(C[c]), y = unpack2(S[c]);
              kahan_add(ks[r][2 * c], kc[r][2 * c], x.x - y.y);
              kahan_add(ks[r][2 * c + 1], kc[r][2 * c + 1], x.y + y.x);
            }
          }
          nb ^= 1;
        }
        const bool last_of_particle = !nxt.valid || nxt.p != cur.p;
        if (last_of_particle && !P.amp_mode) {
#pragma unroll
          for (int r = 0; r < R; ++r) {
            if (!live(r)) continue;
            double I2 = 0.0;
#pragma unroll
            for (int c = 0; c < 6; ++c) {
              const double v = component(r, c);
              I2 = fma(v, v, I2);
            }
            double Sv;
            if (MODE == RAD_CLASSICAL) {
              Sv = I2;
            } else {
              const double u = hw_of(r) / En;
              if (MODE == RAD_SPIN0) {
                Sv = (1.0 - u) * I2;
              } else {
                const double jr = component(r, 6);
                const double ji = component(r, 7);
                Sv = 0.5 * (1.0 + (1.0 - u) * (1.0 - u)) * I2 + (u * u) / (2.0 * gam * gam) * (jr * jr + ji * ji);
              }
            }
            S_acc[r] = fma(wp, Sv, S_acc[r]);
          }
        }
        ++wi;
        if (!nxt.valid) break;
        cur = nxt;
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int64_t e = e0 + 128 * r;
      if (e >= cut) continue;
      if (!P.amp_mode) {
        P.part[(chunk * P.n_angles + jdir) * P.n_omega + e] = S_acc[r];
      } else {
#pragma unroll
        for (int c = 0; c < NC; ++c)
          P.part[((chunk * NC + c) * P.n_angles + jdir) * P.n_omega + e] = component(r, c);
      }
    }
  }
}

template <int MODE, int R>
cudaError_t launch_t(const Params &P, const float *prep, int sms, cudaStream_t st) {
  using L = NodeLayout<MODE, R>;
  auto kern = k_mixed_nodes<MODE, R>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L::kTotal);
  if (e != cudaSuccess) return e;
  int nb = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, kNodeWarps * 32, L::kTotal);
  if (e != cudaSuccess) return e;
  if (nb <= 0) return cudaErrorInvalidConfiguration;
  const int64_t items = ((P.n_omega + 128 * R - 1) / (128 * R)) * P.n_angles * P.n_chunks;
  const int64_t resident = static_cast<int64_t>(nb) * sms;
  kern<<<static_cast<int>(items < resident ? items : resident), kNodeWarps * 32, L::kTotal, st>>>(P, prep);
  return cudaGetLastError();
}

template <int MODE>
cudaError_t launch_r(const Params &P, const float *prep, int r, int sms, cudaStream_t st) {
  if (r == 1) return launch_t<MODE, 1>(P, prep, sms, st);
  if (r == 2) return launch_t<MODE, 2>(P, prep, sms, st);
  return launch_t<MODE, 4>(P, prep, sms, st);
}

// energies per lane: one tile of 128 R energies up to 512
int node_r(int64_t n_omega) { return n_omega <= 128 ? 1 : n_omega <= 256 ? 2 : 4; }

}  // namespace

// Below 96 energies the 64 nodes save too little for the extra launch.
bool node_path_allowed(const LaunchShape &s, int64_t n_omega, int64_t n_angles, int64_t n_chunks) {
  if (s.T != kNodeT || n_omega < 96 || n_omega > INT32_MAX) return false;
  const int64_t tile = 128 * node_r(n_omega), tiles = (n_omega + tile - 1) / tile;
  return n_angles <= (INT32_MAX - 65536) / tiles / n_chunks;  // the 32-bit work counter
}

// Runs reach 56 pi of phase range over the tile's span (twofold oversampling, 56 node spacings). Costs from the measured rates: 17.4 clocks per sample and direction of the 512-energy
// ensemble (classical, runs of about 50), 52 of the 1024-energy batch (spin 1/2, two tiles).
NodeCost node_cost(int mode, int64_t n_omega, int direct_r) {
  const bool spin = mode == RAD_SPIN_HALF;
  NodeCost c;
  c.gran = 32 * direct_r;
  c.tile = 128 * node_r(n_omega);
  c.from_zero = 0;
  c.direct = spin ? 1.0f / 7.6f : 1.0f / 8.5f;
  c.fixed = spin ? 8.5f : 6.8f;
  c.per_energy = spin ? 1.35f : 1.1f;
  c.setup = 46.f;         // window values at a particle energy's w*: some 184 FP64 instructions a warp and 64 energies
  c.margin = 0.85f;
  c.setup_if_differ = 1;  // kept while the particle energy stays
  c.pow2 = 1;
  c.reach = static_cast<float>(56.0 * kPi);
  c.cap = 64.f;
  return c;
}

int64_t node_tiles(int64_t n_omega) { return (n_omega + 128 * node_r(n_omega) - 1) / (128 * node_r(n_omega)); }

cudaError_t launch_mixed_nodes(const Params &P, const float *prep, int sms, cudaStream_t st) {
  const int r = node_r(P.n_omega);
  switch (P.mode) {
    case RAD_CLASSICAL: return launch_r<RAD_CLASSICAL>(P, prep, r, sms, st);
    case RAD_SPIN0: return launch_r<RAD_SPIN0>(P, prep, r, sms, st);
    case RAD_SPIN_HALF: return launch_r<RAD_SPIN_HALF>(P, prep, r, sms, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace rad
