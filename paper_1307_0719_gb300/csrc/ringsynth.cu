// Ring synthesis in single precision: from the per-ring Fourier coefficients
// F^j_m(theta_r) to the derivative maps on the ring's equally spaced pixels (Naess &
// Louis 2013, Sec. II.B: the maps d_theta^j d_phi^k s of Eq. 4 at the pixel centres),
//   D(theta_r, phi_p) = Re[ G_0 + 2 sum_{m>0} G_m e^{i m phi_p} ],  G_m = (i m / L)^k F^j_m.
//
// Every map is one complex-to-real transform of a power-of-two grid of 2 H points, by a
// complex DFT of length H held in registers (RegFft): with S the Hermitian spectrum,
//   Z_m = (S_m + conj S_{H-m}) + i e^{2 pi i m / 2H} (S_m - conj S_{H-m}),  m < H,
// its inverse DFT z_n = x_{2n} + i x_{2n+1} holds the map's values at the grid points.
//
// Rings whose pixels are grid points (the belt: 4 Nside a power of two) store z_n at
// once. The cap rings have 4 i pixels; their function of longitude is band limited (m <= band),
// so it is sampled on a power-of-two grid that oversamples it at least twice and interpolated to the pixels
// with a Kaiser-Bessel window of W = 10 grid points, the coefficients having been divided by the
// window's transform (gridding; Jackson et al. 1991, IEEE Trans. Med. Imaging 10, 473). The method's own
// error is 3e-9 at the band's edge; what counts is the transform's float rounding, which the division
// amplifies at the top of the band (by 3.7 at an oversampling of 2, by 8 at 1.65). Relative RMS error of a map,
// of the rings' rows alone (coefficients ~ (m + 1)^p, p = -1 .. 2, phi-derivatives 0 .. 4, Nside 64 to 2048): caps 1.07 to
// 1.68e-7, no map of a ring above 2.2e-7, belt 1.18 to 1.37e-7. Packed pairs of maps with Bluestein's convolution in
// the caps: 1.41 to 2.5e-7, belt 1.05 to 1.7e-7, and up to 9e-6 where a map shared its transform with a much larger
// one. An oversampling of 1.65 with W = 8 for `twice`: 1.9 to 4.3e-7 on the rings next below a larger
// grid, for 9% less time at Nside 2048; 1.9 instead of 2 up to 12% above Bluestein on single rings, for 3%.
// This takes one transform of one to two times the ring's own length per map; Bluestein's chirp-z
// convolution, exact for any length, takes four of 2 to 4 times the sub-sequence length each (per map of a packed pair).
//
// The rows of F are zero beyond the ring's mcut (see host_ring_bands): the Legendre stage holds
// functions below 2^-32 at zero. Nothing beyond is read. Rows are staged
// once per plane in shared memory, scaled by the window's correction, and multiplied by
// i m / P (a power of two, see synth_power) from one phi-derivative to the next. Where the band limit exceeds half the
// ring's length the aliases are folded while staging (per map, since (m / L)^k is not a
// function of m modulo the length).
//
// What bounds it: instruction issue (Nside 2048 / lmax 3000: the belt 69% issue-active at 23 warps per SM, the caps
// of H = 4096 67% and their two-grid form 78%, of H = 2048 60%, at 31 warps; DRAM below 45% of its copy
// rate). Sixteen T+Q/U realisations of order 4 take 118 ms at
// Nside 2048 / lmax 3000 and 10.4 ms at Nside 512 / lmax 1024, against 232 and 21.9 ms for packed
// pairs of maps with Bluestein's convolution in the caps. One weight for a pixel and
// its mirror image took 6 ms off at Nside 2048 (the cap kernels' instructions per map and pixel fell by
// a fifth), and packed twiddle tables 19 ms (a warp's twiddle loads touched up to 88 lines
// a pass, as much of the load path's time as all shared-memory traffic).
#include <math.h>

#include "regfft.cuh"
#include "ringjobs.cuh"

namespace tl {

// e^{i pi c / 32}, c = 0 .. 31
__device__ __constant__ float2 kRoot64[32] = {
    {1.0f, 0.0f}, {0.99518472667219693f, 0.098017140329560604f}, {0.98078528040323043f, 0.19509032201612825f},
    {0.95694033573220882f, 0.29028467725446233f}, {0.92387953251128674f, 0.38268343236508978f},
    {0.88192126434835505f, 0.47139673682599764f}, {0.83146961230254524f, 0.55557023301960218f},
    {0.77301045336273699f, 0.63439328416364549f}, {0.70710678118654757f, 0.70710678118654757f},
    {0.63439328416364549f, 0.77301045336273699f}, {0.55557023301960218f, 0.83146961230254524f},
    {0.47139673682599764f, 0.88192126434835505f}, {0.38268343236508978f, 0.92387953251128674f},
    {0.29028467725446233f, 0.95694033573220882f}, {0.19509032201612825f, 0.98078528040323043f},
    {0.098017140329560604f, 0.99518472667219693f}, {0.0f, 1.0f}, {-0.098017140329560604f, 0.99518472667219693f},
    {-0.19509032201612825f, 0.98078528040323043f}, {-0.29028467725446233f, 0.95694033573220882f},
    {-0.38268343236508978f, 0.92387953251128674f}, {-0.47139673682599764f, 0.88192126434835505f},
    {-0.55557023301960218f, 0.83146961230254524f}, {-0.63439328416364549f, 0.77301045336273699f},
    {-0.70710678118654757f, 0.70710678118654757f}, {-0.77301045336273699f, 0.63439328416364549f},
    {-0.83146961230254524f, 0.55557023301960218f}, {-0.88192126434835505f, 0.47139673682599764f},
    {-0.92387953251128674f, 0.38268343236508978f}, {-0.95694033573220882f, 0.29028467725446233f},
    {-0.98078528040323043f, 0.19509032201612825f}, {-0.99518472667219693f, 0.098017140329560604f}};

// Modes of a ring group:
//  direct  the ring's pixels are every (2H / N)-th grid point (N = 4 Nside <= 2H);
//  single  one grid of 2H points, at least twice the band's own;
//  twice   the largest rings: two grids of 2H points half a step apart (two transforms of
//          length H = 4096 by two groups of threads), together a grid of 4H points.
enum { kSyDirect = 0, kSySingle = 1, kSyTwice = 2 };

// TG = H / 16 threads hold one transform; a CTA of NT threads holds G of them on one
// ring. Direct CTAs are kept small (the row and the exchange array of H = 4096 take 67 KB:
// three CTAs of 256 threads per SM); the interpolating ones take several maps at a time, which
// share the interpolation weights.
template <int LG, int MODE> struct SyCfg {
  static constexpr int H = 1 << LG, TG = H >> 4;
  static constexpr int NT = MODE == kSyDirect ? 256 : LG >= 11 ? 512 : LG == 8 ? 128 : 256;
  static constexpr int CTAS = MODE == kSyDirect ? (LG == 12 ? 3 : 4) : (LG >= 11 ? 2 : LG == 8 ? 8 : 4);
  static constexpr int G = NT / TG;
  static constexpr int MAPS = MODE == kSyTwice ? 1 : G;  // maps of a CTA at a time
  static constexpr int W = kSyW;
  static constexpr int X = RegFft<LG, +1>::SMEM;  // float2 of an exchange array
};

struct SyArgs {
  const int *nphi;
  const long long *first;
  const double *phi0;
  const float *rsinf;
  const int4 *rings;    // {ring, band, fold, mcut}
  const float2 *tw;     // e^{-2 pi i k / TW}, k < TW / 2
  const float4 *tw4;    // twiddles of the passes of this length (TwidPacked)
  const float *corr;    // 1 / (window's transform) at m / (finest grid)
  int lgtw, mmax, rounds, chunks, rowcap;
  float invL;
  long long tile;       // tile stride of the jobs whose output is tiled (the same for all of them)
};

// Output of one map of an interpolating CTA's round (out: null where there is none)
struct __align__(16) SyOut {
  float *out;
  float scale;
  int tiled;
};

// The aliases of class t (m = t + q N and m = q N - t) of one coefficient row with the
// factor (i m / L)^k, up to the common phase of class t: S_t = sum_q s^q G_{t + qN} +
// sum_{q >= 1} s^q conj G_{qN - t} (0 < t < N/2), s = -1 on half-pixel-shifted rings.
__device__ __forceinline__ float2 sy_fold(const float2 *__restrict__ F, int fs, int t, int N, int mmax, int k, float invL,
                                       bool shifted) {
  float2 s = f2(0.0f, 0.0f);
  int q = 0;
  for (int m = t; m <= mmax; m += N, ++q) {
    const float2 v = __ldg(F + (size_t)m * fs);
    float pw = (shifted && (q & 1)) ? -1.0f : 1.0f;
    const float mm = (float)m * invL;
    for (int i = 0; i < k; ++i) pw *= mm;
    const float2 g = rot_ik(f2(v.x * pw, v.y * pw), k);
    s.x += (t == 0 && q > 0) ? 2.0f * g.x : g.x;
    s.y += g.y;
  }
  if (t > 0 && 2 * t < N) {
    q = 1;
    for (int m = N - t; m <= mmax; m += N, ++q) {
      const float2 v = __ldg(F + (size_t)m * fs);
      float pw = (shifted && (q & 1)) ? -1.0f : 1.0f;
      const float mm = (float)m * invL;
      for (int i = 0; i < k; ++i) pw *= mm;
      const float2 g = rot_ik(f2(v.x * pw, v.y * pw), k);
      s.x += g.x;
      s.y -= g.y;
    }
  }
  return s;
}

template <int LG, int MODE>
__global__ void __launch_bounds__(SyCfg<LG, MODE>::NT, SyCfg<LG, MODE>::CTAS)
    ringfft_synth_kernel(SyArgs A, const __grid_constant__ JobList jobs, const __grid_constant__ SyWindow win) {
  typedef SyCfg<LG, MODE> C;
  typedef RegFft<LG, +1> F;
  constexpr int H = C::H, TG = C::TG, NT = C::NT, N2 = 2 * H;
  constexpr bool INTERP = MODE != kSyDirect;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ SyOut outs[INTERP ? C::MAPS : 1];
  // the next group's blocks may start where this one's leave room (they share nothing; the wait is at
  // the end; see launch_ring_synth)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int tid = threadIdx.x, g = tid / TG, h = tid - g * TG;
  const int ring = blockIdx.x / A.chunks, chunk = blockIdx.x - ring * A.chunks;
  const int4 R = A.rings[ring];
  const int r = R.x, band = R.y;
  const bool fold = R.z != 0;
  const float rs = A.rsinf[r];
  const int N = A.nphi[r];
  const long long first = A.first[r];
  const bool shifted = __double_as_longlong(A.phi0[r]) != 0;  // phi0 >= 0: an integer test
  // rows (one per group; one in all for `twice`), then the exchange arrays
  float2 *rows = (float2 *)smem_raw;
  float2 *xch = rows + (MODE == kSyTwice ? 1 : C::G) * A.rowcap;
  float2 *row = rows + (MODE == kSyTwice ? 0 : g) * A.rowcap;
  float2 *xb = xch + g * C::X;
  const int sm0 = MODE == kSyTwice ? tid : h, sms = MODE == kSyTwice ? NT : TG;  // staging threads of a row
  // the second grid of `twice` sits half a step on; the shifted belt rings' half pixel goes into
  // the staged coefficients, e^{i pi m / 2H}
  const bool half = MODE == kSyTwice && g == 1;
  const bool phase = MODE == kSyDirect && shifted && N == N2;
  const int cstep = INTERP ? (MODE == kSyTwice ? 1 : 1 << (13 - LG)) : 0;  // corr is tabulated on a grid of 2^14
  const int base = (chunk * C::MAPS + (MODE == kSyTwice ? 0 : g)) * A.rounds;  // this group's jobs

  const void *pin = nullptr;
  int pk = 0;
  for (int rd = 0; rd < A.rounds; ++rd) {
    const int jid = base + rd;
    const bool act = jid < jobs.n;
    if (act) {
      const JobDev &J = jobs.job[jid];
      const int k = J.k;
      if (J.in == pin && k == pk + 1 && !fold) {
        for (int m = sm0; m <= band; m += sms) {
          const float2 v = row[m];
          const float mm = (float)m * A.invL;  // exact
          row[m] = f2(-v.y * mm, v.x * mm);
        }
      } else {
        int fs;
        const float2 *FR = job_row<float2>(J, r, A.mmax, fs);
        if (fold) {
          for (int m = sm0; m <= band; m += sms) {
            float2 v = sy_fold(FR, fs, m, N, R.w, k, A.invL, shifted);
            if (INTERP) {
              const float c = __ldg(A.corr + m * cstep);
              v = f2(v.x * c, v.y * c);
            }
            if (m == 0) v.y = 0.0f;
            if (phase) v = cmul(v, conj_if(__ldg(A.tw + (m << (A.lgtw - LG - 2))), true));
            row[m] = v;
          }
        } else {
          constexpr int U = 8;
          for (int m0 = sm0; m0 <= band; m0 += U * sms) {
            float2 v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const int m = m0 + u * sms;
              if (m <= band) v[u] = __ldg(FR + (size_t)m * fs);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const int m = m0 + u * sms;
              if (m > band) break;
              float pw = INTERP ? __ldg(A.corr + m * cstep) : 1.0f;
              const float mm = (float)m * A.invL;
              for (int i = 0; i < k; ++i) pw *= mm;
              float2 w = rot_ik(f2(v[u].x * pw, v[u].y * pw), k);
              if (m == 0) w.y = 0.0f;
              if (phase) w = cmul(w, conj_if(__ldg(A.tw + (m << (A.lgtw - LG - 2))), true));
              row[m] = w;
            }
          }
        }
        pin = J.in;
      }
      pk = k;
    }
    __syncthreads();
    if (INTERP && tid < C::MAPS) {  // (every thread has left the round before)
      const int ji = chunk * C::MAPS * A.rounds + tid * A.rounds + rd;
      SyOut o = {nullptr, 0.0f, 0};
      if (ji < jobs.n) {
        const JobDev &J = jobs.job[ji];
        o.out = (float *)J.out;
        o.scale = J.scalef * (J.div_sint ? rs : 1.0f);
        o.tiled = J.tile != 0;
      }
      outs[tid] = o;
    }
    float2 x[16];
    {
      const float2 wh = conj_if(__ldg(A.tw + (h << (A.lgtw - LG - 1))), true);  // e^{2 pi i h / 2H}
      float2 eh = f2(1.0f, 0.0f);
      if (half) eh = conj_if(__ldg(A.tw + (h << (A.lgtw - LG - 2))), true);  // its square root
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const int m = h + TG * c, pm = H - m;
        const float2 zero = f2(0.0f, 0.0f);
        const float2 a = (act && m <= band) ? row[m] : zero;
        float2 b = (act && pm <= band) ? row[pm] : zero;
        b.y = -b.y;  // conj S_{H-m}
        if (MODE == kSyTwice && half) b = f2(b.y, -b.x);  // times e_{-(H-m)} = -i e_m, below
        const float2 w = cmul(wh, kRoot64[(2 * c) & 31]);  // e^{2 pi i m / 2H}
        const float2 s = cadd(a, b), wd = cmul(w, csub(a, b));
        x[c] = f2(s.x - wd.y, s.y + wd.x);
        if (MODE == kSyTwice && half) x[c] = cmul(x[c], cmul(eh, kRoot64[c]));
      }
      if (MODE == kSyDirect && h == 0 && act && band == H) {
        // the Nyquist term S_H = 2 Re(G_H e^{i H phi0}) (real), beside S_0 in Z_0
        const float s0 = row[0].x, sH = 2.0f * row[H].x;
        x[0] = f2(s0 + sH, s0 - sH);
      }
    }
    F::run(x, xb, h, TwidPacked{A.tw4});
    if (!INTERP) {
      if (act) {
        const JobDev &J = jobs.job[jid];
        const float sc = J.scalef * (J.div_sint ? rs : 1.0f);
        float *out = (float *)J.out;
        if (N == N2 && 2 * TG >= kD3Tile) {
          // slots lie a multiple of the tile's pixels apart: a constant distance in either layout
          const long long p = first + 2 * h;
          float *o = out + (J.tile ? d3_pix(p, J.tile) : p);
          const long long step = J.tile ? (long long)(2 * TG / kD3Tile) * J.tile : 2 * TG;
#pragma unroll
          for (int c = 0; c < 16; ++c) *(float2 *)(o + c * step) = f2(sc * x[c].x, sc * x[c].y);
        } else if (N == N2) {
#pragma unroll
          for (int c = 0; c < 16; ++c) {
            const long long p = first + 2 * (h + TG * c);
            *(float2 *)(out + (J.tile ? d3_pix(p, J.tile) : p)) = f2(sc * x[c].x, sc * x[c].y);
          }
        } else {
          // a ring shorter than the grid: its pixels are every (2H / N)-th point, from half
          // a pixel on for the shifted rings
          const int dec = N2 / N, off = shifted ? dec >> 1 : 0;
#pragma unroll
          for (int c = 0; c < 16; ++c) {
            const int f = 2 * (h + TG * c) - off;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              if (f + e >= 0 && (f + e) % dec == 0) {
                const long long p = first + (f + e) / dec;
                out[J.tile ? d3_pix(p, J.tile) : p] = sc * (e ? x[c].y : x[c].x);
              }
            }
          }
        }
      }
    } else {
      // the grid into the exchange array (every thread's last reads of it lie before the
      // barrier of the last pass), with eight points of the other end at either side
      float *gr = (float *)xb + 8;
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const int n = h + TG * c;
        *(float2 *)(gr + 2 * n) = x[c];
        if (c == 0 && n < 4) *(float2 *)(gr + N2 + 2 * n) = x[c];
        if (c == 15 && n >= H - 4) *(float2 *)(gr + 2 * n - N2) = x[c];
      }
      __syncthreads();
      constexpr int W = C::W, HW = W / 2;
      constexpr int NFL = LG + 1 + (MODE == kSyTwice ? 1 : 0);  // log2 of the fine grid
      const int den = 2 * N;
      const float inv = 1.0f / (float)den, inv2 = 0.5f * inv;
      const float *g0 = (const float *)xch + 8;
      // Pixel p of a half-pixel-shifted ring (every cap ring) sits at (2 p + 1) 2^NFL / (2 N) = i0 +
      // rem / den on the fine grid, and pixel N - 1 - p at its mirror image: the same weights, in
      // reverse, serve both, for all maps of the round
      for (int p = tid; p < N / 2; p += NT) {
        const int num = (2 * p + 1) << NFL;
        int i0 = (int)((float)num * inv);
        int rem = num - i0 * den;
        if (rem < 0) {
          --i0;
          rem += den;
        } else if (rem >= den) {
          ++i0;
          rem -= den;
        }
        // s = rem / den - 1/2, correctly rounded up to the last bit
        const float sn = (float)(2 * rem - den), dn = (float)(2 * den);
        float s = sn * inv2;
        s = fmaf(fmaf(-s, dn, sn), inv2, s);
        const float s2 = s * s;
        float wt[W];
#pragma unroll
        for (int t = 0; t < HW; ++t) {
          const float *pc = win.c[t];
          constexpr int NE = 5, NO = 4;  // even and odd coefficients
          float e = pc[2 * (NE - 1)], o = pc[2 * NO - 1];
#pragma unroll
          for (int i = NE - 2; i >= 0; --i) e = fmaf(e, s2, pc[2 * i]);
#pragma unroll
          for (int i = NO - 2; i >= 0; --i) o = fmaf(o, s2, pc[2 * i + 1]);
          wt[t] = fmaf(s, o, e);
          wt[W - 1 - t] = fmaf(-s, o, e);
        }
        const int b0 = i0 - HW + 1, b1 = (1 << NFL) - i0 - HW;  // the first of the W points of either pixel
        const long long pa = first + p, pb = first + N - 1 - p;
        const long long ta = d3_pix(pa, A.tile), tb = d3_pix(pb, A.tile);
#pragma unroll
        for (int i = 0; i < C::MAPS; ++i) {
          const SyOut o = outs[i];
          if (!o.out) break;  // (the maps of a round are its first ones)
          float va = 0.0f, vb = 0.0f;
          if (MODE == kSyTwice) {
            // fine point f is point f >> 1 of grid f & 1
            const float *a0 = g0 + (b0 & 1) * (2 * C::X) + (b0 >> 1);
            const float *a1 = g0 + ((b0 & 1) ^ 1) * (2 * C::X) + ((b0 + 1) >> 1);
            const float *c0 = g0 + (b1 & 1) * (2 * C::X) + (b1 >> 1);
            const float *c1 = g0 + ((b1 & 1) ^ 1) * (2 * C::X) + ((b1 + 1) >> 1);
#pragma unroll
            for (int t = 0; t < HW; ++t) {
              va = fmaf(wt[2 * t], a0[t], va);
              va = fmaf(wt[2 * t + 1], a1[t], va);
              vb = fmaf(wt[W - 1 - 2 * t], c0[t], vb);
              vb = fmaf(wt[W - 2 - 2 * t], c1[t], vb);
            }
          } else {
            const float *gi = g0 + i * (2 * C::X);
#pragma unroll
            for (int t = 0; t < W; ++t) {
              va = fmaf(wt[t], gi[b0 + t], va);
              vb = fmaf(wt[W - 1 - t], gi[b1 + t], vb);
            }
          }
          o.out[o.tiled ? ta : pa] = va * o.scale;
          o.out[o.tiled ? tb : pb] = vb * o.scale;
        }
      }
      // the next round's first pass stores to the exchange arrays behind a barrier
    }
  }
  // The group before is complete and its maps are visible before this one's blocks end: so this
  // group's completion stands for that of every earlier one (see launch_ring_synth)
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ---------------------------------------------------------------------------
// plan-time tables

// Kaiser-Bessel window I0(beta sqrt(1 - (2x/W)^2)) / I0(beta), |x| < W/2
static double bessel_i0(double x) {
  double t = 1.0, s = 1.0;
  for (int k = 1; k < 200; ++k) {
    t *= (0.5 * x / k) * (0.5 * x / k);
    s += t;
    if (t < 1e-18 * s) break;
  }
  return s;
}
static double kb_window(double x, int W, double beta) {
  const double u = 1.0 - (2.0 * x / W) * (2.0 * x / W);
  return u > 0.0 ? bessel_i0(beta * sqrt(u)) / bessel_i0(beta) : 0.0;
}
// its transform int psi(x) e^{-2 pi i x xi} dx
static double kb_transform(double xi, int W, double beta) {
  const double a = M_PI * W * xi, d = beta * beta - a * a;
  const double v = d > 0.0 ? sinh(sqrt(d)) / sqrt(d) : d < 0.0 ? sin(sqrt(-d)) / sqrt(-d) : 1.0;
  return W * v / bessel_i0(beta);
}
// shape parameter for an oversampling of at least sigma (Beatty et al. 2005, IEEE Trans.
// Med. Imaging 24, 799, at infinite table density: the alias band's edge)
static double kb_beta(int W, double sigma) { return M_PI * W * (1.0 - 0.5 / sigma); }

// Polynomial of degree D through the window at distance c0 - s from a tap, s in
// [-1/2, 1/2], interpolated at Chebyshev nodes: coefficients of s^0 .. s^D
static void kb_poly(int W, double beta, double c0, int D, float *out) {
  const int n = D + 1;
  double node[16], f[16], c[16], p[16], t0[16], t1[16];
  for (int i = 0; i < n; ++i) {
    node[i] = cos(M_PI * (i + 0.5) / n);  // in units of 1/2
    f[i] = kb_window(c0 - 0.5 * node[i], W, beta);
  }
  for (int k = 0; k < n; ++k) {
    c[k] = 0.0;
    for (int i = 0; i < n; ++i) c[k] += f[i] * cos(M_PI * k * (i + 0.5) / n);
    c[k] *= (k ? 2.0 : 1.0) / n;
  }
  // sum c_k T_k(y) in powers of y = 2 s
  for (int i = 0; i < n; ++i) p[i] = t0[i] = t1[i] = 0.0;
  t0[0] = 1.0;
  p[0] += c[0];
  if (n > 1) {
    t1[1] = 1.0;
    p[1] += c[1];
  }
  for (int k = 2; k < n; ++k) {
    double t2[16];
    for (int i = 0; i < n; ++i) t2[i] = (i ? 2.0 * t1[i - 1] : 0.0) - t0[i];
    for (int i = 0; i < n; ++i) {
      p[i] += c[k] * t2[i];
      t0[i] = t1[i];
      t1[i] = t2[i];
    }
  }
  double s = 1.0;
  for (int i = 0; i < n; ++i, s *= 2.0) out[i] = (float)(p[i] * s);
}

constexpr double kSigma = 2.0;  // oversampling of a band at least

// Window polynomials, and the correction corr[m] at m / 2^14 of a grid (a band is at most the
// (2 kSigma)-th part of its grid: kSyCorr entries). They depend on nothing:
// formed once per process.
struct SynthWindow {
  SyWindow win;
  float corr[kSyCorr];
  SynthWindow() {
    const double beta = kb_beta(kSyW, kSigma);
    for (int t = 0; t < kSyW / 2; ++t) kb_poly(kSyW, beta, t - 0.5 * (kSyW - 1), 8, win.c[t]);
    for (int m = 0; m < kSyCorr; ++m) corr[m] = (float)(1.0 / kb_transform(m / 16384.0, kSyW, beta));
  }
};
const float *host_synth_window(SyWindow *w) {
  static const SynthWindow s;  // initialised by the first thread to get here
  *w = s.win;
  return s.corr;
}

// Twiddles of the transforms of length 2^8 .. 2^12 (TwidPacked), one length after another
static constexpr int synth_twiddle_offset(int lg) {
  int n = 0;
  for (int g = 8; g < lg; ++g)
    for (int p = 0; 4 * p + 4 <= g; ++p) n += 1 << (g - 4 * p - 4);
  return n;
}
int host_synth_twiddles(float *out) {
  const int n = synth_twiddle_offset(13);
  if (!out) return n * TwidPacked::PER;
  for (int g = 8; g <= 12; ++g) {
    float *o = out + 4 * TwidPacked::PER * (size_t)synth_twiddle_offset(g);
    for (int p = 0; 4 * p + 4 <= g; ++p) {
      const int L = 1 << (g - 4 * p);
      const int nj = L / 16;
      for (int j = 0; j < nj; ++j) {
        const int qs[6] = {1, 2, 3, 4, 8, 12};
        for (int q = 0; q < 6; ++q) {
          const double a = 2.0 * M_PI * (double)(j * qs[q]) / (double)L;
          float *w = o + 4 * (size_t)((q / 2) * nj + j) + 2 * (q & 1);
          w[0] = (float)cos(a);
          w[1] = (float)sin(a);
        }
      }
      o += 12 * (size_t)nj;
    }
  }
  return n;
}

// Group of one ring, by its length and band (mcut: its coefficients beyond are zero):
// the belt on its own grid; the caps on the smallest grid that oversamples their band kSigma times,
// which is half the ring's length where folding the aliases buys a smaller grid.
// Returns the group key (mode and log2 H), -1 if no grid fits; sets band and fold.
static int synth_key(int nside, int nphi, int mcut, int *band, int *fold) {
  *fold = 0;
  *band = mcut;
  if (nphi == 4 * nside) {
    int lg = 8;
    while ((2 << lg) < nphi) ++lg;
    if (lg > 12) return -1;
    if (mcut > (1 << lg)) {
      *fold = 1;
        *band = nphi / 2;
    }
    return kSyDirect * 16 + lg;
  }
  auto grid = [](int b) {
    for (int lg = 8; lg <= 12; ++lg)
      if ((double)(2 << lg) >= kSigma * 2.0 * b) return kSySingle * 16 + lg;
    return b <= 4095 ? kSyTwice * 16 + 12 : -1;
  };
  int key = grid(mcut);
  if (2 * mcut > nphi) {
    const int kf = grid(nphi / 2);
    if (kf >= 0 && (key < 0 || kf < key)) {
      *fold = 1;
      *band = nphi / 2;
      key = kf;
    }
  }
  return key;
}

// Ring groups of the synthesis kernels: rings[] = {ring, band, fold, mcut} by group, longest
// rings first within a group. Rings that no grid fits go to rest[] (*nrest). Returns the number of groups.
int host_synth_groups(int nside, int nrings, const int *nphi, const int *mcut, SyGroup *groups, int4 *rings, int *rest,
                      int *nrest) {
  int ng = 0, n = 0;
  *nrest = 0;
  for (int key = kSyTwice * 16 + 15; key >= 0; --key) {
    const int first = n;
    int cap = 0;
    // longest first: the belt, then pairs of cap rings from the belt's edges to the poles
    for (int d = 0; d < nrings; ++d) {
      const int r = (nrings / 2) + ((d & 1) ? (d + 1) / 2 : -(d / 2));
      int band, fold;
      if (synth_key(nside, nphi[r], mcut[r], &band, &fold) != key) continue;
      rings[n++] = make_int4(r, band, fold, mcut[r]);
      if (band > cap) cap = band;
    }
    if (n == first) continue;
    groups[ng++] = SyGroup{key >> 4, key & 15, first, n - first, cap};
  }
  for (int r = 0; r < nrings; ++r) {
    int band, fold;
    if (synth_key(nside, nphi[r], mcut[r], &band, &fold) < 0) rest[(*nrest)++] = r;
  }
  return ng;
}

// ---------------------------------------------------------------------------

// The kernels' phi-derivative factor is m / P for the power of two P >= lmax + 1: exact in float, so that
// the k-th derivative's coefficients round k times instead of carrying the k-fold rounding of m / L (and of
// 1 / L, the same for all m). (P / L)^k goes into the map's scale.
static double synth_power(int lmax) {
  double P = 1.0;
  while (P < lmax + 1.0) P *= 2.0;
  return P;
}

template <int LG, int MODE>
static cudaError_t synth_launch(const tl_plan *p, const SyGroup &g, const JobList &jl, bool overlap,
                                cudaStream_t s) {
  typedef SyCfg<LG, MODE> C;
  SyArgs A;
  A.nphi = p->ring.nphi;
  A.first = p->ring.first;
  A.phi0 = p->ring.phi0;
  A.rsinf = p->ring.rsinf;
  A.rings = p->sy_rings + g.first;
  A.tw = (const float2 *)p->twiddle;
  A.tw4 = p->sy_tw4 + TwidPacked::PER * synth_twiddle_offset(LG);
  A.corr = p->sy_corr;
  A.lgtw = 31 - __builtin_clz((unsigned)p->tw_len);
  A.mmax = p->mmax;
  A.rowcap = (g.band + 2) & ~1;
  A.invL = (float)(1.0 / synth_power(p->lmax));
  A.tile = 0;
  for (int i = 0; i < jl.n; ++i)
    if (jl.job[i].tile) {
      if (A.tile && A.tile != jl.job[i].tile) return cudaErrorInvalidValue;
      A.tile = jl.job[i].tile;
    }
  // jobs of a CTA: its groups take `rounds` consecutive jobs each (one plane's maps
  // follow one another, so a row is staged about once per plane and ring), short enough that the
  // launch has about eight CTAs per resident one (16, 5, 3 and 2 measured up to 5% slower)
  const int slots = C::CTAS * p->num_sms;
  const int most = (jl.n + C::MAPS - 1) / C::MAPS;  // rounds with one chunk
  int chunks = (8 * slots + g.count - 1) / g.count;
  if (chunks > most) chunks = most;
  if (chunks < 1) chunks = 1;
  A.rounds = (most + chunks - 1) / chunks;
  A.chunks = (most + A.rounds - 1) / A.rounds;
  const size_t smem =
      sizeof(float2) * ((size_t)(MODE == kSyTwice ? 1 : C::G) * A.rowcap + (size_t)C::G * C::X);
  auto kern = ringfft_synth_kernel<LG, MODE>;
  TL_CUDA_TRY(raise_smem((const void *)kern, smem));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(g.count * A.chunks));
  cfg.blockDim = dim3(C::NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, A, jl, p->sy_win);
}

// The groups write different rings and read only what the stream's work before the first has left, so each
// launch after the first lets its blocks start as the one before runs out of blocks (programmatic
// serialization; the first waits for the stream as usual): otherwise every group ends in a partly empty
// chip. What follows the last group is ordered after that group alone, in a captured graph above all,
// so every block waits for the group before at its end: the groups then complete in order. The
// blocks that wait have all been placed, and those they wait for have all started. Up to Nside 1024: sixteen skies take 0.31 instead of
// 0.40 ms at Nside 32, 0.91 for 1.12 at 128, 2.94 for 3.28 at 256, 10.4 for 11.0 at 512 and 37.9 for 39.1 at
// 1024, but 120.2 for 117.8 at 2048, where the ends weigh little.
cudaError_t launch_ring_synth(const tl_plan *p, JobList &jl, cudaStream_t s) {
  const double c = synth_power(p->lmax) / (double)(p->lmax + 1);
  for (int i = 0; i < jl.n; ++i) jl.job[i].scalef = (float)(jl.job[i].scale * pow(c, jl.job[i].k));
  for (int i = 0; i < p->sy_ngroups; ++i) {
    const SyGroup &g = p->sy_groups[i];
    cudaError_t e = cudaErrorInvalidValue;
#define SY(LG_, MODE_) \
  if (g.lg == LG_ && g.mode == MODE_) e = synth_launch<LG_, MODE_>(p, g, jl, i > 0 && p->nside <= 1024, s);
    SY(8, kSyDirect) SY(9, kSyDirect) SY(10, kSyDirect) SY(11, kSyDirect) SY(12, kSyDirect)
    SY(8, kSySingle) SY(9, kSySingle) SY(10, kSySingle) SY(11, kSySingle) SY(12, kSySingle)
    SY(12, kSyTwice)
#undef SY
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace tl
