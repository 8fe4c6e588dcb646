// Legendre stage in single precision without tensor cores: the kernels of legendre.cu (see there
// and legendre.cuh for the mathematics; Naess & Louis 2013, Sec. II.B, Eq. 4), whose steps are
// bound by instruction issue. Two things keep the instructions per step near the arithmetic's
// own (at order 4: 45 for spin 2, 39 for spin 0 with the potential):
//  - the records of kChunk values of l are staged in shared memory by the block, so that a step reads its
//    factors with two broadcast loads;
//  - once every ring of a warp has reached scale 0 it stays there, and the steps run without
//    the tests for it; before that, a thread whose ring has not reached it does not contract, and
//    a warp whose rings never reach it at this m (host_ring_bands) runs no steps.
// Every value is formed by the same operations in the same order as in the general kernels.
// Order 4, spin 2, Nside 512 / lmax 1024: 2.35 -> 1.64 ms (79% issue-active before and 77% now, 65 -> 55
// instructions per ring and step run, a fifth of the steps not run); spin 0 0.98 -> 0.68 ms; the
// deflection alone to lmax 4096 7.5 -> 4.3 ms. Two rings per thread in packed pairs (f32x2) took
// 2.40 ms: one packed instruction holds its pipe for two cycles, and the pairs' moves ate the rest.
#include <math.h>

#include "legendre.cuh"

namespace tl {

constexpr int kChunk = 32;  // values of l staged at a time (even)

// ---------------------------------------------------------------------------
// spin 0: one north ring per thread, the south ring by parity; the potential's j <= 1 sums from
// the same recurrence with PHI (see legendre_spin0_kernel)

template <int NDER, bool PHI, int NT>
__global__ void __launch_bounds__(NT) legendre_spin0_f32_kernel(RingTable rt, const double *__restrict__ lnorm0,
                                                                int nside, int lmax, int mmax, int nrings,
                                                                const int *__restrict__ mcut,
                                                                const Rec0<float> *__restrict__ rec,
                                                                const float2 *__restrict__ recp,
                                                                float2 *__restrict__ d7, float2 *__restrict__ d7p) {
  constexpr int NJ = NDER + 1, NP = PHI ? 2 : 0;
  __shared__ float4 st[2][kChunk];  // re, im, A, Q
  __shared__ float2 sp[2][PHI ? kChunk : 1];
  const int m = blockIdx.y, t = threadIdx.x;
  const int rn = blockIdx.x * NT + t;
  const bool active = rn < 2 * nside;
  const int r = active ? rn : 0;
  // a warp none of whose rings leaves zero at this m runs no steps, a block of such warps none at all
  const bool live = __any_sync(0xffffffffu, active && (!mcut || m <= mcut[r]));
  const int top = __syncthreads_or(live) ? lmax : -1;
  const double invL = 1.0 / (double)(lmax + 1);
  Leib<float, NDER> LC;
  leibniz_coefs<float, NDER>(rt.z[r], rt.sint[r], invL, LC);
  float d[NJ], v[NJ];
  int sc;
  seed_spin0<float, NDER>(rt, lnorm0, r, m, invL, v, sc);
  rec_init<float, NDER>(d, v);
  const float w = (float)rt.omza[r];
  float s[2][2][NJ], q[2][2][2];  // [parity of l - m][re, im][j]
#pragma unroll
  for (int p = 0; p < 2; ++p)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
#pragma unroll
      for (int j = 0; j < NJ; ++j) s[p][c][j] = 0.0f;
#pragma unroll
      for (int j = 0; j < 2; ++j) q[p][c][j] = 0.0f;
    }
  const long long base = (long long)m * (2 * lmax + 1 - m) / 2;
  auto load = [&](int lb, int buf) {
    for (int i = t; i < kChunk && lb + i <= top; i += NT) {
      st[buf][i] = __ldg((const float4 *)(rec + base + lb + i));
      if (PHI) sp[buf][i] = __ldg(recp + base + lb + i);
    }
  };
  bool plain = false;  // every ring of the warp at scale 0
  load(m, 0);
  int buf = 0;
  for (int lb = m; lb <= top; lb += kChunk, buf ^= 1) {
    const int n = min(kChunk, lmax - lb + 1);
    __syncthreads();  // this chunk is staged, the one before has been read
    if (lb + kChunk <= top) load(lb + kChunk, buf ^ 1);
    auto contract = [&](float4 c, float2 e, int p) {
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        s[p][0][j] = fmaf(c.x, v[j], s[p][0][j]);
        s[p][1][j] = fmaf(c.y, v[j], s[p][1][j]);
      }
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        q[p][0][j] = fmaf(e.x, v[j], q[p][0][j]);
        q[p][1][j] = fmaf(e.y, v[j], q[p][1][j]);
      }
    };
    if (!live) continue;
    int i = 0;
    // kChunk is even: the parity of l - m is that of i
#pragma unroll 1
    for (; i + 1 < n && !plain; i += 2) {
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const float4 c = st[buf][i + p];
        if (sc == 0) contract(c, PHI ? sp[buf][i + p] : make_float2(0.0f, 0.0f), p);
        step_diff<float, NDER, 1>(v, d, LC, w, c.z, c.w);
        rescale<float, NDER>(d, v, v[0], sc);
      }
      plain = __all_sync(0xffffffffu, sc == 0);  // and stays so
    }
#pragma unroll 2
    for (; i + 1 < n; i += 2) {
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const float4 c = st[buf][i + p];
        contract(c, PHI ? sp[buf][i + p] : make_float2(0.0f, 0.0f), p);
        step_diff<float, NDER, 1>(v, d, LC, w, c.z, c.w);
      }
    }
    if (i < n && sc == 0) contract(st[buf][i], PHI ? sp[buf][i] : make_float2(0.0f, 0.0f), 0);  // l = lmax
  }
  if (!active || m > mmax) return;
  const int rs = nrings - 1 - r;
  const size_t ld = (size_t)(mmax + 1);
  auto put = [&](float2 *out, int j, float er, float ei, float orr, float oi) {
    const float sgn = (j & 1) ? -1.0f : 1.0f;
    out[((size_t)j * nrings + r) * ld + m] = make_float2(er + orr, ei + oi);
    if (rs != r) out[((size_t)j * nrings + rs) * ld + m] = make_float2(sgn * (er - orr), sgn * (ei - oi));
  };
#pragma unroll
  for (int j = 0; j < NJ; ++j) put(d7, j, s[0][0][j], s[0][1][j], s[1][0][j], s[1][1][j]);
#pragma unroll
  for (int j = 0; j < NP; ++j) put(d7p, j, q[0][0][j], q[0][1][j], q[1][0][j], q[1][1][j]);
}

// ---------------------------------------------------------------------------
// spin 2: the first half of the threads take north rings, the second half their mirrors
// (see legendre_spin2_kernel)

// a warp's steps through one staged chunk (SG = sign cos theta)
template <int NDER, int SG>
__device__ __forceinline__ void spin2_chunk(const float4 *__restrict__ sc4, const float2 *__restrict__ saq, int n,
                                            bool &plain, const Leib<float, NDER> &LC, float w, float (&v)[NDER + 1],
                                            float (&d)[NDER + 1], int &sc, float (&s1r)[NDER + 1],
                                            float (&s1i)[NDER + 1], float (&s2r)[NDER + 1], float (&s2i)[NDER + 1]) {
  auto contract = [&](float4 c) {
#pragma unroll
    for (int j = 0; j <= NDER; ++j) {
      s1r[j] = fmaf(c.x, v[j], s1r[j]);
      s1i[j] = fmaf(c.y, v[j], s1i[j]);
      s2r[j] = fmaf(c.z, v[j], s2r[j]);
      s2i[j] = fmaf(c.w, v[j], s2i[j]);
    }
  };
  int i = 0;
#pragma unroll 1
  for (; i < n && !plain; ++i) {
    const float2 aq = saq[i];
    if (sc == 0) contract(sc4[i]);
    step_diff<float, NDER, SG>(v, d, LC, w, aq.x, aq.y);
    rescale<float, NDER>(d, v, v[0], sc);
    plain = __all_sync(0xffffffffu, sc == 0);  // and stays so
  }
#pragma unroll 4
  for (; i < n; ++i) {
    const float2 aq = saq[i];
    contract(sc4[i]);
    step_diff<float, NDER, SG>(v, d, LC, w, aq.x, aq.y);
  }
}

template <int NDER, int NT>
__global__ void __launch_bounds__(NT) legendre_spin2_f32_kernel(RingTable rt, const double *__restrict__ lnorm0,
                                                                int nside, int lmax, int mmax, int nrings,
                                                                const int *__restrict__ mcut,
                                                                const Rec2<float> *__restrict__ rec,
                                                                float2 *__restrict__ d7q, float2 *__restrict__ d7u) {
  constexpr int NJ = NDER + 1, HT = NT / 2;
  static_assert(HT % 32 == 0, "mirror threads are whole warps");
  __shared__ float4 st[2][kChunk];      // c1r, c1i, c2r, c2i
  __shared__ float2 aq[2][2][kChunk];   // [buffer][north, mirror] A, Q
  __shared__ float2 xch[NT][NJ];
  const int m = blockIdx.y, t = threadIdx.x;
  const bool mirror = t >= HT;
  const int rn = blockIdx.x * HT + (mirror ? t - HT : t);
  const bool active = rn < 2 * nside;
  const int r = active ? (mirror ? nrings - 1 - rn : rn) : 0;
  // (as for spin 0)
  const bool live = __any_sync(0xffffffffu, active && (!mcut || m <= mcut[r]));
  const int top = __syncthreads_or(live) ? lmax : -1;
  const double invL = 1.0 / (double)(lmax + 1);
  Leib<float, NDER> LC;
  leibniz_coefs<float, NDER>(rt.z[r], rt.sint[r], invL, LC);
  float d[NJ], v[NJ];
  int sc;
  const int l0 = seed_spin2<float, NDER>(rt, lnorm0, r, m, invL, v, sc);
  rec_init<float, NDER>(d, v);
  const float w = (float)rt.omza[r];
  float s1r[NJ], s1i[NJ], s2r[NJ], s2i[NJ];
#pragma unroll
  for (int j = 0; j < NJ; ++j) s1r[j] = s1i[j] = s2r[j] = s2i[j] = 0.0f;
  const Rec2<float> *rm = rec + (long long)m * (2 * lmax + 1 - m) / 2;
  auto load = [&](int lb, int buf) {
    for (int i = t; i < kChunk && lb + i <= top; i += NT) {
      const float4 *p = (const float4 *)(rm + lb + i);
      st[buf][i] = __ldg(p);
      const float4 f = __ldg(p + 1);  // A, m s / (l (l + 1)), Qn, Qs
      aq[buf][0][i] = make_float2(f.x, f.z);
      aq[buf][1][i] = make_float2(f.x, f.w);
    }
  };
  bool plain = false;  // every ring of the warp at scale 0
  load(l0, 0);
  int buf = 0;
  for (int lb = l0; lb <= top; lb += kChunk, buf ^= 1) {
    const int n = min(kChunk, lmax - lb + 1);
    __syncthreads();  // this chunk is staged, the one before has been read
    if (lb + kChunk <= top) load(lb + kChunk, buf ^ 1);
    if (!live) continue;
    if (mirror)
      spin2_chunk<NDER, -1>(st[buf], aq[buf][1], n, plain, LC, w, v, d, sc, s1r, s1i, s2r, s2i);
    else
      spin2_chunk<NDER, 1>(st[buf], aq[buf][0], n, plain, LC, w, v, d, sc, s1r, s1i, s2r, s2i);
  }
#pragma unroll
  for (int j = 0; j < NJ; ++j) xch[t][j] = make_float2(s2r[j], s2i[j]);
  __syncthreads();
  if (!active || m > mmax) return;
  if (mirror && rn == nrings - 1 - rn) return;  // equator: the north thread writes it
  const int partner = mirror ? t - HT : t + HT;
  const size_t ld = (size_t)(mmax + 1);
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    const float2 p = xch[partner][j];
    const float sg = (j & 1) ? -1.0f : 1.0f;
    const float ar = s1r[j] + sg * p.x, ai = s1i[j] + sg * p.y;  // S1 + (-1)^j S2'
    const float br = s1r[j] - sg * p.x, bi = s1i[j] - sg * p.y;  // S1 - (-1)^j S2'
    const size_t o = ((size_t)j * nrings + r) * ld + m;
    d7q[o] = make_float2(-0.5f * ar, -0.5f * ai);
    d7u[o] = make_float2(-0.5f * bi, 0.5f * br);  // i (br + i bi) / 2
  }
}

// ---------------------------------------------------------------------------
// launchers: larger blocks share a staged record between more rings, smaller ones where the rings
// would not fill them

template <int NDER, bool PHI>
static cudaError_t f32_spin0(const tl_plan *p, void *d7, void *d7p, cudaStream_t s) {
  const int rings = 2 * p->nside;
#define RUN(NT)                                                                                            \
  legendre_spin0_f32_kernel<NDER, PHI, NT><<<dim3((rings + NT - 1) / NT, p->mmax + 1), NT, 0, s>>>(        \
      p->ring, p->lnorm0, p->nside, p->lmax, p->mmax, p->nrings, p->mcut, (const Rec0<float> *)p->rec_T,            \
      (const float2 *)p->rec_P, (float2 *)d7, (float2 *)d7p)
  if (rings >= 128) RUN(128);
  else RUN(32);
#undef RUN
  return cudaGetLastError();
}

template <int NDER> static cudaError_t f32_spin2(const tl_plan *p, cudaStream_t s) {
  const int rings = 2 * p->nside;
#define RUN(NT)                                                                                            \
  legendre_spin2_f32_kernel<NDER, NT><<<dim3((rings + NT / 2 - 1) / (NT / 2), p->mmax + 1), NT, 0, s>>>(   \
      p->ring, p->lnorm0, p->nside, p->lmax, p->mmax, p->nrings, p->mcut, (const Rec2<float> *)p->rec_QU,           \
      (float2 *)p->d7_Q, (float2 *)p->d7_U)
  if (rings >= 128) RUN(128);
  else RUN(64);
#undef RUN
  return cudaGetLastError();
}

cudaError_t launch_legendre_spin0_f32(const tl_plan *p, int nder, bool phi, void *d7, void *d7p, cudaStream_t s) {
  switch (nder) {
    case 0: return phi ? cudaErrorInvalidValue : f32_spin0<0, false>(p, d7, d7p, s);
#define CASE(n) \
  case n: return phi ? f32_spin0<n, true>(p, d7, d7p, s) : f32_spin0<n, false>(p, d7, d7p, s);
    CASE(1) CASE(2) CASE(3) CASE(4) CASE(5) CASE(6)
#undef CASE
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_legendre_spin2_f32(const tl_plan *p, int nder, cudaStream_t s) {
  switch (nder) {
#define CASE(n) \
  case n: return f32_spin2<n>(p, s);
    CASE(0) CASE(1) CASE(2) CASE(3) CASE(4) CASE(5) CASE(6)
#undef CASE
  }
  return cudaErrorInvalidValue;
}

}  // namespace tl
