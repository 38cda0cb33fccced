// Register + shared-memory FFT engine of the line lengths P = 1536 and 3072 (P = 3 PB, PB = 512 and
// 1024), and the complex helpers shared with holo_line.cuh.
//
// The Fresnel operator D_z (Appendix A, Eq. defPz/defGz) is a circular convolution on
// the P x P grid; with a separable chirp exp(-i pi lambda z (fx^2 + fy^2)) it factors into
// one pass over rows and one over columns, each "FFT -> chirp -> inverse FFT" along a
// line.
//
// Sub-line of length PB: TB = PB/16 threads, 16 complex values per thread: thread t, register c
// holds element t + TB c ("strided natural" layout).  The forward transform is a mixed-radix
// decimation in frequency with radices 16, 16, R (R = 2 or 4); every stage is a DFT over one digit
// in registers followed by a twiddle and a shared-memory exchange.  The thread/register assignment of each stage is chosen so that the
// forward output is again in strided natural order, so a pointwise multiplier in frequency needs
// no reordering and the inverse transform (the adjoint stages in reverse order) consumes that
// layout directly and returns the same layout.
//
// Exchanges write register k of thread t at t + TB k (contiguous per k) and read the next stage's
// digit; addresses are padded a -> a + a/16 so both phases avoid shared memory bank conflicts.
//
// P = 3 PB.  The T = P/16 threads form three groups of TB; thread t = q TB + i
// holds element i + TB c + PB q (pos).  The forward transform first takes one radix-3
// decimation-in-frequency step through shared memory: group q forms
//   y_q[n] = W_P^{n q} (x[n] + W_3^q x[n + PB] + W_3^{2q} x[n + 2 PB]),  n = i + TB c,
// which is one output of each of the PB three-point butterflies, then group q transforms
// y_q with the power-of-two engine above on its own third of the buffer.  Register rho of
// thread (q, i) then holds frequency 3 (i + TB rho) + q (fpos).  The inverse runs the
// adjoint steps in reverse order and returns the pos layout.
//
// Synchronisation: every thread of a line group calls the transform the same number of
// times.  The buffer must be free when a transform starts and is free again when it returns.

#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace holo {

// --------------------------------------------------------------------- complex helpers

// Packed two-lane FP32 add / subtract (PTX add/sub .f32x2, sm_100 and later): both
// components of a complex value in one instruction, with the same IEEE rounding as two scalar
// operations (outputs are bit-identical to the scalar form; the issue slots of the butterfly
// additions halve).  HOLO_SCALAR_COMPLEX selects the scalar form.
#if !defined(HOLO_SCALAR_COMPLEX)
__device__ __forceinline__ unsigned long long pk(float2 a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ float2 upk(unsigned long long r) {
  float2 a;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
  return a;
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pk(a)), "l"(pk(b)));
  return upk(d);
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
  unsigned long long d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pk(a)), "l"(pk(b)));
  return upk(d);
}
#else
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
#endif
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// a * conj(b)
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.y, b.x, -a.x * b.y));
}
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
// multiply by -i (forward) or +i (inverse)
template <bool INV>
__device__ __forceinline__ float2 mul_mi(float2 a) {
  return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

// --------------------------------------------------------------------- shapes

__host__ __device__ constexpr int ilog2c(int x) { return x <= 1 ? 0 : 1 + ilog2c(x >> 1); }
__host__ __device__ constexpr int ipow16(int s) { return s == 0 ? 1 : 16 * ipow16(s - 1); }

__device__ __forceinline__ int spad(int a) { return a + (a >> 4); }

__host__ __device__ constexpr bool is_pow2c(int x) { return x > 0 && (x & (x - 1)) == 0; }

// A sub-line: two radix-16 stages, then one of radix R.  Stage s: prefix length 16^s, remaining length
// M(s) = PB / 16^(s+1).
template <int PB>
struct SubLine {
  static_assert(PB == 512 || PB == 1024, "sub-line length");
  static constexpr int T = PB / 16;                // threads
  static constexpr int N16 = 2;                    // radix-16 stages
  static constexpr int R = PB / 256;               // radix of the last stage
  static constexpr int SMEM = PB + PB / 16;        // padded exchange buffer, float2 entries
  __host__ __device__ static constexpr int M(int s) { return PB / ipow16(s + 1); }
  // twiddle table in global memory: 15 M(s) entries a stage; in shared memory the roots
  // W_PB^{mu 16^s} (k = 1) of every stage only
  __host__ __device__ static constexpr int tw_off(int s) {
    return s == 0 ? 0 : tw_off(s - 1) + 15 * M(s - 1);
  }
  __host__ __device__ static constexpr int roots_off(int s) {
    return s == 0 ? 0 : roots_off(s - 1) + M(s - 1);
  }
};

template <int P_>
struct Fft {
  static constexpr int P = P_;
  static constexpr int PB = P / 3;                 // sub-line length
  using S = SubLine<PB>;
  static constexpr int T = P / 16;                 // threads per line
  static constexpr int TB = S::T;                  // threads per sub-line
  static constexpr int SMEM = 3 * S::SMEM;
  // radix-3 step: W_P^n and W_P^{2n}, n < PB, appended to both tables
  static constexpr int TW_BASE = S::tw_off(S::N16), TW = TW_BASE + 2 * PB;
  static constexpr int ROOTS_BASE = S::roots_off(S::N16), ROOTS = ROOTS_BASE + 2 * PB;
  // line element held in register c of thread t, and the frequency it holds after fft_fwd
  __host__ __device__ static constexpr int pos(int t, int c) {
    return t % TB + TB * c + PB * (t / TB);
  }
  __host__ __device__ static constexpr int fpos(int t, int c) {
    return 3 * (t % TB + TB * c) + t / TB;
  }
};

// --------------------------------------------------------------------- small DFTs

template <bool INV>
__device__ __forceinline__ void dft2(float2& a, float2& b) {
  float2 s = cadd(a, b), d = csub(a, b);
  a = s;
  b = d;
}

// natural order in, natural order out
template <bool INV>
__device__ __forceinline__ void dft4(float2& x0, float2& x1, float2& x2, float2& x3) {
  const float2 s02 = cadd(x0, x2), d02 = csub(x0, x2);
  const float2 s13 = cadd(x1, x3), e = csub(x1, x3);
  x0 = cadd(s02, s13);
  x2 = csub(s02, s13);
  // d02 +/- (-i e) forward, d02 +/- (i e) inverse, the swap folded into scalar adds
  const float2 p = make_float2(d02.x + e.y, d02.y - e.x), m = make_float2(d02.x - e.y, d02.y + e.x);
  x1 = INV ? m : p;
  x3 = INV ? p : m;
}

// W16^m as (cos, -sin) of 2 pi m / 16 (conjugated for the inverse)
template <bool INV>
__device__ __forceinline__ float2 w16(int m) {
  const float c1 = 0.92387953251128674f, s1 = 0.38268343236508977f, h = 0.70710678118654752f;
  float2 w;
  switch (m) {
    case 1: w = make_float2(c1, -s1); break;
    case 2: w = make_float2(h, -h); break;
    case 3: w = make_float2(s1, -c1); break;
    case 4: w = make_float2(0.f, -1.f); break;
    case 6: w = make_float2(-h, -h); break;
    case 9: w = make_float2(-c1, s1); break;
    default: w = make_float2(1.f, 0.f); break;
  }
  return INV ? cconj(w) : w;
}

template <bool INV>
__device__ __forceinline__ void dft16(float2* v) {
  // 4 x 4: DFT-4 over c2 (elements c1 + 4 c2), twiddle W16^(c1 k2), DFT-4 over c1;
  // output index k2 + 4 k1.
  float2 y[16];
#pragma unroll
  for (int c1 = 0; c1 < 4; ++c1) {
    float2 a = v[c1], b = v[c1 + 4], c = v[c1 + 8], d = v[c1 + 12];
    dft4<INV>(a, b, c, d);
    y[c1 * 4 + 0] = a;
    y[c1 * 4 + 1] = (c1 == 0) ? b : cmul(b, w16<INV>(c1 * 1));
    y[c1 * 4 + 2] = (c1 == 0) ? c : (c1 == 2 ? mul_mi<INV>(c) : cmul(c, w16<INV>(c1 * 2)));
    y[c1 * 4 + 3] = (c1 == 0) ? d : cmul(d, w16<INV>(c1 * 3));
  }
#pragma unroll
  for (int k2 = 0; k2 < 4; ++k2) {
    float2 a = y[0 * 4 + k2], b = y[1 * 4 + k2], c = y[2 * 4 + k2], d = y[3 * 4 + k2];
    dft4<INV>(a, b, c, d);
    v[k2 + 0] = a;
    v[k2 + 4] = b;
    v[k2 + 8] = c;
    v[k2 + 12] = d;
  }
}

template <int R, bool INV>
__device__ __forceinline__ void dft_small(float2* u) {
  if constexpr (R == 2)
    dft2<INV>(u[0], u[1]);
  else
    dft4<INV>(u[0], u[1], u[2], u[3]);
}

// --------------------------------------------------------------------- twiddle tables

// Host-side layout of the twiddle table of one line length P = 3 PB: for each radix-16
// stage s, entries [(k-1) * M(s) + mu] = exp(-2 pi i mu k 16^s / PB), k = 1..15, mu = 0..M(s)-1; then [n] = exp(-2 pi i n / P) and
// [PB + n] = exp(-2 pi i 2n / P), n < PB.  Filled in FP64 on the host.

// v[k] times the k-th power of r (its conjugate for INV), k = 1 .. 15: the powers by a product
// tree of depth <= 4 (rounding error a few ulp).
template <bool INV>
__device__ __forceinline__ void pow_apply(float2 (&v)[16], float2 r) {
  float2 w[16];
  w[1] = r;
  w[2] = cmul(r, r);
  w[3] = cmul(w[2], r);
  w[4] = cmul(w[2], w[2]);
  w[5] = cmul(w[4], r);
  w[6] = cmul(w[4], w[2]);
  w[7] = cmul(w[4], w[3]);
  w[8] = cmul(w[4], w[4]);
#pragma unroll
  for (int k = 9; k < 16; ++k) w[k] = cmul(w[8], w[k - 8]);
#pragma unroll
  for (int k = 1; k < 16; ++k) v[k] = INV ? cmulc(v[k], w[k]) : cmul(v[k], w[k]);
}

// The compact root table (Fft<P>::ROOTS entries: k = 1 of every stage, and the radix-3 step's
// twiddles), small enough to keep in shared memory next to the chirp.
struct TwRoots {
  const float2* roots;
  template <int P>
  __device__ __forceinline__ float2 r3(int idx) const {
    return roots[Fft<P>::ROOTS_BASE + idx];
  }
  template <int PB, int S, bool INV>
  __device__ __forceinline__ void apply(float2 (&v)[16], int mu) const {
    pow_apply<INV>(v, roots[SubLine<PB>::roots_off(S) + mu]);
  }
};

// Copy the roots of every stage from the full table (block-wide).
template <int P>
__device__ __forceinline__ void load_roots(float2* sm_roots, const float2* __restrict__ g_tw) {
  using F = Fft<P>;
  using B = typename F::S;
#pragma unroll
  for (int st = 0; st < B::N16; ++st)
    for (int mu = threadIdx.x; mu < B::M(st); mu += blockDim.x)
      sm_roots[B::roots_off(st) + mu] = g_tw[B::tw_off(st) + mu];
  for (int i = threadIdx.x; i < 2 * F::PB; i += blockDim.x)
    sm_roots[F::ROOTS_BASE + i] = g_tw[F::TW_BASE + i];
}

// --------------------------------------------------------------------- stages

// Barrier over the threads of one line group: the whole block.
struct SyncBlock {
  __device__ __forceinline__ void operator()() const { __syncthreads(); }
};

// The sub-line's forward transform from stage S on; thread t, register c hold element t + T c.
template <int PB, int S, class Sync>
__device__ __forceinline__ void fwd_from(float2 (&v)[16], float2* __restrict__ sm, TwRoots tw, int t,
                                         Sync sync) {
  using F = SubLine<PB>;
  if constexpr (S < F::N16) {
    constexpr int M = F::M(S);
    if constexpr (S > 0) {
      const int mu = t % M, ka = t / M;
#pragma unroll
      for (int c = 0; c < 16; ++c) v[c] = sm[spad(c * M + mu + 16 * M * ka)];
      sync();
    }
    dft16<false>(v);
    tw.template apply<PB, S, false>(v, t % M);
#pragma unroll
    for (int k = 0; k < 16; ++k) sm[spad(t + F::T * k)] = v[k];
    sync();
    fwd_from<PB, S + 1>(v, sm, tw, t, sync);
  } else {
    constexpr int R = F::R, G = 16 / R;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      float2 u[R];
      const int ka = t + F::T * g;
#pragma unroll
      for (int c = 0; c < R; ++c) u[c] = sm[spad(c + R * ka)];
      dft_small<R, false>(u);
#pragma unroll
      for (int k = 0; k < R; ++k) v[g + G * k] = u[k];
    }
    sync();
  }
}

// Its adjoint, stages S, S - 1, ..., 0.
template <int PB, int S, class Sync>
__device__ __forceinline__ void inv_from(float2 (&v)[16], float2* __restrict__ sm, TwRoots tw, int t,
                                         Sync sync) {
  using F = SubLine<PB>;
  if constexpr (S == F::N16) {
    constexpr int R = F::R, G = 16 / R;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      float2 u[R];
#pragma unroll
      for (int k = 0; k < R; ++k) u[k] = v[g + G * k];
      dft_small<R, true>(u);
      const int ka = t + F::T * g;
#pragma unroll
      for (int c = 0; c < R; ++c) sm[spad(c + R * ka)] = u[c];
    }
    sync();
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = sm[spad(t + F::T * k)];
    sync();
    inv_from<PB, S - 1>(v, sm, tw, t, sync);
  } else {
    constexpr int M = F::M(S);
    tw.template apply<PB, S, true>(v, t % M);
    dft16<true>(v);
    if constexpr (S > 0) {
      const int mu = t % M, ka = t / M;
#pragma unroll
      for (int c = 0; c < 16; ++c) sm[spad(c * M + mu + 16 * M * ka)] = v[c];
      sync();
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = sm[spad(t + F::T * k)];
      sync();
      inv_from<PB, S - 1>(v, sm, tw, t, sync);
    }
  }
}

// The radix-3 butterflies of P = 3 PB: group q takes output q of every butterfly of the elements in
// sm (n = i + TB c of thread (q, i)); INV: conjugate roots of unity, no 1/3.
template <int P, bool INV, class Sync>
__device__ __forceinline__ void r3_butterfly_third(float2 (&v)[16], float2* __restrict__ sm, int t,
                                                   Sync sync) {
  using F = Fft<P>;
  constexpr int PB = F::PB, TB = F::TB;
  const float h3 = 0.86602540378443865f;  // sqrt(3)/2
  const int q = t / TB, i = t % TB;
  // output q of the butterfly (x0, x1, x2): x0 + w^q x1 + w^{2q} x2 with w = W_3 (forward)
  // or conj(W_3) (inverse), i.e. x0 - (x1 + x2)/2 -/+ i sqrt(3)/2 (x1 - x2) for q = 1, 2
  const float sg = ((q == 1) != INV) ? -h3 : h3;
#pragma unroll
  for (int c = 0; c < 16; ++c) {
    const int n = i + TB * c;
    const float2 x0 = sm[spad(n)], x1 = sm[spad(n + PB)], x2 = sm[spad(n + 2 * PB)];
    const float2 su = cadd(x1, x2), df = csub(x1, x2);
    float2 y;
    if (q == 0) {
      y = cadd(x0, su);
    } else {
      y.x = fmaf(-0.5f, su.x, x0.x) - sg * df.y;
      y.y = fmaf(-0.5f, su.y, x0.y) + sg * df.x;
    }
    v[c] = y;
  }
  sync();
}

// Forward DFT (e^{-2 pi i}, unnormalised): pos layout in, fpos layout out.
template <int P, class Sync>
__device__ __forceinline__ void fft_fwd_with(float2 (&v)[16], float2* sm, TwRoots tw, int t,
                                             Sync sync) {
  using F = Fft<P>;
  constexpr int PB = F::PB, TB = F::TB;
  const int q = t / TB, i = t % TB;
#pragma unroll
  for (int c = 0; c < 16; ++c) sm[spad(i + TB * c + PB * q)] = v[c];
  sync();
  r3_butterfly_third<P, false>(v, sm, t, sync);
  if (q > 0) {
#pragma unroll
    for (int c = 0; c < 16; ++c) v[c] = cmul(v[c], tw.template r3<P>((q - 1) * PB + i + TB * c));
  }
  fwd_from<PB, 0>(v, sm + q * SubLine<PB>::SMEM, tw, i, sync);
}
// Inverse DFT without the 1/P factor (the adjoint of fft_fwd_with): fpos in, pos out.
template <int P, class Sync>
__device__ __forceinline__ void fft_inv_with(float2 (&v)[16], float2* sm, TwRoots tw, int t,
                                             Sync sync) {
  using F = Fft<P>;
  constexpr int PB = F::PB, TB = F::TB;
  const int q = t / TB, i = t % TB;
  inv_from<PB, SubLine<PB>::N16>(v, sm + q * SubLine<PB>::SMEM, tw, i, sync);
  if (q > 0) {
#pragma unroll
    for (int c = 0; c < 16; ++c) v[c] = cmulc(v[c], tw.template r3<P>((q - 1) * PB + i + TB * c));
  }
#pragma unroll
  for (int c = 0; c < 16; ++c) sm[spad(i + TB * c + PB * q)] = v[c];
  sync();
  r3_butterfly_third<P, true>(v, sm, t, sync);
}

}  // namespace holo
