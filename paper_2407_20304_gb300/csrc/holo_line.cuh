// Line<P>: the transform of one line of length P, for every supported length.
//
// P = 2^k (16 .. 4096).  A line is held by T = P/E threads with E values in registers (E = 32
// from P = 512, 16 below): thread t, register c holds element t + T c.  With n = t + T c and
// k = k1 + E k',
//   X[k1 + E k'] = sum_t W_T^{t k'} W_P^{t k1} ( sum_c x[t + T c] W_E^{c k1} ).
// Stage 1 is a DFT of length E in each thread's registers (twiddles are constants); an exchange
// through shared memory hands row k1 to the threads t = k1 mod E; stage 2 is a DFT over the row,
// its input scaled by w^t.  For P <= 1024 the row has T <= E values and that is all.  For 2048
// and 4096 the row's T = 32 R values take a DFT of length 32 per thread and, after a second
// exchange among the R = 2 or 4 threads of the row (each writes the entries it has read), 32/R
// DFTs of length R, again on scaled inputs (t = u + R w: base W_1024^{k1} over w, then
// W_P^{k1 + 32 k2} over u).  The scaling costs no pass of its own: in a radix-2
// decimation-in-time DFT of a_t w^t the butterfly a +- z b of a level has z = w^{2^l} W^j instead
// of W^j.  Register c of thread t then holds frequency t + T c, the layout the transform started
// from, so a multiplier in frequency and a second transform follow directly.
//
// Butterflies: s = a + z b in four FMAs, and a - z b = 2 a - s in one packed FMA (two lanes): 6
// operations where a complex multiplication and two additions take 8.  The values w^{2^l} and
// W_P^t come from a table built in FP64; every other twiddle is one product of an entry with a
// constant, and a factor -i is a swap.
//
// What bounds it: the FP32 pipe (128 lanes per clock and SM, packed or not: 63 packed FMAs per
// clock measured) at about 36 operations per element, and shared memory (128 bytes per clock) at
// 32 bytes per element and exchange; radix-16 stages with 16 values per thread cost 45
// operations (a power tree of 14 products per twiddled stage), two exchanges at P = 1024 and
// 2048 and one at 256.  Alone on the chip (transform, chirp, inverse, no global memory; ns per
// transform, radix-16 engine -> this): P = 4096 7.2 -> 5.8, 2048 (column form) 5.8 -> 2.8, 1024
// 2.5 -> 1.05.  Why not more values per thread: 64 need one exchange only, but 255 registers (8
// warps per SM) and 32 KB of code per transform.  An SM partition holds 32 KB of instructions;
// up to 128 KB a warp gets one per 2.8 clocks, above one per 6 (measured on straight-line FMAs),
// which made the column pass at P = 4096 three times slower.  For the same reason the inverse is
// the conjugate of the forward transform of the conjugate, and forward and inverse run as two
// turns of a loop over one copy of the code (17 KB).
//
// P = 3 * 2^k, 48 .. 768: the same two stages with E = 24 up to 192 and E = 48 above (stage 1 is 3 x 8
// or 3 x 16 without twiddles).  At P <= 192 all the work is on the chip in one wave, and 48 values in
// half the threads only made it longer (96^2 on 96^2, 2 x 4 planes: pass A 19.6 -> 10 us, B 26.3 ->
// 12.5 us; 98^2 on 192^2, 24 x 3 planes, A and C 33.2 -> 20.0 us).  384 and 768 need rows of 16 values,
// which 24 values do not give a whole number of.
// 1536 and 3072 would need 48 rows over 32 or 64 threads: the radix-3 step and the 16-value engine
// of holo_fft.cuh (E = 16, T = P/16).
//
// ZIN: the inputs outside the middle half P/4 .. 3P/4, i.e. the registers c outside E/4 .. 3E/4,
// are zero and not read.  For E = 2^k stage 1's first two levels become 8 additions per 4 values,
// with the same results as zeros passed to the full form.
//
// Synchronisation: every thread of a line calls fft the same number of times; Sync is a barrier
// over (at least) the threads of the line.  fft starts with a barrier, so the line's buffer may
// still be read by the line's threads when it is called, and the same holds when it returns:
// any other use of the buffer needs a barrier before it.

#pragma once

#include <type_traits>
#include <utility>

#include "holo_fft.cuh"

#define HOLO_INLINE __attribute__((always_inline))

namespace holo {

// ------------------------------------------------------------------ constants

// W_n^j = exp(-2 pi i j / n) for 0 <= j <= n/2 as compile-time constants: Taylor series in FP64
// (28 terms at |x| <= pi: below 1e-16)
constexpr double unit_angle(int j, int n) { return 2.0 * 3.14159265358979323846 * j / n; }
constexpr double unit_cos(int j, int n) {
  const double x = unit_angle(j, n);
  double t = 1.0, s = 1.0;
  for (int k = 1; k < 15; ++k) {
    t *= -x * x / ((2 * k - 1) * (2 * k));
    s += t;
  }
  return s;
}
constexpr double unit_sin(int j, int n) {
  const double x = unit_angle(j, n);
  double t = x, s = x;
  for (int k = 1; k < 15; ++k) {
    t *= -x * x / ((2 * k) * (2 * k + 1));
    s += t;
  }
  return s;
}
template <int J, int N>
struct UnitRoot {
  static constexpr float x = (float)unit_cos(J, N), y = (float)-unit_sin(J, N);
};

// f(0), f(1), ..., f(N - 1) with the index as a compile-time constant (the register arrays below
// are indexed by constants only; unrolled run-time loops give the same code but cost the compiler
// minutes)
template <int I>
struct Idx {
  static constexpr int value = I;
};
template <class F, int... I>
__device__ __forceinline__ void static_for_seq(F&& f, std::integer_sequence<int, I...>) {
  (f(Idx<I>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void static_for(F&& f) {
  static_for_seq(f, std::make_integer_sequence<int, N>{});
}
__host__ __device__ constexpr int bit_reverse(int i, int bits) {
  int r = 0;
  for (int b = 0; b < bits; ++b) r |= ((i >> b) & 1) << (bits - 1 - b);
  return r;
}

// ------------------------------------------------------------------ butterflies

// 2 a - s, both components in one instruction
__device__ __forceinline__ float2 twice_minus(float2 a, float2 s) {
#if !defined(HOLO_SCALAR_COMPLEX)
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(d)
      : "l"(pk(a)), "l"(pk(make_float2(2.f, 2.f))), "l"(pk(make_float2(-s.x, -s.y))));
  return upk(d);
#else
  return make_float2(fmaf(2.f, a.x, -s.x), fmaf(2.f, a.y, -s.y));
#endif
}
// a + z b
__device__ __forceinline__ float2 add_mul(float2 a, float2 b, float zx, float zy) {
  return make_float2(fmaf(zx, b.x, fmaf(-zy, b.y, a.x)), fmaf(zx, b.y, fmaf(zy, b.x, a.y)));
}
// (a, b) <- (a + z b, a - z b)
__device__ __forceinline__ void bfly(float2& a, float2& b, float zx, float zy) {
  const float2 s = add_mul(a, b, zx, zy);
  b = twice_minus(a, s);
  a = s;
}
__device__ __forceinline__ void bfly_one(float2& a, float2& b) {
  const float2 s = cadd(a, b);
  b = csub(a, b);
  a = s;
}
// z = -i
__device__ __forceinline__ void bfly_i(float2& a, float2& b) {
  const float2 s = make_float2(a.x + b.y, a.y - b.x);
  b = make_float2(a.x - b.y, a.y + b.x);
  a = s;
}

// DFT of N values in registers, constants only.  Natural order in; X[k] is left in
// v[bit_reverse(k)].  Levels M, 2M, ... of the radix-2 decimation in time:
template <int N, int M, int END>
__device__ __forceinline__ void dft_const_levels(float2* v) {
  if constexpr (M < END) {
    constexpr int B = ilog2c(N);
    // butterfly i of the level: pair j of group g, elements g + j and M further on
    static_for<N / 2>([&](auto ic) HOLO_INLINE {
      constexpr int i = decltype(ic)::value, j = i / (N / (2 * M)), g = i % (N / (2 * M)) * 2 * M;
      constexpr int ia = bit_reverse(g + j, B), ib = bit_reverse(g + j + M, B);
      if constexpr (j == 0)
        bfly_one(v[ia], v[ib]);
      else if constexpr (2 * j == M)
        bfly_i(v[ia], v[ib]);
      else
        bfly(v[ia], v[ib], UnitRoot<j, 2 * M>::x, UnitRoot<j, 2 * M>::y);
    });
    dft_const_levels<N, 2 * M, END>(v);
  }
}
// ... and the first two levels on values that are zero outside N/4 .. 3N/4: on (0, x1, x2, 0)
// x1 + x2, -i x1 - x2, x2 - x1, i x1 - x2.
template <int N>
__device__ __forceinline__ void dft_const_zin(float2* v) {
  static_for<N / 4>([&](auto ic) HOLO_INLINE {
    constexpr int c = decltype(ic)::value;
    const float2 x1 = v[c + N / 4], x2 = v[c + N / 2];
    v[c] = cadd(x1, x2);
    v[c + N / 4] = csub(x2, x1);
    v[c + N / 2] = make_float2(x1.y - x2.x, -x1.x - x2.y);
    v[c + 3 * N / 4] = make_float2(-x1.y - x2.x, x1.x - x2.y);
  });
}

// DFT of length 3 B (B = 8 or 16) as 3 x B without twiddles (Good-Thomas: element (B a + 3 b) mod
// 3 B, output k with k mod 3 and k mod B the two indices); X[k] is left in v[dft3_at<B>(k)].
template <int B>
__host__ __device__ constexpr int dft3_at(int k) {
  return (B * (k % 3) + 3 * bit_reverse(k % B, ilog2c(B))) % (3 * B);
}
template <int B>
__device__ __forceinline__ void dft3(float2* v) {
  static_for<3>([&](auto ac) HOLO_INLINE {
    constexpr int a = decltype(ac)::value;
    float2 y[B];
    static_for<B>([&](auto bc) HOLO_INLINE {
      constexpr int b = decltype(bc)::value;
      y[b] = v[(B * a + 3 * b) % (3 * B)];
    });
    dft_const_levels<B, 1, B>(y);
    static_for<B>([&](auto bc) HOLO_INLINE {
      constexpr int b = decltype(bc)::value;
      v[(B * a + 3 * b) % (3 * B)] = y[b];
    });
  });
  const float h = 0.86602540378443865f;  // sqrt(3)/2
  static_for<B>([&](auto bc) HOLO_INLINE {
    constexpr int b = decltype(bc)::value;
    float2 &x0 = v[(3 * b) % (3 * B)], &x1 = v[(B + 3 * b) % (3 * B)],
           &x2 = v[(2 * B + 3 * b) % (3 * B)];
    const float2 su = cadd(x1, x2), df = csub(x1, x2);
    const float2 m = make_float2(fmaf(-0.5f, su.x, x0.x), fmaf(-0.5f, su.y, x0.y));
    x0 = cadd(x0, su);
    x1 = make_float2(fmaf(h, df.y, m.x), fmaf(-h, df.x, m.y));
    x2 = make_float2(fmaf(-h, df.y, m.x), fmaf(h, df.x, m.y));
  });
}

// DFT of the T values v[S i] w^i (natural order in, X[k] in v[S bit_reverse(k)]), levels M, 2M,
// ...; tw(l) gives w^{2^l}.
template <int T, int S, int M, class Tw>
__device__ __forceinline__ void dft_scaled_levels(float2* v, Tw tw) {
  if constexpr (M < T) {
    constexpr int B = ilog2c(T);
    const float2 w = tw(ilog2c(T / (2 * M)));
    static_for<(M > 1 ? M / 2 : 1)>([&](auto jc) HOLO_INLINE {
      constexpr int j = decltype(jc)::value;
      float2 z = w;
      if constexpr (j > 0)
        z = cmul(w, make_float2(UnitRoot<j, 2 * M>::x, UnitRoot<j, 2 * M>::y));
      static_for<T / (2 * M)>([&](auto gc) HOLO_INLINE {
        constexpr int g = decltype(gc)::value * 2 * M;
        bfly(v[S * bit_reverse(g + j, B)], v[S * bit_reverse(g + j + M, B)], z.x, z.y);
        // the twiddle M/2 further on is -i z
        if constexpr (M > 1)
          bfly(v[S * bit_reverse(g + j + M / 2, B)], v[S * bit_reverse(g + j + M / 2 + M, B)], z.y,
               -z.x);
      });
    });
    dft_scaled_levels<T, S, 2 * M>(v, tw);
  }
}

// ------------------------------------------------------------------ lines

template <int P_, bool R3_ = (P_ % 3 == 0 && P_ > 768)>
struct Line;

template <int P_>
struct Line<P_, false> {
  static constexpr int P = P_;
  static constexpr bool R3 = false;
  static constexpr bool M3 = P % 3 == 0;            // P = 3 * 2^k: E = 48, up to 192 24
  static_assert(is_pow2c(M3 ? P / 3 : P) && P >= 16 && P <= 4096, "line length");
  static constexpr int E = M3 ? (P > 192 ? 48 : 24) : (P >= 512 ? 32 : 16);
  // where stage 1 leaves output k
  __host__ __device__ static constexpr int at(int k) {
    return M3 ? dft3_at<E / 3>(k) : bit_reverse(k, ilog2c(E));
  }
  static constexpr int T = P / E;
  static constexpr int R = T > E ? T / E : 1;      // radix of the third stage
  static constexpr int NB = R > 1 ? 1 : E / T;     // second-stage DFTs per thread
  static constexpr int T2 = R > 1 ? E : T;         // their length
  // Exchange rows of T values.  Two stages: 16-byte reads of one row per lane, row pitch 4 mod
  // 32 words.  Three stages: 8-byte accesses of one row per lane, odd row pitch.  Either way
  // every access of a warp is free of bank conflicts where a line has 16 threads or more; with
  // fewer, the writes of a block's many columns take two passes.
  static constexpr int RS = R > 1 ? T + 1 : T + 2;
  static constexpr int SMEM = T > 1 ? E * RS : P;  // float2 entries of a line's buffer (>= P)
  static constexpr int B2 = ilog2c(T2);
  // twiddles: [l][k1] = W_{E T2}^{k1 2^l}, l < log2 T2, then (three stages) [t] = W_P^t
  static constexpr int TAB = E * B2 + (R > 1 ? T : 0);
  static constexpr int TABS = TAB;                 // entries kept in shared memory
  __host__ __device__ static constexpr int pos(int t, int c) { return t + T * c; }
  __host__ __device__ static constexpr int fpos(int t, int c) { return t + T * c; }

  __device__ __forceinline__ static void load_table(float2* sm, const float2* __restrict__ g) {
    for (int i = threadIdx.x; i < TAB; i += blockDim.x) sm[i] = g[i];
  }

  // Forward transform, unscaled.  zin (uniform over the line; only where ZIN): the inputs outside
  // the middle half P/4 .. 3P/4 are zero and not read.
  template <bool ZIN, class Sync>
  __device__ __forceinline__ static void fft(float2 (&v)[E], float2* __restrict__ sm,
                                             const float2* __restrict__ tab, int t, Sync sync,
                                             bool zin) {
    if constexpr (T > 1) sync();
    if constexpr (M3) {
      if (ZIN && zin) {
#pragma unroll
        for (int c = 0; c < E; ++c)
          if (c < E / 4 || c >= 3 * E / 4) v[c] = make_float2(0.f, 0.f);
      }
      dft3<E / 3>(v);
    } else {
      if (ZIN && zin)
        dft_const_zin<E>(v);
      else
        dft_const_levels<E, 1, 4>(v);
      dft_const_levels<E, 4, E>(v);
    }
    if constexpr (T > 1) {
      static_for<E>([&](auto ic) HOLO_INLINE {
        constexpr int k = decltype(ic)::value, r = at(k);
        sm[k * RS + t] = v[r];
      });
      sync();
    }
    float2 x[E];
    if constexpr (R == 1) {
      if constexpr (T > 1) {
        static_for<E / 2>([&](auto ic) HOLO_INLINE {
          constexpr int i = decltype(ic)::value, g = i / (T / 2), c = i % (T / 2);
          const float4 q = reinterpret_cast<const float4*>(sm + (t + T * g) * RS)[c];
          v[g + NB * (2 * c)] = make_float2(q.x, q.y);
          v[g + NB * (2 * c + 1)] = make_float2(q.z, q.w);
        });
        static_for<NB>([&](auto ic) HOLO_INLINE {
          constexpr int g = decltype(ic)::value;
          const float2* w = tab + t + T * g;
          dft_scaled_levels<T, NB, 1>(v + g, [&](int l) HOLO_INLINE { return w[E * l]; });
        });
      }
      // to natural order (a renaming of registers)
      static_for<E>([&](auto ic) HOLO_INLINE {
        constexpr int c = decltype(ic)::value;
        constexpr int r = T > 1 ? c % NB + NB * bit_reverse(c / NB, B2) : at(c);
        x[c] = v[r];
      });
    } else {
      // thread t = k1 + 32 u: the values u + R w of row k1, then DFTs of length R over u
      float2* row = sm + (t % E) * RS;
      float2* own = row + t / E;
      static_for<E>([&](auto ic) HOLO_INLINE {
        constexpr int w = decltype(ic)::value;
        v[w] = own[R * w];
      });
      const float2* w2 = tab + t % E;
      dft_scaled_levels<E, 1, 1>(v, [&](int l) HOLO_INLINE { return w2[E * l]; });
      // (the entries a thread writes are those it has read)
      static_for<E>([&](auto ic) HOLO_INLINE {
        constexpr int k = decltype(ic)::value, r = at(k);
        own[R * k] = v[r];
      });
      sync();
      const float2* col = row + t / E * R;
      const float2 w3 = tab[E * B2 + t];
      static_for<E / R>([&](auto ic) HOLO_INLINE {
        constexpr int i = decltype(ic)::value;
        float2 y[R];
#pragma unroll
        for (int u = 0; u < R; ++u) y[u] = col[i * R * R + u];
        // w = W_P^{t + T i} = W_P^t W_32^i
        float2 w = w3;
        if constexpr (i > 0) w = cmul(w3, make_float2(UnitRoot<i, E>::x, UnitRoot<i, E>::y));
        const float2 ww = make_float2(fmaf(w.x, w.x, -w.y * w.y), 2.f * w.x * w.y);
        dft_scaled_levels<R, 1, 1>(y, [&](int l) HOLO_INLINE { return l ? ww : w; });
#pragma unroll
        for (int k = 0; k < R; ++k) x[i + E / R * k] = y[bit_reverse(k, ilog2c(R))];
      });
    }
#pragma unroll
    for (int c = 0; c < E; ++c) v[c] = x[c];
  }
};

template <int P_>
struct Line<P_, true> {
  static constexpr int P = P_;
  static constexpr bool R3 = true, M3 = true;
  using F = Fft<P>;
  static constexpr int E = 16, T = F::T, SMEM = F::SMEM;
  static constexpr int TAB = F::TW, TABS = F::ROOTS;
  __host__ __device__ static constexpr int pos(int t, int c) { return F::pos(t, c); }
  __host__ __device__ static constexpr int fpos(int t, int c) { return F::fpos(t, c); }

  __device__ __forceinline__ static void load_table(float2* sm, const float2* __restrict__ g) {
    load_roots<P>(sm, g);
  }
};

// D = inverse transform of (multiplier x forward transform) of one line: mul(v) multiplies every
// register c by the multiplier at frequency fpos(t, c).  P = 2^k: the inverse is the conjugate of
// the forward transform of the conjugate, so one copy of the transform's code runs twice (it
// shall stay in the 32 KB instruction cache of an SM partition).
template <class L, bool ZIN, class Sync, class Mul>
__device__ __forceinline__ void line_dstep(float2 (&v)[L::E], float2* sm, const float2* tab, int t,
                                           Sync sync, bool zin, Mul mul) {
  if constexpr (L::R3) {
    sync();
    fft_fwd_with<L::P>(v, sm, TwRoots{tab}, t, sync);
    mul(v);
    sync();
    fft_inv_with<L::P>(v, sm, TwRoots{tab}, t, sync);
  } else {
#pragma unroll 1
    for (int turn = 0;; ++turn) {
      L::template fft<ZIN>(v, sm, tab, t, sync, zin && turn == 0);
      if (turn) break;
      mul(v);
#pragma unroll
      for (int c = 0; c < L::E; ++c) v[c] = cconj(v[c]);
    }
#pragma unroll
    for (int c = 0; c < L::E; ++c) v[c] = cconj(v[c]);
  }
}

}  // namespace holo
