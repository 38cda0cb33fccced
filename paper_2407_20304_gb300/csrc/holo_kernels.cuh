// Kernels of the per-plane hot path, templated on the line length P.
//
// Forward model of one (k, j) plane (Eq. fwd_model_cone3 with the shifts of Eq. min1):
//   u_kj = C D_{zhat_j}( p_j * R_kj psi_k ),  zhat_j = zeta_j / m~_j^2,  p_j = D_{omega_j} q.
// The resample is affine, R psi = ext + w with w = R0(psi - ext) supported on a box of
// about n/m~_j pixels per side, so by linearity
//   u_kj = ext * C D_{zhat_j}(p_j) + C D_{zhat_j}(p_j * w_kj) = ext * b + C D_{zhat_j}(p_j * w_kj)
// with b = C D_{zeta_0}(q) the same for every plane (Theorem t3: zhat_j + omega_j = zeta_0).
// Only the box rows need the row transforms, and only box columns of the adjoint field
// are needed for grad_psi and for the w-part of grad_q.  Per plane:
//   pass A (rows of the box): x = p_j * w, row FFT, chirp, row IFFT, keep the n
//           detector columns -> Y[box rows][n]
//   pass B (detector columns): column FFT, chirp, IFFT, keep the n detector rows,
//           u = ext b + (.), residual r = u - a u/|u| (Eq. gradpsi), loss partial,
//           S = sum r kept for the ext-part of grad_q, then the adjoint column transform
//           on C* r, keep box rows -> conj(V) (in place of Y)
//   pass C (rows of the box): adjoint row transform -> v on the box columns;
//           z = conj(p_j) v, x-transpose of the bilinear resample -> h[box rows][n]
//           (in place of V); conj(w) v -> per-plane buffer for grad_q
//   pass D (psi rows, line-length independent): y-transpose, sum over j, times 2.
//
// All passes run persistent blocks (a grid that fills the GPU once) that load the FFT
// twiddles into shared memory once and then walk a flat list of work items.
//
// Every propagation D = inverse . chirp . forward of a line is one line_dstep; its adjoint is
// conj D conj, the chirp being even in frequency.
//
// Probe shifts s_kj (Eq. min1) run the passes' general forms with ramps.  The shift is moved
// off the probe, u_kj = C S_s D_{zhat_j}(p_j * R'_kj psi_k) with R' the resample at object
// shift t - m~_j s, and S_s D_{zhat_j} is one separable Fourier multiplier: the chirp times
// the per-plane phase ramps exp(-2 pi i k s / P) of each axis (ramp_x in the row passes,
// ramp_y in the column pass; at -f for the conjugated adjoints).  The ext-part of the field is then
// shifted per plane as well, so the box is the whole P x P grid, w holds R' psi itself
// (ext added back in pass A) and pass B runs with ext = 0 (no b term, T = w_ref r_ref).

#pragma once

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "holo_internal.h"
#include "holo_line.cuh"
#include "holo_split.h"
#include "holo_tma.cuh"
#include "holo_tmem.cuh"

namespace holo {

// Shared memory of every line kernel: the twiddle table, the half chirp table (P/2 + 1
// entries) and the exchange lines.
template <int P>
struct SmemHead {
  static constexpr int TAB = (Line<P>::TABS + 1) & ~1;
  static constexpr int CHIRP = (P / 2 + 2) & ~1;
  static constexpr int WORDS = TAB + CHIRP;
};

// Row passes.  The threads that exchange with one another form a unit: one line of T >= 32
// threads (four warps at P = 4096, two at 2048, one at 1024) or a warp with 32/T lines below; for
// P = 1536 and 3072 (whose engine holds block barriers) the whole block.  Units of a block share
// the twiddle and chirp tables and are otherwise independent: each has its own barrier, so one
// unit's arithmetic fills the time another spends on its exchange and its loads.  What bounds them
// is the latency of the L2 loads around the transforms at 16 warps per SM (P = 4096: FP32 pipe 45 %
// and 38 %, shared memory 60 % and 55 % busy in A and C).  393k lines of the 2048^2 chunk: pass A
// 9.8 -> 7.9 ms, C 9.4 -> 8.4 ms; 512^2, 180 x 4 planes: about 2.1 -> 1.1 ms each.  Units per block
// (2 at P = 4096, else 4): 4 / 2 / 1 at 4096 took 8.72 / 8.41 / 8.50 ms in pass C, 4 / 2 / 8 at 2048
// 2.76 / 2.82 / 2.91 ms in pass A.
__host__ __device__ constexpr int r3_row_lines(int T) { return T > 128 ? 1 : 256 / T; }

template <int P>
struct RowCfg {
  using L = Line<P>;
  static constexpr int T = L::T;
  static constexpr int GU = L::R3 ? r3_row_lines(T) : (T >= 32 ? 1 : 32 / T);  // lines per unit
  static constexpr int U = GU * T;                                            // threads per unit
  static constexpr int NU = L::R3 ? 1 : (P == 4096 ? 2 : 4);
  static constexpr int NT = NU * U;
  static constexpr int G = NU * GU;  // lines per block
  // line pitch: lines of one half warp on different banks (T < 16 puts several lines in it)
  static constexpr int LS =
      L::SMEM + (L::R3 ? 0 : (T >= 16 ? 0 : (T == 8 ? 8 : (T == 4 ? 4 : 2))));
  static constexpr size_t SMEM_BYTES = (size_t)(SmemHead<P>::WORDS + G * LS) * sizeof(float2);
  static constexpr int MINB = L::R3 ? 2 : (P >= 2048 ? 2 : (L::E == 48 ? 3 : (L::M3 || P >= 512 ? 4 : 6)));
};

// Column passes: C adjacent columns interleaved in the lanes, so that one access covers the C
// columns of consecutive rows; a block is 128 threads, from P = 2048 256 (P = 4096 with four
// columns and 512 threads: pass B 18.6 ms against 17.4; P = 1536, 3072: as their T allows).
template <int P>
struct ColCfg {
  using L = Line<P>;
  static constexpr int T = L::T;
  static constexpr int C =
      L::R3 ? (T >= 192 ? 2 : 4) : (P >= 2048 ? 256 : 128) / T;
  static constexpr int NT = C * T;
  // line pitch: the C lines' runs in one 128-byte bank row side by side
  static constexpr int EXTRA =
      L::R3 ? (P == 1536 ? 3 : 0)
            : (C == 2 ? 8 : (C == 4 ? 4 : 2));
  static constexpr int LS = L::SMEM + EXTRA;
  static constexpr size_t SMEM_BYTES = (size_t)(SmemHead<P>::WORDS + C * LS) * sizeof(float2);
};

// Column D-steps (no per-thread state besides the line): at P = 4096 four columns and 512 threads,
// so that every access covers whole 32-byte sectors (a 4096^2 propagation 262 -> 214 us, with the
// row kernel's prefetch).
template <int P>
struct DColCfg {
  using L = Line<P>;
  static constexpr int C = P == 4096 ? 4 : ColCfg<P>::C;
  static constexpr int NT = C * L::T;
  static constexpr int LS = P == 4096 ? L::SMEM + 4 : ColCfg<P>::LS;
  static constexpr size_t SMEM_BYTES = (size_t)(SmemHead<P>::WORDS + C * LS) * sizeof(float2);
};

// The barrier of a unit of the row passes.
template <int P>
struct UnitSync {
  int unit;
  __device__ __forceinline__ void operator()() const {
    using R = RowCfg<P>;
    if constexpr (R::U == R::NT)
      __syncthreads();
    else if constexpr (R::U == 32)
      __syncwarp();
    else
      asm volatile("bar.sync %0, %1;" ::"r"(unit + 1), "n"(R::U) : "memory");
  }
};

// Sum of per-thread FP64 values over the block; result valid in thread 0.
__device__ __forceinline__ double block_sum_f64(double v, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    for (int i = 0; i < nw; ++i) s += red[i];
  }
  return s;
}

// Builds with HOLO_BOUNDS_CHECK check their table-driven indices on the device: a bad entry
// sets bit 2 of the problem's error word (HOLO_ERR_BOUNDS at the next loss read) and the access
// is skipped; nothing traps.  Other builds compile the checks away.
#if defined(HOLO_BOUNDS_CHECK)
constexpr bool kBoundsCheck = true;
#else
constexpr bool kBoundsCheck = false;
#endif

__device__ __forceinline__ void flag_bounds(unsigned long long* err) { atomicOr(err, 2ull); }

// A plane's box inside the P x P grid and inside the workspace strides of its problem.
__device__ __forceinline__ bool plane_box_ok(const PassArgs& a, const PlaneDesc& d, int P) {
  return d.by0 >= 0 && d.bys >= 0 && d.by0 + d.bys <= P && d.bx0 >= 0 && d.bxs >= 0 &&
         d.bx0 + d.bxs <= P && d.bys <= a.tap_stride && d.bxs <= a.tap_stride &&
         (long long)d.bys * a.n <= a.ystride && (long long)d.bys * d.bxs <= a.gkstride;
}

// A row-pass line (plane gp, box row i): the plane among the chunk's, the row inside its box.
__device__ __forceinline__ bool line_ok(const PassArgs& a, int gp, int i, int P) {
  const int p_lo = a.k0 * a.J;
  if (gp < p_lo || gp >= p_lo + a.nk * a.J) return false;
  const PlaneDesc d = a.planes[gp];
  return i >= 0 && i < d.bys && plane_box_ok(a, d, P);
}

// Chirp exp(-i pi lambda z f^2)/P is even in the signed frequency, so a table of the
// P/2 + 1 non-negative frequencies suffices: entry f for f <= P/2, entry P - f above.  For
// P = 2^k thread t holds the frequencies t + T c: entry t + T c for c < E/2 and entry
// (T - t) + T (E - 1 - c) above (the P/2 entry included), so every lookup is one shared-memory
// load at a constant offset from one of two per-thread addresses.
template <int P>
struct ChirpAt {
  using L = Line<P>;
  const float2* tab;
  int t;
  __device__ __forceinline__ ChirpAt(const float2* tb, int tt) : tab(tb), t(tt) {}
  __host__ __device__ static constexpr int at(int t, int c) {
    if constexpr (L::R3) {
      const int f = L::fpos(t, c);
      return f <= P / 2 ? f : P - f;
    } else {
      return c < L::E / 2 ? t + L::T * c : L::T - t + L::T * (L::E - 1 - c);
    }
  }
  __device__ __forceinline__ float2 operator()(int c) const { return tab[at(t, c)]; }
};

// Copy the half chirp table of one distance into shared memory (block-wide).
template <int P>
__device__ __forceinline__ void load_chirp_half(float2* dst, const float2* __restrict__ src) {
  for (int i = threadIdx.x; i <= P / 2; i += blockDim.x) dst[i] = src[i];
}

// ------------------------------------------------------------------ generic D-step

// One "FFT -> chirp -> inverse FFT" per line, lines = rows (COLS = false) or columns, of every
// source in turn (block-steps of G lines that never span two sources).  One launch for the J
// propagations of a probe, or for the sources of its gradient: what they cost at P <= 1024 is
// launches and half-empty grids (set_probe at P = 256, 4 distances: 9 launches, 55 us).
template <int P, bool COLS>
__global__ void __launch_bounds__(COLS ? DColCfg<P>::NT : RowCfg<P>::NT)
k_line_dstep(const __grid_constant__ LineArgs args, const float2* __restrict__ gtw) {
  using L = Line<P>;
  using H = SmemHead<P>;
  using R = RowCfg<P>;
  constexpr int G = COLS ? DColCfg<P>::C : R::G;
  constexpr int LS = COLS ? DColCfg<P>::LS : R::LS;
  extern __shared__ __align__(16) float2 smem[];
  float2* chs = smem + H::TAB;
  const int g = COLS ? (int)(threadIdx.x % G) : (int)(threadIdx.x / L::T);
  const int t = COLS ? (int)(threadIdx.x / G) : (int)(threadIdx.x % L::T);
  float2* sm = smem + H::WORDS + g * LS;
  L::load_table(smem, gtw);
  const ChirpAt<P> cat(chs, t);
  auto run = [&](auto sync) HOLO_INLINE {
    int s = 0, cur = -1;
    for (int step = blockIdx.x; step < args.step[args.S]; step += gridDim.x) {
      while (step >= args.step[s + 1]) ++s;
      const LineSource& a = args.src[s];
      if (s != cur) {
        __syncthreads();
        load_chirp_half<P>(chs, a.chirp);
        __syncthreads();
        cur = s;
      }
      const float sg = a.conj_chirp ? -1.f : 1.f;
      const int line = (step - args.step[s]) * G + g;
      // a thread group's next row (same source) goes to L2 now
      if (!COLS && t == 0 && line + (int)gridDim.x * G < a.nlines)
        l2_prefetch_bulk(a.in + (long long)(line + (int)gridDim.x * G) * a.in_line_stride,
                         (uint32_t)(a.in_len * sizeof(float2)));
      const bool valid = line < a.nlines;
      const float2* in = a.in + (long long)line * a.in_line_stride;
      float2 v[L::E];
#pragma unroll
      for (int c = 0; c < L::E; ++c) {
        const int rel = L::pos(t, c) - a.in_lo;
        v[c] = (valid && (unsigned)rel < (unsigned)a.in_len) ? in[(long long)rel * a.in_step]
                                                             : make_float2(0.f, 0.f);
      }
      line_dstep<L, false>(v, sm, smem, t, sync, false, [&](float2 (&x)[L::E]) HOLO_INLINE {
#pragma unroll
        for (int c = 0; c < L::E; ++c) {
          float2 ch = cat(c);
          ch.y *= sg;
          x[c] = cmul(x[c], ch);
        }
      });
      float2* out = a.out + (long long)line * a.out_line_stride;
#pragma unroll
      for (int c = 0; c < L::E; ++c) {
        const int rel = L::pos(t, c) - a.out_lo;
        if (valid && (unsigned)rel < (unsigned)a.out_len) out[(long long)rel * a.out_step] = v[c];
      }
    }
  };
  if constexpr (COLS)
    run(SyncBlock{});
  else
    run(UnitSync<P>{(int)(threadIdx.x / R::U)});
}

// The column stage of sum_s D_s(x_s): the rows of every source were propagated already (row
// FFT, chirp, inverse), so D_s = IFFT_y chirp_s FFT_y on columns and the sum needs one inverse
// per column: acc = sum_s chirp_s FFT_y(col_s), out (+)= alpha IFFT_y(acc).  Blocks own C
// columns at a time, as k_line_dstep's column form.  P = 2^k: turn s < S transforms source s,
// turn S the conjugate of the sum (one copy of the transform's code, as line_dstep).
template <int P>
__global__ void __launch_bounds__(DColCfg<P>::NT)
k_cols_sum(const __grid_constant__ SumArgs a, const float2* __restrict__ gtw) {
  using L = Line<P>;
  using H = SmemHead<P>;
  constexpr int G = DColCfg<P>::C, LS = DColCfg<P>::LS, E = L::E;
  extern __shared__ __align__(16) float2 smem[];
  const int g = threadIdx.x % G, t = threadIdx.x / G;
  float2* sm = smem + H::TAB + g * LS;
  L::load_table(smem, gtw);
  __syncthreads();
  const SyncBlock sync;
  for (int base = blockIdx.x * G; base < P; base += gridDim.x * G) {
    const int col = base + g;
    const bool valid = col < P;
    float2 acc[E], v[E];
#pragma unroll
    for (int c = 0; c < E; ++c) acc[c] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int s = 0;; ++s) {
      if (s < a.S) {
        const float2* in = a.in[s] + col;
        const int r_lo = a.r_lo[s], rows = a.rows[s];
#pragma unroll
        for (int c = 0; c < E; ++c) {
          const int rel = L::pos(t, c) - r_lo;
          v[c] = (valid && (unsigned)rel < (unsigned)rows) ? in[(long long)rel * P]
                                                           : make_float2(0.f, 0.f);
        }
      } else {
#pragma unroll
        for (int c = 0; c < E; ++c) v[c] = L::R3 ? acc[c] : cconj(acc[c]);
      }
      if constexpr (L::R3) {
        sync();
        if (s == a.S) {
          fft_inv_with<P>(v, sm, TwRoots{smem}, t, sync);
          break;
        }
        fft_fwd_with<P>(v, sm, TwRoots{smem}, t, sync);
      } else {
        L::template fft<false>(v, sm, smem, t, sync, false);
        if (s == a.S) {
#pragma unroll
          for (int c = 0; c < E; ++c) v[c] = cconj(v[c]);
          break;
        }
      }
      const float2* chg = a.chirp[s];
      const float sg = a.conj_chirp ? -1.f : 1.f;
#pragma unroll
      for (int c = 0; c < E; ++c) {
        float2 ch = __ldg(chg + L::fpos(t, c));
        ch.y *= sg;
        acc[c] = cadd(acc[c], cmul(v[c], ch));
      }
    }
    if (valid) {
#pragma unroll
      for (int c = 0; c < E; ++c) {
        float2* o = a.out + (long long)L::pos(t, c) * P + col;
        float2 r = cscale(v[c], a.alpha);
        if (a.accumulate) r = cadd(r, *o);
        *o = r;
      }
    }
  }
}

// ------------------------------------------------------------------ row passes

// The lines of a chunk run distance-major (distance, angle, box row), so a block's chirp table
// changes J times at most; `s` numbers block-steps of G lines that never span two distances.
// row_item locates step s: its distance, the first line of the calling unit and the end of the
// distance's lines (positions relative to the chunk's lines of that distance).
struct RowItem {
  int j, li, cnt;
};
template <int P>
__device__ __forceinline__ RowItem row_item(const PassArgs& a, int s, int unit) {
  int j = 0;
  while (j + 1 < a.J && s >= a.seg_step[j + 1]) ++j;
  return {j, (s - a.seg_step[j]) * RowCfg<P>::G + unit * RowCfg<P>::GU, a.seg_cnt[j]};
}

// Chirp table of distance j of problem `key` resident in shared memory: loaded unless the
// block's resident table already is that one (block-uniform arguments).
template <int P>
__device__ __forceinline__ void ensure_chirp_key(float2* chs, const float2* __restrict__ tables,
                                                 int j, int key, int& cur) {
  if (key != cur) {
    __syncthreads();
    load_chirp_half<P>(chs, tables + (long long)j * P);
    __syncthreads();
    cur = key;
  }
}

// n = P/2 (P = 2^k >= 64, 192, 384, 768): the crop rows and columns P/4 .. 3P/4 are the registers
// E/4 .. 3E/4 of every thread and the pass-B column groups divide n (HALF forms).
template <int P>
__host__ __device__ constexpr bool half_form_ok() {
  return !Line<P>::R3 && P / 2 % ColCfg<P>::C == 0;
}
// c in the middle half of a thread's registers
template <int P>
__host__ __device__ constexpr bool mid_reg(int c) {
  return c >= Line<P>::E / 4 && c < 3 * Line<P>::E / 4;
}

// One block-step of pass A for the calling unit.  `next` is the block's next step of the same
// problem (its lines are prefetched into L2), or -1.  The resident chirp table is identified by
// pkey * 16 + distance (pkey: the problem's index in a batch, 0 for a single problem).
template <int P, bool HALF>
__device__ __forceinline__ void pass_a_step(const PassArgs& a, int s, int next, float2* smem,
                                            int pkey, int& jcur) {
  using L = Line<P>;
  using R = RowCfg<P>;
  using H = SmemHead<P>;
  constexpr int E = L::E;
  float2* chs = smem + H::TAB;
  const int unit = threadIdx.x / R::U, gu = (threadIdx.x % R::U) / L::T, t = threadIdx.x % L::T;
  const UnitSync<P> sync{unit};
  const RowItem it = row_item<P>(a, s, unit);
  const int j = it.j;
  ensure_chirp_key<P>(chs, a.chirp_zhat, j, pkey * 16 + j, jcur);
  if (it.li >= it.cnt) return;  // (unit-uniform)
  float2* sm = smem + H::WORDS + (unit * R::GU + gu) * R::LS;
  const int n = a.n, lo = P / 2 - n / 2;
  const int p_lo = a.k0 * a.J;
  bool valid = it.li + gu < it.cnt;
  const int2 ln = __ldg(a.lines + a.seg_line0[j] + (valid ? it.li + gu : it.li));
  int gp = ln.x, i = ln.y;
  if constexpr (kBoundsCheck) {
    if (!line_ok(a, gp, i, P) || gp % a.J != j) {
      if (valid) flag_bounds(a.err);
      valid = false;
      gp = p_lo + j;
      i = 0;
    }
  }
  const int lp = gp - p_lo, kl = lp / a.J;
  const PlaneDesc d = a.planes[gp];
  const Tap yt = a.ytap[(long long)gp * a.tap_stride + i];
  const Tap* xt = a.xtap + (long long)gp * a.tap_stride;
  const float2* psi = a.psi + (long long)kl * n * n;
  const float2* prow = a.pj + ((long long)j * P + d.by0 + i) * P;
  float2* wrow = a.gkbuf + (long long)lp * a.gkstride + (long long)i * d.bxs;
  const float2* rmp = a.ramp_x ? a.ramp_x + (long long)gp * P : nullptr;
  // the line's two object rows mixed with its row tap, into the line's exchange buffer:
  //   r[ix] = (1 - fy) (psi[iy0][ix] - ext) + fy (psi[iy0 + 1][ix] - ext)
  // (rows outside psi dropped); the x-interpolation below reads r, so each object pixel
  // costs two coalesced, independent loads instead of four dependent gathers per position
  sync();
  if (valid) {
    const bool r0 = (unsigned)yt.i0 < (unsigned)n, r1 = (unsigned)(yt.i0 + 1) < (unsigned)n;
    const float wy0 = 1.f - yt.f, wy1 = yt.f;
    const float2* p0 = psi + (long long)(r0 ? yt.i0 : 0) * n;
    const float2* p1 = psi + (long long)(r1 ? yt.i0 + 1 : 0) * n;
    auto mix = [&](int ix) {
      float2 r = make_float2(0.f, 0.f);
      if (r0) {
        const float2 q = __ldg(p0 + ix);
        r.x = wy0 * (q.x - a.ext);
        r.y = wy0 * q.y;
      }
      if (r1) {
        const float2 q = __ldg(p1 + ix);
        r.x = fmaf(wy1, q.x - a.ext, r.x);
        r.y = fmaf(wy1, q.y, r.y);
      }
      sm[ix] = r;
    };
    if constexpr (HALF) {
#pragma unroll 8
      for (int c = 0; c < E / 2; ++c) mix(t + L::T * c);
    } else {
#pragma unroll 8
      for (int ix = t; ix < n; ix += L::T) mix(ix);
    }
  }
  sync();
  // the unit's next lines: their probe row and two object rows go to L2 now (one bulk request
  // each, issued by the line's first thread)
  if (t == 0 && next >= 0) {
    const RowItem nx = row_item<P>(a, next, unit);
    if (nx.li + gu < nx.cnt) {
      const int2 nl = __ldg(a.lines + a.seg_line0[nx.j] + nx.li + gu);
      // (a bad entry is flagged when its own line runs)
      if (!kBoundsCheck || line_ok(a, nl.x, nl.y, P)) {
        const int nlp = nl.x - p_lo;
        const PlaneDesc nd = a.planes[nl.x];
        const Tap nyt = a.ytap[(long long)nl.x * a.tap_stride + nl.y];
        l2_prefetch_bulk(a.pj + ((long long)(nlp % a.J) * P + nd.by0 + nl.y) * P + nd.bx0,
                         nd.bxs * (uint32_t)sizeof(float2));
        const float2* npsi = a.psi + (long long)(nlp / a.J) * n * n;
        if ((unsigned)nyt.i0 < (unsigned)n)
          l2_prefetch_bulk(npsi + (long long)nyt.i0 * n, n * (uint32_t)sizeof(float2));
        if ((unsigned)(nyt.i0 + 1) < (unsigned)n)
          l2_prefetch_bulk(npsi + (long long)(nyt.i0 + 1) * n, n * (uint32_t)sizeof(float2));
      }
    }
  }
  // mid: every box of this distance lies in the grid's middle half, so the registers outside
  // E/4 .. 3E/4 hold zeros
  const bool mid = HALF && ((a.mid_x >> j) & 1);
  float2 v[E];
  // the loads of CH registers (a divisor of E/4) are issued together (E = 48: 12 take 372 us where 6
  // took 409, 768^2 on 768^2, 24 x 3 planes)
  constexpr int CH = E == 48 ? 12 : (E / 4 < 8 ? E / 4 : 8);
#pragma unroll
  for (int c0 = 0; c0 < E; c0 += CH) {
    if (HALF && mid && (c0 < E / 4 || c0 >= 3 * E / 4)) {
#pragma unroll
      for (int c = c0; c < c0 + CH; ++c) v[c] = make_float2(0.f, 0.f);
      continue;
    }
    float2 tap[CH], p[CH];  // (tap: the index's bits, the weight)
#pragma unroll
    for (int q = 0; q < CH; ++q) {
      const int X = L::pos(t, c0 + q), rel = X - d.bx0;
      const bool in = valid && (unsigned)rel < (unsigned)d.bxs;
      tap[q] = in ? __ldg(reinterpret_cast<const float2*>(xt + rel)) : make_float2(0.f, 0.f);
      p[q] = in ? __ldg(prow + X) : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int q = 0; q < CH; ++q) {
      const int rel = L::pos(t, c0 + q) - d.bx0;
      const int i0 = __float_as_int(tap[q].x);
      const float f = tap[q].y;
      float2 w = make_float2(0.f, 0.f);
      if (valid && (unsigned)rel < (unsigned)d.bxs) {
        if ((unsigned)i0 < (unsigned)n) {
          const float2 r = sm[i0];
          w.x = (1.f - f) * r.x;
          w.y = (1.f - f) * r.y;
        }
        if ((unsigned)(i0 + 1) < (unsigned)n) {
          const float2 r = sm[i0 + 1];
          w.x = fmaf(f, r.x, w.x);
          w.y = fmaf(f, r.y, w.y);
        }
        if (!HALF && rmp) w.x += a.ext;  // full-grid form: w = R' psi
        wrow[rel] = w;
      }
      v[c0 + q] = cmul(p[q], w);
    }
  }
  const ChirpAt<P> cat(chs, t);
  line_dstep<L, HALF>(v, sm, smem, t, sync, mid, [&](float2 (&x)[E]) HOLO_INLINE {
#pragma unroll
    for (int c = 0; c < E; ++c) x[c] = cmul(x[c], cat(c));
    if (!HALF && rmp) {
#pragma unroll
      for (int c = 0; c < E; ++c) x[c] = cmul(x[c], __ldg(rmp + L::fpos(t, c)));
    }
  });
  float2* yrow = a.ybuf + (long long)lp * a.ystride + (long long)i * n;
#pragma unroll
  for (int c = 0; c < E; ++c) {
    const int rel = L::pos(t, c) - lo;
    if (valid && (HALF ? mid_reg<P>(c) : (unsigned)rel < (unsigned)n)) yrow[rel] = v[c];
  }
}

// One block-step of pass C for the calling unit (arguments as pass_a_step).  The row of V holds
// the conjugate of the adjoint field (pass B), and the chirp is even, so the adjoint row
// transform is the forward one: with x = conj(v) on the box, z = conj(p) v = conj(p x) and
// conj(w) v = conj(w x).
template <int P, bool HALF>
__device__ __forceinline__ void pass_c_step(const PassArgs& a, int s, int next, float2* smem,
                                            int pkey, int& jcur) {
  using L = Line<P>;
  using R = RowCfg<P>;
  using H = SmemHead<P>;
  constexpr int E = L::E;
  float2* chs = smem + H::TAB;
  const int unit = threadIdx.x / R::U, gu = (threadIdx.x % R::U) / L::T, t = threadIdx.x % L::T;
  const UnitSync<P> sync{unit};
  const RowItem it = row_item<P>(a, s, unit);
  const int j = it.j;
  ensure_chirp_key<P>(chs, a.chirp_zhat, j, pkey * 16 + j, jcur);
  if (it.li >= it.cnt) return;  // (unit-uniform)
  float2* sm = smem + H::WORDS + (unit * R::GU + gu) * R::LS;
  const int n = a.n, lo = P / 2 - n / 2;
  const int p_lo = a.k0 * a.J;
  bool valid = it.li + gu < it.cnt;
  const int2 ln = __ldg(a.lines + a.seg_line0[j] + (valid ? it.li + gu : it.li));
  int gp = ln.x, i = ln.y;
  if constexpr (kBoundsCheck) {
    if (!line_ok(a, gp, i, P) || gp % a.J != j) {
      if (valid) flag_bounds(a.err);
      valid = false;
      gp = p_lo + j;
      i = 0;
    }
  }
  const int lp = gp - p_lo;
  float2* yrow = a.ybuf + (long long)lp * a.ystride + (long long)i * n;
  const float2* rmp = a.ramp_x ? a.ramp_x + (long long)gp * P : nullptr;
  float2 v[E];
#pragma unroll
  for (int c = 0; c < E; ++c) {
    const int rel = L::pos(t, c) - lo;
    const bool in = HALF ? mid_reg<P>(c) : (unsigned)rel < (unsigned)n;
    v[c] = (valid && in) ? yrow[rel] : make_float2(0.f, 0.f);
  }
  // the unit's next lines: their adjoint-field row, probe row and w row go to L2 now (one bulk
  // request each, issued by the line's first thread)
  if (t == 0 && next >= 0) {
    const RowItem nx = row_item<P>(a, next, unit);
    if (nx.li + gu < nx.cnt) {
      const int2 nl = __ldg(a.lines + a.seg_line0[nx.j] + nx.li + gu);
      // (a bad entry is flagged when its own line runs)
      if (!kBoundsCheck || line_ok(a, nl.x, nl.y, P)) {
        const int nlp = nl.x - p_lo;
        const PlaneDesc nd = a.planes[nl.x];
        l2_prefetch_bulk(a.ybuf + (long long)nlp * a.ystride + (long long)nl.y * n,
                         n * (uint32_t)sizeof(float2));
        l2_prefetch_bulk(a.pj + ((long long)(nlp % a.J) * P + nd.by0 + nl.y) * P + nd.bx0,
                         nd.bxs * (uint32_t)sizeof(float2));
        l2_prefetch_bulk(a.gkbuf + (long long)nlp * a.gkstride + (long long)nl.y * nd.bxs,
                         nd.bxs * (uint32_t)sizeof(float2));
      }
    }
  }
  const ChirpAt<P> cat(chs, t);
  const PlaneDesc d = a.planes[gp];
  const float2* prow = a.pj + ((long long)j * P + d.by0 + i) * P;
  float2* gk = a.gkbuf + (long long)lp * a.gkstride + (long long)i * d.bxs;
  line_dstep<L, HALF>(v, sm, smem, t, sync, HALF, [&](float2 (&x)[E]) HOLO_INLINE {
#pragma unroll
    for (int c = 0; c < E; ++c) x[c] = cmul(x[c], cat(c));
    if (!HALF && rmp) {
      // (the multiplier of the conjugated line: the ramp at -f)
#pragma unroll
      for (int c = 0; c < E; ++c) {
        const int f = L::fpos(t, c);
        x[c] = cmul(x[c], __ldg(rmp + (f ? P - f : 0)));
      }
    }
  });
  sync();  // the exchange buffer has been read
  // The box holds w = R0(psi - ext) (R' psi with probe shifts) written by pass A; replace it by
  // conj(w) v.  mid: every box of this distance lies in the grid's middle half.
  const bool mid = HALF && ((a.mid_x >> j) & 1);
  // registers [c0, c0 + CH): the loads of all of them are issued together
  auto scatter = [&](auto c0c, auto chc) HOLO_INLINE {
    constexpr int c0 = decltype(c0c)::value, CH = decltype(chc)::value;
    float2 p[CH], w[CH];
#pragma unroll
    for (int q = 0; q < CH; ++q) {
      const int X = L::pos(t, c0 + q), rel = X - d.bx0;
      const bool in = valid && (unsigned)rel < (unsigned)d.bxs;
      p[q] = in ? __ldg(prow + X) : make_float2(0.f, 0.f);
      w[q] = in ? gk[rel] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int q = 0; q < CH; ++q) {
      const int rel = L::pos(t, c0 + q) - d.bx0;
      if (valid && (unsigned)rel < (unsigned)d.bxs) {
        sm[rel] = cmul(p[q], v[c0 + q]);
        gk[rel] = cconj(cmul(w[q], v[c0 + q]));
      }
    }
  };
  if (HALF && mid)
    static_for<(E > 32 ? 2 : 1)>([&](auto ic) HOLO_INLINE {
      constexpr int W = E > 32 ? E / 4 : E / 2;
      scatter(Idx<E / 4 + W * decltype(ic)::value>{}, Idx<W>{});
    });
  else
    static_for<E / 8>([&](auto ic) HOLO_INLINE {
      scatter(Idx<8 * decltype(ic)::value>{}, Idx<8>{});
    });
  // x-transpose of the bilinear resample: h[ip] = w0 z[X0] + w1 z[X0 + 1] with the
  // transposed taps of this plane (same FP64-built weights as the forward taps); the buffer
  // holds conj(z).
  const float4* xa = reinterpret_cast<const float4*>(a.xadj + (long long)gp * n);
  constexpr int EH = HALF ? E / 2 : E, CT = EH < 16 ? EH : (E % 16 || E == 48 ? 12 : 16);
#pragma unroll
  for (int c0 = 0; c0 < EH; c0 += CT) {
    float4 tp[CT];  // (the position's bits, both weights; loaded ahead of the barrier)
#pragma unroll
    for (int q = 0; q < CT; ++q) {
      const int ip = HALF ? t + L::T * (c0 + q) : L::pos(t, c0 + q);
      tp[q] = (valid && ip < n) ? __ldg(xa + ip) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (c0 == 0) sync();
#pragma unroll
    for (int q = 0; q < CT; ++q) {
      const int ip = HALF ? t + L::T * (c0 + q) : L::pos(t, c0 + q);
      if (!valid || ip >= n) continue;
      float2 h = make_float2(0.f, 0.f);
      const int r0 = __float_as_int(tp[q].x) - d.bx0;
      const float w0 = tp[q].y, w1 = tp[q].z;
      if (w0 != 0.f) {
        const float2 z = sm[r0];
        h.x = w0 * z.x;
        h.y = -w0 * z.y;
      }
      if (w1 != 0.f) {
        const float2 z = sm[r0 + 1];
        h.x = fmaf(w1, z.x, h.x);
        h.y = fmaf(-w1, z.y, h.y);
      }
      yrow[ip] = h;
    }
  }
}

template <int P, bool HALF, bool PASS_C>
__device__ __forceinline__ void row_step(const PassArgs& a, int s, int next, float2* smem, int pkey,
                                         int& jcur) {
  if constexpr (PASS_C)
    pass_c_step<P, HALF>(a, s, next, smem, pkey, jcur);
  else
    pass_a_step<P, HALF>(a, s, next, smem, pkey, jcur);
}

// Pass A or C of one problem: persistent blocks over the chunk's block-steps.
template <int P, bool HALF, bool PASS_C>
__global__ void __launch_bounds__(RowCfg<P>::NT, RowCfg<P>::MINB)
k_rows(const __grid_constant__ PassArgs a) {
  extern __shared__ __align__(16) float2 smem[];
  Line<P>::load_table(smem, a.twiddles);
  int jcur = -1;
  const int steps = a.seg_step[a.J];
  for (int s = blockIdx.x; s < steps; s += gridDim.x)
    row_step<P, HALF, PASS_C>(a, s, s + (int)gridDim.x < steps ? s + (int)gridDim.x : -1, smem, 0,
                              jcur);
}

// The arguments of the problem a multi-problem block works on, copied to shared memory (block-wide;
// block-uniform `prob`).
__device__ __forceinline__ void fetch_args(PassArgs& dst, const PassArgs* __restrict__ args, int prob,
                                           int& cur) {
  if (prob == cur) return;
  __syncthreads();
  const int* src = reinterpret_cast<const int*>(args + prob);
  for (int i = threadIdx.x; i < (int)(sizeof(PassArgs) / sizeof(int)); i += blockDim.x)
    reinterpret_cast<int*>(&dst)[i] = __ldg(src + i);
  __syncthreads();
  cur = prob;
}

// Pass A or C of several problems of line length P in one persistent launch: items {problem,
// block-step}, walked by the blocks in a grid-stride loop (args: one PassArgs per problem, in
// device memory).
template <int P, bool HALF, bool PASS_C>
__global__ void __launch_bounds__(RowCfg<P>::NT, RowCfg<P>::MINB)
k_rows_multi(const PassArgs* __restrict__ args, const int2* __restrict__ items, int nitems) {
  extern __shared__ __align__(16) float2 smem[];
  __shared__ PassArgs a;
  Line<P>::load_table(smem, args[items[0].x].twiddles);  // every item has this P
  int jcur = -1, cur = -1;
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    const int2 item = items[it];
    fetch_args(a, args, item.x, cur);
    int next = -1;
    if (it + (int)gridDim.x < nitems) {
      const int2 ni = items[it + gridDim.x];
      if (ni.x == item.x) next = ni.y;
    }
    row_step<P, HALF, PASS_C>(a, item.y, next, smem, item.x, jcur);
  }
}

// ------------------------------------------------------------------ pass B

// Tensor memory of pass B per thread (32-bit columns): b and the residual sum S of its NS crop
// registers; in the HALF form from P = 1024 also its E chirp entries, so that shared memory holds
// the blocks that registers allow together with their Y stages (the chirp read through L1/L2
// instead: pass B 19.2 against 17.4 ms on the 2048^2 chunk, 2.97 against 2.77 at 512^2; below P =
// 1024 neither it nor the stage changed the time).  The general forms of these lengths have no room
// for it there; their chirp is in shared memory unless the Y stage fits only without it, then it is
// read through L1/L2 (see pass_b_chirp_global).
template <int P, bool HALF>
struct PassBMem {
  static constexpr int E = Line<P>::E;
  static constexpr int NS = HALF ? E / 2 : E;
  static constexpr bool CHIRP_TM = HALF && P >= 1024;
  static constexpr bool CHIRP_ANY = !HALF && P >= 1024 && !Line<P>::R3;
  static constexpr int WORDS = 4 * NS + (CHIRP_TM ? 2 * E : 0);
  static constexpr int COLS = tmem_pow2(WORDS * ((ColCfg<P>::NT + 127) / 128));
  static_assert(COLS <= 512, "tensor memory");
  static constexpr int MAXB = 512 / COLS;  // resident blocks per SM
  // in front of the exchange lines: twiddles, and the chirp unless it has a place of its own
  static constexpr int HEAD = CHIRP_TM || CHIRP_ANY ? SmemHead<P>::TAB : SmemHead<P>::WORDS;
};

// Y stage of pass B: whole TMA boxes covering `rows` box rows of C columns.
template <int P>
size_t pass_b_stage_bytes(int rows) {
  constexpr int BOX = stage_box(P);
  return (size_t)((rows + BOX - 1) / BOX) * BOX * ColCfg<P>::C * sizeof(float2);
}

// Shared memory of pass B: head, C exchange lines, with CHIRP_ANY the chirp unless chirp_global; with
// srows > 0 also the Y stage for planes of up to srows box rows (128-byte aligned).
template <int P, bool HALF>
size_t pass_b_smem(int srows, bool chirp_global) {
  using M = PassBMem<P, HALF>;
  const int chirp = M::CHIRP_ANY && !chirp_global ? SmemHead<P>::CHIRP : 0;
  const size_t base = (size_t)(M::HEAD + ColCfg<P>::C * ColCfg<P>::LS + chirp) * sizeof(float2);
  return srows > 0 ? base + 128 + pass_b_stage_bytes<P>(srows) : base;
}

// Crop rows per run of pass B's loads (a divisor of NS, a multiple of 4).
__host__ __device__ constexpr int crop_run(int ns) {
  return ns % 16 == 0 ? 16 : (ns % 12 == 0 ? 12 : 8);
}

// One plane of a block's pass-B work, in shared memory: the block's threads read a field where
// they need it, so that no register holds it through the transforms.
struct PassBPlane {
  int more;            // 0: the block's work is done
  int sg, pp;          // segment, plane (distance, angle order: j * nk + kl)
  int cg, p1;          // column group, end of the segment's planes
  int first;           // first plane of the segment
  int j, lp, by0, bys; // distance, plane slot, box rows
};
__device__ __forceinline__ int peek(const int& x) { return *const_cast<const volatile int*>(&x); }

// What thread 0 keeps (in shared memory) of the plane after the next one: its place in the work
// and its descriptor, on its way from global memory.
struct PassBAhead {
  PlaneDesc desc;
  int more, sg, pp, cg, p1, first, j, kl;
};
struct PassBState {
  PassBPlane plane[2];
  alignas(16) PassBAhead ahead;
};

// The work of block `bid` of `nblk` as segments {column group, planes [p0, p1)}: whole groups
// bid, bid + nblk, ...; with a.pb_split the last, partial round's (group, plane) items in even
// shares over all blocks.
template <int P>
__device__ bool pass_b_segment(const PassArgs& a, int bid, int nblk, int sg, int& cg, int& p0,
                               int& p1) {
  const int ngroups = (a.n + ColCfg<P>::C - 1) / ColCfg<P>::C, per = a.J * a.nk;
  const bool tsplit = a.pb_split != 0 && ngroups % nblk != 0;
  const int rounds = tsplit ? ngroups / nblk : (ngroups - bid + nblk - 1) / nblk;
  if (sg < rounds) {
    cg = bid + sg * nblk;
    p0 = 0;
    p1 = per;
    return true;
  }
  if (!tsplit) return false;
  const long long titems = (long long)(ngroups - rounds * nblk) * per;
  const long long ti0 = split_begin(titems, nblk, bid), ti1 = split_begin(titems, nblk, bid + 1);
  const long long tg = ti0 / per + (sg - rounds), g0 = tg * per;
  if (ti0 >= ti1 || g0 >= ti1) return false;
  cg = rounds * nblk + (int)tg;
  p0 = (int)(ti0 > g0 ? ti0 - g0 : 0);
  p1 = (int)(ti1 - g0 < per ? ti1 - g0 : per);
  return true;
}

// Thread 0: the plane after the one in `ah` (start: the block's first one) into `ah`, its
// descriptor copied asynchronously.
template <int P>
__device__ __forceinline__ void pass_b_advance(const PassArgs& a, int bid, int nblk, PassBAhead& ah,
                                               bool start) {
  int sg = start ? -1 : ah.sg, pp = start ? 0 : ah.pp + 1, p1 = start ? 0 : ah.p1;
  int j = ah.j, kl = ah.kl + 1, first = 0;
  if (pp >= p1) {
    ++sg;
    first = 1;
    int cg = 0;
    ah.more = pass_b_segment<P>(a, bid, nblk, sg, cg, pp, p1) ? 1 : 0;
    if (!ah.more) return;
    ah.cg = cg;
    ah.p1 = p1;
    ah.sg = sg;
    j = pp / a.nk;
    kl = pp - j * a.nk;
  } else if (kl == a.nk) {
    kl = 0;
    ++j;
  }
  ah.pp = pp;
  ah.first = first;
  ah.j = j;
  ah.kl = kl;
  const PlaneDesc* src = a.planes + (long long)(a.k0 + kl) * a.J + j;
  static_assert(sizeof(PlaneDesc) == 32, "two 16-byte copies");
  cp_async16(&ah.desc, src);
  cp_async16(reinterpret_cast<char*>(&ah.desc) + 16, reinterpret_cast<const char*>(src) + 16);
}

// Thread 0: the plane in `ah` into `nx`; for a staged problem its Y tile (every box of the plane's
// box rows; rows past them are not read) is loaded, and its data are fetched into L2.  Then `ah`
// moves on.
template <int P>
__device__ __noinline__ void pass_b_next(const PassArgs& a, int bid, int nblk, PassBAhead& ah,
                                         PassBPlane* nx, float2* stg, uint64_t* bar) {
  constexpr int C = ColCfg<P>::C, BOX = stage_box(P);
  nx->more = ah.more;
  if (!ah.more) return;
  cp_async_wait();
  PlaneDesc d = ah.desc;
  const int lp = ah.kl * a.J + ah.j, cg = ah.cg;
  const long long gplane = (long long)a.k0 * a.J + lp;
  if constexpr (kBoundsCheck) {
    if (!plane_box_ok(a, d, P)) {
      flag_bounds(a.err);
      d.bys = 0;  // the plane's box rows are skipped
    }
  }
  if (a.ymap) {
    const int nb = (d.bys + BOX - 1) / BOX;
    const int row0 = lp * a.yrows;
    mbar_expect_tx(bar, (uint32_t)(nb * BOX * C * sizeof(float2)));
    for (int b = 0; b < nb; ++b)
      tma_load_2d(stg + b * BOX * C, a.ymap, 2 * C * cg, row0 + b * BOX, bar);
  }
  l2_prefetch_bulk(a.dblk + ((gplane - (long long)a.data_k0 * a.J) * a.dgroups + cg) * (long long)a.n * C,
                   (uint32_t)(a.n * C * sizeof(float)));
  nx->sg = ah.sg;
  nx->pp = ah.pp;
  nx->cg = cg;
  nx->p1 = ah.p1;
  nx->first = ah.first;
  nx->j = ah.j;
  nx->lp = lp;
  nx->by0 = d.by0;
  nx->bys = d.bys;
  pass_b_advance<P>(a, bid, nblk, ah, false);
}

// Each block owns whole column groups (C adjacent detector columns) and walks every plane
// of the chunk for them, distance-major: the columns of b = C D_{zeta_0} q are read once,
// and S = sum_kj r_kj is accumulated in a fixed order and written once (with the reference
// residual) as the source of the ext-part of grad_q.  Every S / b slot belongs to one thread
// (its crop rows of its column) and lives in tensor memory.
//
// Per plane the block runs "column transform, chirp, inverse" twice through one loop body: first
// on Y, then on the conjugated residual.  The chirp is even in frequency, so the adjoint of D is
// conj D conj: the second turn yields conj(V), which is what is stored (pass C takes it as is).
//
// What bounds it: the transforms themselves (11.7 of 17.4 ms on the 2048^2 chunk of 240 planes, 1.6
// of 2.8 at 512^2 x 720 planes, alone on the chip), FP32 pipe 48 % and shared memory 51 % busy; the
// 16-byte pieces of V's stores cost 1.6 ms at P = 4096.  The 128 registers of two 256-thread blocks
// (four of 128) do not hold a plane's 32 values and all else: 104 to 180 bytes of spills a thread
// remain in these forms.  Before (b, S and chirp in shared memory, one block per SM, radix-16
// engine): 20.0 and 5.6 ms; 1024^2 x 360 planes 8.9 -> 6.1 ms.  Without the Y stage 22.9 ms.  With the
// block's work list and descriptors in registers the spills (900 bytes a plane) went to L2: 31.8 ms,
// so fields are read from shared memory (peek) where they are used.
//
// The block's FP64 loss partial goes to a.loss_part[bid].  The caller has loaded the twiddle
// table at the head of shared memory and, for a staged problem, initialised the Y-stage barrier.
// The resident chirp table is identified by pkey * 16 + distance; chirp_global (CHIRP_ANY only, one
// value for the whole launch): there is none, its entries are read from global memory.  Returns false
// when a bounded Y-stage wait gave up (the problem's error word is then set).
template <int P, bool HALF>
__device__ __forceinline__ bool pass_b_run(const PassArgs& a, int bid, int nblk, float2* smem,
                                           uint32_t tmem, double* red, uint64_t* ybarp,
                                           PassBState& st, uint32_t& yphase, int pkey,
                                           int& jcur, bool chirp_global) {
  using L = Line<P>;
  using Cc = ColCfg<P>;
  using H = SmemHead<P>;
  using M = PassBMem<P, HALF>;
  constexpr int C = Cc::C, E = L::E, NS = M::NS, S0 = HALF ? E / 4 : 0;
  static_assert(!HALF || half_form_ok<P>(), "HALF form");
  chirp_global = M::CHIRP_ANY && chirp_global;
  float2* chs = smem + (M::CHIRP_ANY ? M::HEAD + C * Cc::LS : H::TAB);
  const int g = threadIdx.x % C, t = threadIdx.x / C;
  float2* sm = smem + M::HEAD + g * Cc::LS;
  const uint32_t tm = tmem_own(tmem, M::WORDS);
  const int n = a.n, lo = P / 2 - n / 2;
  // with probe shifts the ext-part is inside the full-grid rows
  const float ext = !HALF && a.ramp_y ? 0.f : a.ext;
  double dsum = 0.0;
  // Y stage: the tile of the block's next plane is in flight while the current one computes
  // (aligned at run time: the dynamic shared memory of a block starts on a 16-byte boundary only)
  float2* const end = smem + M::HEAD + C * Cc::LS + (M::CHIRP_ANY && !chirp_global ? H::CHIRP : 0);
  float2* stg = reinterpret_cast<float2*>((reinterpret_cast<uintptr_t>(end) + 127) &
                                          ~static_cast<uintptr_t>(127));
  __syncthreads();  // (a multi-problem block's previous work item is done with `st`)
  if (threadIdx.x == 0) {
    pass_b_advance<P>(a, bid, nblk, st.ahead, true);
    pass_b_next<P>(a, bid, nblk, st.ahead, &st.plane[0], stg, ybarp);
  }
  __syncthreads();
  for (int par = 0; peek(st.plane[par].more); par ^= 1) {
    const PassBPlane& pl = st.plane[par];
    if (peek(pl.first)) {
      // (the stores and loads of tensor memory take whole warps)
      const int col = peek(pl.cg) * C + g;
      // (RUN loads in flight: four at a time the twelve rounds of NS = 48 took 5 us of a small problem.
      // The n = P/2 forms of 32 and 48 values have 4 or 6 rounds and keep to four: with longer runs
      // ptxas spills more in the loops below, a batch of sides 256 .. 1024 takes 0.8 % longer)
      constexpr int RUN = HALF && E >= 32 ? 4 : crop_run(NS);
#pragma unroll 1
      for (int k = 0; k < NS; k += RUN) {
        float2 x[RUN / 4][4], zero[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) zero[i] = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < RUN; ++i) {
          const int rr = L::pos(t, S0 + k + i) - lo;
          x[i / 4][i % 4] = (col < n && (unsigned)rr < (unsigned)n && ext != 0.f)
                                ? __ldg(a.bref + (long long)rr * n + col)
                                : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < RUN; i += 4) {
          tmem_store4(tm + 2 * (k + i), x[i / 4]);
          tmem_store4(tm + 2 * NS + 2 * (k + i), zero);
        }
      }
      tmem_store_done();
    }
    {
      const int j = peek(pl.j);
      if constexpr (M::CHIRP_TM) {
        if (pkey * 16 + j != jcur) {
          const float2* chg = a.chirp_zhat + (long long)j * P;
#pragma unroll 1
          for (int k = 0; k < E; k += 16) {
            float2 x[4][4];
#pragma unroll
            for (int i = 0; i < 16; ++i) x[i / 4][i % 4] = __ldg(chg + L::fpos(t, k + i));
#pragma unroll
            for (int i = 0; i < 4; ++i) tmem_store4(tm + 4 * NS + 2 * (k + 4 * i), x[i]);
          }
          tmem_store_done();
          jcur = pkey * 16 + j;
        }
      } else if (!chirp_global) {
        ensure_chirp_key<P>(chs, a.chirp_zhat, j, pkey * 16 + j, jcur);
      }
    }
    float2 v[E];
    // the plane's rows of Y; mid (HALF form only): its box rows lie in P/4 .. 3P/4, i.e. in the
    // registers E/4 .. 3E/4
    auto is_mid = [&](int by0, int bys) HOLO_INLINE {
      return HALF && by0 >= P / 4 && by0 + bys <= 3 * P / 4;
    };
    bool mid;
    {
      const int by0 = peek(pl.by0), bys = peek(pl.bys), col = peek(pl.cg) * C + g;
      const bool valid = HALF || col < n;
      mid = is_mid(by0, bys);
      auto load_y = [&](auto at) HOLO_INLINE {
#pragma unroll
        for (int c0 = 0; c0 < E; c0 += E / 4) {
          if (HALF && mid && (c0 < E / 4 || c0 >= 3 * E / 4)) {
#pragma unroll
            for (int c = c0; c < c0 + E / 4; ++c) v[c] = make_float2(0.f, 0.f);
            continue;
          }
#pragma unroll
          for (int c = c0; c < c0 + E / 4; ++c) {
            const int rel = L::pos(t, c) - by0;
            v[c] = (valid && (unsigned)rel < (unsigned)bys) ? at(rel) : make_float2(0.f, 0.f);
          }
        }
      };
      if (a.ymap != nullptr) {
        const bool ok = mbar_wait(ybarp, yphase);
        yphase ^= 1;
        load_y([&](int rel) HOLO_INLINE { return stg[rel * C + g]; });
        // every thread has its tile entries: the stage is free for the next plane
        if (__syncthreads_or(!ok)) {
          if (threadIdx.x == 0) atomicOr(a.err, 1ull);
          return false;
        }
      } else {
        const float2* yb = a.ybuf + (long long)peek(pl.lp) * a.ystride + col;
        load_y([&](int rel) HOLO_INLINE { return yb[(long long)rel * n]; });
        __syncthreads();
      }
    }
    if (threadIdx.x == 0) pass_b_next<P>(a, bid, nblk, st.ahead, &st.plane[par ^ 1], stg, ybarp);
    if constexpr (L::T == 1) __syncthreads();  // (the transforms of longer lines hold barriers)
#pragma unroll 1
    for (int turn = 0;; ++turn) {
      // zero inputs outside the middle half: Y's box rows (mid), the residual's crop rows (HALF)
      line_dstep<L, HALF>(
          v, sm, smem, t, SyncBlock{}, HALF && (mid || turn), [&](float2 (&x)[E]) HOLO_INLINE {
            if constexpr (M::CHIRP_TM) {
#pragma unroll
              for (int k = 0; k < E; k += 4) {
                float2 ch[4];
                tmem_load4(ch, tm + 4 * NS + 2 * k);
#pragma unroll
                for (int i = 0; i < 4; ++i) x[k + i] = cmul(x[k + i], ch[i]);
              }
            } else {
              // (the first P/2 + 1 entries of the table in global memory are the half table)
              const ChirpAt<P> cat(
                  chirp_global ? a.chirp_zhat + (long long)peek(pl.j) * P : chs, t);
#pragma unroll
              for (int c = 0; c < E; ++c) x[c] = cmul(x[c], cat(c));
            }
            if (!HALF && a.ramp_y) {
              // (the multiplier of the conjugated second turn: the ramp at -f)
              const float2* rmp = a.ramp_y + ((long long)a.k0 * a.J + peek(pl.lp)) * P;
#pragma unroll
              for (int c = 0; c < E; ++c) {
                const int f = L::fpos(t, c);
                x[c] = cmul(x[c], __ldg(rmp + (turn && f ? P - f : f)));
              }
            }
          });
      if (turn) break;
      const int lp = peek(pl.lp), cg = peek(pl.cg), col = cg * C + g;
      const bool valid = HALF || col < n;
      const float* ad =
          a.dblk +
          (((long long)(a.k0 - a.data_k0) * a.J + lp) * a.dgroups + cg) * (long long)n * C + g;
      float2* uo = a.u_out ? a.u_out + (long long)lp * n * n + col : nullptr;
      // The plane's loss terms of the thread: FP32 over groups of four, the groups added in FP32, FP64
      // from there on.  A term meets 3 + NS/4 - 1 roundings at most (6 at NS = 16, 10 at 32, 14 at 48);
      // one chain over all NS would meet NS - 1.
      float lsum = 0.f;
      // (the loads of RUN crop rows' data are issued together, ahead of their use; all NS at once
      // spill at NS = 32 and 48)
      constexpr int RUN = NS == 24 ? 24 : crop_run(NS);
#pragma unroll
      for (int k0 = 0; k0 < NS; k0 += RUN) {
        float dat[RUN];
#pragma unroll
        for (int k = 0; k < RUN; ++k) {
          const int rr = L::pos(t, S0 + k0 + k) - lo;
          dat[k] = (HALF || (valid && (unsigned)rr < (unsigned)n)) ? __ldg(ad + rr * C) : 0.f;
        }
#pragma unroll
        for (int k = 0; k < RUN; k += 4) {
          float2 b[4], S[4];
          tmem_load4x2(b, S, tm + 2 * (k0 + k), tm + 2 * NS + 2 * (k0 + k));
          float l4 = 0.f;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int c = S0 + k0 + k + i;
            const int rr = L::pos(t, c) - lo;
            float2 r = make_float2(0.f, 0.f);
            if (HALF || (valid && (unsigned)rr < (unsigned)n)) {
              float2 u = v[c];
              u.x = fmaf(ext, b[i].x, u.x);
              u.y = fmaf(ext, b[i].y, u.y);
              const float i2 = fmaf(u.x, u.x, u.y * u.y);
              // F2: (|u| - a)^2, r = u - a u/|u| (u/|u| := 0 at |u| = 0);
              // F1: (|u|^2 - d)^2, r = 2 (|u|^2 - d) u
              float diff, f;
              if (a.functional) {
                diff = i2 - dat[k + i];
                f = 2.f * diff;
              } else {
                const float mag = sqrtf(i2);
                diff = mag - dat[k + i];
                f = mag > 0.f ? 1.f - __fdividef(dat[k + i], mag) : 0.f;
              }
              l4 = fmaf(diff, diff, l4);
              if (uo) uo[(long long)rr * n] = u;
              r = cscale(u, f);
            }
            S[i] = cadd(S[i], r);
            v[c] = cconj(r);
          }
          lsum += l4;
          if (a.adj) tmem_store4(tm + 2 * NS + 2 * (k0 + k), S);
        }
      }
      dsum += (double)lsum;
      if (!a.adj) break;
      tmem_store_done();
    }
    if (!a.adj) continue;
    {
      const int by0 = peek(pl.by0), bys = peek(pl.bys), col = peek(pl.cg) * C + g;
      const bool valid = HALF || col < n, md = is_mid(by0, bys);
      float2* yb = a.ybuf + (long long)peek(pl.lp) * a.ystride + col;
#pragma unroll
      for (int c0 = 0; c0 < E; c0 += E / 4) {
        if (HALF && md && (c0 < E / 4 || c0 >= 3 * E / 4)) continue;
#pragma unroll
        for (int c = c0; c < c0 + E / 4; ++c) {
          const int rel = L::pos(t, c) - by0;
          if (valid && (unsigned)rel < (unsigned)bys) yb[(long long)rel * n] = v[c];
        }
      }
    }
    if (peek(pl.pp) + 1 < peek(pl.p1)) continue;
    // the segment's residual sum: T of a whole group; part of a last-round group goes to the
    // block's slot sg - rounds (k_pass_b_tail adds the slots of the group in block order into T)
    const int ngroups = (n + C - 1) / C, slot = peek(pl.sg) - ngroups / nblk;
    const bool part = a.pb_split != 0 && ngroups % nblk != 0 && slot >= 0;
    const int col = peek(pl.cg) * C + g;
    float2* tp = a.tpart + ((long long)bid * a.tslots + slot) * n * C + g;
#pragma unroll 1
    for (int k = 0; k < NS; k += 4) {
      float2 S[4];
      tmem_load4(S, tm + 2 * NS + 2 * k);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int rr = L::pos(t, S0 + k + i) - lo;
        if ((unsigned)rr >= (unsigned)n) continue;
        if (part) {
          tp[rr * C] = S[i];
        } else if (col < n) {
          const long long e = (long long)rr * n + col;
          float2 acc = cscale(S[i], ext);
          if (a.tq_accumulate) acc = cadd(acc, a.tq[e]);
          if (a.rref) {
            const float2 q = __ldg(a.rref + e);
            acc.x = fmaf(a.wref, q.x, acc.x);
            acc.y = fmaf(a.wref, q.y, acc.y);
          }
          a.tq[e] = acc;
        }
      }
    }
  }
  const double s = block_sum_f64(dsum, red);
  if (threadIdx.x == 0) a.loss_part[bid] = s;
  return true;
}

// Resident blocks that the registers must allow, hence the registers a thread may take: 128 at two
// blocks of 256 threads (P = 2048, 4096) or four of 128 (512, 1024), 96 at five (up to 256), 168 at
// three (3 * 2^k) and 255 at two (the general form at 384 and 768, whose b and S leave room for two
// blocks in tensor memory: with the bound at three it kept to 168 registers and spilled 550 bytes, but
// two blocks ran all the same; 768^2 on 768^2, 24 x 3 planes: 1330 -> 710 us).  P = 1536 and 3072: one
// block of 384 threads.
template <int P, bool HALF>
constexpr int pass_b_minb() {
  using L = Line<P>;
  constexpr int b = L::R3 ? 1 : (L::M3 ? 3 : (P >= 2048 ? 2 : (P >= 512 ? 4 : 5)));
  return b < PassBMem<P, HALF>::MAXB ? b : PassBMem<P, HALF>::MAXB;
}

template <int P, bool HALF>
__global__ void __launch_bounds__(ColCfg<P>::NT, pass_b_minb<P, HALF>())
k_pass_b(const __grid_constant__ PassArgs args, int chirp_global) {
  extern __shared__ __align__(16) float2 smem[];
  __shared__ double red[32];
  __shared__ uint64_t ybar;
  __shared__ uint32_t tbase;
  __shared__ PassBState state;
  using M = PassBMem<P, HALF>;
  if (threadIdx.x < 32) tmem_alloc(&tbase, M::COLS);
  // Up to P = 768 the loops read the arguments from shared memory: constant-bank values that do not
  // change are kept in registers or make the compiler copy the loops (at 96 to 168 registers 20 to 550
  // bytes of spills, from shared memory none up to 256 and half at 512; 384^2 on 768^2 206 -> 195 us,
  // 258^2 on 512^2, 24 x 3 planes, 116 -> 107 us).  Longer lines lose by it (512^2 on 1024^2 411 ->
  // 434 us, 2048^2 on 4096^2 2395 -> 2472 us).  The barrier stays for them as well: without it the
  // compiler schedules the code behind it differently, 1 to 4 % slower from P = 1024.
  constexpr bool ARGS_SHARED = P <= 768;
  __shared__ PassArgs sargs;
  const PassArgs& a = ARGS_SHARED ? sargs : args;
  if (ARGS_SHARED) {
    for (int i = threadIdx.x; i < (int)(sizeof(PassArgs) / sizeof(int)); i += blockDim.x)
      reinterpret_cast<int*>(&sargs)[i] = reinterpret_cast<const int*>(&args)[i];
  }
  __syncthreads();
  Line<P>::load_table(smem, a.twiddles);
  if (threadIdx.x == 0) mbar_init(&ybar);
  __syncthreads();
  uint32_t yphase = 0;
  int jcur = -1;
  pass_b_run<P, HALF>(a, blockIdx.x, gridDim.x, smem, tbase, red, &ybar, state, yphase, 0, jcur,
                      chirp_global != 0);
  __syncthreads();
  if (threadIdx.x < 32) tmem_free(tbase, M::COLS);
}

// Pass B of several problems of line length P in one persistent launch: items {problem, b},
// b < the problem's own pass-B grid (a.pb_blocks), each the work of block b of that grid, so
// every problem's results (loss partials included) are those of its own launch bit for bit.
// A Y-stage wait that gives up sets the error word of every problem of the launch.
template <int P, bool HALF>
__global__ void __launch_bounds__(ColCfg<P>::NT, pass_b_minb<P, HALF>())
k_pass_b_multi(const PassArgs* __restrict__ args, const int2* __restrict__ items, int nitems,
               int nprob, int chirp_global) {
  extern __shared__ __align__(16) float2 smem[];
  __shared__ double red[32];
  __shared__ uint64_t ybar;
  __shared__ uint32_t tbase;
  __shared__ PassBState state;
  using M = PassBMem<P, HALF>;
  __shared__ PassArgs a;
  if (threadIdx.x < 32) tmem_alloc(&tbase, M::COLS);
  Line<P>::load_table(smem, args[items[0].x].twiddles);  // every item has this P
  if (threadIdx.x == 0) mbar_init(&ybar);
  __syncthreads();
  uint32_t yphase = 0;
  int jcur = -1, cur = -1;
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    const int2 item = items[it];
    fetch_args(a, args, item.x, cur);
    if (!pass_b_run<P, HALF>(a, item.y, a.pb_blocks, smem, tbase, red, &ybar, state, yphase, item.x,
                             jcur, chirp_global != 0)) {
      if (threadIdx.x == 0)
        for (int p = 0; p < nprob; ++p) atomicOr(args[p].err, 1ull);
      break;
    }
  }
  __syncthreads();
  if (threadIdx.x < 32) tmem_free(tbase, M::COLS);
}

// T of the last round's column groups of a split last round: the slots of every block whose items
// met the group, added in block order, then T = ext S (+ T) (+ w_ref r_ref) as in k_pass_b.
// blockIdx.x: the group, blockIdx.y: a share of its values.  What bounds it is latency: two dozen
// loads in a row at most.  The run of blocks is found once per thread; with the whole grid walked
// and three 64-bit divisions a block and value it took 55 us for 8 items in 152 blocks, now 3 us.
template <int P>
__global__ void k_pass_b_tail(PassArgs a, int nblocks) {
  constexpr int C = ColCfg<P>::C;
  const int n = a.n;
  const int ngroups = (n + C - 1) / C;
  const int rounds = ngroups / nblocks, tail = ngroups - rounds * nblocks;
  const long long per = (long long)a.J * a.nk, titems = (long long)tail * per;
  const int tg = blockIdx.x;
  if (tg >= tail) return;
  const int cg = rounds * nblocks + tg;
  const SplitRun run = split_run(titems, nblocks, per, tg);
  const bool gaps = titems < nblocks;  // blocks without an item
  for (int e = blockIdx.y * blockDim.x + threadIdx.x; e < n * C; e += gridDim.y * blockDim.x) {
    const int rr = e / C, g = e % C, col = cg * C + g;
    float2 S = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int b = run.first; b <= run.last; ++b) {
      if (gaps && split_begin(titems, nblocks, b) == split_begin(titems, nblocks, b + 1)) continue;
      const int slot = b == run.first ? run.slot : 0;
      S = cadd(S, a.tpart[((long long)b * a.tslots + slot) * n * C + e]);
    }
    if (col < n) {
      const long long ie = (long long)rr * n + col;
      float2 acc = cscale(S, a.ext);
      if (a.tq_accumulate) acc = cadd(acc, a.tq[ie]);
      if (a.rref) {
        const float2 q = __ldg(a.rref + ie);
        acc.x = fmaf(a.wref, q.x, acc.x);
        acc.y = fmaf(a.wref, q.y, acc.y);
      }
      a.tq[ie] = acc;
    }
  }
}

// ------------------------------------------------------------------ launchers

inline int sm_count() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
  }
  return sms;
}

// Persistent grid: as many blocks as can be resident at once, capped by the work.
template <class K>
int persistent_blocks(K kernel, int threads, size_t smem, long long items) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  long long b = (long long)per_sm * sm_count();
  if (items < b) b = items;
  return (int)(b < 1 ? 1 : b);
}

// Persistent grid of a multi-problem launch: per_sm (or as many as fit) blocks per SM,
// capped by the items.
template <class K>
int multi_blocks(K kernel, int threads, size_t smem, int nitems, int per_sm) {
  int fit = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kernel, threads, smem) != cudaSuccess ||
      fit < 1) {
    cudaGetLastError();
    fit = 1;
  }
  const int b = (per_sm > 0 && per_sm < fit ? per_sm : fit) * sm_count();
  return b < nitems ? b : (nitems > 0 ? nitems : 1);
}

template <int P, bool COLS>
cudaError_t launch_lines(const LineArgs& args, const float2* tw, cudaStream_t s) {
  constexpr int G = COLS ? DColCfg<P>::C : RowCfg<P>::G;
  constexpr int NT = COLS ? DColCfg<P>::NT : RowCfg<P>::NT;
  constexpr size_t SM = COLS ? DColCfg<P>::SMEM_BYTES : RowCfg<P>::SMEM_BYTES;
  LineArgs a = args;
  a.step[0] = 0;
  for (int i = 0; i < a.S; ++i) a.step[i + 1] = a.step[i] + (a.src[i].nlines + G - 1) / G;
  if (a.step[a.S] <= 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(k_line_dstep<P, COLS>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SM);
  if (e != cudaSuccess) return e;
  const int nb = persistent_blocks(k_line_dstep<P, COLS>, NT, SM, a.step[a.S]);
  k_line_dstep<P, COLS><<<nb, NT, SM, s>>>(a, tw);
  return cudaGetLastError();
}

template <int P>
cudaError_t launch_rows(const LineArgs& a, const float2* tw, cudaStream_t s) {
  return launch_lines<P, false>(a, tw, s);
}
template <int P>
cudaError_t launch_cols(const LineArgs& a, const float2* tw, cudaStream_t s) {
  return launch_lines<P, true>(a, tw, s);
}


template <int P, bool HALF, bool PASS_C>
cudaError_t launch_rows_form(const PassArgs& a, cudaStream_t s) {
  using R = RowCfg<P>;
  const int steps = a.seg_step[a.J];
  if (steps <= 0) return cudaSuccess;
  auto kern = k_rows<P, HALF, PASS_C>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)R::SMEM_BYTES);
  if (e != cudaSuccess) return e;
  const int nb = multi_blocks(kern, R::NT, R::SMEM_BYTES, steps, a.row_per_sm);
  kern<<<nb, R::NT, R::SMEM_BYTES, s>>>(a);
  return cudaGetLastError();
}

// Problems with n = P/2 and no probe shifts run the HALF forms of the passes.
template <int P>
bool use_half(const PassArgs& a) {
  return half_form_ok<P>() && 2 * a.n == P && !a.ramp_x;
}

template <int P, bool PASS_C>
cudaError_t launch_pass_rows(const PassArgs& a, cudaStream_t s) {
  if constexpr (half_form_ok<P>())
    if (use_half<P>(a)) return launch_rows_form<P, true, PASS_C>(a, s);
  return launch_rows_form<P, false, PASS_C>(a, s);
}

template <int P>
int half_form(int n, int shift) {
  return half_form_ok<P>() && 2 * n == P && !shift ? 1 : 0;
}

template <int P>
int pass_b_groups(int n) {
  return (n + ColCfg<P>::C - 1) / ColCfg<P>::C;
}

inline int max_dynamic_smem() {
  static int v = 0;
  if (!v) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (v <= 0) v = 48 * 1024;
  }
  return v;
}

inline int max_sm_smem() {
  static int v = 0;
  if (!v) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (v <= 0) v = 48 * 1024;
  }
  return v;
}

template <int P>
cudaError_t launch_cols_sum(const SumArgs& a, const float2* tw, cudaStream_t s) {
  using Cc = DColCfg<P>;
  if (a.S < 1 || a.S > kMaxSumSources) return cudaErrorNotSupported;
  const size_t sm = (size_t)(SmemHead<P>::TAB + Cc::C * Cc::LS) * sizeof(float2);
  cudaError_t e = cudaFuncSetAttribute(k_cols_sum<P>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sm);
  if (e != cudaSuccess) return e;
  const int nb = persistent_blocks(k_cols_sum<P>, Cc::NT, sm, (P + Cc::C - 1) / Cc::C);
  k_cols_sum<P><<<nb, Cc::NT, sm, s>>>(a, tw);
  return cudaGetLastError();
}

// Resident blocks per SM of pass B with an `rows`-row Y stage (0: plain loads): what fits in
// registers, shared memory and tensor memory.  0: the stage does not fit.  (Counted here: the
// runtime's occupancy query answers 1 for every kernel that allocates tensor memory.)
template <int P, bool HALF>
int pass_b_fit(int rows, bool chirp_global) {
  using Cc = ColCfg<P>;
  const size_t sm = pass_b_smem<P, HALF>(rows, chirp_global);
  if (sm > (size_t)max_dynamic_smem()) return 0;
  // (registers and static shared memory of the kernel, the same on every device: asked for once)
  static std::atomic<int> regs{0}, fixed{0};
  if (regs.load(std::memory_order_acquire) < 1) {
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, k_pass_b<P, HALF>) != cudaSuccess || fa.numRegs < 1) {
      cudaGetLastError();
      return 1;
    }
    fixed.store((int)fa.sharedSizeBytes, std::memory_order_relaxed);
    regs.store(fa.numRegs, std::memory_order_release);
  }
  const int warps = (Cc::NT + 31) / 32;
  const int by_regs = 65536 / ((regs.load() + 7) / 8 * 256 * warps);
  const int by_smem = (int)((size_t)max_sm_smem() / (sm + fixed.load() + 1024));
  const int b = std::min({by_regs, by_smem, PassBMem<P, HALF>::MAXB, 64 / warps, 32});
  return b < 1 ? 1 : b;
}
// Whether the general forms read the chirp from global memory: where a Y stage has room for more
// resident blocks without it in shared memory.  That is the case from P = 2048 for boxes of more
// than about P/4 rows, which had no stage before: pass B of 2050^2 on 4096^2, 8 x 4 planes, 3535 ->
// 2550 us, of 1218^2 on 2048^2, 24 x 3 planes, 2077 -> 1815 us.
template <int P, bool HALF>
bool pass_b_chirp_global(int rows) {
  return PassBMem<P, HALF>::CHIRP_ANY && rows > 0 &&
         pass_b_fit<P, HALF>(rows, false) < pass_b_fit<P, HALF>(rows, true);
}
template <int P, bool HALF>
int pass_b_per_sm(int rows) {
  return pass_b_fit<P, HALF>(rows, pass_b_chirp_global<P, HALF>(rows));
}
template <int P>
int pass_b_per_sm_form(int half, int rows) {
  if constexpr (half_form_ok<P>())
    if (half) return pass_b_per_sm<P, true>(rows);
  return pass_b_per_sm<P, false>(rows);
}

// The persistent grid of pass B (half: the HALF form; rows: box rows of the Y stage).
template <int P>
int pass_b_blocks(int items, int half, int rows) {
  const long long b = (long long)pass_b_per_sm_form<P>(half, rows) * sm_count();
  return (int)(items < b ? items : b);
}

// The Y stage is used from P = 1024 where the box is at most 256 floats wide, the shared memory fits
// and pass B keeps three quarters of its resident blocks per SM, at P = 4096 any.  Loads of Y without
// it wait where they are issued, and at P = 4096 they are pieces of 16 bytes that get slower the more
// memory a chunk covers: full-grid boxes of 2048^2 on 4096^2, 60 x 4 planes, 51.2 ms with two blocks
// without the stage, 35.2 with one and the stage (12 x 4 planes: 7.6, 7.2); 4096^2 on 4096^2, 24 x 3
// planes, 24.1 and 19.4 (2 x 2 planes: 1.34, 1.57).  512^2 on 1024^2 with full-grid boxes, 40 x 4
// planes, four blocks 1.36 ms, three and the stage 1.16.  At P = 2048, where one block with the stage
// would replace two without, 2048^2 on 2048^2, 60 x 3 planes, took 13.0 ms against 10.6.
template <int P>
int pass_b_stage_ok(int half, int rows) {
  if (P < 1024 || rows <= 0 || 2 * ColCfg<P>::C > 256) return 0;
  const int b1 = pass_b_per_sm_form<P>(half, rows);
  const int b0 = pass_b_per_sm_form<P>(half, 0);
  return b1 >= 1 && (4 * b1 >= 3 * b0 || P == 4096) ? 1 : 0;
}

template <int P, bool HALF>
cudaError_t launch_pass_b_form(const PassArgs& a, int nblocks, cudaStream_t s) {
  using Cc = ColCfg<P>;
  const int rows = a.ymap ? a.max_box_rows : 0;
  const bool chirp_global = pass_b_chirp_global<P, HALF>(rows);
  const size_t sm = pass_b_smem<P, HALF>(rows, chirp_global);
  // (the largest carveout: the driver's own choice follows the occupancy query above)
  cudaError_t e = cudaFuncSetAttribute(k_pass_b<P, HALF>,
                                       cudaFuncAttributePreferredSharedMemoryCarveout,
                                       cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_pass_b<P, HALF>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  k_pass_b<P, HALF><<<nblocks, Cc::NT, sm, s>>>(a, chirp_global);
  const int ngroups = (a.n + Cc::C - 1) / Cc::C, tail = ngroups - (ngroups / nblocks) * nblocks;
  if (a.adj && a.pb_split && tail > 0) {
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_pass_b_tail<P><<<dim3(tail, (a.n * Cc::C + 511) / 512), 256, 0, s>>>(a, nblocks);
  }
  return cudaGetLastError();
}

template <int P>
cudaError_t launch_pass_b(const PassArgs& a, int nblocks, cudaStream_t s) {
  if constexpr (half_form_ok<P>())
    if (use_half<P>(a)) return launch_pass_b_form<P, true>(a, nblocks, s);
  return launch_pass_b_form<P, false>(a, nblocks, s);
}

template <int P, bool HALF, bool PASS_C>
cudaError_t launch_rows_multi_form(const PassArgs* args, const int2* items, int nitems, int per_sm,
                                   cudaStream_t s) {
  using R = RowCfg<P>;
  if (nitems <= 0) return cudaSuccess;
  auto kern = k_rows_multi<P, HALF, PASS_C>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)R::SMEM_BYTES);
  if (e != cudaSuccess) return e;
  const int nb = multi_blocks(kern, R::NT, R::SMEM_BYTES, nitems, per_sm);
  kern<<<nb, R::NT, R::SMEM_BYTES, s>>>(args, items, nitems);
  return cudaGetLastError();
}

template <int P>
cudaError_t launch_rows_multi(int pass_c, const PassArgs* args, const int2* items, int nitems,
                              int half, int per_sm, cudaStream_t s) {
  if constexpr (half_form_ok<P>()) {
    if (half)
      return pass_c ? launch_rows_multi_form<P, true, true>(args, items, nitems, per_sm, s)
                    : launch_rows_multi_form<P, true, false>(args, items, nitems, per_sm, s);
  }
  return pass_c ? launch_rows_multi_form<P, false, true>(args, items, nitems, per_sm, s)
                : launch_rows_multi_form<P, false, false>(args, items, nitems, per_sm, s);
}

template <int P, bool HALF>
cudaError_t launch_pass_b_multi_form(const PassArgs* args, const int2* items, int nitems,
                                     int nprob, int max_rows, int per_sm, cudaStream_t s) {
  using Cc = ColCfg<P>;
  if (nitems <= 0) return cudaSuccess;
  const bool chirp_global = pass_b_chirp_global<P, HALF>(max_rows);
  const size_t sm = pass_b_smem<P, HALF>(max_rows, chirp_global);
  auto kern = k_pass_b_multi<P, HALF>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                       cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  const int fit = std::max(pass_b_per_sm<P, HALF>(max_rows), 1);  // (registers as k_pass_b's bound)
  const int nb = std::min((per_sm > 0 ? std::min(per_sm, fit) : fit) * sm_count(), nitems);
  kern<<<nb, Cc::NT, sm, s>>>(args, items, nitems, nprob, chirp_global);
  return cudaGetLastError();
}

template <int P>
cudaError_t launch_pass_b_multi(const PassArgs* args, const int2* items, int nitems, int nprob,
                                int half, int max_rows, int per_sm, cudaStream_t s) {
  if constexpr (half_form_ok<P>())
    if (half)
      return launch_pass_b_multi_form<P, true>(args, items, nitems, nprob, max_rows, per_sm, s);
  return launch_pass_b_multi_form<P, false>(args, items, nitems, nprob, max_rows, per_sm, s);
}

template <int P>
const Ops* make_ops() {
  static const Ops ops = {P,
                          launch_rows<P>,
                          launch_cols<P>,
                          launch_pass_rows<P, false>,
                          launch_pass_b<P>,
                          launch_pass_rows<P, true>,
                          half_form<P>,
                          pass_b_groups<P>,
                          pass_b_blocks<P>,
                          pass_b_stage_ok<P>,
                          Line<P>::TAB,
                          ColCfg<P>::C,
                          RowCfg<P>::G,
                          launch_rows_multi<P>,
                          launch_pass_b_multi<P>,
                          launch_cols_sum<P>};
  return &ops;
}

}  // namespace holo

#define HOLO_INSTANTIATE(P) \
  namespace holo {          \
  const Ops* ops_##P() { return make_ops<P>(); } \
  }

// The long lines' passes are compiled in units of their own (in parallel): HOLO_ROWS, HOLO_ROWS_MULTI
// and HOLO_PASS_B with `template` in those units and with `extern template` beside HOLO_INSTANTIATE.
#define HOLO_ROWS(KIND, P)                                                        \
  namespace holo {                                                                \
  KIND cudaError_t launch_pass_rows<P, false>(const PassArgs&, cudaStream_t);     \
  KIND cudaError_t launch_pass_rows<P, true>(const PassArgs&, cudaStream_t);      \
  }
#define HOLO_ROWS_MULTI(KIND, P)                                                              \
  namespace holo {                                                                            \
  KIND cudaError_t launch_rows_multi<P>(int, const PassArgs*, const int2*, int, int, int,     \
                                        cudaStream_t);                                        \
  }
#define HOLO_PASS_B(KIND, P)                                                                  \
  namespace holo {                                                                            \
  KIND int pass_b_blocks<P>(int, int, int);                                                   \
  KIND int pass_b_stage_ok<P>(int, int);                                                      \
  KIND cudaError_t launch_pass_b<P>(const PassArgs&, int, cudaStream_t);                      \
  KIND cudaError_t launch_pass_b_multi<P>(const PassArgs*, const int2*, int, int, int, int,   \
                                          int, cudaStream_t);                                 \
  }
#define HOLO_INSTANTIATE_SPLIT(P)    \
  HOLO_ROWS(extern template, P)       \
  HOLO_ROWS_MULTI(extern template, P) \
  HOLO_PASS_B(extern template, P)     \
  HOLO_INSTANTIATE(P)
