// packed_kernels.cuh - row, column and RK passes of two-dimensional FP32 groups.
//
// The passes of kernels.cuh in the packed arithmetic of packed.cuh.  Physical
// fields and the state keep the row-major order.  A mixed field is stored
// [member][kx / 4][y / 2][kx % 4][y % 2] (complex, the kept x-modes rounded up to
// four columns Wp; the columns W <= kx < Wp hold zeros): the modes of a row pair
// that neighbouring threads hold make up whole 32-byte sectors, so a row pass
// reads and writes the transposed field straight from and to registers, and a
// column pass reads two samples of four neighbouring columns as 64 bytes.
//
// In both passes a transform belongs to the threads of one warp wherever it
// fits one, so that the kernels need no block barriers; rows of more than 1024
// points and columns of more than 512 use the block.
//
// Against the scalar FP32 passes before them (GB300, 2.0 GHz): a 512-point row
// takes 128 SM-cycles per transform instead of 312 and 336 instructions per
// row instead of about 800; a 256-point column 137 instead of 312; the row pass
// of a 4096 x 2048 grid 168 us per launch instead of 344; a step of 64 256^2 and
// 32 512^2 members 4.40 ms instead of 6.03.
#pragma once

#include <type_traits>

#include "kernels.cuh"
#include "packed.cuh"

namespace sbi {
namespace pk {

// ===========================================================================
// Rows
// ===========================================================================
// 16 elements per thread from 256-point rows up.  128 registers (four blocks
// of 128 threads per SM) hold a transform, the running product of a chain and
// the field that multiplies it (32 registers each at 16 elements): the inner
// loop reads no global memory, and shared memory only for the exchange and the
// twiddles.  Shared-memory bandwidth is what bounds these passes.
template <int NX>
struct RowGeo {
  static constexpr int n = NX / 2;
  static constexpr int R = n >= 128 ? 16 : 8;
  static constexpr int T = n / R;                       // threads per row
  static constexpr bool WARP = T <= 32;
  static constexpr int THREADS = 128;
  static constexpr int MAXR = THREADS / T;              // rows per block
  using F = PackedFft<One, n, R, WARP>;
  using E = typename F::E;
  // exchange elements per row; rows that share half a warp lie T 8-byte banks
  // apart; rows of more than a warp also pass their upper half through it
  static constexpr int XLEN = (F::xlen() + 15) / 16 * 16 + (T < 16 ? T : 0);
  static constexpr bool TAB = n <= 256;                 // e^{-2 pi i k / NX}, k < n / 2, in shared memory
  static constexpr int RTW = (F::TW + (TAB ? n / 2 : 0) + 1) / 2 * 2;   // twiddles of a block
};
template <int NX>
__host__ __device__ constexpr size_t row_smem(int rows, int nslots) {
  using G = RowGeo<NX>;
  return 8 * ((size_t)G::RTW + (size_t)rows * (G::XLEN + nslots * G::n));
}
// Passes are launched so that the blocks of one may start, and form what
// depends on constants alone (twiddle tables, multipliers), while the blocks of
// the pass before still run; nothing a pass wrote may be read, and nothing it
// reads written, before this.  Every thread of every block waits: a pass that is
// complete then has all the earlier ones behind it.
__device__ __forceinline__ void wait_for_previous() {
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
}

// The twiddles of a block's transforms and of the packed real transform: from
// shared memory, or (long rows) products of the thread's own e^{-2 pi i j / NX}
// by roots of unity.
template <int NX>
struct RowTwiddles {
  using G = RowGeo<NX>;
  const float2 *table, *tw;
  int j;
  float2 wj;
  __device__ __forceinline__ RowTwiddles(const void* global, float2* shared, int j_)
      : table(shared), tw(reinterpret_cast<const float2*>(global)), j(j_) {
    G::F::fill_twiddles(shared, tw);
    if constexpr (G::TAB) {
      for (int k = threadIdx.x; k < G::n / 2; k += blockDim.x) shared[G::F::TW + k] = __ldg(tw + tw_off(NX) + k);
    } else {
      wj = __ldg(tw + tw_off(NX) + j);
    }
    __syncthreads();
  }
  __device__ __forceinline__ void run(One (&x)[G::R], typename G::E* xs) const {
    G::F::run(x, xs, j, G::F::twiddles(table, j), tw);
  }
  // e^{-2 pi i (j + r T) / NX}; r < R / 2 with j < T, or r >= R / 2
  __device__ __forceinline__ float2 lower(int r) const {
    if constexpr (G::TAB) return table[G::F::TW + j + r * G::T];
    else return r == 0 ? wj : wmul(wj, unit_root(r, 2 * G::R));
  }
  __device__ __forceinline__ float2 upper(int r) const {
    if constexpr (G::TAB) {
      // e(k) = -conj(e(n - k)), n - k = T - j + (R - 1 - r) T; the one k = n / 2
      // (j = 0, r = R / 2) is multiplied by zero: any entry will do
      const int kk = G::T - j + (G::R - 1 - r) * G::T;
      const float2 e = table[G::F::TW + (r == G::R / 2 ? kk & (G::n / 2 - 1) : kk)];
      return make_float2(-e.x, e.y);
    } else {
      return wmul(wj, unit_root(r, 2 * G::R));
    }
  }
  __device__ __forceinline__ float2 any(int r) const {
    if (r == G::R / 2 && j == 0) return make_float2(0.f, -1.f);
    return r < G::R / 2 ? lower(r) : upper(r);
  }
  // Products by roots of unity are formed where they are used: kept across a
  // loop they would take more registers than there are.  Emits nothing.
  __device__ __forceinline__ void renew() {
    if constexpr (!G::TAB) asm volatile("" : "+f"(wj.x), "+f"(wj.y));
  }
};

// the row of this thread's group; an absent or inactive row reads row 0 of
// member 0 and stores nothing
struct Row {
  int member, y;
  bool act;
};
template <int T>
__device__ __forceinline__ Row row_of(int row_begin, int rows_total, int ny, const int* active, int member0) {
  const int q = row_begin + (int)blockIdx.x * (int)(blockDim.x / T) + (int)threadIdx.x / T;
  Row r;
  r.act = q < rows_total;
  r.member = r.act ? q / ny : 0;
  r.y = r.act ? q - r.member * ny : 0;
  if (r.act && active) r.act = active[member0 + r.member] != 0;
  return r;
}
// mixed field at mode 0 of the row; mode k at + mode_at(k)
__device__ __forceinline__ const unsigned long long* mixed_row(const BufRef& b, const Row& w) {
  return reinterpret_cast<const unsigned long long*>(b.ptr) + (long long)w.member * b.stride + (w.y >> 1) * 8 + (w.y & 1);
}
__device__ __forceinline__ long long mode_at(int k, int ny) { return (long long)(k >> 2) * ny * 4 + (k & 3) * 2; }
// physical row as complex pairs (x[2m], x[2m + 1])
__device__ __forceinline__ float2* real_row(const BufRef& b, const Row& w, int n) {
  return reinterpret_cast<float2*>(reinterpret_cast<float*>(b.ptr) + (long long)w.member * b.stride) + (long long)w.y * n;
}

// Input side of the packed inverse real transform of a row: Z[k] =
// X[k] (1 + i w) for k < W, X[n - k]* (1 - i w) for k > n - W, w = e^{2 pi i k / NX}
// (both terms where more than half of the modes are kept).  The inverse of Z
// is taken as the conjugate of the transform of its conjugate: x = Z*.
// The forms of a row by its width: half of the modes kept (W = n / 2, the default,
// every bound known at compile time), fewer, more, or any of these.  In all but
// the last load_modes brings each element's first term, X[k] for r < R / 2 and
// X[n - k] above, and with more than half more_modes adds the second ones.
enum RowForm : int { kAnyWidth = 0, kHalf = 1, kNarrow = 2, kBroad = 3 };
template <int NX, int FORM>
inline constexpr bool kFastRow = FORM != kAnyWidth && RowGeo<NX>::T >= 4;
template <int NX, int FORM>
inline constexpr bool kEveryMode = kFastRow<NX, FORM> && FORM == kHalf;   // no test against W

// whether the first term of element r is a kept mode
template <int NX, int FORM>
__device__ __forceinline__ bool first_kept(int r, int W, int j) {
  constexpr int R = RowGeo<NX>::R, T = RowGeo<NX>::T;
  if (FORM == kNarrow) return (r < R / 2 ? j + r * T : T - j + (R - 1 - r) * T) < W;
  return FORM == kBroad || r != R / 2 || j != 0;      // kHalf: mode n / 2 is not
}
// AHEAD: the loads of the first buffer stand by themselves
template <int NX, int FORM, bool AHEAD>
__device__ __forceinline__ void load_modes(One (&x)[RowGeo<NX>::R], const BufRef* bufs, int nb, const Row& w, int ny,
                                           int W, int j) {
  constexpr int R = RowGeo<NX>::R, T = RowGeo<NX>::T;
  // k = j + r T: X[k] at lo + r step for r < R / 2; n - k = T - j + (R - 1 - r) T
  const int step = T * ny;
  const long long lo = mode_at(j, ny), hi = mode_at(T - j, ny);
  if constexpr (AHEAD) {
    const unsigned long long* src = mixed_row(bufs[0], w);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      x[r].v = 0;
      if (r < R / 2 && first_kept<NX, FORM>(r, W, j)) x[r].v = src[lo + r * step];
      else if (r >= R / 2 && first_kept<NX, FORM>(r, W, j)) x[r].v = src[hi + (R - 1 - r) * step];
    }
#pragma unroll 1
    for (int q = 1; q < nb; ++q) {
      src = mixed_row(bufs[q], w);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (r < R / 2 && first_kept<NX, FORM>(r, W, j)) x[r] = add(x[r], One{src[lo + r * step]});
        else if (r >= R / 2 && first_kept<NX, FORM>(r, W, j)) x[r] = add(x[r], One{src[hi + (R - 1 - r) * step]});
      }
    }
  } else {
#pragma unroll 1
    for (int q = 0; q < nb; ++q) {
      const unsigned long long* src = mixed_row(bufs[q], w);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        One v = both(0.f);
        if (r < R / 2 && first_kept<NX, FORM>(r, W, j)) v.v = src[lo + r * step];
        else if (r >= R / 2 && first_kept<NX, FORM>(r, W, j)) v.v = src[hi + (R - 1 - r) * step];
        x[r] = q == 0 ? v : add(x[r], v);
      }
    }
  }
}
// conj(X (1 + i w)), 1 + i w = (1 + e.y, e.x) with e = w*
__device__ __forceinline__ One twist_low(One x, float2 e) {
  const float f = 1.f + e.y;
  return fma(both(-e.x), swp(x), mul(f2(f, -f), x));
}
// X (1 - i w)*, 1 - i w = (1 - e.y, -e.x)
__device__ __forceinline__ One twist_high(One x, float2 e) { return cmul(x, make_float2(1.f - e.y, e.x)); }
template <int NX>
__device__ __forceinline__ void twist_modes(One (&x)[RowGeo<NX>::R], const RowTwiddles<NX>& t) {
  constexpr int R = RowGeo<NX>::R;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (r < R / 2) x[r] = twist_low(x[r], t.lower(r));
    else x[r] = twist_high(x[r], t.upper(r));
  }
}
// The same for kBroad with the second terms, X[n - k] for r < R / 2 and X[k] above,
// eight elements at a time, each twiddle used for both.  (With both terms of an
// element loaded side by side the rows spilled 200 bytes per thread from 256
// points up.)
template <int NX>
__device__ __forceinline__ void add_second_modes(One (&x)[RowGeo<NX>::R], const BufRef* bufs, int nb, const Row& w, int ny,
                                           int W, int j, const RowTwiddles<NX>& t) {
  constexpr int R = RowGeo<NX>::R, T = RowGeo<NX>::T, B = 8;
  const int step = T * ny;
  const long long lo = mode_at(j, ny), hi = mode_at(T - j, ny);
#pragma unroll
  for (int r0 = 0; r0 < R; r0 += B) {
    One v[B];
#pragma unroll
    for (int i = 0; i < B; ++i) v[i] = both(0.f);
#pragma unroll 1
    for (int q = 0; q < nb; ++q) {
      const unsigned long long* src = mixed_row(bufs[q], w);
#pragma unroll
      for (int i = 0; i < B; ++i) {
        const int r = r0 + i;
        const bool kept = (r < R / 2 ? T - j + (R - 1 - r) * T : j + r * T) < W;
        const One u{kept ? src[r < R / 2 ? hi + (R - 1 - r) * step : lo + r * step] : 0ull};
        v[i] = q == 0 ? u : add(v[i], u);
      }
    }
#pragma unroll
    for (int i = 0; i < B; ++i) {
      const int r = r0 + i;
      const float2 e = r < R / 2 ? t.lower(r) : t.any(r);
      x[r] = r < R / 2 ? add(twist_low(x[r], e), twist_high(v[i], e)) : add(twist_high(x[r], e), twist_low(v[i], e));
    }
  }
}
template <int NX, int FORM>
__device__ __forceinline__ void inverse_input(One (&x)[RowGeo<NX>::R], const BufRef* bufs, int nb, const Row& w, int ny,
                                              int W, int j, const RowTwiddles<NX>& t) {
  using G = RowGeo<NX>;
  constexpr int n = G::n, R = G::R, T = G::T;
  if constexpr (kFastRow<NX, FORM>) {
    load_modes<NX, FORM, false>(x, bufs, nb, w, ny, W, j);
    if constexpr (FORM == kBroad) add_second_modes<NX>(x, bufs, nb, w, ny, W, j, t);
    else twist_modes<NX>(x, t);
  } else {
    // eight elements at a time: sixteen loads without a branch between them (one
    // after the other they made this form two to three times as slow)
    constexpr int B = R < 8 ? R : 8;
#pragma unroll
    for (int r0 = 0; r0 < R; r0 += B) {
      One a[B], b[B];
      auto load = [&](int q, int i, One& va, One& vb) {
        const unsigned long long* src = mixed_row(bufs[q], w);
        const int k = j + (r0 + i) * T, kk = n - k;
        va.v = k < W ? src[mode_at(k, ny)] : 0ull;
        vb.v = k > 0 && kk < W ? src[mode_at(kk, ny)] : 0ull;
      };
#pragma unroll
      for (int i = 0; i < B; ++i) load(0, i, a[i], b[i]);
#pragma unroll 1
      for (int q = 1; q < nb; ++q) {
#pragma unroll
        for (int i = 0; i < B; ++i) {
          One va, vb;
          load(q, i, va, vb);
          a[i] = add(a[i], va);
          b[i] = add(b[i], vb);
        }
      }
#pragma unroll
      for (int i = 0; i < B; ++i) {
        const int r = r0 + i;
        const float2 e = t.any(r);
        const One o = cmul(sub_conj(a[i], b[i]), make_float2(e.x, -e.y));
        x[r] = conj(addi(add_conj(a[i], b[i]), o));
      }
    }
  }
}

// Output side of the packed forward real transform of a row, Z in x: the kept
// modes X[k] = 1/2 (Z[k] + Z[n-k]*) - i/2 e^{-2 pi i k / NX} (Z[k] - Z[n-k]*),
// k = j + r T < W.  Z[n - k] sits in lane (T - j) mod T, register R - 1 - r
// (thread 0: its own register (R - r) mod R): a shuffle, or, for rows of
// several warps, a pass through the exchange buffer.
// Modes first .. first + COUNT - 1 of a thread's R; where the threads of a row
// share the exchange buffer share_modes goes before.
template <int NX, int FORM>
inline constexpr int kKept = kFastRow<NX, FORM> && FORM != kBroad ? RowGeo<NX>::R / 2 : RowGeo<NX>::R;

template <int NX, int FORM>
__device__ __forceinline__ void share_modes(const One (&x)[RowGeo<NX>::R], int W, int j, typename RowGeo<NX>::E* xs) {
  using G = RowGeo<NX>;
  constexpr int n = G::n, R = G::R, T = G::T;
  if constexpr (!G::WARP) {
    // Z[n - k] of the kept modes: the elements above n - W, and Z[0]
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (r == 0 || (kKept<NX, FORM> < R ? r >= R / 2 : (r + 1) * T > n - W)) xs[j + r * T] = x[r].v;
    __syncthreads();
  }
}
template <int NX, int FORM, int COUNT>
__device__ __forceinline__ void kept_modes(const One (&x)[RowGeo<NX>::R], One (&X)[COUNT], int first, int W, int j,
                                           const typename RowGeo<NX>::E* xs, const RowTwiddles<NX>& t) {
  using G = RowGeo<NX>;
  constexpr int n = G::n, R = G::R, T = G::T;
#pragma unroll
  for (int i = 0; i < COUNT; ++i) {
    const int r = first + i;
    if (!kEveryMode<NX, FORM> && r * T >= W) break;
    const int k = j + r * T;
    One zc;
    if constexpr (!G::WARP) {
      zc.v = xs[(n - k) & (n - 1)];
    } else {
      zc = x[(R - r) & (R - 1)];
      if constexpr (T > 1) {
        const float2 a = parts(x[R - 1 - r]);
        const int lane = (T - j) & (T - 1);
        const One o = f2(__shfl_sync(0xffffffffu, a.x, lane, T), __shfl_sync(0xffffffffu, a.y, lane, T));
        if (j != 0) zc = o;
      }
    }
    const float2 e = kFastRow<NX, FORM> && r < R / 2 ? t.lower(r) : t.any(r);
    const One d = cmul(sub_conj(x[r], zc), e);
    X[i] = scale(0.5f, subi(add_conj(x[r], zc), d));
  }
}
template <int NX, int FORM>
__device__ __forceinline__ void store_modes(const One (&x)[RowGeo<NX>::R], const BufRef& dst, const Row& w, int ny,
                                            int W, int j, typename RowGeo<NX>::E* xs, const RowTwiddles<NX>& t) {
  using G = RowGeo<NX>;
  constexpr bool FAST = kFastRow<NX, FORM>;
  constexpr int KEPT = kKept<NX, FORM>, PART = G::R / 2;     // half of them at a time: registers
  share_modes<NX, FORM>(x, W, j, xs);
  unsigned long long* out = const_cast<unsigned long long*>(mixed_row(dst, w));
  const int step = G::T * ny;
  if (FAST) out += mode_at(j, ny);
#pragma unroll
  for (int first = 0; first < KEPT; first += PART) {
    One X[PART];
    kept_modes<NX, FORM>(x, X, first, W, j, xs, t);
    if (w.act) {
#pragma unroll
      for (int i = 0; i < PART; ++i) {
        const int r = first + i;
        if (!kEveryMode<NX, FORM> && j + r * G::T >= W) continue;
        out[FAST ? r * step : mode_at(j + r * G::T, ny)] = X[i].v;
      }
    }
  }
  if constexpr (!G::WARP) __syncthreads();
}

// v *= f^p, one factor after the other
template <int R>
__device__ __forceinline__ void times_field(One (&v)[R], const One (&f)[R], int p) {
#pragma unroll 1
  for (int i = 0; i < p; ++i) {
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = mul(v[r], f[r]);
  }
}

// Chains of one inverse transform and the products formed from it.  blockIdx.y
// takes a segment of the operations: the whole list, or a few products of one
// chain (the inverse transform and the products before them are then formed
// again without being transformed, in the same order and so with the same
// bits), which spreads a pass over few rows across the SMs.  Both directions
// go through the one transform of the loop (instruction cache).  Rows of more than
// half of the modes are compiled for three blocks per SM: with four they spill 96
// bytes per thread (33 members of 256^2, three quarters of the modes, 950 us a step
// of order 5; with three 854).
template <int NX, int FORM>
__global__ void __launch_bounds__(RowGeo<NX>::THREADS, FORM == kBroad ? 3 : 4)
k_packed_row(const __grid_constant__ RowParams p) {
  using G = RowGeo<NX>;
  constexpr int n = G::n, R = G::R, T = G::T;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  auto* xs = reinterpret_cast<typename G::E*>(smem_raw) + G::RTW + (threadIdx.x / T) * G::XLEN;
  const int j = threadIdx.x % T;
  const int ny = p.ny;
  RowTwiddles<NX> t(p.tw, reinterpret_cast<float2*>(smem_raw), j);
  wait_for_previous();
  const Row w = row_of<T>(p.row_begin, p.rows_total, p.ny, p.active, p.member0);
  One run[R], x[R], f[R];
  int held = 0;      // the field in f: 1 eta, 2 delta
  auto hold = [&](int which) {
    if (held == which) return;
    const float2* src = real_row(which == 1 ? p.eta : p.delta, w, n) + j;
#pragma unroll
    for (int r = 0; r < R; ++r) f[r] = f2(src[r * T]);
    held = which;
  };
  const int first = p.seg[blockIdx.y].first, end = p.seg[blockIdx.y].end, begin = p.seg[blockIdx.y].begin;

#pragma unroll 1
  for (int o = begin; o < end; ++o) {
    t.renew();
    const RowOp op = p.ops[o];
    const bool inverse = op.kind == ROP_C2R;
    if (inverse) {
      inverse_input<NX, FORM>(x, p.buf + op.a, op.b, w, ny, p.W, j, t);
    } else {
      const bool running = (op.c & 2) != 0;
      if (o < first && !running) continue;
      if (!running) {
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = run[r];
      }
#pragma unroll 1
      for (int q = 1; q <= 2; ++q) {
        const int e = q == 1 ? op.a : op.b;
        if (e == 0) continue;
        hold(q);
        if (running) times_field<R>(run, f, e);
        else times_field<R>(x, f, e);
      }
      if (o < first) continue;
      if (running) {
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = run[r];
      }
      if (op.coef_f != 1.f) {
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = scale(op.coef_f, x[r]);
      }
    }
    t.run(x, xs);
    if (inverse) {
#pragma unroll
      for (int r = 0; r < R; ++r) run[r] = conj(x[r]);
      if (op.dst != kNone && w.act) {
        float2* out = real_row(p.buf[op.dst], w, n) + j;
#pragma unroll
        for (int r = 0; r < R; ++r) out[r * T] = parts(run[r]);
      }
    } else {
      store_modes<NX, FORM>(x, p.buf[op.dst], w, ny, p.W, j, xs, t);
    }
  }
}

// The pass that needs V, grad eta and grad phi~ of a row at once (ROP_N2,
// ROP_VFW, ROP_WDOT).  grad eta . grad phi~, |grad eta|^2 and |grad phi~|^2 are
// accumulated as the gradients come back from their transforms, in the
// thread's own slots of shared memory; a derivative of eta waits in registers
// for the one of phi~.  The modes of the next transform are loaded ahead of the
// current one.  The quotients are IEEE divisions, correct to half a unit in the
// last place for every operand.  Load latency bounds the pass (a quarter of the
// issue slots used): 8192 rows of 512 points 66 us, of which the divisions are 6.
// It spills 40 to 140 bytes per thread from 256 points up at three blocks per SM
// (168 registers); with four blocks, 128 registers and no loads ahead it took
// 3 us more.
struct RhsOps {
  int8_t src[5];      // inverse transforms in the order eta_x, phi_x, eta_y, phi_y, V (indices into ops)
  int8_t f, sx, sy;   // the operation; sponge products of phi_x and phi_y (-1: none)
};
__device__ __forceinline__ F2 quotient(F2 a, F2 d) {
  const float2 p = parts(a), q = parts(d);
  return f2(__fdiv_rn(p.x, q.x), __fdiv_rn(p.y, q.y));
}
template <int NX, int FORM>
__global__ void __launch_bounds__(RowGeo<NX>::THREADS, 3)
k_packed_rhs(const __grid_constant__ RowParams p, const RhsOps q) {
  using G = RowGeo<NX>;
  constexpr int n = G::n, R = G::R, T = G::T;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int rows = blockDim.x / T, nt = blockDim.x;
  auto* xs = reinterpret_cast<typename G::E*>(smem_raw) + G::RTW;
  unsigned long long* slot = xs + rows * G::XLEN + threadIdx.x;
  xs += (threadIdx.x / T) * G::XLEN;
  auto S = [&](int s, int r) -> F2& { return reinterpret_cast<F2*>(slot)[(s * R + r) * nt]; };
  const int j = threadIdx.x % T;
  const int ny = p.ny;
  RowTwiddles<NX> t(p.tw, reinterpret_cast<float2*>(smem_raw), j);
  wait_for_previous();
  const Row w = row_of<T>(p.row_begin, p.rows_total, p.ny, p.active, p.member0);

  One e[R], x[R];     // e: eta_x until phi_x is there, eta_y until phi_y
#pragma unroll
  for (int r = 0; r < R; ++r) e[r] = both(0.f);
  // steps 0..4: the inverse transforms; the forward ones follow the step that
  // forms their field.  One transform in the loop serves both.
  constexpr bool AHEAD = kFastRow<NX, FORM> && FORM != kBroad;
  One next[AHEAD ? R : 1];
  auto load_ahead = [&](int step) {
    if constexpr (AHEAD)
      load_modes<NX, FORM, true>(next, p.buf + p.ops[q.src[step]].a, p.ops[q.src[step]].b, w, ny, p.W, j);
  };
  load_ahead(0);
  int s = 0, dst = -1;
#pragma unroll 1
  while (true) {
    t.renew();
    const bool forward = dst >= 0;
    const RowOp c = p.ops[q.src[s < 5 ? s : 4]];
    if (!forward) {
      if constexpr (AHEAD) {
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = next[r];
        twist_modes<NX>(x, t);
        if (s < 4) load_ahead(s + 1);
      } else {
        inverse_input<NX, FORM>(x, p.buf + c.a, c.b, w, ny, p.W, j, t);
      }
    }
    t.run(x, xs);
    if (forward) {
      store_modes<NX, FORM>(x, p.buf[dst], w, ny, p.W, j, xs, t);
      dst = -1;
      if (s == 5) return;
      continue;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = conj(x[r]);
    const int step = s++;
    if (step == 0 || step == 2) {
#pragma unroll
      for (int r = 0; r < R; ++r) e[r] = x[r];
      continue;
    }
    if (step < 4) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const F2 h = x[r], g = e[r];
        if (step == 1) {
          S(0, r) = mul(g, g);
          S(1, r) = mul(g, h);
          S(2, r) = mul(h, h);
        } else {
          S(0, r) = fma(g, g, S(0, r));
          S(1, r) = fma(g, h, S(1, r));
          S(2, r) = fma(h, h, S(2, r));
        }
      }
      const int so = step == 1 ? q.sx : q.sy;
      if (so < 0) continue;
      // w grad phi~ of the damping pressure
      const float2* sponge = real_row(p.wgt, w, n) + j;
#pragma unroll
      for (int r = 0; r < R; ++r) x[r] = mul(x[r], f2(__ldg(sponge + r * T)));
      dst = p.ops[so].dst;
      continue;
    }
    if (c.dst != kNone && w.act) {   // physical V
      float2* out = real_row(p.buf[c.dst], w, n) + j;
#pragma unroll
      for (int r = 0; r < R; ++r) out[r * T] = parts(x[r]);
    }
    const RowOp op = p.ops[q.f];
    const float2* eta = p.eta.ptr ? real_row(p.eta, w, n) + j : nullptr;
    const float2* pg = op.kind == ROP_N2 && p.pg ? reinterpret_cast<const float2*>(p.pg) + j : nullptr;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const F2 dot = S(1, r), den = add(both(1.f), S(0, r));
      if (op.kind == ROP_VFW) {
        x[r] = fma(x[r], den, mul(both(-1.f), dot));
        continue;
      }
      const F2 num = add(x[r], dot);
      if (op.kind == ROP_WDOT) {
        x[r] = quotient(num, den);
        continue;
      }
      x[r] = scale(0.5f, sub(quotient(mul(num, num), den), S(2, r)));
      if (eta) x[r] = axpy(-op.coef_f, f2(eta[r * T]), x[r]);
      if (pg) x[r] = sub(x[r], f2(pg[r * T]));
    }
    if (op.kind == ROP_WDOT) {
      if (w.act) {
        float2* out = real_row(p.buf[op.dst], w, n) + j;
#pragma unroll
        for (int r = 0; r < R; ++r) out[r * T] = parts(x[r]);
      }
      return;
    }
    dst = op.dst;
  }
}

// Wide form for launches of few rows: the five inverse transforms of a row at
// once by five copies of its threads, the products by one copy each; the same
// operations in the same order (the same bits).  A set of threads is a warp, or
// the threads of a longer row.
template <int NX>
struct WideRow {
  static constexpr int SET = RowGeo<NX>::WARP ? 32 : RowGeo<NX>::T;
  static constexpr int ROWS = SET / RowGeo<NX>::T;
};
template <int NX>
__host__ __device__ constexpr size_t row_smem_wide() {
  using G = RowGeo<NX>;
  using H = WideRow<NX>;
  return 8 * ((size_t)G::RTW + 5 * (size_t)H::ROWS * (G::XLEN + G::n));
}
template <int NX, int FORM>
__global__ void __launch_bounds__(5 * WideRow<NX>::SET)
k_packed_rhs_wide(const __grid_constant__ RowParams p, const RhsOps q) {
  using G = RowGeo<NX>;
  using H = WideRow<NX>;
  constexpr int n = G::n, R = G::R, T = G::T, SET = H::SET;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int copy = threadIdx.x / SET, lane = threadIdx.x % SET;
  const int j = lane % T;
  auto* xs = reinterpret_cast<typename G::E*>(smem_raw) + G::RTW + (threadIdx.x / T) * G::XLEN;
  F2* slots = reinterpret_cast<F2*>(reinterpret_cast<typename G::E*>(smem_raw) + G::RTW + 5 * H::ROWS * G::XLEN);
  auto S = [&](int s, int r) -> F2& { return slots[(s * R + r) * SET + lane]; };
  const int row = p.row_begin + (int)blockIdx.x * H::ROWS + lane / T;
  Row w;
  w.act = row < p.rows_total;
  w.member = w.act ? row / p.ny : 0;
  w.y = w.act ? row - w.member * p.ny : 0;
  RowTwiddles<NX> t(p.tw, reinterpret_cast<float2*>(smem_raw), j);
  wait_for_previous();
  if (w.act && p.active) w.act = p.active[p.member0 + w.member] != 0;
  One x[R];
  const RowOp c = p.ops[q.src[copy]];
  inverse_input<NX, FORM>(x, p.buf + c.a, c.b, w, p.ny, p.W, j, t);
  t.run(x, xs);
#pragma unroll
  for (int r = 0; r < R; ++r) S(copy, r) = x[r] = conj(x[r]);
  if (c.dst != kNone && w.act) {   // physical V
    float2* out = real_row(p.buf[c.dst], w, n) + j;
#pragma unroll
    for (int r = 0; r < R; ++r) out[r * T] = parts(x[r]);
  }
  __syncthreads();
  // slots in the order of q.src: eta_x, phi_x, eta_y, phi_y, V
  const RowOp op = p.ops[q.f];
  int dst = -1;
  if (copy == 0) {
    const float2* eta = p.eta.ptr ? real_row(p.eta, w, n) + j : nullptr;
    const float2* pg = op.kind == ROP_N2 && p.pg ? reinterpret_cast<const float2*>(p.pg) + j : nullptr;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const F2 ex = S(0, r), px = S(1, r), ey = S(2, r), py = S(3, r), v = S(4, r);
      const F2 dot = fma(ey, py, mul(ex, px)), den = add(both(1.f), fma(ey, ey, mul(ex, ex)));
      if (op.kind == ROP_VFW) {
        x[r] = fma(v, den, mul(both(-1.f), dot));
        continue;
      }
      const F2 num = add(v, dot);
      if (op.kind == ROP_WDOT) {
        x[r] = quotient(num, den);
        continue;
      }
      x[r] = scale(0.5f, sub(quotient(mul(num, num), den), fma(py, py, mul(px, px))));
      if (eta) x[r] = axpy(-op.coef_f, f2(eta[r * T]), x[r]);
      if (pg) x[r] = sub(x[r], f2(pg[r * T]));
    }
    dst = op.dst;
    if (op.kind == ROP_WDOT && w.act) {
      float2* out = real_row(p.buf[op.dst], w, n) + j;
#pragma unroll
      for (int r = 0; r < R; ++r) out[r * T] = parts(x[r]);
    }
  } else if ((copy == 1 || copy == 3) && (copy == 1 ? q.sx : q.sy) >= 0) {
    const float2* sponge = real_row(p.wgt, w, n) + j;
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = mul(x[r], f2(__ldg(sponge + r * T)));
    dst = p.ops[copy == 1 ? q.sx : q.sy].dst;
  }
  if (op.kind == ROP_WDOT) return;           // the whole block
  if (G::WARP && dst < 0) return;            // the whole warp
  t.run(x, xs);
  if (dst < 0) w.act = false;
  store_modes<NX, FORM>(x, p.buf[dst < 0 ? 0 : dst], w, p.ny, p.W, j, xs, t);
}

// ===========================================================================
// RK pass.  blockIdx.y: the elevation (0) or the potential (1); the two need
// nothing from each other, so a thread holds one transform at a time.  Bound by
// memory: a third of the crossing-sea batch of 96 members in 42 us per launch
// (60 before), 5.4 TB/s of the bytes it cannot do without.
// ===========================================================================
template <int NX, int FORM, typename S>
__global__ void __launch_bounds__(RowGeo<NX>::THREADS, 5)
k_packed_rk(const __grid_constant__ RkParams p) {
  using G = RowGeo<NX>;
  using SP = StatePair<S>;
  constexpr int n = G::n, R = G::R, T = G::T;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  auto* xs = reinterpret_cast<typename G::E*>(smem_raw) + G::RTW + (threadIdx.x / T) * G::XLEN;
  const int j = threadIdx.x % T;
  const int ny = p.ny;
  const bool potential = blockIdx.y != 0;
  RowTwiddles<NX> t(p.tw, reinterpret_cast<float2*>(smem_raw), j);
  wait_for_previous();
  const Row w = row_of<T>(p.row_begin, p.rows_total, p.ny, p.active, 0);

  const BufRef& st = potential ? p.phi0 : p.eta0;
  const BufRef& sum = potential ? p.acc_phi : p.acc_eta;
  const long long off = (long long)w.y * NX;
  char* M = reinterpret_cast<char*>(st.ptr) + (w.member * st.stride + off) * 8;     // 8 bytes per value
  char* A = reinterpret_cast<char*>(sum.ptr) + (w.member * sum.stride + off) * 8;
  One x[R];
  bool bad = false;
  if (p.mode == RK_STAGE && !potential) {
    const float2* v = real_row(p.V, w, n) + j;
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = f2(v[r * T]);
  } else if (p.mode != RK_ENTRY) {
    inverse_input<NX, FORM>(x, potential && p.mode != RK_STAGE ? &p.corr_phi : &p.phit, 1, w, ny, p.W, j, t);
    t.run(x, xs);
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = conj(x[r]);
  }
  const float bw = (p.stage == 1 || p.stage == 4) ? 1.f : 2.f;
  const RkScalar cdt = p.cdt, dt6 = p.dt6;
  const bool sums = p.mode == RK_STAGE && p.stage > 1;
  // the state (and sums) of four elements are loaded before any of them is used
  constexpr int B = R < 4 ? R : 4;
#pragma unroll
  for (int r0 = 0; r0 < R; r0 += B) {
    SP st4[B], sum4[B];
#pragma unroll
    for (int i = 0; i < B; ++i) {
      st4[i] = SP::load(M, j + (r0 + i) * T);
      sum4[i] = sums ? SP::load(A, j + (r0 + i) * T) : SP::zero();
    }
#pragma unroll
    for (int i = 0; i < B; ++i) {
      const int r = r0 + i, m = j + r * T;
      const float2 f = parts(x[r]);
      SP e = st4[i];
      if (p.mode == RK_STAGE) {
        SP a = sum4[i];
        a.add(0, bw * f.x);
        a.add(1, bw * f.y);
        if (p.stage < 4) {
          if (w.act) a.store(A, m);
          x[r] = f2(e.template offset<float>(0, cdt, f.x), e.template offset<float>(1, cdt, f.y));
        } else {
          e.add_scaled(0, a, dt6);
          e.add_scaled(1, a, dt6);
          if (w.act) {
            e.store(M, m);
            bad |= !e.finite();
          }
          x[r] = f2(float(e.value(0)), float(e.value(1)));
        }
      } else {
        if (p.mode != RK_ENTRY) {
          e.add(0, f.x);
          e.add(1, f.y);
          if (p.mode == RK_CORRECT && w.act) {   // RK_OFFSET leaves the state unchanged
            e.store(M, m);
            bad |= !e.finite();
          }
        }
        x[r] = f2(float(e.value(0)), float(e.value(1)));
      }
    }
  }
  if (bad && p.nonfinite) *p.nonfinite = 1;
  if (!p.tail) return;
  if (!potential && w.act) {
    float2* ew = real_row(p.eta_w, w, n) + j;
#pragma unroll
    for (int r = 0; r < R; ++r) ew[r * T] = parts(x[r]);
  }
  t.run(x, xs);
  store_modes<NX, FORM>(x, potential ? p.phi_hat : p.eta_hat, w, ny, p.W, j, xs, t);
}

// ===========================================================================
// Columns.  E[k] and O[k], the transforms of a column's even and odd samples
// (one element holds both), give the modes k and k + ny2 as E +- w^k O, w =
// e^{-2 pi i / ny}.
// HALF: every output carries the dealias mask and at most half of the modes
// are kept: of each pair k, k + ny2 only one can be kept, known at compile time
// per register (r < R / 2: mode k), so only that one is formed, summed and
// transformed back, and the sums of both accumulators stay in registers.
// Otherwise the sums of both modes are kept, with 8 elements per thread.
// CI adjacent columns share a group of threads (lane = j CI + c), so that a
// warp reads whole 64-byte (CI = 4) or 32-byte (CI = 2) runs.
// Every input is copied ahead (cp.async) into the thread's own slots of shared
// memory while the one before it is transformed, and the multipliers of an
// input are loaded before its transform: with twelve warps per SM the loads
// would otherwise take 40 % of the time.  No barrier is needed for either.
// ===========================================================================
// 16 elements per thread from 256 points up, except at 1024 points and for both
// modes' sums: 8 there, twice the threads (a step of a 2048 x 1024 sea of order 5,
// 1.12 -> 0.93 ms; 33 members of 256^2 with three quarters of the modes 1.17 ->
// 0.87, eight of 512^2 1.23 -> 0.91).  LONE: the threads of a column by themselves.
template <int NY, bool HALF, bool LONE = false>
struct ColGeo {
  static constexpr int ny2 = NY / 2;
  static constexpr int R = HALF && (ny2 == 128 || ny2 == 256 || ny2 == 1024) ? 16 : (ny2 >= 8 ? 8 : 4);
  static constexpr int T = ny2 / R;
  static constexpr int CI = LONE || T == 128 ? 1 : (T == 16 || T == 64 || (T == 32 && !HALF) ? 2 : 4);
  static constexpr int GT = T * CI;                       // threads per group
  static constexpr bool WARP = GT <= 32;
  static constexpr int THREADS = 128;
  static constexpr int MAXG = THREADS / GT;               // groups per block
  static constexpr int CPB = CI * MAXG;                   // columns per block
  static constexpr int SG = MAXG * CI >= 4 ? MAXG : 4 / CI;   // the same, staged form (whole tiles)
  using F = PackedFft<Two, ny2, R, WARP, CI>;
  using E = typename F::E;
  static constexpr int XLEN = F::xlen() * CI + (GT < 8 ? GT : 0);   // exchange elements per group
  static constexpr int CTW = (F::TW + 1) / 2;             // twiddles of a block, in elements of 16 bytes
  static constexpr bool STAGEABLE = NY >= 32;
};
template <int NY, bool HALF>
__host__ __device__ constexpr size_t packed_col_smem(int groups) {
  using G = ColGeo<NY, HALF>;
  return sizeof(typename G::E) * ((size_t)G::CTW + (size_t)groups * G::XLEN);
}
// the form that copies its inputs ahead
template <int NY, bool HALF>
__host__ __device__ constexpr size_t packed_col_smem_ahead(int groups) {
  using G = ColGeo<NY, HALF>;
  return packed_col_smem<NY, HALF>(groups) + sizeof(typename G::E) * (size_t)G::R * groups * G::GT;
}
// The staged form adds, 128-byte aligned, the block's tiles of four columns
// and one mbarrier per tile.
template <int NY, bool HALF>
__host__ __device__ constexpr size_t packed_col_smem_staged(int groups) {
  return (packed_col_smem<NY, HALF>(groups) + 127) / 128 * 128 +
         (size_t)(groups * ColGeo<NY, HALF>::CI / 4) * (NY * 32 + 8);
}

// a += v f i^q
__device__ __forceinline__ F2 acc_term(F2 a, F2 v, float f, int q) {
  const float g = q < 2 ? f : -f;
  return (q & 1) ? fma(swp(v), f2(-g, g), a) : fma(both(g), v, a);
}
// (v f i^q)*
__device__ __forceinline__ F2 conj_term(F2 v, float f, int q) {
  const float g = q < 2 ? f : -f;
  return (q & 1) ? mul(both(-g), swp(v)) : mul(f2(g, -g), v);
}


template <int NY, int NACC, bool HALF, bool STAGED>
__global__ void __launch_bounds__(STAGED ? ColGeo<NY, HALF>::SG* ColGeo<NY, HALF>::GT : ColGeo<NY, HALF>::THREADS,
                                  STAGED && ColGeo<NY, HALF>::SG > ColGeo<NY, HALF>::MAXG ? 1 : 3)
k_packed_col(const __grid_constant__ ColParams p) {
  using G = ColGeo<NY, HALF>;
  using E = typename G::E;
  using M = Mem<Two>;
  constexpr int R = G::R, T = G::T, CI = G::CI, GT = G::GT, ny2 = G::ny2;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float2* tab2 = reinterpret_cast<float2*>(smem_raw);
  E* sm = reinterpret_cast<E*>(smem_raw) + G::CTW;
  const int g = threadIdx.x / GT, l = threadIdx.x % GT, c = l % CI, j = l / CI;
  const int groups = blockDim.x / GT;
  E* xs = sm + g * G::XLEN + c;
  E* own = sm + groups * G::XLEN + threadIdx.x;   // not STAGED: the next input, [r][thread]
  const float2* tw = reinterpret_cast<const float2*>(p.tw);
  const int col = p.col_begin + ((int)blockIdx.x * groups + g) * CI + c;
  const bool valid = col < p.cols_total;
  const int member = valid ? col / p.W : 0;
  const int kx = valid ? col - member * p.W : 0;
  const long long at0 = ((long long)(kx >> 2) * ny2 + j) * 4 + (kx & 3);   // element r at + 4 T r
  G::F::fill_twiddles(tab2, tw);
  const auto t = G::F::twiddles(tab2, j);
  float2 wj = __ldg(tw + tw_off(NY) + j);   // w^j; w^{j + r T} = w^j e^{-2 pi i r / 2R}
  wait_for_previous();
  const int gave_up = (STAGED && p.err_flag) ? *(volatile int*)p.err_flag : 0;
  const bool act = valid && (p.active == nullptr || p.active[p.member0 + member] != 0);
  auto field = [&](const BufRef& b) {
    return reinterpret_cast<E*>(reinterpret_cast<float2*>(b.ptr) + (long long)member * b.stride) + at0;
  };
  const long long plane = (long long)p.W * ny2;   // table: modes k < ny2, then k + ny2
  auto copy_ahead = [&](int i) {
    if (act) {
      const E* src = field(p.buf[i]);
#pragma unroll
      for (int r = 0; r < R; ++r)
        cp_async_elem(reinterpret_cast<double2*>(own + r * blockDim.x), reinterpret_cast<const double2*>(src + r * T * 4));
    }
    cp_async_commit();
  };
  if (!STAGED && p.nin > 0) copy_ahead(0);

  // staged form: tiles of four columns (one contiguous run) and barriers
  E* stg = nullptr;
  unsigned long long* bar = nullptr;
  constexpr unsigned kTileBytes = 32u * NY;
  bool live = act, issuer = false;
  auto issue = [&](int i) {
    const char* src = reinterpret_cast<const char*>(reinterpret_cast<const float2*>(p.buf[i].ptr) +
                                                    (long long)member * p.buf[i].stride) +
                      (long long)(kx >> 2) * kTileBytes;
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    mbar_expect_tx(bar, kTileBytes + (unsigned)p.stall_tx);
    bulk_copy_g2s(stg, src, kTileBytes, bar);
  };
  if constexpr (STAGED) {
    const int tile = (g * CI + c) / 4, tiles = groups * CI / 4;
    unsigned char* st0 = smem_raw + (packed_col_smem<NY, HALF>(groups) + 127) / 128 * 128;
    stg = reinterpret_cast<E*>(st0 + (size_t)tile * kTileBytes);
    bar = reinterpret_cast<unsigned long long*>(st0 + (size_t)tiles * kTileBytes) + tile;
    if (gave_up) live = false;
    issuer = (g * CI + c) % 4 == 0 && j == 0;
    if (issuer) {
      mbar_init(bar, 1);
      mbar_init_fence();
    }
  }
  __syncthreads();   // twiddles filled, barriers initialised
  if constexpr (STAGED) {
    if (issuer && live && p.nin > 0) issue(0);
  }

  std::conditional_t<HALF, F2, Two> acc[NACC][R];
#pragma unroll
  for (int q = 0; q < NACC; ++q)
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if constexpr (HALF) acc[q][r] = both(0.f);
      else acc[q][r] = Two{both(0.f), both(0.f)};
    }

  float f[HALF ? R : 2 * R];      // multipliers of a term
  auto load_factors = [&](const ColTerm& m) {
    const float* tab = reinterpret_cast<const float*>(m.tab) + at0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      f[r] = __ldg(tab + r * T * 4 + (!HALF || r < R / 2 ? 0 : plane));
      if constexpr (!HALF) f[R + r] = __ldg(tab + r * T * 4 + plane);
    }
  };
  // inputs, then outputs: both directions go through one transform
#pragma unroll 1
  for (int i = 0; i < p.nin + p.nouts; ++i) {
    // the products of wj are formed where they are used, not kept in registers
    asm volatile("" : "+f"(wj.x), "+f"(wj.y));
    Two x[R];
    const bool forward = i < p.nin;
    if (forward) {
      if constexpr (STAGED) {
        if (live) live = mbar_wait_bounded(bar, (unsigned)(i & 1), p.err_flag);
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = M::from(live ? stg[(j + r * T) * 4 + (kx & 3)] : make_ulonglong2(0, 0));
        __syncthreads();   // the staged tiles are read
        if (issuer && live && i + 1 < p.nin) issue(i + 1);
      } else {
        cp_async_wait_all();
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = M::from(act ? own[r * blockDim.x] : make_ulonglong2(0, 0));
        __syncwarp();      // the slots are read before they are filled again
        if (i + 1 < p.nin) copy_ahead(i + 1);
      }
      if (p.term_begin[i] < p.term_begin[i + 1]) load_factors(p.terms[p.term_begin[i]]);
    } else {
      // even samples from the sums of the modes k and k + ny2, odd ones from
      // their differences times w*; the inverse is the conjugate of the
      // transform of the conjugates
      const ColTerm m = p.outs[i - p.nin];
      const float* tab = reinterpret_cast<const float*>(m.tab) + at0;
      const int ph = (m.gx + m.gy) & 3;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float2 w = r == 0 ? wj : wmul(wj, unit_root(r, 2 * R));
        if constexpr (HALF) {
          const float f = __ldg(tab + r * T * 4 + (r < R / 2 ? 0 : plane));
          const F2 e = conj_term(NACC == 1 || m.acc == 0 ? acc[0][r] : acc[NACC - 1][r], f, ph);
          x[r] = Two{e, cmul(e, r < R / 2 ? w : make_float2(-w.x, -w.y))};
        } else {
          const Two b = NACC == 1 || m.acc == 0 ? acc[0][r] : acc[NACC - 1][r];
          const F2 y0 = conj_term(b.a, __ldg(tab + r * T * 4), ph);
          const F2 y1 = conj_term(b.b, __ldg(tab + r * T * 4 + plane), ph);
          x[r] = Two{add(y0, y1), cmul(sub(y0, y1), w)};
        }
      }
    }
    G::F::run(x, xs, j, t, tw);
    if (forward) {
      F2 v[HALF ? R : 1];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float2 w = r == 0 ? wj : wmul(wj, unit_root(r, 2 * R));
        const F2 o = cmul(x[r].b, w);
        if constexpr (HALF) v[r] = r < R / 2 ? add(x[r].a, o) : sub(x[r].a, o);
        else x[r] = Two{add(x[r].a, o), sub(x[r].a, o)};   // modes (k, k + ny2)
      }
      for (int q = p.term_begin[i]; q < p.term_begin[i + 1]; ++q) {
        const ColTerm m = p.terms[q];
        const int ph = (m.gx + m.gy) & 3;
        if (q > p.term_begin[i]) load_factors(m);
        auto sum = [&](auto& a) {
#pragma unroll
          for (int r = 0; r < R; ++r) {
            if constexpr (HALF) a[r] = acc_term(a[r], v[r], f[r], ph);
            else a[r] = Two{acc_term(a[r].a, x[r].a, f[r], ph), acc_term(a[r].b, x[r].b, f[R + r], ph)};
          }
        };
        if (NACC == 1 || m.acc == 0) sum(acc[0]);
        else sum(acc[NACC - 1]);
      }
      continue;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = Two{conj(x[r].a), conj(x[r].b)};
    if (i == p.nin && act) {
#pragma unroll 2
      for (int q = 0; q < p.npass; ++q) {
        const E* ps = field(p.pass[q]);
        E v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = ps[r * T * 4];
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = add(x[r], M::from(v[r]));
      }
    }
    if (act) {
      E* dst = field(p.buf[p.outs[i - p.nin].in]);
#pragma unroll
      for (int r = 0; r < R; ++r) dst[r * T * 4] = M::to(x[r]);
    }
  }
}

__device__ __forceinline__ void copy_float_ahead(float* dst_smem, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem_u32(dst_smem)), "l"(src) : "memory");
}
// Wide form, for launches of few columns: the threads of a
// set of columns (one warp, or the block's 128 threads where a transform needs
// them) are there p.wide times, each copy transforms its share of the inputs,
// leaves their modes in shared memory, and after one barrier every thread
// sums some modes over all inputs, in the order of the other forms and with the
// same operations (the same bits); the outputs are shared out the same way.
// A pass of eight inputs and one output then takes the time of two transforms
// instead of nine.  Column passes of one 512^2 member: 0.38 ms a step (0.58 in
// the plain form; 0.44 with the multipliers loaded where they are used).
// Columns of 1024 and 2048 points stand alone here, on twice the blocks: a step of a
// 256 x 2048 sea of order 5 0.65 -> 0.47 ms, of 256 x 1024 0.57 -> 0.39.
template <int NY, bool HALF>
struct WideGeo {
  using G = ColGeo<NY, HALF, ColGeo<NY, HALF>::T == 64>;
  static constexpr int SET = G::WARP ? 32 : G::GT;      // threads of one copy
  static constexpr int COLS = G::CI * (SET / G::GT);    // columns of a block
  static constexpr int SX = G::XLEN * (SET / G::GT);    // exchange elements of one copy
};
template <int NY, bool HALF>
__host__ __device__ constexpr size_t packed_col_smem_wide(int copies, int nin, int nterms, int nacc, int npass) {
  using H = WideGeo<NY, HALF>;
  using G = typename H::G;
  const size_t NM = (HALF ? 1 : 2) * G::R;
  const size_t modes = (8 * (size_t)nin + 4 * (size_t)nterms) * NM * H::SET, pass = 16 * (size_t)npass * G::R * H::SET;
  return 16 * ((size_t)G::CTW + (size_t)copies * H::SX) + 8 * (size_t)nacc * NM * H::SET + (modes > pass ? modes : pass);
}
// A thread's modes: HALF the R that can be kept (j + r T, from r = R / 2 on plus
// NY / 2), else j + r T and, from R on, those plus NY / 2.
template <int NY, bool HALF>
__global__ void __launch_bounds__(WideGeo<NY, HALF>::G::WARP ? 256 : 512)
k_packed_col_wide(const __grid_constant__ ColParams p) {
  using H = WideGeo<NY, HALF>;
  using G = typename H::G;
  using E = typename G::E;
  using M = Mem<Two>;
  constexpr int R = G::R, T = G::T, CI = G::CI, GT = G::GT, ny2 = G::ny2, SET = H::SET;
  constexpr int NM = HALF ? R : 2 * R, UP = HALF ? R / 2 : R;   // modes, the first one of the upper plane
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int copies = blockDim.x / SET, copy = threadIdx.x / SET, lane = threadIdx.x % SET;
  const int g = lane / GT, l = lane % GT, c = l % CI, j = l / CI;
  float2* tab2 = reinterpret_cast<float2*>(smem_raw);
  E* xs0 = reinterpret_cast<E*>(smem_raw) + G::CTW;
  E* xs = xs0 + (size_t)copy * H::SX + g * G::XLEN + c;
  F2* sums = reinterpret_cast<F2*>(xs0 + (size_t)copies * H::SX);              // [acc][r][lane]
  F2* modes = sums + (size_t)p.nacc * NM * SET;                                 // [input][r][lane]
  float* factors = reinterpret_cast<float*>(modes + (size_t)p.nin * NM * SET);  // [term][r][lane]
  E* passed = reinterpret_cast<E*>(modes);                                     // later: [pass][r][lane]
  const float2* tw = reinterpret_cast<const float2*>(p.tw);
  const int col = p.col_begin + (int)blockIdx.x * H::COLS + g * CI + c;
  const bool valid = col < p.cols_total;
  const int member = valid ? col / p.W : 0;
  const int kx = valid ? col - member * p.W : 0;
  const long long at0 = ((long long)(kx >> 2) * ny2 + j) * 4 + (kx & 3);
  bool act = valid;
  auto field = [&](const BufRef& b) {
    return reinterpret_cast<E*>(reinterpret_cast<float2*>(b.ptr) + (long long)member * b.stride) + at0;
  };
  const long long plane = (long long)p.W * ny2;
  Two x[R];
  auto load = [&](int i) {
    const E* src = field(p.buf[i]);
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = M::from(act ? src[r * T * 4] : make_ulonglong2(0, 0));
  };
  // the multipliers of an input's terms, for the sums
  auto load_factors = [&](int i) {
    for (int q = p.term_begin[i]; q < p.term_begin[i + 1]; ++q) {
      const float* tab = reinterpret_cast<const float*>(p.terms[q].tab) + at0;
#pragma unroll
      for (int r = 0; r < NM; ++r)
        copy_float_ahead(factors + (q * NM + r) * SET + lane, tab + r % R * T * 4 + (r < UP ? 0 : plane));
    }
    cp_async_commit();
  };
  if (copy < p.nin) load_factors(copy);
  G::F::fill_twiddles(tab2, tw);
  const auto t = G::F::twiddles(tab2, j);
  float2 wj = __ldg(tw + tw_off(NY) + j);
  wait_for_previous();
  act = valid && (p.active == nullptr || p.active[p.member0 + member] != 0);
  if (copy < p.nin) {
    load(copy);
  } else {
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = Two{both(0.f), both(0.f)};
  }
  __syncthreads();
#pragma unroll 1
  for (int i0 = 0; i0 < p.nin; i0 += copies) {     // the same trips for every copy
    asm volatile("" : "+f"(wj.x), "+f"(wj.y));
    const int i = i0 + copy;
    if (i0 > 0 && i < p.nin) {
      load(i);
      load_factors(i);
    }
    if (!G::WARP || i < p.nin) G::F::run(x, xs, j, t, tw);   // a set of several warps has block barriers in it
    if (i < p.nin) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float2 w = r == 0 ? wj : wmul(wj, unit_root(r, 2 * R));
        const F2 o = cmul(x[r].b, w);
        if (HALF) {
          modes[(i * NM + r) * SET + lane] = r < UP ? add(x[r].a, o) : sub(x[r].a, o);
        } else {
          modes[(i * NM + r) * SET + lane] = add(x[r].a, o);
          modes[(i * NM + R + r) * SET + lane] = sub(x[r].a, o);
        }
      }
    }
  }
  // the multipliers of this copy's first output
  float fo[NM];
  if (copy < p.nouts) {
    const float* tab = reinterpret_cast<const float*>(p.outs[copy].tab) + at0;
#pragma unroll
    for (int r = 0; r < NM; ++r) fo[r] = __ldg(tab + r % R * T * 4 + (r < UP ? 0 : plane));
  }
  cp_async_wait_all();
  __syncthreads();
  // copy k sums the modes r = k, k + copies, .., four at a time: their loads
  // from shared memory overlap
  for (int r0 = copy; r0 < NM; r0 += 4 * copies) {
    F2 a0[4], a1[4];
#pragma unroll
    for (int c4 = 0; c4 < 4; ++c4) a0[c4] = a1[c4] = both(0.f);
    for (int i = 0; i < p.nin; ++i) {
      F2 v[4];
#pragma unroll
      for (int c4 = 0; c4 < 4; ++c4) v[c4] = modes[(i * NM + min(r0 + c4 * copies, NM - 1)) * SET + lane];
      for (int q = p.term_begin[i]; q < p.term_begin[i + 1]; ++q) {
        const ColTerm m = p.terms[q];
        const int ph = (m.gx + m.gy) & 3;
        float f[4];
#pragma unroll
        for (int c4 = 0; c4 < 4; ++c4) f[c4] = factors[(q * NM + min(r0 + c4 * copies, NM - 1)) * SET + lane];
#pragma unroll
        for (int c4 = 0; c4 < 4; ++c4) {
          if (m.acc == 0) a0[c4] = acc_term(a0[c4], v[c4], f[c4], ph);
          else a1[c4] = acc_term(a1[c4], v[c4], f[c4], ph);
        }
      }
    }
#pragma unroll
    for (int c4 = 0; c4 < 4; ++c4) {
      const int r = r0 + c4 * copies;
      if (r < NM) {
        sums[r * SET + lane] = a0[c4];
        if (p.nacc > 1) sums[(NM + r) * SET + lane] = a1[c4];
      }
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int o0 = 0; o0 < p.nouts; o0 += copies) {
    asm volatile("" : "+f"(wj.x), "+f"(wj.y));
    const int o = o0 + copy;
    const ColTerm m = p.outs[o < p.nouts ? o : 0];
    if (o == 0 && act) {
      for (int q = 0; q < p.npass; ++q) {
        const E* ps = field(p.pass[q]);
#pragma unroll
        for (int r = 0; r < R; ++r)
          cp_async_elem(reinterpret_cast<double2*>(passed + (q * R + r) * SET + lane),
                        reinterpret_cast<const double2*>(ps + r * T * 4));
      }
      cp_async_commit();
    }
    if (o < p.nouts) {
      const float* tab = reinterpret_cast<const float*>(m.tab) + at0;
      const int ph = (m.gx + m.gy) & 3;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float2 w = r == 0 ? wj : wmul(wj, unit_root(r, 2 * R));
        const F2* sum = sums + ((m.acc ? NM : 0) + r) * SET + lane;
        if (HALF) {
          const float f = o0 == 0 ? fo[r] : __ldg(tab + r * T * 4 + (r < UP ? 0 : plane));
          const F2 e = conj_term(*sum, f, ph);
          x[r] = Two{e, cmul(e, r < UP ? w : make_float2(-w.x, -w.y))};
        } else {
          const F2 y0 = conj_term(*sum, o0 == 0 ? fo[r] : __ldg(tab + r * T * 4), ph);
          const F2 y1 = conj_term(sum[R * SET], o0 == 0 ? fo[NM - R + r] : __ldg(tab + r * T * 4 + plane), ph);
          x[r] = Two{add(y0, y1), cmul(sub(y0, y1), w)};
        }
      }
    }
    if (!G::WARP || o < p.nouts) G::F::run(x, xs, j, t, tw);
    if (o < p.nouts && act) {
#pragma unroll
      for (int r = 0; r < R; ++r) x[r] = Two{conj(x[r].a), conj(x[r].b)};
      if (o == 0) {
        cp_async_wait_all();
        for (int q = 0; q < p.npass; ++q) {
#pragma unroll
          for (int r = 0; r < R; ++r) x[r] = add(x[r], M::from(passed[(q * R + r) * SET + lane]));
        }
      }
      E* dst = field(p.buf[m.in]);
#pragma unroll
      for (int r = 0; r < R; ++r) dst[r * T * 4] = M::to(x[r]);
    }
  }
}

// ===========================================================================
// Launchers
// ===========================================================================
// Launches a pass; chained: behind another pass of the same stream, which it may
// overlap up to its wait_for_previous().
template <typename... P, typename... A>
cudaError_t launch(void (*k)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, bool chained, const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, args...);
}

inline bool rhs_ops(const RowParams& p, RhsOps* q) {
  int slot_op[kMaxSlots] = {-1, -1, -1, -1, -1};
  *q = RhsOps{{-1, -1, -1, -1, -1}, -1, -1, -1};
  for (int o = 0; o < p.nops; ++o) {
    const RowOp& op = p.ops[o];
    if (op.kind == ROP_C2R) slot_op[op.slot] = o;
    else if (op.kind != ROP_PROD) q->f = (int8_t)o;
    else if (op.slot == 3) q->sx = (int8_t)o;
    else if (op.slot == 4) q->sy = (int8_t)o;
  }
  if (q->f < 0) return false;
  const int s = p.ops[q->f].slot;
  if (s != 0 || p.ops[q->f].a != 2) return false;
  const int order[5] = {1, 3, 2, 4, 0};   // slots: V, eta_x, eta_y, phi_x, phi_y
  for (int i = 0; i < 5; ++i) {
    q->src[i] = (int8_t)slot_op[order[i]];
    if (q->src[i] < 0) return false;
  }
  return true;
}

// calls f with the form of rows that keep W modes
template <int NX, typename F>
cudaError_t with_form(int W, F f) {
  using G = RowGeo<NX>;
  if (2 * W == G::n) return f(std::integral_constant<int, kHalf>());
  if constexpr (G::T < 4) return f(std::integral_constant<int, kAnyWidth>());
  else return 2 * W < G::n ? f(std::integral_constant<int, kNarrow>()) : f(std::integral_constant<int, kBroad>());
}

template <int NX>
cudaError_t launch_packed_row_n(const RowParams& p, cudaStream_t st, bool chained) {
  using G = RowGeo<NX>;
  if (p.rpc < 1 || p.rpc > G::MAXR || (p.rpc * G::T) % 32 || p.row_begin < 0 || p.row_begin >= p.rows_total)
    return cudaErrorInvalidValue;
  const unsigned blocks = (unsigned)((p.rows_total - p.row_begin + p.rpc - 1) / p.rpc);
  const int threads = p.rpc * G::T;
  RowParams q = p;
  return with_form<NX>(p.W, [&](auto form) {
    constexpr int FORM = decltype(form)::value;
    if (p.nslots > 1) {
      RhsOps r;
      if (!rhs_ops(q, &r)) return cudaErrorInvalidValue;
      if (p.split > 0) {
        const unsigned wb = (unsigned)((p.rows_total - p.row_begin + WideRow<NX>::ROWS - 1) / WideRow<NX>::ROWS);
        return launch(k_packed_rhs_wide<NX, FORM>, wb, 5 * WideRow<NX>::SET, row_smem_wide<NX>(), st, chained, q, r);
      }
      return launch(k_packed_rhs<NX, FORM>, blocks, threads, row_smem<NX>(p.rpc, 3), st, chained, q, r);
    }
    const int ns = q.nops > 0 && q.ops[0].kind == ROP_C2R ? make_segments(q, p.split) : 0;
    if (ns == 0) return cudaErrorInvalidValue;
    return launch(k_packed_row<NX, FORM>, dim3(blocks, (unsigned)ns), threads, row_smem<NX>(p.rpc, 0), st, chained, q);
  });
}

template <int NX>
cudaError_t launch_packed_rk_n(const RkParams& p, cudaStream_t st, bool chained) {
  using G = RowGeo<NX>;
  if (p.row_begin < 0 || p.row_begin >= p.rows_total) return cudaErrorInvalidValue;
  const dim3 grid((unsigned)((p.rows_total - p.row_begin + G::MAXR - 1) / G::MAXR), 2);
  return with_form<NX>(p.W, [&](auto form) {
    constexpr int FORM = decltype(form)::value;
    return launch(p.state64 ? k_packed_rk<NX, FORM, double> : k_packed_rk<NX, FORM, float>, grid, G::THREADS,
                  row_smem<NX>(G::MAXR, 0), st, chained, p);
  });
}

// every output carries the dealias mask and at most half of the modes are kept
inline bool col_half(const ColParams& p) {
  bool half = p.ky_keep <= p.ny / 4;
  for (int o = 0; o < p.nouts; ++o) half = half && p.outs[o].mask == 1;
  return half;
}
// largest number of copies the wide form of a pass can take (0: none)
template <int NY, bool HALF>
int col_most_wide(const ColParams& p) {
  if (p.staged) return 0;
  const int most = (ColGeo<NY, HALF>::WARP ? 256 : 512) / WideGeo<NY, HALF>::SET;
  for (int k = most; k >= 2; k /= 2)
    if (packed_col_smem_wide<NY, HALF>(k, p.nin, p.nterms, p.nacc, p.npass) <= 227 * 1024) return k;
  return 0;
}

template <int NY, int NACC, bool HALF>
cudaError_t launch_packed_col_a(const ColParams& p, int groups, unsigned blocks, cudaStream_t st, bool chained) {
  using G = ColGeo<NY, HALF>;
  if (!p.staged)
    return launch(k_packed_col<NY, NACC, HALF, false>, blocks, groups * G::GT,
                  packed_col_smem_ahead<NY, HALF>(groups), st, chained, p);
  if constexpr (G::STAGEABLE)
    return launch(k_packed_col<NY, NACC, HALF, true>, blocks, groups * G::GT,
                  packed_col_smem_staged<NY, HALF>(groups), st, chained, p);
  return cudaErrorInvalidValue;
}

template <int NY, bool HALF>
cudaError_t launch_packed_col_h(const ColParams& p, cudaStream_t st, bool chained) {
  using G = ColGeo<NY, HALF>;
  const int most = p.staged ? G::SG : G::MAXG;
  const int cpb = p.cpb > 0 ? p.cpb : most * G::CI;
  const int groups = cpb / G::CI;
  if (cpb % G::CI || groups < 1 || groups > most || (groups * G::GT) % 32 || (p.staged && cpb % 4) ||
      p.col_begin < 0 || p.col_begin % 4 || p.col_begin >= p.cols_total || p.W % 4 || p.nacc < 1 ||
      p.nacc > kMaxColAcc)
    return cudaErrorInvalidValue;
  const unsigned blocks = (unsigned)((p.cols_total - p.col_begin + cpb - 1) / cpb);
  if (p.wide > 0) {
    using H = WideGeo<NY, HALF>;
    const size_t smem = packed_col_smem_wide<NY, HALF>(p.wide, p.nin, p.nterms, p.nacc, p.npass);
    if (p.staged || p.wide * H::SET > (G::WARP ? 256 : 512) || smem > 227 * 1024) return cudaErrorInvalidValue;
    const unsigned wb = (unsigned)((p.cols_total - p.col_begin + H::COLS - 1) / H::COLS);
    return launch(k_packed_col_wide<NY, HALF>, wb, p.wide * H::SET, smem, st, chained, p);
  }
  return p.nacc == 1 ? launch_packed_col_a<NY, 1, HALF>(p, groups, blocks, st, chained)
                     : launch_packed_col_a<NY, 2, HALF>(p, groups, blocks, st, chained);
}
template <int NY>
cudaError_t launch_packed_col_n(const ColParams& p, cudaStream_t st, bool chained) {
  return col_half(p) ? launch_packed_col_h<NY, true>(p, st, chained) : launch_packed_col_h<NY, false>(p, st, chained);
}

template <typename K>
cudaError_t allow_smem(K k, size_t bytes) {
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
template <int NX>
cudaError_t prepare_packed_row_n() {
  using G = RowGeo<NX>;
  auto prepare = [](auto form) {
    constexpr int FORM = decltype(form)::value;
    cudaError_t e = allow_smem(k_packed_row<NX, FORM>, row_smem<NX>(G::MAXR, 0));
    if (e == cudaSuccess) e = allow_smem(k_packed_rhs<NX, FORM>, row_smem<NX>(G::MAXR, 3));
    if (e == cudaSuccess) e = allow_smem(k_packed_rhs_wide<NX, FORM>, row_smem_wide<NX>());
    if (e == cudaSuccess) e = allow_smem(k_packed_rk<NX, FORM, float>, row_smem<NX>(G::MAXR, 0));
    if (e == cudaSuccess) e = allow_smem(k_packed_rk<NX, FORM, double>, row_smem<NX>(G::MAXR, 0));
    return e;
  };
  cudaError_t e = cudaSuccess;
  for (int W : {G::n / 2, G::n / 2 - 1, G::n / 2 + 1})   // one of each form
    if (e == cudaSuccess) e = with_form<NX>(W, prepare);
  return e;
}
template <int NY, int NACC, bool HALF>
cudaError_t prepare_packed_col_a() {
  using G = ColGeo<NY, HALF>;
  cudaError_t e = allow_smem(k_packed_col<NY, NACC, HALF, false>, packed_col_smem_ahead<NY, HALF>(G::MAXG));
  if constexpr (G::STAGEABLE) {
    if (e == cudaSuccess)
      e = allow_smem(k_packed_col<NY, NACC, HALF, true>, packed_col_smem_staged<NY, HALF>(G::SG));
  }
  return e;
}
template <int NY>
cudaError_t prepare_packed_col_n() {
  cudaError_t e = prepare_packed_col_a<NY, 1, true>();
  if (e == cudaSuccess) e = prepare_packed_col_a<NY, 1, false>();
  if (e == cudaSuccess) e = prepare_packed_col_a<NY, 2, true>();
  if (e == cudaSuccess) e = prepare_packed_col_a<NY, 2, false>();
  if (e == cudaSuccess) e = allow_smem(k_packed_col_wide<NY, true>, 227 * 1024);
  if (e == cudaSuccess) e = allow_smem(k_packed_col_wide<NY, false>, 227 * 1024);
  return e;
}

}  // namespace pk
}  // namespace sbi
