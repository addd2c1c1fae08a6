// packed.cuh - FP32 transforms in packed arithmetic.
//
// The FP32 pipe of an SM of this part takes 128 scalar operations per cycle,
// either as four warp instructions or as two of the packed ones (add, mul, fma
// .f32x2: two floats in a register pair).  With one complex number per register
// pair every step of a transform is packed: a sum is one instruction, a product
// by a real or by +-i folded into a sum is one fma (a repeated or exchanged
// half of an operand costs nothing: measured, no extra instruction is issued),
// a complex product is two.  Half of the issue slots are left to everything
// else.
//
// A transform of N elements by T = N / R threads holds R elements per thread (16
// in rows and most columns from N = 128 up, else up to 8): one exchange through
// shared memory up to N = R^2, two up to 8 R^2, three up to 4096 with R = 8.
// Against 8 elements per thread, 16 halve the shared-memory traffic of a
// 256-point transform, which bounds the row passes.
// Elements are in the order x[r] = a[j + r T] on entry and on exit.  An element
// is one complex number (One) or two of independent sequences that share every
// twiddle and index (Two).
#pragma once

#include "fft.cuh"

namespace sbi {
namespace pk {

struct F2 {
  unsigned long long v;
};
__device__ __forceinline__ F2 f2(float a, float b) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ F2 f2(float2 a) { return f2(a.x, a.y); }
__device__ __forceinline__ float2 parts(F2 a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
  return r;
}
__device__ __forceinline__ F2 both(float a) { return f2(a, a); }
__device__ __forceinline__ F2 swp(F2 a) {
  const float2 p = parts(a);
  return f2(p.y, p.x);
}
__device__ __forceinline__ F2 add(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 sub(F2 a, F2 b) {
  F2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 mul(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 fma(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}

// complex operations on a pair (re, im)
__device__ __forceinline__ F2 zero_of(F2) { return both(0.f); }
__device__ __forceinline__ F2 addi(F2 a, F2 b) { return fma(swp(b), f2(-1.f, 1.f), a); }          // a + i b
__device__ __forceinline__ F2 subi(F2 a, F2 b) { return fma(swp(b), f2(1.f, -1.f), a); }          // a - i b
__device__ __forceinline__ F2 axpy(float s, F2 b, F2 c) { return fma(both(s), b, c); }            // c + s b
__device__ __forceinline__ F2 axpyi(float s, F2 b, F2 c) { return fma(swp(b), f2(-s, s), c); }    // c + i s b
__device__ __forceinline__ F2 scale(float s, F2 a) { return mul(both(s), a); }
__device__ __forceinline__ F2 cmul(F2 a, float2 w) { return fma(f2(-w.y, w.y), swp(a), mul(both(w.x), a)); }
__device__ __forceinline__ F2 conj(F2 a) { return mul(a, f2(1.f, -1.f)); }
__device__ __forceinline__ F2 add_conj(F2 a, F2 b) { return fma(b, f2(1.f, -1.f), a); }           // a + b*
__device__ __forceinline__ F2 sub_conj(F2 a, F2 b) { return fma(b, f2(-1.f, 1.f), a); }           // a - b*
// explicit roundings: every instantiation gives the same bits
__device__ __forceinline__ float2 wmul(float2 a, float2 b) {
  return make_float2(fmaf(-a.y, b.y, __fmul_rn(a.x, b.x)), fmaf(a.x, b.y, __fmul_rn(a.y, b.x)));
}

using One = F2;
struct Two {
  F2 a, b;
};
__device__ __forceinline__ Two add(Two x, Two y) { return Two{add(x.a, y.a), add(x.b, y.b)}; }
__device__ __forceinline__ Two sub(Two x, Two y) { return Two{sub(x.a, y.a), sub(x.b, y.b)}; }
__device__ __forceinline__ Two addi(Two x, Two y) { return Two{addi(x.a, y.a), addi(x.b, y.b)}; }
__device__ __forceinline__ Two subi(Two x, Two y) { return Two{subi(x.a, y.a), subi(x.b, y.b)}; }
__device__ __forceinline__ Two axpy(float s, Two y, Two c) { return Two{axpy(s, y.a, c.a), axpy(s, y.b, c.b)}; }
__device__ __forceinline__ Two axpyi(float s, Two y, Two c) { return Two{axpyi(s, y.a, c.a), axpyi(s, y.b, c.b)}; }
__device__ __forceinline__ Two cmul(Two x, float2 w) { return Two{cmul(x.a, w), cmul(x.b, w)}; }

// an element in memory
template <typename V> struct Mem;
template <> struct Mem<One> {
  using T = unsigned long long;
  __device__ __forceinline__ static T to(One v) { return v.v; }
  __device__ __forceinline__ static One from(T m) { return One{m}; }
};
template <> struct Mem<Two> {
  using T = ulonglong2;
  __device__ __forceinline__ static T to(Two v) { return make_ulonglong2(v.a.v, v.b.v); }
  __device__ __forceinline__ static Two from(T m) { return Two{F2{m.x}, F2{m.y}}; }
};

// exp(-2 pi i q / n) for n = 8, 16 or 32 (q and n constants after unrolling)
__device__ __forceinline__ float2 unit_root(int q, int n) {
  constexpr float c[32] = {1.f, 0.98078528040323044913f, 0.92387953251128675613f, 0.83146961230254523708f,
                           0.70710678118654752440f, 0.55557023301960222474f, 0.38268343236508977173f,
                           0.19509032201612826785f, 0.f, -0.19509032201612826785f, -0.38268343236508977173f,
                           -0.55557023301960222474f, -0.70710678118654752440f, -0.83146961230254523708f,
                           -0.92387953251128675613f, -0.98078528040323044913f, -1.f, -0.98078528040323044913f,
                           -0.92387953251128675613f, -0.83146961230254523708f, -0.70710678118654752440f,
                           -0.55557023301960222474f, -0.38268343236508977173f, -0.19509032201612826785f, 0.f,
                           0.19509032201612826785f, 0.38268343236508977173f, 0.55557023301960222474f,
                           0.70710678118654752440f, 0.83146961230254523708f, 0.92387953251128675613f,
                           0.98078528040323044913f};
  const int i = q * (32 / n) & 31;
  return make_float2(c[i], c[(i + 8) & 31]);      // -sin(x) = cos(x + pi / 2)
}

// ---------------------------------------------------------------------------
// Forward DFTs of length R in registers.  The products by (1 -+ i) / sqrt(2)
// are folded into the sums that follow them: 8, 26 and 76 packed operations per
// complex sequence for R = 4, 8 and 16.
// ---------------------------------------------------------------------------
template <typename V>
__device__ __forceinline__ void dft4(V& a, V& b, V& c, V& d) {
  const V t0 = add(a, c), t1 = sub(a, c), t2 = add(b, d), t3 = sub(b, d);
  a = add(t0, t2);
  c = sub(t0, t2);
  b = subi(t1, t3);
  d = addi(t1, t3);
}
constexpr float kH = 0.70710678118654752440f;     // cos(pi / 4)
constexpr float kC1 = 0.92387953251128675613f;    // cos(pi / 8)
constexpr float kS1 = 0.38268343236508977173f;    // sin(pi / 8)

template <int R, typename V> struct PDft;
template <typename V> struct PDft<1, V> {
  __device__ __forceinline__ static void run(V*) {}
};
template <typename V> struct PDft<2, V> {
  __device__ __forceinline__ static void run(V* x) {
    const V t = x[0];
    x[0] = add(t, x[1]);
    x[1] = sub(t, x[1]);
  }
};
template <typename V> struct PDft<4, V> {
  __device__ __forceinline__ static void run(V* x) { dft4(x[0], x[1], x[2], x[3]); }
};
template <typename V> struct PDft<8, V> {
  __device__ __forceinline__ static void run(V* x) {
    V e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6];
    V o0 = x[1], o1 = x[3], o2 = x[5], o3 = x[7];
    dft4(e0, e1, e2, e3);
    dft4(o0, o1, o2, o3);
    x[0] = add(e0, o0);
    x[4] = sub(e0, o0);
    const V u = subi(o1, o1);           // w8 o1 = h (1 - i) o1
    x[1] = axpy(kH, u, e1);
    x[5] = axpy(-kH, u, e1);
    x[2] = subi(e2, o2);                // w8^2 = -i
    x[6] = addi(e2, o2);
    const V v = addi(o3, o3);           // w8^3 o3 = -h (1 + i) o3
    x[3] = axpy(-kH, v, e3);
    x[7] = axpy(kH, v, e3);
  }
};
template <typename V> struct PDft<16, V> {
  __device__ __forceinline__ static void run(V* x) {
    // DFT4 over r2 of x[r1 + 4 r2]: A[r1][q2] in x[r1 + 4 q2]
#pragma unroll
    for (int r = 0; r < 4; ++r) dft4(x[r], x[r + 4], x[r + 8], x[r + 12]);
    // then, for each q2, the DFT4 over r1 of w16^{r1 q2} A[r1][q2], written
    // to x[4 q2 + q1] and put in order (q2 + 4 q1) at the end
    dft4(x[0], x[1], x[2], x[3]);
    {  // q2 = 1
      V* b = x + 4;
      const V p = cmul(b[1], make_float2(kC1, -kS1)), q = cmul(b[3], make_float2(kS1, -kC1));
      const V u = subi(b[2], b[2]);
      const V t0 = axpy(kH, u, b[0]), t1 = axpy(-kH, u, b[0]), t2 = add(p, q), t3 = sub(p, q);
      b[0] = add(t0, t2);
      b[2] = sub(t0, t2);
      b[1] = subi(t1, t3);
      b[3] = addi(t1, t3);
    }
    {  // q2 = 2: w16^2 b1 = h u, w16^4 b2 = -i b2, w16^6 b3 = -h v
      V* b = x + 8;
      const V u = subi(b[1], b[1]), v = addi(b[3], b[3]);
      const V t0 = subi(b[0], b[2]), t1 = addi(b[0], b[2]), t2 = sub(u, v), t3 = add(u, v);
      b[0] = axpy(kH, t2, t0);
      b[2] = axpy(-kH, t2, t0);
      b[1] = axpyi(-kH, t3, t1);
      b[3] = axpyi(kH, t3, t1);
    }
    {  // q2 = 3: w16^6 b2 = -h v
      V* b = x + 12;
      const V p = cmul(b[1], make_float2(kS1, -kC1)), q = cmul(b[3], make_float2(-kC1, kS1));
      const V v = addi(b[2], b[2]);
      const V t0 = axpy(-kH, v, b[0]), t1 = axpy(kH, v, b[0]), t2 = add(p, q), t3 = sub(p, q);
      b[0] = add(t0, t2);
      b[2] = sub(t0, t2);
      b[1] = subi(t1, t3);
      b[3] = addi(t1, t3);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int p = q + 1; p < 4; ++p) {
        const V t = x[4 * q + p];
        x[4 * q + p] = x[q + 4 * p];
        x[q + 4 * p] = t;
      }
  }
};

// ---------------------------------------------------------------------------
// The transform.  WARP: the threads that share a sequence are in one warp
// (exchanges synchronise the warp), else they are in one block and every thread
// of the block runs the transform.  The exchange buffer holds xlen() elements
// per sequence; CI sequences may be interleaved in it (element i of sequence c
// at i CI + c).  Indices are padded by one element per R: the accesses of the
// first pass (stride R) and the contiguous ones then fall into distinct banks.
// ---------------------------------------------------------------------------
template <typename V, int N, int R, bool WARP, int CI = 1>
struct PackedFft {
  static_assert(N % R == 0 && (R == 4 || R == 8 || R == 16) && (N <= 8 * R * R || (R == 8 && N <= 4096)), "length");
  using M = Mem<V>;
  using E = typename M::T;
  static constexpr int T = N / R;
  static constexpr int RP2 = N / R < R ? N / R : R;          // radix of the second pass
  static constexpr int TW = N > R ? (RP2 - 1) * R : 0;       // its twiddles (float2 in shared memory)
  __host__ __device__ static constexpr int xpad(int i) { return i + i / R; }
  __host__ __device__ static constexpr int xlen() { return N > R ? N + N / R : 0; }
  __device__ __forceinline__ static void sync() {
    if constexpr (WARP) __syncwarp();
    else __syncthreads();
  }
  // Second-pass twiddles w_L^{m b}, L = R RP2, m = 1 .. RP2 - 1, of the thread's
  // butterflies b = j + q T (b = j mod R where a third pass follows), from a
  // table [m - 1][b] in shared memory.
  struct Twiddles {
    const float2* t;
    __device__ __forceinline__ float2 operator()(int m, int q) const { return t[(m - 1) * R + q * T]; }
  };
  // the table, by the whole block (the caller synchronises)
  __device__ __forceinline__ static void fill_twiddles(float2* t, const float2* __restrict__ tw) {
    if constexpr (TW > 0) {
      constexpr int L = R * RP2;
      for (int i = threadIdx.x; i < TW; i += blockDim.x) t[i] = __ldg(tw + tw_off(L) + (i / R + 1) * (i % R));
    }
  }
  __device__ __forceinline__ static Twiddles twiddles(const float2* t, int j) {
    return Twiddles{t + (N <= R * R ? j : j & (R - 1))};
  }
  // v[m] *= w^m, w = table[b]
  template <int RP>
  __device__ __forceinline__ static void times_powers(V (&v)[RP], const float2* __restrict__ table, int b) {
    static_assert(RP == 2 || RP == 4 || RP == 8, "later passes of radix 2, 4 and 8");
    const float2 w1 = __ldg(table + b);
    v[1] = cmul(v[1], w1);
    if constexpr (RP >= 4) {
      const float2 w2 = RP == 4 ? __ldg(table + 2 * b) : wmul(w1, w1), w3 = wmul(w1, w2);
      v[2] = cmul(v[2], w2);
      v[3] = cmul(v[3], w3);
      if constexpr (RP >= 8) {
        const float2 w4 = __ldg(table + 4 * b);
        v[4] = cmul(v[4], w4);
        v[5] = cmul(v[5], wmul(w4, w1));
        v[6] = cmul(v[6], wmul(w4, w2));
        v[7] = cmul(v[7], wmul(w4, w3));
      }
    }
  }
  // Butterflies b = j + q T (q < Q) of radix RP on elements v[m] = x[q + m Q].
  // A later pass (512 elements and more with 16 per thread, 128 with 8) loads w_N^b
  // and w_N^{4b} (radix 4: w_N^{2b}) and forms the other powers by products.  With
  // w_N^b itself a product, w_N^j e^{-2 pi i q / R}, the powers carried its error up
  // to three times: a step of a 4096 x 2048 sea was 1.39e-7 from the 64-bit one, and
  // is 1.24e-7.
  template <int RP, bool SECOND>
  __device__ __forceinline__ static void last_pass(V (&x)[R], int j, Twiddles t, const float2* __restrict__ tw) {
    constexpr int Q = R / RP;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      V v[RP];
#pragma unroll
      for (int m = 0; m < RP; ++m) v[m] = x[q + m * Q];
      if constexpr (SECOND) {
#pragma unroll
        for (int m = 1; m < RP; ++m) v[m] = cmul(v[m], t(m, q));
      } else {
        times_powers<RP>(v, tw + tw_off(N), j + q * T);
      }
      PDft<RP, V>::run(v);
#pragma unroll
      for (int m = 0; m < RP; ++m) x[q + m * Q] = v[m];
    }
  }
  // s: the exchange buffer of this thread's sequence (offset by c already);
  // nothing may be in use there on entry, nothing is on exit
  __device__ __forceinline__ static void run(V (&x)[R], E* s, int j, Twiddles t, const float2* __restrict__ tw) {
    PDft<R, V>::run(x);
    if constexpr (N > R) {
      const int wb = j * (R + 1);        // xpad(j R + r) = j (R + 1) + r
#pragma unroll
      for (int r = 0; r < R; ++r) s[(wb + r) * CI] = M::to(x[r]);
      sync();
      // xpad(j + r T) splits: j < T divides R, or R divides T
      const int rb = T < R ? j : xpad(j);
#pragma unroll
      for (int r = 0; r < R; ++r) x[r] = M::from(s[(rb + xpad(r * T)) * CI]);
      sync();
      if constexpr (N <= R * R) {
        last_pass<RP2, true>(x, j, t, tw);
      } else {
        const int k = j & (R - 1);
#pragma unroll
        for (int r = 1; r < R; ++r) x[r] = cmul(x[r], t(r, 0));
        PDft<R, V>::run(x);
        // element (j - k) R + k + r R
        const int sb = xpad((j - k) * R) + k;
#pragma unroll
        for (int r = 0; r < R; ++r) s[(sb + xpad(r * R)) * CI] = M::to(x[r]);
        sync();
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = M::from(s[(rb + xpad(r * T)) * CI]);
        sync();
        if constexpr (N <= 8 * R * R) {
          last_pass<N / (R * R), false>(x, j, t, tw);
        } else {   // a third pass of radix 8, then the last
          const int k3 = j & (R * R - 1);
          times_powers<R>(x, tw + tw_off(R * R * R), k3);
          PDft<R, V>::run(x);
          const int sb3 = xpad((j - k3) * R) + xpad(k3);   // element (j - k3) R + k3 + r R^2
#pragma unroll
          for (int r = 0; r < R; ++r) s[(sb3 + xpad(r * R * R)) * CI] = M::to(x[r]);
          sync();
#pragma unroll
          for (int r = 0; r < R; ++r) x[r] = M::from(s[(rb + xpad(r * T)) * CI]);
          sync();
          last_pass<N / (R * R * R), false>(x, j, t, tw);
        }
      }
    }
  }
};

}  // namespace pk
}  // namespace sbi
