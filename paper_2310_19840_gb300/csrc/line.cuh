// line.cuh - whole steps of one-dimensional FP32 members in one launch (ensembles
// too large for it take one launch per pass: line_pays in line.h).
//
// A one-dimensional member is one row of 16 to 4096 points: a pass over it is
// far below a launch in work, and a step of some 64 dependent launches took 7
// to 27 us each.  Here one launch runs the whole list of passes (a program of
// phases, line.h) with a barrier between phases.  Every transform of a phase
// goes to its own group of threads (packed.cuh), so the products of a level are
// transformed side by side; physical fields stay in shared memory, mixed fields
// (8 KB at most) in global memory, found in L1 and L2.  Rows of 2048 points and
// more run on a cluster of 4 or 8 blocks: the inverse transforms and their
// physical fields are formed in every block, the products and the modes are
// shared out, and the cluster's barrier orders the phases that hand mixed
// fields on.  The results do not depend on the number of blocks.
// What bounds it is the chain of dependent phases, 25 per right-hand side of
// about a microsecond each.
// Measured (GB300, a step): 256 points 102 us (420 us as 64 launches); 4096
// points over a bar 377 us (558 us in one block, 850 us as 64 launches).
#pragma once

#include "line.h"
#include "packed_kernels.cuh"

namespace sbi {
namespace pk {

constexpr int kLineThreads = 512;

template <int NX>
__host__ __device__ constexpr size_t line_smem(int program_bytes) {
  using G = RowGeo<NX>;
  return 8 * ((size_t)G::RTW + (size_t)(kLineThreads / G::T) * G::XLEN + (size_t)kLineSlots * G::n) +
         (program_bytes + 15) / 16 * 16;
}

// MULTI: a cluster of p.cluster blocks per member (else one block, whose code
// then has no shares to work out: 7 % of a 256-point step)
template <int NX, bool EXACT, bool MULTI>
__global__ void __launch_bounds__(kLineThreads, 1) k_line(const __grid_constant__ LineParams p) {
  using G = RowGeo<NX>;
  using SP = StatePair<float>;
  constexpr int n = G::n, R = G::R, T = G::T, GROUPS = kLineThreads / T;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  auto* xs0 = reinterpret_cast<typename G::E*>(smem_raw) + G::RTW;
  F2* slots = reinterpret_cast<F2*>(xs0 + GROUPS * G::XLEN);               // [slot][m]
  unsigned char* prog = reinterpret_cast<unsigned char*>(slots + kLineSlots * n);
  const int tid = threadIdx.x, g = tid / T, j = tid % T;
  auto* xs = xs0 + g * G::XLEN;
  const int C = MULTI ? p.cluster : 1, rank = MULTI ? (int)blockIdx.x % C : 0;
  const int member = p.member0 + (int)blockIdx.x / C;
  for (int i = tid; i < (p.bytes + 15) / 16; i += kLineThreads)
    reinterpret_cast<uint4*>(prog)[i] = reinterpret_cast<const uint4*>(p.program)[i];
  const LineHeader& H = *reinterpret_cast<const LineHeader*>(prog);
  __syncthreads();
  RowTwiddles<NX> t(H.tw, reinterpret_cast<float2*>(smem_raw), j);
  const LinePhase* phases = reinterpret_cast<const LinePhase*>(prog + H.phases);
  const LineJob* jobs = reinterpret_cast<const LineJob*>(prog + H.jobs);
  const LineTerm* terms = reinterpret_cast<const LineTerm*>(prog + H.terms);
  const BufRef* bufs = reinterpret_cast<const BufRef*>(prog + H.bufs);
  const int W = H.W;
  auto mixed = [&](int b) { return reinterpret_cast<F2*>(bufs[b].ptr) + (long long)member * bufs[b].stride; };
  auto real = [&](int b) {
    return reinterpret_cast<F2*>(reinterpret_cast<float*>(bufs[b].ptr) + (long long)member * bufs[b].stride);
  };

#pragma unroll 1
  for (int ip = 0; ip < H.nphases; ++ip) {
    const LinePhase& P = phases[ip];
    // also before a phase that this member skips: the next ones rely on it
    if (MULTI && P.sync) {
      asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
      asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    } else {
      __syncthreads();
    }
    if (P.active && P.active[member] == 0) continue;      // the whole cluster
    if (P.type == LP_INVERSE || P.type == LP_FORWARD) {
      const bool inverse = P.type == LP_INVERSE;
      // every block runs all inverse transforms, and its share of the others
      const int share = inverse ? 1 : C;
#pragma unroll 1
      for (int first = P.begin + (inverse ? 0 : rank); first < P.end; first += share * GROUPS) {
        t.renew();
        const int mine = first + share * g;
        const bool valid = mine < P.end;
        if (G::WARP && first + share * ((tid & ~31) / T) >= P.end) break;   // a warp without a job
        const LineJob job = jobs[valid ? mine : P.begin];
        One x[R];
        if (inverse) {
          // modes k < W and n - k < W of the sum of the sources (inverse_input)
          if constexpr (kFastRow<NX, EXACT>) {
#pragma unroll 1
            for (int q = 0; q < job.nsrc; ++q) {
              const F2* src = mixed(job.buf + q);
#pragma unroll
              for (int r = 0; r < R; ++r) {
                const int k = j + r * T;
                One v = both(0.f);
                if (r < R / 2) v = src[k];
                else if (r > R / 2 || j != 0) v = src[n - k];
                x[r] = q == 0 ? v : add(x[r], v);
              }
            }
            twist_modes<NX>(x, t);
          } else {
#pragma unroll
            for (int r = 0; r < R; ++r) {
              const int k = j + r * T, kk = n - k;
              One a = both(0.f), b = both(0.f);
              for (int q = 0; q < job.nsrc; ++q) {
                const F2* src = mixed(job.buf + q);
                if (k < W) a = add(a, src[k]);
                if (k > 0 && kk < W) b = add(b, src[kk]);
              }
              const float2 e = __ldg(t.tw + tw_off(NX) + k);
              const One o = cmul(sub_conj(a, b), make_float2(e.x, -e.y));
              x[r] = conj(addi(add_conj(a, b), o));
            }
          }
        } else {
          const F2* s = slots + job.slot * n + j;
          const F2* eta = P.eta >= 0 ? real(P.eta) + j : nullptr;
          if (job.op == ROP_PROD) {
#pragma unroll
            for (int r = 0; r < R; ++r) x[r] = s[r * T];
            for (int f = 0; f < 3; ++f) {
              const int e = f == 0 ? job.ea : (f == 1 ? job.eb : job.ew);
              if (e == 0) continue;
              const int b = f == 0 ? P.eta : (f == 1 ? P.delta : P.wgt);
              const F2* src = real(b) + j;
              One v[R];
#pragma unroll
              for (int r = 0; r < R; ++r) v[r] = src[r * T];
              times_field<R>(x, v, e);
            }
            if (job.coef != 1.f) {
#pragma unroll
              for (int r = 0; r < R; ++r) x[r] = scale(job.coef, x[r]);
            }
          } else {
#pragma unroll
            for (int r = 0; r < R; ++r) {
              const F2 v = s[r * T], ex = s[n + r * T], px = s[2 * n + r * T];
              const F2 dot = mul(ex, px), den = fma(ex, ex, both(1.f));
              if (job.op == ROP_VFW) {
                x[r] = fma(v, den, mul(both(-1.f), dot));
              } else {
                const F2 num = add(v, dot);
                x[r] = scale(0.5f, sub(quotient(mul(num, num), den), mul(px, px)));
                if (eta) x[r] = axpy(-job.coef, eta[r * T], x[r]);
                if (job.pg) x[r] = sub(x[r], slots[5 * n + j + r * T]);
              }
            }
          }
        }
        __syncwarp();
        t.run(x, xs);
        if (inverse) {
          if (valid) {
            F2* s = slots + job.slot * n + j;
            F2* out = job.phys >= 0 && rank == 0 ? real(job.phys) + j : nullptr;
#pragma unroll
            for (int r = 0; r < R; ++r) {
              const F2 v = conj(x[r]);
              s[r * T] = v;
              if (out) out[r * T] = v;
            }
          }
        } else {
          One X[kKept<NX, EXACT>];
          share_modes<NX, EXACT>(x, W, j, xs);
          kept_modes<NX, EXACT>(x, X, 0, W, j, xs, t);
          if (valid) {
            F2* out = mixed(job.buf) + j;
#pragma unroll
            for (int r = 0; r < kKept<NX, EXACT>; ++r)
              if (kFastRow<NX, EXACT> || j + r * T < W) out[r * T] = X[r];
          }
          if constexpr (!G::WARP) __syncthreads();
        }
      }
    } else if (P.type == LP_COL) {
      // outputs may overwrite inputs of the same mode: every load of a mode
      // comes before its stores, by the same thread
      for (int k = rank * kLineThreads + tid; k < W; k += C * kLineThreads) {
        F2 a0 = both(0.f), a1 = a0;
#pragma unroll 8
        for (int q = P.begin; q < P.end; ++q) {
          const LineTerm m = terms[q];
          const F2 v = mixed(m.buf)[k];
          const float f = __ldg(reinterpret_cast<const float*>(m.tab) + k);
          if (m.acc == 0) a0 = acc_term(a0, v, f, m.ph);
          else a1 = acc_term(a1, v, f, m.ph);
        }
        F2 extra = both(0.f);
#pragma unroll 4
        for (int q = P.pass_begin; q < P.pass_end; ++q) extra = add(extra, mixed(q)[k]);
        for (int q = P.out_begin; q < P.out_end; ++q) {
          const LineTerm m = terms[q];
          const float f = __ldg(reinterpret_cast<const float*>(m.tab) + k);
          const F2 o = acc_term(both(0.f), m.acc == 0 ? a0 : a1, f, m.ph);
          mixed(m.buf)[k] = q == P.out_begin && P.pass_begin < P.pass_end ? add(o, extra) : o;
        }
      }
    } else if (P.type == LP_RK) {
      const RkParams& q = reinterpret_cast<const RkParams*>(prog + H.rks)[P.out_begin];
      bool bad = false;
      const float bw = (q.stage == 1 || q.stage == 4) ? 1.f : 2.f;
      const RkScalar cdt = p.cdt[q.mode == RK_STAGE ? q.stage - 1 : 0], dt6 = p.dt6;
      // the first block updates the elevation, the second (if there is one) the
      // potential: the blocks that transform slots 2 and 3 (jobs 0 and 1)
      for (int i = tid + (C > 1 ? rank * n : 0); i < (C > 1 ? (rank < 2 ? (rank + 1) * n : 0) : 2 * n);
           i += kLineThreads) {
        const bool potential = i >= n;
        const int m = potential ? i - n : i;
        const BufRef& st = potential ? q.phi0 : q.eta0;
        const BufRef& sum = potential ? q.acc_phi : q.acc_eta;
        char* M = reinterpret_cast<char*>(st.ptr) + (long long)member * st.stride * 8;      // 8 bytes per value
        char* A = reinterpret_cast<char*>(sum.ptr) + (long long)member * sum.stride * 8;
        float2 f = make_float2(0.f, 0.f);
        if (q.mode == RK_STAGE && !potential)
          f = parts(reinterpret_cast<const F2*>(reinterpret_cast<const float*>(q.V.ptr) + (long long)member * q.V.stride)[m]);
        else if (q.mode != RK_ENTRY)
          f = parts(slots[(potential ? 0 : 1) * n + m]);
        float2 res;
        auto update = [&](auto e) {
          using S = decltype(e);
          e = S::load(M, m);
          if (q.mode == RK_STAGE) {
            S a = q.stage > 1 ? S::load(A, m) : S::zero();
            a.add(0, bw * f.x);
            a.add(1, bw * f.y);
            if (q.stage < 4) {
              a.store(A, m);
              res = make_float2(e.template offset<float>(0, cdt, f.x), e.template offset<float>(1, cdt, f.y));
              return;
            }
            e.add_scaled(0, a, dt6);
            e.add_scaled(1, a, dt6);
            e.store(M, m);
            bad |= !e.finite();
          } else if (q.mode != RK_ENTRY) {
            e.add(0, f.x);
            e.add(1, f.y);
            if (q.mode == RK_CORRECT) {   // RK_OFFSET leaves the state unchanged
              e.store(M, m);
              bad |= !e.finite();
            }
          }
          res = make_float2(float(e.value(0)), float(e.value(1)));
        };
        if (q.state64) update(StatePair<double>::zero());
        else update(SP::zero());
        if (q.tail) {
          slots[(potential ? 3 : 2) * n + m] = f2(res);
          if (!potential)
            reinterpret_cast<F2*>(reinterpret_cast<float*>(q.eta_w.ptr) + (long long)member * q.eta_w.stride)[m] = f2(res);
        }
      }
      if (bad && q.nonfinite) *q.nonfinite = 1;
    } else if (P.type == LP_WDOT) {
      F2* out = real(P.dst);
      for (int m = rank * kLineThreads + tid; m < n; m += C * kLineThreads) {
        const F2 ex = slots[n + m];
        out[m] = quotient(fma(ex, slots[2 * n + m], slots[m]), fma(ex, ex, both(1.f)));
      }
    } else if (rank == 0) {   // LP_WMK: FP64 sums and sines, rounded once
      const LineWmk& q = reinterpret_cast<const LineWmk*>(prog + H.wmks)[P.out_begin];
      const double time = *q.t + p.offset[q.stage];
      double* sines = reinterpret_cast<double*>(xs0);       // the exchange buffer is free here
      for (int i = tid; i < q.J; i += kLineThreads) sines[i] = sin(q.omega[i] * time + q.phase[i]);
      __syncthreads();
      for (int x = tid; x < 2 * n; x += kLineThreads) {
        double acc = 0.0;
        for (int i = 0; i < q.J; ++i) acc += q.prof[(size_t)i * 2 * n + x] * sines[i];
        reinterpret_cast<float*>(slots + 5 * n)[x] = float(acc);
      }
    }
  }
}

template <int NX>
cudaError_t prepare_line_n() {
  constexpr bool M = line_cluster(NX) > 1;
  constexpr size_t bytes = line_smem<NX>(kLineMaxBytes);
  cudaError_t e = allow_smem(k_line<NX, true, false>, bytes);
  if (e == cudaSuccess) e = allow_smem(k_line<NX, false, false>, bytes);
  if (e == cudaSuccess) e = allow_smem(k_line<NX, true, M>, bytes);
  if (e == cudaSuccess) e = allow_smem(k_line<NX, false, M>, bytes);
  return e;
}
// Clusters of `cluster` blocks that the device holds at once.  Two blocks do not
// fit an SM, and a cluster lies in one group of SMs, so there are fewer than SMs
// divided by the size: 16 members of 4096 points on clusters of eight took two
// waves, 674 us a step, one member 343.
template <int NX>
cudaError_t line_clusters_n(int cluster, int* most) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)cluster);
  cfg.blockDim = dim3(kLineThreads);
  cfg.dynamicSmemBytes = line_smem<NX>(kLineMaxBytes);
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cluster;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaOccupancyMaxActiveClusters(most, k_line<NX, true, (line_cluster(NX) > 1)>, &cfg);
}
template <int NX>
cudaError_t launch_line_n(const LineParams& p, cudaStream_t st) {
  constexpr bool M = line_cluster(NX) > 1;
  if (p.member0 < 0 || p.member1 <= p.member0 || p.bytes > kLineMaxBytes || p.cluster < 1 ||
      p.cluster > line_cluster(NX))
    return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((p.member1 - p.member0) * p.cluster));
  cfg.blockDim = dim3(kLineThreads);
  cfg.dynamicSmemBytes = line_smem<NX>(p.bytes);
  cfg.stream = st;
  if (p.cluster == 1)
    return p.exact ? cudaLaunchKernelEx(&cfg, k_line<NX, true, false>, p)
                   : cudaLaunchKernelEx(&cfg, k_line<NX, false, false>, p);
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)p.cluster;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return p.exact ? cudaLaunchKernelEx(&cfg, k_line<NX, true, M>, p) : cudaLaunchKernelEx(&cfg, k_line<NX, false, M>, p);
}

}  // namespace pk
}  // namespace sbi
