// Small 2D grids: the whole solve of a field by one thread-block cluster.
//
// A field of some ten thousand points keeps a pass kernel busy for two or
// three microseconds, and the rest of a pass's time goes to its launch, to
// filling and draining the GPU and to the arrival ticket of its dots (8 us per
// pass kernel without dots and 14 with, for 256^2 float32 on a GPU otherwise
// idle). Here one cluster of up to 16 CTAs runs every pass of Algorithms 1-4
// on one field in a single launch: the transforms happen in shared memory,
// the two transpositions of an application of G are stores into the other
// CTAs' shared memory, and the dots are reduced through it. CTA c owns the
// rows y [c ny/C, (c+1) ny/C), its part of every field vector, and in between
// the sequences kx [c KC, (c+1) KC) along y. One application of G:
//   prologue (xfwd_prologue) -> x transform -> stores to the owners of the
//   sequences, cluster barrier -> forward transform along y, x G_hat/P and
//   Parseval dots, inverse transform -> stores back, cluster barrier ->
//   inverse x transform -> epilogue (xinv_epilogue) and dots, cluster barrier.
// The scalar recurrences run in every CTA on the same sums in the same order,
// so all of them take the same decisions. Three equal shared-memory buffers
// serve all phases: x transform U0 <-> U1, received by U2; y transform U2 <->
// U0, received by U1; inverse x transform U0 <-> U2 (the stages of a transform
// alternate between two buffers, one barrier per stage).
// Bound by the latency of the chain of stages and barriers, not by bytes: per
// pass, CG 256^2 float32 40 -> 18 us, Van Cittert 128^2 float64 53 -> 36 us
// (there also by the float64 rate of 16 SMs).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "args.h"
#include "fft.cuh"
#include "launch.h"
#include "passes.cuh"

namespace gad {

__device__ __forceinline__ uint32_t cl_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cl_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Address of this CTA's shared-memory address `a` in the CTA of rank r.
__device__ __forceinline__ uint32_t cl_map(uint32_t a, uint32_t r) {
  uint32_t d;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(r));
  return d;
}
__device__ __forceinline__ void cl_store(uint32_t a, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void cl_store(uint32_t a, double2 v) {
  asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(v.x), "d"(v.y) : "memory");
}
__device__ __forceinline__ void cl_store(uint32_t a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

// One radix-R Stockham stage of nseq sequences from `src` to `dst` (rows of
// stride ld, phys() padding); post(w, i, x) may change output element i of
// sequence w.
template <typename C, int R, bool INV, class Post>
__device__ __forceinline__ void cl_stage(const C* src, C* dst, int ld, int L, int nseq, const FftStage& sg,
                                         const C* tw, int tid, int nthr, Post& post) {
  const int lr = L / R, ns = sg.ns, nb = nseq * lr;
  const bool p2 = (lr & (lr - 1)) == 0;                 // a shift instead of a float quotient
  const int sh = 31 - __clz(lr);
  for (int bi = tid; bi < nb; bi += nthr) {
    const int w = p2 ? bi >> sh : fquot(bi, sg.rcp_lr), j = bi - w * lr;
    const C* s = src + w * ld;
    C v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = s[phys(j + r * lr)];
    const int k = (ns & (ns - 1)) == 0 ? j & (ns - 1) : j - ns * fquot(j, sg.rcp_ns);
    if (ns > 1) {
      const C* twk = tw + sg.tw_off + k;
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = INV ? cmulc(v[r], twk[(r - 1) * ns]) : cmul(v[r], twk[(r - 1) * ns]);
    }
    dft<R, INV>(v);
    C* d = dst + w * ld;
    const int o = (j - k) * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      post(w, o + r * ns, v[r]);
      d[phys(o + r * ns)] = v[r];
    }
  }
}

// Transforms nseq sequences; p (in shared memory) has radices 2, 3, 4 and 8.
// The stages alternate between a and b, starting from a; returns the buffer
// with the result, complete in the whole block. post runs on the outputs of
// the last stage.
struct ClKeep {
  template <typename C> __device__ __forceinline__ void operator()(int, int, C&) const {}
};

template <typename C, bool INV, class Post>
__device__ __forceinline__ C* cl_fft_post(C* a, C* b, int ld, const FftPlan* p, const C* tw, int nseq, int tid,
                                          int nthr, Post& post) {
  ClKeep keep;
  const int L = p->L, n = p->nst;
  for (int q = 0; q < n; ++q) {
    const FftStage sg = p->st[q];
    if (q + 1 < n) {
      switch (sg.radix) {
        case 2: cl_stage<C, 2, INV>(a, b, ld, L, nseq, sg, tw, tid, nthr, keep); break;
        case 3: cl_stage<C, 3, INV>(a, b, ld, L, nseq, sg, tw, tid, nthr, keep); break;
        case 4: cl_stage<C, 4, INV>(a, b, ld, L, nseq, sg, tw, tid, nthr, keep); break;
        default: cl_stage<C, 8, INV>(a, b, ld, L, nseq, sg, tw, tid, nthr, keep); break;
      }
    } else {
      switch (sg.radix) {
        case 2: cl_stage<C, 2, INV>(a, b, ld, L, nseq, sg, tw, tid, nthr, post); break;
        case 3: cl_stage<C, 3, INV>(a, b, ld, L, nseq, sg, tw, tid, nthr, post); break;
        case 4: cl_stage<C, 4, INV>(a, b, ld, L, nseq, sg, tw, tid, nthr, post); break;
        default: cl_stage<C, 8, INV>(a, b, ld, L, nseq, sg, tw, tid, nthr, post); break;
      }
    }
    __syncthreads();
    C* t = a;
    a = b;
    b = t;
  }
  return a;
}

template <typename C, bool INV>
__device__ __noinline__ C* cl_fft(C* a, C* b, int ld, const FftPlan* p, const C* tw, int nseq, int tid, int nthr) {
  ClKeep keep;
  return cl_fft_post<C, INV>(a, b, ld, p, tw, nseq, tid, nthr, keep);
}

// Shared-memory state of the dots: two sets of partials, so that a CTA ahead
// of the others may already write the next reduction's while they read.
struct ClShared {
  FieldState fs;
  double part[2][16][4];
  double red[3][16];
  FftPlan fx, fl;
};

template <typename T>
__device__ __forceinline__ void cl_write_dots(ClShared& sh, const Acc<T>* acc, int nd, double scale, int set, int rank,
                                              int C, int tid) {
  const int lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  for (int d = 0; d < nd; ++d) {
    double v;
    if constexpr (sizeof(T) == 4) {
      const float hi = acc[d].s + acc[d].c;
      const float2 t = warp_sum(make_float2(hi, acc[d].c - (hi - acc[d].s)));
      v = (double)t.x + (double)t.y;
    } else {
      v = warp_sum(acc[d].value());
    }
    if (lane == 0) sh.red[d][warp] = v;
  }
  __syncthreads();
  if (warp < nd) {
    const double v = warp_sum(lane < nw ? sh.red[warp][lane] : 0.0) * scale;
    if (lane < C) {
      const uint32_t a = (uint32_t)__cvta_generic_to_shared(&sh.part[set][rank][warp]);
      cl_store(cl_map(a, (uint32_t)lane), v);
    }
  }
}

// After the barrier that follows cl_write_dots: every CTA adds the C partials
// in the same order and runs the recurrence on its own copy of the state.
__device__ __forceinline__ void cl_finish_dots(ClShared& sh, int stage, const SolveConfig& cfg, int nd, int set, int f,
                                               int C, int tid) {
  if (tid < 32) {
    double t[3] = {0.0, 0.0, 0.0};
    for (int d = 0; d < nd; ++d) t[d] = warp_sum(tid < C ? sh.part[set][tid][d] : 0.0);
    if (tid == 0) scalar_update(stage, sh.fs, t, cfg, f);
  }
  __syncthreads();
}

template <typename T>
__global__ void __launch_bounds__(kClusterThreads, 1) k_cluster(const __grid_constant__ ClusterArgs<T> ca) {
  using C = typename cpx<T>::t;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ ClShared sh;
  const PassArgs<T>& a = ca.a;
  const int tid = threadIdx.x, nthr = blockDim.x, CS = ca.csize;
  const int rank = (int)cl_rank(), f = blockIdx.x / CS;
  const int nx = a.nx, M = nx >> 1, L = a.ny, kxn = a.kxn;
  const int rows = L / CS, l0 = rank * rows;            // this CTA's rows
  const int KC = ca.kc, s0 = min(rank * KC, kxn), ns = min(KC, kxn - s0);   // and its sequences
  C* U0 = reinterpret_cast<C*>(smem_raw);
  C* U1 = U0 + ca.buf;
  C* U2 = U1 + ca.buf;
  C* twx = U2 + ca.buf;                                 // M/2 + 1 factors of the real split
  C* tfx = twx + (M / 2 + 1);
  C* tfl = tfx + (M - 1);
  T* gtab = reinterpret_cast<T*>(tfl + (L - 1));        // G_hat of this CTA's sequences (float64)
  // tables, plans, state
  for (int i = tid; i < M / 2 + 1; i += nthr) twx[i] = reinterpret_cast<const C*>(a.twx)[i];
  for (int i = tid; i < M - 1; i += nthr) tfx[i] = reinterpret_cast<const C*>(ca.fx.tw)[i];
  for (int i = tid; i < L - 1; i += nthr) tfl[i] = reinterpret_cast<const C*>(ca.fl.tw)[i];
  if (tid == 0) {
    sh.fx = ca.fx;
    sh.fl = ca.fl;
    sh.fs = FieldState{};
    sh.fs.active = 1;
  }
  auto k2_of = [&](int kx, int i) {
    const int k = i < (L >> 1) ? i : i - L;
    return kx * kx + k * k;
  };
  if (sizeof(T) == 8)                                   // a float64 divide per element is a visible cost: once per solve
    for (int i = tid; i < ns * L; i += nthr) gtab[i] = ghat(a.kc2, T(k2_of(s0 + i / L, i % L)));
  __syncthreads();
  cl_barrier();                                         // every CTA of the cluster runs before any remote store
  const long long base = (long long)f * a.P + (long long)l0 * nx;
  const uint32_t u1s = (uint32_t)__cvta_generic_to_shared(U1), u2s = (uint32_t)__cvta_generic_to_shared(U2);
  SolveConfig cfg = ca.a.cfg;
  if (rank != 0) cfg.hist = nullptr;
  int set = 0;

  // One application of G with the fused prologue, dots and epilogue of `st`.
  auto apply = [&](const ClusterStep& st, bool force) {
    PassArgs<T> v;
    v.ld = ca.ldx; v.W = rows; v.nx = nx; v.rcp_a = a.rcp_a; v.P = a.P;
    v.ncomp = a.ncomp; v.npairs = a.npairs; v.pair_code = a.pair_code;
    v.op = st.xf;
    v.A = (const T*)st.fA; v.B = (const T*)st.fB; v.O1 = (T*)st.fO1; v.O2 = (T*)st.fO2; v.O3 = (T*)st.fO3;
    xfwd_prologue<T, 2>(v, U0, base, sh.fs.iter == 0, T(sh.fs.alpha), T(sh.fs.beta), T(sh.fs.omega), tid, nthr, f);
    __syncthreads();
    C* x = cl_fft<C, false>(U0, U1, ca.ldx, &sh.fx, tfx, rows, tid, nthr);
    // real split of the packed rows (see xfwd_body), written to the owner of sequence kx
    {
      const int h1 = (M >> 1) + 1;
      auto put = [&](int w, int k, const C& val) {
        const int r = fquot(k, ca.rcp_kc);
        cl_store(cl_map(u2s, (uint32_t)r) + (uint32_t)(((k - r * KC) * ca.ldl + phys(l0 + w)) * sizeof(C)), val);
      };
      for (int idx = tid; idx < rows * h1; idx += nthr) {
        const int k = fquot(idx, ca.rcp_own), w = idx - k * rows;
        const C* row = x + w * ca.ldx;
        if (k == 0) {
          const C z0 = row[0];
          put(w, 0, C{z0.x + z0.y, T(0)});
          put(w, M, C{z0.x - z0.y, T(0)});
        } else {
          const C A = row[phys(k)], B = row[phys(M - k)];
          const C e = {T(0.5) * (A.x + B.x), T(0.5) * (A.y - B.y)};
          const C o = {T(0.5) * (A.y + B.y), T(0.5) * (B.x - A.x)};
          const C wo = cmul(twx[k], o);
          put(w, k, cadd(e, wo));
          if (2 * k != M) put(w, M - k, cconj(csub(e, wo)));
        }
      }
    }
    cl_barrier();
    // along y: forward, x G_hat/P with the Parseval dots, inverse
    Acc<T> pd[3];
    {
      const int op = st.fi;
      const T kc2 = a.kc2, gs = a.gscale;
      auto mul = [&](int w, int i, C& X) {
        const T g = sizeof(T) == 8 ? gtab[w * L + i] : ghat(kc2, T(k2_of(s0 + w, i)));
        if (op != FI_NONE) {
          const T wgt = (s0 + w == 0 || s0 + w == M) ? T(1) : T(2);
          const T wm = wgt * (X.x * X.x + X.y * X.y), gw = g * wm;
          if (op == FI_XGX) {
            pd[0].add(gw);
          } else {
            pd[0].add(wm);
            pd[1].add(gw);
            pd[2].add(g * gw);
          }
        }
        const T sc = g * gs;
        X = C{X.x * sc, X.y * sc};
      };
      C* z = cl_fft_post<C, false>(U2, U0, ca.ldl, &sh.fl, tfl, ns, tid, nthr, mul);
      z = cl_fft<C, true>(z, z == U0 ? U2 : U0, ca.ldl, &sh.fl, tfl, ns, tid, nthr);
      // back to the owners of the rows
      for (int idx = tid; idx < ns * L; idx += nthr) {
        const int w = fquot(idx, ca.rcp_l), i = idx - w * L, r = fquot(i, ca.rcp_own);
        cl_store(cl_map(u1s, (uint32_t)r) + (uint32_t)(((s0 + w) * rows + (i - r * rows)) * sizeof(C)),
                 z[w * ca.ldl + phys(i)]);
      }
    }
    if (st.fi != FI_NONE) {
      cl_write_dots(sh, pd, st.fi == FI_XGX ? 1 : 3, 1.0 / (double)a.P, set, rank, CS, tid);
    }
    cl_barrier();
    if (st.fi != FI_NONE) {
      cl_finish_dots(sh, st.fstage, cfg, st.fi == FI_XGX ? 1 : 3, set, f, CS, tid);
      set ^= 1;
      if (!sh.fs.active && !force) return;
    }
    {
      const int h1 = (M >> 1) + 1;
      for (int idx = tid; idx < rows * h1; idx += nthr) {
        const int k = fquot(idx, ca.rcp_own), w = idx - k * rows;
        C* row = U0 + w * ca.ldx;
        if (k == 0) {
          const T x0 = U1[w].x, xm = U1[M * rows + w].x;   // imaginary parts of DC/Nyquist dropped
          row[0] = C{x0 + xm, x0 - xm};
        } else {
          const C A = U1[k * rows + w], B = U1[(M - k) * rows + w];
          const C e = {A.x + B.x, A.y - B.y};
          const C d = {A.x - B.x, A.y + B.y};
          const C o = cmulc(d, twx[k]);
          row[phys(k)] = C{e.x - o.y, e.y + o.x};
          if (2 * k != M) row[phys(M - k)] = C{e.x + o.y, o.x - e.y};
        }
      }
    }
    __syncthreads();
    const C* y = cl_fft<C, true>(U0, U2, ca.ldx, &sh.fx, tfx, rows, tid, nthr);
    v.op = st.xi;
    v.A = (const T*)st.iA; v.B = (const T*)st.iB; v.C = (const T*)st.iC; v.O1 = (T*)st.iO1; v.O2 = (T*)st.iO2;
    Acc<T> acc[3];
    xinv_epilogue<T, 2>(v, y, base, T(sh.fs.alpha), T(sh.fs.omega), acc[0], acc[1], tid, nthr, f);
    if (st.ndots) {
      cl_write_dots(sh, acc, st.ndots, 1.0, set, rank, CS, tid);
      cl_barrier();
      cl_finish_dots(sh, st.istage, cfg, st.ndots, set, f, CS, tid);
      set ^= 1;
    }
  };

  // steps: init [0, b0), one pass [b0, b1) repeated while the field is active, true residual [b1]
  const int b0 = ca.n_init, b1 = b0 + ca.n_body;
  int i = 0, loop = 0;
  for (bool last = false; !last; ++i) {
    if (i >= b0) {
      if (i == b1 && ca.n_body && sh.fs.active && loop < cfg.maxit) {
        i = b0;
        ++loop;
      }
      if (i == b1 || !sh.fs.active) {
        last = true;
        i = b1;
        if (ca.cg_u && sh.fs.fin_axpy) {                // CG: the last pass's u += alpha p
          const T al = T(sh.fs.alpha);
          T* u = (T*)ca.cg_u + base;
          const T* p = (const T*)ca.cg_p + base;
          for (int q = tid; q < rows * (nx >> 2); q += nthr) {
            V4<T> uu = ld4(u + 4 * q), pp = ld4(p + 4 * q);
#pragma unroll
            for (int e = 0; e < 4; ++e) uu.v[e] = fma(al, pp.v[e], uu.v[e]);
            st4(u + 4 * q, uu);
          }
          __syncthreads();
        }
        if (!ca.n_true) break;
      }
    }
    apply(ca.step[i], last);
  }
  if (ca.a.st && rank == 0 && tid == 0) ca.a.st[f] = sh.fs;
}

}  // namespace gad
