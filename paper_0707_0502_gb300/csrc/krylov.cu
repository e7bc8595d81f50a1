// Krylov-basis kernels: classical Gram-Schmidt twice (CGS2) for the Arnoldi
// recurrence A V_m = V_{m+1} Hbar_m (eq. recurAr / recur0), the fused basis
// combination used by the GMRES-DR restart (eq. recur1) and the multi-shift
// solution updates x_i += V_m d_i (GMRES-DR-Sh step 5), and small vector ops.
//
// Every kernel works on a batch of independent columns (grid.y = column); a
// column whose state says `run == 0` is skipped.  Reductions are
// deterministic: each block writes FP64 partials, the last block to finish
// (atomic ticket) sums them in block order.
#include <type_traits>

#include "kernels.cuh"
#include "vecunits.cuh"

namespace {

constexpr int NT = 256;  // threads of the reduction kernels
constexpr int JB = 8;    // basis vectors per register chunk (update)



DEV c128 ldcg128(const c128* p) {
  double2 v = __ldcg(reinterpret_cast<const double2*>(p));
  return {v.x, v.y};
}

// Sum of a complex value over the warp, by halving: the first exchange splits the parts over
// the half-warps, so each lane adds five times instead of ten.  Valid in every lane.
template <typename R>
DEV cx<R> warp_sum(cx<R> a, int lane) {
  const bool h = lane & 16;
  R k = h ? a.y : a.x;
  k += __shfl_xor_sync(FULL, h ? a.x : a.y, 16);
#pragma unroll
  for (int off = 8; off > 0; off >>= 1) k += __shfl_xor_sync(FULL, k, off);
  const R o = __shfl_xor_sync(FULL, k, 16);
  return h ? cx<R>{o, k} : cx<R>{k, o};
}

// Reduce NV complex values over the block; threads < nvalid write out[t].
template <typename R, int NV>
DEV void block_reduce(cx<R> (&acc)[NV], c128* out, int nvalid) {
  __shared__ c128 sred[NT / 32][NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      acc[i].x += __shfl_down_sync(FULL, acc[i].x, off);
      acc[i].y += __shfl_down_sync(FULL, acc[i].y, off);
    }
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < NV; ++i) sred[warp][i] = up(acc[i]);
  }
  __syncthreads();
  if (threadIdx.x < nvalid) {
    c128 s = {0, 0};
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) s += sred[w][threadIdx.x];
    out[threadIdx.x] = s;
  }
  __syncthreads();
}

// sum of the partials p[bk * stride], bk < count (default: one per block), by
// one warp (fixed order: lanes stride the partials, then a shuffle tree),
// result valid in every lane
DEV c128 warp_sum_partials(const c128* p, long stride, int lane, int count = -1) {
  if (count < 0) count = (int)gridDim.x;
  c128 s = {0, 0};
  for (int bk = lane; bk < count; bk += 32) s += ldcg128(p + (long)bk * stride);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    s.x += __shfl_xor_sync(FULL, s.x, off);
    s.y += __shfl_xor_sync(FULL, s.y, off);
  }
  return s;
}

// true in exactly one block per column: the last one to finish
DEV bool last_block(unsigned* cnt) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = (atomicAdd(cnt, 1u) == gridDim.x - 1);
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// Two-level deterministic sum of the per-slot partials part[s * hs + i] (s < S,
// i < nval) into out[i].  Slots come in groups of RG; the last block to finish
// writing a group's slots (`nblk_group` blocks write into it) sums them, one
// thread per value, into gpart[g * hs + i]; the last group sums the group results.
// FP64 adds are costly on this GPU, so no single block sums all S partials.
// Returns true in the one block that wrote `out` (its threads see `out` after a
// __syncthreads()).
constexpr int RG = 16;
DEV bool reduce2(const c128* part, c128* gpart, int hs, int S, int nval, unsigned* gcnt, unsigned* tcnt, int group,
                 unsigned nblk_group, c128* out) {
  __shared__ bool last_g, last_t;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last_g = (atomicAdd(&gcnt[group], 1u) == nblk_group - 1);
  __syncthreads();
  if (!last_g) return false;
  __threadfence();
  const int s0 = group * RG, s1 = min(S, s0 + RG);
  for (int i = threadIdx.x; i < nval; i += NT) {
    c128 acc = {0, 0};
    for (int q = s0; q < s1; ++q) acc += ldcg128(part + (long)q * hs + i);
    gpart[(long)group * hs + i] = acc;
  }
  __threadfence();
  __syncthreads();
  const int ng = (S + RG - 1) / RG;
  if (threadIdx.x == 0) {
    gcnt[group] = 0;
    last_t = (atomicAdd(tcnt, 1u) == (unsigned)ng - 1);
  }
  __syncthreads();
  if (!last_t) return false;
  __threadfence();
  for (int i = threadIdx.x; i < nval; i += NT) {
    c128 acc = {0, 0};
    for (int g = 0; g < ng; ++g) acc += ldcg128(gpart + (long)g * hs + i);
    out[i] = acc;
  }
  if (threadIdx.x == 0) *tcnt = 0;
  return true;
}

// ------------------------------------------------------------ Gram-Schmidt

// h = V^H w (+ ||w||^2): a block stages a tile of w in shared memory, each warp
// takes whole basis vectors and its lanes stream DU units of that vector
// (coalesced, DU loads in flight per lane); one warp reduction per (vector,
// tile), accumulated in FP64.  The grid is S tile slots x G vector groups: the
// block (slot, group) takes the tiles t = slot (mod S) for the vectors of its
// group, and writes one partial per (slot, vector).  Long vectors use G = 1
// (w and V each read once); short ones, with fewer tiles than blocks, split the
// vectors of a tile over G blocks (w re-read G times from L2).

template <typename R>
__global__ void __launch_bounds__(NT, 3) gs_dot_kernel(Batch<R> b, int nv, const cx<R>* __restrict__ W, long wcs,
                                                    c128* __restrict__ hout, int hstride, int wnorm, int S, int G,
                                                    const cx<R>* __restrict__ Wprev) {
  const int c = blockIdx.y;
  if (!b.st[c].run) return;
  constexpr int K = U<R>::K;
  constexpr int DU = DotTile<R>::DU;
  constexpr int TU = DU * 32;  // units per tile
  __shared__ cx<R> wt[TU * K];
  __shared__ c128 accs[GDR_MAX_M + 2];
  const cx<R>* __restrict__ V = b.V + (c / b.vpp) * b.vcs;
  const cx<R>* __restrict__ w = W + c * wcs;
  const long n = b.nvec ? (long)b.nvec[c] : b.n, nu = nunits<R>(n);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nvec_tot = nv + (wnorm ? 1 : 0);
  const int slot = blockIdx.x % S, grp = blockIdx.x / S;
  const int vpg = (nvec_tot + G - 1) / G;
  const int i0 = grp * vpg, i1 = min(nvec_tot, i0 + vpg);
  for (int i = i0 + threadIdx.x; i < i1; i += NT) accs[i] = {0, 0};
  const long ntiles = (nu + TU - 1) / TU;
  for (long t = slot; t < ntiles && i0 < i1; t += S) {
    const long u0 = t * TU;
    __syncthreads();  // readers of the previous tile are done
    for (int q = threadIdx.x; q < TU; q += NT) {
      cx<R> tmp[K];
      if (u0 + q < nu) {
        ldu<R>(w, u0 + q, n, tmp);
      } else {
#pragma unroll
        for (int kk = 0; kk < K; ++kk) tmp[kk] = {0, 0};
      }
#pragma unroll
      for (int kk = 0; kk < K; ++kk) wt[q * K + kk] = tmp[kk];
    }
    __syncthreads();
    for (int i = i0 + warp; i < i1; i += NT / 32) {
      CSum<R> acc;
      if (i < nv) {
        // lazy step: v_{nv-1} is the previous step's unnormalised vector; scale it
        // and store it into V while it is read
        const bool lazy = Wprev && i == nv - 1;
        const cx<R>* vi = lazy ? Wprev + c * wcs : V + (long)i * b.ldv;
        constexpr int LB = sizeof(R) == 8 ? 8 : DU;  // units loaded together
#pragma unroll
        for (int t0 = 0; t0 < DU; t0 += LB) {
          cx<R> vv[LB][K];
#pragma unroll
          for (int tt = 0; tt < LB; ++tt) {
            const long u = u0 + lane + 32 * (t0 + tt);
            if (u < nu) {
              ldu<R>(vi, u, n, vv[tt]);
            } else {
#pragma unroll
              for (int kk = 0; kk < K; ++kk) vv[tt][kk] = {0, 0};
            }
          }
          if (lazy) {
            const R sc = (R)b.st[c].inv_norm;
            cx<R>* vo = b.V + c * b.vcs + (long)i * b.ldv;
#pragma unroll
            for (int tt = 0; tt < LB; ++tt) {
#pragma unroll
              for (int kk = 0; kk < K; ++kk) vv[tt][kk] = sc * vv[tt][kk];
              const long u = u0 + lane + 32 * (t0 + tt);
              if (u < nu) stu<R>(vo, u, n, vv[tt]);
            }
          }
#pragma unroll
          for (int tt = 0; tt < LB; ++tt)
#pragma unroll
            for (int kk = 0; kk < K; ++kk) acc.macc(vv[tt][kk], wt[(lane + 32 * (t0 + tt)) * K + kk]);
        }
      } else {  // ||w||^2
#pragma unroll
        for (int tt = 0; tt < DU; ++tt)
#pragma unroll
          for (int kk = 0; kk < K; ++kk) acc.norm(wt[(lane + 32 * tt) * K + kk]);
      }
      const cx<R> a = warp_sum(acc.value(), lane);
      if (lane == 0) accs[i] += up(a);
    }
  }
  __syncthreads();
  c128* part = b.part + c * b.pstride;
  for (int i = i0 + threadIdx.x; i < i1; i += NT) part[(long)slot * hstride + i] = accs[i];
  const int rg = slot / RG;
  const unsigned nbg = (unsigned)(min(S, (rg + 1) * RG) - rg * RG) * (unsigned)G;
  reduce2(part, part + (long)b.nblk * hstride, hstride, S, nvec_tot, b.gcnt + 64 * c, b.cnt + 4 * c + 1, rg, nbg,
          hout + (long)c * hstride);
}

// First CGS2 update fused with the second projection: per tile, w' = w - V h
// (all nv vectors; written to Wout by the group-0 block of the tile and staged
// in shared memory), then hout = V^H w' for the block's group of vectors, with
// the tile slot / vector group grid and the partials of gs_dot_kernel.  V is
// read once from HBM for both (the dot re-reads the tile from L1/L2).
template <typename R>
__global__ void __launch_bounds__(NT, 2) gs_update_dot_kernel(Batch<R> b, int nv, const cx<R>* __restrict__ W,
                                                           cx<R>* __restrict__ Wout, long wcs,
                                                           const c128* __restrict__ h, c128* __restrict__ hout,
                                                           int hstride, int S, int G) {
  const int c = blockIdx.y;
  if (!b.st[c].run) return;
  constexpr int K = U<R>::K;
  constexpr int DU = DotTile<R>::DU;
  constexpr int TU = DU * 32;
  __shared__ cx<R> wt[TU * K];
  __shared__ cx<R> hs[GDR_MAX_M + 2];
  __shared__ c128 accs[GDR_MAX_M + 2];
  const cx<R>* __restrict__ V = b.V + c * b.vcs;
  const cx<R>* __restrict__ w = W + c * wcs;
  cx<R>* __restrict__ wo = Wout + c * wcs;
  const long n = b.nvec ? (long)b.nvec[c] : b.n, nu = nunits<R>(n);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int slot = blockIdx.x % S, grp = blockIdx.x / S;
  const int vpg = (nv + G - 1) / G;
  const int i0 = grp * vpg, i1 = min(nv, i0 + vpg);
  for (int i = threadIdx.x; i < nv; i += NT) hs[i] = cvt<R>(h[(long)c * hstride + i]);
  for (int i = i0 + threadIdx.x; i < i1; i += NT) accs[i] = {0, 0};
  const long ntiles = (nu + TU - 1) / TU;
  for (long t = slot; t < ntiles; t += S) {
    const long u0 = t * TU;
    __syncthreads();  // hs ready; readers of the previous tile are done
    for (int q = threadIdx.x; q < TU; q += NT) {
      const long u = u0 + q;
      cx<R> acc[K];
      if (u < nu) {
        ldu<R>(w, u, n, acc);
        CSum<R> sum[K];
        for (int g0 = 0; g0 < nv; g0 += JB) {
          cx<R> vv[JB][K];
#pragma unroll
          for (int qq = 0; qq < JB; ++qq)
            if (g0 + qq < nv) ldu<R>(V + (long)(g0 + qq) * b.ldv, u, n, vv[qq]);
#pragma unroll
          for (int qq = 0; qq < JB; ++qq) {
            if (g0 + qq < nv) {
              const cx<R> hi = hs[g0 + qq];
#pragma unroll
              for (int kk = 0; kk < K; ++kk) sum[kk].mac(vv[qq][kk], hi);
            }
          }
        }
#pragma unroll
        for (int kk = 0; kk < K; ++kk) acc[kk] -= sum[kk].value();
        if (grp == 0) stu<R>(wo, u, n, acc);
      } else {
#pragma unroll
        for (int kk = 0; kk < K; ++kk) acc[kk] = {0, 0};
      }
#pragma unroll
      for (int kk = 0; kk < K; ++kk) wt[q * K + kk] = acc[kk];
    }
    __syncthreads();
    for (int i = i0 + warp; i < i1; i += NT / 32) {
      const cx<R>* vi = V + (long)i * b.ldv;
      CSum<R> acc;
      // the tile in two halves (DU/2 loads in flight per lane; the tile is in L1/L2)
#pragma unroll
      for (int t0 = 0; t0 < DU; t0 += DU / 2) {
        cx<R> vv[DU / 2][K];
#pragma unroll
        for (int tt = 0; tt < DU / 2; ++tt) {
          const long u = u0 + lane + 32 * (t0 + tt);
          if (u < nu) {
            ldu<R>(vi, u, n, vv[tt]);
          } else {
#pragma unroll
            for (int kk = 0; kk < K; ++kk) vv[tt][kk] = {0, 0};
          }
        }
#pragma unroll
        for (int tt = 0; tt < DU / 2; ++tt)
#pragma unroll
          for (int kk = 0; kk < K; ++kk) acc.macc(vv[tt][kk], wt[(lane + 32 * (t0 + tt)) * K + kk]);
      }
      const cx<R> a = warp_sum(acc.value(), lane);
      if (lane == 0) accs[i] += up(a);
    }
  }
  __syncthreads();
  c128* part = b.part + c * b.pstride;
  for (int i = i0 + threadIdx.x; i < i1; i += NT) part[(long)slot * hstride + i] = accs[i];
  const int rg = slot / RG;
  const unsigned nbg = (unsigned)(min(S, (rg + 1) * RG) - rg * RG) * (unsigned)G;
  reduce2(part, part + (long)b.nblk * hstride, hstride, S, nv, b.gcnt + 64 * c, b.cnt + 4 * c + 1, rg, nbg,
          hout + (long)c * hstride);
}

template <typename R>
__global__ void __launch_bounds__(NT) gs_update_kernel(Batch<R> b, int nv, cx<R>* __restrict__ W, long wcs,
                                                       const c128* __restrict__ h, int hstride, int final_step) {
  const int c = blockIdx.y;
  if (!b.st[c].run) return;
  constexpr int K = U<R>::K;
  __shared__ cx<R> hs[GDR_MAX_M + 2];
  for (int i = threadIdx.x; i < nv; i += NT) hs[i] = cvt<R>(h[(long)c * hstride + i]);
  __syncthreads();
  const cx<R>* __restrict__ V = b.V + c * b.vcs;
  cx<R>* __restrict__ w = W + c * wcs;
  const long n = b.nvec ? (long)b.nvec[c] : b.n, nu = nunits<R>(n);
  const long gt = blockIdx.x * (long)NT + threadIdx.x, gs = (long)gridDim.x * NT;
  cx<R> nrm[1] = {{0, 0}};
  for (long u = gt; u < nu; u += gs) {
    cx<R> acc[K];
    CSum<R> sum[K];
    ldu<R>(w, u, n, acc);
    // basis vectors in groups of JB: all loads of a group are in flight together
    for (int i0 = 0; i0 < nv; i0 += JB) {
      cx<R> vv[JB][K];
#pragma unroll
      for (int q = 0; q < JB; ++q) {
        if (i0 + q < nv) ldu<R>(V + (long)(i0 + q) * b.ldv, u, n, vv[q]);
      }
#pragma unroll
      for (int q = 0; q < JB; ++q) {
        if (i0 + q < nv) {
          const cx<R> hi = hs[i0 + q];
#pragma unroll
          for (int kk = 0; kk < K; ++kk) sum[kk].mac(vv[q][kk], hi);
        }
      }
    }
#pragma unroll
    for (int kk = 0; kk < K; ++kk) acc[kk] -= sum[kk].value();
    stu<R>(w, u, n, acc);
#pragma unroll
    for (int kk = 0; kk < K; ++kk) nrm[0].x = fma(acc[kk].y, acc[kk].y, fma(acc[kk].x, acc[kk].x, nrm[0].x));
  }
  if (!final_step) return;
  c128* part = b.part + c * b.pstride;
  block_reduce<R, 1>(nrm, part + (long)blockIdx.x * hstride, 1);
  if (!last_block(b.cnt + 4 * c)) return;
  __shared__ double wn_s;
  if (threadIdx.x < 32) {
    const c128 s = warp_sum_partials(part, hstride, threadIdx.x);
    if (threadIdx.x == 0) wn_s = sqrt(s.x);
  }
  __syncthreads();
  const double wn = wn_s;
  const int j = nv - 1;
  const int m = b.m;
  c128* Hc = b.H + (long)c * (m + 1) * m + (long)j * (m + 1);
  for (int i = threadIdx.x; i < nv; i += NT) Hc[i] = b.h1[(long)c * hstride + i] + b.h2[(long)c * hstride + i];
  if (threadIdx.x == 0) {
    Hc[nv] = {wn, 0.0};
    ColState& st = b.st[c];
    const double w0 = sqrt(b.h1[(long)c * hstride + nv].x);
    st.j = j;
    st.wnorm0 = w0;
    if (!isfinite(wn) || !isfinite(w0)) {
      st.nan = 1;
      st.broke = 1;
      st.run = 0;
      st.m_eff = j + 1;
    } else if (wn <= 1e-12 * w0) {
      st.broke = 1;
      st.run = 0;
      st.m_eff = j + 1;
    } else {
      st.inv_norm = 1.0 / wn;
    }
    b.cnt[4 * c] = 0;
  }
}

template <typename R>
__global__ void scale_kernel(Batch<R> b, int j, const cx<R>* __restrict__ W, long wcs) {
  const int c = blockIdx.y;
  if (!b.st[c].run) return;
  constexpr int K = U<R>::K;
  const long n = b.nvec ? (long)b.nvec[c] : b.n, nu = nunits<R>(n);
  const R s = (R)b.st[c].inv_norm;
  const cx<R>* w = W + c * wcs;
  cx<R>* v = b.V + c * b.vcs + (long)j * b.ldv;
  for (long u = blockIdx.x * (long)blockDim.x + threadIdx.x; u < nu; u += (long)gridDim.x * blockDim.x) {
    cx<R> a[K];
    ldu<R>(w, u, n, a);
#pragma unroll
    for (int kk = 0; kk < K; ++kk) a[kk] = s * a[kk];
    stu<R>(v, u, n, a);
  }
}

// ||x_c||^2 with FP64 block partials; result written by the last block
template <typename T> struct Real;
template <> struct Real<c64> { using R = float; };
template <> struct Real<c128> { using R = double; };

template <typename T>
__global__ void __launch_bounds__(NT) norms2_kernel(long n, const T* __restrict__ x, long xcs, double* out,
                                                    c128* part, unsigned* cnt, const int* nvec) {
  using R = typename Real<T>::R;
  const int c = blockIdx.y;
  if (nvec) n = nvec[c];
  const T* xc = x + c * xcs;
  // FP64 per-thread accumulation.  Complex64 vectors carry 2^-24 relative precision, so
  // their squares are summed in FP32 over groups of four elements (relative error
  // <= 8 * 2^-24 per group) and only the group sums in FP64: the FP64 pipe, slow on this
  // part, would otherwise bound the kernel.  FP64 vectors are summed in FP64 throughout.
  double s = 0;
  const long nu = nunits<R>(n), stride = (long)gridDim.x * NT;
  constexpr int K = U<R>::K;
  if (sizeof(R) == 4) {
    for (long u = blockIdx.x * (long)NT + threadIdx.x; u < nu; u += 4 * stride) {  // four 16-byte units in flight
      T v[4][K];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
#pragma unroll
        for (int kk = 0; kk < K; ++kk) v[q][kk] = {0, 0};
        if (u + q * stride < nu) ldu<R>(xc, u + q * stride, n, v[q]);
      }
#pragma unroll
      for (int h = 0; h < 4; h += 2) {
        float f = 0.f;
#pragma unroll
        for (int q = h; q < h + 2; ++q)
#pragma unroll
          for (int kk = 0; kk < K; ++kk)
            f = fmaf((float)v[q][kk].x, (float)v[q][kk].x, fmaf((float)v[q][kk].y, (float)v[q][kk].y, f));
        s += (double)f;
      }
    }
  } else {
    for (long i = blockIdx.x * (long)NT + threadIdx.x; i < n; i += stride) {
      const T v = xc[i];
      s = fma((double)v.y, (double)v.y, fma((double)v.x, (double)v.x, s));
    }
  }
  c128 d[1] = {{s, 0}};
  block_reduce<double, 1>(d, part + (long)c * gridDim.x + blockIdx.x, 1);
  if (!last_block(cnt + 4 * c)) return;
  if (threadIdx.x < 32) {
    const c128 t = warp_sum_partials(part + (long)c * gridDim.x, 1, threadIdx.x);
    if (threadIdx.x == 0) {
      out[c] = t.x;
      cnt[4 * c] = 0;
    }
  }
}

__global__ void __launch_bounds__(NT) dots128_kernel(long n, const c128* __restrict__ u, long ucs,
                                                     const c128* __restrict__ x, long xcs, c128* out, c128* part,
                                                     unsigned* cnt) {
  const int c = blockIdx.y;
  const c128* uc = u + c * ucs;
  const c128* xc = x + c * xcs;
  CSum<double> sum;
  for (long i = blockIdx.x * (long)NT + threadIdx.x; i < n; i += (long)gridDim.x * NT) sum.macc(uc[i], xc[i]);
  c128 a[1] = {sum.value()};
  block_reduce<double, 1>(a, part + (long)c * gridDim.x + blockIdx.x, 1);
  if (!last_block(cnt + 4 * c)) return;
  if (threadIdx.x < 32) {
    const c128 t = warp_sum_partials(part + (long)c * gridDim.x, 1, threadIdx.x);
    if (threadIdx.x == 0) {
      out[c] = t;
      cnt[4 * c] = 0;
    }
  }
}

// start of a cycle: V[:,0] = r / ||r||  (||r||^2 in rn2[c])
template <typename R>
__global__ void start_scale_kernel(Batch<R> b, const cx<R>* __restrict__ r, long rcs, const double* rn2) {
  const int c = blockIdx.y;
  if (!b.st[c].active) return;
  const double rn = sqrt(rn2[c]);
  if (!(rn > 0)) return;
  const R s = (R)(1.0 / rn);
  const cx<R>* rc = r + c * rcs;
  cx<R>* v = b.V + c * b.vcs;
  const long n = b.nvec ? (long)b.nvec[c] : b.n;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    v[i] = s * rc[i];
}

template <typename R>
__global__ void start_state_kernel(Batch<R> b, const double* rn2) {
  const int c = blockIdx.x;
  const int m = b.m;
  c128* H = b.H + (long)c * (m + 1) * m;
  for (long i = threadIdx.x; i < (long)(m + 1) * m; i += blockDim.x) H[i] = {0, 0};
  c128* cv = b.cvec + (long)c * (m + 1);
  const double rn = sqrt(rn2[c]);
  for (int i = threadIdx.x; i <= m; i += blockDim.x) cv[i] = {i == 0 ? rn : 0.0, 0.0};
  if (threadIdx.x == 0) {
    ColState& st = b.st[c];
    st.broke = 0;
    st.m_eff = m;
    st.rnorm = rn;
    if (!isfinite(rn)) st.nan = 1;
    // a zero residual needs no cycle
    st.run = (st.active && rn > 0 && isfinite(rn)) ? 1 : 0;
  }
}

// ------------------------------------------------------ basis combination

constexpr int CT = 256;  // threads
constexpr int CR = 64;   // rows per tile

template <typename R>
__global__ void __launch_bounds__(CT) combine_kernel(long n, cx<R>* V, long ldv, long vcs, int nv,
                                                     const c128* __restrict__ C, int ldc, long ccs, int nout, int nx,
                                                     int rmode, c128* X, long ldx, long xcs, cx<R>* Rv, long rcs,
                                                     const ColState* st, const int* nvec, int vpp, cx<R>* Xf) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int c = blockIdx.y;
  if (st && !st[c].active) return;
  if (nvec) n = nvec[c];
  if ((long)blockIdx.x * CR >= n) return;
  const int ntot = nout + nx + (rmode ? 1 : 0);
  cx<R>* tile = reinterpret_cast<cx<R>*>(smem_raw);             // CR x nv  (row-fast)
  cx<R>* cf = tile + (long)CR * nv;                              // nv x ntot
  cx<R>* Vc = V + (c / vpp) * vcs;                               // basis of column c (nout == 0 when shared)
  const c128* Cc = C + c * ccs;
  const long r0 = blockIdx.x * (long)CR;
  const int rows = (int)min((long)CR, n - r0);
  for (int t = threadIdx.x; t < nv * ntot; t += CT) {
    const int i = t % nv, o = t / nv;
    cf[t] = cvt<R>(Cc[(long)o * ldc + i]);
  }
  for (int t = threadIdx.x; t < CR * nv; t += CT) {
    const int rr = t % CR, i = t / CR;
    tile[t] = (rr < rows) ? Vc[(long)i * ldv + r0 + rr] : cx<R>{0, 0};
  }
  __syncthreads();
  const int rr = threadIdx.x % CR;
  if (rr >= rows) return;
  const long row = r0 + rr;
  for (int o = threadIdx.x / CR; o < ntot; o += CT / CR) {
    CSum<R> sum;
    const cx<R>* co = cf + (long)o * nv;
    for (int i = 0; i < nv; ++i) sum.mac(tile[(long)i * CR + rr], co[i]);
    const cx<R> acc = sum.value();
    if (o < nout) {
      Vc[(long)o * ldv + row] = acc;
    } else if (o < nout + nx) {
      if (Xf) {
        cx<R>* fp = Xf + c * xcs + (long)(o - nout) * ldx + row;
        *fp = *fp + acc;
      } else {
        c128* xp = X + c * xcs + (long)(o - nout) * ldx + row;
        *xp = *xp + up(acc);
      }
    } else {
      cx<R>* rp = Rv + c * rcs + row;
      if (rmode == 1) *rp = acc;
      else *rp = *rp + acc;
    }
  }
}

// Basis combination without in-place outputs (the solution update x_i += V_m d_i of a
// cycle and the residual r = V_{m+1} s, per column with its own basis): rows are
// independent, so each thread takes rows in a grid-stride loop and reads its row of V
// directly (coalesced across the warp); the block stages the column's coefficients once.
// Same summation order as combine_kernel.
constexpr int CW_MAXO = 12, CW_MAXCF = 1280;
template <typename R, int NO>  // NO >= ntot outputs, so no unrolled work is predicated off for nothing
__global__ void __launch_bounds__(256) combine_rows_kernel(long n, const cx<R>* __restrict__ V, long ldv, long vcs,
                                                           int nv, const c128* __restrict__ C, int ldc, long ccs,
                                                           int nx, int rmode, c128* X, long ldx, long xcs, cx<R>* Rv,
                                                           long rcs, const ColState* st, const int* nvec, int vpp,
                                                           cx<R>* Xf) {
  __shared__ cx<R> cf[CW_MAXCF];  // ntot x nv
  const int c = blockIdx.y;
  if (st && !st[c].active) return;
  if (nvec) n = nvec[c];
  const int ntot = nx + (rmode ? 1 : 0);
  const c128* Cc = C + c * ccs;
  for (int t = threadIdx.x; t < nv * ntot; t += 256) {
    const int i = t % nv, o = t / nv;
    cf[t] = cvt<R>(Cc[(long)o * ldc + i]);
  }
  __syncthreads();
  const cx<R>* Vc = V + (c / vpp) * vcs;
  for (long row = blockIdx.x * 256L + threadIdx.x; row < n; row += (long)gridDim.x * 256) {
    CSum<R> acc[NO];
#pragma unroll 4
    for (int i = 0; i < nv; ++i) {
      const cx<R> v = Vc[(long)i * ldv + row];
#pragma unroll
      for (int o = 0; o < NO; ++o)
        if (o < ntot) acc[o].mac(v, cf[o * nv + i]);
    }
#pragma unroll
    for (int o = 0; o < NO; ++o) {
      if (o >= ntot) break;
      const cx<R> a = acc[o].value();
      if (o < nx) {
        if (Xf) {  // correction accumulated in the vectors' precision
          cx<R>* fp = Xf + c * xcs + (long)o * ldx + row;
          *fp = *fp + a;
        } else {
          c128* xp = X + c * xcs + (long)o * ldx + row;
          *xp = *xp + up(a);
        }
      } else {
        cx<R>* rp = Rv + c * rcs + row;
        if (rmode == 1) *rp = a;
        else *rp = *rp + a;
      }
    }
  }
}

// Basis combination for many columns sharing one basis (vcs = 0, no in-place outputs),
// as in the projection over the kept V_{k+1} of the Proj and refinement stages: a
// persistent block stages every column's coefficients once (complex64 or FP64 as the
// vectors, nv x ntot per column) and, for each of its row tiles, the tile of V once,
// then forms every column's outputs from it -- the basis is read from HBM once instead
// of once per column.
template <typename R>
__global__ void __launch_bounds__(CT) combine_shared_kernel(long n, const cx<R>* __restrict__ V, long ldv, int nv,
                                                            const c128* __restrict__ C, int ldc, long ccs, int nx,
                                                            int rmode, c128* X, long ldx, long xcs, cx<R>* Rv,
                                                            long rcs, const ColState* st, int ncol) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int ntot = nx + (rmode ? 1 : 0);
  cx<R>* tile = reinterpret_cast<cx<R>*>(smem_raw);  // CR x nv (row-fast)
  cx<R>* cf = tile + (long)CR * nv;                   // ncol x (nv x ntot)
  const long per = (long)nv * ntot;
  for (long t = threadIdx.x; t < per * ncol; t += CT) {
    const int c = (int)(t / per);
    const int q = (int)(t % per), i = q % nv, o = q / nv;
    cf[t] = cvt<R>(C[c * ccs + (long)o * ldc + i]);
  }
  const long ntiles = (n + CR - 1) / CR;
  const int rr = threadIdx.x % CR;
  for (long tl = blockIdx.x; tl < ntiles; tl += gridDim.x) {
    const long r0 = tl * CR;
    const int rows = (int)min((long)CR, n - r0);
    __syncthreads();  // the previous tile's readers are done (and the coefficients staged)
    for (int t = threadIdx.x; t < CR * nv; t += CT) {
      const int r = t % CR, i = t / CR;
      tile[t] = (r < rows) ? V[(long)i * ldv + r0 + r] : cx<R>{0, 0};
    }
    __syncthreads();
    if (rr >= rows) continue;
    const long row = r0 + rr;
    // the (column, output) pairs, four independent accumulations per thread at a time;
    // the CT / CR = 4 thread groups of a row take interleaved pairs
    const long P = (long)ncol * ntot;
    for (long p0 = threadIdx.x / CR; p0 < P; p0 += 4 * (CT / CR)) {
      CSum<R> acc[4];
      const cx<R>* co[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const long pq = min(p0 + (long)q * (CT / CR), P - 1);
        co[q] = cf + (pq / ntot) * per + (pq % ntot) * nv;
      }
      for (int i = 0; i < nv; ++i) {
        const cx<R> t = tile[(long)i * CR + rr];
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q].mac(t, co[q][i]);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const long pq = p0 + (long)q * (CT / CR);
        if (pq >= P) break;
        const int c = (int)(pq / ntot), o = (int)(pq % ntot);
        if (st && !st[c].active) continue;
        const cx<R> a = acc[q].value();
        if (o < nx) {
          c128* xp = X + c * xcs + (long)o * ldx + row;
          *xp = *xp + up(a);
        } else {
          cx<R>* rp = Rv + c * rcs + row;
          if (rmode == 1) *rp = a;
          else *rp = *rp + a;
        }
      }
    }
  }
}

// h_c = V^H r_c (nv <= NVM basis vectors) for ncol columns sharing one basis V, as in
// the projection c = V_{k+1}^H r of the Proj and refinement stages.  Block (g, slot)
// stages row tiles of V (32 EPL rows x nv, complex64 or FP64 as the vectors) in shared
// memory; its warp w takes column c = 8 g + w, each lane holding its rows of r_c and
// partial sums for every basis vector in registers, flushed to FP64 in shared memory
// every FL tiles.  The column groups of one tile slot are consecutive blocks, so they
// read the same tiles of V close together (L2 reuse): V comes from HBM about once.
// part[(slot * ncol + c) * nv + i] receives each block's FP64 sums; gs_dot_shared_sum
// adds them over the slots in a fixed order.
constexpr int DS_W = 8, DS_EPL = 4, DS_TR = 32 * DS_EPL, DS_FL = 16;

template <typename R, int NVM>
__global__ void __launch_bounds__(DS_W * 32) gs_dot_shared_kernel(long n, const cx<R>* __restrict__ V, long ldv,
                                                                   int nv, const cx<R>* __restrict__ Rv, long rcs,
                                                                   int ncol, const ColState* st, c128* part) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<R>* vt = reinterpret_cast<cx<R>*>(smem_raw);                       // nv x DS_TR
  c128* accd = reinterpret_cast<c128*>(vt + (long)NVM * DS_TR);          // DS_W x NVM
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grp = blockIdx.x, slot = blockIdx.y;
  const int c = grp * DS_W + warp;
  const bool live = c < ncol && (!st || st[c].run);
  for (int i = lane; i < NVM; i += 32) accd[warp * NVM + i] = {0, 0};
  cx<R> acc[NVM];
#pragma unroll
  for (int i = 0; i < NVM; ++i) acc[i] = {0, 0};
  const cx<R>* r = Rv + (long)(live ? c : 0) * rcs;
  const long ntiles = (n + DS_TR - 1) / DS_TR;
  int cnt = 0;
  auto flush = [&]() {
#pragma unroll
    for (int i = 0; i < NVM; ++i) {
      if (i >= nv) break;
      cx<R> a = acc[i];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        a.x += __shfl_xor_sync(FULL, a.x, off);
        a.y += __shfl_xor_sync(FULL, a.y, off);
      }
      if (lane == (i & 31)) accd[warp * NVM + i] += up(a);
      acc[i] = {0, 0};
    }
  };
  for (long tl = slot; tl < ntiles; tl += gridDim.y) {
    const long r0 = tl * DS_TR;
    const int rows = (int)min((long)DS_TR, n - r0);
    __syncthreads();  // the previous tile's readers are done
    for (int t = threadIdx.x; t < nv * DS_TR; t += DS_W * 32) {
      const int i = t / DS_TR, e = t % DS_TR;
      vt[t] = (e < rows) ? V[(long)i * ldv + r0 + e] : cx<R>{0, 0};
    }
    __syncthreads();
    if (!live) continue;
    cx<R> rv[DS_EPL];
#pragma unroll
    for (int q = 0; q < DS_EPL; ++q) {
      const int e = lane + 32 * q;
      rv[q] = (e < rows) ? r[r0 + e] : cx<R>{0, 0};
    }
#pragma unroll
    for (int i = 0; i < NVM; ++i) {
      if (i >= nv) break;
      if constexpr (sizeof(R) == 8) {
        // a tile's four products as one FMA chain, then a single rounding of the long sum (two
        // accumulators per vector would not fit the registers): 9 FP64 instructions a part, not 12
        cx<R> t = cmulc(vt[i * DS_TR + lane], rv[0]);
#pragma unroll
        for (int q = 1; q < DS_EPL; ++q) t = cfma(t, conj(vt[i * DS_TR + lane + 32 * q]), rv[q]);
        acc[i] += t;
      } else {
#pragma unroll
        for (int q = 0; q < DS_EPL; ++q) acc[i] += cmulc(vt[i * DS_TR + lane + 32 * q], rv[q]);
      }
    }
    if (++cnt == DS_FL) {
      flush();
      cnt = 0;
    }
  }
  if (!live) return;
  flush();
  __syncwarp();
  for (int i = lane; i < nv; i += 32) part[((long)slot * ncol + c) * nv + i] = accd[warp * NVM + i];
}

// hout[c * hs + i] = sum over the S slots of part[(slot * ncol + c) * nv + i]: a block takes 32
// values, eight warps every eighth slot each (coalesced over the values), their sums added in
// a fixed order.  One thread per value walking all slots left most of the GPU idle: 16^4, 31
// vectors x 64 columns, 152 slots: eight blocks, ~40 us.
__global__ void __launch_bounds__(256) gs_dot_shared_sum_kernel(int S, int ncol, int nv, const c128* __restrict__ part,
                                                                c128* hout, int hs, const ColState* st) {
  __shared__ c128 sum[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, tot = ncol * nv;
  const int t = blockIdx.x * 32 + lane;
  c128 acc = {0, 0};
  if (t < tot) {
#pragma unroll 8
    for (int q = w; q < S; q += 8) acc += ldcg128(part + (long)q * tot + t);
  }
  sum[w][lane] = acc;
  __syncthreads();
  if (w != 0 || t >= tot) return;
#pragma unroll
  for (int q = 1; q < 8; ++q) acc += sum[q][lane];
  const int c = t / nv, i = t % nv;
  if (st && !st[c].run) return;
  hout[(long)c * hs + i] = acc;
}

// -------------------------------------------------------- small vector ops

__global__ void cvt_128_64_kernel(long n, const c128* in, long ics, c64* out, long ocs) {
  const int c = blockIdx.y;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    out[c * ocs + i] = to64(in[c * ics + i]);
}
__global__ void cvt_64_128_kernel(long n, const c64* in, long ics, c128* out, long ocs) {
  const int c = blockIdx.y;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    out[c * ocs + i] = to128(in[c * ics + i]);
}
__global__ void copy128_kernel(long n, const c128* in, long ics, c128* out, long ocs) {
  const int c = blockIdx.y;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    out[c * ocs + i] = in[c * ics + i];
}
__global__ void axpy_cols_kernel(long n, const c128* a, const c128* S, long ssc, c128* X, long xcs) {
  const int c = blockIdx.y;
  const c128 ac = a[c];
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    X[c * xcs + i] += ac * S[c * ssc + i];
}
__global__ void scal_cols_kernel(long n, const c128* a, c128* X, long xcs) {
  const int c = blockIdx.y;
  const c128 ac = a[c];
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    X[c * xcs + i] = ac * X[c * xcs + i];
}

unsigned grid_for(gdr_ctx* ctx, long work, int threads) {
  long g = (work + threads - 1) / threads;
  long cap = (long)ctx->num_sms * 8;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return (unsigned)g;
}

}  // namespace

// ------------------------------------------------------------- launchers

double run_share(gdr_ctx* ctx, int ncol, const int* run, int run_stride, const int* nvec) {
  if (!ctx->profile || ncol <= 0 || run == nullptr) return 1.0;
  std::vector<int> rf((size_t)ncol * run_stride), nv(nvec ? ncol : 0);
  GDR_CUDA(cudaMemcpyAsync(rf.data(), run, sizeof(int) * ((size_t)(ncol - 1) * run_stride + 1),
                           cudaMemcpyDeviceToHost, ctx->stream));
  if (nvec) GDR_CUDA(cudaMemcpyAsync(nv.data(), nvec, sizeof(int) * ncol, cudaMemcpyDeviceToHost, ctx->stream));
  GDR_CUDA(cudaStreamSynchronize(ctx->stream));
  double all = 0, on = 0;
  for (int c = 0; c < ncol; ++c) {
    const double len = nvec ? (double)nv[c] : 1.0;
    all += len;
    if (rf[(size_t)c * run_stride]) on += len;
  }
  return all > 0 ? on / all : 1.0;
}

// tile slots S x vector groups G of the dot kernels; S <= nblk bounds the partials
template <typename R>
static void dot_grid(gdr_ctx* ctx, const Batch<R>& b, int nvec, int& S, int& G) {
  constexpr long TU = DotTile<R>::DU * 32;
  const long ntiles = (nunits<R>(b.n) + TU - 1) / TU;
  // as many slots as blocks allow, each slot with the same number of tiles (+-1)
  const long rounds = std::max<long>(1, (ntiles + b.nblk - 1) / b.nblk);
  S = (int)std::max<long>(1, std::min<long>((ntiles + rounds - 1) / rounds, b.nblk));
  const long target = 3L * ctx->num_sms;
  G = 1;
  if (S < target) G = (int)std::min<long>((target + S - 1) / S, (nvec + NT / 32 - 1) / (NT / 32));
  G = std::max(G, 1);
}

// tile slots of the shared-basis dot: about two blocks per SM in all
static int dot_shared_slots(gdr_ctx* ctx, long n, int ncol) {
  const int groups = (ncol + DS_W - 1) / DS_W;
  const long ntiles = (n + DS_TR - 1) / DS_TR;
  return (int)std::max<long>(1, std::min<long>(ntiles, std::max(1, 2 * ctx->num_sms / groups)));
}

template <typename R>
static bool dot_shared_applies(const Batch<R>& b, int nv, bool wnorm, const cx<R>* wprev) {
  return b.vcs == 0 && b.ncol > 1 && b.nvec == nullptr && nv <= 48 && !wnorm && !wprev;
}

void gs_dot_shared_reserve(gdr_ctx* ctx, long n, int ncol, int nv) {
  const int S = std::max(dot_shared_slots(ctx, n, ncol), tc_proj_splits(ctx, n, ncol));
  ctx->get<c128>("dsh.part", (size_t)S * ncol * nv + 64);
  if (!ctx->tc_err) {
    ctx->tc_err = ctx->get<int>("tc.err", 4);
    GDR_CUDA(cudaMemsetAsync(ctx->tc_err, 0, sizeof(int) * 4, ctx->stream));
  }
}

// the tensor-core forms for complex64 columns: from this many columns on (with fewer the
// CUDA-core kernels are memory-bound anyway)
constexpr int TC_MIN_COLS = 8;

// vectors i0 .. i0 + nv - 1 of the basis, into h_out + i0
template <typename R, int NVM>
static void gs_dot_shared_launch(gdr_ctx* ctx, const Batch<R>& b, int i0, int nv, const cx<R>* w, long wcs,
                                 c128* h_out) {
  const int S = dot_shared_slots(ctx, b.n, b.ncol);
  c128* part = ctx->get<c128>("dsh.part", (size_t)S * b.ncol * nv + 64);
  const size_t smem = sizeof(cx<R>) * NVM * DS_TR + sizeof(c128) * DS_W * NVM;
  dim3 grid((unsigned)((b.ncol + DS_W - 1) / DS_W), (unsigned)S);
  {
    KProf kp(ctx, sizeof(R) == 4 ? "gs_dot_shared_c64" : "gs_dot_shared_c128",
             ((double)nv * b.n + col_len(b)) * sizeof(cx<R>) * run_share(ctx, b));
    gs_dot_shared_kernel<R, NVM><<<grid, DS_W * 32, smem, ctx->stream>>>(b.n, b.V + (long)i0 * b.ldv, b.ldv, nv, w, wcs,
                                                                          b.ncol, b.st, part);
    GDR_LAUNCHED(ctx);
  }
  const int tot = b.ncol * nv;
  gs_dot_shared_sum_kernel<<<(tot + 31) / 32, 256, 0, ctx->stream>>>(S, b.ncol, nv, part, h_out + i0, b.m + 2, b.st);
  GDR_LAUNCHED(ctx);
}

// whether every vector starts on a 16-byte boundary, as the kernels that load 16-byte units need
template <typename R>
static bool in_units(const cx<R>* p, long ld, int cols) {
  return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && (cols == 1 || ld * sizeof(cx<R>) % 16 == 0);
}

bool gs_dot_tc(gdr_ctx* ctx, long n, int nv, const c64* V, long ldv, int ncol, const c64* R, long ldr, c128* out,
               int hs, const ColState* st, double prof_bytes) {
  if (ncol < TC_MIN_COLS || !ctx->tc_ok || !ctx->tc_proj || !ctx->tc_err) return false;
  c128* part = ctx->get<c128>("dsh.part", (size_t)tc_proj_splits(ctx, n, ncol) * ncol * nv + 64);
  int S = 0;
  if (!tc_proj_dot(ctx, n, V, ldv, nv, R, ldr, ncol, part, ctx->tc_err, S, prof_bytes)) return false;
  const int tot = ncol * nv;
  gs_dot_shared_sum_kernel<<<(tot + 31) / 32, 256, 0, ctx->stream>>>(S, ncol, nv, part, out, hs, st);
  GDR_LAUNCHED(ctx);
  return true;
}

template <typename R>
void gs_dot(gdr_ctx* ctx, const Batch<R>& b, int nv, const cx<R>* w, long wcs, c128* h_out, bool wnorm,
            const cx<R>* wprev) {
  if constexpr (std::is_same<R, float>::value) {
    if (b.vcs == 0 && b.nvec == nullptr && !wnorm && !wprev) {
      const double bytes = ctx->profile ? ((double)nv * b.n + col_len(b)) * sizeof(cx<R>) * run_share(ctx, b) : 0.0;
      if (gs_dot_tc(ctx, b.n, nv, b.V, b.ldv, b.ncol, w, wcs, h_out, b.m + 2, b.st, bytes)) return;
    }
  }
  // one basis for many columns: read it once; and what the unit kernel below cannot load (the
  // caller's complex64 vectors at odd strides or 8-byte starts), 48 vectors at a time
  const bool units = in_units<R>(b.V, b.ldv, nv) && in_units<R>(w, wcs, b.ncol);
  if (dot_shared_applies(b, nv, wnorm, wprev) || (!units && b.vcs == 0 && !b.nvec && !wnorm && !wprev)) {
    for (int i0 = 0; i0 < nv; i0 += 48) {
      const int ni = std::min(48, nv - i0);
      if (ni <= 24) gs_dot_shared_launch<R, 24>(ctx, b, i0, ni, w, wcs, h_out);
      else gs_dot_shared_launch<R, 48>(ctx, b, i0, ni, w, wcs, h_out);
    }
    return;
  }
  GDR_REQUIRE(units, "Gram-Schmidt dot: vectors must start on 16-byte boundaries");
  int S, G;
  dot_grid(ctx, b, nv + (wnorm ? 1 : 0), S, G);
  dim3 grid((unsigned)(S * G), (unsigned)b.ncol);
  KProf kp(ctx, sizeof(R) == 4 ? "gs_dot_c64" : "gs_dot_c128",
           ((double)nv * basis_len(b) + (wprev ? 2.0 : 1.0) * col_len(b)) * sizeof(cx<R>) * run_share(ctx, b));
  gs_dot_kernel<R><<<grid, NT, 0, ctx->stream>>>(b, nv, w, wcs, h_out, b.m + 2, wnorm ? 1 : 0, S, G, wprev);
  GDR_LAUNCHED(ctx);
}
template <typename R>
void gs_update_dot(gdr_ctx* ctx, const Batch<R>& b, int nv, const cx<R>* w, cx<R>* wout, long wcs, const c128* h,
                   c128* h_out) {
  int S, G;
  dot_grid(ctx, b, nv, S, G);
  dim3 grid((unsigned)(S * G), (unsigned)b.ncol);
  KProf kp(ctx, sizeof(R) == 4 ? "gs_update_dot_c64" : "gs_update_dot_c128",
           (double)(nv + 2) * col_len(b) * sizeof(cx<R>) * run_share(ctx, b));
  gs_update_dot_kernel<R><<<grid, NT, 0, ctx->stream>>>(b, nv, w, wout, wcs, h, h_out, b.m + 2, S, G);
  GDR_LAUNCHED(ctx);
}
template <typename R>
void gs_update(gdr_ctx* ctx, const Batch<R>& b, int nv, cx<R>* w, long wcs, const c128* h, bool final_step) {
  dim3 grid((unsigned)b.nblk, (unsigned)b.ncol);
  KProf kp(ctx, sizeof(R) == 4 ? "gs_update_c64" : "gs_update_c128",
           (double)(nv + 2) * col_len(b) * sizeof(cx<R>) * run_share(ctx, b));
  gs_update_kernel<R><<<grid, NT, 0, ctx->stream>>>(b, nv, w, wcs, h, b.m + 2, final_step ? 1 : 0);
  GDR_LAUNCHED(ctx);
}
template <typename R>
void scale_into(gdr_ctx* ctx, const Batch<R>& b, int j, const cx<R>* w, long wcs) {
  dim3 grid(grid_for(ctx, nunits<R>(b.n), 256), (unsigned)b.ncol);
  KProf kp(ctx, "scale", 2.0 * col_len(b) * sizeof(cx<R>) * run_share(ctx, b));
  scale_kernel<R><<<grid, 256, 0, ctx->stream>>>(b, j, w, wcs);
  GDR_LAUNCHED(ctx);
}

template <typename R>
void arnoldi_step(gdr_ctx* ctx, const gdr_op* A, const Batch<R>& b, int j, int jstart, int jlast, cx<R>*& wlast) {
  const int is = (int)(sizeof(ColState) / sizeof(int)), ds = (int)(sizeof(ColState) / sizeof(double));
  const bool lazy = j > jstart;  // v_j = wlast / h_{j,j-1}, not yet in V
  cx<R>* P = lazy ? wlast : nullptr;
  cx<R>* Wa = (P == b.W) ? b.W2 : b.W;  // receives A v_j
  cx<R>* Wb = (Wa == b.W) ? b.W2 : b.W;  // the other buffer (P itself on a lazy step, free after the first dot)
  if (lazy)
    op_apply_skip(ctx, A, b.ncol, nullptr, P, b.wcs, Wa, b.wcs, nullptr, 0, &b.st[0].run, is, b.cpp,
                  &b.st[0].inv_norm, ds);
  else
    op_apply_skip(ctx, A, b.ncol, nullptr, b.V + (long)j * b.ldv, b.vcs, Wa, b.wcs, nullptr, 0, &b.st[0].run, is,
                  b.cpp);
  gs_dot<R>(ctx, b, j + 1, Wa, b.wcs, b.h1, true, P);
  // fused update + second projection while the basis stays in L2 (its tiles are read
  // twice); separate passes otherwise (each reads V once from HBM)
  const bool fuse = (double)(j + 1) * b.n * sizeof(cx<R>) * b.ncol <= 0.5 * (double)ctx->l2_bytes;
  if (fuse) {
    gs_update_dot<R>(ctx, b, j + 1, Wa, Wb, b.wcs, b.h1, b.h2);
    gs_update<R>(ctx, b, j + 1, Wb, b.wcs, b.h2, true);
    wlast = Wb;
  } else {
    gs_update<R>(ctx, b, j + 1, Wa, b.wcs, b.h1, false);
    gs_dot<R>(ctx, b, j + 1, Wa, b.wcs, b.h2, false);
    gs_update<R>(ctx, b, j + 1, Wa, b.wcs, b.h2, true);
    wlast = Wa;
  }
  if (j == jlast) scale_into<R>(ctx, b, j + 1, wlast, b.wcs);
}

template <typename R>
void start_cycle(gdr_ctx* ctx, const Batch<R>& b, const cx<R>* r, long rcs) {
  double* rn2 = ctx->get<double>("start_rn2", b.ncol);
  norms2<cx<R>>(ctx, b.n, b.ncol, r, rcs, rn2, b.part, b.nblk, b.cnt, b.nvec);
  dim3 grid(grid_for(ctx, b.n, 256), (unsigned)b.ncol);
  start_scale_kernel<R><<<grid, 256, 0, ctx->stream>>>(b, r, rcs, rn2);
  GDR_LAUNCHED(ctx);
  start_state_kernel<R><<<b.ncol, 256, 0, ctx->stream>>>(b, rn2);
  GDR_LAUNCHED(ctx);
}

template <typename T>
void norms2(gdr_ctx* ctx, long n, int cols, const T* x, long xcs, double* out, c128* part, int nblk, unsigned* cnt,
            const int* nvec) {
  // enough blocks for the GPU, no more than give each thread a round of loads (16^4, 64 columns:
  // 456 blocks a column, the most the partials allow, left 1.7 elements of each round of four)
  const long want = std::max<long>((8L * ctx->num_sms + cols - 1) / cols, (n * (long)sizeof(T) / 16 + 4 * NT - 1) / (4 * NT) / 4);
  nblk = (int)std::max<long>(1, std::min<long>(nblk, want));
  dim3 grid((unsigned)nblk, (unsigned)cols);
  KProf kp(ctx, sizeof(T) == 8 ? "norms_c64" : "norms_c128", (double)n * sizeof(T) * cols);
  norms2_kernel<T><<<grid, NT, 0, ctx->stream>>>(n, x, xcs, out, part, cnt, nvec);
  GDR_LAUNCHED(ctx);
}
void dots128(gdr_ctx* ctx, long n, int cols, const c128* u, long ucs, const c128* x, long xcs, c128* out, c128* part,
             int nblk, unsigned* cnt) {
  dim3 grid((unsigned)nblk, (unsigned)cols);
  dots128_kernel<<<grid, NT, 0, ctx->stream>>>(n, u, ucs, x, xcs, out, part, cnt);
  GDR_LAUNCHED(ctx);
}

template <typename R>
void combine(gdr_ctx* ctx, long n, int ncol, cx<R>* V, long ldv, long vcs, int nv, const c128* C, int ldc, long ccs,
             int nout, int nx, int rmode, c128* X, long ldx, long xcs, cx<R>* Rv, long rcs, const ColState* st,
             const int* nvec, int vpp, double lenh, double vlenh, cx<R>* Xf) {
  const int ntot = nout + nx + (rmode ? 1 : 0);
  if (ntot == 0 || ncol == 0) return;
  const size_t smem = sizeof(cx<R>) * ((size_t)CR * nv + (size_t)nv * ntot);
  GDR_REQUIRE(smem <= ctx->combine_smem_limit, "combine: too many basis vectors / outputs for shared memory");
  dim3 grid((unsigned)((n + CR - 1) / CR), (unsigned)ncol);
  // V read once per distinct basis, the rest per column
  const double cl = lenh > 0 ? lenh : (double)n * ncol;
  const double vl = vlenh > 0 ? vlenh : (vcs == 0 ? (double)n : (vpp > 1 ? (double)n * ((ncol + vpp - 1) / vpp) : cl));
  const double act = st ? run_share(ctx, ncol, &st[0].run, (int)(sizeof(ColState) / sizeof(int)), nvec) : 1.0;
  // one basis shared by several columns: stream it once for all of them when their
  // coefficients fit in shared memory beside a row tile
  const size_t smem_sh = sizeof(cx<R>) * ((size_t)CR * nv + (size_t)nv * ntot * ncol);
  if (!Xf && std::is_same<R, float>::value && vcs == 0 && nout == 0 && nx == 0 && (rmode == 1 || rmode == 2) &&
      ncol >= TC_MIN_COLS && nvec == nullptr && vpp == 1 && ctx->tc_ok && ctx->tc_proj && ctx->tc_err) {
    const double bytes = ctx->profile ? act * ((double)n * nv + cl * (rmode == 2 ? 2.0 : 1.0)) * sizeof(cx<R>) : 0.0;
    if (tc_proj_update(ctx, n, reinterpret_cast<const c64*>(V), ldv, nv, C, ccs, rmode, reinterpret_cast<c64*>(Rv),
                       rcs, ncol, st, ctx->tc_err, bytes))
      return;
  }
  if (!Xf && vcs == 0 && nout == 0 && ncol > 1 && nvec == nullptr && smem_sh <= ctx->combine_smem_limit) {
    KProf kp(ctx, sizeof(R) == 4 ? "combine_shared_c64" : "combine_shared_c128",
             act * ((double)n * nv * sizeof(cx<R>) +
                    cl * (2.0 * nx * sizeof(c128) + (rmode == 2 ? 2.0 : (rmode == 1 ? 1.0 : 0.0)) * sizeof(cx<R>))));
    const long ntiles = (n + CR - 1) / CR;
    const unsigned g = (unsigned)std::max<long>(1, std::min<long>(ntiles, 2L * ctx->num_sms));
    combine_shared_kernel<R><<<g, CT, smem_sh, ctx->stream>>>(n, V, ldv, nv, C, ldc, ccs, nx, rmode, X, ldx, xcs, Rv,
                                                              rcs, st, ncol);
    GDR_LAUNCHED(ctx);
    return;
  }
  // profiler names by use: basis restart (in-place outputs), solution update, residual only
  const char* pname = nout > 0 ? (sizeof(R) == 4 ? "combine_restart_c64" : "combine_restart_c128")
                      : nx > 0 ? (sizeof(R) == 4 ? "combine_update_c64" : "combine_update_c128")
                               : (sizeof(R) == 4 ? "combine_resid_c64" : "combine_resid_c128");
  if (nout == 0 && ntot <= CW_MAXO && (long)nv * ntot <= CW_MAXCF) {
    KProf kp(ctx, pname,
             act * (vl * nv * sizeof(cx<R>) + cl * (2.0 * nx * (Xf ? sizeof(cx<R>) : sizeof(c128)) +
                                                   (rmode == 2 ? 2.0 : (rmode == 1 ? 1.0 : 0.0)) * sizeof(cx<R>))));
    // enough blocks per column to fill the GPU on its own: late in a batch few columns
    // are still active, and the blocks of the others return at once
    const long rblk = (n + 255) / 256;
    dim3 g((unsigned)std::max<long>(1, std::min(rblk, 8L * ctx->num_sms)), (unsigned)ncol);
#define GDR_ROWS(NO)                                                                                           \
  combine_rows_kernel<R, NO><<<g, 256, 0, ctx->stream>>>(n, V, ldv, vcs, nv, C, ldc, ccs, nx, rmode, X, ldx, xcs, Rv, \
                                                         rcs, st, nvec, vpp, Xf)
    if (ntot <= 1) GDR_ROWS(1);
    else if (ntot <= 2) GDR_ROWS(2);
    else if (ntot <= 4) GDR_ROWS(4);
    else if (ntot <= 8) GDR_ROWS(8);
    else GDR_ROWS(CW_MAXO);
#undef GDR_ROWS
    GDR_LAUNCHED(ctx);
    return;
  }
  KProf kp(ctx, pname,
           act * (vl * nv * sizeof(cx<R>) + cl * (nout * sizeof(cx<R>) + 2.0 * nx * sizeof(c128) +
                                                 (rmode == 2 ? 2.0 : (rmode == 1 ? 1.0 : 0.0)) * sizeof(cx<R>))));
  if (std::is_same<R, float>::value && nout > 0 && rmode == 0 && vpp == 1 && ctx->tc_proj && ctx->tc_err &&
      tc_restart(ctx, n, ncol, reinterpret_cast<c64*>(V), ldv, vcs, nv, C, ldc, ccs, nout, nx, X, ldx, xcs, st, nvec,
                 ctx->tc_err)) {
    kp.rename("tc_restart_c64");
    return;
  }
  combine_kernel<R><<<grid, CT, smem, ctx->stream>>>(n, V, ldv, vcs, nv, C, ldc, ccs, nout, nx, rmode, X, ldx, xcs,
                                                     Rv, rcs, st, nvec, vpp, Xf);
  GDR_LAUNCHED(ctx);
}

void krylov_init(gdr_ctx* ctx) {
  ctx->combine_smem_limit =
      std::min(set_max_dyn_smem(ctx, combine_kernel<float>), set_max_dyn_smem(ctx, combine_kernel<double>));
  ctx->combine_smem_limit = std::min(ctx->combine_smem_limit, set_max_dyn_smem(ctx, combine_shared_kernel<float>));
  ctx->combine_smem_limit = std::min(ctx->combine_smem_limit, set_max_dyn_smem(ctx, combine_shared_kernel<double>));
  set_max_dyn_smem(ctx, gs_dot_shared_kernel<float, 24>);
  set_max_dyn_smem(ctx, gs_dot_shared_kernel<float, 48>);
  set_max_dyn_smem(ctx, gs_dot_shared_kernel<double, 24>);
  set_max_dyn_smem(ctx, gs_dot_shared_kernel<double, 48>);
}

void cvt_128_to_64(gdr_ctx* ctx, long n, int cols, const c128* in, long ics, c64* out, long ocs) {
  dim3 grid(grid_for(ctx, n, 256), (unsigned)cols);
  cvt_128_64_kernel<<<grid, 256, 0, ctx->stream>>>(n, in, ics, out, ocs);
  GDR_LAUNCHED(ctx);
}
void cvt_64_to_128(gdr_ctx* ctx, long n, int cols, const c64* in, long ics, c128* out, long ocs) {
  dim3 grid(grid_for(ctx, n, 256), (unsigned)cols);
  cvt_64_128_kernel<<<grid, 256, 0, ctx->stream>>>(n, in, ics, out, ocs);
  GDR_LAUNCHED(ctx);
}
void copy128(gdr_ctx* ctx, long n, int cols, const c128* in, long ics, c128* out, long ocs) {
  dim3 grid(grid_for(ctx, n, 256), (unsigned)cols);
  copy128_kernel<<<grid, 256, 0, ctx->stream>>>(n, in, ics, out, ocs);
  GDR_LAUNCHED(ctx);
}
void axpy_cols(gdr_ctx* ctx, long n, int cols, const c128* a, const c128* S, long ssc, c128* X, long xcs) {
  dim3 grid(grid_for(ctx, n, 256), (unsigned)cols);
  axpy_cols_kernel<<<grid, 256, 0, ctx->stream>>>(n, a, S, ssc, X, xcs);
  GDR_LAUNCHED(ctx);
}
void scal_cols(gdr_ctx* ctx, long n, int cols, const c128* a, c128* X, long xcs) {
  dim3 grid(grid_for(ctx, n, 256), (unsigned)cols);
  scal_cols_kernel<<<grid, 256, 0, ctx->stream>>>(n, a, X, xcs);
  GDR_LAUNCHED(ctx);
}

template void gs_dot<float>(gdr_ctx*, const Batch<float>&, int, const c64*, long, c128*, bool, const c64*);
template void gs_dot<double>(gdr_ctx*, const Batch<double>&, int, const c128*, long, c128*, bool, const c128*);
template void gs_update<float>(gdr_ctx*, const Batch<float>&, int, c64*, long, const c128*, bool);
template void gs_update<double>(gdr_ctx*, const Batch<double>&, int, c128*, long, const c128*, bool);
template void scale_into<float>(gdr_ctx*, const Batch<float>&, int, const c64*, long);
template void scale_into<double>(gdr_ctx*, const Batch<double>&, int, const c128*, long);
template void arnoldi_step<float>(gdr_ctx*, const gdr_op*, const Batch<float>&, int, int, int, c64*&);
template void arnoldi_step<double>(gdr_ctx*, const gdr_op*, const Batch<double>&, int, int, int, c128*&);
template void start_cycle<float>(gdr_ctx*, const Batch<float>&, const c64*, long);
template void start_cycle<double>(gdr_ctx*, const Batch<double>&, const c128*, long);
template void norms2<c64>(gdr_ctx*, long, int, const c64*, long, double*, c128*, int, unsigned*, const int*);
template void norms2<c128>(gdr_ctx*, long, int, const c128*, long, double*, c128*, int, unsigned*, const int*);
template void combine<float>(gdr_ctx*, long, int, c64*, long, long, int, const c128*, int, long, int, int, int, c128*,
                             long, long, c64*, long, const ColState*, const int*, int, double, double, c64*);
template void combine<double>(gdr_ctx*, long, int, c128*, long, long, int, const c128*, int, long, int, int, int,
                              c128*, long, long, c128*, long, const ColState*, const int*, int, double, double, c128*);
