// Arnoldi steps of the complex64 stages by classical Gram-Schmidt whose second
// (re)orthogonalisation pass is delayed by one step and merged into the next step's
// projection (DCGS2; eq. recurAr / recur0), so a step reads the basis twice (one dot
// pass, one update pass) instead of four times.
//
// At step j the basis v_0..v_{j-1} is final and u (the provisional v_j) is orthogonalised
// once and unnormalised, with A v_{j-1} = V_j Hbar[0:j, j-1] + u.  With w = A u, one pass
// gives s = V_j^H u, z = V_j^H w, omega = u^H u, zeta = u^H w; then
//   nu = sqrt(omega - |s|^2),  v_j = (u - V_j s) / nu,
//   Hbar[0:j, j-1] += s,  Hbar[j, j-1] = nu                (the delayed pass for step j-1)
//   t = (zeta - s^H z) / nu,  Hbar[0:j+1, j] = ([z ; t] - Hbar[0:j+1, 0:j] s) / nu
//   u' = (w - V_j z - t v_j) / nu = (w - V_j (z - (t/nu) s) - (t/nu) u) / nu,
// u' being the next step's provisional vector (A v_j = V_{j+1} Hbar[0:j+1, j] + u').
// The first step of a cycle starts from a final v_j (s = 0, nu = 1); after the last
// step a finalising pass (dot + update without w) makes v_m from u.  Lucky breakdown
// of step j-1 (nu <= 1e-12 ||A v_{j-1}||) is detected at step j: m_eff = j.
//
// Every kernel works on a batch of columns (grid.y = column); a column whose state says
// `run == 0` is skipped.  Reductions are deterministic: blocks write FP64 partials, the
// last block of a slot group and the last group sum them in order.
//
// What a step hands over, per column, at stride 2m + 8: hd (FP64): s_i, z_i interleaved
// (i < j), nu, t;  dc (as complex64): a = s (m + 1 slots), b = z - (t/nu) s (m + 1
// slots), t/nu, 1/nu -- the update's coefficients in the precision it uses them in.
#include <type_traits>

#include "async.cuh"
#include "kernels.cuh"
#include "vecunits.cuh"

namespace {

constexpr int NT = 256, NW = NT / 32;
constexpr int DC_FIRST = 1, DC_FINAL = 2;
constexpr int DU = 8;    // most 16-byte units per lane of a warp's slab
constexpr int NST = 3;   // vectors in flight per warp
constexpr int RG = 16;   // partial slots per group of the two-level reduction

DEV c128 ldcg128(const c128* p) {
  const double2 v = __ldcg(reinterpret_cast<const double2*>(p));
  return {v.x, v.y};
}
// acc + conj(a) b as FMA chains
DEV c64 fmac(c64 acc, c64 a, c64 b) {
  return {fmaf(a.y, b.y, fmaf(a.x, b.x, acc.x)), fmaf(-a.y, b.x, fmaf(a.x, b.y, acc.y))};
}

// sum over the warp of the four floats (a.x, a.y, w.x, w.y), by halving: two exchanges,
// then one each -- six shuffles instead of twenty.  Lane 8k holds value k.
DEV float warp_sum4(c64 a, c64 w, int lane) {
  const bool h16 = lane & 16, h8 = lane & 8;
  float k0 = h16 ? w.x : a.x, k1 = h16 ? w.y : a.y;
  const float g0 = h16 ? a.x : w.x, g1 = h16 ? a.y : w.y;
  k0 += __shfl_xor_sync(FULL, g0, 16);
  k1 += __shfl_xor_sync(FULL, g1, 16);
  float r = h8 ? k1 : k0;
  r += __shfl_xor_sync(FULL, h8 ? k0 : k1, 8);
  r += __shfl_xor_sync(FULL, r, 4);
  r += __shfl_xor_sync(FULL, r, 2);
  r += __shfl_xor_sync(FULL, r, 1);
  return r;
}

// the same for three FP64 values, six additions instead of fifteen (an FP64 instruction holds
// its pipe for ~64 cycles a warp).  Lanes 0, 8, 16 hold x, y, z.
DEV double warp_sum3(double x, double y, double z, int lane) {
  const bool h16 = lane & 16, h8 = lane & 8;
  double k0 = h16 ? z : x, k1 = h16 ? 0.0 : y;
  k0 += __shfl_xor_sync(FULL, h16 ? x : z, 16);
  k1 += __shfl_xor_sync(FULL, h16 ? y : 0.0, 16);
  double r = h8 ? k1 : k0;
  r += __shfl_xor_sync(FULL, h8 ? k0 : k1, 8);
  r += __shfl_xor_sync(FULL, r, 4);
  r += __shfl_xor_sync(FULL, r, 2);
  r += __shfl_xor_sync(FULL, r, 1);
  return r;
}

// 1/sqrt(x) for a positive normal x: Newton's iteration y <- y + y/2 (1 - x y^2) from an
// FP32 starting value (x scaled by a power of four into its range), 2^-22 -> 2^-43 -> FP64
// rounding: nine dependent FP64 instructions where sqrt and a division take over twenty.
DEV double rsqrt_newton(double x) {
  const long long bits = __double_as_longlong(x);
  const int e = (int)((bits >> 52) & 0x7ff) - 1023, h = e >> 1;  // x = 4^h xs, xs in [1, 4)
  const double xs = __longlong_as_double(bits - (long long)(2 * h) * (1LL << 52));
  double y = (double)rsqrtf((float)xs);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const double r = fma(-xs * y, y, 1.0);
    y = fma(0.5 * y, r, y);
  }
  return y * __longlong_as_double((long long)(1023 - h) * (1LL << 52));
}

// atomicAdd that releases the block's earlier writes (all threads', ordered before by a block
// barrier) and acquires those of the blocks that came before: no fence per thread
DEV unsigned ticket(unsigned* p) {
  unsigned r;
  asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(r) : "l"(p) : "memory");
  return r;
}

// sum over the slots q0..q1-1 of part[q * hs + i], by two neighbouring lanes (even, odd slots),
// valid in both
DEV c128 slot_sum2(const c128* part, int hs, int i, int q0, int q1, int half) {
  c128 acc = {0, 0};
#pragma unroll 8
  for (int q = q0 + half; q < q1; q += 2) acc += ldcg128(part + (long)q * hs + i);
  acc.x += __shfl_xor_sync(FULL, acc.x, 1);
  acc.y += __shfl_xor_sync(FULL, acc.y, 1);
  return acc;
}

// Dot pass.  HBM bounds it (V_j read once, u and w once), so what matters is bytes in
// flight.  Each warp holds its slab of u and w (du <= 8 units per lane) in registers and
// streams the vectors of its group through it from a ring of its own in shared memory,
// NST bulk copies of up to 4 KB ahead: neither registers nor the warp's own reductions
// hold the loads back, and no block barrier is met before the end.  The grid is S slots x
// G vector groups; slab width and groups are chosen by dcgs2_plan.
__global__ void __launch_bounds__(NT, 2) dcgs2_dot_kernel(Batch<float> b, int j, const c64* __restrict__ Uv, long ucs,
                                                       const c64* __restrict__ W, long wcs, int S, int G, int du,
                                                       int mode) {
  const int c = blockIdx.y;
  const int run = b.st[c].run;  // tested once the barriers are set up
  extern __shared__ __align__(128) unsigned char ring_raw[];
  __shared__ c64 accw[NW][2 * GDR_MAX_M + 8];
  __shared__ __align__(8) uint64_t full[NW][NST];
  __shared__ int abort_s;
  const bool hasw = mode != DC_FINAL;
  const c64* __restrict__ V = b.V + c * b.vcs;
  const c64* __restrict__ u = Uv + c * ucs;
  const c64* __restrict__ w = W + c * wcs;
  const long n = b.nvec ? (long)b.nvec[c] : b.n, nu = nunits<float>(n);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nvec_tot = j + 1;  // j basis vectors and the self terms
  const int slot = blockIdx.x % S, grp = blockIdx.x / S;
  const int vpg = (nvec_tot + G - 1) / G;
  const int i0 = grp * vpg, i1 = min(nvec_tot, i0 + vpg), iv1 = min(i1, j);
  const int hs = 2 * b.m + 8;
  const int v0 = 2 * i0, v1 = i0 < i1 ? 2 * i1 + (i1 == nvec_tot ? 1 : 0) : v0;  // value range of this block
  if (threadIdx.x < NW * NST) mbar_init(&full[0][0] + threadIdx.x, 1);
  if (threadIdx.x == 0) abort_s = 0;
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  for (int v = v0 + lane; v < v1; v += 32) accw[warp][v] = {0, 0};
  if (!run) return;
  __syncthreads();
  const int SU = 32 * du;  // units per slab
  const long nslab = i0 < i1 ? (nu + SU - 1) / SU : 0, dsl = (long)S * NW;
  unsigned char* ring = ring_raw + (size_t)warp * NST * SU * 16;
  long psl = (long)slot * NW + warp;  // next copy: slab psl, vector pi
  int pi = i0, issued = 0;
  auto issue = [&]() {
    if (psl >= nslab || i0 >= iv1) return;
    if (lane == 0) {
      const long ub = psl * SU;
      const unsigned bytes = (unsigned)min((long)SU, nu - ub) * 16u;
      uint64_t* bar = &full[warp][issued % NST];
      mbar_arrive_tx(bar, bytes);
      bulk_load(ring + (size_t)(issued % NST) * SU * 16, V + (long)pi * b.ldv + 2 * ub, bytes, bar);
    }
    ++issued;
    if (++pi == iv1) {
      pi = i0;
      psl += dsl;
    }
  };
#pragma unroll
  for (int q = 0; q < NST; ++q) issue();
  int used = 0;
  bool dead = false;
  for (long sl = (long)slot * NW + warp; sl < nslab && !dead; sl += dsl) {
    const long q0 = sl * SU + lane;
    c64 uu[DU][2], ww[DU][2];
#pragma unroll
    for (int t = 0; t < DU; ++t) {
#pragma unroll
      for (int kk = 0; kk < 2; ++kk) uu[t][kk] = ww[t][kk] = {0, 0};
      if (t < du && q0 + 32 * t < nu) {
        ldu<float>(u, q0 + 32 * t, n, uu[t]);
        if (hasw) ldu<float>(w, q0 + 32 * t, n, ww[t]);
      }
    }
    for (int i = i0; i < iv1; ++i, ++used) {
      const int stg = used % NST;
      dead = !__all_sync(FULL, mbar_wait(&full[warp][stg], (unsigned)(used / NST) & 1u, &abort_s));
      if (dead) break;
      const float4* vs = reinterpret_cast<const float4*>(ring + (size_t)stg * SU * 16) + lane;
      c64 au[2] = {{0, 0}, {0, 0}}, aw[2] = {{0, 0}, {0, 0}};  // short chains: FP32 rounding grows with their length
#pragma unroll
      for (int t = 0; t < DU; ++t) {
        if (t < du && q0 + 32 * t < nu) {  // a stage's bytes past the vector's end are stale
          const float4 v = vs[32 * t];
          const c64 a = {v.x, v.y};
          c64 d = {v.z, v.w};
          if ((n & 1) && q0 + 32 * t == nu - 1) d = {0, 0};  // the padding after an odd length
          au[0] = fmac(au[0], a, uu[t][0]);
          au[1] = fmac(au[1], d, uu[t][1]);
          aw[0] = fmac(aw[0], a, ww[t][0]);
          aw[1] = fmac(aw[1], d, ww[t][1]);
        }
      }
      const float r = warp_sum4(au[0] + au[1], aw[0] + aw[1], lane);
      if ((lane & 7) == 0) reinterpret_cast<float*>(accw[warp])[4 * i + (lane >> 3)] += r;
      __syncwarp();
      // refill only now: the store above depends on every value read from the stage
      issue();
    }
    if (i1 == nvec_tot) {  // omega = u^H u, zeta = u^H w, w^H w
      c64 om[2] = {{0, 0}, {0, 0}}, ze[2] = {{0, 0}, {0, 0}};  // om: |u|^2, |w|^2
#pragma unroll
      for (int t = 0; t < DU; ++t)
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) {
          om[kk].x = fmaf(uu[t][kk].y, uu[t][kk].y, fmaf(uu[t][kk].x, uu[t][kk].x, om[kk].x));
          om[kk].y = fmaf(ww[t][kk].y, ww[t][kk].y, fmaf(ww[t][kk].x, ww[t][kk].x, om[kk].y));
          ze[kk] = fmac(ze[kk], uu[t][kk], ww[t][kk]);
        }
      const float r = warp_sum4(om[0] + om[1], ze[0] + ze[1], lane);
      // values 2j: (omega, 0), 2j + 1: zeta, 2j + 2: (w^H w, 0)
      if ((lane & 7) == 0) {
        const int k = lane >> 3;
        reinterpret_cast<float*>(accw[warp])[4 * j + (k == 0 ? 0 : k == 1 ? 4 : k)] += r;
      }
      __syncwarp();
    }
  }
  if (dead) {  // a wait gave up: the column is marked, the copies still in flight are waited for (bounded)
    for (; used < issued; ++used) {
      int own = 0;
      mbar_wait(&full[warp][used % NST], (unsigned)(used / NST) & 1u, &own);
    }
    if (lane == 0) atomicCAS(&b.st[c].err, 0, (int)GDR_ETIMEOUT);
  }
  __syncthreads();
  // the block's sums, the eight warps by a tree of fixed order, FP64: eight lanes per value
  c128* part = b.part + c * b.pstride;
  for (int vb = v0; vb < v1; vb += NT / 8) {
    const int v = vb + (int)(threadIdx.x >> 3);
    c128 a = {0, 0};
    if (v < v1) a = up(accw[threadIdx.x & 7][v]);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      a.x += __shfl_xor_sync(FULL, a.x, o);
      a.y += __shfl_xor_sync(FULL, a.y, o);
    }
    if ((threadIdx.x & 7) == 0 && v < v1) part[(long)slot * hs + v] = a;
  }

  // ---- two-level sum over the slots, into shared memory of the last block
  __shared__ bool last_s;
  __shared__ double red_s[NW][4];  // |s|^2, Re and Im of s^H z
  __shared__ double wn_s;
  __shared__ c128 t_s;
  __shared__ int brk_s;
  c128* sval = reinterpret_cast<c128*>(ring_raw);  // the ring has been read
  const int nval = 2 * j + 3, ng = (S + RG - 1) / RG, rg = slot / RG;
  c128* gpart = part + (long)b.nblk * hs;
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned nbg = (unsigned)(min(S, (rg + 1) * RG) - rg * RG) * (unsigned)G;
    last_s = ticket(&b.gcnt[64 * c + rg]) == nbg - 1;
  }
  __syncthreads();
  if (!last_s) return;
  const int half = threadIdx.x & 1;
  for (int ib = 0; ib < nval; ib += NT / 2) {
    const int i = ib + (int)(threadIdx.x >> 1), s0 = rg * RG, s1 = i < nval ? min(S, s0 + RG) : s0;
    const c128 acc = slot_sum2(part, hs, i, s0, s1, half);
    if (half || i >= nval) continue;
    if (ng == 1) sval[i] = acc;
    else gpart[(long)rg * hs + i] = acc;
  }
  if (ng > 1) {
    __syncthreads();
    if (threadIdx.x == 0) {
      b.gcnt[64 * c + rg] = 0;
      last_s = ticket(&b.cnt[4 * c + 1]) == (unsigned)ng - 1;
    }
    __syncthreads();
    if (!last_s) return;
    for (int ib = 0; ib < nval; ib += NT / 2) {
      const int i = ib + (int)(threadIdx.x >> 1);
      const c128 acc = slot_sum2(gpart, hs, i, 0, i < nval ? ng : 0, half);
      if (!half && i < nval) sval[i] = acc;
    }
    if (threadIdx.x == 0) b.cnt[4 * c + 1] = 0;
  } else if (threadIdx.x == 0) {
    b.gcnt[64 * c + rg] = 0;
  }
  __syncthreads();

  // ---- coefficients.  FP64 instructions occupy their pipe for ~64 cycles a warp here, so each
  // value is formed once, in as few warps as hold the j values; Hbar's columns, which no
  // one waits for, are formed by the update kernel's extra block.
  const int m = b.m, i = threadIdx.x;
  const bool first = mode == DC_FIRST;
  const int nwj = (j + 31) / 32;  // warps that hold values (j <= 96)
  c128 si = {0, 0}, zi = {0, 0};
  if (warp < nwj) {
    if (i < j) {
      if (!first) si = sval[2 * i];
      zi = sval[2 * i + 1];
    }
    const c128 szp = cmulc(si, zi);
    const double r = warp_sum3(norm2(si), szp.x, szp.y, lane);
    if ((lane & 7) == 0) red_s[warp][lane >> 3] = r;
  }
  // beside it, on another warp's pipe: ||w||
  if (threadIdx.x == NT - 32) wn_s = mode != DC_FINAL ? sqrt(sval[2 * j + 2].x) : 0.0;
  __syncthreads();
  ColState& st = b.st[c];
  c128* hv = b.hd + (long)c * hs;
  c64* df = reinterpret_cast<c64*>(b.dc + (long)c * hs);
  if (threadIdx.x == 0) {
    double ss = 0;
    c128 sz = {0, 0};
    for (int q = 0; q < nwj; ++q) {
      ss += red_s[q][0];
      sz += c128{red_s[q][1], red_s[q][2]};
    }
    const double omega = sval[2 * j].x;
    // nu and 1/nu by the iteration where nu^2 is in its range, else by sqrt and a division
    const double nu2 = fmax(omega - ss, 0.0);
    const bool plain = nu2 > 1e-290 && nu2 < 1e290;
    double inu = first ? 1.0 : plain ? rsqrt_newton(nu2) : 0.0;
    const double nuv = first ? 1.0 : plain ? nu2 * inu : sqrt(nu2);
    int brk = 0;
    if (!first) {
      if (!isfinite(nuv) || !isfinite(omega)) {
        st.nan = 1;
        brk = 1;
      } else if (nuv <= 1e-12 * st.wnorm0) {
        brk = 1;
      }
      if (brk) {
        b.H[(long)c * (m + 1) * m + (long)(j - 1) * (m + 1) + j] = {nuv, 0.0};
        st.broke = 1;
        st.run = 0;
        st.m_eff = j;
      }
    }
    if (!brk) {
      if (!first && !plain) inu = 1.0 / nuv;
      st.inv_norm = inu;
      st.j = j;
      hv[2 * j] = {nuv, 0.0};
      if (mode != DC_FINAL) {
        const c128 t = inu * (sval[2 * j + 1] - sz);
        const c128 tn = inu * t;
        df[2 * (m + 1)] = to64(tn);
        hv[2 * j + 1] = t;
        t_s = tn;
        st.wnorm0 = wn_s * inu;
        if (!isfinite(wn_s)) {
          st.nan = 1;
          st.broke = 1;
          st.run = 0;
          st.m_eff = j + 1;
          brk = 1;
        }
      }
      df[2 * (m + 1) + 1] = {(float)inu, 0.f};
    }
    brk_s = brk;
  }
  __syncthreads();
  if (brk_s || i >= j) return;
  df[i] = to64(si);
  hv[2 * i] = si;
  if (mode == DC_FINAL) return;
  hv[2 * i + 1] = zi;
  df[(m + 1) + i] = to64(zi - t_s * si);
}

// Hbar of step j: the delayed pass completes column j-1 and column j follows.  H s is of
// rounding size, so it is formed in FP32 from a copy of Hbar (rebuilt on a cycle's first
// step, since the restart may have rewritten the kept columns).  Not inlined: the update
// kernel's registers (58: four blocks per SM) are its streaming loop's own.
__device__ __noinline__ void dcgs2_hbar(const Batch<float>& b, int c, int j, int mode) {
  __shared__ c64 s32[GDR_MAX_M + 1];
  const int m = b.m;
  const bool first = mode == DC_FIRST;
  c128* H = b.H + (long)c * (m + 1) * m;
  c64* Hf = b.Hf + (long)c * (m + 1) * m;
  const c128* hv = b.hd + (long)c * (2 * m + 8);
  const double nuv = hv[2 * j].x;
  if (first)
    for (int q = threadIdx.x; q < j * (m + 1); q += NT) Hf[q] = to64(H[q]);
  if (!first)
    for (int i = threadIdx.x; i <= j; i += NT) {
      c128& hij = H[(long)(j - 1) * (m + 1) + i];
      hij = i < j ? hij + hv[2 * i] : c128{nuv, 0.0};
      Hf[(long)(j - 1) * (m + 1) + i] = to64(hij);
    }
  if (mode == DC_FINAL) return;
  for (int i = threadIdx.x; i < j; i += NT) s32[i] = to64(hv[2 * i]);
  __syncthreads();
  // the copy's rows below the subdiagonal are zero, as H's are
  for (int i = j + 1 + threadIdx.x; i <= m; i += NT) Hf[(long)j * (m + 1) + i] = {0.f, 0.f};
  const double inu = 1.0 / nuv;
  for (int i = threadIdx.x; i <= j; i += NT) {
    c64 hsum = {0.f, 0.f};
    if (!first) {
#pragma unroll 8
      for (int l = 0; l < j; ++l) hsum += Hf[(long)l * (m + 1) + i] * s32[l];
    }
    const c128 zi = i < j ? hv[2 * i + 1] : hv[2 * j + 1];
    const c128 hnew = inu * (zi - to128(hsum));
    H[(long)j * (m + 1) + i] = hnew;
    Hf[(long)j * (m + 1) + i] = to64(hnew);
  }
}

// DCGS2 update pass of step j (every unit of every running column):
//   v_j = (u - V_j a) / nu      into V[:, j]   (not on the first step: v_j is final)
//   u'  = (w - V_j b - (t/nu) u) / nu  into Unew (may alias u; not on the finalising pass)
// and, in one extra block per column, Hbar.  JB vectors are loaded together.
template <int JB>
__global__ void __launch_bounds__(NT) dcgs2_update_kernel(Batch<float> b, int j, const c64* Uv, long ucs,
                                                          const c64* __restrict__ W, c64* Unew, int mode) {
  const int c = blockIdx.y;
  if (!b.st[c].run) return;
  if (blockIdx.x == 0) {  // first, so that it runs beside the others
    dcgs2_hbar(b, c, j, mode);
    return;
  }
  const int m = b.m, hs = 2 * m + 8;
  __shared__ c64 sa[GDR_MAX_M + 1], sb[GDR_MAX_M + 1];
  const c64* df = reinterpret_cast<const c64*>(b.dc + (long)c * hs);
  const bool first = mode == DC_FIRST, fin = mode == DC_FINAL;
  for (int i = threadIdx.x; i < j; i += NT) {
    sa[i] = df[i];
    if (!fin) sb[i] = df[(m + 1) + i];
  }
  const c64 tnu = fin ? c64{0, 0} : df[2 * (m + 1)];
  const float inu = df[2 * (m + 1) + 1].x;
  __syncthreads();
  const c64* __restrict__ V = b.V + c * b.vcs;
  const c64* u = Uv + c * ucs;
  const c64* __restrict__ w = W + c * b.wcs;
  c64* un = Unew + c * b.wcs;
  c64* vj = b.V + c * b.vcs + (long)j * b.ldv;
  const long n = b.nvec ? (long)b.nvec[c] : b.n, nu = nunits<float>(n);
  const long gt = (blockIdx.x - 1) * (long)NT + threadIdx.x, gs = (long)(gridDim.x - 1) * NT;
  for (long q = gt; q < nu; q += gs) {
    c64 uu[2], acc_a[2], acc_b[2];
    ldu<float>(u, q, n, uu);
    if (!fin) {
      ldu<float>(w, q, n, acc_b);
    } else {
      acc_b[0] = acc_b[1] = {0, 0};
    }
    acc_a[0] = uu[0];
    acc_a[1] = uu[1];
    for (int g0 = 0; g0 < j; g0 += JB) {
      c64 vv[JB][2];
#pragma unroll
      for (int qq = 0; qq < JB; ++qq)
        if (g0 + qq < j) ldu<float>(V + (long)(g0 + qq) * b.ldv, q, n, vv[qq]);
#pragma unroll
      for (int qq = 0; qq < JB; ++qq) {
        if (g0 + qq < j) {
          const c64 ai = sa[g0 + qq], bi = sb[g0 + qq];
#pragma unroll
          for (int kk = 0; kk < 2; ++kk) {
            // the product first: one rounding at the accumulator's magnitude per vector (as two
            // chained FMAs each component takes two, and v_j's error grew by a third)
            if (!first) acc_a[kk] -= vv[qq][kk] * ai;
            if (!fin) acc_b[kk] -= vv[qq][kk] * bi;
          }
        }
      }
    }
    if (!first) {
      const c64 o[2] = {inu * acc_a[0], inu * acc_a[1]};
      stu<float>(vj, q, n, o);
    }
    if (!fin) {
      const c64 o[2] = {inu * (acc_b[0] - tnu * uu[0]), inu * (acc_b[1] - tnu * uu[1])};
      stu<float>(un, q, n, o);
    }
  }
}

// Slots S, vector groups G and slab width du of the dot pass: those that need the fewest
// (waves of the two blocks resident per SM) x (rounds x vectors x units per lane + a fixed
// part), the fixed part (u, w, the block's sums) being worth about three vectors.  One
// column of 24^3x32 has 10,368 slabs of eight units for 2,432 resident warps, five rounds
// for 4.3 of work: seven units give 4.9; one column of 16^4 or 8^4 fills the GPU only with
// its vectors split over several blocks.  At most four rounds for several columns: late in
// a batch few are still active, and their blocks alone should fill the GPU.
struct DotPlan {
  int S, G, du;
};
DotPlan dcgs2_plan(const gdr_ctx* ctx, const Batch<float>& b, int nvec) {
  const long nu = nunits<float>(b.n), resident = 2L * ctx->num_sms;
  DotPlan best{1, 1, DU};
  double cost = 1e300;
  auto consider = [&](int du, long rounds, int G) {
    const long tiles = (nu + 32L * du * NW - 1) / (32L * du * NW), S = (tiles + rounds - 1) / rounds;
    if (S > b.nblk) return;
    const int vpg = (nvec + G - 1) / G;
    if (G > 1 && (nvec + vpg - 1) / vpg != G) return;  // an empty group
    const long waves = (S * G * b.ncol + resident - 1) / resident;
    const double t = (double)waves * (24.0 + (double)rounds * vpg * du);
    if (t < cost) {
      cost = t;
      best = {(int)S, G, du};
    }
  };
  const long most = b.ncol > 1 ? 4 : 64;
  for (int du = DU; du >= 2; --du) {
    for (int G = 2; G <= std::min(nvec, 32); ++G) consider(du, 1, G);
    const long tiles = (nu + 32L * du * NW - 1) / (32L * du * NW);
    for (long r = 1; r <= std::min(tiles, most); ++r) consider(du, r, 1);
  }
  if (cost == 1e300) {  // a vector longer than `most` rounds of nblk blocks: as many rounds as it takes
    const long tiles = (nu + 32L * DU * NW - 1) / (32L * DU * NW);
    best.S = (int)std::min<long>(tiles, b.nblk);
  }
  return best;
}

}  // namespace

void dcgs2_init(gdr_ctx* ctx) { set_max_dyn_smem(ctx, dcgs2_dot_kernel); }

template <>
void arnoldi_dcgs2<double>(gdr_ctx*, const gdr_op*, const Batch<double>&, int, int) {
  GDR_REQUIRE(false, "arnoldi_dcgs2: complex64 stages only");
}

template <>
void arnoldi_dcgs2<float>(gdr_ctx* ctx, const gdr_op* A, const Batch<float>& b, int jstart, int jend) {
  GDR_REQUIRE(b.hd && b.dc && b.Hf, "arnoldi_dcgs2: batch without DCGS2 buffers");
  const int is = (int)(sizeof(ColState) / sizeof(int));
  const double sv = sizeof(c64);
  for (int j = jstart; j <= jend; ++j) {
    const int mode = (j == jend) ? DC_FINAL : (j == jstart ? DC_FIRST : 0);
    // u: the final v_j on the first step, else the provisional vector in W2
    const c64* Uv = (mode == DC_FIRST) ? b.V + (long)j * b.ldv : b.W2;
    const long ucs = (mode == DC_FIRST) ? b.vcs : b.wcs;
    if (mode != DC_FINAL)
      op_apply_skip(ctx, A, b.ncol, nullptr, Uv, ucs, b.W, b.wcs, nullptr, 0, &b.st[0].run, is, b.cpp);
    const DotPlan p = dcgs2_plan(ctx, b, j + 1);
    const double act = run_share(ctx, b);
    {
      KProf kp(ctx, "dcgs2_dot_c64", ((double)j + (mode == DC_FINAL ? 1.0 : 2.0)) * col_len(b) * sv * act);
      dcgs2_dot_kernel<<<dim3((unsigned)(p.S * p.G), (unsigned)b.ncol), NT, (size_t)NW * NST * p.du * 512,
                         ctx->stream>>>(b, j, Uv, ucs, b.W, b.wcs, p.S, p.G, p.du, mode);
      GDR_LAUNCHED(ctx);
    }
    {
      const double reads = (double)j + (mode == DC_FINAL ? 1.0 : 2.0);
      const double writes = (mode == 0) ? 2.0 : 1.0;
      KProf kp(ctx, "dcgs2_update_c64", (reads + writes) * col_len(b) * sv * run_share(ctx, b));
      // four blocks are resident per SM; every block the same number of rounds
      const long ub = (nunits<float>(b.n) + NT - 1) / NT, rounds = (ub + 4L * ctx->num_sms - 1) / (4L * ctx->num_sms);
      const dim3 grid((unsigned)((ub + rounds - 1) / rounds) + 1, (unsigned)b.ncol);
      dcgs2_update_kernel<8><<<grid, NT, 0, ctx->stream>>>(b, j, Uv, ucs, b.W, b.W2, mode);
      GDR_LAUNCHED(ctx);
    }
  }
}
