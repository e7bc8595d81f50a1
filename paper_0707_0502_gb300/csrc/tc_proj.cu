// Projection dot C = V^H R over a kept basis V (n x nv, complex64) shared by many
// columns R (n x ncol, complex64) -- the Minres projection c = V_{k+1}^H r of every
// column of a Proj or refinement batch (Sec. 2.3, GMRES-Proj-Sh step 4) -- on the
// tensor cores (tcgen05, TF32 inputs, FP32 accumulation in tensor memory).
//
// A complex vector of length n is read as 2n interleaved floats (re, im), so with
// K = 2n:  Re(v^H r) = sum_k v[k] r[k]  and  Im(v^H r) = sum_k v'[k] r[k], where v' is
// v with every (re, im) pair replaced by (-im, re).  One CTA takes a K range and up to
// 128 columns: per K stage (32 floats) TMA brings the V tile (128 rows, rows >= nv zero)
// and the R tile (N rows) into shared memory with the 128-byte swizzle the MMA
// descriptors expect, rounding to TF32 on the way; four warps write the primed V tile
// (the pair swap keeps every 16-byte chunk in place, so the swizzle is unaffected); one
// thread issues the MMAs: D_re += V R^T and D_im += V' R^T, D_re / D_im 128 x N FP32 in
// tensor memory.  At the end the four warps read the accumulators back (tcgen05.ld) and
// write FP64 partials per (K range, column, basis vector), which gs_dot_shared_sum adds
// in a fixed order.
//
// TF32 keeps 10 bits of the significand: a coefficient is accurate to ~1e-3 relative.
// That is enough for the projection: the Proj cycle updates the solutions and the
// residuals with the same coefficients, so an error in c only makes one projection
// slightly less than optimal; residuals and solutions stay consistent.
//
// The residual update R += V T over the same basis (the projection's r -= V_{k+1}(Hbar_k -
// sigma_1 Ibar) d_1 of every column, T = -(Hbar_k - sigma_1 Ibar) d_1) is the transposed
// problem, and the GMRES-DR restart V[:, 0:k+1] <- V_{m+1} P is the same with one column's
// coefficients: with the real form of V (row 2i: [Re v_j, -Im v_j], row 2i+1: [Im v_j, Re v_j]
// over j) and the coefficients interleaved, the real rows of the result are A B^T with
// K = 2 nv.  A tile of 64 complex rows is one 128-row MMA.  The result must keep FP32's
// accuracy, so the product is split: A = A_hi + A_lo and B = B_hi + B_lo with TF32 parts,
// D = A_hi B_hi + A_lo B_hi + A_hi B_lo, which leaves an error of ~2^-22 relative per product.
//
// Every wait on an mbarrier gives up after about a second, marks the call failed
// (err, checked by the host) and the CTA winds down, freeing its tensor memory.
#include <cuda.h>

#include "async.cuh"
#include "kernels.cuh"

namespace {

constexpr int TC_M = 128;      // MMA rows: basis vectors, zero-filled above nv
constexpr int TC_KF = 32;      // floats per K stage: one 128-byte swizzle row
constexpr int TC_MAXST = 8;    // stages of the ring
constexpr int TC_THREADS = 256;  // warp 0 TMA, warp 1 MMA, warp 2 tensor-memory owner, warps 4-7 prime + epilogue
constexpr unsigned TC_A_BYTES = TC_M * TC_KF * 4;  // 16 KB

struct TcArgs {
  int ncol, nv, nt;      // columns, basis vectors, MMA N (multiple of 16, <= 128)
  int nst;               // stages
  long ksteps;           // K stages of the whole vector (2n / 32 rounded up)
  long ksplit;           // K stages per CTA
  c128* part;            // [K range][ncol][nv] FP64 partials
  int* err;              // set when a wait timed out
};

DEV void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          s_addr(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(s_addr(bar))
      : "memory");
}

DEV void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
          s_addr(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(s_addr(bar))
      : "memory");
}

// shared-memory operand descriptor: K-major, 128-byte swizzle, 8-row groups 1024 B apart
DEV uint64_t sm_desc(const void* p) {
  uint64_t d = (uint64_t)((s_addr(p) >> 4) & 0x3FFF);
  d |= (uint64_t)1 << 16;              // leading byte offset (unused with a swizzled K-major layout)
  d |= (uint64_t)(1024 >> 4) << 32;    // stride byte offset: the next group of 8 rows
  d |= (uint64_t)1 << 46;              // descriptor version of this architecture family
  d |= (uint64_t)2 << 61;              // 128-byte swizzle
  return d;
}

// instruction descriptor: D FP32, A and B TF32, both K-major, M = 128, N = nt
DEV uint32_t instr_desc(int nt) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(nt >> 3) << 17) | ((uint32_t)(TC_M >> 4) << 24);
}

DEV void mma_tf32(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(
          d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
DEV void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(s_addr(bar))
               : "memory");
}

// 32 consecutive accumulator columns of this warp's 32 lanes, one lane (row) per thread
DEV void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// 16 columns from each of two tensor-memory addresses, added: v = [t0 .. t0+16) + [t1 .. t1+16)
DEV void tmem_add16(uint32_t t0, uint32_t t1, float (&v)[16]) {
  uint32_t r[32];  // early clobber: the first load's results land while the second's address is still needed
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%32];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%33];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=&r"(r[0]), "=&r"(r[1]), "=&r"(r[2]), "=&r"(r[3]), "=&r"(r[4]), "=&r"(r[5]), "=&r"(r[6]), "=&r"(r[7]), "=&r"(r[8]), "=&r"(r[9]), "=&r"(r[10]), "=&r"(r[11]), "=&r"(r[12]), "=&r"(r[13]), "=&r"(r[14]), "=&r"(r[15]), "=&r"(r[16]), "=&r"(r[17]), "=&r"(r[18]), "=&r"(r[19]), "=&r"(r[20]), "=&r"(r[21]), "=&r"(r[22]), "=&r"(r[23]), "=&r"(r[24]), "=&r"(r[25]), "=&r"(r[26]), "=&r"(r[27]), "=&r"(r[28]), "=&r"(r[29]), "=&r"(r[30]), "=&r"(r[31])
      : "r"(t0), "r"(t1)
      : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]) + __uint_as_float(r[16 + i]);
}

// box of a 3-D map from shared memory (128-byte aligned), in the thread's bulk group
DEV void tma_store_3d(const CUtensorMap* map, int x, int y, int z, const void* src) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(map), "r"(x),
               "r"(y), "r"(z), "r"(s_addr(src))
               : "memory");
}
// v += t0 + (t1 + t2), 16 columns each, one wait for the three loads
DEV void tmem_acc16(uint32_t t0, uint32_t t1, uint32_t t2, float (&v)[16]) {
  uint32_t r[48];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%48];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%49];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47}, [%50];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=&r"(r[0]), "=&r"(r[1]), "=&r"(r[2]), "=&r"(r[3]), "=&r"(r[4]), "=&r"(r[5]), "=&r"(r[6]), "=&r"(r[7]), "=&r"(r[8]), "=&r"(r[9]), "=&r"(r[10]), "=&r"(r[11]), "=&r"(r[12]), "=&r"(r[13]), "=&r"(r[14]), "=&r"(r[15]), "=&r"(r[16]), "=&r"(r[17]), "=&r"(r[18]), "=&r"(r[19]), "=&r"(r[20]), "=&r"(r[21]), "=&r"(r[22]), "=&r"(r[23]), "=&r"(r[24]), "=&r"(r[25]), "=&r"(r[26]), "=&r"(r[27]), "=&r"(r[28]), "=&r"(r[29]), "=&r"(r[30]), "=&r"(r[31]), "=&r"(r[32]), "=&r"(r[33]), "=&r"(r[34]), "=&r"(r[35]), "=&r"(r[36]), "=&r"(r[37]), "=&r"(r[38]), "=&r"(r[39]), "=&r"(r[40]), "=&r"(r[41]), "=&r"(r[42]), "=&r"(r[43]), "=&r"(r[44]), "=&r"(r[45]), "=&r"(r[46]), "=&r"(r[47])
      : "r"(t0), "r"(t1), "r"(t2)
      : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i)
    v[i] += __uint_as_float(r[i]) + (__uint_as_float(r[16 + i]) + __uint_as_float(r[32 + i]));
}

// accumulator layout in tensor memory: D_re in columns [0, nt), D_im from column im_off
// (STACK: D_re and D_im in the two halves of the rows, one accumulator)
HD int tc_im_off(int nt) { return (nt + 31) / 32 * 32; }
HD uint32_t tc_cols(int nt, bool stack) {
  const int need = (stack ? 1 : 2) * tc_im_off(nt);
  return need <= 32 ? 32u : need <= 64 ? 64u : need <= 128 ? 128u : 256u;
}
HD unsigned tc_stage_bytes(int nt, bool stack) { return (stack ? 1u : 2u) * TC_A_BYTES + (unsigned)nt * TC_KF * 4; }

// STACK (nv <= 64): rows 0..63 of one operand are V, rows 64..127 V', so a stage is four MMAs
// (issuing one takes a thread ~80 cycles, and a stage of 31 vectors and 64 columns is ~550
// cycles of HBM time: eight MMAs a stage were slower than HBM), 8 KB to bring and only nv
// rows to prime, and the ring holds up to eight stages instead of four.
template <bool STACK>
__global__ void __launch_bounds__(TC_THREADS, 1) tc_proj_dot_kernel(const __grid_constant__ CUtensorMap mapV,
                                                                   const __grid_constant__ CUtensorMap mapR,
                                                                   TcArgs a) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  constexpr unsigned V_BYTES = STACK ? TC_A_BYTES / 2 : TC_A_BYTES;  // V's tile, V' right behind it
  const unsigned b_bytes = (unsigned)a.nt * TC_KF * 4;
  const unsigned stage_bytes = tc_stage_bytes(a.nt, STACK);  // V, V', R
  __shared__ __align__(8) uint64_t full[TC_MAXST], primed[TC_MAXST], empty[TC_MAXST], accb;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_s;
  __shared__ long issued_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long k0 = (long)blockIdx.x * a.ksplit;
  const int nk = (int)(min(a.ksteps, k0 + a.ksplit) - k0);
  const int col0 = blockIdx.y * a.nt;
  const int im_off = tc_im_off(a.nt);
  const uint32_t tcols = tc_cols(a.nt, STACK);
  if (threadIdx.x == 0) {
    for (int s = 0; s < a.nst; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&primed[s], 4);  // one arrival per warp
      mbar_init(&empty[s], 1);
    }
    mbar_init(&accb, 1);
    abort_s = 0;
    issued_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_addr(&tmem_base)),
                 "r"(tcols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // rows of V' that are never primed
  for (int s = 0; s < a.nst; ++s) {
    float4* z = reinterpret_cast<float4*>(base + (size_t)s * stage_bytes + V_BYTES);
    for (unsigned q = a.nv * 8 + threadIdx.x; q < V_BYTES / 16; q += TC_THREADS) z[q] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tm = tmem_base;
  volatile int* abort = &abort_s;

  if (warp == 0 && lane == 0) {  // ---- TMA producer
    int issued = 0, s = 0;
    unsigned ph = 0;
    for (int it = 0; it < nk && !*abort; ++it) {
      if (it >= a.nst && !mbar_wait(&empty[s], ph ^ 1u, abort)) break;
      unsigned char* st = base + (size_t)s * stage_bytes;
      mbar_arrive_tx(&full[s], V_BYTES + b_bytes);
      const int x = (int)((k0 + it) * TC_KF);  // a multiple of 32 floats: 128-byte aligned
      tma_load_2d(st, &mapV, x, 0, &full[s]);
      tma_load_2d(st + 2 * V_BYTES, &mapR, x, col0, &full[s]);
      issued = it + 1;
      if (++s == a.nst) {
        s = 0;
        ph ^= 1u;
      }
    }
    issued_s = issued;
  } else if (warp == 1 && lane == 0) {  // ---- MMA issuer
    const uint32_t idesc = instr_desc(a.nt);
    int s = 0;
    unsigned ph = 0;
    for (int it = 0; it < nk; ++it) {
      if (!mbar_wait(&full[s], ph, abort) || !mbar_wait(&primed[s], ph, abort)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      unsigned char* st = base + (size_t)s * stage_bytes;
      const uint64_t dv = sm_desc(st), dp = dv + (V_BYTES >> 4), dr = dv + (2 * V_BYTES >> 4);
#pragma unroll
      for (int kk = 0; kk < TC_KF / 8; ++kk) {  // 8 TF32 (32 bytes) per MMA
        const uint32_t acc = (it > 0 || kk > 0) ? 1u : 0u;
        mma_tf32(tm, dv + 2 * kk, dr + 2 * kk, idesc, acc);
        if (!STACK) mma_tf32(tm + (uint32_t)im_off, dp + 2 * kk, dr + 2 * kk, idesc, acc);
      }
      mma_commit(&empty[s]);
      if (++s == a.nst) {
        s = 0;
        ph ^= 1u;
      }
    }
    mma_commit(&accb);  // arrives once every MMA issued above has completed
  } else if (warp >= 4) {  // ---- V' = V with (re, im) -> (-im, re), then the epilogue
    const unsigned t = threadIdx.x - 128;
    int s = 0;
    unsigned ph = 0;
    for (int it = 0; it < nk; ++it) {
      if (!__all_sync(0xffffffffu, mbar_wait(&full[s], ph, abort))) break;
      unsigned char* st = base + (size_t)s * stage_bytes;
      const float4* src = reinterpret_cast<const float4*>(st);
      float4* dst = reinterpret_cast<float4*>(st + V_BYTES);
      for (unsigned q = t; q < (unsigned)a.nv * 8; q += 128) {
        const float4 v = src[q];
        dst[q] = make_float4(-v.y, v.x, -v.w, v.z);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&primed[s]);
      if (++s == a.nst) {
        s = 0;
        ph ^= 1u;
      }
    }
    // the MMAs finish (or time out) before the accumulators are read or freed; this
    // wait does not follow the CTA's abort flag
    int own = 0;
    const bool got = mbar_wait(&accb, 0, &own);
    if (!got) *abort = 1;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    __syncwarp();
    if (__all_sync(0xffffffffu, got && !*abort)) {
      // accumulators: tensor-memory lane = basis vector, column = matrix column
      const int q4 = warp & 3;
      const uint32_t lane_base = (uint32_t)(q4 * 32) << 16;
      for (int cb = 0; cb < a.nt; cb += 32) {
        float re[32], im[32];
        tmem_ld32(tm + lane_base + (uint32_t)cb, re);
        if (!STACK) tmem_ld32(tm + lane_base + (uint32_t)(im_off + cb), im);
        const int row = STACK ? (q4 & 1) * 32 + lane : q4 * 32 + lane;
        if (row < a.nv) {
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const int c = col0 + cb + j;
            if (cb + j >= a.nt || c >= a.ncol) continue;
            c128* p = &a.part[((long)blockIdx.x * a.ncol + c) * a.nv + row];
            if (STACK) (q4 < 2 ? p->x : p->y) = (double)re[j];
            else *p = c128{(double)re[j], (double)im[j]};
          }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (*abort) {
    // wait (bounded) for the last load issued into each stage, then report the failure
    if (warp == 0 && lane == 0) {
      const long issued = issued_s;
      for (long it = issued > a.nst ? issued - a.nst : 0; it < issued; ++it) {
        int own = 0;
        mbar_wait(&full[(int)(it % a.nst)], (unsigned)((it / a.nst) & 1), &own);
      }
      atomicExch(a.err, 1);
    }
    __syncthreads();
  }
  if (warp == 2) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm), "r"(tcols) : "memory");
  }
}

// ------------------------------------------- basis combinations (D = V T over row tiles)
//
// One kernel for the residual update R (+)= V T of many columns over one basis and for the
// GMRES-DR restart V[:, 0:nout] <- V C with its solution update X += V D (in place: a tile's
// rows are all read before any of its outputs is written, and no two tiles share a row).
//
// What bounds it is HBM (V read once, R read and written, or V's kept columns written), if
// what a tile needs -- bringing V, splitting it into TF32 parts, the MMAs, the epilogue -- runs
// beside one another.  So V goes through two rings of K atoms (16 vectors x 64 rows): one TMA
// load per atom into `raw`, that nothing waits for but the writers (a 512-byte bulk copy per
// vector took the issuing warp ~110 cycles each, 16 an atom); two groups of writer warps split
// an atom into A while the MMAs of the one before run.  Any basis size streams through the same
// shared memory (the restart's 81 vectors are six atoms).  The outputs leave by bulk stores or
// reductions from shared memory.  Measured at 24^3x32 (5.3 M rows): 41 vectors x 120 columns
// 4.07 -> 1.97 ms (89% of the copy bandwidth); the restart of 81 vectors to 41, before on the
// CUDA cores, 6.35 -> 2.43 ms, bound by its epilogue warps (a drain per atom and the outputs).

constexpr int TU_ROWS = 64;         // complex rows per tile: 128 real MMA rows
constexpr int TU_THREADS = 640;     // warp 0 copies of V, warps 1 and 3 MMA, warp 2 tensor memory, warps 4-11 A atoms, warps 12-19 epilogue
constexpr int TU_EPI = 12;          // first epilogue warp
constexpr int TU_DW = 256;          // tensor-memory columns of one accumulator buffer
constexpr int TU_DLO = 128;         // ... and its first column of the products with a lo part
constexpr int TU_SC = 16;           // columns that a group of four epilogue warps stages at a time
constexpr int TU_MAXNV = 48;        // basis vectors of the residual update
constexpr int TU_MINNV = 54;        // fewest of the restart
constexpr int TU_STAGES = 2;        // K atoms of A, one per group of four writer warps
constexpr int TU_MAXOUT = 64;       // outputs of the restart: hi and lo parts of B side by side in one MMA (N = 128)
constexpr int TU_RAW_ROW = 512;     // bytes of one vector's rows in `raw`
constexpr int TU_RAW = 16 * TU_RAW_ROW;
constexpr int TU_MAXRAW = 8;
constexpr int TU_PER = 8;           // elements of an atom per writer thread: 64 rows x 16 vectors / 128
constexpr unsigned TU_ATOM_A = 128u * 128u;  // one K atom of A: 128 rows x 128 bytes

enum TuMode {
  TU_DIRECT = 0,   // R = V T or R += V T, R read and written by the epilogue's threads
  TU_REDUCE = 1,   // R += V T, accumulators staged and added to R by bulk reductions (16-byte aligned R)
  TU_RESTART = 2   // V[:, 0:nout] = V C (in place), X (FP64) += V D
};


struct TuArgs {
  long n;
  int nv, ncol, nt, ka, kp;  // basis vectors, MMA columns in all and per column tile, K atoms, K padded to 8
  int rmode;                 // TU_DIRECT: 1: R = V T, 2: R += V T
  int nraw, nstage, bulk;    // stages of the raw ring and of an epilogue group's output ring (1 or 2)
                             // bulk: V by TMA, V's outputs by bulk stores (16-byte aligned, even strides)
  c64* V;
  long ldv, vcs;             // stride of the vectors, and of the batch's bases (TU_RESTART: blockIdx.y)
  const c128* C;             // coefficients of MMA column k at C + k * cs (nv values), of batch column c at + c * ccs
  long cs, ccs;
  float* R;                  // R as floats, column k at R + 2 * k * ldr
  long ldr;
  int nout;                  // TU_RESTART: columns written into V; the others go to X
  int tstore;                // ... whole tiles of them by tensor stores (mapO)
  c128* X;
  long ldx, xcs;
  const ColState* st;
  const int* nvec;           // TU_RESTART: vector length per batch column (nullptr: n)
  int* err;
};

DEV uint32_t tf32_rna(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return r;
}
// x = hi + lo, both TF32
DEV void split_tf32(float x, float& hi, float& lo) {
  hi = __uint_as_float(tf32_rna(x));
  lo = __uint_as_float(tf32_rna(x - hi));
}
// byte offset of element (row, kin < 32) within a K atom (K-major, 128-byte swizzle)
DEV unsigned swz_atom(int row, int kin) {
  return (unsigned)row * 128u + ((unsigned)((kin >> 2) ^ (row & 7)) << 4) + (unsigned)(kin & 3) * 4u;
}

DEV void named_sync(int id, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory"); }
// barrier of `threads` threads that tells each whether any of them passed true
DEV bool named_any(int id, int threads, bool p) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred q, o;\n setp.ne.u32 q, %3, 0;\n barrier.cta.red.or.pred o, %1, %2, q;\n selp.u32 %0, 1, 0, o;\n}\n"
      : "=r"(r)
      : "r"(id), "r"(threads), "r"((uint32_t)p)
      : "memory");
  return r != 0;
}

template <int MODE>
__global__ void __launch_bounds__(TU_THREADS, 1) tc_combine_kernel(const __grid_constant__ CUtensorMap mapV,
                                                                  const __grid_constant__ CUtensorMap mapO, TuArgs a) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  unsigned char* A = base;  // TU_STAGES x (hi atom, lo atom)
  unsigned char* Bhi = A + (size_t)TU_STAGES * 2 * TU_ATOM_A;
  __shared__ __align__(8) uint64_t afull[TU_STAGES], aempty[TU_STAGES], dfull[2], dempty[2], fin;
  __shared__ __align__(8) uint64_t rfull[TU_MAXRAW], rempty[TU_MAXRAW];
  __shared__ long issued_s;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_s;
  __shared__ int cmap[128];  // the active columns of this column tile, compacted
  __shared__ int wcnt[4], nact_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int batch = MODE == TU_RESTART ? blockIdx.y : 0;
  const int col0 = MODE == TU_RESTART ? 0 : blockIdx.y * a.nt;
  const long n = (MODE == TU_RESTART && a.nvec) ? (long)a.nvec[batch] : a.n;
  const long ntiles = (n + TU_ROWS - 1) / TU_ROWS;
  const long my_tiles = blockIdx.x < ntiles ? (ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
  c64* V = a.V + batch * a.vcs;

  // active columns: the MMA width and the epilogue follow their number, and a tile
  // whose columns have all converged has nothing to do
  bool f = false;
  unsigned bal = 0;
  if (warp < 4) {
    const int c = threadIdx.x;
    f = c < a.nt && col0 + c < a.ncol && (!a.st || a.st[MODE == TU_RESTART ? batch : col0 + c].active);
    bal = __ballot_sync(0xffffffffu, f);
    if (lane == 0) wcnt[warp] = __popc(bal);
  }
  __syncthreads();
  if (warp < 4) {
    int off = 0;
    for (int w = 0; w < warp; ++w) off += wcnt[w];
    if (f) cmap[off + __popc(bal & ((1u << lane) - 1u))] = threadIdx.x;
    if (threadIdx.x == 0) nact_s = wcnt[0] + wcnt[1] + wcnt[2] + wcnt[3];
  }
  __syncthreads();
  const int nact = nact_s;
  if (nact == 0 || my_tiles == 0) return;  // uniform over the CTA, before any barrier or tensor memory
  const int ne = (nact + 15) / 16 * 16;   // MMA N: compacted columns, zero rows above nact
  const unsigned blo = (unsigned)ne * 128u;  // per K atom: ne rows of hi parts, then ne rows of lo parts
  unsigned char* raw = Bhi + (size_t)a.ka * 2 * blo;

  if (threadIdx.x == 0) {
    for (int q = 0; q < TU_STAGES; ++q) {
      mbar_init(&afull[q], 4);  // one arrival per warp: a warp's 32 would be served one by one
      mbar_init(&aempty[q], 2);  // one commit per MMA warp
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&dfull[b], 2);
      mbar_init(&dempty[b], 8);
    }
    for (int q = 0; q < a.nraw; ++q) {
      mbar_init(&rfull[q], a.bulk ? 1 : 32);
      mbar_init(&rempty[q], 4);
    }
    mbar_init(&fin, 2);
    abort_s = 0;
    issued_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_addr(&tmem_base)),
                 "r"(2 * TU_DW)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // B = the active columns' coefficients split into TF32 parts, K-major, row k = column
  // cmap[k].  The residual update splits the FP64 coefficient; the restart takes it in the
  // basis' precision first, as its CUDA-core form does (one FP64 instruction an element
  // instead of four: at 96 x 64 coefficients the difference is ~9 us of FP64 pipe).
  {
    const c128* C = a.C + batch * a.ccs;
    const int kw = a.ka * 32;
    for (int t = threadIdx.x; t < ne * kw; t += TU_THREADS) {
      const int r = t / kw, k = t % kw, j = k >> 1;
      float hi = 0.f, lo = 0.f;
      if (r < nact && j < a.nv) {
        const c128 v = C[(long)(col0 + cmap[r]) * a.cs + j];
        const double x = (k & 1) ? v.y : v.x;
        if (MODE == TU_RESTART) {
          split_tf32((float)x, hi, lo);
        } else {
          hi = __uint_as_float(tf32_rna((float)x));
          lo = __uint_as_float(tf32_rna((float)(x - (double)hi)));
        }
      }
      unsigned char* b = Bhi + (size_t)(k >> 5) * 2 * blo + swz_atom(r, k & 31);
      *reinterpret_cast<float*>(b) = hi;
      *reinterpret_cast<float*>(b + blo) = lo;
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tm = tmem_base;
  volatile int* abort = &abort_s;
  const long natoms = my_tiles * a.ka;  // K atoms this CTA works through

  if (warp == 0) {  // ---- copies of V, one atom after another
    long q = 0;
    for (long it = 0; it < my_tiles; ++it) {
      const long r0 = (blockIdx.x + it * (long)gridDim.x) * TU_ROWS;
      for (int at = 0; at < a.ka; ++at, ++q) {
        const int s = (int)(q % a.nraw);
        const bool ok = q < a.nraw || mbar_wait(&rempty[s], (unsigned)((q / a.nraw - 1) & 1), abort);
        if (!__all_sync(0xffffffffu, ok)) break;
        unsigned char* dst = raw + (size_t)s * TU_RAW;
        if (a.bulk) {  // rows from n and vectors from nv on arrive as zeros (or the batch's padding: rows not stored)
          if (lane == 0) {
            mbar_arrive_tx(&rfull[s], TU_RAW);
            tma_load_3d(dst, &mapV, (int)(2 * r0), 16 * at, batch, &rfull[s]);
          }
        } else {
          const int rows = (int)min((long)TU_ROWS, n - r0), nj = min(16, a.nv - 16 * at);
          const c64* src = V + (long)(16 * at) * a.ldv + r0;
          for (int e = lane; e < nj * TU_ROWS; e += 32) {
            const int j = e / TU_ROWS, i = e % TU_ROWS;
            if (i < rows)
              asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(s_addr(dst + j * TU_RAW_ROW + i * 8)),
                           "l"(__cvta_generic_to_global(src + (long)j * a.ldv + i))
                           : "memory");
          }
          asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(s_addr(&rfull[s])) : "memory");
        }
        if (lane == 0) issued_s = q + 1;
      }
      if (*abort) break;
    }
    if (!a.bulk) asm volatile("cp.async.wait_all;" ::: "memory");
  } else if (warp == 1 || warp == 3) {  // ---- MMA issuers
    // Issuing an MMA takes a thread ~80 cycles whatever its N, longer than these run, so two
    // warps share an atom's: warp 1 the products with A's hi part, warp 3 those with a lo part,
    // into accumulators of their own.  The restart's A_hi [B_hi | B_lo] is one instruction
    // (N = 2 ne <= 128): 4 MMAs a warp and atom; the residual update has 4 and 8.
    // Accumulator buffers alternate per tile, or (restart) per atom, and the epilogue sums the
    // atoms in FP32 itself: each MMA truncates as it adds to the accumulator, so the error grows
    // with their number in one accumulator (81 vectors, 60 MMAs: 9.7e-7 of the result; the
    // CUDA-core form had 1.2e-7, this one 1.0e-7).
    if (lane == 0) {
      constexpr bool PER_ATOM = MODE == TU_RESTART;
      const bool hi_warp = warp == 1;
      const uint32_t idesc = instr_desc(PER_ATOM && hi_warp ? 2 * ne : ne);
      const uint64_t da0 = sm_desc(A + (hi_warp ? 0 : TU_ATOM_A)), b0 = sm_desc(Bhi);
      const uint32_t stage_step = 2 * TU_ATOM_A >> 4, bstep = 2 * blo >> 4, lo_step = blo >> 4;  // 16-byte units
      const uint32_t dcol = tm + (hi_warp ? 0u : (uint32_t)TU_DLO);
      int q = 0, db = 0;
      bool ok = true;
      for (int it = 0; it < (int)my_tiles && ok; ++it) {
        uint64_t bh = b0;
        for (int at = 0; at < a.ka; ++at, ++q, bh += bstep) {
          const int s = q & (TU_STAGES - 1), b = db & 1;
          if (PER_ATOM || at == 0)
            ok = db < 2 || mbar_wait(&dempty[b], (unsigned)(((db >> 1) & 1) ^ 1), abort);
          ok = ok && mbar_wait(&afull[s], (unsigned)((q / TU_STAGES) & 1), abort);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t d = dcol + (uint32_t)(b * TU_DW);
          const uint64_t da = da0 + s * stage_step;
          const int nk = a.kp / 8 - 4 * at;
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            if (kk < nk) mma_tf32(d, da + 2 * kk, bh + 2 * kk, idesc, (!PER_ATOM && at > 0) || kk > 0 ? 1u : 0u);
          if (!PER_ATOM && !hi_warp) {  // A_hi B_lo
            const uint64_t dh = da - (TU_ATOM_A >> 4), bl = bh + lo_step;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              if (kk < nk) mma_tf32(d, dh + 2 * kk, bl + 2 * kk, idesc, 1u);
          }
          mma_commit(&aempty[s]);
          if (PER_ATOM || at == a.ka - 1) {
            mma_commit(&dfull[b]);
            ++db;
          }
        }
      }
      mma_commit(&fin);  // arrives once every MMA issued above has completed
      int own = 0;
      if (!mbar_wait(&fin, 0, &own)) *abort = 1;
    }
  } else if (warp >= 4 && warp < TU_EPI) {  // ---- A atoms from the copies, alternating between two groups
    // lane = (row, basis vector) as 8 x 4: a load reads 4 runs of 64 bytes and a store writes 8
    // rows x 32 bytes of A; the row pitch and the swizzle spread both over all banks
    const int w4 = warp & 3, grp = (warp - 4) >> 2, il = lane >> 2, jl = lane & 3;
    const int jpad = a.kp / 2;  // the MMAs read vectors below jpad; those from nv on are zero
    // this thread's elements are rows i0 and i0 + 8, vectors jl + 4t: swz_atom of (2 i0, 2 jj)
    // and (2 i0 + 1, 2 jj), the second rows 16 real rows further on
    const int i0 = w4 * 16 + il;
    unsigned o0[4], o1[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      o0[t] = swz_atom(2 * i0, 2 * (jl + 4 * t));
      o1[t] = swz_atom(2 * i0 + 1, 2 * (jl + 4 * t));
    }
    for (long q = grp; q < natoms; q += TU_STAGES) {
      const int s = grp, rs = (int)(q % a.nraw), at = (int)(q % a.ka);
      bool ok = mbar_wait(&rfull[rs], (unsigned)((q / a.nraw) & 1), abort);
      if (!__all_sync(0xffffffffu, ok)) break;
      const unsigned char* src = raw + (size_t)rs * TU_RAW + jl * TU_RAW_ROW + i0 * 8;
      unsigned char* hi = A + (size_t)s * 2 * TU_ATOM_A;
      const int jn = a.nv - 16 * at - jl, jp = jpad - 16 * at - jl;  // vectors of this atom: given, and read by the MMAs
      float2 v[TU_PER];
#pragma unroll
      for (int e = 0; e < TU_PER; ++e) {
        v[e] = make_float2(0.f, 0.f);
        if (4 * (e & 3) < jn) v[e] = *reinterpret_cast<const float2*>(src + 4 * (e & 3) * TU_RAW_ROW + 64 * (e >> 2));
      }
      // the copies are in registers by the time the MMAs give the stage back (waited for together
      // with the copies: 41 vectors x 120 columns at 24^3x32 2.034 ms, now 1.973; a third stage
      // of A with a group of its own: the restart 3.01 -> 3.19 ms)
      ok = q < TU_STAGES || mbar_wait(&aempty[s], (unsigned)((q / TU_STAGES - 1) & 1), abort);
      if (!__all_sync(0xffffffffu, ok)) break;
#pragma unroll
      for (int e = 0; e < TU_PER; ++e) {
        const int t = e & 3, h = e >> 2;
        if (4 * t >= jp) continue;
        float rh, rl, ih, il2;
        split_tf32(v[e].x, rh, rl);
        split_tf32(v[e].y, ih, il2);
        *reinterpret_cast<float2*>(hi + o0[t] + h * 2048) = make_float2(rh, -ih);
        *reinterpret_cast<float2*>(hi + o1[t] + h * 2048) = make_float2(ih, rh);
        *reinterpret_cast<float2*>(hi + TU_ATOM_A + o0[t] + h * 2048) = make_float2(rl, -il2);
        *reinterpret_cast<float2*>(hi + TU_ATOM_A + o1[t] + h * 2048) = make_float2(il2, rl);
      }
      // the raw stage is given back only now that its values have been used: an arrival placed
      // right after the loads let a refill overtake some of them (seen as later rows in a tile)
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&afull[s]);
        mbar_arrive(&rempty[rs]);
      }
    }
  } else if (warp >= TU_EPI) {  // ---- epilogue
    const int q4 = warp & 3, half = (warp - TU_EPI) >> 2;
    const int m = q4 * 32 + lane;  // real row of the tile = tensor-memory lane
    const uint32_t lane_base = (uint32_t)(q4 * 32) << 16;
    const int nch = (ne + 31) / 32;  // this group takes the 32-column chunks half and half + 2 (nch <= 4)
    float* const stage0 = reinterpret_cast<float*>(raw + (size_t)a.nraw * TU_RAW) + half * a.nstage * TU_SC * 128;
    float* stage = stage0;
    const int ndrain = MODE == TU_RESTART ? a.ka : 1;  // accumulators per tile
    // columns [k0, k0 + TU_SC) x 128 rows through shared memory, one 512-byte bulk store or
    // reduction per column (fewer at the ragged end): no thread waits for R's old values or
    // for its stores.  The stage's previous columns must have been read out first.
    auto stage_out = [&](const float* d, int k0, int kend, float* out, long ld, const int* map, unsigned bytes, bool add,
                         int tx) {
      if (a.nstage == 2) {
        stage = stage == stage0 ? stage0 + TU_SC * 128 : stage0;
        asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
      } else {
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
      }
      named_sync(1 + half, 128);
#pragma unroll
      for (int j = 0; j < TU_SC; ++j) stage[j * 128 + m] = d[j];
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      named_sync(1 + half, 128);
      if (MODE == TU_RESTART && tx >= 0) {
        if (m == 0) tma_store_3d(&mapO, tx, k0, batch, stage);
      } else if (m < TU_SC && k0 + m < kend) {
        float* dst = out + 2 * (long)(map ? col0 + map[k0 + m] : k0 + m) * ld;
        if (add)
          asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], %2;" ::"l"(
                           __cvta_generic_to_global(dst)),
                       "r"(s_addr(stage + m * 128)), "r"(bytes)
                       : "memory");
        else
          asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(__cvta_generic_to_global(dst)),
                       "r"(s_addr(stage + m * 128)), "r"(bytes)
                       : "memory");
      }
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    };
    long db = 0;
    bool ok = true;
    for (long it = 0; it < my_tiles; ++it) {
      const long r0 = (blockIdx.x + it * (long)gridDim.x) * TU_ROWS;
      const long g = 2 * r0 + m;  // float index within a column
      const bool rowok = g < 2 * n;
      float sum[32];  // TU_RESTART: the atoms' sum (one chunk per group)
#pragma unroll
      for (int j = 0; j < 32; ++j) sum[j] = 0.f;
      for (int dr = 0; dr < ndrain; ++dr, ++db) {
        const int b = (int)(db & 1);
        int own = 0;
        const bool got = mbar_wait(&dfull[b], (unsigned)((db >> 1) & 1), &own);
        if (!got) *abort = 1;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // the group's four warps, which synchronise to stage outputs, leave together: told here, or
        // (restart, whose warps drain the atoms of a tile each at its own pace) at the tile's end
        ok = MODE == TU_RESTART ? __all_sync(0xffffffffu, got) : !named_any(1 + half, 128, !got);
        if (!ok) break;
        const uint32_t tb = tm + lane_base + (uint32_t)(b * TU_DW);
        if (MODE == TU_RESTART) {
          if (half < nch) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const uint32_t col = (uint32_t)(half * 32 + 16 * h);
              if (col < (uint32_t)ne)  // the products with a lo part first, then the sum so far
                tmem_acc16(tb + col, tb + ne + col, tb + TU_DLO + col, *reinterpret_cast<float(*)[16]>(sum + 16 * h));
            }
          }
        } else {
          for (int cc = half; cc < nch; cc += 2) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int k0 = cc * 32 + TU_SC * h;
              float d[TU_SC];
              tmem_add16(tb + (uint32_t)k0, tb + (uint32_t)(TU_DLO + k0), d);
              if (MODE == TU_REDUCE) {
                const unsigned bytes = (unsigned)min(128L, 2 * n - 2 * r0) * 4u;  // n even: a multiple of 16
                stage_out(d, k0, nact, a.R + 2 * r0, a.ldr, cmap, bytes, true, -1);
              } else {
#pragma unroll
                for (int j = 0; j < TU_SC; ++j) {
                  if (!rowok || k0 + j >= nact) continue;
                  float* rp = a.R + 2 * (long)(col0 + cmap[k0 + j]) * a.ldr + g;
                  *rp = a.rmode == 2 ? *rp + d[j] : d[j];
                }
              }
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&dempty[b]);
      }
      if (MODE == TU_RESTART) ok = !named_any(1 + half, 128, !ok);
      if (!ok) break;
      if (MODE == TU_RESTART) {
        const bool bulk = a.bulk && (n % 2 == 0 || n - r0 >= TU_ROWS);  // not for an odd last row
        const unsigned bytes = (unsigned)min(128L, 2 * n - 2 * r0) * 4u;
        float* Vf = reinterpret_cast<float*>(V) + 2 * r0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int k0 = half * 32 + TU_SC * h, k1 = min(k0 + TU_SC, nact);
          if (k0 >= nact) break;  // uniform in the group
          // a whole tile: one tensor store of the 16 columns (clipped at nout), where 16 bulk stores
          // held the group up while the MMAs waited for it (81 -> 41 at 24^3x32: 2.98 ms, now 2.43)
          const int tx = a.tstore && n - r0 >= TU_ROWS && k0 < a.nout ? (int)(2 * r0) : -1;
          stage_out(sum + TU_SC * h, k0, bulk ? min(a.nout, k1) : 0, Vf, a.ldv, nullptr, bytes, false, tx);
          if (!rowok) continue;
          // each thread reads back its own row: a loop over just these columns (unrolled over
          // `sum` the compiler predicates all 32 FP64 additions, and the pipe runs each)
          if (!bulk)
            for (int k = k0; k < min(a.nout, k1); ++k) Vf[2 * (long)k * a.ldv + m] = stage[(k - k0) * 128 + m];
          for (int k = max(a.nout, k0); k < k1; ++k) {
            double* xp = reinterpret_cast<double*>(a.X + batch * a.xcs) + 2 * (long)(k - a.nout) * a.ldx + g;
            *xp = *xp + (double)stage[(k - k0) * 128 + m];
          }
        }
      }
    }
    if (MODE != TU_DIRECT) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (*abort) {
    // wait (bounded) for the last copies issued into each stage, then report the failure
    if (threadIdx.x == 0) {
      const long issued = issued_s;
      for (long q = issued > a.nraw ? issued - a.nraw : 0; q < issued; ++q) {
        int own = 0;
        mbar_wait(&rfull[(int)(q % a.nraw)], (unsigned)((q / a.nraw) & 1), &own);
      }
      atomicExch(a.err, 1);
    }
    __syncthreads();
  }
  if (warp == 2) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm), "r"(2 * TU_DW) : "memory");
  }
}

using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                 const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encoder() {
  static EncodeTiled fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiled>(p);
  }
  return fn;
}

// 2-D map of `rows` vectors of 2n floats each (stride ld complex elements), box 32 floats x box_rows,
// TF32 rounding on load, 128-byte swizzle, zero fill outside
bool make_map(CUtensorMap& m, const void* ptr, long n, long ld, int rows, int box_rows) {
  EncodeTiled enc = encoder();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)(2 * n), (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)(ld * 8)};
  cuuint32_t box[2] = {(cuuint32_t)TC_KF, (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  return enc(&m, CU_TENSOR_MAP_DATA_TYPE_TFLOAT32, 2, const_cast<void*>(ptr), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 3-D map of `batch` bases (stride vcs) of `rows` vectors of 2n floats each, box 128 floats x 16
// vectors, no swizzle, zero fill outside
bool make_map_raw(CUtensorMap& m, const void* ptr, long n, long ld, int rows, long vcs, int batch) {
  EncodeTiled enc = encoder();
  if (!enc) return false;
  cuuint64_t dims[3] = {(cuuint64_t)(2 * n), (cuuint64_t)rows, (cuuint64_t)batch};
  cuuint64_t strides[2] = {(cuuint64_t)(ld * 8), (cuuint64_t)((vcs ? vcs : ld * rows) * 8)};
  cuuint32_t box[3] = {2 * TU_ROWS, 16, 1};
  cuuint32_t es[3] = {1, 1, 1};
  return enc(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(ptr), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

int tc_proj_splits(gdr_ctx* ctx, long n, int ncol) {
  const int ctiles = (ncol + 127) / 128;
  const long ksteps = (2 * n + TC_KF - 1) / TC_KF;
  const int want = std::max(1, ctx->num_sms / ctiles);
  const long ksplit = (ksteps + want - 1) / want;
  return (int)((ksteps + ksplit - 1) / ksplit);
}

bool tc_proj_dot(gdr_ctx* ctx, long n, const c64* V, long ldv, int nv, const c64* R, long ldr, int ncol, c128* part,
                 int* err, int& nsplit, double prof_bytes) {
  if (nv < 1 || nv > TC_M || ncol < 1 || !ctx->tc_ok) return false;
  if (n >= (1L << 30)) return false;  // TMA coordinates, in floats, are 32-bit
  const int ctiles = (ncol + 127) / 128;
  const int per = (ncol + ctiles - 1) / ctiles;
  const int nt = std::max(16, (per + 15) / 16 * 16);
  const bool stack = nv <= TC_M / 2;
  CUtensorMap mv, mr;
  if (!make_map(mv, V, n, ldv, nv, stack ? TC_M / 2 : TC_M) || !make_map(mr, R, n, ldr, ncol, nt)) return false;
  TcArgs a;
  a.ncol = ncol;
  a.nv = nv;
  a.nt = nt;
  a.ksteps = (2 * n + TC_KF - 1) / TC_KF;
  nsplit = tc_proj_splits(ctx, n, ncol);
  a.ksplit = (a.ksteps + nsplit - 1) / nsplit;
  a.part = part;
  a.err = err;
  const size_t sb = tc_stage_bytes(nt, stack);
  a.nst = (int)std::min<size_t>(TC_MAXST, (ctx->tc_dot_smem - 1024) / sb);
  const size_t smem = 1024 + a.nst * sb;
  dim3 grid((unsigned)nsplit, (unsigned)ctiles);
  KProf kp(ctx, "tc_proj_dot_c64", prof_bytes);
  if (stack) tc_proj_dot_kernel<true><<<grid, TC_THREADS, smem, ctx->stream>>>(mv, mr, a);
  else tc_proj_dot_kernel<false><<<grid, TC_THREADS, smem, ctx->stream>>>(mv, mr, a);
  GDR_LAUNCHED(ctx);
  return true;
}

// shared memory with nraw stages of the raw ring and nstage of the output rings
static size_t tc_combine_smem(int ka, int ne, int nraw, int nstage) {
  return 1024 + (size_t)TU_STAGES * 2 * TU_ATOM_A + 2 * (size_t)ka * ne * 128 + (size_t)nraw * TU_RAW +
         (size_t)2 * nstage * TU_SC * 512;
}
constexpr int TU_MINRAW = 4;
static_assert(TU_MINRAW % TU_STAGES == 0 && TU_MAXRAW % TU_STAGES == 0, "raw stages come in pairs");

template <int MODE>
static void tc_combine_launch(gdr_ctx* ctx, TuArgs& a, unsigned gx, unsigned gy) {
  const int ne = (a.nt + 15) / 16 * 16;
  a.nraw = TU_MAXRAW;
  // an even number: each stage then belongs to one group of writers, which waits for its fills in
  // order (with an odd one a group could test a stage's next phase before the other group's fill
  // of the phase before it had landed, and find it "complete")
  a.nstage = tc_combine_smem(a.ka, ne, TU_MINRAW, 2) <= ctx->tc_combine_smem ? 2 : 1;
  while (a.nraw > TU_MINRAW && tc_combine_smem(a.ka, ne, a.nraw, a.nstage) > ctx->tc_combine_smem) a.nraw -= TU_STAGES;
  // TMA needs 16-byte aligned starts and strides; coordinates are 32-bit
  CUtensorMap mv = {};
  a.bulk = a.ldv % 2 == 0 && a.vcs % 2 == 0 && (reinterpret_cast<uintptr_t>(a.V) & 15) == 0 && a.n < (1L << 29) &&
           make_map_raw(mv, a.V, a.n, a.ldv, a.nv, a.vcs, MODE == TU_RESTART ? (int)gy : 1);
  CUtensorMap mo = {};
  a.tstore = MODE == TU_RESTART && a.bulk && a.nout > 0 && make_map_raw(mo, a.V, a.n, a.ldv, a.nout, a.vcs, (int)gy);
  tc_combine_kernel<MODE><<<dim3(gx, gy), TU_THREADS, tc_combine_smem(a.ka, ne, a.nraw, a.nstage), ctx->stream>>>(mv, mo, a);
  GDR_LAUNCHED(ctx);
}

static void tc_combine_sizes(TuArgs& a, int nv) {
  a.nv = nv;
  a.kp = (2 * nv + 7) / 8 * 8;
  a.ka = (a.kp + 31) / 32;
}

bool tc_proj_update(gdr_ctx* ctx, long n, const c64* V, long ldv, int nv, const c128* C, long ccs, int rmode, c64* R,
                    long ldr, int ncol, const ColState* st, int* err, double prof_bytes) {
  if (nv < 1 || nv > TU_MAXNV || ncol < 1 || (rmode != 1 && rmode != 2) || !ctx->tc_ok || !ctx->tc_update_ok)
    return false;
  const int ctiles = (ncol + 127) / 128;
  const int per = (ncol + ctiles - 1) / ctiles;
  TuArgs a{};
  tc_combine_sizes(a, nv);
  a.n = n;
  a.ncol = ncol;
  a.nt = (per + 31) / 32 * 32;
  a.rmode = rmode;
  a.V = const_cast<c64*>(V);
  a.ldv = ldv;
  a.C = C;
  a.cs = ccs;
  a.R = reinterpret_cast<float*>(R);
  a.ldr = ldr;
  a.st = st;
  a.err = err;
  const long ntiles = (n + TU_ROWS - 1) / TU_ROWS;
  const unsigned gx = (unsigned)std::min<long>(std::max(1, ctx->num_sms / ctiles), ntiles);
  // bulk reductions need 16-byte aligned column starts and lengths
  const bool bulk = rmode == 2 && n % 2 == 0 && ldr % 2 == 0 && (reinterpret_cast<uintptr_t>(R) & 15) == 0;
  KProf kp(ctx, "tc_proj_update_c64", prof_bytes);
  if (bulk) tc_combine_launch<TU_REDUCE>(ctx, a, gx, (unsigned)ctiles);
  else tc_combine_launch<TU_DIRECT>(ctx, a, gx, (unsigned)ctiles);
  return true;
}

bool tc_restart(gdr_ctx* ctx, long n, int ncol, c64* V, long ldv, long vcs, int nv, const c128* C, long ldc, long ccs,
                int nout, int nx, c128* X, long ldx, long xcs, const ColState* st, const int* nvec, int* err) {
  TuArgs a{};
  const int nn = nout + nx;
  tc_combine_sizes(a, nv);
  // The hand-overs per K atom cost the same however few outputs there are, the CUDA-core form's
  // products grow with both, and its row tile of many vectors leaves fewer blocks on an SM.  us,
  // CUDA cores -> here (one figure: both), at n = 3,072 / 49,152 / 786,432:
  //   54 vectors, 12 outputs   8.2 -> 10.3 / 19.5 -> 22.5 / 201 -> 215;  16  10.3 / 23.6 -> 22.9 / 248 -> 217
  //               20 outputs  11.1 -> 12.2 / 28.7 -> 26.6 / 301 -> 260;  26  14.3 -> 12.3 / 37.9 -> 26.7 / 396 -> 261
  //   61 vectors, 12 outputs  10.3 -> 10.3 / 20.7 -> 23.3 / 223 -> 220;  16  11.3 -> 10.3 / 28.9 -> 23.7 / 306 -> 220
  //   81 vectors, 12 outputs  10.3 -> 12.3 / 29.5 -> 30.7 / 341 -> 313;  16  12.3 / 35.1 -> 30.7 / 406 -> 313
  // 16 is the line above 60 vectors; up to 60 the line of 26 keeps to what wins at every length.
  // And the error: each MMA truncates where an FP32 FMA rounds, so this form's is about 1.4e-7 of
  // the result (rms) at any basis size, the CUDA cores' grows with the vectors: 1.04e-7 at 26, 1.25 at
  // 41, 1.38 at 51, 1.41 at 54 (here 1.36), 1.49 at 61 (1.41), 1.69 at 81 (1.41).
  if (nv < TU_MINNV || nn < (nv > 60 ? 16 : 26)) return false;
  if (nv < 1 || nv > GDR_MAX_M + 1 || nn > TU_MAXOUT || !ctx->tc_ok || !ctx->tc_update_ok ||
      tc_combine_smem(a.ka, (nn + 15) / 16 * 16, TU_MINRAW, 1) > ctx->tc_combine_smem)
    return false;
  a.n = n;
  a.ncol = nn;
  a.nt = nn;
  a.V = V;
  a.ldv = ldv;
  a.vcs = vcs;
  a.C = C;
  a.cs = ldc;
  a.ccs = ccs;
  a.nout = nout;
  a.X = X;
  a.ldx = ldx;
  a.xcs = xcs;
  a.st = st;
  a.nvec = nvec;
  a.err = err;
  const long ntiles = (n + TU_ROWS - 1) / TU_ROWS;
  const unsigned gx = (unsigned)std::min<long>(std::max(1, ctx->num_sms / ncol), ntiles);
  tc_combine_launch<TU_RESTART>(ctx, a, gx, (unsigned)ncol);
  return true;
}

// ------------------------------------------------------- waits that gave up

// Wait for the stream and for the word that a kernel above sets when one of its waits gives up,
// and, when given, for a batch's first column state -- behind the queued kernels, through the
// context's pinned memory.
ColState fetch_state(gdr_ctx* ctx, const ColState* st, bool& tc_failed) {
  struct Host {
    ColState st;
    int err;
  };
  Host* h = static_cast<Host*>(ctx->host_status(sizeof(Host)));
  *h = Host{};
  if (st) GDR_CUDA(cudaMemcpyAsync(&h->st, st, sizeof(ColState), cudaMemcpyDeviceToHost, ctx->stream));
  if (ctx->tc_err) GDR_CUDA(cudaMemcpyAsync(&h->err, ctx->tc_err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
  GDR_CUDA(cudaStreamSynchronize(ctx->stream));
  tc_failed = h->err != 0;
  return h->st;
}

void tc_fail(gdr_ctx* ctx) {
  GDR_CUDA(cudaMemsetAsync(ctx->tc_err, 0, sizeof(int), ctx->stream));
  GDR_CUDA(cudaStreamSynchronize(ctx->stream));
  throw gdr_error(GDR_ETIMEOUT,
                  "a tensor-core wait gave up, in this call or in a gdr_basis_update queued since the last call that "
                  "synchronised");
}

void tc_check(gdr_ctx* ctx) {
  bool failed;
  fetch_state(ctx, nullptr, failed);
  if (failed) tc_fail(ctx);
}

namespace {
// one wait for an arrival that never comes, ended by its limit (about a second)
__global__ void tc_wait_selftest_kernel(int* err) {
  __shared__ __align__(8) uint64_t bar;
  int own = 0;
  mbar_init(&bar, 1);
  if (!mbar_wait(&bar, 0, &own)) atomicExch(err, 1);
}
}  // namespace

void tc_wait_selftest(gdr_ctx* ctx) {
  tc_wait_selftest_kernel<<<1, 1, 0, ctx->stream>>>(ctx->tc_err);
  GDR_LAUNCHED(ctx);
}

void tc_proj_init(gdr_ctx* ctx) {
  ctx->tc_ok = false;
  if (!encoder()) return;
  cudaFuncAttributes at;
  auto allow = [&](auto kernel) {  // dynamic shared memory this kernel may use
    if (cudaFuncGetAttributes(&at, kernel) != cudaSuccess || at.sharedSizeBytes >= ctx->max_smem_optin) return (size_t)0;
    const size_t dyn = ctx->max_smem_optin - at.sharedSizeBytes;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn) == cudaSuccess ? dyn : 0;
  };
  ctx->tc_dot_smem = std::min(allow(tc_proj_dot_kernel<true>), allow(tc_proj_dot_kernel<false>));
  if (ctx->tc_dot_smem < 1024 + 3 * (size_t)tc_stage_bytes(128, false)) return;
  ctx->tc_ok = true;
  ctx->tc_update_ok = false;
  const int ka = (2 * TU_MAXNV + 31) / 32;
  ctx->tc_combine_smem = std::min({allow(tc_combine_kernel<TU_RESTART>), allow(tc_combine_kernel<TU_DIRECT>),
                                   allow(tc_combine_kernel<TU_REDUCE>)});
  ctx->tc_update_ok = ctx->tc_combine_smem >= tc_combine_smem(ka, 128, TU_MINRAW, 1);
  // the waits' error word, here rather than on first use: the step-level calls may be captured
  ctx->tc_err = ctx->get<int>("tc.err", 4);
  GDR_CUDA(cudaMemset(ctx->tc_err, 0, sizeof(int) * 4));
}
