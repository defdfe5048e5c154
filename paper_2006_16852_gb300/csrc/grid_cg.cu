// grid_cg.cu -- the whole preconditioned CG or BiCGSTAB solve (Section 3.1,
// criteria of Section 2.5) in ONE launch whose CTAs are resident for the whole
// solve, the phases separated by reductions over all CTAs that are the only
// barriers: a cooperative launch of one CTA per SM for mid-size systems, a
// 16-CTA thread-block cluster for small ones.
//
// Between the cluster form's sizes and a few hundred thousand rows, an
// iteration of the graph form is bound by launch and reduction latency (~20
// us for CG's three launches, ~35 us for BiCGSTAB's five) rather than by its
// bytes or FP64 work.  Here an iteration is two (CG) or three (BiCGSTAB)
// grid reductions plus the work spread over all 152 SMs.
//
// Rows: CTA b owns rows [b R, (b + 1) R), thread t the CTA's rows t, t + 256,
// ...; a row's vector entries and Jacobi diagonal stay in the owning thread's
// registers.  The vector an SpMV reads lies in the CTA's shared memory: its
// own rows, and its halo -- every other CTA's row that one of its rows
// refers to (listed once, when the solver is generated).  The halo's
// direction vector is not exchanged: every CTA carries the entries of its
// halo along with the owner's operations, from z = M^{-1} r (and M^{-1} v),
// which the owners publish in global memory (L2).
//
// Whatever crosses CTAs is a 16-byte word {value, sequence number}, stored
// and loaded whole: a reader polls a word until it carries the number it
// waits for, so neither a fence nor a barrier stands between a vector entry
// and its reader, and the halo is fetched by the warps that would otherwise
// idle while the reduction after it is in flight.  A reduction is the same:
// each CTA stores its sum as a word, one warp per value polls all the CTAs'
// words and adds them in one fixed order.  So all CTAs hold bit-identical
// totals and take identical stop decisions, and the two words a CTA may have
// outstanding alternate between two buffers: word b + 2 overwrites word b
// only after reduction b + 1, which every CTA enters only after it has read
// its words of b.  Sequence numbers start at a value of the solve's own, so
// no word needs clearing.
//
// What bounds an iteration is latency.  CG on 65,536 rows, 5-point, about
// 17,900 cycles: direction 1,060, SpMV 2,400, update 1,440 (these three are
// near the FP64 pipe's time for them), and per reduction 1,200 for the CTA's
// sum, 2,300 - 3,700 until the last CTA's word is there, 990 for the sum of
// the words, 980 for a division (260 where none is left).  A dependent FP64
// add takes 68 cycles, a butterfly step 145, and a warp instruction holds its
// quarter of the SM's FP64 pipe for about 64 cycles whatever its lanes do:
// hence one warp per value in a reduction (a quarter each) and scalars
// derived by one thread per CTA.  CG, Jacobi, 256 x 256: 14.7 -> 8.4 ms to
// 1e-12 (15.6 -> 8.9 us per iteration; before: an arrival counter and a
// release word per barrier, vectors re-read from L2); BiCGSTAB, 201 x 199:
// 10.2 -> 4.0 ms (graph form before).
//
// Small systems (the cluster sizes of cluster_cg.cu, whose kernels keep the
// matrices whose halo does not fit): the same kernels on 16 CTAs, the
// reductions' words pushed straight into every CTA's shared memory
// (distributed shared memory) and polled there; the vectors' words stay in
// L2, fetched while a reduction is in flight.  CG, Jacobi, Poisson 64 x 64 to
// 1e-12: 1.40 -> 1.10 ms (6.0 -> 4.7 us per iteration; before: three cluster
// barriers, p gathered across the cluster), 128 x 128 diffusion 4.64 -> 3.82
// ms, BiCGSTAB 128 x 128 3.37 -> 2.68 ms.
//
// Every wait is bounded: one that gives up sets the error bit and an abort
// word that ends every other CTA's waits at once, so the launch always
// returns.
#include <algorithm>
#include <vector>

#include "gk_device.cuh"
#include "gk_internal.h"
#include "solver_state.cuh"

namespace gk {
namespace {

constexpr int kGrThreads = 256;
constexpr int kGrWarps = kGrThreads / 32;
constexpr int kGrMaxCtas = 160;          // 5 words per polling lane
constexpr int kGrMaxRptCg = 8;           // rows per thread: registers of the row's vectors
constexpr int kGrMaxRptBi = 4;
// Below: the cluster form, for BiCGSTAB (whose cluster form ends at 16,384
// rows) the graph form; the line is CG's, BiCGSTAB's own has not been measured.
constexpr int64_t kGrMinRows = 32769;
constexpr int64_t kGrMaxRows = 262144;   // above: the graph form's SpMV kernels win
constexpr int kGrMaxRowLen = 64;         // one thread per row: no long rows
constexpr int kGrMaxK = 3;               // values per reduction
// Copies of a reduction's words, CTA b polling copy b % 8: with one copy the
// polls of 152 CTAs queue on the same few L2 lines (CG on 65,536 rows:
// 21,400 cycles per iteration with 1 copy, 17,900 with 8, 18,400 with 19,
// 18,500 with one per CTA, whose stores cost more than the polls save).
constexpr int kGrCopies = 8;
constexpr int kGrClusterCtas = 16;
constexpr int kGrPlanThreads = 1024;

struct GridArgs {
  const int32_t* rowptr;
  const int32_t* code;   // per entry: the column's place in the CTA's slice (own rows, then halo)
  const double* val;
  const double* b;
  double* x;
  const double* dinv;
  SolverState* st;
  const int32_t* halo_n;    // [grid] halo entries of a CTA
  const int32_t* halo_col;  // [grid][halo_cap] their rows, increasing
  int halo_cap;
  ulonglong2* zw[2];     // z = M^{-1} r as words, step k in buffer k % 2
  ulonglong2* vw[2];     // BiCGSTAB: M^{-1} v
  ulonglong2* words;     // [kGrCopies][2][kGrMaxK][grid] the reductions' words
  unsigned int* abort_;  // nonzero: a wait gave up somewhere
  unsigned long long seq0;
  int n;
  int rows_per_cta;
  int stage_nnz;  // STAGE: room for this many entries of the CTA's rows in shared memory
};

__device__ __forceinline__ void store_word(ulonglong2* p, double v, unsigned long long seq) {
  asm volatile("{\n .reg .b128 w;\n mov.b128 w, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], w;\n}\n" ::"l"(p),
               "l"(static_cast<unsigned long long>(__double_as_longlong(v))), "l"(seq)
               : "memory");
}

__device__ __forceinline__ double load_word(const ulonglong2* p, unsigned long long& seq) {
  unsigned long long v;
  asm volatile("{\n .reg .b128 w;\n ld.relaxed.gpu.global.b128 w, [%2];\n mov.b128 {%0, %1}, w;\n}\n"
               : "=l"(v), "=l"(seq)
               : "l"(p)
               : "memory");
  return __longlong_as_double(static_cast<long long>(v));
}

// The reductions' shared memory.
struct GridRed {
  double part[kGrMaxK][kGrThreads];
  double tot[kGrMaxK];
  // CLUSTER: the CTAs' sums, pushed by their owners: each double as two 8-byte
  // words {half, sequence number}, zero (no number) at the start
  unsigned long long push[2][kGrMaxK][kGrClusterCtas][2];
  int ok;
};

// An 8-byte store into another CTA's shared memory (cluster address), and the
// owner's load of it; each 8-byte word arrives whole.
__device__ __forceinline__ void push_word(uint32_t addr, uint32_t half, uint32_t seq) {
  asm volatile("{\n .reg .b64 w;\n mov.b64 w, {%1, %2};\n st.relaxed.cluster.shared::cluster.b64 [%0], w;\n}\n" ::"r"(addr),
               "r"(half), "r"(seq)
               : "memory");
}
__device__ __forceinline__ uint2 pushed_word(const unsigned long long* p) {
  uint2 w;
  asm volatile("{\n .reg .b64 w;\n ld.relaxed.cluster.shared::cta.b64 w, [%2];\n mov.b64 {%0, %1}, w;\n}\n"
               : "=r"(w.x), "=r"(w.y)
               : "r"(smem_u32(p))
               : "memory");
  return w;
}
__device__ __forceinline__ uint32_t cluster_addr(const void* p, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Bounds a polling loop: true when the wait has to be given up (this one's
// limit, or another wait's).
struct GrWait {
  long long t0 = 0;
  uint32_t polls = 0;
  __device__ __forceinline__ bool give_up(const GridArgs& a) {
    if (polls++ == 0) t0 = clock64();
    if (*static_cast<volatile unsigned int*>(a.abort_) != 0u) return true;
    if (polls <= kMaxPolls && clock64() - t0 <= kMaxWaitCycles) return false;
    atomicOr(&a.st->err, kErrTimeout);
    atomicExch(a.abort_, 1u);
    return true;
  }
};

// dst[h] = the halo's words (buffer w, sequence number seq), by threads
// [first, 256) of the block, four words of a thread in flight.
__device__ __forceinline__ void fetch_halo(const GridArgs& a, GridRed& red, const ulonglong2* w,
                                           unsigned long long seq, const int32_t* cols, int H, double* dst,
                                           int first) {
  const int nt = kGrThreads - first;
  for (int h0 = static_cast<int>(threadIdx.x) - first; h0 < H; h0 += 4 * nt) {
    double v[4];
    const ulonglong2* src[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) src[j] = w + __ldg(cols + min(h0 + j * nt, H - 1));
    GrWait wait;
    for (;;) {
      bool here = true;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        unsigned long long q;
        v[j] = load_word(src[j], q);
        here = here && q == seq;
      }
      if (here) break;
      if (wait.give_up(a)) {
        red.ok = 0;
        return;
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (h0 + j * nt < H) dst[h0 + j * nt] = v[j];
  }
}

// Sums v over the grid; then lanes 0 and 1 of warp k < K of every CTA run
// post(k, lane, totals) (the iteration's scalars are derived once per CTA, in
// parallel where they are independent: FP64 divisions and square roots are
// long, and two quotients in two lanes take the time of one); false if the solve is being aborted.  Warp k sums value k: 8
// threads' values per lane, one butterfly, then the CTAs' words, 5 per lane,
// and one butterfly.  Meanwhile the other warps run idle(32 K).
template <bool CLUSTER, int K, typename Idle, typename Post>
__device__ __forceinline__ bool grid_total(const GridArgs& a, GridRed& red, unsigned long long& seq,
                                           const double (&v)[K], Idle idle, Post post) {
  // the warp's index from lane 0, so that the branch on it is uniform: the
  // shuffles under a branch on threadIdx.x took 620 cycles a step
  const int lane = threadIdx.x & 31, warp = warp_uniform(threadIdx.x >> 5);
#pragma unroll
  for (int k = 0; k < K; ++k) red.part[k][threadIdx.x] = v[k];
  ++seq;
  __syncthreads();
  if (warp < K) {
    const int G = gridDim.x;
    const int slot = (static_cast<int>(seq & 1) * kGrMaxK + warp) * G;
    const int copy = 2 * kGrMaxK * G;  // words per copy
    double u[kGrWarps];
#pragma unroll
    for (int w = 0; w < kGrWarps; ++w) u[w] = red.part[warp][lane + 32 * w];
#pragma unroll
    for (int h = kGrWarps / 2; h > 0; h >>= 1) {
#pragma unroll
      for (int w = 0; w < h; ++w) u[w] += u[w + h];
    }
    double s[1] = {u[0]};
    warp_sum<1, double>(s);
    GrWait wait;
    bool ok = true;
    if constexpr (CLUSTER) {
      const uint32_t seq32 = static_cast<uint32_t>(seq);
      unsigned long long(*slot)[2] = red.push[seq & 1][warp];
      if (lane < kGrClusterCtas) {
        const uint32_t to = cluster_addr(slot[blockIdx.x], static_cast<uint32_t>(lane));
        push_word(to, static_cast<uint32_t>(__double2loint(s[0])), seq32);
        push_word(to + 8, static_cast<uint32_t>(__double2hiint(s[0])), seq32);
      }
      uint2 w0, w1;
      for (;;) {
        w0 = pushed_word(&slot[lane & (kGrClusterCtas - 1)][0]);
        w1 = pushed_word(&slot[lane & (kGrClusterCtas - 1)][1]);
        if (__all_sync(0xffffffffu, w0.y == seq32 && w1.y == seq32)) break;
        const int stop = lane == 0 ? static_cast<int>(wait.give_up(a)) : 0;
        if (__shfl_sync(0xffffffffu, stop, 0)) {
          ok = false;
          break;
        }
      }
      s[0] = __hiloint2double(static_cast<int>(w1.x), static_cast<int>(w0.x));
#pragma unroll
      for (int o = kGrClusterCtas / 2; o > 0; o >>= 1) s[0] += __shfl_xor_sync(0xffffffffu, s[0], o);
    } else {
      if (lane < kGrCopies) store_word(a.words + lane * copy + slot + blockIdx.x, s[0], seq);
      __syncwarp();
      const ulonglong2* words = a.words + static_cast<int>(blockIdx.x % kGrCopies) * copy + slot;
      double c[kGrMaxCtas / 32];
      bool got[kGrMaxCtas / 32];
#pragma unroll
      for (int j = 0; j < kGrMaxCtas / 32; ++j) {
        c[j] = 0.0;
        got[j] = lane + 32 * j >= G;
      }
      for (;;) {
        bool here = true;
#pragma unroll
        for (int j = 0; j < kGrMaxCtas / 32; ++j) {
          if (!got[j]) {
            unsigned long long q;
            c[j] = load_word(words + lane + 32 * j, q);
            got[j] = q == seq;
          }
        }
#pragma unroll
        for (int j = 0; j < kGrMaxCtas / 32; ++j) here = here && got[j];
        if (__all_sync(0xffffffffu, here)) break;
        const int stop = lane == 0 ? static_cast<int>(wait.give_up(a)) : 0;
        if (__shfl_sync(0xffffffffu, stop, 0)) {
          ok = false;
          break;
        }
      }
      s[0] = c[0];
#pragma unroll
      for (int j = 1; j < kGrMaxCtas / 32; ++j) s[0] += c[j];
      warp_sum<1, double>(s);
    }
    if (lane == 0) {
      red.tot[warp] = s[0];
      if (!ok) red.ok = 0;
    }
    if (K > 1) asm volatile("bar.sync 1, %0;" ::"n"(32 * K) : "memory");
    else __syncwarp();
    if (lane < 2) post(warp, lane, red.tot);
  } else {
    idle(32 * K);
  }
  __syncthreads();
  return red.ok != 0;
}

// The CTA's rows of the matrix (row pointers relative to the CTA's first
// entry, codes, values), in shared memory if they fit (SRC_STAGED), and its
// halo.
enum GridSrc { SRC_STAGED = 0, SRC_SHORT = 1, SRC_LONG = 2 };
constexpr int kGrLongRow = 16;  // SRC_LONG: some row has more entries

template <int SRC>
struct GridRows {
  static constexpr bool STAGE = SRC == SRC_STAGED;
  const int32_t* rp;
  const int32_t* code;
  const double* val;
  const int32_t* halo;
  int row0, rows, H;

  __device__ __forceinline__ void init(const GridArgs& a, double* s_val) {
    const int R = a.rows_per_cta;
    row0 = min(static_cast<int>(blockIdx.x) * R, a.n);
    rows = min(R, a.n - row0);
    H = __ldg(a.halo_n + blockIdx.x);
    halo = a.halo_col + static_cast<int64_t>(blockIdx.x) * a.halo_cap;
    if (STAGE) {
      int32_t* s_rp = reinterpret_cast<int32_t*>(s_val + a.stage_nnz);
      int32_t* s_code = s_rp + R + 1;
      const int e0 = __ldg(a.rowptr + row0);
      for (int l = threadIdx.x; l <= R; l += kGrThreads) s_rp[l] = __ldg(a.rowptr + row0 + min(l, rows)) - e0;
      const int ne = __ldg(a.rowptr + row0 + rows) - e0;
      for (int k = threadIdx.x; k < ne; k += kGrThreads) {
        s_code[k] = __ldg(a.code + e0 + k);
        s_val[k] = __ldg(a.val + e0 + k);
      }
      rp = s_rp;
      code = s_code;
      val = s_val;
    } else {
      rp = a.rowptr + row0;
      code = a.code;
      val = a.val;
    }
  }

  // sum_k val_k loc[code_k] of the local row l in increasing k (the oracle's
  // ordered SpMV); entries in groups of 8 so that their loads are in flight
  // together.  Rows read from memory are bound by the L1 lookups, one per
  // thread and load, since a warp's rows lie far apart: from the first entry
  // on a 16-byte boundary of the codes on, long rows are read 16 bytes at a
  // time, 6 loads for 8 entries instead of 16.  Us per iteration, one entry a
  // load / this form / the kernels of cluster_cg.cu: CG on 61 diagonals,
  // 16,000 rows 76.8 / 42.6 / 66.5, 81 diagonals, 4,000 rows 40.0 / 19.7 /
  // 32.8, 27-point 32^3 59.8 / 36.4 / 53.1; BiCGSTAB on the first two 142 / 81 / 111
  // and 77.7 / 37.4 / 57.3.  Rows of up to kGrLongRow entries are two groups
  // at most, and the steps to and from the boundary cost them more (9
  // diagonals 19.4 against 21.5); matrices of such rows alone have kernels
  // without the other form, whose code costs theirs 1 to 4 %.
  __device__ __forceinline__ double apply(int l, const double* loc) const {
    double s = 0.0;
    int k = STAGE ? rp[l] : __ldg(rp + l);
    const int k1 = STAGE ? rp[l + 1] : __ldg(rp + l + 1);
    if (SRC == SRC_LONG && k1 - k > kGrLongRow) {
      const int ka = (k + 3) & ~3;
      int cp[3];
      double vp[3];
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        cp[u] = 0;
        vp[u] = 0.0;
        if (k + u < ka) {
          cp[u] = __ldg(code + k + u);
          vp[u] = __ldg(val + k + u);
        }
      }
#pragma unroll
      for (int u = 0; u < 3; ++u)
        if (k + u < ka) s = fma(vp[u], loc[cp[u]], s);
      for (k = ka; k + 8 <= k1; k += 8) {
        int4 c[2];
        double2 v[4];
#pragma unroll
        for (int u = 0; u < 2; ++u) c[u] = __ldg(reinterpret_cast<const int4*>(code + k) + u);
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = __ldg(reinterpret_cast<const double2*>(val + k) + u);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          s = fma(v[2 * u].x, loc[c[u].x], s);
          s = fma(v[2 * u].y, loc[c[u].y], s);
          s = fma(v[2 * u + 1].x, loc[c[u].z], s);
          s = fma(v[2 * u + 1].y, loc[c[u].w], s);
        }
      }
    }
    for (; k < k1; k += 8) {
      double v[8], w[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        v[u] = w[u] = 0.0;
        if (k + u < k1) {
          v[u] = STAGE ? val[k + u] : __ldg(val + k + u);
          w[u] = loc[STAGE ? code[k + u] : __ldg(code + k + u)];
        }
      }
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (k + u < k1) s = fma(v[u], w[u], s);
    }
    return s;
  }
};

// The iteration's scalars, derived by one thread of each CTA.  A division or
// a square root there is about 650 cycles that every thread waits for, so
// beta's divisor is inverted along with an earlier quotient, in another lane
// (scale), and a norm's square root is taken only where the criteria may
// hold: rr > tol2 implies ||r|| > tol.  An inverse that is no normal number
// (the divisor below 5.6e-309 or above 4.5e307, as with a right-hand side
// scaled near 1e-150 or 1e150) is not used: beta is then the quotient itself,
// by a call, so that its divisions stay out of the way (inlined, and with the
// inverse's factors checked one by one, BiCGSTAB on 100 x 110 took 2,345 us,
// 2,334 so, 2,327 without any check).
__device__ __forceinline__ bool gr_normal(double v) {
  return ((static_cast<unsigned int>(__double2hiint(v)) >> 20) & 0x7ffu) - 1u < 0x7feu;
}

__device__ __noinline__ double gr_slow_beta(double rho, double prev, double alpha, double omega) {
  return (rho / prev) * (alpha / omega);
}

struct GrScalars {
  double rho, rho_prev, alpha, omega, beta, scale, rr, ss, rnorm0, bnorm, ref, tol, tol2;
  long long iter, spmvs;
  int stop, half, om_stop;
};

__device__ __forceinline__ void gr_init_scalars(GrScalars& sc) {
  sc.rnorm0 = sc.bnorm = sc.rr = sc.ss = sc.rho = sc.tol = sc.tol2 = 0.0;
  sc.ref = sc.alpha = sc.omega = sc.rho_prev = sc.scale = 1.0;
  sc.beta = 0.0;
  sc.iter = 0;
  sc.spmvs = 1;
  sc.stop = GK_STOP_NONE;
  sc.half = 0;
  sc.om_stop = GK_STOP_NONE;
}

// The solve's shared state; CLUSTER: every CTA of the cluster has started (and
// its words are clear) before any is written to.
template <bool CLUSTER>
__device__ __forceinline__ void gr_start(GrScalars& sc, GridRed& red) {
  if (threadIdx.x == 0) {
    gr_init_scalars(sc);
    red.ok = 1;
  }
  if constexpr (CLUSTER) {
    unsigned long long* w = &red.push[0][0][0][0];
    for (int i = threadIdx.x; i < 2 * kGrMaxK * kGrClusterCtas * 2; i += kGrThreads) w[i] = 0ull;
    cluster_barrier();
  } else {
    __syncthreads();
  }
}

// ||r0||^2 and ||b||^2 to the reference norm and the tolerance
__device__ __forceinline__ void gr_setup_norms(GrScalars& sc, const double* tt, int rel_to_b, double factor) {
  sc.rr = tt[0];
  sc.rnorm0 = sqrt(tt[0]);
  sc.bnorm = sqrt(tt[1]);
  double ref = rel_to_b ? sc.bnorm : sc.rnorm0;
  if (ref == 0.0) ref = 1.0;
  sc.ref = ref;
  sc.tol = factor * ref;
  sc.tol2 = sc.tol * sc.tol * (1.0 + 0x1p-49);  // the margin covers the roundings of the product and the square root
}

// The criteria on a squared norm: NaN, residual, iteration count.
__device__ __forceinline__ int gr_criteria(const GrScalars& sc, double rr, long long k, long long max_iters) {
  if (rr > sc.tol2 && isfinite(rr)) return k >= max_iters ? GK_STOP_MAX_ITERS : GK_STOP_NONE;
  const double rn = sqrt(rr);
  if (!isfinite(rn)) return GK_STOP_NAN;
  if (rn <= sc.tol) return GK_STOP_CONVERGED;
  if (k >= max_iters) return GK_STOP_MAX_ITERS;
  return GK_STOP_NONE;
}

__device__ __forceinline__ void gr_store_state(SolverState* st, const GrScalars& sc, bool ok) {
  st->rnorm = sqrt(sc.rr);
  st->snorm = sqrt(sc.ss);
  st->rnorm0 = sc.rnorm0;
  st->bnorm = sc.bnorm;
  st->ref = sc.ref;
  st->tol = sc.tol;
  st->rho = sc.rho;
  st->rho_prev = sc.rho_prev;
  st->alpha = sc.alpha;
  st->omega = sc.omega;
  st->beta = sc.beta;
  st->half = sc.half;
  st->iter = sc.iter;
  st->iter_guard = sc.iter;
  st->spmvs = sc.spmvs;
  st->stop = ok ? sc.stop : GK_STOP_NAN;
}

// CG.  An iteration:
//   p = z + beta p (own rows and halo), q = A p, sigma = p.q   -> reduction
//   alpha = rho / sigma; x += alpha p; r -= alpha q;
//   z = M^{-1} r (published); rho' = r.z, ||r||^2              -> reduction,
//                                       the halo's z fetched meanwhile
//   criteria; beta = rho' / rho
// Shared memory: p of own rows and halo, z of the halo, the staged rows.
template <int PK, int RPT, int SRC, bool CLUSTER>
__global__ void __launch_bounds__(kGrThreads, 1) cg_grid_kernel(GridArgs a) {
  extern __shared__ double loc[];
  __shared__ GridRed red;
  __shared__ GrScalars sc;
  const int t = threadIdx.x;
  const int R = a.rows_per_cta;
  double* const ph = loc + R;            // p of the halo
  double* const zh = ph + a.halo_cap;    // z of the halo
  GridRows<SRC> A;
  A.init(a, zh + a.halo_cap);
  const int row0 = A.row0, H = A.H;
  SolverState* st = a.st;
  const double factor = st->factor;
  const long long max_iters = st->max_iters;
  const int rel_to_b = st->rel_to_b;
  unsigned long long seq = a.seq0;

  double x[RPT], r[RPT], d[RPT], z[RPT], p[RPT];
  bool own[RPT];
#pragma unroll
  for (int u = 0; u < RPT; ++u) {
    const int l = t + u * kGrThreads;
    own[u] = l < A.rows;
    x[u] = own[u] ? a.x[row0 + l] : 0.0;
    d[u] = (PK == PREC_SCALAR && own[u]) ? __ldg(a.dinv + row0 + l) : 1.0;
    r[u] = z[u] = p[u] = 0.0;
    if (own[u]) loc[l] = x[u];
  }
  // x0 itself is not written before the end of the solve
  for (int h = t; h < H; h += kGrThreads) ph[h] = a.x[__ldg(A.halo + h)];
  gr_start<CLUSTER>(sc, red);
  unsigned long long zseq = a.seq0 + 1;  // sequence number of z_k's words
  bool ok;
  {
    double v[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int u = 0; u < RPT; ++u) {
      if (!own[u]) continue;
      const int l = t + u * kGrThreads;
      const double bi = a.b[row0 + l];
      r[u] = bi - A.apply(l, loc);
      z[u] = PK == PREC_SCALAR ? d[u] * r[u] : r[u];
      store_word(a.zw[0] + row0 + l, z[u], zseq);
      v[0] = fma(r[u], r[u], v[0]);
      v[1] = fma(bi, bi, v[1]);
      v[2] = fma(r[u], z[u], v[2]);
    }
    ok = grid_total<CLUSTER, 3>(
        a, red, seq, v, [&](int first) { fetch_halo(a, red, a.zw[0], zseq, A.halo, H, zh, first); },
        [&](int w, int lane, const double* tt) {
          if (w != 0 || lane != 0) return;
          gr_setup_norms(sc, tt, rel_to_b, factor);
          sc.rho = tt[2];
          sc.stop = gr_criteria(sc, sc.rr, 0, max_iters);
        });
  }
  for (long long k = 0; ok && sc.stop == GK_STOP_NONE; ++k) {
    const double beta = sc.beta;
#pragma unroll
    for (int u = 0; u < RPT; ++u) {
      if (!own[u]) continue;
      p[u] = k == 0 ? z[u] : fma(beta, p[u], z[u]);
      loc[t + u * kGrThreads] = p[u];
    }
    for (int h = t; h < H; h += kGrThreads) ph[h] = k == 0 ? zh[h] : fma(beta, ph[h], zh[h]);
    __syncthreads();
    double q[RPT];
    double v[1] = {0.0};
#pragma unroll
    for (int u = 0; u < RPT; ++u) {
      q[u] = 0.0;
      if (!own[u]) continue;
      q[u] = A.apply(t + u * kGrThreads, loc);
      v[0] = fma(p[u], q[u], v[0]);
    }
    if (!(ok = grid_total<CLUSTER, 1>(a, red, seq, v, [](int) {}, [&](int, int lane, const double* tt) {
            // lane 0: alpha = rho / sigma; lane 1: the next beta's factor 1 / rho
            const double sigma = tt[0];
            const double q = (lane == 0 ? sc.rho : 1.0) / (lane == 0 ? sigma : sc.rho);
            if (lane == 1) {
              sc.scale = q;
              return;
            }
            sc.spmvs += 1;
            if (!isfinite(sigma)) sc.stop = GK_STOP_NAN;
            else if (sigma <= 0.0) sc.stop = GK_STOP_BREAKDOWN;
            else sc.alpha = q;
          })))
      break;
    if (sc.stop != GK_STOP_NONE) break;
    const double alpha = sc.alpha;
    ulonglong2* const zw = a.zw[(k + 1) & 1];
    ++zseq;
    double w[2] = {0.0, 0.0};
#pragma unroll
    for (int u = 0; u < RPT; ++u) {
      if (!own[u]) continue;
      r[u] = fma(-alpha, q[u], r[u]);
      z[u] = PK == PREC_SCALAR ? d[u] * r[u] : r[u];
      store_word(zw + row0 + t + u * kGrThreads, z[u], zseq);
      x[u] = fma(alpha, p[u], x[u]);
      w[0] = fma(r[u], z[u], w[0]);
      w[1] = fma(r[u], r[u], w[1]);
    }
    if (!(ok = grid_total<CLUSTER, 2>(
              a, red, seq, w, [&](int first) { fetch_halo(a, red, zw, zseq, A.halo, H, zh, first); },
              [&](int warp, int lane, const double* tt) {
                if (lane != 0) return;
                if (warp == 0) {
                  sc.beta = gr_normal(sc.scale) ? tt[0] * sc.scale : gr_slow_beta(tt[0], sc.rho, 1.0, 1.0);
                  sc.rho = tt[0];
                } else {
                  sc.iter += 1;
                  sc.rr = tt[1];
                  sc.stop = gr_criteria(sc, sc.rr, sc.iter, max_iters);
                }
              })))
      break;
  }
#pragma unroll
  for (int u = 0; u < RPT; ++u)
    if (own[u]) a.x[row0 + t + u * kGrThreads] = x[u];
  if (blockIdx.x == 0 && t == 0) gr_store_state(st, sc, ok);
  if (CLUSTER) cluster_barrier();  // no CTA leaves while others may still write to its shared memory
}

// BiCGSTAB (the Templates form, as the graph form computes it, with the
// direction kept in the preconditioned space: p^ = M^{-1} p obeys the same
// recurrence with M^{-1} r and M^{-1} v, and p itself enters nothing else).
// With z = M^{-1} r and v^ = M^{-1} v, an iteration:
//   p^ = z + beta (p^ - omega v^), v = A p^, v^ (published);
//   r^.v                                  -> reduction, the halo's v^ fetched
//   alpha; s = r - alpha v, s^ = z - alpha v^, t = A s^;
//   s.t, ||s||, t.t                       -> reduction
//   half-step exit; omega; x += alpha p^ + omega s^;
//   r = s - omega t, z (published); r^.r, ||r||  -> reduction, the halo's z
//   criteria; rho, beta
// (t is computed before the half-step test is known, which saves a grid
// reduction in every iteration and costs one SpMV in the last.)
// Shared memory: the SpMV's input on own rows and halo; p^, z and v^ of the
// halo; the staged rows.
template <int PK, int RPT, int SRC, bool CLUSTER>
__global__ void __launch_bounds__(kGrThreads, 1) bicg_grid_kernel(GridArgs a) {
  extern __shared__ double loc[];
  __shared__ GridRed red;
  __shared__ GrScalars sc;
  const int t = threadIdx.x;
  const int R = a.rows_per_cta;
  double* const in_h = loc + R;
  double* const ph_h = in_h + a.halo_cap;
  double* const z_h = ph_h + a.halo_cap;
  double* const vh_h = z_h + a.halo_cap;
  GridRows<SRC> A;
  A.init(a, vh_h + a.halo_cap);
  const int row0 = A.row0, H = A.H;
  SolverState* st = a.st;
  const double factor = st->factor;
  const long long max_iters = st->max_iters;
  const int rel_to_b = st->rel_to_b;
  unsigned long long seq = a.seq0;

  double x[RPT], r[RPT], rh[RPT], d[RPT], z[RPT], ph[RPT], v[RPT], vh[RPT], tv[RPT];
  bool own[RPT];
#pragma unroll
  for (int u = 0; u < RPT; ++u) {
    const int l = t + u * kGrThreads;
    own[u] = l < A.rows;
    x[u] = own[u] ? a.x[row0 + l] : 0.0;
    d[u] = (PK == PREC_SCALAR && own[u]) ? __ldg(a.dinv + row0 + l) : 1.0;
    r[u] = rh[u] = z[u] = ph[u] = v[u] = vh[u] = tv[u] = 0.0;
    if (own[u]) loc[l] = x[u];
  }
  for (int h = t; h < H; h += kGrThreads) in_h[h] = a.x[__ldg(A.halo + h)];
  gr_start<CLUSTER>(sc, red);
  // a fresh rho = r^.r either fails (NaN, zero) or yields the next beta
  auto new_rho = [&](double rho) {
    if (!isfinite(rho)) sc.stop = GK_STOP_NAN;
    else if (rho == 0.0) sc.stop = GK_STOP_BREAKDOWN;
    else {
      // scale = (alpha / omega) / the previous rho = (1 / r^.v) (t.t / s.t).
      // The first factor loses 4 bits at most where it is subnormal, the
      // second more where omega is that large.
      const bool usable = gr_normal(sc.scale) && fabs(sc.omega) < 0x1p1000;
      sc.beta = usable ? rho * sc.scale : gr_slow_beta(rho, sc.rho, sc.alpha, sc.omega);
      sc.rho = rho;
    }
  };
  unsigned long long wseq = a.seq0 + 1;  // sequence number of step k's words
  bool ok;
  {
    double w[2] = {0.0, 0.0};
#pragma unroll
    for (int u = 0; u < RPT; ++u) {
      if (!own[u]) continue;
      const int l = t + u * kGrThreads;
      const double bi = a.b[row0 + l];
      r[u] = bi - A.apply(l, loc);
      rh[u] = r[u];
      z[u] = PK == PREC_SCALAR ? d[u] * r[u] : r[u];
      store_word(a.zw[0] + row0 + l, z[u], wseq);
      w[0] = fma(r[u], r[u], w[0]);
      w[1] = fma(bi, bi, w[1]);
    }
    // r^ = r0: rho = r^.r is ||r0||^2
    ok = grid_total<CLUSTER, 2>(
        a, red, seq, w, [&](int first) { fetch_halo(a, red, a.zw[0], wseq, A.halo, H, z_h, first); },
        [&](int warp, int lane, const double* tt) {
          if (warp != 0 || lane != 0) return;
          gr_setup_norms(sc, tt, rel_to_b, factor);
          sc.stop = gr_criteria(sc, sc.rr, 0, max_iters);
          if (sc.stop == GK_STOP_NONE) new_rho(tt[0]);
        });
  }
  for (long long k = 0; ok && sc.stop == GK_STOP_NONE; ++k) {
    const int cur = static_cast<int>(k & 1);
    {
      const double beta = sc.beta, omega = sc.omega;
#pragma unroll
      for (int u = 0; u < RPT; ++u) {
        if (!own[u]) continue;
        ph[u] = k == 0 ? z[u] : fma(beta, fma(-omega, vh[u], ph[u]), z[u]);
        loc[t + u * kGrThreads] = ph[u];
      }
      for (int h = t; h < H; h += kGrThreads) {
        const double p = k == 0 ? z_h[h] : fma(beta, fma(-omega, vh_h[h], ph_h[h]), z_h[h]);
        ph_h[h] = p;
        in_h[h] = p;
      }
      __syncthreads();
      double w[1] = {0.0};
#pragma unroll
      for (int u = 0; u < RPT; ++u) {
        if (!own[u]) continue;
        const int l = t + u * kGrThreads;
        v[u] = A.apply(l, loc);
        vh[u] = PK == PREC_SCALAR ? d[u] * v[u] : v[u];
        store_word(a.vw[cur] + row0 + l, vh[u], wseq);
        w[0] = fma(rh[u], v[u], w[0]);
      }
      if (!(ok = grid_total<CLUSTER, 1>(
                a, red, seq, w,
                [&](int first) { fetch_halo(a, red, a.vw[cur], wseq, A.halo, H, vh_h, first); },
                [&](int, int lane, const double* tt) {
                  // lane 0: alpha = rho / r^.v; lane 1: 1 / r^.v for the next beta
                  const double rhv = tt[0];
                  const double q = (lane == 0 ? sc.rho : 1.0) / rhv;
                  if (lane == 1) {
                    sc.scale = q;
                    return;
                  }
                  sc.spmvs += 1;
                  if (!isfinite(rhv)) sc.stop = GK_STOP_NAN;
                  else if (rhv == 0.0) sc.stop = GK_STOP_BREAKDOWN;
                  else sc.alpha = q;
                })))
        break;
    }
    if (sc.stop != GK_STOP_NONE) break;
    const double alpha = sc.alpha;
    {
      // s in r's place, s^ in z's
#pragma unroll
      for (int u = 0; u < RPT; ++u) {
        if (!own[u]) continue;
        r[u] = fma(-alpha, v[u], r[u]);
        z[u] = fma(-alpha, vh[u], z[u]);
        loc[t + u * kGrThreads] = z[u];
      }
      for (int h = t; h < H; h += kGrThreads) in_h[h] = fma(-alpha, vh_h[h], z_h[h]);
      __syncthreads();
      double w[3] = {0.0, 0.0, 0.0};
#pragma unroll
      for (int u = 0; u < RPT; ++u) {
        if (!own[u]) continue;
        tv[u] = A.apply(t + u * kGrThreads, loc);
        w[0] = fma(r[u], tv[u], w[0]);
        w[1] = fma(r[u], r[u], w[1]);
        w[2] = fma(tv[u], tv[u], w[2]);
      }
      // warp 0: omega and its failures; warp 1: the half-step test, which
      // comes first where both hold
      if (!(ok = grid_total<CLUSTER, 3>(a, red, seq, w, [](int) {}, [&](int warp, int lane, const double* tt) {
              if (warp == 0) {
                // lane 0: omega = s.t / t.t; lane 1: the next beta's factor
                // (alpha / omega) / rho = (1 / r^.v) (t.t / s.t)
                const double q = tt[lane == 0 ? 0 : 2] / tt[lane == 0 ? 2 : 0];
                if (lane == 1) {
                  sc.scale *= q;
                  return;
                }
                if (!isfinite(tt[2]) || !isfinite(tt[0])) sc.om_stop = GK_STOP_NAN;
                else if (tt[2] == 0.0) sc.om_stop = GK_STOP_BREAKDOWN;
                else sc.omega = q;
              } else if (warp == 1 && lane == 0) {
                sc.ss = tt[1];
                if (gr_criteria(sc, sc.ss, 0, 1) == GK_STOP_CONVERGED) {
                  sc.half = 1;
                  sc.iter += 1;
                  sc.rr = sc.ss;
                  sc.stop = GK_STOP_CONVERGED;
                } else {
                  sc.spmvs += 1;
                }
              }
            })))
        break;
    }
    if (sc.half) {
#pragma unroll
      for (int u = 0; u < RPT; ++u) x[u] = fma(alpha, ph[u], x[u]);
      break;
    }
    if (sc.om_stop != GK_STOP_NONE) break;
    const double omega = sc.omega;
    {
      ulonglong2* const zw = a.zw[cur ^ 1];
      ++wseq;
      double w[2] = {0.0, 0.0};
#pragma unroll
      for (int u = 0; u < RPT; ++u) {
        if (!own[u]) continue;
        const double zs = z[u];
        r[u] = fma(-omega, tv[u], r[u]);
        z[u] = PK == PREC_SCALAR ? d[u] * r[u] : r[u];
        store_word(zw + row0 + t + u * kGrThreads, z[u], wseq);
        x[u] = fma(omega, zs, fma(alpha, ph[u], x[u]));
        w[0] = fma(rh[u], r[u], w[0]);
        w[1] = fma(r[u], r[u], w[1]);
      }
      if (!(ok = grid_total<CLUSTER, 2>(
                a, red, seq, w,
                [&](int first) { fetch_halo(a, red, zw, wseq, A.halo, H, z_h, first); },
                [&](int warp, int lane, const double* tt) {
                  if (warp != 0 || lane != 0) return;
                  sc.iter += 1;
                  sc.rho_prev = sc.rho;
                  sc.rr = tt[1];
                  int stop = gr_criteria(sc, sc.rr, sc.iter, max_iters);
                  if (stop == GK_STOP_NONE && sc.omega == 0.0) stop = GK_STOP_BREAKDOWN;
                  sc.stop = stop;
                  if (stop == GK_STOP_NONE) new_rho(tt[0]);
                })))
        break;
    }
  }
#pragma unroll
  for (int u = 0; u < RPT; ++u)
    if (own[u]) a.x[row0 + t + u * kGrThreads] = x[u];
  if (blockIdx.x == 0 && t == 0) {
    if (sc.stop == GK_STOP_NONE) sc.stop = sc.om_stop;
    gr_store_state(st, sc, ok);
  }
  if (CLUSTER) cluster_barrier();
}

// The halo of every CTA: a bitmap of the columns of its rows that other CTAs
// own (n bits of shared memory), and their ranks.  With halo_col null only
// counts are written, of the halos, then of the CTAs' entries and of those of
// their longest rows (halo_n[3][grid]); else the halos' counts, their columns
// in increasing order and, per entry of the matrix, the place of its column
// in the CTA's slice.
__global__ void __launch_bounds__(kGrPlanThreads) gr_halo_kernel(const int32_t* __restrict__ rowptr,
                                                                 const int32_t* __restrict__ col, int n, int R,
                                                                 int halo_cap, int32_t* __restrict__ halo_n,
                                                                 int32_t* __restrict__ halo_col,
                                                                 int32_t* __restrict__ code) {
  extern __shared__ uint32_t bits[];  // ceil(n / 32) words, then as many ranks
  __shared__ int wsum[kGrPlanThreads / 32];
  __shared__ int s_longest;
  const int nw = (n + 31) / 32;
  int* rank = reinterpret_cast<int*>(bits + nw);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int row0 = min(static_cast<int>(blockIdx.x) * R, n), rows = min(R, n - row0);
  const int e0 = rowptr[row0], e1 = rowptr[row0 + rows];
  for (int w = t; w < nw; w += kGrPlanThreads) bits[w] = 0u;
  if (t == 0) s_longest = 0;
  __syncthreads();
  if (!halo_col) {
    int longest = 0;
    for (int l = t; l < rows; l += kGrPlanThreads) longest = max(longest, rowptr[row0 + l + 1] - rowptr[row0 + l]);
    atomicMax(&s_longest, longest);
  }
  for (int k = e0 + t; k < e1; k += kGrPlanThreads) {
    const int c = col[k];
    if (c < row0 || c >= row0 + rows) atomicOr(bits + (c >> 5), 1u << (c & 31));
  }
  __syncthreads();
  // exclusive ranks of the words: each thread a run of consecutive words
  const int per = (nw + kGrPlanThreads - 1) / kGrPlanThreads;
  const int w0 = min(t * per, nw), w1 = min(w0 + per, nw);
  int sum = 0;
  for (int w = w0; w < w1; ++w) sum += __popc(bits[w]);
  int incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += up;
  }
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  int base = 0;
  for (int w = 0; w < warp; ++w) base += wsum[w];
  int at = base + incl - sum;
  for (int w = w0; w < w1; ++w) {
    rank[w] = at;
    at += __popc(bits[w]);
  }
  if (t == kGrPlanThreads - 1) halo_n[blockIdx.x] = at;
  if (!halo_col) {
    if (t == 0) {
      halo_n[gridDim.x + blockIdx.x] = e1 - e0;
      halo_n[2 * gridDim.x + blockIdx.x] = s_longest;
    }
    return;
  }
  __syncthreads();
  int32_t* out = halo_col + static_cast<int64_t>(blockIdx.x) * halo_cap;
  for (int w = t; w < nw; w += kGrPlanThreads) {
    uint32_t m = bits[w];
    int i = rank[w];
    while (m) {
      const int bit = __ffs(static_cast<int>(m)) - 1;
      out[i++] = w * 32 + bit;
      m &= m - 1;
    }
  }
  for (int k = e0 + t; k < e1; k += kGrPlanThreads) {
    const int c = col[k];
    code[k] = (c >= row0 && c < row0 + rows)
                  ? c - row0
                  : R + rank[c >> 5] + __popc(bits[c >> 5] & ((1u << (c & 31)) - 1u));
  }
}

// The waits' failure path (gk_wait_selftest): thread 0 polls a word that
// nobody writes, through the halo's fetch, until it gives up; then every
// thread's wait has to end at the abort word.  *result: 0 if all of it went
// as designed.
__global__ void __launch_bounds__(kGrThreads) grid_wait_selftest_kernel(GridArgs a, int* result) {
  __shared__ GridRed red;
  __shared__ double dst[4 * kGrThreads];
  if (threadIdx.x == 0) red.ok = 1;
  __syncthreads();
  fetch_halo(a, red, a.words, a.seq0, a.halo_col, 1, dst, 0);
  __syncthreads();
  const bool first = red.ok == 0 && *a.abort_ == 1u && (a.st->err & kErrTimeout) != 0;
  __syncthreads();
  if (threadIdx.x == 0) {
    red.ok = 1;
    a.st->err = 0;
  }
  __syncthreads();
  const long long t0 = clock64();
  fetch_halo(a, red, a.words, a.seq0, a.halo_col, 4 * kGrThreads, dst, 0);
  const bool soon = clock64() - t0 < kMaxWaitCycles / 8;
  const bool all_soon = __syncthreads_and(soon) != 0;
  if (threadIdx.x == 0) *result = first && all_soon && red.ok == 0 && a.st->err == 0 ? 0 : 1;
}

using GrKernel = void (*)(GridArgs);

template <int PK, int SRC, bool CLUSTER>
GrKernel pick_rpt(int kind, int rpt) {
  if (kind == GK_BICGSTAB) {
    switch (rpt) {
      case 1: return bicg_grid_kernel<PK, 1, SRC, CLUSTER>;
      case 2: return bicg_grid_kernel<PK, 2, SRC, CLUSTER>;
      default: return bicg_grid_kernel<PK, 4, SRC, CLUSTER>;
    }
  }
  switch (rpt) {
    case 1: return cg_grid_kernel<PK, 1, SRC, CLUSTER>;
    case 2: return cg_grid_kernel<PK, 2, SRC, CLUSTER>;
    case 4: return cg_grid_kernel<PK, 4, SRC, CLUSTER>;
    default: return cg_grid_kernel<PK, 8, SRC, CLUSTER>;
  }
}

template <int PK, bool CLUSTER>
GrKernel pick_src(int kind, int rpt, int src) {
  if (src == SRC_STAGED) return pick_rpt<PK, SRC_STAGED, CLUSTER>(kind, rpt);
  // fewer rows a thread, or BiCGSTAB's half as many, are staged unless they are long
  if (src == SRC_SHORT && kind == GK_CG && rpt == 4) return cg_grid_kernel<PK, 4, SRC_SHORT, CLUSTER>;
  if (src == SRC_SHORT && kind == GK_CG && rpt == 8) return cg_grid_kernel<PK, 8, SRC_SHORT, CLUSTER>;
  return pick_rpt<PK, SRC_LONG, CLUSTER>(kind, rpt);
}

template <bool CLUSTER>
GrKernel pick_pk(int kind, int pk, int rpt, int src) {
  return pk == PREC_SCALAR ? pick_src<PREC_SCALAR, CLUSTER>(kind, rpt, src)
                           : pick_src<PREC_NONE, CLUSTER>(kind, rpt, src);
}

GrKernel pick(const Solver& S, int rpt, int src, bool cluster) {
  return cluster ? pick_pk<true>(S.kind, S.pk, rpt, src) : pick_pk<false>(S.kind, S.pk, rpt, src);
}

cudaLaunchConfig_t cluster_config(size_t smem, cudaStream_t s, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kGrClusterCtas, 1, 1);
  cfg.blockDim = dim3(kGrThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kGrClusterCtas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

// Dynamic shared memory a CTA may use (of 227 KB, next to the 7.7 KB of the
// reductions and the scalars): the vectors must fit, the rows of the matrix
// are staged if they do.
constexpr size_t kGrSmemMax = 216 * 1024;
static_assert(sizeof(GridRed) + sizeof(GrScalars) + kGrSmemMax <= 227 * 1024, "a CTA's shared memory");

}  // namespace

int grid_wait_selftest(bool* ok, cudaStream_t s) {
  // one array: the state, the abort word, the result, one word, 4 * 256 halo columns (all of them 0)
  struct Scratch {
    SolverState st;
    unsigned int abort_;
    int result;
    alignas(16) ulonglong2 word;
    int32_t cols[4 * kGrThreads];
  };
  Scratch* d = nullptr;
  GK_TRY_CUDA(cudaMalloc(&d, sizeof(Scratch)));
  GridArgs a = {};
  a.st = &d->st;
  a.abort_ = &d->abort_;
  a.words = &d->word;
  a.halo_col = d->cols;
  a.seq0 = 1ull << 40;
  int result = 1;
  cudaError_t e = cudaMemsetAsync(d, 0, sizeof(Scratch), s);
  if (e == cudaSuccess) {
    grid_wait_selftest_kernel<<<1, kGrThreads, 0, s>>>(a, &d->result);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&result, &d->result, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(d);
  if (e != cudaSuccess) return cuda_error(e, "gk_wait_selftest");
  *ok = result == 0;
  return GK_OK;
}

// cluster: the plan of the 16-CTA form (the caller has checked that the
// cluster form applies); else of the cooperative grid.
int grid_cg_plan(Solver* S, bool cluster) {
  S->gr_grid = 0;
  if ((S->kind != GK_CG && S->kind != GK_BICGSTAB) || S->pk == PREC_BLOCK) return GK_OK;
  const bool bi = S->kind == GK_BICGSTAB;
  const int64_t n = S->n;
  if (!cluster) {
    if (n < kGrMinRows || n > kGrMaxRows) return GK_OK;
    int coop = 0;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, S->device) != cudaSuccess || !coop) {
      cudaGetLastError();
      return GK_OK;
    }
  }
  const int G = cluster ? kGrClusterCtas : sm_count();
  const int64_t R = (n + G - 1) / G;
  int rpt = 1;
  while (static_cast<int64_t>(rpt) * kGrThreads < R) rpt *= 2;
  if (G > kGrMaxCtas || rpt > (bi ? kGrMaxRptBi : kGrMaxRptCg)) return GK_OK;
  // the CTAs' halos, entries and longest rows, then the lists
  const size_t plan_smem = 8 * static_cast<size_t>((n + 31) / 32);
  GK_TRY(set_smem(gr_halo_kernel, plan_smem));
  GK_TRY(dalloc_n(&S->gr_halo_n, static_cast<size_t>(3 * G), &S->device_bytes));
  gr_halo_kernel<<<G, kGrPlanThreads, plan_smem>>>(S->A->rowptr, S->A->col, static_cast<int>(n), static_cast<int>(R),
                                                   0, S->gr_halo_n, nullptr, nullptr);
  GK_TRY_CUDA(cudaGetLastError());
  std::vector<int32_t> info(static_cast<size_t>(3 * G));
  GK_TRY_CUDA(cudaMemcpy(info.data(), S->gr_halo_n, sizeof(int32_t) * info.size(), cudaMemcpyDeviceToHost));
  const auto most_of = [&](int k) { return *std::max_element(info.begin() + k * G, info.begin() + (k + 1) * G); };
  const int64_t cap = std::max<int32_t>(1, most_of(0)), most = most_of(1);
  const int32_t longest = most_of(2);
  if (longest > kGrMaxRowLen && !cluster) return GK_OK;  // one thread per row: no long rows
  const size_t vectors = sizeof(double) * static_cast<size_t>(R + (bi ? 4 : 2) * cap);
  // Scattered columns, whose halo does not fit: the graph form.  Measured with
  // halos gathered from global memory instead (us per iteration, graph form
  // in brackets): 65,536 rows of 50 random columns 58.9 (35.2), 130,000 of
  // 20 48.1 (33.7), 260,000 of 8 40.8 (37.7).
  if (vectors > kGrSmemMax) return GK_OK;
  const size_t staged = 12 * static_cast<size_t>(most) + 4 * static_cast<size_t>(R + 1);
  const bool stage = vectors + staged <= kGrSmemMax;
  const size_t smem = vectors + (stage ? staged : 0);
  const int src = stage ? SRC_STAGED : longest > kGrLongRow ? SRC_LONG : SRC_SHORT;
  GrKernel k = pick(*S, rpt, src, cluster);
  bool fits = set_smem(k, smem) == GK_OK;
  if (fits && cluster) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = cluster_config(smem, nullptr, attr);
    int clusters = 0;
    fits = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
           cudaOccupancyMaxActiveClusters(&clusters, k, &cfg) == cudaSuccess && clusters >= 1;
  } else if (fits) {
    int per_sm = 0;
    fits = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kGrThreads, smem) == cudaSuccess && per_sm >= 1;
  }
  if (!fits) {
    cudaGetLastError();
    return GK_OK;
  }
  const size_t n_words = static_cast<size_t>(2) * kGrCopies * kGrMaxK * G + 1, n_vec = static_cast<size_t>(bi ? 4 : 2) * n;
  const size_t n_col = static_cast<size_t>(G) * cap, n_code = static_cast<size_t>(S->A->nnz);
  GK_TRY(dalloc_async(&S->gr_plan, (n_words + n_vec) * sizeof(ulonglong2) + (n_col + n_code) * sizeof(int32_t),
                      &S->device_bytes, nullptr));
  S->gr_words = static_cast<ulonglong2*>(S->gr_plan);
  // (codes on a 16-byte boundary)
  S->gr_code = reinterpret_cast<int32_t*>(S->gr_words + n_words + n_vec);
  S->gr_halo_col = S->gr_code + n_code;
  GK_TRY_CUDA(cudaMemset(S->gr_words, 0, (n_words + n_vec) * sizeof(ulonglong2)));
  gr_halo_kernel<<<G, kGrPlanThreads, plan_smem>>>(S->A->rowptr, S->A->col, static_cast<int>(n), static_cast<int>(R),
                                                   static_cast<int>(cap), S->gr_halo_n, S->gr_halo_col, S->gr_code);
  GK_TRY_CUDA(cudaGetLastError());
  // (the caller waits for the null stream; the device's wait, which was here,
  // breaks other threads' captures)
  S->gr_grid = G;
  S->gr_rpt = rpt;
  S->gr_rows = static_cast<int>(R);
  S->gr_halo_cap = static_cast<int>(cap);
  S->gr_src = src;
  S->gr_nnz = stage ? static_cast<int>(most) : 0;
  S->gr_smem = smem;
  S->gr_epoch = 1;
  return GK_OK;
}

int grid_cg_solve(Solver* S, bool cluster, cudaStream_t s) {
  const bool bi = S->kind == GK_BICGSTAB;
  GridArgs a;
  a.rowptr = S->A->rowptr;
  a.code = S->gr_code;
  a.val = S->A->val;
  a.b = S->b;
  a.x = S->x;
  a.dinv = S->P ? S->P->dinv : nullptr;
  a.st = S->st;
  a.halo_n = S->gr_halo_n;
  a.halo_col = S->gr_halo_col;
  a.halo_cap = S->gr_halo_cap;
  const size_t n_words = static_cast<size_t>(2) * kGrCopies * kGrMaxK * S->gr_grid + 1;
  a.words = S->gr_words;
  a.abort_ = reinterpret_cast<unsigned int*>(S->gr_words + n_words - 1);
  ulonglong2* vec = S->gr_words + n_words;
  a.zw[0] = vec;
  a.zw[1] = vec + S->n;
  a.vw[0] = bi ? vec + 2 * S->n : nullptr;
  a.vw[1] = bi ? vec + 3 * S->n : nullptr;
  // every solve has its own 2^40 sequence numbers (the reductions of months),
  // so the words of earlier solves match none of this one's; after 2^24
  // solves the words are cleared and the numbers start over
  if (S->gr_epoch >> 24) {
    GK_TRY_CUDA(cudaMemsetAsync(S->gr_words, 0, (n_words + static_cast<size_t>(bi ? 4 : 2) * S->n) * sizeof(ulonglong2), s));
    S->gr_epoch = 1;
  }
  a.seq0 = S->gr_epoch << 40;
  S->gr_epoch += 1;
  a.n = static_cast<int>(S->n);
  a.rows_per_cta = S->gr_rows;
  a.stage_nnz = S->gr_nnz;
  GK_TRY_CUDA(cudaMemsetAsync(a.abort_, 0, sizeof(unsigned int), s));
  GrKernel k = pick(*S, S->gr_rpt, S->gr_src, cluster);
  if (cluster) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = cluster_config(S->gr_smem, s, attr);
    GK_TRY_CUDA(cudaLaunchKernelEx(&cfg, k, a));
  } else {
    void* args[] = {&a};
    GK_TRY_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(k), dim3(S->gr_grid), dim3(kGrThreads), args,
                                            S->gr_smem, s));
  }
  return GK_OK;
}

}  // namespace gk
