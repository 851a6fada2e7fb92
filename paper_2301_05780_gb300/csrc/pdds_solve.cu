// FP64 BiCGSTAB (van der Vorst 1992) for the PDDSparse system G u = b
// (Eq. 23), one persistent cooperative launch per call.  The paper solves
// this system on one core after assembly (Sec. 4.3, Sec. 5.2.2).
//
// What bounds it: GB300's FP64 unit (1.25 TFLOP/s: two FMAs a cycle and SM, so
// one FP64 instruction holds an SM's unit for 16 cycles however few of its
// lanes count) and, for small systems, the grid-wide dependencies.  Hence
//  - the whole recurrence is one kernel, at most one 1024-thread CTA per SM,
//    with grid barriers instead of launches:
//      p = r + beta (p - omega v)            | v = A p, (rh, v)        |
//      s = r - alpha v                       | t = A s, (t, s), (t, t) |
//      x += alpha p + omega s, r = s - omega t, (rh, r), (r, r)        |
//    (forming p and s at the gather would save two barriers, but costs three
//    and two FP64 instructions per nonzero instead of one: measured slower);
//  - a row's sum is spread over only as many lanes as coalescing needs (4 more
//    while threads are idle), since the shuffle tree's adds are FP64 instructions too; dot products
//    are taken one row per lane after the product, not on each row's lane;
//  - the recurrence's divisions run on one thread of each CTA.
// A barrier carries the dot products: each CTA leaves its partial sums before
// it arrives, and every CTA adds all of them in the same order after it, so
// that all CTAs see the same bits, decide alike, and a solve repeats exactly.
// Several problems share a launch, each on its own CTAs with its own barrier.
// A barrier's wait is bounded (CTAs that other streams' work keeps from
// starting); a problem whose wait has run out is solved again on one CTA,
// which waits for no other.
// Measured on one GB300 against six launches per iteration (one warp per row,
// host read every eight iterations): 68 us per iteration instead of 200 on
// 113,665 unknowns / 8.3e6 nonzeros (27 us of FP64 FMAs), 44 instead of 75 on
// 11,241 / 4.5e6 (FP64 unit 42 % busy); 26 on 833 / 5.1e4 either way (the
// latency of five barriers); 16 systems of 57 to 15,000 unknowns 52 -> 9 ms.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdio>
#include <mutex>
#include <string>
#include <vector>

#include "pdds.h"
#include "pdds_internal.h"

namespace pdds {

constexpr int kSolveMaxCtas = 512;   // CTAs of one problem

struct SolveScalars {
  double relres;
  int32_t converged, breakdown, iters, timeout;
  unsigned arrived;                   // barrier: arrivals so far
  int32_t pad_;
  double part[3][2 * kSolveMaxCtas];  // per phase: the CTAs' two partial sums
};

namespace {

constexpr int kThreads = 1024;

struct SolveDesc {
  const int32_t* rp;
  const int32_t* ci;
  const double* val;
  const double* b;
  double* x;
  double* work;       // r, rh, p, v, s, t: 6 n
  SolveScalars* sc;   // up to the partial sums zeroed before the launch
  int64_t n;
  double rtol;
  uint64_t wait_ns;   // bound on a barrier's wait (0: a CTA that would wait gives up at once)
  int32_t maxit, cta0, ctas, lanes;  // lanes of a warp that share a row
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The recurrence's scalars, the same in every CTA (written by its thread 0).
struct Shared {
  double a[kThreads], b[kThreads];  // the threads' partial dot products
  double sum_b[1];
  double bb, rho, rv, alpha, omega, beta, relres;
  int iters, converged, breakdown, ok;
};

// One problem's CTAs and the barrier between them.
struct Team {
  SolveScalars* sc;
  int rank, ctas;
  uint64_t wait_ns;
  unsigned target;  // arrivals that complete the next barrier

  // Thread 0: arrive and wait for the team; false when the wait ran out.
  __device__ bool meet() {
    __threadfence();  // this CTA's vectors and sums before its arrival
    atomicAdd(&sc->arrived, 1u);
    uint64_t t0 = 0;
    for (int spin = 0;; ++spin) {
      unsigned seen;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&sc->arrived) : "memory");
      if ((int)(seen - target) >= 0) break;
      if ((spin & 255) == 255 || wait_ns == 0) {
        uint64_t t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t0 == 0) t0 = t;
        if (t - t0 >= wait_ns || __ldcg(&sc->timeout) != 0) return false;
      }
    }
    __threadfence();
    return true;
  }

  __device__ bool barrier(Shared& S) {
    __syncthreads();
    if (ctas > 1) {
      if (threadIdx.x == 0) S.ok = meet();
      __syncthreads();
      target += ctas;
    }
    return S.ok != 0;
  }

  // Sums a and b over the team (set: which of the three slots; live: threads
  // of this CTA that can hold a nonzero), hands them to `fin` on thread 0.
  template <class Fin>
  __device__ bool reduce(Shared& S, int set, int live, double a, double b, Fin fin) {
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    S.a[threadIdx.x] = a;
    S.b[threadIdx.x] = b;
    __syncthreads();
    double sum = 0.0;
    if (w < 2) {  // warp 0 sums a, warp 1 b
      const double* x = w == 0 ? S.a : S.b;
      double s0 = 0.0, s1 = 0.0;
      int i = l;
      for (; i + 32 < live; i += 64) { s0 += x[i]; s1 += x[i + 32]; }
      if (i < live) s0 += x[i];
      sum = warp_sum(s0 + s1);
      if (w == 1 && l == 0) S.sum_b[0] = sum;
    }
    if (ctas > 1) {
      double* part = sc->part[set];
      if (w < 2 && l == 0) part[2 * rank + w] = sum;
      __syncthreads();
      if (threadIdx.x == 0) S.ok = meet();
      __syncthreads();
      target += ctas;
      if (w < 2) {
        sum = 0.0;
        for (int i = l; i < ctas; i += 32) sum += __ldcg(part + 2 * i + w);
        sum = warp_sum(sum);
        if (w == 1 && l == 0) S.sum_b[0] = sum;
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) fin(sum, S.sum_b[0]);
    __syncthreads();
    return S.ok != 0;
  }
};

// The rows of a CTA: blocks of kRun rows, dealt to the team's CTAs in turn, so
// that every CTA gets its share of long (interior) and short rows, and a warp's
// vector accesses still come in 64-byte runs.
constexpr int kRun = 8;
__device__ __forceinline__ int64_t team_row(const Team& M, int64_t j) {
  return ((j / kRun) * M.ctas + M.rank) * kRun + j % kRun;
}
__device__ __forceinline__ int64_t team_rows(const Team& M, int64_t n) {
  const int64_t blocks = (n + kRun - 1) / kRun;
  return blocks > M.rank ? (blocks - M.rank + M.ctas - 1) / M.ctas * kRun : 0;
}

// y = A x on the CTA's rows, T lanes per row.
template <int T>
__device__ __forceinline__ void spmv(const SolveDesc& D, const Team& M, int64_t mine,
                                     const double* x, double* y) {
  const int sub = threadIdx.x & (T - 1);
  // every lane of a warp runs the same number of rounds (the shuffles below)
  for (int64_t j0 = 0; j0 < mine; j0 += kThreads / T) {
    const int64_t j = j0 + threadIdx.x / T;
    const int64_t row = team_row(M, j);
    const bool live = j < mine && row < D.n;
    double s = 0.0;
    if (live) {
      const int end = __ldg(D.rp + row + 1);
#pragma unroll 4
      for (int q = __ldg(D.rp + row) + sub; q < end; q += T)
        s = fma(__ldg(D.val + q), x[__ldg(D.ci + q)], s);
    }
#pragma unroll
    for (int o = T / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (sub == 0 && live) y[row] = s;
  }
}

template <int T>
__device__ void bicgstab(const SolveDesc& D, Team M, Shared& S) {
  const int64_t n = D.n;
  double* const r = D.work;
  double* const rh = D.work + n;
  double* const p = D.work + 2 * n;
  double* const v = D.work + 3 * n;
  double* const s = D.work + 4 * n;
  double* const t = D.work + 5 * n;
  double* const x = D.x;
  // this CTA's rows, one per thread
  const int64_t mine = team_rows(M, n);
  const int live = (int)(mine < kThreads ? mine : kThreads);
  auto each_row = [&](auto f) {
    for (int64_t j = threadIdx.x; j < mine; j += kThreads) {
      const int64_t i = team_row(M, j);
      if (i < n) f(i);
    }
  };
  if (threadIdx.x == 0) S.ok = 1;
  double d0 = 0.0, d1 = 0.0;
  each_row([&](int64_t i) {
    const double bi = D.b[i];
    x[i] = 0.0; r[i] = bi; rh[i] = bi; p[i] = 0.0; v[i] = 0.0;
    d0 += bi * bi;
  });
  bool ok = M.reduce(S, 0, live, d0, 0.0, [&](double bb, double) {
    S.bb = S.rho = bb;
    S.omega = 1.0;
    S.beta = bb;  // (rho / 1) (1 / 1)
    S.relres = bb > 0 ? 1.0 : 0.0;
    S.iters = S.breakdown = 0;
    S.converged = bb == 0.0;
  });
  while (ok && !S.converged && !S.breakdown && S.iters < D.maxit) {
    const double beta = S.beta, om = S.omega;
    each_row([&](int64_t i) { p[i] = r[i] + beta * (p[i] - om * v[i]); });
    if (!(ok = M.barrier(S))) break;
    spmv<T>(D, M, mine, p, v);
    __syncthreads();
    d0 = 0.0;
    each_row([&](int64_t i) { d0 += rh[i] * v[i]; });
    ok = M.reduce(S, 1, live, d0, 0.0, [&](double rv, double) {
      S.rv = rv;
      S.alpha = S.rho / rv;
    });
    if (!ok) break;
    const double alpha = S.alpha;
    each_row([&](int64_t i) { s[i] = r[i] - alpha * v[i]; });
    if (!(ok = M.barrier(S))) break;
    spmv<T>(D, M, mine, s, t);
    __syncthreads();
    d0 = d1 = 0.0;
    each_row([&](int64_t i) {
      const double ti = t[i];
      d0 += ti * s[i];
      d1 += ti * ti;
    });
    ok = M.reduce(S, 2, live, d0, d1,
                  [&](double ts, double tt) { S.omega = tt > 0.0 ? ts / tt : 0.0; });
    if (!ok) break;
    const double omega = S.omega;
    d0 = d1 = 0.0;
    each_row([&](int64_t i) {
      const double si = s[i];
      x[i] += alpha * p[i] + omega * si;
      const double ri = si - omega * t[i];
      r[i] = ri;
      d0 += rh[i] * ri;
      d1 += ri * ri;
    });
    ok = M.reduce(S, 0, live, d0, d1, [&](double rr, double rr2) {
      S.iters += 1;
      S.converged = rr2 <= D.rtol * D.rtol * S.bb;
      S.relres = rr2;  // its root and quotient are taken at the end
      if (!S.converged) {
        // breakdown codes: 1 (rh, v) = 0, 2 omega = 0, 3 (rh, r) = 0, 4 residual not finite
        if (!(S.rv != 0.0)) S.breakdown = 1;
        else if (!(S.omega != 0.0)) S.breakdown = 2;
        else if (!(rr != 0.0)) S.breakdown = 3;
        else if (!(rr2 < 1e200 && S.bb > 1e-100) && !(sqrt(rr2 / S.bb) <= 1e300)) S.breakdown = 4;
      }
      S.beta = (rr / S.rho) * (S.alpha / S.omega);
      S.rho = rr;
    });
  }
  if (threadIdx.x == 0) {
    if (M.rank == 0) {
      D.sc->relres = S.iters > 0 ? sqrt(S.relres / S.bb) : S.relres;
      D.sc->converged = S.converged;
      D.sc->breakdown = S.breakdown;
      D.sc->iters = S.iters;
    }
    if (!ok) atomicExch(&D.sc->timeout, 1);
  }
}

constexpr int kInline = 32;  // problems of one launch (their descriptors are its parameter)
struct SolveParams {
  SolveDesc inl[kInline];
  int count;
};

__global__ void __launch_bounds__(kThreads, 1) k_bicgstab(const __grid_constant__ SolveParams P) {
  int i = 0;
  while (i + 1 < P.count && (int)blockIdx.x >= P.inl[i + 1].cta0) ++i;
  const SolveDesc& D = P.inl[i];
  __shared__ Shared S;
  const Team M{D.sc, (int)blockIdx.x - D.cta0, D.ctas, D.wait_ns, (unsigned)D.ctas};
  switch (D.lanes) {
    case 4: bicgstab<4>(D, M, S); break;
    case 8: bicgstab<8>(D, M, S); break;
    case 16: bicgstab<16>(D, M, S); break;
    default: bicgstab<32>(D, M, S); break;
  }
}

}  // namespace

size_t bicgstab_work_doubles(int64_t n) { return (size_t)6 * (size_t)n; }
size_t bicgstab_scalars_bytes() { return sizeof(SolveScalars); }

namespace {

// One launch (for up to kInline problems) that solves jobs[which[0 .. count)] on at
// most `most` CTAs, or on more if each problem gets just one; outcomes to
// heads[which[..]] once the stream has been synchronized with.  `again`: after
// a run of the same jobs, whose b may have been overwritten (u may be b's own
// memory) and is taken from where that run kept it.
struct SolveHead { double relres; int32_t converged, breakdown, iters, timeout; };

cudaError_t launch_solves(const SolveJob* jobs, const std::vector<int>& which, int most, bool again,
                          double rtol, int32_t maxit, uint64_t wait_ns, SolveHead* heads,
                          int* launches, cudaStream_t st) {
  cudaError_t e;
  const int count = (int)which.size();
  for (int base = 0; base < count;) {
    SolveParams P{};
    // A context given twice has one scratch: its second solve goes into the
    // next launch.
    auto in_launch = [&](const SolveScalars* sc) {
      for (int i = 0; i < P.count; ++i)
        if (jobs[which[base + i]].sc == sc) return true;
      return false;
    };
    while (P.count < kInline && base + P.count < count && !in_launch(jobs[which[base + P.count]].sc))
      ++P.count;
    int64_t total = 0;
    for (int i = 0; i < P.count; ++i) total += std::max<int64_t>(jobs[which[base + i]].nnz, 1);
    for (int limit = most;; limit /= 2) {
      int ctas = 0;
      for (int i = 0; i < P.count; ++i) {
        const SolveJob& J = jobs[which[base + i]];
        SolveDesc& D = P.inl[i];
        // (the recurrence's shadow residual is b)
        D = SolveDesc{J.rp, J.ci, J.val, again ? J.work + J.n : J.b, J.x, J.work, J.sc, J.n, rtol,
                      wait_ns, maxit, 0, 0, 0};
        // One CTA up to 12 nonzeros a thread (its barriers stay inside the SM),
        // else one per two nonzeros a thread, at most its share of the SMs.
        const int64_t want = J.nnz <= 12 * kThreads ? 1 : (J.nnz + 2 * kThreads - 1) / (2 * kThreads);
        const int64_t share = std::max<int64_t>(1, (int64_t)(limit - P.count + 1) * J.nnz / total);
        D.cta0 = ctas;
        D.ctas = (int)std::max<int64_t>(1, std::min<int64_t>({want, share, (int64_t)kSolveMaxCtas}));
        // Lanes per row: as many as keep the CTA's threads busy in one round,
        // from 4 (32-byte runs of a row) to about one per nonzero.
        const int64_t mine = (J.n + D.ctas - 1) / D.ctas, per_row = J.nnz / std::max<int64_t>(J.n, 1);
        D.lanes = 4;
        while (D.lanes < 32 && 2 * D.lanes * mine <= kThreads + kThreads / 8 && D.lanes < per_row)
          D.lanes *= 2;
        ctas += D.ctas;
      }
      for (int i = 0; i < P.count; ++i)
        if ((e = cudaMemsetAsync(P.inl[i].sc, 0, offsetof(SolveScalars, part), st)) != cudaSuccess)
          return e;
      void* args[] = {&P};
      // one CTA per problem: none waits for another, an ordinary launch will do
      const void* fn = reinterpret_cast<const void*>(k_bicgstab);
      e = ctas == P.count ? cudaLaunchKernel(fn, dim3(ctas), dim3(kThreads), args, 0, st)
                          : cudaLaunchCooperativeKernel(fn, dim3(ctas), dim3(kThreads), args, 0, st);
      // fewer SMs than the device has (a partition), or no cooperative
      // launches: smaller teams, in the end of one CTA each
      if ((e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) && limit > 1) {
        (void)cudaGetLastError();
        continue;
      }
      if (e != cudaSuccess) return e;
      break;
    }
    if (launches) *launches += 1;
    for (int i = 0; i < P.count; ++i)
      if ((e = cudaMemcpyAsync(&heads[which[base + i]], P.inl[i].sc, sizeof(SolveHead),
                               cudaMemcpyDeviceToHost, st)) != cudaSuccess)
        return e;
    base += P.count;
  }
  return cudaStreamSynchronize(st);
}

}  // namespace

cudaError_t bicgstab_batch(SolveJob* jobs, int count, double rtol, int32_t maxit, int* launches,
                           cudaStream_t st, uint64_t wait_ns) {
  int dev = 0, sms = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if (launches) *launches = 0;
  std::vector<SolveHead> h(count);
  std::vector<int> which(count);
  for (int i = 0; i < count; ++i) which[i] = i;
  if ((e = launch_solves(jobs, which, sms, false, rtol, maxit, wait_ns, h.data(), launches, st)) !=
      cudaSuccess)
    return e;
  which.clear();
  for (int i = 0; i < count; ++i)
    if (h[i].timeout) which.push_back(i);
  if (!which.empty() && (e = launch_solves(jobs, which, 1, true, rtol, maxit, wait_ns, h.data(),
                                           launches, st)) != cudaSuccess)
    return e;
  for (int i = 0; i < count; ++i) {
    jobs[i].iters = h[i].iters;
    jobs[i].relres = h[i].relres;
    jobs[i].converged = h[i].converged ? 1 : -h[i].breakdown;
  }
  return cudaSuccess;
}

cudaError_t bicgstab_device(const int32_t* rp, const int32_t* ci, const double* val,
                            const double* b, double* x, int64_t n, int64_t nnz, double* work,
                            SolveScalars* sc, double rtol, int32_t maxit, int32_t* iters,
                            double* relres, int* converged, int* launches, cudaStream_t st,
                            uint64_t wait_ns) {
  SolveJob J{rp, ci, val, b, x, n, nnz, work, sc, 0, 0.0, 0};
  const cudaError_t e = bicgstab_batch(&J, 1, rtol, maxit, launches, st, wait_ns);
  if (e != cudaSuccess) return e;
  if (iters) *iters = J.iters;
  if (relres) *relres = J.relres;
  if (converged) *converged = J.converged;
  return cudaSuccess;
}

}  // namespace pdds

// ===========================================================================
// Allocation-free solve.
//
// Some callers of this library cannot allocate device memory: applications
// that own all device memory through their own pool or arena under a fixed
// budget (a library-side cudaMalloc would bypass their accounting, or fail),
// and latency-critical code where the implicit device synchronization of
// cudaMalloc/cudaFree is not acceptable.  pdds_solve_noalloc serves them: it
// runs the same BiCGSTAB kernels as pdds_solve, but its scratch -- six work
// vectors and the recurrence scalars -- lives in the file-scope device array
// below, which every GPU that loads this library holds until the process
// exits (6.3 MB).  The caller still passes G, b and u.
// ===========================================================================
namespace pdds {
namespace {

constexpr int64_t kNoAllocMaxN = 131072;           // largest system size served
constexpr int64_t kNoAllocScalarSlots = 4096;      // >= sizeof(SolveScalars) / 8
static_assert(sizeof(pdds::SolveScalars) <= kNoAllocScalarSlots * sizeof(double), "scratch");

static __device__ __align__(256) double g_noalloc_scratch[6 * kNoAllocMaxN + kNoAllocScalarSlots];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
double* g_noalloc_ptr[kMaxDevices] = {nullptr};

}  // namespace
}  // namespace pdds

extern "C" pdds_status pdds_internal_solve_noalloc(const pdds_csr* G, const double* b, double* u,
                                                   double rtol, int32_t maxit, int32_t* iters,
                                                   void* cuda_stream, uint64_t wait_ns) {
  using namespace pdds;
  if (!G || !b || !u || !G->row_ptr || !G->col || !G->val) {
    set_global_error("solve_noalloc: NULL matrix/vector");
    return PDDS_EINVAL;
  }
  if (G->n > kNoAllocMaxN) {
    char buf[200];
    std::snprintf(buf, sizeof buf,
                  "solve_noalloc: n = %lld exceeds the static scratch limit of %lld unknowns; "
                  "use pdds_solve", (long long)G->n, (long long)kNoAllocMaxN);
    set_global_error(buf);
    return PDDS_EINVAL;
  }
  if (G->n < 1 || G->nnz < G->n) {
    set_global_error("solve_noalloc: need n >= 1 and nnz >= n");
    return PDDS_EINVAL;
  }
  if (!(rtol > 0) || maxit < 1) {
    set_global_error("solve_noalloc: need rtol > 0, maxit >= 1");
    return PDDS_EINVAL;
  }
  (void)cudaGetLastError();
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    set_global_error(std::string("solve_noalloc: cudaGetDevice: ") + cudaGetErrorString(e));
    return PDDS_ECUDA;
  }
  double* scratch = nullptr;
  {
    // First call on this device (the current one): look up the array's device
    // address.  Host code cannot use g_noalloc_scratch's name as a pointer.
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
      void* p = nullptr;
      e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
      if (e != cudaSuccess || !p) {
        set_global_error(std::string("solve_noalloc: cudaGetSymbolAddress: ") +
                         cudaGetErrorString(e));
        return PDDS_ECUDA;
      }
      g_noalloc_ptr[dev] = static_cast<double*>(p);
    }
    scratch = g_noalloc_ptr[dev];
  }
  auto* sc = reinterpret_cast<SolveScalars*>(scratch + 6 * kNoAllocMaxN);
  int32_t it = 0;
  double rel = 0;
  int conv = 0, nl = 0;
  // bicgstab_device zeroes the scalars and initialises every work vector it
  // reads, so the previous call's contents never leak into this one.
  e = bicgstab_device(G->row_ptr, G->col, G->val, b, u, G->n, G->nnz, scratch, sc, rtol, maxit, &it, &rel,
                      &conv, &nl, (cudaStream_t)cuda_stream, wait_ns);
  if (e != cudaSuccess) {
    set_global_error(std::string("solve_noalloc: ") + cudaGetErrorString(e));
    return PDDS_ECUDA;
  }
  if (iters) *iters = it;
  if (conv != 1) {
    char buf[200];
    std::snprintf(buf, sizeof buf,
                  "solve_noalloc: no convergence after %d iterations (relres %.3e)%s", it, rel,
                  bicgstab_stop_reason(conv));
    set_global_error(buf);
    return PDDS_ENOCONV;
  }
  return PDDS_OK;
}

extern "C" pdds_status pdds_solve_noalloc(const pdds_csr* G, const double* b, double* u,
                                          double rtol, int32_t maxit, int32_t* iters,
                                          void* cuda_stream) {
  return pdds_internal_solve_noalloc(G, b, u, rtol, maxit, iters, cuda_stream, pdds::kSolveWaitNs);
}
