// One preconditioned CG step per right-hand side (Eq. stern on the shifted
// operator): a thread-block cluster per RHS.
//
// The step reads p, A p, r, x and K once, in 16-byte loads that a thread keeps
// in registers, and writes x, r and p: 7 vector passes.  Its two reductions are
// per-warp sums in the vectors' precision, summed in FP64 over the warps and,
// through distributed shared memory, over the cluster.
//
// Why clusters: with a handful of RHS a step's time is the latency of one
// block walking one vector.  Against the streaming block per RHS this replaced:
// three RHS of 64^3 one CG application 13.4 -> 9.9 ms, eight of 24^3 2.19 -> 1.61 ms.
// More than CG_TAIL_MAX RHS are streamed (k_cg_stream below).
//
// Two forms for few RHS: PROJ adds the projection term sum_w sigma_w |w><w| p
// to A p first (the RHS's cluster has p in registers, the states come from L2),
// and with 'tail' the last cluster to finish compacts the active list and takes
// the loop decision, so that a CG step is the transform and this kernel.
#include <cooperative_groups.h>

#include <algorithm>

#include "linalg.cuh"
#include "profile.cuh"

namespace cg = cooperative_groups;

namespace pdep {
namespace {

template <typename R>
__device__ __forceinline__ R warp_sum(R v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <typename R>
struct Vec;
template <>
struct Vec<float> {
  static constexpr int n = 4;
  static __device__ __forceinline__ void ld(const float* p, float (&v)[4]) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x;
    v[1] = q.y;
    v[2] = q.z;
    v[3] = q.w;
  }
  static __device__ __forceinline__ void st(float* p, const float (&v)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  }
};
template <>
struct Vec<double> {
  static constexpr int n = 2;
  static __device__ __forceinline__ void ld(const double* p, double (&v)[2]) {
    const double2 q = *reinterpret_cast<const double2*>(p);
    v[0] = q.x;
    v[1] = q.y;
  }
  static __device__ __forceinline__ void st(double* p, const double (&v)[2]) {
    *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
  }
};

// per-warp sums of a and b (in R) into FP64 block totals at out (thread 0
// writes; the caller synchronises)
template <typename R, int T>
__device__ __forceinline__ void block_totals(R a, R b, double (&sh)[2][T / 32], double2* out) {
  a = warp_sum(a);
  b = warp_sum(b);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) {
    sh[0][w] = (double)a;
    sh[1][w] = (double)b;
  }
  __syncthreads();
  if (w == 0) {
    double x = l < T / 32 ? sh[0][l] : 0.0, y = l < T / 32 ? sh[1][l] : 0.0;
#pragma unroll
    for (int o = T / 64; o > 0; o >>= 1) {
      x += __shfl_xor_sync(0xffffffffu, x, o);
      y += __shfl_xor_sync(0xffffffffu, y, o);
    }
    if (l == 0) *out = make_double2(x, y);
  }
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// V 16-byte vectors per thread: cluster * T * V vectors cover n_pw; the blocks
// of a cluster take interleaved stripes of T vectors.
template <typename R, int T, int V, bool PROJ>
__global__ void __launch_bounds__(T)
    k_cg_step(CgArgs<R> a, const int* __restrict__ list, CgProj<R> pj, CgTail tail) {
  constexpr int E = Vec<R>::n;
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int slot = blockIdx.x / C;
  const int listed = a.list_count ? *a.list_count : (int)gridDim.x / C;
  if (slot >= listed) return;  // the whole cluster
  const int i = list ? list[slot] : slot;
  __shared__ double sh[2][T / 32];
  __shared__ double2 tot[2];
  __shared__ R coef[2];  // alpha, then beta
  __shared__ int flag;   // 1: breakdown, 2: converged
  __shared__ int last;
  const CgScal s = a.sc[i];
  const int tid = threadIdx.x;
  if (s.active) {
    const long long o = (long long)i * a.ld;
    const R* K = a.kprec + (long long)(i % a.n_occ) * a.ld;
    R pv[V][E], av[V][E], rv[V][E];
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const int j = ((v * C + rank) * T + tid) * E;
      if (j < a.n_pw) {
        Vec<R>::ld(a.p + o + j, pv[v]);
        Vec<R>::ld(a.ap + o + j, av[v]);
        Vec<R>::ld(a.r + o + j, rv[v]);
#pragma unroll
        for (int e = 0; e < E; ++e)
          if (j + e >= a.n_pw) pv[v][e] = av[v][e] = rv[v][e] = R(0);
      } else {
#pragma unroll
        for (int e = 0; e < E; ++e) pv[v][e] = av[v][e] = rv[v][e] = R(0);
      }
    }
    if constexpr (PROJ) {
      // S_w = sigma_w <w|p> over the cluster, then A p += sum_w S_w |w>.  The
      // block's stripe of p goes through shared memory and each warp takes whole
      // states of it: a warp sum per state and block instead of one per warp
      // (in FP64 its five additions take 320 clocks)
      __shared__ __align__(16) R stripe[T * V * E];
      __shared__ R S[CG_PROJ_MAX], sums[CG_PROJ_MAX];
#pragma unroll
      for (int v = 0; v < V; ++v) Vec<R>::st(stripe + (v * T + tid) * E, pv[v]);
      __syncthreads();
      for (int w = tid >> 5; w < pj.n; w += T / 32) {
        const R* P = pj.states + (long long)w * a.ld;
        R d = R(0);
#pragma unroll 4
        for (int q = tid & 31; q < T * V; q += 32) {
          const int j = ((q / T * C + rank) * T + q % T) * E;
          if (j < a.n_pw) {
            R x[E], y[E];
            Vec<R>::ld(P + j, x);
            Vec<R>::ld(stripe + q * E, y);
#pragma unroll
            for (int e = 0; e < E; ++e) d += x[e] * y[e];
          }
        }
        d = warp_sum(d);
        if ((tid & 31) == 0) sums[w] = d;
      }
      if (C > 1)
        cl.sync();
      else
        __syncthreads();
      for (int w = tid; w < pj.n; w += T) {
        R t = R(0);
        for (int c = 0; c < C; ++c) t += cl.map_shared_rank(sums, c)[w];
        S[w] = pj.sigma[w] * t;
      }
      __syncthreads();
#pragma unroll 4
      for (int w = 0; w < pj.n; ++w) {
        const R* P = pj.states + (long long)w * a.ld;
        const R f = S[w];
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const int j = ((v * C + rank) * T + tid) * E;
          if (j < a.n_pw) {
            R q[E];
            Vec<R>::ld(P + j, q);
#pragma unroll
            for (int e = 0; e < E; ++e)
              if (j + e < a.n_pw) av[v][e] += q[e] * f;
          }
        }
      }
    }
    R pap = R(0);
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
      for (int e = 0; e < E; ++e) pap += pv[v][e] * av[v][e];
    block_totals<R, T>(pap, R(0), sh, &tot[0]);
    if (C > 1) cl.sync();
    if (tid == 0) {
      double t = 0.0;
      for (int c = 0; c < C; ++c) t += cl.map_shared_rank(tot, c)[0].x;
      const double al = s.rz / t;
      flag = (!(t > 0.0) || !isfinite(al)) ? 1 : 0;
      coef[0] = (R)al;
      if (flag && rank == 0) {
        atomicOr(a.status, isfinite(t) ? (unsigned)DEV_BREAKDOWN : (unsigned)DEV_NONFINITE);
        a.sc[i].active = 0;
      }
    }
    __syncthreads();
    if (!flag) {  // the same in every block: each sums the same totals in order
      const R alpha = coef[0];
      R rr = R(0), rkr = R(0);
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int j = ((v * C + rank) * T + tid) * E;
        if (j < a.n_pw) {
          R xv[E], kv[E];
          Vec<R>::ld(a.x + o + j, xv);
          Vec<R>::ld(K + j, kv);
#pragma unroll
          for (int e = 0; e < E; ++e) {
            const bool in = j + e < a.n_pw;
            xv[e] = in ? xv[e] + alpha * pv[v][e] : R(0);
            const R r = rv[v][e] - alpha * av[v][e];
            rv[v][e] = r;
            rr += r * r;
            av[v][e] = in ? kv[e] * r : R(0);  // K r, A p is no longer needed
            rkr += av[v][e] * r;
          }
          Vec<R>::st(a.x + o + j, xv);
          Vec<R>::st(a.r + o + j, rv[v]);
        }
      }
      block_totals<R, T>(rr, rkr, sh, &tot[1]);
      if (C > 1) cl.sync();
      if (tid == 0) {
        double tr = 0.0, tk = 0.0;
        for (int c = 0; c < C; ++c) {
          const double2 q = cl.map_shared_rank(tot, c)[1];
          tr += q.x;
          tk += q.y;
        }
        const double rn = sqrt(tr);
        const bool done = rn <= (a.tolv ? a.tolv[i] : a.tol) * s.bnorm;
        flag = done ? 2 : 0;
        coef[1] = (R)(tk / s.rz);
        if (rank == 0) {
          CgScal n = s;
          n.iters = s.iters + 1;
          n.rnorm = rn;
          n.rz = tk;
          n.active = done ? 0 : 1;
          if (!isfinite(rn)) {
            n.active = 0;
            atomicOr(a.status, (unsigned)DEV_NONFINITE);
          }
          a.sc[i] = n;
          if (n.active && !tail.on) atomicAdd(a.n_active, 1);
        }
      }
      __syncthreads();
      if (flag != 2) {
        const R beta = coef[1];
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const int j = ((v * C + rank) * T + tid) * E;
          if (j < a.n_pw) {
#pragma unroll
            for (int e = 0; e < E; ++e) pv[v][e] = av[v][e] + beta * pv[v][e];
            Vec<R>::st(a.p + o + j, pv[v]);
          }
        }
      }
    }
    if (C > 1) cl.sync();  // no block leaves while another reads its totals
  }
  if (!tail.on || rank != 0) return;
  // loop control by the last cluster of the step
  if (tid == 0) {
    __threadfence();
    last = atomicAdd(tail.ticket, 1) == listed - 1 ? 1 : 0;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  // ordered compaction of the active RHS (n <= CG_TAIL_MAX)
  constexpr int PER = CG_TAIL_MAX / T;
  __shared__ int warp_count[T / 32];
  int act[PER], mine = 0;
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int q = tid * PER + k;
    act[k] = q < a.n_rhs ? __ldcg(&a.sc[q].active) != 0 : 0;
    mine += act[k];
  }
  int pre = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, pre, d);
    if ((tid & 31) >= d) pre += u;
  }
  if ((tid & 31) == 31) warp_count[tid >> 5] = pre;
  __syncthreads();
  int off = pre - mine, total = 0;
#pragma unroll
  for (int w = 0; w < T / 32; ++w) {
    if (w < (tid >> 5)) off += warp_count[w];
    total += warp_count[w];
  }
#pragma unroll
  for (int k = 0; k < PER; ++k)
    if (act[k]) tail.list[off++] = tid * PER + k;
  if (tid == 0) {
    CgLoopState* ls = tail.loop;
    *tail.ticket = 0;
    ls->active = total;
    const int it = ls->iter + 1;
    ls->iter = it;
    ls->launches += tail.launches;
    bool go = total > 0 && it < tail.max_iter;
    if (go && tail.budget_ns > 0 && global_ns() - ls->t0 > tail.budget_ns) {
      go = false;
      atomicOr(a.status, (unsigned)DEV_TIMEOUT);
    }
    ls->listed = go ? total : 0;  // a further step of the same graph pass is empty
    ls->go = go ? 1 : 0;
    if (tail.has_handle) cudaGraphSetConditional(tail.handle, go ? 1u : 0u);
  }
}

// --- many RHS -----------------------------------------------------------------
// One block per RHS leaves the memory idle while the block reduces, and what its
// registers hold in flight is too little to begin with (8192 RHS of 6859 FP32 at
// 2.8 TB/s).  Here persistent blocks stream the RHS: p, A p, r and x of the next
// two come by bulk copies into two shared-memory stages while one is worked on,
// some 110 KB in flight per SM whatever the row length (short rows: several
// blocks per SM).  K comes from L2, outputs go from registers to memory.  58 steps
// of up to 8192 RHS of 6859 FP32: 20.5 -> 10.8 ms (5.2 TB/s); 41 of up to 1408
// RHS of 1935: 0.95 -> 0.66 ms.
constexpr int CG_STREAM_V = 4;
constexpr size_t CG_STREAM_SMEM = 224 * 1024;
constexpr long long CG_WAIT_CYCLES = 2000000000ll;  // about a second

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
// bounded wait for the phase of the given parity; false when it ran out
__device__ __forceinline__ bool stage_wait(unsigned long long* bar, uint32_t parity) {
  const long long t0 = clock64();
  for (;;) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    if (done) return true;
    if (clock64() - t0 > CG_WAIT_CYCLES) return false;
  }
}

// TIMED: the form inside graphs captured while profiling
template <typename R, int T, bool TIMED>
__global__ void __launch_bounds__(T)
    k_cg_stream(CgArgs<R> a, const int* __restrict__ list, int rowb, DevTimer* timer) {
  constexpr int E = Vec<R>::n, V = CG_STREAM_V;
  extern __shared__ __align__(128) unsigned char stages[];
  __shared__ __align__(8) unsigned long long full[2];
  __shared__ double sh[2][T / 32];
  __shared__ double2 tot[2];
  __shared__ R coef[2];
  __shared__ int flag, dead;
  const int tid = threadIdx.x, G = gridDim.x;
  const int listed = a.list_count ? *a.list_count : a.n_listed;
  int k = blockIdx.x;
  if (k >= listed) return;
  if (TIMED && k == 0 && tid == 0) dev_timer_first(timer);
  auto rhs = [&](int q) { return q < listed ? (list ? list[q] : q) : -1; };
  // by one thread: the four rows of RHS i into a stage
  auto issue = [&](int st, int i) {
    const R* src[4] = {a.p, a.ap, a.r, a.x};
    const uint32_t bar = smem_addr(&full[st]);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(4 * rowb)
                 : "memory");
#pragma unroll
    for (int q = 0; q < 4; ++q)
      asm volatile(
          "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
              smem_addr(stages + (st * 4 + q) * (size_t)rowb)),
          "l"(src[q] + (long long)i * a.ld), "r"(rowb), "r"(bar)
          : "memory");
  };
  const bool feeder = tid == 32;
  int i0 = rhs(k), i1 = rhs(k + G);
  if (feeder) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&full[0])) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&full[1])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    dead = 0;
    issue(0, i0);
    if (i1 >= 0) issue(1, i1);
  }
  __syncthreads();
  int it = 0;
#pragma unroll 1
  for (; i0 >= 0; k += G, ++it) {
    const int st = it & 1, i = i0;
    const CgScal s = a.sc[i];
    const int i2 = rhs(k + 2 * G);
    const R* K = a.kprec + (long long)(i % a.n_occ) * a.ld;
    R pv[V][E], av[V][E], rv[V][E], xv[V][E], kv[V][E];
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const int j = (v * T + tid) * E;
#pragma unroll
      for (int e = 0; e < E; ++e) kv[v][e] = R(0);
      if (j < a.n_pw) Vec<R>::ld(K + j, kv[v]);
    }
    if (!stage_wait(&full[st], (it >> 1) & 1)) {
      dead = 1;
      atomicOr(a.status, (unsigned)DEV_TIMEOUT);
    }
    const R* row = reinterpret_cast<const R*>(stages + st * 4 * (size_t)rowb);
    const int rn_ = rowb / (int)sizeof(R);
    R pap = R(0);
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const int j = (v * T + tid) * E;
      if (j < a.n_pw) {
        Vec<R>::ld(row + j, pv[v]);
        Vec<R>::ld(row + rn_ + j, av[v]);
        Vec<R>::ld(row + 2 * rn_ + j, rv[v]);
        Vec<R>::ld(row + 3 * rn_ + j, xv[v]);
      }
#pragma unroll
      for (int e = 0; e < E; ++e)
        if (j + e >= a.n_pw) pv[v][e] = av[v][e] = rv[v][e] = xv[v][e] = kv[v][e] = R(0);
#pragma unroll
      for (int e = 0; e < E; ++e) pap += pv[v][e] * av[v][e];
    }
    block_totals<R, T>(pap, R(0), sh, &tot[0]);  // its barrier: the stage has been read
    if (feeder && i2 >= 0 && !dead) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      issue(st, i2);
    }
    if (tid == 0) {
      const double t = tot[0].x, al = s.rz / t;
      flag = !s.active || dead ? 3 : (!(t > 0.0) || !isfinite(al)) ? 1 : 0;
      coef[0] = (R)al;
      if (flag == 1) {
        atomicOr(a.status, isfinite(t) ? (unsigned)DEV_BREAKDOWN : (unsigned)DEV_NONFINITE);
        a.sc[i].active = 0;
      }
    }
    __syncthreads();
    if (dead) break;
    if (!flag) {
      const R alpha = coef[0];
      const long long o = (long long)i * a.ld;
      R rr = R(0), rkr = R(0);
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int j = (v * T + tid) * E;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          xv[v][e] += alpha * pv[v][e];
          const R r = rv[v][e] - alpha * av[v][e];
          rv[v][e] = r;
          rr += r * r;
          av[v][e] = kv[v][e] * r;  // K r, A p is no longer needed
          rkr += av[v][e] * r;
        }
        if (j < a.n_pw) {
          Vec<R>::st(a.x + o + j, xv[v]);
          Vec<R>::st(a.r + o + j, rv[v]);
        }
      }
      block_totals<R, T>(rr, rkr, sh, &tot[1]);
      if (tid == 0) {
        const double2 q = tot[1];
        const double rn = sqrt(q.x);
        const bool done = rn <= (a.tolv ? a.tolv[i] : a.tol) * s.bnorm;
        flag = done ? 2 : 0;
        coef[1] = (R)(q.y / s.rz);
        CgScal n = s;
        n.iters = s.iters + 1;
        n.rnorm = rn;
        n.rz = q.y;
        n.active = done ? 0 : 1;
        if (!isfinite(rn)) {
          n.active = 0;
          atomicOr(a.status, (unsigned)DEV_NONFINITE);
        }
        a.sc[i] = n;
        if (n.active) atomicAdd(a.n_active, 1);
      }
      __syncthreads();
      if (flag != 2) {
        const R beta = coef[1];
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const int j = (v * T + tid) * E;
#pragma unroll
          for (int e = 0; e < E; ++e) pv[v][e] = av[v][e] + beta * pv[v][e];
          if (j < a.n_pw) Vec<R>::st(a.p + o + j, pv[v]);
        }
      }
    }
    i0 = i1;
    i1 = i2;
  }
  if (dead && feeder) {
    // a wait ran out: the other stage's copies end before the block leaves
    const int nx = it + 1;
    if (i1 >= 0) stage_wait(&full[nx & 1], (nx >> 1) & 1);
    stage_wait(&full[it & 1], (it >> 1) & 1);
  }
  if (TIMED && tid == 0)
    dev_timer_done(timer, min(listed, G), blockIdx.x == 0, 12.0 * listed * (double)a.n_pw,
                   7.0 * listed * (double)a.n_pw * sizeof(R));
}

template <typename R, int T, bool TIMED>
cudaError_t launch_stream_form(const CgArgs<R>& a, const int* list, int nb, int rowb, DevTimer* timer,
                               cudaStream_t st) {
  auto kern = k_cg_stream<R, T, TIMED>;
  static OncePerDevice limit;  // per instantiation
  if (const cudaError_t e = raise_smem_limit(limit, kern, (int)CG_STREAM_SMEM)) return e;
  const size_t smem = 8 * (size_t)rowb;
  static const int sms = [] {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 152;
  }();
  int per = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, T, smem);
  if (e != cudaSuccess) return e;
  kern<<<std::min(nb, std::max(per, 1) * sms), T, smem, st>>>(a, list, rowb, timer);
  return cudaGetLastError();
}
template <typename R, int T>
cudaError_t launch_stream(const CgArgs<R>& a, const int* list, int nb, int rowb, cudaStream_t st) {
  DevTimer* timer = capture_timer(sizeof(R) == 8 ? PC_CG_F64 : PC_CG_F32);
  return timer ? launch_stream_form<R, T, true>(a, list, nb, rowb, timer, st)
               : launch_stream_form<R, T, false>(a, list, nb, rowb, nullptr, st);
}

// bytes of a row in a stage
int stream_row(int n_pw, int elem) { return (n_pw * elem + 15) / 16 * 16; }

template <typename R, int T, int V, bool PROJ>
cudaError_t launch(const CgArgs<R>& a, const int* list, int nb, int C, const CgProj<R>& pj,
                   const CgTail& tail, cudaStream_t st) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)nb * C);
  cfg.blockDim = dim3(T);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_cg_step<R, T, V, PROJ>, a, list, pj, tail);
}

// smallest cluster (1, 2, 4, 8) of T-thread blocks with V vectors per thread
// that covers nvec vectors; 0 when none does
int cluster_for(int nvec, int T, int V) {
  for (int c = 1; c <= 8; c *= 2)
    if ((long long)c * T * V >= nvec) return c;
  return 0;
}

}  // namespace

bool cg_streams(int n_rhs, int n_pw, int elem) {
  return n_rhs > CG_TAIL_MAX && 8 * (size_t)stream_row(n_pw, elem) <= CG_STREAM_SMEM;
}

template <typename R>
cudaError_t cg_step(const CgArgs<R>& a, const int* list, int n_list, cudaStream_t st,
                    const CgProj<R>* proj, const CgTail* tail) {
  const int nb = list ? n_list : a.n_rhs;
  if (nb <= 0) return cudaSuccess;
  // x, r, p, Ap read once; x, r, p written once: 7 vector passes per active RHS
  ProfScope ps(sizeof(R) == 8 ? PC_CG_F64 : PC_CG_F32, st, 12.0 * nb * (double)a.n_pw,
               7.0 * nb * (double)a.n_pw * sizeof(R), list ? a.list_count : nullptr, nb);
  count_launch();
  const int nvec = (a.n_pw + Vec<R>::n - 1) / Vec<R>::n;
  const CgProj<R> pj = proj ? *proj : CgProj<R>{};
  const CgTail tl = tail ? *tail : CgTail{};
  if (!proj && !tl.on && cg_streams(a.n_rhs, a.n_pw, sizeof(R))) {
    CgArgs<R> b = a;
    b.n_listed = nb;
    const int rowb = stream_row(a.n_pw, sizeof(R));
    if (nvec <= 64 * CG_STREAM_V) return launch_stream<R, 64>(b, list, nb, rowb, st);
    if (nvec <= 128 * CG_STREAM_V) return launch_stream<R, 128>(b, list, nb, rowb, st);
    if (nvec <= 256 * CG_STREAM_V) return launch_stream<R, 256>(b, list, nb, rowb, st);
    return launch_stream<R, 512>(b, list, nb, rowb, st);
  }
  // shapes of the autotuner (cg_start's default CG_FEW: as many blocks per RHS
  // as help, for few RHS)
  struct Shape {
    int T, V;
  };
  static const Shape shapes[CG_NUM_VARIANTS] = {{256, 4}, {256, 8}, {512, 4}, {128, 8}};
  Shape sh{256, 1};
  if (!proj && a.variant >= 0 && a.variant < CG_NUM_VARIANTS) sh = shapes[a.variant];
  int C = cluster_for(nvec, sh.T, sh.V);
  while (!C && sh.V < 8) {
    sh.V *= 2;
    C = cluster_for(nvec, sh.T, sh.V);
  }
  if (!C) {
    sh = Shape{512, 8};
    C = cluster_for(nvec, sh.T, sh.V);
  }
  if (!C) return cudaErrorInvalidValue;
  if (proj) {
    switch (sh.T * 16 + sh.V) {
      case 256 * 16 + 1: return launch<R, 256, 1, true>(a, list, nb, C, pj, tl, st);
      case 256 * 16 + 2: return launch<R, 256, 2, true>(a, list, nb, C, pj, tl, st);
      case 256 * 16 + 4: return launch<R, 256, 4, true>(a, list, nb, C, pj, tl, st);
      case 256 * 16 + 8: return launch<R, 256, 8, true>(a, list, nb, C, pj, tl, st);
    }
    return cudaErrorInvalidValue;
  }
  switch (sh.T * 16 + sh.V) {
    case 256 * 16 + 1: return launch<R, 256, 1, false>(a, list, nb, C, pj, tl, st);
    case 256 * 16 + 2: return launch<R, 256, 2, false>(a, list, nb, C, pj, tl, st);
    case 256 * 16 + 4: return launch<R, 256, 4, false>(a, list, nb, C, pj, tl, st);
    case 256 * 16 + 8: return launch<R, 256, 8, false>(a, list, nb, C, pj, tl, st);
    case 512 * 16 + 4: return launch<R, 512, 4, false>(a, list, nb, C, pj, tl, st);
    case 512 * 16 + 8: return launch<R, 512, 8, false>(a, list, nb, C, pj, tl, st);
    case 128 * 16 + 8: return launch<R, 128, 8, false>(a, list, nb, C, pj, tl, st);
  }
  return cudaErrorInvalidValue;
}
template cudaError_t cg_step<double>(const CgArgs<double>&, const int*, int, cudaStream_t,
                                     const CgProj<double>*, const CgTail*);
template cudaError_t cg_step<float>(const CgArgs<float>&, const int*, int, cudaStream_t,
                                    const CgProj<float>*, const CgTail*);

bool cg_proj_fits(int n_pw, int elem, int n_ext) {
  if (n_ext > CG_PROJ_MAX) return false;
  return cluster_for((n_pw * elem + 15) / 16, 256, 8) > 0;
}

}  // namespace pdep
