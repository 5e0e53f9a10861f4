// Solve-phase CUDA kernels for sm_103a: blocked SELL-32 and plain-BSR SpMV,
// the fused residual + polynomial smoothing step, multicolour Gauss-Seidel,
// the coarse solves and the CGS2 Arnoldi reductions.  The float32 sparse work
// is bound by HBM bandwidth (small coarse levels by latency), the float64
// matvec and CGS2 passes by GB300's FP64 rate; loads of a warp are contiguous
// per slot and every reduction has a fixed order.
#include "kernels.cuh"

#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <mutex>
#include <type_traits>

namespace mfs {
namespace dev {

namespace {

constexpr int kThreads = 256;
// CTAs of the one-thread-per-row SELL-32 kernels: two slices, so that a grid
// of a few thousand CTAs spreads evenly over the SMs (with 256-thread CTAs
// the busiest SM held 8 where the average was 7.1)
constexpr int kSellThreads = 64;
// plain-BSR matrices with at most kCtaRowsMax rows averaging at least
// kCtaRowBlocks blocks per row take one CTA per row instead of one warp
constexpr int64_t kCtaRowsMax = 4096;
constexpr int64_t kCtaRowBlocks = 128;
constexpr int64_t kCtaRowsMax64 = 1024;  // the same for float64 (cta_rows)
constexpr int64_t kCtaRowBlocks64 = 768;
constexpr int kGsCtaThreads = 1024;  // threads of the one-CTA Gauss-Seidel kernel for small levels
LaunchHook *g_hook = nullptr;
// > 0 while this thread's launches must bypass the process-wide hook
thread_local int g_hook_off = 0;

// While set, this thread's launches are appended here instead of issued.
thread_local Recorder *g_rec = nullptr;
// While set, this thread's solve-phase launches are programmatic dependent
// launches where they directly follow another of its kernel launches on the
// same stream (g_pdl_prev): a kernel after a copy, an event or a graph launch
// is launched normally.
thread_local unsigned g_pdl = 0;    // largest grid (CTAs) launched this way; 0: none
thread_local unsigned g_pdl64 = 0;  // the same for kernels bound by the FP64 pipe (K::kFp64)
thread_local cudaStream_t g_pdl_prev = nullptr;
// accounting of the launch being issued (HookScope fills it for the recorder)
thread_local RecOp g_acct;

struct HookScope {
  cudaStream_t s;
  int cls;
  double bytes;
  int sig;
  int64_t rows;
  double flops;
  bool on = false;
  HookScope(cudaStream_t s_, int c, double b, int sg, int64_t r, double f)
      : s(s_), cls(c), bytes(b), sig(sg), rows(r), flops(f) {
    if (g_rec) {
      g_acct.cls = c;
      g_acct.sig = sg;
      g_acct.rows = r;
      g_acct.bytes = b;
      g_acct.flops = f;
      return;
    }
    if (g_hook && !g_hook_off) on = g_hook->before(s, cls, sig, rows);
    if (on) g_pdl_prev = nullptr;  // an event precedes the launch
  }
  ~HookScope() {
    if (on) {
      g_hook->after(s, cls, bytes, sig, rows, flops);
      g_pdl_prev = nullptr;
    }
  }
};

// Every solve-phase kernel is a traits struct K: K::Args (its arguments),
// K::run(args, block, blocks) (its body for one block of a grid of `blocks`)
// and K::kMaxThreads.  k_solo runs it over a normal grid; k_multi runs many
// independent launches of K (one per system of a batch) as ONE grid: CTA c
// runs block map[c].bid of the launch whose arguments are tab[map[c].t],
// unless that launch's system map[c].g is inactive.
// Launched as a programmatic dependent launch (set_pdl), a kernel may be
// scheduled while its predecessor in the stream still runs: it first waits
// until that predecessor has completed and its writes are visible, then lets
// its own successor start launching.  Launched normally, both are no-ops.
// Kernels with K::kEarly take the wait as a functor and call it (once, by
// every thread) after their first loads of matrix data, which no launch of a
// solve writes: a chain of dependent small launches then pays for the row
// pointer, the columns and the blocks while the predecessor still runs (a
// 13-CTA gather chain: 1.24 -> 0.97 us a launch).
// Loads of matrix data that stay before the wait: volatile, so that the
// compiler does not move them behind it (as __ldg they were: 1.82 -> 1.72 ms
// for a solve of the 3,267-dof system)
__device__ __forceinline__ int32_t ld_pin(const int32_t *p) {
  int32_t v;
  asm volatile("ld.global.nc.b32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ float ld_pin(const float *p) {
  float v;
  asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ double ld_pin(const double *p) {
  double v;
  asm volatile("ld.global.nc.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}
// a plain-BSR block, in the loads of ldg_block
template <int N, typename T> __device__ __forceinline__ void ld_pin_block(const T *p, T (&o)[N]) {
  constexpr int B = N * (int)sizeof(T);
  if constexpr (sizeof(T) == 8 && B % 16 == 0) {
#pragma unroll
    for (int i = 0; i < N; i += 2)
      asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];" : "=d"(o[i]), "=d"(o[i + 1]) : "l"(p + i));
  } else if constexpr (sizeof(T) == 4 && B % 16 == 0) {
#pragma unroll
    for (int i = 0; i < N; i += 4)
      asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];"
                   : "=f"(o[i]), "=f"(o[i + 1]), "=f"(o[i + 2]), "=f"(o[i + 3])
                   : "l"(p + i));
  } else if constexpr (sizeof(T) == 4 && B % 8 == 0) {
#pragma unroll
    for (int i = 0; i < N; i += 2)
      asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(o[i]), "=f"(o[i + 1]) : "l"(p + i));
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) o[i] = ld_pin(p + i);
  }
}
// A vector that an earlier launch of the solve wrote: an ordinary load.  Under
// a programmatic launch this grid is resident while its predecessor still
// writes x, so x is not read-only for the life of the kernel and must not be
// read through the non-coherent path (__ldg, ld.global.nc), whose loads the
// compiler may also move across the wait; ordinary loads stay behind the
// wait's memory clobber as long as x is not __restrict__ in the function that
// waits.  __ldg and ld_pin are for matrix data, which only the setup writes.
template <typename T> __device__ __forceinline__ T ld_vec(const T *p) { return *p; }
struct PdlWait {
  __device__ __forceinline__ void operator()() const {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }
};
struct NoWait {
  __device__ __forceinline__ void operator()() const {}
};
template <class K, class = void> struct IsEarly : std::false_type {};
template <class K> struct IsEarly<K, std::void_t<decltype(K::kEarly)>> : std::true_type {};

// Kernels that the FP64 pipe bounds have K::kFp64 = true.  A CTA launched ahead
// takes its place while the predecessor's CTAs still hold theirs, so a grid
// of a few CTAs per SM ends up uneven, and the SM with the most float64 work
// sets the time; the float32 kernels wait for memory and do not mind.
template <class K, class = void> struct IsFp64 : std::false_type {};
template <class K> struct IsFp64<K, std::void_t<decltype(K::kFp64)>> : std::bool_constant<K::kFp64> {};

template <class K>
__global__ void __launch_bounds__(K::kMaxThreads) k_solo(const __grid_constant__ typename K::Args a) {
  if constexpr (IsEarly<K>::value) {
    K::run(a, (int)blockIdx.x, (int)gridDim.x, PdlWait());
  } else {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    K::run(a, (int)blockIdx.x, (int)gridDim.x);
  }
}

// CTAs per SM the multi-system form of K must fit (K::kMinBlocks, default 1):
// its arguments come from a table instead of the constant bank, which costs
// registers (112 instead of 32 in the coupled matvec); the kernels of large
// grids are held to about the registers of their single-system form so that as
// many CTAs stay resident (256 boxes 607 -> 561 ms; the small float64 sparse
// kernels, which wait for their own chains, lost 2 % and are not)
template <class K, class = void> struct MinBlocks {
  static constexpr int value = 1;
};
template <class K> struct MinBlocks<K, std::void_t<decltype(K::kMinBlocks)>> {
  static constexpr int value = K::kMinBlocks;
};

template <class K>
__global__ void __launch_bounds__(K::kMaxThreads, MinBlocks<K>::value)
k_multi(const typename K::Args *__restrict__ tab, const MsBlock *__restrict__ map, const int *__restrict__ active) {
  const MsBlock m = map[blockIdx.x];
  if (active != nullptr && active[m.g] == 0) return;
  if constexpr (IsEarly<K>::value) K::run(tab[m.t], m.bid, m.nb, NoWait());
  else K::run(tab[m.t], m.bid, m.nb);
}

// issue one launch of K, or record it (with the accounting of the enclosing
// HookScope) when this thread has a recorder
template <class K>
void go(unsigned grid, unsigned threads, size_t smem, cudaStream_t s, const typename K::Args &a) {
  if (g_rec) {
    RecOp op = g_acct;
    op.fn = (const void *)&k_multi<K>;
    op.grid = grid;
    op.threads = threads;
    op.smem = smem;
    op.args.assign((const unsigned char *)&a, (const unsigned char *)&a + sizeof(a));
    g_rec->ops.push_back(std::move(op));
    g_acct = RecOp();
    return;
  }
  const bool pdl = grid <= (IsFp64<K>::value ? g_pdl64 : g_pdl) && g_pdl_prev == s;
  g_pdl_prev = g_pdl ? s : nullptr;
  if (pdl) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_solo<K>, a);
    return;
  }
  k_solo<K><<<grid, threads, smem, s>>>(a);
}

template <typename T> int sparse_sig(const Sell &A) {
  // 3 / 9: SELL-32 with 4 / 8 slots in flight, 8: several threads per row
  if (A.kind == 0 && A.split > 1) return 8000 + A.br * 100 + A.bc * 10 + (sizeof(T) == 8 ? 1 : 0);
  const int layout = A.kind == 0 && A.unroll == 4 ? 3 : (A.kind == 0 && A.unroll == 8 ? 9 : A.kind);
  return layout * 1000 + A.br * 100 + A.bc * 10 + (sizeof(T) == 8 ? 1 : 0);
}

// algorithmic bytes of one pass over a block matrix: values + block-column
// indices + row lengths, each read once
template <typename T> double matrix_bytes(const Sell &A) {
  return (double)A.nnzb * (A.br * A.bc * sizeof(T) + sizeof(int32_t)) + (double)A.nbr * sizeof(int32_t);
}

// The N entries of one plain-BSR block (row-major, consecutive) in the widest
// loads its size allows: 16-byte loads when N * sizeof(T) is a multiple of
// 16, 8-byte ones when a multiple of 8, else one load per entry.  Block k
// starts k * N * sizeof(T) bytes into a value array that starts on a 16-byte
// boundary (every value array is its own allocation; the setup checks it), so
// every vector is aligned.  Fewer, wider loads keep the load queue of the plain-BSR
// kernels from filling (6x6 float blocks: 9 loads instead of 36).
template <int N, typename T>
__device__ __forceinline__ void ldg_block(const T *__restrict__ p, T (&o)[N]) {
  constexpr int B = N * (int)sizeof(T);
  if constexpr (sizeof(T) == 8 && B % 16 == 0) {
    const double2 *q = reinterpret_cast<const double2 *>(p);
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
      const double2 v = __ldg(q + i);
      o[2 * i] = v.x;
      o[2 * i + 1] = v.y;
    }
  } else if constexpr (sizeof(T) == 4 && B % 16 == 0) {
    const float4 *q = reinterpret_cast<const float4 *>(p);
#pragma unroll
    for (int i = 0; i < N / 4; ++i) {
      const float4 v = __ldg(q + i);
      o[4 * i] = v.x;
      o[4 * i + 1] = v.y;
      o[4 * i + 2] = v.z;
      o[4 * i + 3] = v.w;
    }
  } else if constexpr (sizeof(T) == 4 && B % 8 == 0) {
    const float2 *q = reinterpret_cast<const float2 *>(p);
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
      const float2 v = __ldg(q + i);
      o[2 * i] = v.x;
      o[2 * i + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) o[i] = __ldg(p + i);
  }
}

inline unsigned grid_for(int64_t n, int threads = kThreads) {
  return (unsigned)((n + threads - 1) / threads);
}

template <int BR, int BC, typename T, int U>
__device__ __forceinline__ void sell_row(const int32_t *__restrict__ sp, const int32_t *__restrict__ rl,
                                         const int32_t *__restrict__ col, const T *__restrict__ val,
                                         const T *__restrict__ x, int64_t row, T (&acc)[BR]) {
  const int lane = (int)(row & 31);
  const int64_t slice = row >> 5;
  const int64_t base = sp[slice];
  const int len = rl[row];
  const int32_t *cp = col + base * 32 + lane;
  const T *vp = val + base * (BR * BC * 32) + lane;
#pragma unroll
  for (int r = 0; r < BR; ++r) acc[r] = T(0);
  // U slots in flight per thread (chosen per matrix by the layout autotuner)
#pragma unroll U
  for (int t = 0; t < len; ++t) {
    const int64_t c = __ldg(cp + (int64_t)t * 32);
    T xv[BC];
#pragma unroll
    for (int q = 0; q < BC; ++q) xv[q] = ld_vec(x + c * BC + q);
    const T *v = vp + (int64_t)t * (BR * BC * 32);
#pragma unroll
    for (int r = 0; r < BR; ++r)
#pragma unroll
      for (int q = 0; q < BC; ++q) acc[r] += __ldg(v + (r * BC + q) * 32) * xv[q];
  }
}

// A plain-BSR block row by a group of L = 2^ls lanes (8, 16 or 32): the lanes
// stride over the row's blocks.  The first block of a lane is loaded before
// `wait` (see k_solo), the next column while the current block is used, so
// that a further block costs one load latency instead of two.  (Two or four
// blocks of a lane at a time cost registers: 23^3 box AMG(BGS) 9.8 -> 10.1-12.1 ms.)
template <int BR, int BC, typename T, class W>
__device__ __forceinline__ void bsr_row(const int32_t *__restrict__ rp, const int32_t *__restrict__ col,
                                        const T *__restrict__ val, const T *x, int64_t row, bool active,
                                        int gl, int ls, W wait, T (&acc)[BR]) {
  int k = 0, hi = 0;
  if (active) {
    k = ld_pin(rp + row) + gl;
    hi = ld_pin(rp + row + 1);
  }
  int64_t c = 0;
  T blk[BR * BC];
  if (k < hi) {
    c = ld_pin(col + k);
    ld_pin_block<BR * BC, T>(val + (int64_t)k * (BR * BC), blk);
  }
  wait();
#pragma unroll
  for (int r = 0; r < BR; ++r) acc[r] = T(0);
  while (k < hi) {
    const int kn = k + (1 << ls);
    T xv[BC];
#pragma unroll
    for (int q = 0; q < BC; ++q) xv[q] = ld_vec(x + c * BC + q);
    if (kn < hi) c = __ldg(col + kn);
#pragma unroll
    for (int r = 0; r < BR; ++r)
#pragma unroll
      for (int q = 0; q < BC; ++q) acc[r] += blk[r * BC + q] * xv[q];
    if (kn < hi) ldg_block<BR * BC, T>(val + (int64_t)kn * (BR * BC), blk);
    k = kn;
  }
}

// Sums of the BR entries over a group of 2^ls lanes (8, 16 or 32).  With R the
// power of two >= BR: while a lane still holds several entries it keeps one
// half, adds the partner's and hands the other half over, so 6 adds instead
// of 15 for three entries and 32 lanes (in float64 every add of a warp takes
// 64 cycles of an SM quarter).  Lane gl returns the sum of entry
// sum_entry<BR>(gl, ls); entries past BR - 1 are zero.
template <int BR> constexpr int kSumRows = BR <= 1 ? 1 : BR <= 2 ? 2 : BR <= 4 ? 4 : 8;
template <int BR> __device__ __forceinline__ int sum_entry(int gl, int ls) { return (gl * kSumRows<BR>) >> ls; }
template <int BR> __device__ __forceinline__ bool sum_owner(int gl, int ls) {
  return (gl & ((1 << ls) / kSumRows<BR> - 1)) == 0 && sum_entry<BR>(gl, ls) < BR;
}
template <int BR, typename T>
__device__ __forceinline__ T group_sum(const T (&acc)[BR], int gl, int ls) {
  constexpr int R = kSumRows<BR>;
  T a[R];
#pragma unroll
  for (int r = 0; r < R; ++r) a[r] = r < BR ? acc[r < BR ? r : 0] : T(0);
  int o = 1 << (ls - 1);
#pragma unroll
  for (int m = R / 2; m > 0; m /= 2, o >>= 1) {
    const bool up = (gl & o) != 0;
#pragma unroll
    for (int r = 0; r < m; ++r) {
      const T keep = up ? a[r + m] : a[r], give = up ? a[r] : a[r + m];
      a[r] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  for (; o > 0; o >>= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
  return a[0];
}

// dx of one node from its row sums acc (see gs_sweeps), written into x
template <int BR, typename T>
__device__ __forceinline__ void gs_update(const T (&acc)[BR], int64_t node, const T *__restrict__ dblk,
                                          const T *__restrict__ b, T *x, T omega, bool backward) {
  const T *D = dblk + node * (BR * BR);
  T dx[BR];
  if (!backward) {
#pragma unroll
    for (int r = 0; r < BR; ++r) {
      T res = b[node * BR + r] - acc[r];
#pragma unroll
      for (int c = 0; c < r; ++c) res -= D[r * BR + c] * dx[c];
      dx[r] = omega * res / D[r * BR + r];
    }
  } else {
#pragma unroll
    for (int r = BR - 1; r >= 0; --r) {
      T res = b[node * BR + r] - acc[r];
#pragma unroll
      for (int c = r + 1; c < BR; ++c) res -= D[r * BR + c] * dx[c];
      dx[r] = omega * res / D[r * BR + r];
    }
  }
#pragma unroll
  for (int r = 0; r < BR; ++r) x[node * BR + r] += dx[r];
}

template <int BR, int BC, typename T>
struct KSpmvWarp {
  static constexpr int kMaxThreads = kThreads;
  static constexpr int kMinBlocks = sizeof(T) == 4 && BR * BC <= 9 ? 5 : 1;  // multi-system form: <= 48 registers
  static constexpr bool kFp64 = sizeof(T) == 8;
  static constexpr bool kEarly = true;
  struct Args {
    int64_t nbr;
    const int32_t *rp;
    const int32_t *col;
    const T *val;
    const T *x;
    T *y;
    T alpha;
    T beta;
    const T *z;
    int ls;  // log2 of the lanes per row
  };
  template <class W> static __device__ __forceinline__ void run(const Args &a, int bid, int nb, W wait) {
    const int64_t row = ((int64_t)bid * blockDim.x + threadIdx.x) >> a.ls;
    const int gl = threadIdx.x & ((1 << a.ls) - 1);
    T acc[BR];
    bsr_row<BR, BC, T>(a.rp, a.col, a.val, a.x, row, row < a.nbr, gl, a.ls, wait, acc);
    const bool own = row < a.nbr && sum_owner<BR>(gl, a.ls);
    const int64_t i = row * BR + sum_entry<BR>(gl, a.ls);
    const T zi = own && a.z != nullptr ? a.z[i] : T(0);
    const T s = group_sum<BR, T>(acc, gl, a.ls);
    if (own) a.y[i] = a.z != nullptr ? a.alpha * s + a.beta * zi : a.alpha * s;
  }
};

// One CTA per block row, for few and long rows (restrictions to small coarse
// levels): threads stride over the row's blocks, then a fixed butterfly per
// warp and a fixed-order sum over the warps.
template <int BR, int BC, typename T>
__device__ __forceinline__ void cta_row(const int32_t *__restrict__ rp, const int32_t *__restrict__ col,
                                        const T *__restrict__ val, const T *__restrict__ x, int64_t row,
                                        T (*part)[BR]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T acc[BR];
#pragma unroll
  for (int r = 0; r < BR; ++r) acc[r] = T(0);
  for (int k = rp[row] + threadIdx.x; k < rp[row + 1]; k += blockDim.x) {
    const int64_t c = __ldg(col + k);
    T xv[BC];
#pragma unroll
    for (int q = 0; q < BC; ++q) xv[q] = ld_vec(x + c * BC + q);
    T blk[BR * BC];
    ldg_block<BR * BC, T>(val + (int64_t)k * (BR * BC), blk);
#pragma unroll
    for (int r = 0; r < BR; ++r)
#pragma unroll
      for (int q = 0; q < BC; ++q) acc[r] += blk[r * BC + q] * xv[q];
  }
#pragma unroll
  for (int r = 0; r < BR; ++r) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
    if (lane == 0) part[warp][r] = acc[r];
  }
  __syncthreads();
}

template <int BR, int BC, typename T>
__device__ __forceinline__ void d_spmv_cta(int64_t nbr, const int32_t *__restrict__ rp, const int32_t *__restrict__ col,
           const T *__restrict__ val, const T *__restrict__ x, T *y, T alpha, T beta, const T *z, int bid_, int nb_) {
  __shared__ T part[kThreads / 32][BR];
  const int64_t row = bid_;
  cta_row<BR, BC, T>(rp, col, val, x, row, part);
  if (threadIdx.x < BR) {
    T a = T(0);
    for (int w = 0; w < kThreads / 32; ++w) a += part[w][threadIdx.x];
    const int64_t i = row * BR + threadIdx.x;
    y[i] = z != nullptr ? alpha * a + beta * z[i] : alpha * a;
  }
}
template <int BR, int BC, typename T>
struct KSpmvCta {
  static constexpr int kMaxThreads = kThreads;
  static constexpr bool kFp64 = sizeof(T) == 8;
  struct Args {
    int64_t nbr;
    const int32_t *rp;
    const int32_t *col;
    const T *val;
    const T *x;
    T *y;
    T alpha;
    T beta;
    const T *z;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    d_spmv_cta<BR, BC, T>(a.nbr, a.rp, a.col, a.val, a.x, a.y, a.alpha, a.beta, a.z, bid, nb);
  }
};

// the same row per CTA for a smoothing step
template <int BR, typename T>
struct KSmoothCta {
  static constexpr int kMaxThreads = kThreads;
  static constexpr bool kFp64 = sizeof(T) == 8;
  struct Args {
    int64_t nbr;
    const int32_t *rp;
    const int32_t *col;
    const T *val;
    const T *dinv;
    const T *b;
    const T *x;
    T *xout;
    T *d;
    T c1;
    T c2;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    __shared__ T part[kThreads / 32][BR];
    const int64_t i = (int64_t)bid * BR + threadIdx.x;
    T bi = T(0), xi = T(0), dd = T(0), di = T(0);
    if (threadIdx.x < BR) {
      bi = a.b[i];
      xi = a.x[i];
      dd = a.d[i];
      di = a.dinv[i];
    }
    cta_row<BR, BR, T>(a.rp, a.col, a.val, a.x, bid, part);
    if (threadIdx.x < BR) {
      T s = T(0);
      for (int w = 0; w < kThreads / 32; ++w) s += part[w][threadIdx.x];
      dd = a.c1 * dd + a.c2 * di * (bi - s);
      a.d[i] = dd;
      a.xout[i] = xi + dd;
    }
  }
};

template <int BR, typename T>
struct KSmoothWarp {
  static constexpr int kMaxThreads = kThreads;
  static constexpr int kMinBlocks = sizeof(T) == 4 && BR <= 3 ? 5 : 1;  // multi-system form: <= 48 registers
  static constexpr bool kFp64 = sizeof(T) == 8;
  static constexpr bool kEarly = true;
  struct Args {
    int64_t nbr;
    const int32_t *rp;
    const int32_t *col;
    const T *val;
    const T *dinv;
    const T *b;
    const T *x;
    T *xout;
    T *d;
    T c1;
    T c2;
    int ls;  // log2 of the lanes per row
  };
  template <class W> static __device__ __forceinline__ void run(const Args &a, int bid, int nb, W wait) {
    const int64_t row = ((int64_t)bid * blockDim.x + threadIdx.x) >> a.ls;
    const int gl = threadIdx.x & ((1 << a.ls) - 1);
    const bool own = row < a.nbr && sum_owner<BR>(gl, a.ls);
    const int64_t i = row * BR + sum_entry<BR>(gl, a.ls);
    const T di = own ? ld_pin(a.dinv + i) : T(0);
    T acc[BR];
    bsr_row<BR, BR, T>(a.rp, a.col, a.val, a.x, row, row < a.nbr, gl, a.ls, wait, acc);
    T bi = T(0), xi = T(0), dd = T(0);
    if (own) {
      bi = a.b[i];
      xi = a.x[i];
      dd = a.d[i];
    }
    const T s = group_sum<BR, T>(acc, gl, a.ls);
    if (own) {
      const T res = bi - s;
      dd = a.c1 * dd + a.c2 * di * res;
      a.d[i] = dd;
      a.xout[i] = xi + dd;
    }
  }
};

template <int BR, int BC, typename T, int U>
__device__ __forceinline__ void d_spmv(int64_t nbr, const int32_t *__restrict__ sp, const int32_t *__restrict__ rl,
       const int32_t *__restrict__ col, const T *__restrict__ val, const T *__restrict__ x, T *y,
       T alpha, T beta, const T *z, int bid_, int nb_) {
  const int64_t row = (int64_t)bid_ * blockDim.x + threadIdx.x;
  if (row >= nbr) return;
  T acc[BR];
  sell_row<BR, BC, T, U>(sp, rl, col, val, x, row, acc);
  T *yp = y + row * BR;
  if (z != nullptr) {
    const T *zp = z + row * BR;
    T zv[BR];
#pragma unroll
    for (int r = 0; r < BR; ++r) zv[r] = zp[r];
#pragma unroll
    for (int r = 0; r < BR; ++r) yp[r] = alpha * acc[r] + beta * zv[r];
  } else {
#pragma unroll
    for (int r = 0; r < BR; ++r) yp[r] = alpha * acc[r];
  }
}
template <int BR, int BC, typename T, int U>
struct KSpmvSell {
  static constexpr int kMaxThreads = kThreads;
  static constexpr bool kFp64 = sizeof(T) == 8;
  static constexpr int kMinBlocks = BR * BC <= 9 ? 8 : 1;  // multi-system form: <= 32 registers
  struct Args {
    int64_t nbr;
    const int32_t *sp;
    const int32_t *rl;
    const int32_t *col;
    const T *val;
    const T *x;
    T *y;
    T alpha;
    T beta;
    const T *z;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    d_spmv<BR, BC, T, U>(a.nbr, a.sp, a.rl, a.col, a.val, a.x, a.y, a.alpha, a.beta, a.z, bid, nb);
  }
};

// SELL-32 with H = blockDim.x / 32 threads per block row, for matrices whose
// rows alone do not fill the GPU: a CTA takes one slice, its warp h the slots
// h, h + H, ... of the 32 rows; the H partial sums of an entry meet in shared
// memory and are added in the order of h by the thread that finishes the
// entry (entry e of the slice: row e / BR, component e % BR, so that the
// vectors are read and written in whole segments; up to BR entries a thread).
// One thread per row left 68,921 rows of 27 3x3 float32 blocks with 453
// threads per SM, each walking its slots: 22.8 us a product, the best other
// layout 20.1 us, with H = 4 11.9 us (launch and events: 5.5 us of each).
// (Loading the finishing entry's vectors ahead of the row cost registers:
// 18.1 instead of 17.3 ms for the SIMPLE solve of the 40^3 box.)
constexpr int kSellSplitMax = 8;
constexpr int kSellPad = 33;  // row pitch of the partial sums (bank conflicts)

template <int BR, int BC, typename T, class W>
__device__ __forceinline__ void sell_split_row(int64_t nbr, const int32_t *__restrict__ sp,
                                               const int32_t *__restrict__ rl, const int32_t *__restrict__ col,
                                               const T *__restrict__ val, const T *x, int64_t slice,
                                               W wait, T (&acc)[BR]) {
  const int lane = threadIdx.x & 31, h = threadIdx.x >> 5, H = blockDim.x >> 5;
  const int64_t row = slice * 32 + lane;
  const int64_t base = ld_pin(sp + slice);
  const int len = row < nbr ? ld_pin(rl + row) : 0;
  const int32_t *cp = col + base * 32 + lane;
  const T *vp = val + base * (BR * BC * 32) + lane;
  // first slot: before the wait (see k_solo)
  int64_t c = 0;
  T v0[BR * BC];
#pragma unroll
  for (int e = 0; e < BR * BC; ++e) v0[e] = T(0);
  if (h < len) {
    c = ld_pin(cp + (int64_t)h * 32);
#pragma unroll
    for (int e = 0; e < BR * BC; ++e) v0[e] = ld_pin(vp + ((int64_t)h * (BR * BC) + e) * 32);
  }
  wait();
#pragma unroll
  for (int r = 0; r < BR; ++r) acc[r] = T(0);
  if (h < len) {
    T xv[BC];
#pragma unroll
    for (int q = 0; q < BC; ++q) xv[q] = ld_vec(x + c * BC + q);
#pragma unroll
    for (int r = 0; r < BR; ++r)
#pragma unroll
      for (int q = 0; q < BC; ++q) acc[r] += v0[r * BC + q] * xv[q];
  }
#pragma unroll 2
  for (int t = h + H; t < len; t += H) {
    const int64_t ct = __ldg(cp + (int64_t)t * 32);
    T xv[BC];
#pragma unroll
    for (int q = 0; q < BC; ++q) xv[q] = ld_vec(x + ct * BC + q);
    const T *v = vp + (int64_t)t * (BR * BC * 32);
#pragma unroll
    for (int r = 0; r < BR; ++r)
#pragma unroll
      for (int q = 0; q < BC; ++q) acc[r] += __ldg(v + (r * BC + q) * 32) * xv[q];
  }
}

template <int BR, int BC, typename T, class W>
__device__ __forceinline__ void sell_split_sums(int64_t nbr, const int32_t *__restrict__ sp,
                                                const int32_t *__restrict__ rl, const int32_t *__restrict__ col,
                                                const T *__restrict__ val, const T *x, int64_t slice,
                                                W wait, T (*part)[BR][kSellPad]) {
  T acc[BR];
  sell_split_row<BR, BC, T>(nbr, sp, rl, col, val, x, slice, wait, acc);
#pragma unroll
  for (int r = 0; r < BR; ++r) part[threadIdx.x >> 5][r][threadIdx.x & 31] = acc[r];
  __syncthreads();
}

template <int BR, typename T>
__device__ __forceinline__ T sell_split_entry(T (*part)[BR][kSellPad], int e) {
  const int H = blockDim.x >> 5;
  T a = part[0][e % BR][e / BR];
  for (int h = 1; h < H; ++h) a += part[h][e % BR][e / BR];
  return a;
}

template <int BR, int BC, typename T>
struct KSpmvSellSplit {
  static constexpr int kMaxThreads = 32 * kSellSplitMax;
  static constexpr int kMinBlocks = sizeof(T) == 4 && BR * BC <= 9 ? 6 : 1;  // multi-system form: <= 40 registers
  static constexpr bool kFp64 = sizeof(T) == 8;
  static constexpr bool kEarly = true;
  struct Args {
    int64_t nbr;
    const int32_t *sp;
    const int32_t *rl;
    const int32_t *col;
    const T *val;
    const T *x;
    T *y;
    T alpha;
    T beta;
    const T *z;
  };
  template <class W> static __device__ __forceinline__ void run(const Args &a, int bid, int nb, W wait) {
    __shared__ T part[kSellSplitMax][BR][kSellPad];
    sell_split_sums<BR, BC, T>(a.nbr, a.sp, a.rl, a.col, a.val, a.x, bid, wait, part);
    const int64_t i0 = (int64_t)bid * 32 * BR, n = a.nbr * BR;
    for (int e = threadIdx.x; e < 32 * BR && i0 + e < n; e += blockDim.x) {
      const T s = sell_split_entry<BR, T>(part, e);
      a.y[i0 + e] = a.z != nullptr ? a.alpha * s + a.beta * a.z[i0 + e] : a.alpha * s;
    }
  }
};

template <int BR, typename T>
struct KSmoothSellSplit {
  static constexpr int kMaxThreads = 32 * kSellSplitMax;
  static constexpr int kMinBlocks = sizeof(T) == 4 && BR <= 3 ? 6 : 1;  // multi-system form: <= 40 registers
  static constexpr bool kFp64 = sizeof(T) == 8;
  static constexpr bool kEarly = true;
  struct Args {
    int64_t nbr;
    const int32_t *sp;
    const int32_t *rl;
    const int32_t *col;
    const T *val;
    const T *dinv;
    const T *b;
    const T *x;
    T *xout;
    T *d;
    T c1;
    T c2;
  };
  template <class W> static __device__ __forceinline__ void run(const Args &a, int bid, int nb, W wait) {
    __shared__ T part[kSellSplitMax][BR][kSellPad];
    sell_split_sums<BR, BR, T>(a.nbr, a.sp, a.rl, a.col, a.val, a.x, bid, wait, part);
    const int64_t i0 = (int64_t)bid * 32 * BR, n = a.nbr * BR;
    for (int e = threadIdx.x; e < 32 * BR && i0 + e < n; e += blockDim.x) {
      const int64_t i = i0 + e;
      const T res = a.b[i] - sell_split_entry<BR, T>(part, e);
      const T dd = a.c1 * a.d[i] + a.c2 * a.dinv[i] * res;
      a.d[i] = dd;
      a.xout[i] = a.x[i] + dd;
    }
  }
};

// Sums of products with their V-cycle epilogue (spmv_terms).  The couplings,
// residuals and first smoothing steps of a small or mid-size level are
// launches of 2 to 4 us whose work takes a fraction of that; one launch does
// what 2 to 4 did (and the vectors in between are written and read once less).
template <typename T> struct TermArgs {
  const int32_t *rp, *rl, *col;  // rp: slice offsets in SELL-32
  const T *val, *x;
  int bc;
};
template <typename T> struct EpiArgs {
  T alpha, beta, c1, c2;
  const T *z, *dinv, *x;  // x: kRowSmooth's vector of the level
  T *y, *d, *xout;
  int mode;
};
// operands of one entry, loaded ahead of its sum
template <typename T> struct EpiVals {
  T z, dinv, d, x;
};
template <bool SM, typename T>
__device__ __forceinline__ EpiVals<T> epi_load(const EpiArgs<T> &e, int64_t i) {
  EpiVals<T> v;
  if constexpr (SM) {
    v.z = e.z[i];
    v.dinv = e.dinv[i];
    v.d = e.d[i];
    v.x = e.x[i];
  } else {
    v.z = e.mode == kRowSub ? e.y[i] : e.z != nullptr ? e.z[i] : T(0);
    v.dinv = e.mode != kRowPlain ? e.dinv[i] : T(0);
  }
  return v;
}
// s: the sum (SM: without the last term), t: the last term (SM)
template <bool SM, typename T>
__device__ __forceinline__ void epi_store(const EpiArgs<T> &e, int64_t i, const EpiVals<T> &v, T s, T t) {
  if constexpr (SM) {
    const T c = v.z - s;
    const T res = c - t;
    const T dd = e.c1 * v.d + e.c2 * v.dinv * res;
    e.y[i] = c;
    e.d[i] = dd;
    e.xout[i] = v.x + dd;
  } else if (e.mode == kRowSub) {
    e.y[i] = v.z - v.dinv * s;
  } else {
    const T y = e.z != nullptr ? e.alpha * s + e.beta * v.z : e.alpha * s;
    e.y[i] = y;
    if (e.mode == kRowFirst) {
      const T dd = e.c2 * v.dinv * y;
      e.d[i] = dd;
      e.xout[i] = dd;
    }
  }
}

#define MFS_BC_SWITCH(BCV, CALL)                     \
  switch (BCV) {                                     \
    case 1: { constexpr int BC_ = 1; CALL; } break;  \
    case 2: { constexpr int BC_ = 2; CALL; } break;  \
    case 3: { constexpr int BC_ = 3; CALL; } break;  \
    default: { constexpr int BC_ = 6; CALL; } break; \
  }

template <int BR, typename T, bool SM>
struct KTermsBsr {
  static constexpr int kMaxThreads = kThreads;
  static constexpr bool kFp64 = sizeof(T) == 8;
  static constexpr bool kEarly = true;
  struct Args {
    int64_t nbr;
    int nt, ls;
    TermArgs<T> t[kMaxTerms];
    EpiArgs<T> e;
  };
  template <class W> static __device__ __forceinline__ void run(const Args &a, int bid, int nb, W wait) {
    const int64_t row = ((int64_t)bid * blockDim.x + threadIdx.x) >> a.ls;
    const int gl = threadIdx.x & ((1 << a.ls) - 1);
    const bool act = row < a.nbr, own = act && sum_owner<BR>(gl, a.ls);
    const int64_t i = row * BR + sum_entry<BR>(gl, a.ls);
    T acc[BR], last[BR];
    MFS_BC_SWITCH(a.t[0].bc, (bsr_row<BR, BC_, T>(a.t[0].rp, a.t[0].col, a.t[0].val, a.t[0].x, row, act, gl, a.ls,
                                                  wait, acc)));
    for (int k = 1; k < a.nt; ++k) {
      MFS_BC_SWITCH(a.t[k].bc, (bsr_row<BR, BC_, T>(a.t[k].rp, a.t[k].col, a.t[k].val, a.t[k].x, row, act, gl, a.ls,
                                                    NoWait(), last)));
      if (!SM || k + 1 < a.nt)
#pragma unroll
        for (int r = 0; r < BR; ++r) acc[r] += last[r];
    }
    EpiVals<T> v{};
    if (own) v = epi_load<SM, T>(a.e, i);
    const T s = group_sum<BR, T>(acc, gl, a.ls);
    T t = T(0);
    if constexpr (SM) t = group_sum<BR, T>(last, gl, a.ls);
    if (own) epi_store<SM, T>(a.e, i, v, s, t);
  }
};

template <int BR, typename T, bool SM>
struct KTermsSell {
  static constexpr int kMaxThreads = 32 * kSellSplitMax;
  static constexpr bool kFp64 = sizeof(T) == 8;
  static constexpr bool kEarly = true;
  using Args = typename KTermsBsr<BR, T, SM>::Args;  // ls unused
  template <class W> static __device__ __forceinline__ void run(const Args &a, int bid, int nb, W wait) {
    __shared__ T part[kSellSplitMax][BR][kSellPad];
    __shared__ T part2[SM ? kSellSplitMax : 1][BR][kSellPad];
    const int lane = threadIdx.x & 31, h = threadIdx.x >> 5;
    T acc[BR], last[BR];
    MFS_BC_SWITCH(a.t[0].bc, (sell_split_row<BR, BC_, T>(a.nbr, a.t[0].rp, a.t[0].rl, a.t[0].col, a.t[0].val,
                                                         a.t[0].x, bid, wait, acc)));
    for (int k = 1; k < a.nt; ++k) {
      MFS_BC_SWITCH(a.t[k].bc, (sell_split_row<BR, BC_, T>(a.nbr, a.t[k].rp, a.t[k].rl, a.t[k].col, a.t[k].val,
                                                           a.t[k].x, bid, NoWait(), last)));
      if (!SM || k + 1 < a.nt)
#pragma unroll
        for (int r = 0; r < BR; ++r) acc[r] += last[r];
    }
#pragma unroll
    for (int r = 0; r < BR; ++r) {
      part[h][r][lane] = acc[r];
      if constexpr (SM) part2[h][r][lane] = last[r];
    }
    __syncthreads();
    const int64_t i0 = (int64_t)bid * 32 * BR, n = a.nbr * BR;
    for (int e = threadIdx.x; e < 32 * BR && i0 + e < n; e += blockDim.x) {
      const EpiVals<T> v = epi_load<SM, T>(a.e, i0 + e);
      const T s = sell_split_entry<BR, T>(part, e);
      T t = T(0);
      if constexpr (SM) t = sell_split_entry<BR, T>(part2, e);
      epi_store<SM, T>(a.e, i0 + e, v, s, t);
    }
  }
};

// Merged coupled rows in float64, H threads per block row.  H = 1: one
// thread per row, 64-thread CTAs (two slices).  H > 1: a CTA of 32 H threads
// takes one slice of 32 rows, its warp h the slots h, h + H, ...; the H
// partial sums of a row are added in the fixed order h = 0, 1, ... through
// shared memory.  More threads per row keep more FP64 FMAs in flight (the
// FP64 pipe bounds this kernel on GB300).
template <int BR, int B0, int B1, int B2, int H>
__device__ __forceinline__ void d_spmv_rows(int64_t nbr, const int32_t *__restrict__ sp, const int32_t *__restrict__ rl,
            const int32_t *__restrict__ col, const double *__restrict__ val, const double *__restrict__ x0,
            const double *__restrict__ x1, const double *__restrict__ x2, double *__restrict__ y, int bid_, int nb_) {
  constexpr int BCT = B0 + B1 + B2;
  const int lane = threadIdx.x & 31, h = H == 1 ? 0 : threadIdx.x >> 5;
  const int64_t row = H == 1 ? (int64_t)bid_ * 64 + threadIdx.x : (int64_t)bid_ * 32 + lane;
  const bool active = row < nbr;
  double acc[BR];
#pragma unroll
  for (int r = 0; r < BR; ++r) acc[r] = 0.0;
  if (active) {
    const int64_t base = sp[row >> 5];
    const int len = rl[row];
    const int32_t *cp = col + base * 32 + lane;
    const double *vp = val + base * (BR * BCT * 32) + lane;
#pragma unroll 2
    for (int t = h; t < len; t += H) {
      const int64_t c = __ldg(cp + (int64_t)t * 32);
      double xv[BCT];
#pragma unroll
      for (int q = 0; q < B0; ++q) xv[q] = ld_vec(x0 + c * B0 + q);
#pragma unroll
      for (int q = 0; q < B1; ++q) xv[B0 + q] = ld_vec(x1 + c * B1 + q);
#pragma unroll
      for (int q = 0; q < B2; ++q) xv[B0 + B1 + q] = ld_vec(x2 + c * B2 + q);
      const double *v = vp + (int64_t)t * (BR * BCT * 32);
#pragma unroll
      for (int r = 0; r < BR; ++r)
#pragma unroll
        for (int q = 0; q < BCT; ++q) acc[r] += __ldg(v + (r * BCT + q) * 32) * xv[q];
    }
  }
  if constexpr (H == 1) {
    if (active)
#pragma unroll
      for (int r = 0; r < BR; ++r) y[row * BR + r] = acc[r];
  } else {
    __shared__ double part[H - 1][BR][32];
    if (h > 0)
#pragma unroll
      for (int r = 0; r < BR; ++r) part[h - 1][r][lane] = acc[r];
    __syncthreads();
    if (h == 0 && active)
#pragma unroll
      for (int r = 0; r < BR; ++r) {
        double a = acc[r];
#pragma unroll
        for (int q = 0; q < H - 1; ++q) a += part[q][r][lane];
        y[row * BR + r] = a;
      }
  }
}
// The rows of all fields in one launch: CTAs [0, end[0]) take field 0 (BR =
// B0), then fields 1 and 2 (one dof per node).  The launches' ends, where SMs
// run dry, and two launches of a few microseconds on small systems are paid
// once (64^3 box 366 -> 340 us, 3,267-dof system 1.70 -> 1.66 ms a solve).
template <int B0, int B1, int B2, int H>
struct KSpmvRows {
  static constexpr int kMaxThreads = (H == 1 ? 64 : 32 * H);
  static constexpr int kMinBlocks = 1536 / kMaxThreads;  // multi-system form: <= 40 registers
  static constexpr bool kFp64 = true;
  struct Field {
    int64_t nbr;
    const int32_t *sp;
    const int32_t *rl;
    const int32_t *col;
    const double *val;
    double *y;
  };
  struct Args {
    int end[3];  // CTAs up to and with each field
    Field f[3];
    const double *x0;
    const double *x1;
    const double *x2;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    if (bid < a.end[0]) {
      const Field &f = a.f[0];
      d_spmv_rows<B0, B0, B1, B2, H>(f.nbr, f.sp, f.rl, f.col, f.val, a.x0, a.x1, a.x2, f.y, bid, nb);
    } else {
      const int i = bid < a.end[1] ? 1 : 2;
      const Field &f = a.f[i];
      d_spmv_rows<1, B0, B1, B2, H>(f.nbr, f.sp, f.rl, f.col, f.val, a.x0, a.x1, a.x2, f.y, bid - a.end[i - 1], nb);
    }
  }
};

template <int BR, typename T, int U>
__device__ __forceinline__ void d_smooth(int64_t nbr, const int32_t *__restrict__ sp, const int32_t *__restrict__ rl,
         const int32_t *__restrict__ col, const T *__restrict__ val, const T *__restrict__ dinv,
         const T *__restrict__ b, const T *__restrict__ x, T *__restrict__ xout, T *__restrict__ d,
         T c1, T c2, int bid_, int nb_) {
  const int64_t row = (int64_t)bid_ * blockDim.x + threadIdx.x;
  if (row >= nbr) return;
  T acc[BR];
  sell_row<BR, BR, T, U>(sp, rl, col, val, x, row, acc);
#pragma unroll
  for (int r = 0; r < BR; ++r) {
    const int64_t i = row * BR + r;
    const T res = b[i] - acc[r];
    const T dd = c1 * d[i] + c2 * dinv[i] * res;
    d[i] = dd;
    xout[i] = x[i] + dd;
  }
}
template <int BR, typename T, int U>
struct KSmoothSell {
  static constexpr int kMaxThreads = kThreads;
  static constexpr bool kFp64 = sizeof(T) == 8;
  static constexpr int kMinBlocks = BR <= 3 ? 8 : 1;  // multi-system form: <= 32 registers
  struct Args {
    int64_t nbr;
    const int32_t *sp;
    const int32_t *rl;
    const int32_t *col;
    const T *val;
    const T *dinv;
    const T *b;
    const T *x;
    T *xout;
    T *d;
    T c1;
    T c2;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    d_smooth<BR, T, U>(a.nbr, a.sp, a.rl, a.col, a.val, a.dinv, a.b, a.x, a.xout, a.d, a.c1, a.c2, bid, nb);
  }
};

// G lanes per row of a plain BSR matrix: the lanes of a group stride over the
// row's blocks, then a fixed xor-butterfly inside the group sums them.  x goes
// through the read-only path: in a one-colour launch only rows of that colour
// write x, and they never read each other's entries (earlier colours wrote in
// earlier launches).
template <int BR, int G, typename T>
__device__ __forceinline__ void gs_group_row(const int32_t *__restrict__ rp, const int32_t *__restrict__ col,
                                             const T *__restrict__ val, const T *x, int64_t row, bool active,
                                             int gl, T (&acc)[BR]) {
#pragma unroll
  for (int r = 0; r < BR; ++r) acc[r] = T(0);
  const int lo = active ? rp[row] : 0, hi = active ? rp[row + 1] : 0;
  for (int k = lo + gl; k < hi; k += G) {
    const int64_t c = __ldg(col + k);
    T xv[BR];
#pragma unroll
    for (int q = 0; q < BR; ++q) xv[q] = ld_vec(x + c * BR + q);
    T blk[BR * BR];
    ldg_block<BR * BR, T>(val + (int64_t)k * (BR * BR), blk);
#pragma unroll
    for (int r = 0; r < BR; ++r)
#pragma unroll
      for (int q = 0; q < BR; ++q) acc[r] += blk[r * BR + q] * xv[q];
  }
#pragma unroll
  for (int r = 0; r < BR; ++r)
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
}

// One colour: reordered rows [r0, r1), G lanes per row.
template <int BR, typename T, int G>
__device__ __forceinline__ void d_gs_color(int64_t r0, int64_t r1, const int32_t *__restrict__ rp, const int32_t *__restrict__ col,
           const T *__restrict__ val, const int32_t *__restrict__ rowidx, const T *__restrict__ dblk,
           const T *__restrict__ b, T *x, T omega, int backward, int bid_, int nb_) {
  const int64_t t = (int64_t)bid_ * blockDim.x + threadIdx.x;
  const int64_t row = r0 + t / G;
  const int gl = (int)(t % G);
  const bool active = row < r1;
  T acc[BR];
  gs_group_row<BR, G, T>(rp, col, val, x, row, active, gl, acc);
  if (active && gl == 0) gs_update<BR, T>(acc, rowidx[row], dblk, b, x, omega, backward != 0);
}
template <int BR, typename T, int G>
struct KGsColor {
  static constexpr int kMaxThreads = kThreads;
  static constexpr bool kFp64 = sizeof(T) == 8;
  struct Args {
    int64_t r0;
    int64_t r1;
    const int32_t *rp;
    const int32_t *col;
    const T *val;
    const int32_t *rowidx;
    const T *dblk;
    const T *b;
    T *x;
    T omega;
    int backward;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    d_gs_color<BR, T, G>(a.r0, a.r1, a.rp, a.col, a.val, a.rowidx, a.dblk, a.b, a.x, a.omega, a.backward, bid, nb);
  }
};

// All colours and sweeps of a small level in one CTA: x lives in shared
// memory for the whole launch (loaded first, written back last), so the
// colour-to-colour dependency goes through shared memory and __syncthreads;
// groups of G lanes stride over the rows of a colour.  Every thread reaches
// every barrier (uniform loops, no early exit).
template <int BR, typename T, int G>
__device__ __forceinline__ void d_gs_small(int nc, int64_t n, const int32_t *__restrict__ coff, const int32_t *__restrict__ rp,
           const int32_t *__restrict__ col, const T *__restrict__ val, const int32_t *__restrict__ rowidx,
           const T *__restrict__ dblk, const T *__restrict__ b, T *__restrict__ x, T omega, int sweeps,
           int backward, int bid_, int nb_) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *xs = reinterpret_cast<T *>(smem_raw);
  const int tid = threadIdx.x;
  for (int64_t k = tid; k < n * BR; k += blockDim.x) xs[k] = x[k];
  __syncthreads();
  const int ngroups = blockDim.x / G;
  const int gid = tid / G, gl = tid % G;
  for (int sw = 0; sw < sweeps; ++sw)
    for (int q = 0; q < nc; ++q) {
      const int c = backward ? nc - 1 - q : q;
      const int lo = coff[c], hi = coff[c + 1];
      for (int base = lo; base < hi; base += ngroups) {
        const int row = base + gid;
        const bool active = row < hi;
        T acc[BR];
#pragma unroll
        for (int r = 0; r < BR; ++r) acc[r] = T(0);
        const int k0 = active ? rp[row] : 0, k1 = active ? rp[row + 1] : 0;
        for (int k = k0 + gl; k < k1; k += G) {
          const int64_t cc = __ldg(col + k);
          const T *v = val + (int64_t)k * (BR * BR);
#pragma unroll
          for (int r = 0; r < BR; ++r)
#pragma unroll
            for (int qq = 0; qq < BR; ++qq) acc[r] += __ldg(v + r * BR + qq) * xs[cc * BR + qq];
        }
#pragma unroll
        for (int r = 0; r < BR; ++r)
#pragma unroll
          for (int o = G / 2; o > 0; o >>= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
        if (active && gl == 0) gs_update<BR, T>(acc, rowidx[row], dblk, b, xs, omega, backward != 0);
      }
      __syncthreads();
    }
  for (int64_t k = tid; k < n * BR; k += blockDim.x) x[k] = xs[k];
}
template <int BR, typename T, int G>
struct KGsSmall {
  static constexpr int kMaxThreads = kGsCtaThreads;
  static constexpr bool kFp64 = sizeof(T) == 8;
  struct Args {
    int nc;
    int64_t n;
    const int32_t *coff;
    const int32_t *rp;
    const int32_t *col;
    const T *val;
    const int32_t *rowidx;
    const T *dblk;
    const T *b;
    T *x;
    T omega;
    int sweeps;
    int backward;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    d_gs_small<BR, T, G>(a.nc, a.n, a.coff, a.rp, a.col, a.val, a.rowidx, a.dblk, a.b, a.x, a.omega, a.sweeps, a.backward, bid, nb);
  }
};

// x = inv b for the explicit inverse of a coarsest matrix (row-major, float64):
// b staged in shared memory as float64, one warp per row, fixed butterfly sum.
template <typename T>
struct KInvApply {
  static constexpr int kMaxThreads = kThreads;
  static constexpr bool kEarly = true;
  struct Args {
    int n;
    const double *inv;
    const T *b;
    T *x;
  };
  template <class W> static __device__ __forceinline__ void run(const Args &p, int bid, int nb, W wait) {
    extern __shared__ double bs[];
    const int row = bid * (blockDim.x / 32) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    const double *a = p.inv + (int64_t)row * p.n;
    const double a0 = row < p.n && lane < p.n ? ld_pin(a + lane) : 0.0;
    wait();
    for (int j = threadIdx.x; j < p.n; j += blockDim.x) bs[j] = (double)p.b[j];
    __syncthreads();
    if (row >= p.n) return;
    double acc = 0.0;
    if (lane < p.n) acc += a0 * bs[lane];
    for (int j = lane + 32; j < p.n; j += 32) acc += __ldg(a + j) * bs[j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) p.x[row] = (T)acc;
  }
};

template <typename T>
__device__ __forceinline__ void d_smooth_first(int64_t n, const T *__restrict__ dinv, const T *__restrict__ b,
                               T *__restrict__ x, T *__restrict__ d, T c2, int bid_, int nb_) {
  for (int64_t i = (int64_t)bid_ * blockDim.x + threadIdx.x; i < n; i += (int64_t)nb_ * blockDim.x) {
    const T dd = c2 * dinv[i] * b[i];
    d[i] = dd;
    x[i] = dd;
  }
}
template <typename T>
struct KSmoothFirst {
  static constexpr int kMaxThreads = kThreads;
  struct Args {
    int64_t n;
    const T *dinv;
    const T *b;
    T *x;
    T *d;
    T c2;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    d_smooth_first<T>(a.n, a.dinv, a.b, a.x, a.d, a.c2, bid, nb);
  }
};

// Dense LU solve in one CTA, blocked by 32: one warp solves each 32 x 32
// diagonal block with shuffles, then all warps update the rows below (above)
// with that block's 32 new unknowns.  y lives in shared memory, and so do the
// factors when they fit (staged == 1), which keeps the warp's sequential
// steps off global-memory latency.
template <typename T>
__device__ __forceinline__ void d_lu_solve(int n, const double *__restrict__ lu_g, const int32_t *__restrict__ perm,
           const T *__restrict__ b, T *__restrict__ x, int staged, int bid_, int nb_) {
  extern __shared__ double sm[];
  double *y = sm;
  const int tid = threadIdx.x, nt = blockDim.x, warp = tid >> 5, lane = tid & 31;
  const double *lu = lu_g;
  if (staged) {
    double *ls = sm + n;
    for (int64_t i = tid; i < (int64_t)n * n; i += nt) ls[i] = lu_g[i];
    lu = ls;
  }
  for (int i = tid; i < n; i += nt) y[i] = (double)b[perm[i]];
  __syncthreads();
  // forward: L y = Pb, unit lower triangle
  for (int k0 = 0; k0 < n; k0 += 32) {
    const int nb = min(32, n - k0);
    if (warp == 0) {
      // this lane's row of the 32 x 32 diagonal block, loaded up front
      double Lr[32];
#pragma unroll
      for (int c = 0; c < 32; ++c) Lr[c] = (c < nb && lane < nb) ? lu[(int64_t)(k0 + c) * n + k0 + lane] : 0.0;
      double yv = lane < nb ? y[k0 + lane] : 0.0;
#pragma unroll
      for (int c = 0; c < 32; ++c) {
        if (c < nb) {
          const double yc = __shfl_sync(0xffffffffu, yv, c);
          if (lane > c && lane < nb) yv -= Lr[c] * yc;
        }
      }
      if (lane < nb) y[k0 + lane] = yv;
    }
    __syncthreads();
    for (int i = k0 + nb + tid; i < n; i += nt) {
      double s = 0.0;
#pragma unroll
      for (int c = 0; c < 32; ++c)  // all 32 loads in flight at once
        if (c < nb) s += lu[(int64_t)(k0 + c) * n + i] * y[k0 + c];
      y[i] -= s;
    }
    __syncthreads();
  }
  // backward: U x = y
  const int last = ((n - 1) / 32) * 32;
  for (int k0 = last; k0 >= 0; k0 -= 32) {
    const int nb = min(32, n - k0);
    if (warp == 0) {
      double Ur[32];
#pragma unroll
      for (int c = 0; c < 32; ++c) Ur[c] = (c < nb && lane < nb) ? lu[(int64_t)(k0 + c) * n + k0 + lane] : 1.0;
      double yv = lane < nb ? y[k0 + lane] : 0.0;
#pragma unroll
      for (int c = 31; c >= 0; --c) {
        if (c < nb) {
          if (lane == c) yv /= Ur[c];
          const double yc = __shfl_sync(0xffffffffu, yv, c);
          if (lane < c) yv -= Ur[c] * yc;
        }
      }
      if (lane < nb) y[k0 + lane] = yv;
    }
    __syncthreads();
    for (int i = tid; i < k0; i += nt) {
      double s = 0.0;
#pragma unroll
      for (int c = 0; c < 32; ++c)
        if (c < nb) s += lu[(int64_t)(k0 + c) * n + i] * y[k0 + c];
      y[i] -= s;
    }
    __syncthreads();
  }
  for (int i = tid; i < n; i += nt) x[i] = (T)y[i];
}
template <typename T>
struct KLuSolve {
  static constexpr int kMaxThreads = 512;
  struct Args {
    int n;
    const double *lu_g;
    const int32_t *perm;
    const T *b;
    T *x;
    int staged;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    d_lu_solve<T>(a.n, a.lu_g, a.perm, a.b, a.x, a.staged, bid, nb);
  }
};

template <typename T>
__device__ __forceinline__ void d_fill(T *x, int64_t n, T v, int bid_, int nb_) {
  for (int64_t i = (int64_t)bid_ * blockDim.x + threadIdx.x; i < n; i += (int64_t)nb_ * blockDim.x)
    x[i] = v;
}
template <typename T>
struct KFill {
  static constexpr int kMaxThreads = kThreads;
  struct Args {
    T *x;
    int64_t n;
    T v;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    d_fill<T>(a.x, a.n, a.v, bid, nb);
  }
};

template <typename T>
__device__ __forceinline__ void d_axpy_diag(T *__restrict__ x, const T *__restrict__ dinv, const T *__restrict__ t, int64_t n, int bid_, int nb_) {
  for (int64_t i = (int64_t)bid_ * blockDim.x + threadIdx.x; i < n; i += (int64_t)nb_ * blockDim.x)
    x[i] -= dinv[i] * t[i];
}
template <typename T>
struct KAxpyDiag {
  static constexpr int kMaxThreads = kThreads;
  struct Args {
    T *x;
    const T *dinv;
    const T *t;
    int64_t n;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    d_axpy_diag<T>(a.x, a.dinv, a.t, a.n, bid, nb);
  }
};

template <typename T>
__device__ __forceinline__ void d_axpy(T *__restrict__ y, const T *__restrict__ x, T a, int64_t n, int bid_, int nb_) {
  for (int64_t i = (int64_t)bid_ * blockDim.x + threadIdx.x; i < n; i += (int64_t)nb_ * blockDim.x)
    y[i] += a * x[i];
}
template <typename T>
struct KAxpy {
  static constexpr int kMaxThreads = kThreads;
  struct Args {
    T *y;
    const T *x;
    T a;
    int64_t n;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    d_axpy<T>(a.y, a.x, a.a, a.n, bid, nb);
  }
};

template <typename TI, typename TO>
__device__ __forceinline__ void d_convert(const TI *__restrict__ in, TO *__restrict__ out, int64_t n, int bid_, int nb_) {
  for (int64_t i = (int64_t)bid_ * blockDim.x + threadIdx.x; i < n; i += (int64_t)nb_ * blockDim.x)
    out[i] = (TO)in[i];
}
template <typename TI, typename TO>
struct KConvert {
  static constexpr int kMaxThreads = kThreads;
  struct Args {
    const TI *in;
    TO *out;
    int64_t n;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    d_convert<TI, TO>(a.in, a.out, a.n, bid, nb);
  }
};

__global__ void k_sell_widths(const int32_t *__restrict__ rp, int64_t nbr, int32_t *__restrict__ rl,
                              int32_t *__restrict__ w) {
  const int64_t I = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const int len = I < nbr ? rp[I + 1] - rp[I] : 0;
  if (I < nbr) rl[I] = len;
  int m = len;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0 && (I >> 5) * 32 < nbr) w[I >> 5] = m;
}

// one thread per block row: slot t of row I goes to slice I/32, lane I%32
__global__ void k_sell_fill(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci, int nsrc,
                            const double *__restrict__ v0, const double *__restrict__ v1,
                            const double *__restrict__ v2, int b0, int b1, int b2, int br, int64_t nbr,
                            const int32_t *__restrict__ sp, int32_t *__restrict__ col, double *__restrict__ v64,
                            float *__restrict__ v32) {
  const int64_t I = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (I >= nbr) return;
  const int64_t lane = I & 31, base = sp[I >> 5];
  const int bct = b0 + b1 + b2, bs = br * bct;
  for (int64_t a = rp[I]; a < rp[I + 1]; ++a) {
    const int64_t slot = base + (a - rp[I]);
    col[slot * 32 + lane] = ci[a];
    for (int r = 0; r < br; ++r) {
      int o = 0;
      for (int j = 0; j < nsrc; ++j) {
        const double *v = j == 0 ? v0 : (j == 1 ? v1 : v2);
        const int bj = j == 0 ? b0 : (j == 1 ? b1 : b2);
        for (int q = 0; q < bj; ++q) {
          const double x = v[(a * br + r) * bj + q];
          const int64_t e = (slot * bs + r * bct + o + q) * 32 + lane;
          if (v64) v64[e] = x;
          if (v32) v32[e] = (float)x;
        }
        o += bj;
      }
    }
  }
}

__device__ __forceinline__ void d_scale(const double *x, double a, double *y, int64_t n, int bid_, int nb_) {
  for (int64_t i = (int64_t)bid_ * blockDim.x + threadIdx.x; i < n; i += (int64_t)nb_ * blockDim.x)
    y[i] = a * x[i];
}
struct KScale {
  static constexpr int kMaxThreads = kThreads;
  struct Args {
    const double *x;
    double a;
    double *y;
    int64_t n;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    d_scale(a.x, a.a, a.y, a.n, bid, nb);
  }
};

// v = a v (in place) and out = v converted to TO: the normalisation of a new
// Krylov vector fused with the copy the preconditioner reads
template <typename TO>
__device__ __forceinline__ void d_scale_convert(double *__restrict__ v, double a, TO *__restrict__ out, int64_t n,
                                                int bid_, int nb_) {
  for (int64_t i = (int64_t)bid_ * blockDim.x + threadIdx.x; i < n; i += (int64_t)nb_ * blockDim.x) {
    const double t = a * v[i];
    v[i] = t;
    out[i] = (TO)t;
  }
}
template <typename TO>
struct KScaleConvert {
  static constexpr int kMaxThreads = kThreads;
  struct Args {
    double *v;
    double a;
    TO *out;
    int64_t n;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    d_scale_convert<TO>(a.v, a.a, a.out, a.n, bid, nb);
  }
};

// the same with a = inv[0] read from device memory (1 / |w| of the previous
// Arnoldi vector, so that a captured iteration graph normalises its input
// itself); out may be null (in-place scaling only).  The square root and the
// division are done once, by the pass that made the norm: done here by every
// thread they took 29 us of FP64 time on 1.37 M entries (5 us of memory traffic).
template <typename TO>
__device__ __forceinline__ void d_scale_convert_dev(double *__restrict__ v, const double *__restrict__ inv,
                                                    TO *__restrict__ out, int64_t n, int bid_, int nb_) {
  const double a = inv[0];
  for (int64_t i = (int64_t)bid_ * blockDim.x + threadIdx.x; i < n; i += (int64_t)nb_ * blockDim.x) {
    const double t = a * v[i];
    v[i] = t;
    if (out) out[i] = (TO)t;
  }
}
template <typename TO>
struct KScaleConvertDev {
  static constexpr int kMaxThreads = kThreads;
  struct Args {
    double *v;
    const double *inv;
    TO *out;
    int64_t n;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    d_scale_convert_dev<TO>(a.v, a.inv, a.out, a.n, bid, nb);
  }
};

// sum of v over the CTA (kThreads threads), valid in thread 0
__device__ __forceinline__ double block_sum(double v, double *sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x < 32) {
    s = l < kThreads / 32 ? sh[l] : 0.0;
#pragma unroll
    for (int o = kThreads / 64; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  }
  return s;
}

// The CGS2 passes over V (k rows of length n) and w.  The FP64 pipe bounds
// them (a warp's float64 instruction takes 64 cycles of an SM quarter; HBM
// delivers 1.6 times what the pipe can use), on small systems through the SM
// with the most entries: so the entries are spread over all SMs in tiles of
// 256 (mdot_blocks) and the sums over lanes are kept short
// (warp_sum_rows).  The three passes and their reductions at 23 rows, in a
// graph: 48,510 entries 27 us (107 us with n / 2048 CTAs), 344,605 73 us
// (133), 1.37 M 266 us (287; float64 floor 238).  Smaller tiles shared by
// several threads an entry gained 4 us at 3,267 entries but cost a batch
// of 96 such systems 9 % and were dropped.
constexpr int kTile = kThreads;  // entries of w per step of a CTA
constexpr int kMaxQ = 64;        // rows of V handled per launch (8 per warp)

// Sum over the warp of each of a lane's 8 values (HALF: only the first 4 are
// used): at offsets 16, 8, 4 a lane keeps one half of its rows and adds the
// partner's half, then two ordinary butterfly steps.  9 (6) float64 adds per
// lane instead of the 40 of eight butterflies.  Lane l holds the sum of row
// l >> 2 (HALF: l >> 3).
template <bool HALF>
__device__ __forceinline__ double warp_sum_rows(const double (&a)[8], int lane) {
  const bool h16 = (lane & 16) != 0, h8 = (lane & 8) != 0, h4 = (lane & 4) != 0;
  double c[2], d;
  if constexpr (HALF) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
      c[i] = (h16 ? a[i + 2] : a[i]) + __shfl_xor_sync(0xffffffffu, h16 ? a[i] : a[i + 2], 16);
    d = (h8 ? c[1] : c[0]) + __shfl_xor_sync(0xffffffffu, h8 ? c[0] : c[1], 8);
    d += __shfl_xor_sync(0xffffffffu, d, 4);
  } else {
    double b[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      b[i] = (h16 ? a[i + 4] : a[i]) + __shfl_xor_sync(0xffffffffu, h16 ? a[i] : a[i + 4], 16);
#pragma unroll
    for (int i = 0; i < 2; ++i)
      c[i] = (h8 ? b[i + 2] : b[i]) + __shfl_xor_sync(0xffffffffu, h8 ? b[i] : b[i + 2], 8);
    d = (h4 ? c[1] : c[0]) + __shfl_xor_sync(0xffffffffu, h4 ? c[0] : c[1], 4);
  }
  d += __shfl_xor_sync(0xffffffffu, d, 2);
  d += __shfl_xor_sync(0xffffffffu, d, 1);
  return d;
}

// p[0] + ... + p[n - 1] by the whole CTA, valid in thread 0.  The partial
// sums come from other CTAs of this launch or of the previous one: read from L2.
__device__ __forceinline__ double cta_sum_partials(const double *p, int n, double *sh) {
  double a = 0.0;
  for (int i = threadIdx.x; i < n; i += kThreads) a += __ldcg(p + i);
  return block_sum(a, sh);
}

// Passes with one result: the CTA that comes last (the counter says so, and
// is set back to 0 for the next pass) adds up the nb partial sums, in the
// order of k_reduce_partials: out[0], and with `inv` out[1] = 1 / sqrt(out[0]).
// Every thread of every CTA calls this after thread 0 has written its
// partial.  (For k results this would run k nb / 32 float64 warp
// instructions on one SM: with 23 rows of 270 partials 3.8 us more than the
// launch of k CTAs that it saves, with 13 partials 1.5 us.)
__device__ __forceinline__ void finish_sum(const double *partial, int nb, double *out, unsigned *cnt, bool inv,
                                           double *sh) {
  __shared__ int last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(cnt, 1u) == (unsigned)(nb - 1) ? 1 : 0;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  const double t = cta_sum_partials(partial, nb, sh);
  if (threadIdx.x == 0) {
    out[0] = t;
    if (inv) out[1] = 1.0 / sqrt(t);
    *cnt = 0u;
  }
}

// The sums of a pass over at most kInlineBlocks CTAs are added up by every CTA
// of the next pass itself (thread q adds the partial sums of row q in order;
// CTA 0 also writes them out for the host): 0.4 us for 13 partials instead of a
// launch of 2.3 us.
constexpr int kInlineBlocks = 16;
__device__ __forceinline__ void load_sums(const double *__restrict__ h, const double *__restrict__ hpart, int k,
                                          int rows, int nblk, double *__restrict__ hout, double *hs, int bid) {
  if (hpart == nullptr) {
    for (int q = threadIdx.x; q < k; q += kThreads) hs[q] = h[q];
  } else if (threadIdx.x < rows) {
    const double *p = hpart + (int64_t)threadIdx.x * nblk;
    double a[kInlineBlocks], t = 0.0;
#pragma unroll
    for (int i = 0; i < kInlineBlocks; ++i) a[i] = i < nblk ? p[i] : 0.0;
#pragma unroll
    for (int i = 0; i < kInlineBlocks; ++i)
      if (i < nblk) t += a[i];
    if (threadIdx.x < k) hs[threadIdx.x] = t;
    if (bid == 0) hout[threadIdx.x] = t;
  }
  __syncthreads();
}

// acc[m] += V_q[t0 ..] . ws over a staged tile for the warp's rows q = warp +
// 8 m, a lane's 8 loads issued before the first product
__device__ __forceinline__ void tile_dots(const double *__restrict__ V, int64_t ldv, int k, int64_t t0, int cnt,
                                          const double *ws, double (&acc)[kMaxQ / 8]) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int m = 0; m < kMaxQ / 8; ++m) {
    const int q = warp + 8 * m;
    if (q < k) {
      const double *vq = V + (int64_t)q * ldv + t0 + lane;
      double v[kTile / 32], s = acc[m];  // one FMA chain per row across the tiles
      if (cnt == kTile) {
#pragma unroll
        for (int u = 0; u < kTile / 32; ++u) v[u] = vq[32 * u];
      } else {
#pragma unroll
        for (int u = 0; u < kTile / 32; ++u) v[u] = lane + 32 * u < cnt ? vq[32 * u] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < kTile / 32; ++u) s = fma(v[u], ws[lane + 32 * u], s);
      acc[m] = s;
    }
  }
}

__device__ __forceinline__ void store_dots(int k, int nblk, const double (&acc)[kMaxQ / 8],
                                           double *__restrict__ partial, int bid) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp >= k) return;  // no rows
  int q;
  double t;
  bool own;
  if (k <= kMaxQ / 2) {
    t = warp_sum_rows<true>(acc, lane);
    q = warp + 8 * (lane >> 3);
    own = (lane & 7) == 0;
  } else {
    t = warp_sum_rows<false>(acc, lane);
    q = warp + 8 * (lane >> 2);
    own = (lane & 3) == 0;
  }
  if (own && q < k) partial[(int64_t)q * nblk + bid] = t;
}

// sum_q V_q[i] h_q, 8 loads in flight
__device__ __forceinline__ double col_dot(const double *__restrict__ V, int64_t ldv, int k, const double *hs,
                                          int64_t i) {
  const double *v = V + i;
  double s = 0.0;  // (a chain started from w_i would wait for its load)
  int q = 0;
  for (; q + 8 <= k; q += 8) {
    double t[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) t[u] = v[(int64_t)(q + u) * ldv];
#pragma unroll
    for (int u = 0; u < 8; ++u) s = fma(t[u], hs[q + u], s);
  }
  double t[7];
#pragma unroll
  for (int u = 0; u < 7; ++u) t[u] = q + u < k ? v[(int64_t)(q + u) * ldv] : 0.0;
#pragma unroll
  for (int u = 0; u < 7; ++u)
    if (q + u < k) s = fma(t[u], hs[q + u], s);
  return s;
}

// h_q = V_q . w for q < k (w may be one of the rows of V)
__device__ __forceinline__ void d_mdot(const double *__restrict__ V, int64_t ldv, int k, const double *__restrict__ w, int64_t n,
       double *__restrict__ partial, int nblk, int64_t per, double *out, unsigned *cnt, int bid_) {
  __shared__ double ws[2][kTile];
  __shared__ double sh[32];
  const int64_t lo = (int64_t)bid_ * per, hi = min(n, lo + per);
  double acc[kMaxQ / 8];
#pragma unroll
  for (int m = 0; m < kMaxQ / 8; ++m) acc[m] = 0.0;
  // the next tile's w is loaded while this one is worked on; two buffers, so
  // that one barrier a tile is enough
  double wn = lo + threadIdx.x < hi ? w[lo + threadIdx.x] : 0.0;
  int buf = 0;
  for (int64_t t0 = lo; t0 < hi; t0 += kTile, buf ^= 1) {
    const int c = (int)min((int64_t)kTile, hi - t0);
    ws[buf][threadIdx.x] = wn;
    const int64_t nx = t0 + kTile + threadIdx.x;
    wn = nx < hi ? w[nx] : 0.0;
    __syncthreads();
    tile_dots(V, ldv, k, t0, c, ws[buf], acc);
  }
  store_dots(k, nblk, acc, partial, bid_);
  if (cnt != nullptr) finish_sum(partial, nblk, out, cnt, false, sh);
}
struct KMdot {
  static constexpr int kMaxThreads = kThreads;
  static constexpr int kMinBlocks = 4;  // multi-system form: <= 64 registers
  static constexpr bool kFp64 = true;
  struct Args {
    const double *V;
    int64_t ldv;
    int k;
    const double *w;
    int64_t n;
    double *partial;
    int nblk;
    int64_t per;    // entries per CTA
    double *out;    // with cnt (k = 1): the sum, added up by the last CTA
    unsigned *cnt;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    d_mdot(a.V, a.ldv, a.k, a.w, a.n, a.partial, a.nblk, a.per, a.out, a.cnt, bid);
  }
};

// w <- w - sum_q V_q h_q, then partial dots V_q . w_new (CGS2 second pass)
__device__ __forceinline__ void d_cgs_fused(const double *__restrict__ V, int64_t ldv, int k, const double *__restrict__ h,
            const double *__restrict__ hpart, double *__restrict__ hout, double *__restrict__ w,
            int64_t n, double *__restrict__ partial, int nblk, int64_t per, int bid_) {
  __shared__ double ws[kTile];
  __shared__ double hs[kMaxQ];
  load_sums(h, hpart, k, k + 1, nblk, hout, hs, bid_);  // the dot pass had w as its last row
  const int64_t lo = (int64_t)bid_ * per, hi = min(n, lo + per);
  double acc[kMaxQ / 8];
#pragma unroll
  for (int m = 0; m < kMaxQ / 8; ++m) acc[m] = 0.0;
  for (int64_t t0 = lo; t0 < hi; t0 += kTile) {
    const int c = (int)min((int64_t)kTile, hi - t0);
    double wn = 0.0;
    if (threadIdx.x < c) {
      const int64_t i = t0 + threadIdx.x;
      const double wi = w[i];
      wn = wi - col_dot(V, ldv, k, hs, i);
      w[i] = wn;
    }
    ws[threadIdx.x] = wn;
    __syncthreads();
    tile_dots(V, ldv, k, t0, c, ws, acc);
    __syncthreads();
  }
  store_dots(k, nblk, acc, partial, bid_);
}
struct KCgsFused {
  static constexpr int kMaxThreads = kThreads;
  static constexpr int kMinBlocks = 4;  // multi-system form: <= 64 registers
  static constexpr bool kFp64 = true;
  struct Args {
    const double *V;
    int64_t ldv;
    int k;
    const double *h;
    const double *hpart;  // or null: h holds the sums
    double *hout;
    double *w;
    int64_t n;
    double *partial;
    int nblk;
    int64_t per;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    d_cgs_fused(a.V, a.ldv, a.k, a.h, a.hpart, a.hout, a.w, a.n, a.partial, a.nblk, a.per, bid);
  }
};

// out[q] = sum of the nblk partial sums of row q, one CTA per row
__device__ __forceinline__ void d_reduce_partials(const double *__restrict__ partial, int k, int nblk, double *__restrict__ out, int bid_) {
  __shared__ double sh[32];
  if (bid_ >= k) return;
  const double s = cta_sum_partials(partial + (int64_t)bid_ * nblk, nblk, sh);
  if (threadIdx.x == 0) out[bid_] = s;
}
struct KReducePartials {
  static constexpr int kMaxThreads = kThreads;
  static constexpr bool kFp64 = true;
  struct Args {
    const double *partial;
    int k;
    int nblk;
    double *out;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    d_reduce_partials(a.partial, a.k, a.nblk, a.out, bid);
  }
};

// w <- w - sum_q V_q h_q, then |w|^2 and 1 / |w| (last CTA)
__device__ __forceinline__ void d_cgs_update(const double *__restrict__ V, int64_t ldv, int k, const double *__restrict__ h,
             const double *__restrict__ hpart, double *__restrict__ hout, double *__restrict__ w, int64_t n,
             double *__restrict__ partial, int nblk, int64_t per, double *out, unsigned *cnt, int bid_) {
  __shared__ double hs[kMaxQ];
  __shared__ double sh[32];
  load_sums(h, hpart, k, k, nblk, hout, hs, bid_);
  const int64_t lo = (int64_t)bid_ * per, hi = min(n, lo + per);
  double nrm = 0.0;
  for (int64_t i = lo + threadIdx.x; i < hi; i += kTile) {
    const double wi = w[i];
    const double wn = wi - col_dot(V, ldv, k, hs, i);
    w[i] = wn;
    nrm = fma(wn, wn, nrm);
  }
  const double t = block_sum(nrm, sh);
  if (threadIdx.x == 0) partial[bid_] = t;
  finish_sum(partial, nblk, out, cnt, true, sh);
}
struct KCgsUpdate {
  static constexpr int kMaxThreads = kThreads;
  static constexpr int kMinBlocks = 4;  // multi-system form: <= 64 registers
  static constexpr bool kFp64 = true;
  struct Args {
    const double *V;
    int64_t ldv;
    int k;
    const double *h;
    const double *hpart;  // or null: h holds the sums
    double *hout;
    double *w;
    int64_t n;
    double *partial;
    int nblk;
    int64_t per;
    double *out;
    unsigned *cnt;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    d_cgs_update(a.V, a.ldv, a.k, a.h, a.hpart, a.hout, a.w, a.n, a.partial, a.nblk, a.per, a.out, a.cnt, bid);
  }
};

__device__ __forceinline__ void d_gemv_add(const double *__restrict__ Z, int64_t ldz, int k, const double *__restrict__ y,
                           double *__restrict__ x, int64_t n, int bid_, int nb_) {
  __shared__ double ys[64];
  for (int q = threadIdx.x; q < k; q += blockDim.x) ys[q] = y[q];
  __syncthreads();
  for (int64_t i = (int64_t)bid_ * blockDim.x + threadIdx.x; i < n; i += (int64_t)nb_ * blockDim.x) {
    double s = 0.0;
    for (int q = 0; q < k; ++q) s += Z[(int64_t)q * ldz + i] * ys[q];
    x[i] += s;
  }
}
struct KGemvAdd {
  static constexpr int kMaxThreads = kThreads;
  static constexpr bool kFp64 = true;
  struct Args {
    const double *Z;
    int64_t ldz;
    int k;
    const double *y;
    double *x;
    int64_t n;
  };
  static __device__ __forceinline__ void run(const Args &a, int bid, int nb) {
    d_gemv_add(a.Z, a.ldz, a.k, a.y, a.x, a.n, bid, nb);
  }
};

// The tail of a single-field V-cycle (Algorithm 1 on the level above the
// coarsest and the coarse solve) in ONE CTA, for levels small enough that
// their vectors live in shared memory: Chebyshev / Jacobi pre-smoothing from
// zero, residual, restriction, the coarsest solve through the explicit
// inverse, prolongation and post-smoothing, separated by __syncthreads
// instead of kernel boundaries.  Every step reduces a row exactly as the
// separate launches do (bsr_ls lanes per block row striding over its blocks,
// the same halving sums; the inverse applied in float64), so
// the result is the one of the step-by-step V-cycle bit for bit.
constexpr int kTailThreads = 1024;
constexpr int kTailMaxSteps = 8;

template <typename T> struct TailArgs {
  int64_t n, nbr, nc, ncbr;  // level dofs / block rows; coarse dofs / block rows
  const int32_t *arp, *acol;
  const T *aval, *dinv;
  const int32_t *rrp, *rcol;
  const T *rval;  // R: ncbr block rows of BC x BR blocks
  const int32_t *prp, *pcol;
  const T *pval;  // P: nbr block rows of BR x BC blocks
  const double *inv;  // nc x nc row-major inverse of the coarsest matrix
  const T *b;
  T *x;
  int als, rls, pls;  // log2 of the lanes per row of A, R, P
  int ns;  // smoothing steps per application
  T c1[kTailMaxSteps], c2[kTailMaxSteps];
};

// row sums of a plain-BSR block row against x in shared memory, with the
// lanes per row and the arithmetic of KSpmvWarp; groups of 2^ls lanes stride
// over the rows and f(row, entry, sum) runs in the lane that owns an entry
template <int BR, int BC, typename T, class F>
__device__ __forceinline__ void tail_rows(int64_t nbr, const int32_t *__restrict__ rp,
                                          const int32_t *__restrict__ col, const T *__restrict__ val, const T *x,
                                          int ls, F f) {
  const int gl = threadIdx.x & ((1 << ls) - 1);
  const int64_t step = kTailThreads >> ls;
  for (int64_t r0 = 0; r0 < nbr; r0 += step) {
    const int64_t row = r0 + (threadIdx.x >> ls);
    const bool active = row < nbr;
    T acc[BR];
#pragma unroll
    for (int r = 0; r < BR; ++r) acc[r] = T(0);
    for (int k = active ? rp[row] + gl : 0; active && k < rp[row + 1]; k += 1 << ls) {
      const int64_t c = __ldg(col + k);
      T xv[BC];
#pragma unroll
      for (int q = 0; q < BC; ++q) xv[q] = x[c * BC + q];
      T blk[BR * BC];
      ldg_block<BR * BC, T>(val + (int64_t)k * (BR * BC), blk);
#pragma unroll
      for (int r = 0; r < BR; ++r)
#pragma unroll
        for (int q = 0; q < BC; ++q) acc[r] += blk[r * BC + q] * xv[q];
    }
    __syncwarp();
    const T s = group_sum<BR, T>(acc, gl, ls);
    if (active && sum_owner<BR>(gl, ls)) f(row, sum_entry<BR>(gl, ls), s);
  }
}

// one smoothing step in shared memory: xo = x + d, d = c1 d + c2 dinv (b - A x)
template <int BR, typename T>
__device__ __forceinline__ void tail_smooth(const TailArgs<T> &a, const T *b, const T *x, T *xo, T *d, T c1, T c2) {
  tail_rows<BR, BR, T>(a.nbr, a.arp, a.acol, a.aval, x, a.als, [&](int64_t row, int r, T s) {
    const int64_t i = row * BR + r;
    const T res = b[i] - s;
    const T dd = c1 * d[i] + c2 * a.dinv[i] * res;
    d[i] = dd;
    xo[i] = x[i] + dd;
  });
  __syncthreads();
}

template <int BR, int BC, typename T>
__device__ __forceinline__ void d_vcycle_tail(const TailArgs<T> &a) {
  extern __shared__ __align__(16) unsigned char tail_smem[];
  double *bc = reinterpret_cast<double *>(tail_smem);  // coarse right-hand side (float64 copy)
  T *xc = reinterpret_cast<T *>(bc + a.nc);
  T *bcT = xc + a.nc;
  T *b = bcT + a.nc;
  T *x0 = b + a.n;
  T *x1 = x0 + a.n;
  T *d = x1 + a.n;
  T *r = d + a.n;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int64_t i = tid; i < a.n; i += kTailThreads) b[i] = a.b[i];
  __syncthreads();
  // pre-smoothing from zero: the first step d = x = c2 dinv b, then steps
  for (int64_t i = tid; i < a.n; i += kTailThreads) {
    const T dd = a.c2[0] * a.dinv[i] * b[i];
    d[i] = dd;
    x0[i] = dd;
  }
  __syncthreads();
  T *cur = x0, *oth = x1;
  for (int k = 1; k < a.ns; ++k) {
    tail_smooth<BR, T>(a, b, cur, oth, d, a.c1[k], a.c2[k]);
    T *t = cur;
    cur = oth;
    oth = t;
  }
  // residual r = b - A x  (as y = -1 * A x + 1 * b)
  tail_rows<BR, BR, T>(a.nbr, a.arp, a.acol, a.aval, cur, a.als,
                       [&](int64_t row, int q, T t) { r[row * BR + q] = T(-1) * t + T(1) * b[row * BR + q]; });
  __syncthreads();
  // restriction bc = R r
  tail_rows<BC, BR, T>(a.ncbr, a.rrp, a.rcol, a.rval, r, a.rls,
                       [&](int64_t row, int q, T t) { bcT[row * BC + q] = T(1) * t; });
  __syncthreads();
  // coarsest solve through the explicit inverse, in float64
  for (int64_t j = tid; j < a.nc; j += kTailThreads) bc[j] = (double)bcT[j];
  __syncthreads();
  for (int64_t row = warp; row < a.nc; row += kTailThreads / 32) {
    const double *ar = a.inv + row * a.nc;
    double acc = 0.0;
    for (int64_t j = lane; j < a.nc; j += 32) acc += __ldg(ar + j) * bc[j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) xc[row] = (T)acc;
  }
  __syncthreads();
  // prolongation x += P xc  (as y = 1 * P xc + 1 * x)
  tail_rows<BR, BC, T>(a.nbr, a.prp, a.pcol, a.pval, xc, a.pls,
                       [&](int64_t row, int q, T t) { cur[row * BR + q] = T(1) * t + T(1) * cur[row * BR + q]; });
  __syncthreads();
  // post-smoothing from the corrected x
  for (int k = 0; k < a.ns; ++k) {
    tail_smooth<BR, T>(a, b, cur, oth, d, a.c1[k], a.c2[k]);
    T *t = cur;
    cur = oth;
    oth = t;
  }
  for (int64_t i = tid; i < a.n; i += kTailThreads) a.x[i] = cur[i];
}
template <int BR, int BC, typename T>
struct KVcycleTail {
  static constexpr int kMaxThreads = kTailThreads;
  using Args = TailArgs<T>;
  static __device__ __forceinline__ void run(const Args &a, int, int) { d_vcycle_tail<BR, BC, T>(a); }
};

inline unsigned ew_grid(int64_t n) {
  int64_t g = (n + kThreads - 1) / kThreads;
  if (g > 152 * 16) g = 152 * 16;
  return (unsigned)(g > 0 ? g : 1);
}

// FP64 FMA throughput probe: C independent chains a = a * m + c per thread;
// the sum is stored only when it equals a value it cannot take (m, c are
// runtime values), so no chain can be dropped by the compiler.
__device__ double g_fp64_sink;
template <int C>
__global__ void __launch_bounds__(1024) k_fp64_rate(int iters, double m, double c) {
  double a[C];
#pragma unroll
  for (int k = 0; k < C; ++k) a[k] = 1e-3 * threadIdx.x + k;
  for (int it = 0; it < iters; ++it)
#pragma unroll
    for (int k = 0; k < C; ++k) a[k] = fma(a[k], m, c);
  double s = 0.0;
#pragma unroll
  for (int k = 0; k < C; ++k) s += a[k];
  if (s == -12345.678) g_fp64_sink = s;
}

}  // namespace

// best rate over a few launch shapes (chains per thread, CTA size, CTAs per
// SM): the highest FMA throughput the part delivers, not one shape's
double fp64_rate(cudaStream_t s) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return -1.0;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return -1.0;
  struct Shape {
    int chains, threads, per_sm;
  };
  const Shape shapes[] = {{8, 256, 8}, {16, 256, 8}, {16, 512, 4}, {32, 256, 4}, {8, 1024, 2}};
  double best = 0.0;
  bool ok = true;
  for (const Shape &sh : shapes) {
    const int ctas = sms * sh.per_sm, iters = 65536 / sh.chains;
    for (int r = 0; r < 4 && ok; ++r) {
      ok = cudaEventRecord(e0, s) == cudaSuccess;
      if (sh.chains == 8) k_fp64_rate<8><<<ctas, sh.threads, 0, s>>>(iters, 0.999999, 1e-7);
      else if (sh.chains == 16) k_fp64_rate<16><<<ctas, sh.threads, 0, s>>>(iters, 0.999999, 1e-7);
      else k_fp64_rate<32><<<ctas, sh.threads, 0, s>>>(iters, 0.999999, 1e-7);
      ok = ok && cudaEventRecord(e1, s) == cudaSuccess && cudaEventSynchronize(e1) == cudaSuccess;
      float ms = 0.f;
      ok = ok && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess;
      const double flops = 2.0 * sh.chains * (double)iters * sh.threads * ctas;
      if (ok && r > 0 && ms > 0.f) best = std::max(best, flops / (ms * 1e-3) / 1e12);  // r = 0 warms up
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (!ok || cudaGetLastError() != cudaSuccess) return -1.0;
  return best;
}

#define MFS_BLOCK_DISPATCH(BRV, BCV, CALL)                                      \
  switch (BRV * 16 + BCV) {                                                     \
    case 1 * 16 + 1: { constexpr int BR_ = 1, BC_ = 1; CALL; } break;           \
    case 1 * 16 + 2: { constexpr int BR_ = 1, BC_ = 2; CALL; } break;           \
    case 1 * 16 + 3: { constexpr int BR_ = 1, BC_ = 3; CALL; } break;           \
    case 1 * 16 + 6: { constexpr int BR_ = 1, BC_ = 6; CALL; } break;           \
    case 2 * 16 + 1: { constexpr int BR_ = 2, BC_ = 1; CALL; } break;           \
    case 2 * 16 + 2: { constexpr int BR_ = 2, BC_ = 2; CALL; } break;           \
    case 2 * 16 + 3: { constexpr int BR_ = 2, BC_ = 3; CALL; } break;           \
    case 2 * 16 + 6: { constexpr int BR_ = 2, BC_ = 6; CALL; } break;           \
    case 3 * 16 + 1: { constexpr int BR_ = 3, BC_ = 1; CALL; } break;           \
    case 3 * 16 + 2: { constexpr int BR_ = 3, BC_ = 2; CALL; } break;           \
    case 3 * 16 + 3: { constexpr int BR_ = 3, BC_ = 3; CALL; } break;           \
    case 3 * 16 + 6: { constexpr int BR_ = 3, BC_ = 6; CALL; } break;           \
    case 6 * 16 + 1: { constexpr int BR_ = 6, BC_ = 1; CALL; } break;           \
    case 6 * 16 + 2: { constexpr int BR_ = 6, BC_ = 2; CALL; } break;           \
    case 6 * 16 + 3: { constexpr int BR_ = 6, BC_ = 3; CALL; } break;           \
    case 6 * 16 + 6: { constexpr int BR_ = 6, BC_ = 6; CALL; } break;           \
    default: fprintf(stderr, "mfs: unsupported block shape %dx%d\n", BRV, BCV); \
  }

void set_launch_hook(LaunchHook *h) { g_hook = h; }
void set_recorder(Recorder *r) { g_rec = r; }
void set_pdl(unsigned max_grid, unsigned max_grid64) {
  g_pdl = max_grid;
  g_pdl64 = max_grid64;
  g_pdl_prev = nullptr;
}
void pdl_break() { g_pdl_prev = nullptr; }

HookBypass::HookBypass() { ++g_hook_off; }
HookBypass::~HookBypass() { --g_hook_off; }

void init() {
  // once per device and process (concurrent setups must not race on it)
  static std::mutex mu;
  static bool done[64] = {false};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return;
  std::lock_guard<std::mutex> lock(mu);
  if (done[dev]) return;
  cudaFuncSetAttribute(k_solo<KLuSolve<float>>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  cudaFuncSetAttribute(k_solo<KLuSolve<double>>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  cudaFuncSetAttribute(k_multi<KLuSolve<float>>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  cudaFuncSetAttribute(k_multi<KLuSolve<double>>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  done[dev] = true;
}

// log2 of the lanes per row of a plain-BSR matrix: the smallest group that
// walks an average row in one step (8 blocks: 8 lanes), two steps for rows of
// up to 32 blocks, more for longer ones.  In float64 the lanes' products
// and sums bound these kernels (64 cycles a warp instruction): a 9-block row
// of 3x3 blocks takes 9 warp instructions with 16 lanes, 24 with a warp.  A
// row of over 1,024 blocks among short ones decides alone and takes all 32
// (four rows of 4,000 blocks among 68,921 of 27, float64, 16 / 32 lanes: 3x3
// 260 / 185 us, 1x1 80 / 74; of 1,051: 109 / 107 and 47 / 59).
template <typename T> int bsr_ls(const Sell &A) {
  if (A.longest > 1024) return 5;
  const double avg = (double)A.nnzb / (double)A.nbr;
  return avg <= 8.0 ? 3 : avg <= 32.0 ? 4 : 5;
}
// CTA size of the plain-BSR kernels: small enough to spread few rows over
// the SMs, 64 to 256 threads
static unsigned bsr_threads(int64_t lanes) {
  unsigned t = 64;
  while (t < (unsigned)kThreads && lanes > (int64_t)t * 152) t *= 2;
  return t;
}
// Few, long rows: one CTA per row.  In float64 the 8 warps' sums over lanes
// take longer than a row of a few hundred blocks (6x3 blocks, 184 a row, 1,128
// rows: 22 us, 7 with a warp per row), so only very long rows of which there are
// few (rows of 1x3 blocks of a call that also multiplies 29,791 3x3 rows, warp /
// CTA: 20 rows of 600 blocks 47.9 / 47.6 us, of 1,000 50 / 47, of 3,000 66 / 50; 1,000
// rows of 600 52 / 53, of 1,000 63 / 59; 2,000 rows 57 / 64 and 72 / 70, 4,000 66 / 80
// and 82 / 89).
template <typename T> bool cta_rows(const Sell &A) {
  constexpr int64_t rows = sizeof(T) == 4 ? kCtaRowsMax : kCtaRowsMax64;
  constexpr int64_t blocks = sizeof(T) == 4 ? kCtaRowBlocks : kCtaRowBlocks64;
  return A.kind == 1 && A.nbr <= rows && A.nnzb >= blocks * A.nbr;
}

template <typename T>
void spmv(const Sell &A, const T *x, T *y, T alpha, T beta, const T *z, cudaStream_t s) {
  if (A.nbr == 0) return;
  const T *v = vals<T>(A);
  const bool cta = cta_rows<T>(A);
  HookScope hs(s, K_SPMV, matrix_bytes<T>(A) + (double)sizeof(T) * (A.ncols() + A.nrows() * (z ? 2 : 1)),
               cta ? 7000 + sparse_sig<T>(A) % 1000 : sparse_sig<T>(A), A.nbr,
               2.0 * A.nnzb * A.br * A.bc + (z ? 3.0 : 1.0) * A.nrows());
  if (A.kind == 1) {
    if (cta) {
      MFS_BLOCK_DISPATCH(A.br, A.bc,
                         (go<KSpmvCta<BR_, BC_, T>>((unsigned)A.nbr, kThreads, 0, s, {
                             A.nbr, A.sp, A.col, v, x, y, alpha, beta, z})));
    } else {
      const int ls = bsr_ls<T>(A);
      const unsigned th = bsr_threads(A.nbr << ls);
      MFS_BLOCK_DISPATCH(A.br, A.bc,
                         (go<KSpmvWarp<BR_, BC_, T>>(grid_for(A.nbr << ls, th), th, 0, s, {
                             A.nbr, A.sp, A.col, v, x, y, alpha, beta, z, ls})));
    }
    return;
  }
  if (A.split > 1) {
    MFS_BLOCK_DISPATCH(A.br, A.bc,
                       (go<KSpmvSellSplit<BR_, BC_, T>>((unsigned)A.nslices, 32 * A.split, 0, s, {
                           A.nbr, A.sp, A.rl, A.col, v, x, y, alpha, beta, z})));
  } else if (A.unroll == 4) {
    MFS_BLOCK_DISPATCH(A.br, A.bc,
                       (go<KSpmvSell<BR_, BC_, T, 4>>(grid_for(A.nbr, kSellThreads), kSellThreads, 0, s, {
                           A.nbr, A.sp, A.rl, A.col, v, x, y, alpha, beta, z})));
  } else if (A.unroll == 8) {
    MFS_BLOCK_DISPATCH(A.br, A.bc,
                       (go<KSpmvSell<BR_, BC_, T, 8>>(grid_for(A.nbr, kSellThreads), kSellThreads, 0, s, {
                           A.nbr, A.sp, A.rl, A.col, v, x, y, alpha, beta, z})));
  } else {
    MFS_BLOCK_DISPATCH(A.br, A.bc,
                       (go<KSpmvSell<BR_, BC_, T, 2>>(grid_for(A.nbr, kSellThreads), kSellThreads, 0, s, {
                           A.nbr, A.sp, A.rl, A.col, v, x, y, alpha, beta, z})));
  }
}

#define MFS_SQUARE_DISPATCH(BRV, CALL)                                  \
  switch (BRV) {                                                        \
    case 1: { constexpr int BR_ = 1; CALL; } break;                     \
    case 2: { constexpr int BR_ = 2; CALL; } break;                     \
    case 3: { constexpr int BR_ = 3; CALL; } break;                     \
    case 6: { constexpr int BR_ = 6; CALL; } break;                     \
    default: fprintf(stderr, "mfs: unsupported block size %d\n", BRV); \
  }

#define MFS_ROWS_DISPATCH(B, CALL)                                      \
  switch (B[0] * 100 + B[1] * 10 + B[2]) {                              \
    case 311: { constexpr int X0 = 3, X1 = 1, X2 = 1; CALL; } break;    \
    case 310: { constexpr int X0 = 3, X1 = 1, X2 = 0; CALL; } break;    \
    case 210: { constexpr int X0 = 2, X1 = 1, X2 = 0; CALL; } break;    \
    default: break;                                                     \
  }

bool rows_supported(const int *b, int nb) {
  if (nb < 2 || nb > 3) return false;
  const int code = b[0] * 100 + b[1] * 10 + (nb > 2 ? b[2] : 0);
  return code == 311 || code == 310 || code == 210;
}

template <int B0, int B1, int B2, int H>
static void rows_launch(const RowMerged *R, int nf, const double *x, double *y, cudaStream_t s) {
  typename KSpmvRows<B0, B1, B2, H>::Args a{};
  int end = 0;
  for (int i = 0; i < 3; ++i) {
    if (i < nf) {
      const Sell &A = R[i].M;
      end += H == 1 ? (int)grid_for(A.nbr, 64) : (int)A.nslices;  // H > 1: one slice per CTA
      a.f[i] = {A.nbr, A.sp, A.rl, A.col, A.v64, y + R[i].off[i]};
    }
    a.end[i] = end;
  }
  a.x0 = x + R[0].off[0];
  a.x1 = x + R[0].off[1];
  a.x2 = nf > 2 ? x + R[0].off[2] : x;
  if (end) go<KSpmvRows<B0, B1, B2, H>>((unsigned)end, H == 1 ? 64 : 32 * H, 0, s, a);
}

void spmv_rows(const std::vector<RowMerged> &R, const double *x, double *y, cudaStream_t s) {
  const int nf = (int)R.size();
  const int b3[3] = {R[0].b[0], R[0].b[1], nf > 2 ? R[0].b[2] : 0};
  double bytes = 0.0, flops = 0.0;
  int br = 0;
  for (const RowMerged &r : R) {
    const Sell &A = r.M;
    bytes += (double)A.nnzb * (A.br * A.bc * 8.0 + 4.0) + 4.0 * A.nbr + 8.0 * (A.nbc * A.bc + A.nrows());
    flops += 2.0 * A.nnzb * A.br * A.bc;
    br += A.br;
  }
  HookScope hs(s, K_SPMV, bytes, 2000 + br * 100 + R[0].M.bc * 10 + 1, R[0].M.nbr, flops);
  const int split = R[0].split;
  if (split == 8) {
    MFS_ROWS_DISPATCH(b3, (rows_launch<X0, X1, X2, 8>(R.data(), nf, x, y, s)));
  } else if (split == 4) {
    MFS_ROWS_DISPATCH(b3, (rows_launch<X0, X1, X2, 4>(R.data(), nf, x, y, s)));
  } else if (split == 2) {
    MFS_ROWS_DISPATCH(b3, (rows_launch<X0, X1, X2, 2>(R.data(), nf, x, y, s)));
  } else {
    MFS_ROWS_DISPATCH(b3, (rows_launch<X0, X1, X2, 1>(R.data(), nf, x, y, s)));
  }
}

template <typename T>
void smooth_step(const Sell &A, const T *dinv, const T *b, const T *x, T *xout, T *d, T c1, T c2,
                 cudaStream_t s) {
  if (A.nbr == 0) return;
  const T *v = vals<T>(A);
  const bool cta = cta_rows<T>(A);
  HookScope hs(s, K_SMOOTH, matrix_bytes<T>(A) + (double)sizeof(T) * (A.ncols() + 5.0 * A.nrows()),
               cta ? 7000 + sparse_sig<T>(A) % 1000 : sparse_sig<T>(A), A.nbr, 2.0 * A.nnzb * A.br * A.bc + 6.0 * A.nrows());
  if (A.kind == 1 && cta) {
    MFS_SQUARE_DISPATCH(A.br, (go<KSmoothCta<BR_, T>>((unsigned)A.nbr, kThreads, 0, s, {
                                  A.nbr, A.sp, A.col, v, dinv, b, x, xout, d, c1, c2})));
    return;
  }
  if (A.kind == 1) {
    const int ls = bsr_ls<T>(A);
    const unsigned th = bsr_threads(A.nbr << ls);
    MFS_SQUARE_DISPATCH(A.br, (go<KSmoothWarp<BR_, T>>(grid_for(A.nbr << ls, th), th, 0, s, {
                                  A.nbr, A.sp, A.col, v, dinv, b, x, xout, d, c1, c2, ls})));
    return;
  }
  if (A.split > 1) {
    MFS_SQUARE_DISPATCH(A.br, (go<KSmoothSellSplit<BR_, T>>((unsigned)A.nslices, 32 * A.split, 0, s, {
                                  A.nbr, A.sp, A.rl, A.col, v, dinv, b, x, xout, d, c1, c2})));
  } else if (A.unroll == 4) {
    MFS_SQUARE_DISPATCH(A.br, (go<KSmoothSell<BR_, T, 4>>(grid_for(A.nbr, kSellThreads), kSellThreads, 0, s, {
                                  A.nbr, A.sp, A.rl, A.col, v, dinv, b, x, xout, d, c1, c2})));
  } else if (A.unroll == 8) {
    MFS_SQUARE_DISPATCH(A.br, (go<KSmoothSell<BR_, T, 8>>(grid_for(A.nbr, kSellThreads), kSellThreads, 0, s, {
                                  A.nbr, A.sp, A.rl, A.col, v, dinv, b, x, xout, d, c1, c2})));
  } else {
    MFS_SQUARE_DISPATCH(A.br, (go<KSmoothSell<BR_, T, 2>>(grid_for(A.nbr, kSellThreads), kSellThreads, 0, s, {
                                  A.nbr, A.sp, A.rl, A.col, v, dinv, b, x, xout, d, c1, c2})));
  }
}

template <typename T>
void smooth_first(int64_t n, const T *dinv, const T *b, T *x, T *d, T c2, cudaStream_t s) {
  if (n == 0) return;
  HookScope hs(s, K_VECTOR, 4.0 * n * sizeof(T), 1, n, 2.0 * n);
  go<KSmoothFirst<T>>(ew_grid(n), kThreads, 0, s, {n, dinv, b, x, d, c2});
}

template <typename T> bool rows_fusable(const RowTerm<T> *t, int n) {
  if (n < 1 || n > kMaxTerms) return false;
  for (int k = 0; k < n; ++k) {
    const Sell &A = *t[k].A;
    if (A.nbr == 0 || A.nbr != t[0].A->nbr || A.br != t[0].A->br || A.kind != t[0].A->kind) return false;
    if (A.br != 1 && A.br != 2 && A.br != 3 && A.br != 6) return false;
    if (A.bc != 1 && A.bc != 2 && A.bc != 3 && A.bc != 6) return false;
    // one thread per row (large systems: the launches are long) and one CTA per row stay separate
    if (A.kind == 0 ? A.split <= 1 : cta_rows<T>(A)) return false;
  }
  return true;
}
template bool rows_fusable<float>(const RowTerm<float> *, int);
template bool rows_fusable<double>(const RowTerm<double> *, int);

template <int BR, typename T, bool SM>
static void terms_launch(const RowTerm<T> *t, int n, const RowOut<T> &o, int split, int ls, cudaStream_t s) {
  typename KTermsBsr<BR, T, SM>::Args a{};
  const Sell &A = *t[0].A;
  a.nbr = A.nbr;
  a.nt = n;
  a.ls = ls;
  for (int k = 0; k < n; ++k) {
    const Sell &M = *t[k].A;
    a.t[k] = {M.sp, M.rl, M.col, vals<T>(M), t[k].x, M.bc};
  }
  a.e = {o.alpha, o.beta, o.c1, o.c2, o.z, o.dinv, SM ? t[n - 1].x : nullptr, o.y, o.d, o.xout, o.mode};
  if (A.kind == 0) {
    go<KTermsSell<BR, T, SM>>((unsigned)A.nslices, 32 * split, 0, s, a);
  } else {
    const unsigned th = bsr_threads(A.nbr << ls);
    go<KTermsBsr<BR, T, SM>>(grid_for(A.nbr << ls, th), th, 0, s, a);
  }
}

template <typename T> void spmv_terms(const RowTerm<T> *t, int n, const RowOut<T> &o, cudaStream_t s) {
  const Sell &A = *t[0].A;
  double bytes = 0.0, flops = 0.0;
  int split = 1, ls = 0;
  for (int k = 0; k < n; ++k) {
    const Sell &M = *t[k].A;
    bytes += matrix_bytes<T>(M) + (double)sizeof(T) * M.ncols();
    flops += 2.0 * M.nnzb * M.br * M.bc;
    split = std::max(split, M.split);
    ls = std::max(ls, M.kind == 1 ? bsr_ls<T>(M) : 0);
  }
  const double vecs = o.mode == kRowSmooth ? 6.0 : o.mode == kRowFirst ? 4.0 + (o.z ? 1 : 0) : o.mode == kRowSub ? 3.0 : o.z ? 2.0 : 1.0;
  HookScope hs(s, o.mode == kRowSmooth ? K_SMOOTH : K_SPMV, bytes + sizeof(T) * vecs * A.nrows(),
               (A.kind == 0 ? 11000 : 10000) + A.br * 100 + n * 10 + (sizeof(T) == 8 ? 1 : 0), A.nbr,
               flops + vecs * A.nrows());
  if (o.mode == kRowSmooth) {
    MFS_SQUARE_DISPATCH(A.br, (terms_launch<BR_, T, true>(t, n, o, split, ls, s)));
  } else {
    MFS_SQUARE_DISPATCH(A.br, (terms_launch<BR_, T, false>(t, n, o, split, ls, s)));
  }
}
template void spmv_terms<float>(const RowTerm<float> *, int, const RowOut<float> &, cudaStream_t);
template void spmv_terms<double>(const RowTerm<double> *, int, const RowOut<double> &, cudaStream_t);

#define MFS_GS_G_DISPATCH(GV, CALL)                              \
  switch (GV) {                                                  \
    case 4: { constexpr int G_ = 4; CALL; } break;               \
    case 8: { constexpr int G_ = 8; CALL; } break;               \
    case 16: { constexpr int G_ = 16; CALL; } break;             \
    default: { constexpr int G_ = 32; CALL; } break;             \
  }

template <typename T>
void gs_sweeps(const GsLevel &g, const T *dblk, const T *b, T *x, T omega, int sweeps, bool backward,
               cudaStream_t s) {
  const Sell &A = g.M;
  if (A.nbr == 0) return;
  const T *v = vals<T>(A);
  const int bw = backward ? 1 : 0;
  const int sig = (A.kind == 1 ? 5 : 4) * 1000 + sparse_sig<T>(A) % 1000;
  if (!g.small) {
    const int nc = g.ncolors();
    for (int sw = 0; sw < sweeps; ++sw)
      for (int q = 0; q < nc; ++q) {
        const int c = backward ? nc - 1 - q : q;
        const int64_t r0 = g.hoff[c], r1 = g.hoff[c + 1], nr = r1 - r0;
        // this colour's blocks + gathered x + diagonal blocks + b and x of its rows
        HookScope hs(s, K_SMOOTH,
                     (double)g.cnnzb[c] * (A.br * A.bc * sizeof(T) + sizeof(int32_t)) +
                         (double)sizeof(T) * (g.cnnzb[c] * A.bc + (A.br + 2.0) * A.br * nr) + 8.0 * nr,
                     sig, nr, 2.0 * g.cnnzb[c] * A.br * A.bc + 2.0 * A.br * A.br * nr);
        MFS_GS_G_DISPATCH(g.G, MFS_SQUARE_DISPATCH(A.br, (go<KGsColor<BR_, T, G_>>(grid_for(nr * G_), kThreads, 0, s, {
                                                             r0, r1, A.sp, A.col, v, g.rowidx, dblk, b, x, omega, bw}))));
      }
    return;
  }
  HookScope hs(s, K_SMOOTH,
               sweeps * (matrix_bytes<T>(A) + (double)sizeof(T) * ((A.br + 2.0) * A.nrows())) +
                   2.0 * sizeof(T) * A.nrows(),
               sig, A.nbr, sweeps * (2.0 * A.nnzb * A.br * A.bc + 2.0 * A.br * A.nrows()));
  const int nc = g.ncolors();
  const size_t shm = (size_t)A.nrows() * sizeof(T);
  MFS_GS_G_DISPATCH(g.G, MFS_SQUARE_DISPATCH(A.br, (go<KGsSmall<BR_, T, G_>>(1, kGsCtaThreads, shm, s, {
                                                       nc, A.nbr, g.coff, A.sp, A.col, v, g.rowidx, dblk, b, x,
                                                       omega, sweeps, bw}))));
}

template <typename T>
void lu_solve(const DenseLU &lu, const T *b, T *x, cudaStream_t s) {
  if (lu.n == 0) return;
  if (lu.inv) {
    HookScope hs(s, K_COARSE, 8.0 * lu.n * (double)lu.n + 2.0 * sizeof(T) * lu.n, 2, lu.n, 2.0 * lu.n * (double)lu.n);
    constexpr int kRowsPerCta = kThreads / 32;
    go<KInvApply<T>>((unsigned)((lu.n + kRowsPerCta - 1) / kRowsPerCta), kThreads, (size_t)lu.n * sizeof(double), s, {
        lu.n, lu.inv, b, x});
    return;
  }
  HookScope hs(s, K_COARSE, 8.0 * lu.n * (double)lu.n + (4.0 + 2 * sizeof(T)) * lu.n, 1, lu.n,
               2.0 * lu.n * (double)lu.n);
  // stage the factors in shared memory when y and LU fit in 200 KB
  const int staged = (size_t)lu.n * (lu.n + 1) * sizeof(double) <= 200 * 1024 ? 1 : 0;
  const size_t smem = (size_t)lu.n * (staged ? lu.n + 1 : 1) * sizeof(double);
  const int threads = lu.n <= 64 ? 256 : 512;
  go<KLuSolve<T>>(1, threads, smem, s, {lu.n, lu.lu, lu.perm, b, x, staged});
}

size_t tail_smem_bytes(int64_t n, int64_t nc, size_t tsize) {
  return (size_t)nc * (sizeof(double) + 2 * tsize) + (size_t)n * 5 * tsize;
}

bool tail_supported(int br, int bc) { return br == bc && (br == 1 || br == 2 || br == 3 || br == 6); }

template bool cta_rows<float>(const Sell &);
template bool cta_rows<double>(const Sell &);

template <typename T>
void vcycle_tail(const Sell &A, const T *dinv, const Sell &R, const Sell &P, const DenseLU &lu, int ns,
                 const T *c1, const T *c2, const T *b, T *x, cudaStream_t s) {
  TailArgs<T> a{};
  a.n = A.nrows();
  a.nbr = A.nbr;
  a.nc = lu.n;
  a.ncbr = R.nbr;
  a.arp = A.sp;
  a.acol = A.col;
  a.aval = vals<T>(A);
  a.dinv = dinv;
  a.rrp = R.sp;
  a.rcol = R.col;
  a.rval = vals<T>(R);
  a.prp = P.sp;
  a.pcol = P.col;
  a.pval = vals<T>(P);
  a.als = bsr_ls<T>(A);
  a.rls = bsr_ls<T>(R);
  a.pls = bsr_ls<T>(P);
  a.inv = lu.inv;
  a.b = b;
  a.x = x;
  a.ns = ns;
  for (int k = 0; k < ns && k < kTailMaxSteps; ++k) {
    a.c1[k] = c1[k];
    a.c2[k] = c2[k];
  }
  const size_t smem = tail_smem_bytes(a.n, a.nc, sizeof(T));
  const double bytes = ns * 2.0 * matrix_bytes<T>(A) + matrix_bytes<T>(A) + matrix_bytes<T>(R) + matrix_bytes<T>(P) +
                       8.0 * lu.n * (double)lu.n + 2.0 * sizeof(T) * A.nrows();
  HookScope hs(s, K_COARSE, bytes, 3, A.nbr, 0.0);
  switch (A.br) {
    case 1: go<KVcycleTail<1, 1, T>>(1, kTailThreads, smem, s, a); break;
    case 2: go<KVcycleTail<2, 2, T>>(1, kTailThreads, smem, s, a); break;
    case 3: go<KVcycleTail<3, 3, T>>(1, kTailThreads, smem, s, a); break;
    case 6: go<KVcycleTail<6, 6, T>>(1, kTailThreads, smem, s, a); break;
    default: break;
  }
}
template void vcycle_tail<float>(const Sell &, const float *, const Sell &, const Sell &, const DenseLU &, int,
                                 const float *, const float *, const float *, float *, cudaStream_t);
template void vcycle_tail<double>(const Sell &, const double *, const Sell &, const Sell &, const DenseLU &, int,
                                  const double *, const double *, const double *, double *, cudaStream_t);

template <typename T>
void fill(T *x, int64_t n, T v, cudaStream_t s) {
  HookScope hs(s, K_VECTOR, (double)n * sizeof(T), 2, n, 0.0);
  if (n) go<KFill<T>>(ew_grid(n), kThreads, 0, s, {x, n, v});
}
template <typename T>
void axpy_diag(T *x, const T *dinv, const T *t, int64_t n, cudaStream_t s) {
  HookScope hs(s, K_VECTOR, 4.0 * n * sizeof(T), 3, n, 2.0 * n);
  if (n) go<KAxpyDiag<T>>(ew_grid(n), kThreads, 0, s, {x, dinv, t, n});
}
template <typename T>
void axpy(T *y, const T *x, T a, int64_t n, cudaStream_t s) {
  HookScope hs(s, K_VECTOR, 3.0 * n * sizeof(T), 4, n, 2.0 * n);
  if (n) go<KAxpy<T>>(ew_grid(n), kThreads, 0, s, {y, x, a, n});
}
void sell_widths(const int32_t *rp, int64_t nbr, int32_t *rl, int32_t *w, cudaStream_t s) {
  if (nbr) k_sell_widths<<<grid_for(nbr), kThreads, 0, s>>>(rp, nbr, rl, w);
}

void sell_fill(const int32_t *rp, const int32_t *ci, int nsrc, const double *v0, const double *v1,
               const double *v2, const int *bcs, int br, int64_t nbr, const int32_t *sp, int32_t *col,
               double *v64, float *v32, cudaStream_t s) {
  if (nbr)
    k_sell_fill<<<grid_for(nbr), kThreads, 0, s>>>(rp, ci, nsrc, v0, v1, v2, bcs[0], nsrc > 1 ? bcs[1] : 0,
                                                   nsrc > 2 ? bcs[2] : 0, br, nbr, sp, col, v64, v32);
}

template <typename TI, typename TO>
void convert(const TI *in, TO *out, int64_t n, cudaStream_t s) {
  HookScope hs(s, K_VECTOR, (double)n * (sizeof(TI) + sizeof(TO)), 5, n, 0.0);
  if (n) go<KConvert<TI, TO>>(ew_grid(n), kThreads, 0, s, {in, out, n});
}
template <typename TO>
void scale_convert(double *v, double a, TO *out, int64_t n, cudaStream_t s) {
  HookScope hs(s, K_VECTOR, (16.0 + sizeof(TO)) * n, 7, n, (double)n);
  if (n) go<KScaleConvert<TO>>(ew_grid(n), kThreads, 0, s, {v, a, out, n});
}
template void scale_convert<float>(double *, double, float *, int64_t, cudaStream_t);
template void scale_convert<double>(double *, double, double *, int64_t, cudaStream_t);
template <typename TO>
void scale_convert_dev(double *v, const double *inv, TO *out, int64_t n, cudaStream_t s) {
  HookScope hs(s, K_VECTOR, (16.0 + (out ? sizeof(TO) : 0)) * n, 8, n, (double)n);
  if (n) go<KScaleConvertDev<TO>>(ew_grid(n), kThreads, 0, s, {v, inv, out, n});
}
template void scale_convert_dev<float>(double *, const double *, float *, int64_t, cudaStream_t);
template void scale_convert_dev<double>(double *, const double *, double *, int64_t, cudaStream_t);

void scale(const double *x, double a, double *y, int64_t n, cudaStream_t s) {
  HookScope hs(s, K_VECTOR, 16.0 * n, 6, n, (double)n);
  if (n) go<KScale>(ew_grid(n), kThreads, 0, s, {x, a, y, n});
}

// CTAs of the CGS2 passes over a length-n basis and entries (whole tiles)
// per CTA.  The SM with the most work sets the time: per CTA the three passes
// run 32 float64 warp instructions a tile and row (768 at 24 rows, the middle
// of a 50-column cycle), and its sums over lanes and its launch cost as much
// as 120 such instructions (fitted to timings of 972 to 1.37 M entries).
// More than two tiles per CTA only with 3 CTAs per SM, which hide the load
// latency (1.37 M entries, 47 rows: 2 per SM 597 us, 3 per SM 500 us).
// Systems solved in batches fill the GPU together: four tiles a CTA there (the
// sums over lanes are 4 % of a CTA's float64 work instead of 14 %).
// (The count is per system, so a batch and a solo solve reduce in the same order.)
int mdot_blocks(int64_t n, bool batch) {
  const int64_t tiles = std::max<int64_t>(1, (n + kTile - 1) / kTile);
  if (batch) {
    const int64_t per = std::max<int64_t>(4, (tiles + 152 * 4 - 1) / (152 * 4));
    return (int)((tiles + per - 1) / per);
  }
  int best = 1;
  double tbest = 1e300;
  for (int ctas = 1; ctas <= kMdotBlocksMax / 152; ++ctas) {  // CTAs per SM
    const int64_t per = (tiles + 152 * ctas - 1) / (152 * ctas);
    const int64_t nblk = (tiles + per - 1) / per;
    if (per > 1 && ctas < (per > 2 ? 3 : 2)) continue;
    const double t = (double)((nblk + 151) / 152) * (768.0 * per + 120.0);
    if (t < tbest) {
      tbest = t;
      best = (int)nblk;
    }
  }
  return best;
}
// entries (whole tiles) per CTA
static int64_t mdot_per(int64_t n, int nblk) {
  const int64_t tiles = std::max<int64_t>(1, (n + kTile - 1) / kTile);
  return (tiles + nblk - 1) / nblk * kTile;
}

void mdot(const double *V, int64_t ldv, int k, const double *w, int64_t n, double *partial, int nblk,
          cudaStream_t s, double *out, unsigned *cnt) {
  const int64_t per = mdot_per(n, nblk);
  if (k != 1 || !out) cnt = nullptr;
  {
    HookScope hs(s, K_ARNOLDI, 8.0 * n * (k + 1), 1, n, 2.0 * n * k);
    go<KMdot>(nblk, kThreads, 0, s, {V, ldv, k, w, n, partial, nblk, per, out, cnt});
  }
  if (out && !cnt) reduce_partials(partial, k, nblk, out, s);
}

void reduce_partials(const double *partial, int k, int nblk, double *out, cudaStream_t s) {
  HookScope hs(s, K_ARNOLDI, 8.0 * (double)k * nblk, 2, k, (double)k * nblk);
  // recorded launches take a grid that does not depend on k (blocks >= k return)
  go<KReducePartials>(g_rec ? (unsigned)kMaxQ : (unsigned)k, kThreads, 0, s, {partial, k, nblk, out});
}

// One CGS2 step (see kernels.cuh)
void cgs2(const double *V, int64_t ldv, int k, double *w, int64_t n, double *partial, int nblk, double *out,
          unsigned *cnt, cudaStream_t s) {
  const int64_t per = mdot_per(n, nblk);
  const bool inl = nblk <= kInlineBlocks;
  double *p1 = partial, *p2 = partial + (int64_t)64 * nblk;
  mdot(V, ldv, k + 1, w, n, p1, nblk, s, inl ? nullptr : out, nullptr);
  {
    HookScope hs(s, K_ARNOLDI, 8.0 * n * (k + 2), 3, n, 4.0 * n * k);
    go<KCgsFused>(nblk, kThreads, 0, s, {V, ldv, k, out, inl ? p1 : nullptr, out, w, n, p2, nblk, per});
  }
  if (!inl) reduce_partials(p2, k, nblk, out + 64, s);
  HookScope hs(s, K_ARNOLDI, 8.0 * n * (k + 2), 4, n, 2.0 * n * k + 2.0 * n);
  go<KCgsUpdate>(nblk, kThreads, 0, s,
                 {V, ldv, k, out + 64, inl ? p2 : nullptr, out + 64, w, n, p1, nblk, per, out + 128, cnt});
}

void gemv_add(const double *Z, int64_t ldz, int k, const double *y, double *x, int64_t n, cudaStream_t s) {
  HookScope hs(s, K_ARNOLDI, 8.0 * n * (k + 2), 5, n, 2.0 * n * k);
  go<KGemvAdd>(ew_grid(n), kThreads, 0, s, {Z, ldz, k, y, x, n});
}

#define MFS_INST(T)                                                                                   \
  template void spmv<T>(const Sell &, const T *, T *, T, T, const T *, cudaStream_t);                 \
  template void smooth_step<T>(const Sell &, const T *, const T *, const T *, T *, T *, T, T,         \
                               cudaStream_t);                                                         \
  template void smooth_first<T>(int64_t, const T *, const T *, T *, T *, T, cudaStream_t);            \
  template void gs_sweeps<T>(const GsLevel &, const T *, const T *, T *, T, int, bool, cudaStream_t);   \
  template void lu_solve<T>(const DenseLU &, const T *, T *, cudaStream_t);                           \
  template void fill<T>(T *, int64_t, T, cudaStream_t);                                               \
  template void axpy_diag<T>(T *, const T *, const T *, int64_t, cudaStream_t);                       \
  template void axpy<T>(T *, const T *, T, int64_t, cudaStream_t);
MFS_INST(double)
MFS_INST(float)
template void convert<double, float>(const double *, float *, int64_t, cudaStream_t);
template void convert<float, double>(const float *, double *, int64_t, cudaStream_t);
template void convert<double, double>(const double *, double *, int64_t, cudaStream_t);
template void convert<float, float>(const float *, float *, int64_t, cudaStream_t);

}  // namespace dev
}  // namespace mfs
