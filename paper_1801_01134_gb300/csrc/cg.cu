// Conjugate gradients over beta(r,c) SpMV, in float64 and as mixed-precision
// iterative refinement (float64 residual / update / norms, float32 or bfloat16
// matrix with float32 vectors inside).
//
// The paper motivates fast SpMV by iterative solvers such as CG, which apply
// one matrix many times (Introduction). CG is Hestenes & Stiefel's; the
// refinement loop is the classical one (Wilkinson; Moler 1967):
//     r = b - A x (float64);  solve A d ~= r / ||r|| in float32;  x += ||r|| d.
// A third mode keeps one float32 CG recurrence and replaces its residual by the
// float64 one from time to time (reliable updates, Sleijpen & van der Vorst
// 1996), which needs about the float64 iteration count instead of paying for
// restarts.
// On GB300 float64 arithmetic is issue-bound (one float64 FMA warp-instruction
// per ~16 SM cycles), so moving the bulk of the work to float32 pays twice:
// half the bytes per SpMV and no float64 pipe in the inner loop.
//
// The iteration is ordered so that it takes two passes. With beta from the
// previous iteration (0 at the start, p = q = 0):
//     q = A r + beta q,  p = r + beta p,  alpha = rho / (p.q)     (pass 1)
//     x += alpha p,  r -= alpha q,  rho' = r.r,  beta = rho'/rho  (pass 2)
// which is Hestenes-Stiefel CG with A p_k formed as A r_k + beta A p_{k-1}
// (equal in exact arithmetic), so the SpMV reads r and the p update rides in
// its epilogue instead of a third pass.
// Scalars (rho, p.q, alpha, beta) never leave the device inside an iteration,
// and dot products are summed in a fixed order (so results repeat run to run).
// Matrices without long intervals iterate inside one resident kernel (see
// k_cg_resident); the others run the SpMV and two vector kernels per
// iteration, whose last block to finish sums the partials and writes the
// derived scalar; that iteration can be captured once into a CUDA graph and
// replayed, and the host reads the residual norm every `check_every`
// iterations.
#include <algorithm>
#include <climits>
#include <cmath>
#include <vector>

#include "spmv_beta.cuh"

namespace spc5 {
namespace {

constexpr int kThreads = 256;
// Grid cap of the vector updates (beyond it, warps stride over the work).
// Every block adds one same-address atomic to the reduction ticket, and those
// serialise at about 2.5 ns each on GB300, so a smaller grid finishes the
// reduction sooner: measured best at 2 blocks per SM (7-point Poisson 96^3).
constexpr int kVecBlocksPerSm = 2;
// S_ITERS / S_STATUS: iterations of the last resident launch; 1 when one of its waits gave up
enum { S_RHO = 0, S_PQ, S_ALPHA, S_BETA, S_RHONEW, S_NORM, S_ITERS, S_STATUS, S_COUNT = 8 };
constexpr double kReliableDelta = 0.1;  // update when the recurred norm fell by this factor

template <class A>
__device__ __forceinline__ A block_sum(A v) {
  __shared__ A ws[kThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  if (lane == 0) ws[w] = v;
  __syncthreads();
  A t = threadIdx.x < kThreads / 32 ? ws[threadIdx.x] : A(0);
  if (w == 0) {
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) t += __shfl_xor_sync(0xffffffffu, t, d);
  }
  __syncthreads();
  return t;  // valid in thread 0
}

// part[block] = sum_i a[i] b[i] (grid-stride, accumulation type A)
template <class T, class A>
__global__ void __launch_bounds__(kThreads) k_dot_part(const T* __restrict__ a, const T* __restrict__ b, int64_t n,
                                                       A* __restrict__ part) {
  A s = 0;
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads)
    s = fma((A)a[i], (A)b[i], s);
  s = block_sum<A>(s);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// One thread-block sums the partials in float64 in a fixed order and writes
// the scalar `what`, with its derived scalar:
//   S_PQ     -> alpha = rho / pq      (0 when pq == 0)
//   S_RHONEW -> beta = rhonew / rho, then rho = rhonew
//   S_RHO / S_NORM -> plain sum
template <class A>
__global__ void __launch_bounds__(kThreads) k_dot_final(const A* __restrict__ part, int nb, double* __restrict__ scal,
                                                        int what) {
  double s = 0;
  for (int i = threadIdx.x; i < nb; i += kThreads) s += (double)part[i];
  s = block_sum<double>(s);
  if (threadIdx.x == 0) {
    if (what == S_PQ) {
      scal[S_PQ] = s;
      scal[S_ALPHA] = s != 0.0 ? scal[S_RHO] / s : 0.0;
    } else if (what == S_RHONEW) {
      scal[S_RHONEW] = s;
      scal[S_BETA] = scal[S_RHO] != 0.0 ? s / scal[S_RHO] : 0.0;
      scal[S_RHO] = s;
    } else {
      scal[what] = s;
    }
  }
}

// r = b - t (float64) and its partial r.r
__global__ void __launch_bounds__(kThreads) k_residual(double* __restrict__ r, const double* __restrict__ b,
                                                       const double* __restrict__ t, int64_t n,
                                                       double* __restrict__ part) {
  double s = 0;
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads) {
    const double ri = b[i] - t[i];
    r[i] = ri;
    s = fma(ri, ri, s);
  }
  s = block_sum<double>(s);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// start of an inner solve: r32 = r64 / ||r64||, p32 = q32 = x32 = 0, beta = 0
__global__ void __launch_bounds__(kThreads) k_inner_start(const double* __restrict__ r64, float* __restrict__ r32,
                                                          float* __restrict__ p32, float* __restrict__ q32,
                                                          float* __restrict__ x32, int64_t n, double* __restrict__ scal) {
  const double inv = scal[S_NORM] > 0.0 ? 1.0 / sqrt(scal[S_NORM]) : 0.0;
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads) {
    r32[i] = (float)(r64[i] * inv);
    p32[i] = 0.0f;
    q32[i] = 0.0f;
    x32[i] = 0.0f;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) scal[S_BETA] = 0.0;
}

// x64 += ||r|| * x32
__global__ void __launch_bounds__(kThreads) k_inner_apply(double* __restrict__ x64, const float* __restrict__ x32,
                                                          int64_t n, const double* __restrict__ scal) {
  const double nr = sqrt(scal[S_NORM]);
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads)
    x64[i] = fma(nr, (double)x32[i], x64[i]);
}

// reliable update: x64 += x32, x32 = 0
__global__ void __launch_bounds__(kThreads) k_fold_x(double* __restrict__ x64, float* __restrict__ x32, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads) {
    x64[i] += (double)x32[i];
    x32[i] = 0.0f;
  }
}

// r32 = (float) r64
__global__ void __launch_bounds__(kThreads) k_narrow(const double* __restrict__ r64, float* __restrict__ r32,
                                                     int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads)
    r32[i] = (float)r64[i];
}

template <class T>
__global__ void __launch_bounds__(kThreads) k_copy_vec(T* __restrict__ d, const T* __restrict__ s, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads) d[i] = s[i];
}

template <class T>
__global__ void __launch_bounds__(kThreads) k_zero_vec(T* __restrict__ d, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads) d[i] = T(0);
}

// Last-block-done finish of a grid reduction: every block has stored its
// partial in part[blockIdx.x]; the block that arrives last (atomic ticket)
// sums all partials in index order - the same order on every run - and
// resets the ticket for the next kernel. Returns the total in that block
// (thread 0), and whether this block is the last one.
template <class A>
__device__ __forceinline__ bool finish_last_block(A* part, A mine, unsigned* ticket, double* total) {
  __shared__ bool last;
  if (threadIdx.x == 0) {
    part[blockIdx.x] = mine;
    __threadfence();
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return false;
  double s = 0;
  for (unsigned j = threadIdx.x; j < gridDim.x; j += kThreads) s += (double)__ldcg(part + j);
  s = block_sum<double>(s);
  if (threadIdx.x == 0) {
    *total = s;
    *ticket = 0u;
  }
  return true;
}

// reliable update after t = A x: r64 = b - t, r32 = (float) r64 and the
// partials of both squared norms; the last block writes scal[NORM] and, for
// the replaced recurrence, beta = rho_new / rho_previous = s * beta / rho and
// rho = s
__global__ void __launch_bounds__(kThreads) k_replace_residual(double* __restrict__ r64, float* __restrict__ r32,
                                                               const double* __restrict__ b,
                                                               const double* __restrict__ t, int64_t n,
                                                               double* __restrict__ scal, double* part, float* part32,
                                                               unsigned* ticket) {
  double s = 0;
  float s32 = 0;
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads) {
    const double ri = b[i] - t[i];
    const float rf = (float)ri;
    r64[i] = ri;
    r32[i] = rf;
    s = fma(ri, ri, s);
    s32 = fmaf(rf, rf, s32);
  }
  s32 = block_sum<float>(s32);
  if (threadIdx.x == 0) part32[blockIdx.x] = s32;  // before the ticket's fence
  s = block_sum<double>(s);
  double tot;
  if (!finish_last_block<double>(part, s, ticket, &tot)) return;
  double tot32 = 0;
  for (unsigned j = threadIdx.x; j < gridDim.x; j += kThreads) tot32 += (double)__ldcg(part32 + j);
  tot32 = block_sum<double>(tot32);
  if (threadIdx.x == 0) {
    scal[S_NORM] = tot;
    scal[S_BETA] = scal[S_RHO] != 0.0 ? tot32 * scal[S_BETA] / scal[S_RHO] : 0.0;
    scal[S_RHO] = tot32;
  }
}

// 16-byte vector of T (float4 / double2) for the streaming kernels
template <class T>
struct Vec16;
template <>
struct Vec16<float> {
  using type = float4;
  static constexpr int N = 4;
};
template <>
struct Vec16<double> {
  using type = double2;
  static constexpr int N = 2;
};

template <class T>
__device__ __forceinline__ T& lane_of(typename Vec16<T>::type& v, int k) {
  return reinterpret_cast<T*>(&v)[k];
}

// After the SpMV (matrices with long intervals): w = A r came from the
// SpMV; q = w + beta q, p = r + beta p, p.q finished by the last block.
template <class T, class A>
__global__ void __launch_bounds__(kThreads) k_cg_pq(T* __restrict__ p, T* __restrict__ q, const T* __restrict__ r,
                                                    const T* __restrict__ w, int64_t n, double* __restrict__ scal,
                                                    A* part, unsigned* ticket) {
  const T beta = (T)scal[S_BETA];
  A prod = 0;
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads) {
    const T qn = fma(beta, q[i], w[i]);
    const T pn = fma(beta, p[i], r[i]);
    q[i] = qn;
    p[i] = pn;
    prod = fma((A)pn, (A)qn, prod);
  }
  prod = block_sum<A>(prod);
  double tot;
  if (finish_last_block<A>(part, prod, ticket, &tot) && threadIdx.x == 0) {
    scal[S_PQ] = tot;
    scal[S_ALPHA] = tot != 0.0 ? scal[S_RHO] / tot : 0.0;
  }
}

// x += alpha p; r -= alpha q; r.r finished by the last block, which writes
// rhonew, beta = rhonew / rho and rho = rhonew. 16-byte loads and stores;
// element i's arithmetic is the same whichever thread does it.
template <class T, class A>
__global__ void __launch_bounds__(kThreads) k_cg_xr_fused(T* __restrict__ x, T* __restrict__ r,
                                                          const T* __restrict__ p, const T* __restrict__ q, int64_t n,
                                                          double* __restrict__ scal, A* part, unsigned* ticket) {
  using V = typename Vec16<T>::type;
  constexpr int N = Vec16<T>::N;
  const T alpha = (T)scal[S_ALPHA];
  A s = 0;
  const bool aligned = ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(r) |
                         reinterpret_cast<uintptr_t>(p) | reinterpret_cast<uintptr_t>(q)) & 15u) == 0;
  const int64_t nv = aligned ? n / N : 0;  // a caller's x may start anywhere: then all scalar
  const int64_t stride = (int64_t)gridDim.x * kThreads;
  for (int64_t v = (int64_t)blockIdx.x * kThreads + threadIdx.x; v < nv; v += stride) {
    V xv = reinterpret_cast<const V*>(x)[v], rv = reinterpret_cast<const V*>(r)[v];
    const V pv = reinterpret_cast<const V*>(p)[v], qv = reinterpret_cast<const V*>(q)[v];
#pragma unroll
    for (int k = 0; k < N; ++k) {
      lane_of<T>(xv, k) = fma(alpha, lane_of<T>(const_cast<V&>(pv), k), lane_of<T>(xv, k));
      const T ri = fma(-alpha, lane_of<T>(const_cast<V&>(qv), k), lane_of<T>(rv, k));
      lane_of<T>(rv, k) = ri;
      s = fma((A)ri, (A)ri, s);
    }
    reinterpret_cast<V*>(x)[v] = xv;
    reinterpret_cast<V*>(r)[v] = rv;
  }
  for (int64_t i = nv * N + (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += stride) {
    x[i] = fma(alpha, p[i], x[i]);
    const T ri = fma(-alpha, q[i], r[i]);
    r[i] = ri;
    s = fma((A)ri, (A)ri, s);
  }
  s = block_sum<A>(s);
  double tot;
  if (finish_last_block<A>(part, s, ticket, &tot) && threadIdx.x == 0) {
    scal[S_RHONEW] = tot;
    scal[S_BETA] = scal[S_RHO] != 0.0 ? tot / scal[S_RHO] : 0.0;
    scal[S_RHO] = tot;
  }
}

// ------------------------------------------------------- resident iterations
// Many CG iterations in one cooperative launch (matrices without long
// intervals). The blocks stay: a phase ends with a barrier over the grid after
// which every block sums all blocks' partials itself, in the same order (so
// all hold the same scalars and results repeat run to run), and the residual
// norm is tested after every iteration.
//   * The rows are unpacked once per solve (k_rows_fill): 32 rows side by
//     side, value j of row i at offset 32 j + i, with the column of every
//     value. A mask walk costs over 200 instructions per row and waits for
//     memory five times in turn (row pointer, mask, x, next masks, x); here a
//     row's columns and values come in one wait and its x entries in a second.
//     The products are added in the same order.
//   * A warp keeps its rows through all phases. p, q and x are read and
//     written only by their own lane, so they stay in shared memory as far as
//     that reaches; r is gathered by others, through the L1, which the
//     barrier's fence empties.
//   * What follows from a sum is computed by one thread per block: a float64
//     division by every warp of an SM costs more than the barrier (16 cycles
//     per warp instruction: 15 us an iteration).
// Measured per iteration against two kernels each (SpMV with the p, q update;
// x, r update): 7-point Poisson 96^3 float32 31.0 -> 20.5 us, float64 48.5 ->
// 44, 20 thousand rows float64 14.9 -> 11. What is left of the 20.5: 5 to 9 us
// the product (blocks finish unevenly), 1.3 the updates, 3 and 6 the two
// barriers (the second waits until the new r can be read everywhere); float64
// spends 19 us on its pipe's multiply-adds alone.
// Waits are bounded: a block that gives up sets the status and all leave. The
// solve is then done again with the separate kernels, and so is one whose launch
// is refused (a context that owns fewer SMs than the device has).
constexpr int kResThreads = 512;
constexpr int kResPerSm = 2;
constexpr size_t kResReserve = 16384;  // shared memory left to the block's own words and the system
// Rows of a thread held in shared memory, at most. The L1 takes what they leave,
// and a float64 product that gathers all over r needs room there for its loads
// on the way: two million rows of 8 scattered entries, an iteration 208 us with
// the seven rows that fit, 122 with five, 118 with four; 7-point 128^3 98.7, 102
// and 104 (float32 there 45, and 53 with half of its rows).
template <class X>
constexpr int kResHeld = sizeof(X) == 8 ? 5 : INT_MAX;
// A float64 thread with more rows than this many times those it holds streams
// its vectors through the L2 like the separate kernels do, with half their
// threads on the way: 7-point 160^3 (4.1 million rows, 27 of them per thread)
// 185 us an iteration against 174 to 178, 128^3 (14 per thread) 102 against 101.
// In float32 the resident kernel stays ahead (200^3: 198 against 248 us).
constexpr int kResStream = 4;
constexpr long long kSpinClocks = 4000000000ll;  // a wait's limit, about two seconds

// Unpacked rows of a matrix (device), 32 rows per slice.
struct Rows {
  const int32_t* len;   // entries of each row
  const int64_t* off;   // first element of each slice
  const int32_t* col;
  const void* val;
};

// entries of each row; *slots += the longest row of every slice
template <int R, int C>
__global__ void __launch_bounds__(kThreads) k_rows_count(int64_t I, const int32_t* __restrict__ brp,
                                                         const uint8_t* __restrict__ bmask, int32_t* __restrict__ len,
                                                         unsigned long long* __restrict__ slots) {
  constexpr int MB = (R * C + 7) / 8;
  const int64_t row = (int64_t)blockIdx.x * kThreads + threadIdx.x;  // its interval: row / R
  const int64_t it = row / R;
  const int i = (int)(row % R);
  int n = 0;
  if (it < I) {
    for (int32_t b = __ldg(brp + it), e = __ldg(brp + it + 1); b < e; ++b)
      n += __popc(row_bits<C>(load_mask<MB>(bmask, b), i));
    len[row] = n;
  }
  const int most = __reduce_max_sync(0xffffffffu, n);
  __shared__ int wide[kThreads / 32];
  if ((threadIdx.x & 31) == 0) wide[threadIdx.x >> 5] = most;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long t = 0;
    for (int w = 0; w < kThreads / 32; ++w) t += (unsigned long long)wide[w];
    if (t) atomicAdd(slots, t);
  }
}

// the rows' columns and values; the slices take their places as they come
template <int R, int C, class V>
__global__ void __launch_bounds__(kThreads) k_rows_fill(int64_t I, const int32_t* __restrict__ brp,
                                                        const int32_t* __restrict__ bcol,
                                                        const uint8_t* __restrict__ bmask, const V* __restrict__ val,
                                                        const int64_t* __restrict__ valptr,
                                                        const int32_t* __restrict__ len, int64_t* __restrict__ off,
                                                        int32_t* __restrict__ col, V* __restrict__ out,
                                                        unsigned long long* __restrict__ slots) {
  constexpr int MB = (R * C + 7) / 8;
  const int64_t row = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  const int64_t it = row / R;
  const int i = (int)(row % R), lane = threadIdx.x & 31;
  const int most = __reduce_max_sync(0xffffffffu, it < I ? len[row] : 0);
  unsigned long long at = 0;
  if (lane == 0) at = atomicAdd(slots, (unsigned long long)most);
  at = __shfl_sync(0xffffffffu, at, 0) * 32ull;
  if (it >= I) return;
  if (lane == 0) off[row >> 5] = (int64_t)at;
  col += at + lane;
  out += at + lane;
  const V* __restrict__ v = val + __ldg(valptr + it);
  int64_t j = 0;
  for (int32_t b = __ldg(brp + it), e = __ldg(brp + it + 1); b < e; ++b) {
    const Mask<MB> mk = load_mask<MB>(bmask, b);
    const int32_t c0 = __ldg(bcol + b);
    const V* __restrict__ w = v + popc_below<C>(mk, i);
    for (uint32_t bits = row_bits<C>(mk, i); bits; bits &= bits - 1, j += 32) {
      col[j] = c0 + __ffs(bits) - 1;
      out[j] = *w++;
    }
    v += popc_all(mk);
  }
}

struct ResState {  // device words of one launch
  int status;  // 1: a wait gave up
  int pad[3];
};
// After it, the blocks' words for the two sums of an iteration: each block
// publishes its partial sum in 8-byte words that carry half the bits and the
// number of the sum, so that one read tells whether the sum is there and what
// it is (an 8-byte store arrives whole).
constexpr int kResWords = 2;
inline size_t res_bytes(int blocks) { return sizeof(ResState) + sizeof(unsigned long long) * 2 * kResWords * (size_t)blocks; }

// Sum of v over the block, in thread 0. All values are laid down and one warp
// adds them up: a shuffle tree in every warp would keep the float64 pipe busy
// four times as long.
template <class A>
__device__ __forceinline__ A res_block_sum(A v) {
  __shared__ A all[kResThreads];
  all[threadIdx.x] = v;
  __syncthreads();
  A t = 0;
  if (threadIdx.x < 32) {
    A a[4] = {A(0), A(0), A(0), A(0)};
#pragma unroll
    for (int k = 0; k < kResThreads / 32; ++k) a[k & 3] += all[32 * k + threadIdx.x];
    t = (a[0] + a[1]) + (a[2] + a[3]);
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) t += __shfl_xor_sync(0xffffffffu, t, d);
  }
  return t;
}

// an 8-byte read that what its writer wrote before can be read after
__device__ __forceinline__ unsigned long long load_acquire(const volatile unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// Every block's `mine` (thread 0) summed over the grid in block order and
// handed to `then` in thread 0 after all blocks have arrived; false when the
// wait gave up. `phase` counts the calls from 1. Thread t waits for block t's
// words (one memory round trip after the last block has come), one warp adds.
// With FENCE, what the blocks wrote before the call can be read after it;
// without, only the sum passes between them.
template <class A, bool FENCE, class Then>
__device__ __forceinline__ bool grid_sum(A mine, ResState* st, unsigned phase, long long limit, Then then) {
  constexpr bool kWide = sizeof(A) == 8;
  __shared__ A parts[kResThreads];
  // the two sums of an iteration have words of their own: a block publishes
  // its next one of a kind only after all have read the last
  volatile unsigned long long* const word =
      reinterpret_cast<volatile unsigned long long*>(st + 1) + (phase & 1u) * kResWords * gridDim.x;
  if (threadIdx.x == 0) {
    if (FENCE) asm volatile("fence.acq_rel.gpu;" ::: "memory");
    if constexpr (kWide) {
      const unsigned long long bits = (unsigned long long)__double_as_longlong(mine);
      word[kResWords * blockIdx.x] = (bits << 32) | phase;
      word[kResWords * blockIdx.x + 1] = (bits & 0xffffffff00000000ull) | phase;
    } else {
      word[kResWords * blockIdx.x] = ((unsigned long long)__float_as_uint(mine) << 32) | phase;
    }
  }
  bool bad = false;
  if (threadIdx.x < gridDim.x) {
    const volatile unsigned long long* const w = word + kResWords * threadIdx.x;
    unsigned long long lo = w[0], hi = kWide ? w[1] : phase;
    const long long t0 = clock64();
    while ((unsigned)lo != phase || (unsigned)hi != phase) {
      if (clock64() - t0 > limit || *(volatile int*)&st->status) {
        // given up only if the words, read once more, are not there (the clock
        // runs on while the whole process is suspended)
        lo = w[0];
        if (kWide) hi = w[1];
        if ((unsigned)lo == phase && (unsigned)hi == phase) break;
        st->status = 1;
        bad = true;
        break;
      }
      lo = w[0];
      if (kWide) hi = w[1];
    }
    if constexpr (kWide)
      parts[threadIdx.x] = __longlong_as_double((long long)((hi & 0xffffffff00000000ull) | (lo >> 32)));
    else
      parts[threadIdx.x] = __uint_as_float((unsigned)(lo >> 32));
    if (FENCE) load_acquire(w);  // what the poll has seen is there
  }
  if (__syncthreads_or(bad)) return false;
  if (threadIdx.x < 32) {
    double a[2] = {0.0, 0.0};
    int k = 0;
    for (unsigned j = threadIdx.x; j < gridDim.x; j += 32, k ^= 1) {
      if (k)
        a[1] += (double)parts[j];
      else
        a[0] += (double)parts[j];
    }
    double s = a[0] + a[1];
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
    if (threadIdx.x == 0) then(s);
  }
  __syncthreads();
  return true;
}

// acc = row `row` of A times x, its `len` entries from col and val (stride 32)
// on, eight (float64: four, for the registers) at a time: their loads are all
// on the way before the first is used. Values stay as they are stored until
// then: widening bfloat16 at the load made every load wait for the one before
// (27-point 96^3, beta(2,4), an iteration 85 us; now 47, float32 52).
// x changes while the kernel runs: ordinary loads, not read-only ones.
template <class T>
__device__ __forceinline__ typename T::A row_dot(int len, const int32_t* __restrict__ col,
                                                 const typename T::V* __restrict__ val, const typename T::X* x) {
  constexpr int U = sizeof(typename T::X) == 8 ? 4 : 8;
  typename T::A acc = 0;
  for (int j = 0; j < len; j += U) {
    int32_t c[U];
    typename T::V v[U];
    typename T::A xx[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (j + u < len) {
        c[u] = __ldg(col + 32 * (j + u));
        v[u] = __ldg(val + 32 * (j + u));
      }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (j + u < len) xx[u] = x[c[u]];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (j + u < len) acc = fmadd<T>(sval<T>(v, u), xx[u], acc);
  }
  return acc;
}

template <class T>
__global__ void __launch_bounds__(kResThreads, kResPerSm)
    k_cg_resident(int64_t n, const Rows rows, typename T::X* x, typename T::X* r, typename T::X* p, typename T::X* q,
                  double* scal, ResState* st, double stop, double fall, int every, int held, int max_it,
                  long long limit) {
  using A = typename T::A;
  using X = typename T::X;
  const int64_t nrows = (int64_t)gridDim.x * kResThreads;  // rows of one round
  const int64_t first = (int64_t)blockIdx.x * kResThreads + threadIdx.x;
  const int32_t* __restrict__ lens = rows.len;
  const int64_t* __restrict__ offs = rows.off;
  const int32_t* __restrict__ cols = rows.col + (threadIdx.x & 31);
  const typename T::V* __restrict__ vals = static_cast<const typename T::V*>(rows.val) + (threadIdx.x & 31);
  // p, q and x of the thread's first `held` rows live in shared memory from
  // here to the end of the launch (slot j * kResThreads + threadIdx.x is the
  // j-th row's); those of further rows stay where they are
  extern __shared__ __align__(16) unsigned char held_raw[];
  X* const hp = reinterpret_cast<X*>(held_raw);
  X* const hq = hp + (int64_t)held * kResThreads;
  X* const hx = hq + (int64_t)held * kResThreads;
  {
    int j = threadIdx.x;
    for (int64_t row = first; row < n && j < held * kResThreads; row += nrows, j += kResThreads) {
      hp[j] = p[row];
      hq[j] = q[row];
      hx[j] = x[row];
    }
  }
  // the solve's scalars, kept by thread 0
  __shared__ double rho, alpha, beta, pq, target;
  __shared__ X alpha_x, beta_x;
  __shared__ bool more;
  if (threadIdx.x == 0) {
    // down to `stop`; with fall > 0 to half of `stop`, or until the norm, seen
    // every `every` iterations, has fallen by `fall` from the float64
    // residual's (scal[S_NORM]); nothing to do where that has reached `stop`
    target = stop;
    more = true;
    if (fall > 0.0) {
      const double rn = sqrt(scal[S_NORM]);
      more = rn > stop;
      target = fall * rn;
      target *= target;
      stop *= 0.5;
    }
    stop *= stop;  // squared norms from here on
    rho = scal[S_RHO];
    beta = scal[S_BETA];
    alpha = pq = 0.0;
    beta_x = (X)beta;
  }
  __syncthreads();
  unsigned phase = 0;
  int k = 0;
  while (more && k < max_it) {
    // q = A r + beta q, p = r + beta p, p.q (only the sum passes to other
    // blocks, and all have read their r entries when it is complete)
    const X bx = beta_x;
    A prod = 0;
    int j = threadIdx.x;
    int len = first < n ? __ldg(lens + first) : 0;
    int64_t off = first < n ? __ldg(offs + (first >> 5)) : 0;
    for (int64_t row = first; row < n; row += nrows, j += kResThreads) {
      const int len0 = len;
      const int64_t off0 = off;
      if (row + nrows < n) {  // the next row's place, one row ahead
        len = __ldg(lens + row + nrows);
        off = __ldg(offs + ((row + nrows) >> 5));
      }
      const A acc = row_dot<T>(len0, cols + off0, vals + off0, r);
      X qn, pn;
      if (j < held * kResThreads) {
        hq[j] = qn = fma(bx, hq[j], (X)acc);
        hp[j] = pn = fma(bx, hp[j], r[row]);
      } else {
        q[row] = qn = fma(bx, q[row], (X)acc);
        p[row] = pn = fma(bx, p[row], r[row]);
      }
      prod = fma((A)pn, (A)qn, prod);
    }
    prod = res_block_sum<A>(prod);
    if (!grid_sum<A, false>(prod, st, ++phase, limit, [&](double sum) {
          pq = sum;
          alpha = sum != 0.0 ? rho / sum : 0.0;
          alpha_x = (X)alpha;
        })) {
      if (threadIdx.x == 0) scal[S_STATUS] = 1.0;
      return;
    }
    // x += alpha p, r -= alpha q, r.r
    const X ax = alpha_x;
    A s = 0;
    j = threadIdx.x;
#pragma unroll 2
    for (int64_t row = first; row < n; row += nrows, j += kResThreads) {
      X ri;
      if (j < held * kResThreads) {
        hx[j] = fma(ax, hp[j], hx[j]);
        ri = fma(-ax, hq[j], r[row]);
      } else {
        x[row] = fma(ax, p[row], x[row]);
        ri = fma(-ax, q[row], r[row]);
      }
      r[row] = ri;
      s = fma((A)ri, (A)ri, s);
    }
    s = res_block_sum<A>(s);
    if (!grid_sum<A, true>(s, st, ++phase, limit, [&](double sum) {
          beta = rho != 0.0 ? sum / rho : 0.0;
          beta_x = (X)beta;
          rho = sum;
          more = sum > stop && !(fall > 0.0 && (k + 1) % every == 0 && sum <= target);  // not on NaN
        })) {
      if (threadIdx.x == 0) scal[S_STATUS] = 1.0;
      return;
    }
    ++k;
  }
  {
    int j = threadIdx.x;
    for (int64_t row = first; row < n && j < held * kResThreads; row += nrows, j += kResThreads) {
      p[row] = hp[j];
      q[row] = hq[j];
      x[row] = hx[j];
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    scal[S_PQ] = pq;
    scal[S_ALPHA] = alpha;
    scal[S_RHONEW] = rho;
    scal[S_RHO] = rho;
    scal[S_BETA] = beta;
    scal[S_ITERS] = (double)k;
  }
}

// the resident kernel for a handle's rows and its grid (all blocks resident at once)
struct ResLaunch {
  const void* kern = nullptr;
  int blocks = 0;  // 0: the handle's iterations run as separate kernels
  int held = 0;    // rows per thread whose p, q and x fit the shared memory
  size_t smem = 0;
  long long limit = kSpinClocks;
  Rows rows{};
};

template <class T>
ResLaunch resident_kernel(int64_t n) {
  ResLaunch l;
  l.kern = (const void*)k_cg_resident<T>;
  int dev = 0, per_sm = 0, smem_sm = 0, smem_block = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, l.kern, kResThreads, 0) != cudaSuccess || per_sm < 1 ||
      cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&smem_block, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
    return l;
  per_sm = std::min(per_sm, kResPerSm);
  // a thread per block waits in the barrier
  const int64_t blocks = std::min({(n + kResThreads - 1) / kResThreads, (int64_t)sm_count() * per_sm, (int64_t)kResThreads});
  const size_t row = 3 * sizeof(typename T::X) * kResThreads;  // one row of every thread
  const size_t room = std::min((size_t)smem_block, (size_t)smem_sm / (size_t)per_sm) - kResReserve;
  const int64_t each = (n + blocks * kResThreads - 1) / (blocks * kResThreads);  // rows of a thread
  l.held = (int)std::min({each, (int64_t)(room / row), (int64_t)kResHeld<typename T::X>});
  if (sizeof(typename T::X) == 8 && each > kResStream * (int64_t)l.held) return l;
  l.smem = row * (size_t)l.held;
  int fit = 0;
  if (cudaFuncSetAttribute(l.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)room) == cudaSuccess &&
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, l.kern, kResThreads, l.smem) == cudaSuccess &&
      (int64_t)fit * sm_count() >= blocks)
    l.blocks = (int)blocks;
  return l;
}

// workspace from the library's pool, in the order of the solve's stream (a
// dozen cudaMalloc / cudaFree pairs of a few MB took about a millisecond)
struct Buf {
  void* p = nullptr;
  cudaStream_t s = nullptr;
  ~Buf() { release(); }
  cudaError_t alloc(size_t bytes, cudaStream_t st) {
    s = st;
    return pool_alloc(&p, bytes, st);
  }
  void release() {
    if (p) cudaFreeAsync(p, s);
    p = nullptr;
  }
};

cudaError_t spmv_any(const spc5_matrix* h, const void* x, void* y, cudaStream_t s) {
  switch (h->vt) {
    case SPC5_F64: return launch_spmv_f64(h, x, y, false, s);
    case SPC5_F32: return launch_spmv_f32(h, x, y, false, s);
    default: return launch_spmv_bf16(h, x, y, false, s);
  }
}

// One CG iteration on the stream (vector type T, accumulation type A), in
// the order of the file comment, for the matrices the resident kernel does not
// take: the SpMV into w, then q = w + beta q, p = r + beta p, p.q, then the
// x, r update with r.r.
template <class T, class A>
cudaError_t cg_iteration(const spc5_matrix* M, T* x, T* r, T* p, T* q, T* w, int64_t n, double* scal, A* part,
                         int nb, unsigned* ticket, cudaStream_t s) {
  cudaError_t e = spmv_any(M, r, w, s);
  if (e == cudaSuccess) k_cg_pq<T, A><<<nb, kThreads, 0, s>>>(p, q, r, w, n, scal, part, ticket);
  if (e != cudaSuccess) return e;
  k_cg_xr_fused<T, A><<<nb, kThreads, 0, s>>>(x, r, p, q, n, scal, part, ticket);
  return cudaGetLastError();
}

// At most `steps` resident iterations queued on s (see k_cg_resident).
template <class T>
cudaError_t launch_resident(const ResLaunch& l, int64_t n, T* x, T* r, T* p, T* q, double* scal, ResState* res,
                            double stop, double fall, int every, int steps, cudaStream_t s) {
  Rows rows = l.rows;
  int held = l.held;
  long long limit = l.limit;
  void* args[] = {&n, &rows, &x, &r, &p, &q, &scal, &res, &stop, &fall, &every, &held, &steps, &limit};
  cudaError_t e = cudaMemsetAsync(res, 0, res_bytes(l.blocks), s);
  if (e == cudaSuccess) e = cudaLaunchCooperativeKernel(l.kern, dim3((unsigned)l.blocks), dim3(kResThreads), args, l.smem, s);
  return e;
}

// The unpacked rows of the handle that the iterations multiply by, for one solve.
struct UnpackedRows {
  Buf words, len, off, col, val;  // words: slots in use, then those handed out
  int64_t rows = 0;

  // first pass, queued; the caller reads words[0] with its next synchronisation
  cudaError_t count(const spc5_matrix* M, cudaStream_t s) {
    rows = (M->I * M->r + 31) / 32 * 32;
    cudaError_t e = words.alloc(2 * sizeof(unsigned long long), s);
    if (e == cudaSuccess) e = len.alloc(sizeof(int32_t) * (size_t)rows, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(words.p, 0, 2 * sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    const unsigned grid = (unsigned)((rows + kThreads - 1) / kThreads);
#define SPC5_CASE(RR, CC)         \
  if (M->r == RR && M->c == CC)   \
    k_rows_count<RR, CC><<<grid, kThreads, 0, s>>>(M->I, M->block_rowptr, M->block_masks, (int32_t*)len.p, \
                                                   (unsigned long long*)words.p);
    SPC5_CASE(1, 4) SPC5_CASE(1, 8) SPC5_CASE(1, 16)
    SPC5_CASE(2, 4) SPC5_CASE(2, 8) SPC5_CASE(2, 16)
    SPC5_CASE(4, 4) SPC5_CASE(4, 8) SPC5_CASE(4, 16)
    SPC5_CASE(8, 4) SPC5_CASE(8, 8) SPC5_CASE(8, 16)
#undef SPC5_CASE
    return cudaGetLastError();
  }

  template <class V>
  cudaError_t fill_as(const spc5_matrix* M, cudaStream_t s) {
    const unsigned grid = (unsigned)((rows + kThreads - 1) / kThreads);
#define SPC5_CASE(RR, CC)         \
  if (M->r == RR && M->c == CC)   \
    k_rows_fill<RR, CC, V><<<grid, kThreads, 0, s>>>(                                                          \
        M->I, M->block_rowptr, M->block_colidx, M->block_masks, (const V*)M->values, M->valptr, (int32_t*)len.p, \
        (int64_t*)off.p, (int32_t*)col.p, (V*)val.p, (unsigned long long*)words.p + 1);
    SPC5_CASE(1, 4) SPC5_CASE(1, 8) SPC5_CASE(1, 16)
    SPC5_CASE(2, 4) SPC5_CASE(2, 8) SPC5_CASE(2, 16)
    SPC5_CASE(4, 4) SPC5_CASE(4, 8) SPC5_CASE(4, 16)
    SPC5_CASE(8, 4) SPC5_CASE(8, 8) SPC5_CASE(8, 16)
#undef SPC5_CASE
    return cudaGetLastError();
  }

  void release() {
    for (Buf* b : {&words, &len, &off, &col, &val}) b->release();
  }

  // second pass; false where the rows are too uneven (or the memory too short)
  // to be laid side by side
  bool fill(const spc5_matrix* M, unsigned long long slots, cudaStream_t s, Rows* out) {
    // 32 rows padded to the longest of them: at most three times the entries
    if (slots == 0 || slots * 32ull > 3ull * (unsigned long long)M->nnz + 65536ull) return false;
    const size_t vs = value_size(M->vt);
    cudaError_t e = off.alloc(sizeof(int64_t) * (size_t)(rows / 32), s);
    if (e == cudaSuccess) e = col.alloc(sizeof(int32_t) * 32 * (size_t)slots, s);
    if (e == cudaSuccess) e = val.alloc(vs * 32 * (size_t)slots, s);
    if (e != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    e = vs == 8 ? fill_as<uint64_t>(M, s) : vs == 4 ? fill_as<uint32_t>(M, s) : fill_as<uint16_t>(M, s);
    *out = Rows{(const int32_t*)len.p, (const int64_t*)off.p, (const int32_t*)col.p, val.p};
    return e == cudaSuccess;
  }
};

// The resident kernel, launched for at most kResIterations iterations at a
// time, until sqrt(rho) <= stop or max_it. SPC5_ETIMEOUT: it was refused or gave
// up (the caller of cg_solve starts again without it).
constexpr int kResIterations = 4096;
constexpr size_t kSolveKeep = 1ull << 30;  // bytes the pool may keep after a solve that may have used more

spc5_status refused(cudaError_t e) {
  cudaGetLastError();
  return fail(SPC5_ETIMEOUT, std::string("cg: resident iterations: ") + cudaGetErrorName(e));
}

template <class T>
spc5_status cg_resident_loop(const ResLaunch& l, int64_t n, T* x, T* r, T* p, T* q, double* scal, ResState* res,
                             double stop, int max_it, double* host_scal, cudaStream_t s, int* iters) {
  *iters = 0;
  while (*iters < max_it) {
    const int steps = max_it - *iters < kResIterations ? max_it - *iters : kResIterations;
    cudaError_t e = launch_resident<T>(l, n, x, r, p, q, scal, res, stop, 0.0, 1, steps, s);
    if (e != cudaSuccess) return refused(e);
    e = cudaMemcpyAsync(host_scal, scal, sizeof(double) * S_COUNT, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "cg: resident iterations");
    if (host_scal[S_STATUS] != 0.0) return fail(SPC5_ETIMEOUT, "cg: a grid barrier gave up");
    *iters += (int)host_scal[S_ITERS];
    if (!(sqrt(host_scal[S_RHO]) > stop)) break;  // also stops on NaN
  }
  return SPC5_OK;
}

// Runs CG iterations until sqrt(rho) <= stop or max_it; iteration body
// replayed from a CUDA graph when use_graph. Returns iterations done.
// `keep`: when not NULL the instantiated graph is taken from / left in *keep
// for later calls with the same vectors (the caller destroys it).
template <class T, class A>
spc5_status cg_loop(const spc5_matrix* M, T* x, T* r, T* p, T* q, T* w, int64_t n, double* scal, A* part, int nb,
                    unsigned* ticket, const ResLaunch& l, ResState* res, double stop, int max_it, int check_every, bool use_graph,
                    double* host_scal, cudaStream_t s, int* iters, cudaGraphExec_t* keep = nullptr) {
  if (l.blocks > 0) return cg_resident_loop<T>(l, n, x, r, p, q, scal, res, stop, max_it, host_scal, s, iters);
  cudaGraphExec_t exec = keep ? *keep : nullptr;
  if (use_graph && !exec) {
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return cuda_fail(e, "cg: begin capture");
    cudaError_t e2 = cg_iteration<T, A>(M, x, r, p, q, w, n, scal, part, nb, ticket, s);
    e = cudaStreamEndCapture(s, &g);
    if (e2 != cudaSuccess) {
      if (g) cudaGraphDestroy(g);
      return cuda_fail(e2, "cg: capture");
    }
    if (e != cudaSuccess) return cuda_fail(e, "cg: end capture");
    e = cudaGraphInstantiate(&exec, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return cuda_fail(e, "cg: instantiate");
  }
  // Residual checks: the first after check_every iterations; then the
  // observed convergence rate predicts how many more are needed, and the next
  // check is placed there (between 2 and 8 x check_every iterations away).
  int k = 0, next = check_every;
  double prev_norm = -1.0;
  int prev_k = 0;
  spc5_status st = SPC5_OK;
  while (k < max_it) {
    int batch = next;
    if (batch > max_it - k) batch = max_it - k;
    cudaError_t e = cudaSuccess;
    for (int j = 0; j < batch && e == cudaSuccess; ++j)
      e = use_graph ? cudaGraphLaunch(exec, s) : cg_iteration<T, A>(M, x, r, p, q, w, n, scal, part, nb, ticket, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(host_scal, scal, sizeof(double) * S_COUNT, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
      st = cuda_fail(e, "cg: iteration");
      break;
    }
    k += batch;
    const double nr = sqrt(host_scal[S_RHO]);
    if (!(nr > stop)) break;  // also stops on NaN
    next = check_every;
    if (check_every > 1 && prev_norm > 0.0 && nr < prev_norm) {
      const double rate = log(nr / prev_norm) / (double)(k - prev_k);  // < 0
      const double need = log(stop / nr) / rate;
      int pred = (int)ceil(need);
      const int lo = check_every > 2 ? check_every / 4 : 1, hi = 8 * check_every;
      next = pred < lo ? lo : (pred > hi ? hi : pred);
    }
    prev_norm = nr;
    prev_k = k;
  }
  if (keep)
    *keep = exec;
  else if (exec)
    cudaGraphExecDestroy(exec);
  *iters = k;
  return st;
}

// One solve; `resident` allows the resident kernel.
spc5_status cg_solve(const spc5_matrix* A, const spc5_matrix* L, const double* b, double* x, const spc5_cg_opts* o,
                     spc5_cg_info* info, cudaStream_t user, bool resident) {
  const int64_t n = A->n;
  // vector kernels: grid-stride, at most kVecBlocksPerSm CTAs per SM (each
  // CTA adds one partial and one ticket to the reductions)
  int64_t nb64 = (n + kThreads - 1) / kThreads;
  if (nb64 > (int64_t)sm_count() * kVecBlocksPerSm) nb64 = (int64_t)sm_count() * kVecBlocksPerSm;
  const int nb = nb64 > 0 ? (int)nb64 : 1;
  const double tol = o->tol > 0 ? o->tol : 1e-10;
  const int max_it = o->max_iters > 0 ? o->max_iters : 100000;
  const int max_outer = o->max_outer > 0 ? o->max_outer : 30;
  const double inner_tol = o->inner_tol > 0 ? o->inner_tol : 1e-6;
  const int inner_max = o->inner_max_iters > 0 ? o->inner_max_iters : 2000;
  const int every = o->check_every > 0 ? o->check_every : 8;
  const bool use_graph = o->use_graph != 0;

  // private stream ordered after the caller's work (capture needs a real stream)
  cudaStream_t s = nullptr;
  cudaEvent_t ev = nullptr;
  cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventRecord(ev, user);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(s, ev, 0);
  if (e != cudaSuccess) {
    if (s) cudaStreamDestroy(s);
    if (ev) cudaEventDestroy(ev);
    return cuda_fail(e, "cg: stream");
  }
  struct Cleanup {
    cudaStream_t s;
    cudaEvent_t ev;
    cudaStream_t user;
    ~Cleanup() {
      cudaEventRecord(ev, s);
      cudaStreamWaitEvent(user, ev, 0);
      cudaStreamSynchronize(s);
      cudaStreamDestroy(s);
      cudaEventDestroy(ev);
    }
  } cleanup{s, ev, user};

  // partials: one per block of the vector updates
  const int64_t nparts = nb + 8;
  Buf scal_b, part_b, r_b, p_b, q_b, t_b, ticket_b, res_b;
  e = scal_b.alloc(sizeof(double) * S_COUNT, s);
  if (e == cudaSuccess) e = part_b.alloc(sizeof(double) * (size_t)nparts, s);
  if (e == cudaSuccess) e = ticket_b.alloc(sizeof(unsigned), s);
  if (e == cudaSuccess) e = cudaMemsetAsync(ticket_b.p, 0, sizeof(unsigned), s);
  if (e == cudaSuccess) e = res_b.alloc(res_bytes(sm_count() * kResPerSm), s);
  if (e == cudaSuccess) e = r_b.alloc(sizeof(double) * (size_t)n, s);
  if (e == cudaSuccess) e = p_b.alloc(sizeof(double) * (size_t)n, s);
  if (e == cudaSuccess) e = q_b.alloc(sizeof(double) * (size_t)n, s);
  if (e == cudaSuccess) e = t_b.alloc(sizeof(double) * (size_t)n, s);
  if (e != cudaSuccess) return cuda_fail(e, "cg: workspace");
  double* scal = (double*)scal_b.p;
  double* part = (double*)part_b.p;
  double* r = (double*)r_b.p;
  double* p = (double*)p_b.p;
  double* q = (double*)q_b.p;
  double* t = (double*)t_b.p;
  unsigned* ticket = (unsigned*)ticket_b.p;
  ResState* res = (ResState*)res_b.p;
  double hs[S_COUNT];
  e = cudaMemsetAsync(scal, 0, sizeof(double) * S_COUNT, s);
  if (e != cudaSuccess) return cuda_fail(e, "cg: init");

  // ||b||^2 into S_RHONEW's slot via a plain sum (b.b)
  k_dot_part<double, double><<<nb, kThreads, 0, s>>>(b, b, n, part);
  k_dot_final<double><<<1, kThreads, 0, s>>>(part, nb, scal, S_NORM);
  k_zero_vec<double><<<nb, kThreads, 0, s>>>(x, n);
  // the matrix of the iterations: its rows unpacked where the resident kernel can take them
  const spc5_matrix* M = L ? L : A;
  ResLaunch lres;
  UnpackedRows unpacked;
  unsigned long long slots = 0;
  if (resident && M->nseg == 0 && M->I > 0) {
    lres = M->vt == SPC5_F64 ? resident_kernel<F64>(n) : M->vt == SPC5_F32 ? resident_kernel<F32>(n) : resident_kernel<BF16>(n);
    if (o->wait_us > 0) lres.limit = 2000ll * o->wait_us;  // clocks: at most 2.07 per nanosecond
    if (lres.blocks > 0) {
      e = unpacked.count(M, s);
      if (e == cudaSuccess) e = cudaMemcpyAsync(&slots, unpacked.words.p, sizeof(slots), cudaMemcpyDeviceToHost, s);
      if (e != cudaSuccess) return cuda_fail(e, "cg: row lengths");
    }
  }
  e = cudaMemcpyAsync(hs, scal, sizeof(hs), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(e, "cg: norm of b");
  const double bnorm = sqrt(hs[S_NORM]);
  info->iterations = info->outer = info->inner_total = 0;
  info->converged = 0;
  info->rel_residual = 0.0;
  if (bnorm == 0.0) {  // x = 0 solves A x = 0
    info->converged = 1;
    return SPC5_OK;
  }
  if (lres.blocks > 0 && !unpacked.fill(M, slots, s, &lres.rows)) {
    unpacked.release();
    lres.blocks = 0;
  }
  const double stop = tol * bnorm;
  double rn_true = -1.0;  // the returned x's residual norm, once a solver has computed it
  spc5_status st = SPC5_OK;
  if (!L) {
    // float64 CG from x = 0: r = b, p = q = 0, beta = 0 (scal cleared), rho = b.b
    k_copy_vec<double><<<nb, kThreads, 0, s>>>(r, b, n);
    k_zero_vec<double><<<nb, kThreads, 0, s>>>(p, n);
    k_zero_vec<double><<<nb, kThreads, 0, s>>>(q, n);
    k_dot_part<double, double><<<nb, kThreads, 0, s>>>(r, r, n, part);
    k_dot_final<double><<<1, kThreads, 0, s>>>(part, nb, scal, S_RHO);
    int it = 0;
    st = cg_loop<double, double>(A, x, r, p, q, t, n, scal, part, nb, ticket, lres, res, stop, max_it, every, use_graph, hs, s,
                                 &it);
    info->iterations = it;
  } else if (o->reliable) {
    // float32 CG with reliable updates: one recurrence, never restarted; when
    // its residual norm has fallen by kReliableDelta since the last update,
    // x += x32 and r = b - A x in float64 replace the recurred quantities
    // (the search direction is kept, beta rescaled to the new residual)
    Buf r32_b, p32_b, q32_b, x32_b, w32_b, part32_b;
    e = r32_b.alloc(sizeof(float) * (size_t)n, s);
    if (e == cudaSuccess) e = p32_b.alloc(sizeof(float) * (size_t)n, s);
    if (e == cudaSuccess) e = q32_b.alloc(sizeof(float) * (size_t)n, s);
    if (e == cudaSuccess) e = x32_b.alloc(sizeof(float) * (size_t)n, s);
    if (e == cudaSuccess) e = w32_b.alloc(sizeof(float) * (size_t)n, s);
    if (e == cudaSuccess) e = part32_b.alloc(sizeof(float) * (size_t)nparts, s);
    if (e != cudaSuccess) return cuda_fail(e, "cg: workspace");
    float* r32 = (float*)r32_b.p;
    float* p32 = (float*)p32_b.p;
    float* q32 = (float*)q32_b.p;
    float* x32 = (float*)x32_b.p;
    float* w32 = (float*)w32_b.p;
    float* part32 = (float*)part32_b.p;
    // x = 0 (done), r = b; r32 = b, p32 = q32 = x32 = 0, beta = 0, rho = r32.r32
    k_copy_vec<double><<<nb, kThreads, 0, s>>>(r, b, n);
    k_narrow<<<nb, kThreads, 0, s>>>(b, r32, n);
    k_zero_vec<float><<<nb, kThreads, 0, s>>>(p32, n);
    k_zero_vec<float><<<nb, kThreads, 0, s>>>(q32, n);
    k_zero_vec<float><<<nb, kThreads, 0, s>>>(x32, n);
    k_dot_part<float, float><<<nb, kThreads, 0, s>>>(r32, r32, n, part32);
    k_dot_final<float><<<1, kThreads, 0, s>>>(part32, nb, scal, S_RHO);
    double rn_upd = bnorm;
    struct GraphKeep {
      cudaGraphExec_t g = nullptr;
      ~GraphKeep() {
        if (g) cudaGraphExecDestroy(g);
      }
    } keep;  // one captured iteration for all stretches between updates
    for (;;) {
      int it = 0;
      if (lres.blocks > 0) {
        // the kernel works out the target itself, and the update follows it
        // on the stream: the host looks once per stretch
        const int steps = max_it - info->inner_total < kResIterations ? max_it - info->inner_total : kResIterations;
        e = launch_resident<float>(lres, n, x32, r32, p32, q32, scal, res, stop, kReliableDelta, every, steps, s);
        if (e != cudaSuccess) return refused(e);
      } else {
        const double target = kReliableDelta * rn_upd > 0.5 * stop ? kReliableDelta * rn_upd : 0.5 * stop;
        st = cg_loop<float, float>(L, x32, r32, p32, q32, w32, n, scal, part32, nb, ticket, lres, res, target,
                                   max_it - info->inner_total, every, use_graph, hs, s, &it, &keep.g);
        if (st != SPC5_OK) return st;
      }
      // reliable update in float64
      k_fold_x<<<nb, kThreads, 0, s>>>(x, x32, n);
      e = spmv_any(A, x, t, s);
      if (e != cudaSuccess) return cuda_fail(e, "cg: residual spmv");
      k_replace_residual<<<nb, kThreads, 0, s>>>(r, r32, b, t, n, scal, part, part32, ticket);
      e = cudaMemcpyAsync(hs, scal, sizeof(hs), cudaMemcpyDeviceToHost, s);
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
      if (e != cudaSuccess) return cuda_fail(e, "cg: reliable update");
      if (hs[S_STATUS] != 0.0) return fail(SPC5_ETIMEOUT, "cg: a grid barrier gave up");
      if (lres.blocks > 0) it = (int)hs[S_ITERS];
      info->inner_total += it;
      info->outer += 1;
      rn_upd = sqrt(hs[S_NORM]);
      if (!(rn_upd > stop) || info->inner_total >= max_it || it == 0) break;
    }
    rn_true = rn_upd;  // of the x that is returned
    info->iterations = info->inner_total;
  } else {
    Buf r32_b, p32_b, q32_b, x32_b, w32_b, part32_b;
    e = r32_b.alloc(sizeof(float) * (size_t)n, s);
    if (e == cudaSuccess) e = p32_b.alloc(sizeof(float) * (size_t)n, s);
    if (e == cudaSuccess) e = w32_b.alloc(sizeof(float) * (size_t)n, s);
    if (e == cudaSuccess) e = q32_b.alloc(sizeof(float) * (size_t)n, s);
    if (e == cudaSuccess) e = x32_b.alloc(sizeof(float) * (size_t)n, s);
    if (e == cudaSuccess) e = part32_b.alloc(sizeof(float) * (size_t)nparts, s);
    if (e != cudaSuccess) return cuda_fail(e, "cg: workspace");
    float* r32 = (float*)r32_b.p;
    float* p32 = (float*)p32_b.p;
    float* q32 = (float*)q32_b.p;
    float* x32 = (float*)x32_b.p;
    float* w32 = (float*)w32_b.p;
    float* part32 = (float*)part32_b.p;
    // r = b (x = 0)
    k_copy_vec<double><<<nb, kThreads, 0, s>>>(r, b, n);
    k_dot_part<double, double><<<nb, kThreads, 0, s>>>(r, r, n, part);
    k_dot_final<double><<<1, kThreads, 0, s>>>(part, nb, scal, S_NORM);
    for (int outer = 0; outer < max_outer; ++outer) {
      e = cudaMemcpyAsync(hs, scal, sizeof(hs), cudaMemcpyDeviceToHost, s);
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
      if (e != cudaSuccess) return cuda_fail(e, "cg: residual norm");
      if (!(sqrt(hs[S_NORM]) > stop)) break;
      if (info->inner_total >= max_it) break;
      const double hs_norm = hs[S_NORM];
      // inner CG in float32 on A_low d = r / ||r||, from d = 0
      k_inner_start<<<nb, kThreads, 0, s>>>(r, r32, p32, q32, x32, n, scal);
      k_dot_part<float, float><<<nb, kThreads, 0, s>>>(r32, r32, n, part32);
      k_dot_final<float><<<1, kThreads, 0, s>>>(part32, nb, scal, S_RHO);
      e = cudaMemcpyAsync(hs, scal, sizeof(hs), cudaMemcpyDeviceToHost, s);
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
      if (e != cudaSuccess) return cuda_fail(e, "cg: inner start");
      int it = 0;
      const int budget = inner_max < max_it - info->inner_total ? inner_max : max_it - info->inner_total;
      // solve only as far as the final tolerance needs: a relative reduction of
      // half of tol * ||b|| / ||r||, but never looser than inner_tol allows
      // from below (float32 cannot reach much further than about 1e-6)
      double itol = 0.5 * stop / sqrt(hs_norm);
      if (itol < inner_tol) itol = inner_tol;
      if (itol > 0.5) itol = 0.5;
      st = cg_loop<float, float>(L, x32, r32, p32, q32, w32, n, scal, part32, nb, ticket, lres, res, itol * sqrt(hs[S_RHO]), budget,
                                 every, use_graph, hs, s, &it);
      if (st != SPC5_OK) return st;
      info->inner_total += it;
      // x += ||r|| d; r = b - A x in float64
      k_inner_apply<<<nb, kThreads, 0, s>>>(x, x32, n, scal);
      e = spmv_any(A, x, t, s);
      if (e != cudaSuccess) return cuda_fail(e, "cg: residual spmv");
      k_residual<<<nb, kThreads, 0, s>>>(r, b, t, n, part);
      k_dot_final<double><<<1, kThreads, 0, s>>>(part, nb, scal, S_NORM);
      info->outer = outer + 1;
    }
    info->iterations = info->inner_total;
  }
  if (st != SPC5_OK) return st;
  if (rn_true >= 0.0) {
    info->rel_residual = rn_true / bnorm;
    info->converged = info->rel_residual <= tol ? 1 : 0;
    return SPC5_OK;
  }
  // true residual of the returned x, in float64
  e = spmv_any(A, x, t, s);
  if (e != cudaSuccess) return cuda_fail(e, "cg: final residual");
  k_residual<<<nb, kThreads, 0, s>>>(r, b, t, n, part);
  k_dot_final<double><<<1, kThreads, 0, s>>>(part, nb, scal, S_NORM);
  e = cudaMemcpyAsync(hs, scal, sizeof(hs), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(e, "cg: final residual");
  info->rel_residual = sqrt(hs[S_NORM]) / bnorm;
  info->converged = info->rel_residual <= tol ? 1 : 0;
  return SPC5_OK;
}

}  // namespace

spc5_status cg_impl(const spc5_matrix* A, const spc5_matrix* L, const double* b, double* x, const spc5_cg_opts* o,
                    spc5_cg_info* info, cudaStream_t user) {
  spc5_status st = cg_solve(A, L, b, x, o, info, user, true);
  if (st == SPC5_ETIMEOUT) st = cg_solve(A, L, b, x, o, info, user, false);
  // A large solve's workspace does not stay in the pool: it is several times the
  // matrix, and the program may not solve again.
  const spc5_matrix* M = L ? L : A;
  const double bytes = (L ? 52.0 : 32.0) * (double)A->n + 3.0 * (double)M->nnz * (double)(4 + value_size(M->vt));
  if (bytes > (double)kSolveKeep) trim_scratch(kSolveKeep);
  return st;
}

}  // namespace spc5
