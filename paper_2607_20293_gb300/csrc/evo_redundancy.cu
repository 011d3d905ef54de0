// Redundancy-aware initialisation (Sec. 3.3): the dissimilarity map of Eq. 6
// from the residual activations of the uncached policy, its MSE / L1 /
// Wasserstein-1 variants, and guided sampling of fixed-budget schedules
// (Eq. 7).
//
// Activations come from evo_denoise_trace with the all-refresh lattice:
// trace [T][U][N][H][E] fp32.  For every unit b and sample r the T activations
// a_{r,b,t} (n = H*E entries each) give the pairwise terms
//   cosine : 1 - <a_t, a_t'> / (|a_t| |a_t'|)      (zero vector: 1)
//   mse    : mean (a_t - a_t')^2
//   l1     : mean |a_t - a_t'|
//   w1     : mean |sort(a_t) - sort(a_t')|          (Wasserstein-1 of the entries)
// and d_{r,b,t} = 1/(T-1) sum_{t' != t} of the term; d_{b,t} = mean over r.
//
// Pair kernel: a block per (b, r) streams its T rows through shared memory in
// chunks; every thread owns a register tile of (t, t') pairs of the symmetric
// matrix and keeps every sum in entry order.  Per-sample maps go to scratch and
// are averaged in a second pass in a fixed order (deterministic).
//
// Guided sampling: one block per schedule.  The Eq. 7 weights are taken in
// fixed point, q = floor((eps + d/max d)^gamma * 2^40) with IEEE double
// operations that are never contracted, and each draw picks, among the
// positions not yet drawn in index order, the first whose running sum of q
// exceeds rnd mod (sum of the remaining q) (only zero weights left: the
// first position not yet drawn).  All sums are exact 64-bit
// integers, so the schedule does not depend on the order of the warp's scan.

#include <cstdint>
#include <cuda_runtime.h>

#include "evo_internal.h"

namespace evo {

namespace {

constexpr int RM_MAX_T = 128;

enum { M_COS = 0, M_MSE = 1, M_L1 = 2, M_W1 = 3 };

__device__ __forceinline__ void cp16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// Cosine, mean square and mean absolute difference (of sorted rows:
// Wasserstein-1): one block per (b, r).
// Every pair's sum runs over the entries in index order, and every row's over
// the steps in order, so that the map is a fixed function of the trace whatever
// the tiling: a guided draw takes a 64-bit remainder by the sum of the weights,
// so a map that differs in its last bits draws other schedules.  The matrix is
// symmetric: a thread owns an RA x CB tile (rows RA i .. of t, CB j .. of t',
// on or above the diagonal) in registers.  8 x 4 for long loops: four entries
// take 12 16-byte loads for 128 multiply-adds.  Shorter loops have too few such
// tiles to fill their warps: 4 x 2 up to 64 steps (50 steps x 15 units x 7
// samples of 3,516 entries, mean square: 217 us with 8 x 4, 125 us), 2 x 2 up to
// 32 (25 steps x 15 x 7: 211 us with 8 x 4, 72 us).
// Groups of four rows lie 16 bytes off a multiple of 128, so neighbouring j
// start in distinct banks.
// Bound by FP32 issue and the shared loads.  Cosine map of 24 units x 16 samples
// x 100 steps x 4,096 entries: 1,279 us as the full matrix in 4 x 4 tiles ->
// 665 us in 8 x 8 packed tiles with the entries cut over blocks (which changed
// the sums) -> 580 us.  Wasserstein-1 of 24 units x 4 samples x 100 steps x 4,096
// entries, sort included: 735 us, and 632 with the entries cut over a cluster of
// blocks, whose sums depended on how many maps shared the call.
constexpr int OP_CH = 32, OP_STAGES = 4, OP_GROUP = 4 * OP_CH + 4;

__host__ __device__ constexpr int op_groups(int T) { return (T + 7) / 8 * 2; }   // groups of four rows
// tiles of T rows: row group i pairs with the column groups j >= i RA / CB
__host__ __device__ constexpr int op_tiles(int T, int RA, int CB) {
  const int nr = (T + RA - 1) / RA, f = RA / CB;
  return f * nr * (nr + 1) / 2;
}
constexpr int OP_SMALL_T = 32, OP_MID_T = 64;
constexpr int op_max_threads(int RA) { return RA == 2 ? 160 : 288; }
static_assert(op_tiles(RM_MAX_T, 8, 4) <= op_max_threads(8) && op_tiles(OP_MID_T, 4, 2) <= op_max_threads(4) &&
                  op_tiles(OP_SMALL_T, 2, 2) <= op_max_threads(2),
              "a tile per thread");
size_t op_smem(int T) {
  const size_t ring = (size_t)OP_STAGES * op_groups(T) * OP_GROUP, mat = (size_t)T * (T | 1) + T;
  return (ring > mat ? ring : mat) * sizeof(float);
}

template <int METRIC>
__device__ __forceinline__ float pair_op(float x, float y, float acc) {
  if constexpr (METRIC == M_COS) return fmaf(x, y, acc);
  if constexpr (METRIC == M_MSE) {
    const float e = x - y;
    return fmaf(e, e, acc);
  }
  return acc + fabsf(x - y);
}

template <int METRIC, int RA, int CB>
__global__ void __launch_bounds__(op_max_threads(RA), 2) ordered_pair_kernel(const float* rows, int T, int U, int N,
                                                                             int n, float* dr /* [U][N][T] */) {
  extern __shared__ __align__(16) float rm_smem[];
  const int b = blockIdx.x / N, r = blockIdx.x % N;
  const int ng = op_groups(T);
  constexpr int F = RA / CB;
  const int nr = (T + RA - 1) / RA;
  int ti = 0, tj = threadIdx.x;                         // tile number -> (i, j); row i holds F (nr - i) tiles
  while (ti < nr && tj >= F * (nr - ti)) {
    tj -= F * (nr - ti);
    ++ti;
  }
  const bool mine = ti < nr;
  tj += F * ti;
  float acc[RA][CB];
#pragma unroll
  for (int a = 0; a < RA; ++a)
#pragma unroll
    for (int c = 0; c < CB; ++c) acc[a][c] = 0.f;
  auto row = [](int t) { return (t >> 2) * OP_GROUP + (t & 3) * OP_CH; };
  const int nch = (n + OP_CH - 1) / OP_CH;
  const bool vec = (n & 3) == 0 && (reinterpret_cast<uintptr_t>(rows) & 15) == 0;
  const long long step = (long long)U * N * n;          // floats between rows t and t + 1
  const float* base = rows + ((long long)b * N + r) * n;
  // chunk c -> buffer c % OP_STAGES; a ragged or unaligned row by plain loads, zero-padded
  auto load_chunk = [&](int c) {
    if (c < nch) {
      float* xs = rm_smem + (c % OP_STAGES) * ng * OP_GROUP;
      const int c0 = c * OP_CH;
      for (int v = threadIdx.x; v < T * (OP_CH / 4); v += blockDim.x) {
        const int t = v / (OP_CH / 4), k = 4 * (v % (OP_CH / 4)), w = n - c0 - k;
        const float* src = base + t * step + c0 + k;
        float* dst = xs + row(t) + k;
        if (w > 3 && vec) {
          cp16(dst, src);
        } else {
          float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
          if (w > 0) f.x = src[0];
          if (w > 1) f.y = src[1];
          if (w > 2) f.z = src[2];
          if (w > 3) f.w = src[3];
          *reinterpret_cast<float4*>(dst) = f;
        }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int s = 0; s < OP_STAGES - 1; ++s) load_chunk(s);
  for (int c = 0; c < nch; ++c) {
    asm volatile("cp.async.wait_group %0;" ::"n"(OP_STAGES - 2) : "memory");
    __syncthreads();                                    // chunk c is there, chunk c - 1 has been read
    load_chunk(c + OP_STAGES - 1);
    if (mine) {
      const float* xs = rm_smem + (c % OP_STAGES) * ng * OP_GROUP;
      const float *xr = xs + row(RA * ti), *yr = xs + row(CB * tj);
#pragma unroll(RA == 8 ? 1 : 8 / RA)
      for (int k = 0; k < OP_CH; k += 4) {
        float4 y[CB];
#pragma unroll
        for (int q = 0; q < CB; ++q) y[q] = *reinterpret_cast<const float4*>(yr + q * OP_CH + k);
#pragma unroll
        for (int a = 0; a < RA; ++a) {
          const float4 x = *reinterpret_cast<const float4*>(xr + (a >> 2) * OP_GROUP + (a & 3) * OP_CH + k);
#pragma unroll
          for (int q = 0; q < CB; ++q) {
            float v = acc[a][q];
            v = pair_op<METRIC>(x.x, y[q].x, v);
            v = pair_op<METRIC>(x.y, y[q].y, v);
            v = pair_op<METRIC>(x.z, y[q].z, v);
            v = pair_op<METRIC>(x.w, y[q].w, v);
            acc[a][q] = v;
          }
        }
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // the matrix takes the ring's place: rows of T | 1 floats, then the norms
  const int ld = T | 1;
  float* norm = rm_smem + T * ld;
  if (mine) {
#pragma unroll
    for (int a = 0; a < RA; ++a)
#pragma unroll
      for (int c = 0; c < CB; ++c) {
        const int t = RA * ti + a, t2 = CB * tj + c;
        if (t < T && t2 < T) {
          rm_smem[t * ld + t2] = acc[a][c];
          rm_smem[t2 * ld + t] = acc[a][c];             // (within the diagonal tiles: the same value twice)
        }
      }
  }
  __syncthreads();
  if (METRIC == M_COS) {
    for (int t = threadIdx.x; t < T; t += blockDim.x) norm[t] = sqrtf(rm_smem[t * ld + t]);
    __syncthreads();
  }
  for (int i = threadIdx.x; i < T * T; i += blockDim.x) {
    const int t = i / T, t2 = i - t * T;
    float* g = rm_smem + t * ld + t2;
    if (METRIC == M_COS) {
      const float nn = norm[t] * norm[t2];
      *g = nn == 0.f ? 1.f : 1.f - *g / nn;
    } else {
      *g = *g / (float)n;
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < T; t += blockDim.x) {
    float s = 0.f;
    for (int t2 = 0; t2 < T; ++t2)
      if (t2 != t) s += rm_smem[t * ld + t2];
    dr[((long long)b * N + r) * T + t] = s / (float)(T - 1);
  }
}

// d[b][t] = mean over r of dr[b][r][t], summed in order r = 0..N-1
__global__ void mean_kernel(const float* dr, int T, int U, int N, float* d) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= U * T) return;
  const int b = i / T, t = i % T;
  float s = 0.f;
  for (int r = 0; r < N; ++r) s += dr[((long long)b * N + r) * T + t];
  d[i] = s / (float)N;
}

// A float's place in the order, as a signed integer (and back): a sort by
// integer minimum and maximum moves every value, NaN among them, and loses none.
__device__ __forceinline__ int order_key(float f) {
  const int i = __float_as_int(f);
  return i ^ ((i >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float key_value(int k) { return __int_as_float(k ^ ((k >> 31) & 0x7fffffff)); }

constexpr int SR_V = 16, SR_LV = 4;   // entries per thread

// shared index of entry i: one word of padding per 32, so that a thread's 16
// entries and a stride-16 set of them both spread over the banks
__device__ __forceinline__ int sr_at(int i) { return i + (i >> 5); }

// Ascending bitonic sort of rows of n = 2^LN entries, 2^(LN - 4) threads per
// row, 16 entries of the row per thread in registers.  The compare distances of
// a merge are taken four at a time: in layout s a thread holds the 16 entries
// whose index differs in bits s .. s + 3, so four distances need one exchange
// through shared memory.  Bound by shared-memory exchanges and integer min/max.
// 9,600 rows of 4,096: 1,634 us in shared memory alone -> 345 us; 480 rows of
// 16,384: 960 -> 180 us.
template <int LN>
__global__ void __launch_bounds__(LN <= 12 ? 256 : (1 << (LN - SR_LV))) sort_rows_reg_kernel(const float* in, float* out,
                                                                                          long long n_rows) {
  constexpr int N = 1 << LN, TPR = N / SR_V;            // threads per row
  constexpr int RPB = LN <= 12 ? 256 / TPR : 1;         // rows per block
  extern __shared__ __align__(16) float srt[];
  const int sub = threadIdx.x / TPR, tr = threadIdx.x % TPR;
  const long long row = (long long)blockIdx.x * RPB + sub;
  const bool live = row < n_rows;
  int* sh = reinterpret_cast<int*>(srt) + sub * (N + N / 32);
  // coalesced load into shared memory
  if (live)
    for (int i = tr; i < N; i += TPR) sh[sr_at(i)] = order_key(in[row * N + i]);
  __syncthreads();
  int v[SR_V];
  // entry e of this thread in layout s: the thread number's low s bits, then e, then its other bits
  auto index = [&](int s, int e) { return (tr & ((1 << s) - 1)) | (e << s) | ((tr >> s) << (s + SR_LV)); };
  auto load = [&](int s) {
#pragma unroll
    for (int e = 0; e < SR_V; ++e) v[e] = sh[sr_at(index(s, e))];
  };
  auto store = [&](int s) {
#pragma unroll
    for (int e = 0; e < SR_V; ++e) sh[sr_at(index(s, e))] = v[e];
  };
  load(0);
#pragma unroll
  for (int k = 1; k <= LN; ++k) {                       // merges of 2^k entries
    int cur = 0;                                        // layout at hand
#pragma unroll
    for (int hi = k - 1; hi >= 0; hi -= SR_LV) {        // distances 2^hi .. 2^lo
      const int s = hi - (SR_LV - 1) > 0 ? hi - (SR_LV - 1) : 0;
      if (s != cur) {
        store(cur);
        __syncthreads();
        load(s);                                        // the entries it stores next: no barrier needed in between
        cur = s;
      }
#pragma unroll
      for (int j = hi; j >= s; --j) {
        const int d = 1 << (j - s);
#pragma unroll
        for (int e = 0; e < SR_V; ++e)
          if (!(e & d)) {
            const bool up = (index(s, e) & (1 << k)) == 0;
            const int lo = min(v[e], v[e | d]), up_v = max(v[e], v[e | d]);
            v[e] = up ? lo : up_v;
            v[e | d] = up ? up_v : lo;
          }
      }
      if (s == 0 && cur == 0) break;
    }
  }
  store(0);
  __syncthreads();
  if (live)
    for (int i = tr; i < N; i += TPR) out[row * N + i] = key_value(sh[sr_at(i)]);
}

template <int LN>
cudaError_t sort_rows_reg(const float* in, float* out, long long n_rows, cudaStream_t st) {
  constexpr int N = 1 << LN, TPR = N / SR_V, RPB = LN <= 12 ? 256 / TPR : 1;
  const int sm = RPB * (N + N / 32) * (int)sizeof(int);
  const cudaError_t e =
      cudaFuncSetAttribute(sort_rows_reg_kernel<LN>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
  if (e != cudaSuccess) return e;
  sort_rows_reg_kernel<LN><<<(unsigned)((n_rows + RPB - 1) / RPB), RPB * TPR, sm, st>>>(in, out, n_rows);
  return cudaGetLastError();
}

// The same in shared memory alone, one block per row: rows of fewer than 256
// entries, which do not fill a warp of the register sort.
__global__ void sort_rows_kernel(const float* in, float* out, int n) {
  extern __shared__ __align__(16) float srt[];
  const float* src = in + (long long)blockIdx.x * n;
  for (int i = threadIdx.x; i < n; i += blockDim.x) srt[i] = src[i];
  __syncthreads();
  for (int k = 2; k <= n; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int l = i ^ j;
        if (l > i) {
          const float a = srt[i], c = srt[l];
          const bool up = (i & k) == 0;
          if ((a > c) == up) {
            srt[i] = c;
            srt[l] = a;
          }
        }
      }
      __syncthreads();
    }
  float* dst = out + (long long)blockIdx.x * n;
  for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = srt[i];
}

constexpr int GS_MAX_CELLS = 4096;

constexpr int GS_THREADS = 128;

// One block per schedule p.  All warps set the weights up; warp 0 draws.  The
// cells are cut into 32 runs of `ch` cells; lane l holds the inclusive sum of
// the remaining weights of runs 0 .. l, and `pre` the inclusive sums within
// each run, so a draw finds its run with one ballot and its cell with at most
// four, and then takes the drawn weight off the sums behind it: a few dozen
// dependent instructions per draw instead of a pass over every cell.  Bound by
// that chain (64-bit remainder, two shared-memory round trips): 64 schedules of
// 240 of 2,400 cells 1,283 -> 134 us, of which about 20 us are the weights
// (double precision, which this chip does at two operations per clock and SM).
__global__ void __launch_bounds__(GS_THREADS) guided_kernel(const float* d, int cells, int K, float eps, int gamma,
                                                            const unsigned long long* rnd, uint8_t* S) {
  __shared__ unsigned long long pre[GS_MAX_CELLS];
  __shared__ uint8_t taken[GS_MAX_CELLS];
  __shared__ float wmax[GS_THREADS / 32];
  const int p = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float mx = 0.f;
  for (int i = threadIdx.x; i < cells; i += GS_THREADS) mx = fmaxf(mx, d[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) wmax[warp] = mx;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < GS_THREADS / 32; ++w) mx = fmaxf(mx, wmax[w]);
  const double e = (double)eps, dm = (double)mx;
  for (int i = threadIdx.x; i < cells; i += GS_THREADS) {
    const double base = __dadd_rn(e, __ddiv_rn((double)d[i], dm));
    double v = base;
    for (int g = 1; g < gamma; ++g) v = __dmul_rn(v, base);
    pre[i] = (unsigned long long)(long long)floor(__dmul_rn(v, 1099511627776.0));
    taken[i] = 0;
  }
  __syncthreads();
  if (warp == 0) {
    const int ch = (cells + 31) / 32, lo = min(cells, lane * ch), hi = min(cells, lo + ch);
    unsigned long long part = 0;
    for (int i = lo; i < hi; ++i) {
      part += pre[i];
      pre[i] = part;
    }
    unsigned long long incl = part;                     // of runs 0 .. lane
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long up = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += up;
    }
    __syncwarp();
    unsigned long long next = K > 0 ? rnd[(long long)p * K] : 0ull;
    for (int k = 0; k < K; ++k) {
      const unsigned long long total = __shfl_sync(0xffffffffu, incl, 31);
      const unsigned long long rk = next;
      if (k + 1 < K) next = rnd[(long long)p * K + k + 1];
      if (total == 0) {
        // only zero weights left: the first position not yet drawn
        for (int i0 = 0; i0 < cells; i0 += 32) {
          const unsigned has = __ballot_sync(0xffffffffu, i0 + lane < cells && !taken[i0 + lane]);
          if (has) {
            if (lane == 0) taken[i0 + __ffs(has) - 1] = 1;
            break;
          }
        }
        __syncwarp();
        continue;
      }
      const unsigned long long target = rk % total;
      const int run = __ffs(__ballot_sync(0xffffffffu, incl > target)) - 1;
      // sum of the runs in front; the comparison below adds to it, so that sums that
      // wrap around (large eps and gamma) pick what a plain running sum picks
      const unsigned long long front = __shfl_sync(0xffffffffu, incl, run > 0 ? run - 1 : 0);
      const unsigned long long before = run > 0 ? front : 0ull;
      const int c0 = run * ch, cn = min(ch, cells - c0);
      int sel = -1;
      unsigned long long mine[4];                       // this lane's cells of the run: lane, lane + 32, ...
#pragma unroll
      for (int j = 0; j < 4; ++j) mine[j] = lane + 32 * j < cn ? pre[c0 + lane + 32 * j] : 0ull;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const unsigned hit = __ballot_sync(0xffffffffu, lane + 32 * j < cn && before + mine[j] > target);
        if (sel < 0 && hit) sel = 32 * j + __ffs(hit) - 1;
      }
      const unsigned long long w = pre[c0 + sel] - (sel > 0 ? pre[c0 + sel - 1] : 0ull);
      __syncwarp();
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (lane + 32 * j < cn && lane + 32 * j >= sel) pre[c0 + lane + 32 * j] = mine[j] - w;
      if (lane == 0) taken[c0 + sel] = 1;
      if (lane >= run) incl -= w;
      __syncwarp();
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < cells; i += GS_THREADS) S[(long long)p * cells + i] = taken[i];
}

template <int METRIC, int RA, int CB>
cudaError_t launch_ordered_pair_as(const float* rows, int T, int U, int N, int n, float* dr, cudaStream_t st) {
  const cudaError_t e = cudaFuncSetAttribute(ordered_pair_kernel<METRIC, RA, CB>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)op_smem(RM_MAX_T));
  if (e != cudaSuccess) return e;
  const int threads = (op_tiles(T, RA, CB) + 31) / 32 * 32;
  ordered_pair_kernel<METRIC, RA, CB><<<U * N, threads, op_smem(T), st>>>(rows, T, U, N, n, dr);
  return cudaGetLastError();
}

template <int METRIC>
cudaError_t launch_ordered_pair(const float* rows, int T, int U, int N, int n, float* dr, cudaStream_t st) {
  return T > OP_MID_T     ? launch_ordered_pair_as<METRIC, 8, 4>(rows, T, U, N, n, dr, st)
         : T > OP_SMALL_T ? launch_ordered_pair_as<METRIC, 4, 2>(rows, T, U, N, n, dr, st)
                          : launch_ordered_pair_as<METRIC, 2, 2>(rows, T, U, N, n, dr, st);
}

}  // namespace

// floats of the per-sample maps at the start of the scratch, a multiple of 16
// bytes: the sorted rows behind them are read by 16-byte copies
static size_t map_floats(int T, int U, int N) { return ((size_t)U * N * T + 3) & ~size_t(3); }

size_t redundancy_scratch_bytes(int T, int U, int N, int n, int metric) {
  size_t b = map_floats(T, U, N) * sizeof(float);
  if (metric == M_W1) b += (size_t)T * U * N * n * sizeof(float);
  return b;
}

bool redundancy_shape_ok(int T, int U, int N, int n, int metric) {
  if (T < 2 || T > RM_MAX_T || U <= 0 || N <= 0 || n <= 0 || metric < 0 || metric > M_W1) return false;
  if (metric == M_W1 && ((n & (n - 1)) != 0 || n > 16384)) return false;   // bitonic sort in shared memory
  return true;
}

cudaError_t launch_redundancy(const float* trace, int T, int U, int N, int n, int metric, float* d, void* scratch,
                              cudaStream_t st) {
  float* dr = static_cast<float*>(scratch);
  const float* rows = trace;
  if (metric == M_W1) {
    float* sorted = dr + map_floats(T, U, N);
    const long long n_rows = (long long)T * U * N;
    cudaError_t e = cudaSuccess;
    switch (n) {
      case 256: e = sort_rows_reg<8>(trace, sorted, n_rows, st); break;
      case 512: e = sort_rows_reg<9>(trace, sorted, n_rows, st); break;
      case 1024: e = sort_rows_reg<10>(trace, sorted, n_rows, st); break;
      case 2048: e = sort_rows_reg<11>(trace, sorted, n_rows, st); break;
      case 4096: e = sort_rows_reg<12>(trace, sorted, n_rows, st); break;
      case 8192: e = sort_rows_reg<13>(trace, sorted, n_rows, st); break;
      case 16384: e = sort_rows_reg<14>(trace, sorted, n_rows, st); break;
      default: sort_rows_kernel<<<T * U * N, 128, n * sizeof(float), st>>>(trace, sorted, n);
    }
    if (e != cudaSuccess) return e;
    rows = sorted;
  }
  cudaError_t e = cudaSuccess;
  switch (metric) {
    case M_COS: e = launch_ordered_pair<M_COS>(rows, T, U, N, n, dr, st); break;
    case M_MSE: e = launch_ordered_pair<M_MSE>(rows, T, U, N, n, dr, st); break;
    default: e = launch_ordered_pair<M_L1>(rows, T, U, N, n, dr, st);   // (w1: of the sorted rows)
  }
  if (e != cudaSuccess) return e;
  mean_kernel<<<(U * T + 255) / 256, 256, 0, st>>>(dr, T, U, N, d);
  return cudaGetLastError();
}

bool guided_shape_ok(int U, int T, int K, int gamma, int P) {
  return U > 0 && T > 0 && U * T <= GS_MAX_CELLS && K >= 0 && K <= U * T && gamma >= 1 && gamma <= 16 && P > 0;
}

cudaError_t launch_guided(const float* d, int U, int T, int K, float eps, int gamma, const uint64_t* rnd, int P,
                          uint8_t* S, cudaStream_t st) {
  guided_kernel<<<P, GS_THREADS, 0, st>>>(d, U * T, K, eps, gamma, reinterpret_cast<const unsigned long long*>(rnd), S);
  return cudaGetLastError();
}

}  // namespace evo
