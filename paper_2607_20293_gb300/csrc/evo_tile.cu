// The tile path: one persistent kernel in which a CTA runs the whole T-step
// loop of a job -- up to 8 samples (128 action-token rows) of one lattice -- on
// the fifth-generation tensor cores (tcgen05), with no other CTA involved.
// Models of n_emb 256, 4 heads of 64, horizon 16 (a sample is 16 rows).
//
// Why this shape.  Between a refreshed unit and the next nothing crosses a
// sample, so a job needs no grid-wide step; what the batch-wide path pays per
// lattice cell (three or four launches over the rows of every sample, of which
// few are live when the lattices differ, and a round trip of the residual
// stream, of r, q|k|v and the hidden layer through L2) is gone.  128 rows fill
// one tcgen05 M, and the residual stream fits the registers of eight warps.
//
// On chip:
//   * residual stream: fp32 in registers.  A compute warp owns one sample (16
//     rows), in the layout of mma.sync accumulators (tcgen05.ld 16x256b): lane
//     4 g + q holds columns 8 j + 2 q, + 1 of rows g and g + 8.  Row sums need
//     two shuffles and no other warp, and a bias is loaded once for two rows.
//     (A thread per row half, the 32x32b layout, loads every bias as a
//     broadcast, whose 16 bytes a lane cost as much as any other 512-byte load,
//     and exchanges its sums through shared memory: LayerNorm 7,200 cycles.)
//   * tensor memory, 512 columns: R (256: the second GEMM's accumulator) and
//     two accumulators of 128 columns for the first GEMM, so that the epilogue
//     of one chunk overlaps the MMAs of the next;
//   * shared memory: the normalised rows (64 KiB, 128-byte-swizzled A operand),
//     two 32 KiB buffers of the second GEMM's A operand (attention output,
//     hidden-layer chunks), a ring of five 16 KiB weight slots, and the vectors
//     (LayerNorm, biases) of this unit and the next.
// Weights are packed at creation in the order in which the MMAs consume them,
// as swizzled shared-memory images, and stream through the ring by one bulk
// copy (cp.async.bulk) per slot; skipped units move no weights.  The vectors
// come the same way: read where they are used, from L2 through the 20 KiB of
// L1 that are left, they cost more than everything else (a LayerNorm 7,900
// cycles; a call of 8 samples at full refresh 43.4 ms).  The tables of the
// output head and the input embedding are copied into the free operand buffers
// at each step's end.
//
// A refreshed unit: LayerNorm -> first GEMM in chunks of 128 columns ->
// per-chunk epilogue -> second GEMM accumulating in R -> r: a += r, c_b <- bf16(r).
//   SA   chunks q|k of heads 0, 1, v of both, q|k of 2, 3, v of both; the warp
//        does its sample's causal attention in registers (q, k and v arrive as
//        fragments);
//   CA   q of heads 0|1 and 2|3, at most 8 memory tokens;
//   FFN  8 chunks of the hidden layer with GELU; the second GEMM consumes chunk
//        c while chunk c + 2 is computed.
// The unit caches live in global memory in the order of the threads that own
// the values (a thread reads back only what it wrote itself).
//
// Bound by instruction issue and its dependent chains on two compute warps per
// SM sub-partition (the register file holds no more of them beside the stream:
// with sixteen warps of half a row the compiler spills it).  A unit takes about
// 14 us.  64 candidates x 16 observations and their reference (n_emb 256, 8
// layers, 100 steps): 97.5 ms batch-wide -> 33.9 ms, the reference's 2,400
// units; 300 samples at refresh fraction 0.125: 10.3 -> 7.1 ms.
//
// Warps 0-7 compute, warp 8 streams weights, warp 9 issues the MMAs (10 and 11
// only complete the third warpgroup, which gives its registers away).  Every
// wait on an mbarrier is bounded, and once one was in vain none waits any more
// (mbar_wait_live, evo_tc.cuh): no copy is issued from then on, the copying and
// the issuing warp leave after their unit, and the compute warps, which meet at
// barriers of their own, leave together at the next step's end.  What is computed
// until then stays in bounds and is worthless; the status word says so.

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "evo_internal.h"
#include "evo_tc.cuh"

namespace evo {

namespace {

using namespace tc;

constexpr int TE = 256, TH = 16;                      // n_emb (4 heads of 64), horizon
constexpr int TROWS = 128, TG = TROWS / TH;           // rows and samples of a job
constexpr int TCW = 8, TCT = TCW * 32;                // compute warps, threads
// three warpgroups; registers per thread after the split: 256 x 200 + 128 x 104
// = 384 x 168, what the block is launched with
constexpr int TTHREADS = TCT + 128;
constexpr int SLOT = 16384, NSLOTS = 5;
constexpr int XLN_BYTES = TROWS * TE * 2;             // four 64-column blocks of 16 KiB
constexpr int HID_BYTES = TROWS * 128 * 2;            // one chunk: two 64-column blocks
// vectors of a unit: LayerNorm gain, shift, second bias (256 each), first bias
__host__ __device__ constexpr int n_bias1(int u) { return u == 0 ? 768 : (u == 1 ? 256 : 1024); }
__host__ __device__ constexpr int vec_floats(int u) { return 768 + n_bias1(u); }
__host__ __device__ constexpr int vec_off(int u) {
  return u == 0 ? 0 : (u == 1 ? vec_floats(0) : vec_floats(0) + vec_floats(1));
}
constexpr int VEC_LAYER = vec_floats(0) + vec_floats(1) + vec_floats(2);
constexpr int VEC_BYTES = vec_floats(2) * 4;
constexpr int TILE_SMEM = 1024 + XLN_BYTES + 2 * HID_BYTES + NSLOTS * SLOT + 2 * VEC_BYTES + 256;
// step-end tables: W_head^T and W_in [A][256], b_in + P_pos [32][16][8], LN_f gain and shift
__host__ __device__ constexpr int tab_floats(int A) { return 2 * A * TE + 64 * TH * 4 + 2 * TE; }
static_assert(tab_floats(16) * 4 <= 2 * HID_BYTES, "step-end tables in the operand buffers");
static_assert(TILE_SMEM <= 232448, "shared memory per block");

// chunks of the first GEMM (128 columns, K = 256) and of the second (K = 128,
// 256 columns) by unit kind (SA, CA, FFN); a slot is a 128-row, 64-column block
__host__ __device__ constexpr int n_first(int u) { return u == 0 ? 6 : (u == 1 ? 2 : 8); }
__host__ __device__ constexpr int n_second(int u) { return u == 2 ? 8 : 2; }
__host__ __device__ constexpr int unit_slots(int u) { return 4 * (n_first(u) + n_second(u)); }
__host__ __device__ constexpr int unit_slot0(int u) {   // first slot of the kind inside a layer
  return u == 0 ? 0 : (u == 1 ? unit_slots(0) : unit_slots(0) + unit_slots(1));
}
constexpr int LAYER_SLOTS = unit_slots(0) + unit_slots(1) + unit_slots(2);

struct TileParams {
  int L, A, n_obs, T, U;
  int n_jobs, jobs_per_lat, per_sched, obs_mod, sampler;
  const int* order;                // lattices in the order in which their jobs are taken, or null
  const uint64_t* mask;            // [n_sched][T][2]: units refreshed at t, units whose cache holds a value
  const uint8_t* wpack;            // [L][LAYER_SLOTS][SLOT]
  const float* vec;                // [L][VEC_LAYER]
  const float* tab;                // [tab_floats(A)]
  const float* head_b;             // [A]
  const float* stab;               // [T][8]
  const float* noise;              // [n_noise][obs_mod][16][A]
  // memory keys | values in bf16, the 64 values of a head in the order in which
  // a lane reads them (tile_kv_column)
  const __nv_bfloat16* kv_time;    // [T][L][512]
  const __nv_bfloat16* kv_obs;     // [obs_mod][n_obs][L][512]
  uint4* cache;                    // [grid][U][16][256]: thread-ordered bf16
  float* out;                      // [samples][16][A]
  float* trace;                    // TRACE: [T][U][rows][256], what every cell adds to the stream
  long long rows;                  // rows of the call
  float scale;
  int* status;
  long long wait_limit;
};

__device__ __forceinline__ void bar_compute() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
// the same; true in every thread if x is in one
__device__ __forceinline__ bool bar_compute_any(bool x) {
  uint32_t r;
  asm volatile("{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, 1, 256, p;\n selp.u32 %0, 1, 0, q;\n}\n"
               : "=r"(r)
               : "r"((uint32_t)x)
               : "memory");
  return r != 0;
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ uint64_t desc64(uint32_t lo, uint32_t hi) { return ((uint64_t)hi << 32) | lo; }
__device__ __noinline__ void wait_slow(uint32_t bar, uint32_t parity, int* status, long long limit, uint32_t dead) {
  mbar_wait_live(bar, parity, status, limit, dead);
}

// 16 rows x 32 (64) fp32 columns in the layout of mma.sync accumulators: tile j
// (columns 8 j ..) holds rows lane / 4 (v[j][0..1]) and + 8 (v[j][2..3]),
// columns 2 (lane % 4) and + 1
__device__ __forceinline__ void tmem_ld_frag(uint32_t taddr, float (&v)[4][4]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
      "[%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i >> 2][i & 3] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld_frag(uint32_t taddr, float (&v)[8][4]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i >> 2][i & 3] = __uint_as_float(r[i]);
}

// 16 columns of it, issued ahead: the registers hold them after tmem_wait
__device__ __forceinline__ void tmem_ld_ahead(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
               :
               : "memory");
}

__device__ __forceinline__ uint32_t pk2(float x, float y) {
  __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  return *reinterpret_cast<uint32_t*>(&h);
}

__device__ __forceinline__ uint32_t movm(uint32_t x) {   // 8 x 8 bf16 transpose across the warp
  uint32_t y;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}

__device__ __forceinline__ void mma_k16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void mma_k8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5}, {%6}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(b0));
}

__device__ __forceinline__ float2 bf2(uint32_t u) {
  return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u));
}

__device__ __forceinline__ float2 fma_x2(float2 a, float2 b, float2 c) {   // packed, IEEE (no flush)
  float2 d;
  asm("{\n .reg .b64 ra, rb, rc, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n mov.b64 rc, {%6, %7};\n"
      " fma.rn.f32x2 rd, ra, rb, rc;\n mov.b64 {%0, %1}, rd;\n}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ float2 mul_x2(float2 a, float2 b) {
  float2 d;
  asm("{\n .reg .b64 ra, rb, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n"
      " mul.rn.f32x2 rd, ra, rb;\n mov.b64 {%0, %1}, rd;\n}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }

// four 8 x 8 bf16 tiles (rows 0-7 | 8-15 of tile n, the same of n + 1) into a
// 64-column block of 128-byte swizzled rows, from row row0 (a multiple of 16)
__device__ __forceinline__ void put_tiles(uint8_t* blk, int row0, int n, int lane, uint32_t t0, uint32_t t1, uint32_t t2,
                                          uint32_t t3) {
  const int r = lane & 15;                 // lane's row address: matrix lane / 8, its row lane % 8
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(
                   su32(blk + (row0 + r) * 128 + (((n + (lane >> 4)) ^ (r & 7)) << 4))),
               "r"(t0), "r"(t1), "r"(t2), "r"(t3)
               : "memory");
}

__device__ __forceinline__ void arrive_warp(uint64_t* bar, int lane) {
  __syncwarp();
  if (lane == 0) mbar_arrive1(bar);
}

// the same value in every lane, and known to the compiler to be
__device__ __forceinline__ uint64_t uniform64(uint64_t v) {
  const uint32_t lo = __shfl_sync(0xffffffffu, (uint32_t)v, 0), hi = __shfl_sync(0xffffffffu, (uint32_t)(v >> 32), 0);
  return ((uint64_t)hi << 32) | lo;
}

struct Bars {
  uint64_t full[NSLOTS], empty[NSLOTS];   // weight ring
  uint64_t vfull[2], vempty[2];           // vectors of a unit: landed / read (8 warps)
  uint64_t xready;                        // normalised rows written (8 warps)
  uint64_t afull[2], aempty[2];           // first-GEMM accumulators: finished (commit) / drained (8 warps)
  uint64_t hready[2], hempty[2];          // second-GEMM operand buffers: written (8 warps) / consumed (commit)
  uint64_t rfull;                         // R finished (commit)
  uint32_t tslot;
  uint32_t dead;                          // a wait was in vain
};

// mean and 1/std of the lane's two rows (64 columns each, the rest in the quad's
// other lanes)
__device__ __forceinline__ void tile_stats(const float2 (&a)[2][32], float (&mean)[2], float (&rstd)[2]) {
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    float2 s[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) s[j] = a[r][j];
#pragma unroll
    for (int j = 4; j < 32; ++j) s[j & 3] = add2(s[j & 3], a[r][j]);
    s[0] = add2(add2(s[0], s[1]), add2(s[2], s[3]));
    mean[r] = s[0].x + s[0].y;
  }
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
    mean[0] += __shfl_xor_sync(0xffffffffu, mean[0], o);
    mean[1] += __shfl_xor_sync(0xffffffffu, mean[1], o);
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    mean[r] *= 1.f / TE;
    const float2 nm = both(-mean[r]);
    float2 s[4] = {};
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      const float2 d = add2(a[r][j], nm);
      s[j & 3] = fma_x2(d, d, s[j & 3]);
    }
    s[0] = add2(add2(s[0], s[1]), add2(s[2], s[3]));
    rstd[r] = s[0].x + s[0].y;
  }
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
    rstd[0] += __shfl_xor_sync(0xffffffffu, rstd[0], o);
    rstd[1] += __shfl_xor_sync(0xffffffffu, rstd[1], o);
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    rstd[r] = rsqrtf(rstd[r] * (1.f / TE) + 1e-5f);
    // opaque: else the compiler keeps the 128 differences of the variance pass
    // for the caller's a - mean, and spills the stream for them
    asm volatile("" : "+f"(mean[r]));
  }
}

// softmax of one head's scores (rows lane / 4 and + 8; NT key tiles of 8) on
// the accumulators; returns the reciprocal row sums
template <int NT, bool CAUSAL>
__device__ __forceinline__ void tile_softmax(float (&s)[NT][4], float scale, int nkeys, int lane, float (&inv)[2]) {
  const int g = lane >> 2, tq = lane & 3;
  float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int r = g + (e >> 1) * 8, col = n * 8 + 2 * tq + (e & 1);
      const bool keep = CAUSAL ? col <= r : col < nkeys;
      const float v = keep ? s[n][e] * scale : -INFINITY;
      s[n][e] = v;
      mx[e >> 1] = fmaxf(mx[e >> 1], v);
    }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 1));
    mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 2));
  }
  float sum[2] = {0.f, 0.f};
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float v = s[n][e] == -INFINITY ? 0.f : __expf(s[n][e] - mx[e >> 1]);
      s[n][e] = v;
      sum[e >> 1] += v;
    }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    sum[h] += __shfl_xor_sync(0xffffffffu, sum[h], 1);
    sum[h] += __shfl_xor_sync(0xffffffffu, sum[h], 2);
    inv[h] = 1.f / sum[h];
  }
}

__device__ __forceinline__ int lattice_of(const TileParams& p, int j) {
  const int k = j / p.jobs_per_lat;
  return p.order ? __ldg(p.order + k) : k;
}

// TRACE: the debug variant, which also stores every cell's residual
template <bool TRACE>
__global__ void __launch_bounds__(TTHREADS, 1) tile_kernel(const TileParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* xln = smem;
  uint8_t* hid = xln + XLN_BYTES;
  uint8_t* ring = hid + 2 * HID_BYTES;
  float* vecs = reinterpret_cast<float*>(ring + NSLOTS * SLOT);     // [2][VEC_BYTES / 4]
  Bars* B = reinterpret_cast<Bars*>(vecs + 2 * VEC_BYTES / 4);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 9) tmem_alloc(&B->tslot, 512);
  if (threadIdx.x == 0) {
    for (int s = 0; s < NSLOTS; ++s) {
      mbar_init1(&B->full[s], 1);
      mbar_init1(&B->empty[s], 1);
    }
    mbar_init1(&B->xready, TCW);
    for (int i = 0; i < 2; ++i) {
      mbar_init1(&B->vfull[i], 1);
      mbar_init1(&B->vempty[i], TCW);
      mbar_init1(&B->afull[i], 1);
      mbar_init1(&B->aempty[i], TCW);
      mbar_init1(&B->hready[i], TCW);
      mbar_init1(&B->hempty[i], 1);
    }
    mbar_init1(&B->rfull, 1);
    B->dead = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = B->tslot, tR = tmem, tA = tmem + 256;

  if (warp >= 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 104;");
    // Both walk the refreshed units as the compute warps do.  Their loops set
    // the pace of the weights (a slot is 256 cycles of MMAs), so they count
    // slots and phases instead of dividing, work on 32-bit shared addresses and
    // descriptor words, leave a wait that does not pass at once to a call, and
    // run uniformly over the warp with one elected lane issuing (1,000 samples at
    // full refresh: 39.4 ms with one lane in a divergent branch, 35.0).
    const uint32_t bfull = su32(B->full), bempty = su32(B->empty), dead = su32(&B->dead);
    bool leave = false;                                // the block gives up (uniform)
    uint32_t s = 0, ph = 0;                            // ring slot, its phase
    auto next_slot = [&]() {
      if (++s == NSLOTS) {
        s = 0;
        ph ^= 1u;
      }
    };
    auto wait = [&](uint32_t bar, uint32_t parity) {
      if (!mbar_test(bar, parity)) wait_slow(bar, parity, p.status, p.wait_limit, dead);
    };
    if (warp == 8) {
      // ------------------------------------------------ weights and vectors: bulk copies
      const uint32_t bvfull = su32(B->vfull), bvempty = su32(B->vempty), dring = su32(ring), dvec = su32(vecs);
      uint32_t units = 0;
      for (int j = blockIdx.x; j < p.n_jobs && !leave; j += gridDim.x) {
        const uint64_t* mk = p.mask + (long long)lattice_of(p, j) * p.T * 2;
        uint64_t nxt = __ldg(mk);
        for (int t = 0; t < p.T && !leave; ++t) {
          uint64_t m = uniform64(nxt);
          if (t + 1 < p.T) nxt = __ldg(mk + 2 * (t + 1));
          while (m && !leave) {
            const int b = __ffsll((long long)m) - 1, l = b / 3, u = b - 3 * l;
            m &= m - 1;
            const uint32_t vb = units & 1;
            wait(bvempty + 8 * vb, ((units >> 1) & 1u) ^ 1u);
            if (elect_one() && !block_dead(dead)) {
              expect_tx(bvfull + 8 * vb, vec_floats(u) * 4);
              bulk_load(dvec + vb * VEC_BYTES, p.vec + (long long)l * VEC_LAYER + vec_off(u), vec_floats(u) * 4,
                        bvfull + 8 * vb);
            }
            ++units;
            const uint8_t* src = p.wpack + ((long long)l * LAYER_SLOTS + unit_slot0(u)) * SLOT;
            const uint8_t* end = src + unit_slots(u) * SLOT;
#pragma unroll 1
            for (; src != end; src += SLOT) {
              wait(bempty + 8 * s, ph ^ 1u);
              if (elect_one() && !block_dead(dead)) {
                expect_tx(bfull + 8 * s, SLOT);
                bulk_load(dring + s * SLOT, src, SLOT, bfull + 8 * s);
              }
              next_slot();
            }
            leave = __any_sync(0xffffffffu, block_dead(dead));
          }
        }
      }
    } else if (warp == 9) {
      // ------------------------------------------------ MMA issue
      constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TROWS >> 4) << 24);
      constexpr uint32_t ID128 = IDESC | ((128u >> 3) << 17), ID256 = IDESC | ((256u >> 3) << 17);
      const uint64_t d0 = sw128_desc(0);
      const uint32_t dhi = (uint32_t)(d0 >> 32), dlo = (uint32_t)d0;     // + (address >> 4)
      const uint32_t dx = dlo + (su32(xln) >> 4), dh = dlo + (su32(hid) >> 4), dr = dlo + (su32(ring) >> 4);
      const uint32_t baf = su32(B->afull), bae = su32(B->aempty), bhr = su32(B->hready), bhe = su32(B->hempty);
      const uint32_t bx = su32(&B->xready), brf = su32(&B->rfull);
      uint32_t units = 0, na = 0, nh = 0;               // phases: units, first-GEMM chunks; second-GEMM chunks / 2
      for (int j = blockIdx.x; j < p.n_jobs && !leave; j += gridDim.x) {
        const uint64_t* mk = p.mask + (long long)lattice_of(p, j) * p.T * 2;
        uint64_t nxt = __ldg(mk);
        for (int t = 0; t < p.T && !leave; ++t) {
          uint64_t m = uniform64(nxt);
          if (t + 1 < p.T) nxt = __ldg(mk + 2 * (t + 1));
          while (m && !leave) {
            const int b = __ffsll((long long)m) - 1, u = b % 3;
            m &= m - 1;
            wait(bx, units & 1u);
            tc_fence_after();
            const int nf = n_first(u), n_ops = nf + n_second(u);
            int c2 = 0;                                 // second-GEMM chunk
            // the order in which pack_unit lays out the slots
#pragma unroll 1
            for (int i = 0; i < n_ops; ++i) {
              const bool first = u == 2 ? i < 3 || ((i & 1) == 0 && i < 14) : i < nf;
              if (first) {
                const uint32_t a = na & 1u;
                wait(bae + 8 * a, ((na >> 1) & 1u) ^ 1u);
                tc_fence_after();
                ++na;
#pragma unroll 1
                for (uint32_t k = 0; k < 4; ++k) {      // K block k
                  wait(bfull + 8 * s, ph);
                  tc_fence_after();
                  const uint32_t ak = dx + k * (16384 >> 4), bk = dr + s * (SLOT >> 4);
                  if (elect_one()) {
#pragma unroll
                    for (uint32_t e = 0; e < 4; ++e)
                      mma_f16(tA + a * 128, desc64(ak + 2 * e, dhi), desc64(bk + 2 * e, dhi), ID128, k | e);
                    commit(bempty + 8 * s);
                    if (k == 3) commit(baf + 8 * a);
                  }
                  next_slot();
                }
              } else {
                const uint32_t buf = c2 & 1u;
                wait(bhr + 8 * buf, nh & 1u);
                tc_fence_after();
#pragma unroll 1
                for (uint32_t k = 0; k < 2; ++k) {      // K block k: its 256 columns in two slots
                  const uint32_t s0 = s, p0 = ph;
                  next_slot();
                  const uint32_t s1 = s, p1 = ph;
                  next_slot();
                  wait(bfull + 8 * s0, p0);
                  wait(bfull + 8 * s1, p1);
                  tc_fence_after();
                  const uint32_t ak = dh + buf * (HID_BYTES >> 4) + k * (16384 >> 4);
                  const uint32_t b0 = dr + s0 * (SLOT >> 4), b1 = dr + s1 * (SLOT >> 4), acc = (uint32_t)c2 | k;
                  if (elect_one()) {
                    // one MMA of 256 columns takes 128 cycles, two of 128 take
                    // 196; a pair that wraps around the ring has to
                    if (s1) {
#pragma unroll
                      for (uint32_t e = 0; e < 4; ++e)
                        mma_f16(tR, desc64(ak + 2 * e, dhi), desc64(b0 + 2 * e, dhi), ID256, acc | e);
                    } else {
#pragma unroll
                      for (uint32_t e = 0; e < 4; ++e) {
                        mma_f16(tR, desc64(ak + 2 * e, dhi), desc64(b0 + 2 * e, dhi), ID128, acc | e);
                        mma_f16(tR + 128, desc64(ak + 2 * e, dhi), desc64(b1 + 2 * e, dhi), ID128, acc | e);
                      }
                    }
                    commit(bempty + 8 * s0);
                    commit(bempty + 8 * s1);
                    if (k == 1) {
                      commit(bhe + 8 * buf);
                      if (i == n_ops - 1) commit(brf);
                    }
                  }
                }
                nh += buf;                              // the buffers alternate
                ++c2;
              }
            }
            ++units;
            leave = __any_sync(0xffffffffu, block_dead(dead));
          }
        }
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 200;");
    // ------------------------------------------------ compute warps
    const int quad = warp & 3;
    const int row0 = quad * 32 + (warp >> 2) * 16;     // this warp's sample: rows row0 .. row0 + 15
    const uint32_t lanes = (uint32_t)row0 << 16;
    const int g = lane >> 2, tq = lane & 3, tid = threadIdx.x;
    uint4* cache = p.cache + (long long)blockIdx.x * p.U * 16 * TCT + tid;
    uint32_t na = 0, nh[2] = {0, 0}, units = 0;
    float2 a[2][32];                                   // columns 8 j + 2 tq, + 1 of rows g, g + 8
    auto wait = [&](uint64_t* bar, uint32_t parity) {
      mbar_wait_live(su32(bar), parity, p.status, p.wait_limit, su32(&B->dead));
    };

    for (int j = blockIdx.x; j < p.n_jobs; j += gridDim.x) {
      const int lat = lattice_of(p, j), part = j % p.jobs_per_lat;
      const int ns = min(TG, p.per_sched - part * TG); // samples of this job
      const bool live = (row0 >> 4) < ns;              // (a warp without a sample repeats the first one's inputs)
      const int sample = lat * p.per_sched + part * TG + (live ? row0 >> 4 : 0);
      const uint64_t* mk = p.mask + (long long)lat * p.T * 2;
      // sampler: lane -> row lane % 16, actions lane / 16 + 2 i
      const int srow = lane & 15, sact = lane >> 4;
      const float* nz = p.noise + ((long long)(sample % p.obs_mod) * TH + srow) * p.A;
      float* xo = p.out + ((long long)sample * TH + srow) * p.A;
      // (in this warp's own rows of the first column block)
      float* xs = reinterpret_cast<float*>(xln + row0 * 128);   // [16][16]: the running sample, at step ends
      float* es = xs + 256;                                     // [16][16]: the output head's sums

      const float* tab = reinterpret_cast<const float*>(hid);
      // the step-end tables -> operand buffers (free between units); false: the block gives up
      auto load_tab = [&]() -> bool {
        if (bar_compute_any(block_dead(su32(&B->dead)))) return false;   // (nobody reads the buffers)
        for (int i = tid; i < tab_floats(p.A) / 4; i += TCT)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(su32(hid + 16 * i)), "l"(p.tab + 4 * i) : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
        return true;
      };
      auto wait_tab = [&]() {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        bar_compute();
      };
      // a <- x W_in + b_in + P_pos (xs holds x)
      auto embed = [&]() {
        const float2* bs = reinterpret_cast<const float2*>(tab + 2 * p.A * TE) + lane;
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          a[0][i] = bs[i * 64];
          a[1][i] = bs[i * 64 + 32];
        }
        const float2* w = reinterpret_cast<const float2*>(tab + p.A * TE) + tq;
        for (int c = 0; c < p.A; ++c, w += TE / 2) {
          const float2 x0 = both(xs[g * 16 + c]), x1 = both(xs[(g + 8) * 16 + c]);
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const float2 v = w[4 * i];
            a[0][i] = fma_x2(x0, v, a[0][i]);
            a[1][i] = fma_x2(x1, v, a[1][i]);
          }
        }
      };

      if (!load_tab()) break;
      // x <- noise[0]
      for (int c = sact; c < p.A; c += 2) {
        const float v = nz[c];
        if (live) xo[c] = v;
        xs[srow * 16 + c] = v;
      }
      wait_tab();
      embed();

      for (int t = 0; t < p.T; ++t) {
        const uint64_t ref = __ldg(mk + 2 * t), val = __ldg(mk + 2 * t + 1);
        uint64_t rest = ref, skip = ~ref & val;
        // the lane's place in cell (t, k): columns 2 tq, + 1 of row g
        auto trace_cell = [&](int k) {
          return p.trace + (((long long)t * p.U + k) * p.rows + (long long)sample * TH + g) * TE + 2 * tq;
        };
        if (TRACE && live)
          for (int k = 0; k < p.U; ++k)                 // a cache never written adds nothing
            if (!((ref | val) >> k & 1ull))
              for (int i = 0; i < 32; ++i) {
                *reinterpret_cast<float2*>(trace_cell(k) + 8 * i) = make_float2(0.f, 0.f);
                *reinterpret_cast<float2*>(trace_cell(k) + 8 * TE + 8 * i) = make_float2(0.f, 0.f);
              }
        for (;;) {
          const int b = rest ? __ffsll((long long)rest) - 1 : p.U;
          // Eq. 1: the skipped units before b whose cache holds a value
          uint64_t m = b >= 64 ? skip : skip & ((1ull << b) - 1ull);
          skip &= ~m;
          while (m) {
            const int k = __ffsll((long long)m) - 1;
            m &= m - 1;
            const uint4* src = cache + (long long)k * 16 * TCT;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              uint4 raw[8];
#pragma unroll
              for (int i = 0; i < 8; ++i) raw[i] = src[(8 * h + i) * TCT];
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                const int c = 16 * h + 2 * i;
                a[0][c] = add2(a[0][c], bf2(raw[i].x));
                a[1][c] = add2(a[1][c], bf2(raw[i].y));
                a[0][c + 1] = add2(a[0][c + 1], bf2(raw[i].z));
                a[1][c + 1] = add2(a[1][c + 1], bf2(raw[i].w));
                if (TRACE && live) {
                  float* tr = trace_cell(k) + 8 * c;
                  *reinterpret_cast<float2*>(tr) = bf2(raw[i].x);
                  *reinterpret_cast<float2*>(tr + 8 * TE) = bf2(raw[i].y);
                  *reinterpret_cast<float2*>(tr + 8) = bf2(raw[i].z);
                  *reinterpret_cast<float2*>(tr + 8 * TE + 8) = bf2(raw[i].w);
                }
              }
            }
          }
          if (!rest) break;
          rest &= rest - 1;
          const int l = b / 3, u = b - 3 * l;

          // LayerNorm -> xln
          const float* vec = vecs + (units & 1) * (VEC_BYTES / 4);
          {
            float mean[2], rstd[2];
            tile_stats(a, mean, rstd);
            wait(&B->vfull[units & 1], (units >> 1) & 1u);
            const float2 nm0 = both(-mean[0]), nm1 = both(-mean[1]), rs0 = both(rstd[0]), rs1 = both(rstd[1]);
            const float2 *gv = reinterpret_cast<const float2*>(vec) + tq, *bv = gv + TE / 2;
#pragma unroll
            for (int i = 0; i < 32; i += 2) {
              uint32_t w[4];
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                const float2 gg = gv[4 * (i + e)], be = bv[4 * (i + e)];
                const float2 y0 = fma_x2(mul_x2(add2(a[0][i + e], nm0), rs0), gg, be);
                const float2 y1 = fma_x2(mul_x2(add2(a[1][i + e], nm1), rs1), gg, be);
                w[2 * e] = pk2(y0.x, y0.y);
                w[2 * e + 1] = pk2(y1.x, y1.y);
              }
              put_tiles(xln + (i >> 3) * 16384, row0, i & 7, lane, w[0], w[1], w[2], w[3]);
            }
          }
          fence_async_smem();
          tc_fence_before();
          arrive_warp(&B->xready, lane);

          auto wait_acc = [&]() -> uint32_t {           // the next chunk's accumulator
            const uint32_t acc = na & 1u;
            wait(&B->afull[acc], (na >> 1) & 1u);
            tc_fence_after();
            return acc;
          };
          auto free_acc = [&](uint32_t acc) {
            tc_fence_before();
            arrive_warp(&B->aempty[acc], lane);
            ++na;
          };
          auto wait_hid = [&](int buf) {                // the operand buffer's previous chunk is consumed
            wait(&B->hempty[buf], (nh[buf] & 1u) ^ 1u);
            ++nh[buf];
          };
          auto put_hid = [&](int buf) {
            fence_async_smem();
            arrive_warp(&B->hready[buf], lane);
          };

          if (u == 2) {
            for (int c = 0; c < 8; ++c) {
              const uint32_t acc = wait_acc();
              const int buf = c & 1;
              // 16 columns at a time, the next ones on their way: four pairs of
              // GELUs side by side are what the registers leave room for
              const uint32_t src = tA + acc * 128 + lanes;
              const float2* bb = reinterpret_cast<const float2*>(vec + 768 + c * 128) + tq;
              uint32_t v[2][8];
              tmem_ld_ahead(src, v[0]);
              wait_hid(buf);
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                uint32_t(&w)[8] = v[i & 1];
                tmem_wait(w);
                if (i < 7) tmem_ld_ahead(src + 16 * (i + 1), v[(i + 1) & 1]);
                else free_acc(acc);
                const float2 b0 = bb[8 * i], b1 = bb[8 * i + 4];
                const float2 y0 = gelu_as2(add2(make_float2(__uint_as_float(w[0]), __uint_as_float(w[1])), b0));
                const float2 y1 = gelu_as2(add2(make_float2(__uint_as_float(w[2]), __uint_as_float(w[3])), b0));
                const float2 y2 = gelu_as2(add2(make_float2(__uint_as_float(w[4]), __uint_as_float(w[5])), b1));
                const float2 y3 = gelu_as2(add2(make_float2(__uint_as_float(w[6]), __uint_as_float(w[7])), b1));
                put_tiles(hid + buf * HID_BYTES + (i >> 2) * 16384, row0, 2 * (i & 3), lane, pk2(y0.x, y0.y),
                          pk2(y1.x, y1.y), pk2(y2.x, y2.y), pk2(y3.x, y3.y));
              }
              put_hid(buf);
            }
          } else if (u == 0) {
            const float* bq = vec + 768;
#pragma unroll 1
            for (int hp = 0; hp < 2; ++hp) {            // heads 2 hp, 2 hp + 1
              uint32_t pa[2][4];
              float inv[2][2];
#pragma unroll
              for (int hh = 0; hh < 2; ++hh) {
                const int h = 2 * hp + hh;
                const uint32_t acc = wait_acc();
                float sc[2][4] = {};
#pragma unroll
                for (int half = 0; half < 2; ++half) {  // 32 head dims at a time
                  float qv[4][4], kv[4][4];
                  tmem_ld_frag(tA + acc * 128 + half * 32 + lanes, qv);
                  tmem_ld_frag(tA + acc * 128 + 64 + half * 32 + lanes, kv);
                  if (half == 1) free_acc(acc);
                  const float* bqh = bq + h * 64 + half * 32 + 2 * tq;
#pragma unroll
                  for (int i = 0; i < 4; ++i) {
                    const float2 b0 = *reinterpret_cast<const float2*>(bqh + 8 * i);
                    const float2 b1 = *reinterpret_cast<const float2*>(bqh + TE + 8 * i);
                    qv[i][0] += b0.x;
                    qv[i][1] += b0.y;
                    qv[i][2] += b0.x;
                    qv[i][3] += b0.y;
                    kv[i][0] += b1.x;
                    kv[i][1] += b1.y;
                    kv[i][2] += b1.x;
                    kv[i][3] += b1.y;
                  }
#pragma unroll
                  for (int ks = 0; ks < 2; ++ks) {
                    const uint32_t aq[4] = {pk2(qv[2 * ks][0], qv[2 * ks][1]), pk2(qv[2 * ks][2], qv[2 * ks][3]),
                                            pk2(qv[2 * ks + 1][0], qv[2 * ks + 1][1]),
                                            pk2(qv[2 * ks + 1][2], qv[2 * ks + 1][3])};
                    mma_k16(sc[0], aq, pk2(kv[2 * ks][0], kv[2 * ks][1]), pk2(kv[2 * ks + 1][0], kv[2 * ks + 1][1]));
                    mma_k16(sc[1], aq, pk2(kv[2 * ks][2], kv[2 * ks][3]), pk2(kv[2 * ks + 1][2], kv[2 * ks + 1][3]));
                  }
                }
                tile_softmax<2, true>(sc, p.scale, 16, lane, inv[hh]);
                pa[hh][0] = pk2(sc[0][0], sc[0][1]);
                pa[hh][1] = pk2(sc[0][2], sc[0][3]);
                pa[hh][2] = pk2(sc[1][0], sc[1][1]);
                pa[hh][3] = pk2(sc[1][2], sc[1][3]);
              }
              wait_hid(hp);
              const uint32_t acc = wait_acc();          // v of both heads
#pragma unroll
              for (int hh = 0; hh < 2; ++hh)
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                  float vv[4][4];
                  tmem_ld_frag(tA + acc * 128 + hh * 64 + half * 32 + lanes, vv);
                  if (hh == 1 && half == 1) free_acc(acc);
                  const float* bv = bq + 2 * TE + (2 * hp + hh) * 64 + half * 32 + 2 * tq;
                  uint32_t w[8];
#pragma unroll
                  for (int i = 0; i < 4; ++i) {
                    const float2 b0 = *reinterpret_cast<const float2*>(bv + 8 * i);
                    const uint32_t v0 = movm(pk2(vv[i][0] + b0.x, vv[i][1] + b0.y));   // tokens 0 .. 7
                    const uint32_t v1 = movm(pk2(vv[i][2] + b0.x, vv[i][3] + b0.y));   // tokens 8 .. 15
                    float o[4] = {};
                    mma_k16(o, pa[hh], v0, v1);
                    w[2 * i] = pk2(o[0] * inv[hh][0], o[1] * inv[hh][0]);
                    w[2 * i + 1] = pk2(o[2] * inv[hh][1], o[3] * inv[hh][1]);
                  }
                  uint8_t* blk = hid + hp * HID_BYTES + hh * 16384;
                  put_tiles(blk, row0, 4 * half, lane, w[0], w[1], w[2], w[3]);
                  put_tiles(blk, row0, 4 * half + 2, lane, w[4], w[5], w[6], w[7]);
                }
              put_hid(hp);
            }
          } else {
            const int nkeys = 1 + p.n_obs;
            const float* bq = vec + 768;
            // keys and values of memory token j: the timestep token, then the sample's observation tokens
            auto mem_row = [&](int jk) -> const __nv_bfloat16* {
              return jk == 0 ? p.kv_time + ((long long)t * p.L + l) * 2 * TE
                             : p.kv_obs + (((long long)(sample % p.obs_mod) * p.n_obs + (jk - 1)) * p.L + l) * 2 * TE;
            };
            // lanes whose token does not exist read the timestep token's row and drop it
            const bool k_ok = g < nkeys, v0_ok = 2 * tq < nkeys, v1_ok = 2 * tq + 1 < nkeys;
            const uint4* kr = reinterpret_cast<const uint4*>(mem_row(k_ok ? g : 0)) + 2 * tq;
            const uint4* v0r = reinterpret_cast<const uint4*>(mem_row(v0_ok ? 2 * tq : 0) + TE) + g;
            const uint4* v1r = reinterpret_cast<const uint4*>(mem_row(v1_ok ? 2 * tq + 1 : 0) + TE) + g;
            uint4 k0, k1, v0, v1;                       // the next head's
            auto load_kv = [&](int h) {
              const uint4 z = make_uint4(0u, 0u, 0u, 0u);
              k0 = k_ok ? __ldg(kr + 8 * h) : z;
              k1 = k_ok ? __ldg(kr + 8 * h + 1) : z;
              v0 = v0_ok ? __ldg(v0r + 8 * h) : z;
              v1 = v1_ok ? __ldg(v1r + 8 * h) : z;
            };
            load_kv(0);
#pragma unroll 1
            for (int h = 0; h < 4; ++h) {
              const uint32_t acc = na & 1u;
              const uint32_t kf[8] = {k0.x, k0.y, k0.z, k0.w, k1.x, k1.y, k1.z, k1.w};
              const uint32_t va[4] = {v0.x, v0.y, v0.z, v0.w}, vb[4] = {v1.x, v1.y, v1.z, v1.w};
              if (h < 3) load_kv(h + 1);
              if (!(h & 1)) wait_acc();
              float sc[1][4] = {};
#pragma unroll
              for (int half = 0; half < 2; ++half) {
                float qv[4][4];
                tmem_ld_frag(tA + acc * 128 + (h & 1) * 64 + half * 32 + lanes, qv);
                const float* bqh = bq + h * 64 + half * 32 + 2 * tq;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  const float2 b0 = *reinterpret_cast<const float2*>(bqh + 8 * i);
                  qv[i][0] += b0.x;
                  qv[i][1] += b0.y;
                  qv[i][2] += b0.x;
                  qv[i][3] += b0.y;
                }
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) {
                  const uint32_t aq[4] = {pk2(qv[2 * ks][0], qv[2 * ks][1]), pk2(qv[2 * ks][2], qv[2 * ks][3]),
                                          pk2(qv[2 * ks + 1][0], qv[2 * ks + 1][1]),
                                          pk2(qv[2 * ks + 1][2], qv[2 * ks + 1][3])};
                  mma_k16(sc[0], aq, kf[4 * half + 2 * ks], kf[4 * half + 2 * ks + 1]);
                }
              }
              if (h & 1) free_acc(acc);
              float inv[2];
              tile_softmax<1, false>(sc, p.scale, nkeys, lane, inv);
              const uint32_t p0 = pk2(sc[0][0], sc[0][1]), p1 = pk2(sc[0][2], sc[0][3]);
              if (!(h & 1)) wait_hid(h >> 1);
              uint8_t* blk = hid + (h >> 1) * HID_BYTES + (h & 1) * 16384;
#pragma unroll
              for (int i = 0; i < 8; i += 2) {
                uint32_t w[4];
#pragma unroll
                for (int e = 0; e < 2; ++e) {           // tokens 2 tq | 2 tq + 1 of head dim 8 (i + e) + g
                  float o[4] = {};
                  mma_k8(o, p0, p1, __byte_perm(va[i >> 1], vb[i >> 1], e ? 0x7632 : 0x5410));
                  w[2 * e] = pk2(o[0] * inv[0], o[1] * inv[0]);
                  w[2 * e + 1] = pk2(o[2] * inv[1], o[3] * inv[1]);
                }
                put_tiles(blk, row0, i, lane, w[0], w[1], w[2], w[3]);
              }
              if (h & 1) put_hid(h >> 1);
            }
          }

          // r = R + bias: a += r, c_b <- bf16(r)
          wait(&B->rfull, units & 1u);
          tc_fence_after();
          const uint32_t vb = units & 1u;
          ++units;
          uint4* dst = cache + (long long)b * 16 * TCT;
          const float2* b2 = reinterpret_cast<const float2*>(vec + 2 * TE) + tq;
#pragma unroll
          for (int c = 0; c < 4; ++c) {                 // 64 columns at a time
            float v[8][4];
            tmem_ld_frag(tR + c * 64 + lanes, v);
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
              uint32_t w[4];
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                const float2 bi = b2[4 * (8 * c + i + e)];
                const float2 r0 = add2(make_float2(v[i + e][0], v[i + e][1]), bi);
                const float2 r1 = add2(make_float2(v[i + e][2], v[i + e][3]), bi);
                w[2 * e] = pk2(r0.x, r0.y);
                w[2 * e + 1] = pk2(r1.x, r1.y);
                a[0][8 * c + i + e] = add2(a[0][8 * c + i + e], r0);
                a[1][8 * c + i + e] = add2(a[1][8 * c + i + e], r1);
                if (TRACE && live) {
                  float* tr = trace_cell(b) + 8 * (8 * c + i + e);
                  *reinterpret_cast<float2*>(tr) = r0;
                  *reinterpret_cast<float2*>(tr + 8 * TE) = r1;
                }
              }
              dst[(4 * c + (i >> 1)) * TCT] = make_uint4(w[0], w[1], w[2], w[3]);
            }
          }
          arrive_warp(&B->vempty[vb], lane);
        }

        // step end: eps = LN_f(a) W_head + b_head, the sampler step, the next embedding
        if (!load_tab()) break;
        {
          float xv[8], zv[8];                           // x and the step's noise of this lane's actions
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int c = sact + 2 * i;
            xv[i] = c < p.A ? xo[c] : 0.f;
            zv[i] = c < p.A && p.sampler == 0 ? nz[(long long)(1 + t) * p.obs_mod * TH * p.A + c] : 0.f;
          }
          float mean[2], rstd[2];
          tile_stats(a, mean, rstd);
          wait_tab();
          {
            const float2 nm0 = both(-mean[0]), nm1 = both(-mean[1]), rs0 = both(rstd[0]), rs1 = both(rstd[1]);
            const float2 *gv = reinterpret_cast<const float2*>(tab + 2 * p.A * TE + 64 * TH * 4) + tq, *bv = gv + TE / 2;
#pragma unroll
            for (int i = 0; i < 32; ++i) {
              const float2 gg = gv[4 * i], be = bv[4 * i];
              a[0][i] = fma_x2(mul_x2(add2(a[0][i], nm0), rs0), gg, be);
              a[1][i] = fma_x2(mul_x2(add2(a[1][i], nm1), rs1), gg, be);
            }
          }
          const float2* w = reinterpret_cast<const float2*>(tab) + tq;
          for (int c = 0; c < p.A; ++c, w += TE / 2) {
            float2 d0[2] = {}, d1[2] = {};
#pragma unroll
            for (int i = 0; i < 32; ++i) {
              const float2 v = w[4 * i];
              d0[i & 1] = fma_x2(a[0][i], v, d0[i & 1]);
              d1[i & 1] = fma_x2(a[1][i], v, d1[i & 1]);
            }
            d0[0] = add2(d0[0], d0[1]);
            d1[0] = add2(d1[0], d1[1]);
            float e0 = d0[0].x + d0[0].y, e1 = d1[0].x + d1[0].y;
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
              e0 += __shfl_xor_sync(0xffffffffu, e0, o);
              e1 += __shfl_xor_sync(0xffffffffu, e1, o);
            }
            if (tq == 0) {
              es[g * 16 + c] = e0;
              es[(g + 8) * 16 + c] = e1;
            }
          }
          __syncwarp();
          const float* tb = p.stab + t * 8;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int c = sact + 2 * i;
            if (c < p.A) {
              const float eps = es[srow * 16 + c] + __ldg(p.head_b + c);
              float x0 = (xv[i] - tb[1] * eps) * tb[0];
              x0 = fminf(1.0f, fmaxf(-1.0f, x0));
              float xn;
              if (p.sampler == 0)
                xn = tb[2] * x0 + tb[3] * xv[i] + tb[4] * zv[i];
              else
                xn = tb[6] * x0 + tb[7] * ((xv[i] - tb[5] * x0) / tb[1]);
              if (live) xo[c] = xn;
              xs[srow * 16 + c] = xn;
            }
          }
          __syncwarp();
        }
        if (t + 1 < p.T) embed();
      }
    }
  }
  __syncwarp();
  settle_after_timeout(p.status, block_dead(su32(&B->dead)));   // then copies and MMAs may still be in flight
  tc_fence_before();
  __syncthreads();
  if (warp == 9) tmem_dealloc(tmem, 512);
}

}  // namespace

struct TileState {
  int L = 0, A = 0, n_obs = 0, T = 0, sampler = 0;
  int num_sms = 0, cache_slots = 0;
  uint8_t* wpack = nullptr;       // [L][LAYER_SLOTS][SLOT]
  float* vec = nullptr;           // [L][VEC_LAYER], then the step-end tables, then b_head
  uint4* cache = nullptr;         // [cache_slots][3L][16][256]
  GuardList guards;
};

namespace {

uint16_t bf16_of(float f) {
  uint32_t u;
  std::memcpy(&u, &f, 4);
  if ((u & 0x7f800000u) == 0x7f800000u) return (uint16_t)(u >> 16);
  u += 0x7fffu + ((u >> 16) & 1u);
  return (uint16_t)(u >> 16);
}

float bf16_round(float f) {
  const uint32_t u = (uint32_t)bf16_of(f) << 16;
  float r;
  std::memcpy(&r, &u, 4);
  return r;
}

// element (n, kk) of a 64-column K block: 128-byte rows, 16-byte chunks XOR-swizzled by row
void put(uint8_t* blk, int n, int kk, float v) {
  const uint16_t h = bf16_of(v);
  std::memcpy(blk + n * 128 + (((kk >> 3) ^ (n & 7)) << 4) + (kk & 7) * 2, &h, 2);
}

// The unit's weight slots in the order in which the MMA warp consumes them.
// W1 [256][n1] -> chunks of 128 columns (col(c, n) = column of row n of chunk
// c), W2 [K2][256].
template <class Col>
uint8_t* pack_unit(uint8_t* dst, int u, const float* W1, int n1, const float* W2, Col col) {
  auto first = [&](int c) {
    for (int kb = 0; kb < 4; ++kb, dst += SLOT)
      for (int n = 0; n < 128; ++n)
        for (int kk = 0; kk < 64; ++kk) put(dst, n, kk, W1[(size_t)(kb * 64 + kk) * n1 + col(c, n)]);
  };
  auto second = [&](int c) {
    for (int i = 0; i < 4; ++i, dst += SLOT)
      for (int n = 0; n < 128; ++n)
        for (int kk = 0; kk < 64; ++kk)
          put(dst, n, kk, W2[(size_t)(c * 128 + (i >> 1) * 64 + kk) * TE + (i & 1) * 128 + n]);
  };
  if (u == 2) {                     // the first GEMM two chunks ahead: its accumulator is free before the GELUs are done
    first(0);
    first(1);
    for (int c = 2; c < 8; ++c) {
      first(c);
      second(c - 2);
    }
    second(6);
    second(7);
  } else {
    for (int c = 0; c < n_first(u); ++c) first(c);
    second(0);
    second(1);
  }
  return dst;
}

}  // namespace

bool tile_supported(const evo_config* c) {
  return c->dtype == EVO_DTYPE_BF16 && c->n_emb == TE && c->n_head == 4 && c->horizon == TH && c->action_dim <= 16 &&
         1 + c->n_obs <= 8 && 3 * c->n_layer <= 64;
}

int tile_smem_bytes() { return TILE_SMEM; }

// Place p of a head's 64 values in the tile path's keys (part 0) and values
// (part 1): the head dim that stands there.  Keys: quad lane q of a fragment
// reads dims 8 i + 2 q, + 1 (i = 0 .. 7) as 32 bytes; values: row g reads dims
// 8 i + g as 16 bytes.
int tile_kv_column(int part, int p) {
  return part == 0 ? 8 * ((p >> 1) & 7) + 2 * (p >> 4) + (p & 1) : 8 * (p & 7) + (p >> 3);
}

int tile_create(TileState** out, const evo_config* c, const float* weights, const int* woff, int max_batch) {
  *out = nullptr;
  if (!tile_supported(c)) return EVO_ERR_UNSUPPORTED;
  TileState* s = new TileState();
  auto fail = [&](int e) {
    tile_destroy(s);
    return e;
  };
  s->L = c->n_layer;
  s->A = c->action_dim;
  s->n_obs = c->n_obs;
  s->T = c->n_steps;
  s->sampler = c->sampler;
  const int L = s->L, U = 3 * L;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&s->num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || s->num_sms <= 0)
    return fail(EVO_ERR_CUDA);
  std::vector<uint8_t> wp((size_t)L * LAYER_SLOTS * SLOT);
  const int A = s->A;
  std::vector<float> vec((size_t)L * VEC_LAYER + tab_floats(A) + A);
  uint8_t* dst = wp.data();
  for (int l = 0; l < L; ++l) {
    auto W = [&](int id) { return weights + woff[W_LAYER0] + (size_t)l * woff[W_LAYER_STRIDE] + woff[id]; };
    dst = pack_unit(dst, 0, W(WL_SA_WQKV), 3 * TE, W(WL_SA_WO), [](int ch, int n) {
      const int hp = ch / 3, i = ch % 3;                 // heads 2 hp, 2 hp + 1: q|k, q|k, v|v
      return i == 2 ? 2 * TE + hp * 128 + n : (n < 64 ? (2 * hp + i) * 64 + n : TE + (2 * hp + i) * 64 + n - 64);
    });
    dst = pack_unit(dst, 1, W(WL_CA_WQ), TE, W(WL_CA_WO), [](int ch, int n) { return ch * 128 + n; });
    dst = pack_unit(dst, 2, W(WL_FF_W1), 4 * TE, W(WL_FF_W2), [](int ch, int n) { return ch * 128 + n; });
    static const int id[3][4] = {{WL_LN1G, WL_LN1B, WL_SA_BO, WL_SA_BQKV},
                                 {WL_LN2G, WL_LN2B, WL_CA_BO, WL_CA_BQ},
                                 {WL_LN3G, WL_LN3B, WL_FF_B2, WL_FF_B1}};
    for (int u = 0; u < 3; ++u) {
      float* d = vec.data() + (size_t)l * VEC_LAYER + vec_off(u);
      for (int k = 0; k < 4; ++k) std::memcpy(d + k * TE, W(id[u][k]), (size_t)(k < 3 ? TE : n_bias1(u)) * 4);
    }
  }
  float* tab = vec.data() + (size_t)L * VEC_LAYER;
  for (int k = 0; k < A; ++k)
    for (int e = 0; e < TE; ++e) {   // the weight matrices in bf16, like every other
      tab[k * TE + e] = bf16_round(weights[woff[W_HEAD_W] + e * A + k]);
      tab[(A + k) * TE + e] = bf16_round(weights[woff[W_IN_W] + k * TE + e]);
    }
  float* base = tab + 2 * A * TE;
  for (int i = 0; i < 32; ++i)
    for (int tok = 0; tok < TH; ++tok)
      for (int e = 0; e < 8; ++e)
        base[(i * TH + tok) * 8 + e] = weights[woff[W_IN_B] + 8 * i + e] + weights[woff[W_POS] + tok * TE + 8 * i + e];
  std::memcpy(base + 64 * TH * 4, weights + woff[W_LNF_G], TE * 4);
  std::memcpy(base + 64 * TH * 4 + TE, weights + woff[W_LNF_B], TE * 4);
  std::memcpy(base + 64 * TH * 4 + 2 * TE, weights + woff[W_HEAD_B], (size_t)A * 4);
  // a job holds a sample at least, so no call has more jobs than samples
  s->cache_slots = std::min(s->num_sms, max_batch);
  const size_t cache_bytes = (size_t)s->cache_slots * U * 16 * TCT * sizeof(uint4);
  if (cudaMalloc(&s->wpack, wp.size()) != cudaSuccess || cudaMalloc(&s->vec, vec.size() * 4) != cudaSuccess ||
      guarded_malloc(reinterpret_cast<void**>(&s->cache), cache_bytes, &s->guards) != cudaSuccess)
    return fail(EVO_ERR_OOM);
  if (cudaMemcpy(s->wpack, wp.data(), wp.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(s->vec, vec.data(), vec.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaFuncSetAttribute(tile_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, TILE_SMEM) != cudaSuccess ||
      cudaFuncSetAttribute(tile_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, TILE_SMEM) != cudaSuccess)
    return fail(EVO_ERR_CUDA);
  *out = s;
  return EVO_OK;
}

void tile_destroy(TileState* s) {
  if (!s) return;
  cudaFree(s->wpack);
  cudaFree(s->vec);
  guarded_free(s->cache);
  delete s;
}

const GuardList* tile_guards(const TileState* s) { return &s->guards; }

cudaError_t tile_run(const TileState* s, const TileCall& c) {
  TileParams p{};
  p.L = s->L;
  p.A = s->A;
  p.n_obs = s->n_obs;
  p.T = s->T;
  p.U = 3 * s->L;
  p.jobs_per_lat = (c.per_sched + TG - 1) / TG;
  p.n_jobs = p.jobs_per_lat * c.n_sched;
  p.per_sched = c.per_sched;
  p.obs_mod = c.obs_mod;
  p.sampler = s->sampler;
  p.mask = c.mask;
  p.order = c.order;
  p.wpack = s->wpack;
  p.vec = s->vec;
  p.tab = s->vec + (size_t)s->L * VEC_LAYER;
  p.head_b = p.tab + tab_floats(s->A);
  p.stab = c.stab;
  p.noise = c.noise;
  p.kv_time = c.kv_time;
  p.kv_obs = c.kv_obs;
  p.cache = s->cache;
  p.out = c.out;
  p.trace = c.trace;
  p.rows = (long long)c.n_sched * c.per_sched * TH;
  p.scale = 0.125f;               // 1 / sqrt(64)
  p.status = c.status;
  p.wait_limit = WAIT_CYCLES_DEFAULT;
  const int grid = std::min(p.n_jobs, s->cache_slots);
  if (c.trace)
    tile_kernel<true><<<grid, TTHREADS, TILE_SMEM, c.st>>>(p);
  else
    tile_kernel<false><<<grid, TTHREADS, TILE_SMEM, c.st>>>(p);
  return cudaGetLastError();
}

}  // namespace evo
