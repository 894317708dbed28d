// Activation and weight quantizers (Sec. 4, "Quantization": FP8 / NVFP4
// post-training quantization; activations are quantized at run time, weights
// once).  All kernels here are HBM-bandwidth bound streaming kernels:
//
// Dynamic tensor scale, by the size of x (launch_dynamic):
//   cluster_quant_kernel  up to 1 MB: every cluster of eight CTAs reads all of
//                         x, so no grid-wide barrier
//   regpass_kernel        (NVFP4) x held in registers: one read of x, the amax
//                         reduced across the grid
//   onepass_kernel        the same with x in shared memory
//   two_phase_kernel      larger x: amax, then the tiles again in reverse order,
//                         in one launch
// Static tensor scale:
//   quant_nvfp4_kernel    bf16 -> packed e2m1 codes + E4M3 block scales in the
//                         tensor-core scale layout + FP32 tensor scale
//   quant_nvfp4_small_kernel the same of an x of at most 32 bytes per thread
//   quant_nvfp4_ring_kernel  the same of an x that was just written
//   quant_fp8_kernel      bf16 -> E4M3 codes with one tensor scale
// Weights:
//   quant_fp8_rows_kernel bf16 -> E4M3 codes with one scale per row
//
// The [M, K] input is a flat array of 16-byte chunks (8 bf16); a unit is the
// two chunks of one NVFP4 block, and four neighbouring lanes hold one
// 64-element group (because K % 64 == 0 a group never straddles a row).
// quant_nvfp4_kernel and two_phase_kernel load straight to registers; the static
// FP8 quantizer and the dynamic chain's NVFP4 one (stream_tiles) cut x into 16 KB
// tiles that a persistent grid (three CTAs per SM) takes through a four-deep
// shared-memory ring filled by bulk copies, ~192 KB per SM of input in flight.
#include "qlin_internal.h"

namespace qlin {

namespace {

constexpr int kThreads = 512;
constexpr int kTileChunks = 1024;             // 16 KB of input per tile
constexpr int kStages = 4;
constexpr int kSmem = kStages * kTileChunks * 16 + 64;
constexpr int kBlocksPerSm = 3;

// Largest |bf16| in a 16-byte chunk or in the two chunks of an NVFP4 block, as
// the bit pattern of a bf16 magnitude (any NaN: 0x7FFF, above infinity).
// Packed bf16 absolute maxima, one reduction of the two halves per block; with
// masks and integer maxima of halves dynamic NVFP4 took 5.31 us (now 5.13) at
// 1000 x 3072, 11.4 (11.2) at 4608 x 3072 and 39.4 (39.0) at 18432 x 3072; the
// static kernels measured the same.  (Not so in the GEMM's re-quantizing
// epilogue, which keeps the integer form: there these take 59.5 us to 61.7.)
__device__ __forceinline__ uint32_t abs_max2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("{\n\t.reg .b32 x, y;\n\tabs.bf16x2 x, %1;\n\tabs.bf16x2 y, %2;\n\t"
      "max.NaN.bf16x2 %0, x, y;\n\t}"
      : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ uint32_t chunk_abs_max_bits(const uint4 v) {
  const uint32_t m = abs_max2(abs_max2(v.x, v.y), abs_max2(v.z, v.w));
  return max(m & 0xFFFFu, m >> 16);
}
__device__ __forceinline__ uint32_t block_abs_max_bits(const uint4 v, const uint4 w) {
  const uint32_t m = abs_max2(abs_max2(abs_max2(v.x, v.y), abs_max2(v.z, v.w)),
                              abs_max2(abs_max2(w.x, w.y), abs_max2(w.z, w.w)));
  return max(m & 0xFFFFu, m >> 16);
}

__device__ __forceinline__ void unpack8(const uint4 v, float (&f)[8]) {
  f[0] = bf16_lo(v.x); f[1] = bf16_hi(v.x);
  f[2] = bf16_lo(v.y); f[3] = bf16_hi(v.y);
  f[4] = bf16_lo(v.z); f[5] = bf16_hi(v.z);
  f[6] = bf16_lo(v.w); f[7] = bf16_hi(v.w);
}

__device__ __forceinline__ uint4 lds128(const uint4* p) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(smem_u32(p)));
  return v;
}

// A load that stays after the grid dependency wait (volatile, as that is).
__device__ __forceinline__ uint4 ldg128(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// The per-tile work of each kernel (called by every thread for each tile).
// One lane per 16-element block (two chunks); each lane stores its block's
// scale code as one byte of the atom layout (one store instruction per warp,
// instead of gathering a 64-element group's four codes by shuffles: measured
// 2-7% faster).  r_b = S_enc / s_b comes from a per-CTA table over the 127
// finite E4M3 codes, filled with the same fp32 division.
template <typename Idx>
struct Nvfp4Op {
  static constexpr int kUnit = 2;
  static constexpr bool kBlockMax = true;   // the one-read kernel keeps block maxima
  float s_enc;
  Idx chunks_per_row;
  // row = chunk / chunks_per_row without a division (32-bit indices):
  // t = umulhi(div_m, c), row = (t + ((c - t) >> div_s1)) >> div_s2
  // (Granlund and Montgomery, PLDI 1994, division by invariant integers)
  uint32_t div_m, div_s1, div_s2;
  int64_t K;
  uint32_t* codes;
  uint8_t* scales;
  float* r_table;   // shared memory, 128 entries
  __device__ __forceinline__ void bind(float* table) { r_table = table; }
  __device__ __forceinline__ void init() {
    if (threadIdx.x < 128) {
      const uint32_t c = threadIdx.x;
      r_table[c] = (c == 0u) ? 0.0f : __fdiv_rn(s_enc, e4m3_value(c));
    }
  }
  // The codes of one 16-element block (block amax bits mb) and its scale
  // code (in `word`).
  // kDivide: r_b by its division instead of the table (one block per thread).
  template <bool kDivide = false>
  __device__ __forceinline__ void quantize_block(const uint4 (&v)[2], uint32_t mb,
                                                 uint32_t& code0, uint32_t& code1,
                                                 uint32_t& word) const {
    const float t = __fmul_rn(__uint_as_float(mb << 16), s_enc);
    const uint32_t sb = e4m3_code_div6(t);
    const float r_b = !kDivide ? r_table[sb]
                      : sb == 0u ? 0.0f
                                 : __fdiv_rn(s_enc, e4m3_value(sb));
    float f[8];
    unpack8(v[0], f);
#pragma unroll
    for (int i = 0; i < 8; i += 2) mul2_rn(f[i], f[i + 1], r_b);
    code0 = e2m1x8(f);
    unpack8(v[1], f);
#pragma unroll
    for (int i = 0; i < 8; i += 2) mul2_rn(f[i], f[i + 1], r_b);
    code1 = e2m1x8(f);
    word = sb;
  }
  template <bool kDivide = false>
  __device__ __forceinline__ void unit(const uint4 (&v)[2], uint64_t c, bool valid) {
    uint32_t code0, code1, word;
    quantize_block<kDivide>(v, block_abs_max_bits(v[0], v[1]), code0, code1,
                            word);
    if (valid) {
      reinterpret_cast<uint2*>(codes)[c >> 1] = make_uint2(code0, code1);
      {
        if constexpr (sizeof(Idx) == 4) {
          const uint32_t ci = (uint32_t)c;
          const uint32_t t = __umulhi(div_m, ci);
          const uint32_t row = (t + ((ci - t) >> div_s1)) >> div_s2;
          const uint32_t colc = ci - row * (uint32_t)chunks_per_row;   // in chunks
          scales[((row >> 7) * (uint32_t)(K >> 6) + (colc >> 3)) * 512u +
                 (row & 31u) * 16u + ((row >> 5) & 3u) * 4u + ((colc >> 1) & 3u)] = (uint8_t)word;
        } else {
          const Idx ci = (Idx)c;
          const Idx row = ci / chunks_per_row;
          const Idx col = (ci - row * chunks_per_row) << 3;
          scales[scale_offset((int64_t)row, (int64_t)(col >> 4), K)] = (uint8_t)word;
        }
      }
    }
  }
  // The thread's units of two chunks, kStride chunks apart, held in registers
  // (bm: their block amax bits); row and column are tracked without dividing.
  template <int kUnits, uint32_t kStride>
  __device__ __forceinline__ void run_units(const uint4 (&v)[kUnits][2],
                                            const uint32_t (&bm)[kUnits / 2], uint32_t n,
                                            uint64_t c0) const {
    const uint32_t cpr = (uint32_t)chunks_per_row;
    const uint32_t dq = kStride / cpr, dr = kStride % cpr;
    const uint64_t cg = c0 + 2u * threadIdx.x;
    uint32_t row = (uint32_t)(cg / cpr), col = (uint32_t)(cg % cpr);   // col in chunks
    const uint32_t kgroups = (uint32_t)(K >> 6);
#pragma unroll
    for (int u = 0; u < kUnits; ++u) {
      if ((uint32_t)u * kStride >= n) break;   // block-uniform
      const uint32_t cl = (uint32_t)u * kStride + 2u * threadIdx.x;
      uint32_t a0, a1, aw;
      quantize_block(v[u], (u & 1) ? bm[u / 2] >> 16 : bm[u / 2] & 0xFFFFu, a0, a1, aw);
      if (cl < n) {
        reinterpret_cast<uint2*>(codes)[(c0 + cl) >> 1] = make_uint2(a0, a1);
        scales[((row >> 7) * kgroups + (col >> 3)) * 512u + (row & 31u) * 16u +
               ((row >> 5) & 3u) * 4u + ((col >> 1) & 3u)] = (uint8_t)aw;
      }
      row += dq;
      col += dr;
      if (col >= cpr) {
        col -= cpr;
        ++row;
      }
    }
  }
  __device__ __forceinline__ void pair(const uint4 (&v)[2], uint64_t c, bool valid) {
    unit(v, c, valid);
  }
  // The two chunks of one thread, with no table.
  __device__ __forceinline__ void block(const uint4 (&v)[2], uint32_t c, bool valid) {
    unit<true>(v, c, valid);
  }
  // A slice of n chunks held in shared memory, global chunks [c0, c0 + n)
  // (c0 and n multiples of 8): each thread takes units of two chunks at a
  // stride of the block, two units per step for instruction-level
  // parallelism, and tracks its row and column without dividing.  The
  // block amax bits of step s's two units are bm[s] (low, high halves), as
  // gathered by block_max_pass.
  template <int kThreadsPerBlock, int kSteps>
  __device__ __forceinline__ void run_slice(const uint4* buf, uint32_t n, uint64_t c0,
                                            const uint32_t (&bm)[kSteps]) const {
    constexpr uint32_t kStride = 2u * kThreadsPerBlock;          // chunks per step and unit
    const uint32_t cpr = (uint32_t)chunks_per_row;
    const uint32_t dq = (2u * kStride) / cpr, dr = (2u * kStride) % cpr;
    const uint32_t kq = kStride / cpr, kr = kStride % cpr;
    const uint64_t cg = c0 + 2u * threadIdx.x;
    uint32_t row = (uint32_t)(cg / cpr), col = (uint32_t)(cg % cpr);   // col in chunks
    const uint32_t kgroups = (uint32_t)(K >> 6);
    // the loop bound is block-uniform
#pragma unroll
    for (int s = 0; s < kSteps; ++s) {
      const uint32_t base = (uint32_t)s * 2u * kStride;
      if (base >= n) break;
      const uint32_t cl = base + 2u * threadIdx.x;
      uint4 va[2], vb[2];
      const bool ok_a = cl < n, ok_b = cl + kStride < n;   // units never straddle n
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        va[k] = ok_a ? lds128(buf + cl + k) : make_uint4(0u, 0u, 0u, 0u);
        vb[k] = ok_b ? lds128(buf + cl + kStride + k) : make_uint4(0u, 0u, 0u, 0u);
      }
      uint32_t a0, a1, aw, b0, b1, bw;
      quantize_block(va, bm[s] & 0xFFFFu, a0, a1, aw);
      quantize_block(vb, bm[s] >> 16, b0, b1, bw);
      uint32_t row_b = row + kq, col_b = col + kr;
      if (col_b >= cpr) {
        col_b -= cpr;
        ++row_b;
      }
      if (ok_a) {
        reinterpret_cast<uint2*>(codes)[(c0 + cl) >> 1] = make_uint2(a0, a1);
        scales[((row >> 7) * kgroups + (col >> 3)) * 512u + (row & 31u) * 16u +
               ((row >> 5) & 3u) * 4u + ((col >> 1) & 3u)] = (uint8_t)aw;
      }
      if (ok_b) {
        reinterpret_cast<uint2*>(codes)[(c0 + cl + kStride) >> 1] = make_uint2(b0, b1);
        scales[((row_b >> 7) * kgroups + (col_b >> 3)) * 512u + (row_b & 31u) * 16u +
               ((row_b >> 5) & 3u) * 4u + ((col_b >> 1) & 3u)] = (uint8_t)bw;
      }
      row += dq;
      col += dr;
      if (col >= cpr) {
        col -= cpr;
        ++row;
      }
    }
  }
};

struct Fp8Op {
  static constexpr int kUnit = 1;
  static constexpr bool kBlockMax = false;
  float s_enc;
  uint2* codes;
  __device__ __forceinline__ void bind(float*) {}
  __device__ __forceinline__ void init() {}
  __device__ __forceinline__ void unit(const uint4 (&v)[1], uint64_t c, bool valid) {
    if (!valid) return;
    float f[8];
    unpack8(v[0], f);
#pragma unroll
    for (int i = 0; i < 8; ++i) f[i] = __fmul_rn(f[i], s_enc);
    codes[c] = make_uint2(e4m3x4(f[0], f[1], f[2], f[3]), e4m3x4(f[4], f[5], f[6], f[7]));
  }
  __device__ __forceinline__ void pair(const uint4 (&v)[2], uint64_t c, bool valid) {
    if (!valid) return;
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      float f[8];
      unpack8(v[k], f);
#pragma unroll
      for (int i = 0; i < 8; ++i) f[i] = __fmul_rn(f[i], s_enc);
      w[2 * k] = e4m3x4(f[0], f[1], f[2], f[3]);
      w[2 * k + 1] = e4m3x4(f[4], f[5], f[6], f[7]);
    }
    *reinterpret_cast<uint4*>(codes + c) = make_uint4(w[0], w[1], w[2], w[3]);
  }
  __device__ __forceinline__ void block(const uint4 (&v)[2], uint32_t c, bool valid) {
    const uint4 a[1] = {v[0]}, b[1] = {v[1]};
    unit(a, c, valid);
    unit(b, c + 1, valid);
  }
  template <int kThreadsPerBlock>
  __device__ __forceinline__ void run_slice(const uint4* buf, uint32_t n, uint64_t c0) const {
    for (uint32_t cl = threadIdx.x; cl < n; cl += kThreadsPerBlock) {
      float f[8];
      unpack8(lds128(buf + cl), f);
#pragma unroll
      for (int i = 0; i < 8; ++i) f[i] = __fmul_rn(f[i], s_enc);
      codes[c0 + cl] =
          make_uint2(e4m3x4(f[0], f[1], f[2], f[3]), e4m3x4(f[4], f[5], f[6], f[7]));
    }
  }
};

// Persistent tile loop: thread 0 keeps kStages bulk copies of 16 KB tiles in
// flight; every thread applies `op` to its chunks of each landed tile.
// `setup(op)` runs once the first copies are on their way (reads that only
// the arithmetic needs, such as the tensor scale, overlap the loads).
// Returns false if a bounded wait expired (recorded in *err).
template <typename Op, typename Setup>
__device__ __forceinline__ bool stream_tiles(const uint4* __restrict__ x, uint64_t n_chunks,
                                             Op& op, Setup setup, unsigned* err,
                                             uint64_t timeout_ns) {
  extern __shared__ __align__(128) uint8_t qsm[];
  uint4* buf = reinterpret_cast<uint4*>(qsm);
  uint64_t* full = reinterpret_cast<uint64_t*>(qsm + kStages * kTileChunks * 16);
  __shared__ int abort_flag;
  const uint64_t n_tiles = (n_chunks + kTileChunks - 1) / kTileChunks;
  const int tid = threadIdx.x;

  auto issue = [&](uint64_t t, int s) {
    const uint64_t c0 = t * kTileChunks;
    const uint64_t left = n_chunks - c0;
    const uint32_t nc = left < (uint64_t)kTileChunks ? (uint32_t)left : (uint32_t)kTileChunks;
    mbar_arrive_expect_tx(&full[s], nc * 16u);
    bulk_load(buf + s * kTileChunks, x + c0, nc * 16u, &full[s]);
  };

  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) mbar_init(&full[s], 1);
    abort_flag = 0;
    mbar_fence_init();
    for (int s = 0; s < kStages; ++s) {
      const uint64_t t = blockIdx.x + (uint64_t)s * gridDim.x;
      if (t < n_tiles) issue(t, s);
    }
  }
  setup(op);
  op.init();
  __syncthreads();
  int s = 0;
  uint32_t phase = 0;
  bool ok = true;
  uint64_t t_stop = 0;
  for (uint64_t t = blockIdx.x; t < n_tiles; t += gridDim.x) {
    if (tid == 0) {
      const WaitCtl ctl{&abort_flag, err, timeout_ns};
      if (!mbar_wait(&full[s], phase, ctl)) abort_flag = 1;
    }
    __syncthreads();
    if (abort_flag) {
      ok = false;
      t_stop = t;
      break;
    }
    const uint64_t c0 = t * kTileChunks;
    constexpr int kU = Op::kUnit;
#pragma unroll
    for (int u = 0; u < kTileChunks / (kU * kThreads); ++u) {
      const int cl = (u * kThreads + tid) * kU;   // first chunk of this thread's unit
      const uint64_t c = c0 + cl;
      const bool valid = c < n_chunks;           // units never straddle n_chunks
      uint4 v[kU];
#pragma unroll
      for (int k = 0; k < kU; ++k)
        v[k] = valid ? lds128(buf + s * kTileChunks + cl + k) : make_uint4(0u, 0u, 0u, 0u);
      op.unit(v, c, valid);
    }
    __syncthreads();   // every thread is done with this stage
    if (tid == 0) {
      const uint64_t nt = t + (uint64_t)kStages * gridDim.x;
      if (nt < n_tiles) issue(nt, s);
    }
    if (++s == kStages) {
      s = 0;
      phase ^= 1u;
    }
  }
  if (!ok && tid == 0) {
    // Let every copy already issued land before the CTA exits: the tiles
    // t_stop, t_stop + G, ... (at most kStages of them) sit in stages
    // s, s + 1, ... with the current phase, flipping on wrap-around.
    uint64_t tt = t_stop;
    for (int i = 0; i < kStages && tt < n_tiles; ++i, tt += gridDim.x) {
      const uint32_t a = smem_u32(&full[s]);
      const uint64_t t0 = global_timer_ns();
      while (!mbar_try_wait(a, phase) && global_timer_ns() - t0 < timeout_ns) {
      }
      if (++s == kStages) {
        s = 0;
        phase ^= 1u;
      }
    }
  }
  return ok;
}

// The first 16 KB per CTA of x into L2 (one bulk prefetch from thread 0 of
// each), issued before grid_dep_wait: a prefetch is a hint that returns no
// data, so it is correct even while the previous kernel still writes x, and the
// DRAM reads overlap that kernel's tail.  (Static NVFP4 through the ring,
// 4608 x 3072: 9.1 -> 8.0 us in a chain of launches, 9.3 -> 8.3 us right after a
// fused GEMM, unchanged alone after an L2 flush.  The kernels that load straight
// to registers have 32 KB tiles; prefetching those whole measured 7.5 -> 7.8 us
// there, 38.9 -> 38.6 in two_phase_kernel at 18432 x 3072.)
__device__ __forceinline__ void l2_prefetch_first_tile(const uint4* x, uint64_t n_chunks) {
  if (threadIdx.x == 0 && (uint64_t)blockIdx.x * kTileChunks < n_chunks) {
    const uint64_t c0 = (uint64_t)blockIdx.x * kTileChunks;
    const uint64_t left = n_chunks - c0;
    const uint32_t nc = left < (uint64_t)kTileChunks ? (uint32_t)left : (uint32_t)kTileChunks;
    l2_prefetch_bulk(x + c0, nc * 16u);
  }
}

// Block 0 records the static tensor scale S_dec.
__device__ __forceinline__ float static_scale(const float* scale_src, float* sdec_out) {
  const float s_dec = *scale_src;
  if (blockIdx.x == 0 && threadIdx.x == 0 && sdec_out != scale_src) *sdec_out = s_dec;
  return s_dec;
}

// NVFP4 with a static scale: x goes straight to registers (32 bytes, one block,
// per load where x is 32-byte aligned), each thread loading its next tile's
// units while it quantizes this one's.  Two CTAs of 512 threads per SM keep
// 64 KB per SM of loads in flight.  Bound by HBM: 18432 x 3072 in 22.4-23.2 us
// (6.2-6.5 TB/s), through the shared-memory ring 24.1-25.5 (its block reads have
// two-way bank conflicts); 4608 x 3072 7.5 us, through the ring 7.8.  256-thread
// CTAs with one to three units measured 22.3-23.6 us and 7.7-8.6 us.
constexpr int kDirectPerSm = 2;
constexpr int kDirectUnits = 2;                                       // per thread and tile
constexpr uint32_t kDirectTile = 2u * kThreads * kDirectUnits;        // chunks: 32 KB

__device__ __forceinline__ void ldg256(const uint4* p, uint4 (&v)[2]) {
  asm volatile("ld.global.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0].x), "=r"(v[0].y), "=r"(v[0].z), "=r"(v[0].w), "=r"(v[1].x),
                 "=r"(v[1].y), "=r"(v[1].z), "=r"(v[1].w)
               : "l"(p));
}

// The same of a small x: one block per thread, no table (its barrier and
// division come before the first block), as long as every block has a thread at
// once.  Bound by latency: 128 x 256 1.91 us in the persistent kernel, 1.26 here
// (1.74 through the ring); 300 x 3072 2.23 -> 1.64, 1333 x 3072 2.95 -> 2.58.  CTAs
// of 128 and 512 threads measured within 0.3 us of it.
constexpr int kSmallThreads = 256;
constexpr uint64_t kSmallPerSm = 2 * 2048;   // chunks: a block per resident thread

__global__ void __launch_bounds__(kSmallThreads)
    quant_nvfp4_small_kernel(const uint4* __restrict__ x, uint32_t n_chunks,
                             const float* scale_src, float* sdec_out, Nvfp4Op<uint32_t> op) {
  grid_dep_wait();
  grid_dep_launch();
  const uint32_t c = 2u * (blockIdx.x * kSmallThreads + threadIdx.x);
  const bool own = c < n_chunks;   // blocks never straddle n_chunks
  uint4 v[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) v[k] = own ? ldg128(x + c + k) : make_uint4(0u, 0u, 0u, 0u);
  op.s_enc = encode_scale(static_scale(scale_src, sdec_out));
  op.block(v, c, own);
}

template <typename Idx>
__global__ void __launch_bounds__(kThreads, kDirectPerSm)
    quant_nvfp4_kernel(const uint4* __restrict__ x, uint64_t n_chunks, int64_t K,
                       const float* scale_src, float* sdec_out, uint32_t* __restrict__ codes,
                       uint8_t* __restrict__ scales, uint3 row_div) {
  l2_prefetch_first_tile(x, n_chunks);
  grid_dep_wait();
  grid_dep_launch();
  __shared__ float r_table[128];
  Nvfp4Op<Idx> op;
  op.r_table = r_table;
  op.chunks_per_row = (Idx)(K >> 3);
  op.div_m = row_div.x;
  op.div_s1 = row_div.y;
  op.div_s2 = row_div.z;
  op.K = K;
  op.codes = codes;
  op.scales = scales;
  const uint64_t n_tiles = (n_chunks + kDirectTile - 1) / kDirectTile;
  const bool v8 = (reinterpret_cast<uintptr_t>(x) & 31u) == 0;
  auto first = [&](uint64_t t, int k) {   // first chunk of unit k of tile t
    return t * kDirectTile + 2u * (uint32_t)(k * kThreads + threadIdx.x);
  };
  auto load = [&](uint64_t t, uint4 (&v)[kDirectUnits][2]) {
#pragma unroll
    for (int k = 0; k < kDirectUnits; ++k) {
      const uint64_t c = first(t, k);   // units never straddle n_chunks
      if (c >= n_chunks) {
        v[k][0] = v[k][1] = make_uint4(0u, 0u, 0u, 0u);
      } else if (v8) {
        ldg256(x + c, v[k]);
      } else {
        v[k][0] = ldg128(x + c);
        v[k][1] = ldg128(x + c + 1);
      }
    }
  };
  auto quantize = [&](uint64_t t, const uint4 (&v)[kDirectUnits][2]) {
#pragma unroll
    for (int k = 0; k < kDirectUnits; ++k) {
      const uint64_t c = first(t, k);
      op.unit(v[k], c, c < n_chunks);
    }
  };
  uint4 v[kDirectUnits][2], w[kDirectUnits][2];
  uint64_t t = blockIdx.x;
  if (t < n_tiles) load(t, v);
  op.s_enc = encode_scale(static_scale(scale_src, sdec_out));
  op.init();
  __syncthreads();
  while (t < n_tiles) {
    uint64_t nt = t + gridDim.x;
    if (nt < n_tiles) load(nt, w);
    quantize(t, v);
    t = nt;
    if (t >= n_tiles) break;
    nt = t + gridDim.x;
    if (nt < n_tiles) load(nt, v);
    quantize(t, w);
    t = nt;
  }
}

// NVFP4 with a static scale, of an x that the kernel before has just written (the
// dynamic chain's y): through the ring, whose 192 KB per SM of bulk copies in
// flight start on x as soon as that kernel ends.  The direct loads above are
// faster on an x that comes from HBM alone, but took 25.3 us instead of 20.6
// right after a 4608 x 12288 GEMM (chains: 4608 x 12288 x 256 61.0 -> 56.7 us,
// 4608 x 9216 x 3072 60.8 -> 59.7, 18432 x 6144 x 256 117 -> 111).
__global__ void __launch_bounds__(kThreads, kBlocksPerSm)
    quant_nvfp4_ring_kernel(const uint4* __restrict__ x, uint64_t n_chunks,
                            const float* scale_src, float* sdec_out, Nvfp4Op<uint32_t> op,
                            unsigned* err, uint64_t timeout_ns) {
  l2_prefetch_first_tile(x, n_chunks);
  grid_dep_wait();
  grid_dep_launch();
  __shared__ float r_table[128];
  op.bind(r_table);
  stream_tiles(
      x, n_chunks, op,
      [&](Nvfp4Op<uint32_t>& o) { o.s_enc = encode_scale(static_scale(scale_src, sdec_out)); },
      err, timeout_ns);
}

__global__ void __launch_bounds__(kThreads, kBlocksPerSm)
    quant_fp8_kernel(const uint4* __restrict__ x, uint64_t n_chunks, const float* scale_src,
                     float* sdec_out, Fp8Op op, unsigned* err, uint64_t timeout_ns) {
  l2_prefetch_first_tile(x, n_chunks);
  grid_dep_wait();
  grid_dep_launch();
  stream_tiles(
      x, n_chunks, op,
      [&](Fp8Op& o) { o.s_enc = encode_scale(static_scale(scale_src, sdec_out)); }, err,
      timeout_ns);
}

// FP8 weights, one scale per row: one warp per row, held in kRegs chunks per lane
// (kTwoPass: longer rows in two passes, the second of which hits L1/L2).  Short
// rows take an instance of their own, with as many CTAs per SM as its registers
// allow: through the twelve-chunk one 100003 x 64 took 42.8 us (14.6 with two
// chunks, 18.7 in two passes) and 12288 x 1024 9.6 (7.2 with four chunks, 8.1).
// 12288 x 3072: 18.3 us, in two passes 21.2.  Offline, once per layer.
template <int kRegs, int kPerSm, bool kTwoPass = false>
__global__ void __launch_bounds__(kThreads, kPerSm)
    quant_fp8_rows_kernel(const uint4* __restrict__ w, int64_t rows, int64_t K,
                          float* __restrict__ s_rows, uint2* __restrict__ codes) {
  grid_dep_wait();
  grid_dep_launch();
  const int lane = threadIdx.x & 31;
  const int64_t cpr = K >> 3;
  const int64_t warp = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * kThreads) >> 5;
  for (int64_t r = warp; r < rows; r += nwarps) {
    const uint4* wr = w + r * cpr;
    uint32_t m = 0;
    if (!kTwoPass || cpr <= 32 * kRegs) {
      uint4 v[kRegs];
#pragma unroll
      for (int i = 0; i < kRegs; ++i)
        v[i] = lane + 32 * i < cpr ? ldg128(wr + lane + 32 * i) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
      for (int i = 0; i < kRegs; ++i) m = max(m, chunk_abs_max_bits(v[i]));
      m = __reduce_max_sync(0xFFFFFFFFu, m);
      const float amax = __uint_as_float(m << 16);
      const float s_dec = (amax == 0.0f) ? 1.0f : __fdiv_rn(amax, 448.0f);
      const float s_enc = encode_scale(s_dec);
      if (lane == 0) s_rows[r] = s_dec;
#pragma unroll
      for (int i = 0; i < kRegs; ++i) {
        if (lane + 32 * i >= cpr) continue;
        float f[8];
        unpack8(v[i], f);
#pragma unroll
        for (int e = 0; e < 8; ++e) f[e] = __fmul_rn(f[e], s_enc);
        codes[r * cpr + lane + 32 * i] =
            make_uint2(e4m3x4(f[0], f[1], f[2], f[3]), e4m3x4(f[4], f[5], f[6], f[7]));
      }
      continue;
    }
    if constexpr (kTwoPass) {
      for (int64_t c = lane; c < cpr; c += 32) m = max(m, chunk_abs_max_bits(__ldg(wr + c)));
      m = __reduce_max_sync(0xFFFFFFFFu, m);
      const float amax = __uint_as_float(m << 16);
      const float s_dec = (amax == 0.0f) ? 1.0f : __fdiv_rn(amax, 448.0f);
      const float s_enc = encode_scale(s_dec);
      if (lane == 0) s_rows[r] = s_dec;
      for (int64_t c = lane; c < cpr; c += 32) {
        float f[8];
        unpack8(__ldg(wr + c), f);
#pragma unroll
        for (int i = 0; i < 8; ++i) f[i] = __fmul_rn(f[i], s_enc);
        codes[r * cpr + c] =
            make_uint2(e4m3x4(f[0], f[1], f[2], f[3]), e4m3x4(f[4], f[5], f[6], f[7]));
      }
    }
  }
}

// ------------------------------------------------ one-pass dynamic scale ---
// The tensor scale depends on max |x| over the whole tensor, and the codes
// depend on the tensor scale, so a streaming quantizer reads x twice.  When x
// fits in the aggregate shared memory (or registers) of the grid, one CTA per
// SM, each CTA loads its slice once, the grid combines the slice maxima through
// two words of global memory, and each CTA quantizes its slice from where it
// holds it.
constexpr int kOnePassThreads = 1024;
constexpr int kOnePassSmem = 225 * 1024;
constexpr int kOnePassSliceMax = 14 * 1024;       // chunks: 224 KB of data at most
// NVFP4 steps of run_slice: two 2-chunk units per thread and step
constexpr int kOnePassSteps = (kOnePassSliceMax + 4 * kOnePassThreads - 1) / (4 * kOnePassThreads);

// The amax word and the arrival count as one 64-bit acquire load (they are
// adjacent words of one 8-byte-aligned pair, low word first).
__device__ __forceinline__ uint64_t ld_acquire_gpu_pair(const unsigned* p) {
  uint64_t v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// Wait until at most `pending` (0-3) of this thread's cp.async groups are
// still in flight (the operand must be an immediate; a constant argument
// folds the switch).
__device__ __forceinline__ void cp_async_wait_pending(int pending) {
  switch (pending) {
    case 3: asm volatile("cp.async.wait_group 3;" ::: "memory"); break;
    case 2: asm volatile("cp.async.wait_group 2;" ::: "memory"); break;
    case 1: asm volatile("cp.async.wait_group 1;" ::: "memory"); break;
    default: asm volatile("cp.async.wait_group 0;" ::: "memory"); break;
  }
}

// How often a CTA gave up waiting for its grid: CTAs that helped, pieces they
// read, CTAs that read all of x alone.  Counted on that path only.
__device__ unsigned g_grid_counts[3];

constexpr uint32_t kPieceChunks = 4096;       // 64 KB of x per ticket
constexpr unsigned kAllRead = 1u << 30;       // added to the arrivals (a grid has fewer CTAs)
constexpr uint32_t kMet = 0xFFFFFFFFu, kHelp = 0xFFFFFFFEu, kAlone = 0xFFFFFFFDu;

// The maximum of the grid's warp maxima (max |x|, as bits) into *s_amax (shared
// memory, for every thread): combine the CTA's, publish, arrive, wait for every
// CTA, depart.  The grid is no larger than the machine, so its CTAs are resident
// together unless other streams' kernels hold SMs -- for long, or waiting, as
// another grid like this one would.  So a CTA waits wait.help_ns only; then it
// takes pieces of x by ticket, with every other CTA that waits, and when all of x
// has been read that way the grid has met without the CTAs that are missing: they
// find it so when they start.  Nothing then waits on a CTA that is not running,
// and x is read once more in all.  (With 20 of 152 SMs held by another kernel,
// 4608 x 3072 takes 50 us and 18432 x 3072 89; waiting 1 ms for the missing CTAs
// and then reading all of x in every CTA took 1360 and 2820.  A cooperative
// launch, which keeps the grid together, costs about 2 us outside a graph: 2.5 MB
// of FP8 6.2 us instead of 4.5.)  The wait for the last pieces, which running CTAs
// hold, is bounded by wait.stop_ns; a CTA whose wait expires there reads all of x
// for itself.
//
// sync[0]: amax bits (fp32), sync[1]: arrivals, sync[2]: departures, sync[3]: the
// next ticket, sync[4]: pieces read.
template <int kThreadsPerBlock>
__device__ __forceinline__ void grid_amax(const uint4* x, uint64_t n_chunks, uint32_t* warp_max,
                                          unsigned* sync, float* s_amax, uint32_t* s_state,
                                          GridWait wait) {
  const int tid = threadIdx.x;
  __syncthreads();   // warp_max is written
  auto combine = [&] {
    uint32_t b = 0;
#pragma unroll
    for (int w = 0; w < kThreadsPerBlock / 32; ++w) b = max(b, warp_max[w]);
    return b;
  };
  // The count and the amax are read together: a load that sees every CTA's
  // arrival (or that all of x has been read) also sees every maximum released
  // before it, which saves the second round trip to L2 that reading the amax
  // afterwards took.
  auto met = [&] {
    const uint64_t pair = ld_acquire_gpu_pair(&sync[0]);
    if ((uint32_t)(pair >> 32) < gridDim.x) return false;
    *s_amax = __uint_as_float((uint32_t)pair);
    return true;
  };
  // Poll until the grid has met or limit_ns have passed (0: no poll).
  auto poll = [&](uint64_t limit_ns, uint32_t expired) {
    if (limit_ns == 0) return expired;
    const uint64_t t0 = global_timer_ns();
    while (!met())
      if (global_timer_ns() - t0 > limit_ns) return expired;
    return kMet;
  };
  if (tid == 0) {
    const uint32_t b = combine();
    if (b) atomicMax(&sync[0], b << 16);
    // the arrival releases the maximum above to every CTA that sees it
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&sync[1]) : "memory");
    // (a loop of its own, the common case: through poll() below 0.1 us slower)
    const uint64_t t0 = global_timer_ns();
    uint64_t pair = ld_acquire_gpu_pair(&sync[0]);
    bool expired = false;
    while ((uint32_t)(pair >> 32) < gridDim.x && !expired) {
      expired = global_timer_ns() - t0 > wait.help_ns;
      pair = ld_acquire_gpu_pair(&sync[0]);
    }
    *s_state = wait.help_ns == 0 || (uint32_t)(pair >> 32) < gridDim.x ? kHelp : kMet;
    *s_amax = __uint_as_float((uint32_t)pair);
  }
  __syncthreads();
  const uint32_t state = *s_state;
  // Depart (by 1, a CTA that helped by 1 and 65536); the last CTA out resets the
  // words, those of the pieces only if one helped.  The other warps do not wait
  // for this atomic's round trip.
  auto depart = [&](unsigned by) {
    if (tid == 0) {
      const unsigned before = atomicAdd(&sync[2], by);
      if ((before & 0xFFFFu) == gridDim.x - 1u) {
        sync[0] = 0u;
        sync[1] = 0u;
        sync[2] = 0u;
        if ((before + by) >> 16) {
          sync[3] = 0u;
          sync[4] = 0u;
        }
      }
    }
  };
  if (state == kMet) depart(1u);
  if (state == kHelp) {
    __syncthreads();   // every thread has read s_state
    const uint32_t pieces = (uint32_t)((n_chunks + kPieceChunks - 1) / kPieceChunks);
    bool done = false;   // thread 0: the grid has met
    if (tid == 0) atomicAdd(&g_grid_counts[0], 1u);
    for (;;) {
      if (tid == 0) {
        uint32_t t = kMet;
        if (!done && (t = atomicAdd(&sync[3], 1u)) >= pieces) t = poll(wait.stop_ns, kAlone);
        *s_state = t;
      }
      __syncthreads();
      const uint32_t t = *s_state;
      if (t >= pieces) break;
      // the last pieces first: the CTAs that are missing are mostly the last ones
      const uint64_t c0 = (uint64_t)(pieces - 1u - t) * kPieceChunks;
      uint32_t m = 0;
#pragma unroll 4
      for (uint32_t i = tid; i < kPieceChunks; i += kThreadsPerBlock)
        if (c0 + i < n_chunks) m = max(m, chunk_abs_max_bits(ldg128(x + c0 + i)));
      m = __reduce_max_sync(0xFFFFFFFFu, m);
      if ((tid & 31) == 0) warp_max[tid >> 5] = m;
      __syncthreads();
      if (tid == 0) {
        atomicAdd(&g_grid_counts[1], 1u);
        const uint32_t b = combine();
        if (b) atomicMax(&sync[0], b << 16);
        __threadfence();
        if (atomicAdd(&sync[4], 1u) == pieces - 1u) {
          __threadfence();
          asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(&sync[1]), "r"(kAllRead)
                       : "memory");
        }
        done = met();
      }
    }
    if (*s_state == kAlone) {
      if (tid == 0) atomicAdd(&g_grid_counts[2], 1u);
      uint32_t m = 0;
      for (uint64_t c = tid; c < n_chunks; c += kThreadsPerBlock)
        m = max(m, chunk_abs_max_bits(ldg128(x + c)));
      m = __reduce_max_sync(0xFFFFFFFFu, m);
      if ((tid & 31) == 0) warp_max[tid >> 5] = m;
      __syncthreads();
      if (tid == 0) *s_amax = __uint_as_float(combine() << 16);
      __syncthreads();
    }
    depart(0x10001u);
  }
}

// sync: the words of grid_amax, all zero at launch; the last CTA to depart zeroes
// them again, so back-to-back launches (graph replays included) need no clearing
// between.
template <typename Op>
__global__ void __launch_bounds__(kOnePassThreads, 1)
    onepass_kernel(const uint4* __restrict__ x, uint64_t n_chunks, uint32_t slice, Op op,
                   float qmax, float* sdec_out, unsigned* sync, GridWait wait) {
  extern __shared__ __align__(128) uint8_t qsm[];
  uint4* buf = reinterpret_cast<uint4*>(qsm);
  __shared__ uint32_t warp_max[kOnePassThreads / 32];
  __shared__ float op_table[128];
  __shared__ float s_amax;
  __shared__ uint32_t state;
  grid_dep_wait();
  const int tid = threadIdx.x;
  const uint64_t c_begin = (uint64_t)blockIdx.x * slice;
  const uint32_t n = c_begin >= n_chunks ? 0u
                     : (uint32_t)(n_chunks - c_begin < slice ? n_chunks - c_begin : slice);
  // every thread copies its chunks (a dozen 16-byte asynchronous copies in
  // flight per thread), then takes their amax; it reads only the chunks it
  // copied itself, so waiting for its own copies suffices.  NVFP4 copies in
  // the units run_slice quantizes (two adjacent chunks, a warp covering 1 KB),
  // one copy group per step of block maxima, so that each step's maxima are
  // taken while the later steps' copies are still landing (4608 x 3072, which
  // regpass_kernel takes now: 12.46 -> 12.23 us)
  const uint4* xs = x + c_begin;
  if constexpr (Op::kBlockMax) {
#pragma unroll
    for (int s = 0; s < 2 * kOnePassSteps; ++s) {
      const uint32_t c = (uint32_t)s * 2u * kOnePassThreads + 2u * tid;
      if (c < n) {
        cp_async16(smem_u32(buf + c), xs + c);
        cp_async16(smem_u32(buf + c + 1), xs + c + 1);
      }
      if (s & 1) asm volatile("cp.async.commit_group;" ::: "memory");   // step s / 2
    }
  } else {
    for (uint32_t i = tid; i < n; i += kOnePassThreads) cp_async16(smem_u32(buf + i), xs + i);
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_all;" ::: "memory");
    grid_dep_launch();   // x is on chip: the next kernel may begin launching
  }
  uint32_t m = 0;
  uint32_t bm[kOnePassSteps] = {};
  if constexpr (Op::kBlockMax) {
    // NVFP4: the amax of each 16-element block this thread will quantize
    // (the units of run_slice), kept for after the barrier
    static_assert(kOnePassSteps <= 4, "cp_async_wait_pending takes 0-3 groups");
#pragma unroll
    for (int s = 0; s < kOnePassSteps; ++s) {
      cp_async_wait_pending(kOnePassSteps - 1 - s);   // steps 0..s have landed
      if (s == kOnePassSteps - 1) grid_dep_launch();  // x is on chip
      const uint32_t ca = (uint32_t)s * 4u * kOnePassThreads + 2u * tid;
      const uint32_t cb = ca + 2u * kOnePassThreads;
      const uint32_t a =
          ca < n ? block_abs_max_bits(lds128(buf + ca), lds128(buf + ca + 1))
                 : 0u;
      const uint32_t b =
          cb < n ? block_abs_max_bits(lds128(buf + cb), lds128(buf + cb + 1))
                 : 0u;
      bm[s] = a | (b << 16);
      m = max(m, max(a, b));
    }
  } else {
    for (uint32_t i = tid; i < n; i += kOnePassThreads)
      m = max(m, chunk_abs_max_bits(lds128(buf + i)));
  }
  m = __reduce_max_sync(0xFFFFFFFFu, m);
  if ((tid & 31) == 0) warp_max[tid >> 5] = m;
  grid_amax<kOnePassThreads>(x, n_chunks, warp_max, sync, &s_amax, &state, wait);
  const float amax = s_amax;
  const float s_dec = (amax == 0.0f) ? 1.0f : __fdiv_rn(amax, qmax);
  if (blockIdx.x == 0 && tid == 0) *sdec_out = s_dec;
  op.s_enc = encode_scale(s_dec);
  op.bind(op_table);
  op.init();
  __syncthreads();
  if constexpr (Op::kBlockMax)
    op.template run_slice<kOnePassThreads, kOnePassSteps>(buf, n, c_begin, bm);
  else
    op.template run_slice<kOnePassThreads>(buf, n, c_begin);
}

// NVFP4, x held in registers instead of shared memory (up to kRegUnits 32-byte
// units, one block each, per thread): no trip through shared memory, whose
// 32-byte-strided reads (each block twice, with two-way bank conflicts) made up
// 6500 of the 21 000 cycles of the shared-memory kernel.  4608 x 3072: 12.2 ->
// 11.2 us, 1000 x 3072: 5.45 -> 5.1 us.  (FP8 in this form: 11.1 -> 10.9 us,
// but 3.9 -> 4.6 us at 2.5 MB, so it keeps the shared-memory kernel.)  Reading
// x from HBM takes ~6 us of it, the grid barrier ~1.3 us.  (32-byte loads:
// 1000 x 3072 5.1 -> 4.95 us, but 4608 x 3072 11.2 -> 11.4.)
constexpr int kRegThreads = 512;
constexpr int kRegUnits = 12;
constexpr uint32_t kRegStride = 2u * kRegThreads;               // chunks between a thread's units
constexpr uint32_t kRegSliceMax = kRegUnits * kRegStride;       // 192 KB of x per CTA

template <typename Op>
__global__ void __launch_bounds__(kRegThreads, 1)
    regpass_kernel(const uint4* __restrict__ x, uint64_t n_chunks, uint32_t slice, Op op,
                   float qmax, float* sdec_out, unsigned* sync, GridWait wait) {
  __shared__ uint32_t warp_max[kRegThreads / 32];
  __shared__ float op_table[128];
  __shared__ float s_amax;
  __shared__ uint32_t state;
  grid_dep_wait();
  const uint32_t tid = threadIdx.x;
  const uint64_t c_begin = (uint64_t)blockIdx.x * slice;
  const uint32_t n = c_begin >= n_chunks ? 0u
                     : (uint32_t)(n_chunks - c_begin < slice ? n_chunks - c_begin : slice);
  const uint4* xs = x + c_begin + 2u * tid;
  uint4 v[kRegUnits][2];
#pragma unroll
  for (int u = 0; u < kRegUnits; ++u) {
    const bool in = (uint32_t)u * kRegStride + 2u * tid < n;   // units never straddle n
#pragma unroll
    for (int k = 0; k < 2; ++k)
      v[u][k] = in ? ldg128(xs + u * kRegStride + k) : make_uint4(0u, 0u, 0u, 0u);
  }
  uint32_t m = 0;
  uint32_t bm[kRegUnits / 2];   // block maxima, two to a word
#pragma unroll
  for (int u = 0; u < kRegUnits; ++u) {
    const uint32_t b = block_abs_max_bits(v[u][0], v[u][1]);
    if (u & 1)
      bm[u / 2] |= b << 16;
    else
      bm[u / 2] = b;
    m = max(m, b);
  }
  grid_dep_launch();   // x is on chip: the next kernel may begin launching
  m = __reduce_max_sync(0xFFFFFFFFu, m);
  if ((tid & 31u) == 0u) warp_max[tid >> 5] = m;
  grid_amax<kRegThreads>(x, n_chunks, warp_max, sync, &s_amax, &state, wait);
  const float amax = s_amax;
  const float s_dec = (amax == 0.0f) ? 1.0f : __fdiv_rn(amax, qmax);
  if (blockIdx.x == 0 && tid == 0) *sdec_out = s_dec;
  op.s_enc = encode_scale(s_dec);
  op.bind(op_table);
  op.init();
  __syncthreads();
  op.template run_units<kRegUnits, kRegStride>(v, bm, n, c_begin);
}

// Dynamic scale of an x that does not fit on chip: one launch reads x for its
// amax, meets at the grid barrier and quantizes its tiles in reverse order: the
// last three of every CTA (29 MB in all) wait in shared memory, and the ones
// before them are the lines most recently in L2.  Loads as in
// quant_nvfp4_kernel.  Bound by HBM and latency: 18432 x 3072 reads its 113 MB in
// 19 us (of 165 MB read in all: L2 keeps ~30 MB of them) and quantizes in 20.
// NVFP4 39.0 us, FP8 38.1 us (6000 x 3072: 14.7 and 13.2); without the tiles
// kept 39.2 and 39.3 (15.1 and 14.2); an amax kernel and the quantizer after it
// took 48.1 and 50.1.
constexpr int kKeep = 3;                                             // tiles of 32 KB per CTA
constexpr int kKeepSmem = kKeep * (int)kDirectTile * 16;

template <typename Op>
__global__ void __launch_bounds__(kThreads, kDirectPerSm)
    two_phase_kernel(const uint4* __restrict__ x, uint64_t n_chunks, Op op, float qmax,
                     float* sdec_out, unsigned* sync, GridWait wait) {
  extern __shared__ __align__(128) uint8_t qsm[];
  uint4* const keep = reinterpret_cast<uint4*>(qsm);
  __shared__ uint32_t warp_max[kThreads / 32];
  __shared__ float op_table[128];
  __shared__ float s_amax;
  __shared__ uint32_t state;
  l2_prefetch_first_tile(x, n_chunks);
  grid_dep_wait();
  grid_dep_launch();
  const uint32_t tid = threadIdx.x;
  const int64_t n_tiles = (int64_t)((n_chunks + kDirectTile - 1) / kDirectTile);
  const bool v8 = (reinterpret_cast<uintptr_t>(x) & 31u) == 0;
  auto first = [&](int64_t t, int k) {
    return (uint64_t)t * kDirectTile + 2u * (uint32_t)(k * kThreads + tid);
  };
  auto load = [&](int64_t t, uint4 (&v)[kDirectUnits][2]) {
#pragma unroll
    for (int k = 0; k < kDirectUnits; ++k) {
      const uint64_t c = first(t, k);
      if (t >= n_tiles || t < 0 || c >= n_chunks) {
        v[k][0] = v[k][1] = make_uint4(0u, 0u, 0u, 0u);
      } else if (v8) {
        ldg256(x + c, v[k]);
      } else {
        v[k][0] = ldg128(x + c);
        v[k][1] = ldg128(x + c + 1);
      }
    }
  };
  uint32_t m = 0;
  auto amax = [&](const uint4 (&v)[kDirectUnits][2]) {
#pragma unroll
    for (int k = 0; k < kDirectUnits; ++k)
      m = max(m, block_abs_max_bits(v[k][0], v[k][1]));
  };
  // The CTA's last kKeep tiles also stay in shared memory (each thread keeps and
  // reads back its own units; 16-byte accesses side by side).
  auto slot = [&](int r, int k, int h) {
    return keep + ((r * kDirectUnits + k) * 2 + h) * kThreads + tid;
  };
  const int64_t g = gridDim.x;
  const int64_t own = (n_tiles - (int64_t)blockIdx.x + g - 1) / g;   // tiles of this CTA
  const int64_t kept = own - kKeep;                                  // the first one kept
  auto tile = [&](int64_t i) { return (int64_t)blockIdx.x + i * g; };
  auto take = [&](int64_t i, const uint4 (&v)[kDirectUnits][2]) {
    amax(v);
    if (i < kept) return;
#pragma unroll
    for (int k = 0; k < kDirectUnits; ++k)
#pragma unroll
      for (int h = 0; h < 2; ++h) *slot((int)(i - kept), k, h) = v[k][h];
  };
  uint4 v[kDirectUnits][2], w[kDirectUnits][2];
  {
    uint4 u[kDirectUnits][2];   // two tiles in flight beside the one taken
    load(tile(0), v);
    load(tile(1), w);
    for (int64_t i = 0; i < own; i += 3) {
      load(tile(i + 2), u);
      take(i, v);
      if (i + 1 >= own) break;
      load(tile(i + 3), v);
      take(i + 1, w);
      if (i + 2 >= own) break;
      load(tile(i + 4), w);
      take(i + 2, u);
    }
  }
  m = __reduce_max_sync(0xFFFFFFFFu, m);
  if ((tid & 31) == 0) warp_max[tid >> 5] = m;
  load(kept > 0 ? tile(kept - 1) : -1, v);   // the first tile not kept, while the grid meets
  grid_amax<kThreads>(x, n_chunks, warp_max, sync, &s_amax, &state, wait);
  const float am = s_amax;
  const float s_dec = (am == 0.0f) ? 1.0f : __fdiv_rn(am, qmax);
  if (blockIdx.x == 0 && tid == 0) *sdec_out = s_dec;
  op.s_enc = encode_scale(s_dec);
  op.bind(op_table);
  op.init();
  __syncthreads();
  auto quantize = [&](int64_t t, const uint4 (&v)[kDirectUnits][2]) {
#pragma unroll
    for (int k = 0; k < kDirectUnits; ++k) {
      const uint64_t c = first(t, k);
      op.pair(v[k], c, c < n_chunks);
    }
  };
  for (int64_t i = own - 1; i >= 0 && i >= kept; --i) {
#pragma unroll
    for (int k = 0; k < kDirectUnits; ++k)
#pragma unroll
      for (int h = 0; h < 2; ++h) w[k][h] = *slot((int)(i - kept), k, h);
    quantize(tile(i), w);
  }
  for (int64_t i = kept - 1; i >= 0; i -= 2) {
    load(i >= 1 ? tile(i - 1) : -1, w);
    quantize(tile(i), v);
    if (i < 1) break;
    load(i >= 2 ? tile(i - 2) : -1, v);
    quantize(tile(i - 1), w);
  }
}

// Small x: every cluster of eight CTAs reads all of x (an eighth per CTA, from
// L2 after the first), combines the maxima through distributed shared memory
// and quantizes its share, so the grid needs no grid-wide barrier.  One
// 16-element block (two chunks) per thread, loaded first and kept in registers.
// Bound by latency: launch, one load, one cluster barrier (128 x 256: NVFP4 4.46
// -> 2.2 us, FP8 3.4 -> 2.0 us against the grid-wide routes).
constexpr int kClusterCtas = 8;
constexpr int kClusterThreads = 512;
constexpr uint32_t kClusterSub = 2 * kClusterThreads;   // chunks a CTA quantizes at most

__device__ __forceinline__ void st_shared_cluster_u32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// range: chunks of a CTA's eighth of x; sub: chunks of it that each of the
// grid's clusters quantizes (both multiples of 8, sub <= kClusterSub).
template <typename Op>
__global__ void __launch_bounds__(kClusterThreads, 1)
    cluster_quant_kernel(const uint4* __restrict__ x, uint32_t n_chunks, uint32_t range,
                         uint32_t sub, Op op, float qmax, float* sdec_out) {
  __shared__ uint32_t warp_max[kClusterThreads / 32];
  __shared__ uint32_t cta_max[kClusterCtas];
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  grid_dep_wait();
  const uint32_t tid = threadIdx.x;
  const uint32_t rank = cluster_ctarank();
  const uint32_t r0 = min(rank * range, n_chunks), r1 = min(r0 + range, n_chunks);
  const uint32_t s0 = r0 + (blockIdx.x / kClusterCtas) * sub;
  const uint32_t s1 = min(s0 + sub, r1);
  const uint32_t c = s0 + 2u * tid;
  const bool own = c < s1;
  uint4 v[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) v[k] = own ? ldg128(x + c + k) : make_uint4(0u, 0u, 0u, 0u);
  uint32_t m = 0;
  uint32_t i = r0 + tid;
  for (; i + 7u * kClusterThreads < r1; i += 8u * kClusterThreads) {   // eight loads in flight
    uint4 t[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) t[k] = ldg128(x + i + k * kClusterThreads);
#pragma unroll
    for (int k = 0; k < 8; ++k) m = max(m, chunk_abs_max_bits(t[k]));
  }
  for (; i < r1; i += kClusterThreads) m = max(m, chunk_abs_max_bits(ldg128(x + i)));
  grid_dep_launch();
  m = __reduce_max_sync(0xFFFFFFFFu, m);
  if ((tid & 31u) == 0u) warp_max[tid >> 5] = m;
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");   // the peers have started
  __syncthreads();
  if (tid < (uint32_t)kClusterCtas) {
    uint32_t b = 0;
#pragma unroll
    for (int w = 0; w < kClusterThreads / 32; ++w) b = max(b, warp_max[w]);
    st_shared_cluster_u32(mapa_shared(&cta_max[rank], tid), b);
  }
  __syncwarp();
  cluster_sync();
  uint32_t b = 0;
#pragma unroll
  for (int r = 0; r < kClusterCtas; ++r) b = max(b, cta_max[r]);
  const float amax = __uint_as_float(b << 16);
  const float s_dec = (amax == 0.0f) ? 1.0f : __fdiv_rn(amax, qmax);
  if (blockIdx.x == 0 && tid == 0) *sdec_out = s_dec;
  op.s_enc = encode_scale(s_dec);
  op.block(v, c, own);
}

// Opt a kernel into `smem` bytes of dynamic shared memory and find how many of its
// CTAs an SM holds, once per device.
struct Setup {
  cudaError_t err;
  int resident;
};
template <auto kKern>
const Setup& setup(Device dev, int threads, int smem) {
  static PerDevice<Setup> per_device;
  return per_device.get(dev.index, [&] {
    Setup t{cudaFuncSetAttribute(kKern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem), 0};
    if (t.err == cudaSuccess && cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                                    &t.resident, kKern, threads, smem) != cudaSuccess)
      t.resident = 0;
    return t;
  });
}

// Launch with programmatic stream serialization (see grid_dep_wait).
template <typename... Params, typename... Args>
cudaError_t launch_pdl(void (*kern)(Params...), int grid, int block, int smem, cudaStream_t s,
                       Args... args) {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3((unsigned)block, 1, 1);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

int stream_grid(uint64_t n_chunks, int num_sms) {
  const uint64_t tiles = (n_chunks + kTileChunks - 1) / kTileChunks;
  return (int)std::max<uint64_t>(1, std::min<uint64_t>(tiles, (uint64_t)num_sms * kBlocksPerSm));
}

}  // namespace

// One-pass dynamic quantization when x fits on chip: returns
// cudaErrorNotSupported (nothing launched) when it does not, or when the
// device cannot hold the grid resident.
template <typename Op>
static cudaError_t launch_onepass(const void* x, uint64_t n_chunks, const Op& op, float qmax,
                                  float* sdec_out, unsigned* sync, bool clear, cudaStream_t s,
                                  Device dev, GridWait wait) {
  // slices of whole 64-element groups (8 chunks), one per SM
  uint64_t slice = (n_chunks + dev.num_sms - 1) / dev.num_sms;
  slice = (slice + 7) / 8 * 8;
  if (slice > (uint64_t)kOnePassSliceMax || slice == 0) return cudaErrorNotSupported;
  const int grid = (int)((n_chunks + slice - 1) / slice);
  // NVFP4: held in registers where the slice fits, else in shared memory
  const bool reg = Op::kBlockMax && slice <= (uint64_t)kRegSliceMax;
  const int threads = reg ? kRegThreads : kOnePassThreads, smem = reg ? 0 : kOnePassSmem;
  auto kern = onepass_kernel<Op>;
  const Setup* st = nullptr;
  if constexpr (Op::kBlockMax) {
    if (reg) {
      kern = regpass_kernel<Op>;
      st = &setup<regpass_kernel<Op>>(dev, threads, smem);
    }
  }
  if (st == nullptr) st = &setup<onepass_kernel<Op>>(dev, threads, smem);
  if (st->err != cudaSuccess) return st->err;
  if (st->resident < 1 || grid > dev.num_sms * st->resident) return cudaErrorNotSupported;
  if (clear) {
    const cudaError_t e = cudaMemsetAsync(sync, 0, kGridSyncWords * sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
  }
  return launch_pdl(kern, grid, threads, smem, s, static_cast<const uint4*>(x), n_chunks,
                    (uint32_t)slice, op, qmax, sdec_out, sync, wait);
}

// x of any size: two phases over it in one launch.
template <typename Op>
static cudaError_t launch_two_phase(const void* x, uint64_t n_chunks, const Op& op, float qmax,
                                    float* sdec_out, unsigned* sync, bool clear, cudaStream_t s,
                                    Device dev, GridWait wait) {
  const Setup& st = setup<two_phase_kernel<Op>>(dev, kThreads, kKeepSmem);
  cudaError_t e = st.err;
  if (e != cudaSuccess) return e;
  if (st.resident < 1) return cudaErrorLaunchOutOfResources;
  if (clear && (e = cudaMemsetAsync(sync, 0, kGridSyncWords * sizeof(unsigned), s)) != cudaSuccess) return e;
  const uint64_t tiles = (n_chunks + kDirectTile - 1) / kDirectTile;
  const int grid = (int)std::min<uint64_t>(tiles, (uint64_t)dev.num_sms * std::min(st.resident, kDirectPerSm));
  return launch_pdl(two_phase_kernel<Op>, grid, kThreads, kKeepSmem, s, static_cast<const uint4*>(x),
                    n_chunks, op, qmax, sdec_out, sync, wait);
}

// The cluster route takes x of up to 1 MB: there every CTA's eighth of x takes
// as long to read as the grid barrier it saves (NVFP4: 1 MB 3.9 us against 4.7
// on the grid-wide routes, 2 MB 6.2 against 4.8; FP8: 3.6 against 3.55 and 5.6
// against 3.7).
constexpr uint64_t kClusterMaxChunks = 1024 * 64;

template <typename Op>
static cudaError_t launch_cluster_quant(const void* x, uint32_t n_chunks, const Op& op,
                                        float qmax, float* sdec_out, cudaStream_t s) {
  const uint32_t range = ((n_chunks + kClusterCtas - 1) / kClusterCtas + 7) / 8 * 8;
  const uint32_t clusters = (range + kClusterSub - 1) / kClusterSub;
  const uint32_t sub = ((range + clusters - 1) / clusters + 7) / 8 * 8;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kClusterCtas;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3(clusters * kClusterCtas, 1, 1);
  cfg.blockDim = dim3(kClusterThreads, 1, 1);
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, cluster_quant_kernel<Op>, static_cast<const uint4*>(x), n_chunks,
                            range, sub, op, qmax, sdec_out);
}

// Multiplier and shifts that divide a 32-bit index by d (1 <= d < 2^31)
// without a division instruction: the round-up form of Granlund and
// Montgomery (PLDI 1994), exact for every 32-bit dividend.
static uint3 invariant_divisor(uint32_t d) {
  int l = 0;
  while ((1ull << l) < d) ++l;   // ceil(log2 d)
  const uint64_t m = ((1ull << 32) * ((1ull << l) - d)) / d + 1;
  return make_uint3((uint32_t)m, (uint32_t)(l < 1 ? l : 1), (uint32_t)(l > 1 ? l - 1 : 0));
}

// The arithmetic and addressing of an NVFP4 quantizer of x [M, K] into `out`;
// s_enc and the table are set in the kernel.
template <typename Idx>
static Nvfp4Op<Idx> nvfp4_op(int64_t K, const qlin_nvfp4_t& out) {
  Nvfp4Op<Idx> op;
  op.s_enc = 0.0f;
  op.chunks_per_row = (Idx)(K >> 3);
  const uint3 row_div = invariant_divisor((uint32_t)(K >> 3));
  op.div_m = row_div.x;
  op.div_s1 = row_div.y;
  op.div_s2 = row_div.z;
  op.K = K;
  op.codes = reinterpret_cast<uint32_t*>(out.codes);
  op.scales = out.scales;
  op.r_table = nullptr;
  return op;
}

static Fp8Op fp8_op(const qlin_fp8_t& out) {
  Fp8Op op;
  op.s_enc = 0.0f;
  op.codes = reinterpret_cast<uint2*>(out.codes);
  return op;
}

// By size: every cluster reads x (latency), x held on chip (one read), two
// phases over x.
template <typename Op>
static cudaError_t launch_dynamic(const void* x, uint64_t n_chunks, const Op& op, float qmax,
                                  float* sdec_out, unsigned* sync, bool clear, cudaStream_t s,
                                  Device dev, GridWait wait) {
  if (n_chunks <= kClusterMaxChunks)
    return launch_cluster_quant(x, (uint32_t)n_chunks, op, qmax, sdec_out, s);
  const cudaError_t e = launch_onepass(x, n_chunks, op, qmax, sdec_out, sync, clear, s, dev,
                                       wait);
  if (e != cudaErrorNotSupported) return e;
  return launch_two_phase(x, n_chunks, op, qmax, sdec_out, sync, clear, s, dev,
                          wait);
}

cudaError_t launch_quant_nvfp4_dynamic(const void* x, int64_t M, int64_t K,
                                       const qlin_nvfp4_t& out, unsigned* sync, bool clear,
                                       cudaStream_t s, Device dev, GridWait wait) {
  const uint64_t n_chunks = (uint64_t)M * (uint64_t)K / 8;
  if (n_chunks < (1ull << 32))   // 32-bit index math is enough
    return launch_dynamic(x, n_chunks, nvfp4_op<uint32_t>(K, out), 2688.0f, out.tensor_scale, sync,
                          clear, s, dev, wait);
  return launch_two_phase(x, n_chunks, nvfp4_op<uint64_t>(K, out), 2688.0f, out.tensor_scale, sync,
                          clear, s, dev, wait);
}

cudaError_t launch_quant_fp8_dynamic(const void* x, int64_t M, int64_t K, const qlin_fp8_t& out,
                                     unsigned* sync, bool clear, cudaStream_t s, Device dev,
                                     GridWait wait) {
  return launch_dynamic(x, (uint64_t)M * (uint64_t)K / 8, fp8_op(out), 448.0f, out.scale, sync,
                        clear, s, dev, wait);
}

cudaError_t launch_quant_nvfp4_after(const void* x, int64_t M, int64_t K, const float* scale_src,
                                     const qlin_nvfp4_t& out, cudaStream_t s, Device dev,
                                     unsigned* err, uint64_t timeout_ns) {
  const uint64_t n_chunks = (uint64_t)M * (uint64_t)K / 8;
  if (n_chunks >= (1ull << 32)) return launch_quant_nvfp4(x, M, K, scale_src, out, s, dev);
  const cudaError_t e = setup<quant_nvfp4_ring_kernel>(dev, kThreads, kSmem).err;
  if (e != cudaSuccess) return e;
  return launch_pdl(quant_nvfp4_ring_kernel, stream_grid(n_chunks, dev.num_sms), kThreads, kSmem, s,
                    static_cast<const uint4*>(x), n_chunks, scale_src, out.tensor_scale,
                    nvfp4_op<uint32_t>(K, out), err, timeout_ns);
}

cudaError_t launch_quant_nvfp4(const void* x, int64_t M, int64_t K, const float* scale_src,
                               const qlin_nvfp4_t& out, cudaStream_t s, Device dev) {
  const uint64_t n_chunks = (uint64_t)M * (uint64_t)K / 8;
  auto* xin = static_cast<const uint4*>(x);
  if (n_chunks <= kSmallPerSm * (uint64_t)dev.num_sms)
    return launch_pdl(quant_nvfp4_small_kernel,
                      (int)((n_chunks / 2 + kSmallThreads - 1) / kSmallThreads), kSmallThreads, 0,
                      s, xin, (uint32_t)n_chunks, scale_src, out.tensor_scale,
                      nvfp4_op<uint32_t>(K, out));
  const uint64_t tiles = (n_chunks + kDirectTile - 1) / kDirectTile;
  const int grid = (int)std::min<uint64_t>(tiles, (uint64_t)dev.num_sms * kDirectPerSm);
  auto* codes = reinterpret_cast<uint32_t*>(out.codes);
  const uint3 row_div = invariant_divisor((uint32_t)(K >> 3));
  auto kern = n_chunks < (1ull << 32) ? quant_nvfp4_kernel<uint32_t>   // 32-bit index math is enough
                                      : quant_nvfp4_kernel<uint64_t>;
  return launch_pdl(kern, grid, kThreads, 0, s, xin, n_chunks, K, scale_src, out.tensor_scale,
                    codes, out.scales, row_div);
}

cudaError_t launch_quant_fp8(const void* x, int64_t M, int64_t K, const float* scale_src,
                             const qlin_fp8_t& out, cudaStream_t s, Device dev, unsigned* err,
                             uint64_t timeout_ns) {
  const uint64_t n_chunks = (uint64_t)M * (uint64_t)K / 8;
  const cudaError_t e = setup<quant_fp8_kernel>(dev, kThreads, kSmem).err;
  if (e != cudaSuccess) return e;
  return launch_pdl(quant_fp8_kernel, stream_grid(n_chunks, dev.num_sms), kThreads, kSmem, s,
                    static_cast<const uint4*>(x), n_chunks, scale_src, out.scale, fp8_op(out), err,
                    timeout_ns);
}

cudaError_t launch_quant_fp8_rows(const void* w, int64_t N, int64_t K, const qlin_fp8_t& out,
                                  cudaStream_t s, Device dev) {
  const int64_t want = (N + kThreads / 32 - 1) / (kThreads / 32);
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)dev.num_sms * 8));
  auto kern = K <= 2 * 256   ? quant_fp8_rows_kernel<2, 4>   // a chunk per lane: 256 of K
              : K <= 4 * 256 ? quant_fp8_rows_kernel<4, 3>
                             : quant_fp8_rows_kernel<12, 2, true>;
  return launch_pdl(kern, grid, kThreads, 0, s, static_cast<const uint4*>(w), N, K, out.scale,
                    reinterpret_cast<uint2*>(out.codes));
}

cudaError_t take_grid_counts(unsigned (&counts)[3]) {
  static const unsigned zero[3] = {};
  cudaError_t e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = cudaMemcpyFromSymbol(counts, g_grid_counts, sizeof counts);
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_grid_counts, zero, sizeof zero);
  return e;
}

}  // namespace qlin
