// Fifth-generation tensor-core path (tcgen05, accumulators in tensor memory) for the two dense
// contractions of the library: the observation-window scores S_w of the static heads and the
// text-centric attention rows of the head classification.  Both are "queries x keys^T" with
// head_dim 128: a block of up to 256 query rows stays in shared memory, 128-key tiles stream through
// a ring of stages, every tile is one complete accumulation (K = 128 = 8 instructions of K = 16).
//
// Operands are bf16, K-major, in the 128-byte-swizzled canonical layout of the matrix descriptors:
// a row's 128 elements are split into two halves of 64 (128 bytes); each half-plane is
// [row][128 B] with the eight 16-byte pieces of a row XOR-permuted by (row & 7); planes are 1024-byte
// aligned.  Shared-memory descriptor: start address >> 4 in bits 0..13, leading byte offset (unused
// for swizzled K-major, set to 1) in bits 16..29, stride byte offset (1024 B between 8-row groups)
// >> 4 in bits 32..45, descriptor version 1 in bits 46..47, layout type 2 (128-byte swizzle) in
// bits 61..63.  Instruction descriptor (kind::f16): D format f32 (1) in bits 4..5, A and B format
// bf16 (1) in bits 7..9 and 10..12, both K-major (bits 15, 16 clear), N >> 3 in bits 17..22, M >> 4
// in bits 24..28.  An M = 128 accumulator puts row i in tensor-memory lane i and column j in column
// base + j; warp w of the CTA may read lanes 32 * (w % 4) .. + 31.
#pragma once
#include <cuda.h>

#include "hkv_device.cuh"

namespace hkv {
namespace tc {

constexpr int kKeysPerTile = 128;                   // keys of one streamed tile
constexpr int kQRows = 256;                         // query rows resident per CTA (two M = 128 blocks)
constexpr int kPlaneBytesK = kKeysPerTile * 128;    // one 64-element half of a key tile
constexpr int kPlaneBytesQ = kQRows * 128;
constexpr int kStageBytes = 2 * kPlaneBytesK;       // 32 KB
constexpr int kQBytes = 2 * kPlaneBytesQ;           // 64 KB
constexpr int kStages = 3;
constexpr int kTmemCols = 512;                      // two accumulator buffers of 256 columns
constexpr int kDrainWarps = 16;                     // four per lane quarter, 64 accumulator columns each
constexpr int kBarBytes = 256;
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(cols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t addr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols) : "memory");
}
__device__ __forceinline__ void fence_before_sync() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after_sync() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// D[tmem] (+)= A[smem] * B[smem]^T, one thread issues
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "setp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
      "}\n" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// the barrier gets one arrival once every tensor-core instruction issued so far by this thread is done
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  return static_cast<uint64_t>((addr >> 4) & 0x3FFFu) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
template <int M, int N>
struct InstrDesc {
  static constexpr uint32_t value = (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(N >> 3) << 17) |
                                    (static_cast<uint32_t>(M >> 4) << 24);
};

// One 16-byte piece of row `row` (piece 0..15 of its 256 bytes) inside a two-plane operand block.
__device__ __forceinline__ uint32_t piece_offset(int row, int piece, int plane_bytes) {
  return static_cast<uint32_t>((piece >> 3) * plane_bytes + row * 128 + (((piece & 7) ^ (row & 7)) << 4));
}

// ---- packed pairs of floats (one instruction for two elements) ----
__device__ __forceinline__ uint64_t pack_f32x2(float lo, float hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ void unpack_f32x2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// sum += x with the rounding error carried in comp (compensated summation; no fast-math in this library)
__device__ __forceinline__ void add_compensated(float& sum, float& comp, float x) {
  const float y = x - comp, t = sum + y;
  comp = (t - sum) - y;
  sum = t;
}

// ---------------------------------------------------------------------------------------------
// The segment engine.  A CTA walks a list of SEGMENTS -- a block of up to kQRows query rows against a run of key tiles
// of the same head -- so that work can be cut into equal shares of the whole launch's tiles whatever the heads'
// lengths, with one tensor-memory allocation and one pipeline per CTA: the key tiles of the next segment are already
// arriving while the last ones of the current are drained, and only the 64 KB of query rows are exchanged between two
// segments (by the draining warps, behind a named barrier they share with the issuer).
// The last warp brings in key tiles (TMA, two boxes of 64 elements x 128 keys in the operands' swizzled layout), warp 0
// feeds the tensor core; sixteen warps drain.  (With one warp for both, a tile's instructions held it for 1250 cycles and
// the next tile's copies for 500 more.)  Without any drain a tile takes 1610 cycles as one product of N = 256 and 1830 as two of
// N = 128, without the copies as well 1300 and 1670.
// Hand-overs.  What one role passes on to another travels over an mbarrier: a landed tile (full), a tile's completed
// instructions (acc_full for the draining warps, stage_free for the copies), a drained accumulator (acc_free).  Every
// wait on one is bounded.  A role whose wait runs out, or that sees that another's has, signals nothing more and waits for
// none of these any more, so that nobody is told of something that did not happen.  Named barriers are only used where
// every participant both arrives and waits, and are met the same number of times by all of them whether they have given up
// or not: by the draining warps among themselves (the caller's) and once per segment by them and warp 0.  So every role
// gets to the end, where each waits (bounded) for the copies or instructions it has started before the CTA may leave.
//   map               tensor map over all keys as rows of 128 bf16, boxes of 64 x 128 (key_map below)
//   segment(s, seg)   the CTA's s-th segment; false behind the last.  Seg has n_rows (query rows that exist: at most 128
//                     need only half of the instructions), tile_begin, tile_end and key_row0, the row
//                     of tile 0's first key in the map.  Rows behind the head's last key hold whatever the tensor holds
//                     there (zero behind its end): the caller masks them
//   q_row(seg, row)   pointer to a query row's 128 bf16, or nullptr for a zero row
//   begin(seg, lane_row, part), tile(seg, tile, lane_row, part, taddr), end(seg, lane_row, part, ok): called by the
//                     512 draining threads; a thread owns accumulator lane lane_row (0..127), columns
//                     64 part .. 64 part + 63 (part 0..3), at tensor-memory address taddr (drain_raw); ok: no wait has
//                     run out so far
// kKeysAsRows: false: accumulator rows = query rows (two M = 128 blocks side by side, block t in columns 128 t ..
// 128 t + 127 = the tile's keys); true: accumulator rows = the tile's keys, columns = the 256 query rows.
// kRing: key tiles of shared memory.  *user: shared memory behind the barriers' page, the caller's.  kSegThreads threads.
// ---------------------------------------------------------------------------------------------
constexpr int kSegThreads = (2 + kDrainWarps) * 32;
// named barriers; kBarDrain, kBarUser and above are the caller's
constexpr int kBarDrainIssue = 1, kBarDrain = 2, kBarUser = 3;
__device__ __forceinline__ void named_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// mbar_try_wait that may sleep for up to `ns` before it answers no: a warp that asks again and again takes issue slots from
// the draining warps of its scheduler
__device__ __forceinline__ bool mbar_try_wait_ns(uint64_t* bar, uint32_t parity, uint32_t ns) {
  uint32_t ok;
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
      "selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(ns)
      : "memory");
  return ok != 0;
}
constexpr uint32_t kWaitNs = 20000;
constexpr int seg_smem_fixed(int stages) { return kQBytes + stages * kStageBytes + kBarBytes + 1024; }   // + the caller's bytes

// 32 lanes x 16 columns, waited for: the four warps of a scheduler hide each other's latency, and the values need no copy
// between the read and its wait.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
// A draining thread's 64 columns as four groups of 16: fn(group, r) with columns 16 group ..
template <int kUnroll = 4, class Fn>
__device__ __forceinline__ void drain_raw(uint32_t taddr, Fn fn) {
#pragma unroll kUnroll
  for (int g = 0; g < 4; ++g) {
    uint32_t r[16];
    tmem_ld16(taddr + 16u * g, r);
    fn(g, r);
  }
}

// Loads the box at (x, y) of a two-dimensional tensor map into shared memory; bytes are credited to `bar`.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

template <bool kKeysAsRows, int kRing, class Seg, class SegmentFn, class QRowFn, class BeginFn, class TileFn, class EndFn>
__device__ bool segments_cta(uint8_t* smem_raw, const CUtensorMap* map, SegmentFn segment, QRowFn q_row, BeginFn begin,
                             TileFn tile_fn, EndFn end, uint8_t** user) {
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);   // operand planes are 1024-byte aligned
  uint8_t* qs = smem;
  uint8_t* ks = smem + kQBytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(ks + kRing * kStageBytes);
  uint64_t* stage_free = full + kRing;
  uint64_t* acc_full = stage_free + kRing;
  uint64_t* acc_free = acc_full + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_free + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  *user = ks + kRing * kStageBytes + kBarBytes;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  static_assert((2 * kRing + 4) * 8 + 8 <= kBarBytes, "the barriers' page");

  if (tid == 0) {
    for (int s = 0; s < kRing; ++s) {
      mbar_init(full + s, 1);
      mbar_init(stage_free + s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(acc_full + b, 1);
      mbar_init(acc_free + b, kDrainWarps);
    }
    mbar_fence_init();
    *abort_flag = 0;
  }
  if (warp == 0) {
    tmem_alloc(tmem_slot, kTmemCols);
    tmem_relinquish();
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  bool ok = true;   // no wait of this warp has run out, and it has not seen that another's has; the same in all its lanes
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    if (!ok || __all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return;
    const long long start = clock64();
    for (uint32_t it = 1; !__all_sync(0xffffffffu, mbar_try_wait_ns(bar, parity, kWaitNs)); ++it) {
      if ((it & 15u) == 0u && __any_sync(0xffffffffu, *abort_flag || clock64() - start > HKV_WAIT_CYCLES)) {
        *abort_flag = 1;
        ok = false;
        return;
      }
    }
  };
  // what this warp has started itself, waited for whatever has become of the rest
  auto settle = [&](uint64_t* bar, uint32_t parity) {
    const long long start = clock64();
    while (!__all_sync(0xffffffffu, mbar_try_wait_ns(bar, parity, kWaitNs))) {
      if (__any_sync(0xffffffffu, clock64() - start > HKV_WAIT_CYCLES)) {
        ok = false;
        return;
      }
    }
  };

  if (warp == 0) {
    constexpr uint32_t idesc = kKeysAsRows ? InstrDesc<128, 256>::value : InstrDesc<128, 128>::value;
    const uint32_t q_addr = smem_u32(qs), k_addr0 = smem_u32(ks);
    Seg seg;
    int i = 0;
    for (int sg = 0; segment(sg, seg); ++sg) {
      named_sync(kBarDrainIssue, (kDrainWarps + 1) * 32);   // the segment's query rows are in place
      const bool both = seg.n_rows > 128;
      fence_after_sync();
      for (int tile = seg.tile_begin; ok && tile < seg.tile_end; ++tile) {
        const int s = i % kRing, buf = i & 1;
        if (i >= 2) wait(acc_free + buf, ((i >> 1) - 1) & 1);   // tile i - 2 has been drained
        wait(full + s, (i / kRing) & 1);
        if (!ok) break;
        fence_after_sync();
        if (lane == 0) {
          const uint32_t k_addr = k_addr0 + static_cast<uint32_t>(s * kStageBytes);
          const uint32_t d = tmem_base + static_cast<uint32_t>(buf * 256);
#pragma unroll
          for (int kk = 0; kk < 8; ++kk) {   // K = 16 elements = 32 bytes per instruction; 4 per half-plane
            const uint32_t koff = static_cast<uint32_t>((kk >> 2) * kPlaneBytesK + (kk & 3) * 32);
            const uint32_t qoff = static_cast<uint32_t>((kk >> 2) * kPlaneBytesQ + (kk & 3) * 32);
            if (kKeysAsRows) {
              umma_bf16(d, smem_desc(k_addr + koff), smem_desc(q_addr + qoff), idesc, kk != 0);
            } else {
              umma_bf16(d, smem_desc(q_addr + qoff), smem_desc(k_addr + koff), idesc, kk != 0);
              if (both) umma_bf16(d + 128u, smem_desc(q_addr + qoff + 128u * 128u), smem_desc(k_addr + koff), idesc, kk != 0);
            }
          }
          umma_commit(stage_free + s);   // the stage may be refilled
          umma_commit(acc_full + buf);   // the accumulator is complete
        }
        __syncwarp();
        ++i;
      }
    }
    for (int t = max(0, i - 2); t < i; ++t) settle(acc_full + (t & 1), (t >> 1) & 1);
  } else if (warp == kDrainWarps + 1) {
    // ---- loads, kRing tiles ahead of the tensor core ----
    Seg seg;
    int n = 0;
    for (int sg = 0; ok && segment(sg, seg); ++sg) {
      for (int tile = seg.tile_begin; ok && tile < seg.tile_end; ++tile) {
        const int s = n % kRing;
        if (n >= kRing) wait(stage_free + s, (n / kRing - 1) & 1);   // the instructions of tile n - kRing have completed
        if (!ok) break;
        if (lane == 0) {
          const uint32_t dst = smem_u32(ks) + static_cast<uint32_t>(s * kStageBytes);
          mbar_arrive_expect_tx(full + s, kStageBytes);
          tma_load_2d(dst, map, 0, seg.key_row0 + tile * kKeysPerTile, full + s);
          tma_load_2d(dst + kPlaneBytesK, map, 64, seg.key_row0 + tile * kKeysPerTile, full + s);
        }
        __syncwarp();
        ++n;
      }
    }
    for (int t = max(0, n - kRing); t < n; ++t) settle(full + t % kRing, (t / kRing) & 1);
  } else {
    // ---- drain: warp w owns lane quarter w % 4 (the hardware's rule) and column part (w - 1) / 4 ----
    const int quarter = warp & 3, part = (warp - 1) >> 2;
    const int row = quarter * 32 + lane;
    const int dtid = tid - 32;
    int i = 0;
    Seg seg;
    for (int sg = 0; segment(sg, seg); ++sg) {
      // the query block, all of a thread's loads in flight; every instruction that read the previous block has
      // completed, because this thread has seen the segment's last accumulator
      {
        constexpr int kPieces = kQRows * 16 / (kDrainWarps * 32);
        uint4 v[kPieces];
#pragma unroll
        for (int u = 0; u < kPieces; ++u) {
          const int idx = dtid + u * kDrainWarps * 32;
          const __nv_bfloat16* src = q_row(seg, idx >> 4);
          v[u] = src ? __ldg(reinterpret_cast<const uint4*>(src) + (idx & 15)) : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int u = 0; u < kPieces; ++u) {
          const int idx = dtid + u * kDrainWarps * 32;
          *reinterpret_cast<uint4*>(qs + piece_offset(idx >> 4, idx & 15, kPlaneBytesQ)) = v[u];
        }
      }
      fence_proxy_async();   // written by ordinary stores, read by the tensor core
      fence_before_sync();
      named_sync(kBarDrainIssue, (kDrainWarps + 1) * 32);
      begin(seg, row, part);
      for (int tile = seg.tile_begin; tile < seg.tile_end; ++tile, ++i) {
        const int buf = i & 1;
        wait(acc_full + buf, (i >> 1) & 1);
        fence_after_sync();
        const uint32_t taddr =
            tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + static_cast<uint32_t>(buf * 256 + part * 64);
        tile_fn(seg, tile, row, part, taddr);
        fence_before_sync();
        __syncwarp();
        if (ok && lane == 0) mbar_arrive(acc_free + buf);
      }
      end(seg, row, part, ok);
    }
  }
  const bool all_ok = !__syncthreads_or(!ok);
  fence_after_sync();
  if (warp == 0) tmem_dealloc(tmem_base, kTmemCols);
  return all_ok;
}

// Host: the tensor map segments_cta takes, over `rows` keys of 128 bf16 from `keys` on.
inline cudaError_t key_map(CUtensorMap* map, const void* keys, uint64_t rows) {
  using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                              const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                              CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static Encode encode = [] {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult found;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found) != cudaSuccess ||
        found != cudaDriverEntryPointSuccess)
      fn = nullptr;
    return reinterpret_cast<Encode>(fn);
  }();
  if (!encode) return cudaErrorNotSupported;
  const cuuint64_t dims[2] = {128, rows}, strides[1] = {256};
  const cuuint32_t box[2] = {64, kKeysPerTile}, step[2] = {1, 1};
  const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(keys), dims, strides, box, step,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace tc
}  // namespace hkv
