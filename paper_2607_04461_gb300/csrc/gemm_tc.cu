// tcgen05 / TMEM GEMM for sm_103a: out[M][N] = epilogue(A[M][K] * W[N][K]^T).
//
// The dense projections of the DiT block (Eq. 7's B_l: QKV, attention output, cross
// query, cross output, FFN up and down) and the text projection run here.
//
// Design (one CTA per SM, persistent over output tiles of 128 x BN):
//  * warp 0, one thread: TMA producer. Loads 128x64 tiles of A and BNx64 tiles of W
//    (bf16, 128-byte swizzle) into a ring of STAGES shared-memory stages; each stage
//    has a "full" mbarrier (TMA transaction bytes) and an "empty" one (MMA done).
//  * warp 1: allocates 2*BN TMEM columns (two fp32 accumulators of 128 lanes x BN);
//    one thread issues tcgen05.mma (M=128, N=BN, K=16, bf16 -> fp32), commits each
//    stage back to its "empty" barrier and each finished tile to "tmem_full".
//  * warps 2-9: epilogue. Warp w reads TMEM lanes 32*(w%4).. (its lane quarter) and one
//    half of the tile's columns ((w-2)/4) with tcgen05.ld, applies bias / GELU / gated
//    residual / contribution write, stores to global, and releases the accumulator
//    ("tmem_empty") so that the MMA of the tile after next can start while this
//    epilogue runs. Two warps per lane quarter keep twice the epilogue's loads in
//    flight, which the fp32 residual epilogues need to keep up with the mainloop.
// Every mbarrier wait is bounded (mbar_wait): on timeout the kernel records the error,
// stops issuing work, waits (bounded) for its own TMA loads, frees TMEM and returns.
#include <cudaTypedefs.h>

#include <atomic>
#include <string.h>

#include "kernels.h"

namespace {

constexpr int BM = 128;
constexpr int BK = 64;  // 64 bf16 = 128 bytes: one swizzle row
constexpr int NUM_THREADS = 320;       // producer, MMA, 8 epilogue warps
constexpr int EPI_THREADS = 256;

template <int BN>
struct TcCfg {
  static constexpr int STAGES = (BN == 256) ? 4 : 6;
  static constexpr int A_BYTES = BM * BK * 2;
  static constexpr int B_BYTES = BN * BK * 2;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int TMEM_COLS = 2 * BN;  // 256 or 512 (power of two >= 32)
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 /*align*/ + 256 /*barriers*/;
};

// Instruction descriptor, kind::f16: D fp32, A and B bf16, both K-major, M=128, N=BN.
template <int BN>
__device__ __forceinline__ uint32_t idesc_bf16() {
  return (1u << 4)                     // D format: f32
         | (1u << 7)                   // A format: bf16
         | (1u << 10)                  // B format: bf16
         | ((uint32_t)(BN >> 3) << 17) // N >> 3
         | ((uint32_t)(BM >> 4) << 24);// M >> 4
}

template <int BN, int KIND>
__global__ void __launch_bounds__(NUM_THREADS, 1)
    gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW,
                   int M, int N, int K, GemmEpi epi, int* err) {
  using C = TcCfg<BN>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::STAGES * C::STAGE_BYTES);
  uint64_t* empty = full + C::STAGES;
  uint64_t* tmem_full = empty + C::STAGES;
  uint64_t* tmem_empty = tmem_full + 2;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(tmem_empty + 2);

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int n_mt = (M + BM - 1) / BM, n_nt = N / BN, n_tiles = n_mt * n_nt;
  const int nk = K / BK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&tmem_full[a], 1);
      mbar_init(&tmem_empty[a], EPI_THREADS);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmW);
  }
  if (warp == 1) tmem_alloc(tmem_holder, C::TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_holder;
  // The weights do not depend on the previous kernel: the producer starts loading the W
  // tiles of its first tile's first stages before waiting for its predecessor.
  const int pre = (int)blockIdx.x < n_tiles ? (nk < C::STAGES ? nk : C::STAGES) : 0;
  if (warp == 0 && elect_one())
    for (int kb = 0; kb < pre; ++kb) {
      uint8_t* sa = smem + kb * C::STAGE_BYTES;
      mbar_expect_tx(&full[kb], C::STAGE_BYTES);
      tma_load_2d(sa + C::A_BYTES, &tmW, &full[kb], kb * BK, ((int)blockIdx.x % n_nt) * BN);
    }
  griddep_wait();  // inputs written by the previous kernel are visible from here on
  griddep_launch();

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    int issued = 0;  // loads' K blocks so far
    for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
      const int m0 = (tile / n_nt) * BM, n0 = (tile % n_nt) * BN;
      for (int kb = 0; kb < nk; ++kb) {
        uint8_t* sa = smem + stage * C::STAGE_BYTES;
        const bool have_w = tile == (int)blockIdx.x && kb < pre;  // W already requested
        if (!have_w && !mbar_wait_warp(&empty[stage], phase ^ 1u, err)) { ok = false; break; }
        if (elect_one()) {
          if (!have_w) {
            mbar_expect_tx(&full[stage], C::STAGE_BYTES);
            tma_load_2d(sa + C::A_BYTES, &tmW, &full[stage], kb * BK, n0);
          }
          tma_load_2d(sa, &tmA, &full[stage], kb * BK, m0);
        }
        ++issued;
        if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
      }
    }
    if (!ok && lane == 0) {
      // Let this CTA's loads in flight land before the CTA exits: the last use of every
      // stage so far (stage s's u-th use completes phase u - 1 of its barrier).
      for (int s = 0; s < C::STAGES && s < issued; ++s) {
        const int uses = (issued - s + C::STAGES - 1) / C::STAGES;
        const uint32_t a = smem_u32(&full[s]);
        const uint64_t t0 = fb_globaltimer();
        while (!mbar_try(a, (uses - 1) & 1u) && fb_globaltimer() - t0 < fb_wait_limit()) {
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    const uint32_t idesc = idesc_bf16<BN>();
    const uint32_t ring_lo = desc_lo_k(smem_u32(smem));
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    int it = 0;
    for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x, ++it) {
      const int acc = it & 1;
      const uint32_t acc_phase = (it >> 1) & 1;
      if (!mbar_wait_warp(&tmem_empty[acc], acc_phase ^ 1u, err)) break;
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + acc * BN;
      for (int kb = 0; kb < nk; ++kb) {
        if (!mbar_wait_warp(&full[stage], phase, err)) { ok = false; break; }
        tc_fence_after();
        const uint32_t alo = ring_lo + (uint32_t)stage * (C::STAGE_BYTES >> 4);
        const uint32_t blo = alo + (C::A_BYTES >> 4);
        if (elect_one()) {
          // +32 bytes per K=16 step inside the swizzle row (encoded >> 4 -> +2)
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)
            tc_mma_ss_lo(d_tmem, alo + 2 * k, blo + 2 * k, DESC_HI, idesc, (kb | k) ? 1u : 0u);
          tc_commit(&empty[stage]);
          if (kb + 1 == nk) tc_commit(&tmem_full[acc]);
        }
        if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
      }
    }
  } else {
    // ---------------- epilogue (warps 2..9) ----------------
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    int it = 0;
    for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ++it) {
      const int acc = it & 1;
      const uint32_t acc_phase = (it >> 1) & 1;
      const int m0 = (tile / n_nt) * BM, n0 = (tile % n_nt) * BN;
      // short-K tiles only: over a long mainloop the streamed operands evict the rows
      if (nk <= 48 && m0 + quarter * 32 + lane < M)
        epi_prefetch<KIND>(epi, m0 + quarter * 32 + lane, n0 + half * (BN / 2), BN / 2);
      // every lane waits; the warp leaves together if any lane gave up, so the
      // .sync.aligned tcgen05.ld below is always executed by the whole warp
      const bool ok = mbar_wait(&tmem_full[acc], acc_phase, err);
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after();
      const int row = m0 + quarter * 32 + lane;
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * BN;
#pragma unroll 1
      for (int c = half * (BN / 64); c < (half + 1) * (BN / 64); ++c) {
        uint32_t r[32];
        tmem_ld32(taddr + c * 32, r);
        tmem_ld_wait();
        reg_fence32(r);
        if (row < M) {
          float v[32];
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
          epi_apply32<KIND>(epi, row, n0 + c * 32, v);
        }
      }
      tc_fence_before();
      mbar_arrive(&tmem_empty[acc]);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, C::TMEM_COLS);
  }
}

// ---- 2-SM variant -------------------------------------------------------------------
// A cluster of two CTAs computes a tile of 256 output features x T tokens (rows of A) with
// tcgen05.mma.cta_group::2: the features are the MMA's M dimension (256, CTA r of the pair
// holds features 128 r .. 128 r + 127 of the W tile and receives their accumulators in its
// TMEM, one feature per lane, one token per column), the tokens its N dimension (any
// multiple of 16 up to 256; CTA r holds T / 2 of the A rows). The even CTA issues the MMAs;
// its "full" barriers count the TMA bytes of both CTAs (the odd CTA's loads complete on
// them across the pair), its commits arrive on the "empty" / "tmem_full" barriers of both
// CTAs, and both CTAs' epilogue warps release an accumulator on its "tmem_empty" barrier.
//
// T is a launch parameter (see choose_tile): with the tokens along N the split follows the
// row count in steps of 16, so that few rows (one candidate's 1560) neither leave SM pairs
// idle nor compute padding. Stages and barriers are laid out for T at run time.
constexpr int C2_BN = 256;                           // output features of a tile
constexpr int C2_W_BYTES = 128 * BK * 2;             // 16 KB: this CTA's 128 W rows x 64 bf16
constexpr int C2_TMEM_COLS = 512;                    // two accumulators of up to 256 tokens
constexpr int C2_MAX_STAGES = 8;
constexpr int C2_MAX_ACCS = 8;
// TMEM columns from one accumulator to the next, and accumulators of the ring
__host__ __device__ __forceinline__ int c2_acc_cols(int T) { return (T + 31) / 32 * 32; }
__host__ __device__ __forceinline__ int c2_accs(int T) {
  const int n = C2_TMEM_COLS / c2_acc_cols(T);
  return n < C2_MAX_ACCS ? n : C2_MAX_ACCS;
}
// Shared memory of a CTA: 2.5 KB less than an SM can give it, which lets two blocks of the
// normalisation kernels that follow most GEMMs start beside it and wait there (1 KB each is
// reserved by the system): one candidate's block 224.5 -> 221.9 us.
constexpr int C2_SMEM_BYTES = 229888;
// Epilogue tiles and operand ring per epilogue: each of the 8 epilogue warps owns NBUF tiles
// of CHUNK tokens x 32 features, through which results leave by TMA store and (fp32 residual)
// residual rows arrive by TMA load. A chunk costs its warp about 300 clocks of buffer wait,
// proxy fence and store issue, so the bf16 epilogues take 32 tokens at a time; the fp32 ones
// take 16, which leaves the operand ring its stages.
template <int KIND>
struct C2Cfg {
  static constexpr bool F32 = KIND == EPI_RESID || KIND == EPI_RESID_DELTA;
  static constexpr int CHUNK = F32 ? 16 : 32;
  static constexpr int NBUF = F32 ? 3 : 2;
  static constexpr int TILE_BYTES = CHUNK * 32 * (F32 ? 4 : 2);
  static constexpr int EPI_BYTES = 8 * NBUF * TILE_BYTES;
  static constexpr int RING_BYTES = C2_SMEM_BYTES - 512 /*barriers*/ - EPI_BYTES;
};
__host__ __device__ __forceinline__ int c2_stages(int T, int ring_bytes) {
  const int n = ring_bytes / (C2_W_BYTES + T / 2 * BK * 2);
  return n < C2_MAX_STAGES ? n : C2_MAX_STAGES;
}
// Warps: 0 and 10 load (even and odd K blocks: one warp needs about 370 clocks from a free
// stage to its two TMA loads, more than the MMAs of a narrow tile's K block take, 288 at
// T = 144), 1 issues the MMAs, 2-9 run the epilogue.
constexpr int C2_THREADS = 352;

// ---- work split of the 2-SM kernel --------------------------------------------------
// Data-parallel: cluster c computes whole tiles c, c + G, c + 2G, ... (G clusters).
// Stream-K: the U = tiles x nk (tile, K-block) units, tile-major, are cut into G
// contiguous ranges of floor(c U / G) .. floor((c + 1) U / G); a cluster walks its range
// as segments (one tile, K-blocks kb0..kb1). With U >= G every range is non-empty, so the
// parts of a cut tile are held by consecutive clusters, the first as the last segment of its
// range and the others as the first of theirs. Partials go through the workspace in fp32, are
// counted on the tile's counter per epilogue warp, and are added in K order, so the sum does
// not depend on arrival order. The cut tiles are finished in one of two ways:
// * Ranges no longer than a tile (U <= G nk, at most two segments): every contributor
//   finishes a share of the tile's tokens in proportion to its K blocks, so that all clusters
//   finish about the same amount after equal ranges. It publishes the tokens of the others'
//   shares, waits (bounded) for the tile's count, and adds the others' partials of its own
//   share to its accumulators, which stay in TMEM. One finisher per tile instead was the last
//   to leave by far: 256 x 1536 x 8960 (13 contributors a tile) 18.6 us, 60.8 with one.
//   If a contributor does not turn up, the others make room for it (sk_wait_all).
// * Longer ranges: the first contributor finishes the tile alone as the others, which reach
//   it at the start of their ranges, have published long before. (Sharing it too would put
//   two more trips through the workspace at the end: 1040 x 5120 x 5120 50.3 us, 59.6.)
struct Seg {
  int tile, kb0, kb1;
};
struct WorkIter {
  long long u, u0, u1;
  int tile, n_tiles, nk, G;
  bool sk;
  __device__ WorkIter(bool sk_, int c, int G_, int n_tiles_, int nk_)
      : tile(c), n_tiles(n_tiles_), nk(nk_), G(G_), sk(sk_) {
    const long long U = (long long)n_tiles_ * nk_;
    u = u0 = (long long)c * U / G_;
    u1 = (long long)(c + 1) * U / G_;
  }
  __device__ bool next(Seg& g) {
    if (!sk) {
      if (tile >= n_tiles) return false;
      g.tile = tile;
      g.kb0 = 0;
      g.kb1 = nk;
      tile += G;
      return true;
    }
    if (u >= u1) return false;
    g.tile = (int)(u / nk);
    g.kb0 = (int)(u % nk);
    const long long rest = u1 - u;
    g.kb1 = rest < nk - g.kb0 ? g.kb0 + (int)rest : nk;
    u += g.kb1 - g.kb0;
    return true;
  }
};
// the cluster whose stream-K range holds unit u
__device__ __forceinline__ int sk_owner(long long u, long long U, int G) {
  return (int)(((u + 1) * G - 1) / U);
}
// Workspace slot `slot` (2c: the first segment of cluster c's range, 2c + 1: the last; a range
// meets at most two cut tiles). Per slot and CTA of the pair, 8 epilogue warps x 4096 floats:
// the warp's chunks of CH tokens [chunk][j/4][lane 32][4].
__device__ __forceinline__ float* sk_part(float* ws, int slot, int rank, int we) {
  return ws + ((size_t)(slot * 2 + rank) * 8 + we) * 4096;
}
// A cut tile: its first contributor, the number of them, whether the first holds it as the
// last segment of a longer range, this cluster's accumulator of it
struct CutTile {
  int tile = -1, lo = 0, n = 0, last = 0, acc = 0;
};
// A cut tile's counter, one per CTA of the pair and epilogue warp, zero between launches:
//   bits 0-9    contributors whose shares for the others are published
//   bits 10-19  contributors that have seen all of them (the last one zeroes the counter)
//   bits 20-29  contributors that have handed their own share over (the last one finishes the
//               tile and zeroes the counter)
//   bit 30      SK_HANDOVER, set while some contributor is missing
constexpr int SK_SEEN = 1 << 10, SK_HANDED = 1 << 20, SK_COUNT = 0x3ff;
// counts `n` on a cut tile's counter after this warp's (syncwarp'ed) writes; the old value
__device__ __forceinline__ int sk_count(int* ctr, int n) {
  int old;
  asm volatile("atom.add.release.gpu.global.s32 %0, [%1], %2;"
               : "=r"(old) : "l"(ctr), "r"(n) : "memory");
  return old;
}
// the same, ordered before this warp's later reads of what others counted in too
__device__ __forceinline__ int sk_count_acquire(int* ctr, int n) {
  int old;
  asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], %2;"
               : "=r"(old) : "l"(ctr), "r"(n) : "memory");
  return old;
}
__device__ __forceinline__ int sk_load(const int* ctr) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
  return v;
}
// waits (bounded) until `n` contributors are in
__device__ __forceinline__ bool sk_wait(const int* ctr, int n, int* err) {
  const uint64_t t0 = fb_globaltimer();
  uint32_t i = 0;
  for (int c; (c = sk_load(ctr)) < 0 || (c & SK_COUNT) != n;) {
    if ((++i & 7u) != 0) continue;  // error word and clock now and then: short polls
    if (*(volatile int*)err != 0) return false;
    if (fb_globaltimer() - t0 > fb_wait_limit()) {
      fb_report(err, FB_DEVERR_WAIT_TIMEOUT);
      return false;
    }
  }
  return true;
}
// Waits (bounded) until all `n` contributors of a shared tile are in, SK_SHARE. They may never
// be while this grid waits: launches of other streams can hold the SMs that its missing clusters
// need, waiting in the same way. So a contributor that has waited a 20000th of the wait limit
// (100 us) for a missing one sets SK_HANDOVER: nobody waits any more, every contributor publishes
// its own share too and counts that, and the last one to do so finishes the tile.
enum { SK_GAVE_UP = 0, SK_SHARE, SK_HAND_OVER };
__device__ __forceinline__ int sk_wait_all(int* ctr, int n, int* err) {
  const uint64_t t0 = fb_globaltimer();
  for (uint32_t i = 1;; ++i) {
    const int c = sk_load(ctr);
    if (c >= 0) {
      if (c & SK_HANDOVER) return SK_HAND_OVER;
      if ((c & SK_COUNT) == n) return SK_SHARE;
    }
    if ((i & 7u) != 0) continue;
    if (*(volatile int*)err != 0) return SK_GAVE_UP;
    const uint64_t waited = fb_globaltimer() - t0;
    if (waited > fb_wait_limit()) {
      fb_report(err, FB_DEVERR_WAIT_TIMEOUT);
      return SK_GAVE_UP;
    }
    // (only while one is missing: the counter is still what was read)
    if (c >= 0 && waited * 20000 > fb_wait_limit()) atomicCAS(ctr, c, c | SK_HANDOVER);
  }
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void ld_shared_v4(uint32_t a, uint32_t* r) {
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
constexpr int SK_SLOTS = 8;  // 2 KB slots of an epilogue warp: 16 KB of the operand ring

// ---- epilogue of the 2-SM kernel ----------------------------------------------------
// A lane owns one output feature, so bias and gate are one register each, and a warp's
// access to one token of a shared-memory tile or of global memory is one row of 32
// consecutive features (128 bytes of fp32: no bank conflicts without a swizzle). A warp
// takes every other chunk of the tile's tokens. The residual chunks load two ahead, the
// first ones while the mainloop runs; the contribution epilogue (Delta) reads the base rows
// into registers one chunk ahead and stores the contribution directly.

// Two tokens' values (j, j + 1) of each lane's feature as one 4-byte store per lane: lanes
// exchange with their neighbour, even lanes then hold two adjacent features of token j,
// odd lanes of token j + 1 (64 contiguous bytes per token and warp).
__device__ __forceinline__ uint32_t pair_pack_bf16(float v0, float v1, int lane) {
  const float got = __shfl_xor_sync(0xffffffffu, (lane & 1) ? v0 : v1, 1);
  return (lane & 1) ? pack_bf16x2(got, v1) : pack_bf16x2(v0, got);
}

// CH (16 or 32) TMEM columns of this warp's lanes, waited for
template <int CH>
__device__ __forceinline__ void tmem_ld_chunk(uint32_t taddr, uint32_t* r) {
  if (CH == 32) {
    tmem_ld32(taddr, r);
    tmem_ld_wait();
    reg_fence32(r);
  } else {
    tmem_ld16(taddr, r);
    tmem_ld_wait();
    reg_fence16(r);
  }
}

template <int KIND>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(C2_THREADS, 1)
    gemm_tc2_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW,
                    const __grid_constant__ CUtensorMap tmO, const __grid_constant__ CUtensorMap tmR,
                    int M, int N, int K, int T, int parts, GemmEpi epi, SkArgs sk, int* err) {
  using CC = C2Cfg<KIND>;
  extern __shared__ __align__(1024) uint8_t smem[];  // (operand tiles need the alignment)
  if ((smem_u32(smem) & 1023u) != 0) {
    if (threadIdx.x == 0) fb_report(err, FB_DEVERR_BAD_ARG);
    return;
  }
  // (RING_BYTES and EPI_BYTES are multiples of 512: tiles and barriers stay aligned)
  uint8_t* epi_smem = smem + CC::RING_BYTES;
  uint64_t* full = reinterpret_cast<uint64_t*>(epi_smem + CC::EPI_BYTES);
  uint64_t* empty = full + C2_MAX_STAGES;
  uint64_t* tmem_full = empty + C2_MAX_STAGES;
  uint64_t* tmem_empty = tmem_full + C2_MAX_ACCS;
  uint64_t* rload = tmem_empty + C2_MAX_ACCS;  // residual tile loads: NBUF per epilogue warp
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(rload + 8 * 3);
  uint32_t* gave_up = tmem_holder + 1;  // a role of this CTA gave up a wait

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const uint32_t rank = cluster_ctarank();
  const int cluster = blockIdx.x >> 1, n_clusters = gridDim.x >> 1;
  const int n_mt = (M + T - 1) / T, n_nt = (N + C2_BN - 1) / C2_BN, n_tiles = n_mt * n_nt;
  const int nk = K / BK;
  const int stage_bytes = C2_W_BYTES + T / 2 * BK * 2;
  const int stages = c2_stages(T, CC::RING_BYTES);
  const int acc_cols = c2_acc_cols(T), n_accs = c2_accs(T);
  bool failed = false;

  if (threadIdx.x == 0) {
    *gave_up = 0;
    for (int s = 0; s < stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < n_accs; ++a) {
      mbar_init(&tmem_full[a], 1);
      mbar_init(&tmem_empty[a], 16);  // 8 epilogue warps x 2 CTAs
    }
    for (int b = 0; b < 8 * 3; ++b) mbar_init(&rload[b], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmW);
    tma_prefetch_desc(&tmO);
    if (CC::F32) tma_prefetch_desc(&tmR);
  }
  if (warp == 1) tmem_alloc_cg2(tmem_holder, C2_TMEM_COLS);
  tc_fence_before();
  cluster_sync();  // both CTAs' barriers initialised, TMEM allocated
  tc_fence_after();
  const uint32_t tmem_base = *tmem_holder;
  const bool use_sk = sk.on != 0;
  const long long U = (long long)n_tiles * nk;
  // As in the 1-SM kernel: W tiles of the first segment's first stages before the wait.
  int pre = 0;
  if (warp == 0 || warp == 10) {
    WorkIter w0(use_sk, cluster, n_clusters, n_tiles, nk);
    Seg first;
    if (w0.next(first)) {
      const int len = first.kb1 - first.kb0;
      pre = len < stages ? len : stages;
      const int n0 = (first.tile % n_nt) * C2_BN + 128 * (int)rank;
      if (warp == 0 && elect_one())
        for (int i = 0; i < pre; ++i) {
          if (rank == 0) mbar_expect_tx(&full[i], 2 * stage_bytes);
          tma_load_2d_cg2(smem + i * stage_bytes, &tmW, mapa_shared(smem_u32(&full[i]), 0),
                          (first.kb0 + i) * BK, n0);
        }
    }
  }
  griddep_wait();
  // Dependents may start once every CTA of this grid has passed here: with the stream-K
  // split all contributors are then resident, so a finisher's wait cannot be starved.
  griddep_launch();

  if (warp == 0 || warp == 10) {
    // ---------------- TMA producers (both CTAs) ----------------
    int stage = 0;
    uint32_t phase = 0;
    bool mine = warp == 0;  // K blocks alternate between the two warps
    WorkIter wi(use_sk, cluster, n_clusters, n_tiles, nk);
    Seg sg;
    for (int it = 0; !failed && wi.next(sg); ++it) {
      const int m0 = (sg.tile / n_nt) * T + T / 2 * (int)rank;
      const int n0 = (sg.tile % n_nt) * C2_BN + 128 * (int)rank;
      for (int kb = sg.kb0; kb < sg.kb1; ++kb, mine = !mine) {
        if (mine) {
          uint8_t* sw = smem + stage * stage_bytes;
          const uint32_t fb = mapa_shared(smem_u32(&full[stage]), 0);
          const bool have_w = it == 0 && kb - sg.kb0 < pre;  // requested before the wait
          if (!have_w && !mbar_wait_warp(&empty[stage], phase ^ 1u, err)) { failed = true; break; }
          if (elect_one()) {
            if (!have_w) {
              if (rank == 0) mbar_expect_tx(&full[stage], 2 * stage_bytes);
              tma_load_2d_cg2(sw, &tmW, fb, kb * BK, n0);
            }
            tma_load_2d_cg2(sw + C2_W_BYTES, &tmA, fb, kb * BK, m0);
          }
        }
        if (++stage == stages) { stage = 0; phase ^= 1u; }
      }
    }
  } else if (warp == 1) {
    if (rank == 0) {
      // ---------------- MMA issuer (even CTA) ----------------
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(T >> 3) << 17) |
                             ((uint32_t)(C2_BN >> 4) << 24);
      const uint32_t ring_lo = desc_lo_k(smem_u32(smem));
      int stage = 0;
      uint32_t phase = 0;
      WorkIter wi(use_sk, cluster, n_clusters, n_tiles, nk);
      Seg sg;
      const int part_len = (nk + parts - 1) / parts;
      int acc = 0;
      uint32_t acc_phase = 0;
      while (!failed && wi.next(sg)) {
        // the tile's K parts (one, with the stream-K split), each in the ring's next accumulator
        for (int kb = sg.kb0; !failed && kb < sg.kb1;) {
          if (!mbar_wait_warp(&tmem_empty[acc], acc_phase ^ 1u, err)) { failed = true; break; }
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + acc * acc_cols;
          const int first = kb, end = sg.kb1 - kb < part_len ? sg.kb1 : kb + part_len;
          for (; kb < end; ++kb) {
            if (!mbar_wait_warp(&full[stage], phase, err)) { failed = true; break; }
            tc_fence_after();
            const uint32_t wlo = ring_lo + (uint32_t)(stage * (stage_bytes >> 4));
            const uint32_t alo = wlo + (C2_W_BYTES >> 4);
            if (elect_one()) {
#pragma unroll
              for (int k = 0; k < BK / 16; ++k)
                tc_mma_cg2_lo(d_tmem, wlo + 2 * k, alo + 2 * k, DESC_HI, idesc,
                              (kb > first || k > 0) ? 1u : 0u);
              tc_commit_mc(&empty[stage], 0x3);
              if (kb + 1 == end) tc_commit_mc(&tmem_full[acc], 0x3);
            }
            if (++stage == stages) { stage = 0; phase ^= 1u; }
          }
          if (++acc == n_accs) { acc = 0; acc_phase ^= 1u; }
        }
      }
    }
  } else {
    // ---------------- epilogue (warps 2..9 of both CTAs) ----------------
    // warp: features quarter * 32 .. + 31 of this CTA's 128 (its TMEM lanes), every other
    // 16-token chunk of the tile
    const int quarter = warp & 3, half = (warp - 2) >> 2, we = warp - 2;
    const uint32_t te_remote = mapa_shared(smem_u32(&tmem_empty[0]), 0);
    constexpr int NBUF = CC::NBUF, CH = CC::CHUNK;
    const bool has_r = CC::F32 && epi.resid != nullptr;
    uint8_t* wtiles = epi_smem + we * NBUF * CC::TILE_BYTES;
    uint64_t* wload = rload + we * 3;
    uint32_t rl_phase = 0;  // bit b: parity of tile b's next load
    WorkIter wi(use_sk, cluster, n_clusters, n_tiles, nk);
    // the cut tiles of this cluster's range (at most two: newest, older): published when
    // their segment is done, this cluster's share of their chunks finished after the range
    CutTile cut0, cut1, ct;
    int fin = 0;
    // lanes 0 and 1 (cut0's, cut1's): how the tile is finished, whether this warp zeroes its
    // counter at the end
    int how = SK_SHARE;
    bool reset_ctr = false;
    // ranges of at most two segments: the accumulators stay in TMEM to the end, and a
    // cluster's own share is neither published nor read back
    const bool keep = U <= (long long)n_clusters * nk;
    auto counter = [&](const CutTile& c) { return sk.ctr + ((size_t)c.lo * 2 + rank) * 8 + we; };
    // chunks of a tile's accumulators into this cluster's slot of the workspace: its own share,
    // i0 .. i1 - 1, or all others
    auto publish_chunks = [&](const CutTile& c, uint32_t taddr, int nch, int i0, int i1, bool own) {
      const int part_slot = 2 * cluster + (c.lo == cluster && c.last);
      float4* part = reinterpret_cast<float4*>(sk_part(sk.ws, part_slot, (int)rank, we)) + lane;
#pragma unroll 1
      for (int i = 0; i < nch; ++i) {
        if ((i >= i0 && i < i1) != own) continue;
        uint32_t r[CH];
        tmem_ld_chunk<CH>(taddr + i * 2 * CH, r);
#pragma unroll
        for (int j4 = 0; j4 < CH / 4; ++j4)
          part[(i * (CH / 4) + j4) * 32] = make_float4(
              __uint_as_float(r[4 * j4]), __uint_as_float(r[4 * j4 + 1]),
              __uint_as_float(r[4 * j4 + 2]), __uint_as_float(r[4 * j4 + 3]));
      }
      __syncwarp();
    };
    int next_acc = 0;
    uint32_t next_phase = 0;
    while (true) {
      Seg sg;
      const bool seg = wi.next(sg);
      if (!seg) {
        ct = fin == 0 ? cut0 : cut1;
        if (fin++ > 1 || ct.tile < 0) break;
        sg.tile = ct.tile;
      }
      const int tile = sg.tile;
      // the accumulator of the tile's first K part; the others follow it in the ring
      const int acc = seg ? next_acc : ct.acc;
      const bool is_cut = seg && (sg.kb0 != 0 || sg.kb1 != nk);
      const bool publish = is_cut && (keep || sg.kb0 != 0);
      const bool from_parts = !seg || (is_cut && !publish);  // a cut tile is finished now
      const int m0 = (tile / n_nt) * T;
      const int f0 = (tile % n_nt) * C2_BN + 128 * (int)rank + quarter * 32;
      const int nv = M - m0 < T ? M - m0 : T;  // valid tokens of the tile
      // this warp's chunks: i = 0, 1, ... covers tokens (half + 2 i) * CH ..
      // (none if its features lie past N, a multiple of 128)
      const int ncht = (nv + CH - 1) / CH, nch = f0 < N ? (ncht + 1 - half) / 2 : 0;
      // the chunks that this step finishes: all of a whole tile's, a share of a cut one's
      int i0 = 0, i1 = nch, own = -1;
      if (is_cut || !seg) {
        if (seg) {
          ct.tile = tile;
          ct.lo = sk_owner((long long)tile * nk, U, n_clusters);
          ct.n = sk_owner((long long)(tile + 1) * nk - 1, U, n_clusters) - ct.lo + 1;
          ct.last = (long long)ct.lo * U / n_clusters < (long long)tile * nk;
          ct.acc = acc;
        }
        if (keep) {
          // in proportion to its K blocks: every cluster's shares add up to about the same
          const long long k0 = wi.u0 - (long long)tile * nk, k1 = wi.u1 - (long long)tile * nk;
          i0 = k0 <= 0 ? 0 : ((int)k0 * nch + nk / 2) / nk;
          i1 = k1 >= nk ? nch : ((int)k1 * nch + nk / 2) / nk;
          own = cluster - ct.lo;
        } else if (from_parts) {
          own = 0;
        } else {
          i1 = 0;
        }
      }
      const size_t off0 = (size_t)(m0 + half * CH) * epi.ldo + f0 + lane;
      const bool work = !publish && i0 < i1, any = !publish && nch > 0;
      const float bias = any && epi.bias ? __ldg(epi.bias + f0 + lane) : 0.f;
      const float gate = CC::F32 && any && epi.gate ? __ldg(epi.gate + f0 + lane) : 1.f;
      // residual chunk i into tile (i - i0) % NBUF (one lane)
      auto rload_issue = [&](int i) {
        const int t = (i - i0) % NBUF;
        mbar_expect_tx(&wload[t], CC::TILE_BYTES);
        tma_load_2d(wtiles + t * CC::TILE_BYTES, &tmR, &wload[t], f0, m0 + (half + 2 * i) * CH);
      };
      float bv[16];
      auto load_base = [&](int i) {  // Delta: base rows of chunk i
        const int left = nv - (half + 2 * i) * CH;  // tokens from this chunk to the tile's end
        const float* p = epi.base + off0 + (size_t)i * 2 * CH * epi.ldo;
#pragma unroll
        for (int j = 0; j < 16; ++j) bv[j] = j < left ? __ldcg(p + (size_t)j * epi.ldo) : 0.f;
      };
      auto first_loads = [&] {
        if (elect_one()) {
          bulk_wait_read<0>();  // the previous output tile's stores have left the tiles
          if (has_r) rload_issue(i0);
          if (has_r && i0 + 1 < i1) rload_issue(i0 + 1);
        }
        __syncwarp();
        if (KIND == EPI_RESID_DELTA) load_base(i0);
      };
      if (work) first_loads();
      const uint32_t taddr =
          tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * acc_cols + half * CH;
      if (seg) {
        // the last part's accumulator is complete after all others of the tile
        int last = acc + parts - 1;
        uint32_t last_phase = next_phase;
        if (last >= n_accs) { last -= n_accs; last_phase ^= 1u; }
        const bool ok = mbar_wait(&tmem_full[last], last_phase, err);
        if (!__all_sync(0xffffffffu, ok)) { failed = true; break; }
        tc_fence_after();
        if (publish) {
          publish_chunks(ct, taddr, nch, i0, i1, false);
          if (lane == 0) sk_count(counter(ct), 1);
          if (keep) {
            cut1 = cut0;
            cut0 = ct;
          }
        } else if (is_cut) {
          // the other contributors computed their parts at the start of their ranges
          bool in = true;
          if (lane == 0) {
            in = sk_wait(counter(ct), ct.n - 1, err);
            if (in) *(volatile int*)counter(ct) = 0;  // every contributor is in: ready for reuse
          }
          if (!__all_sync(0xffffffffu, in)) { failed = true; break; }
        }
      } else {
        bool ok = true;
        if (fin == 1) {
          // Wait (bounded) until every contributor's warp has counted in, for both cut tiles
          // at once (lanes 0 and 1). All publish before they wait, at the ends of ranges of
          // one length. With no other launch on its SMs every contributor is running: the grid
          // is at most the resident-cluster count, and a dependent grid starts only after all of
          // this grid's CTAs have started.
          const CutTile w = lane == 0 ? cut0 : cut1;
          if (lane < 2 && w.tile >= 0) {
            how = sk_wait_all(counter(w), w.n, err);
            ok = how != SK_GAVE_UP;
            // seen by this warp; whoever is the last to see it zeroes the counter (at the end)
            if (how == SK_SHARE)
              reset_ctr = ((sk_count(counter(w), SK_SEEN) >> 10) & SK_COUNT) == w.n - 1;
          }
          if (!__all_sync(0xffffffffu, ok)) { failed = true; break; }
        }
        if (__shfl_sync(0xffffffffu, how, fin - 1) == SK_HAND_OVER) {
          // the residual rows of this share have been asked for and are not used
          for (int t = 0; t < 2 && has_r && i0 + t < i1; ++t) {
            ok = mbar_wait(&wload[t], (rl_phase >> t) & 1u, err) && ok;
            rl_phase ^= 1u << t;
          }
          if (!__all_sync(0xffffffffu, ok)) { failed = true; break; }
          publish_chunks(ct, taddr, nch, i0, i1, true);
          int handed = 0;
          if (lane == 0) {
            handed = (sk_count_acquire(counter(ct), SK_HANDED) >> 20) & SK_COUNT;
            if (handed == ct.n - 1) *(volatile int*)counter(ct) = 0;  // nobody reads it any more
          }
          if (__shfl_sync(0xffffffffu, handed, 0) != ct.n - 1) continue;
          i0 = 0;  // the last one: everything is published
          i1 = nch;
          if (nch > 0) first_loads();
        }
      }
      if (!publish) {
        // TMEM columns from the tile's first accumulator to that of K part p
        auto acc_col = [&](int p) { return (acc + p < n_accs ? p : p - n_accs) * acc_cols; };
        // A cut tile's partials come through this warp's 16 KB of the operand ring, idle now
        // (every MMA that read it has completed and no load follows), in the order they are
        // summed and SK_SLOTS - 1 of 2 KB (16 tokens) in flight: lanes copy what they read.
        int pi = i0, ph = 0, pq = own == 0 ? 1 : 0, slot = 0;
        const uint32_t ring = smem_u32(smem) + we * (SK_SLOTS * 2048) + lane * 16;
        auto fetch = [&](int into) {
          if (pi < i1) {
            const int part_slot = 2 * (ct.lo + pq) + (pq == 0 && ct.last);
            const float* src = sk_part(sk.ws, part_slot, (int)rank, we) +
                               (pi * (CH * 8) + ph * 8 + lane) * 4;
#pragma unroll
            for (int j4 = 0; j4 < 4; ++j4) cp_async16(ring + into * 2048 + j4 * 512, src + j4 * 128);
            if (++pq == own) ++pq;
            if (pq >= ct.n) {
              pq = own == 0 ? 1 : 0;
              ph += 16;
              if (ph == CH) { ph = 0; ++pi; }
            }
          }
          cp_async_commit();
        };
        if (from_parts)
          for (int i = 0; i < SK_SLOTS - 1; ++i) fetch(i);
        // chunk i's sums: the accumulators, or a cut tile's parts in K order
        auto chunk_sums = [&](int i, float* v) {
          if (!from_parts) {
            if (parts == 1) {
              uint32_t r[CH];
              tmem_ld_chunk<CH>(taddr + i * 2 * CH, r);
#pragma unroll
              for (int j = 0; j < CH; ++j) v[j] = __uint_as_float(r[j]);
              return;
            }
#pragma unroll
            for (int h = 0; h < CH; h += 16) {
#pragma unroll 1
              for (int p = 0; p < parts; p += 2) {  // two parts' loads in flight
                uint32_t r[16], r2[16];
                const bool two = p + 1 < parts;
                tmem_ld16(taddr + acc_col(p) + i * 2 * CH + h, r);
                if (two) tmem_ld16(taddr + acc_col(p + 1) + i * 2 * CH + h, r2);
                tmem_ld_wait();
                reg_fence16(r);
                reg_fence16(r2);
#pragma unroll
                for (int j = 0; j < 16; ++j)
                  v[h + j] = p == 0 ? __uint_as_float(r[j]) : v[h + j] + __uint_as_float(r[j]);
                if (two) {
#pragma unroll
                  for (int j = 0; j < 16; ++j) v[h + j] += __uint_as_float(r2[j]);
                }
              }
            }
            return;
          }
#pragma unroll
          for (int h = 0; h < CH; h += 16) {
#pragma unroll 1
            for (int q = 0; q < ct.n; ++q) {
              uint32_t r[16];
              if (q == own) {
                tmem_ld_chunk<16>(taddr + i * 2 * CH + h, r);
              } else {
                cp_async_wait<SK_SLOTS - 2>();
#pragma unroll
                for (int j4 = 0; j4 < 4; ++j4)
                  ld_shared_v4(ring + slot * 2048 + j4 * 512, r + 4 * j4);
                // into the slot that was read one part ago
                fetch((slot + SK_SLOTS - 1) % SK_SLOTS);
                slot = (slot + 1) % SK_SLOTS;
              }
#pragma unroll
              for (int j = 0; j < 16; ++j)
                v[h + j] = q == 0 ? __uint_as_float(r[j]) : v[h + j] + __uint_as_float(r[j]);
            }
          }
        };
#pragma unroll 1
        for (int i = i0; i < i1; ++i) {
          float v[CH];
          chunk_sums(i, v);
          const int b = (i - i0) % NBUF;
          uint8_t* tile_b = wtiles + b * CC::TILE_BYTES;
          if (CC::F32) {
            float* tf = reinterpret_cast<float*>(tile_b) + lane;
            if (has_r) {
              const bool lok = mbar_wait(&wload[b], (rl_phase >> b) & 1u, err);
              rl_phase ^= 1u << b;
              if (!__all_sync(0xffffffffu, lok)) { failed = true; break; }
#pragma unroll
              for (int j = 0; j < CH; ++j) v[j] = tf[j * 32] + gate * (v[j] + bias);
              // its tile was stored from one chunk ago: free for chunk i + 2
              if (i + 2 < i1 && elect_one()) {
                bulk_wait_read<0>();
                rload_issue(i + 2);
              }
            } else {
              // no residual: the store from this tile three chunks ago has been read
              if (elect_one()) bulk_wait_read<2>();
              __syncwarp();
#pragma unroll
              for (int j = 0; j < CH; ++j) v[j] = gate * (v[j] + bias);
            }
#pragma unroll
            for (int j = 0; j < CH; ++j) tf[j * 32] = v[j];
          } else {
            // the store from this tile two chunks ago has left shared memory
            if (elect_one()) bulk_wait_read<1>();
            __syncwarp();
            uint32_t* tw = reinterpret_cast<uint32_t*>(tile_b) + (lane & 1) * 16 + (lane >> 1);
#pragma unroll
            for (int j = 0; j < CH; j += 2) {
              float y0 = v[j] + bias, y1 = v[j + 1] + bias;
              if (KIND == EPI_GELU_BF16) gelu_tanh_f2(y0, y1);
              tw[j * 16] = pair_pack_bf16(y0, y1, lane);
            }
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (elect_one()) {
            // boxes of 16 tokens; a second one past the tile's end belongs to the next tile
            const int t0 = (half + 2 * i) * CH;
            tma_store_2d(&tmO, smem_u32(tile_b), f0, m0 + t0);
            if (CH == 32 && t0 + 16 < nv)
              tma_store_2d(&tmO, smem_u32(tile_b) + CC::TILE_BYTES / 2, f0, m0 + t0 + 16);
            bulk_commit();
          }
          if (KIND == EPI_RESID_DELTA) {
            const int left = nv - (half + 2 * i) * CH;
            bf16* dl = epi.delta + off0 + (size_t)i * 2 * CH * epi.ldo - lane + (lane & ~1) +
                       (size_t)(lane & 1) * epi.ldo;
#pragma unroll
            for (int j = 0; j < CH; j += 2) {
              const uint32_t w = pair_pack_bf16(v[j] - bv[j], v[j + 1] - bv[j + 1], lane);
              if (j + (lane & 1) < left) *reinterpret_cast<uint32_t*>(dl + (size_t)j * epi.ldo) = w;
            }
            if (i + 1 < i1) load_base(i + 1);
          }
        }
        if (failed) break;
      }
      if (seg) {
        if (own < 0) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0)
            for (int p = 0; p < parts; ++p) {
              const int a = acc + p < n_accs ? acc + p : acc + p - n_accs;
              mbar_arrive_cluster(te_remote + a * (uint32_t)sizeof(uint64_t));
            }
        }
        next_acc += parts;
        if (next_acc >= n_accs) { next_acc -= n_accs; next_phase ^= 1u; }
      }
    }
    if (reset_ctr)  // the last to see this cut tile's count: ready for reuse
      *(volatile int*)counter(lane == 0 ? cut0 : cut1) = 0;
  }

  // own TMA stores complete (one lane issued them all)
  if (warp >= 2 && warp < 10 && elect_one()) bulk_wait<0>();
  if (failed) *gave_up = 1;
  tc_fence_before();
  cluster_sync();
  if (*gave_up != 0) {
    // After a timeout, give TMA loads that may still be in flight time to land before
    // the shared memory they target is released (they complete within microseconds). A CTA
    // with loads in flight has unfinished tiles, so its own epilogue gave up too.
    const uint64_t t0 = fb_globaltimer();
    while (fb_globaltimer() - t0 < 100000ull) __nanosleep(1000);
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_cg2(tmem_base, C2_TMEM_COLS);
  }
}

PFN_cuTensorMapEncodeTiled_v12000 get_encode() {
  // looked up once; a function-local static is initialised thread-safely (the bench
  // drives two models from two host threads)
  static const PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    cudaDriverEntryPointQueryResult q;
    void* p = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    cudaGetLastError();
    return static_cast<PFN_cuTensorMapEncodeTiled_v12000>(nullptr);
  }();
  return fn;
}

// 2-D bf16 tensor map over rows x cols (row stride ld elements), box box_rows x 64.
bool make_map(CUtensorMap* map, const bf16* ptr, int rows, int cols, int ld, int box_rows) {
  auto enc = get_encode();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * sizeof(bf16)};
  cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16*>(ptr), dims,
                   strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

template <int BN, int KIND>
cudaError_t launch(const GemmArgs& g, int* err, int num_sms, cudaStream_t st) {
  using C = TcCfg<BN>;
  CUtensorMap ma, mw;
  if (!make_map(&ma, g.A, g.M, g.K, g.lda, BM) || !make_map(&mw, g.W, g.N, g.K, g.ldw, BN))
    return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(gemm_tc_kernel<BN, KIND>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_BYTES);
  if (e != cudaSuccess) return e;
  const int tiles = ((g.M + BM - 1) / BM) * (g.N / BN);
  const int grid = tiles < num_sms ? tiles : num_sms;
  return launch_k(gemm_tc_kernel<BN, KIND>, dim3(grid), dim3(NUM_THREADS), C::SMEM_BYTES, st, ma,
                  mw, g.M, g.N, g.K, g.epi, err);
}

template <int BN>
cudaError_t dispatch_kind(const GemmArgs& g, int* err, int num_sms, cudaStream_t st) {
  switch (g.kind) {
    case EPI_BF16: return launch<BN, EPI_BF16>(g, err, num_sms, st);
    case EPI_GELU_BF16: return launch<BN, EPI_GELU_BF16>(g, err, num_sms, st);
    case EPI_RESID: return launch<BN, EPI_RESID>(g, err, num_sms, st);
    case EPI_RESID_DELTA: return launch<BN, EPI_RESID_DELTA>(g, err, num_sms, st);
  }
  return cudaErrorInvalidValue;
}

// 2-D map over an epilogue matrix [rows][cols] (row stride ld elements) with 16 x 32 boxes
bool make_epi_map(CUtensorMap* map, const void* ptr, bool f32, int rows, int cols, int ld) {
  auto enc = get_encode();
  if (!enc) return false;
  const size_t es = f32 ? 4 : 2;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * es};
  cuuint32_t box[2] = {32, 16};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16,
                   2, const_cast<void*>(ptr), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// Token width T of the 2-SM kernel's tiles on mc SM pairs: the multiple of 16 with the least
// estimated time in SM clocks. A K block's operands, 128 W rows and T / 2 token rows of 128
// bytes per SM, arrive at about 64 bytes per clock and SM, 256 + T clocks, which is also the
// MMAs' time (2 T) at T = 256 and more than it below; 313 clocks is the loading and issuing
// threads' time per K block (163 ns at 64 to 160 tokens x 1536 x 8960). As many rounds as the
// fullest pair has tiles: the first one's mainloop, for each further one its mainloop or, if
// that is longer, the epilogue that runs beside it (a fixed part per tile, 12 clocks per
// token, 30 with fp32 residual and output), and the last round's epilogue alone (16 or 28 per
// token). Measured (us, chosen T first): 1560 x 4608 x 1536 18.3 at T = 208 (20.4 at 256,
// 19.8 at 160), 1560 x 8960 x 1536 29.7 at 208 (32.0 at 256), 1560 x 1536 x 1536 with
// residual 11.4 at 144 (14.9 at 256), 4096 x 1536 x 1536 18.8 at 176 (22.3 at 256), 49920 x
// 1536 x 1536 185 at 256 (197 at 208). Bound by the epilogue: 3259 x 768 x 256 9.2 at 48, 7.3
// at 128, 6.4 at 160; 9965 x 768 x 256 14.4 at 80, 9.9 at 224, 10.3 at 256.
struct TileChoice {
  int T, rounds;
  double clocks;
};
TileChoice choose_tile(int M, int N, int nk, int mc, bool f32) {
  TileChoice best{0, 0, 0};
  for (int T = 256; T >= 16; T -= 16) {
    const long tiles = (long)((M + T - 1) / T) * ((N + C2_BN - 1) / C2_BN);
    const long rounds = (tiles + mc - 1) / mc;
    const double main = (double)nk * (256 + T > 313 ? 256 + T : 313);
    const double epilogue = f32 ? 3300 + 30.0 * T : 2900 + 12.0 * T;
    const double last = (f32 ? 28.0 : 16.0) * T + 400;
    const double est = main + (rounds - 1) * (main > epilogue ? main : epilogue) + last;
    if (best.T == 0 || est < best.clocks) best = {T, (int)rounds, est};
  }
  return best;
}

// Clusters of the 2-SM kernel that the current device can hold at once (pairs must share a GPC),
// asked once per device for the whole device, whatever SM budget the first launch has; without an
// answer, the launch's SMs in pairs.
template <int KIND>
int resident_clusters(int num_sms) {
  constexpr int DEVICES = 64;
  static std::atomic<int> known[DEVICES];  // zero until a launch has asked (any thread)
  int dev = 0, sms = 0, n = 0;
  if (cudaGetDevice(&dev) == cudaSuccess && dev < DEVICES) {
    n = known[dev].load(std::memory_order_relaxed);
    if (n > 0) return n;
  }
  cudaLaunchConfig_t cfg = {};
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess) {
    cfg.gridDim = dim3(sms / 2 * 2, 1, 1);
    cfg.blockDim = dim3(C2_THREADS, 1, 1);
    cfg.dynamicSmemBytes = C2_SMEM_BYTES;
    if (cudaOccupancyMaxActiveClusters(&n, gemm_tc2_kernel<KIND>, &cfg) == cudaSuccess && n > 0) {
      if (dev < DEVICES) known[dev].store(n, std::memory_order_relaxed);
      return n;
    }
  }
  cudaGetLastError();
  return num_sms / 2;
}

template <int KIND>
cudaError_t launch2(const GemmArgs& g, int* err, int num_sms, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(gemm_tc2_kernel<KIND>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, C2_SMEM_BYTES);
  if (e != cudaSuccess) return e;
  // as many clusters as can be resident at once, and no more than the num_sms SMs that this launch
  // may use allow
  const int occ = resident_clusters<KIND>(num_sms);
  const int mc = occ < num_sms / 2 ? occ : num_sms / 2;
  const int nk = g.K / BK;
  // Stream-K automatically (sk_mode 0, the single-op calls) only for a few rounds of
  // 256 x 256 tiles (<= 4) whose last round leaves at least 24 K blocks' worth of work per
  // pair idle ((rounds - tiles / pairs) * nk >= 24), with A and W together within half of
  // L2 (or one row of tiles, which reads W once however it is cut): the cut tiles' partials
  // are written and summed at a cost that a short K does not repay, and the contiguous unit
  // ranges spread each round over far-apart tiles, so operands larger than L2 are read
  // several times.
  const long tiles256 = (long)((g.M + 255) / 256) * (g.N / C2_BN);
  const long rounds256 = (tiles256 + mc - 1) / mc;
  const double operand_bytes = 2.0 * ((double)g.M + g.N) * g.K;
  const bool sk_ok =
      g.N % C2_BN == 0 && g.sk_ws && g.sk_ctr && mc <= g.sk_clusters && tiles256 * (long long)nk >= 4LL * mc;
  const bool sk_pays = rounds256 <= 4 && (rounds256 * mc - tiles256) * nk >= 24LL * mc &&
                       (operand_bytes <= 64.0 * 1024 * 1024 || g.M <= 256);
  if (g.sk_mode == 2 && !sk_ok) return cudaErrorInvalidValue;
  const TileChoice whole = choose_tile(g.M, g.N, nk, mc, C2Cfg<KIND>::F32);
  // stream-K keeps T = 256 (all rows of fewer): fewer tiles to cut, shorter K ranges to sum
  const int sk_T = g.M < 256 ? (g.M + 15) / 16 * 16 : 256;
  // Whole tiles where the split would pay sum K in parts with accumulators of their own,
  // whose ranges are 0.9 of a pair's under the split or shorter, as far as TMEM goes: the
  // tensor core's fp32 sums lose 7e-8 of the result per K block, and the shorter ranges keep
  // the error no larger than the split's (1560 x 1536 x 8960: 3.2e-6 in 3 parts, 4.6e-6
  // split, 1.0e-5 in one; 34.5 us in 3 parts, 32.7 in one).
  int parts = 1;
  if (sk_ok && sk_pays) {
    parts = (int)(mc / (0.9 * tiles256)) + 1;
    if (parts < 2) parts = 2;
    if (parts > c2_accs(whole.T)) parts = c2_accs(whole.T);
    const int len = (nk + parts - 1) / parts;  // K blocks of a part; the kernel takes as many
    parts = (nk + len - 1) / len;
  }
  bool use_sk = g.sk_mode == 2 || (g.sk_mode != 1 && sk_ok && sk_pays);
  // The model's own launches (sk_mode 3) take the faster of the two: a range of the split in
  // the clocks of choose_tile and 15 % (full-width tiles stay short of the rate), then
  // publishing, waiting for and summing the parts; a further accumulator about 1500. Measured
  // (us, split / whole tiles): rows x 1536 x 8960, 32 rows 12.4 / 29.8, 256 18.6 / 31.0, 640
  // 24.5 / 31.5, 1040 31.4 / 31.6, 1560 38.6 / 34.5; rows x 5120 x 5120, 100 rows 15.6 / 20.6,
  // 256 22.2 / 22.4, 400 28.2 / 23.1. More than one round of tiles: whole (1040 x 5120 x 5120
  // 50.3 / 44.7).
  if (g.sk_mode == 3 && use_sk) {
    const double range = (double)((tiles256 * nk + mc - 1) / mc);
    use_sk = rounds256 == 1 &&
             1.15 * range * (256 + sk_T > 313 ? 256 + sk_T : 313) + 51 * sk_T + 9500 <
                 whole.clocks + 1500 * (parts - 1);
  }
  if (use_sk) parts = 1;
  const SkArgs sk{use_sk ? 1 : 0, g.sk_ws, g.sk_ctr};
  const int T = use_sk ? sk_T : whole.T;
  const int tiles = (g.M + T - 1) / T * ((g.N + C2_BN - 1) / C2_BN);
  CUtensorMap ma, mw, mo, mr{};  // mr: unused without a residual
  if (!make_map(&ma, g.A, g.M, g.K, g.lda, T / 2) || !make_map(&mw, g.W, g.N, g.K, g.ldw, 128) ||
      !make_epi_map(&mo, g.epi.out, C2Cfg<KIND>::F32, g.M, g.N, g.epi.ldo) ||
      (C2Cfg<KIND>::F32 && g.epi.resid &&
       !make_epi_map(&mr, g.epi.resid, true, g.M, g.N, g.epi.ldo)))
    return cudaErrorInvalidValue;
  const int clusters = sk.on ? mc : (tiles < mc ? tiles : mc);
  return launch_k(gemm_tc2_kernel<KIND>, dim3(2 * clusters), dim3(C2_THREADS), C2_SMEM_BYTES, st,
                  ma, mw, mo, mr, g.M, g.N, g.K, T, parts, g.epi, sk, err);
}

cudaError_t dispatch2(const GemmArgs& g, int* err, int num_sms, cudaStream_t st) {
  switch (g.kind) {
    case EPI_BF16: return launch2<EPI_BF16>(g, err, num_sms, st);
    case EPI_GELU_BF16: return launch2<EPI_GELU_BF16>(g, err, num_sms, st);
    case EPI_RESID: return launch2<EPI_RESID>(g, err, num_sms, st);
    case EPI_RESID_DELTA: return launch2<EPI_RESID_DELTA>(g, err, num_sms, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

bool gemm_tc_supported(const GemmArgs& g) {
  auto al16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  return g.M >= 1 && g.N % 128 == 0 && g.K % BK == 0 && g.K >= BK && g.lda % 8 == 0 &&
         g.ldw % 8 == 0 && g.epi.ldo % 8 == 0 && al16(g.A) && al16(g.W) && al16(g.epi.out) &&
         (g.kind < EPI_RESID || al16(g.epi.resid)) && (g.kind != EPI_RESID_DELTA || g.epi.resid) &&
         (g.kind != EPI_RESID_DELTA || (al16(g.epi.base) && al16(g.epi.delta)));
}

cudaError_t gemm_tc_set_wait_limit(unsigned long long ns) { return fb_set_wait_limit_tu(ns); }

cudaError_t gemm_tc(const GemmArgs& g, int* err, int num_sms, cudaStream_t st, bool force_1sm) {
  if (!gemm_tc_supported(g)) return cudaErrorInvalidValue;
  // 2-SM tiles of 256 features x T tokens; where N leaves half of the last feature tile empty
  // (N % 256 == 128) only from K = 1536 and past one 128-row tile, where T spreads the rows
  // over more SMs than the 1-SM kernel's 128 x BN tiles (BN = 256 when that still gives every
  // SM a tile), and with every tile half empty (N = 128) up to 2048 rows. Measured (us, 1-SM /
  // 2-SM): N = 128, 1560 rows: K = 512 5.3 / 6.0, K = 1536 (the head) 9.1 / 8.7, K = 5120 22.3
  // / 17.9; 12480 rows, K = 1536: 9.9 / 10.8, N = 384 17.4 / 16.2.
  const bool half_tile = g.N % C2_BN != 0;
  const bool half_ok =
      g.K >= 1536 && g.M > BM && (g.N > 128 || g.M <= 16 * BM) && g.sk_mode != 2;
  if (!force_1sm && num_sms >= 2 && (!half_tile || half_ok)) return dispatch2(g, err, num_sms, st);
  if (g.sk_mode == 2) return cudaErrorInvalidValue;  // stream-K exists in the 2-SM kernel only
  const int mt = (g.M + BM - 1) / BM;
  if (g.N % 256 == 0 && mt * (g.N / 256) >= num_sms) return dispatch_kind<256>(g, err, num_sms, st);
  return dispatch_kind<128>(g, err, num_sms, st);
}
