// tcgen05 flash attention (head_dim 128) for the DiT block's self- and cross-attention:
// O = softmax(Q K^T / sqrt(128)) V per (batch, head), non-causal, ragged tails masked.
//
// One CTA = one 128-query tile of one (batch, head); 6 warps:
//  * warp 0: TMA producers. Lane 0 loads Q once (2 x [128 rows][64 cols] boxes) and then
//    128-key K tiles into a 3-slot ring; lane 1 loads the V tiles into a 2-slot ring
//    (128-byte swizzle). A K slot is released as soon as the S MMA that read it is done,
//    a V slot when its PV MMA is done, so K tiles load up to two tiles ahead.
//  * warp 1: TMEM owner (512 columns: S0, S1, O) and, one thread, the MMA issuer:
//    S_j = Q K_j^T into S[j % 2] (M=128, N=128 keys, K=128, both operands K-major),
//    then, once the softmax has written P_j, O += P_j V_j (A = P from shared memory,
//    K-major over keys; B = V, MN-major: the V tile is read as stored, [key][dim]).
//  * warps 2-5: softmax, one query row per thread (TMEM lane = row). Each reads its S
//    row (128 fp32), keeps the running row max m and sum l in registers, writes
//    P = exp2(S * log2(e)/sqrt(d) - m) as bf16 into the swizzled P tile, and rescales its
//    O row in TMEM only when the max grew by more than 2^8 since the last rescale
//    (every term of O and l always uses the same m, so the result is exact). At the end
//    each thread normalises its O row and stores it. The exponent arguments and the row
//    sum run on key pairs with packed fp32 FMA / add (one instruction per two keys).
// Ragged ends: the last key tile's S MMA is only as wide as its 32-key chunks of real keys
// and its PV MMA reads only those keys; in the 256-query kernel a second query tile that
// lies wholly past Lq is neither loaded nor computed.
// All waits are bounded; on a timeout the kernel records the error and drains.
#include <cudaTypedefs.h>

#include <cfloat>
#include <cmath>

#include "kernels.h"

namespace {

constexpr int TB = 128;                    // queries per CTA = keys per KV tile
constexpr int SUB = TB * 64 * 2;           // 16 KB: 128 rows x 64 bf16 (one swizzle width)
constexpr int Q_BYTES = 2 * SUB;           // 32 KB
constexpr int K_BYTES = 2 * SUB;           // one K tile (2 sub-tiles of 64 columns)
constexpr int V_BYTES = 2 * SUB;           // one V tile
constexpr int P_BYTES = 2 * SUB;
constexpr int KSLOT = 3, VSLOT = 2;        // K and V ring depths
constexpr int SMEM_BYTES = Q_BYTES + KSLOT * K_BYTES + VSLOT * V_BYTES + P_BYTES + 1024 + 256;
constexpr int THREADS = 192;
constexpr uint32_t TMEM_COLS = 512;        // S0 [0,128), S1 [128,256), O [256,384)
constexpr uint32_t O_COL = 256;

struct Params {
  int Lq, Lkv, kv_batch_rows;
  bf16* O;
  int ldo;
  float scale_log2;
  int* err;
  int batch, heads;
  // the persistent kernel's work split (see SplitPlan)
  int n_full_qb;     // 256-query items per head among the first n_full items
  int n_full, n_items;         // of all items; those behind the first n_full have one query tile
  int lone_qb;       // and among the first n_full those of this pair have (-1: none)
  unsigned div_qb, div_heads;  // ceil(2^32 / n_full_qb), ceil(2^32 / heads): see div_by
  int split;         // != 0: the items from `rounds` full rounds on are cut into equal shares
  int rounds;
  float* ws;         // per CTA: 8 warps x ATTN_WS_WARP floats (a cut item's partial)
  int* flags;        // per CTA and warp: 1 = its partial is in ws (0 between launches)
};

// Operand layouts (descriptors from desc_lo_k / desc_lo_mn): Q, K and P are K-major with
// 128-byte swizzle, 8-row groups 1024 B apart; V is MN-major with 128-byte swizzle, 64
// consecutive head dims per 128-byte row (one row per key), the next 64 dims SUB bytes on.

// instruction descriptor of the S MMA with N = 32 * nch keys (N field: N >> 3 at bit 17)
__device__ __forceinline__ uint32_t idesc_keys(uint32_t idesc128, int nch) {
  return (idesc128 & ~(0x3Fu << 17)) | ((uint32_t)(4 * nch) << 17);
}

// three-input maximum (one instruction on sm_100 and later)
__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
// maximum of a 128-score row: eight independent chains of three-input maxima, so the
// reduction is a few dependent steps instead of 128. At least the lowest finite value: a row
// whose scores are all -inf (masked keys) then has exponentials of exp2(-inf) = 0 and joins
// other tiles and parts with a factor of 0, where a maximum of -inf would give -inf + inf.
__device__ __forceinline__ float rowmax128(const float* s) {
  float m[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) m[k] = fmax3(s[k], s[k + 8], s[k + 16]);
#pragma unroll
  for (int i = 24; i + 16 <= 120; i += 16) {
#pragma unroll
    for (int k = 0; k < 8; ++k) m[k] = fmax3(m[k], s[i + k], s[i + 8 + k]);
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) m[k] = fmaxf(m[k], s[120 + k]);
  return fmax3(fmax3(m[0], m[1], m[2]), fmax3(fmax3(m[3], m[4], m[5]), m[6], m[7]), -FLT_MAX);
}

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}



__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
      "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]),
      "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]),
      "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]),
      "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, uint32_t src, int x, int y,
                                             int z) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];"
               ::"l"(reinterpret_cast<uint64_t>(map)), "r"(src), "r"(x), "r"(y), "r"(z)
               : "memory");
}

// The O rows of one warp (lane = row y0 + lane of batch b, its 128 columns at TMEM address
// t_o) to global memory: scaled by inv, rounded to bf16, written into a 4 KB staging tile
// (32 rows x 64 columns in the TMA 128-byte swizzle: 16-byte chunk c of row r at chunk
// position c ^ (r & 7), so a warp's writes fall in distinct banks) and stored by two 3-D
// TMA stores (64 columns each) that drop rows at or past Lq. Whole 128-byte row segments
// reach memory instead of one 16-byte piece per row per store instruction. Lane 0 waits
// until the first store has read the tile before it is refilled; the caller waits for the
// stores (bulk_wait) before the CTA exits or before the tile is used again.
__device__ __forceinline__ void store_o_warp(uint8_t* stage, const CUtensorMap* tmO, uint32_t t_o,
                                             float inv, int x0, int y0, int b, int Lq, int lane) {
  if (y0 >= Lq) return;  // every row of this warp lies past Lq
#pragma unroll 1
  for (int half = 0; half < 2; ++half) {
    uint32_t u[64];
    tmem_ld32(t_o + half * 64, u);
    tmem_ld32(t_o + half * 64 + 32, u + 32);
    tmem_ld_wait();
    reg_fence32(u);
    reg_fence32(u + 32);
    if (half == 1) {
      if (lane == 0) bulk_wait_read<0>();
      __syncwarp();
    }
    uint8_t* row = stage + lane * 128;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      uint4 w;
      w.x = pack_bf16x2(__uint_as_float(u[8 * c + 0]) * inv, __uint_as_float(u[8 * c + 1]) * inv);
      w.y = pack_bf16x2(__uint_as_float(u[8 * c + 2]) * inv, __uint_as_float(u[8 * c + 3]) * inv);
      w.z = pack_bf16x2(__uint_as_float(u[8 * c + 4]) * inv, __uint_as_float(u[8 * c + 5]) * inv);
      w.w = pack_bf16x2(__uint_as_float(u[8 * c + 6]) * inv, __uint_as_float(u[8 * c + 7]) * inv);
      *reinterpret_cast<uint4*>(row + ((c ^ (lane & 7)) * 16)) = w;
    }
    fence_async_smem();
    __syncwarp();
    if (lane == 0) {
      tma_store_3d(tmO, smem_u32(stage), x0 + half * 64, y0, b);
      bulk_commit();
    }
  }
}


__global__ void __launch_bounds__(THREADS, 1)
    attn_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                   const __grid_constant__ CUtensorMap tmV,
                   const __grid_constant__ CUtensorMap tmO, Params p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* Qs = smem;
  uint8_t* Ks = smem + Q_BYTES;
  uint8_t* Vs = Ks + KSLOT * K_BYTES;
  uint8_t* Ps = Vs + VSLOT * V_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(Ps + P_BYTES);
  uint64_t* q_full = bars;
  uint64_t* k_full = bars + 1;        // [3]
  uint64_t* k_empty = bars + 4;       // [3]
  uint64_t* v_full = bars + 7;        // [2]
  uint64_t* v_empty = bars + 9;       // [2]
  uint64_t* s_full = bars + 11;       // [2]
  uint64_t* p_full = bars + 13;
  uint64_t* o_done = bars + 14;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + 15);

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int qt = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
  const int q_row0 = b * p.Lq + qt * TB;
  const int kv_row0 = b * p.kv_batch_rows;
  const int n_kv = (p.Lkv + TB - 1) / TB;
  // the last key tile holds last_nch 32-key chunks of real keys: its S MMA is that many
  // chunks wide and its PV MMA reads only those keys
  const int last_nch = (p.Lkv - (n_kv - 1) * TB + 31) >> 5;
  int* err = p.err;
  bool failed = false;

  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    for (int s = 0; s < KSLOT; ++s) {
      mbar_init(&k_full[s], 1);
      mbar_init(&k_empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&v_full[s], 1);
      mbar_init(&v_empty[s], 1);
      mbar_init(&s_full[s], 1);
    }
    mbar_init(p_full, 4);   // one arrival per softmax warp
    mbar_init(o_done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    tma_prefetch_desc(&tmQ);
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmV);
  }
  if (warp == 1) tmem_alloc(tmem_holder, TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;
  griddep_wait();
  griddep_launch();

  if (warp == 0) {
    // ---------------- TMA producers: lane 0 Q and K, lane 1 V ----------------
    const int xq = h * 128;
    if (lane == 0) {
      mbar_expect_tx(q_full, Q_BYTES);
      tma_load_2d(Qs, &tmQ, q_full, xq, q_row0);
      tma_load_2d(Qs + SUB, &tmQ, q_full, xq + 64, q_row0);
      for (int j = 0; j < n_kv; ++j) {
        const int s = j % KSLOT;
        if (!mbar_wait(&k_empty[s], ((j / KSLOT) & 1) ^ 1u, err)) { failed = true; break; }
        uint8_t* st = Ks + s * K_BYTES;
        const int y = kv_row0 + j * TB;
        mbar_expect_tx(&k_full[s], K_BYTES);
        tma_load_2d(st, &tmK, &k_full[s], xq, y);
        tma_load_2d(st + SUB, &tmK, &k_full[s], xq + 64, y);
      }
    } else if (lane == 1) {
      for (int j = 0; j < n_kv; ++j) {
        const int s = j & 1;
        if (!mbar_wait(&v_empty[s], ((j >> 1) & 1) ^ 1u, err)) { failed = true; break; }
        uint8_t* st = Vs + s * V_BYTES;
        const int y = kv_row0 + j * TB;
        mbar_expect_tx(&v_full[s], V_BYTES);
        tma_load_2d(st, &tmV, &v_full[s], xq, y);
        tma_load_2d(st + SUB, &tmV, &v_full[s], xq + 64, y);
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    const uint32_t idesc_s = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TB >> 3) << 17) |
                             ((uint32_t)(TB >> 4) << 24);
    const uint32_t idesc_pv = idesc_s | (1u << 16);  // B (V) is MN-major
    const uint32_t dhi = DESC_HI;
    const uint32_t q_lo = desc_lo_k(smem_u32(Qs)), p_lo = desc_lo_k(smem_u32(Ps));
    const uint32_t k_lo = desc_lo_k(smem_u32(Ks)), v_lo = desc_lo_mn(smem_u32(Vs), SUB);
    auto issue_s = [&](int j) {
      const uint32_t ka = k_lo + (j % KSLOT) * (K_BYTES >> 4);
      if (j + 1 < n_kv || last_nch == 4) {
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          const uint32_t off = ((kk >> 2) * SUB + (kk & 3) * 32) >> 4;
          tc_mma_ss_lo(tmem + (j & 1) * TB, q_lo + off, ka + off, dhi, idesc_s, kk ? 1u : 0u);
        }
      } else {
        const uint32_t idesc = idesc_keys(idesc_s, last_nch);
#pragma unroll 1
        for (int kk = 0; kk < 8; ++kk) {
          const uint32_t off = ((kk >> 2) * SUB + (kk & 3) * 32) >> 4;
          tc_mma_ss_lo(tmem + (j & 1) * TB, q_lo + off, ka + off, dhi, idesc, kk ? 1u : 0u);
        }
      }
      tc_commit(&s_full[j & 1]);
    };
    if (mbar_wait_warp(q_full, 0, err) && mbar_wait_warp(&k_full[0], 0, err)) {
      tc_fence_after();
      if (elect_one()) issue_s(0);
      for (int j = 0; j < n_kv; ++j) {
        if (j + 1 < n_kv) {
          if (!mbar_wait_warp(&k_full[(j + 1) % KSLOT], ((j + 1) / KSLOT) & 1, err)) { failed = true; break; }
          tc_fence_after();
          if (elect_one()) issue_s(j + 1);
        }
        if (!mbar_wait_warp(p_full, j & 1, err)) { failed = true; break; }
        if (!mbar_wait_warp(&v_full[j & 1], (j >> 1) & 1, err)) { failed = true; break; }
        tc_fence_after();
        const uint32_t va = v_lo + (j & 1) * (V_BYTES >> 4);
        if (elect_one()) {
          if (j + 1 < n_kv || last_nch == 4) {
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
              const uint32_t off = ((kk >> 2) * SUB + (kk & 3) * 32) >> 4;
              tc_mma_ss_lo(tmem + O_COL, p_lo + off, va + kk * (2048 >> 4), dhi, idesc_pv,
                           (j | kk) ? 1u : 0u);
            }
          } else {
#pragma unroll 1
            for (int kk = 0; kk < 2 * last_nch; ++kk) {  // 16 keys per step
              const uint32_t off = ((kk >> 2) * SUB + (kk & 3) * 32) >> 4;
              tc_mma_ss_lo(tmem + O_COL, p_lo + off, va + kk * (2048 >> 4), dhi, idesc_pv,
                           (j | kk) ? 1u : 0u);
            }
          }
          tc_commit(o_done);
        }
      }
    } else {
      failed = true;
    }
  } else {
    // ---------------- softmax (warps 2..5), one query row per thread ----------------
    const int quarter = warp & 3;
    const int r = quarter * 32 + lane;
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
    float m_used = -INFINITY, l = 0.f;
    uint8_t* prow = Ps + r * 128;  // this row inside each 64-key sub-tile
    // one softmax thread releases K_j once S_j is done and V_{j-1} once PV_{j-1} is, so
    // the MMA issuer commits only what the softmax waits for (each tcgen05.commit holds up
    // the issuing thread while softmax warps share its SM sub-partition)
    const bool lead = warp == 2 && lane == 0;
    for (int j = 0; j < n_kv && !failed; ++j) {
      const bool ok = mbar_wait(&s_full[j & 1], (j >> 1) & 1, err);
      if (!__all_sync(0xffffffffu, ok)) { failed = true; break; }
      if (lead) mbar_arrive(&k_empty[j % KSLOT]);
      tc_fence_after();
      float s[128];
      {
        // all four loads in flight, one wait; scores stay unscaled (the scale is > 0, so the
        // row max commutes with it and is scaled once)
        uint32_t u[128];
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(lane_base + (j & 1) * TB + c * 32, u + c * 32);
        tmem_ld_wait();
#pragma unroll
        for (int c = 0; c < 4; ++c) reg_fence32(u + c * 32);
#pragma unroll
        for (int i = 0; i < 128; ++i) s[i] = __uint_as_float(u[i]);
      }
      const int valid = p.Lkv - j * TB;  // keys of this tile that exist
      if (valid < TB) {
#pragma unroll
        for (int i = 0; i < 128; ++i)
          if (i >= valid) s[i] = -INFINITY;
      }
      const float mx = rowmax128(s) * p.scale_log2;
      if (j > 0) {
        // PV_{j-1} must be done before P is overwritten and before O is touched
        const bool ok2 = mbar_wait(o_done, (j - 1) & 1, err);
        if (!__all_sync(0xffffffffu, ok2)) { failed = true; break; }
        if (lead) mbar_arrive(&v_empty[(j - 1) & 1]);
        tc_fence_after();
      }
      if (j == 0) {
        m_used = mx;
      } else if (__any_sync(0xffffffffu, mx > m_used + 8.f)) {
        const float m_new = fmaxf(m_used, mx);
        const float alpha = ex2(m_used - m_new);
        m_used = m_new;
        l *= alpha;
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
          uint32_t u[32];
          tmem_ld32(lane_base + O_COL + c * 32, u);
          tmem_ld_wait();
          reg_fence32(u);
#pragma unroll
          for (int i = 0; i < 32; ++i) u[i] = __float_as_uint(__uint_as_float(u[i]) * alpha);
          tmem_st32(lane_base + O_COL + c * 32, u);
        }
        tmem_st_wait();
      }
      // exponent arguments and the row sum on key pairs (packed FMA and add)
      const uint64_t sc2 = f2_join(p.scale_log2, p.scale_log2);
      const uint64_t nm2 = f2_join(-m_used, -m_used);
      uint64_t ls2[4] = {0ull, 0ull, 0ull, 0ull};  // independent partial sums
#pragma unroll
      for (int ch = 0; ch < 16; ++ch) {  // 16-byte chunks of 8 keys
        uint32_t w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float t0, t1;
          f2_split(f2_fma(f2_join(s[ch * 8 + 2 * q], s[ch * 8 + 2 * q + 1]), sc2, nm2), t0, t1);
          const float e0 = ex2(t0), e1 = ex2(t1);
          ls2[q] = f2_add(ls2[q], f2_join(e0, e1));
          w[q] = pack_bf16x2(e0, e1);
        }
        const int sub = ch >> 3, c16 = (ch & 7) ^ (r & 7);
        *reinterpret_cast<uint4*>(prow + sub * SUB + c16 * 16) = make_uint4(w[0], w[1], w[2], w[3]);
      }
      {
        float a0, a1, b0, b1;
        f2_split(f2_add(ls2[0], ls2[1]), a0, a1);
        f2_split(f2_add(ls2[2], ls2[3]), b0, b1);
        l += (a0 + a1) + (b0 + b1);
      }
      fence_async_smem();  // P visible to the tensor core (async proxy)
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(p_full);
    }
    if (!failed) {
      const bool ok = mbar_wait(o_done, (n_kv - 1) & 1, err);
      if (__all_sync(0xffffffffu, ok)) {
        tc_fence_after();
        // every MMA is done: the P tile is free for the O staging tiles (4 KB per warp)
        store_o_warp(Ps + (warp - 2) * 4096, &tmO, lane_base + O_COL, 1.f / l, h * 128,
                     qt * TB + quarter * 32, b, p.Lq, lane);
        if (lane == 0) bulk_wait<0>();
      } else {
        failed = true;
      }
    }
  }

  tc_fence_before();
  if (__syncthreads_or(failed)) {  // a role gave up: loads in flight land before the CTA exits
    const uint64_t t0 = fb_globaltimer();
    while (fb_globaltimer() - t0 < 100000ull) __nanosleep(1000);
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

// ---- two query tiles per CTA ---------------------------------------------------------
// Same computation with 256 queries per CTA: tiles A and B share every K/V tile (half
// the K/V traffic per FLOP). P is written back into the TMEM columns of its S tile
// (bf16 pairs) and read from there as the A operand of the PV MMA, so shared memory only
// holds Q_A, Q_B and the K/V ring. TMEM: S_A|P_A [0,128), S_B|P_B [128,256), O_A
// [256,384), O_B [384,512). MMA order per KV tile j: PV_A(j), S_A(j+1), PV_B(j), S_B(j+1),
// so each softmax group works while the tensor core runs the other group's MMAs.
// tcgen05 operations of one thread execute in order, so S_A(j+1) overwrites P_A(j) only
// after PV_A(j) has read it, and the commit that announces S_g(j+1) also covers PV_g(j)
// (the softmax may then rescale O_g).
constexpr int THREADS2 = 320;
constexpr int SMEM2_BYTES = 2 * Q_BYTES + KSLOT * K_BYTES + VSLOT * V_BYTES + 1024 + 256;


__global__ void __launch_bounds__(THREADS2, 1)
    attn_tc2_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                    const __grid_constant__ CUtensorMap tmV,
                   const __grid_constant__ CUtensorMap tmO, Params p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* Qs = smem;                  // [2 tiles][2 sub-tiles]
  uint8_t* Ks = smem + 2 * Q_BYTES;
  uint8_t* Vs = Ks + KSLOT * K_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(Vs + VSLOT * V_BYTES);
  uint64_t* q_full = bars;
  uint64_t* k_full = bars + 1;         // [3]
  uint64_t* k_empty = bars + 4;        // [3]
  uint64_t* v_full = bars + 7;         // [2]
  uint64_t* v_empty = bars + 9;        // [2]
  uint64_t* s_full = bars + 11;        // [2 groups]
  uint64_t* p_full = bars + 13;        // [2 groups]
  uint64_t* o_done = bars + 15;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + 16);

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int qb = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
  const int q_row0 = b * p.Lq + qb * 2 * TB;
  const int kv_row0 = b * p.kv_batch_rows;
  const int n_kv = (p.Lkv + TB - 1) / TB;
  int* err = p.err;
  bool failed = false;

  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    for (int s = 0; s < KSLOT; ++s) {
      mbar_init(&k_full[s], 1);
      mbar_init(&k_empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&v_full[s], 1);
      mbar_init(&v_empty[s], 1);
      mbar_init(&s_full[s], 1);
      mbar_init(&p_full[s], 4);
    }
    mbar_init(o_done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    tma_prefetch_desc(&tmQ);
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmV);
  }
  if (warp == 1) tmem_alloc(tmem_holder, TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;
  griddep_wait();
  griddep_launch();

  if (warp == 0) {
    // ---------------- TMA producers: lane 0 Q and K, lane 1 V ----------------
    const int xq = h * 128;
    if (lane == 0) {
      // a second query tile with no query in range (the ragged end of Lq) does no work
      const int ngroups = qb * 2 * TB + TB < p.Lq ? 2 : 1;
      mbar_expect_tx(q_full, ngroups * Q_BYTES);
      for (int g = 0; g < ngroups; ++g) {
        tma_load_2d(Qs + g * Q_BYTES, &tmQ, q_full, xq, q_row0 + g * TB);
        tma_load_2d(Qs + g * Q_BYTES + SUB, &tmQ, q_full, xq + 64, q_row0 + g * TB);
      }
      for (int j = 0; j < n_kv; ++j) {
        const int s = j % KSLOT;
        if (!mbar_wait(&k_empty[s], ((j / KSLOT) & 1) ^ 1u, err)) { failed = true; break; }
        uint8_t* st = Ks + s * K_BYTES;
        const int y = kv_row0 + j * TB;
        mbar_expect_tx(&k_full[s], K_BYTES);
        tma_load_2d(st, &tmK, &k_full[s], xq, y);
        tma_load_2d(st + SUB, &tmK, &k_full[s], xq + 64, y);
      }
    } else if (lane == 1) {
      for (int j = 0; j < n_kv; ++j) {
        const int s = j & 1;
        if (!mbar_wait(&v_empty[s], ((j >> 1) & 1) ^ 1u, err)) { failed = true; break; }
        uint8_t* st = Vs + s * V_BYTES;
        const int y = kv_row0 + j * TB;
        mbar_expect_tx(&v_full[s], V_BYTES);
        tma_load_2d(st, &tmV, &v_full[s], xq, y);
        tma_load_2d(st + SUB, &tmV, &v_full[s], xq + 64, y);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc_s = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TB >> 3) << 17) |
                               ((uint32_t)(TB >> 4) << 24);
      const uint32_t idesc_pv = idesc_s | (1u << 16);
      const uint32_t dhi = DESC_HI;
      const uint32_t q_lo[2] = {desc_lo_k(smem_u32(Qs)), desc_lo_k(smem_u32(Qs + Q_BYTES))};
      const uint32_t k_lo = desc_lo_k(smem_u32(Ks)), v_lo = desc_lo_mn(smem_u32(Vs), SUB);
      const int two = qb * 2 * TB + TB < p.Lq;  // both tiles hold queries (as for the Q load)
      // real keys of the last key tile, in 32-key chunks (see attn_tc_kernel)
      const int last_nch = (p.Lkv - (n_kv - 1) * TB + 31) >> 5;
      // full key tiles take the constant-folded loops; the last tile of a ragged Lkv
      // (last_nch < 4 chunks of 32 keys) issues S with N = 32 * last_nch and PV over those
      // keys only
      auto issue_s = [&](int g, int j) {
        const uint32_t ka = k_lo + (j % KSLOT) * (K_BYTES >> 4);
        const uint32_t qg = q_lo[g];
        if (j + 1 < n_kv || last_nch == 4) {
#pragma unroll
          for (int kk = 0; kk < 8; ++kk) {
            const uint32_t off = ((kk >> 2) * SUB + (kk & 3) * 32) >> 4;
            tc_mma_ss_lo(tmem + g * TB, qg + off, ka + off, dhi, idesc_s, kk ? 1u : 0u);
          }
        } else {
          const uint32_t idesc = idesc_keys(idesc_s, last_nch);
#pragma unroll 1
          for (int kk = 0; kk < 8; ++kk) {
            const uint32_t off = ((kk >> 2) * SUB + (kk & 3) * 32) >> 4;
            tc_mma_ss_lo(tmem + g * TB, qg + off, ka + off, dhi, idesc, kk ? 1u : 0u);
          }
        }
        tc_commit(&s_full[g]);
        if (g == 1 || two == 0) tc_commit(&k_empty[j % KSLOT]);  // every tile's S_j done
      };
      auto issue_pv = [&](int g, int j) {
        const uint32_t va = v_lo + (j & 1) * (V_BYTES >> 4);
        if (j + 1 < n_kv || last_nch == 4) {
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            tc_mma_ts_lo(tmem + O_COL + g * TB, tmem + g * TB + kk * 8, va + kk * (2048 >> 4),
                         dhi, idesc_pv, (j | kk) ? 1u : 0u);
        } else {
#pragma unroll 1
          for (int kk = 0; kk < 2 * last_nch; ++kk)  // 16 keys per step
            tc_mma_ts_lo(tmem + O_COL + g * TB, tmem + g * TB + kk * 8, va + kk * (2048 >> 4),
                         dhi, idesc_pv, (j | kk) ? 1u : 0u);
        }
      };
      bool ok = mbar_wait(q_full, 0, err) && mbar_wait(&k_full[0], 0, err);
      if (ok && two) {
        tc_fence_after();
        issue_s(0, 0);
        issue_s(1, 0);
        for (int j = 0; j < n_kv && ok; ++j) {
          const bool more = j + 1 < n_kv;
          if (!(ok = mbar_wait(&p_full[0], j & 1, err))) break;
          if (!(ok = mbar_wait(&v_full[j & 1], (j >> 1) & 1, err))) break;
          tc_fence_after();
          issue_pv(0, j);
          if (more) {
            if (!(ok = mbar_wait(&k_full[(j + 1) % KSLOT], ((j + 1) / KSLOT) & 1, err))) break;
            tc_fence_after();
            issue_s(0, j + 1);
          }
          if (!(ok = mbar_wait(&p_full[1], j & 1, err))) break;
          tc_fence_after();
          issue_pv(1, j);
          tc_commit(&v_empty[j & 1]);
          if (more) issue_s(1, j + 1);
        }
      } else if (ok) {
        // one tile (the second lies past Lq): the same chain without the other group
        tc_fence_after();
        issue_s(0, 0);
        for (int j = 0; j < n_kv && ok; ++j) {
          if (!(ok = mbar_wait(&p_full[0], j & 1, err))) break;
          if (!(ok = mbar_wait(&v_full[j & 1], (j >> 1) & 1, err))) break;
          tc_fence_after();
          issue_pv(0, j);
          tc_commit(&v_empty[j & 1]);
          if (j + 1 < n_kv) {
            if (!(ok = mbar_wait(&k_full[(j + 1) % KSLOT], ((j + 1) / KSLOT) & 1, err))) break;
            tc_fence_after();
            issue_s(0, j + 1);
          }
        }
      }
      if (ok) tc_commit(o_done);
      failed = !ok;
    }
  } else {
    // ---------------- softmax groups: warps 2-5 -> tile A, warps 6-9 -> tile B ----------
    const int g = (warp - 2) >> 2;
    const int quarter = warp & 3;
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
    const uint32_t s_col = g * TB, o_col = O_COL + g * TB;
    float m_used = -INFINITY, l = 0.f;
    // a tile with no query in range (the ragged end of Lq) has no MMAs and no softmax
    if (qb * 2 * TB + g * TB < p.Lq) {
      for (int j = 0; j < n_kv && !failed; ++j) {
        const bool ok = mbar_wait(&s_full[g], j & 1, err);
        if (!__all_sync(0xffffffffu, ok)) { failed = true; break; }
        tc_fence_after();
        float s[128];
        {
          // all four loads in flight, one wait; scores stay unscaled (the scale is > 0, so the
          // row max commutes with it and is scaled once)
          uint32_t u[128];
#pragma unroll
          for (int c = 0; c < 4; ++c) tmem_ld32(lane_base + s_col + c * 32, u + c * 32);
          tmem_ld_wait();
#pragma unroll
          for (int c = 0; c < 4; ++c) reg_fence32(u + c * 32);
#pragma unroll
          for (int i = 0; i < 128; ++i) s[i] = __uint_as_float(u[i]);
        }
        const int valid = p.Lkv - j * TB;  // keys of this tile that exist
        if (valid < TB) {
#pragma unroll
          for (int i = 0; i < 128; ++i)
            if (i >= valid) s[i] = -INFINITY;
        }
        const float mx = rowmax128(s) * p.scale_log2;
        if (j == 0) {
          m_used = mx;
        } else if (__any_sync(0xffffffffu, mx > m_used + 8.f)) {
          const float m_new = fmaxf(m_used, mx);
          const float alpha = ex2(m_used - m_new);
          m_used = m_new;
          l *= alpha;
#pragma unroll 1
          for (int c = 0; c < 4; ++c) {
            uint32_t u[32];
            tmem_ld32(lane_base + o_col + c * 32, u);
            tmem_ld_wait();
            reg_fence32(u);
#pragma unroll
            for (int i = 0; i < 32; ++i) u[i] = __float_as_uint(__uint_as_float(u[i]) * alpha);
            tmem_st32(lane_base + o_col + c * 32, u);
          }
        }
        const uint64_t sc2 = f2_join(p.scale_log2, p.scale_log2);
        const uint64_t nm2 = f2_join(-m_used, -m_used);
        uint64_t ls2[2] = {0ull, 0ull};  // independent partial sums
        // keys 0-63 from the registers; P of those keys fills TMEM columns 0-31 only, so
        // keys 64-127 are read again from their S columns instead of staying live in
        // registers through the first half (register room for the item loop)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          float h[64];
          if (c == 0) {
#pragma unroll
            for (int i = 0; i < 64; ++i) h[i] = s[i];
          } else {
            uint32_t u2[64];
            tmem_ld32(lane_base + s_col + 64, u2);
            tmem_ld32(lane_base + s_col + 96, u2 + 32);
            tmem_ld_wait();
            reg_fence32(u2);
            reg_fence32(u2 + 32);
#pragma unroll
            for (int i = 0; i < 64; ++i) h[i] = __uint_as_float(u2[i]);
            if (valid < TB) {
#pragma unroll
              for (int i = 0; i < 64; ++i)
                if (64 + i >= valid) h[i] = -INFINITY;
            }
          }
          uint32_t u[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            float t0, t1;
            f2_split(f2_fma(f2_join(h[2 * i], h[2 * i + 1]), sc2, nm2), t0, t1);
            const float e0 = ex2(t0), e1 = ex2(t1);
            ls2[i & 1] = f2_add(ls2[i & 1], f2_join(e0, e1));
            u[i] = pack_bf16x2(e0, e1);
          }
          tmem_st32(lane_base + s_col + c * 32, u);
        }
        {
          float a0, a1;
          f2_split(f2_add(ls2[0], ls2[1]), a0, a1);
          l += a0 + a1;
        }
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_full[g]);
      }
      if (!failed) {
        const bool ok = mbar_wait(o_done, 0, err);
        if (__all_sync(0xffffffffu, ok)) {
          tc_fence_after();
          // every MMA is done: the Q tiles are free for the O staging tiles (4 KB per warp)
          store_o_warp(Qs + (warp - 2) * 4096, &tmO, lane_base + o_col, 1.f / l, h * 128,
                       qb * 2 * TB + g * TB + quarter * 32, b, p.Lq, lane);
          if (lane == 0) bulk_wait<0>();
        } else {
          failed = true;
        }
      }
    }
  }

  if (failed || *(volatile int*)err != 0) {
    const uint64_t t0 = fb_globaltimer();
    while (fb_globaltimer() - t0 < 100000ull) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

// ---- persistent 256-query kernel ----------------------------------------------------
// attn_tc2_kernel's computation with at most one CTA per SM, each working through segments:
// whole items (batch b, head h, query-tile pair qb) and, where whole items would leave SMs
// idle in the last round, parts of the key range of one item. Items are numbered with the
// pairs of two query tiles first (qb fastest, so that the CTAs running at the same time
// share their K/V tiles in L2), then the items of a last single tile, or by head throughout
// (single_tiles_in_place). Per CTA the work of
// consecutive segments overlaps:
//  * the producer loads the next segment's Q as soon as the current one's last S MMAs are
//    done (q_empty) and carries on through the K/V rings, whose slots and phases count
//    across segments; the slots are released by a softmax thread that has seen a tile's last
//    S MMAs done, so the MMA issuer commits only what the softmax groups wait for (each
//    tcgen05.commit holds up the issuing thread while softmax warps share its SM
//    sub-partition);
//  * the MMA issuer starts the next segment's S MMAs right after the current one's last PV
//    (the tensor pipe runs in order, so S_g overwrites P_g only after PV_g has read it);
//  * each softmax group stores its O rows (o_done, one phase per segment of the group) while
//    those S MMAs run, each thread its row in 32-byte stores (whole sectors); its first P
//    of the next segment is announced only after those TMEM reads, so the first PV of the
//    next segment (accumulate = 0) cannot overwrite O early.
// Group B has no work in items whose second query tile lies past Lq; the issuer and the
// group count the phases of their own barriers.
//
// Work split. G CTAs; `rounds` full rounds of items (CTA c: items c, c + G, ...), then, with
// p.split, the rest as G contiguous ranges of equal cost over the (item, 128-key step) units:
// 4 per step of an item with two query tiles, 3 with one (measured about 0.75). An item cut
// between CTAs c_lo .. c_hi is finished by c_hi, the others leave the group's unnormalised O
// rows, row maxima and sums (fp32) in the workspace; c_hi adds them in CTA order, so the
// result does not depend on timing. A CTA works on the part that it contributes first and
// finishes another's item last, so the finisher's wait is normally over before it begins;
// and it waits only for CTAs of lower index, which started before it.
constexpr int ATTN_WS_WARP = 32 * 128 + 64;  // O rows [chunk 4][4-column group 8][lane][4], (m, l)
static_assert(8 * ATTN_WS_WARP == ATTN_WS_FLOATS_PER_CTA && 8 == ATTN_FLAGS_PER_CTA, "attention workspace");

enum { SEG_WHOLE = 0, SEG_PART = 1, SEG_FINISH = 2 };
struct Seg {
  int item, j0, j1, kind;  // key tiles j0 .. j1 - 1 of the item
};
// One CTA's segments in order: a contributed part, whole items of the full rounds, whole
// items of its range, the tail of an item that it finishes.
struct SplitPlan {
  int part_item, part_j0, part_j1;  // part_j1 == 0: none
  int whole_first, n_whole;
  int tail_item, tail_j0;           // tail_item < 0: none
  int c_lo;                         // first contributor of tail_item
};
// The split region's unit arithmetic.
struct SplitUnits {
  int n_kv, n_full, n_items, r0;    // r0: first item of the region
  unsigned full_units, units;       // (units x G fits 32 bits: plan_split)
  __device__ SplitUnits(const Params& p, int n_kv_, int G) : n_kv(n_kv_) {
    n_full = p.n_full;
    n_items = p.n_items;
    r0 = p.rounds * G;              // <= n_full
    full_units = (unsigned)(n_full - r0) * 4 * n_kv;
    units = full_units + (unsigned)(n_items - n_full) * 3 * n_kv;
  }
  // where CTA c's range begins
  __device__ void at(unsigned c, unsigned G, int& item, int& j) const {
    const unsigned u = c * units / G;
    if (u >= units) {
      item = n_items;
      j = 0;
    } else if (u < full_units) {
      item = r0 + (int)(u / (4u * n_kv));
      j = (int)(u % (4u * n_kv)) / 4;
    } else {
      item = n_full + (int)((u - full_units) / (3u * n_kv));
      j = (int)((u - full_units) % (3u * n_kv)) / 3;
    }
  }
};
__device__ void make_split_plan(const Params& p, int n_kv, int G, int c, SplitPlan* pl) {
  const SplitUnits su(p, n_kv, G);
  pl->part_j1 = 0;
  pl->n_whole = 0;
  pl->tail_item = -1;
  int i0, j0, i1, j1;
  su.at(c, G, i0, j0);
  su.at(c + 1, G, i1, j1);
  if (i0 == i1) {                   // inside one item, which another CTA finishes
    pl->part_item = i0;
    pl->part_j0 = j0;
    pl->part_j1 = j1 > j0 ? j1 : 0;
    return;
  }
  if (j0 > 0) {
    pl->tail_item = i0;
    pl->tail_j0 = j0;
    // the contributors are the CTAs before this one down to the first whose range reaches
    // the item's first key tile (a share is more than a step, so each holds some of it,
    // except one whose range ends within the item's first step)
    int lo = c, ilo = i0, jlo = j0;
    while (ilo == i0 && jlo > 0) {
      --lo;
      su.at(lo, G, ilo, jlo);
    }
    pl->c_lo = lo;
  }
  pl->whole_first = j0 > 0 ? i0 + 1 : i0;
  pl->n_whole = i1 - pl->whole_first;
  pl->part_item = i1;
  pl->part_j0 = 0;
  pl->part_j1 = j1;
}
// Segment s of the CTA; false past the last.
template <bool SPLIT>
__device__ __forceinline__ bool get_seg(const Params& p, const SplitPlan& pl, int s, int n_kv,
                                        Seg& g) {
  g.j0 = 0;
  g.j1 = n_kv;
  g.kind = SEG_WHOLE;
  if (!SPLIT) {
    g.item = (int)blockIdx.x + s * (int)gridDim.x;
    return g.item < p.n_items;
  }
  if (pl.part_j1) {
    if (s == 0) {
      g = Seg{pl.part_item, pl.part_j0, pl.part_j1, SEG_PART};
      return true;
    }
    --s;
  }
  if (s < p.rounds) {
    g.item = (int)blockIdx.x + s * (int)gridDim.x;
    return true;
  }
  s -= p.rounds;
  if (s < pl.n_whole) {
    g.item = pl.whole_first + s;
    return true;
  }
  if (s > pl.n_whole || pl.tail_item < 0) return false;
  g = Seg{pl.tail_item, pl.tail_j0, n_kv, SEG_FINISH};
  return true;
}
// Waits (bounded, as mbar_wait) until another CTA has raised its flag from 0 to 1 (any other
// value, as a crashed launch could leave it, is waited on until the time limit).
__device__ __forceinline__ bool wait_flag(int* flag, int* err) {
  const uint64_t t0 = fb_globaltimer();
  while (*(volatile int*)flag != 1) {
    if (*(volatile int*)err != 0) return false;
    if (fb_globaltimer() - t0 > fb_wait_limit()) {
      fb_report(err, FB_DEVERR_WAIT_TIMEOUT);
      return false;
    }
    __nanosleep(64);
  }
  return true;
}
// Whole warp: makes its earlier stores visible and raises the flag.
__device__ __forceinline__ void raise_flag(int* flag, int lane) {
  __threadfence();
  __syncwarp();
  if (lane == 0) atomicAdd(flag, 1);
}
// The finisher of a cut item waits for the parts of CTAs c_lo .. blockIdx.x - 1 (this warp's
// rows: flags by lane), updates the row's maximum m and sum l with theirs, in CTA order, and
// returns in a_own the factor of the rows that it has in TMEM itself. False if a wait gave up.
__device__ __forceinline__ bool join_parts(const Params& p, int c_lo, int ww, int lane, float& m,
                                           float& l, float& a_own, int* err) {
  const int n = (int)blockIdx.x - c_lo;
  int* flags = p.flags + (size_t)c_lo * 8 + ww;
  bool ok = true;
  for (int i = lane; i < n && ok; i += 32) ok = wait_flag(flags + i * 8, err);
  if (!__all_sync(0xffffffffu, ok)) return false;
  __threadfence();
  for (int i = lane; i < n; i += 32) flags[i * 8] = 0;  // free for the next launch
  const float* part = p.ws + ((size_t)c_lo * 8 + ww) * ATTN_WS_WARP;
  float m_all = m;
#pragma unroll 4
  for (int i = 0; i < n; ++i)
    m_all = fmaxf(m_all, __ldcg(part + (size_t)i * 8 * ATTN_WS_WARP + 4096 + 2 * lane));
  a_own = ex2(m - m_all);
  l *= a_own;
  m = m_all;
#pragma unroll 4
  for (int i = 0; i < n; ++i) {
    const float2 ml = __ldcg(
        reinterpret_cast<const float2*>(part + (size_t)i * 8 * ATTN_WS_WARP + 4096) + lane);
    l += ml.y * ex2(ml.x - m_all);
  }
  return true;
}
// Adds 64 columns (half 0 or 1) of the parts' rows, scaled to the maximum m, to f in CTA order.
// A part's 16 loads are in flight together.
__device__ __forceinline__ void add_parts(const Params& p, int c_lo, int ww, int lane, float m,
                                          int half, float4* f) {
  const float* part = p.ws + ((size_t)c_lo * 8 + ww) * ATTN_WS_WARP;
#pragma unroll 1
  for (int c = c_lo; c < (int)blockIdx.x; ++c, part += 8 * ATTN_WS_WARP) {
    const float a = ex2(__ldcg(part + 4096 + 2 * lane) - m);
    float4 v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q)
      v[q] = __ldcg(reinterpret_cast<const float4*>(part) + (half * 16 + q) * 32 + lane);
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      f[q].x += a * v[q].x;
      f[q].y += a * v[q].y;
      f[q].z += a * v[q].z;
      f[q].w += a * v[q].w;
    }
  }
}
// x / d by the rounded-up reciprocal ceil(2^32 / d): exact while x d < 2^32 (plan_split
// checks the largest item number); d = 1 has no 32-bit reciprocal and is passed as 0
__device__ __forceinline__ int div_by(int x, unsigned recip) {
  return recip ? (int)__umulhi((unsigned)x, recip) : x;
}
// item -> query-tile pair qb, head h, batch b, groups with work
__device__ __forceinline__ int decode_item(const Params& p, int item, int& qb, int& h, int& b) {
  const bool full = item < p.n_full;
  int bh = item - p.n_full;
  qb = p.n_full_qb;
  if (full) {
    bh = div_by(item, p.div_qb);
    qb = item - bh * p.n_full_qb;
  }
  b = div_by(bh, p.div_heads);
  h = bh - b * p.heads;
  return full && qb != p.lone_qb ? 2 : 1;
}
// groups with work of an item
template <bool SPLIT>
__device__ __forceinline__ int item_tiles(const Params& p, int item) {
  if (item >= p.n_full) return 1;
  if (SPLIT) return 2;  // (cut items: single query tiles are the last items)
  return item - div_by(item, p.div_qb) * p.n_full_qb != p.lone_qb ? 2 : 1;
}

// One O row: 32 columns at a time, scaled by inv and rounded to bf16, in 32-byte stores (whole
// sectors) where the rows are 32-byte aligned.
struct ORow {
  bf16* row;
  bool in, st32;
  __device__ __forceinline__ ORow(const Params& p, int item, int q) {
    int qb, h, b;
    decode_item(p, item, qb, h, b);
    const int qrow = qb * 2 * TB + q;
    in = qrow < p.Lq;
    row = p.O + (size_t)(b * p.Lq + qrow) * p.ldo + h * 128;
    st32 = ((reinterpret_cast<uintptr_t>(p.O) & 31) | (p.ldo & 15)) == 0;
  }
  __device__ __forceinline__ void store32(int c, const uint32_t* u, float inv) const {
    if (!in) return;
    if (st32) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        uint32_t w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
          w[i] = pack_bf16x2(__uint_as_float(u[q * 16 + 2 * i]) * inv,
                             __uint_as_float(u[q * 16 + 2 * i + 1]) * inv);
        store_b32x8(row + c * 32 + q * 16, w);
      }
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(u[q * 8 + i]) * inv;
        store_bf16x8(row + c * 32 + q * 8, v);
      }
    }
  }
};

template <bool SPLIT>
__global__ void __launch_bounds__(THREADS2, 1)
    attn_tc2p_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                     const __grid_constant__ CUtensorMap tmV, Params p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* Qs = smem;                  // [2 tiles][2 sub-tiles]
  constexpr int KS = KSLOT;            // K ring slots
  uint8_t* Ks = smem + 2 * Q_BYTES;
  uint8_t* Vs = Ks + KS * K_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(Vs + VSLOT * V_BYTES);
  uint64_t* q_full = bars;
  uint64_t* q_empty = bars + 1;
  uint64_t* k_full = bars + 2;         // [KS]
  uint64_t* k_empty = bars + 5;        // [KS]
  uint64_t* v_full = bars + 8;         // [2]
  // bars + 10, + 11: unused (a V slot is released by the K slot release of the next tile)
  uint64_t* s_full = bars + 12;        // [2 groups]
  uint64_t* p_full = bars + 14;        // [2 groups]
  uint64_t* o_done = bars + 16;        // [2 groups]
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + 18);

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int n_kv = (p.Lkv + TB - 1) / TB;
  __shared__ SplitPlan plan;
  int* err = p.err;
  bool failed = false;

  if (SPLIT && threadIdx.x == 64) make_split_plan(p, n_kv, gridDim.x, blockIdx.x, &plan);
  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    mbar_init(q_empty, 1);
    for (int s = 0; s < KS; ++s) {
      mbar_init(&k_full[s], 1);
      mbar_init(&k_empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&v_full[s], 1);
      mbar_init(&s_full[s], 1);
      mbar_init(&p_full[s], 4);
      mbar_init(&o_done[s], 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    tma_prefetch_desc(&tmQ);
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmV);
  }
  if (warp == 1) tmem_alloc(tmem_holder, TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;
  griddep_wait();
  griddep_launch();

  if (warp == 0) {
    // ---------------- TMA producers: lane 0 Q and K, lane 1 V ----------------
    if (lane == 0) {
      uint32_t kt = 0;  // K tiles loaded by this CTA
      Seg sg;
      for (int it = 0; !failed && get_seg<SPLIT>(p, plan, it, n_kv, sg); ++it) {
        int qb, h, b;
        const int ng = decode_item(p, sg.item, qb, h, b);
        const int xq = h * 128, q_row0 = b * p.Lq + qb * 2 * TB, kv_row0 = b * p.kv_batch_rows;
        if (!mbar_wait(q_empty, (it & 1) ^ 1u, err)) { failed = true; break; }
        mbar_expect_tx(q_full, ng * Q_BYTES);
        for (int g = 0; g < ng; ++g) {
          tma_load_2d(Qs + g * Q_BYTES, &tmQ, q_full, xq, q_row0 + g * TB);
          tma_load_2d(Qs + g * Q_BYTES + SUB, &tmQ, q_full, xq + 64, q_row0 + g * TB);
        }
        for (int j = sg.j0; j < sg.j1; ++j, ++kt) {
          const int s = kt % KS;
          if (!mbar_wait(&k_empty[s], ((kt / KS) & 1) ^ 1u, err)) { failed = true; break; }
          uint8_t* st = Ks + s * K_BYTES;
          const int y = kv_row0 + j * TB;
          mbar_expect_tx(&k_full[s], K_BYTES);
          tma_load_2d(st, &tmK, &k_full[s], xq, y);
          tma_load_2d(st + SUB, &tmK, &k_full[s], xq + 64, y);
        }
      }
    } else if (lane == 1) {
      uint32_t vt = 0;  // V tiles loaded by this CTA
      Seg sg;
      for (int it = 0; !failed && get_seg<SPLIT>(p, plan, it, n_kv, sg); ++it) {
        int qb, h, b;
        decode_item(p, sg.item, qb, h, b);
        const int xq = h * 128, kv_row0 = b * p.kv_batch_rows;
        for (int j = sg.j0; j < sg.j1; ++j, ++vt) {
          const int s = vt & 1;
          // slot s last held tile vt - 2; its PV MMAs are done once the S MMAs of tile
          // vt - 1 are (the issuer issues those after them): the K slot release of tile
          // vt - 1 (K and V tiles are counted alike)
          if (vt >= 2) {
            const uint32_t t = vt - 1;
            if (!mbar_wait(&k_empty[t % KS], (t / KS) & 1, err)) { failed = true; break; }
          }
          uint8_t* st = Vs + s * V_BYTES;
          const int y = kv_row0 + j * TB;
          mbar_expect_tx(&v_full[s], V_BYTES);
          tma_load_2d(st, &tmV, &v_full[s], xq, y);
          tma_load_2d(st + SUB, &tmV, &v_full[s], xq + 64, y);
        }
      }
    }
  } else if (warp == 1) {
    const uint32_t idesc_s = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TB >> 3) << 17) |
                             ((uint32_t)(TB >> 4) << 24);
    const uint32_t idesc_pv = idesc_s | (1u << 16);
    const int last_nch = (p.Lkv - (n_kv - 1) * TB + 31) >> 5;
    // descriptor lower words of the Q buffers, K slot 0 and V slot 0 (the other slots lie
    // K_BYTES / V_BYTES further on)
    const uint32_t dhi = DESC_HI;
    const uint32_t q_lo[2] = {desc_lo_k(smem_u32(Qs)), desc_lo_k(smem_u32(Qs + Q_BYTES))};
    const uint32_t k_lo = desc_lo_k(smem_u32(Ks)), v_lo = desc_lo_mn(smem_u32(Vs), SUB);
    // Everything the MMAs' operands depend on is counted under warp-uniform control flow (the
    // segment's bounds, read from shared memory, only enter votes).
    uint32_t ks = 0, kph = 0;           // K ring slot and phase of the current key tile
    uint32_t vt = 0;                    // V tiles consumed (slot vt & 1)
    uint32_t pph[2] = {0u, 0u};         // P phases per group
    bool ok = true;
    // S_g of the key tile in K slot `slot`; `last`: the last key tile (its real keys only)
    auto issue_s = [&](int g, uint32_t slot, bool last) {
      const uint32_t ka = k_lo + slot * (K_BYTES >> 4);
      const uint32_t qg = q_lo[g];
      if (!last || last_nch == 4) {
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          const uint32_t off = ((kk >> 2) * SUB + (kk & 3) * 32) >> 4;
          tc_mma_ss_lo(tmem + g * TB, qg + off, ka + off, dhi, idesc_s, kk ? 1u : 0u);
        }
      } else {
        const uint32_t idesc = idesc_keys(idesc_s, last_nch);
#pragma unroll 1
        for (int kk = 0; kk < 8; ++kk) {
          const uint32_t off = ((kk >> 2) * SUB + (kk & 3) * 32) >> 4;
          tc_mma_ss_lo(tmem + g * TB, qg + off, ka + off, dhi, idesc, kk ? 1u : 0u);
        }
      }
      tc_commit(&s_full[g]);
    };
    auto issue_pv = [&](int g, uint32_t acc, bool last) {
      const uint32_t va = v_lo + (vt & 1) * (V_BYTES >> 4);
      if (!last || last_nch == 4) {
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)
          tc_mma_ts_lo(tmem + O_COL + g * TB, tmem + g * TB + kk * 8, va + kk * (2048 >> 4),
                       dhi, idesc_pv, kk ? 1u : acc);
      } else {
#pragma unroll 1
        for (int kk = 0; kk < 2 * last_nch; ++kk)
          tc_mma_ts_lo(tmem + O_COL + g * TB, tmem + g * TB + kk * 8, va + kk * (2048 >> 4),
                       dhi, idesc_pv, kk ? 1u : acc);
      }
    };
    for (int it = 0; ok; ++it) {
      Seg sg;
      if (!__all_sync(0xffffffffu, get_seg<SPLIT>(p, plan, it, n_kv, sg))) break;
      const bool two = __all_sync(0xffffffffu, item_tiles<SPLIT>(p, sg.item) == 2);
      int j = sg.j0;
      bool last = __all_sync(0xffffffffu, j + 1 == n_kv);
      if (!(ok = mbar_wait_warp(q_full, it & 1, err))) break;
      if (!(ok = mbar_wait_warp(&k_full[ks], kph, err))) break;
      tc_fence_after();
      if (elect_one()) {
        issue_s(0, ks, last);
        if (two) issue_s(1, ks, last);
      }
      uint32_t acc = 0;
      for (bool more = true; more; acc = 1) {
        ++j;
        more = __all_sync(0xffffffffu, j < sg.j1);
        const bool next_last = __all_sync(0xffffffffu, j + 1 == n_kv);
        const uint32_t ks1 = ks + 1 == KS ? 0 : ks + 1, kph1 = ks + 1 == KS ? kph ^ 1u : kph;
        // this step's V and next step's K tiles first: they are normally there already,
        // and these waits then overlap the tensor pipe's last instructions of the
        // previous batch instead of following the softmax's hand-off (the pipe holds
        // about one instruction, so every wait between batches is idle pipe time)
        if (!(ok = mbar_wait_warp(&v_full[vt & 1], (vt >> 1) & 1, err))) break;
        if (more && !(ok = mbar_wait_warp(&k_full[ks1], kph1, err))) break;
        if (!(ok = mbar_wait_warp(&p_full[0], pph[0], err))) break;
        pph[0] ^= 1u;
        tc_fence_after();
        // a group's O rows are complete with its last PV: its epilogue may start while
        // the other group's last PV runs
        if (elect_one()) {
          issue_pv(0, acc, last);
          if (more) issue_s(0, ks1, next_last);
          else tc_commit(&o_done[0]);
        }
        if (two) {
          if (!(ok = mbar_wait_warp(&p_full[1], pph[1], err))) break;
          pph[1] ^= 1u;
          tc_fence_after();
          if (elect_one()) {
            issue_pv(1, acc, last);
            if (more) issue_s(1, ks1, next_last);
            else tc_commit(&o_done[1]);
          }
        }
        ks = ks1;
        kph = kph1;
        ++vt;
        last = next_last;
      }
    }
    failed = !ok;
  } else {
    // ---------------- softmax groups: warps 2-5 -> tile A, warps 6-9 -> tile B ----------
    const int g = (warp - 2) >> 2;
    const int quarter = warp & 3;
    const int r = quarter * 32 + lane;
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
    const uint32_t s_col = g * TB, o_col = O_COL + g * TB;
    uint32_t cnt = 0;  // segments this group has worked on
    uint32_t sc = 0;   // S tiles this group has seen
    uint32_t kt = 0;   // K tiles of the CTA so far (numbered as the producer does)
    // the group whose S MMAs come last in a key tile (B, or A where B has no work) releases
    // the tile's K slot, and at the segment's last tile the Q buffer, once its S is done: the
    // issuer's S MMAs of a tile follow its PV MMAs of the tile before, so this also frees
    // that tile's V slot
    const bool lead = (warp & 3) == 2 && lane == 0;  // one thread per group
    bool flag_due = false;  // this group's part is stored, its flag not yet raised
    auto raise_due = [&] {
      if (flag_due) raise_flag(p.flags + blockIdx.x * 8 + warp - 2, lane);
      flag_due = false;
    };
    float m_used = -INFINITY, l = 0.f;  // the row's maximum and sum in the current segment
    bool finish = false;                // the last segment completes an item cut between CTAs
    for (int it = 0;; ++it) {
      int j, j_end;
      bool last_group;
      {
        Seg sg;
        if (!get_seg<SPLIT>(p, plan, it, n_kv, sg)) break;
        const int ng = item_tiles<SPLIT>(p, sg.item);
        if (g >= ng) {  // this tile lies past Lq: no work
          kt += sg.j1 - sg.j0;
          if (SPLIT) raise_due();
          continue;
        }
        j = sg.j0;
        j_end = sg.j1;
        last_group = g == ng - 1;
      }
      m_used = -INFINITY;
      l = 0.f;
      for (; j < j_end; ++j, ++sc, ++kt) {
        const bool ok = mbar_wait(&s_full[g], sc & 1, err);
        if (!__all_sync(0xffffffffu, ok)) { failed = true; break; }
        if (lead && last_group) {
          mbar_arrive(&k_empty[kt % KS]);
          if (j == j_end - 1) mbar_arrive(q_empty);
        }
        tc_fence_after();
        float s[128];
        {
          uint32_t u[128];
#pragma unroll
          for (int c = 0; c < 4; ++c) tmem_ld32(lane_base + s_col + c * 32, u + c * 32);
          tmem_ld_wait();
#pragma unroll
          for (int c = 0; c < 4; ++c) reg_fence32(u + c * 32);
#pragma unroll
          for (int i = 0; i < 128; ++i) s[i] = __uint_as_float(u[i]);
        }
        const int valid = p.Lkv - j * TB;
        if (valid < TB) {
#pragma unroll
          for (int i = 0; i < 128; ++i)
            if (i >= valid) s[i] = -INFINITY;
        }
        const float mx = rowmax128(s) * p.scale_log2;
        // The segment's first tile: every lane's m_used is still -inf, which no maximum is. The
        // vote keeps the branch, which is warp-wide (the rescale), uniform. (Comparing the tile's
        // number instead takes 2 % longer: 8 x 1560 queries x 12 heads 103.6 -> 105.9 us.)
        if (__all_sync(0xffffffffu, m_used == -INFINITY)) {
          m_used = mx;
        } else if (__any_sync(0xffffffffu, mx > m_used + 8.f)) {
          const float m_new = fmaxf(m_used, mx);
          const float alpha = ex2(m_used - m_new);
          m_used = m_new;
          l *= alpha;
#pragma unroll 1
          for (int c = 0; c < 4; ++c) {
            uint32_t u[32];
            tmem_ld32(lane_base + o_col + c * 32, u);
            tmem_ld_wait();
            reg_fence32(u);
#pragma unroll
            for (int i = 0; i < 32; ++i) u[i] = __float_as_uint(__uint_as_float(u[i]) * alpha);
            tmem_st32(lane_base + o_col + c * 32, u);
          }
        }
        const uint64_t sc2 = f2_join(p.scale_log2, p.scale_log2);
        const uint64_t nm2 = f2_join(-m_used, -m_used);
        uint64_t ls2[2] = {0ull, 0ull};  // independent partial sums
        // keys 0-63 from the registers; P of those keys fills TMEM columns 0-31 only, so
        // keys 64-127 are read again from their S columns instead of staying live in
        // registers through the first half (register room for the item loop)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          float h[64];
          if (c == 0) {
#pragma unroll
            for (int i = 0; i < 64; ++i) h[i] = s[i];
          } else {
            uint32_t u2[64];
            tmem_ld32(lane_base + s_col + 64, u2);
            tmem_ld32(lane_base + s_col + 96, u2 + 32);
            tmem_ld_wait();
            reg_fence32(u2);
            reg_fence32(u2 + 32);
#pragma unroll
            for (int i = 0; i < 64; ++i) h[i] = __uint_as_float(u2[i]);
            if (valid < TB) {
#pragma unroll
              for (int i = 0; i < 64; ++i)
                if (64 + i >= valid) h[i] = -INFINITY;
            }
          }
          uint32_t u[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            float t0, t1;
            f2_split(f2_fma(f2_join(h[2 * i], h[2 * i + 1]), sc2, nm2), t0, t1);
            const float e0 = ex2(t0), e1 = ex2(t1);
            ls2[i & 1] = f2_add(ls2[i & 1], f2_join(e0, e1));
            u[i] = pack_bf16x2(e0, e1);
          }
          tmem_st32(lane_base + s_col + c * 32, u);
        }
        {
          float a0, a1;
          f2_split(f2_add(ls2[0], ls2[1]), a0, a1);
          l += a0 + a1;
        }
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_full[g]);
      }
      if (failed) break;
      Seg sg;
      get_seg<SPLIT>(p, plan, it, n_kv, sg);
      if (SPLIT) raise_due();
      // the segment's O rows: PV_g of its last key tile done
      const bool ok = mbar_wait(&o_done[g], cnt & 1, err);
      if (!__all_sync(0xffffffffu, ok)) { failed = true; break; }
      tc_fence_after();
      if (SPLIT && sg.kind == SEG_PART) {
        // publish the rows, maxima and sums; the flag goes up after the next segment's last
        // key tile (its stores have then long been performed), or after the last segment
        float* part = p.ws + ((size_t)blockIdx.x * 8 + warp - 2) * ATTN_WS_WARP;
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
          uint32_t u[32];
          tmem_ld32(lane_base + o_col + c * 32, u);
          tmem_ld_wait();
          reg_fence32(u);
#pragma unroll
          for (int q = 0; q < 8; ++q)
            reinterpret_cast<float4*>(part)[(c * 8 + q) * 32 + lane] =
                make_float4(__uint_as_float(u[4 * q]), __uint_as_float(u[4 * q + 1]),
                            __uint_as_float(u[4 * q + 2]), __uint_as_float(u[4 * q + 3]));
        }
        reinterpret_cast<float2*>(part + 4096)[lane] = make_float2(m_used, l);
        flag_due = true;
      } else if (SPLIT && sg.kind == SEG_FINISH) {  // always the CTA's last segment
        finish = true;
        break;
      } else {
        const ORow out(p, sg.item, g * TB + r);
        const float inv = 1.f / l;
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
          uint32_t u[32];
          tmem_ld32(lane_base + o_col + c * 32, u);
          tmem_ld_wait();
          reg_fence32(u);
          out.store32(c, u, inv);
        }
      }
      ++cnt;
    }
    if (SPLIT && !failed) raise_due();
    float a_own = 1.f;
    if (SPLIT && finish) {
      if (!join_parts(p, plan.c_lo, warp - 2, lane, m_used, l, a_own, err)) {
        failed = true;
        finish = false;
      }
    }
    if (SPLIT && finish) {
      const ORow out(p, plan.tail_item, g * TB + r);
      const float inv = 1.f / l;
#pragma unroll 1
      for (int half = 0; half < 2; ++half) {
        float4 f[16];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t u[32];
          tmem_ld32(lane_base + o_col + half * 64 + c * 32, u);
          tmem_ld_wait();
          reg_fence32(u);
#pragma unroll
          for (int q = 0; q < 8; ++q)
            f[c * 8 + q] = make_float4(
                __uint_as_float(u[4 * q]) * a_own, __uint_as_float(u[4 * q + 1]) * a_own,
                __uint_as_float(u[4 * q + 2]) * a_own, __uint_as_float(u[4 * q + 3]) * a_own);
        }
        add_parts(p, plan.c_lo, warp - 2, lane, m_used, half, f);
        out.store32(half * 2, reinterpret_cast<const uint32_t*>(f), inv);
        out.store32(half * 2 + 1, reinterpret_cast<const uint32_t*>(f + 8), inv);
      }
    }
  }

  tc_fence_before();
  if (__syncthreads_or(failed)) {  // a role gave up: loads in flight land before the CTA exits
    const uint64_t t0 = fb_globaltimer();
    while (fb_globaltimer() - t0 < 100000ull) __nanosleep(1000);
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encoder() {
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

bool map_128x64(CUtensorMap* m, const bf16* ptr, int rows, int cols, int ld) {
  auto enc = encoder();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * sizeof(bf16)};
  cuuint32_t box[2] = {64, (cuuint32_t)TB};
  cuuint32_t estr[2] = {1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16*>(ptr), dims, strides, box,
             estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// O as a 3-D tensor [batch][Lq][cols] (row stride ld, batch stride Lq ld): a TMA store box
// of 32 rows x 64 columns (128-byte swizzle) stops at each batch's Lq
bool map_o(CUtensorMap* m, const bf16* ptr, int batch, int Lq, int cols, int ld) {
  auto enc = encoder();
  if (!enc) return false;
  cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)Lq, (cuuint64_t)batch};
  cuuint64_t strides[2] = {(cuuint64_t)ld * sizeof(bf16), (cuuint64_t)Lq * ld * sizeof(bf16)};
  cuuint32_t box[3] = {64, 32, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<bf16*>(ptr), dims, strides, box,
             estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Whole items: whether the single query tiles (Lq's last one) run behind the other tiles of their
// head instead of after all pairs. Last they fill the last round better, but read their head's
// K / V again: from DRAM where the K / V of all heads are more than about half of L2, once more
// per n_pairs reads. Measured (us, last / in place; 12 heads): 16 x 384 queries (38 MB of K / V)
// 20.4 / 21.5, 24 x 384 29.0 / 30.8, 16 x 600 41.9 / 41.8, 16 x 640 (63 MB) 42.3 / 41.0, 32 x 384
// 43.2 / 42.2, 64 x 384 81.1 / 73.2, 64 x 600 156.1 / 148.7, 64 x 640 159.7 / 148.2, 32 x 896
// 141.7 / 136.7, 32 x 1100 209.4 / 204.7, 32 x 1408 302.7 / 299.3; from six pairs on within 1.5 %
// either way (8 x 1560 105.0 / 106.7, 32 x 1560 390.6 / 389.8, on 112 SMs 478.4 / 481.7, 8 x 3200
// 341.4 / 344.8). Shared K / V stay in L2: 64 x 384 x 77 keys 39.1 / 43.5.
bool single_tiles_in_place(const AttnArgs& a, int n_pairs) {
  const double kv = 4.0 * 128 * a.heads * (double)a.Lkv * (a.kv_batch_rows ? a.batch : 1);
  return n_pairs <= 5 && kv > 60e6;
}

// Chooses the persistent kernel's split and grid. Times in 128-key steps of a 256-query item
// (1.45-1.55 us): whole items take their rounds; with the split every CTA takes an equal share,
// its steps are about 5 % longer (the ranges share less K / V, the loop keeps more registers),
// and storing, waiting for and adding the parts of cut items takes about 4.5 steps and one
// more per part. Measured (us, whole items / split): 1 x 1560 x 12 heads 23.4 / 25.5, 2 x 1560
// 40.8 / 35.2, 4 x 1560 60.9 / 57.8, 8 x 1560 103.3 / 102.7, 16 x 1560 186.9 / 202.9, 1 x 4096
// 93.8 / 71.8, 4 x 4096 279.7 / 258.6, 1 x 1560 on 40 SMs 58.3 / 51.4, cross-attention (4 key
// tiles) 4 x 1560 23.9 / 27.5.
int plan_split(const AttnArgs& a, int sms, Params* p) {
  const int n_kv = (a.Lkv + TB - 1) / TB;
  const long bh = (long)a.heads * a.batch, items = (a.Lq + 2 * TB - 1) / (2 * TB) * bh;
  p->n_full_qb = (a.Lq + TB - 1) / (2 * TB);
  const long n_full = p->n_full_qb * bh, lone = items - n_full;
  p->n_full = (int)n_full;
  p->n_items = (int)items;
  auto recip = [](int d) { return d > 1 ? (unsigned)((0x100000000ull + d - 1) / d) : 0u; };
  p->div_qb = recip(p->n_full_qb);
  p->div_heads = recip(a.heads);
  p->lone_qb = -1;
  p->ws = a.ws;
  p->flags = a.flags;
  p->split = 0;
  p->rounds = 0;
  const int grid = (int)(items < sms ? items : sms);
  auto whole = [&] {
    if (lone > 0 && single_tiles_in_place(a, p->n_full_qb)) {
      p->n_full_qb += 1;
      p->n_full = p->n_items;
      p->lone_qb = p->n_full_qb - 1;
      p->div_qb = recip(p->n_full_qb);
    }
    return grid;
  };
  if (!a.ws || !a.flags || sms > a.ws_ctas) return whole();
  // full rounds of two-tile items but one, so that every CTA's share of the rest is at least
  // about one item and an item is cut in few parts
  const double total = (4.0 * n_full + 3.0 * lone) * n_kv / 4;  // steps
  long rounds = (long)(total / sms / n_kv) - 1;
  if (rounds > n_full / sms) rounds = n_full / sms;
  if (rounds < 0) rounds = 0;
  const double rest = total - (double)rounds * sms * n_kv;
  long G = sms;
  if (rounds == 0 && rest / G < 3) G = (long)(rest / 3);  // at least 3 steps per CTA
  if (G < 1) G = 1;
  const double share = rest / G, parts = std::ceil(n_kv / share) + 1;
  const double t_split = 1.05 * (rounds * n_kv + share) + 4.5 + parts;
  const double t_whole = (double)((items + sms - 1) / sms) * n_kv;
  // (the split's 32-bit unit arithmetic: see SplitUnits)
  if (G <= 1 || t_split >= 0.98 * t_whole || total * 4 * sms > 4e9) return whole();
  p->split = 1;
  p->rounds = (int)rounds;
  return (int)G;
}

int sms_of(const AttnArgs& a) {
  int dev = 0, sms = a.sms;
  if (sms <= 0 && (cudaGetDevice(&dev) != cudaSuccess ||
                   cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess))
    sms = 148;
  return sms;
}

enum Form { Q128, Q256, PERSISTENT };
Form choose_form(const AttnArgs& a, int sms) {
  // 256-query items share each K/V tile between two query tiles and overlap one tile's
  // softmax with the other's MMAs; in the persistent kernel one costs about 1.25 times a
  // 128-query CTA (measured on a 40-SM partition, 1 x 1560 queries x 12 heads: 4 waves of
  // 128-query CTAs 68.3 us self / 30.9 us cross, 3 items per CTA 64.7 / 25.6 us). The
  // choice compares waves (for the persistent kernel, items per CTA): on 152 SMs that
  // shape is 2 waves of 128-query CTAs (156) or 1 item per CTA (84), on 40 SMs 4 against
  // 3. The shorter 128-query CTAs remain only where the 256-query form saves no waves
  // (both fit one wave, or Lq <= 128).
  const long ctas1 = (long)((a.Lq + TB - 1) / TB) * a.heads * a.batch;
  const long nqb = (a.Lq + 2 * TB - 1) / (2 * TB), ctas2 = nqb * a.heads * a.batch;
  const long w1 = (ctas1 + sms - 1) / sms, w2 = (ctas2 + sms - 1) / sms;
  const bool two = a.tc_variant >= 2 || (a.tc_variant == 0 && 4 * w1 >= 5 * w2);
  // 256-query items run in the persistent kernel (one CTA per SM looping over them, or one
  // item per CTA when they fit one wave: its MMA issue and slot releases are the leaner
  // ones, 1 x 1560 queries x 12 heads 25.8 -> 24.5 us); tc_variant 2 keeps the one-item
  // kernel
  const bool persistent = (a.tc_variant >= 3 || (two && a.tc_variant == 0)) &&
                          ctas2 * (a.heads > nqb ? a.heads : nqb) < (1ll << 32);  // see div_by
  return persistent ? PERSISTENT : two ? Q256 : Q128;
}

}  // namespace

cudaError_t attention_tc_set_wait_limit(unsigned long long ns) {
  return fb_set_wait_limit_tu(ns);
}

bool attention_tc_supported(const AttnArgs& a) {
  auto al16 = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15) == 0; };
  return a.head_dim == 128 && a.Lq >= 1 && a.Lkv >= 1 && a.batch >= 1 && a.ldq % 8 == 0 &&
         a.ldk % 8 == 0 && a.ldv % 8 == 0 && a.ldo % 8 == 0 && al16(a.Q) && al16(a.K) &&
         al16(a.V) && al16(a.O);
}

int attention_tc_split(const AttnArgs& a) {
  const int sms = sms_of(a);
  Params p;
  if (!attention_tc_supported(a) || choose_form(a, sms) != PERSISTENT) return 0;
  const int grid = plan_split(a, sms, &p);
  return p.split ? grid : 0;
}

cudaError_t attention_tc(const AttnArgs& a, int* err, cudaStream_t st) {
  if (!attention_tc_supported(a)) return cudaErrorInvalidValue;
  const int cols = a.heads * 128;
  const int kv_rows = a.kv_batch_rows ? (a.batch - 1) * a.kv_batch_rows + a.Lkv : a.Lkv;
  CUtensorMap mq, mk, mv, mo;
  if (!map_128x64(&mq, a.Q, a.batch * a.Lq, cols, a.ldq) ||
      !map_128x64(&mk, a.K, kv_rows, cols, a.ldk) || !map_128x64(&mv, a.V, kv_rows, cols, a.ldv) ||
      !map_o(&mo, a.O, a.batch, a.Lq, cols, a.ldo))
    return cudaErrorInvalidValue;
  const int sms = sms_of(a);
  Params p;
  p.Lq = a.Lq;
  p.Lkv = a.Lkv;
  p.kv_batch_rows = a.kv_batch_rows;
  p.O = a.O;
  p.ldo = a.ldo;
  p.scale_log2 = 1.4426950408889634f / sqrtf(128.f);
  p.err = err;
  p.batch = a.batch;
  p.heads = a.heads;
  const Form form = choose_form(a, sms);
  if (form == PERSISTENT) {
    const int grid = plan_split(a, sms, &p);
    auto kern = p.split ? attn_tc2p_kernel<true> : attn_tc2p_kernel<false>;
    cudaError_t e =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM2_BYTES);
    if (e != cudaSuccess) return e;
    e = launch_k(kern, dim3(grid), dim3(THREADS2), SMEM2_BYTES, st, mq, mk, mv, p);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
  }
  if (form == Q256) {
    cudaError_t e = cudaFuncSetAttribute(attn_tc2_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM2_BYTES);
    if (e != cudaSuccess) return e;
    dim3 grid((a.Lq + 2 * TB - 1) / (2 * TB), a.heads, a.batch);
    e = launch_k(attn_tc2_kernel, grid, dim3(THREADS2), SMEM2_BYTES, st, mq, mk, mv, mo, p);
    if (e != cudaSuccess) return e;
  } else {
    cudaError_t e = cudaFuncSetAttribute(attn_tc_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    if (e != cudaSuccess) return e;
    dim3 grid((a.Lq + TB - 1) / TB, a.heads, a.batch);
    e = launch_k(attn_tc_kernel, grid, dim3(THREADS), SMEM_BYTES, st, mq, mk, mv, mo, p);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}
