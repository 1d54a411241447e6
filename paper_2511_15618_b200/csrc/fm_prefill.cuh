// Prefill: BOS + prompt of all sequences as one packed multi-row forward.
//
// The rows of a chunk are the coordinate positions of up to a few thousand prompt tokens, sequence
// segments one after the other; segments start at multiples of 9, so every vertex and face of a
// segment has its children in the same chunk, and only the two hiddens before the segment come from
// the carry rings.  Each projection is then a real GEMM (weights read once per chunk instead of once
// per D + 1 tokens), and the attention of a segment streams a key once per 128 query rows.
#pragma once
#include "fm_common.cuh"
#include "fm_gemm_tc.cuh"
#include "fm_kernels.cuh"
#include "fm_ptx.cuh"

namespace pf {

// One sequence's share of a chunk: level-local positions [p0, p0 + n) at rows [r0, r0 + n).
struct Seg {
  int b, last;                   // sequence; last != 0: the segment ends with the prompt
  int p0[3], n[3], r0[3];
};
typedef PackedRow Row;

// Pointers of one layer, for launches that span layers.
struct LayerPtr { const bf16* Wqkv; const float* g1; bf16* K; bf16* V; int level, pad; };

// ------------------------------------------------------------------------------------------
// GEMM
// ------------------------------------------------------------------------------------------
// y[n][m] = sum_k W[m, k] A[n, k].  Tile: 128 output features per CTA (the MMA's M axis) x NT rows (N axis).
// Operand rows with two bfloat16 terms lie as [hi | lo] tiles behind one another and form one operand of
// 2 NT rows, so a weight slab is loaded once for both.  Persistent CTAs walk over the tiles
// (feature tiles innermost: neighbouring CTAs share their operand rows in L2); a ring of shared-memory
// stages decouples the copies from the warp that issues the MMAs, and two accumulators in tensor memory let the
// epilogue of a tile run under the MMAs of the next.
// CG = 2: two CTAs of a cluster multiply together (tcgen05 cta_group::2, M = 256).  Each keeps its own 128 features of
// weights; of the operand rows the first holds the hi and the second the lo tile, so an SM copies 32 instead of
// 48 KB per slab and its MMAs read a third less shared memory.  The first CTA issues; both CTAs' copies count on its barriers.
// tiled_cut (flashmesh.cu) says where that is faster: long K or many rows.
// What a slab (512 MMA clocks) waited for, 6994 rows, d = 1024, K = 4096: one thread per role behind `lane == 0`, whose
// every descriptor went from general to uniform registers: 970 clocks; whole warps in step with one elected lane: 740.
// The epilogue runs beside that, and must not take longer than a tile's MMAs (8 200 clocks at K = 1024).  A warp turns
// CW rows x 32 features in shared memory so that a lane works on four neighbouring features of a row (no shuffles, 8- and
// 16-byte stores, a row's address once for all of them), sixteen warps hide each other's latencies, the rows' scales
// come from a warp of their own, and what an epilogue reads is requested a step ahead.
// QKV / output projection / first / second FFN matrix, 6994 rows, d = 1024, us: 99 / 41 / 125 / 110 before these, 63 / 32 / 85 / 83
// now (without any epilogue 57 / 22 / 73 / 69; tensor pipe 75 % active in the last).
enum Mode { PF_F32 = 0, PF_GELU = 1, PF_RESID = 2, PF_QKV = 3, PF_PREFIX = 4 };

constexpr int EPI_WARPS = 16, CW = 16;           // epilogue warps; rows a warp takes at a time
constexpr int THREADS = 128 + 32 * EPI_WARPS;    // weight producer, operand producer, MMA warp, the rows' scales, the epilogue
constexpr int MAX_STAGES = 6;

struct Gemm {
  const bf16* W; const CUtensorMap* tmA;
  int M, K, R, NT, stages, slabs;  // slabs of 64 k per stage: 1 or 2
  int tiles_m, tiles_n, tiles;   // tiles = tiles_m * tiles_n * layers (PF_PREFIX), else tiles_m * tiles_n; a pair's tile has 256 features
  const bf16* w_base; const CUtensorMap* tmW;      // pairs: weights through one map over the workspace [bytes / 128][64]
  int w_tile0, w_tiles;          // first and number of 128-feature tiles of the matrix
  const int* n_active;           // skip when *n_active == 0 (may be null)
  int* status;
};
struct Epi {
  const float* ssq_in; int ssq_n, ld_ssq; float inv_d, eps;     // RMSNorm scale of the operand rows (null: none)
  void* out; int ldo, lo_off;                                   // PF_F32: fp32 (rows a multiple of 4 apart), PF_GELU: [hi | lo] bf16
  float* x; int ldx, add; const float* gain; bf16* a_out; int lda; float* ssq_out;      // PF_RESID
  Dims dm; const Row* rows; int level; const float2* rope; float qscale;                // PF_QKV
  bf16 *q, *kbuf, *vbuf, *Kc, *Vc;                              // keys and values: into the cache, or (Kc null) into kbuf / vbuf
  const LayerPtr* layers; int row_first, rows_layer;            // PF_PREFIX: operand rows of layer z at z * rows_layer
};

inline int stage_slabs(int NT, int parts) { return parts * NT > 128 ? 1 : 2; }      // slabs of 64 k per stage
inline int stage_bytes(int NT, int parts, int cg) { return stage_slabs(NT, parts) * (tc::BM * 128 + parts * NT / cg * 128); }
// behind the ring: the epilogue's scratch, the rows' scales of two tiles, barriers, room to align
constexpr int SMEM_MOST = 227 * 1024, SMEM_REST = EPI_WARPS * CW * 32 * 4 + 2 * 128 * 4 + 256 + 1024;
inline int ring_stages(int NT, int parts, int cg) {
  const int n = (SMEM_MOST - SMEM_REST) / stage_bytes(NT, parts, cg);
  return n < MAX_STAGES ? n : MAX_STAGES;
}
inline int smem_bytes(int NT, int parts, int cg, int stages) { return stages * stage_bytes(NT, parts, cg) + SMEM_REST; }

// tcgen05 instructions of a CTA (CG = 1) or of a pair of CTAs (CG = 2)
template <int CG>
__device__ inline void tmem_alloc(uint32_t* slot, uint32_t ncols) {
  if (CG == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(ptx::smem_u32(slot)), "r"(ncols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  } else {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(ptx::smem_u32(slot)), "r"(ncols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
}
template <int CG>
__device__ inline void tmem_free(uint32_t tmem, uint32_t ncols) {
  if (CG == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
  else asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
}
template <int CG>
__device__ inline void mma(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t accumulate) {
  if (CG == 1) tc::mma_ss(tmem_d, da, db, idesc, accumulate);
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
        : "memory");
}
// arrives on the barrier (of both CTAs of a pair) once the MMAs issued so far are done
template <int CG>
__device__ inline void commit(uint64_t* bar) {
  if (CG == 1) tc::commit(bar);
  else
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(ptx::smem_u32(bar)),
                 "h"((uint16_t)3)
                 : "memory");
}

__device__ inline void ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,"
      "%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]),
        "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
__device__ inline void ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ inline void ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
template <int MODE, int PARTS, int CG>
__global__ void __launch_bounds__(THREADS, 1) gemm_kernel(const Gemm g, const Epi e) {
  if (g.n_active != nullptr && *g.n_active == 0) {           // the whole grid leaves; keep the launch chain ordered
    ptx::grid_dep_launch();
    ptx::grid_dep_wait();
    return;
  }
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int NT = g.NT, ST = g.stages, SLABS = g.slabs;
  const int HN = PARTS * NT / CG;                            // operand rows of a slab in this CTA
  const int w_slab = tc::BM * 128, a_slab = HN * 128, stage = SLABS * (w_slab + a_slab);
  float* s_turn = reinterpret_cast<float*>(sm + ST * stage);                 // [epilogue warp][CW rows][32 features]
  float* s_inv = s_turn + EPI_WARPS * CW * 32;               // [2][128]
  uint64_t* full = reinterpret_cast<uint64_t*>(s_inv + 2 * 128);
  uint64_t* empty = full + MAX_STAGES;
  uint64_t* acc_full = empty + MAX_STAGES;
  uint64_t* acc_empty = acc_full + 2;
  uint64_t *inv_full = acc_empty + 2, *inv_empty = inv_full + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(inv_empty + 2);
  int& s_fail = *reinterpret_cast<int*>(tmem_slot + 1);
  const int tid = threadIdx.x, warp = (int)ptx::uniform(tid >> 5), lane = tid & 31;
  const int rank = CG == 2 ? (int)ptx::uniform(tc::cluster_rank()) : 0;    // place in the pair
  const int worker = (int)blockIdx.x / CG, workers = (int)gridDim.x / CG;
  const int slabs = g.K / tc::BK, steps = (slabs + SLABS - 1) / SLABS;
  uint32_t ncols = 32;
  while ((int)ncols < 2 * PARTS * NT) ncols <<= 1;
  const int acc_cols = (int)ncols / 2;
  if (tid == 0) {
    s_fail = 0;
    for (int i = 0; i < ST; ++i) { ptx::mbar_init(full + i, 2); ptx::mbar_init(empty + i, 1); }
    for (int i = 0; i < 2; ++i) { ptx::mbar_init(acc_full + i, 1); ptx::mbar_init(acc_empty + i, CG * EPI_WARPS); ptx::mbar_init(inv_full + i, 1); ptx::mbar_init(inv_empty + i, EPI_WARPS); }
    ptx::fence_mbar_init();
    ptx::prefetch_tmap(g.tmA);
    if (CG == 2) ptx::prefetch_tmap(g.tmW);
  }
  if (warp == 2) tmem_alloc<CG>(tmem_slot, ncols);
  tc::fence_before();
  __syncthreads();
  if (CG == 2) tc::cluster_sync();                           // the peer's barriers are initialised
  tc::fence_after();
  const uint32_t tmem = ptx::uniform(*tmem_slot);
  ptx::grid_dep_launch();
  const bool scaled = MODE != PF_PREFIX && MODE != PF_RESID && e.ssq_in != nullptr;
  bool failed = false;                                       // a bounded wait of this warp gave up
  const int per_z = g.tiles_m * g.tiles_n;
  auto tile_of = [&](int t, int& z, int& tm, int& tn) {
    z = MODE == PF_PREFIX ? t / per_z : 0;
    const int u = t - z * per_z;
    tn = u / g.tiles_m;
    tm = u - tn * g.tiles_m;
  };
  auto wait = [](uint64_t* bar, uint32_t parity) { return __all_sync(0xffffffffu, ptx::mbar_wait(bar, parity)) != 0; };
  if (warp == 0) {
    // ---- weights: they do not depend on the previous kernel and start before the dependency wait
    int st = 0, round = 0;                                   // stage, times the ring has been walked through
    for (int t = worker; t < g.tiles && !failed; t += workers) {
      int z, tm, tn;
      tile_of(t, z, tm, tn);
      // (an odd number of 128-feature tiles: the last pair's second CTA repeats the first one's weights and stores nothing)
      const int tw = CG == 2 ? min(CG * tm + rank, g.w_tiles - 1) : tm;
      const bf16* W = (MODE == PF_PREFIX ? e.layers[z].Wqkv : g.W) + (size_t)(g.w_tile0 + tw) * slabs * (tc::BM * tc::BK);
      const int w_row = CG == 2 ? (int)((W - g.w_base) / tc::BK) : 0;
      for (int s = 0; s < steps; ++s) {
        if (round > 0 && !wait(empty + st, (round - 1) & 1)) { failed = true; break; }
        if (ptx::elect_one()) {
          if (CG == 1) {
            const int bytes = min(SLABS, slabs - s * SLABS) * w_slab;
            ptx::mbar_expect_tx(full + st, bytes);
            ptx::bulk_load(sm + st * stage, W + (size_t)s * SLABS * (tc::BM * tc::BK), bytes, full + st);
          } else {                                           // (behind the last slab: whatever follows, never multiplied)
            if (rank == 0) ptx::mbar_expect_tx(full + st, CG * SLABS * w_slab);
            ptx::tma_load_2d_pair(sm + st * stage, g.tmW, 0, w_row + s * SLABS * tc::BM, tc::map_peer(ptx::smem_u32(full + st), 0));
          }
        }
        if (++st == ST) { st = 0; ++round; }
      }
    }
    // the last arrivals of the MMAs (the first CTA's, for both CTAs of a pair) land before this CTA leaves
    for (int i = 0; CG == 2 && i < ST && !failed; ++i) {
      const int uses = round + (i < st ? 1 : 0);
      if (uses > 0 && !wait(empty + i, (uses - 1) & 1)) failed = true;
    }
    if (failed) s_fail = 1;
  } else if (warp == 1) {
    // ---- operand rows: one copy brings the hi and lo tiles of a stage (zeros behind the last slab); of a pair, the first
    // CTA holds the hi and the second the lo tile (one term: half of the rows each)
    ptx::grid_dep_wait();
    int st = 0, round = 0;                                   // stage, times the ring has been walked through
    for (int t = worker; t < g.tiles && !failed; t += workers) {
      int z, tm, tn;
      tile_of(t, z, tm, tn);
      const int row = tn * NT + (MODE == PF_PREFIX ? z * e.rows_layer : 0) + (CG == 2 && PARTS == 1 ? rank * HN : 0);
      for (int s = 0; s < steps; ++s) {
        if (round > 0 && !wait(empty + st, (round - 1) & 1)) { failed = true; break; }
        if (ptx::elect_one()) {
          if (rank == 0) ptx::mbar_expect_tx(full + st, CG * SLABS * a_slab);
          unsigned char* dst = sm + st * stage + SLABS * w_slab;
          if (CG == 1) ptx::tma_load_4d(dst, g.tmA, 0, row, 0, s * SLABS, full + st);
          else ptx::tma_load_4d_pair(dst, g.tmA, 0, row, PARTS == 2 ? rank : 0, s * SLABS, tc::map_peer(ptx::smem_u32(full + st), 0));
        }
        if (++st == ST) { st = 0; ++round; }
      }
    }
    if (failed) s_fail = 1;
  } else if (warp == 2 && rank == 0) {
    // ---- MMA issuer
    const uint32_t idesc = tc::instr_desc_bf16(PARTS * NT, CG * tc::BM);
    int st = 0, round = 0, k = 0;
    for (int t = worker; t < g.tiles; t += workers, ++k) {
      const int buf = k & 1;
      if (k >= 2 && !(CG == 2 ? __all_sync(0xffffffffu, tc::mbar_wait_cluster(acc_empty + buf, ((k >> 1) - 1) & 1)) != 0 : wait(acc_empty + buf, ((k >> 1) - 1) & 1))) { failed = true; break; }
      tc::fence_after();
      for (int s = 0; s < steps; ++s) {
        const int n = min(SLABS, slabs - s * SLABS);
        if (!wait(full + st, round & 1)) { failed = true; break; }
        tc::fence_after();
        const uint32_t base = ptx::smem_u32(sm + st * stage);
        if (ptx::elect_one()) {
          for (int j = 0; j < n; ++j) {
            const uint64_t da = tc::smem_desc_sw128(base + j * w_slab), db = tc::smem_desc_sw128(base + SLABS * w_slab + j * a_slab);
#pragma unroll
            for (int kk = 0; kk < tc::BK / 16; ++kk)
              mma<CG>(tmem + buf * acc_cols, da + 2 * kk, db + 2 * kk, idesc, (s > 0 || j > 0 || kk > 0) ? 1u : 0u);
          }
          commit<CG>(empty + st);
          if (s == steps - 1) commit<CG>(acc_full + buf);
        }
        __syncwarp();
        if (++st == ST) { st = 0; ++round; }
      }
      if (failed) break;
    }
    if (failed) s_fail = 1;
  } else if (warp == 3 && scaled) {
    // ---- scales of the operand rows, a tile ahead of the epilogue (its own loads cost it 2 us a tile: nothing hides their latency there)
    ptx::grid_dep_wait();
    int k = 0;
    for (int t = worker; t < g.tiles; t += workers, ++k) {
      int z, tm, tn;
      tile_of(t, z, tm, tn);
      const int buf = k & 1, n0 = tn * NT, nrows = min(NT, g.R - n0);
      if (k >= 2 && !wait(inv_empty + buf, ((k >> 1) - 1) & 1)) { failed = true; break; }
      for (int r0 = 0; r0 < nrows; r0 += 32) {               // eight lanes add the partial sums of a row
        float ss[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        const float* sq = e.ssq_in + (size_t)(n0 + r0 + (lane >> 3)) * e.ld_ssq;
        const int rows = nrows - r0 - (lane >> 3);           // (the eight requests of a round travel together)
        if ((e.ssq_n & 3) == 0) {
          for (int s0 = 0; s0 < e.ssq_n; s0 += 32) {
            const int s = s0 + 4 * (lane & 7);
            float4 q[8];
#pragma unroll
            for (int i = 0; i < 8; ++i)
              q[i] = 4 * i < rows && s < e.ssq_n ? __ldcg(reinterpret_cast<const float4*>(sq + (size_t)4 * i * e.ld_ssq + s)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int i = 0; i < 8; ++i) ss[i] += (q[i].x + q[i].y) + (q[i].z + q[i].w);
          }
        } else {
          for (int s = lane & 7; s < e.ssq_n; s += 8)
#pragma unroll
            for (int i = 0; i < 8; ++i) ss[i] += 4 * i < rows ? __ldcg(sq + (size_t)4 * i * e.ld_ssq + s) : 0.f;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          ss[i] += __shfl_xor_sync(0xffffffffu, ss[i], 1);
          ss[i] += __shfl_xor_sync(0xffffffffu, ss[i], 2);
          ss[i] += __shfl_xor_sync(0xffffffffu, ss[i], 4);
          if ((lane & 7) == 0) s_inv[buf * 128 + r0 + 4 * i + (lane >> 3)] = rsqrtf(ss[i] * e.inv_d + e.eps);
        }
      }
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(inv_full + buf);
    }
    if (failed) s_fail = 1;
  } else if (warp >= 4) {
    // ---- epilogue: warp w reads tensor-memory lanes 32 (w mod 4) .. + 31 (a feature each); four warps share the rows, CW
    // at a time.  A warp turns its CW rows x 32 features in a scratch of its own: behind that a lane holds four
    // neighbouring features of rows tl, tl + 4, .., and everything it reads and writes is 8 or 16 bytes wide.
    const int w4 = warp & 3, tl = lane >> 3, f4 = 4 * (lane & 7);
    float* turn = s_turn + (warp - 4) * (CW * 32);
    ptx::grid_dep_wait();
    auto release = [&](int buf) {                            // this warp has read its share of the accumulator
      if (rank == 0) ptx::mbar_arrive(acc_empty + buf);
      else ptx::mbar_arrive_peer(tc::map_peer(ptx::smem_u32(acc_empty + buf), 0));
    };
    int k = 0;
    for (int t = worker; t < g.tiles; t += workers, ++k) {
      int z, tm, tn;
      tile_of(t, z, tm, tn);
      tm = CG * tm + rank;                                   // this CTA's tile of 128 features
      const int buf = k & 1, n0 = tn * NT, nrows = min(NT, g.R - n0);
      const int m = tm * tc::BM + w4 * 32 + f4;              // this lane's features m .. m + 3 (M is a multiple of 4 but for plain stores)
      const bool m_ok = m < g.M;
      const int c_first = CW * ((warp - 4) >> 2);
      // ---- under the tile's MMAs: residual values of the warp's first rows
      float4 gain = make_float4(1.f, 1.f, 1.f, 1.f);
      float4 x0[4];                                          // PF_RESID: residual values, PF_QKV: rotary angles of the lane's two pairs
      Row rw[4];
      const int dh = e.dm.dh, H = e.dm.H, Hkv = e.dm.Hkv;
      const int head = MODE == PF_QKV || MODE == PF_PREFIX ? m / dh : 0, f = m - head * dh;       // (the same head for the whole warp: dh is 64 or 128)
      const bool rotate = MODE == PF_QKV && head < H + Hkv && e.dm.theta != 0.f;
      auto load_x = [&](float4 (&x)[4], int c0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int n = c0 + tl + 4 * i;
          x[i] = e.add && n < nrows && m_ok ? __ldcg(reinterpret_cast<const float4*>(e.x + (size_t)(n0 + n) * e.ldx + m)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      };
      auto load_rows = [&](int c0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) rw[i] = e.rows[min(n0 + c0 + tl + 4 * i, g.R - 1)];
      };
      if (MODE == PF_RESID) {
        if (e.gain != nullptr && m_ok) gain = *reinterpret_cast<const float4*>(e.gain + m);
        load_x(x0, c_first);
      }
      if (MODE == PF_QKV) load_rows(c_first);
      if (!__all_sync(0xffffffffu, ptx::mbar_wait(acc_full + buf, (k >> 1) & 1))) { s_fail = 1; break; }
      tc::fence_after();
      float inv[2][4];
      if (scaled) {
        if (!__all_sync(0xffffffffu, ptx::mbar_wait(inv_full + buf, (k >> 1) & 1))) { s_fail = 1; break; }
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int i = 0; i < 4; ++i) inv[c][i] = s_inv[buf * 128 + ((c_first + c * 4 * CW + tl + 4 * i) & 127)];
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(inv_empty + buf);
      }
      if (c_first >= nrows && lane == 0) release(buf);       // nothing to read for this warp
#pragma unroll 1
      for (int c0 = c_first; c0 < nrows; c0 += 4 * CW) {
        if (MODE == PF_QKV) {
#pragma unroll
          for (int i = 0; i < 4; ++i) x0[i] = rotate ? *reinterpret_cast<const float4*>(e.rope + (size_t)rw[i].p * (dh >> 1) + (f >> 1)) : make_float4(1.f, 0.f, 1.f, 0.f);
        }
        {
          uint32_t r[CW];
          ld16(tmem + buf * acc_cols + ((uint32_t)(w4 * 32) << 16) + c0, r);
          if (PARTS == 2) {
            uint32_t r2[CW];
            ld16(tmem + buf * acc_cols + ((uint32_t)(w4 * 32) << 16) + NT + c0, r2);
            ld_wait();
#pragma unroll
            for (int j = 0; j < CW; ++j) turn[j * 32 + lane] = __uint_as_float(r[j]) + __uint_as_float(r2[j]);
          } else {
            ld_wait();
#pragma unroll
            for (int j = 0; j < CW; ++j) turn[j * 32 + lane] = __uint_as_float(r[j]);
          }
        }
        tc::fence_before();
        __syncwarp();
        if (c0 + 4 * CW >= nrows && lane == 0) release(buf); // this warp's share has been read
        const bool more = c0 + 4 * CW < nrows;
        float4 xn[4];                                        // of the next rows, under the work on these
        if (MODE == PF_RESID && more) load_x(xn, c0 + 4 * CW);
        float4 v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = *reinterpret_cast<const float4*>(turn + (tl + 4 * i) * 32 + f4);
        __syncwarp();                                        // the scratch may be written again
        if (scaled) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float s = c0 == c_first ? inv[0][i] : inv[1][i];
            v[i].x *= s; v[i].y *= s; v[i].z *= s; v[i].w *= s;
          }
        }
        if (MODE == PF_RESID) {
#pragma unroll
          for (int i = 0; i < 4; ++i) { v[i].x += x0[i].x; v[i].y += x0[i].y; v[i].z += x0[i].z; v[i].w += x0[i].w; x0[i] = xn[i]; }
        }
        int pb = 0, ps = 0;                                  // PF_PREFIX: sequence and prefix slot of the lane's first row
        if (MODE == PF_PREFIX) { const int r = e.row_first + n0 + c0 + tl; pb = r / e.dm.P; ps = r - pb * e.dm.P; }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int n = c0 + tl + 4 * i;
          const size_t row = (size_t)(n0 + n);
          const bool ok = n < nrows && m_ok;
          if (MODE == PF_F32) {
            float* o = reinterpret_cast<float*>(e.out) + row * e.ldo + m;
            if (ok && m + 3 < g.M) *reinterpret_cast<float4*>(o) = v[i];
            else if (ok) {                                   // the last columns of a width that is not a multiple of 4
              o[0] = v[i].x;
              if (m + 1 < g.M) o[1] = v[i].y;
              if (m + 2 < g.M) o[2] = v[i].z;
            }
          } else if (MODE == PF_GELU) {
            const float2 a = tc::gelu2(v[i].x, v[i].y), b = tc::gelu2(v[i].z, v[i].w);
            if (ok) tc::store_hi_lo4(reinterpret_cast<bf16*>(e.out) + row * e.ldo + m, a.x, a.y, b.x, b.y, e.lo_off);
          } else if (MODE == PF_RESID) {
            if (ok) {
              *reinterpret_cast<float4*>(e.x + row * e.ldx + m) = v[i];
              if (e.a_out != nullptr)
                tc::store_hi_lo4(e.a_out + row * e.lda + m, __fmul_rn(v[i].x, gain.x), __fmul_rn(v[i].y, gain.y), __fmul_rn(v[i].z, gain.z),
                             __fmul_rn(v[i].w, gain.w), e.lo_off);
            }
            if (e.ssq_out != nullptr) {                      // sum of squares over the warp's 32 features
              float ss = m_ok ? (v[i].x * v[i].x + v[i].y * v[i].y) + (v[i].z * v[i].z + v[i].w * v[i].w) : 0.f;
              ss += __shfl_xor_sync(0xffffffffu, ss, 1);
              ss += __shfl_xor_sync(0xffffffffu, ss, 2);
              ss += __shfl_xor_sync(0xffffffffu, ss, 4);
              if (f4 == 0 && n < nrows && tm < g.w_tiles) e.ssq_out[row * e.ld_ssq + tm * 4 + w4] = ss;
            }
          } else if (MODE == PF_QKV) {
            // Q and K heads are stored with their rotary pairs side by side
            const float4 cs = x0[i];
            float4 y = v[i];
            if (rotate) y = make_float4(v[i].x * cs.x - v[i].y * cs.y, v[i].y * cs.x + v[i].x * cs.y, v[i].z * cs.z - v[i].w * cs.w, v[i].w * cs.z + v[i].z * cs.w);
            bf16* o;
            bool there = ok;
            if (head < H) {
              o = e.q + row * (size_t)(H * dh) + m;
              y.x *= e.qscale; y.y *= e.qscale; y.z *= e.qscale; y.w *= e.qscale;
            } else {
              const bool is_k = head < H + Hkv;
              const int hk = head - H - (is_k ? 0 : Hkv);
              if (e.Kc == nullptr) o = (is_k ? e.kbuf : e.vbuf) + row * (size_t)(Hkv * dh) + hk * dh + f;
              else {
                there = ok && rw[i].b >= 0;
                o = (is_k ? e.Kc : e.Vc) + (size_t)((rw[i].b * Hkv + hk) * (e.dm.P + e.dm.cap[e.level]) + e.dm.P + rw[i].slot) * dh + f;
              }
            }
            if (there) *reinterpret_cast<uint2*>(o) = make_uint2(ptx::pack_bf16(y.x, y.y), ptx::pack_bf16(y.z, y.w));
          } else {  // PF_PREFIX
            const LayerPtr& L = e.layers[z];
            bf16* o = (head < Hkv ? L.K : L.V) + (size_t)((pb * Hkv + (head < Hkv ? head : head - Hkv)) * (e.dm.P + e.dm.cap[L.level]) + ps) * dh + f;
            if (ok) *reinterpret_cast<uint2*>(o) = make_uint2(ptx::pack_bf16(v[i].x, v[i].y), ptx::pack_bf16(v[i].z, v[i].w));
            for (ps += 4; ps >= e.dm.P; ps -= e.dm.P) ++pb;
          }
        }
        if (MODE == PF_QKV && more) load_rows(c0 + 4 * CW);
      }
    }
  }
  __syncwarp();
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (s_fail) {
    if (tid == 0) atomicExch(g.status, -5);
    ptx::drain_delay();                                      // stages already requested may still be landing
  }
  if (CG == 2) {                                             // the pair's MMAs read this CTA's shared memory
    tc::cluster_sync();
    tc::fence_after();
  }
  if (warp == 1) tmem_free<CG>(tmem, ncols);
}

// ------------------------------------------------------------------------------------------
// row-wise kernels
// ------------------------------------------------------------------------------------------
// (b, p, segment, cache slot) of every row of the three levels; grid (segments, 3)
__global__ void map_kernel(Dims dm, const Seg* __restrict__ segs, Row* m0, Row* m1, Row* m2) {
  const int l = blockIdx.y;
  const Seg& s = segs[blockIdx.x];
  Row* m = (l == 0 ? m0 : l == 1 ? m1 : m2) + s.r0[l];
  for (int i = threadIdx.x; i < s.n[l]; i += blockDim.x) m[i] = Row{s.b, s.p0[l] + i, (int)blockIdx.x, (s.p0[l] + i) % dm.cap[l]};
}

// operand row [hi | lo] of x * g and the row's sum of squares, four columns per thread and step
__device__ inline void entry_row(const float4* xr, int row, int d, const float* __restrict__ g, bf16* __restrict__ a,
                                 float* __restrict__ ssq, int ld_ssq) {
  __shared__ float sh[32];
  float ss = 0.f;
  for (int i = threadIdx.x; i < d / 4; i += blockDim.x) {
    const float4 v = xr[i];
    const float4 gg = g != nullptr ? reinterpret_cast<const float4*>(g)[i] : make_float4(1.f, 1.f, 1.f, 1.f);
    ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
    bf16* p = a + (size_t)row * 2 * d + 4 * i;
    tc::store_hi_lo2(p, __fmul_rn(v.x, gg.x), __fmul_rn(v.y, gg.y), d);
    tc::store_hi_lo2(p + 2, __fmul_rn(v.z, gg.z), __fmul_rn(v.w, gg.w), d);
  }
  ss = block_sum(ss, sh);
  if (threadIdx.x == 0) ssq[(size_t)row * ld_ssq] = ss;
}

__global__ void embed_kernel(Dims dm, SeqState st, const Row* __restrict__ rows, const int* __restrict__ prompt,
                             const int* __restrict__ prompt_off, const bf16* __restrict__ E, float* __restrict__ x,
                             const float* __restrict__ g, bf16* __restrict__ a, float* __restrict__ ssq, int ld_ssq) {
  ptx::grid_dep_launch();
  ptx::grid_dep_wait();
  const int row = blockIdx.x, d = dm.d;
  const Row r = rows[row];
  int tok = r.p == 0 ? dm.n_bins : prompt[prompt_off[r.b] + r.p - 1];
  if (tok < 0 || tok >= dm.V) {                      // never index outside the table
    if (threadIdx.x == 0) atomicExch(st.status, -1);
    tok = dm.n_bins + 2;
  }
  float4* xr = reinterpret_cast<float4*>(x + (size_t)row * d);
  const __nv_bfloat162* er = reinterpret_cast<const __nv_bfloat162*>(E + (size_t)tok * d);
  for (int i = threadIdx.x; i < d / 4; i += blockDim.x) {
    const float2 lo = __bfloat1622float2(er[2 * i]), hi = __bfloat1622float2(er[2 * i + 1]);
    xr[i] = make_float4(lo.x, lo.y, hi.x, hi.y);
  }
  entry_row(xr, row, d, g, a, ssq, ld_ssq);                  // every thread reads the columns it wrote
}

// operand rows of a shorten GEMM: row u of level `lu` <- hiddens 3u-2, 3u-1, 3u of the level below,
// from its residual rows or, before the segment, from the carry ring; grid (rows of the level, 3)
__global__ void gather_kernel(Dims dm, const Seg* __restrict__ segs, const Row* __restrict__ rows, int lu,
                              const float* x_low, const float* ring, bf16* __restrict__ out) {
  ptx::grid_dep_launch();
  ptx::grid_dep_wait();
  const int row = blockIdx.x, part = blockIdx.y, d = dm.d, lb = lu - 1, rs = fm_ring(lb);
  const Row r = rows[row];
  const Seg& s = segs[r.seg];
  const int pos = 3 * r.p - 2 + part;
  const float4* src = reinterpret_cast<const float4*>(pos >= s.p0[lb] ? x_low + (size_t)(s.r0[lb] + pos - s.p0[lb]) * d
                                                                      : ring + ((size_t)r.b * rs + ((pos + rs) % rs)) * d);
  bf16* o = out + (size_t)row * 6 * d + part * d;
  for (int i = threadIdx.x; i < d / 4; i += blockDim.x) {
    const float4 v = pos >= 0 ? __ldcg(src + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    tc::store_hi_lo2(o + 4 * i, v.x, v.y, 3 * d);
    tc::store_hi_lo2(o + 4 * i + 2, v.z, v.w, 3 * d);
  }
}

// x[row] (the pre-shorten hidden) += its parent's upsampled slot; the last hiddens and triples of a
// segment go into the carry rings for what comes after it; operand row and sum of squares for the stack
// above.  The parent of every row is a row of the same segment.
__global__ void upsample_kernel(Dims dm, const Seg* __restrict__ segs, const Row* __restrict__ rows, int level,
                                const float* tri, float* __restrict__ h_ring, float* __restrict__ tri_ring,
                                float* x, const float* __restrict__ g, bf16* __restrict__ a, float* __restrict__ ssq, int ld_ssq) {
  ptx::grid_dep_launch();
  ptx::grid_dep_wait();
  const int row = blockIdx.x, d = dm.d, rs = fm_ring(level), rsu = fm_ring(level + 1);
  const Row r = rows[row];
  const Seg& s = segs[r.seg];
  const int up = r.p / 3, slot = r.p - 3 * up;
  const float4* t = reinterpret_cast<const float4*>(tri + ((size_t)(s.r0[level + 1] + up - s.p0[level + 1]) * 3 + slot) * d);
  float4* xr = reinterpret_cast<float4*>(x + (size_t)row * d);
  float4* hr = r.p >= s.p0[level] + s.n[level] - rs ? reinterpret_cast<float4*>(h_ring + ((size_t)r.b * rs + r.p % rs) * d) : nullptr;
  // a triple is stored whole, by the block of its first child (its other children may lie behind the segment)
  float4* tr = slot == 0 && up >= s.p0[level + 1] + s.n[level + 1] - rsu ? reinterpret_cast<float4*>(tri_ring + ((size_t)r.b * rsu + up % rsu) * 3 * d) : nullptr;
  for (int i = threadIdx.x; i < d / 4; i += blockDim.x) {
    const float4 h = __ldcg(xr + i), u = __ldcg(t + i);
    if (hr != nullptr) hr[i] = h;
    if (tr != nullptr) { tr[i] = u; tr[d / 4 + i] = __ldcg(t + d / 4 + i); tr[d / 2 + i] = __ldcg(t + d / 2 + i); }
    xr[i] = make_float4(h.x + u.x, h.y + u.y, h.z + u.z, h.w + u.w);
  }
  entry_row(xr, row, d, g, a, ssq, ld_ssq);
}

// the residual row of a prompt's last position, as it enters the last layer of a stack (split node)
__global__ void stash_kernel(Dims dm, const Seg* __restrict__ segs, int level, const float* x, float* __restrict__ ring) {
  ptx::grid_dep_launch();
  ptx::grid_dep_wait();
  const Seg& s = segs[blockIdx.x];
  if (!s.last) return;
  const int k = s.n[level] - 1, p = s.p0[level] + k, rs = fm_ring(level);
  const float4* src = reinterpret_cast<const float4*>(x + (size_t)(s.r0[level] + k) * dm.d);
  float4* dst = reinterpret_cast<float4*>(ring + ((size_t)s.b * rs + p % rs) * dm.d);
  for (int i = threadIdx.x; i < dm.d / 4; i += blockDim.x) dst[i] = __ldcg(src + i);
}

// keys and values of the chunk -> cache, where its attention still needed entries that they replace
__global__ void cache_kernel(Dims dm, const Seg* __restrict__ segs, const Row* __restrict__ rows, int level, const bf16* kbuf,
                             const bf16* vbuf, bf16* __restrict__ Kc, bf16* __restrict__ Vc) {
  ptx::grid_dep_launch();
  ptx::grid_dep_wait();
  const int row = blockIdx.x, cap = dm.cap[level], kvw = dm.Hkv * dm.dh;
  const Row r = rows[row];
  const Seg& s = segs[r.seg];
  if (r.p < s.p0[level] + s.n[level] - cap) return;          // a later row of the segment takes this slot
  const int slots = dm.P + cap;
  for (int i = threadIdx.x; i < kvw / 8; i += blockDim.x) {
    const int hk = 8 * i / dm.dh, c = 8 * i - hk * dm.dh;
    const size_t to = (((size_t)r.b * dm.Hkv + hk) * slots + dm.P + r.slot) * dm.dh + c;
    *reinterpret_cast<uint4*>(Kc + to) = __ldcg(reinterpret_cast<const uint4*>(kbuf + (size_t)row * kvw) + i);
    *reinterpret_cast<uint4*>(Vc + to) = __ldcg(reinterpret_cast<const uint4*>(vbuf + (size_t)row * kvw) + i);
  }
}

// attention output and residual row of a prompt's last position -> row b of the decode buffers
__global__ void last_rows_kernel(Dims dm, const Seg* __restrict__ segs, const bf16* attn, const float* x,
                                 bf16* __restrict__ attn_out, float* __restrict__ x_out) {
  ptx::grid_dep_launch();
  ptx::grid_dep_wait();
  const Seg& s = segs[blockIdx.x];
  if (!s.last) return;
  const size_t row = s.r0[0] + s.n[0] - 1;
  const int hd = dm.H * dm.dh;
  for (int i = threadIdx.x; i < hd / 4; i += blockDim.x)
    reinterpret_cast<uint4*>(attn_out + (size_t)s.b * 2 * hd)[i] = __ldcg(reinterpret_cast<const uint4*>(attn + row * 2 * hd) + i);
  for (int i = threadIdx.x; i < dm.d / 4; i += blockDim.x)
    reinterpret_cast<float4*>(x_out + (size_t)s.b * dm.d)[i] = __ldcg(reinterpret_cast<const float4*>(x + row * dm.d) + i);
}

// state behind the prompt: the first main token is the argmax of the last position
__global__ void finish_kernel(Dims dm, SeqState st, const float* logits, const int* __restrict__ prompt,
                              const int* __restrict__ prompt_off) {
  ptx::grid_dep_launch();
  ptx::grid_dep_wait();
  const int b = blockIdx.x, n = st.plen[b];
  const Top2 t = block_top2(logits + (size_t)b * dm.Vpad, dm, n);
  for (int i = max(0, n - FM_HIST) + threadIdx.x; i < n; i += blockDim.x) st.hist[b * FM_HIST + (i & (FM_HIST - 1))] = prompt[prompt_off[b] + i];
  if (threadIdx.x == 0) { st.L[b] = n + 1; st.main_tok[b] = t.i1; }
}

// ------------------------------------------------------------------------------------------
// conditioning
// ------------------------------------------------------------------------------------------
// operand rows of the prefix projections: a[z][row] = bf16(rms(c_row) * g1 of layer z); grid (rows, layer groups)
__global__ void prefix_norm_kernel(const float* __restrict__ c, const LayerPtr* __restrict__ layers, int n_layers, int rows_layer,
                                   bf16* __restrict__ a, int d, float eps) {
  __shared__ float sh[32];
  const float* xr = c + (size_t)blockIdx.x * d;              // caller memory: only known to be float-aligned
  float ss = 0.f;
  for (int i = threadIdx.x; i < d / 4; i += blockDim.x) { const float4 v = make_float4(xr[4 * i], xr[4 * i + 1], xr[4 * i + 2], xr[4 * i + 3]); ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w; }
  ss = block_sum(ss, sh);
  const float inv = rsqrtf(ss / (float)d + eps);
  for (int i = threadIdx.x; i < d / 4; i += blockDim.x) {
    const float4 v = make_float4(xr[4 * i], xr[4 * i + 1], xr[4 * i + 2], xr[4 * i + 3]);
#pragma unroll 4
    for (int z = blockIdx.y; z < n_layers; z += gridDim.y) {
      const float4 g = reinterpret_cast<const float4*>(layers[z].g1)[i];
      uint2 o;
      o.x = ptx::pack_bf16(v.x * inv * g.x, v.y * inv * g.y);
      o.y = ptx::pack_bf16(v.z * inv * g.z, v.w * inv * g.w);
      *reinterpret_cast<uint2*>(a + ((size_t)z * rows_layer + blockIdx.x) * d + 4 * i) = o;
    }
  }
}

// ------------------------------------------------------------------------------------------
// attention
// ------------------------------------------------------------------------------------------
// Causal attention of a chunk's rows.  A CTA takes 128 query rows (eight warps of 16) of one segment and
// head; a producer warp streams first the cache entries of earlier chunks (prefix slots included),
// then the keys and values of the chunk itself through a ring of TMA stages.  The chunk's own entries
// come from the cache too, except where a windowed level's ring would give a slot to a new position
// while an earlier row of the chunk still needs the old one: then they come from the projection's
// output, and the cache is written afterwards.
struct Attn {
  Dims dm;
  const Seg* segs; const int2* tiles;        // (segment, first query row)
  int level;
  const bf16* q;                             // [rows, H*dh], rotated and scaled by log2(e)/sqrt(dh)
  const CUtensorMap *tmK, *tmV;              // cache as 2-D [B*Hkv*slots, dh], box C x 64
  const CUtensorMap *tmKn, *tmVn;            // the chunk's [rows, Hkv*dh], same box; null: they are in the cache already
  bf16* out;                                 // [rows, 2*H*dh] as [hi | lo]
  int* status;
};

// QW of the eight warps share a key, the others split the keys of a tile among them and are merged at
// the end: few rows then still make enough CTAs, each with a short chain of key steps.
template <int DH, int C, int QW>
struct AttnCfg {
  static constexpr int NW = 8, KW = NW / QW, STAGES = 3, SUB = C / KW < 64 ? C / KW : 64, HALVES = DH / 64;
  static_assert(SUB >= 16, "a warp takes at least 16 keys of a tile");
  static constexpr int ROWS = QW * 16;
  static constexpr int TILE = C * DH * 2, STAGE = 2 * TILE;
  static constexpr int BYTES = STAGES * STAGE + 64 + 1024;
  static constexpr int THREADS = (NW + 1) * 32;
};

// word t of the quad's lane c -> word c of its lane t
__device__ inline void quad_transpose(uint4& v, int t4) {
  const bool odd = t4 & 1, high = t4 & 2;
  uint32_t a = __shfl_xor_sync(0xffffffffu, odd ? v.x : v.y, 1), b = __shfl_xor_sync(0xffffffffu, odd ? v.z : v.w, 1);
  if (odd) { v.x = a; v.z = b; } else { v.y = a; v.w = b; }
  a = __shfl_xor_sync(0xffffffffu, high ? v.x : v.z, 2), b = __shfl_xor_sync(0xffffffffu, high ? v.y : v.w, 2);
  if (high) { v.x = a; v.y = b; } else { v.z = a; v.w = b; }
}

template <int DH, int C, int QW>
__global__ void __launch_bounds__(AttnCfg<DH, C, QW>::THREADS, DH == 64 ? 2 : 1) attn_kernel(const Attn a) {
  using CF = AttnCfg<DH, C, QW>;
  constexpr int NW = CF::NW, KS = DH / 16, SUB = CF::SUB, KW = CF::KW;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + CF::STAGES * CF::STAGE);
  uint64_t* empty = full + CF::STAGES;
  __shared__ int s_fail;
  const Dims& dm = a.dm;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t4 = lane & 3;
  const int h = blockIdx.x, hk = h / (dm.H / dm.Hkv), level = a.level;
  ptx::grid_dep_launch();
  // (segments and tiles were written before the pass)
  const int2 tile = a.tiles[blockIdx.y];
  const Seg& sg = a.segs[tile.x];
  const int b = sg.b, p0 = sg.p0[level], n = sg.n[level], r0 = sg.r0[level], q0 = tile.y, nq = min(CF::ROWS, n - q0);
  const int P = dm.P, cap = dm.cap[level], W = dm.window[level], slots = P + cap;
  const int used = P + min(cap, p0);                         // cache slots that earlier chunks have filled
  const bool linear = p0 <= cap;
  const int q_last = q0 + nq - 1, vis_lo = W > 0 ? max(0, p0 + q0 - W + 1) : 0;      // lowest position any row sees
  // key tiles: [0, tp) prefix (and what shares its last tile), [tc0, tc1) cache, [tn0, tn1) this chunk
  const int tc1 = (used + C - 1) / C, tp = min(tc1, (P + C - 1) / C);
  const int tc0 = linear ? max(tp, min(tc1, (P + vis_lo) / C)) : tp;
  const int tn0 = max(0, vis_lo - p0) / C, tn1 = q_last / C + 1;
  const int n_old = tp + tc1 - tc0, n_tiles = n_old + tn1 - tn0;
  if (threadIdx.x == 0) {
    s_fail = 0;
    for (int i = 0; i < CF::STAGES; ++i) { ptx::mbar_init(full + i, 1); ptx::mbar_init(empty + i, NW); }
    ptx::fence_mbar_init();
  }
  __syncthreads();
  if (warp == NW) {
    if (lane == 0) {
      auto issue = [&](int i) {
        const int st = i % CF::STAGES;
        unsigned char* Ks = sm + st * CF::STAGE;
        unsigned char* Vs = Ks + CF::TILE;
        ptx::mbar_expect_tx(full + st, CF::STAGE);
        const bool old = i < n_old, cached = old || a.tmKn == nullptr;
        const int row = !cached ? r0 + (tn0 + i - n_old) * C
                                : (b * dm.Hkv + hk) * slots + (i < tp ? i * C : old ? (tc0 + i - tp) * C : P + p0 + (tn0 + i - n_old) * C);
        const CUtensorMap* mk = cached ? a.tmK : a.tmKn;
        const CUtensorMap* mv = cached ? a.tmV : a.tmVn;
#pragma unroll
        for (int hf = 0; hf < CF::HALVES; ++hf) {
          const int x = cached ? hf * 64 : hk * DH + hf * 64;
          ptx::tma_load_2d(Ks + hf * C * 128, mk, x, row, full + st);
          ptx::tma_load_2d(Vs + hf * C * 128, mv, x, row, full + st);
        }
      };
      // Entries of the prefix and of earlier chunks were complete before this chunk's first launch: they are requested
      // before the dependency wait.  (Slots behind them in a shared tile may be written meanwhile; they are masked.)
      const int pre = min(n_old, CF::STAGES);
      for (int i = 0; i < pre; ++i) issue(i);
      ptx::grid_dep_wait();
      for (int i = pre; i < n_tiles; ++i) {
        if (i >= CF::STAGES && !ptx::mbar_wait(empty + i % CF::STAGES, ((i / CF::STAGES) - 1) & 1)) { s_fail = 1; break; }
        issue(i);
      }
    }
    __syncwarp();
  } else {
    ptx::grid_dep_wait();
    uint32_t qa[KS][4];
    const int qw = warp % QW, kw = warp / QW;
    const int w0 = q0 + qw * 16;                             // this warp's first query row of the segment
    const bool live = qw * 16 < nq;
    // A lane takes 16-byte chunks of its two rows, the quad transposes them into fragments.  (A 4-byte load per fragment
    // register asks L2 for every sector twice: 0.8 us a launch at 73 rows.)  All requests first: one L2 latency, not two.
    uint4 v[2][KS / 2];
#pragma unroll
    for (int hr = 0; hr < 2; ++hr) {
      const int i = w0 + g + hr * 8;
      const bf16* qp = a.q + ((size_t)(r0 + (i < q0 + nq ? i : q0)) * dm.H + h) * DH;      // (rows behind the tile: any row of it)
#pragma unroll
      for (int k = 0; k < KS / 2; ++k) v[hr][k] = __ldcg(reinterpret_cast<const uint4*>(qp) + 4 * k + t4);
    }
#pragma unroll
    for (int hr = 0; hr < 2; ++hr) {
      const bool ok = w0 + g + hr * 8 < q0 + nq;
#pragma unroll
      for (int k = 0; k < KS / 2; ++k) {
        quad_transpose(v[hr][k], t4);
        qa[2 * k][hr] = ok ? v[hr][k].x : 0u;
        qa[2 * k][2 + hr] = ok ? v[hr][k].y : 0u;
        qa[2 * k + 1][hr] = ok ? v[hr][k].z : 0u;
        qa[2 * k + 1][2 + hr] = ok ? v[hr][k].w : 0u;
      }
    }
    float o[DH / 8][4];
    float mrun[2] = {-INFINITY, -INFINITY}, lrun[2] = {0.f, 0.f};
#pragma unroll
    for (int i = 0; i < DH / 8; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
    const int wrap_q = p0 > 0 ? (p0 - 1) / cap : 0, wrap_r = p0 - 1 - wrap_q * cap;
    const int pr_lo = p0 + w0, pr_hi = pr_lo + 15;           // positions of the warp's rows
    for (int i = 0; i < n_tiles; ++i) {
      const int st = i % CF::STAGES;
      const bool old = i < n_old;
      const int k0 = old ? (i < tp ? i : tc0 + i - tp) * C : (tn0 + i - n_old) * C;    // first slot, or first chunk row
      if (!__all_sync(0xffffffffu, ptx::mbar_wait(full + st, (i / CF::STAGES) & 1))) { s_fail = 1; break; }
      const uint32_t Ks_u = ptx::smem_u32(sm + st * CF::STAGE), Vs_u = Ks_u + CF::TILE;
#pragma unroll 1
      for (int sub = kw; sub < C / SUB; sub += KW) {
        const int s_lo = k0 + sub * SUB, s_hi = s_lo + SUB - 1;
        bool skip, all_vis;
        if (old) {
          skip = s_lo >= used || (linear && s_lo >= P && W > 0 && s_hi - P < pr_lo - W + 1);
          all_vis = s_hi < P || (linear && s_hi < used && (W == 0 || max(s_lo - P, 0) >= pr_hi - W + 1));
        } else {
          skip = p0 + s_lo > pr_hi || (W > 0 && p0 + s_hi < pr_lo - W + 1);
          all_vis = p0 + s_hi <= pr_lo && (W == 0 || p0 + s_lo >= pr_hi - W + 1);
        }
        if (skip || !live) continue;                         // the same for the whole warp
        float s[SUB / 8][4];
#pragma unroll
        for (int nt = 0; nt < SUB / 8; ++nt) s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
#pragma unroll
        for (int kb = 0; kb < SUB / 16; ++kb)
#pragma unroll
          for (int ks = 0; ks < KS; ++ks) {
            const int key = sub * SUB + kb * 16 + (lane & 7) + (lane >> 4) * 8;
            const int ch = ks * 2 + ((lane >> 3) & 1);
            uint32_t b0, b1, b2, b3;
            ptx::ldmatrix_x4(b0, b1, b2, b3, Ks_u + (ch >> 3) * C * 128 + ptx::swz128(key, ch & 7));
            ptx::mma_bf16_16816(s[2 * kb], qa[ks], b0, b1);
            ptx::mma_bf16_16816(s[2 * kb + 1], qa[ks], b2, b3);
          }
        if (!all_vis) {
#pragma unroll
          for (int nt = 0; nt < SUB / 8; ++nt)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const int k = s_lo + nt * 8 + 2 * t4 + e;      // slot or chunk row
              int kp;                                        // its position; -1 prefix, -2 nothing there
              if (old) {
                const int r = k - P;
                kp = k < P ? -1 : (k >= used ? -2 : (linear ? r : r + (r <= wrap_r ? wrap_q : wrap_q - 1) * cap));
              } else {
                kp = p0 + k;
              }
#pragma unroll
              for (int hr = 0; hr < 2; ++hr) {
                const int pr = pr_lo + g + hr * 8;
                const bool vis = kp == -1 || (kp >= 0 && kp <= pr && (W == 0 || kp >= pr - W + 1));
                if (!vis) s[nt][hr * 2 + e] = -INFINITY;
              }
            }
        }
        float scale[2], base[2];
#pragma unroll
        for (int hr = 0; hr < 2; ++hr) {
          float mx = -INFINITY;
#pragma unroll
          for (int nt = 0; nt < SUB / 8; ++nt) mx = fmaxf(mx, fmaxf(s[nt][hr * 2], s[nt][hr * 2 + 1]));
          mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
          mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
          const float mnew = fmaxf(mrun[hr], mx);
          base[hr] = mnew == -INFINITY ? 0.f : mnew;
          scale[hr] = mnew == mrun[hr] ? 1.f : exp2f(mrun[hr] - base[hr]);
          mrun[hr] = mnew;
        }
        float ls[2] = {0.f, 0.f};
#pragma unroll
        for (int nt = 0; nt < SUB / 8; ++nt)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            s[nt][e] = exp2f(s[nt][e] - base[e >> 1]);
            ls[e >> 1] += s[nt][e];
          }
#pragma unroll
        for (int hr = 0; hr < 2; ++hr) lrun[hr] = lrun[hr] * scale[hr] + ls[hr];     // per lane; the quad is added at the end
        if (__any_sync(0xffffffffu, scale[0] != 1.f || scale[1] != 1.f)) {
#pragma unroll
          for (int i2 = 0; i2 < DH / 8; ++i2) {
            o[i2][0] *= scale[0]; o[i2][1] *= scale[0];
            o[i2][2] *= scale[1]; o[i2][3] *= scale[1];
          }
        }
#pragma unroll
        for (int kb = 0; kb < SUB / 16; ++kb) {
          uint32_t pa[4];
          pa[0] = ptx::pack_bf16(s[2 * kb][0], s[2 * kb][1]);
          pa[1] = ptx::pack_bf16(s[2 * kb][2], s[2 * kb][3]);
          pa[2] = ptx::pack_bf16(s[2 * kb + 1][0], s[2 * kb + 1][1]);
          pa[3] = ptx::pack_bf16(s[2 * kb + 1][2], s[2 * kb + 1][3]);
#pragma unroll
          for (int dp = 0; dp < DH / 16; ++dp) {
            const int key = sub * SUB + kb * 16 + (lane & 7) + ((lane >> 3) & 1) * 8;
            const int ch = dp * 2 + (lane >> 4);
            uint32_t b0, b1, b2, b3;
            ptx::ldmatrix_x4_trans(b0, b1, b2, b3, Vs_u + (ch >> 3) * C * 128 + ptx::swz128(key, ch & 7));
            ptx::mma_bf16_16816(o[2 * dp], pa, b0, b1);
            ptx::mma_bf16_16816(o[2 * dp + 1], pa, b2, b3);
          }
        }
      }
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(empty + st);
    }
#pragma unroll
    for (int hr = 0; hr < 2; ++hr) {
      lrun[hr] += __shfl_xor_sync(0xffffffffu, lrun[hr], 1);
      lrun[hr] += __shfl_xor_sync(0xffffffffu, lrun[hr], 2);
    }
    if (KW == 1) {
#pragma unroll
      for (int hr = 0; hr < 2; ++hr) {
        const float inv = 1.f / lrun[hr];
        const int i = g + hr * 8;
        if (qw * 16 + i < nq) {
          bf16* op = a.out + ((size_t)(r0 + w0 + i) * 2 * dm.H + h) * DH;
#pragma unroll
          for (int c = 0; c < DH / 8; ++c) tc::store_hi_lo2(op + c * 8 + 2 * t4, o[c][hr * 2] * inv, o[c][hr * 2 + 1] * inv, dm.H * DH);
        }
      }
    } else {
      asm volatile("bar.sync 1, 256;" ::: "memory");         // the compute warps are done with the ring
      float* mine = reinterpret_cast<float*>(sm) + warp * 16 * (DH + 2);      // [16][DH + 2]: output, maximum, sum
#pragma unroll
      for (int hr = 0; hr < 2; ++hr) {
        float* row = mine + (g + hr * 8) * (DH + 2);
#pragma unroll
        for (int c = 0; c < DH / 8; ++c) *reinterpret_cast<float2*>(row + c * 8 + 2 * t4) = make_float2(o[c][hr * 2], o[c][hr * 2 + 1]);
        if (t4 == 0) { row[DH] = mrun[hr]; row[DH + 1] = lrun[hr]; }
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
      const float* base = reinterpret_cast<const float*>(sm);
      for (int e = threadIdx.x; e < nq * (DH / 2); e += NW * 32) {
        const int i = e / (DH / 2), c = 2 * (e - i * (DH / 2));
        const float* row = base + ((i >> 4) * 16 + (i & 15)) * (DH + 2);
        float m = -INFINITY;
#pragma unroll
        for (int k = 0; k < KW; ++k) m = fmaxf(m, row[k * QW * 16 * (DH + 2) + DH]);
        float l = 0.f, o0 = 0.f, o1 = 0.f;
#pragma unroll
        for (int k = 0; k < KW; ++k) {
          const float* r = row + k * QW * 16 * (DH + 2);
          const float w = r[DH] == -INFINITY ? 0.f : exp2f(r[DH] - m);
          l += w * r[DH + 1];
          o0 += w * r[c];
          o1 += w * r[c + 1];
        }
        const float inv = 1.f / l;
        tc::store_hi_lo2(a.out + ((size_t)(r0 + q0 + i) * 2 * dm.H + h) * DH + c, o0 * inv, o1 * inv, dm.H * DH);
      }
    }
  }
  __syncthreads();
  if (s_fail) {                                              // a bounded wait gave up: report
    if (threadIdx.x == 0) atomicExch(a.status, -5);
    ptx::drain_delay();
  }
}


// The same for many rows and heads of 64, on the tensor cores: a CTA takes 128 query rows of a head, two threads per
// row.  S = Q K^T goes to tensor memory; a thread reads its half of a row once, the two exchange maxima, and P
// (bfloat16) goes back to tensor memory as the A operand of O += P V.  V is multiplied as it lies (keys x features: the
// B operand's MN-major form).  S of the next tile is multiplied as soon as S is in registers, i.e. under the
// exponentials.  The output is rescaled only when a row's maximum has grown by more than 2^8 (the conditional rescaling of
// FlashAttention-4, T. Dao et al., Hot Chips 2025).  Nearest bound: the special-function units (1024 clocks for a tile's
// exponentials, which two CTAs per SM share; 65 % of their rate in use), beside them the issue slots of the softmax warps: hence
// sums and differences in pairs, maxima of three, one barrier a tile.  6994 rows, 16 heads: 180 us a launch (187 without these,
// 201 with copies and MMAs issued behind `lane == 0`; MMAs of warps, attn_kernel: 505 us; a thread per row without the overlap: 462 us).
namespace fa {
constexpr int THREADS = 320;     // producer warp, MMA warp, eight softmax warps
constexpr int STAGES = 2, TILE = 128 * 128, STAGE = 2 * TILE;            // bytes of 128 keys (or values) of 64
constexpr int BYTES = TILE + STAGES * STAGE + 512 * 4 + 128 + 1024;
constexpr float GROW = 8.f;

__device__ inline float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ inline uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ inline float2 unpack2(uint64_t r) {
  float2 v;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(r));
  return v;
}
__device__ inline uint64_t add2(uint64_t a, uint64_t b) {              // two sums in one instruction
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ inline float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ inline void st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15};" ::"r"(r[0]), "r"(r[1]),
               "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]),
               "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(taddr)
               : "memory");
}
__device__ inline void st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ inline void mma_ts(uint32_t d, uint32_t a, uint64_t db, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
      "r"(a), "l"(db), "r"(idesc), "r"(accumulate)
      : "memory");
}
}  // namespace fa

__global__ void __launch_bounds__(fa::THREADS, 2) attn_tc_kernel(const Attn a, const CUtensorMap* tmQ) {
  using namespace fa;
  constexpr int DH = 64, C = 128;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  unsigned char* ring = sm + TILE;                           // behind the query tile
  float* s_pair = reinterpret_cast<float*>(ring + STAGES * STAGE);         // [tile mod 2][half][row]
  uint64_t* full = reinterpret_cast<uint64_t*>(s_pair + 512);
  uint64_t *empty = full + STAGES, *q_full = empty + STAGES, *s_full = q_full + 1, *s_read = s_full + 1, *p_full = s_read + 1, *o_full = p_full + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(o_full + 1);
  __shared__ int s_fail;
  const Dims& dm = a.dm;
  const int warp = (int)ptx::uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int h = blockIdx.x, hk = h / (dm.H / dm.Hkv), level = a.level;
  const int2 tile = a.tiles[blockIdx.y];
  const Seg& sg = a.segs[tile.x];
  const int b = sg.b, p0 = sg.p0[level], n = sg.n[level], r0 = sg.r0[level], q0 = tile.y, nq = min(128, n - q0);
  const int P = dm.P, cap = dm.cap[level], W = dm.window[level], slots = P + cap;
  const int used = P + min(cap, p0);                         // cache slots that earlier chunks have filled
  const bool linear = p0 <= cap;
  const int q_last = q0 + nq - 1, vis_lo = W > 0 ? max(0, p0 + q0 - W + 1) : 0;      // lowest position any row sees
  // key tiles, as in attn_kernel: prefix, cache, this chunk
  const int tc1 = (used + C - 1) / C, tp = min(tc1, (P + C - 1) / C);
  const int tc0 = linear ? max(tp, min(tc1, (P + vis_lo) / C)) : tp;
  const int tn0 = max(0, vis_lo - p0) / C, tn1 = q_last / C + 1;
  const int n_old = tp + tc1 - tc0, n_tiles = n_old + tn1 - tn0;
  if (threadIdx.x == 0) {
    s_fail = 0;
    for (int i = 0; i < STAGES; ++i) { ptx::mbar_init(full + i, 1); ptx::mbar_init(empty + i, 1); }
    ptx::mbar_init(q_full, 1); ptx::mbar_init(s_full, 1); ptx::mbar_init(s_read, 8); ptx::mbar_init(p_full, 8); ptx::mbar_init(o_full, 1);
    ptx::fence_mbar_init();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(ptx::smem_u32(tmem_slot)), "r"(256) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = ptx::uniform(*tmem_slot), tO = tmem + 128, tP = tmem + 192;        // S in columns 0..127, then O, then P
  ptx::grid_dep_launch();
  auto wait = [](uint64_t* bar, uint32_t parity) { return __all_sync(0xffffffffu, ptx::mbar_wait(bar, parity)) != 0; };
  if (warp == 0) {
    auto issue = [&](int i) {
      if (!ptx::elect_one()) return;
      const int st = i % STAGES;
      const bool old = i < n_old, cached = old || a.tmKn == nullptr;
      const int row = !cached ? r0 + (tn0 + i - n_old) * C
                              : (b * dm.Hkv + hk) * slots + (i < tp ? i * C : old ? (tc0 + i - tp) * C : P + p0 + (tn0 + i - n_old) * C);
      const int x = cached ? 0 : hk * DH;
      ptx::mbar_expect_tx(full + st, STAGE);
      ptx::tma_load_2d(ring + st * STAGE, cached ? a.tmK : a.tmKn, x, row, full + st);
      ptx::tma_load_2d(ring + st * STAGE + TILE, cached ? a.tmV : a.tmVn, x, row, full + st);
    };
    const int pre = min(n_old, STAGES);                      // as in attn_kernel: old entries before the dependency wait
    for (int i = 0; i < pre; ++i) issue(i);
    ptx::grid_dep_wait();
    if (ptx::elect_one()) {
      ptx::mbar_expect_tx(q_full, TILE);
      ptx::tma_load_2d(sm, tmQ, h * DH, r0 + q0, q_full);
    }
    for (int i = pre; i < n_tiles; ++i) {
      if (i >= STAGES && !wait(empty + i % STAGES, ((i / STAGES) - 1) & 1)) { s_fail = 1; break; }
      issue(i);
    }
  } else if (warp == 1) {
    const uint32_t id_s = tc::instr_desc_bf16(128), id_o = tc::instr_desc_bf16(DH) | (1u << 16);       // B of P V is MN-major
    const uint64_t dq = tc::smem_desc_sw128(ptx::smem_u32(sm));
    bool ok = wait(q_full, 0);
    auto scores = [&](int i) {
      const int st = i % STAGES;
      if (!wait(full + st, (i / STAGES) & 1)) return false;
      tc::fence_after();
      const uint64_t dk = tc::smem_desc_sw128(ptx::smem_u32(ring + st * STAGE));
      if (ptx::elect_one()) {
#pragma unroll
        for (int k = 0; k < DH / 16; ++k) tc::mma_ss(tmem, dq + 2 * k, dk + 2 * k, id_s, k > 0 ? 1u : 0u);
        tc::commit(s_full);
      }
      return true;
    };
    ok = ok && scores(0);
    for (int i = 0; i < n_tiles && ok; ++i) {
      if (!(ok = wait(s_read, i & 1))) break;
      if (i + 1 < n_tiles && !(ok = scores(i + 1))) break;
      if (!(ok = wait(p_full, i & 1))) break;
      tc::fence_after();
      const uint64_t dv = tc::smem_desc_sw128(ptx::smem_u32(ring + (i % STAGES) * STAGE + TILE));
      if (ptx::elect_one()) {
#pragma unroll
        for (int k = 0; k < C / 16; ++k) mma_ts(tO, tP + 8 * k, dv + 128 * k, id_o, (i > 0 || k > 0) ? 1u : 0u);
        tc::commit(empty + i % STAGES);
        tc::commit(o_full);
      }
    }
    if (!ok) {
      s_fail = 1;
      if (ptx::elect_one()) tc::commit(q_full);              // what was issued ends before the CTA does
      wait(q_full, 1);
    }
  } else if (warp >= 2) {
    // ---- softmax: warps w and w + 4 share 32 query rows, 64 of a tile's keys each
    const int w4 = warp & 3, half = (warp - 2) >> 2, i_row = w4 * 32 + lane;
    const uint32_t lanes = (uint32_t)(w4 * 32) << 16;
    const int pr = p0 + q0 + i_row;                          // the row's position
    const int wrap_q = p0 > 0 ? (p0 - 1) / cap : 0, wrap_r = p0 - 1 - wrap_q * cap;
    float m = -INFINITY, l = 0.f;                            // the maximum in use, the sum
    bool ok = true;
    for (int i = 0; i < n_tiles; ++i) {
      const bool old = i < n_old;
      const int k0 = old ? (i < tp ? i : tc0 + i - tp) * C : (tn0 + i - n_old) * C, k1 = k0 + C - 1;     // slots, or chunk rows
      // every key of the tile visible to every row of the tile?
      const bool all_vis = old ? k1 < P || (linear && k1 < used && (W == 0 || max(k0 - P, 0) >= p0 + q_last - W + 1))
                               : k1 <= q0 && (W == 0 || p0 + k0 >= p0 + q_last - W + 1);
      auto visible = [&](int k) {                            // slot or chunk row k
        int kp;
        if (old) {
          const int r = k - P;
          if (k < P) return true;
          if (k >= used) return false;
          kp = linear ? r : r + (r <= wrap_r ? wrap_q : wrap_q - 1) * cap;
        } else {
          kp = p0 + k;
        }
        return kp >= 0 && kp <= pr && (W == 0 || kp >= pr - W + 1);
      };
      ok = ok && __all_sync(0xffffffffu, ptx::mbar_wait(s_full, i & 1));             // (goes on: its partner waits at the barrier)
      tc::fence_after();
      uint32_t r0[32], r1[32];
      const int kh = k0 + 64 * half;
      ld32(tmem + lanes + 64 * half, r0);
      ld32(tmem + lanes + 64 * half + 32, r1);
      ld_wait();
      tc::fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(s_read);
      if (!all_vis) {
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          if (!visible(kh + j)) r0[j] = 0xff800000u;         // -inf: exponential 0
          if (!visible(kh + 32 + j)) r1[j] = 0xff800000u;
        }
      }
      float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int j = 0; j < 32; j += 4) {
        m4[0] = max3(m4[0], __uint_as_float(r0[j]), __uint_as_float(r0[j + 1])); m4[1] = max3(m4[1], __uint_as_float(r0[j + 2]), __uint_as_float(r0[j + 3]));
        m4[2] = max3(m4[2], __uint_as_float(r1[j]), __uint_as_float(r1[j + 1])); m4[3] = max3(m4[3], __uint_as_float(r1[j + 2]), __uint_as_float(r1[j + 3]));
      }
      float mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
      float* pair = s_pair + (i & 1) * 256;                  // (two of them: written again behind the next tile's barrier)
      pair[half * 128 + i_row] = mx;
      asm volatile("bar.sync %0, 64;" ::"r"(1 + w4) : "memory");
      mx = fmaxf(mx, pair[(half ^ 1) * 128 + i_row]);
      // P of the tile before has been multiplied: its place, and O, are free
      if (i > 0) ok = ok && __all_sync(0xffffffffu, ptx::mbar_wait(o_full, (i - 1) & 1));
      tc::fence_after();
      const bool grow = mx > m + GROW || (m == -INFINITY && mx != -INFINITY);
      if (__any_sync(0xffffffffu, grow)) {
        const float mn = grow ? mx : m, f = m == -INFINITY ? (grow ? 0.f : 1.f) : ex2(m - mn);
        m = mn;
        l *= f;
        if (i > 0) {                                         // this half's 32 columns of the output
#pragma unroll 1
          for (int c = 0; c < 2; ++c) {
            uint32_t o[16];
            tc::ld16(tO + lanes + 32 * half + 16 * c, o);
#pragma unroll
            for (int j = 0; j < 16; ++j) o[j] = __float_as_uint(__uint_as_float(o[j]) * f);
            st16(tO + lanes + 32 * half + 16 * c, o);
          }
        }
      }
      const float base = m == -INFINITY ? 0.f : m;
      const uint64_t nb = pack2(-base, -base);
      uint64_t s2[2] = {0ull, 0ull};
      uint32_t pk[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float2 d = unpack2(add2(pack2(__uint_as_float(r0[2 * j]), __uint_as_float(r0[2 * j + 1])), nb));
        const float e0 = ex2(d.x), e1 = ex2(d.y);
        s2[0] = add2(s2[0], pack2(e0, e1));
        pk[j] = ptx::pack_bf16(e0, e1);
      }
      st16(tP + lanes + 32 * half, pk);
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float2 d = unpack2(add2(pack2(__uint_as_float(r1[2 * j]), __uint_as_float(r1[2 * j + 1])), nb));
        const float e0 = ex2(d.x), e1 = ex2(d.y);
        s2[1] = add2(s2[1], pack2(e0, e1));
        pk[j] = ptx::pack_bf16(e0, e1);
      }
      st16(tP + lanes + 32 * half + 16, pk);
      const float2 sa = unpack2(s2[0]), sb = unpack2(s2[1]);
      l += (sa.x + sa.y) + (sb.x + sb.y);
      st_wait();
      tc::fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(p_full);
    }
    float* pair = s_pair + (n_tiles & 1) * 256;
    pair[half * 128 + i_row] = l;
    asm volatile("bar.sync %0, 64;" ::"r"(1 + w4) : "memory");
    l += pair[(half ^ 1) * 128 + i_row];
    ok = ok && __all_sync(0xffffffffu, ptx::mbar_wait(o_full, (n_tiles - 1) & 1));
    if (!ok) s_fail = 1;
    else {
      tc::fence_after();
      const float inv = 1.f / l;
      bf16* op = a.out + ((size_t)(r0 + q0 + i_row) * 2 * dm.H + h) * DH;
      uint32_t r[32];
      ld32(tO + lanes + 32 * half, r);
      ld_wait();
      if (i_row < nq) {
#pragma unroll
        for (int j = 0; j < 32; j += 8) {
          uint32_t hi[4], lo[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float x = __uint_as_float(r[j + 2 * k]) * inv, y = __uint_as_float(r[j + 2 * k + 1]) * inv;
            const __nv_bfloat162 hv = __floats2bfloat162_rn(x, y);
            hi[k] = *reinterpret_cast<const uint32_t*>(&hv);
            lo[k] = ptx::pack_bf16(__fsub_rn(x, __bfloat162float(hv.x)), __fsub_rn(y, __bfloat162float(hv.y)));
          }
          *reinterpret_cast<uint4*>(op + 32 * half + j) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
          *reinterpret_cast<uint4*>(op + dm.H * DH + 32 * half + j) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
      }
    }
  }
  __syncwarp();
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (s_fail) {                                              // a bounded wait gave up: report
    if (threadIdx.x == 0) atomicExch(a.status, -5);
    ptx::drain_delay();
  }
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256) : "memory");
}

}  // namespace pf
