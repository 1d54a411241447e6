// The projections of a pass with few rows (up to 16), one launch without any exchange between CTAs.
//
//   y[n][m] = sum_k W[m, k] A[n, k]
//
// With few rows a launch is a chain of latencies, not a stream: the weights are on chip before the
// previous kernel has ended, and what counts is the time from its end to the last store.  So a CTA owns
// FT output features (8, 16 or 32) with their whole K range: its weights come into shared memory
// by bulk copies before the dependency wait; behind it every warp reads its share of K of the operand
// rows from L2 straight into the registers of warp MMAs (no copy engine, no tensor memory), the warps'
// partial tiles are added through shared memory in warp order, and the epilogue follows.  (The tensor-memory
// form with K split over a cluster, fm_gemm_tc.cuh, spends 0.8 us on the operand copy, 0.5 us on the
// round trip through tensor memory and 1 us on the exchange between the CTAs, and hardly more for more rows.)  From one
// launch's dependency wait to the next one's, d = 1024, 2 rows, here / there: QKV 3.2 / 3.3 us, output projection 2.5 / 3.7, first
// FFN matrix 3.3 / 3.5, second 4.0 / 5.6; more rows at rows_cut in flashmesh.cu.
//
// The token rows are the MMA's M axis: the hi terms of the R rows, then their lo terms, so 10 rows with two
// terms take 20 of 32 MMA rows.  Eight features are the N axis.  Within a block of 32 k, lane t of a quad
// holds k = 8t .. 8t + 7 of its row (one 16-byte load) and serves two MMA steps with it, four k each;
// the weights' lanes do the same, so the MMAs see a permuted but consistent order of k.
//
// 256 threads of at most 128 registers (80 were slower: 4.4 against 3.9 us per launch) and as a rule at most
// 64 KB of shared memory: the next launch's CTA, with its weights, fits beside this one.
#pragma once
#include "fm_common.cuh"
#include "fm_gemm_tc.cuh"
#include "fm_ptx.cuh"

namespace rg {

constexpr int MAX_ROWS = 16;
constexpr int THREADS = 256, NW = THREADS / 32;

struct Args {
  const bf16* W;                 // packed weight slabs (see fm_gemm_tc.cuh)
  const bf16* A; int lda;        // operand rows [.., parts * K]
  int M, K, R, parts;            // R: rows per problem
  int w_tile0, a_row0;
  int z_rows, z_w_tiles;         // blockIdx.y: stacked problem z uses weight tiles from w_tile0 + z*z_w_tiles, rows from z*z_rows
  const int* n_active;           // skip when *n_active == 0 (may be null)
  int* status;
};

inline __host__ __device__ int red_stride(int FT) { return FT == 8 ? 8 : FT + 8; }          // floats; conflict-free quad stores
inline int smem_bytes(int FT, int K, int mtn) {
  const int w = FT * K * 2, r = NW * mtn * 16 * red_stride(FT) * 4;
  return (w > r ? w : r) + 128;
}

// D[16 x 8] += A[16 x 16] B[16 x 8] (not volatile: the compiler may interleave independent ones)
__device__ inline void mma(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

template <int MODE, int MTN, int FJ>
__global__ void __launch_bounds__(THREADS, 2) gemm_rows_kernel(const Args g, const tc::Epi e) {
  using namespace tc;
  constexpr int FT = FJ * 8, PAIRS = FT / 2, S = FT == 8 ? 8 : FT + 8;
  constexpr bool IS_RESID = MODE == EPI_RESID || MODE == EPI_RESID_CAT;
  constexpr bool ROW_MAPS = MODE == EPI_QKV || MODE == EPI_RESID_CAT || MODE == EPI_UP;
  constexpr bool SCALED = MODE != EPI_UP && !IS_RESID;
  constexpr int CARRY_MAX = MODE == EPI_UP ? 128 : 1;
  if (g.n_active != nullptr && *g.n_active == 0) {           // the whole grid leaves; keep the launch chain ordered
    ptx::grid_dep_launch();
    ptx::grid_dep_wait();
    return;
  }
  extern __shared__ __align__(128) unsigned char sm[];
  float* red = reinterpret_cast<float*>(sm);                 // [warp][MTN * 16][S], over the weights once they are used up
  __shared__ uint64_t full;
  __shared__ float s_inv[MAX_ROWS];
  __shared__ int s_rb[MAX_ROWS], s_rp[MAX_ROWS], s_ra[MAX_ROWS], s_rl[MAX_ROWS];
  __shared__ int s_carry[CARRY_MAX], s_ncarry;
  const int tid = threadIdx.x, warp = (int)ptx::uniform(tid >> 5), lane = tid & 31, gq = lane >> 2, t4 = lane & 3;
  const int f0 = blockIdx.x * FT, slabs = g.K / BK, R = g.R;
  const int row0 = e.row0 + (int)blockIdx.y * g.z_rows;      // first output row
  if (tid == 0) {
    ptx::mbar_init(&full, 1);
    ptx::fence_mbar_init();
    ptx::mbar_expect_tx(&full, (uint32_t)(FT * g.K * 2));
  }
  if (warp == 0) {
    __syncwarp();
    const bf16* src = g.W + ((size_t)(g.w_tile0 + (int)blockIdx.y * g.z_w_tiles + f0 / BM) * slabs * BM + f0 % BM) * BK;
    if (ptx::elect_one())                                    // (one lane of a warp in step: the copies' operands stay in uniform registers)
      for (int s = 0; s < slabs; ++s) ptx::bulk_load(sm + s * FT * 128, src + (size_t)s * (BM * BK), FT * 128, &full);
    __syncwarp();
  }
  ptx::grid_dep_launch();
  // ---- what does not depend on the previous kernel: row maps (positions are per-pass state), the first item's gain and angle
  if (ROW_MAPS && warp == 1 && lane < R) {
    int b = 0, p = 0;
    const bool valid = row_of(e, row0 + lane, b, p);
    s_rb[lane] = valid ? b : -1;
    s_rp[lane] = p;
    if ((MODE == EPI_RESID_CAT || MODE == EPI_UP) && valid) {
      // first position of the sequence at the other level of the pair, last position at the lower one
      const int Lb = e.st.L[b], nr = e.st.nrow[b];
      const int rl = fm_ratio(MODE == EPI_UP ? e.level - 1 : e.level), ru = 3 * rl;
      s_ra[lane] = MODE == EPI_UP ? (Lb + rl - 1) / rl : (Lb + ru - 1) / ru;
      s_rl[lane] = (Lb + nr - 1) / rl;
    }
  }
  if (MODE == EPI_UP && warp == 2 && lane == 0) {
    // child rows of this tile's slot whose parent was computed in an earlier pass
    const int lvl = e.level - 1, rl = fm_ratio(lvl), m_low = fm_rows_per_seq(e.dm, lvl), slot = f0 / e.d_model;
    int cnt = 0;
    for (int b = 0; b < e.batch; ++b) {
      const int nr = e.st.nrow[b], Lb = e.st.L[b];
      if (nr <= 0) continue;
      const int p0l = (Lb + rl - 1) / rl, plast = (Lb + nr - 1) / rl, p0u = (Lb + 3 * rl - 1) / (3 * rl);
      for (int p = p0l; p < 3 * p0u && p <= plast; ++p)
        if (p % 3 == slot && cnt < CARRY_MAX) s_carry[cnt++] = b * m_low + (p - p0l);
    }
    s_ncarry = cnt;
  }
  const int items = R * PAIRS;
  const int my_pair = tid % PAIRS;                           // the same in every item: THREADS is a multiple of PAIRS
  const int ma = f0 + 2 * my_pair, mb = ma + 1;
  const bool a_ok = ma < g.M, b_ok = mb < g.M;
  float ga = 1.f, gb = 1.f;
  if ((IS_RESID || MODE == EPI_UP) && e.gain != nullptr) {
    if (a_ok) ga = e.gain[MODE == EPI_UP ? ma % e.d_model : ma];
    if (b_ok) gb = e.gain[MODE == EPI_UP ? mb % e.d_model : mb];
  }
  float2 cs0 = make_float2(1.f, 0.f);
  const bool rot = MODE == EPI_QKV && e.dm.theta != 0.f && a_ok && ma / e.dm.dh < e.dm.H + e.dm.Hkv;
  if (rot && tid < items) {
    int b, p;
    if (row_of(e, row0 + tid / PAIRS, b, p)) cs0 = e.rope_tab[(size_t)p * (e.dm.dh >> 1) + ((ma % e.dm.dh) >> 1)];
  }
  // ---- operand rows: this lane's two rows per MMA tile
  const int NR = g.parts * R;
  const bf16* ap[MTN][2];
  bool av[MTN][2];
#pragma unroll
  for (int mt = 0; mt < MTN; ++mt)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = mt * 16 + gq + 8 * h, r = c < R ? c : c - R;
      av[mt][h] = c < NR;
      ap[mt][h] = g.A + (size_t)(g.a_row0 + (int)blockIdx.y * g.z_rows + (av[mt][h] ? r : 0)) * g.lda + (c < R ? 0 : g.K) + 8 * t4;
    }
  const int nkb = g.K / 32, kb0 = nkb * warp / NW, kb1 = nkb * (warp + 1) / NW;
  __syncthreads();                                           // barrier and row maps are initialised
  ptx::grid_dep_wait();                                      // everything below touches activations
  // The partial sums of squares of rows warp and warp + NW are requested first, 16 bytes a lane (rows of ssq are a multiple
  // of 16 floats; 4 bytes at a time a row of 128 slots took four round trips).
  float4 sq[2];
  if (SCALED && e.ssq_in != nullptr) {
#pragma unroll
    for (int j = 0; j < 2; ++j)
      sq[j] = warp + NW * j < R && 4 * lane < e.ssq_n ? __ldcg(reinterpret_cast<const float4*>(e.ssq_in + (size_t)(row0 + warp + NW * j) * e.ld_ssq) + lane) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  constexpr int CB = 2;                                      // blocks of 32 k per request, two requests in flight
  uint4 va[2][CB][MTN][2];
  auto load = [&](int buf, int kb) {
#pragma unroll
    for (int c = 0; c < CB; ++c)
#pragma unroll
      for (int mt = 0; mt < MTN; ++mt)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          va[buf][c][mt][h] = (av[mt][h] && kb + c < kb1) ? __ldcg(reinterpret_cast<const uint4*>(ap[mt][h] + (size_t)(kb + c) * 32)) : make_uint4(0, 0, 0, 0);
  };
  load(0, kb0);
  load(1, kb0 + CB);
  // residual values of the first item, and the rows' scales, while the operands travel
  float2 x0 = make_float2(0.f, 0.f);
  if (IS_RESID && e.add && tid < items && b_ok) x0 = __ldcg(reinterpret_cast<const float2*>(e.x + (size_t)(row0 + tid / PAIRS) * e.ldx + ma));
  if (SCALED && warp < R) {
    float ss[2] = {0.f, 0.f};
    if (e.ssq_in != nullptr) {
      const int left = e.ssq_n - 4 * lane;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        ss[j] = (sq[j].x + (left > 1 ? sq[j].y : 0.f)) + ((left > 2 ? sq[j].z : 0.f) + (left > 3 ? sq[j].w : 0.f));
        if (warp + NW * j < R)
          for (int s = 128 + lane; s < e.ssq_n; s += 32) ss[j] += __ldcg(e.ssq_in + (size_t)(row0 + warp + NW * j) * e.ld_ssq + s);     // more than 128 slots
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float a = __shfl_xor_sync(0xffffffffu, ss[0], o), b = __shfl_xor_sync(0xffffffffu, ss[1], o);
        ss[0] += a;
        ss[1] += b;
      }
    }
    if (lane < 2 && warp + NW * lane < R) s_inv[warp + NW * lane] = e.ssq_in != nullptr ? rsqrtf((lane == 0 ? ss[0] : ss[1]) * e.inv_d_in + e.eps) : 1.f;
  }
  float acc[MTN][FJ][4];
#pragma unroll
  for (int mt = 0; mt < MTN; ++mt)
#pragma unroll
    for (int j = 0; j < FJ; ++j) acc[mt][j][0] = acc[mt][j][1] = acc[mt][j][2] = acc[mt][j][3] = 0.f;
  const bool ok = ptx::mbar_wait(&full, 0);
  // MMA column q takes feature q / 2 + 4 (q mod 2) of its eight: the two features that eight lanes read together then lie in
  // different halves of the swizzled 128 bytes (in order, every such read took two passes over the banks).
  const int fq = (gq >> 1) | ((gq & 1) << 2);
  auto block = [&](int buf, int kb) {
#pragma unroll
    for (int c = 0; c < CB; ++c) {
      if (kb + c >= kb1) break;
      const int k = kb + c;
      uint4 w[FJ];
#pragma unroll
      for (int j = 0; j < FJ; ++j) w[j] = *reinterpret_cast<const uint4*>(sm + ((k >> 1) * FT + j * 8 + fq) * 128 + (((4 * (k & 1) + t4) ^ fq) << 4));
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int j = 0; j < FJ; ++j)
#pragma unroll
          for (int mt = 0; mt < MTN; ++mt) {
            const uint4 &p = va[buf][c][mt][0], &q = va[buf][c][mt][1];
            if (s == 0) mma(acc[mt][j], p.x, q.x, p.y, q.y, w[j].x, w[j].y);
            else mma(acc[mt][j], p.z, q.z, p.w, q.w, w[j].z, w[j].w);
          }
    }
  };
  for (int kb = kb0; kb < kb1; kb += 2 * CB) {
    block(0, kb);
    load(0, kb + 2 * CB);
    block(1, kb + CB);
    load(1, kb + 3 * CB);
  }
  __syncthreads();                                           // the weights are used up: their place becomes `red`
#pragma unroll
  for (int mt = 0; mt < MTN; ++mt)
#pragma unroll
    for (int j = 0; j < FJ; ++j) {
      float* p = red + ((warp * MTN + mt) * 16 + gq) * S + j * 8 + t4;        // MMA columns 2 t4 and 2 t4 + 1
      p[0] = acc[mt][j][0]; p[4] = acc[mt][j][1];
      p[8 * S] = acc[mt][j][2]; p[8 * S + 4] = acc[mt][j][3];
    }
  __syncthreads();
  if (!ok && tid == 0) atomicExch(g.status, -5);
  // ---- epilogue: one item = a row and two neighbouring features (in the QKV projection a rotary pair)
  for (int it0 = 0; it0 + warp * 32 < items; it0 += THREADS) {
    const int it = it0 + tid;
    const bool active = it < items, first = it0 == 0;
    const int n = active ? it / PAIRS : 0;
    const float* p = red + n * S + 2 * my_pair;
    float ya = 0.f, yb = 0.f, la = 0.f, lb = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) {                           // warp order: hi products, lo products
      const float2 h = *reinterpret_cast<const float2*>(p + w * (MTN * 16 * S));
      ya += h.x;
      yb += h.y;
    }
    if (g.parts == 2) {
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        const float2 l = *reinterpret_cast<const float2*>(p + w * (MTN * 16 * S) + R * S);
        la += l.x;
        lb += l.y;
      }
    }
    ya += la;
    yb += lb;
    if (MODE != EPI_UP && !IS_RESID) {
      const float inv = s_inv[n];
      ya *= inv;
      yb *= inv;
    }
    const size_t row = (size_t)(row0 + n);
    if (MODE == EPI_F32) {
      float* o = reinterpret_cast<float*>(e.out) + row * e.ldo + ma;
      if (active && b_ok && (e.ldo & 1) == 0) *reinterpret_cast<float2*>(o) = make_float2(ya, yb);
      else if (active) {
        if (a_ok) o[0] = ya;
        if (b_ok) o[1] = yb;
      }
    } else if (MODE == EPI_BF16 || MODE == EPI_GELU) {
      if (MODE == EPI_GELU) {
        const float2 y = gelu2(ya, yb);
        ya = y.x;
        yb = y.y;
      }
      bf16* o = reinterpret_cast<bf16*>(e.out) + row * e.ldo + ma;
      if (active && b_ok) store_hi_lo2(o, ya, yb, e.lo_off);
      else if (active && a_ok) store_hi_lo(o, ya, e.lo_off);
    } else if (IS_RESID) {
      float xa = 0.f, xb = 0.f;
      if (active && b_ok) {                                  // both columns (M is even wherever the residual is used)
        float* xr = e.x + row * e.ldx + ma;
        if (!first && e.add) x0 = __ldcg(reinterpret_cast<const float2*>(xr));
        xa = x0.x + ya;
        xb = x0.y + yb;
        if (MODE == EPI_RESID_CAT && s_rb[n] >= 0) {
          // (xa, xb) is the level's final hidden of position p: into the carry ring, into the operand row of
          // the parent that pools it (if that parent is a row of this pass), and, where the position's own
          // parent p / 3 was computed in an earlier pass, that parent's stored slot is added at once
          const int b = s_rb[n], pos = s_rp[n], dd = e.d_model, rs = fm_ring(e.level), rsu = fm_ring(e.level + 1);
          *reinterpret_cast<float2*>(e.cat_ring + ((size_t)b * rs + pos % rs) * dd + ma) = make_float2(xa, xb);
          const int u = (pos + 2) / 3, part = pos - 3 * u + 2;
          if (3 * u <= s_rl[n])
            store_hi_lo2(e.cat_out + ((size_t)(b * fm_rows_per_seq(e.dm, e.level + 1) + u - s_ra[n]) * 6 + part) * dd + ma, xa, xb, 3 * dd);
          if (pos < 3 * s_ra[n]) {
            const float2 t = __ldcg(reinterpret_cast<const float2*>(e.cat_tri + (((size_t)b * rsu + (pos / 3) % rsu) * 3 + pos % 3) * dd + ma));
            xa += t.x;
            xb += t.y;
          }
        }
        *reinterpret_cast<float2*>(xr) = make_float2(xa, xb);
        if (e.a_out != nullptr) store_hi_lo2(e.a_out + row * e.lda + ma, __fmul_rn(xa, ga), __fmul_rn(xb, gb), e.lo_off);
      }
      if (e.ssq_out != nullptr) {                            // sum of squares of this CTA's features, for the next norm
        float sq = __fmaf_rn(xa, xa, __fmul_rn(xb, xb));
#pragma unroll
        for (int o = PAIRS / 2; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        if (active && my_pair == 0) e.ssq_out[row * e.ld_ssq_out + blockIdx.x] = sq;
      }
    } else if (MODE == EPI_UP) {
      // (ya, yb): columns (ma, ma + 1) of the triple of parent row n = slot ma / d, column ma % d
      const int dd = e.d_model, slot = ma / dd, col = ma - slot * dd;
      float xa = 0.f, xb = 0.f;
      bool child = false;
      size_t crow = 0;
      if (active && b_ok && s_rb[n] >= 0) {
        const int b = s_rb[n], pu = s_rp[n], rsu = fm_ring(e.level), pos = 3 * pu + slot;
        *reinterpret_cast<float2*>(e.tri_ring + ((size_t)b * rsu + pu % rsu) * 3 * dd + ma) = make_float2(ya, yb);
        if (pos <= s_rl[n]) {                                // the child is a row of this pass
          child = true;
          crow = (size_t)b * fm_rows_per_seq(e.dm, e.level - 1) + (pos - s_ra[n]);
          float* xr = e.x + crow * e.ldx + col;
          const float2 xc = __ldcg(reinterpret_cast<const float2*>(xr));
          xa = xc.x + ya;
          xb = xc.y + yb;
          *reinterpret_cast<float2*>(xr) = make_float2(xa, xb);
          store_hi_lo2(e.a_out + crow * e.lda + col, __fmul_rn(xa, ga), __fmul_rn(xb, gb), e.lo_off);
        }
      }
      float sq = __fmaf_rn(xa, xa, __fmul_rn(xb, xb));
#pragma unroll
      for (int o = PAIRS / 2; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
      if (child && my_pair == 0) e.ssq_out[crow * e.ld_ssq_out + (f0 % dd) / FT] = sq;
    } else {  // EPI_QKV: the rotary pair (i, i + dh/2) of one head, stored at (c, c + 1), c = 2i
      const int dh = e.dm.dh, H = e.dm.H, Hkv = e.dm.Hkv, head = ma / dh, c = ma - head * dh;
      if (active && a_ok) {
        const int b = s_rb[n], pos = s_rp[n];
        const bool valid = b >= 0;
        if (rot) {
          const float2 cs = first ? cs0 : (valid ? e.rope_tab[(size_t)pos * (dh >> 1) + (c >> 1)] : make_float2(1.f, 0.f));
          const float y1 = ya * cs.x - yb * cs.y, y2 = yb * cs.x + ya * cs.y;
          ya = y1;
          yb = y2;
        }
        if (head < H) {
          *reinterpret_cast<__nv_bfloat162*>(e.q_out + (row * H + head) * dh + c) =
              valid ? __floats2bfloat162_rn(ya * e.qscale, yb * e.qscale) : __floats2bfloat162_rn(0.f, 0.f);
        } else if (valid) {
          const int cap = e.dm.cap[e.level], hk = head - H < Hkv ? head - H : head - H - Hkv;
          bf16* dst = (head - H < Hkv ? e.Kc : e.Vc) + (((size_t)b * Hkv + hk) * (e.dm.P + cap) + e.dm.P + pos % cap) * dh + c;
          *reinterpret_cast<__nv_bfloat162*>(dst) = __floats2bfloat162_rn(ya, yb);
        }
      }
    }
  }
  if (MODE == EPI_QKV && e.stash_ring != nullptr) {
    // the rows' residual values, as they enter this layer, go into the carry ring (the draft heads read
    // them after the pass); the CTAs share the columns
    const int cols = (e.stash_d + (int)gridDim.x - 1) / (int)gridDim.x, c0 = (int)blockIdx.x * cols;
    for (int i = tid; i < R * cols; i += THREADS) {
      const int n = i / cols, col = c0 + i - n * cols;
      if (col < e.stash_d && s_rb[n] >= 0)
        e.stash_ring[((size_t)s_rb[n] * e.stash_rs + s_rp[n] % e.stash_rs) * e.stash_d + col] = __ldcg(e.stash_x + (size_t)(row0 + n) * e.stash_d + col);
    }
  }
  if (MODE == EPI_UP) {
    // children whose parent was computed in an earlier pass: their residual rows are final already (the
    // last layer below added the stored slot); what is missing is the next operand and the sums of squares
    const int dd = e.d_model, nci = s_ncarry * PAIRS, col = ma % dd;
    for (int it0 = 0; it0 + warp * 32 < nci; it0 += THREADS) {
      const int it = it0 + tid;
      const bool active = it < nci;
      const size_t crow = active ? (size_t)s_carry[it / PAIRS] : 0;
      float2 xc = make_float2(0.f, 0.f);
      if (active) {
        xc = __ldcg(reinterpret_cast<const float2*>(e.x + crow * e.ldx + col));
        store_hi_lo2(e.a_out + crow * e.lda + col, __fmul_rn(xc.x, ga), __fmul_rn(xc.y, gb), e.lo_off);
      }
      float sq = __fmaf_rn(xc.x, xc.x, __fmul_rn(xc.y, xc.y));
#pragma unroll
      for (int o = PAIRS / 2; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
      if (active && my_pair == 0) e.ssq_out[crow * e.ld_ssq_out + (f0 % dd) / FT] = sq;
    }
  }
  if (!ok) ptx::drain_delay();                               // a wait gave up: copies already requested may still be landing
}

}  // namespace rg
