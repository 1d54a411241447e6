// Few-row causal attention over one level's KV cache (Sec. 3.3: the candidates of a pass are
// masked causally among themselves; conditioning enters as prefix keys visible to every row).
//
// Streaming split-KV design.  The cache of a (sequence, kv-head) is cut into chunks of C slots; chunk c
// belongs to group c mod NG (NG is fixed per level when the context is created), so that all groups have
// work and nearly the same amount at any fill of the cache.  One CTA streams one group: a producer warp
// brings the K and V tiles of its chunks in with TMA (2-D tensor maps over the cache, 128-byte swizzle)
// through a ring of shared-memory stages; NW compute warps each own a fixed slice of every chunk
// and keep their own running softmax state (max, sum, output) across the group's chunks, so warps never
// wait for one another while streaming.  All query rows of the sequence that share the kv-head (rows of
// the pass x heads of the group, 16 per CTA) form the M axis of warp-level bf16 MMAs, so the cache is
// read once per pass, not once per row.
// At the end of the group the warps' states are merged in warp order.  One group: the result is final.
// Several: the groups' states go to a scratch buffer, and a second small launch (attn_merge_kernel, a warp
// per row and head) merges them in group order.  (Merging by the CTA that takes the last ticket of a
// counter cost 1.1 us for the ticket and 1.4 us for the merge by a single CTA; a thread-block cluster
// per head was slower still: CTAs this large are gang-scheduled microseconds apart.)
// Slices, chunks and groups are fixed by slot index, so a row's result does not depend on how many
// other rows or sequences the launch holds, nor on the cache length at the time it is computed.
// Programmatic dependent launch: cache entries written by earlier passes do not depend on the
// previous kernel, so chunks that hold none of this pass's new slots are requested before
// griddepcontrol.wait.
#pragma once
#include "fm_common.cuh"
#include "fm_ptx.cuh"

struct AttnArgs {
  Dims dm;
  SeqState st;
  int batch, level;
  const bf16* q;              // [rows, H*dh] bf16, rotated and scaled by log2(e)/sqrt(dh)
  const CUtensorMap* tmK;     // cache as 2-D [B*Hkv*slots, dh], box C x 64
  const CUtensorMap* tmV;
  float* part;                // [B*Hkv*MT, max_groups, 16, dh + 2]
  bf16* out;                  // [rows, 2*H*dh]: the next GEMM's operand rows as [hi | lo] bfloat16 terms
  int max_groups;             // NG, the number of groups of this level (= gridDim.x)
  int MT;                     // 16-row query tiles per (sequence, kv-head)
  // Draft mode (SP-Block / HF-Block queries, Sec. 3.1): draft_nq > 0 query rows per sequence, none of
  // them in the cache; every row sees what the last accepted position of the level sees (the prefix
  // and positions max(0, p - W + 1) .. p with p = floor((L - 1) / ratio)).  Row r of sequence b is
  // read at q[(b * draft_nq + r)] and written to out row r * out_row_stride + b.
  int draft_nq;
  int out_row_stride;
};

template <int DH, int C, int NW, int ST>
struct AttnCfg {
  static_assert(C % (16 * NW) == 0, "a compute warp owns a multiple of 16 slots of a chunk");
  // Stages of 32 KB.  Five: with the 64 KB of the projection in front (few rows, d = 1024) exactly what an SM
  // holds, so that most of a group is on chip before the queries are.  Three: two CTAs per SM.
  static constexpr int STAGES = ST;
  static constexpr int KPW = C / NW;                        // slots of a chunk per warp
  static constexpr int HALVES = DH / 64;
  static constexpr int TILE = C * DH * 2;                   // bytes of one K (or V) tile
  static constexpr int STAGE = 2 * TILE;
  static constexpr int RING = STAGES * STAGE;               // also holds the warps' states for their merge
  static_assert(RING >= NW * 16 * (DH + 2) * 4, "");
  static constexpr int BYTES = RING + 128;                  // + barriers
  static constexpr int MAX_GROUPS = 24;                     // a lane per group in the merge
  static constexpr int THREADS = (NW + 1) * 32;
  // CTAs per SM that the ring depth was chosen for.  The launch bound holds the registers to it (at most 200 per thread
  // for two; 143 and 168 are in use), this the shared memory: 228 KB per SM, of which a CTA takes 1 KB for itself.
  static constexpr int CTAS = STAGES <= 3 ? 2 : 1;
  static_assert(CTAS * (BYTES + 1024) <= 228 * 1024, "the CTAs of an SM share its shared memory");
};

namespace attn {
__device__ inline void store_out2(bf16* out, float a, float b, int lo_off) {
  const __nv_bfloat162 hi = __floats2bfloat162_rn(a, b);
  *reinterpret_cast<__nv_bfloat162*>(out) = hi;
  *reinterpret_cast<__nv_bfloat162*>(out + lo_off) = __floats2bfloat162_rn(__fsub_rn(a, __bfloat162float(hi.x)), __fsub_rn(b, __bfloat162float(hi.y)));
}
// (volatile: a batch of these is issued before anything that waits for one of them)
__device__ inline float2 load2(const float* p) {
  float2 v;
  asm volatile("ld.global.cg.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
__device__ inline int div_ratio(int x, int level) { return level == 0 ? x : (level == 1 ? x / 3 : x / 9); }
}  // namespace attn

// What a (sequence, kv-head) has to do at a level in this pass.
struct AttnWork {
  int n, p0, nq, p_max, n_chunks, n_groups, M, m_rows;
  bool dmode;
};
__device__ inline AttnWork attn_work(const AttnArgs& a, int b, int C) {
  AttnWork w;
  const Dims& dm = a.dm;
  const int level = a.level, ratio = fm_ratio(level);
  w.n = b < a.batch ? a.st.nrow[b] : 0;
  const int Lb = b < a.batch ? a.st.L[b] : 0;
  w.dmode = a.draft_nq > 0;
  w.p0 = w.dmode ? attn::div_ratio(Lb - 1, level) : attn::div_ratio(Lb + ratio - 1, level);
  w.nq = w.n > 0 ? (w.dmode ? a.draft_nq : attn::div_ratio(Lb + w.n - 1, level) - w.p0 + 1) : 0;
  w.p_max = w.dmode ? w.p0 : w.p0 + w.nq - 1;
  w.n_chunks = (dm.P + min(dm.cap[level], w.p_max + 1) + C - 1) / C;
  w.n_groups = min(w.n_chunks, a.max_groups);
  w.M = w.nq * (dm.H / dm.Hkv);
  w.m_rows = w.dmode ? a.draft_nq : fm_rows_per_seq(dm, level);
  return w;
}
// where query idx (= r * heads per group + head of the group) of sequence b writes its output columns
__device__ inline size_t attn_out_at(const AttnArgs& a, const AttnWork& w, int b, int hk, int idx, int DH) {
  const int group = a.dm.H / a.dm.Hkv, r = group == 1 ? idx : idx / group, gh = idx - r * group;
  const size_t row = a.out_row_stride > 0 ? (size_t)r * a.out_row_stride + b : (size_t)(b * w.m_rows + r);
  return (row * 2 * a.dm.H + hk * group + gh) * DH;
}

// grid (max_groups, Hkv * MT, batch); block (NW + 1) warps: NW compute warps and one producer warp.
template <int DH, int C, int NW, int ST>
__global__ void __launch_bounds__(AttnCfg<DH, C, NW, ST>::THREADS, AttnCfg<DH, C, NW, ST>::CTAS) attn_stream_kernel(const AttnArgs a) {
  using CF = AttnCfg<DH, C, NW, ST>;
  constexpr int KS = DH / 16, KB = CF::KPW / 16, NT = CF::KPW / 8;     // k-steps of Q K^T; 16-slot blocks and 8-slot tiles per warp
  const Dims& dm = a.dm;
  const int u = blockIdx.x, NG = a.max_groups;
  const int hk = a.MT == 1 ? (int)blockIdx.y : (int)blockIdx.y / a.MT;
  const int mt = (int)blockIdx.y - hk * a.MT;
  const int b = blockIdx.z;
  const int warp = (int)ptx::uniform(threadIdx.x >> 5), lane = threadIdx.x & 31, g = lane >> 2, t4 = lane & 3;
  ptx::grid_dep_launch();
  // ---- what this CTA has to do (per-pass state is final before the pass's first kernel starts)
  const AttnWork w = attn_work(a, b, C);
  if (w.nq <= 0 || mt * 16 >= w.M || u >= w.n_groups) {      // nothing of the cache falls into this group yet
    ptx::grid_dep_wait();                                    // keep the launch chain ordered
    return;
  }
  const int level = a.level, p0 = w.p0, p_max = w.p_max, M = w.M;
  const int P = dm.P, cap = dm.cap[level], W = dm.window[level], slots = P + cap;
  const int group = dm.H / dm.Hkv;
  const int n_my = (w.n_chunks - u + NG - 1) / NG;           // chunks u, u + NG, ...

  extern __shared__ __align__(1024) unsigned char sm[];
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + CF::RING);
  uint64_t* empty = full + CF::STAGES;
  int& s_fail = *reinterpret_cast<int*>(empty + CF::STAGES);   // (no static shared memory: the ring must start at a 1024-byte boundary)

  // slots written by this pass: P + (p mod cap), p = p0..p_max: one run of nq slots from new_lo,
  // which may wrap around the end of the ring once
  const int new_lo = P + p0 % cap;
  const int n_new = w.dmode ? 0 : w.nq;                      // draft queries append nothing
  auto has_new = [&](int c) {
    const int lo = c * C, hi = lo + C;                       // [lo, hi)
    const int e1 = min(new_lo + n_new, slots);               // first part [new_lo, e1)
    const int n2 = new_lo + n_new - e1;                      // wrapped part [P, P + n2)
    return (new_lo < hi && e1 > lo) || (n2 > 0 && P < hi && P + n2 > lo);
  };
  const int row_base = (b * dm.Hkv + hk) * slots;
  auto issue = [&](int i) {
    if (!ptx::elect_one()) return;                           // one lane of the producer warp, which stays in step
    const int st = i % CF::STAGES;
    unsigned char* Ks = sm + st * CF::STAGE;
    unsigned char* Vs = Ks + CF::TILE;
    ptx::mbar_expect_tx(full + st, CF::STAGE);
    const int row0 = row_base + (u + i * NG) * C;
#pragma unroll
    for (int h = 0; h < CF::HALVES; ++h) {
      ptx::tma_load_2d(Ks + h * C * 128, a.tmK, h * 64, row0, full + st);
      ptx::tma_load_2d(Vs + h * C * 128, a.tmV, h * 64, row0, full + st);
    }
  };
  int n_pre = 0;                                             // producer: chunks requested
  if (warp == NW) {
    if (lane == 0) {
      s_fail = 0;
      for (int i = 0; i < CF::STAGES; ++i) { ptx::mbar_init(full + i, 1); ptx::mbar_init(empty + i, NW); }
      ptx::fence_mbar_init();
    }
    __syncwarp();
    // chunks that hold old entries only are requested at once, before the dependency wait
    const int pre = n_my < CF::STAGES ? n_my : CF::STAGES;
    while (n_pre < pre && !has_new(u + n_pre * NG)) { issue(n_pre); __syncwarp(); ++n_pre; }
  }
  __syncthreads();

  // running state of this warp's slices: rows g and g+8 of the query tile
  float o[DH / 8][4];
  float mrun[2] = {-INFINITY, -INFINITY}, lrun[2] = {0.f, 0.f};
#pragma unroll
  for (int i = 0; i < DH / 8; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;

  if (warp == NW) {
    // ---- producer
    ptx::grid_dep_wait();
    for (int i = n_pre; i < n_my; ++i) {
      if (i >= CF::STAGES && !__all_sync(0xffffffffu, ptx::mbar_wait(empty + i % CF::STAGES, ((i / CF::STAGES) - 1) & 1))) { s_fail = 1; break; }
      issue(i);
      __syncwarp();
    }
  } else {
    // ---- compute warps
    ptx::grid_dep_wait();                          // queries come from the previous kernel
    // Q fragments of this CTA's query tile (rows idx = mt*16 + g, +8; idx = r*group + gh)
    uint32_t qa[KS][4];
    int prow[2];
#pragma unroll
    for (int hrow = 0; hrow < 2; ++hrow) {
      const int idx = mt * 16 + g + hrow * 8;
      const bool ok = idx < M;
      const int r = ok ? (group == 1 ? idx : idx / group) : 0, gh = ok ? idx - r * group : 0;
      prow[hrow] = ok ? (w.dmode ? p0 : p0 + r) : -100;
      const bf16* qp = a.q + ((size_t)(b * w.m_rows + r) * dm.H + hk * group + gh) * DH;
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        qa[ks][hrow] = ok ? __ldcg(reinterpret_cast<const unsigned int*>(qp + ks * 16 + 2 * t4)) : 0u;
        qa[ks][2 + hrow] = ok ? __ldcg(reinterpret_cast<const unsigned int*>(qp + ks * 16 + 8 + 2 * t4)) : 0u;
      }
    }
    // slot -> position: behind the prefix, slot P + r holds position r + k*cap with
    // k = floor((p_max - r) / cap) = wrap_q if r <= wrap_r else wrap_q - 1
    const int wrap_q = p_max / cap, wrap_r = p_max - wrap_q * cap;
    for (int i = 0; i < n_my; ++i) {
      const int st = i % CF::STAGES;
      // is every slot of the chunk visible to every row of the pass?  (the common case: prefix, or
      // old positions inside every row's window) -- then no masks are needed
      const int s_lo = (u + i * NG) * C, s_hi = s_lo + C - 1;
      bool all_vis = s_hi < P;
      if (!all_vis && s_lo >= P) {
        const int r_lo = s_lo - P, r_hi = s_hi - P;
        if (r_hi < cap && r_hi <= p_max && (r_hi <= wrap_r || r_lo > wrap_r)) {
          const int k = r_hi <= wrap_r ? wrap_q : wrap_q - 1;
          all_vis = r_hi + k * cap <= p0 && (W == 0 || r_lo + k * cap >= p_max - W + 1);
        }
      }
      if (!__all_sync(0xffffffffu, ptx::mbar_wait(full + st, (i / CF::STAGES) & 1))) { s_fail = 1; break; }
      const uint32_t Ks_u = ptx::smem_u32(sm + st * CF::STAGE), Vs_u = Ks_u + CF::TILE;
      // All fragments of the warp's slice are requested first: a chunk is then one shared-memory latency, two
      // groups of independent MMAs and the softmax between them, not a chain of loads and MMAs.
      uint32_t kf[KB][KS][4], vf[KB][DH / 16][4];
#pragma unroll
      for (int kb = 0; kb < KB; ++kb)
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
          const int key = warp * CF::KPW + kb * 16 + (lane & 7) + (lane >> 4) * 8;
          const int ch = ks * 2 + ((lane >> 3) & 1);
          ptx::ldmatrix_x4(kf[kb][ks][0], kf[kb][ks][1], kf[kb][ks][2], kf[kb][ks][3], Ks_u + (ch >> 3) * C * 128 + ptx::swz128(key, ch & 7));
        }
#pragma unroll
      for (int kb = 0; kb < KB; ++kb)
#pragma unroll
        for (int dp = 0; dp < DH / 16; ++dp) {
          const int key = warp * CF::KPW + kb * 16 + (lane & 7) + ((lane >> 3) & 1) * 8;
          const int ch = dp * 2 + (lane >> 4);
          ptx::ldmatrix_x4_trans(vf[kb][dp][0], vf[kb][dp][1], vf[kb][dp][2], vf[kb][dp][3], Vs_u + (ch >> 3) * C * 128 + ptx::swz128(key, ch & 7));
        }
      // ---- S = Q K^T over this warp's slots
      float s[NT][4];
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
#pragma unroll
      for (int ks = 0; ks < KS; ++ks)
#pragma unroll
        for (int kb = 0; kb < KB; ++kb) {
          ptx::mma_bf16_16816(s[2 * kb], qa[ks], kf[kb][ks][0], kf[kb][ks][1]);
          ptx::mma_bf16_16816(s[2 * kb + 1], qa[ks], kf[kb][ks][2], kf[kb][ks][3]);
        }
      if (!all_vis) {
        // positions of this thread's key columns: n-tile nt, element e -> slot base + nt*8 + 2*t4 + e
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int slot = s_lo + warp * CF::KPW + nt * 8 + 2 * t4 + e;
            const int r = slot - P;
            const int kp = slot < P ? -1 : ((r >= cap || r > p_max) ? -2 : r + (r <= wrap_r ? wrap_q : wrap_q - 1) * cap);
#pragma unroll
            for (int hrow = 0; hrow < 2; ++hrow) {
              const int pr = prow[hrow];
              const bool vis = kp == -1 || (kp >= 0 && kp <= pr && (W == 0 || kp >= pr - W + 1));
              if (!(vis && pr >= 0)) s[nt][hrow * 2 + e] = -INFINITY;
            }
          }
      }
      // ---- running max and exponentials (rows g and g+8; quad = the 4 lanes sharing g); the sums stay per lane
      float scale[2], base[2];
#pragma unroll
      for (int hrow = 0; hrow < 2; ++hrow) {
        float mx = -INFINITY;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) mx = fmaxf(mx, fmaxf(s[nt][hrow * 2], s[nt][hrow * 2 + 1]));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        const float mnew = fmaxf(mrun[hrow], mx);
        base[hrow] = mnew == -INFINITY ? 0.f : mnew;
        scale[hrow] = mnew == mrun[hrow] ? 1.f : exp2f(mrun[hrow] - base[hrow]);
        mrun[hrow] = mnew;
      }
      float ls[2] = {0.f, 0.f};
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          s[nt][e] = exp2f(s[nt][e] - base[e >> 1]);
          ls[e >> 1] += s[nt][e];
        }
      lrun[0] = lrun[0] * scale[0] + ls[0];
      lrun[1] = lrun[1] * scale[1] + ls[1];
      // the running output only needs rescaling when a row's maximum moved (scale 1 changes nothing)
      if (__any_sync(0xffffffffu, scale[0] != 1.f || scale[1] != 1.f)) {
#pragma unroll
        for (int i2 = 0; i2 < DH / 8; ++i2) {
          o[i2][0] *= scale[0]; o[i2][1] *= scale[0];
          o[i2][2] *= scale[1]; o[i2][3] *= scale[1];
        }
      }
      // ---- O += P V
#pragma unroll
      for (int kb = 0; kb < KB; ++kb) {
        uint32_t pa[4];
        pa[0] = ptx::pack_bf16(s[2 * kb][0], s[2 * kb][1]);
        pa[1] = ptx::pack_bf16(s[2 * kb][2], s[2 * kb][3]);
        pa[2] = ptx::pack_bf16(s[2 * kb + 1][0], s[2 * kb + 1][1]);
        pa[3] = ptx::pack_bf16(s[2 * kb + 1][2], s[2 * kb + 1][3]);
#pragma unroll
        for (int dp = 0; dp < DH / 16; ++dp) {
          ptx::mma_bf16_16816(o[2 * dp], pa, vf[kb][dp][0], vf[kb][dp][1]);
          ptx::mma_bf16_16816(o[2 * dp + 1], pa, vf[kb][dp][2], vf[kb][dp][3]);
        }
      }
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(empty + st);           // this warp is done with the stage
    }
#pragma unroll
    for (int hrow = 0; hrow < 2; ++hrow) {
      lrun[hrow] += __shfl_xor_sync(0xffffffffu, lrun[hrow], 1);
      lrun[hrow] += __shfl_xor_sync(0xffffffffu, lrun[hrow], 2);
    }
  }
  // ---- the warps' states -> shared memory (the ring is idle once every warp is here), merged in warp order
  __syncthreads();
  if (s_fail) {                                              // a bounded wait gave up: report, write nothing
    if (threadIdx.x == 0) atomicExch(a.st.status, -5);
    ptx::drain_delay();                                      // chunks already requested may still be landing
    return;
  }
  float* pw = reinterpret_cast<float*>(sm);                  // [NW][16][DH] outputs
  float* ml = pw + NW * 16 * DH;                             // [NW][16][2] maxima and sums
  if (warp < NW) {
    float* mine = pw + warp * 16 * DH;
#pragma unroll
    for (int i = 0; i < DH / 8; ++i) {
      *reinterpret_cast<float2*>(mine + g * DH + i * 8 + 2 * t4) = make_float2(o[i][0], o[i][1]);
      *reinterpret_cast<float2*>(mine + (g + 8) * DH + i * 8 + 2 * t4) = make_float2(o[i][2], o[i][3]);
    }
    if (t4 == 0) {
      *reinterpret_cast<float2*>(ml + (warp * 16 + g) * 2) = make_float2(mrun[0], lrun[0]);
      *reinterpret_cast<float2*>(ml + (warp * 16 + g + 8) * 2) = make_float2(mrun[1], lrun[1]);
    }
  }
  __syncthreads();
  const int rows_here = min(16, M - mt * 16);
  const size_t pt = ((size_t)(b * dm.Hkv + hk) * a.MT + mt);
  float* gpart = a.part + (pt * NG + u) * 16 * (DH + 2);
  const bool single = w.n_groups == 1;
  for (int e = threadIdx.x; e < rows_here * (DH / 2); e += CF::THREADS) {      // two neighbouring columns of a row
    const int i = e / (DH / 2), c = 2 * (e - i * (DH / 2));
    float2 st[NW];
    float mm = -INFINITY, l = 0.f, o0 = 0.f, o1 = 0.f;
#pragma unroll
    for (int k = 0; k < NW; ++k) { st[k] = *reinterpret_cast<const float2*>(ml + (k * 16 + i) * 2); mm = fmaxf(mm, st[k].x); }
#pragma unroll
    for (int k = 0; k < NW; ++k) {
      const float f = st[k].x == -INFINITY ? 0.f : exp2f(st[k].x - mm);
      const float2 v = *reinterpret_cast<const float2*>(pw + (k * 16 + i) * DH + c);
      l += f * st[k].y;
      o0 += f * v.x;
      o1 += f * v.y;
    }
    if (single) {
      const float inv = 1.f / l;
      attn::store_out2(a.out + attn_out_at(a, w, b, hk, mt * 16 + i, DH) + c, o0 * inv, o1 * inv, dm.H * DH);
    } else {
      float* row = gpart + (size_t)i * (DH + 2);             // columns: output, maximum, sum
      *reinterpret_cast<float2*>(row + c) = make_float2(o0, o1);
      if (c == 0) *reinterpret_cast<float2*>(row + DH) = make_float2(mm, l);
    }
  }
}

// Merge of the groups, in group order: a warp per (sequence, kv-head, query); grid (B*Hkv*MT, 4), 4 warps.
template <int DH, int C>
__global__ void __launch_bounds__(128) attn_merge_kernel(const AttnArgs a) {
  ptx::grid_dep_launch();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int pt = blockIdx.x, mt = pt % a.MT, hk = pt / a.MT % a.dm.Hkv, b = pt / (a.MT * a.dm.Hkv), i = blockIdx.y * 4 + warp;
  const AttnWork w = attn_work(a, b, C);
  const bool live = w.nq > 0 && mt * 16 + i < w.M && w.n_groups > 1;
  const float* src = a.part + (size_t)pt * a.max_groups * 16 * (DH + 2) + (size_t)i * (DH + 2);
  constexpr int GS = 16 * (DH + 2), CL = DH / 32;            // floats per group; columns per lane
  ptx::grid_dep_wait();
  if (!live) return;
  const float2 ml = lane < w.n_groups ? attn::load2(src + lane * GS + DH) : make_float2(-INFINITY, 0.f);
  float2 v[12][CL / 2], acc[CL / 2];
  auto load = [&](int k0) {
#pragma unroll
    for (int k = 0; k < 12; ++k)
#pragma unroll
      for (int j = 0; j < CL / 2; ++j)
        v[k][j] = k0 + k < w.n_groups ? attn::load2(src + (k0 + k) * GS + lane * CL + 2 * j) : make_float2(0.f, 0.f);
  };
  load(0);
  const float mm = warp_max(ml.x), f = ml.x == -INFINITY ? 0.f : exp2f(ml.x - mm);
  const float inv = 1.f / warp_sum(f * ml.y);                // (absent groups add exact zeros: the sum does not depend on how many there are)
#pragma unroll
  for (int j = 0; j < CL / 2; ++j) acc[j] = make_float2(0.f, 0.f);
  for (int k0 = 0; k0 < w.n_groups; k0 += 12) {
    if (k0 > 0) load(k0);
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const float fk = __shfl_sync(0xffffffffu, f, k0 + k);
#pragma unroll
      for (int j = 0; j < CL / 2; ++j) { acc[j].x = fmaf(fk, v[k][j].x, acc[j].x); acc[j].y = fmaf(fk, v[k][j].y, acc[j].y); }
    }
  }
  bf16* out = a.out + attn_out_at(a, w, b, hk, mt * 16 + i, DH) + lane * CL;
#pragma unroll
  for (int j = 0; j < CL / 2; ++j) attn::store_out2(out + 2 * j, acc[j].x * inv, acc[j].y * inv, a.dm.H * DH);
}
