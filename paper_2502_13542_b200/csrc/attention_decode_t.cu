// Step 5 for short steps (decode, Eq. 3) of at most 32 query rows per KV head (rows = new tokens x G):
// attention over
//   [initial tokens | local past | the new tokens (causal) | selected blocks]
// for bf16, D = 128, pages of 16 to 128 tokens.  The work per key is 4 * D * rows flops against 4 * D bytes
// of K and V: the stage is bound by the K / V stream, and by latency when there are few sequences.
//
// The products are transposed, so that the wide operand of the tensor core is the cache and the few queries
// are the narrow one:  S^T [128 keys x N] = K Q^T  and  O^T [128 channels x 2N] = V^T [P_hi | P_lo],
// N = 16 or 32.  Against queries padded to 128 rows (attention_decode.cu, which serves more than 32 rows) a
// tile takes a sixth of the tensor-pipe time, its softmax 128 x rows exponentials spread over 128 threads (thread =
// key) instead of 128 x 128 on a few warps, TMEM 4 N columns instead of 512 and Q 4 KiB of shared memory
// instead of 32, so that two CTAs fit an SM and one's start and end hide behind the other's stream.
// P is two bf16 terms (hi + lo, 16 significant bits) side by side as the columns of one operand: V is read once.
//
// One CTA = one KV head of one (sequence, layer) and every n-th 128-key tile of its key stream, n = CTAs
// of the cluster (up to 8, chosen so that the CTAs fill the SMs); the ranks' partial results meet in
// distributed shared memory.  The selected blocks come last: everything else is known before this step's
// selection exists, so the kernel starts while the selection is still being computed (programmatic dependent
// launch) and each role takes the dependency wait where the selected blocks begin.
//
// Roles: softmax and epilogue in groups of four warps, one group for up to 8 rows, two for 16, four for 32 (each
// takes 8 rows: one group with 32 rows apiece needs 2,400 clk per tile, and its unrolled code is fetched anew by
// every CTA: 91.5 us for two layers of four sequences with five drafted tokens, 80.9 with four groups); then one warp
// each: K producer (and Q), V producer, issuer of Q K^T, issuer of P V (one issuer for both holds the next Q K^T back
// behind the wait for P; with it and a merge of one row per round: 158.9 us for six layers of one sequence, 152.9
// without).  K and V tiles share one ring of 32 KiB slots, K0 V0 K1 V1 ...; a tile is eight boxes of one 16-token
// granule.  The running maximum moves only when a score exceeds it by 2^32 (P has fp32's range), which is a vote per
// tile; the reduction over the 128 threads that a new maximum takes is the rare path.
// Measured against the padded form, whole decode steps as graphs: 64 sequences of 2k-8k tokens 528 -> 390 us for
// two layers (the K / V stream alone 385 us at the measured copy bandwidth), 16 of 32k-131k 202 -> 166 us, one
// sequence 208 -> 148 us for six layers (its partial results then took a second kernel), four sequences of five
// drafted tokens 153 -> 81 us for two layers (no cut without a workspace then).
// Every wait on an mbarrier is bounded; on expiry the CTA flags ACTQKV_DEV_TIMEOUT, drains, and its partial
// result counts as empty.
#include <algorithm>

#include "tc_common.cuh"

using namespace actqkv;
using namespace actqkv::tc;

namespace {

constexpr int kBN = 128, kD = 128;
constexpr int kMaxRanks = 8;
constexpr int kMaxRows = 32;
constexpr uint32_t kTileBytes = 32 * 1024;               // one K or V tile

// P may reach 2^32 before the running maximum has to move, as in the padded kernel: what it may reach is taken from the
// range of V (six layers of one sequence 151.0 us with 2^64, 151.4 with this, 152.2 with 2^15, 153.9 with 2^8).
constexpr float kMaxLag = kRescaleThreshold;

// R: rows rounded up to 4, 8, 16 or 32; N: columns of S^T (a multiple of 16).  kDeep: one CTA per SM with six
// ring slots, for grids that leave the SMs to one CTA each (and for 32 rows); else two CTAs of three.
template <int R, bool kDeep> struct Cfg {
  static constexpr int N = R < 16 ? 16 : R;
  static constexpr int SG = R < 16 ? 1 : R / 8, RS = R / SG;       // softmax groups of four warps, rows of each
  static constexpr int kThreads = 128 * SG + 128;
  static constexpr int kCtasPerSm = kDeep ? 1 : 2;
  static constexpr int kRing = kDeep ? 6 : 3;
  static constexpr uint32_t kQBytes = N * 256, kPBytes = 2 * N * 256;
  static constexpr uint32_t kCols = 4 * N;               // S 2 x N, O 2 N
  static constexpr int kNumBars = 1 + 4 * kRing + 4 + 4;
  static constexpr uint32_t kBarBytes = 320;
  static constexpr uint32_t kSmall = (4 * R + 2 * R) * 4;           // per-warp maxima / sums, then (m, l)
  static constexpr uint32_t kNeeded = kRing * kTileBytes + kQBytes + kPBytes + kBarBytes + kSmall;
  static constexpr uint32_t kBytes = kNeeded + 1024;
  static_assert(8 * kNumBars + 16 <= kBarBytes, "barrier area too small");
  static_assert(kCtasPerSm * (kBytes + 1024) <= 228 * 1024, "shared memory budget");
  static_assert(R * kD * 4 <= kTileBytes, "the partial result must fit in a ring slot");
};

template <int n> struct Tmem;                            // n columns of the warp's 32 lanes
template <> struct Tmem<4> {
  __device__ static __forceinline__ void ld(uint32_t a, uint32_t (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n\ttcgen05.wait::ld.sync.aligned;"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
  }
  __device__ static __forceinline__ void st(uint32_t a, const uint32_t (&r)[4]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%4], {%0, %1, %2, %3};"
                 :: "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(a) : "memory");
  }
};
template <> struct Tmem<8> {
  __device__ static __forceinline__ void ld(uint32_t a, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\ttcgen05.wait::ld.sync.aligned;"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(a) : "memory");
  }
  __device__ static __forceinline__ void st(uint32_t a, const uint32_t (&r)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};"
                 :: "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(a) : "memory");
  }
};

struct DecodeTParams {
  uint32_t spin_limit;       // polls a device-side wait may take
  int drop_k_tile;           // test hook: the K copy of this tile of every CTA is not issued (-1: none)
  int n_ranks;
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ float ld_peer(uint32_t local, uint32_t rank) {
  uint32_t a;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap* tm) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(tm) : "memory");
}
// Barrier 1 over the softmax warps; returns the OR of the predicate.
template <int kThreads> __device__ __forceinline__ bool softmax_sync_or(bool p) {
  uint32_t res;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 q, %1, 0;\n\t"
      "bar.red.or.pred p, 1, %2, q;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(res) : "r"(uint32_t(p)), "n"(kThreads) : "memory");
  return res != 0;
}
__device__ __forceinline__ void ld_peer4(uint32_t local, uint32_t rank, float (&v)[4]) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(a) : "memory");
}

// The two 16-bit halves of v to two places of shared memory.
__device__ __forceinline__ void st_pair(uint32_t a0, uint32_t a1, uint32_t v) {
  asm volatile("{\n\t.reg .b16 a, b;\n\tmov.b32 {a, b}, %2;\n\tst.shared.b16 [%0], a;\n\tst.shared.b16 [%1], b;\n\t}"
               ::"r"(a0), "r"(a1), "r"(v) : "memory");
}
// For every row r the reduction of v[r] over the warp, in 31 (R = 32) instead of 5 R shuffles: halves of the
// warp swap halves of the rows, quarters quarters, ...  Lane l ends up with row row_of_lane<R>(l); when R < 32,
// 32 / R neighbouring lanes hold the same one.
template <int R> __device__ __forceinline__ int row_of_lane(int lane) { return lane / (32 / R); }
template <int R, bool kMax>
__device__ __forceinline__ float reduce_rows(float (&v)[R], int lane) {
  auto op = [](float a, float b) { return kMax ? fmaxf(a, b) : a + b; };
  int o = 16;
#pragma unroll
  for (int h = R / 2; h >= 1; h >>= 1, o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const float send = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
      v[i] = op(keep, __shfl_xor_sync(0xffffffffu, send, o));
    }
  }
  float x = v[0];
#pragma unroll
  for (int q = 16 / R; q >= 1; q >>= 1) x = op(x, __shfl_xor_sync(0xffffffffu, x, q));
  return x;
}

template <int R, bool kDeep>
__global__ void __launch_bounds__(Cfg<R, kDeep>::kThreads, Cfg<R, kDeep>::kCtasPerSm)
attention_decode_t_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_kw,
                          const __grid_constant__ CUtensorMap tm_vw, const __grid_constant__ CUtensorMap tm_kp,
                          const __grid_constant__ CUtensorMap tm_vp, TcParams p, DecodeTParams dp) {
  using C = Cfg<R, kDeep>;
  constexpr int N = C::N, kRing = C::kRing, RS = C::RS, kThreads = C::kThreads, W0 = 4 * C::SG;      // W0: first warp after the softmax's
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  const uint32_t ring = base, q_smem = base + kRing * kTileBytes, p_smem = q_smem + C::kQBytes, bars = p_smem + C::kPBytes;
  const uint32_t bar_q = bars;
  // Position pos of the stream (K of tile i at 2 i, V at 2 i + 1) uses slot pos % kRing.  In an odd ring a slot
  // holds K and V tiles in turn, so the two have barriers of their own: whoever waits for a use has then itself
  // waited for the use before it on the same barrier, or issued a copy after such a wait, and cannot mistake the one
  // for the other.
  auto bar_full = [&](int pos) { return bars + 8u * (1 + 2 * (pos % kRing) + (pos & 1)); };
  auto bar_empty = [&](int pos) { return bars + 8u * (1 + 2 * kRing + 2 * (pos % kRing) + (pos & 1)); };
  auto parity = [](int pos) { return uint32_t(pos / (kRing % 2 ? 2 * kRing : kRing)) & 1u; };
  auto bar_sfull = [&](int b) { return bars + 8u * (1 + 4 * kRing + b); };
  auto bar_sfree = [&](int b) { return bars + 8u * (3 + 4 * kRing + b); };
  const uint32_t bar_pfull = bars + 8u * (5 + 4 * kRing), bar_pvdone = bar_pfull + 8u, bar_done = bar_pvdone + 8u,
                 bar_drain = bar_done + 8u;              // the Q K^T issuer's own, after a failed wait
  unsigned char* base_generic = smem_raw + (base - raw);
  unsigned char* bars_generic = base_generic + (bars - base);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars_generic + 8 * C::kNumBars);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bars_generic + 8 * C::kNumBars + 4);
  float* wred = reinterpret_cast<float*>(bars_generic + C::kBarBytes);   // [warp][row]
  float* ml = wred + 4 * R;                                              // [row] maximum, then [row] sum
  float* part = reinterpret_cast<float*>(base_generic);                  // [row][channel], over the ring at the end

  const int n_ranks = dp.n_ranks;
  const int rank = n_ranks > 1 ? int(cluster_rank()) : 0;
  const int g = blockIdx.x / n_ranks, unit = blockIdx.y;
  const int seq = unit / p.n_layers, layer_local = unit - seq * p.n_layers;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nt = p.a.n_tokens, G = p.group, rows = nt * G;

  grid_launch_dependents();          // the append makes its loads while this kernel runs
  // ---- the key stream
  const Geometry geo = make_geometry(p.a.pos0[seq], p.n_init, p.block, p.n_local_prev);
  const int local_len = int(geo.p0 - geo.local_start);
  GranuleKeys ks;
  ks.sel = p.a.sel_idx + (size_t(unit) * p.n_kv_heads + g) * p.cap_blocks;
  ks.pt = p.a.page_table + size_t(seq) * p.max_pages;
  ks.gpb = p.block / 16;
  ks.gpp_log2 = __ffs(p.page_tokens / 16) - 1;
  ks.g_init = geo.init_len / 16;
  ks.g_a = ks.g_init + (local_len + 15) / 16;            // the last local page may be partly filled
  ks.g_b = 0;
  ks.local0 = int(geo.local_start / 16);
  ks.n_cand = geo.n_cand; ks.block0 = p.n_init / 16; ks.max_pages = p.max_pages;
  ks.n_phys_pages = p.n_phys_pages; ks.page_base = layer_local * p.n_phys_pages;
  ks.n_heads = p.n_kv_heads; ks.head = g;
  ks.oob = (p.n_layers * p.n_phys_pages * p.n_kv_heads) << ks.gpp_log2;
  const int n_a = geo.init_len + local_len;               // exact: the tail of the last page is masked
  const int tiles_a = (n_a + kBN - 1) / kBN;
  const int n1 = tiles_a + 1;                             // tiles before the dependency wait: the past, the new tokens
  const int ksteps_new = (nt + 15) / 16;                  // 16-key steps of the tile of the new tokens
  int n_b = 0;
  auto share = [&](int n) { return (n - rank + n_ranks - 1) / n_ranks; };      // tiles j = i * n_ranks + rank < n
  const int early = share(n1);
  auto total_after_wait = [&](bool report) -> int {
    grid_dependency_wait();            // the selection is complete from here on
    int c = p.a.sel_count ? p.a.sel_count[unit] : 0;
    if (c < 0 || c > p.cap_blocks || c > geo.n_cand) {
      if (report) set_status(p.a.status, ACTQKV_DEV_BAD_SELECTION);
      c = max(0, min(c, min(p.cap_blocks, geo.n_cand)));
    }
    n_b = c * p.block;
    ks.g_b = c * ks.gpb;
    return share(n1 + (n_b + kBN - 1) / kBN);
  };
  auto wait_bar = [&](uint32_t bar, uint32_t parity) { return mbar_wait(bar, parity, abort_flag, dp.spin_limit); };

  // ---- set-up that depends on no earlier kernel
  if (warp == W0 && lane == 0) { prefetch_tensormap(&tm_q); prefetch_tensormap(&tm_kp); prefetch_tensormap(&tm_kw); }
  if (warp == W0 + 1 && lane == 0) { prefetch_tensormap(&tm_vp); prefetch_tensormap(&tm_vw); }
  const int first_row = warp == W0 || warp == W0 + 1       // the producers' first look-up, one granule per lane
      ? granule_a(ks, ((lane >> 3) * n_ranks + rank) * 8 + (lane & 7), p.a.status, warp == W0) : 0;
  if (tid == 0) {
    mbar_init(bar_q, 1);
    for (int s = 0; s < 2 * kRing; ++s) { mbar_init(bars + 8u * (1 + s), 1); mbar_init(bars + 8u * (1 + 2 * kRing + s), 1); }
    mbar_init(bar_sfull(0), 1); mbar_init(bar_sfull(1), 1);
    mbar_init(bar_sfree(0), W0); mbar_init(bar_sfree(1), W0);
    mbar_init(bar_pfull, W0); mbar_init(bar_pvdone, 1); mbar_init(bar_done, 1); mbar_init(bar_drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (rows < R) {           // rows of Q that hold no query: zeros
    for (int i = tid; i < 2 * (R - rows) * 8; i += kThreads) {
      const int half = i / ((R - rows) * 8), v = i % ((R - rows) * 8);
      *reinterpret_cast<uint4*>(base_generic + (q_smem - base) + half * (N * 128) + rows * 128 + v * 16) = make_uint4(0, 0, 0, 0);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == W0 + 3) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(C::kCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;                       // S buffers at 0 and N, O (hi columns, lo columns) at 2 N

  auto row_out = [&](int r) { return ((size_t(unit) * nt + r / G) * p.n_q_heads + g * G + r % G) * kD; };
  auto store_lse = [&](int r, float mm, float ll) {
    if (p.a.lse)
      p.a.lse[(size_t(unit) * p.n_q_heads + g * G + r % G) * nt + r / G] =
          ll == 0.f ? -INFINITY : (mm + log2f(ll)) * 0.6931471805599453f;
  };
  int issued = 0;                                         // tiles a producer has issued copies for
  if (warp == W0 || warp == W0 + 1) {
    // =========================== TMA producers ===========================
    const int is_v = warp - W0;
    const CUtensorMap* tm_pages = is_v ? &tm_vp : &tm_kp;
    const CUtensorMap* tm_win = is_v ? &tm_vw : &tm_kw;
    if (!is_v && lane == 0) {
      mbar_expect_tx(bar_q, 2u * uint32_t(rows) * 128u);
      tma_load_3d(q_smem, &tm_q, bar_q, 0, g * G, unit * nt);              // box: 64 channels x G heads x nt tokens
      tma_load_3d(q_smem + N * 128u, &tm_q, bar_q, 64, g * G, unit * nt);
    }
    __syncwarp();
    bool ok = true;
    auto claim = [&](int i, uint32_t bytes, uint32_t& full) -> uint32_t {
      const int pos = 2 * i + is_v, s = pos % kRing;
      if (pos >= kRing) ok = wait_bar(bar_empty(pos - kRing), parity(pos - kRing));
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) return 0;
      full = bar_full(pos);
      if (lane == 0 && (is_v || i != dp.drop_k_tile)) mbar_expect_tx(full, bytes);
      __syncwarp();
      return ring + s * kTileBytes;
    };
    // Tiles [i0, i1) of this CTA; the look-ups are taken 32 granules = 4 tiles at a time, one granule per
    // lane, ahead of their use.
    auto paged = [&](int i0, int i1, int first, auto&& row_of) {
      int cur = 0, next = first;
      for (int i = i0; i < i1 && ok; ++i) {
        if (((i - i0) & 3) == 0) cur = next;
        uint32_t full = 0;
        const uint32_t sbase = claim(i, kTileBytes, full);
        if (!ok) break;
        const int row = __shfl_sync(0xffffffffu, cur, ((i - i0) & 3) * 8 + (lane & 7));
        if (lane < 8 && (is_v || i != dp.drop_k_tile)) tma_load_5d(sbase + lane * 4096u, tm_pages, full, 0, 0, 0, 0, row);
        issued = i + 1;
        if (((i - i0) & 3) == 0) next = row_of(i + 4 + (lane >> 3), lane & 7);
      }
    };
    const int a_end = share(tiles_a);
    paged(0, a_end, first_row, [&](int i, int k) { return granule_a(ks, (i * n_ranks + rank) * 8 + k, p.a.status, !is_v); });
    if (a_end < early && ok) {                            // this rank has the new tokens
      uint32_t full = 0;
      const uint32_t sbase = claim(a_end, uint32_t(2 * ksteps_new) * 2048u, full);
      if (ok && lane < 2 * ksteps_new && (is_v || a_end != dp.drop_k_tile))
        tma_load_5d(sbase + lane * 2048u, tm_win, full, 0, lane * 8, 0, g, unit);      // (rows behind the unit's last token: zeros)
      __syncwarp();
      if (ok) issued = early;
    }
    if (ok) {
      // the page-table entries of every candidate block start their way into L2 while this warp waits
      if (!is_v) {
        const char* pt0 = reinterpret_cast<const char*>(ks.pt + p.n_init / p.page_tokens);
        const int lines = min(ks.max_pages - p.n_init / p.page_tokens, (ks.n_cand * ks.gpb) >> ks.gpp_log2) / 32;   // 32 entries per 128 bytes
        for (int l = lane; l < lines; l += 32)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(pt0 + size_t(l) * 128));
      }
      // the first entries of the selection are loaded together with its count
      const int gi0 = ((early + (lane >> 3)) * n_ranks + rank - n1) * 8 + (lane & 7), e0 = gi0 / ks.gpb;
      grid_dependency_wait();
      const int blk0 = e0 < p.cap_blocks ? ks.sel[e0] : -1;
      const int n_tiles = total_after_wait(!is_v && lane == 0);
      auto row_b = [&](int i, int k) { return granule_b(ks, (i * n_ranks + rank - n1) * 8 + k, p.a.status, !is_v); };
      paged(early, n_tiles, granule_b_of_block(ks, gi0, blk0, p.a.status, !is_v), row_b);
    }
  } else if (warp == W0 + 2) {
    // =========================== issuer of Q K^T ===========================
    constexpr uint32_t idesc_qk = make_idesc(false, 128, N);
    bool ok = wait_bar(bar_q, 0);
    int n_tiles = early;
    for (int i = 0; ok; ++i) {
      if (i == early) n_tiles = total_after_wait(false);
      if (i >= n_tiles) break;
      const int pos = 2 * i, s = pos % kRing;
      ok = wait_bar(bar_full(pos), parity(pos));
      if (i >= 2) ok = ok && wait_bar(bar_sfree(i & 1), (i / 2 - 1) & 1);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const uint32_t k_tile = ring + s * kTileBytes;
      if (elect_one()) {
#pragma unroll
        for (int k = 0; k < kD / 16; ++k)
          mma_ss(tmem + (i & 1) * N, make_desc(k_tile + (k >> 2) * 1024u + (k & 3) * 32u, 16u, 2048u),
                 make_desc(q_smem + (k >> 2) * (N * 128u) + (k & 3) * 32u, 16u, 1024u), idesc_qk, k > 0 ? 1u : 0u);
        tc_commit(bar_empty(pos));
        tc_commit(bar_sfull(i & 1));
      }
      __syncwarp();
    }
    if (!ok) {      // the products issued must be through before TMEM is freed
      if (elect_one()) tc_commit(bar_drain);
      __syncwarp();
      for (uint32_t n = 0; n < dp.spin_limit && !mbar_try_wait(bar_drain, 0); ++n) {}
    }
  } else if (warp == W0 + 3) {
    // =========================== issuer of P V ===========================
    constexpr uint32_t idesc_pv = make_idesc(false, 128, 2 * N) | (1u << 15);      // A (V) is MN-major
    bool ok = true;
    int n_tiles = early;
    for (int i = 0; ok; ++i) {
      if (i == early) n_tiles = total_after_wait(false);
      if (i >= n_tiles) break;
      const int pos = 2 * i + 1, s = pos % kRing, j = i * n_ranks + rank;
      ok = wait_bar(bar_full(pos), parity(pos));
      if (ok && j == tiles_a - 1 && (n_a & 15)) {
        // The rows behind p0 in the last granule of the local past may hold anything.  Their weight is 0, but 0 x NaN
        // is NaN: they become zeros here, where the tile is waited for anyway.
        uint4* granule = reinterpret_cast<uint4*>(base_generic + s * kTileBytes + ((n_a - j * kBN) >> 4) * 4096);
        for (int v = lane; v < 256; v += 32)              // [group of 8 rows][channel half][row][vector]
          if ((v >> 7) * 8 + ((v >> 3) & 7) >= (n_a & 15)) granule[v] = make_uint4(0, 0, 0, 0);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      }
      ok = ok && wait_bar(bar_pfull, i & 1);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const uint32_t v_tile = ring + s * kTileBytes;
      const int ksteps = j == n1 - 1 ? ksteps_new : kBN / 16;    // of the new tokens' tile only these keys were copied
      if (elect_one()) {
        for (int k = 0; k < ksteps; ++k)
          mma_ss(tmem + 2 * N, make_desc(v_tile + k * 4096u, 1024u, 2048u),
                 make_desc(p_smem + (k >> 2) * (2 * N * 128u) + (k & 3) * 32u, 16u, 1024u), idesc_pv, (i > 0 || k > 0) ? 1u : 0u);
        tc_commit(bar_empty(pos));
        tc_commit(bar_pvdone);
      }
      __syncwarp();
    }
    // the last P V depends, through the softmax, on every Q K^T
    if (elect_one()) tc_commit(bar_done);
    __syncwarp();
    if (!ok) for (uint32_t n = 0; n < dp.spin_limit && !mbar_try_wait(bar_done, 0); ++n) {}
  } else if (warp < W0) {
    // =========================== softmax ===========================
    // Thread = key of the tile.  P (hi rows, lo rows) goes to shared memory as the K-major operand of P V.
    const int q4 = warp & 3, g0 = (warp >> 2) * RS, mine = rows - g0;      // TMEM lane quadrant; the group's first row; rows from there on
    const uint32_t lane_addr = uint32_t(q4 * 32) << 16;
    const int key = q4 * 32 + lane;
    float m[RS], l[RS];
#pragma unroll
    for (int r = 0; r < RS; ++r) { m[r] = r < mine ? -INFINITY : 0.f; l[r] = 0.f; }      // (the score of a row without a query is 0)
    const uint32_t p_key = p_smem + uint32_t(key >> 6) * (2 * N * 128u) + uint32_t(g0 >> 3) * 1024u;
    const uint32_t p_col = uint32_t(key & 63) * 2u;
    bool ok = true;
    int n_tiles = early;
    for (int i = 0;; ++i) {
      if (i == early) n_tiles = total_after_wait(false);
      if (i >= n_tiles) break;
      const int j = i * n_ranks + rank;
      ok = ok && wait_bar(bar_sfull(i & 1), (i >> 1) & 1);
      ok = __all_sync(0xffffffffu, ok);
      tc_fence_after();
      uint32_t sr[RS];
      if (ok) {
        Tmem<RS>::ld(tmem + lane_addr + (i & 1) * N + g0, sr);
        tc_fence_before();
      }
      __syncwarp();
      if (ok && lane == 0) mbar_arrive(bar_sfree(i & 1));
      // d: the score in powers of two over the maximum in use.  Key k is valid for row r up to the tile's end, in the
      // new tokens' tile up to the row's own token; most tiles are valid as a whole.
      const int left = j < tiles_a ? n_a - j * kBN : j < n1 ? 0 : n_b - (j - n1) * kBN;      // valid keys; 0: new tokens
      auto on = [&](int r) { return left > 0 ? key < left : key < nt && key * G <= g0 + r; };
      float d[RS];
      bool grow = false;
      auto weigh = [&]() {
#pragma unroll
        for (int r = 0; r < RS; ++r) d[r] = fmaf(__uint_as_float(sr[r]), p.scale_log2, -m[r]);
        if (left < kBN)
#pragma unroll
          for (int r = 0; r < RS; ++r) d[r] = on(r) ? d[r] : -INFINITY;
#pragma unroll
        for (int r = 0; r < RS; ++r) grow |= d[r] > kMaxLag;
      };
      weigh();
      if (softmax_sync_or<128 * C::SG>(grow || !ok)) {
        // a new maximum for every row, over the tile and the old one
        {
          float top[RS];
#pragma unroll
          for (int r = 0; r < RS; ++r) top[r] = on(r) ? __uint_as_float(sr[r]) * p.scale_log2 : -INFINITY;
          const float w = reduce_rows<RS, true>(top, lane);
          wred[q4 * R + g0 + row_of_lane<RS>(lane)] = w;
        }
        if (softmax_sync_or<128 * C::SG>(!ok)) { ok = false; break; }
        float f[RS];
        bool moved = false;
#pragma unroll
        for (int r = 0; r < RS; ++r) {
          const float top = fmaxf(fmaxf(wred[g0 + r], wred[R + g0 + r]), fmaxf(wred[2 * R + g0 + r], wred[3 * R + g0 + r]));
          f[r] = 1.f;
          if (top > m[r]) {
            f[r] = m[r] == -INFINITY ? 0.f : ex2(m[r] - top);
            m[r] = top;
            l[r] *= f[r];
            moved = true;
          }
        }
        if (i > 0 && moved) {                             // the same for all threads of the group
          ok = wait_bar(bar_pvdone, (i - 1) & 1);         // O must be quiescent
          ok = __all_sync(0xffffffffu, ok);
          if (ok) {
            tc_fence_after();
#pragma unroll
            for (int part_i = 0; part_i < 2; ++part_i) {
              const uint32_t a = tmem + lane_addr + (2 + part_i) * N + g0;
              uint32_t o[RS];
              Tmem<RS>::ld(a, o);
#pragma unroll
              for (int r = 0; r < RS; ++r) o[r] = __float_as_uint(__uint_as_float(o[r]) * f[r]);
              Tmem<RS>::st(a, o);
            }
            tmem_wait_st();
          }
        }
        if (softmax_sync_or<128 * C::SG>(!ok)) { ok = false; break; }  // (also: wred is read before the next tile writes it)
        weigh();
      }
      uint32_t hi[RS / 2], lo[RS / 2];
#pragma unroll
      for (int r = 0; r < RS; r += 2) {
        const float e0 = ex2(d[r]), e1 = ex2(d[r + 1]);
        l[r] += e0;
        l[r + 1] += e1;
        const uint32_t h = pack_bf16(e0, e1);
        hi[r / 2] = h;
        lo[r / 2] = pack_bf16(e0 - __uint_as_float(h << 16), e1 - __uint_as_float(h & 0xFFFF0000u));
      }
      if (i > 0) {                                        // P V of the tile before has read its P
        ok = ok && wait_bar(bar_pvdone, (i - 1) & 1);
        ok = __all_sync(0xffffffffu, ok);
      }
      if (ok) {
#pragma unroll
        for (int r = 0; r < RS; r += 2) {
          constexpr uint32_t kLo = N * 128u;              // rows N .. 2N - 1
          const uint32_t row = p_key + r * 128u;
          st_pair(row + (p_col ^ (r * 16u)), row + 128u + (p_col ^ (r * 16u + 16u)), hi[r / 2]);
          st_pair(row + kLo + (p_col ^ (r * 16u)), row + kLo + 128u + (p_col ^ (r * 16u + 16u)), lo[r / 2]);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
      }
      __syncwarp();
      if (ok && lane == 0) mbar_arrive(bar_pfull);
      // a warp that gave up here leaves through the vote of the next tile, or of the end
      if (!ok) *abort_flag = 1;
    }
    if (ok && n_tiles > 0) ok = wait_bar(bar_done, 0);
    ok = __all_sync(0xffffffffu, ok);
    // ---- sums over the keys, then thread = channel
    wred[q4 * R + g0 + row_of_lane<RS>(lane)] = reduce_rows<RS, false>(l, lane);
    ok = !softmax_sync_or<128 * C::SG>(!ok);
    tc_fence_after();
    const bool have = ok && n_tiles > 0;
    float o[RS];
    if (have) {
      uint32_t hi[RS], lo[RS];
      Tmem<RS>::ld(tmem + lane_addr + 2 * N + g0, hi);
      Tmem<RS>::ld(tmem + lane_addr + 3 * N + g0, lo);
#pragma unroll
      for (int r = 0; r < RS; ++r) o[r] = __uint_as_float(hi[r]) + __uint_as_float(lo[r]);
    } else {
#pragma unroll
      for (int r = 0; r < RS; ++r) o[r] = 0.f;
    }
#pragma unroll
    for (int r = 0; r < RS; ++r) l[r] = have ? (wred[g0 + r] + wred[R + g0 + r]) + (wred[2 * R + g0 + r] + wred[3 * R + g0 + r]) : 0.f;
    if (n_ranks == 1) {
#pragma unroll
      for (int r = 0; r < RS; ++r) {
        if (r >= mine) break;
        const size_t at = row_out(g0 + r) + key;
        const float v = l[r] == 0.f ? 0.f : o[r] / l[r];      // (a sum that is not a number stays one)
        if (p.out_bf16) static_cast<__nv_bfloat16*>(p.a.out)[at] = __float2bfloat16_rn(v);
        else static_cast<float*>(p.a.out)[at] = v;
        if (key == r) store_lse(g0 + r, m[r], l[r]);
      }
    } else {
      // the ranks' partial results meet: O over the ring, which no copy or product uses any more -- unless a wait gave
      // up: copies may then still be landing there, and the merge reads from the rank's sum of 0 that there is nothing
#pragma unroll
      for (int r = 0; r < RS; ++r) {
        part[(g0 + r) * kD + key] = o[r];
        if (key == r) { ml[g0 + r] = have ? m[r] : -INFINITY; ml[R + g0 + r] = l[r]; }
      }
      __syncwarp();
      cluster_sync_all();
    }
  }
  __syncwarp();
  if (n_ranks > 1) {
    if (warp >= W0) cluster_sync_all();      // the softmax warps' first one
    // every rank finishes an equal share of the (row, V channels) items
    constexpr int V = R < 16 ? 1 : 4;                   // few rows: one channel each is a single round, with fewer registers
    const int items = rows * (kD / V), chunk = (items + n_ranks - 1) / n_ranks, end = min(items, (rank + 1) * chunk);
    for (int e = rank * chunk + tid; e < end; e += kThreads) {
      const int r = e / (kD / V), ch = V * (e % (kD / V));
      float pm[kMaxRanks], pl[kMaxRanks], po[kMaxRanks][V], mm = -INFINITY;
#pragma unroll
      for (int k = 0; k < kMaxRanks; ++k)
        if (k < n_ranks) {
          pm[k] = ld_peer(smem_u32(ml + r), k);
          pl[k] = ld_peer(smem_u32(ml + R + r), k);
          if constexpr (V == 1) po[k][0] = ld_peer(smem_u32(part + r * kD + ch), k);
          else ld_peer4(smem_u32(part + r * kD + ch), k, reinterpret_cast<float(&)[4]>(po[k]));
        }
#pragma unroll
      for (int k = 0; k < kMaxRanks; ++k)
        if (k < n_ranks) mm = fmaxf(mm, pm[k]);
      float ll = 0.f, oo[V] = {};
#pragma unroll
      for (int k = 0; k < kMaxRanks; ++k)
        if (k < n_ranks) {
          if (pl[k] == 0.f) continue;       // an empty partial result, whatever its O holds
          const float w = ex2(pm[k] - mm);
          ll = fmaf(w, pl[k], ll);
#pragma unroll
          for (int v = 0; v < V; ++v) oo[v] = fmaf(w, po[k][v], oo[v]);
        }
#pragma unroll
      for (int v = 0; v < V; ++v) oo[v] = ll == 0.f ? 0.f : oo[v] / ll;
      const size_t at = row_out(r) + ch;
      if constexpr (V == 1) {
        if (p.out_bf16) static_cast<__nv_bfloat16*>(p.a.out)[at] = __float2bfloat16_rn(oo[0]);
        else static_cast<float*>(p.a.out)[at] = oo[0];
      } else if (p.out_bf16) {
        *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(p.a.out) + at) =
            make_uint2(pack_bf16(oo[0], oo[1]), pack_bf16(oo[2], oo[3]));
      } else {
        *reinterpret_cast<float4*>(static_cast<float*>(p.a.out) + at) = make_float4(oo[0], oo[1], oo[2], oo[3]);
      }
      if (ch == 0) store_lse(r, mm, ll);
    }
    cluster_sync_all();                     // a peer may still read this CTA's part
  }

  // ---- teardown
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // a wait gave up: what the producers issued must have landed before the CTA leaves (in the normal course
    // every tile was consumed)
    if (tid == 0) set_status(p.a.status, ACTQKV_DEV_TIMEOUT);
    if (warp == W0 || warp == W0 + 1) {
      for (int i = max(0, issued - (kRing + 1) / 2); i < issued; ++i) {
        if (warp == W0 && i == dp.drop_k_tile) continue;
        const int pos = 2 * i + (warp - W0);
        for (uint32_t n = 0; n < dp.spin_limit && !mbar_try_wait(bar_full(pos), parity(pos)); ++n) {}
      }
      if (warp == W0) for (uint32_t n = 0; n < dp.spin_limit && !mbar_try_wait(bar_q, 0); ++n) {}
    }
    __syncthreads();
  }
  if (warp == W0 + 3) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::kCols));
  }
}

template <int R, bool kDeep>
int launch(const CUtensorMap* tm, const TcParams& p, const DecodeTParams& dp, int units, cudaStream_t st) {
  auto kern = attention_decode_t_kernel<R, kDeep>;
  static std::atomic<bool> opted_in[kMaxDevices];
  if (!opt_in_shared_memory(kern, int(Cfg<R, kDeep>::kBytes), opted_in)) return ACTQKV_ERR_LAUNCH;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(p.n_kv_heads * dp.n_ranks, units, 1);
  lc.blockDim = dim3(Cfg<R, kDeep>::kThreads, 1, 1);
  lc.dynamicSmemBytes = Cfg<R, kDeep>::kBytes;
  lc.stream = st;
  cudaLaunchAttribute attr[2];
  allow_early_launch(attr[0]);
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = dp.n_ranks;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  lc.attrs = attr;
  lc.numAttrs = 2;
  if (cudaLaunchKernelEx(&lc, kern, tm[0], tm[1], tm[2], tm[3], tm[4], p, dp) != cudaSuccess) return ACTQKV_ERR_LAUNCH;
  return launch_status();
}

}  // namespace

namespace actqkv {

bool attention_decode_t_supported(const actqkv_config* cfg, int n_tokens) {
  const int P = cfg->page_tokens;
  return cfg->dtype == ACTQKV_BF16 && cfg->head_dim == kD && (P == 16 || P == 32 || P == 64 || P == 128) &&
         cfg->n_local_prev % 16 == 0 && n_tokens * (cfg->n_q_heads / cfg->n_kv_heads) <= kMaxRows;
}

// n_ranks: CTAs that share a key stream (at most 8); 0 chooses: doubled as long as all CTAs are resident at once.
int launch_attention_decode_t(const actqkv_config* cfg, const Batch& b, const AttnArgs& a, int n_ranks, cudaStream_t st) {
  const int U = b.units(), nt = a.n_tokens, Hq = cfg->n_q_heads, Hkv = cfg->n_kv_heads, G = Hq / Hkv, rows = nt * G;
  CUtensorMap tm[5];
  const cuuint64_t dims[3] = {cuuint64_t(kD), cuuint64_t(Hq), cuuint64_t(U) * nt};
  const cuuint64_t str[2] = {cuuint64_t(kD) * 2, cuuint64_t(Hq) * kD * 2};
  const cuuint32_t box[3] = {64, cuuint32_t(G), cuuint32_t(nt)};
  const uint64_t granules = uint64_t(b.n_layers) * cfg->n_phys_pages * Hkv * (cfg->page_tokens / 16);
  if (!encode(&tm[0], a.q, 3, dims, str, box) || !encode_unit_groups(&tm[1], a.k_win, U, nt, Hkv) ||
      !encode_unit_groups(&tm[2], a.v_win, U, nt, Hkv) || !encode_granules(&tm[3], a.k_pages, granules) ||
      !encode_granules(&tm[4], a.v_pages, granules))
    return ACTQKV_ERR_LAUNCH;
  TcParams p;
  p.a = a;
  p.n_q_heads = Hq; p.n_kv_heads = Hkv; p.group = G; p.block = cfg->block; p.n_init = cfg->n_init;
  p.n_local_prev = cfg->n_local_prev; p.cap_blocks = cfg->cap_blocks; p.max_pages = cfg->max_pages;
  p.n_phys_pages = cfg->n_phys_pages; p.n_layers = b.n_layers; p.out_bf16 = cfg->out_dtype == ACTQKV_BF16;
  p.page_tokens = cfg->page_tokens;
  const float scale = cfg->sm_scale > 0.f ? cfg->sm_scale : 1.f / sqrtf(float(kD));
  p.scale_log2 = scale * 1.4426950408889634f;
  DecodeTParams dp;
  dp.spin_limit = cfg->test_wait_limit > 0 ? uint32_t(cfg->test_wait_limit) : 1u << 20;
  dp.drop_k_tile = cfg->test_wait_limit > 0 ? cfg->test_drop_k_tile : -1;
  // Ranks: doubled while all clusters are resident with an SM to each CTA (two sequences of 8 KV heads, 2,500 / 30,000
  // tokens: 22.5 / 28.6 us over 8 CTAs each, which are two waves, 15.0 / 20.4 us over 4); one more doubling where two CTAs share an SM only then
  // (75 to 148 streams), so that no SM is left idle beside a busy one.
  const int64_t pairs = int64_t(U) * Hkv;
  if (n_ranks <= 0) {
    n_ranks = 1;
    while (n_ranks < kMaxRanks && pairs <= resident_clusters(n_ranks * 2)) n_ranks *= 2;
    if (rows <= 16 && n_ranks == 1 && pairs <= kNumSMs) n_ranks = 2;
  }
  dp.n_ranks = std::min(n_ranks, kMaxRanks);
  const bool deep = pairs * dp.n_ranks <= kNumSMs;
#define ACTQKV_DECODE_T(R) (deep ? launch<R, true>(tm, p, dp, U, st) : launch<R, false>(tm, p, dp, U, st))
  return rows <= 4 ? ACTQKV_DECODE_T(4) : rows <= 8 ? ACTQKV_DECODE_T(8) : rows <= 16 ? ACTQKV_DECODE_T(16)
       : launch<32, true>(tm, p, dp, U, st);
#undef ACTQKV_DECODE_T
}

}  // namespace actqkv
