// Step 4: dynamic KV cut-off (Eq. 12) and top-c block selection (Algorithm 1, last loop).
//
// No host round trip.  A call that batches several layers runs two kernels:
//   cutoff_chain_kernel  one CTA per sequence.  Warps evaluate (or read) the per-head
//                        information densities of every batched layer, then one thread walks
//                        the layers shallow -> deep in fp64: B^l from Eq. 12, the granted
//                        integer c^l, the running B_kv and the density history.
//   select_kernel        one CTA per (unit, KV head).  Scores become order-preserving 32-bit
//                        keys in shared memory; up to 384 keys (256 where 256 threads hold
//                        them) are ranked against one another, of more the c-th largest is found
//                        by a search on the bits; equal keys are admitted lowest index first; the
//                        survivors are compacted in ascending block order.
// A call for one layer (the usual layer-by-layer use) runs select_kernel alone: the Hkv CTAs of a
// sequence form a thread-block cluster, each takes its head's density, they exchange the values
// through distributed shared memory, every CTA evaluates Eq. 12 for itself and the first one
// writes the budget state back.  Behind bias + probe of a window it takes the scores of a small table, too.
#include "common.cuh"
#include "stages.cuh"

using namespace actqkv;

namespace {

constexpr int kChainThreads = 1024;

struct ChainParams {
  const float* scores;
  const float* theta_in;   // NULL: compute from scores
  float* theta_out;        // written when computed here
  const int32_t* n_cand;
  double* state;
  int32_t* sel_count;
  float* budget_real;
  int n_kv_heads, n_cap, L, Lb, layer0, k_blocks, cap_blocks, thetabar_mode;
  float beta;
  uint32_t polls;          // bound of a device-side wait
  int drop;                // test hook: what select_kernel never sends (-1: nothing)
};

// Eq. 12 for one layer with n > 0 candidates: returns the granted count c and the un-rounded
// budget; `rest` = sum over the deeper layers of their mean density (theta-bar).
struct Grant { int c; double real; };
__device__ __forceinline__ Grant grant_layer(double th, double rest, double b_rem, int layers_left, int n, int cap) {
  Grant gr;
  const double den = th + rest;
  gr.real = den > 0.0 ? th / den * b_rem : b_rem / double(layers_left);
  const double fl = floor(gr.real + 0.5);
  int c = fl > 2.0e9 ? 2000000000 : (fl < -2.0e9 ? -2000000000 : int(fl));
  gr.c = max(min(1, n), min(c, min(cap, n)));
  return gr;
}

__global__ void __launch_bounds__(kChainThreads) cutoff_chain_kernel(ChainParams p) {
  extern __shared__ float theta_h[];   // [Lb][Hkv]
  const int seq = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  grid_launch_dependents();
  grid_dependency_wait();            // scores / densities come from the stream's previous kernels
  const int n = min(p.n_cand[seq], p.n_cap);
  if (p.theta_in) {                  // one load per thread, all in flight together
    const float* src = p.theta_in + size_t(seq) * p.Lb * p.n_kv_heads;
    for (int pair = threadIdx.x; pair < p.Lb * p.n_kv_heads; pair += kChainThreads) theta_h[pair] = src[pair];
  } else {
    for (int pair = warp; pair < p.Lb * p.n_kv_heads; pair += kChainThreads / 32) {
      const size_t uh = size_t(seq) * p.Lb * p.n_kv_heads + pair;
      const float th = warp_entropy(p.scores + uh * p.n_cap, n, p.beta);
      if (lane == 0) {
        if (p.theta_out) p.theta_out[uh] = th;
        theta_h[pair] = th;
      }
    }
  }
  __syncthreads();

  // Shared work arrays after the densities: doubles [Lb] th, [L + 1] suffix of known theta-bars,
  // [L + 1] suffix count of layers without one, [Lb] ratio.
  double* th_l = reinterpret_cast<double*>(theta_h + ((p.Lb * p.n_kv_heads + 1) & ~1));
  double* suf_known = th_l + p.Lb;
  double* suf_open = suf_known + p.L + 1;
  double* ratio = suf_open + p.L + 1;
  double* st = p.state + size_t(seq) * (1 + 2 * p.L);
  double* hist_sum = st + 1;
  double* hist_cnt = st + 1 + p.L;
  const int tid = threadIdx.x;
  // ---- in parallel: each batched layer's density (mean over its KV heads, fixed order)
  if (tid < p.Lb) {
    double s = 0.0;
    for (int g = 0; g < p.n_kv_heads; ++g) s += double(theta_h[tid * p.n_kv_heads + g]);
    th_l[tid] = s / double(p.n_kv_heads);
  }
  __syncthreads();
  // ---- in parallel: theta-bar of every model layer that has one (its history mean, or this call's
  // own density in the Algorithm-1 reading); the others will take the current layer's density
  if (tid < p.L) {
    double known = 0.0, open = 0.0;
    if (p.thetabar_mode == ACTQKV_THETABAR_ALG1) known = th_l[tid - p.layer0];
    else if (hist_cnt[tid] > 0.0) known = hist_sum[tid] / hist_cnt[tid];
    else open = 1.0;
    suf_known[tid] = known;          // turned into suffix sums below
    suf_open[tid] = open;
  }
  __syncthreads();
  if (tid < 2) {                     // suffix[j] = sum over layers >= j (additions only, running sum in a register)
    double* suf = tid == 0 ? suf_known : suf_open;
    double run = 0.0;
    suf[p.L] = 0.0;
    for (int j = p.L - 1; j >= 0; --j) {
      run += suf[j];
      suf[j] = run;
    }
  }
  __syncthreads();
  // ---- in parallel: the share theta / (theta + sum of deeper theta-bars) of Eq. 12, which does
  // not depend on the running budget
  if (tid < p.Lb) {
    const int layer = p.layer0 + tid;
    const double th = th_l[tid];
    const double den = th + suf_known[layer + 1] + suf_open[layer + 1] * th;
    ratio[tid] = den > 0.0 ? th / den : -1.0;
  }
  __syncthreads();
  // ---- serial: the budget walks the layers shallow -> deep
  if (tid == 0) {
    double b_rem = st[0];
    const double lo_d = double(min(1, n)), hi_d = double(min(p.cap_blocks, n));
    for (int l = 0; l < p.Lb; ++l) {
      const int layer = p.layer0 + l;
      if (layer == 0) b_rem = double(p.L) * double(p.k_blocks);
      int c = 0;
      double real = 0.0;
      if (n > 0) {
        // The count stays a double on the path from one layer's budget to the next (the clamp
        // bounds are small integers, so clamping the double and converting gives the same count
        // as converting and clamping; a NaN budget counts as 0 before the clamp, as a conversion
        // to int would make it); the integer for the store is taken off that path.
        real = ratio[l] >= 0.0 ? ratio[l] * b_rem : b_rem / double(p.L - layer);
        const double fl = floor(real + 0.5);
        const double cd = fmax(lo_d, fmin(fl == fl ? fl : 0.0, hi_d));
        b_rem -= cd;
        c = int(cd);
      }
      const size_t unit = size_t(seq) * p.Lb + l;
      p.sel_count[unit] = c;
      if (p.budget_real) p.budget_real[unit] = float(real);
    }
    st[0] = b_rem;
  }
  if (tid < p.Lb && n > 0) {         // density history of the layers of this call
    hist_sum[p.layer0 + tid] += th_l[tid];
    hist_cnt[p.layer0 + tid] += 1.0;
  }
}

// Order-preserving key: larger score <-> larger unsigned key; NaN lowest; -0 == +0.
__device__ __forceinline__ uint32_t score_key(float f) {
  if (f != f) return 0u;
  if (f == 0.f) f = 0.f;
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// The threads of select_kernel that hold keys (the control warp behind them takes no part).
template <int kKeys>
__device__ __forceinline__ void key_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kKeys) : "memory"); }

// Exclusive scan of one int per key thread; returns the prefix.
template <int kKeys>
__device__ __forceinline__ int key_exclusive_scan(int v, int* warp_tot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  key_sync<kKeys>();
  if (lane == 31) warp_tot[warp] = inc;
  key_sync<kKeys>();
  const int before = __reduce_add_sync(0xffffffffu, lane < warp ? warp_tot[lane] : 0);
  return before + inc - v;
}

// The largest threshold thr that at least c of the keys reach (0 < c < their number), three or four bits per step: warp
// w counts the keys of at least thr | w << shift (w >= 1), all of them, the first 256 from registers.  Done
// early when exactly c keys reach thr.  Returns thr; at: the number of keys that reach it.  keys: padded with
// zeros to 4 * n4, n4 a multiple of 32; tot: one count per warp, two sets used in turn.
template <int kKeys>
__device__ __forceinline__ uint32_t search_cth(int c, const uint32_t* keys, int n4, int (*tot)[kKeys / 32], int& at) {
  constexpr int kWarps = kKeys / 32, kBits = kWarps == 16 ? 4 : 3;
  static_assert(kWarps == 1 << kBits, "a threshold per warp");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint4* k4 = reinterpret_cast<const uint4*>(keys) + lane;
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u), a = k4[0], b = n4 > 32 ? k4[32] : zero;
  uint32_t thr = 0u;
  int turn = 0;
  for (int shift = 32 - kBits;; shift -= kBits) {
    const int sh = max(shift, 0), top = (1 << (kBits + min(shift, 0))) - 1;      // the last step may have fewer bits
    const uint32_t t = thr | (uint32_t(warp) << sh);
    auto reach = [&](const uint4& x) { return (int(x.x >= t) + int(x.y >= t)) + (int(x.z >= t) + int(x.w >= t)); };
    int cnt = reach(a) + reach(b);
    for (int i = 64; i < n4; i += 32) cnt += reach(k4[i]);
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0) tot[turn][warp] = cnt;
    key_sync<kKeys>();
    const int mine = tot[turn][lane & (kWarps - 1)];                   // counts fall with w
    const int w = __popc(__ballot_sync(0xffffffffu, lane >= 1 && lane <= top && mine >= c));
    const int reached = __shfl_sync(0xffffffffu, mine, w);
    if (w > 0) { thr |= uint32_t(w) << sh; at = reached; }
    if (at == c || sh == 0) return thr;
    turn ^= 1;
  }
}

// How many of the n keys (padded with zeros to a multiple of 4) come before key k of index i: larger ones, and equal
// ones of a lower index.  The keys of the warps before and behind the own one need one comparison each.
__device__ __forceinline__ int rank_of(uint32_t k, int i, const uint32_t* keys, int n) {
  const uint4* k4 = reinterpret_cast<const uint4*>(keys);
  const int own = (i & ~31) >> 2, end = (n + 3) >> 2;
  int r = 0;
#pragma unroll 4
  for (int j = 0; j < own; ++j) {
    const uint4 x = k4[j];
    r += (int(x.x >= k) + int(x.y >= k)) + (int(x.z >= k) + int(x.w >= k));
  }
#pragma unroll 4
  for (int j = own; j < end; ++j) {
    const uint4 x = k4[j];
    r += (int(x.x > k) + int(x.y > k)) + (int(x.z > k) + int(x.w > k));
  }
  const uint32_t same = __match_any_sync(0xffffffffu, k);              // equal keys inside the warp
  return r + __popc(same & ((1u << (i & 31)) - 1u));
}

// Waits (bounded) for phase 0 of an mbarrier.
__device__ __forceinline__ bool wait_phase0(uint32_t bar, uint32_t polls) {
  for (uint32_t i = 0; i < polls; ++i) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\tselp.b32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar) : "memory");
    if (ok) return true;
  }
  return false;
}

// kFused: the call holds one layer; the grid is launched as clusters of n_kv_heads CTAs (one
// sequence each) and the cut-off chain of that layer is evaluated here (ch), else sel_count is
// an input written by cutoff_chain_kernel.
//
// A chain of short phases on the critical path of a step, once per launch.  kKeys threads hold the keys, one warp
// behind them (control) the chain: the key warps fetch the scores and leave one (maximum, Z, sum e x) per slot; control
// merges these into the head's density, hands it to the cluster's CTAs by asynchronous remote stores that complete on
// their barriers, adds up theirs and grants the count in fp64.  Meanwhile the key warps rank their keys against all
// others, which needs no count; with the count a key is taken if its rank is below it, and one scan over the warps'
// ballots places it.  Beyond kRankMax candidates (or a key per thread) the n^2 comparisons are longer than the chain beside them, and the
// c-th largest key is found instead by a search on its bits (a threshold per warp and step), which ends as soon as a
// threshold separates exactly c keys.  Score and selection of one layer, 60 of these pairs chained in a graph, us per pair
// at 128 / 251 / 313 / 384 / 450 / 512 candidates: ranks 4.6 / 5.6 / 6.2 / 7.0 / 8.2 / 8.7, search 5.9 / 6.0 / 6.6 / 6.8 / 6.9 /
// 6.6; with four sequences ranks 5.3 / 6.8 / 9.2 / 10.5 / 15.6 / 18.0, search 6.4 / 9.0 / 11.1 / 11.7 / 13.6 / 14.5.  With one thread
// taking the density, a cluster barrier and a three-bit search after the count: 6.9 / 7.5 / 8.0 / 8.2 / 8.4 / 8.3 and 7.5 /
// 9.5 / 12.9 / 13.7 / 14.9 / 15.2.
// What is left is bound by the first fetch of the instructions, so the kernel goes through all
// phases once before the dependency wait, on 32 made-up scores and without a global access (the rehearsal), and again
// after it.
constexpr int kRankMax = 384;

// The scores of one layer taken inside the selection (D > 0): blocks of 1 KiB, mean aggregation.
struct ScoreArgs {
  const float* probe_kv;
  const void* repr_k;
  const float* repr_inv_norm;
  float* scores_out;
  int r;
};
constexpr uint32_t kGroupBytes = 4096;               // four blocks
constexpr int kScoreKeys = 256;                      // key threads of that form
constexpr int kScoreMaxCap = 128, kScoreMaxHeads = 16;
constexpr int kScoreSlots = kScoreMaxCap / 4 / (kScoreKeys / 32);       // groups of a key warp at most
constexpr int kScoreSmem = 136 * 1024;               // 1 + 4 + 128.3 KiB at kScoreMaxCap and eight rows a block
constexpr int kMaxKeysSmem = 200 * 1024;             // 25,600 rows
// scores and keys, then the inverse norms, the groups and a barrier for each
__host__ __device__ inline size_t keys_bytes(int n_cap) { return (size_t(n_cap) + 127) / 128 * 128 * 8; }
__host__ __device__ inline size_t norms_bytes(int n_cap, int r) { return (size_t(n_cap) * r * 4 + 127) / 128 * 128; }
__host__ __device__ inline int slots_of(int n_cap) { return (n_cap + 4 * (kScoreKeys / 32) - 1) / (4 * (kScoreKeys / 32)); }

// kCols: slots of the density that a key warp sums.
template <bool kFused, int kKeys, int kCols, typename T, int D>
__global__ void __launch_bounds__(kKeys + 32)
select_kernel(const float* __restrict__ scores, const int32_t* __restrict__ n_cand,
              int32_t* __restrict__ sel_count, int32_t* __restrict__ sel_idx, int n_kv_heads,
              int n_cap, int cap_blocks, int n_layers, int32_t* status, ChainParams ch, ScoreArgs sa) {
  extern __shared__ __align__(128) uint32_t sel_smem[];       // the head's scores [n_cap] (fp32), then their keys, each padded to a multiple of 128
  constexpr int kWarps = kKeys / 32;
  __shared__ int warp_tot[2][kWarps];
  __shared__ float sh_thetas[2][8];            // the densities of the cluster's heads (written by their CTAs), one set per pass
  __shared__ __align__(8) uint64_t sh_bar[2];  // a pass's densities have arrived
  // Eq. 11 is summed in 16 slots, the scores i = 32 v .. 32 v + 31 (mod 512) in slot v, one per warp or two, so that a density
  // does not depend on the number of key threads, which goes by the size of the batch.  (256 candidates fill 8 slots.)
  constexpr int kSlots = kWarps * kCols;
  __shared__ float red_m[kSlots], red_z[kSlots], red_e[kSlots];
  __shared__ int sh_count, sh_late;            // the granted count; a wait ran out
  const int g = blockIdx.x, unit = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool control = warp == kWarps;
  auto smem = [](const void* x) { return uint32_t(__cvta_generic_to_shared(x)); };
  // A peer's shared memory may be written only once that peer runs: every CTA says so here, and waits for
  // the others just ahead of its first remote store.
  if constexpr (kFused) {
    if (tid == 0) sh_late = 0;
    if (control && lane < 2) {
      const uint32_t bytes = 4u * uint32_t(n_kv_heads), bar = smem(sh_bar + lane);
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar));
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
    }
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  }
  grid_launch_dependents();
  const int n_given = n_cand[unit / n_layers], n_real = min(n_given, n_cap);
  const bool ranked = n_real <= min(kRankMax, kKeys);
  const float* s = scores + (size_t(unit) * n_kv_heads + g) * n_cap;
  int32_t* out = sel_idx + (size_t(unit) * n_kv_heads + g) * cap_blocks;
  float* sc = reinterpret_cast<float*>(sel_smem);
  uint32_t* keys = sel_smem + (n_cap + 127) / 128 * 128;
  // ---- the scores' table: key warp w owns groups w, w + kWarps, ... of four blocks; they and the inverse norms come ahead
  // of the dependency wait
  constexpr int VN = 16 / sizeof(T), DD = D > 0 ? D : 128, LPR = DD / VN, RPP = 32 / LPR;
  const size_t head = size_t(unit) * n_kv_heads + g;
  unsigned char* after_keys = reinterpret_cast<unsigned char*>(sel_smem) + keys_bytes(n_cap);
  float* norms = reinterpret_cast<float*>(after_keys);
  unsigned char* groups = after_keys + norms_bytes(n_cap, sa.r);
  uint64_t* group_bar = reinterpret_cast<uint64_t*>(groups + size_t(kWarps) * slots_of(n_cap) * kGroupBytes) + warp * kScoreSlots;
  groups += size_t(warp) * slots_of(n_cap) * kGroupBytes;
  if constexpr (D > 0) {
    static_assert(kKeys == kScoreKeys, "the groups are laid out for its warps");
    if (!control) {
      if (lane < kScoreSlots) {                      // a lane per group
        const uint32_t bar = smem(group_bar + lane);
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        const int b = 4 * (warp + lane * kWarps), nb = min(4, n_real - b);
        if (nb > 0 && !(b == 0 && ch.drop == n_kv_heads + g)) {
          const uint32_t bytes = uint32_t(nb) * 1024u;
          const unsigned char* src = static_cast<const unsigned char*>(sa.repr_k) + (head * n_cap + b) * 1024;
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
          asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                       ::"r"(smem(groups + lane * kGroupBytes)), "l"(src), "r"(bytes), "r"(bar) : "memory");
        }
      }
      __syncwarp();
      const float* inv = sa.repr_inv_norm + head * n_cap * sa.r;
      for (int i = tid; i < n_real * sa.r; i += kKeys) norms[i] = __ldg(inv + i);
    } else if (lane == 0 && g == 0 && n_given > n_cap) {
      set_status(status, ACTQKV_DEV_NCAND_CLAMPED);
    }
  }
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    asm volatile("" : "+r"(pass));             // one body for both passes
    const bool real = pass != 0;
    if (real) grid_dependency_wait();          // scores / densities / counts come from the stream's previous kernels
    const int n = real ? n_real : min(n_real, 32);
    const int n4 = (n + 127) / 128 * 32;       // 16-byte groups of keys, padded for the search
    const int seq = unit, layer = ch.layer0;   // kFused: one layer per call
    double* st = ch.state + size_t(seq) * (1 + 2 * ch.L);
    double b_rem = 0.0, rest = 0.0;
    int no_hist = 0;
    if (!control) {
      if constexpr (D > 0) {
        float pv[VN], sq = 0.f;
        const float* pg = sa.probe_kv + head * DD + (lane % LPR) * VN;
#pragma unroll
        for (int e = 0; e < VN; e += 4) {
          const float4 x = real ? __ldg(reinterpret_cast<const float4*>(pg + e)) : make_float4(1.f, 1.f, 1.f, 1.f);
          pv[e] = x.x; pv[e + 1] = x.y; pv[e + 2] = x.z; pv[e + 3] = x.w;
        }
        // the probe's norm: every group of LPR lanes holds the whole probe
#pragma unroll
        for (int e = 0; e < VN; ++e) sq = fmaf(pv[e], pv[e], sq);
#pragma unroll
        for (int o = LPR >> 1; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        const bool bad = !(sq > 0.f) || !isfinite(sq);
        if (bad && lane == 0 && 4 * warp < n) set_status(status, ACTQKV_DEV_BAD_PROBE);
        const float inv_pn = bad ? 0.f : rsqrtf(sq);
        if (!real) key_sync<kKeys>();            // the norms are written
        for (int i = 0; 4 * (warp + i * kWarps) < n; ++i) {
          const int b = 4 * (warp + i * kWarps);
          if (real && !wait_phase0(smem(group_bar + i), ch.polls)) {            // goes on with whatever arrived
            if (lane == 0) { sh_late = 1; set_status(status, ACTQKV_DEV_TIMEOUT); }
          }
          __syncwarp();
          const uint4* rows = reinterpret_cast<const uint4*>(groups + i * kGroupBytes) + lane;
          float accb[4];
#pragma unroll
          for (int bi = 0; bi < 4; ++bi) {
            accb[bi] = 0.f;
#pragma unroll
            for (int k = 0; k < 2; ++k) {                      // the block's two vectors
              const int u = 2 * bi + k, row = b * sa.r + u * RPP + lane / LPR;
              float x[VN];
              Vec16<T>::unpack(rows[u * 32], x);
              float dot = 0.f;
#pragma unroll
              for (int e = 0; e < VN; ++e) dot = fmaf(pv[e], x[e], dot);
              accb[bi] = fmaf(dot, row < n * sa.r ? norms[row] : 0.f, accb[bi]);
            }
          }
          // the four block sums are reduced together: halves swap block pairs, quarters swap blocks, then three steps
          // inside each quarter
          const bool up16 = lane & 16, up8 = lane & 8;
          const float t0 = __shfl_xor_sync(0xffffffffu, up16 ? accb[0] : accb[2], 16);
          const float t1 = __shfl_xor_sync(0xffffffffu, up16 ? accb[1] : accb[3], 16);
          const float k0 = (up16 ? accb[2] : accb[0]) + t0, k1 = (up16 ? accb[3] : accb[1]) + t1;
          float k = (up8 ? k1 : k0) + __shfl_xor_sync(0xffffffffu, up8 ? k0 : k1, 8);
          k += __shfl_xor_sync(0xffffffffu, k, 4);
          k += __shfl_xor_sync(0xffffffffu, k, 2);
          k += __shfl_xor_sync(0xffffffffu, k, 1);
          const int blk = b + 2 * (lane >> 4) + ((lane >> 3) & 1);
          if ((lane & 7) == 0 && blk < n) {
            const float score = k * inv_pn / float(sa.r);
            sc[blk] = score;
            if (real) sa.scores_out[head * n_cap + blk] = score;
          }
        }
        key_sync<kKeys>();                       // the scores are complete
      }
      // the scores are fetched once, by all threads at a time; density and selection read them from here
      float m[2] = {-INFINITY, -INFINITY};       // per column of key threads
      static_assert(kCols == 1 || (kCols == 2 && kKeys == 256), "every second fetch is of the other slot");
      for (int i0 = tid; i0 < 4 * n4; i0 += 4 * kKeys) {
        float x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + u * kKeys;
          x[u] = i < n ? (D > 0 ? sc[i] : real ? s[i] : float(i) * 0.03f) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + u * kKeys;
          if (u > 0 && i >= 4 * n4) break;
          if (kFused && i < n) {
            if (D == 0) sc[i] = x[u];
            m[u & (kCols - 1)] = fmaxf(m[u & (kCols - 1)], ch.beta * x[u]);
          }
          keys[i] = i < n ? score_key(x[u]) : 0u;
        }
      }
      if (kFused && warp * 32 < n) {           // Eq. 11 over a slot's scores, about the slot's own maximum; both slots of a warp at a time
        float top[kCols], z[kCols], e_x[kCols];
#pragma unroll
        for (int col = 0; col < kCols; ++col) { top[col] = warp_max_redux(m[col]); z[col] = e_x[col] = 0.f; }
#pragma unroll 2
        for (int i = tid; i < n; i += kKeys * kCols) {
#pragma unroll
          for (int col = 0; col < kCols; ++col) {
            if (col > 0 && i + col * kKeys >= n) break;
            const float x = fmaf(ch.beta, sc[i + col * kKeys], -top[col]), e = expf(x);
            z[col] += e;
            e_x[col] = fmaf(e, x, e_x[col]);
          }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
          for (int col = 0; col < kCols; ++col) {
            z[col] += __shfl_xor_sync(0xffffffffu, z[col], o);
            e_x[col] += __shfl_xor_sync(0xffffffffu, e_x[col], o);
          }
        if (lane == 0)
#pragma unroll
          for (int col = 0; col < kCols; ++col) {
            const int v = warp + col * kWarps;
            red_m[v] = top[col]; red_z[v] = z[col]; red_e[v] = e_x[col];
          }
      }
    } else if constexpr (kFused) {
      // The old state: the mean densities of the deeper layers that have a history (a lane per layer, then a
      // butterfly over the lanes).  Every CTA reads it before it hands out its density, CTA 0 writes it after all have.
      b_rem = real && layer > 0 ? st[0] : double(ch.L) * double(ch.k_blocks);
      for (int j = layer + 1 + lane; j < ch.L; j += 32) {
        const double cnt = real ? st[1 + ch.L + j] : 2.0;
        if (cnt > 0.0) rest += (real ? st[1 + j] : 1.0) / cnt; else ++no_hist;
      }
#pragma unroll 1
      for (int o = 16; o > 0; o >>= 1) rest += __shfl_xor_sync(0xffffffffu, rest, o);
      b_rem = __shfl_sync(0xffffffffu, b_rem, 0);       // has arrived
      no_hist = __reduce_add_sync(0xffffffffu, no_hist);
    }
    __syncthreads();
    if constexpr (kFused) if (!real) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    int rank = 0;
    if (!control) {
      if (ranked && warp * 32 < n) rank = rank_of(keys[tid], tid, keys, n);
    } else if constexpr (kFused) {
      const size_t uh = size_t(unit) * n_kv_heads + g;
      float th_own;
      if (ch.theta_in && real) {
        th_own = ch.theta_in[uh];
      } else {                                 // the slots' sums, moved to the common maximum
        const bool on = lane < kSlots && lane * 32 < n;
        const float m = on ? red_m[lane] : -INFINITY, top = warp_max_redux(m);
        const float x = on ? m - top : 0.f, f = on ? expf(x) : 0.f, zw = on ? red_z[lane] : 0.f;
        float z = f * zw, e_x = on ? f * fmaf(zw, x, red_e[lane]) : 0.f;
        z = warp_sum(z);
        e_x = warp_sum(e_x);
        th_own = n > 0 ? fmaxf(logf(z) - e_x / z, 0.f) : 0.f;
        if (lane == 0 && !ch.theta_in && ch.theta_out && real) ch.theta_out[uh] = th_own;
      }
      const uint32_t bar = smem(sh_bar + pass);
      if (lane < n_kv_heads && !(real && ch.drop == g)) {
        uint32_t dst, far;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(smem(&sh_thetas[pass][g])), "r"(lane));
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(far) : "r"(bar), "r"(lane));
        asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];"
                     ::"r"(dst), "r"(__float_as_uint(th_own)), "r"(far) : "memory");
      }
      if (!wait_phase0(bar, ch.polls) && lane == 0) { sh_late = 1; set_status(status, ACTQKV_DEV_TIMEOUT); }
      double sum = 0.0;
      for (int h = 0; h < n_kv_heads; ++h) sum += double(sh_thetas[pass][h]);
      const double th = sum / double(n_kv_heads);
      Grant gr{0, 0.0};
      // layers without history count with this layer's density; with every layer in the call
      // (L == 1) there is no deeper layer and both theta-bar readings coincide
      if (n > 0) gr = grant_layer(th, rest + double(no_hist) * th, b_rem, ch.L - layer, n, ch.cap_blocks);
      if (lane == 0) {
        sh_count = real ? gr.c : 5;
        if (g == 0 && real) {
          st[0] = n > 0 ? b_rem - double(gr.c) : b_rem;
          if (n > 0) {
            st[1 + layer] += th;
            st[1 + ch.L + layer] += 1.0;
          }
          sel_count[unit] = gr.c;
          if (ch.budget_real) ch.budget_real[unit] = float(gr.real);
        }
      }
    } else {
      if (lane == 0) {
        int c = real ? sel_count[unit] : 5;
        if (real && (c < 0 || c > min(cap_blocks, n))) {
          set_status(status, ACTQKV_DEV_BAD_SELECTION);
          c = max(0, min(c, min(cap_blocks, n)));
        }
        sh_count = c;
      }
    }
    __syncthreads();
    const int c = sh_count;
    if (control) {
      if (real)
        for (int i = max(c, 0) + lane; i < cap_blocks; i += 32) out[i] = -1;
    } else if (ranked) {
      const bool take = tid < n && rank < c;
      const uint32_t votes = __ballot_sync(0xffffffffu, take);
      if (lane == 0) warp_tot[0][warp] = __popc(votes);
      key_sync<kKeys>();
      const int pos = __reduce_add_sync(0xffffffffu, lane < warp ? warp_tot[0][lane] : 0) + __popc(votes & ((1u << lane) - 1u));
      if (take && pos < cap_blocks && real) out[pos] = tid;
    } else if (c >= n) {
      if (real)
        for (int i = tid; i < min(n, c); i += kKeys) out[i] = i;
    } else if (c > 0) {
      // ---- the largest threshold that at least c keys reach; done early when exactly c do
      int at = n;                                // keys >= thr
      const uint32_t thr = search_cth<kKeys>(c, keys, n4, warp_tot, at);
      // at > c: thr is the c-th largest key itself and at - c too many keys equal it; of those the first
      // by index are admitted
      int need_eq = n;
      if (at > c) {
        int above = 0;
        for (int i = tid; i < n; i += kKeys) above += keys[i] > thr;
        above = __reduce_add_sync(0xffffffffu, above);
        key_sync<kKeys>();
        if (lane == 0) warp_tot[0][warp] = above;
        key_sync<kKeys>();
        need_eq = c - __reduce_add_sync(0xffffffffu, lane < kWarps ? warp_tot[0][lane] : 0);
      }
      const int per = (n + kKeys - 1) / kKeys;
      const int i0 = min(n, tid * per), i1 = min(n, i0 + per);
      int eq_before = 0;
      if (at > c) {
        int eq = 0;
        for (int i = i0; i < i1; ++i) eq += keys[i] == thr;
        eq_before = key_exclusive_scan<kKeys>(eq, warp_tot[0]);
      }
      // compacted in ascending block order
      int cnt = 0, e = eq_before;
      for (int i = i0; i < i1; ++i) {
        const uint32_t x = keys[i];
        cnt += at > c ? (x > thr || (x == thr && e++ < need_eq)) : x >= thr;
      }
      int pos = key_exclusive_scan<kKeys>(cnt, warp_tot[0]);
      e = eq_before;
      for (int i = i0; i < i1; ++i) {
        const uint32_t x = keys[i];
        const bool take = at > c ? (x > thr || (x == thr && e++ < need_eq)) : x >= thr;
        if (take && pos < cap_blocks && real) out[pos++] = i;
      }
    }
    __syncthreads();                             // the next pass writes what this one reads
  }
  // A CTA whose wait ran out may not leave before what is still on its way to its shared memory has arrived: its own
  // copies, and the densities of peers that are late (they have sent theirs once they are at this barrier or have exited,
  // which counts as arriving).  Where all densities arrived no peer has anything left to send.
  if constexpr (kFused) {
    if (sh_late) {
      if constexpr (D > 0)
        for (int i = 0; !control && 4 * (warp + i * kWarps) < n_real; ++i) wait_phase0(smem(group_bar + i), ch.polls);
      asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
      wait_phase0(smem(sh_bar), ch.polls);
      wait_phase0(smem(sh_bar + 1), ch.polls);
    }
  }
}

// One layer whose scores the selection takes itself: small tables of 1 KiB blocks, which the CTA of a KV head
// brings into shared memory while bias + probe of the window runs.  It saves a launch and the hand-over of the scores, and
// costs a head's products on one SM instead of eight.  Steps of 2 to 512 tokens in tables of 104 rows, one kernel against two, us
// a layer at 4 / 40 / 96 candidates: one sequence of 8 KV heads -0.7 to -1.8 / -0.3 to -1.1 / -0.1 to -4.1, two -2.2 to +0.9 / -2.2 to
// +1.0 / -2.1 to +0.5 (the losses at 64 and 128 tokens), three -2.9 to +0.5 / -2.4 to +3.3 / -3.1 to +5.5, four +0.7 to +2.0 / +1.0 to +4.0 /
// -0.6 to +2.2; 2 KV heads (fp32) gain up to four sequences.  So it is taken up to 16 heads in all.  At 120 candidates of a table
// of 128 it is even (-2 to +2.9), but a prompt comes through all the smaller counts first.  The line goes by the rows of the table,
// which the host knows, and not by the candidates in it: a prompt in a state sized for more than 16k tokens takes two kernels.
// Behind anything shorter than bias + probe the copies are exposed (the append of the step before lets nothing start
// early): a decode step with attention and append takes 14.6 / 17.9 / 18.5 us as two kernels and 15.2 / 19.4 / 20.6 as one at
// 8 / 40 / 96 candidates, 27.5 and 29.3 with four sequences at 96, a drafted step of 5 tokens 21.0 and 23.9.
bool scores_in_selection(const actqkv_config* cfg, const Batch& b) {
  const size_t block_bytes = size_t(cfg->n_repr) * cfg->head_dim * elt_size(cfg);
  return b.n_layers == 1 && cfg->n_kv_heads <= 8 && cfg->cap_blocks > 0 && cfg->agg_mode != ACTQKV_AGG_MAX && block_bytes == 1024 &&
         cfg->n_cap > 0 && cfg->n_cap <= kScoreMaxCap && b.n_seq * cfg->n_kv_heads <= kScoreMaxHeads;
}

int launch_cutoff(const actqkv_config* cfg, const Batch& b, const float* scores, const float* theta_in,
                  float* theta_out, const int32_t* n_cand, void* budget_state, int32_t* sel_idx,
                  int32_t* sel_count, float* budget_real, int32_t* status, cudaStream_t st, const ScoreArgs* score_args = nullptr) {
  if (cfg->thetabar_mode == ACTQKV_THETABAR_ALG1 && (b.layer0 != 0 || b.n_layers != cfg->n_layers))
    return ACTQKV_ERR_UNSUPPORTED;
  if (keys_bytes(cfg->n_cap) > kMaxKeysSmem) return ACTQKV_ERR_SHAPE;
  ChainParams p;
  p.scores = scores; p.theta_in = theta_in; p.theta_out = theta_out; p.n_cand = n_cand;
  p.state = static_cast<double*>(budget_state);
  p.sel_count = sel_count; p.budget_real = budget_real;
  p.n_kv_heads = cfg->n_kv_heads; p.n_cap = cfg->n_cap; p.L = cfg->n_layers; p.Lb = b.n_layers;
  p.layer0 = b.layer0; p.k_blocks = cfg->k_blocks; p.cap_blocks = cfg->cap_blocks;
  p.thetabar_mode = cfg->thetabar_mode; p.beta = cfg->beta;
  p.polls = cfg->test_wait_limit > 0 ? uint32_t(cfg->test_wait_limit) : 1u << 20;
  p.drop = cfg->test_wait_limit > 0 ? cfg->test_drop_k_tile : -1;
  const bool fused = b.n_layers == 1 && cfg->n_kv_heads <= 8 && cfg->cap_blocks > 0;
  // 512 key threads where 256 would hold several candidates each and the CTAs have the SMs to themselves; a grid that fills
  // the SMs keeps the narrow form, which becomes resident beside two CTAs of the streaming scores (288 threads x 56
  // registers; 16 sequences of 32k-131k tokens, a decode step of two layers: 168 us).
  const bool wide = cfg->n_cap > 256 && b.units() * cfg->n_kv_heads <= kNumSMs / 2;
  using bf16 = __nv_bfloat16;
  // Two slots of the density per warp where 256 threads may have more than 256 scores: 0.2 to 0.5 us a launch (16 sequences at 313 / 500
  // / 900 candidates 16.0 -> 16.2, 19.7 -> 20.1, 28.5 -> 28.8 with the scores), which smaller tables do not pay.  (The 8 slots of the narrow
  // form in the wide one, too: 0.3 us on every single sequence above 256.)
  const bool two_slots = fused && !wide && cfg->n_cap > 256;
  auto kern = fused ? (wide        ? select_kernel<true, 512, 1, float, 0>
                       : two_slots ? select_kernel<true, 256, 2, float, 0> : select_kernel<true, 256, 1, float, 0>)
                    : (wide ? select_kernel<false, 512, 1, float, 0> : select_kernel<false, 256, 1, float, 0>);
  ScoreArgs sa = {};
  size_t sm_sel = keys_bytes(cfg->n_cap);
  if (score_args) {
    sa = *score_args;
    const bool half = cfg->dtype == ACTQKV_BF16;
    kern = cfg->head_dim == 128 ? (half ? select_kernel<true, kScoreKeys, 1, bf16, 128> : select_kernel<true, kScoreKeys, 1, float, 128>)
                                : (half ? select_kernel<true, kScoreKeys, 1, bf16, 64> : select_kernel<true, kScoreKeys, 1, float, 64>);
    sm_sel += norms_bytes(cfg->n_cap, sa.r) + size_t(kScoreKeys / 32) * (slots_of(cfg->n_cap) * kGroupBytes + kScoreSlots * 8);
  }
  static std::atomic<bool> carved[9][kMaxDevices], opted_in[9][kMaxDevices];
  const int form = score_args ? 4 + 2 * (cfg->head_dim == 128) + (cfg->dtype == ACTQKV_BF16) : two_slots ? 8 : 2 * wide + fused;
  // one opt-in at the largest size of the form: a size per call could be lowered by another thread ahead of the launch
  if (sm_sel > 40 * 1024 && !opt_in_shared_memory(kern, score_args ? kScoreSmem : kMaxKeysSmem, opted_in[form])) return ACTQKV_ERR_LAUNCH;
  if (!fused) {
    const size_t sm_chain = sizeof(float) * ((size_t(b.n_layers) * cfg->n_kv_heads + 1) & ~size_t(1)) +
                            sizeof(double) * (2 * size_t(b.n_layers) + 2 * (size_t(cfg->n_layers) + 1));
    if (sm_chain > 48 * 1024) return ACTQKV_ERR_SHAPE;
    if (!p.theta_in && theta_out && b.n_layers * cfg->n_kv_heads >= 64) {
      // many (layer, head) densities: take them with one warp each in a kernel of their own
      const int rc = launch_entropy(cfg, b, scores, n_cand, theta_out, st);
      if (rc) return rc;
      p.theta_in = theta_out;
    }
    static std::atomic<bool> carved_chain[kMaxDevices];
    prefer_max_shared(cutoff_chain_kernel, carved_chain);
    cudaLaunchConfig_t lcc = {};
    lcc.gridDim = dim3(b.n_seq, 1, 1);
    lcc.blockDim = dim3(kChainThreads, 1, 1);
    lcc.dynamicSmemBytes = sm_chain;
    lcc.stream = st;
    cudaLaunchAttribute cattr[1];
    allow_early_launch(cattr[0]);
    lcc.attrs = cattr;
    lcc.numAttrs = 1;
    if (cudaLaunchKernelEx(&lcc, cutoff_chain_kernel, p) != cudaSuccess) return ACTQKV_ERR_LAUNCH;
    if (cfg->cap_blocks == 0) return ACTQKV_OK;
  }
  prefer_max_shared(kern, carved[form]);
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(cfg->n_kv_heads, b.units(), 1);
  lc.blockDim = dim3((wide ? 512 : 256) + 32, 1, 1);
  lc.dynamicSmemBytes = sm_sel;
  lc.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = fused ? cfg->n_kv_heads : 1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  allow_early_launch(attr[1]);
  lc.attrs = attr;
  lc.numAttrs = 2;                  // every kernel of the chain waits for its predecessor before it reads
  if (cudaLaunchKernelEx(&lc, kern, scores, n_cand, sel_count, sel_idx, cfg->n_kv_heads, cfg->n_cap,
                         cfg->cap_blocks, b.n_layers, status, p, sa) != cudaSuccess)
    return ACTQKV_ERR_LAUNCH;
  return launch_status();
}

}  // namespace

extern "C" int actqkv_select_cutoff(const actqkv_config* cfg, const actqkv_batch* batch, const float* scores,
                                    const float* theta, const int32_t* n_cand, void* budget_state,
                                    int32_t* sel_idx, int32_t* sel_count, float* budget_real,
                                    int32_t* status, void* stream) {
  const Batch b = get_batch(batch);
  int rc = check_config(cfg, b);
  if (rc) return rc;
  ACTQKV_REQUIRE_PTR(scores);
  if (!theta || !n_cand || !budget_state || !sel_count) return ACTQKV_ERR_NULL;
  ACTQKV_REQUIRE_PTR(sel_idx);
  return launch_cutoff(cfg, b, scores, theta, nullptr, n_cand, budget_state, sel_idx, sel_count,
                       budget_real, status, reinterpret_cast<cudaStream_t>(stream));
}

int actqkv::score_select(const actqkv_config* cfg, const actqkv_batch* batch, const float* probe_kv, const void* repr_k,
                         const float* repr_inv_norm, const int32_t* n_cand, void* budget_state, float* scores, float* theta,
                         int32_t* sel_idx, int32_t* sel_count, float* budget_real, int32_t* status, bool behind_probe,
                         cudaStream_t st) {
  const Batch b = get_batch(batch);
  int rc = check_config(cfg, b);
  if (rc) return rc;
  ACTQKV_REQUIRE_PTR(probe_kv);
  ACTQKV_REQUIRE_PTR(repr_k);
  ACTQKV_REQUIRE_PTR(repr_inv_norm);
  ACTQKV_REQUIRE_PTR(scores);
  ACTQKV_REQUIRE_PTR(sel_idx);
  if (!n_cand || !budget_state || !sel_count) return ACTQKV_ERR_NULL;
  if (behind_probe && scores_in_selection(cfg, b)) {
    const ScoreArgs sa = {probe_kv, repr_k, repr_inv_norm, scores, cfg->n_repr};
    return launch_cutoff(cfg, b, scores, nullptr, theta, n_cand, budget_state, sel_idx, sel_count, budget_real, status, st, &sa);
  }
  rc = launch_scores(cfg, b, probe_kv, repr_k, repr_inv_norm, n_cand, scores, status, st);
  if (rc) return rc;
  return launch_cutoff(cfg, b, scores, nullptr, theta, n_cand, budget_state, sel_idx, sel_count, budget_real, status, st);
}

extern "C" int actqkv_score_select(const actqkv_config* cfg, const actqkv_batch* batch, const float* probe_kv,
                                   const void* repr_k, const float* repr_inv_norm, const int32_t* n_cand,
                                   void* budget_state, float* scores, float* theta, int32_t* sel_idx,
                                   int32_t* sel_count, float* budget_real, int32_t* status, void* stream) {
  return score_select(cfg, batch, probe_kv, repr_k, repr_inv_norm, n_cand, budget_state, scores, theta, sel_idx, sel_count,
                      budget_real, status, false, reinterpret_cast<cudaStream_t>(stream));
}
