// Step 5, general kernel: attention of the step's queries over
//   [initial tokens | selected blocks | local past | step tokens (causal)]     (Eq. 2, Eq. 3)
// gathered from the paged cache.  fp32 products and sums on CUDA cores, any supported dtype / head
// dim / page size / alignment; serves fp32 caches and what the tensor-core kernels do not take.
//
// One CTA = 32 rows of one KV head: the (token, query head) pairs of the group, row = token * G + head,
// so that K and V are read once per group.  Keys go through shared memory in chunks, as they come, two buffers: a producer
// warp looks the keys up (position -> page table, behind the selection's entries), brings chunk c + 1 and waits for it while
// the four compute warps work on chunk c; one CTA barrier per chunk.
// A compute warp has 8 rows; its lanes have one or two keys each in Q K^T (one: fp32 at D = 128) and D / 32 channels each in P V.
// Bound by what two compute warps a scheduler can hide of shared memory and arithmetic (four sequences of 256 tokens, 32
// heads: issue slots busy 58 to 71 %, FMA pipe 43 to 55 %, shared memory 54 and 60 % in fp32, 46 and 45 % in bf16).  Q and P
// are read by broadcast, one 128-byte wavefront per 16-byte load, K and V by 32 lanes apart.  Wavefronts per 64 FMAs of a warp,
// Q K^T and P V: fp32 16 and 16 at D = 64, 24 and 12 at D = 128; bf16, which is unpacked at its use (8 rows share that), 12
// and 12, 12 and 8.  (4 rows x 4 keys per thread, 16 lanes to a row: 32.)
//
// The initial tokens, the local past and the step's own tokens come first and the selected blocks last: the former are
// known before this step's selection exists, so their chunks run ahead of the dependency wait (programmatic dependent
// launch).  Few tiles: the chunks are cut over the CTAs of a cluster (chunk c goes to rank c % n) and the partial
// results are merged through distributed shared memory.
// Launches one behind the other, us, 4 x 4 tiles with all 128 threads staging fp32 between two barriers and every key behind the
// wait -> this (one producer warp that unpacks bf16 into fp32, as it was at first, in brackets):
//                                            fp32 D = 64     fp32 D = 128    bf16 D = 64              bf16 D = 128
//   1 token, 32 / 8 heads, 4,096 behind        17 ->  13        27 ->  19       17 ->   13  (15)         27 ->   18  (22)
//   256 tokens, 4 / 2 heads, 1,472 behind      29 ->  22        39 ->  35       29 ->   21  (24)         37 ->   31  (38)
//   256 tokens, 32 / 8 heads, 1,472 behind    161 ->  99       224 -> 200      166 ->   97 (111)        217 ->  160 (227)
//   16 sequences of that                    1,492 -> 1,405   2,983 -> 2,837  1,487 -> 1,371 (1,586)   2,839 -> 2,267 (3,197)
//   64 sequences of 1 token, 1,472 behind     286 -> 180       442 -> 359      290 ->  176 (221)        397 ->  290 (410)
// An SM holds two of these CTAs where it held four at D = 64: grids that leave some SMs one and some two (80 to 100, 180 to 200 and
// 320 CTAs) are 1 to 8 % slower in fp32 at D = 64 (45 -> 48, 88 -> 93, 174 -> 182), the ones beside them up to 1.8 times as fast.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "stages.cuh"

using namespace actqkv;

namespace {

constexpr int kRows = 32;
constexpr int kComputeWarps = 4, kRowsPerWarp = kRows / kComputeWarps;
constexpr int kThreads = 32 * (kComputeWarps + 1);
constexpr int kMaxSplits = 8;

// Bytes.  K and V lie there as they come (bf16 is unpacked at its use), Q and P as fp32.
template <typename T, int D> struct Smem {
  static constexpr int kChunk = D * sizeof(T) > 256 ? 32 : 64;          // keys; two CTAs per SM
  static constexpr int kKStride = D + Vec16<T>::N;   // elements; 8 consecutive keys at one 16-byte vector hit distinct banks
  static constexpr int kPStride = kChunk + 4;        // floats
  static constexpr int kKV = kChunk * (kKStride + D) * int(sizeof(T));  // one buffer: K, then V
  static constexpr int kQ = 0, kBuf = kQ + kRows * D * 4, kP = kBuf + 2 * kKV, kBytes = kP + kRows * kPStride * 4;
};

struct SimtParams {
  AttnArgs a;
  int n_q_heads, n_kv_heads, group, block, page_tokens, n_init, n_local_prev, cap_blocks;
  int max_pages, n_phys_pages, n_layers, n_splits;
  float scale_log2;
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// 16 bytes / 4 bytes of CTA `rank`'s shared memory at the address that `local` has in this CTA
__device__ __forceinline__ float4 ld_peer4(const float* local, uint32_t rank) {
  uint32_t a;
  float4 v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(uint32_t(__cvta_generic_to_shared(local))), "r"(rank));
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float ld_peer(const float* local, uint32_t rank) {
  uint32_t a;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(uint32_t(__cvta_generic_to_shared(local))), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(uint32_t(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
}

template <typename T, typename TO, int D>
__global__ void __launch_bounds__(kThreads, 2) attention_simt_kernel(SimtParams p) {
  using S = Smem<T, D>;
  constexpr int kChunk = S::kChunk, KPL = kChunk / 32, CPL = D / 32;   // keys and channels per lane
  constexpr int VN = Vec16<T>::N, VPR = D / VN, R = kRowsPerWarp;
  extern __shared__ __align__(16) unsigned char sm[];
  float *Qs = reinterpret_cast<float*>(sm + S::kQ), *Ps = reinterpret_cast<float*>(sm + S::kP);
  __shared__ float part_m[kRows], part_l[kRows];

  grid_launch_dependents();          // the append makes its loads while this kernel runs
  const uint32_t rank = p.n_splits > 1 ? cluster_rank() : 0u;
  const int tile = blockIdx.x / p.n_splits, g = blockIdx.y, unit = blockIdx.z;
  const int G = p.group, seq = unit / p.n_layers, layer_local = unit - seq * p.n_layers;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nt = p.a.n_tokens, n_rows = nt * G;

  const Geometry geo = make_geometry(p.a.pos0[seq], p.n_init, p.block, p.n_local_prev);
  const T* qb = static_cast<const T*>(p.a.q) + size_t(unit) * nt * p.n_q_heads * D;
  for (int i = tid; i < kRows * VPR; i += kThreads) {
    const int r = i / VPR, cv = i - r * VPR, gr = tile * kRows + r;
    float qf[VN];
    if (gr < n_rows) {
      Vec16<T>::load_nc(qb + (size_t(gr / G) * p.n_q_heads + g * G + gr % G) * D + cv * VN, qf);
    } else {
#pragma unroll
      for (int e = 0; e < VN; ++e) qf[e] = 0.f;
    }
#pragma unroll
    for (int e = 0; e < VN; ++e) Qs[r * D + cv * VN + e] = qf[e];
  }

  // ---- the key stream: [initial | local past | step's tokens], filled up to whole chunks, then the selected blocks
  const int64_t n_past = int64_t(geo.init_len) + (geo.p0 - geo.local_start);
  const int last_row = min(n_rows, (tile + 1) * kRows) - 1;
  const int64_t n_early = n_past + last_row / G + 1;
  const int64_t early = (n_early + kChunk - 1) / kChunk;               // chunks ahead of the wait
  int64_t total = early;                                               // all chunks, known after it
  int sel_len = 0;
  bool open = false;
  // Every warp that comes to the selected blocks takes the wait itself (it is the launch dependency, so it always ends).
  auto wait_selection = [&]() {
    grid_dependency_wait();
    int c = p.a.sel_count ? p.a.sel_count[unit] : 0;
    if (c < 0 || c > p.cap_blocks || c > geo.n_cand) {
      if (tid == 0) set_status(p.a.status, ACTQKV_DEV_BAD_SELECTION);
      c = max(0, min(c, min(p.cap_blocks, geo.n_cand)));
    }
    sel_len = c * p.block;
    total = early + (sel_len + kChunk - 1) / kChunk;
    open = true;
  };
  __syncthreads();                                     // Q is written

  float m[R], l[R], o[R][CPL];                         // l: this lane's share of the row's sum
#pragma unroll
  for (int r = 0; r < R; ++r) {
    m[r] = -INFINITY; l[r] = 0.f;
#pragma unroll
    for (int q = 0; q < CPL; ++q) o[r][q] = 0.f;
  }

  if (warp == kComputeWarps) {
    // =========================== producer ===========================
    const int32_t* sel = p.a.sel_idx + (size_t(unit) * p.n_kv_heads + g) * p.cap_blocks;
    const size_t page_elems = size_t(p.n_kv_heads) * p.page_tokens * D;
    const T* kp = static_cast<const T*>(p.a.k_pages) + size_t(layer_local) * p.n_phys_pages * page_elems;
    const T* vp = static_cast<const T*>(p.a.v_pages) + size_t(layer_local) * p.n_phys_pages * page_elems;
    const int32_t* pt = p.a.page_table + size_t(seq) * p.max_pages;
    const T* kw = static_cast<const T*>(p.a.k_win) + size_t(unit) * nt * p.n_kv_heads * D;
    const T* vw = static_cast<const T*>(p.a.v_win) + size_t(unit) * nt * p.n_kv_heads * D;
    // the place of key i: its element offset in the cache pool or (n_past <= i < n_early) in the step's own keys; -1: none
    auto find = [&](int64_t i) -> int64_t {
      int64_t tok;
      if (i >= early * kChunk) {
        const int64_t r = i - early * kChunk;
        if (r >= sel_len) return -1;
        const int blk = sel[int(r) / p.block];
        if (blk < 0 || blk >= geo.n_cand) {
          set_status(p.a.status, ACTQKV_DEV_BAD_SELECTION);
          return -1;
        }
        tok = int64_t(p.n_init) + int64_t(blk) * p.block + int(r) % p.block;
      } else {
        if (i >= n_early) return -1;
        if (i >= n_past) return ((i - n_past) * p.n_kv_heads + g) * D;
        tok = i < geo.init_len ? i : geo.local_start + (i - geo.init_len);
      }
      const int64_t lp = tok / p.page_tokens;
      const int phys = lp < p.max_pages ? pt[lp] : -1;
      if (phys < 0 || phys >= p.n_phys_pages) {
        set_status(p.a.status, ACTQKV_DEV_BAD_PAGE);
        return -1;
      }
      return (int64_t(phys) * p.n_kv_heads + g) * p.page_tokens * D + (tok - lp * p.page_tokens) * D;
    };
    struct Places { int64_t at[KPL]; };
    auto look_up = [&](int64_t c) {
      Places x;
#pragma unroll
      for (int j = 0; j < KPL; ++j) x.at[j] = find(c * kChunk + 32 * j + lane);
      return x;
    };
    // Two lanes per key, 16 keys at a time: whole 32-byte sectors, and no address arithmetic between a row's copies.
    auto bring = [&](int64_t c, const Places& x, T* Ks) {
      T* Vs = Ks + kChunk * S::kKStride;
      const int half = lane & 1;
#pragma unroll
      for (int j = 0; j < 2 * KPL; ++j) {
        const int in = 16 * (j & 1) + (lane >> 1), row = 32 * (j >> 1) + in;
        const int64_t at = __shfl_sync(0xffffffffu, x.at[j >> 1], in);
        const bool past = c >= early || c * kChunk + row < n_past;
        const T *ks = (past ? kp : kw) + at + half * VN, *vs = (past ? vp : vw) + at + half * VN;
        T *kd = Ks + row * S::kKStride + half * VN, *vd = Vs + row * D + half * VN;
        if (at < 0) {
#pragma unroll 1
          for (int e = 0; e < D; e += 2 * VN)
            *reinterpret_cast<uint4*>(kd + e) = *reinterpret_cast<uint4*>(vd + e) = make_uint4(0, 0, 0, 0);
        } else {
#pragma unroll
          for (int e = 0; e < D; e += 2 * VN) {
            cp_async16(kd + e, ks + e);
            cp_async16(vd + e, vs + e);
          }
        }
      }
    };
    int64_t c = rank;
    if (c >= early) wait_selection();
    Places x = look_up(c);
    for (int buf = 0; c < total; buf ^= 1) {
      bring(c, x, reinterpret_cast<T*>(sm + S::kBuf + buf * S::kKV));
      c += p.n_splits;
      const bool known = c < early || open;
      if (known && c < total) x = look_up(c);          // while the copies fly
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncthreads();                                 // the chunk is there, and the other buffer has been read
      if (!known) {
        wait_selection();
        if (c < total) x = look_up(c);
      }
    }
  } else {
    // =========================== compute ===========================
    int lim[R];                                        // the warp's rows see the step's tokens [0, lim)
#pragma unroll
    for (int r = 0; r < R; ++r) lim[r] = min((tile * kRows + warp * R + r) / G, last_row / G) + 1;
    const float* q_rows = Qs + warp * R * D;
    float* p_rows = Ps + warp * R * S::kPStride;
    int64_t c = rank;
    for (int buf = 0;; buf ^= 1, c += p.n_splits) {
      if (c >= early && !open) wait_selection();
      if (c >= total) break;
      __syncthreads();                                 // the chunk is there
      const T *Ks = reinterpret_cast<const T*>(sm + S::kBuf + buf * S::kKV), *Vs = Ks + kChunk * S::kKStride;
      // ---- S = Q K^T: keys lane + 32 j
      float s[R][KPL];
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int j = 0; j < KPL; ++j) s[r][j] = 0.f;
#pragma unroll 2
      for (int d = 0; d < D; d += VN) {
        float kv[KPL][VN];
#pragma unroll
        for (int j = 0; j < KPL; ++j) Vec16<T>::load(Ks + (lane + 32 * j) * S::kKStride + d, kv[j]);
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int e = 0; e < VN; e += 4) {
            const float4 qv = *reinterpret_cast<const float4*>(q_rows + r * D + d + e);
#pragma unroll
            for (int j = 0; j < KPL; ++j) {
              s[r][j] = fmaf(qv.x, kv[j][e], s[r][j]);
              s[r][j] = fmaf(qv.y, kv[j][e + 1], s[r][j]);
              s[r][j] = fmaf(qv.z, kv[j][e + 2], s[r][j]);
              s[r][j] = fmaf(qv.w, kv[j][e + 3], s[r][j]);
            }
          }
      }
      // ---- running softmax of the warp's rows
      // row r sees the chunk's keys [0, lim_r): all of the past, its own part of the step's tokens, the selected blocks
      const bool window = c < early;
      const int64_t rest = window ? n_past - c * kChunk : sel_len - (c - early) * kChunk;
      const int past_lim = int(min(rest, int64_t(kChunk)));            // negative: behind the past
#pragma unroll
      for (int r = 0; r < R; ++r) {
        float mx = -INFINITY;
        const int lim_r = window ? past_lim + (past_lim < kChunk ? lim[r] : 0) : past_lim;
#pragma unroll
        for (int j = 0; j < KPL; ++j) {
          s[r][j] = lane + 32 * j < lim_r ? s[r][j] * p.scale_log2 : -INFINITY;
          mx = fmaxf(mx, s[r][j]);
        }
        const float m_new = fmaxf(m[r], warp_max_redux(mx));
        const float corr = m_new == -INFINITY ? 1.f : exp2f(m[r] - m_new);
        float sum = 0.f;
#pragma unroll
        for (int j = 0; j < KPL; ++j) {
          const float e = m_new == -INFINITY ? 0.f : exp2f(s[r][j] - m_new);
          p_rows[r * S::kPStride + lane + 32 * j] = e;
          sum += e;
        }
        l[r] = l[r] * corr + sum;
        m[r] = m_new;
#pragma unroll
        for (int q = 0; q < CPL; ++q) o[r][q] *= corr;
      }
      __syncwarp();                                    // a row's weights are written and read by one warp
      // ---- O += P V: channels CPL * lane ..
#pragma unroll 2
      for (int k = 0; k < kChunk; k += 4) {
        float4 pv[R];
#pragma unroll
        for (int r = 0; r < R; ++r) pv[r] = *reinterpret_cast<const float4*>(p_rows + r * S::kPStride + k);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          float v[CPL];
          if constexpr (sizeof(T) == 2) {              // bf16 is the upper half of an fp32
            uint32_t raw[CPL / 2];
            if constexpr (CPL == 2) {
              raw[0] = *reinterpret_cast<const uint32_t*>(Vs + (k + kk) * D + 2 * lane);
            } else {
              const uint2 t = *reinterpret_cast<const uint2*>(Vs + (k + kk) * D + 4 * lane);
              raw[0] = t.x; raw[1] = t.y;
            }
#pragma unroll
            for (int q = 0; q < CPL / 2; ++q) {
              v[2 * q] = __uint_as_float(raw[q] << 16);
              v[2 * q + 1] = __uint_as_float(raw[q] & 0xFFFF0000u);
            }
          } else if constexpr (CPL == 2) {
            const float2 t = *reinterpret_cast<const float2*>(Vs + (k + kk) * D + 2 * lane);
            v[0] = t.x; v[1] = t.y;
          } else {
            const float4 t = *reinterpret_cast<const float4*>(Vs + (k + kk) * D + 4 * lane);
            v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
          }
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const float w = kk == 0 ? pv[r].x : kk == 1 ? pv[r].y : kk == 2 ? pv[r].z : pv[r].w;
#pragma unroll
            for (int q = 0; q < CPL; ++q) o[r][q] = fmaf(w, v[q], o[r][q]);
          }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) l[r] = warp_sum(l[r]);
  }

  TO* ob = static_cast<TO*>(p.a.out) + size_t(unit) * nt * p.n_q_heads * D;
  auto store = [&](int row, int col, const auto& v) {  // sizeof(v) / 4 channels
    constexpr int N = sizeof(v) / 4;
    const int gr = tile * kRows + row;
    TO* dst = ob + (size_t(gr / G) * p.n_q_heads + g * G + gr % G) * D + col;
    __align__(16) TO t[N];
#pragma unroll
    for (int e = 0; e < N; ++e) t[e] = from_f32<TO>(v[e]);
    using Raw = typename std::conditional<sizeof(t) == 16, uint4, typename std::conditional<sizeof(t) == 8, uint2, uint32_t>::type>::type;
    *reinterpret_cast<Raw*>(dst) = *reinterpret_cast<const Raw*>(t);
  };
  auto store_lse = [&](int row, float mm, float ll) {
    const int gr = tile * kRows + row;
    if (p.a.lse) p.a.lse[(size_t(unit) * p.n_q_heads + g * G + gr % G) * nt + gr / G] = (mm + log2f(ll)) * 0.6931471805599453f;
  };
  if (p.n_splits == 1) {
    if (warp == kComputeWarps) return;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int row = warp * R + r;
      if (tile * kRows + row >= n_rows) continue;
      const float inv = l[r] > 0.f ? 1.f / l[r] : 0.f;
      float v[CPL];
#pragma unroll
      for (int q = 0; q < CPL; ++q) v[q] = o[r][q] * inv;
      store(row, CPL * lane, v);
      if (lane == 0) store_lse(row, m[r], l[r]);
    }
    return;
  }
  // ---- the ranks' partial results: O where Q was (its rows were this warp's alone), maxima and sums beside it; rank k
  // finishes rows [32 k / n, 32 (k + 1) / n), adding the ranks in order
  if (warp < kComputeWarps) {
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float* dst = Qs + (warp * R + r) * D + CPL * lane;
#pragma unroll
      for (int q = 0; q < CPL; ++q) dst[q] = o[r][q];
      if (lane == 0) { part_m[warp * R + r] = m[r]; part_l[warp * R + r] = l[r]; }
    }
  }
  __syncwarp();
  cluster_sync_all();
  const int own = kRows / p.n_splits;
  for (int i = tid; i < own * (D / 4); i += kThreads) {
    const int row = int(rank) * own + i / (D / 4), col = 4 * (i % (D / 4));
    if (tile * kRows + row >= n_rows) continue;
    float pm[kMaxSplits], pl[kMaxSplits], mm = -INFINITY;
    float4 po[kMaxSplits];
#pragma unroll
    for (int k = 0; k < kMaxSplits; ++k)
      if (k < p.n_splits) {
        pm[k] = ld_peer(part_m + row, k);
        pl[k] = ld_peer(part_l + row, k);
        po[k] = ld_peer4(Qs + row * D + col, k);
      }
#pragma unroll
    for (int k = 0; k < kMaxSplits; ++k)
      if (k < p.n_splits) mm = fmaxf(mm, pm[k]);
    float ll = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < kMaxSplits; ++k)
      if (k < p.n_splits) {
        const float w = pm[k] == -INFINITY ? 0.f : exp2f(pm[k] - mm);
        ll = fmaf(w, pl[k], ll);
        acc.x = fmaf(w, po[k].x, acc.x); acc.y = fmaf(w, po[k].y, acc.y);
        acc.z = fmaf(w, po[k].z, acc.z); acc.w = fmaf(w, po[k].w, acc.w);
      }
    const float inv = ll > 0.f ? 1.f / ll : 0.f;
    const float v[4] = {acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv};
    store(row, col, v);
    if (col == 0) store_lse(row, mm, ll);
  }
  __syncwarp();
  cluster_sync_all();                                  // a peer may still read this CTA's part
}

template <typename T, typename TO, int D>
int launch(const SimtParams& p, dim3 grid, cudaStream_t st) {
  static std::atomic<bool> opted_in[kMaxDevices];
  auto kern = attention_simt_kernel<T, TO, D>;
  constexpr int kBytes = Smem<T, D>::kBytes;
  if (!opt_in_shared_memory(kern, kBytes, opted_in)) return ACTQKV_ERR_LAUNCH;
  static std::atomic<bool> carved[kMaxDevices];
  prefer_max_shared(kern, carved);
  cudaLaunchConfig_t lc = {};
  lc.gridDim = grid;
  lc.blockDim = dim3(kThreads, 1, 1);
  lc.dynamicSmemBytes = kBytes;
  lc.stream = st;
  cudaLaunchAttribute attr[2];
  allow_early_launch(attr[0]);
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = p.n_splits;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  lc.attrs = attr;
  lc.numAttrs = 2;
  if (cudaLaunchKernelEx(&lc, kern, p) != cudaSuccess) return ACTQKV_ERR_LAUNCH;
  return launch_status();
}

}  // namespace

namespace actqkv {

int launch_attention_simt(const actqkv_config* cfg, const Batch& b, const AttnArgs& a, cudaStream_t st) {
  SimtParams p;
  p.a = a;
  p.n_q_heads = cfg->n_q_heads; p.n_kv_heads = cfg->n_kv_heads; p.group = cfg->n_q_heads / cfg->n_kv_heads;
  p.block = cfg->block; p.page_tokens = cfg->page_tokens; p.n_init = cfg->n_init;
  p.n_local_prev = cfg->n_local_prev; p.cap_blocks = cfg->cap_blocks; p.max_pages = cfg->max_pages;
  p.n_phys_pages = cfg->n_phys_pages; p.n_layers = b.n_layers;
  const float scale = cfg->sm_scale > 0.f ? cfg->sm_scale : 1.f / sqrtf(float(cfg->head_dim));
  p.scale_log2 = scale * 1.4426950408889634f;
  const int tiles = (a.n_tokens * p.group + kRows - 1) / kRows;
  // ranks per key stream: doubled as long as all CTAs are resident at once (two per SM)
  const int64_t slots = int64_t(kNumSMs) * 2;
  p.n_splits = 1;
  while (p.n_splits < kMaxSplits && int64_t(tiles) * cfg->n_kv_heads * b.units() * p.n_splits * 2 <= slots) p.n_splits *= 2;
  const dim3 grid(tiles * p.n_splits, cfg->n_kv_heads, b.units());
  const bool bf = cfg->dtype == ACTQKV_BF16, obf = cfg->out_dtype == ACTQKV_BF16;
#define ACTQKV_SIMT_D(T, TO) (cfg->head_dim == 128 ? launch<T, TO, 128>(p, grid, st) : launch<T, TO, 64>(p, grid, st))
  if (bf && obf) return ACTQKV_SIMT_D(__nv_bfloat16, __nv_bfloat16);
  if (bf) return ACTQKV_SIMT_D(__nv_bfloat16, float);
  if (obf) return ACTQKV_SIMT_D(float, __nv_bfloat16);
  return ACTQKV_SIMT_D(float, float);
#undef ACTQKV_SIMT_D
}

}  // namespace actqkv
