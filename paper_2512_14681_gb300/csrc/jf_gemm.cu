// Weight-streaming projections of the forward pass (Eq. 3: one pass over all in-flight rows):
// Y[m, n] = sum_k X[m, k] W[n, k] for the QKV, O, gate/up, down and LM-head matrices.
//
// bf16 path: tcgen05 tensor cores, "swap-AB" so that 128 weight rows form the MMA's M side and
// the (few) in-flight tokens its N side. A persistent, warp-specialised kernel: one CTA per SM
// walks its share of (tile, split) work units; a producer warp streams weight and activation
// tiles by TMA (128-byte swizzle) through a 4-12 stage mbarrier ring that never drains between
// units; an MMA warp accumulates into one of two TMEM accumulators; eight epilogue warps drain
// the other accumulator (fused epilogue, split-K reduction) while the next unit streams in.
// fp32 path (small fp32 models): a SIMT mainloop over 128-feature tiles with the same epilogues.
//
// Split-K is deterministic: partial tiles go to a workspace and the last CTA of a tile (atomic
// ticket, no waiting) adds them in split order. Every output element's reduction order is fixed
// by the weight shape alone, so a row's result does not depend on how many rows are in flight.
#include "jf_device.cuh"
#include "jf_internal.h"
#include "jf_once.h"

namespace jf {
namespace {

constexpr int A_STAGE_BYTES = kTileN * kTileK * 2;  // 16 KB of weights per stage

constexpr int EPI_STAGE_BYTES = 9216;               // epilogue exchange buffers (argmax)
constexpr int SMEM_LIMIT = 232448;                  // 227 KB per CTA

// PAIR: two CTAs (a cluster) share a tile of 256 weight rows; each stages its 128 rows of A and half of
// the tile's tokens.
template <int BN, bool PAIR>
struct TcCfg {
  static constexpr int B_ROWS = PAIR ? BN / 2 : BN;
  static constexpr int B_STAGE_BYTES = B_ROWS * kTileK * 2;
  static constexpr int STAGE_BYTES = A_STAGE_BYTES + B_STAGE_BYTES;
  static constexpr int S0 = (SMEM_LIMIT - 1024 - EPI_STAGE_BYTES - 512) / STAGE_BYTES;
  static constexpr int STAGES = S0 > 12 ? 12 : S0 / 2 * 2;  // two 64-k blocks a stage pair
  static_assert(STAGES >= 4, "at least two stage pairs");
  static constexpr int ACC_COLS = BN;   // one accumulator; two are allocated (double buffer)
  static constexpr int TMEM_COLS = 2 * BN <= 32 ? 32 : (2 * BN <= 64 ? 64 : (2 * BN <= 128 ? 128 : (2 * BN <= 256 ? 256 : 512)));
  static constexpr int SMEM = 1024 + STAGES * STAGE_BYTES + EPI_STAGE_BYTES + 512;
  static_assert(SMEM <= SMEM_LIMIT, "shared memory budget");
};

// The epilogue's threads: NH groups of 128, group `half` takes the 16-column chunks half, half + NH, ...
// sync(): the group's barrier; sync_all(): that of all groups (barrier 0 is __syncthreads).
template <int NH>
struct EpiThreads {
  int half, row;  // row: this thread's weight row of the tile
  JF_DEV void sync() const { asm volatile("bar.sync %0, 128;" ::"r"(1 + half) : "memory"); }
  JF_DEV void sync_all() const {
    if constexpr (NH == 1) sync();
    else asm volatile("bar.sync 3, %0;" ::"n"(128 * NH) : "memory");
  }
  JF_DEV bool first() const { return half == 0 && row == 0; }
};

constexpr int kMaxSplits = 8;  // split-K never exceeds this (enforced by the host)

JF_DEV uint8_t* align1024(uint8_t* p) {
  return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~uintptr_t(1023));
}

// ---------------------------------------------------------------------------------------------
// Greedy argmax. Logits are compared through keys that preserve their order as unsigned integers (-0
// counts as +0, NaN as the lowest, key 0). A row without a number gets the index kAmNoIndex, which no
// vocabulary holds: the callers see it, and the next forward's embedding reports it. Every CTA keeps a
// running entry (best key, its lowest index,
// runner-up key) of every row over the vocabulary tiles it takes: in shared memory for up to
// kAmTableRows rows, otherwise in its global slot; k_argmax_finish merges the CTAs' slots. The merge is
// associative and commutative, so the result does not depend on which CTA took which tile. With
// 15 shuffles a column and the entries in global memory the epilogue, not the weights, set the pace of
// the LM head above 32 rows, and one CTA merged all slots at the end (8 layers and head of the 7B shape,
// 32 rows 941 -> 929 us, 160 rows 1286 -> 1189, 512 rows 2427 -> 2072; 1.5B, 64 rows 499 -> 449).
// ---------------------------------------------------------------------------------------------
JF_DEV uint32_t am_key(float v) {
  const uint32_t u = __float_as_uint(v + 0.0f);
  return v != v ? 0u : ((u & 0x80000000u) ? ~u : (u | 0x80000000u));
}
// (no number under a key of 0: -infinity)
JF_DEV float am_value(uint32_t key) {
  return key == 0u ? -INFINITY : __uint_as_float((key & 0x80000000u) ? key ^ 0x80000000u : ~key);
}
JF_DEV void am_merge(uint32_t& b1, uint32_t& bi, uint32_t& b2, uint32_t o1, uint32_t oi, uint32_t o2) {
  if (o1 > b1 || (o1 == b1 && oi < bi)) {
    b2 = b1 > o2 ? b1 : o2;
    b1 = o1;
    bi = oi;
  } else {
    b2 = b2 > o1 ? b2 : o1;
  }
}

constexpr int kAmRedWords = 2 * 2 * 4 * 16 * 3;  // [group][parity of its chunk][warp][column][3]
constexpr int kAmTableRows = 512;
static_assert((kAmRedWords + 3 * kAmTableRows) * 4 <= EPI_STAGE_BYTES, "argmax tables fit the epilogue's staging");
constexpr uint32_t kAmNoIndex = 0x7fffffffu;

// Running entries of a CTA: entry of row m at [m * stride].
struct AmEntries {
  uint32_t *red, *k1, *idx, *k2;
  size_t stride;
};
JF_DEV AmEntries am_global(const GemmEpi& e, uint32_t* red, int slot, int n_slots) {
  return AmEntries{red, reinterpret_cast<uint32_t*>(e.am_v1) + slot, reinterpret_cast<uint32_t*>(e.am_i1) + slot,
                   reinterpret_cast<uint32_t*>(e.am_v2) + slot, (size_t)n_slots};
}
JF_DEV AmEntries am_shared(uint32_t* words) {
  uint32_t* t = words + kAmRedWords;
  return AmEntries{words, t, t + kAmTableRows, t + 2 * kAmTableRows, 1};
}
JF_DEV void am_clear(const AmEntries& am, int m_begin, int m_end, int tid, int nthreads) {
  for (int m = m_begin + tid; m < m_end; m += nthreads) {
    am.k1[m * am.stride] = 0u;
    am.idx[m * am.stride] = kAmNoIndex;
    am.k2[m * am.stride] = 0u;
  }
}

// One warp per row: the slots of all CTAs, eight a lane in flight.
__global__ void __launch_bounds__(128) k_argmax_finish(const uint32_t* k1, const uint32_t* idx, const uint32_t* k2,
                                                       int n_slots, int M, int* out, float* top2) {
  JF_TL_ENTRY();
  pdl_launch_dependents();
  const int m = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  pdl_wait();
  JF_TL_WAITED();
  if (m < M) {
    uint32_t b1 = 0, bi = kAmNoIndex, b2 = 0;
    for (int s0 = 0; s0 < n_slots; s0 += 8 * 32) {
      uint32_t a[8], i[8], c[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int s = s0 + 32 * k + lane;
        const size_t at = (size_t)m * n_slots + s;
        a[k] = s < n_slots ? __ldcg(k1 + at) : 0u;
        i[k] = s < n_slots ? __ldcg(idx + at) : kAmNoIndex;
        c[k] = s < n_slots ? __ldcg(k2 + at) : 0u;
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) am_merge(b1, bi, b2, a[k], i[k], c[k]);
    }
    const uint32_t top = __reduce_max_sync(0xffffffffu, b1);
    const uint32_t best = __reduce_min_sync(0xffffffffu, b1 == top ? bi : 0xffffffffu);
    const uint32_t second = __reduce_max_sync(0xffffffffu, (b1 == top && bi == best) ? b2 : b1);
    if (lane == 0) {
      out[m] = (int)(top == 0u ? kAmNoIndex : best);
      if (top2) {
        top2[2 * m] = am_value(top);
        top2[2 * m + 1] = am_value(second);
      }
    }
  }
  JF_TL_EXIT(TL_ARGMAX);
}

cudaError_t launch_argmax_finish(const GemmEpi& e, int M, int n_slots, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((M + 3) / 4);
  cfg.blockDim = dim3(128);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_argmax_finish, reinterpret_cast<const uint32_t*>(e.am_v1),
                            reinterpret_cast<const uint32_t*>(e.am_i1), reinterpret_cast<const uint32_t*>(e.am_v2), n_slots,
                            M, e.am_out, e.top2_out);
}

// ---------------------------------------------------------------------------------------------
// Epilogue on one 16-column chunk: thread `row` (0..127) holds v[j] = Y[m0 + c0 + j, n0 + row].
// xs: shared staging [16][128] fp32 (exchange between the two halves of a tile).
// ---------------------------------------------------------------------------------------------
template <typename T, int EPI, int NH>
JF_DEV void epilogue_chunk(const GemmEpi& e, const float (&v)[16], const EpiThreads<NH>& th, int n0, int m0, int c0, float* xs,
                           int n_tile, const AmEntries& am) {
  const int row = th.row, n = n0 + row;
  constexpr int kind = EPI;
  if constexpr (kind == EPI_STORE || kind == EPI_RESID) {
    if (n < e.N) {
      if constexpr (kind == EPI_RESID) {
        // all residual loads first (independent), then the stores
        float old[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int m = m0 + c0 + j;
          old[j] = (m < e.M) ? e.x[(size_t)m * e.ldx + n] : 0.0f;
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int m = m0 + c0 + j;
          if (m < e.M) e.x[(size_t)m * e.ldx + n] = old[j] + v[j];
        }
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int m = m0 + c0 + j;
          if (m < e.M) e.y[(size_t)m * e.ldy + n] = v[j];
        }
      }
    }
    return;
  } else if constexpr (kind == EPI_SWIGLU) {
    // rows 2i (gate) and 2i+1 (up) of the tile are feature 64 * n_tile + i, held by adjacent lanes:
    // the even lane finishes columns 0..7 of the chunk, the odd lane columns 8..15
    const bool odd = (row & 1) != 0;
    const int f = n_tile * 64 + (row >> 1);
    T* act = reinterpret_cast<T*>(e.act);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float mine = odd ? v[k] : v[8 + k];
      const float other = __shfl_xor_sync(0xffffffffu, mine, 1);
      const float g = odd ? other : v[k];
      const float u = odd ? v[8 + k] : other;
      const int m = m0 + c0 + (odd ? 8 + k : k);
      if (m < e.M && n < e.N) act[(size_t)m * e.ld_act + f] = to_act<T>(silu_f(g) * u);
    }
    return;
  } else if constexpr (kind == EPI_QKV) {
    // the feature's bias (if any) before the rotation, so that the partner reads biased values
    const float b = (e.bias != nullptr && n < e.N) ? act_to_f32(reinterpret_cast<const T*>(e.bias)[n]) : 0.f;
#pragma unroll
    for (int j = 0; j < 16; ++j) xs[j * 128 + row] = v[j] + b;
    th.sync();
    {
      const int hd = e.head_dim, half = hd >> 1;
      const int i = n % hd;
      const bool is_q = n < e.n_q;
      const bool is_k = !is_q && n < e.n_q + e.n_kv;
      const bool rot = is_q || is_k;
      const int partner = (i < half) ? row + half : row - half;
      T* dst;
      size_t stride;
      if (is_q) { dst = reinterpret_cast<T*>(e.q_out) + n; stride = (size_t)e.n_q; }
      else if (is_k) { dst = reinterpret_cast<T*>(e.k_out) + (n - e.n_q); stride = (size_t)e.n_kv; }
      else { dst = reinterpret_cast<T*>(e.v_out) + (n - e.n_q - e.n_kv); stride = (size_t)e.n_kv; }
      if (n < e.N) {
        // positions, then rotary coefficients: two rounds of independent loads for 16 tokens
        int pm[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int m = m0 + c0 + j;
          pm[j] = (rot && m < e.M) ? e.pos[m] : 0;
        }
        float2 cs[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) cs[j] = rot ? e.rope[(size_t)pm[j] * half + (i % half)] : make_float2(1.f, 0.f);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int m = m0 + c0 + j;
          float out = xs[j * 128 + row];
          if (rot) {
            const float x2 = xs[j * 128 + partner];
            out = (i < half) ? (out * cs[j].x - x2 * cs[j].y) : (out * cs[j].x + x2 * cs[j].y);
          }
          if (m < e.M) dst[(size_t)m * stride] = to_act<T>(out);
        }
      }
    }
    th.sync();
    return;
  } else {
    // EPI_ARGMAX: best (value, lowest index) and runner-up over this tile's 128 vocabulary rows. A warp
    // reduces a column with two redux instructions on order-preserving keys; lane j keeps column j.
    const int warp = row >> 5, lane = row & 31;
    uint32_t b1 = 0, b2 = 0, bi = 0;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const uint32_t key = n < e.N ? am_key(v[j]) : 0u;
      const uint32_t top = __reduce_max_sync(0xffffffffu, key);
      const int win = __ffs((int)__ballot_sync(0xffffffffu, key == top)) - 1;
      const uint32_t second = __reduce_max_sync(0xffffffffu, lane == win ? 0u : key);
      if (lane == j) {
        b1 = top;
        bi = (uint32_t)(n - lane + win);
        b2 = second;
      }
    }
    // (alternates from one of the group's chunks to the next: one barrier a chunk is enough)
    uint32_t* red = am.red + (th.half * 2 + (c0 / (16 * NH) & 1)) * (4 * 16 * 3);
    if (lane < 16) {
      uint32_t* mine = red + (warp * 16 + lane) * 3;
      mine[0] = b1;
      mine[1] = bi;
      mine[2] = b2;
    }
    th.sync();
    const int m = m0 + c0 + row;
    if (row < 16 && m < e.M) {
#pragma unroll
      for (int w = 1; w < 4; ++w) {
        const uint32_t* o = red + (w * 16 + row) * 3;
        am_merge(b1, bi, b2, o[0], o[1], o[2]);
      }
      // fold this tile into the CTA's running entry of row m; the same thread owns the row's entry for
      // every tile of the CTA, so program order orders the updates
      const size_t at = (size_t)m * am.stride;
      am_merge(b1, bi, b2, am.k1[at], am.idx[at], am.k2[at]);
      am.k1[at] = b1;
      am.idx[at] = bi;
      am.k2[at] = b2;
    }
  }
}

// A split tile's CTAs draw tickets with atomicDec, which starts anew from 0 and from any word above the split
// count. jf_op_gemm's tickets lie behind its partial tiles, at a place that depends on the shape, and another
// shape's call on the same workspace may have left partials there: they are stored complemented, so that none
// of them reads as 1 .. 7 (the complements of those are NaNs that no sum gives: a sum's NaN is 0x7fffffff).
JF_DEV float complement(float v) { return __uint_as_float(~__float_as_uint(v)); }

// Shared tail of both mainloops, run by the epilogue threads: the partial tile for EPI_PARTIAL;
// otherwise ticketing for split-K, then the epilogue. get(c0, v) fills this thread's 16 accumulator
// values of columns c0..c0+15. am: this CTA's argmax entries.
template <typename T, int BN, int EPI, int NH, typename Get>
JF_DEV void finish_tile(const GemmParams& p, Get get, float* xs, int* sflag, int n_tile, int split, int m_tile,
                        const EpiThreads<NH>& th, const AmEntries& am) {
  const int n0 = n_tile * kTileN, m0 = m_tile * BN;
  const int tile_lin = n_tile * p.m_tiles + m_tile;
  int ncols = p.M - m0;
  if (ncols > BN) ncols = BN;
  const int nchunks = (ncols + 15) >> 4;
  auto store_partial = [&](auto word) {
    float* mine = p.ws + ((size_t)tile_lin * p.k_splits + split) * (size_t)BN * kTileN;
    for (int c = th.half; c < nchunks; c += NH) {
      float v[16];
      get(c * 16, v);
#pragma unroll
      for (int j = 0; j < 16; ++j) mine[(c * 16 + j) * kTileN + th.row] = word(v[j]);
    }
  };
  if constexpr (EPI == EPI_PARTIAL) {
    store_partial([](float v) { return v; });
  } else if (p.k_splits == 1) {
    for (int c = th.half; c < nchunks; c += NH) {
      float v[16];
      get(c * 16, v);
      epilogue_chunk<T, EPI>(p.epi, v, th, n0, m0, c * 16, xs, n_tile, am);
    }
  } else {
    store_partial(complement);
    __threadfence();
    th.sync_all();
    if (th.first()) {
      // 0 or a stale word -> k_splits - 1 -> ... -> 1 -> 0
      *sflag = atomicDec(reinterpret_cast<unsigned*>(p.tile_counter) + tile_lin, (unsigned)p.k_splits - 1u) == 1u;
    }
    th.sync_all();
    const bool last = *sflag != 0;
    th.sync_all();
    if (!last) return;
    __threadfence();
    const float* base = p.ws + (size_t)tile_lin * p.k_splits * (size_t)BN * kTileN;
    for (int c = th.half; c < nchunks; c += NH) {
      // partials of four splits in flight together, added in split order
      float v[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = 0.0f;
#pragma unroll
      for (int s0 = 0; s0 < kMaxSplits; s0 += 4) {
        float part[4][16];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const float* src = base + (size_t)(s0 + s) * BN * kTileN;
#pragma unroll
          for (int j = 0; j < 16; ++j)
            part[s][j] = (s0 + s < p.k_splits) ? complement(__ldcg(src + (c * 16 + j) * kTileN + th.row)) : 0.0f;
        }
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          if (s0 + s < p.k_splits) {
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] += part[s][j];
          }
        }
      }
      epilogue_chunk<T, EPI>(p.epi, v, th, n0, m0, c * 16, xs, n_tile, am);
    }
  }
}

// Work unit u of the persistent schedule: split = u % k_splits; the k_splits units of a tile are
// consecutive (their partials meet soon), and so are the m tiles of a weight tile (its second
// read hits L2). n_tile counts pairs of tiles when two CTAs share one.
struct Unit {
  int n_tile, m_tile, split, kb0, kb1;
};
JF_DEV Unit unit_of(const GemmParams& p, int u) {
  Unit w;
  w.split = u % p.k_splits;
  const int t = u / p.k_splits;
  w.m_tile = t % p.m_tiles;
  w.n_tile = t / p.m_tiles;
  w.kb0 = (int)((unsigned)(p.kb_total * w.split) / (unsigned)p.k_splits);  // (at most 8 splits)
  w.kb1 = (int)((unsigned)(p.kb_total * (w.split + 1)) / (unsigned)p.k_splits);
  return w;
}

// ---------------------------------------------------------------------------------------------
// bf16 tcgen05 persistent kernel, 320 threads: warps 0-7 epilogue (warp w reads TMEM lanes
// 32(w%4) .. 32(w%4)+31 and every other 16-column chunk: the last unit's epilogue is not hidden, and
// eight warps halve it), warp 8 = TMA producer, warp 9 = MMA issuer (and the TMEM allocation).
// (8 layers and head of the 7B shape: 64 rows 990 -> 978 us, 160 rows 1198 -> 1167; 32 rows as before).
//
// PAIR (more than 160 rows): two CTAs on neighbouring SMs take a tile of 256 weight rows together
// (cta_group::2). Each loads its own 128 weight rows and half of the tokens (at 256 tokens 32 KB a 64-k
// stage instead of 48), rank 0 issues the MMAs of both, and each drains its own 128 rows. With
// one CTA per tile the operands, not the tensor cores, bounded it: 48 KB a 512-cycle stage is more than
// an SM draws from L2, and only four such stages fit. gate/up (37888 x 3584) at 512 rows: 110.6 ->
// 104.9 us a call, the launch 103.5 -> 87 (ncu; 1.6 PFLOP/s, tensor pipe 77% of the active cycles); prefill of
// 4,000 tokens through one 7B layer 2.39 -> 2.29 ms.
// ---------------------------------------------------------------------------------------------
constexpr int EPI_HALVES = 2, PRODUCER_WARP = 4 * EPI_HALVES, MMA_WARP = PRODUCER_WARP + 1;
constexpr int TC_THREADS = 32 * (MMA_WARP + 1);

template <int BN, int EPI, bool PAIR>
__global__ void __launch_bounds__(TC_THREADS, 1)
    k_gemm_tc(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const GemmParams p) {
  using Cfg = TcCfg<BN, PAIR>;
  // The ring's unit is a stage pair: two 64-k blocks (one at an odd unit's end) with one full and one
  // empty barrier, so that a wait, an arrival and a commit (about 100-200 cycles each) serve 128 k.
  constexpr int S = Cfg::STAGES, D = S / 2;
  constexpr int kCtas = PAIR ? 2 : 1;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  uint8_t* sA = smem;
  uint8_t* sB = smem + S * A_STAGE_BYTES;
  float* xs = reinterpret_cast<float*>(sB + S * Cfg::B_STAGE_BYTES);
  uint64_t* bars = reinterpret_cast<uint64_t*>(reinterpret_cast<uint8_t*>(xs) + EPI_STAGE_BYTES);
  const uint32_t idle = smem_u32(bars + 2 * D + 4);  // never completes: a wait for its odd phase passes
  const uint32_t sink = smem_u32(bars + 2 * D + 5);  // nobody waits for it
  const uint32_t all_done = smem_u32(bars + 2 * D + 6);  // every MMA of this CTA (of the pair, in rank 0)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * D + 7);
  int* sflag = reinterpret_cast<int*>(tmem_slot + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + D);
  const uint32_t tfull0 = smem_u32(bars + 2 * D), tempty0 = smem_u32(bars + 2 * D + 2);
  const int rank = PAIR ? (int)cluster_rank() : 0;
  // a pair's full and tempty barriers are rank 0's
  const uint32_t lead_full0 = PAIR ? map_to_rank(full0, 0) : full0;
  const int first_unit = (int)blockIdx.x / kCtas, unit_step = (int)gridDim.x / kCtas;
  const int total_units = ((p.n_tiles + kCtas - 1) / kCtas) * p.m_tiles * p.k_splits;
  JF_TL_ENTRY();
  // The next kernel may launch as soon as every CTA of this grid is resident: its CTAs take the
  // SMs this grid leaves, prefetch their own weights and park in their dependency wait, so no
  // launch latency is paid after the last tile (it writes nothing before that wait).
  pdl_launch_dependents();

  int total_iters = 0;  // stage pairs of this CTA
  for (int u = first_unit; u < total_units; u += unit_step) {
    const Unit w = unit_of(p, u);
    total_iters += (w.kb1 - w.kb0 + 1) / 2;
  }
  const int pre = total_iters < D ? total_iters : D;
  // k blocks kb and kb + 1 (if it belongs to the unit) into stage pair d (predicated off when `on` is false)
  auto load_a = [&](const Unit& w, int kb, int d, uint64_t pol, bool on) {
    const int n0 = (w.n_tile * kCtas + rank) * kTileN;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t dst = smem_u32(sA + (2 * d + h) * A_STAGE_BYTES);
      const bool live = on && kb + h < w.kb1;
      if constexpr (PAIR) tma_load_2d_pair(dst, &tmA, lead_full0 + 8 * d, (kb + h) * kTileK, n0, pol, live);
      else tma_load_2d(dst, &tmA, full0 + 8 * d, (kb + h) * kTileK, n0, pol, live);
    }
  };
  auto load_b = [&](const Unit& w, int kb, int d, uint64_t pol, bool on) {
    const int m0 = w.m_tile * BN + rank * Cfg::B_ROWS;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t dst = smem_u32(sB + (2 * d + h) * Cfg::B_STAGE_BYTES);
      const bool live = on && kb + h < w.kb1;
      if constexpr (PAIR) tma_load_2d_pair(dst, &tmB, lead_full0 + 8 * d, (kb + h) * kTileK, m0, pol, live);
      else tma_load_2d(dst, &tmB, full0 + 8 * d, (kb + h) * kTileK, m0, pol, live);
    }
  };
  // rank 0 expects the bytes of both CTAs
  auto expect = [&](const Unit& w, int kb, int d, bool on) {
    mbar_arrive_expect_tx(full0 + 8 * d, (kb + 1 < w.kb1 ? 2 : 1) * kCtas * Cfg::STAGE_BYTES, on && rank == 0);
  };
  if (tid == 32 * PRODUCER_WARP) {
    for (int d = 0; d < D; ++d) {
      mbar_init(full0 + 8 * d, 1);
      mbar_init(empty0 + 8 * d, 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull0 + 8 * a, 1);
      mbar_init(tempty0 + 8 * a, kCtas);
    }
    mbar_init(idle, 1);
    mbar_init(sink, 1);
    mbar_init(all_done, 1);
    fence_mbar_init();
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
  }
  if (warp == MMA_WARP) {
    if constexpr (PAIR) {
      tmem_alloc_pair(smem_u32(tmem_slot), Cfg::TMEM_COLS);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(smem_u32(tmem_slot), Cfg::TMEM_COLS);
      tmem_relinquish();
    }
  }
  __syncwarp();
  tc_fence_before();
  if constexpr (PAIR) {
    __syncthreads();
    cluster_sync();  // both CTAs' barriers exist, and both hold their TMEM
  } else if (warp == PRODUCER_WARP) {
    asm volatile("bar.arrive 2, %0;" ::"n"(TC_THREADS) : "memory");  // the producer starts without waiting for the others
  } else {
    asm volatile("bar.sync 2, %0;" ::"n"(TC_THREADS) : "memory");
  }
  tc_fence_after();

  if (warp == PRODUCER_WARP) {
    // Stage pairs 0 .. pre-1: lane j requests the weights of pair j before the dependency wait (a forward's
    // weights were complete before it began, so they stream in while the previous kernel finishes; the W of
    // jf_op_gemm may be the previous kernel's output and is requested after the wait: a launch of 4608 x 3584,
    // 32 rows, inside a graph takes 11.0 us, 12 as a full boundary, 8.9 with the weights first) and its
    // activations right after it; from then on one lane requests both of a pair as it comes free. Round
    // -1 of the loop goes through all of it with the requests predicated off, so that the code is in the
    // instruction cache when the wait ends: the weights that stream through L2 push code out of it, and
    // fetching it there put the first refill 2.5 us after the wait (now 0.8).
    const uint64_t polA = l2_policy_evict_first(), polB = l2_policy_evict_last();
    Unit w0 = unit_of(p, first_unit);
    int u = first_unit, kb0 = w0.kb0 + 2 * lane;  // stage pair `lane`
    while (lane < pre && kb0 >= w0.kb1) {
      u += unit_step;
      const int over = kb0 - (w0.kb1 + ((w0.kb1 - w0.kb0) & 1));  // (a unit takes whole pairs)
      w0 = unit_of(p, u);
      kb0 = w0.kb0 + over;
    }
    if (!p.w_ready) pdl_wait();
    if (lane < pre) {
      expect(w0, kb0, lane, true);
      load_a(w0, kb0, lane, polA, true);
    }
    __syncwarp();
    u = __shfl_sync(0xffffffffu, u, pre - 1);
    int kb = __shfl_sync(0xffffffffu, kb0, pre - 1) + 2;
    Unit w = unit_of(p, u);
    int d = pre == D ? 0 : pre, issued = pre;
    uint32_t parity = 0u;
#pragma unroll 1
    for (int q = -1; q <= 0 || pre + q < total_iters; ++q) {
      const bool on = q >= 0;
      if (q <= 0) {
        if (on) pdl_wait();
        if (lane < pre) load_b(w0, kb0, lane, polB, on);
        __syncwarp();
        if (on && pre >= total_iters) break;
      }
      if (on && kb >= w.kb1) {
        u += unit_step;
        w = unit_of(p, u);
        kb = w.kb0;
      }
      const bool ok = mbar_wait_bounded(on ? empty0 + 8 * d : idle, on ? parity : 1u, p.wait_ns);
      if (!__all_sync(0xffffffffu, ok)) {
        if (lane == 0) jf_set_error(p.err, JF_DERR_TIMEOUT_MMA);
        break;
      }
      if (elect_one()) {
        expect(w, kb, d, on);
        load_a(w, kb, d, polA, on);
        load_b(w, kb, d, polB, on);
      }
      __syncwarp();
      if (on) {
        ++issued;
        kb += 2;
        if (++d == D) {
          d = 0;
          parity ^= 1u;
        }
      }
    }
    // Every copy has landed before the CTA may leave, also after a wait that gave up (a pair's complete on rank
    // 0's barriers; when a wait gives up here too, the copies have had its limit to land).
    if (rank == 0)
      for (int q = issued > D ? issued - D : 0; q < issued; ++q)
        if (!mbar_wait_bounded(full0 + 8 * (q % D), (uint32_t)(q / D) & 1u, p.wait_ns)) break;
    if constexpr (PAIR) {  // rank 0's last arrivals on this CTA's barriers, before it may leave
      for (int q = total_iters > D ? total_iters - D : 0; q < total_iters; ++q)
        if (!mbar_wait_bounded(empty0 + 8 * (q % D), (uint32_t)(q / D) & 1u, p.wait_ns)) break;
    }
    __syncwarp();
  } else if (warp == MMA_WARP) {
    // The whole warp walks the stage pairs, one elected lane issues (a wait behind issued MMAs takes as
    // long as they queue); descriptors are a base plus constants. The first pass over the loop computes
    // on whatever the stages hold, into an accumulator that the first real MMA overwrites, and its waits
    // pass: it fetches the code while the stages are on their way.
    const uint32_t tmem = *tmem_slot;
    if (rank == 0) {
      constexpr uint32_t idesc = idesc_bf16_f32(kCtas * kTileN, BN);
      const uint64_t da = sdesc_k_sw128(smem_u32(sA)), db = sdesc_k_sw128(smem_u32(sB));
      int d = 0, i = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int u = first_unit; u < total_units && ok; u += unit_step, ++i) {
        const Unit w = unit_of(p, u);
        const int acc = i & 1;
        const uint32_t prev = (uint32_t)((i >> 1) - 1) & 1u;  // phase of the accumulator's previous use
        if (i >= 2 && !__all_sync(0xffffffffu, mbar_wait_bounded(tempty0 + 8 * acc, prev, p.wait_ns))) {
          if (lane == 0) jf_set_error(p.err, JF_DERR_TIMEOUT_EPI);
          break;
        }
        tc_fence_after();
        const uint32_t dacc = tmem + (uint32_t)(acc * Cfg::ACC_COLS);
#pragma unroll 1
        for (int kb = w.kb0 - (i == 0 ? 2 : 0); kb < w.kb1; kb += 2) {
          const bool on = kb >= w.kb0;  // (a unit has at least one k block: the last round is on)
          ok = mbar_wait_bounded(on ? full0 + 8 * d : idle, on ? phase : 1u, p.wait_ns);
          if (!__all_sync(0xffffffffu, ok)) {
            if (lane == 0) jf_set_error(p.err, JF_DERR_TIMEOUT_TMA);
            ok = false;
            break;
          }
          tc_fence_after();
          if (elect_one()) {
            const uint64_t a0 = da + (uint64_t)(d * (2 * A_STAGE_BYTES >> 4));
            const uint64_t b0 = db + (uint64_t)(d * (2 * Cfg::B_STAGE_BYTES >> 4));
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              if (h == 1 && kb + 1 >= w.kb1) break;
#pragma unroll
              for (int kk = 0; kk < kTileK / 16; ++kk) {
                const uint64_t a = a0 + h * (A_STAGE_BYTES >> 4) + kk * 2, b = b0 + h * (Cfg::B_STAGE_BYTES >> 4) + kk * 2;
                const uint32_t add = (h > 0 || kk > 0 || kb != w.kb0) ? 1u : 0u;
                if constexpr (PAIR) tc_mma_bf16_pair(dacc, a, b, idesc, add);
                else tc_mma_bf16(dacc, a, b, idesc, add);
              }
            }
            const uint32_t bar = on ? empty0 + 8 * d : sink;
            if constexpr (PAIR) tc_commit_pair(bar);
            else tc_commit(bar);
            if (kb + 2 >= w.kb1) {
              if constexpr (PAIR) tc_commit_pair(tfull0 + 8 * acc);
              else tc_commit(tfull0 + 8 * acc);
            }
          }
          __syncwarp();
          if (on && ++d == D) {
            d = 0;
            phase ^= 1u;
          }
        }
      }
      // every MMA is complete before the tensor memory is given back, also after a wait that gave up
      if (elect_one()) {
        if constexpr (PAIR) tc_commit_pair_local(all_done);
        else tc_commit(all_done);
      }
      __syncwarp();
      mbar_wait_bounded(all_done, 0u, p.wait_ns);
    }
    __syncwarp();
  } else {
    // epilogue warps
    pdl_wait();
    JF_TL_WAITED();
    uint32_t* words = reinterpret_cast<uint32_t*>(xs);
    const bool table = p.M <= kAmTableRows;
    const EpiThreads<EPI_HALVES> th{warp >> 2, tid & 127};
    AmEntries am = {};
    if constexpr (EPI == EPI_ARGMAX) {
      am = table ? am_shared(words) : am_global(p.epi, words, blockIdx.x, gridDim.x);
      am_clear(am, 0, p.M, tid, 128 * EPI_HALVES);
      th.sync_all();
    }
    const uint32_t tmem = *tmem_slot;
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    int i = 0;
    for (int u = first_unit; u < total_units; u += unit_step, ++i) {
      const Unit w = unit_of(p, u);
      const int acc = i & 1;
      // agreed on by all epilogue threads: they share barriers below
      const bool ready = mbar_wait_bounded(tfull0 + 8 * acc, (uint32_t)(i >> 1) & 1u, p.wait_ns);
      if (!sync_and<3, 128 * EPI_HALVES>(ready)) {
        if (!ready) jf_set_error(p.err, JF_DERR_TIMEOUT_EPI);
        break;
      }
      tc_fence_after();
      const uint32_t dacc = tmem + (uint32_t)(acc * Cfg::ACC_COLS) + lane_base;
      auto get = [&](int c0, float (&v)[16]) { tmem_ld16(dacc + (uint32_t)c0, v); };
      const int n_tile = w.n_tile * kCtas + rank;
      if (n_tile < p.n_tiles)  // (the last pair's second tile may not exist)
        finish_tile<bf16, BN, EPI>(p, get, xs, sflag, n_tile, w.split, w.m_tile, th, am);
      if (u + unit_step >= total_units) break;  // nobody waits for the last accumulator to be free
      tc_fence_before();
      th.sync_all();
      if (tid == 0) {
        if constexpr (PAIR) mbar_arrive_cluster(map_to_rank(tempty0 + 8 * acc, 0));
        else mbar_arrive(tempty0 + 8 * acc);
      }
    }
    if constexpr (EPI == EPI_ARGMAX) {
      if (table) {
        th.sync_all();
        const AmEntries out = am_global(p.epi, words, blockIdx.x, gridDim.x);
        for (int m = tid; m < p.M; m += 128 * EPI_HALVES) {
          out.k1[m * out.stride] = am.k1[m];
          out.idx[m * out.stride] = am.idx[m];
          out.k2[m * out.stride] = am.k2[m];
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) {
    cluster_sync();  // neither CTA leaves while the other may use its shared or tensor memory
    if (warp == MMA_WARP) tmem_dealloc_pair(*tmem_slot, Cfg::TMEM_COLS);
  } else {
    if (warp == MMA_WARP) tmem_dealloc(*tmem_slot, Cfg::TMEM_COLS);
  }
  JF_TL_EXIT(TL_GEMM + EPI);
}

// ---------------------------------------------------------------------------------------------
// fp32 SIMT kernel: a cluster of n_splits CTAs per tile of 128 features x BN tokens, each CTA on its
// share of K. Weight and token tiles of 32 k stream through shared memory by cp.async (four stages);
// thread (row, h) sums Y[m0 .. m0+BN-1, n0 + row] over the k of half h of every tile; the halves, then
// the CTAs of the cluster in rank order (read from their shared memory), are added in a fixed order that
// depends on N and K alone. These models' matrices are small (a 256 x 1024 one is two feature tiles), so
// latency bounds the kernel: it is spread over 8-152 SMs instead of one CTA per tile whose threads each
// walked a weight row (a jf_op_gemm call of 4096 x 1024, 40 rows: 150 -> 53 us, of which a launch takes 26-35;
// the tiny fp32 decoder's generation, with the fp32 attention: 33.0 -> 5.3 ms).
// ---------------------------------------------------------------------------------------------
constexpr int F32_BK = 32;
constexpr int F32_STAGES = 4;
constexpr int F32_PITCH = F32_BK + 4;  // floats per tile row: 16-byte aligned, conflict-free 16-byte reads
constexpr int F32_THREADS = 256;
constexpr int f32_stage_floats(int bn) { return (kTileN + bn) * F32_PITCH; }
constexpr int f32_smem(int bn) { return F32_STAGES * f32_stage_floats(bn) * 4; }

// Four consecutive floats of a row (k .. k+3, zeros past K) into shared memory: one 16-byte copy when
// every row is 16-byte aligned, otherwise four 4-byte ones.
JF_DEV void f32_copy4(uint32_t dst, const float* row, int k, int K, bool ok, bool vec) {
  const int left = ok ? K - k : 0;
  if (vec) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(row + (left > 0 ? k : 0)),
                 "r"(left > 0 ? 16 : 0)
                 : "memory");
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + 4 * i), "l"(row + (left > i ? k + i : 0)),
                   "r"(left > i ? 4 : 0)
                   : "memory");
  }
}

JF_DEV float ld_cluster_f32(const float* p, uint32_t rank) {  // *p of the cluster's CTA `rank`
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(map_to_rank(smem_u32(p), rank)) : "memory");
  return v;
}

template <int BN, int EPI>
__global__ void __launch_bounds__(F32_THREADS) k_gemm_f32(const float* __restrict__ W, const float* __restrict__ X,
                                                          const GemmParams p, int n_splits, bool vec) {
  extern __shared__ __align__(16) float tiles[];  // F32_STAGES x {W [128][PITCH], X [BN][PITCH]}
  __shared__ float part[BN * kTileN];
  __shared__ float xs[16 * 128];
  __shared__ int sflag;
  const int tid = threadIdx.x, row = tid & 127, half = tid >> 7;
  const int n_tile = blockIdx.x / n_splits, split = blockIdx.x % n_splits;
  const int n0 = n_tile * kTileN, m0 = blockIdx.z * BN;
  const int kb0 = (int)((long long)p.kb_total * split / n_splits), kb1 = (int)((long long)p.kb_total * (split + 1) / n_splits);
  pdl_launch_dependents();
  auto load = [&](int kb, int first, int last) {  // rows [first, last) of the stage: weights, then tokens
    const uint32_t base = smem_u32(tiles + ((kb - kb0) % F32_STAGES) * f32_stage_floats(BN));
    for (int i = first * (F32_BK / 4) + tid; i < last * (F32_BK / 4); i += F32_THREADS) {
      const int r = i / (F32_BK / 4), c = (i % (F32_BK / 4)) * 4;
      const bool w = r < kTileN;
      const int g = w ? n0 + r : m0 + r - kTileN;
      const bool ok = g < (w ? p.N : p.M);
      f32_copy4(base + (uint32_t)(r * F32_PITCH + c) * 4, (w ? W : X) + (ok ? (size_t)g * p.K : 0), kb * F32_BK + c, p.K, ok,
                vec);
    }
  };
  // A forward's weights were complete before it began: their first tiles are fetched before the
  // dependency wait (the tiny decoder's generation 6.63 -> 6.23 ms). jf_op_gemm's W may be the previous
  // call's Y, so EPI_STORE waits first.
  constexpr bool kEarly = EPI != EPI_STORE;
  if (kEarly) {
    for (int s = 0; s < F32_STAGES - 1; ++s)
      if (kb0 + s < kb1) load(kb0 + s, 0, kTileN);
  }
  pdl_wait();
  for (int s = 0; s < F32_STAGES - 1; ++s) {
    if (kb0 + s < kb1) load(kb0 + s, kEarly ? kTileN : 0, kTileN + BN);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  float acc[BN];
#pragma unroll
  for (int j = 0; j < BN; ++j) acc[j] = 0.0f;
  for (int kb = kb0; kb < kb1; ++kb) {
    asm volatile("cp.async.wait_group %0;" ::"n"(F32_STAGES - 2) : "memory");
    __syncthreads();  // this tile has landed; the one before it has been read by everyone
    if (kb + F32_STAGES - 1 < kb1) load(kb + F32_STAGES - 1, 0, kTileN + BN);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float* wt = tiles + ((kb - kb0) % F32_STAGES) * f32_stage_floats(BN) + half * (F32_BK / 2);
    const float* xt = wt + kTileN * F32_PITCH;
#pragma unroll
    for (int k = 0; k < F32_BK / 2; k += 4) {
      const float4 w = *reinterpret_cast<const float4*>(wt + row * F32_PITCH + k);
#pragma unroll
      for (int j = 0; j < BN; ++j) {
        const float4 x = *reinterpret_cast<const float4*>(xt + j * F32_PITCH + k);
        acc[j] = fmaf(w.x, x.x, acc[j]);
        acc[j] = fmaf(w.y, x.y, acc[j]);
        acc[j] = fmaf(w.z, x.z, acc[j]);
        acc[j] = fmaf(w.w, x.w, acc[j]);
      }
    }
  }
  if (half == 1) {
#pragma unroll
    for (int j = 0; j < BN; ++j) part[j * kTileN + row] = acc[j];
  }
  __syncthreads();
  if (half == 0) {
#pragma unroll
    for (int j = 0; j < BN; ++j) part[j * kTileN + row] += acc[j];
  }
  if (n_splits > 1) cluster_sync();  // every CTA's partial tile is visible to rank 0
  if (split == 0 && half == 0) {
    auto get = [&](int c0, float (&v)[16]) {
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = part[(c0 + j) * kTileN + row];
      for (int r0 = 1; r0 < n_splits; r0 += 4) {  // four CTAs' values in flight, added in rank order
        float q[4][16];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            q[r][j] = r0 + r < n_splits ? ld_cluster_f32(part + (c0 + j) * kTileN + row, (uint32_t)(r0 + r)) : 0.f;
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          if (r0 + r < n_splits) {
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] += q[r][j];
          }
        }
      }
    };
    const EpiThreads<1> th{0, row};
    AmEntries am = {};
    if constexpr (EPI == EPI_ARGMAX) {
      am = am_global(p.epi, reinterpret_cast<uint32_t*>(xs), n_tile, p.n_tiles);
      am_clear(am, m0, m0 + BN < p.M ? m0 + BN : p.M, tid, 128);
      th.sync_all();
    }
    finish_tile<float, BN, EPI>(p, get, xs, &sflag, n_tile, 0, blockIdx.z, th, am);
  }
  if (n_splits > 1) cluster_sync();  // the other CTAs keep their partial tiles until rank 0 has read them
}

template <int BN, int EPI, bool PAIR>
cudaError_t launch_tc_epi(const CUtensorMap& tmA, const CUtensorMap& tmB, const GemmParams& p, cudaStream_t st) {
  using Cfg = TcCfg<BN, PAIR>;
  constexpr int kCtas = PAIR ? 2 : 1;
  cudaLaunchConfig_t cfg = {};
  const int units = ((p.n_tiles + kCtas - 1) / kCtas) * p.m_tiles * p.k_splits;
  const int groups = p.grid / kCtas;
  cfg.gridDim = dim3(kCtas * (units < groups ? units : groups));
  cfg.blockDim = dim3(TC_THREADS);
  cfg.dynamicSmemBytes = Cfg::SMEM;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = kCtas;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = PAIR ? 2 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_gemm_tc<BN, EPI, PAIR>, tmA, tmB, p);
  if (EPI != EPI_ARGMAX || e != cudaSuccess) return e;
  return launch_argmax_finish(p.epi, p.M, (int)cfg.gridDim.x, st);
}

template <int BN, bool PAIR = false>
cudaError_t launch_tc(const CUtensorMap& tmA, const CUtensorMap& tmB, const GemmParams& p, cudaStream_t st) {
  switch (p.epi.kind) {
    case EPI_STORE: return launch_tc_epi<BN, EPI_STORE, PAIR>(tmA, tmB, p, st);
    case EPI_SWIGLU: return launch_tc_epi<BN, EPI_SWIGLU, PAIR>(tmA, tmB, p, st);
    case EPI_ARGMAX: return launch_tc_epi<BN, EPI_ARGMAX, PAIR>(tmA, tmB, p, st);
    case EPI_PARTIAL: return launch_tc_epi<BN, EPI_PARTIAL, PAIR>(tmA, tmB, p, st);
    default: return cudaErrorInvalidValue;
  }
}

template <typename K>
cudaError_t opt_in(K kernel, int smem) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

template <int BN, bool PAIR = false>
cudaError_t prep_tc() {
  cudaError_t e;
  const int sm = TcCfg<BN, PAIR>::SMEM;
  if ((e = opt_in(k_gemm_tc<BN, EPI_STORE, PAIR>, sm)) || (e = opt_in(k_gemm_tc<BN, EPI_SWIGLU, PAIR>, sm)) ||
      (e = opt_in(k_gemm_tc<BN, EPI_ARGMAX, PAIR>, sm)))
    return e;
  return opt_in(k_gemm_tc<BN, EPI_PARTIAL, PAIR>, sm);
}

}  // namespace

#ifdef JF_TIMELINE
JF_TL_SETTER(tl_set_gemm)
#endif

template <int BN>
static cudaError_t prep_f32() {
  cudaError_t e;
  const int sm = f32_smem(BN);
  if ((e = cudaFuncSetAttribute(k_gemm_f32<BN, EPI_STORE>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm))) return e;
  if ((e = cudaFuncSetAttribute(k_gemm_f32<BN, EPI_RESID>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm))) return e;
  if ((e = cudaFuncSetAttribute(k_gemm_f32<BN, EPI_QKV>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm))) return e;
  if ((e = cudaFuncSetAttribute(k_gemm_f32<BN, EPI_SWIGLU>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm))) return e;
  return cudaFuncSetAttribute(k_gemm_f32<BN, EPI_ARGMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
}

// Opt the kernels into their dynamic shared-memory sizes on the current device.
static cudaError_t gemm_prepare_current() {
  cudaError_t e;
  if ((e = prep_f32<16>()) != cudaSuccess) return e;
  if ((e = prep_f32<32>()) != cudaSuccess) return e;
  if ((e = prep_tc<16>()) != cudaSuccess) return e;
  if ((e = prep_tc<32>()) != cudaSuccess) return e;
  if ((e = prep_tc<64>()) != cudaSuccess) return e;
  if ((e = prep_tc<128>()) != cudaSuccess) return e;
  if ((e = prep_tc<160>()) != cudaSuccess) return e;
  if ((e = prep_tc<160, true>()) != cudaSuccess) return e;
  if ((e = prep_tc<192, true>()) != cudaSuccess) return e;
  if ((e = prep_tc<224, true>()) != cudaSuccess) return e;
  return prep_tc<256, true>();
}

// The attributes are per device: set them once for each device the process uses (outside any
// stream capture), whichever entry point reaches that device first.
cudaError_t gemm_prepare() {
  static PerDeviceOnce once;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const int r = once.run(dev, [] { return gemm_prepare_current(); });
  return r < 0 ? cudaErrorInvalidDevice : static_cast<cudaError_t>(r);
}

// Token-tile width. Up to 256 rows one tile, the narrowest that holds them; above, as few tiles as 256-wide
// ones would be (every further tile is another pass over the weights) and among the widths that give that
// count the narrowest (the tensor cores' work grows with the padded rows). 8 layers and head of the 7B
// shape, us: 16-wide against 32-wide tiles at one row 867 / 879 (twelve stages instead of ten, half the
// activation copies); 192 against 256 at 192 rows 1248 / 1275, at 384 (two tiles) 1750 / 1899; 224 against
// 256 at 224 rows 1293 / 1308, at 448 1900 / 1990. Three 128-wide tiles at 384 rows were slower than two of
// 256.
int gemm_bn_for(int M) {
  if (M <= 16) return 16;
  if (M <= 32) return 32;
  if (M <= 64) return 64;
  if (M <= 128) return 128;
  const int tiles = (M + 255) / 256;
  for (int bn : {128, 160, 192, 224})
    if ((M + bn - 1) / bn == tiles) return bn;
  return 256;
}

// Token rows of one TMA box of the activations: above 160 rows CTA pairs run, whose CTAs load half of a
// tile's tokens each (320 rows as two 160-wide tiles: 1568 us by pairs, 1660 by single CTAs; pairs at 32,
// 64, 128 and 160 rows: 0-1% slower, 3% on the 1.5B shape, whose short projections pay for the cluster).
int gemm_box_rows(int bn, int M) { return M > 160 ? bn / 2 : bn; }

cudaError_t launch_gemm_bf16(const CUtensorMap& tmA, const CUtensorMap& tmB, const GemmParams& p, int bn,
                             cudaStream_t st) {
  switch (bn) {
    case 16: return launch_tc<16>(tmA, tmB, p, st);
    case 32: return launch_tc<32>(tmA, tmB, p, st);
    case 64: return launch_tc<64>(tmA, tmB, p, st);
    case 128: return launch_tc<128>(tmA, tmB, p, st);
    case 160: return p.M > 160 ? launch_tc<160, true>(tmA, tmB, p, st) : launch_tc<160>(tmA, tmB, p, st);
    case 192: return launch_tc<192, true>(tmA, tmB, p, st);
    case 224: return launch_tc<224, true>(tmA, tmB, p, st);
    case 256: return launch_tc<256, true>(tmA, tmB, p, st);
    default: return cudaErrorInvalidValue;
  }
}

// CTAs per tile of the fp32 kernel (from N and K alone, so that a row's sums do not depend on the rows in
// flight): a power of two up to 8, at least 64 k each, about one CTA per SM of a 152-SM GPU at the most.
static int f32_splits(int n_tiles, int K) {
  int s = 1;
  while (s < 8 && 2 * s * 64 <= K && 2 * s * n_tiles <= 152) s *= 2;
  return s;
}

template <int BN, int EPI>
static cudaError_t launch_f32_epi(const float* W, const float* X, GemmParams p, cudaStream_t st) {
  p.m_tiles = (p.M + BN - 1) / BN;
  p.kb_total = (p.K + F32_BK - 1) / F32_BK;
  const int splits = f32_splits(p.n_tiles, p.K);
  const bool vec = p.K % 4 == 0 && ((reinterpret_cast<uintptr_t>(W) | reinterpret_cast<uintptr_t>(X)) & 15) == 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.n_tiles * splits, 1, p.m_tiles);
  cfg.blockDim = dim3(F32_THREADS);
  cfg.dynamicSmemBytes = f32_smem(BN);
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = splits;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = splits > 1 ? 2 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_gemm_f32<BN, EPI>, W, X, p, splits, vec);
  if (EPI != EPI_ARGMAX || e != cudaSuccess) return e;
  return launch_argmax_finish(p.epi, p.M, p.n_tiles, st);
}

template <int BN>
static cudaError_t launch_f32(const float* W, const float* X, const GemmParams& p, cudaStream_t st) {
  switch (p.epi.kind) {
    case EPI_STORE: return launch_f32_epi<BN, EPI_STORE>(W, X, p, st);
    case EPI_RESID: return launch_f32_epi<BN, EPI_RESID>(W, X, p, st);
    case EPI_QKV: return launch_f32_epi<BN, EPI_QKV>(W, X, p, st);
    case EPI_SWIGLU: return launch_f32_epi<BN, EPI_SWIGLU>(W, X, p, st);
    case EPI_ARGMAX: return launch_f32_epi<BN, EPI_ARGMAX>(W, X, p, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_gemm_f32(const float* W, const float* X, const GemmParams& p, cudaStream_t st) {
  // 32-token tiles once they fill the GPU (half the weight reads), 16-token ones below that
  const long long ctas32 = (long long)p.n_tiles * f32_splits(p.n_tiles, p.K) * ((p.M + 31) / 32);
  return ctas32 >= 304 ? launch_f32<32>(W, X, p, st) : launch_f32<16>(W, X, p, st);
}

}  // namespace jf
