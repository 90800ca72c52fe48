// Attention of the in-flight rows over the exact committed KV cache (Sec. 2.1, Eq. 3: the
// block's n conditionals come out of one pass with a causal mask) and the block-causal tree mask
// of multi-block decoding and rejection recycling (Sec. 3.2, Algorithm 1).
//
// Rows are grouped into chains (jf_internal.h): a chain's rows sit at consecutive positions
// starting at the sequence's committed length P, and a row at position p attends to cache
// positions [0, P) and to the chain's own rows at positions P .. p. A real-active draft followed
// by its pseudo-active blocks is one chain; each recycled candidate is a chain of its own. Hence
// every row attends to exactly the positions 0 .. p, each position resolved either to a KV page
// (p < P) or to an in-flight row of its chain.
//
// bf16 path: split-KV flash decoding on the tcgen05 tensor cores with a fixed reduction tree.
// Work unit = (chain, KV head, tile of up to 128 (token, head) query rows of whole tokens). Key positions are cut into
// absolute 128-key chunks, and chunk c belongs to lane c mod 8; a lane's chunks are taken in
// increasing order with one online-softmax state per row, and the 8 lane states (O, maximum, sum) are
// folded in lane order. The tree depends only on absolute key positions, never on how many rows share
// the forward or how many chunks a unit has, so a row's result is the same in every batch. The lanes
// of a unit are spread over a cluster of 8, 4 or 2 CTAs, or one CTA takes them all (jf_attn_form.h).
// fp32 path: four warps per (row, head) on absolute 32-key groups, online softmax in fp32, folded in
// warp order.
#include "jf_device.cuh"
#include "jf_internal.h"

namespace jf {
namespace {

constexpr int HD = 128;
constexpr int ROWS_PER_BLOCK = kAttnQRows / kAttnLanes;  // rows folded together (16)

JF_DEV void cp_async16(uint32_t dst, const void* src, bool valid) {
  const int n = valid ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
JF_DEV void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
JF_DEV void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

JF_DEV uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);  // one cvt.rn.bf16x2.f32
  return *reinterpret_cast<const uint32_t*>(&v);
}

JF_DEV uint32_t pack_f16(float lo, float hi) {
  const __half2 v = __floats2half2_rn(lo, hi);  // one cvt.rn.f16x2.f32
  return *reinterpret_cast<const uint32_t*>(&v);
}

// 2^x by the MUFU ex2 instruction (flushes results below 2^-126 to zero; 2^-inf = 0).
JF_DEV float ex2_ftz(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Fold of two softmax states (m, l, O) in the log2 domain: m = max(ma, mb),
// O = 2^(ma-m) Oa + 2^(mb-m) Ob, l likewise; an empty state has m = -inf and weight 0.
JF_DEV void fold_weights(float ma, float mb, float& wa, float& wb, float& m) {
  m = fmaxf(ma, mb);
  wa = (ma == -INFINITY) ? 0.f : exp2f(ma - m);
  wb = (mb == -INFINITY) ? 0.f : exp2f(mb - m);
}
// wa a + wb b, rounded the same way wherever it is compiled (every form folds to the same bits).
JF_DEV float fold_value(float wa, float a, float wb, float b) { return __fmaf_rn(wa, a, __fmul_rn(wb, b)); }

// Unit ui of the forward (chains in order, then KV heads, then query tiles), looked up
// by warp 0 into s_unit; s_unit.pad stays 0 past the last unit. Every CTA of cluster ui gets the
// same unit. The chain table was written by a kernel or graph launch that was complete
// before this forward's first kernel (k_embed, no programmatic launch) began, so this runs before the
// dependency wait.
JF_DEV void resolve_unit(const AttnParams& a, int ui, int j, int n_units, int G, int warp, int lane, AttnUnit& s_unit) {
  if (threadIdx.x == 0) s_unit.pad = 0;
  __syncthreads();
  if (warp == 0) {
    const int n_ch = *a.n_chains_dev;
    const int tile = attn_tile_rows(G);
    int base = 0;
    for (int c0 = 0; c0 < n_ch; c0 += 32) {
      const int c = c0 + lane;
      Chain ch = {0, 0, 0, 0};
      int nqt = 0;
      if (c < n_ch) {
        ch = a.chains[c];
        nqt = (ch.nrows * G + tile - 1) / tile;
      }
      const int nu = a.Hkv * nqt;
      int incl = nu;
#pragma unroll
      for (int sh = 1; sh < 32; sh <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, sh);
        if (lane >= sh) incl += v;
      }
      const int first = base + incl - nu;
      if (nu > 0 && ui >= first && ui < base + incl) {
        const int k = ui - first, kvh = k / nqt, qt = k % nqt;
        int qrows = ch.nrows * G - qt * tile;
        if (qrows > tile) qrows = tile;
        const int nch = (ch.pos0 + (qt * tile + qrows - 1) / G) / kAttnChunk + 1;
        if (nch > kAttnLanes * kAttnLaneChunks) {
          if (j == 0) jf_set_error(a.err, JF_DERR_BOUNDS);
        } else {
          s_unit = AttnUnit{ch.seq, ch.row0, ch.nrows, ch.pos0, kvh, qt, nch, 1};
        }
      }
      base += __shfl_sync(0xffffffffu, incl, 31);
    }
    // the launch must cover every unit
    if (lane == 0 && j == 0 && ui == n_units - 1 && base > ui + 1)
      jf_set_error(a.err, JF_DERR_BOUNDS);
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------------------------
// Warp roles of a CTA: warps 0-7 take the softmax steps (warp w: query rows 32(w%4).., key columns
// 64(w/4)..+63 of a chunk), warp 8 issues the tensor-core MMAs, warp 9 loads K, warp 10 V. Per 128-key
// chunk t: S = Q K^T (M = 128 query rows, N = 128 keys, K = 128) into one of two TMEM buffers while
// the softmax of the chunks before it runs; the softmax warps read S out of TMEM, write P in fp16 to
// one of two TMEM buffers (the A operand of the second MMA) and P V accumulates into O, which stays in
// TMEM for
// the whole lane. Q, K and V sit in 64-column atoms of 8 rows with the 128-byte swizzle, Q as two
// 128-row column blocks, K and V in the pages' own layout (kv_page_offset), so that a page is one
// contiguous copy: Q and K are read K-major, V (fp16 in the cache: the QKV finish stores the
// bf16-rounded values as fp16) MN-major as it arrives, dims along N. Q K^T runs on bf16 operands, P V on fp16 ones
// (both operands of one MMA share their type).
// ---------------------------------------------------------------------------------------------
constexpr int SOFTMAX_THREADS = 256;
constexpr int ATT_THREADS = SOFTMAX_THREADS + 3 * 32;
constexpr int TC_BLK = 16384;                     // one 128-row x 64-column 16-bit operand block
constexpr int TC_OPND = 2 * TC_BLK;               // 128 rows x 128 columns
constexpr int K_STAGES = 3, V_STAGES = 2;         // V_STAGES: one per parity of the step
constexpr int TC_OFF_K = TC_OPND, TC_OFF_V = TC_OFF_K + K_STAGES * TC_OPND;  // after Q
constexpr int TC_SMEM = TC_OFF_V + V_STAGES * TC_OPND + 1024;                // + slack for 1024-byte alignment
constexpr int TM_S = 0, TM_P = 256, TM_O = 384;   // TMEM columns: S 2 x 128, P 2 x 64 (fp16 pairs), O 128
constexpr int TC_TMEM_COLS = 512;
constexpr int PAGES_PER_CHUNK = kAttnChunk / kPage, PAGE_BYTES = kPage * HD * 2;
// A row's reference maximum follows its scores only when they exceed it by more than this (log2
// units): until then its probabilities are at most 2^8, which fp16 holds with the same 11 bits, and
// O needs no rescaling.
constexpr float RESCALE_LAG = 8.0f;

// byte offset of 16-byte chunk c16 (0..15) of row r of Q (two 128-row column blocks)
JF_DEV uint32_t tc_swz(int r, int c16) {
  return (uint32_t)((c16 >> 3) * TC_BLK + r * 128 + (((c16 & 7) ^ (r & 7)) << 4));
}

// The steps of one CTA: the chunks of its lanes j, j + n_ctas, ..., lane after lane.
struct Cursor {
  int ln, chunk;
  JF_DEV void advance(int n_chunks, int n_ctas) {
    chunk += kAttnLanes;
    if (chunk >= n_chunks) {
      ln += n_ctas;
      chunk = ln;
    }
  }
  JF_DEV bool first() const { return chunk < kAttnLanes; }  // of its lane
};

// The loads of one operand (K or V) of every step of a CTA, by one warp, up to n_stages chunks ahead: a
// chunk's cached pages are contiguous copies from the page pool (lane l: page l, its id read one chunk
// ahead); a page of in-flight keys is four TMA boxes from the in-flight rows; the pages that hold the
// last cached and the first in-flight key or end past the tile's last key (at most two of a unit) are
// copied row by row, with zeros past the last key; pages wholly past it are not read by anyone. Cached
// pages of the first chunks are requested before the dependency wait. full[s] completes when stage s
// is loaded; freed[s] when its MMAs are done. Returns false when a wait gave up. (Loops are kept rolled:
// between two layers' weights the kernel's code is often fetched again from memory.)
JF_DEV bool load_steps(const AttnParams& a, const AttnUnit& u, int j, int n_ctas, int n_steps, int max_kp,
                       const CUtensorMap* tm_inf, const uint16_t* pages, const uint16_t* inflight, uint32_t stages,
                       int n_stages, uint64_t* full, uint64_t* freed) {
  const int lane = threadIdx.x & 31;
  const int* page_row = a.page_table + (size_t)u.seq * a.pages_per_seq;
  auto page_of = [&](int id) { return pages + ((size_t)id * a.Hkv + u.kvh) * (kPage * HD); };
  auto page_id = [&](int chunk) {  // of this lane's page; -1: no cached keys in it
    const int kp = chunk * kAttnChunk + lane * kPage;
    if (lane >= PAGES_PER_CHUNK || kp >= u.pos0) return -1;
    const int id = page_row[kp / kPage];
    if (id >= 0 && id < a.n_pages) return id;
    jf_set_error(a.err, JF_DERR_BOUNDS);
    return 0;
  };
  auto cached_page = [&](int chunk) {
    return lane < PAGES_PER_CHUNK && chunk * kAttnChunk + lane * kPage + kPage <= u.pos0;
  };
  auto copy_cached = [&](int chunk, int id, int stage) {
    if (cached_page(chunk))
      bulk_load(stages + (uint32_t)(stage * TC_OPND + lane * PAGE_BYTES), page_of(id), PAGE_BYTES, smem_u32(&full[stage]));
  };
  Cursor c{j, j};
#pragma unroll 1
  for (int t = 0; t < n_stages && t < n_steps; ++t, c.advance(u.n_chunks, n_ctas))
    copy_cached(c.chunk, page_id(c.chunk), t);
  c = Cursor{j, j};
  int id_next = n_steps > 0 ? page_id(c.chunk) : -1, stage = 0;
  uint32_t parity = 1u;  // of the stage's previous use
  bool done = true;
  pdl_wait();  // in-flight keys come from the QKV projection
#pragma unroll 1
  for (int t = 0; t < n_steps; ++t) {
    const int chunk = c.chunk, id = id_next, kp0 = chunk * kAttnChunk;
    c.advance(u.n_chunks, n_ctas);
    if (t + 1 < n_steps) id_next = page_id(c.chunk);
    if (t >= n_stages) {
      const bool ok = mbar_wait_bounded(smem_u32(&freed[stage]), parity, a.wait_ns);
      if (!__all_sync(0xffffffffu, ok)) {
        n_steps = t;
        done = false;
        break;
      }
      copy_cached(chunk, id, stage);
    }
    const uint32_t dst = stages + (uint32_t)(stage * TC_OPND), bar = smem_u32(&full[stage]);
    uint32_t bytes = cached_page(chunk) ? PAGE_BYTES : 0u;
    if (kp0 + kAttnChunk > u.pos0) {
      const int kp = kp0 + (lane >> 2) * kPage;  // lane: quarter lane % 4 of page lane / 4
      if (kp >= u.pos0 && kp + kPage - 1 <= max_kp) {
        tma_load_3d_plain(dst + lane * (PAGE_BYTES / 4), tm_inf, bar, (lane & 1) * 64, u.kvh,
                          u.row0 + kp - u.pos0 + ((lane >> 1) & 1) * 8);
        bytes += PAGE_BYTES / 4;
      }
      __syncwarp();
      bool rows = false;
#pragma unroll 1
      for (int pg = 0; pg < PAGES_PER_CHUNK; ++pg) {
        const int kp1 = kp0 + pg * kPage;
        if (kp1 + kPage <= u.pos0 || kp1 > max_kp || (kp1 >= u.pos0 && kp1 + kPage - 1 <= max_kp)) continue;
        rows = true;
        const int page = __shfl_sync(0xffffffffu, id, pg);
#pragma unroll
        for (int k = 0; k < kPage / 2; ++k) {
          const int r = 2 * k + (lane >> 4), piece = lane & 15, key = kp1 + r;
          const uint16_t* src = nullptr;
          if (key < u.pos0) src = page_of(page) + kv_page_offset(r, piece) / 2;
          else if (key <= max_kp) src = inflight + ((size_t)(u.row0 + key - u.pos0) * a.Hkv + u.kvh) * HD + piece * 8;
          cp_async16(dst + pg * PAGE_BYTES + kv_page_offset(r, piece), src ? src : pages, src != nullptr);
        }
      }
      if (rows) {
        cp_async_commit();
        cp_async_wait<0>();
        fence_proxy_async_smem();  // this thread's cp.async writes -> tensor-core operand reads
        __syncwarp();              // every lane's, before lane 0's arrival
      }
    }
    const uint32_t total = __reduce_add_sync(0xffffffffu, bytes);
    if (lane == 0) mbar_arrive_expect_tx(bar, total);
    if (++stage == n_stages) {
      stage = 0;
      parity ^= 1u;
    }
  }
  // every copy has landed before the CTA may leave, also after a wait that gave up
  for (int t = n_steps > n_stages ? n_steps - n_stages : 0; t < n_steps; ++t)
    if (!mbar_wait_bounded(smem_u32(&full[t % n_stages]), (uint32_t)(t / n_stages) & 1u, a.wait_ns)) break;
  return done;
}

// Fold of rows rb*16 .. rb*16+15 of unit ui over its 8 lane states in lane order (thread: row
// tid % 16, dims 8 (tid / 16) ..), normalised and stored in bf16. The same arithmetic whichever CTA
// of the unit runs it.
JF_DEV void fold_row_block(const AttnParams& a, const AttnUnit& u, int ui, int rb, int qr0, int qrows, int G, int tid) {
  const int lr = tid & 15, rw = rb * ROWS_PER_BLOCK + lr;
  const int d = (tid >> 4) * 8;
  if (rw >= qrows) return;
  const float* x0 = a.xchg + (size_t)ui * kAttnLanes * kAttnXchgFloats;
  const int n_lanes = u.n_chunks < kAttnLanes ? u.n_chunks : kAttnLanes;  // the others are empty
  float ov[kAttnLanes][8], mv[kAttnLanes], lv[kAttnLanes];
#pragma unroll
  for (int q = 0; q < kAttnLanes; ++q) {
    if (q >= n_lanes) break;
    const float* xq = x0 + (size_t)q * kAttnXchgFloats;
#pragma unroll
    for (int e = 0; e < 8; e += 4) {
      const float4 v = __ldcg(reinterpret_cast<const float4*>(xq) + ((d + e) >> 2) * kAttnQRows + rw);
      ov[q][e] = v.x;
      ov[q][e + 1] = v.y;
      ov[q][e + 2] = v.z;
      ov[q][e + 3] = v.w;
    }
    mv[q] = __ldcg(xq + HD * kAttnQRows + rw);
    lv[q] = __ldcg(xq + HD * kAttnQRows + kAttnQRows + rw);
  }
  float M = mv[0], L = lv[0];
  float acc[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) acc[e] = ov[0][e];
#pragma unroll
  for (int q = 1; q < kAttnLanes; ++q) {
    if (q >= n_lanes) break;
    float wa, wb, mm;
    fold_weights(M, mv[q], wa, wb, mm);
    M = mm;
    L = fold_value(wa, L, wb, lv[q]);
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = fold_value(wa, acc[e], wb, ov[q][e]);
  }
  const float il = L > 0.f ? 1.f / L : 0.f;
  const int qr = qr0 + rw, tq = qr / G, g = qr % G;
  bf16* dst = reinterpret_cast<bf16*>(a.out) + ((size_t)(u.row0 + tq) * a.Hq + u.kvh * G + g) * HD + d;
  *reinterpret_cast<uint4*>(dst) = make_uint4(pack_bf16(acc[0] * il, acc[1] * il), pack_bf16(acc[2] * il, acc[3] * il),
                                              pack_bf16(acc[4] * il, acc[5] * il), pack_bf16(acc[6] * il, acc[7] * il));
}

// A unit's key lanes are spread over `n_ctas` CTAs (1, 2, 4 or 8): CTA j walks lanes j, j + n_ctas, ...
// one after the other, each with its own softmax state. kWhole (n_ctas = 1): the CTA folds each
// finished lane into a running state in registers. Otherwise the CTAs of a unit are one cluster:
// each writes its lanes' states to the unit's scratch slots and, after a cluster barrier, folds
// 128 / n_ctas of the rows. Every form computes the same lane states and folds them in lane order,
// so their results are bit-identical.
//
// What bounds it: a 128-key chunk takes about 2000 cycles of a CTA (ncu, 32,768 keys: the tensor pipe is busy
// for 1020 of them, ex2 and the issue slots for 21% and 41%), the chain of the softmax warps (scores out of
// tensor memory, the row maxima's barrier, 64 exponentials a thread, P back). With every warp
// loading K/V by cp.async, waiting for each MMA and adding P V in registers a chunk took 4900 (30% of
// it the copies' issue). One 7B layer at P = 32768: 32 rows 204 -> 147 us, 128 rows 330 -> 198 us; 512
// rows at 4096: 398 -> 309 us. Long units are bound by the chunk step. At decode sizes (P = 1024, 32
// rows: 9.2 us of attention a layer, as before) the prologue and the fold dominate: lane states pass through
// L2 in 16-byte pieces ([dim / 4][row][4]; one value a store took 1 us more), and the code is kept small
// (unrolled loaders made a first pass over a layer 4 us slower).
template <bool kWhole>
__global__ void __launch_bounds__(ATT_THREADS, 1)
    k_attn_tc(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_ki,
              const __grid_constant__ CUtensorMap tm_vi, const AttnParams a, int n_ctas) {
  extern __shared__ uint8_t sm_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(sm_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sQ = smem_u32(sm), sK = smem_u32(sm + TC_OFF_K), sV = smem_u32(sm + TC_OFF_V);
  // per K stage: loaded / read; per V stage: loaded; per parity of the step: S ready, P ready, P V done
  // (which also frees the V stage); Q loaded; all MMAs done
  __shared__ __align__(8) uint64_t b_kfull[K_STAGES], b_kfree[K_STAGES], b_vfull[V_STAGES], b_s[2], b_p[2], b_o[2], b_q, b_all;
  __shared__ uint32_t tmem_slot;
  __shared__ AttnUnit s_unit;
  __shared__ float red_max[2][2][kAttnQRows];  // [step parity][column half][row]
  __shared__ float red_l[2][2][kAttnQRows];

  JF_TL_ENTRY();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if constexpr (kWhole) n_ctas = 1;
  const int j = (int)(blockIdx.x % n_ctas);  // = rank in the cluster
  const int ui = (int)(blockIdx.x / n_ctas);
  const int G = a.Hq / a.Hkv;
  const bool by_token = G <= kAttnQRows;  // the tile holds whole tokens: Q arrives by TMA
  pdl_launch_dependents();  // the next kernel may launch now
  if (tid == 0) {
    for (int i = 0; i < K_STAGES; ++i) {
      mbar_init(smem_u32(&b_kfull[i]), 1);
      mbar_init(smem_u32(&b_kfree[i]), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&b_vfull[i]), 1);
      mbar_init(smem_u32(&b_s[i]), 1);
      mbar_init(smem_u32(&b_p[i]), SOFTMAX_THREADS / 32);
      mbar_init(smem_u32(&b_o[i]), 1);
    }
    mbar_init(smem_u32(&b_all), 1);
    mbar_init(smem_u32(&b_q), by_token ? 1 : SOFTMAX_THREADS / 32);
    fence_mbar_init();
  }
  resolve_unit(a, ui, j, (int)(gridDim.x / n_ctas), G, warp, lane, s_unit);
  const AttnUnit u = s_unit;
  if (!u.pad) return;  // past the last unit: the whole unit (cluster) leaves together
  if (warp == 8) {
    tmem_alloc(smem_u32(&tmem_slot), TC_TMEM_COLS);
    tmem_relinquish();
  }
  const int tile = attn_tile_rows(G), qr0 = u.qt * tile;
  int qrows = u.nrows * G - qr0;
  if (qrows > tile) qrows = tile;
  const int max_kp = u.pos0 + (qr0 + qrows - 1) / G;
  auto lane_chunks = [&](int ln) { return u.n_chunks > ln ? (u.n_chunks - 1 - ln) / kAttnLanes + 1 : 0; };
  int n_steps = 0;
  for (int ln = j; ln < kAttnLanes; ln += n_ctas) n_steps += lane_chunks(ln);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  bool ok = true;

  if (warp > 8) {
    // ---- loads
    const bool k = warp == 9;
    const bool done = load_steps(a, u, j, n_ctas, n_steps, max_kp, k ? &tm_ki : &tm_vi,
                                 reinterpret_cast<const uint16_t*>(k ? a.k_pages : a.v_pages),
                                 reinterpret_cast<const uint16_t*>(k ? a.k_inf : a.v_inf), k ? sK : sV,
                                 k ? K_STAGES : V_STAGES, k ? b_kfull : b_vfull, k ? b_kfree : b_o);
    if (!done && lane == 0) jf_set_error(a.err, JF_DERR_TIMEOUT_MMA);
  } else if (warp == 8) {
    // ---- MMAs: once the softmax of step t has left its S buffer, P V of step t and S of step t+2 go in
    // together, after every wait they need (a wait behind issued MMAs takes as long as they queue). The
    // whole warp walks the steps, one elected lane issues; the operand descriptors are a base plus
    // constants (16-byte units), which keeps the issue of a chunk's MMAs shorter than they run.
    if (lane == 0) tma_prefetch_desc(&tm_q);
    pdl_wait();  // queries come from the QKV projection
    if (by_token && n_steps > 0 && elect_one()) {
      // rows (token, head of the group) of whole tokens, two 64-dim halves; rows past the tile's last
      // token are never stored
      const uint32_t bar = smem_u32(&b_q);
      mbar_arrive_expect_tx(bar, (uint32_t)(tile * HD * 2));
      tma_load_3d_plain(sQ, &tm_q, bar, 0, u.kvh * G, u.row0 + qr0 / G);
      tma_load_3d_plain(sQ + TC_BLK, &tm_q, bar, 64, u.kvh * G, u.row0 + qr0 / G);
    }
    __syncwarp();
    constexpr uint32_t idesc = idesc_bf16_f32(128, 128);
    constexpr uint32_t idesc_pv = idesc_f16_f32(128, 128) | (1u << 16);  // fp16 P, fp16 V MN-major
    const uint64_t dq = sdesc_k_sw128(sQ), dk = sdesc_k_sw128(sK, 2048u), dv = sdesc_mn_sw128(sV, 1024u, 2048u);
    const uint32_t tm_s = tmem + TM_S, tm_p = tmem + TM_P, tm_o = tmem + TM_O;
    auto issue_s = [&](int t, int stage) {  // by one lane
      const uint64_t dks = dk + (uint64_t)(stage * (TC_OPND >> 4));
      const uint32_t d = tm_s + (t & 1) * 128;
#pragma unroll
      for (int kk = 0; kk < 8; ++kk)
        tc_mma_bf16(d, dq + (uint64_t)((kk >> 2) * (TC_BLK >> 4) + (kk & 3) * 2),
                    dks + (uint64_t)((kk >> 2) * 64 + (kk & 3) * 2), idesc, kk > 0 ? 1u : 0u);
      tc_commit(smem_u32(&b_s[t & 1]));
      tc_commit(smem_u32(&b_kfree[stage]));
    };
    if (n_steps > 0) {
      ok = __all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(&b_q), 0u, a.wait_ns));
      Cursor c{j, j};
      int stage = 0;  // K stage and phase of step t+2
      uint32_t parity = 0;
      for (int t = -2; t < n_steps && ok; ++t) {
        const bool next = t + 2 < n_steps;
        if (next) ok = mbar_wait_bounded(smem_u32(&b_kfull[stage]), parity, a.wait_ns);
        if (t >= 0)
          ok = ok && mbar_wait_bounded(smem_u32(&b_vfull[t & 1]), (uint32_t)(t >> 1) & 1u, a.wait_ns) &&
               mbar_wait_bounded(smem_u32(&b_p[t & 1]), (uint32_t)(t >> 1) & 1u, a.wait_ns);
        if (!__all_sync(0xffffffffu, ok)) {
          ok = false;
          break;
        }
        tc_fence_after();
        if (t >= 0) {
          const uint64_t dvs = dv + (uint64_t)((t & 1) * (TC_OPND >> 4));
          const uint32_t ap = tm_p + (t & 1) * 64;
          const uint32_t acc = c.first() ? 0u : 1u;
          const int groups = (max_kp - c.chunk * kAttnChunk) / 16;  // 16-key groups with a key the tile sees, less one
          if (elect_one()) {
            // keys 16kk .. 16kk+15: 8 packed P columns, one page of V (its two 64-dim atoms 1024 bytes, its
            // two 8-key groups 2048 bytes apart)
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
              if (kk <= groups)
                tc_mma_f16_ts(tm_o, ap + kk * 8, dvs + (uint64_t)(kk * (PAGE_BYTES >> 4)), idesc_pv, kk > 0 ? 1u : acc);
            tc_commit(smem_u32(&b_o[t & 1]));
          }
          __syncwarp();
          c.advance(u.n_chunks, n_ctas);
        }
        if (next) {
          // (its completion also tells the softmax that P V of step t has read its P buffer)
          if (elect_one()) issue_s(t + 2, stage);
          __syncwarp();
          if (++stage == K_STAGES) {
            stage = 0;
            parity ^= 1u;
          }
        }
      }
      if (!ok && lane == 0) jf_set_error(a.err, JF_DERR_TIMEOUT_MMA);
      // Q has landed and every MMA is complete before the CTA may leave, also after a wait that gave up
      if (elect_one()) tc_commit(smem_u32(&b_all));
      __syncwarp();
      mbar_wait_bounded(smem_u32(&b_q), 0u, a.wait_ns);
      mbar_wait_bounded(smem_u32(&b_all), 0u, a.wait_ns);
    }
    __syncwarp();
  } else {
    // ---- softmax
    pdl_wait();
    JF_TL_WAITED();
    if (!by_token && n_steps > 0) {
      const bf16* Q = reinterpret_cast<const bf16*>(a.q);
      for (int i = tid; i < kAttnQRows * 16; i += SOFTMAX_THREADS) {
        const int r = i >> 4, c = i & 15;
        const bool in = r < qrows;
        const int qr = qr0 + (in ? r : 0);
        const int t = qr / G, g = qr % G;
        cp_async16(sQ + tc_swz(r, c), Q + ((size_t)(u.row0 + t) * a.Hq + u.kvh * G + g) * HD + c * 8, in);
      }
      cp_async_commit();
      cp_async_wait<0>();
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&b_q));
    }
    const int quad = warp & 3, half = warp >> 2;
    const int r = quad * 32 + lane;  // this thread's query row (TMEM lane)
    const bool live = quad * 32 < qrows;  // the warp holds rows of the tile
    const int pos_r = r < qrows ? u.pos0 + (qr0 + r) / G : -1;
    const int pos_first = u.pos0 + qr0 / G;  // the tile's first row sees the fewest keys
    const uint32_t t_row = tmem + ((uint32_t)(quad * 32) << 16);
    const uint32_t t_o = t_row + TM_O + 64 * half;
    const float scale = a.scale_log2;
    float m_ref = -INFINITY, l_run = 0.f;
    float acc[kWhole ? 64 : 1], M_all = -INFINITY, L_all = 0.f;  // running fold of the finished lanes

    // A finished lane (its last step was t_end, its maximum m): kWhole folds it into the running
    // state, otherwise its state (O, m, l over both column halves) goes to its scratch slot of the
    // unit, O stored as [dim / 4][row][4] (a warp writes 512 contiguous bytes for 4 dimensions).
    auto finish_lane = [&](int ln, int t_end, float m) {
      if (!mbar_wait_bounded(smem_u32(&b_o[t_end & 1]), (uint32_t)(t_end >> 1) & 1u, a.wait_ns)) {
        jf_set_error(a.err, JF_DERR_TIMEOUT_MMA);
        ok = false;
      }
      tc_fence_after();
      if (!live) return;
      const float l = red_l[t_end & 1][0][r] + red_l[t_end & 1][1][r];
      if constexpr (kWhole) {
        float wa = 0.f, wb = 1.f, mm = m;
        if (ln > 0) fold_weights(M_all, m, wa, wb, mm);
        M_all = mm;
        L_all = ln > 0 ? fold_value(wa, L_all, wb, l) : l;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float t32[32];
          tmem_ld32(t_o + 32 * h, t32);
#pragma unroll
          for (int i = 0; i < 32; ++i)
            acc[32 * h + i] = ln > 0 ? fold_value(wa, acc[32 * h + i], wb, t32[i]) : t32[i];
        }
      } else {
        float* xs = a.xchg + ((size_t)ui * kAttnLanes + ln) * kAttnXchgFloats;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float t32[32];
          tmem_ld32(t_o + 32 * h, t32);
          if (r < qrows) {
#pragma unroll
            for (int i = 0; i < 32; i += 4)
              reinterpret_cast<float4*>(xs)[((64 * half + 32 * h + i) >> 2) * kAttnQRows + r] =
                  make_float4(t32[i], t32[i + 1], t32[i + 2], t32[i + 3]);
          }
        }
        if (half == 0 && r < qrows) {
          xs[HD * kAttnQRows + r] = m;
          xs[HD * kAttnQRows + kAttnQRows + r] = l;
        }
      }
    };

    Cursor c{j, j};
    int ln = j;  // lane of the previous step
    for (int t = 0; t <= n_steps; ++t) {
      const bool step = t < n_steps;  // after the last step only the last lane is finished
      if (step && !mbar_wait_bounded(smem_u32(&b_s[t & 1]), (uint32_t)(t >> 1) & 1u, a.wait_ns)) {
        jf_set_error(a.err, JF_DERR_TIMEOUT_MMA);
        ok = false;
      }
      tc_fence_after();
      const bool first = !step || c.first();
      const float m_prev = m_ref;  // of the lane that the previous step finished, if it did
      if (first) {
        m_ref = -INFINITY;
        l_run = 0.f;
      }
      // scores of this row, keys 64*half .. 64*half+63 of the chunk; keys past the row's own position are
      // masked. The scale (> 0) goes into the maximum and into one fma per exponential:
      // p = 2^(s * scale - m). kWhole reads them a second time for the exponentials: its running fold
      // takes the registers that would keep them.
      const bool busy = live && step;
      const uint32_t t_s = t_row + TM_S + (t & 1) * 128 + 64 * half;
      const bool masked = c.chunk * kAttnChunk + kAttnChunk - 1 > pos_first;  // for some row
      const int n_seen = pos_r + 1 - (c.chunk * kAttnChunk + 64 * half);       // keys of these 64 the row sees
      auto scores = [&](int h, float (&v)[32]) {
        tmem_ld32(t_s + 32 * h, v);
        if (masked) {
#pragma unroll
          for (int i = 0; i < 32; ++i) v[i] = (32 * h + i < n_seen) ? v[i] : -INFINITY;
        }
      };
      float sv[kWhole ? 1 : 2][32];
      if (busy) {
        float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float(&v)[32] = sv[kWhole ? 0 : h];
          scores(h, v);
#pragma unroll
          for (int i = 0; i < 32; ++i) mx[i & 3] = fmaxf(mx[i & 3], v[i]);
        }
        red_max[t & 1][half][r] = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * scale;
      }
      ok = sync_and<1, SOFTMAX_THREADS>(ok);  // (barrier 0 is __syncthreads)
      if (!ok) break;
      bool raise = false;
      float mc = -INFINITY;
      if (busy) {
        mc = fmaxf(red_max[t & 1][0][r], red_max[t & 1][1][r]);
        raise = mc > m_ref + RESCALE_LAG;  // (also from -inf)
      }
      if (!first && __any_sync(0xffffffffu, raise)) {
        // the same for both column halves of the warp's rows; alpha = 1 leaves a row as it is
        if (!mbar_wait_bounded(smem_u32(&b_o[(t - 1) & 1]), (uint32_t)((t - 1) >> 1) & 1u, a.wait_ns)) {
          jf_set_error(a.err, JF_DERR_TIMEOUT_MMA);
          ok = false;
        }
        tc_fence_after();
        const float al = raise ? (m_ref == -INFINITY ? 0.f : ex2_ftz(m_ref - mc)) : 1.f;
        l_run *= al;
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          float t16[16];
          uint32_t w[16];
          tmem_ld16(t_o + 16 * h, t16);
#pragma unroll
          for (int i = 0; i < 16; ++i) w[i] = __float_as_uint(t16[i] * al);
          tmem_st16(t_o + 16 * h, w);
        }
      }
      if (raise) m_ref = mc;
      if (busy) {
        const float nb = (m_ref == -INFINITY) ? 0.f : -m_ref;
        // P in fp16: fp16 keeps 11 significant bits of P, where bf16's 8 would move the attention
        // output by up to half a bf16 unit, as much as its own rounding. The row sum in four
        // independent partial sums, added in a fixed order.
        float ls[4] = {0.f, 0.f, 0.f, 0.f};
        const uint32_t t_p = t_row + TM_P + (t & 1) * 64 + 32 * half;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t w[16];
          float(&v)[32] = sv[kWhole ? 0 : h];
          if constexpr (kWhole) scores(h, v);
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float p0 = ex2_ftz(fmaf(v[2 * i], scale, nb));
            const float p1 = ex2_ftz(fmaf(v[2 * i + 1], scale, nb));
            ls[(2 * i) & 3] += p0;
            ls[(2 * i + 1) & 3] += p1;
            w[i] = pack_f16(p0, p1);
          }
          tmem_st16(t_p + 16 * h, w);
        }
        l_run += (ls[0] + ls[1]) + (ls[2] + ls[3]);
        red_l[t & 1][half][r] = l_run;
        tmem_wait_st();
      }
      // a finished lane's state leaves before this step's P V overwrites O
      if (first && t > 0) finish_lane(ln, t - 1, m_prev);
      if (!step) break;
      ln = c.ln;
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&b_p[t & 1]));
      c.advance(u.n_chunks, n_ctas);
    }
    if constexpr (kWhole) {
      if (ok && r < qrows) {
        const float il = L_all > 0.f ? 1.f / L_all : 0.f;
        const int qr = qr0 + r, tq = qr / G, g = qr % G;
        bf16* dst = reinterpret_cast<bf16*>(a.out) + ((size_t)(u.row0 + tq) * a.Hq + u.kvh * G + g) * HD + 64 * half;
#pragma unroll
        for (int e = 0; e < 64; e += 8)
          *reinterpret_cast<uint4*>(dst + e) =
              make_uint4(pack_bf16(acc[e] * il, acc[e + 1] * il), pack_bf16(acc[e + 2] * il, acc[e + 3] * il),
                         pack_bf16(acc[e + 4] * il, acc[e + 5] * il), pack_bf16(acc[e + 6] * il, acc[e + 7] * il));
      }
    }
  }
  if constexpr (!kWhole) {
    __syncwarp();
    cluster_sync();  // release / acquire: every lane's state of the unit is visible
    if (ok && warp < 8) {
      const int blocks = kAttnLanes / n_ctas;
      for (int rb = j * blocks; rb < (j + 1) * blocks; ++rb) fold_row_block(a, u, ui, rb, qr0, qrows, G, tid);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 8) tmem_dealloc(tmem, TC_TMEM_COLS);
  JF_TL_EXIT(TL_ATTN);
}

// fp32 path: one CTA per (row, query head); warp w takes the absolute 32-key groups w, w + 4, ... in
// increasing order, and the four states are folded in warp order, so a row's result does not depend on
// the other rows. Latency bounds it (small models, short contexts): a lane has its whole key row in
// flight at once (four partial dot products), and value rows are loaded 64 registers at a time before
// their sums. Against one warp per (row, head) on every group, two layers and the head: iteration of 32
// rows at 1,000 tokens 354 -> 196 us, at 3,000 854 -> 363 us, one row at 3,000 721 -> 240 us (heads of 64
// dims; 411 -> 280, 979 -> 592 and 928 -> 486 us for 128); error against 64 bits at 3,000 tokens 1.7e-6
// -> 1.1e-6, at 33 and 200 the same within a tenth.
constexpr int F32_WARPS = 4;
template <int HDT>
__global__ void __launch_bounds__(32 * F32_WARPS) k_attn_f32(const AttnParams a) {
  constexpr int NV = HDT / 32;  // dims per lane of the output
  constexpr int VB = 64 / NV;   // value rows in flight (64 registers)
  __shared__ float4 s_q[HDT / 4];
  __shared__ float s_o[F32_WARPS][HDT], s_m[F32_WARPS], s_l[F32_WARPS];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = blockIdx.x / a.Hq, h = blockIdx.x % a.Hq;
  pdl_launch_dependents();
  pdl_wait();
  const int kvh = h / (a.Hq / a.Hkv);
  const int n_ch = *a.n_chains_dev;
  int ci = 0;
  for (; ci < n_ch; ++ci) {
    const Chain c = a.chains[ci];
    if (r >= c.row0 && r < c.row0 + c.nrows) break;
  }
  if (ci == n_ch) return;
  const Chain ch = a.chains[ci];
  const int pos = ch.pos0 + (r - ch.row0);
  const float4* q = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(a.q) + ((size_t)r * a.Hq + h) * HDT);
  if (threadIdx.x < HDT / 4) s_q[threadIdx.x] = q[threadIdx.x];
  __syncthreads();
  const float* Kp = reinterpret_cast<const float*>(a.k_pages);
  const float* Vp = reinterpret_cast<const float*>(a.v_pages);
  const float* Ki = reinterpret_cast<const float*>(a.k_inf);
  const float* Vi = reinterpret_cast<const float*>(a.v_inf);
  const float scale = a.scale_log2;
  float m = -INFINITY, l = 0.f, o[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) o[i] = 0.f;
  for (int kb = 32 * warp; kb <= pos; kb += 32 * F32_WARPS) {
    const int kp = kb + lane;
    float s = -INFINITY;
    unsigned long long v_row = 0;  // this lane's key's value row
    if (kp <= pos) {
      size_t off;
      if (kp < ch.pos0) {
        const int page = a.page_table[(size_t)ch.seq * a.pages_per_seq + (kp >> 4)];
        off = (((size_t)page * a.Hkv + kvh) * kPage + (kp & 15)) * HDT;
      } else {
        off = ((size_t)(ch.row0 + kp - ch.pos0) * a.Hkv + kvh) * HDT;
      }
      const float4* kr = reinterpret_cast<const float4*>((kp < ch.pos0 ? Kp : Ki) + off);
      v_row = reinterpret_cast<unsigned long long>((kp < ch.pos0 ? Vp : Vi) + off);
      float d[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int i0 = 0; i0 < HDT / 4; i0 += 16) {
        float4 kv[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) kv[i] = kr[i0 + i];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float4 x = s_q[i0 + i];
          d[0] = fmaf(x.x, kv[i].x, d[0]);
          d[1] = fmaf(x.y, kv[i].y, d[1]);
          d[2] = fmaf(x.z, kv[i].z, d[2]);
          d[3] = fmaf(x.w, kv[i].w, d[3]);
        }
      }
      s = ((d[0] + d[1]) + (d[2] + d[3])) * scale;
    }
    float mx = s;
#pragma unroll
    for (int sh = 16; sh > 0; sh >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, sh));
    const float mn = fmaxf(m, mx);
    const float al = (m == -INFINITY) ? 0.f : exp2f(m - mn);
    const float p = (s == -INFINITY) ? 0.f : exp2f(s - mn);
    l = l * al + warp_sum(p);
#pragma unroll
    for (int i = 0; i < NV; ++i) o[i] *= al;
#pragma unroll 1
    for (int j0 = 0; j0 < 32 && kb + j0 <= pos; j0 += VB) {
      float v[VB][NV];
#pragma unroll
      for (int j = 0; j < VB; ++j) {
        const float* vr = reinterpret_cast<const float*>(__shfl_sync(0xffffffffu, v_row, j0 + j));
#pragma unroll
        for (int i = 0; i < NV; ++i) v[j][i] = (kb + j0 + j <= pos) ? vr[lane + 32 * i] : 0.f;
      }
#pragma unroll
      for (int j = 0; j < VB; ++j) {
        const float pj = __shfl_sync(0xffffffffu, p, j0 + j);
        if (kb + j0 + j <= pos) {
#pragma unroll
          for (int i = 0; i < NV; ++i) o[i] = fmaf(pj, v[j][i], o[i]);
        }
      }
    }
    m = mn;
  }
  if (lane == 0) {
    s_m[warp] = m;
    s_l[warp] = l;
  }
#pragma unroll
  for (int i = 0; i < NV; ++i) s_o[warp][lane + 32 * i] = o[i];
  __syncthreads();
  const int dim = threadIdx.x;
  if (dim < HDT) {
    float M = s_m[0], L = s_l[0], acc = s_o[0][dim];  // group 0 holds key 0: never empty
#pragma unroll
    for (int w = 1; w < F32_WARPS; ++w) {
      float wa, wb, mm;
      fold_weights(M, s_m[w], wa, wb, mm);
      M = mm;
      L = fold_value(wa, L, wb, s_l[w]);
      acc = fold_value(wa, acc, wb, s_o[w][dim]);
    }
    reinterpret_cast<float*>(a.out)[((size_t)r * a.Hq + h) * HDT + dim] = acc * (L > 0.f ? 1.f / L : 0.f);
  }
}

}  // namespace

#ifdef JF_TIMELINE
JF_TL_SETTER(tl_set_attn)
#endif

// n_ctas: CTAs per unit (1, 2, 4 or 8; one cluster when more than one).
cudaError_t launch_attn_tc(const AttnMaps& tm, const AttnParams& a, int units_bound, int n_ctas, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_ctas * units_bound);
  cfg.blockDim = dim3(ATT_THREADS);
  cfg.dynamicSmemBytes = TC_SMEM;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = n_ctas;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = n_ctas > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, n_ctas > 1 ? k_attn_tc<false> : k_attn_tc<true>, tm.q, tm.k_inf, tm.v_inf, a, n_ctas);
}

// Shared-memory limits of both forms; max_clusters[i] = how many clusters of 2^i CTAs can be resident
// at once (none of the 8-CTA ones is an error).
cudaError_t attn_prepare(int max_clusters[4]) {
  cudaError_t e = cudaFuncSetAttribute(k_attn_tc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_attn_tc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
  if (e != cudaSuccess) return e;
  int dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&max_clusters[0], cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  for (int i = 1; i < 4; ++i) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1 << i);
    cfg.blockDim = dim3(ATT_THREADS);
    cfg.dynamicSmemBytes = TC_SMEM;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1 << i;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if ((e = cudaOccupancyMaxActiveClusters(&max_clusters[i], k_attn_tc<false>, &cfg)) != cudaSuccess) return e;
    if (max_clusters[i] < 1) return cudaErrorInvalidConfiguration;
  }
  return cudaSuccess;
}

cudaError_t launch_attn_f32(const AttnParams& a, int n_rows, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_rows * a.Hq);
  cfg.blockDim = dim3(32 * F32_WARPS);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, a.hd == 64 ? k_attn_f32<64> : k_attn_f32<128>, a);
}

}  // namespace jf
