// Part of the ST^3 library for sm_100a; included by st3.cu only.
#ifndef ST3_FINISH_CUH_
#define ST3_FINISH_CUH_
#include "st3_common.cuh"

namespace {

// ------------------------------------------------------------------------------------------
// Merge partials, visual scores, top-k (Eq. 3), in-place compaction (Eq. 7's eviction)
// ------------------------------------------------------------------------------------------
// Two or more blocks per (layer, sequence), on different SMs, that never wait for each other:
//   OUT block   merges the chunk partials of its heads into the attention output (a warp per head);
//   TRIM block  merges only the (max, sum) pairs, turns the raw logits into head-summed
//               probabilities, selects the rows to keep, pairs holes with kept tail rows and
//               moves the rows.
// Both are chains of dependent memory round trips, so every phase issues all its loads first.
// (max, sum) of one head's merged softmax from its chunk partials; every lane gets both, and in `w` the weights
// exp2(max_i - max) of partials `lane` and `lane + 32`.
__device__ __forceinline__ void merge_stats(const float2* ml, long long item0, int nit, int H, int h, int lane,
                                            float& M, float& L, float (&w)[2]) {
  float2 v[2];  // the first 64 partials stay in registers
#pragma unroll
  for (int j = 0; j < 2; ++j)
    v[j] = lane + 32 * j < nit ? ml[(item0 + lane + 32 * j) * H + h] : make_float2(-INFINITY, 0.f);
  M = fmaxf(v[0].x, v[1].x);
  for (int i = lane + 64; i < nit; i += 32) M = fmaxf(M, ml[(item0 + i) * H + h].x);
  M = warp_max(M);
#pragma unroll
  for (int j = 0; j < 2; ++j) w[j] = fast_exp2(v[j].x - M);
  L = v[0].y * w[0] + v[1].y * w[1];
  for (int i = lane + 64; i < nit; i += 32) {
    const float2 u = ml[(item0 + i) * H + h];
    L += u.y * fast_exp2(u.x - M);
  }
  L = warp_sum(L);
}

constexpr int kSelBins = 256;   // bins of the selection's histogram, over the range of the scores; eight to a lane
constexpr int kSelCand = 64;    // keys of the bin that the cut falls into that are ranked directly

// BPS blocks of NT threads to an SM: one of 512 with 128 registers a thread, one of 1024, or two of 512, as the launch has
// more (layer, sequence) units (st3.cu has the rule: the work of a unit is a chain of round trips, and more units in flight
// end sooner).  Bound by latency: two round trips, the flag, and dependent integer work in
// between, which a warp issues at 6-10 cycles an instruction; threads that have no row only take issue slots.  The same code
// with 1024 threads of 64 registers: 7B layers one a call 9 760 against 9 190 us a generation, 13B layers of 16 sequences
// 26 680 against 25 670.
template <typename T, int D, int BPS, int NT>
__global__ void __launch_bounds__(NT, BPS) st3_finish_kernel(const __grid_constant__ StepParams p) {
  constexpr int kFinishThreads = NT, kFinishWarps = NT / 32;
  constexpr int ROWB = D * sizeof(T);
  constexpr int VPR = ROWB / 16;  // 16-byte vectors per row
  constexpr int DPL = D / 32;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ float2 s_ML[kMaxHeads];  // (max, 1/sum) of a head's merged softmax
  __shared__ __align__(16) int s_hist[kSelBins];
  __shared__ unsigned s_lo, s_hi;
  __shared__ unsigned long long s_cand[kSelCand];
  __shared__ int s_ncand, s_again;
  __shared__ unsigned s_word[kMaxVisual / 32];  // a bit per row: moves (or, of a prompt, is kept)

  const int tid = threadIdx.x, lane = tid & 31;
  const int B = p.B, H = p.H, Nv = p.Nv;
  // grid (sequences, layers, 1 + output blocks): the first plane trims, the others write the output.  No division: a small
  // launch starts little ahead of the end of its wait.
  const int b = blockIdx.x, l_rel = blockIdx.y, out_part = (int)blockIdx.z - 1;
  const bool out_role = out_part >= 0;
  const int l = p.layer_begin + l_rel;
  const long long lb = (long long)l * B + b;
  const LayerParams y = p.layer[l_rel];
  const int nit = y.cv + p.ct;
  const long long item0 = (long long)y.lstart + (long long)b * nit;
  const float2* ml = reinterpret_cast<const float2*>(p.part_ml);
  // the scores that decide come from this layer, or from its stage's pruning layer (same rows, same order)
  const int src = y.src_layer;
  const bool src_here = src >= p.layer_begin && src < p.layer_begin + p.layer_count;
  const int nit_s = src_here ? p.layer[src - p.layer_begin].cv + p.ct : 0;
  const long long item0_s = src_here ? (long long)p.layer[src - p.layer_begin].lstart + (long long)b * nit_s : 0;
  if (!out_role) {
    for (int i = tid; i < kSelBins; i += kFinishThreads) s_hist[i] = 0;
    if (tid == 0) { s_ncand = 0; s_lo = 0xffffffffu; s_hi = 0u; }
  }
  // The parameters a block needs are read before it waits: they are cold in the constant cache (one 7B layer a call
  // 11.07 -> 10.88 us, a small fp32 layer 10.1 -> 9.7, a 13B layer of 16 sequences 44.6 -> 43.5).
  asm volatile("" ::"l"(ml), "l"(p.part_acc), "l"(p.out), "l"(p.logits_copy[y.src_copy]), "l"(p.ids), "l"(p.n_cur),
               "l"(p.flags), "l"(p.ext_scores), "l"(item0 + item0_s), "l"(p.mass_by_id), "r"(p.fresh), "r"(nit + nit_s),
               "r"(p.stage_rows));
  // This launch may have been set up while the attention launch before it was still running: wait for that
  // whole grid (and, through it, for everything earlier in the stream).  Then the next step's attention launch
  // may start; it waits on p.flags for what this launch changes.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (out_role) {
    // ===================== OUT block: attention output of every head =====================
    constexpr int kMergeBatch = 8 * 1024 / (BPS * NT);  // partials in flight per round trip, as the registers allow
    for (int h = out_part * kFinishWarps + (tid >> 5); h < H; h += ((int)gridDim.z - 1) * kFinishWarps) {
      float a[kMergeBatch][DPL];
      auto load_batch = [&](int i0) {
#pragma unroll
        for (int i = 0; i < kMergeBatch; ++i) {
          if (i0 + i < nit) {
            const float* src = p.part_acc + ((item0 + i0 + i) * H + h) * D + lane * DPL;
            if (DPL == 4) {
              const float4 v = *reinterpret_cast<const float4*>(src);
              a[i][0] = v.x; a[i][1] = v.y; a[i][DPL - 2] = v.z; a[i][DPL - 1] = v.w;
            } else {
              const float2 v = *reinterpret_cast<const float2*>(src);
              a[i][0] = v.x; a[i][DPL - 1] = v.y;
            }
          }
        }
      };
      load_batch(0);
      float M, Lh, w[2];
      merge_stats(ml, item0, nit, H, h, lane, M, Lh, w);
      float o[DPL];
#pragma unroll
      for (int j = 0; j < DPL; ++j) o[j] = 0.f;
      for (int i0 = 0; i0 < nit; i0 += kMergeBatch) {
        if (i0) load_batch(i0);
#pragma unroll
        for (int i = 0; i < kMergeBatch; ++i) {
          if (i0 + i < nit) {
            const int it = i0 + i;
            const float wgt = it < 64 ? __shfl_sync(0xffffffffu, it < 32 ? w[0] : w[1], it & 31)
                                      : fast_exp2(ml[(item0 + it) * H + h].x - M);
#pragma unroll
            for (int j = 0; j < DPL; ++j) o[j] = fmaf(wgt, a[i][j], o[j]);
          }
        }
      }
      const float invL = 1.f / Lh;
      T* out = reinterpret_cast<T*>(p.out) + (((long long)l_rel * B + b) * H + h) * D;
#pragma unroll
      for (int j = 0; j < DPL; ++j) store_out(out + lane * DPL + j, o[j] * invL);
    }
    return;
  }

  // ===================== TRIM block =====================
  const int tt = tid, warp = tid >> 5;
  // Signals that this launch is done with the visual rows, ids and logits of (l, b).
  auto done = [&]() {
    __syncthreads();
    if (tt == 0) st_release(p.flags + lb, p.seq);  // what the block wrote is ordered before it by the barrier
  };
  const int n_host = y.ncur;
  const int k = min(n_host, (int)y.ntgt);
  const bool evicts = k < n_host;  // same answer in every thread
  const int n_dev = p.n_cur[lb];
  const bool fresh = p.fresh;  // a new prompt: row i is visual token i, whatever the bookkeeping says
  if (!evicts) {
    if (fresh) {
      for (int i = tt; i < n_host; i += kFinishThreads) { p.ids[lb * Nv + i] = i; p.mass_by_id[lb * Nv + i] = 0.f; }
      if (tt == 0) p.n_cur[lb] = n_host;
    } else if (tt == 0) {
      if (n_dev != y.nold) atomicOr(p.status, ST3_DEV_COUNT_MISMATCH);
      else if (n_host != n_dev) p.n_cur[lb] = n_host;  // static-rank cut: only the count changes
    }
    done();
    return;
  }
  int* ids = p.ids + lb * Nv;
  float* mass_by_id = p.mass_by_id + lb * Nv;
  const long long lb_src = (long long)src * B + b;
  const float* logits = p.logits_copy[y.src_copy] + lb_src * H * logit_pitch(Nv);
  unsigned long long* s_key = reinterpret_cast<unsigned long long*>(smem);  // [Nv]
  int* s_hole = reinterpret_cast<int*>(smem + (size_t)Nv * 8);              // [Nv], the ids until the scores are known
  int* s_mover = s_hole + Nv;                                               // [Nv]
  const int n_cur = n_host;

  // The (max, sum) pairs, the logits of all heads (as many rows as the stage holds) and the ids are requested now: one round
  // trip for all of them, and no registers to hold the logits.
  const bool own_scores = p.ext_scores == nullptr;
  const int pitch = p.stage_rows;  // 16 (mod 32): a quarter of a warp reads two heads without bank conflicts
  float* s_log = reinterpret_cast<float*>(smem + ((size_t)Nv * 12 + 15) / 16 * 16);  // [H][pitch], over the list of movers
  auto stage = [&](int c0) {
    const int rows = min(pitch, n_cur - c0);
    for (int h = warp; h < H; h += kFinishWarps)
      for (int i = 4 * lane; i < rows; i += 128) copy_async<16>(s_log + h * pitch + i, logits + (h * logit_pitch(Nv) + c0 + i));
  };
  if (own_scores) {
    // (max, sum) of the heads: a warp takes eight heads, four lanes to a head
    constexpr int kStatBatch = 4;  // pairs of a lane in flight
    static_assert(kFinishWarps * 8 >= kMaxHeads, "one pass over the heads");
    const int h = warp * 8 + (lane & 7), part = lane >> 3;
    const bool merges = src_here && warp * 8 < H;
    float2 u[kStatBatch];
    auto load_pairs = [&](int c0) {
#pragma unroll
      for (int j = 0; j < kStatBatch; ++j)
        u[j] = h < H && c0 + 4 * j < nit_s ? ml[(item0_s + c0 + 4 * j) * H + h] : make_float2(-INFINITY, 0.f);
    };
    if (merges) load_pairs(part);
    stage(0);
    if (!fresh)
      for (int i = tt; i < n_cur; i += kFinishThreads) copy_async<4>(s_hole + i, ids + i);
    if (merges) {
      float M = -INFINITY, L = 0.f;
      for (int c0 = part;;) {
        float m = M;
#pragma unroll
        for (int j = 0; j < kStatBatch; ++j) m = fmaxf(m, u[j].x);
        const float ref = m > -INFINITY ? m : 0.f;  // a lane without pairs keeps zeros
        L *= fast_exp2(M - ref);
#pragma unroll
        for (int j = 0; j < kStatBatch; ++j) L = fmaf(u[j].y, fast_exp2(u[j].x - ref), L);
        M = m;
        c0 += 4 * kStatBatch;
        if (c0 >= nit_s) break;
        load_pairs(c0);
      }
      __syncwarp();
      float m = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, 8));
      m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 16));
      L *= fast_exp2(M - m);
      L += __shfl_xor_sync(0xffffffffu, L, 8);
      L += __shfl_xor_sync(0xffffffffu, L, 16);
      if (part == 0 && h < H) {
        const float2 st = make_float2(m, 1.f / L);
        s_ML[h] = st;
        if (src == l) *reinterpret_cast<float2*>(p.head_stat + 2 * (lb * H + h)) = st;
      }
    } else if (!src_here) {  // the pruning layer ran in an earlier launch of this step: its statistics were kept
      for (int i = tt; i < H; i += kFinishThreads) s_ML[i] = *reinterpret_cast<const float2*>(p.head_stat + 2 * (lb_src * H + i));
    }
  } else {  // scores of the caller, of a new prompt: each thread fetches what it will read
    const float* ext = p.ext_scores + ((long long)l_rel * B + b) * Nv;
    for (int i = tt; i < n_cur; i += kFinishThreads) copy_async<4>(s_log + i, ext + i);
  }
  copies_landed();
  __syncthreads();
  if (!fresh && n_dev != n_host) {  // host bookkeeping and device state disagree: flag, do not touch
    if (tt == 0) atomicOr(p.status, ST3_DEV_COUNT_MISMATCH);
    done();
    return;
  }

  // ---- visual scores: probability of every visual row summed over heads ----
  bool bad = false;
  unsigned lo = 0xffffffffu, hi = 0u;  // range of the keys' high words
  if (!own_scores) {
    // scores supplied by the caller (any finite float): order-preserving map of the bits to unsigned
    for (int i = tt; i < n_cur; i += kFinishThreads) {
      float sc = s_log[i];
      if (!(fabsf(sc) <= 3.0e38f)) { bad = true; sc = -3.0e38f; }
      mass_by_id[i] = sc;
      unsigned u = __float_as_uint(sc);
      u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
      lo = min(lo, u); hi = max(hi, u);
      s_key[i] = ((unsigned long long)u << 32) | (unsigned long long)(0xffffffffu - (unsigned)i);
    }
  }
  // A lane sums every eighth head of four rows (a warp: 16 rows); the sums meet in shuffles that leave a lane with one row, and
  // take a third of the shared-memory reads that a row per lane takes (1 540 -> 700 cycles a pass of 256 rows of 32 heads).
  // Every fourth head (32 rows) where 16 warps of 16 rows do not hold all rows: a small fp32 layer 186 -> 183.5 us a
  // generation, a prompt of 32 7B layers 1 227 -> 1 206; with 40 heads, ten to a lane, it loses (24 590 -> 24 690 us).  One
  // choice for all passes and for every size of the block and its stage: it decides the order in which a row's heads are added, and rows with equal logits
  // must get equal scores, also in two layers of a stage that are selected in different launches.
  const int lq = n_cur > 256 && H <= 32 ? 3 : 2;  // log2 of the row quads of a warp
  for (int c0 = 0; own_scores && c0 < n_cur; c0 += pitch) {
    if (c0) {
      __syncthreads();
      stage(c0);
      copies_landed();
      __syncthreads();
    }
    const int rows = min(pitch, n_cur - c0);
    const int span = 4 << lq, groups = 32 >> lq, quad = lane & ((1 << lq) - 1), g = lane >> lq;
    for (int r0 = warp * span; r0 < rows; r0 += kFinishWarps * span) {
      const float* at = s_log + min(r0 + quad * 4, (rows - 1) & ~3);
      float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll 4
      for (int h = g; h < H; h += groups) {
        const float2 st = s_ML[h];
        const float4 x = *reinterpret_cast<const float4*>(at + h * pitch);
        a0 += fast_exp2(x.x - st.x) * st.y;
        a1 += fast_exp2(x.y - st.x) * st.y;
        a2 += fast_exp2(x.z - st.x) * st.y;
        a3 += fast_exp2(x.w - st.x) * st.y;
      }
      __syncwarp();
      const bool up = lane & 16, odd = lane & 8;
      const float b0 = (up ? a2 : a0) + __shfl_xor_sync(0xffffffffu, up ? a0 : a2, 16);
      const float b1 = (up ? a3 : a1) + __shfl_xor_sync(0xffffffffu, up ? a1 : a3, 16);
      float mass = (odd ? b1 : b0) + __shfl_xor_sync(0xffffffffu, odd ? b0 : b1, 8);
      if (lq == 2) mass += __shfl_xor_sync(0xffffffffu, mass, 4);
      const int r = r0 + quad * 4 + (up ? 2 : 0) + (odd ? 1 : 0), i = c0 + r;
      if ((lq == 3 || !(lane & 4)) && r < rows) {
        if (!(mass >= 0.f) || !(mass <= 3.0e38f)) { bad = true; mass = 0.f; }
        const int id = fresh ? i : s_hole[i];
        mass_by_id[id] = mass;
        const unsigned u = __float_as_uint(mass);
        lo = min(lo, u); hi = max(hi, u);
        s_key[i] = ((unsigned long long)u << 32) | (unsigned long long)(0xffffffffu - (unsigned)id);
      }
    }
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(p.status, ST3_DEV_NONFINITE);
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) { atomicMin(&s_lo, lo); atomicMax(&s_hi, hi); }
  __syncthreads();

  // From here on row i belongs to thread i; the warps without rows go straight to the barriers and leave the issue slots to
  // the others.
  const bool works = warp * 32 < n_cur;

  // ---- the k-th largest 64-bit key (keys are unique: ids are) ----
  // A histogram over the range of the keys finds the bin of the cut, and the keys in it are ranked against one another.
  // Where too many share it (narrow or equal scores), the same once more over that bin's range.  Every working warp
  // derives the bin and the cut by itself.
  unsigned long long prefix = ~0ull;  // k = 0: no key reaches this value (ids are < 2^31)
  if (k > 0) {
    lo = s_lo;
    unsigned long long base = (unsigned long long)lo << 32;  // first key of bin 0
    int sh = 32 + max(0, 24 - __clz((int)(s_hi - lo)));      // log2 of a bin's keys: the high words make 256 bins
    int width = 64, need = k;                                // log2 of all bins' keys; how many of them are kept
    for (;;) {
      auto inside = [&](unsigned long long key) { return width == 64 || (key - base) >> width == 0; };
      if (works) {
        for (int i = tt; i < n_cur; i += kFinishThreads) {
          const unsigned long long key = s_key[i];
          const unsigned d = width == 64 ? ((unsigned)(key >> 32) - lo) >> (sh - 32) : (unsigned)((key - base) >> sh);
          if (inside(key)) atomicAdd(&s_hist[(d & 4) * 32 + (d >> 3) * 4 + (d & 3)], 1);  // a lane's bins as two vectors
        }
      }
      __syncthreads();
      int inbin = 0;
      if (works) {
        const int4 a = reinterpret_cast<const int4*>(s_hist)[lane], c4 = reinterpret_cast<const int4*>(s_hist)[32 + lane];
        // keys of this lane's bins j and above (and none: f[8])
        const int f7 = c4.w, f6 = f7 + c4.z, f5 = f6 + c4.y, f4 = f5 + c4.x, f3 = f4 + a.w, f2 = f3 + a.z, f1 = f2 + a.y, f0 = f1 + a.x;
        int S = f0;  // inclusive suffix sum over lanes (this lane and the higher ones)
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int x = __shfl_down_sync(0xffffffffu, S, o);
          if (lane + o < 32) S += x;
        }
        const int want = need - (S - f0);  // of this lane's bins
        const unsigned who = __ballot_sync(0xffffffffu, 0 < want && want <= f0);
        // the highest bin j with want <= f[j]
        const int f[9] = {f0, f1, f2, f3, f4, f5, f6, f7, 0};
        int digit = -1, upto = f0, above = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          digit += want <= f[j];
          upto = want <= f[j] ? f[j] : upto;
        }
#pragma unroll
        for (int j = 8; j >= 1; --j) above = want > f[j] ? f[j] : above;
        const int from = __ffs(who) - 1;
        digit = __shfl_sync(0xffffffffu, digit + lane * 8, from);
        inbin = __shfl_sync(0xffffffffu, upto - above, from);
        need = __shfl_sync(0xffffffffu, want - above, from);
        base += (unsigned long long)digit << sh;
        width = sh;
        sh = max(0, sh - 8);
        if (need < inbin && inbin <= kSelCand) {
          for (int i = tt; i < n_cur; i += kFinishThreads) {
            const unsigned long long key = s_key[i];
            if (inside(key)) s_cand[atomicAdd(&s_ncand, 1)] = key;
          }
        }
        if (tt == 0) s_again = need < inbin && inbin > kSelCand;
      }
      __syncthreads();
      if (!s_again) {
        prefix = base;  // the whole bin is kept
        if (works && need < inbin) {
          const unsigned long long k0 = lane < inbin ? s_cand[lane] : 0ull, k1 = lane + 32 < inbin ? s_cand[lane + 32] : 0ull;
          int l0 = 0, l1 = 0;  // larger keys
          for (int j = 0; j < inbin; ++j) {
            const unsigned long long x = s_cand[j];
            l0 += x > k0; l1 += x > k1;
          }
          const unsigned b0 = __ballot_sync(0xffffffffu, lane < inbin && l0 == need - 1);
          const unsigned b1 = __ballot_sync(0xffffffffu, lane + 32 < inbin && l1 == need - 1);
          prefix = __shfl_sync(0xffffffffu, b0 ? k0 : k1, __ffs(b0 ? b0 : b1) - 1);
        }
        break;
      }
      for (int i = tt; i < kSelBins; i += kFinishThreads) s_hist[i] = 0;
      __syncthreads();
    }
  }

  if (fresh && p.static_rank) {
    // ---- top-index order: the kept token with r larger keys comes r-th.  st3_gather_kernel copies the rows.
    for (int i = tt; i < n_cur; i += kFinishThreads) {
      const unsigned long long key = s_key[i];
      if (key >= prefix) {
        int r = 0;
        for (int j = 0; j < n_cur; ++j) r += s_key[j] > key;
        ids[r] = i;
      }
    }
    if (tt == 0) p.n_cur[lb] = k;
    done();
    return;
  }

  // ---- pair every hole among the first k rows with a kept row of the tail (of a prompt: number the kept rows) ----
  if (works) {
    for (int i0 = warp * 32; i0 < n_cur; i0 += kFinishThreads) {
      const int i = i0 + lane;
      const bool keep = i < n_cur && s_key[i] >= prefix;
      const unsigned word = __ballot_sync(0xffffffffu, i < n_cur && (fresh ? keep : keep != (i < k)));
      if (lane == 0) s_word[i0 >> 5] = word;
    }
  }
  __syncthreads();
  const int low_words = fresh ? kMaxVisual / 32 : k >> 5;  // words of the first k rows, and the bits of the word across
  const unsigned low_bits = (1u << (k & 31)) - 1;          // the border
  auto low_of = [&](int x) { return x < low_words ? 0xffffffffu : x == low_words ? low_bits : 0u; };
  const int nwords = (n_cur + 31) >> 5;
  // A warp takes a run of words, so that it adds up those below only once; its first one is requested together with them
  // (after the sums: 7B layers one a call 8 746 -> 8 804 us a generation).
  const int run = (nwords + kFinishWarps - 1) / kFinishWarps, first = warp * run;
  unsigned word = first < nwords ? s_word[first] : 0u;
  auto bits_of = [&](unsigned x, unsigned m) { return __popc(x & m) | __popc(x & ~m) << 16; };
  int total = 0, before = 0;  // set bits (holes | movers << 16) of all words, and of the words below w0
  for (int x = lane; x < nwords; x += 32) {
    const int c = bits_of(s_word[x], low_of(x));
    total += c;
    before += x < first ? c : 0;
  }
  total = __reduce_add_sync(0xffffffffu, total);
  before = __reduce_add_sync(0xffffffffu, before);
  for (int w0 = first;;) {
    const unsigned m = low_of(w0), lt = (1u << lane) - 1;
    if (word >> lane & 1u) {
      const int i = w0 * 32 + lane;
      if (fresh) ids[before + __popc(word & lt)] = i;  // the prompt's order; st3_gather_kernel copies the rows
      else if (m >> lane & 1u) s_hole[(before & 0xffff) + __popc(word & m & lt)] = i;
      else s_mover[(before >> 16) + __popc(word & ~m & lt)] = i;
    }
    if (++w0 >= min(first + run, nwords)) break;
    before += bits_of(word, m);
    word = s_word[w0];
  }
  if (fresh) {
    if (tt == 0) {
      p.n_cur[lb] = k;
      if (total != k) atomicOr(p.status, ST3_DEV_RANGE);  // cannot happen: exactly k keys pass the threshold
    }
    done();
    return;
  }
  __syncthreads();
  const int nmove = total & 0xffff;
  if (nmove != (total >> 16)) {  // cannot happen when exactly k keys pass the threshold
    if (tt == 0) atomicOr(p.status, ST3_DEV_RANGE);
    done();
    return;
  }

  // ---- move the rows (sources are rows >= k, destinations rows < k: disjoint) ----
  // A thread's vectors are the same 16 bytes of the key or value row of one (row, head) pair after another.
  constexpr int VPP = 2 * VPR, kPairs = kFinishThreads / VPP;  // vectors of a pair, pairs side by side
  unsigned char* blk0 = reinterpret_cast<unsigned char*>(p.cache) + (size_t)(lb * H) * p.lbh_stride * sizeof(T) +
                        (size_t)(tt / VPR % 2) * Nv * ROWB + tt % VPR * 16;
  const int npair = nmove * H;
  const size_t head_bytes = (size_t)p.lbh_stride * sizeof(T);
  auto place = [&](int x, const int* rows) {
    const unsigned r = fast_div((unsigned)x, p.h_mul, p.h_shift);
    return reinterpret_cast<uint4*>(blk0 + (x - r * H) * head_bytes + rows[r] * ROWB);
  };
  constexpr int kMoveBatch = 8 / (BPS * NT / 512);  // vectors of a thread in flight
  for (int x0 = tt / VPP; x0 < npair; x0 += kMoveBatch * kPairs) {
    uint4 val[kMoveBatch];
#pragma unroll
    for (int j = 0; j < kMoveBatch; ++j)
      if (x0 + j * kPairs < npair) val[j] = *place(x0 + j * kPairs, s_mover);
    if (x0 == tt / VPP)  // under the loads: the ids, each the low word of its key
      for (int j = tt; j < nmove; j += kFinishThreads) ids[s_hole[j]] = (int)(0xffffffffu - (unsigned)s_key[s_mover[j]]);
#pragma unroll
    for (int j = 0; j < kMoveBatch; ++j)
      if (x0 + j * kPairs < npair) *place(x0 + j * kPairs, s_hole) = val[j];
  }
  proxy_fence();  // the next attention launch reads the moved rows with bulk copies once it sees the flag
  if (tt == 0) p.n_cur[lb] = k;
  done();
}

// ------------------------------------------------------------------------------------------
// Prompt rows -> cache regions: [S | I] to the text region, the kept visual rows (ids) to the visual region
// ------------------------------------------------------------------------------------------
// Runs after the selection and copies what it kept, spread over the whole GPU: bound by memory bandwidth for a batch,
// by one round trip for ids and one for the rows for a single layer.  The selection blocks used to move the kept rows
// inside the cache, one block per (layer, sequence): 105-118 us for 32 heads and 576 visual tokens, 515 us for 2880.
// st3_prefill_select of one 7B layer, one sequence: 105 -> 28 us; 32 layers in one call: 298 -> 137 us; a 13B layer of
// 16 sequences: 269 -> 104 us; three NeXT layers of 8 sequences that prune: 1099 -> 415 us, that keep all: 589 -> 577 us.
constexpr int kGatherBlocks = 16;  // per (layer, sequence, head); 4, 8, 16 and 32 blocks and 1, 2 or 4 vectors in flight
                                   // per thread are within 3 % of one another on a batch, 16 or more best for one layer

// Where the attention launch has not cached them (p.store_rows), the text rows and the visual rows of layers that keep
// them all are copied as well, under the selection launch: what they need was complete before a block of it let this
// launch start.
template <typename T, int D>
__global__ void __launch_bounds__(kThreads) st3_gather_kernel(const __grid_constant__ StepParams p) {
  constexpr int VPR = D * sizeof(T) / 16;
  const int H = p.H, B = p.B, Nv = p.Nv;
  // grid (kGatherBlocks, heads x layers, sequences): all of it in y would exceed the 65535 a dimension holds
  const int h = blockIdx.y % H, l_rel = blockIdx.y / H, b = blockIdx.z;
  const long long lb = (long long)(p.layer_begin + l_rel) * B + b;
  const int n_txt = p.store_rows ? 0 : p.sys_len + __ldg(p.text_len + b);
  const bool all = p.layer[l_rel].ntgt == Nv;
  const int n_vis = all && p.store_rows ? 0 : p.layer[l_rel].ntgt;
  const int* ids = p.ids + lb * Nv;
  const long long in0 = (((long long)l_rel * B + b) * H + h) * p.t0_max * VPR;
  const uint4* srcK = reinterpret_cast<const uint4*>(p.k_in) + in0;
  const uint4* srcV = reinterpret_cast<const uint4*>(p.v_in) + in0;
  uint4* dst = reinterpret_cast<uint4*>(reinterpret_cast<T*>(p.cache) + (lb * H + h) * p.lbh_stride);
  const int total = (n_txt + n_vis) * VPR;
  bool selected = all;  // the kept rows are known
  for (int i = blockIdx.x * kThreads + threadIdx.x; i < total; i += kGatherBlocks * kThreads) {
    const int row = i / VPR, c = i % VPR;
    const bool vis = row >= n_txt;
    int src;  // row of the prompt
    if (vis) {
      if (!selected) asm volatile("griddepcontrol.wait;" ::: "memory");
      selected = true;
      const int id = all ? row - n_txt : ids[row - n_txt];
      if ((unsigned)id >= (unsigned)Nv) {  // a selection that failed: reported, not used
        atomicOr(p.status, ST3_DEV_RANGE);
        continue;
      }
      src = p.sys_len + id;
    } else {
      src = row < p.sys_len ? row : row + Nv;
    }
    const uint4 kk = __ldg(srcK + src * VPR + c), vv = __ldg(srcV + src * VPR + c);
    // K_vis | V_vis | K_txt | V_txt
    const long long d = vis ? i - n_txt * VPR : 2LL * Nv * VPR + i;
    dst[d] = kk;
    dst[d + (long long)(vis ? Nv : p.cap_txt) * VPR] = vv;
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");  // this grid ends after the one ahead of it
}

}  // namespace

#endif  // ST3_FINISH_CUH_
