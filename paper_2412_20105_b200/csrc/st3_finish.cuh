// Part of the ST^3 library for sm_100a; included by st3.cu only.
#ifndef ST3_FINISH_CUH_
#define ST3_FINISH_CUH_
#include "st3_common.cuh"

namespace {

// ------------------------------------------------------------------------------------------
// Merge partials, visual scores, top-k (Eq. 3), in-place compaction (Eq. 7's eviction)
// ------------------------------------------------------------------------------------------
// Two blocks per (layer, sequence), on different SMs, that never wait for each other:
//   OUT block   merges the chunk partials of every head into the attention output (a warp per head);
//   TRIM block  merges only the (max, sum) pairs, turns the raw logits into head-summed
//               probabilities, selects the rows to keep, pairs holes with kept tail rows and
//               moves the rows.
// Both are chains of dependent memory round trips, so every phase issues all its loads first.
constexpr int kHeadBatch = 16;  // logits of one visual row a thread keeps in flight

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

constexpr int kSelBins = 2048;  // bins of the selection's histogram, over the range of the scores
constexpr int kSelCand = 64;    // keys of the bin that the cut falls into that are ranked directly

// NT threads per block: 1024, or 512 (two blocks per SM) when a launch has more (layer, sequence) units than the GPU
// can hold blocks: the work of a unit is a chain of memory round trips, and more units in flight end sooner.
template <typename T, int D, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) st3_finish_kernel(const __grid_constant__ StepParams p) {
  constexpr int kFinishThreads = NT, kFinishWarps = NT / 32;
  constexpr int ROWB = D * sizeof(T);
  constexpr int VPR = ROWB / 16;  // 16-byte vectors per row
  constexpr int DPL = D / 32;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ float2 s_ML[kMaxHeads];  // (max, 1/sum) of a head's merged softmax
  __shared__ int s_hist[kSelBins];
  __shared__ int s_scan[kFinishWarps];
  __shared__ unsigned s_lo[kFinishWarps], s_hi[kFinishWarps];
  __shared__ unsigned long long s_cand[kSelCand], s_cut;
  __shared__ int s_ncand;
  __shared__ float s_half[kFinishThreads / 2];
  __shared__ int s_sel[3];  // digit, count above, count in bin

  const int tid = threadIdx.x, lane = tid & 31;
  const int B = p.B, H = p.H, Nv = p.Nv;
  const int units = p.layer_count * B;  // blocks [0, units) trim, blocks [units, 2 units) write the output
  const bool out_role = (int)blockIdx.x >= units;
  const int unit = out_role ? blockIdx.x - units : blockIdx.x;
  const int l_rel = unit / B, b = unit % B;
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
    if (tid == 0) s_ncand = 0;
  }
  // The parameters a block needs are read before it waits: they are cold in the constant cache (one 7B layer a call
  // 11.07 -> 10.88 us, a small fp32 layer 10.1 -> 9.7, a 13B layer of 16 sequences 44.6 -> 43.5).
  asm volatile("" ::"l"(ml), "l"(p.part_acc), "l"(p.out), "l"(p.logits_copy[y.src_copy]), "l"(p.ids), "l"(p.n_cur),
               "l"(p.flags), "l"(p.ext_scores), "l"(item0 + item0_s), "l"(p.mass_by_id), "r"(p.fresh), "r"(nit + nit_s));
  // This launch may have been set up while the attention launch before it was still running: wait for that
  // whole grid (and, through it, for everything earlier in the stream).  Then the next step's attention launch
  // may start; it waits on p.flags for what this launch changes.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (out_role) {
    if (p.ext_scores) return;  // selection-only launch: nothing to merge yet
    // ===================== OUT block: attention output of every head =====================
    constexpr int kMergeBatch = 8;  // partials in flight per round trip
    for (int h = tid >> 5; h < H; h += kFinishWarps) {
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
  const float* logits = p.logits_copy[y.src_copy] + lb_src * H * Nv;
  unsigned long long* s_key = reinterpret_cast<unsigned long long*>(smem);  // [Nv]
  int* s_hole = reinterpret_cast<int*>(smem + (size_t)Nv * 8);              // [Nv]
  int* s_mover = s_hole + Nv;                                               // [Nv]
  const int n_cur = n_host;

  // Thread (row r, half g) of a pass sums every second batch of 16 heads of its row; half 1 hands its
  // sum to half 0 through shared memory, so the order of the additions is fixed.  The first batch of
  // the first pass is requested now, together with the (max, sum) pairs: one round trip for both.
  constexpr int kRowsPerPass = kFinishThreads / 2;
  const int ri = tt % kRowsPerPass, hg = tt / kRowsPerPass;
  float pre[kHeadBatch];
  int id0 = 0;
  const bool own_scores = p.ext_scores == nullptr;
  if (own_scores) {
    if (ri < n_cur) {
      if (hg == 0) id0 = fresh ? ri : ids[ri];
#pragma unroll
      for (int j = 0; j < kHeadBatch; ++j) {
        const int h = hg * kHeadBatch + j;
        pre[j] = h < H ? logits[(long long)h * Nv + ri] : -INFINITY;
      }
    }
    if (src_here) {
      for (int h = warp; h < H; h += kFinishWarps) {
        float M, Lh, w[2];
        merge_stats(ml, item0_s, nit_s, H, h, lane, M, Lh, w);
        if (lane == 0) {
          s_ML[h] = make_float2(M, 1.f / Lh);
          if (src == l) { p.head_stat[2 * (lb * H + h)] = M; p.head_stat[2 * (lb * H + h) + 1] = 1.f / Lh; }
        }
      }
    } else {  // the pruning layer ran in an earlier launch of this step: its statistics were kept
      for (int h = tt; h < H; h += kFinishThreads) {
        s_ML[h] = make_float2(p.head_stat[2 * (lb_src * H + h)], p.head_stat[2 * (lb_src * H + h) + 1]);
      }
    }
  }
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
    const float* ext = p.ext_scores + ((long long)l_rel * B + b) * Nv;
    for (int i = tt; i < n_cur; i += kFinishThreads) {
      const int id = fresh ? i : ids[i];
      float sc = ext[id];
      if (!(fabsf(sc) <= 3.0e38f)) { bad = true; sc = -3.0e38f; }
      mass_by_id[id] = sc;
      unsigned u = __float_as_uint(sc);
      u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
      lo = min(lo, u); hi = max(hi, u);
      s_key[i] = ((unsigned long long)u << 32) | (unsigned long long)(0xffffffffu - (unsigned)id);
    }
  }
  for (int i0 = 0; own_scores && i0 < n_cur; i0 += kRowsPerPass) {
    const int i = i0 + ri;
    float pm = 0.f;
    int id = id0;
    if (i < n_cur) {
      if (i0 && hg == 0) id = fresh ? i : ids[i];
      for (int h0 = hg * kHeadBatch; h0 < H; h0 += 2 * kHeadBatch) {
        float v[kHeadBatch];
        if (i0 == 0 && h0 == hg * kHeadBatch) {
#pragma unroll
          for (int j = 0; j < kHeadBatch; ++j) v[j] = pre[j];
        } else {
#pragma unroll
          for (int j = 0; j < kHeadBatch; ++j) v[j] = h0 + j < H ? logits[(long long)(h0 + j) * Nv + i] : -INFINITY;
        }
#pragma unroll
        for (int j = 0; j < kHeadBatch; ++j)
          if (h0 + j < H) {
            const float2 st = s_ML[h0 + j];
            pm += fast_exp2(v[j] - st.x) * st.y;
          }
      }
    }
    if (hg == 1) s_half[ri] = pm;
    __syncthreads();
    if (hg == 0 && i < n_cur) {
      float mass = pm + s_half[ri];
      if (!(mass >= 0.f) || !(mass <= 3.0e38f)) { bad = true; mass = 0.f; }
      mass_by_id[id] = mass;
      const unsigned u = __float_as_uint(mass);
      lo = min(lo, u); hi = max(hi, u);
      s_key[i] = ((unsigned long long)u << 32) | (unsigned long long)(0xffffffffu - (unsigned)id);
    }
    if (i0 + kRowsPerPass < n_cur) __syncthreads();  // s_half is written again
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) { s_lo[warp] = lo; s_hi[warp] = hi; }
  __syncthreads();
  if (bad) atomicOr(p.status, ST3_DEV_NONFINITE);

  // ---- the k-th largest 64-bit key (keys are unique: ids are) ----
  // One histogram over the range of the scores (2048 bins: a few keys in each) finds the bin of the cut, and the keys
  // in it are ranked against one another.  Where too many share it (equal scores), a radix select over all digits.
  unsigned long long prefix = 0ull, mask = 0ull;
  bool found = true;
  if (k > 0) {
    lo = __reduce_min_sync(0xffffffffu, lane < kFinishWarps ? s_lo[lane] : 0xffffffffu);
    hi = __reduce_max_sync(0xffffffffu, lane < kFinishWarps ? s_hi[lane] : 0u);
    const int sh = max(0, 32 - __clz((int)(hi - lo)) - 11);  // (hi - lo) >> sh < 2048
    for (int i = tt; i < n_cur; i += kFinishThreads)
      atomicAdd(&s_hist[((unsigned)(s_key[i] >> 32) - lo) >> sh], 1);
    __syncthreads();
    constexpr int kPer = kSelBins / kFinishThreads;  // consecutive bins of a thread
    int c[kPer], t = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) { c[j] = s_hist[tt * kPer + j]; t += c[j]; }
    int S = t;  // inclusive suffix sum over lanes (this lane and the higher ones)
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_down_sync(0xffffffffu, S, o);
      if (lane + o < 32) S += v;
    }
    if (lane == 0) s_scan[warp] = S;
    __syncthreads();
    int above = S - t + __reduce_add_sync(0xffffffffu, lane > warp && lane < kFinishWarps ? s_scan[lane] : 0);
    if (above < k && k <= above + t) {
#pragma unroll
      for (int j = kPer - 1; j >= 0; --j) {
        if (above + c[j] >= k) { s_sel[0] = tt * kPer + j; s_sel[1] = above; s_sel[2] = c[j]; break; }
        above += c[j];
      }
    }
    __syncthreads();
    const unsigned digit = (unsigned)s_sel[0];
    const int need = k - s_sel[1], inbin = s_sel[2];
    if (need == inbin) {  // the whole bin is kept
      prefix = (unsigned long long)(lo + (digit << sh)) << 32;
    } else if (inbin <= kSelCand) {
      for (int i = tt; i < n_cur; i += kFinishThreads) {
        const unsigned long long key = s_key[i];
        if (((unsigned)(key >> 32) - lo) >> sh == digit) s_cand[atomicAdd(&s_ncand, 1)] = key;
      }
      __syncthreads();
      if (tt < inbin) {
        const unsigned long long key = s_cand[tt];
        int larger = 0;
        for (int j = 0; j < inbin; ++j) larger += s_cand[j] > key;
        if (larger == need - 1) s_cut = key;
      }
      __syncthreads();
      prefix = s_cut;
    } else {
      found = false;
    }
  }
  if (k > 0 && !found) {
    int need = k;
    for (int shift = 56; shift >= 0; shift -= 8) {
      if (tt < 256) s_hist[tt] = 0;
      __syncthreads();
      for (int i = tt; i < n_cur; i += kFinishThreads) {
        const unsigned long long key = s_key[i];
        if ((key & mask) == prefix) atomicAdd(&s_hist[(int)((key >> shift) & 0xffull)], 1);
      }
      __syncthreads();
      if (warp == 0) {
        int c[8], t = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) { c[j] = s_hist[lane * 8 + j]; t += c[j]; }
        int S = t;  // inclusive suffix sum over lanes (this lane and the higher ones)
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_down_sync(0xffffffffu, S, o);
          if (lane + o < 32) S += v;
        }
        int above = S - t;
        if (above < need && need <= S) {
#pragma unroll
          for (int j = 7; j >= 0; --j) {
            if (above + c[j] >= need) { s_sel[0] = lane * 8 + j; s_sel[1] = above; s_sel[2] = c[j]; break; }
            above += c[j];
          }
        }
      }
      __syncthreads();
      const int digit = s_sel[0], above = s_sel[1], inbin = s_sel[2];
      need -= above;
      prefix |= (unsigned long long)digit << shift;
      mask |= 0xffull << shift;
      if (need == inbin) break;  // the whole bin is kept: keys >= prefix are exactly the top k
    }
  }
  if (k == 0) {
    prefix = ~0ull;  // keep nothing (ids are < 2^31, so no key reaches this value)
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

  // ---- pair every hole among the first k rows with a kept row of the tail ----
  const int per = (n_cur + kFinishThreads - 1) / kFinishThreads;
  const int i0 = min(n_cur, tt * per), i1 = min(n_cur, i0 + per);
  int nh = 0, nm = 0;
  for (int i = i0; i < i1; ++i) {
    const bool keep = s_key[i] >= prefix;
    nh += fresh ? keep : (i < k && !keep);
    nm += !fresh && i >= k && keep;
  }
  const int packed = nh | (nm << 16);
  int incl = packed;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) s_scan[warp] = incl;
  __syncthreads();
  int wsum = lane < kFinishWarps ? s_scan[lane] : 0;  // inclusive prefix sums of the warps' totals, in every warp
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, wsum, o);
    if (lane >= o) wsum += v;
  }
  const int total = __shfl_sync(0xffffffffu, wsum, 31);
  const int woff = warp ? __shfl_sync(0xffffffffu, wsum, warp - 1) : 0;
  const int excl = woff + incl - packed;
  int ph = excl & 0xffff, pm = excl >> 16;
  if (fresh) {  // the kept tokens in the prompt's order; st3_gather_kernel copies the rows
    for (int i = i0; i < i1; ++i)
      if (s_key[i] >= prefix) ids[ph++] = i;
    if (tt == 0) {
      p.n_cur[lb] = k;
      if ((total & 0xffff) != k) atomicOr(p.status, ST3_DEV_RANGE);  // cannot happen: exactly k keys pass the threshold
    }
    done();
    return;
  }
  for (int i = i0; i < i1; ++i) {
    const bool keep = s_key[i] >= prefix;
    if (i < k && !keep) s_hole[ph++] = i;
    if (i >= k && keep) s_mover[pm++] = i;
  }
  __syncthreads();
  const int nmove = total & 0xffff;
  if (nmove != (total >> 16)) {  // cannot happen when exactly k keys pass the threshold
    if (tt == 0) atomicOr(p.status, ST3_DEV_RANGE);
    done();
    return;
  }

  // ---- move the rows (sources are rows >= k, destinations rows < k: disjoint) ----
  const int id_moved = tt < nmove ? ids[s_mover[tt]] : 0;  // in flight together with the rows
  unsigned char* blk0 = reinterpret_cast<unsigned char*>(p.cache) + (size_t)(lb * H) * p.lbh_stride * sizeof(T);
  const unsigned nvec = (unsigned)(nmove * H * 2 * VPR);
  auto place = [&](unsigned v, const int* rows) {  // vector v of the moves: (row, head, K or V, 16 bytes of it)
    const unsigned x = v / (2 * VPR), j = fast_div(x, p.h_mul, p.h_shift);
    return reinterpret_cast<uint4*>(blk0 + (size_t)(x - j * H) * p.lbh_stride * sizeof(T) +
                                    ((size_t)(v / VPR % 2) * Nv + rows[j]) * ROWB) + v % VPR;
  };
  constexpr int kMoveBatch = 8;  // vectors of a thread in flight: one round trip for 8 rows of 32 heads
  for (unsigned v0 = tt; v0 < nvec; v0 += kMoveBatch * kFinishThreads) {
    uint4 val[kMoveBatch];
#pragma unroll
    for (int j = 0; j < kMoveBatch; ++j)
      if (v0 + j * kFinishThreads < nvec) val[j] = *place(v0 + j * kFinishThreads, s_mover);
#pragma unroll
    for (int j = 0; j < kMoveBatch; ++j)
      if (v0 + j * kFinishThreads < nvec) *place(v0 + j * kFinishThreads, s_hole) = val[j];
  }
  proxy_fence();  // the next attention launch reads the moved rows with bulk copies once it sees the flag
  if (tt < nmove) ids[s_hole[tt]] = id_moved;
  for (int j = tt + kFinishThreads; j < nmove; j += kFinishThreads) ids[s_hole[j]] = ids[s_mover[j]];
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
