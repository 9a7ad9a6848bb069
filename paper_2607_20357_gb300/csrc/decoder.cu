// Device-side schedule of the gated decoder (Sec. 3.2) and the row kernels
// around the GEMMs: RMSNorm, final norm of the last rows, RoPE table.
//
// For every layer l the setup kernel turns the gates into work lists, so
// that gated-off work is never issued and the host never learns k or T:
//  * e_{b,l,j} = (l < P) or (layer_gate[b,l] and group_gate[b,l,j]);
//  * consecutive samples with the same non-zero group mask form one row
//    segment (samples with mask 0 skip the layer: residual bypass);
//  * QKV tiles cover only the Q/K/V columns of active groups, gate/up tiles
//    only active FFN channels. These N-sparse lists are built per group, over
//    maximal runs of consecutive samples in which that group runs (other
//    groups' bits do not cut a run), and adjacent groups whose on/off pattern
//    over the samples is the same share one column block; so mixed masks do
//    not fragment the row tiles, and all-on batches get the segment tiles;
//  * O and down tiles carry the segment mask so their K loop visits only
//    active groups' rows of W_O / W_down;
//  * attention items are (sample, active head, block of kAttnQ queries).
#include "kernels.cuh"

namespace svl {

constexpr int kSetupThreads = 512;
constexpr int kSetupRows = kSetupThreads / 32;  // rows of X per block (one warp each)
constexpr int kVtRows = 512;                    // rows of V^T per zeroing block

// The persistent GEMM runs tiles in waves of num_sms. When the last wave is
// at most half full, each of its tiles is cut into two half-width tiles
// (which then still fit in one wave and finish in about half the time).
// `head` > 0: halves must hold whole heads of that width (RoPE epilogue).
// Called by the whole block once the list is complete; the appended halves
// keep the order of their tiles (a ballot prefix over the eligible ones).
// s_scan: blockDim.x / 32 ints of shared memory. Returns the new count.
__device__ int split_tail(int4* tiles, int count, int cap, int num_sms, int head, int* s_scan) {
  const int r = count % num_sms;
  if (r == 0 || 2 * r > num_sms) return count;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int eligible = 0;  // in the chunks before this one
  for (int c0 = count - r; c0 < count; c0 += blockDim.x) {
    const int i = c0 + static_cast<int>(threadIdx.x);
    int4 t = make_int4(0, 0, 0, 0);
    bool e = false;
    if (i < count) {
      t = tiles[i];
      const int nc = t.w & 0xFFFF, half = nc / 2;
      e = nc >= 64 && !(half & 15) && !(head > 0 && half % head);
    }
    const unsigned bal = __ballot_sync(0xffffffffu, e);
    if (lane == 0) s_scan[warp] = __popc(bal);
    __syncthreads();
    int before = eligible + __popc(bal & ((1u << lane) - 1u)), chunk = 0;
    for (int w = 0; w < nw; ++w) {
      if (w < warp) before += s_scan[w];
      chunk += s_scan[w];
    }
    __syncthreads();  // s_scan is reused by the next chunk
    if (e && count + before < cap) {
      const int nc = t.w & 0xFFFF, half = nc / 2;
      tiles[i] = make_int4(t.x, t.y, t.z, (t.w & ~0xFFFF) | half);
      tiles[count + before] = make_int4(t.x, t.y, t.z + half, (t.w & ~0xFFFF) | (nc - half));
    }
    eligible += chunk;
  }
  return count + min(eligible, cap - count);
}

// Residual GEMMs (O, down) cut the tiles of a last wave that is at most half
// full along K instead: each of the r tail tiles is repeated s times (s =
// num_sms / r, at most 8, within the list capacity and the partial buffer),
// the copies compute shares of the tile's K blocks side by side in that wave
// and the last to finish sums them. Full-width tiles keep the tensor core's
// widest MMAs. Called by the whole block once the list is complete; thread 0
// writes {first copy index, r, s} to info. Returns the count.
__device__ int split_k_tail(int4* tiles, int count, int cap, int num_sms, int units, int* info) {
  const int sp = ksplit_shares(count, cap, num_sms, units);
  const int r = sp < 2 ? 0 : count % num_sms;
  const int first = count - r;
  if (threadIdx.x == 0) {
    info[0] = first;
    info[1] = r;
    info[2] = sp < 2 ? 1 : sp;
  }
  if (sp < 2) return count;
  // copy `part` (1 .. sp-1) of tail tile i goes to count + (part - 1) r + i
  for (int idx = threadIdx.x; idx < r * (sp - 1); idx += blockDim.x) tiles[count + idx] = tiles[first + idx % r];
  return count + r * (sp - 1);
}

// Shared memory of a list block: the non-empty samples of the batch in order
// (rows [cu0, cu1), group mask: bit j set if group j runs) and the row runs of
// the list being built with their first entry's index. Sized for B samples.
struct ListShared {
  int *cu0, *cu1, *r0, *r1, *off;
  uint8_t *mask, *key;
  int n;  // non-empty samples
  SVL_DEVINL ListShared(int* base, int B)
      : cu0(base), cu1(cu0 + B), r0(cu1 + B), r1(r0 + B), off(r1 + B), mask(reinterpret_cast<uint8_t*>(off + B + 1)),
        key(mask + B), n(0) {}
};
size_t list_shared_bytes(int B) { return (5 * static_cast<size_t>(B) + 1) * sizeof(int) + 2 * static_cast<size_t>(B); }

// Maximal runs of consecutive samples with the same non-zero key: the group
// mask (bit < 0), or whether group `bit` runs. Fills r0, r1 and key of every
// run; returns their number. Called by the whole block.
__device__ int find_runs(ListShared& sh, int bit, int* s_scan) {
  auto key = [&](int i) -> int { return bit < 0 ? sh.mask[i] : (sh.mask[i] >> bit) & 1; };
  int nrun = 0;
  for (int c0 = 0; c0 < sh.n; c0 += blockDim.x) {
    const int i = c0 + static_cast<int>(threadIdx.x);
    const int k = i < sh.n ? key(i) : 0;
    const int start = (k && (i == 0 || key(i - 1) != k)) ? 1 : 0;
    int total;
    const int id = nrun + block_exclusive_scan(start, &total, s_scan) + start - 1;
    if (start) {
      sh.r0[id] = sh.cu0[i];
      sh.key[id] = static_cast<uint8_t>(k);
    }
    if (k && (i == sh.n - 1 || key(i + 1) != k)) sh.r1[id] = sh.cu1[i];
    nrun += total;
  }
  __syncthreads();
  return nrun;
}

// off[i] = sum of count(0 .. i-1) over n entries, off[n] = the total (returned).
template <class Count>
__device__ int prefix_offsets(ListShared& sh, int n, int* s_scan, Count count) {
  int acc = 0;
  for (int c0 = 0; c0 < n; c0 += blockDim.x) {
    const int i = c0 + static_cast<int>(threadIdx.x);
    int total;
    const int ex = block_exclusive_scan(i < n ? count(i) : 0, &total, s_scan);
    if (i < n) sh.off[i] = acc + ex;
    acc += total;
  }
  if (threadIdx.x == 0) sh.off[n] = acc;
  __syncthreads();
  return acc;
}

// The columns of a tile list's n-tiles: up to three matrices (Q, K, V), each
// a run of columns [c0, c1) cut into tiles of `step`.
struct ColSet {
  int c0[3], c1[3], nt[3], step;
  SVL_DEVINL int total() const { return nt[0] + nt[1] + nt[2]; }
  SVL_DEVINL void set(int mat, int a, int b) {
    c0[mat] = a;
    c1[mat] = b;
    nt[mat] = (b - a + step - 1) / step;
  }
  // n-tile ni as (n0, ncols | mat << 16)
  SVL_DEVINL int2 tile(int ni) const {
    const int mat = ni < nt[0] ? 0 : (ni < nt[0] + nt[1] ? 1 : 2);
    const int k = ni - (mat > 0 ? nt[0] : 0) - (mat > 1 ? nt[1] : 0);
    const int a = mat == 0 ? c0[0] : (mat == 1 ? c0[1] : c0[2]), b = mat == 0 ? c1[0] : (mat == 1 ? c1[1] : c1[2]);
    const int n0 = a + k * step;
    return make_int2(n0, min(step, b - n0) | (mat << 16));
  }
};

// Writes the tiles of the block's runs from list index `base` on, each run's
// mt x nt tiles in raster bands. mband > 0: bands of `mband` m-tiles, each
// sweeping all n-tiles while its input rows stay in L2 (the tiles of one n-tile
// follow each other, so concurrent CTAs share its weights too). Otherwise bands
// of `nband` n-tiles, each sweeping all m-tiles while its weight columns stay
// in L2. `kmask`: tiles carry their run's key as the K mask. All tiles of all
// runs are written by one flat loop over the block's threads (a binary search
// finds a tile's run). Returns the number of tiles.
__device__ int emit_runs(ListShared& sh, int nrun, int4* tiles, int base, int cap, const ColSet& cs, bool kmask,
                         uint32_t* status, int* s_scan, int nband, int mband) {
  const int n_nt = cs.total();
  const int total = prefix_offsets(
      sh, nrun, s_scan, [&](int i) { return ((sh.r1[i] - sh.r0[i] + kBM_SCHED - 1) / kBM_SCHED) * n_nt; });
  for (int t = threadIdx.x; t < total; t += blockDim.x) {
    int lo = 0, hi = nrun;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (sh.off[mid] <= t) lo = mid; else hi = mid;
    }
    const int u = t - sh.off[lo], r0 = sh.r0[lo], r1 = sh.r1[lo];
    const int mt = (r1 - r0 + kBM_SCHED - 1) / kBM_SCHED;
    int mi, ni;
    if (mband > 0) {
      const int band = u / (mband * n_nt);
      const int rem = u - band * mband * n_nt;
      const int bh = min(mband, mt - band * mband);
      ni = rem / bh;
      mi = band * mband + rem % bh;
    } else {
      const int band = u / (mt * nband);
      const int rem = u - band * mt * nband;
      const int bw = min(nband, n_nt - band * nband);
      mi = rem / bw;
      ni = band * nband + rem % bw;
    }
    const int m0 = r0 + mi * kBM_SCHED;
    const int idx = base + t;
    if (idx >= cap) {
      report(status, SVL_DEV_BAD_INDEX);
      continue;
    }
    const int2 n = cs.tile(ni);
    tiles[idx] = make_int4(m0, min(m0 + kBM_SCHED, r1), n.x, n.y | (kmask ? static_cast<int>(sh.key[lo]) << 24 : 0));
  }
  __syncthreads();  // off, r0, r1 and key are reused by the caller
  return total;
}

// The list of CTA pairs: entries 2i and 2i + 1 are the 128-row tiles of one
// pair, which share their columns (the B operand) but need not adjoin. The
// m-tiles of all runs are numbered through, so only the last of an odd number
// has no partner (an entry without rows), and go in bands of `mband` (even)
// m-tiles, each sweeping all n-tiles. (With 256 adjoining rows to a pair, every
// run that ended in a pair's first half cost a whole pair: 16 samples with masks
// of their own, 970 rows in all, a forward of four layers 1,125 us against 920
// on single CTAs.) Returns the number of entries.
__device__ int emit_pairs(ListShared& sh, int nrun, int4* tiles, int base, int cap, const ColSet& cs, uint32_t* status,
                          int* s_scan, int mband) {
  const int n_nt = cs.total();
  const int mt =
      prefix_offsets(sh, nrun, s_scan, [&](int i) { return (sh.r1[i] - sh.r0[i] + kBM_SCHED - 1) / kBM_SCHED; });
  const int mt2 = mt + (mt & 1), total = mt2 * n_nt;
  for (int t = threadIdx.x; t < total; t += blockDim.x) {
    const int band = t / (mband * n_nt);
    const int rem = t - band * mband * n_nt;
    const int bh = min(mband, mt2 - band * mband);
    const int ni = rem / bh, mi = band * mband + rem % bh;
    const int m = min(mi, mt - 1);  // (the missing partner loads its neighbour's rows and stores none)
    int lo = 0, hi = nrun;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (sh.off[mid] <= m) lo = mid; else hi = mid;
    }
    const int m0 = sh.r0[lo] + (m - sh.off[lo]) * kBM_SCHED;
    const int idx = base + t;
    if (idx >= cap) {
      report(status, SVL_DEV_BAD_INDEX);
      continue;
    }
    const int2 n = cs.tile(ni);
    tiles[idx] = make_int4(m0, mi < mt ? min(m0 + kBM_SCHED, sh.r1[lo]) : m0, n.x, n.y);
  }
  __syncthreads();  // off, r0, r1 and key are reused by the caller
  return total;
}

// One work list of layer l: kind kListQkv / kListGateUp (N-sparse), kListO /
// kListDown (K-sparse) or kListAttn. Nothing here is walked by one thread:
// runs and offsets come from block-wide scans and every entry from the flat
// loops. (The walk by thread 0 with block barriers per run that this replaces
// took 63 us for one layer of 16 samples with mixed masks, this 6 us; the
// lists of a layer are built by separate blocks.)
__device__ void build_list(const ScheduleArgs& a, int l, int kind, int* dyn) {
  __shared__ int s_scan[32];
  __shared__ unsigned s_neq;
  const int tid = threadIdx.x, B = a.B, G = a.G;
  ListShared sh(dyn, B);
  if (tid == 0) s_neq = 0;
  __syncthreads();
  // the non-empty samples, and for every pair of adjacent groups whether
  // their on/off patterns over the samples differ
  unsigned neq = 0;
  for (int c0 = 0; c0 < B; c0 += blockDim.x) {
    const int b = c0 + tid;
    int q0 = 0, q1 = 0, mask = 0;
    if (b < B) {
      q0 = a.tokens ? b : a.cu_seqlens[b];
      q1 = a.tokens ? b + 1 : a.cu_seqlens[b + 1];
      if (l < a.P) {
        mask = (1 << G) - 1;
      } else {
        // every gate is requested before the first is looked at (G <= 8):
        // reading them one after the other cost most of a list's 5 us
        const size_t at = static_cast<size_t>(b) * a.L + l;
        const uint8_t on = a.layer_gate[at];
        uint8_t e[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) e[j] = j < G ? a.group_gate[at * G + j] : 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) mask |= (on && e[j]) ? (1 << j) : 0;
      }
    }
    const int some = q1 > q0 ? 1 : 0;
    int total;
    const int i = sh.n + block_exclusive_scan(some, &total, s_scan);
    if (some) {
      sh.cu0[i] = q0;
      sh.cu1[i] = q1;
      sh.mask[i] = static_cast<uint8_t>(mask);
      neq |= mask ^ (mask >> 1);
    }
    sh.n += total;
  }
  if (neq) atomicOr(&s_neq, neq);
  __syncthreads();
  neq = s_neq;

  if (kind == kListQkv || kind == kListGateUp) {
    // N-sparse: per block of adjacent groups with the same pattern, the
    // maximal row runs of samples where the block runs times its columns
    const bool qkv = kind == kListQkv;
    int4* tiles = qkv ? a.qkv_tiles + static_cast<size_t>(l) * a.qkv_cap : a.gu_tiles + static_cast<size_t>(l) * a.gu_cap;
    // (CTA pairs: an even number of entries, whole pairs)
    const int cap = (qkv ? a.qkv_cap : a.gu_cap) & (a.pairs ? ~1 : ~0);
    const int hq = (a.A / G) * a.dh, hk = (a.Akv / G) * a.dh;
    int off = 0;
    for (int j0 = 0; j0 < G;) {
      int j1 = j0;
      while (j1 + 1 < G && !((neq >> j1) & 1)) ++j1;
      ColSet cs{};
      cs.step = qkv ? a.qkv_step : 128;
      if (qkv) {
        cs.set(0, j0 * hq, (j1 + 1) * hq);
        cs.set(1, j0 * hk, (j1 + 1) * hk);
        cs.set(2, j0 * hk, (j1 + 1) * hk);
      } else {
        cs.set(0, j0 * (a.Di / G), (j1 + 1) * (a.Di / G));
      }
      const int nrun = find_runs(sh, j0, s_scan);
      off += a.pairs ? emit_pairs(sh, nrun, tiles, off, cap, cs, a.status, s_scan, a.mband)
                     : emit_runs(sh, nrun, tiles, off, cap, cs, false, a.status, s_scan, 0, a.mband);
      j0 = j1 + 1;
    }
    off = min(off, cap);
    if (qkv) off = split_tail(tiles, off, cap, a.nsparse_wave, a.dh, s_scan);
    if (tid == 0) (qkv ? a.qkv_count : a.gu_count)[l] = off;
  } else if (kind == kListO || kind == kListDown) {
    // K-sparse: segments of consecutive samples with the same mask, all D
    // columns; the tiles carry the mask
    const bool o = kind == kListO;
    int4* tiles = o ? a.o_tiles + static_cast<size_t>(l) * a.o_cap : a.dn_tiles + static_cast<size_t>(l) * a.dn_cap;
    const int cap = o ? a.o_cap : a.dn_cap;
    ColSet cs{};
    cs.step = 256;
    cs.set(0, 0, a.D);
    const int nrun = find_runs(sh, -1, s_scan);
    int off = emit_runs(sh, nrun, tiles, 0, cap, cs, true, a.status, s_scan, o ? kNBandO : kNBand, 0);
    off = split_k_tail(tiles, min(off, cap), cap, a.num_sms, a.ks_units,
                       a.ks_info + static_cast<size_t>(l) * 8 + (o ? 0 : 4));
    if (tid == 0) (o ? a.o_count : a.dn_count)[l] = off;
    int* ticket = a.ks_ticket + (2 * static_cast<size_t>(l) + (o ? 0 : 1)) * a.ks_ticket_ld;
    for (int i = tid; i < a.ks_ticket_ld; i += blockDim.x) ticket[i] = 0;
  } else {
    // Attention items: per active sample and active head, blocks of kAttnQ
    // queries, head by head and latest block first: the kernel takes units from
    // the front of the list, so one head's blocks run at about the same time
    // and share its keys in L2. A block's work grows with its index, so with few
    // long samples the largest units of the last heads would start last and the
    // CTAs end far apart: then the latest blocks of all heads come first, in
    // chunks of samples whose keys and values stay in L2. With many units the
    // spread at the end is small and the shared keys count for more.
    // Stage calls at LLaVA-7B / Qwen2-VL-7B widths, head by head's time over by
    // size: one sample of 2,300 rows 1.23 / 1.25, two of 3,000 1.08 / 1.12, four of
    // 2,300 1.03 / 1.09, six of 1,500 1.02 / 1.06, eight of 1,024 to 3,000 1.00 to 1.02,
    // one of 2,300 among seven short ones 1.09 / 1.06. The other way round: ten of
    // 1,024 0.99, sixteen of 769 0.96, of 2,500 0.99, one of 2,300 among 15 short
    // ones 0.95 / 0.97, 64 of 1,024 0.91; eight of 900 0.97, four of 800 0.95 / 1.00,
    // one of 900 0.91 / 0.98 (the short ones within the timer's 1 us).
    int4* items = a.attn_items + static_cast<size_t>(l) * a.attn_cap;
    const int hpg = a.A / G;
    const int total = prefix_offsets(sh, sh.n, s_scan, [&](int i) {
      return ((sh.cu1[i] - sh.cu0[i] + kAttnQ - 1) / kAttnQ) * __popc(sh.mask[i]) * hpg;
    });
    const int longest = tid < min(sh.n, kAttnSorted) ? sh.cu1[tid] - sh.cu0[tid] : 0;
    const bool sorted = __syncthreads_or(longest > kAttnLong) && sh.n <= kAttnSorted;
    if (sorted) {
      const int chunk_rows = max(static_cast<int>(kAttnChunkBytes / (4ll * a.Akv * a.dh)), 1);
      for (int i = tid; i < sh.n; i += blockDim.x) {
        sh.r0[i] = (sh.cu1[i] - sh.cu0[i] + kAttnQ - 1) / kAttnQ;  // blocks
        sh.r1[i] = __popc(sh.mask[i]) * hpg;                       // heads
        sh.key[i] = static_cast<uint8_t>(min(sh.cu0[i] / chunk_rows, 255));
      }
      __syncthreads();
    }
    for (int t = tid; t < total; t += blockDim.x) {
      int lo = 0, hi = sh.n;
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (sh.off[mid] <= t) lo = mid; else hi = mid;
      }
      const int u = t - sh.off[lo], r0 = sh.cu0[lo], r1 = sh.cu1[lo];
      const int nq = (r1 - r0 + kAttnQ - 1) / kAttnQ;
      const int hi_ = u / nq, qi = nq - 1 - (u - hi_ * nq);
      int grp = hi_ / hpg;  // the grp-th active group
      const int within = hi_ - grp * hpg;
      int j = 0;
      for (int m = sh.mask[lo]; j < G; ++j)
        if (((m >> j) & 1) && grp-- == 0) break;
      const int q0 = r0 + qi * kAttnQ;
      int at = t;
      if (sorted) {
        // before this item: earlier chunks, and of its own chunk the later
        // blocks and the same block of earlier samples
        at = hi_;
        for (int i = 0; i < sh.n; ++i) {
          const int nb = sh.r0[i], nh = sh.r1[i];
          if (sh.key[i] < sh.key[lo]) at += nb * nh;
          else if (sh.key[i] == sh.key[lo]) at += nh * (max(nb - 1 - qi, 0) + (i < lo && nb > qi ? 1 : 0));
        }
      }
      if (at < a.attn_cap) items[at] = make_int4(q0, min(q0 + kAttnQ, r1), r0, j * hpg + within);
      else report(a.status, SVL_DEV_BAD_INDEX);
    }
    if (tid == 0) {
      a.attn_count[l] = min(total, a.attn_cap);
      a.attn_next[l] = 0;
    }
  }
}

// Everything the first GEMM of a forward needs, in one launch:
//   blocks [0, n_lists * n_layers): one work list of one layer each;
//   then the V^T zeroing blocks (z_blocks per sample boundary) and the row
//   blocks (kSetupRows rows each): sums of squares of the packed rows, and
//   for a decode step first the rows themselves.
// V^T: attention reads 64-key tiles that start up to 7 keys before a sample
// and run up to 63 past its end. Those keys are masked (P = 0) but must be
// finite, and a neighbouring sample whose group is off in a layer has none
// written there, so the windows around every sample boundary are zeroed once
// per call (at b = 1 and 16 samples 10 MB instead of the whole 84 MB of V^T).
__global__ void __launch_bounds__(kSetupThreads) setup_kernel(ScheduleArgs a) {
  extern __shared__ int setup_dyn[];
  pdl_begin(false);
  int blk = blockIdx.x;
  const int n_list_blocks = a.n_lists * a.n_layers;
  if (blk < n_list_blocks) {
    // layers vary fastest: the lists needed first are built first
    const int li = blk / a.n_layers;
    build_list(a, a.l0 + blk - li * a.n_layers, (a.list_kinds >> (4 * li)) & 15, setup_dyn);
    return;
  }
  blk -= n_list_blocks;
  if (a.vt) {
    const int zb = (a.dkv + kVtRows - 1) / kVtRows, n_z = zb * (a.B + 1);
    if (blk < n_z) {
      const int b = blk / zb, v0 = (blk - b * zb) * kVtRows, rows = min(kVtRows, a.dkv - v0);
      const int c = a.cu_seqlens[b];
      const int w0 = max(c - 8, 0) >> 3, w1 = min(c + 64 + 7, a.t_pad) >> 3, nw = w1 - w0;  // 16-byte words
      for (int i = threadIdx.x; i < rows * nw; i += blockDim.x) {
        const int r = i / nw, w = i - r * nw;
        reinterpret_cast<uint4*>(a.vt + static_cast<size_t>(v0 + r) * a.t_pad)[w0 + w] = make_uint4(0, 0, 0, 0);
      }
      return;
    }
    blk -= n_z;
  }
  if (!a.ss) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = blk * kSetupRows + warp;
  __nv_bfloat16* x = a.X + static_cast<size_t>(r) * a.D;
  const uint4* src = reinterpret_cast<const uint4*>(x);
  bool bad = false;
  if (a.tokens) {
    // decode: row b is the embedding of the fed token at position cache_len[b]
    if (blk == 0 && threadIdx.x == 0) a.cu_out[0] = 0;
    if (r >= a.B) return;
    const int id = a.tokens[r], len = a.cache_len[r];
    bad = id < 0 || id >= a.V;
    if (lane == 0) {
      a.cu_out[r + 1] = r + 1;
      a.pos_out[r] = len;
      if (bad || len < 0 || len >= a.max_len) report(a.status, SVL_DEV_BAD_INDEX);
    }
    src = reinterpret_cast<const uint4*>(a.embed + static_cast<size_t>(bad ? 0 : id) * a.D);
  } else if (r >= a.cu_seqlens[a.B] || r >= a.t_cap) {
    return;
  }
  // sum of squares of the row into slot 0 of ss ([slots][ss_ld]), the other
  // slots zeroed: the first layer's fused RMSNorm reads these
  float acc = 0.f;
  for (int c = lane; c < a.D / 8; c += 32) {
    const uint4 u = bad ? make_uint4(0, 0, 0, 0) : src[c];
    if (a.tokens) reinterpret_cast<uint4*>(x)[c] = u;
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 f = unpack_bf16x2(w[i]);
      acc = fmaf(f.x, f.x, fmaf(f.y, f.y, acc));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  for (int i = lane; i < a.ss_slots; i += 32) a.ss[static_cast<size_t>(i) * a.ss_ld + r] = i == 0 ? acc : 0.f;
}

cudaError_t launch_setup(const ScheduleArgs& a, cudaStream_t s) {
  const size_t smem = list_shared_bytes(a.B);
  if (smem > 48 * 1024) {
    // per call: the attribute belongs to the current device's function
    const cudaError_t e =
        cudaFuncSetAttribute(setup_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
  }
  const int zb = a.vt ? ((a.dkv + kVtRows - 1) / kVtRows) * (a.B + 1) : 0;
  const int rows = a.ss ? ((a.tokens ? a.B : a.t_cap) + kSetupRows - 1) / kSetupRows : 0;
  const int grid = a.n_lists * a.n_layers + zb + rows;
  return grid > 0 ? launch_pdl(setup_kernel, grid, kSetupThreads, smem, s, a) : cudaSuccess;
}

// LLM-side compute controller (Sec. 3.2), one block per sample:
//   h~ = h_b^(P) + W_k2 SiLU(W_k1 PE(kappa))          (Eq. 7; h_b^(P) = the budget
//                                                     token's row after P layers)
//   logit[l - P][j] = W_h[(l - P) G + j] . h~ + c_h    (gate head)
//   group (l, j) runs if l < P or logit > 0 (sigma > 0.5; no noise at inference)
// With `project` and b < 1, the token count being committed, the fewest
// active groups of layers >= P are switched off, lowest logit first (equal
// logits: lower l * G + j first), until Eq. 8 at S = S_text + k is within
// b * C_full (Sec. 3.3 "Inference").
constexpr int kCtlThreads = 256;
__global__ void __launch_bounds__(kCtlThreads) controller_kernel(CtlArgs a) {
  extern __shared__ float ctl_smem[];
  float* ht = ctl_smem;           // [D] fused state
  float* lg = ctl_smem + a.D;     // [(L - P) * G] gate logits
  __shared__ double pe[256], hid[256];
  __shared__ int keep_groups;
  __shared__ long long n_on_sh;
  pdl_begin(false);
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int L = a.L, G = a.G, P = min(a.P, a.L), H = a.H, D = a.D;
  const int ng = (L - P) * G;
  const int row = a.cu_seqlens[b + 1] - 1;
  // e_kappa = W_k2 SiLU(W_k1 PE(kappa)), PE as Eq. 5
  if (tid < H) {
    const int half = H / 2, f = tid < half ? tid : tid - half;
    const double arg = 1000.0 * static_cast<double>(a.kappa[b]) * pow(10000.0, -2.0 * f / H);
    pe[tid] = tid < half ? sin(arg) : cos(arg);
  }
  if (tid == 0) {
    keep_groups = -1;
    n_on_sh = 0;
  }
  __syncthreads();
  if (tid < H) {
    double s = 0.0;
    for (int j = 0; j < H; ++j) s += static_cast<double>(__bfloat162float(a.kap_w1[tid * H + j])) * pe[j];
    hid[tid] = s / (1.0 + exp(-s));
  }
  __syncthreads();
  for (int d = tid; d < D; d += blockDim.x) {
    double s = row >= 0 ? static_cast<double>(__bfloat162float(a.X[static_cast<size_t>(row) * D + d])) : 0.0;
    for (int j = 0; j < H; ++j) s += static_cast<double>(__bfloat162float(a.kap_w2[static_cast<size_t>(d) * H + j])) * hid[j];
    ht[d] = static_cast<float>(s);
  }
  __syncthreads();
  // gate head: one warp per logit, lanes along D
  for (int o = warp; o < ng; o += blockDim.x / 32) {
    const __nv_bfloat16* wr = a.gate_w + static_cast<size_t>(o) * D;
    float acc = 0.f;
    for (int d = lane; d < D; d += 32) acc = fmaf(__bfloat162float(wr[d]), ht[d], acc);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (lane == 0) {
      lg[o] = acc + a.gate_c[o];
      if (a.gate_logits) a.gate_logits[static_cast<size_t>(b) * ng + o] = lg[o];
    }
  }
  __syncthreads();
  // raw gates and their count (prefix groups always on)
  int on = 0;
  for (int idx = tid; idx < L * G; idx += blockDim.x) on += (idx < P * G || lg[idx - P * G] > 0.f) ? 1 : 0;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) on += __shfl_xor_sync(0xffffffffu, on, off);
  if (lane == 0 && on) atomicAdd(reinterpret_cast<unsigned long long*>(&n_on_sh), static_cast<unsigned long long>(on));
  __syncthreads();
  uint32_t flags = 0;
  int drop = 0;
  if (a.project && a.budget[b] < 1.0f) {
    const long long D64 = D, Dkv = a.Dkv, Di = a.Di, V = a.V, G64 = G, L64 = L;
    const long long lin = 4 * D64 * D64 + 4 * D64 * Dkv + 6 * D64 * Di;
    const long long nv = a.vis_off[b + 1] - a.vis_off[b], st = a.text_len[b];
    const long long S_full = nv + st, S = st + a.k[b];
    const long long c_full = G64 * L64 * (lin * S_full + 4 * D64 * S_full * S_full) + G64 * 2 * D64 * V * S_full;
    const double limit = static_cast<double>(a.budget[b]) * static_cast<double>(c_full);
    const long long per = lin * S + 4 * D64 * S * S, lm = G64 * 2 * D64 * V * S;
    const long long n_on = n_on_sh, n_min = static_cast<long long>(P) * G;
    if (static_cast<double>(n_on * per + lm) > limit) {
      for (long long nk = n_min + tid; nk < n_on; nk += blockDim.x)
        if (static_cast<double>(nk * per + lm) <= limit) atomicMax(&keep_groups, static_cast<int>(nk));
      __syncthreads();
      if (n_on > n_min) flags |= SVL_FLAG_GROUPS_DROPPED;
      if (keep_groups < 0) flags |= SVL_FLAG_OVER_BUDGET;
      drop = static_cast<int>(n_on - (keep_groups < 0 ? n_min : keep_groups));
    }
  }
  uint8_t* go = a.group_gate + static_cast<size_t>(b) * L * G;
  for (int idx = tid; idx < L * G; idx += blockDim.x) {
    bool active = idx < P * G || lg[idx - P * G] > 0.f;
    if (active && drop > 0 && idx >= P * G) {
      const float v = lg[idx - P * G];
      int rank = 0;
      for (int j = P * G; j < L * G; ++j) {
        const float w = lg[j - P * G];
        if (w > 0.f && (w < v || (w == v && j < idx))) ++rank;
      }
      active = rank >= drop;
    }
    go[idx] = active ? 1 : 0;
  }
  __syncthreads();
  for (int l = tid; l < L; l += blockDim.x) {
    int any = 0;
    for (int j = 0; j < G; ++j) any |= go[l * G + j];
    a.layer_gate[static_cast<size_t>(b) * L + l] = any ? 1 : 0;
  }
  if (tid == 0 && a.flags) a.flags[b] |= flags;
}

void launch_controller(const CtlArgs& a, cudaStream_t s) {
  const size_t smem = sizeof(float) * (static_cast<size_t>(a.D) + static_cast<size_t>(a.L - min(a.P, a.L)) * a.G);
  static bool configured = false;
  if (!configured && smem > 48 * 1024) {
    cudaFuncSetAttribute(controller_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
    configured = true;
  }
  launch_pdl(controller_kernel, a.B, kCtlThreads, smem, s, a);
}

// ---------------------------------------------------------------- RMSNorm

// 1 / rms of a row of D values, by one warp.
SVL_DEVINL float row_inv_rms(const uint4* xv, int D, float eps, int lane) {
  float ss = 0.f;
  for (int c = lane; c < D / 8; c += 32) {
    const uint4 u = xv[c];
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 f = unpack_bf16x2(w[i]);
      ss += f.x * f.x + f.y * f.y;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  return rsqrtf(ss / static_cast<float>(D) + eps);
}

// Eight values times inv times their gains, rounded to bf16.
SVL_DEVINL uint4 norm8(const uint4 u, const uint4 gg, float inv) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
  const uint32_t q[4] = {gg.x, gg.y, gg.z, gg.w};
  uint32_t o[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = unpack_bf16x2(w[i]), h = unpack_bf16x2(q[i]);
    o[i] = pack_bf16x2(f.x * inv * h.x, f.y * inv * h.y);
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}

SVL_DEVINL void norm_row(const __nv_bfloat16* x, const __nv_bfloat16* g, __nv_bfloat16* y, int D, float eps,
                         int lane) {
  const uint4* xv = reinterpret_cast<const uint4*>(x);
  const float inv = row_inv_rms(xv, D, eps, lane);
  for (int c = lane; c < D / 8; c += 32)
    reinterpret_cast<uint4*>(y)[c] = norm8(xv[c], reinterpret_cast<const uint4*>(g)[c], inv);
}

__global__ void rmsnorm_kernel(NormArgs a) {
  pdl_begin(true);  // the LM head loads weights before it waits
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = blockIdx.x * (blockDim.x >> 5) + warp;
  const int T = a.cu_seqlens[a.B];
  if (r >= T || r >= a.t_cap) return;
  norm_row(a.X + static_cast<size_t>(r) * a.D, a.gain, a.Y + static_cast<size_t>(r) * a.D, a.D, a.eps, lane);
}

// One block per sample: the final norm of its last row, staged in shared
// memory by the whole block; every warp then sums the squares in the order of
// a single warp (a warp per row reading global memory took 10 us, all of it
// load latency). Rows B .. n_pad - 1 are zeroed.
constexpr int kFinalThreads = 256;
__global__ void __launch_bounds__(kFinalThreads) final_rows_kernel(NormArgs a) {
  extern __shared__ uint4 final_row[];  // [D / 8]
  pdl_begin(true);  // the LM head loads weights before it waits
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
  uint4* y = reinterpret_cast<uint4*>(a.Y + static_cast<size_t>(b) * a.D);
  const int r1 = b < a.B ? a.cu_seqlens[b + 1] : 0, r0 = b < a.B ? a.cu_seqlens[b] : 0;
  if (r1 <= r0) {
    for (int c = tid; c < a.D / 8; c += kFinalThreads) y[c] = make_uint4(0, 0, 0, 0);
    return;
  }
  const uint4* x = reinterpret_cast<const uint4*>(a.X + static_cast<size_t>(r1 - 1) * a.D);
  const uint4* g = reinterpret_cast<const uint4*>(a.gain);
  for (int c = tid; c < a.D / 8; c += kFinalThreads) final_row[c] = x[c];
  __syncthreads();
  const float inv = row_inv_rms(final_row, a.D, a.eps, lane);
  for (int c = tid; c < a.D / 8; c += kFinalThreads) y[c] = norm8(final_row[c], g[c], inv);
}

// W'[r][c] = W[r][c] * g[c] (a norm gain folded into the projection after it)
__global__ void fold_gain_kernel(const __nv_bfloat16* W, const __nv_bfloat16* g, __nv_bfloat16* out, int64_t rows,
                                 int cols) {
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= rows * cols) return;
  const int c = static_cast<int>(i % cols);
  out[i] = __float2bfloat16_rn(__bfloat162float(W[i]) * __bfloat162float(g[c]));
}

// flag = 0 unless every gain is exactly 1
__global__ void gain_is_one_kernel(const __nv_bfloat16* g, int n, int* flag) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    if (__bfloat162float(g[i]) != 1.f) *flag = 0;
}

cudaError_t fold_gain(const __nv_bfloat16* W, const __nv_bfloat16* g, __nv_bfloat16* out, int64_t rows, int cols,
                      cudaStream_t s) {
  const int64_t n = rows * cols;
  fold_gain_kernel<<<static_cast<unsigned>((n + 255) / 256), 256, 0, s>>>(W, g, out, rows, cols);
  return cudaGetLastError();
}

cudaError_t gain_is_one(const __nv_bfloat16* g, int n, int* flag, cudaStream_t s) {
  gain_is_one_kernel<<<(n + 255) / 256, 256, 0, s>>>(g, n, flag);
  return cudaGetLastError();
}

void launch_rmsnorm(const NormArgs& a, cudaStream_t s) {
  const int grid = (a.t_cap + 7) / 8;
  if (grid > 0) launch_pdl(rmsnorm_kernel, grid, 256, 0, s, a);
}

void launch_final_last_rows(const NormArgs& a, int n_pad, cudaStream_t s) {
  const size_t smem = 2 * static_cast<size_t>(a.D);
  if (smem > 48 * 1024)
    cudaFuncSetAttribute(final_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  launch_pdl(final_rows_kernel, n_pad, kFinalThreads, smem, s, a);
}

__global__ void selftest_wait_kernel(uint32_t* status, long long cycles) {
  __shared__ uint64_t bar;
  __shared__ int abort;
  if (threadIdx.x == 0) {
    abort = 0;
    mbar_init(&bar, 1);
    fence_barrier_init();
  }
  __syncthreads();
  if (threadIdx.x == 0 && !mbar_wait(&bar, 0, &abort, cycles)) report(status, SVL_DEV_TIMEOUT);
}

void launch_selftest_wait(uint32_t* status, long long cycles, cudaStream_t s) {
  selftest_wait_kernel<<<1, 32, 0, s>>>(status, cycles);
}

__global__ void rope_table_kernel(float2* cs, int max_seq, int dh, double theta) {
  const int half = dh / 2;
  const long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (i >= static_cast<long long>(max_seq) * half) return;
  const int f = static_cast<int>(i / max_seq), p = static_cast<int>(i % max_seq);
  const double ang = static_cast<double>(p) * pow(theta, -2.0 * f / dh);
  cs[i] = make_float2(static_cast<float>(cos(ang)), static_cast<float>(sin(ang)));
}

void launch_rope_table(float2* cs, int max_seq, int dh, double theta, cudaStream_t s) {
  const long long n = static_cast<long long>(max_seq) * (dh / 2);
  rope_table_kernel<<<static_cast<int>((n + 255) / 256), 256, 0, s>>>(cs, max_seq, dh, theta);
}

}  // namespace svl
