// Token controller (Sec. 3.1; Sec. 3.3 "Inference"): budget embedding,
// budget -> k from Eq. 8, per-sample top-k by radix select, stable compaction.
// The token scores themselves come from the tcgen05 GEMM (EPI_SCORE).
#include "kernels.cuh"

namespace svl {

// e_b = W_b2 SiLU(W_b1 PE(b)), PE(b) = [sin(1000 b w_i) | cos(1000 b w_i)],
// w_i = 10000^(-2i/H) (Eq. 5; `omega`, kept by the model: a double-precision
// pow per call took 2 us). One block per sample. The argument reaches 1000 rad,
// so it is formed and reduced to [-pi, pi] in double precision before the
// single-precision sine and cosine (error about 1e-7 either way); the two H x H
// products run in fp32 from shared memory, four threads per output.
constexpr double kTwoPi = 6.283185307179586;
constexpr int kFrontThreads = 256;

SVL_DEVINL void budget_matvec(const __nv_bfloat16* w, const float* x, int H, float* y, bool silu) {
  const int i = threadIdx.x, part = i & 3;
  for (int o0 = 0; o0 < H; o0 += kFrontThreads / 4) {
    const int o = o0 + i / 4;
    float s = 0.f;
    if (o < H) {
#pragma unroll 8
      for (int j = part; j < H; j += 4) s = fmaf(__bfloat162float(w[o * H + j]), x[j], s);
    }
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    if (o < H && part == 0) y[o] = silu ? s / (1.f + expf(-s)) : s;
  }
}

__global__ void budget_omega_kernel(double* omega, int H) {
  const int f = threadIdx.x;
  if (f < H / 2) omega[f] = pow(10000.0, -2.0 * f / H);
}

void launch_budget_omega(double* omega, int H, cudaStream_t s) { budget_omega_kernel<<<1, 128, 0, s>>>(omega, H); }

// Eq. 8 for one sample, times G so that it is an exact integer.
struct CostModel {
  long long lin, D4, lm, GL;
  SVL_DEVINL CostModel(const SelectArgs& a)
      : lin(4 * a.D * a.D + 4 * a.D * a.Dkv + 6 * a.D * a.Di), D4(4 * a.D), lm(a.G * 2 * a.D * a.V),
        GL(static_cast<long long>(a.G) * a.L) {}
  SVL_DEVINL long long cost(long long n_on, long long S) const { return n_on * (lin * S + D4 * S * S) + lm * S; }
};

// Blocks 0 .. B-1: the budget embedding of a sample. Blocks B .. 2B-1, when the
// counts do not depend on the scores (`counts`: gates given): k and the flags of
// a sample, beside the score GEMM instead of after it. (One block for all
// samples with a thread each took 10 us for 64 samples.)
__global__ void __launch_bounds__(kFrontThreads) front_kernel(FrontArgs f) {
  extern __shared__ __align__(16) uint8_t front_smem[];
  __shared__ float pe[256];
  __shared__ float hid[256];
  const int b = blockIdx.x, i = threadIdx.x, H = f.H;
  __nv_bfloat16* sw1 = reinterpret_cast<__nv_bfloat16*>(front_smem);
  __nv_bfloat16* sw2 = sw1 + H * H;
  pdl_begin(true);  // the score GEMM loads its operands before it waits
  if (b < f.B) {
    // (after the wait: the launch before may be the caller's update of these weights)
    if (f.w_vec) {
      for (int c = i; c < H * H / 8; c += kFrontThreads) {
        reinterpret_cast<uint4*>(sw1)[c] = reinterpret_cast<const uint4*>(f.w1)[c];
        reinterpret_cast<uint4*>(sw2)[c] = reinterpret_cast<const uint4*>(f.w2)[c];
      }
    } else {
      for (int c = i; c < H * H; c += kFrontThreads) {
        sw1[c] = f.w1[c];
        sw2[c] = f.w2[c];
      }
    }
    if (i < H) {
      const int half = H / 2;
      const double arg = 1000.0 * static_cast<double>(f.budget[b]) * f.omega[i < half ? i : i - half];
      const float r = static_cast<float>(arg - rint(arg / kTwoPi) * kTwoPi);
      pe[i] = i < half ? sinf(r) : cosf(r);
    }
    __syncthreads();
    budget_matvec(sw1, pe, H, hid, true);
    __syncthreads();
    budget_matvec(sw2, hid, H, f.e_b + static_cast<size_t>(b) * H, false);
    return;
  }
  const SelectArgs& a = f.sel;
  const int s = b - f.B;
  __shared__ int on_groups, best_k;
  if (i == 0) {
    on_groups = 0;
    best_k = -1;
  }
  __syncthreads();
  const int n = max(0, a.vis_off[s + 1] - a.vis_off[s]);
  const int kc = a.keep_count ? a.keep_count[s] : -1;
  const long long st = a.text_len[s];
  const double budget = static_cast<double>(a.budget[s]);
  const uint8_t* lg = a.layer_gate + static_cast<size_t>(s) * a.L;
  const uint8_t* gg = a.group_gate + static_cast<size_t>(s) * a.L * a.G;
  int on = 0;  // active (layer, group) pairs
  for (int idx = i; idx < a.L * a.G; idx += kFrontThreads) {
    const int l = idx / a.G;
    on += (l < a.P || (gg[idx] && lg[l])) ? 1 : 0;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) on += __shfl_xor_sync(0xffffffffu, on, o);
  if ((i & 31) == 0 && on) atomicAdd(&on_groups, on);
  __syncthreads();
  const CostModel cm(a);
  const double limit = budget * static_cast<double>(cm.cost(cm.GL, n + st));
  // the cost grows with k, so the feasible counts are a prefix: take the largest
  int mine = -1;
  for (int kk = i; kk <= n; kk += kFrontThreads)
    if (static_cast<double>(cm.cost(on_groups, st + kk)) <= limit) mine = kk;
  mine = __reduce_max_sync(0xffffffffu, mine);
  if ((i & 31) == 0 && mine >= 0) atomicMax(&best_k, mine);
  __syncthreads();
  if (i == 0) {
    a.k_out[s] = kc >= 0 ? min(kc, n) : max(best_k, 0);
    if (a.flags) a.flags[s] = (kc < 0 && best_k < 0) ? SVL_FLAG_OVER_BUDGET : 0;
  }
}

void launch_front(const FrontArgs& f, cudaStream_t s) {
  const size_t smem = 2 * sizeof(__nv_bfloat16) * static_cast<size_t>(f.H) * f.H;
  if (smem > 40 * 1024)
    cudaFuncSetAttribute(front_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  launch_pdl(front_kernel, f.B * (f.counts ? 2 : 1), kFrontThreads, smem, s, f);
}

// Orderable key: unsigned comparison of keys matches float comparison.
SVL_DEVINL uint32_t order_key(float z) {
  if (z == 0.0f) z = 0.0f;  // -0 and +0 are equal logits
  const uint32_t u = __float_as_uint(z);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Selection of one sample by a whole block: the k largest logits of z[0..n)
// (equal logits: lower index first), as ascending indices to out. The keys are
// read once, into shared memory while they fit (kKeysShared).
constexpr int kKeysShared = 4096;

SVL_DEVINL void load_keys(const float* z, int n, uint32_t* skeys) {
  if (n <= kKeysShared)
    for (int i = threadIdx.x; i < n; i += blockDim.x) skeys[i] = order_key(z[i]);
}

// (skeys: load_keys of the same logits)
__device__ void top_k(const float* z, int n, int k, int* out, const uint32_t* skeys) {
  __shared__ int hist[256];
  __shared__ int warp_sums[32];
  __shared__ int s_prefix_cnt[3];
  const int tid = threadIdx.x, lane = tid & 31;
  if (k == 0) return;
  if (k >= n) {
    for (int i = tid; i < n; i += blockDim.x) out[i] = i;
    return;
  }
  const bool shared = n <= kKeysShared;
  auto key_at = [&](int i) -> uint32_t { return shared ? skeys[i] : order_key(z[i]); };

  // ---- radix select of the k-th largest key, 8 bits per pass, MSB first
  uint32_t prefix = 0, mask = 0;
  int remaining = k;  // keys still to take among those matching `prefix`
  for (int shift = 24; shift >= 0; shift -= 8) {
    for (int i = tid; i < 256; i += blockDim.x) hist[i] = 0;
    __syncthreads();
    // logits share their leading digits: the lanes of a warp with the same one
    // count together (32 atomics on one address made a pass 2 us)
    for (int base = 0; base < n; base += blockDim.x) {
      const int i = base + tid;
      const uint32_t key = i < n ? key_at(i) : 0;
      const bool in = i < n && (key & mask) == prefix;
      const int digit = in ? static_cast<int>((key >> shift) & 0xFF) : -1;
      const unsigned same = __match_any_sync(0xffffffffu, digit);
      if (in && lane == __ffs(same) - 1) atomicAdd(&hist[digit], __popc(same));
    }
    __syncthreads();
    if (tid < 32) {
      // warp 0: counts above each digit (suffix sums from 255 down), then the
      // largest digit d whose keys with digit >= d reach `remaining`
      int cnt[8], sum = 0;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        cnt[u] = hist[255 - (tid * 8 + u)];  // lane t holds digits 255-8t .. 248-8t
        sum += cnt[u];
      }
      int incl = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (tid >= o) incl += y;
      }
      int above = incl - sum;  // keys with a digit above this lane's first digit
      int found = -1, found_above = 0;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (found < 0 && above + cnt[u] >= remaining) {
          found = 255 - (tid * 8 + u);
          found_above = above;
        }
        above += cnt[u];
      }
      const unsigned ballot = __ballot_sync(0xffffffffu, found >= 0);
      const int first = ballot ? __ffs(ballot) - 1 : 31;
      const int d = __shfl_sync(0xffffffffu, found, first);
      const int ab = __shfl_sync(0xffffffffu, found_above, first);
      if (tid == 0) {
        s_prefix_cnt[0] = d < 0 ? 0 : d;
        s_prefix_cnt[1] = remaining - (d < 0 ? 0 : ab);
        s_prefix_cnt[2] = hist[d < 0 ? 0 : d];
      }
    }
    __syncthreads();
    prefix |= static_cast<uint32_t>(s_prefix_cnt[0]) << shift;
    mask |= 0xFFu << shift;
    remaining = s_prefix_cnt[1];
    if (s_prefix_cnt[2] == remaining) break;  // every key with this prefix is kept: lower digits do not matter
  }
  const uint32_t tau = prefix;  // the digits read so far of the k-th largest key
  // keys > tau (in these digits) are kept; of the keys == tau, the `remaining` lowest indices

  // ---- ordered pass: per chunk the ranks of equal keys and the output
  // positions by index from one scan of both counts (16 bits each: a chunk has
  // at most 1,024 keys)
  int eq_before = 0, kept_before = 0;
  for (int base = 0; base < n; base += blockDim.x) {
    const int i = base + tid;
    const uint32_t key = i < n ? key_at(i) & mask : 0;
    const int gt = (i < n && key > tau) ? 1 : 0, eq = (i < n && key == tau) ? 1 : 0;
    int total;
    const int ex = block_exclusive_scan(gt | (eq << 16), &total, warp_sums);
    const int eq_rank = eq_before + (ex >> 16);
    // kept before this key: the greater ones and the equal ones taken so far
    const int pos = kept_before + (ex & 0xFFFF) + min(eq_rank, remaining) - min(eq_before, remaining);
    if (gt || (eq && eq_rank < remaining)) out[pos] = i;
    const int eq_after = eq_before + (total >> 16);
    kept_before += (total & 0xFFFF) + min(eq_after, remaining) - min(eq_before, remaining);
    eq_before = eq_after;
  }
}

// One block per sample whose k is known (front_kernel): its kept offset is the
// sum of the k before it, and its indices go to their final place. Bound by the
// latency of its radix passes over shared memory. A fourth launch that moved the
// indices took 3.9 us; the controller of one 576-token sample went from 20.7 to
// 18.4 us, of 64 samples from 33.5 to 28.9 us.
__global__ void __launch_bounds__(kSelectThreads) topk_kernel(int B, const float* scores, const int* vis_off,
                                                              const int* k, int* kept_off, int* kept_idx) {
  __shared__ uint32_t topk_keys[kKeysShared];
  __shared__ int off;
  pdl_begin(false);
  const int b = blockIdx.x, tid = threadIdx.x, v0 = vis_off[b], n = max(0, vis_off[b + 1] - v0), kb = k[b];
  if (tid == 0) off = 0;
  int part = 0;
  for (int i = tid; i < b; i += kSelectThreads) part += k[i];
  load_keys(scores + v0, n, topk_keys);
  __syncthreads();
  part = __reduce_add_sync(0xffffffffu, part);
  if ((tid & 31) == 0 && part) atomicAdd(&off, part);
  __syncthreads();
  if (tid == 0) {
    kept_off[b] = off;
    if (b == B - 1) kept_off[B] = off + kb;
  }
  top_k(scores + v0, n, kb, kept_idx + off, topk_keys);
}

void launch_topk(int B, const float* scores, const int* vis_off, const int* k, int* kept_off, int* kept_idx,
                 cudaStream_t s) {
  launch_pdl(topk_kernel, B, kSelectThreads, 0, s, B, scores, vis_off, k, kept_off, kept_idx);
}

// One block per sample, for the rules whose k depends on the scores: k, then
// the k largest logits (ties: lower index), written in ascending index order to
// kept_local[vis_off[b] ...].
//
// Under the paper's own rule (a.gate_logits set; Sec. 3.1 and Sec. 3.3
// "Inference") the gates are the compute controller's logits > 0 (prefix
// layers always on), k is capped by the number of logits z > 0 (sigma > 0.5),
// and when no visual token fits the budget, the fewest active groups of layers
// l >= P that make it fit are switched off, lowest logit first (equal logits:
// lower (l, j) first); the projected gates are written out.
__global__ void __launch_bounds__(kSelectThreads) select_kernel(SelectArgs a) {
  __shared__ uint32_t topk_keys[kKeysShared];
  __shared__ int best_k;
  __shared__ long long n_on_sum;  // updated with 64-bit atomics
  __shared__ int n_pos, keep_groups;
  __shared__ double kappa_sum;
  pdl_begin(false);

  const int b = blockIdx.x, tid = threadIdx.x;
  const int v0 = a.vis_off[b], v1 = a.vis_off[b + 1];
  const int n = max(0, v1 - v0);
  const long long s_text = a.text_len[b];

  // ---- k from the budget (Eq. 8, exact integers scaled by G)
  if (tid == 0) {
    n_on_sum = 0;
    best_k = -1;
    n_pos = 0;
    keep_groups = -1;
    kappa_sum = 0.0;
  }
  __syncthreads();
  const float* gl = a.gate_logits ? a.gate_logits + static_cast<size_t>(b) * a.L * a.G : nullptr;
  auto active = [&](int idx) -> bool { return idx / a.G < a.P || gl[idx] > 0.f; };
  {
    // active (layer, group) pairs of this sample; not needed (and no gates
    // given) when the gates are decided later
    int on = 0;
    if (!a.threshold_only)
      for (int idx = tid; idx < a.L * a.G; idx += blockDim.x) on += active(idx) ? 1 : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) on += __shfl_xor_sync(0xffffffffu, on, o);
    if ((tid & 31) == 0 && on) atomicAdd(reinterpret_cast<unsigned long long*>(&n_on_sum), static_cast<unsigned long long>(on));
    int pos = 0;  // logits z > 0, i.e. sigma(z) > 0.5
    for (int i = tid; i < n; i += blockDim.x) pos += a.scores[v0 + i] > 0.f ? 1 : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) pos += __shfl_xor_sync(0xffffffffu, pos, o);
    if ((tid & 31) == 0 && pos) atomicAdd(&n_pos, pos);
    if (a.kappa) {
      // survival rate kappa = sum sigma(z_i) / N that conditions the compute controller (Sec. 3.2)
      double sg = 0.0;
      for (int i = tid; i < n; i += blockDim.x) sg += 1.0 / (1.0 + exp(-static_cast<double>(a.scores[v0 + i])));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sg += __shfl_xor_sync(0xffffffffu, sg, o);
      if ((tid & 31) == 0) atomicAdd(&kappa_sum, sg);
    }
  }
  __syncthreads();
  int k;
  uint32_t flags = 0;
  const int kc = a.keep_count ? a.keep_count[b] : -1;
  if (tid == 0 && a.kappa) a.kappa[b] = n > 0 ? static_cast<float>(kappa_sum / n) : 0.f;
  if (kc >= 0) {
    k = min(kc, n);
  } else if (a.threshold_only) {
    k = n_pos;  // the compute controller decides the gates later
  } else {
    const long long D = a.D, Dkv = a.Dkv, Di = a.Di, V = a.V, G = a.G, L = a.L;
    const long long lin = 4 * D * D + 4 * D * Dkv + 6 * D * Di;
    const long long S_full = n + s_text;
    const long long c_full = G * L * (lin * S_full + 4 * D * S_full * S_full) + G * 2 * D * V * S_full;
    const double limit = static_cast<double>(a.budget[b]) * static_cast<double>(c_full);
    long long mine = -1;
    for (int kk = tid; kk <= n; kk += blockDim.x) {
      const long long S = s_text + kk;
      const long long cost = n_on_sum * (lin * S + 4 * D * S * S) + G * 2 * D * V * S;
      if (static_cast<double>(cost) <= limit) mine = max(mine, static_cast<long long>(kk));
    }
    // cost grows with k, so the feasible set is a prefix: take the max
    if (mine >= 0) atomicMax(&best_k, static_cast<int>(mine));
    __syncthreads();
    if (best_k >= 0) {
      k = min(best_k, n_pos);
    } else {
      // paper rule: no visual token fits, so head groups go. The most groups
      // that still fit with the text alone (prefix groups cannot go):
      k = 0;
      const long long n_min = static_cast<long long>(min(a.P, a.L)) * G;
      const long long per = lin * s_text + 4 * D * s_text * s_text, lm = G * 2 * D * V * s_text;
      for (long long nk = n_min + tid; nk < n_on_sum; nk += blockDim.x)
        if (static_cast<double>(nk * per + lm) <= limit) atomicMax(&keep_groups, static_cast<int>(nk));
      __syncthreads();
      if (n_on_sum > n_min) flags |= SVL_FLAG_GROUPS_DROPPED;
      const bool over = keep_groups < 0;  // even the prefix layers alone exceed the budget
      if (over) flags |= SVL_FLAG_OVER_BUDGET;
      __syncthreads();
      if (over && tid == 0) keep_groups = static_cast<int>(n_min);
    }
  }
  if (gl) {
    // projected gates: the (n_on - keep_groups) lowest-logit active groups
    // of layers >= P are off (none unless the fallback ran)
    __syncthreads();
    const int drop = keep_groups < 0 ? 0 : static_cast<int>(n_on_sum) - keep_groups;
    uint8_t* go = a.group_gate_out + static_cast<size_t>(b) * a.L * a.G;
    for (int idx = tid; idx < a.L * a.G; idx += blockDim.x) {
      bool on = active(idx);
      if (on && drop > 0 && idx >= a.P * a.G) {
        const float v = gl[idx];
        int rank = 0;
        for (int j = a.P * a.G; j < a.L * a.G; ++j)
          if (active(j) && (gl[j] < v || (gl[j] == v && j < idx))) ++rank;
        on = rank >= drop;
      }
      go[idx] = on ? 1 : 0;
    }
    __syncthreads();
    for (int l = tid; l < a.L; l += blockDim.x) {
      int any = 0;
      for (int j = 0; j < a.G; ++j) any |= go[l * a.G + j];
      a.layer_gate_out[static_cast<size_t>(b) * a.L + l] = any ? 1 : 0;
    }
  }
  if (tid == 0) {
    a.k_out[b] = k;
    if (a.flags) a.flags[b] = flags;
  }

  load_keys(a.scores + v0, n, topk_keys);
  top_k(a.scores + v0, n, k, a.kept_local + v0, topk_keys);
}

// Compacts the per-sample kept lists: kept_off[b] = k_0 + ... + k_{b-1}.
__global__ void compact_kernel(int B, const int* vis_off, const int* k, const int* kept_local, int* kept_idx,
                               int* kept_off) {
  __shared__ int off;
  pdl_begin(false);
  const int b = blockIdx.x;
  if (threadIdx.x == 0) off = 0;
  __syncthreads();
  int part = 0;  // k of the samples before b, summed by all threads
  for (int i = threadIdx.x; i < b; i += blockDim.x) part += k[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if ((threadIdx.x & 31) == 0 && part) atomicAdd(&off, part);
  __syncthreads();
  if (threadIdx.x == 0) {
    kept_off[b] = off;
    if (b == B - 1) kept_off[B] = off + k[b];
  }
  const int kb = k[b];
  const int* src = kept_local + vis_off[b];
  for (int i = threadIdx.x; i < kb; i += blockDim.x) kept_idx[off + i] = src[i];
}

void launch_select(const SelectArgs& a, int B, cudaStream_t s) {
  launch_pdl(select_kernel, B, kSelectThreads, 0, s, a);
}

void launch_compact(int B, const int* vis_off, const int* k, const int* kept_local, int* kept_idx, int* kept_off,
                    cudaStream_t s) {
  launch_pdl(compact_kernel, B, 256, 0, s, B, vis_off, k, kept_local, kept_idx, kept_off);
}

}  // namespace svl
