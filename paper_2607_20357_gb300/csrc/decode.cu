// Gated decode with a KV cache: one new token per sample and step, under the
// sample's prefill gates (Sec. 3.2: a gated-off head group has no keys or
// values to cache and nothing to compute; a skipped layer is bypassed). The
// paper leaves decode open (Sec. 5); the projections and the MLP run on the
// same gated tcgen05 GEMMs as the prefill with one row per sample.
//
// Cache layout (caller-owned): K then V, each [L][B][max_len][A_kv * d_head]
// bf16, position p of sample b at row p. Only the columns of KV heads of
// active groups are written and read.
#include "kernels.cuh"

namespace svl {

// Prefill: rows of the packed K [t_cap, dkv] and V^T [dkv, t_pad] of one
// layer to the cache at each row's position. 32 x 32 tiles through shared
// memory so that both the V^T reads and the cache writes are coalesced.
__global__ void kv_store_kernel(KvArgs a) {
  __shared__ __nv_bfloat16 tile[32][33];
  pdl_begin(false);
  const int T = a.cu_seqlens[a.B];
  const int r0 = blockIdx.x * 32, c0 = blockIdx.y * 32;  // packed rows, kv columns
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8 threads
  // K: row-major already, copy row by row
  for (int i = ty; i < 32; i += 8) {
    const int r = r0 + i, c = c0 + tx;
    if (r < T && c < a.dkv) {
      const int b = find_sample(a.cu_seqlens, a.B, r);
      const int p = a.pos[r];
      if (p >= 0 && p < a.max_len)
        a.k_cache[(static_cast<size_t>(b) * a.max_len + p) * a.dkv + c] = a.k[static_cast<size_t>(r) * a.dkv + c];
    }
  }
  // V: read 32 columns of V^T (rows c) x 32 keys, write transposed
  for (int i = ty; i < 32; i += 8) {
    const int c = c0 + i, r = r0 + tx;
    tile[i][tx] = (c < a.dkv && r < T) ? a.vt[static_cast<size_t>(c) * a.t_pad + r] : __float2bfloat16(0.f);
  }
  __syncthreads();
  for (int i = ty; i < 32; i += 8) {
    const int r = r0 + i, c = c0 + tx;
    if (r < T && c < a.dkv) {
      const int b = find_sample(a.cu_seqlens, a.B, r);
      const int p = a.pos[r];
      if (p >= 0 && p < a.max_len) a.v_cache[(static_cast<size_t>(b) * a.max_len + p) * a.dkv + c] = tile[tx][i];
    }
  }
}

void launch_kv_store(const KvArgs& a, int t_cap, cudaStream_t s) {
  const dim3 grid((t_cap + 31) / 32, (a.dkv + 31) / 32);
  if (grid.x > 0) launch_pdl(kv_store_kernel, grid, 256, 0, s, a);
}

// Attention of the new tokens: each query head of an active group against the
// cached keys 0..len-1 and the token's own key (position len), softmax in
// float32, output row of O. The positions form kRuns contiguous runs, each
// walked by one warp 32 at a time: lane j scores key j on its own (one chain
// over the head's dimensions), the warp folds the 32 scores into its online
// softmax, then every lane accumulates its d_head / 32 output dimensions over
// the 32 V rows in order. The runs are merged in order at the end.
// Memory-bound on the cache (2 * (len + 1) * d_head * 2 bytes per KV head), so
// what matters is that rows are read whole and many at a time. With a key's
// row read by one lane, 16 bytes at a time, and a block per query head also under
// GQA, a decode step of 16 samples of about 350 rows took 642 us (555 now, with the
// argmax and the final norm below) and one of a single 1,900-row sample with seven
// heads per KV head 979 us (712; both over four layers, with their GEMMs):
//  - d_head / 8 lanes copy a K row with 16 bytes each into a swizzled tile in
//    shared memory, from which the lanes read their own rows (a lane reading
//    its row straight from global memory touches 32 lines per instruction);
//  - one query head per KV head: a block per head, a warp per run, and the V
//    rows are requested into registers before the scores are formed;
//  - several (GQA): a cluster of kRuns blocks per KV head, a block per run, a
//    warp per query head, so the cache is read once for all of them; 32 or 128
//    positions at a time (the score chains of four tiles side by side; the rule
//    is at launch_dec) while the next ones load, and the runs meet through
//    distributed shared memory.
constexpr int kRuns = 8;
constexpr int kDecThreads = kRuns * 32;

SVL_DEVINL void cp_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(smem)), "l"(gmem) : "memory");
}
SVL_DEVINL void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
SVL_DEVINL void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Whether head group g of sample b runs in this layer.
SVL_DEVINL bool dec_group_on(const DecAttnArgs& a, int b, int g) {
  return a.l < a.P || (a.layer_gate[b * a.L + a.l] && a.group_gate[(static_cast<size_t>(b) * a.L + a.l) * a.G + g]);
}

// One run's softmax state: the running max, the row sum and this lane's
// d_head / 32 output dimensions.
template <int PER>
struct RunState {
  float m = -INFINITY, l = 0.f, o[PER];
};

// Scores of key `lane` of KT consecutive K tiles (`pitch` bytes apart) against
// sq (q * scale): one chain over the dimensions per tile, the tiles' chains side
// by side, operands read four 16-byte chunks at a time so that only the first
// read's latency is exposed.
template <int DH, int KT>
SVL_DEVINL void tile_scores(const uint8_t* ktile, int pitch, const float* sq, int lane, float* acc) {
  const uint8_t* row = ktile + lane * DH * 2;
  const int sw = (lane & 7) << 4;
  constexpr int CB = KT > 1 ? 4 : 8;  // chunks per batch
#pragma unroll
  for (int t = 0; t < KT; ++t) acc[t] = 0.f;
#pragma unroll
  for (int c0 = 0; c0 < DH / 8; c0 += CB) {
    uint4 u[KT][CB];
#pragma unroll
    for (int t = 0; t < KT; ++t)
#pragma unroll
      for (int c = 0; c < CB; ++c)
        u[t][c] = *reinterpret_cast<const uint4*>(row + t * pitch + (((c0 + c) << 4) ^ sw));
#pragma unroll
    for (int c = 0; c < CB; ++c) {
      const float4 q0 = *reinterpret_cast<const float4*>(sq + 8 * (c0 + c));
      const float4 q1 = *reinterpret_cast<const float4*>(sq + 8 * (c0 + c) + 4);
#pragma unroll
      for (int t = 0; t < KT; ++t) {
        const float2 k0 = unpack_bf16x2(u[t][c].x), k1 = unpack_bf16x2(u[t][c].y), k2 = unpack_bf16x2(u[t][c].z),
                     k3 = unpack_bf16x2(u[t][c].w);
        float s = acc[t];
        s = fmaf(q0.x, k0.x, s);
        s = fmaf(q0.y, k0.y, s);
        s = fmaf(q0.z, k1.x, s);
        s = fmaf(q0.w, k1.y, s);
        s = fmaf(q1.x, k2.x, s);
        s = fmaf(q1.y, k2.y, s);
        s = fmaf(q1.z, k3.x, s);
        acc[t] = fmaf(q1.w, k3.y, s);
      }
    }
  }
}

SVL_DEVINL float warp_max(float x) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, off));
  return x;
}
SVL_DEVINL float warp_sum(float x) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
  return x;
}

// Folds a tile's 32 scores into the run's max and row sum, given their max
// over the warp; returns this lane's probability (0 where not `in`).
template <int PER>
SVL_DEVINL float fold_scores(RunState<PER>& r, float sc, float mx, bool in) {
  const float mn = fmaxf(r.m, mx);
  const float e = in ? __expf(sc - mn) : 0.f;
  const float es = warp_sum(e);
  const float corr = __expf(r.m - mn);  // 0 while m is -inf
  r.l = r.l * corr + es;
#pragma unroll
  for (int i = 0; i < PER; ++i) r.o[i] *= corr;
  r.m = mn;
  return e;
}

// PER packed bf16 values of a row.
template <int PER>
SVL_DEVINL uint2 row_part(const void* p) {
  if constexpr (PER == 4) return *reinterpret_cast<const uint2*>(p);
  else return make_uint2(*reinterpret_cast<const uint32_t*>(p), 0u);
}

// O += probability times this lane's dimensions (packed bf16, from row(j)) for
// the rows j < n of a tile, eight at a time without branches between them: the
// rows past n of the last eight count as zeros.
template <int PER, class Row>
SVL_DEVINL void fold_rows(RunState<PER>& r, float e, int n, Row row) {
#pragma unroll
  for (int j0 = 0; j0 < 32; j0 += 8) {
    if (j0 >= n) break;
    float ej[8];
    uint2 w[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      ej[j] = __shfl_sync(0xffffffffu, e, j0 + j);
      w[j] = row(j0 + j);
      if (j0 + j >= n) {
        ej[j] = 0.f;
        w[j] = make_uint2(0, 0);
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float2 v0 = unpack_bf16x2(w[j].x);
      r.o[0] = fmaf(ej[j], v0.x, r.o[0]);
      r.o[1] = fmaf(ej[j], v0.y, r.o[1]);
      if constexpr (PER == 4) {
        const float2 v1 = unpack_bf16x2(w[j].y);
        r.o[2] = fmaf(ej[j], v1.x, r.o[2]);
        r.o[3] = fmaf(ej[j], v1.y, r.o[3]);
      }
    }
  }
}

// One query head per KV head: block (b, head), warp = run.
template <int DH>
__global__ void __launch_bounds__(kDecThreads, 2) decode_attn_kernel(DecAttnArgs a) {
  constexpr int PER = DH / 32, CH = DH / 8;  // dimensions per lane, 16-byte chunks per row
  extern __shared__ __align__(128) uint8_t dec_smem[];  // K tiles [kRuns][32 rows]
  __shared__ __align__(16) float sq[DH];                // q * scale
  __shared__ __align__(16) __nv_bfloat16 snv[DH];       // the new value row
  __shared__ float sm_m[kRuns], sm_l[kRuns];
  __shared__ float sm_o[kRuns][DH];
  pdl_begin(a.late);
  const int b = blockIdx.x, h = blockIdx.y;
  if (!dec_group_on(a, b, h / (a.A / a.G))) return;  // gated off: no keys, no values, no output
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
  const int len = a.cache_len[b];
  if (len < 0 || len >= a.max_len) {
    // full (or corrupt) cache, reported by setup_kernel: the head's output is
    // zero, so the step's logits for this sample are defined, and nothing is
    // appended
    if (tid < DH) a.out[static_cast<size_t>(b) * a.ldo + h * DH + tid] = __float2bfloat16(0.f);
    return;
  }
  const __nv_bfloat16* knew = a.k + static_cast<size_t>(b) * a.dkv + h * DH;
  const size_t cbase = static_cast<size_t>(b) * a.max_len * a.dkv + static_cast<size_t>(h) * DH;
  const int n = len + 1, per_run = (n + kRuns - 1) / kRuns;
  const int p_begin = warp * per_run, p_end = min(n, p_begin + per_run);
  uint8_t* ktile = dec_smem + warp * 32 * DH * 2;
  uint2 vv[32];
  // requests the K tile and this lane's part of the V rows of positions
  // [p0, p0 + 32) of the run (the new token's V row comes from snv), eight V
  // rows at a time as far as the run goes
  const __nv_bfloat16* kc = a.k_cache + cbase + (lane % CH) * 8;
  const __nv_bfloat16* vc = a.v_cache + cbase + lane * PER;
  auto request_k = [&](int p0) {
    constexpr int RI = 32 / CH;  // rows per instruction
#pragma unroll
    for (int it = 0; it < CH; ++it) {
      const int row = it * RI + lane / CH, p = p0 + row;
      if (p < p_end)
        cp_async16(ktile + row * DH * 2 + (((lane % CH) ^ (row & 7)) << 4),
                   p < len ? kc + static_cast<size_t>(p) * a.dkv : knew + (lane % CH) * 8);
    }
    cp_async_commit();
  };
  auto request_v = [&](int p0) {
    const int cached = min(p_end, len) - p0;
#pragma unroll
    for (int j0 = 0; j0 < 32; j0 += 8) {
      if (j0 >= cached) break;
#pragma unroll
      for (int j = j0; j < j0 + 8; ++j)  // rows past the cached ones repeat the last: never used
        vv[j] = row_part<PER>(vc + static_cast<size_t>(p0 + min(j, cached - 1)) * a.dkv);
    }
  };
  request_k(p_begin);
  request_v(p_begin);
  if (tid < DH) {
    sq[tid] = __bfloat162float(a.q[static_cast<size_t>(b) * a.ldq + h * DH + tid]) * a.scale;
    const __nv_bfloat16 vnew = a.vt[static_cast<size_t>(h * DH + tid) * a.t_pad + b];
    snv[tid] = vnew;
    // append the new key and value to the cache
    const size_t at = (static_cast<size_t>(b) * a.max_len + len) * a.dkv + h * DH + tid;
    a.k_cache[at] = knew[tid];
    a.v_cache[at] = vnew;
  }
  __syncthreads();
  RunState<PER> r;
#pragma unroll
  for (int i = 0; i < PER; ++i) r.o[i] = 0.f;
  for (int p0 = p_begin; p0 < p_end; p0 += 32) {
    cp_async_wait<0>();
    __syncwarp();
    const bool in = p0 + lane < p_end;
    float sc;
    tile_scores<DH, 1>(ktile, 0, sq, lane, &sc);
    __syncwarp();  // the tile is read before it is filled again
    if (p0 + 32 < p_end) request_k(p0 + 32);  // lands while this tile is folded
    if (!in) sc = -INFINITY;
    const float e = fold_scores<PER>(r, sc, warp_max(sc), in);
    fold_rows<PER>(r, e, min(p_end, len) - p0, [&](int j) { return vv[j]; });
    if (len >= p0 && len < p0 + 32 && len < p_end) {  // the new token, last of the last run
      const float en = __shfl_sync(0xffffffffu, e, len - p0);
      const uint2 w = row_part<PER>(snv + lane * PER);
      const float2 v0 = unpack_bf16x2(w.x), v1 = unpack_bf16x2(w.y);
      r.o[0] = fmaf(en, v0.x, r.o[0]);
      r.o[1] = fmaf(en, v0.y, r.o[1]);
      if constexpr (PER == 4) {
        r.o[2] = fmaf(en, v1.x, r.o[2]);
        r.o[3] = fmaf(en, v1.y, r.o[3]);
      }
    }
    if (p0 + 32 < p_end) request_v(p0 + 32);
  }
  if (lane == 0) {
    sm_m[warp] = r.m;
    sm_l[warp] = r.l;
  }
#pragma unroll
  for (int i = 0; i < PER; ++i) sm_o[warp][lane * PER + i] = r.o[i];
  __syncthreads();
  if (tid < DH) {
    float M = -INFINITY;
    for (int w = 0; w < kRuns; ++w) M = fmaxf(M, sm_m[w]);
    float L = 0.f, acc = 0.f;
    for (int w = 0; w < kRuns; ++w) {
      const float f = sm_m[w] == -INFINITY ? 0.f : __expf(sm_m[w] - M);
      L += sm_l[w] * f;
      acc += sm_o[w][tid] * f;
    }
    const float inv = L > 0.f ? 1.f / L : 0.f;
    a.out[static_cast<size_t>(b) * a.ldo + h * DH + tid] = __float2bfloat16_rn(acc * inv);
  }
}

// Several query heads per KV head: cluster of kRuns blocks, block = run, warp
// = query head; blockIdx.y = KV head times passes of kRuns query heads. A step is
// KT tiles of 32 positions (16 KB each at d_head 128); two steps in shared memory.
template <int DH, int KT>
__global__ void __launch_bounds__(kDecThreads, KT == 1 ? 3 : 1) decode_attn_gqa_kernel(DecAttnArgs a) {
  constexpr int PER = DH / 32, CH = DH / 8, TB = 32 * DH * 2;
  extern __shared__ __align__(128) uint8_t dec_smem[];  // [2][KT] of 32 K rows and 32 V rows
  __shared__ __align__(16) float sq[kRuns][DH];
  __shared__ float sm_m[kRuns], sm_l[kRuns];  // per query head, read by the cluster
  __shared__ float sm_o[kRuns][DH];
  pdl_begin(a.late);
  const int run = blockIdx.x, b = blockIdx.z;
  const int grp = a.A / a.Akv, npass = (grp + kRuns - 1) / kRuns;
  const int kvh = blockIdx.y / npass, h0 = kvh * grp + (blockIdx.y - kvh * npass) * kRuns;
  const int nh = min(kRuns, (kvh + 1) * grp - h0);
  if (!dec_group_on(a, b, h0 / (a.A / a.G))) return;  // the whole cluster
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
  const int len = a.cache_len[b];
  __nv_bfloat16* out = a.out + static_cast<size_t>(b) * a.ldo + h0 * DH;
  if (len < 0 || len >= a.max_len) {  // the whole cluster; see decode_attn_kernel
    if (run == 0)
      for (int i = tid; i < nh * DH; i += kDecThreads) out[i] = __float2bfloat16(0.f);
    return;
  }
  const __nv_bfloat16* knew = a.k + static_cast<size_t>(b) * a.dkv + kvh * DH;
  const __nv_bfloat16* vnew = a.vt + static_cast<size_t>(kvh) * DH * a.t_pad + b;
  const size_t cbase = static_cast<size_t>(b) * a.max_len * a.dkv + static_cast<size_t>(kvh) * DH;
  const int n = len + 1, per_run = (n + kRuns - 1) / kRuns;
  const int p_begin = run * per_run, p_end = min(n, p_begin + per_run);
  auto request = [&](int p0, int buf) {  // the tiles of one step into half `buf` of the ring
    uint8_t* tiles = dec_smem + buf * KT * 2 * TB;
    for (int idx = tid; idx < 32 * KT * CH; idx += kDecThreads) {
      const int row = idx / CH, c = idx % CH, p = p0 + row;
      if (p >= p_end) break;  // rows only grow
      uint8_t* kt = tiles + (row >> 5) * 2 * TB + (row & 31) * DH * 2;
      const size_t at = cbase + static_cast<size_t>(p) * a.dkv + c * 8;
      cp_async16(kt + ((c ^ (row & 7)) << 4), p < len ? a.k_cache + at : knew + c * 8);
      if (p < len) cp_async16(kt + TB + c * 16, a.v_cache + at);
    }
    cp_async_commit();
    const int jn = len - p0;  // the new token's V row (transposed in this step's V^T)
    if (jn >= 0 && jn < 32 * KT && len < p_end && tid < DH)
      reinterpret_cast<__nv_bfloat16*>(tiles + (jn >> 5) * 2 * TB + TB)[(jn & 31) * DH + tid] =
          vnew[static_cast<size_t>(tid) * a.t_pad];
  };
  request(p_begin, 0);
  for (int i = tid; i < nh * DH; i += kDecThreads)
    sq[i / DH][i % DH] = __bfloat162float(a.q[static_cast<size_t>(b) * a.ldq + h0 * DH + i]) * a.scale;
  if (run == 0 && h0 == kvh * grp && tid < DH) {  // append the new key and value to the cache
    const size_t at = (static_cast<size_t>(b) * a.max_len + len) * a.dkv + kvh * DH + tid;
    a.k_cache[at] = knew[tid];
    a.v_cache[at] = vnew[static_cast<size_t>(tid) * a.t_pad];
  }
  RunState<PER> r;
#pragma unroll
  for (int i = 0; i < PER; ++i) r.o[i] = 0.f;
  int buf = 0;
  for (int p0 = p_begin; p0 < p_end; p0 += 32 * KT) {
    cp_async_wait<0>();
    __syncthreads();  // this step's tiles have landed, and the previous step's are read
    request(p0 + 32 * KT, buf ^ 1);
    if (warp < nh) {
      const uint8_t* kt = dec_smem + buf * KT * 2 * TB;
      float sc[KT], mx[KT];
      tile_scores<DH, KT>(kt, 2 * TB, sq[warp], lane, sc);
#pragma unroll
      for (int t = 0; t < KT; ++t) {
        if (p0 + 32 * t + lane >= p_end) sc[t] = -INFINITY;
        mx[t] = warp_max(sc[t]);
      }
#pragma unroll
      for (int t = 0; t < KT; ++t) {
        const int n = p_end - (p0 + 32 * t);
        if (n <= 0) break;
        const float e = fold_scores<PER>(r, sc[t], mx[t], lane < n);
        const uint8_t* vrows = kt + t * 2 * TB + TB + lane * PER * 2;
        fold_rows<PER>(r, e, min(32, n), [&](int j) { return row_part<PER>(vrows + j * DH * 2); });
      }
    }
    buf ^= 1;
  }
  cp_async_wait<0>();
  if (warp < nh) {
    if (lane == 0) {
      sm_m[warp] = r.m;
      sm_l[warp] = r.l;
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) sm_o[warp][lane * PER + i] = r.o[i];
  }
  // merge the runs in order: every block writes d_head / kRuns dimensions
  cluster_sync();
  constexpr int DW = DH / kRuns;
  for (int i = tid; i < nh * DW; i += kDecThreads) {
    const int h = i / DW, d = run * DW + i % DW;
    float mw[kRuns], M = -INFINITY;
#pragma unroll
    for (int w = 0; w < kRuns; ++w) {
      mw[w] = ld_cluster(mapa_shared(&sm_m[h], w));
      M = fmaxf(M, mw[w]);
    }
    float L = 0.f, acc = 0.f;
#pragma unroll
    for (int w = 0; w < kRuns; ++w) {
      const float f = mw[w] == -INFINITY ? 0.f : __expf(mw[w] - M);
      L += ld_cluster(mapa_shared(&sm_l[h], w)) * f;
      acc += ld_cluster(mapa_shared(&sm_o[h][d], w)) * f;
    }
    const float inv = L > 0.f ? 1.f / L : 0.f;
    out[h * DH + d] = __float2bfloat16_rn(acc * inv);
  }
  cluster_sync();  // the others have read this block's run
}

template <int DH, int KT>
static cudaError_t launch_gqa(const DecAttnArgs& a, int kv_blocks, cudaStream_t s) {
  constexpr int ring = 2 * KT * 2 * 32 * DH * 2;
  const cudaError_t e =
      cudaFuncSetAttribute(decode_attn_gqa_kernel<DH, KT>, cudaFuncAttributeMaxDynamicSharedMemorySize, ring);
  if (e != cudaSuccess) return e;
  return launch_pdl_cluster(decode_attn_gqa_kernel<DH, KT>, dim3(kRuns, kv_blocks, a.B), kDecThreads, ring, kRuns, s,
                            a);
}

// Steps of four tiles while the rings of all blocks find room at once in 128 KB
// per SM: every block has its SM (nearly) to itself then, and what counts is how
// much of its run is in flight. With more blocks, steps of one tile: four blocks
// fit on an SM and cover each other's latency. A decode step of four layers at
// Qwen2-VL-7B widths (four KV heads), one tile / four: 1 sample of 2,000 rows
// 579 / 522 us, 4 of 1,000 542 / 536, 8 of 30 475 / 520 and of 2,000 622 / 656, 64 of
// 200 669 / 1,018, 256 of 30 1,012 / 2,244 (two tiles: 542, 507, 479, 561, 756, 1,334).
template <int DH>
static cudaError_t launch_dec(const DecAttnArgs& a, cudaStream_t s) {
  const int grp = a.A / a.Akv;
  if (grp > 1) {
    const int kv_blocks = a.Akv * ((grp + kRuns - 1) / kRuns);
    const int64_t rings = static_cast<int64_t>(kRuns) * kv_blocks * a.B * (4 * 2 * 2 * 32 * DH * 2);
    return rings <= static_cast<int64_t>(a.num_sms) * (128 << 10) ? launch_gqa<DH, 4>(a, kv_blocks, s)
                                                                  : launch_gqa<DH, 1>(a, kv_blocks, s);
  }
  constexpr int smem = kRuns * 32 * DH * 2;
  const cudaError_t e =
      cudaFuncSetAttribute(decode_attn_kernel<DH>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(decode_attn_kernel<DH>, dim3(a.B, a.A), kDecThreads, smem, s, a);
}

cudaError_t launch_decode_attn(const DecAttnArgs& a, cudaStream_t s) {
  return a.dh == 128 ? launch_dec<128>(a, s) : launch_dec<64>(a, s);
}

// Greedy next token per sample (largest logit; equal logits: lower id) and
// the cache length advanced by the fed token. A cluster of kFinSplit CTAs
// scans a sample's logits in contiguous parts (one block took 11 us for
// 152,064 logits); with V a multiple of 4 and 16-byte aligned logits (`vec`)
// each thread reads float4s (4 consecutive ids, kept in id order, so the tie
// rule holds).
constexpr int kFinThreads = 512, kFinSplit = 8;

SVL_DEVINL void arg_better(float x, int v, float& best, int& idx) {
  if (x > best || (x == best && v < idx)) {
    best = x;
    idx = v;
  }
}

__global__ void __launch_bounds__(kFinThreads) decode_finish_kernel(int B, int V, const float* logits, bool vec,
                                                                    int* next_token, int* cache_len, int max_len) {
  __shared__ float bv[kFinThreads / 32];
  __shared__ int bi[kFinThreads / 32];
  __shared__ float cta_v;
  __shared__ int cta_i;
  pdl_begin(false);
  const int b = blockIdx.y, part = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float* row = logits + static_cast<size_t>(b) * V;
  float best = -INFINITY;
  int idx = 0x7fffffff;
  if (vec) {
    const float4* r4 = reinterpret_cast<const float4*>(row);
    const int n4 = V / 4, per = (n4 + kFinSplit - 1) / kFinSplit, c1 = min(n4, (part + 1) * per);
#pragma unroll 4
    for (int c = part * per + tid; c < c1; c += kFinThreads) {
      const float4 x = r4[c];
      arg_better(x.x, 4 * c, best, idx);
      arg_better(x.y, 4 * c + 1, best, idx);
      arg_better(x.z, 4 * c + 2, best, idx);
      arg_better(x.w, 4 * c + 3, best, idx);
    }
  } else {
    const int per = (V + kFinSplit - 1) / kFinSplit, v1 = min(V, (part + 1) * per);
    for (int v = part * per + tid; v < v1; v += kFinThreads) arg_better(row[v], v, best, idx);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float ob = __shfl_xor_sync(0xffffffffu, best, off);
    const int oi = __shfl_xor_sync(0xffffffffu, idx, off);
    arg_better(ob, oi, best, idx);
  }
  if (lane == 0) {
    bv[warp] = best;
    bi[warp] = idx;
  }
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < kFinThreads / 32; ++w) arg_better(bv[w], bi[w], best, idx);
    cta_v = best;
    cta_i = idx;
  }
  cluster_sync();
  if (part == 0 && tid == 0) {
    for (int c = 1; c < kFinSplit; ++c)
      arg_better(ld_cluster(mapa_shared(&cta_v, c)),
                 __float_as_int(ld_cluster(mapa_shared(&cta_i, c))), best, idx);
    // a sample whose cache was already full took no step: its length stays
    // and it has no next token
    const int len = cache_len[b];
    const bool stepped = len >= 0 && len < max_len;
    if (next_token) next_token[b] = !stepped ? -1 : (idx == 0x7fffffff ? 0 : idx);
    if (stepped) cache_len[b] = len + 1;
  }
  cluster_sync();  // the first CTA has read the others' results
}

cudaError_t launch_decode_finish(int B, int V, const float* logits, int* next_token, int* cache_len, int max_len,
                                 cudaStream_t s) {
  // (the ABI asks for no alignment of the caller's logits beyond a float's)
  const bool vec = (V & 3) == 0 && (reinterpret_cast<uintptr_t>(logits) & 15) == 0;
  return launch_pdl_cluster(decode_finish_kernel, dim3(kFinSplit, B), kFinThreads, 0, kFinSplit, s, B, V, logits, vec,
                            next_token, cache_len, max_len);
}

}  // namespace svl
