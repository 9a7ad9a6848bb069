// Packing (Sec. 3: S = S_text + S_vis; Sec. 3.1: kept tokens form a
// compressed contiguous sequence with positions 0..S-1). Sample b occupies
// rows cu_seqlens[b]..cu_seqlens[b+1) of X: kept visual rows in ascending
// token order, then its text rows, then (with the compute controller,
// Sec. 3.2) its budget token at position S.
#include "kernels.cuh"

namespace svl {

constexpr int kPackThreads = 512;
constexpr int kPackRows = kPackThreads / 32;  // a warp per output row

constexpr int kPackScan = 4096;  // samples up to which every gather block forms the offsets itself

// Row offsets of all samples into cu[0..B], by a whole block; `out` (or
// nullptr) gets a copy. Samples past t_cap rows are cut off and reported.
__device__ void row_offsets(const PackArgs& a, int* cu, int* out) {
  __shared__ int warp_sums[32];
  int before = 0;
  bool over = false;
  for (int b0 = 0; b0 < a.B; b0 += kPackThreads) {
    const int b = b0 + threadIdx.x;
    int rows = 0;
    if (b < a.B)
      rows = max(a.kept_off[b + 1] - a.kept_off[b], 0) + max(a.text_off[b + 1] - a.text_off[b], 0) +
             (a.tok_rows ? 1 : 0);
    int total;
    const int end = before + block_exclusive_scan(rows, &total, warp_sums) + rows;
    if (b < a.B) {
      over = over || end > a.t_cap;
      cu[b + 1] = min(end, a.t_cap);
      if (out) out[b + 1] = min(end, a.t_cap);
    }
    before += total;
  }
  if (threadIdx.x == 0) {
    cu[0] = 0;
    if (out) out[0] = 0;
  }
  if (out && over) report(a.status, SVL_DEV_BAD_INDEX);
}

__global__ void __launch_bounds__(kPackThreads) pack_offsets_kernel(PackArgs a) {
  pdl_begin(false);
  row_offsets(a, a.cu_seqlens, a.cu_seqlens);
}

// Every block forms the row offsets of all samples in shared memory (a launch
// of one thread that walked them cost 4 us before this one); the first block
// writes them out. Beyond kPackScan samples they come from their own launch.
// Bound by memory: rows in, rows out, once each.
__global__ void __launch_bounds__(kPackThreads) pack_gather_kernel(PackArgs a) {
  extern __shared__ int pack_cu[];  // [B + 1], up to kPackScan samples
  pdl_begin(a.use_projector);  // the projector GEMM loads weights before it waits
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int* cu = a.cu_seqlens;
  if (a.B <= kPackScan) {
    row_offsets(a, pack_cu, blockIdx.x == 0 ? a.cu_seqlens : nullptr);
    cu = pack_cu;
  }
  __syncthreads();
  const int r = blockIdx.x * kPackRows + warp;
  if (r >= cu[a.B]) return;
  const int b = find_sample(cu, a.B, r);
  const int i = r - cu[b];
  const int kb = a.kept_off[b + 1] - a.kept_off[b];
  if (lane == 0) a.pos[r] = i;
  const uint4* src;
  uint4* dst;
  int width;
  bool bad = false;
  if (i < kb) {
    const int j = a.kept_off[b] + i;
    const int n_b = a.vis_off[b + 1] - a.vis_off[b];
    int tok = a.kept_idx[j];
    if (tok < 0 || tok >= n_b) { bad = true; tok = 0; }
    src = reinterpret_cast<const uint4*>(a.vis + static_cast<size_t>(a.vis_off[b] + tok) * a.c_vis);
    width = a.c_vis;
    if (a.use_projector) {
      dst = reinterpret_cast<uint4*>(a.stage + static_cast<size_t>(j) * a.c_vis);
      if (lane == 0) a.row_map[j] = r;
    } else {
      dst = reinterpret_cast<uint4*>(a.X + static_cast<size_t>(r) * a.D);
    }
  } else if (a.tok_rows && i == kb + (a.text_off[b + 1] - a.text_off[b])) {
    src = reinterpret_cast<const uint4*>(a.tok_rows + static_cast<size_t>(b) * a.D);  // budget token
    dst = reinterpret_cast<uint4*>(a.X + static_cast<size_t>(r) * a.D);
    width = a.D;
  } else {
    int id = a.text_ids[a.text_off[b] + (i - kb)];
    if (id < 0 || id >= a.V) { bad = true; id = 0; }
    src = reinterpret_cast<const uint4*>(a.embed + static_cast<size_t>(id) * a.D);
    dst = reinterpret_cast<uint4*>(a.X + static_cast<size_t>(r) * a.D);
    width = a.D;
  }
  if (bad && lane == 0) report(a.status, SVL_DEV_BAD_INDEX);
  // four 16-byte pieces per lane in flight
  const int n = width / 8;
  for (int c0 = lane; c0 < n; c0 += 128) {
    uint4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (c0 + 32 * u < n) v[u] = bad ? make_uint4(0, 0, 0, 0) : src[c0 + 32 * u];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (c0 + 32 * u < n) dst[c0 + 32 * u] = v[u];
  }
}

__global__ void offsets_diff_kernel(const int* off, int* len, int B) {
  pdl_begin(false);
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < B) len[b] = off[b + 1] - off[b];
}

void launch_offsets_diff(const int* off, int* len, int B, cudaStream_t s) {
  launch_pdl(offsets_diff_kernel, (B + 255) / 256, 256, 0, s, off, len, B);
}

// One block per sample: PE(b) and the hidden layer in double, then D outputs.
__global__ void llm_budget_embed_kernel(const float* budget, const __nv_bfloat16* w1, const __nv_bfloat16* w2, int H,
                                        int D, __nv_bfloat16* out) {
  __shared__ double pe[256];
  __shared__ double hid[256];
  pdl_begin(false);
  const int b = blockIdx.x, i = threadIdx.x;
  const double bv = static_cast<double>(budget[b]);
  if (i < H) {
    const int half = H / 2;
    const int f = i < half ? i : i - half;
    const double arg = 1000.0 * bv * pow(10000.0, -2.0 * f / H);
    pe[i] = i < half ? sin(arg) : cos(arg);
  }
  __syncthreads();
  if (i < H) {
    double s = 0.0;
    for (int j = 0; j < H; ++j) s += static_cast<double>(__bfloat162float(w1[i * H + j])) * pe[j];
    hid[i] = s / (1.0 + exp(-s));
  }
  __syncthreads();
  for (int d = i; d < D; d += blockDim.x) {
    double s = 0.0;
    for (int j = 0; j < H; ++j) s += static_cast<double>(__bfloat162float(w2[static_cast<size_t>(d) * H + j])) * hid[j];
    out[static_cast<size_t>(b) * D + d] = __float2bfloat16_rn(static_cast<float>(s));
  }
}

void launch_llm_budget_embed(const float* budget, const __nv_bfloat16* w1, const __nv_bfloat16* w2, int H, int D,
                             int B, __nv_bfloat16* out, cudaStream_t s) {
  launch_pdl(llm_budget_embed_kernel, B, 256, 0, s, budget, w1, w2, H, D, out);
}

cudaError_t launch_pack_gather(const PackArgs& a, cudaStream_t s) {
  const int grid = (a.t_cap + kPackRows - 1) / kPackRows;
  // (one block at least: it writes cu_seqlens)
  return launch_pdl(pack_gather_kernel, grid > 0 ? grid : 1, kPackThreads,
                    a.B <= kPackScan ? sizeof(int) * (static_cast<size_t>(a.B) + 1) : 0, s, a);
}

bool pack_needs_offsets(int B) { return B > kPackScan; }
void launch_pack_offsets(const PackArgs& a, cudaStream_t s) {
  launch_pdl(pack_offsets_kernel, 1, kPackThreads, 0, s, a);
}

}  // namespace svl
