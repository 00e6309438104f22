// FP32 GEMM on the CUDA cores (FFMA): the dense node-wise linear layers of
// the PNA convolution (message layer W_M, update layer W_U) and their weight
// and input gradients, for the full-FP32 path.
//
// Operands are "virtual": each is assembled while it is staged into shared
// memory from up to kMaxSeg segments along the feature dimension, each with an
// optional per-node scale (the degree scalers) and an optional ReLU mask (the
// backward of the update's ReLU).  So [x ; agg ; amp*agg ; att*agg] (16H
// wide) is never materialised, and a "ones" segment appends a row that
// yields bias gradients as column sums inside the weight-gradient GEMM.
//
// Tiling: 8 TM x 128 x 8 block tile (TM rows and 8 columns per thread, 128
// threads), register-staged double buffering of the shared-memory tiles.
// Split-K writes per-split partial tiles that a second kernel sums in split
// order (deterministic) and finishes with bias / ReLU.
//
// Measured (2,174 atoms, H = 200; us per launch, before: an 8 x 8 thread tile
// that looked its operands up and scaled them at each load, after): message
// 22 -> 13, update 147 -> 80, dW_U 147 -> 88, dagg 83 -> 66, dW_M 22 -> 16,
// dx 22 -> 21; the update of 64,427 atoms 3,370 -> 1,885 (44 of the 78
// TFLOP/s that plain FFMA chains reach).  ncu there: FFMA pipe 90% busy on the
// SMs that hold two CTAs throughout, 65% on average; what is left is the
// last wave and the columns past N (200 fill 6.25 of 7 warps).
#include <algorithm>
#include <mutex>

#include "kernels.cuh"

namespace gcnn {
namespace {

constexpr int BN = 128, BK = 8, kThreads = 128, kCtasPerSm = 2;
// shared-memory pitches (floats): the transposing stores of a warp (16 rows,
// two k's four rows of the tile apart) fall into 32 different banks
constexpr int kLdB = BN + 4;
constexpr int lda_of(int TM) { return 8 * TM + 4; }
constexpr int kReduceThreads = 256;
// The K-chunks of a product are part of its arithmetic (a chunk is summed in
// k order, the chunks in chunk order), so their number depends on the
// product's sizes alone and not on the tile of the kernel that runs them:
// kPlanTile and kPlanK are the plan's own units.
constexpr int kPlanTile = 128, kPlanK = 8;
// Row-invariant products: chunks of this many k's whatever the rows, so that
// one molecule's update (K = 3,200) runs in 13 CTAs and not one after the
// other (6-layer forward of one molecule: 3,377 -> 284 us).
constexpr int kInvariantChunk = 256;

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

struct Sizes {
  int M, K;
};

__device__ __forceinline__ Sizes actual_sizes(const GemmDesc &d, DevDims dims) {
  Sizes s{d.M, d.K};
  if (d.node_dim == kNodeM) s.M = min(d.M, dims.nodes(d.M));
  if (d.node_dim == kNodeK) s.K = min(d.K, dims.nodes(d.K));
  return s;
}

__device__ __forceinline__ int find_seg(const Operand &op, int f) {
  int s = 0;
#pragma unroll
  for (int q = 1; q < kMaxSeg; ++q)
    if (q < op.nseg && op.seg[q].begin <= f) s = q;
  return s;
}

// v where the mask is positive, 0 elsewhere
__device__ __forceinline__ float4 keep_positive(float4 v, float4 mk) {
  return make_float4(mk.x > 0.f ? v.x : 0.f, mk.y > 0.f ? v.y : 0.f, mk.z > 0.f ? v.z : 0.f, mk.w > 0.f ? v.w : 0.f);
}

// Two FP32 fused multiply-adds in one instruction, each rounded as fmaf:
// (c.x, c.y) += (a.x b.x, a.y b.y) on register pairs.
__device__ __forceinline__ void fma2(unsigned long long &c, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long pair(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpair(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

// Bias and ReLU of the final value, then its store (the ones row keeps only
// its first last_row_cols columns).
__device__ __forceinline__ void finish4(const GemmDesc &d, int M, int m, int n, float4 v) {
  if (d.bias) {
    v.x += (n + 0 < d.bias_n) ? d.bias[n + 0] : 0.f;
    v.y += (n + 1 < d.bias_n) ? d.bias[n + 1] : 0.f;
    v.z += (n + 2 < d.bias_n) ? d.bias[n + 2] : 0.f;
    v.w += (n + 3 < d.bias_n) ? d.bias[n + 3] : 0.f;
  }
  if (d.relu) {
    v.x = fmaxf(v.x, 0.f); v.y = fmaxf(v.y, 0.f); v.z = fmaxf(v.z, 0.f); v.w = fmaxf(v.w, 0.f);
  }
  float *c = d.C + (size_t)m * d.ldc + n;
  if (d.last_row_cols > 0 && m == M - 1) {
    const float t[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (n + q < d.last_row_cols) c[q] = t[q];
  } else {
    *reinterpret_cast<float4 *>(c) = v;
  }
}

// One BM x 128 output tile (BM = 8 TM) per CTA of four warps, one per 32
// columns; a thread holds TM x 8 sums as pairs of neighbouring rows.
//   * The kernel is bound by the FFMA pipe, with the shared-memory read port
//     (128 B per cycle and SM, whatever the broadcast) close behind: an 8 x 8
//     thread tile needs as many read cycles as FFMA cycles, 16 x 8 three
//     quarters of them; two FMAs per instruction leave the issue slots for
//     the reads and the duplicated B operands.
//   * Pointers, scales and masks of the virtual operands move along with the
//     k loop and are looked up again only where a segment begins; looked up
//     per load they took more instructions than the FMAs.  Applied at the
//     load they made each k tile wait for it; they are applied when the tile
//     is stored.
//   * Rows and columns past the end repeat the last one (their results are
//     not stored); k's past the end read as zero.
//   * Warps whose columns lie past N only help with the loads.
// CHUNKS: the CTA runs all `splits` K-chunks itself and adds their sums in
// chunk order (running totals in shared memory), the additions that the
// reduction kernel makes over partial tiles; otherwise CTA z runs chunk z.
template <int TM, bool AK, bool BNC, bool CHUNKS>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
sgemm_kernel(GemmDesc d, DevDims dims, float *__restrict__ partial, int splits, int kps) {
  pdl_entry(GCNN_K_GEMM_SIMT);
  constexpr int BM = 8 * TM, kLdA = lda_of(TM), NA = (2 * BM + kThreads - 1) / kThreads;
  __shared__ __align__(16) float As[2][BK][kLdA];
  __shared__ __align__(16) float Bs[2][BK][kLdB];
  extern __shared__ __align__(16) float4 s_tot[];  // CHUNKS: 2 TM float4 per thread
  const Sizes sz = actual_sizes(d, dims);
  const int M = sz.M, K = sz.K, N = d.N;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  if (m0 >= M) return;  // block-uniform
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ty = lane >> 2, tx = lane & 3;
  const bool active = n0 + 32 * warp < N;

  // ---- A: slot i of a thread is row a_row (K-contiguous; k's a_k .. a_k + 3)
  // or k a_k (M-contiguous; rows a_row .. a_row + 3) of the tile
  constexpr bool kMaskA = AK && !BNC, kMaskB = !AK;  // the forms that may carry a ReLU mask
  const float *pa[NA];
  int astep[NA];                    // floats to the slot's next k tile
  const float *ps[AK ? 1 : NA];     // M-contiguous: scale of the slot's next k, or null
  float sc[NA];                     // the loaded tile's scales
  bool scaled = false;
  long long amask = 0;              // mask minus operand address, in floats
  bool am = false;
  int a_end = 0;                    // K-contiguous: first k past the current segment
  float4 ra[NA], ma[kMaskA ? NA : 1];
  auto a_row = [&](int i) { return AK ? (tid >> 1) + 64 * i : (tid + kThreads * i) % (BM / 4) * 4; };
  auto a_k = [&](int i) { return AK ? (tid & 1) * 4 : (tid + kThreads * i) / (BM / 4); };
  auto a_on = [&](int i) { return tid + kThreads * i < 2 * BM; };
  auto seek_a = [&](int k) {
    if (AK) {
      const int q = find_seg(d.A, k);
      const Seg &sg = d.A.seg[q];
      a_end = q + 1 < d.A.nseg ? d.A.seg[q + 1].begin : 0x7fffffff;
      am = kMaskA && sg.mask != nullptr;
      amask = am ? sg.mask - sg.ptr : 0;
      scaled = sg.rowscale != nullptr;
#pragma unroll
      for (int i = 0; i < NA; ++i) {
        const int m = min(m0 + a_row(i), M - 1);
        pa[i] = sg.ptr + (size_t)m * sg.ld + (k - sg.begin) + a_k(i);
        sc[i] = scaled ? sg.rowscale[m] : 1.f;
        astep[i] = BK;
      }
    } else {
      scaled = true;
#pragma unroll
      for (int i = 0; i < NA; ++i) {
        const int m = m0 + a_row(i);
        const Seg &sg = d.A.seg[find_seg(d.A, min(m, M - 1))];
        pa[i] = sg.ptr && m < M ? sg.ptr + (size_t)(k + a_k(i)) * sg.ld + (m - sg.begin) : nullptr;
        ps[i] = sg.rowscale && m < M ? sg.rowscale + k + a_k(i) : nullptr;
        astep[i] = BK * sg.ld;
      }
    }
  };
  // ---- B: slot h is column b_n (K-contiguous) or k b_k (N-contiguous)
  const float *pb[2];
  int bstep = 0;
  long long bmask = 0;
  bool bm = false;
  int b_end = 0;
  float4 rb[2], mb[kMaskB ? 2 : 1];
  auto seek_b = [&](int k) {
    const int q = BNC ? 0 : find_seg(d.B, k);
    const Seg &sg = d.B.seg[q];
    b_end = !BNC && q + 1 < d.B.nseg ? d.B.seg[q + 1].begin : 0x7fffffff;
    bstep = BNC ? BK * sg.ld : BK;
    bm = kMaskB && sg.mask != nullptr;
    bmask = bm ? sg.mask - sg.ptr : 0;
#pragma unroll
    for (int h = 0; h < 2; ++h)
      pb[h] = BNC ? sg.ptr + (size_t)(k + warp + 4 * h) * sg.ld + min(n0 + lane * 4, N - 4)
                  : sg.ptr + (size_t)min(n0 + (tid >> 1) + 64 * h, N - 1) * sg.ld + (k - sg.begin) + (tid & 1) * 4;
  };
  int kend = 0;
  // ---- global -> registers: loads only; masks and scales are applied when
  // the tile is stored, so that the FMAs in between hide the loads' latency
  auto load = [&](int k0) {
    if (AK && k0 >= a_end) seek_a(k0);
    if (!BNC && k0 >= b_end) seek_b(k0);
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int k = k0 + a_k(i);
      ra[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (!AK) sc[i] = 1.f;
      if (a_on(i) && k < kend) {
        if (AK || pa[i]) {
          ra[i] = ld4(pa[i]);
          if (kMaskA && am) ma[i] = ld4(pa[i] + amask);
          if (!AK && ps[i]) sc[i] = *ps[i];
        } else {  // the ones row: the tile's rows below M
          const int m = m0 + a_row(i);
          ra[i] = make_float4(m < M, m + 1 < M, m + 2 < M, m + 3 < M);
        }
      }
      if (AK || pa[i]) pa[i] += astep[i];
      if (!AK && ps[i]) ps[i] += BK;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = k0 + (BNC ? warp + 4 * h : (tid & 1) * 4);
      rb[h] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (k < kend) {
        rb[h] = ld4(pb[h]);
        if (kMaskB && bm) mb[h] = ld4(pb[h] + bmask);
      }
      pb[h] += bstep;
    }
  };
  // ---- registers -> shared
  auto store = [&](int buf) {
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      if (!a_on(i)) continue;
      const int r = a_row(i), k = a_k(i);
      if (kMaskA && am) ra[i] = keep_positive(ra[i], ma[i]);
      if (scaled) {
        ra[i].x *= sc[i]; ra[i].y *= sc[i]; ra[i].z *= sc[i]; ra[i].w *= sc[i];
      }
      if (AK) {
        As[buf][k + 0][r] = ra[i].x; As[buf][k + 1][r] = ra[i].y;
        As[buf][k + 2][r] = ra[i].z; As[buf][k + 3][r] = ra[i].w;
      } else {
        *reinterpret_cast<float4 *>(&As[buf][k][r]) = ra[i];
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (kMaskB && bm) rb[h] = keep_positive(rb[h], mb[h]);
      if (BNC) {
        *reinterpret_cast<float4 *>(&Bs[buf][warp + 4 * h][lane * 4]) = rb[h];
      } else {
        const int r = (tid >> 1) + 64 * h, kq = (tid & 1) * 4;
        Bs[buf][kq + 0][r] = rb[h].x; Bs[buf][kq + 1][r] = rb[h].y;
        Bs[buf][kq + 2][r] = rb[h].z; Bs[buf][kq + 3][r] = rb[h].w;
      }
    }
  };

  // acc[i][j]: rows 32 (i / 2) + ty*4 + 2 (i % 2) + {0, 1}, column
  // 32 warp + 16 (j / 4) + tx*4 + j % 4
  unsigned long long acc[TM / 2][8];
  const int z0 = CHUNKS ? 0 : (int)blockIdx.z, z1 = CHUNKS ? splits : z0 + 1;
  for (int z = z0; z < z1; ++z) {
    const int kbeg = z * kps;
    kend = min(K, kbeg + kps);
#pragma unroll
    for (int i = 0; i < TM / 2; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = 0ull;
    if (kbeg < kend) {
      seek_a(kbeg);
      seek_b(kbeg);
      load(kbeg);
      store(0);
      __syncthreads();
      int buf = 0;
      for (int k0 = kbeg; k0 < kend; k0 += BK) {
        const bool more = k0 + BK < kend;
        if (more) load(k0 + BK);
        if (active) {
#pragma unroll
          for (int kk = 0; kk < BK; ++kk) {
            ulonglong2 a[TM / 4];
#pragma unroll
            for (int i = 0; i < TM / 4; ++i)
              a[i] = *reinterpret_cast<const ulonglong2 *>(&As[buf][kk][32 * i + ty * 4]);
            const float4 b0 = *reinterpret_cast<const float4 *>(&Bs[buf][kk][32 * warp + tx * 4]);
            const float4 b1 = *reinterpret_cast<const float4 *>(&Bs[buf][kk][32 * warp + 16 + tx * 4]);
            const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const unsigned long long bb = pair(b[j], b[j]);
#pragma unroll
              for (int i = 0; i < TM / 4; ++i) {
                fma2(acc[2 * i][j], a[i].x, bb);
                fma2(acc[2 * i + 1][j], a[i].y, bb);
              }
            }
          }
        }
        if (more) store(buf ^ 1);
        __syncthreads();
        buf ^= 1;
      }
    }
    if (CHUNKS && splits > 1 && active) {  // total += chunk z, in chunk order
#pragma unroll
      for (int i = 0; i < TM / 2; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 u = unpair(acc[i][2 * q]), w = unpair(acc[i][2 * q + 1]);
          float4 v = make_float4(u.x, u.y, w.x, w.y);
          float4 *t = s_tot + (4 * i + q) * kThreads + tid;
          if (z > 0) {
            const float4 o = *t;
            v = make_float4(o.x + v.x, o.y + v.y, o.z + v.z, o.w + v.w);
          }
          if (z + 1 < splits) {
            *t = v;
          } else {
            acc[i][2 * q] = pair(v.x, v.y);
            acc[i][2 * q + 1] = pair(v.z, v.w);
          }
        }
    }
  }

  // ---- epilogue
  if (!active) return;
#pragma unroll
  for (int i = 0; i < TM / 2; ++i)
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int m = m0 + 32 * (i / 2) + ty * 4 + 2 * (i % 2) + r;
      if (m >= M) continue;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int n = n0 + 32 * warp + 16 * h + tx * 4;
        if (n >= N) continue;
        float e[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 u = unpair(acc[i][4 * h + q]);
          e[q] = r ? u.y : u.x;
        }
        const float4 v = make_float4(e[0], e[1], e[2], e[3]);
        if (!CHUNKS && splits > 1)
          *reinterpret_cast<float4 *>(partial + ((size_t)blockIdx.z * d.M + m) * N + n) = v;
        else
          finish4(d, M, m, n, v);
      }
    }
}

// C = epilogue(sum_z partial[z]); one thread per 4 outputs
__global__ void __launch_bounds__(kReduceThreads)
splitk_reduce_kernel(GemmDesc d, DevDims dims, const float *__restrict__ partial, int splits) {
  pdl_entry(GCNN_K_GEMM_SIMT_REDUCE);
  const Sizes sz = actual_sizes(d, dims);
  const int M = sz.M, N = d.N, N4 = N / 4;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)M * N4) return;
  const int m = (int)(t / N4), n = (int)(t % N4) * 4;
  float4 v = ld4(partial + (size_t)m * N + n);
  for (int z = 1; z < splits; ++z) {
    const float4 p = ld4(partial + ((size_t)z * d.M + m) * N + n);
    v.x += p.x; v.y += p.y; v.z += p.z; v.w += p.w;
  }
  finish4(d, M, m, n, v);
}

int g_num_sms = 0;

}  // namespace

int num_sms() {
  if (g_num_sms == 0) {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0)
      g_num_sms = n;
    else
      g_num_sms = 148;
  }
  return g_num_sms;
}

namespace {

int choose_splits(int M, int N, int K) {
  const long long tiles = (long long)ceil_div(M, kPlanTile) * ceil_div(N, kPlanTile);
  const int ktiles = (int)ceil_div(K, kPlanK);
  const long long target = 2LL * num_sms();
  int s = (int)std::max<long long>(1, (target + tiles - 1) / tiles);
  s = std::min(s, std::max(1, ktiles / 8));  // at least 8 k-tiles per split
  return std::min(s, 32);
}

// along_k: the segments run along K, in steps of whole k tiles
bool operand_ok(const Operand &op, bool along_k) {
  if (op.nseg < 1 || op.nseg > kMaxSeg || op.seg[0].begin != 0) return false;
  for (int q = 0; q < op.nseg; ++q) {
    const Seg &s = op.seg[q];
    if (s.begin % (along_k ? BK : 4)) return false;
    if (along_k && !s.ptr) return false;
    if (q > 0 && s.begin <= op.seg[q - 1].begin) return false;
    if (s.ptr && (s.ld % 4 || reinterpret_cast<uintptr_t>(s.ptr) % 16)) return false;
    if (s.mask && (!s.ptr || reinterpret_cast<uintptr_t>(s.mask) % 16)) return false;
  }
  return true;
}

using Kernel = void (*)(GemmDesc, DevDims, float *, int, int);

// chunks: all K-chunks in one CTA (the forward products only)
template <int TM>
Kernel kernel_of(const GemmDesc &d, bool chunks) {
  constexpr int most = TM <= 16 ? TM : 16;  // with masks or per-k scales in registers
  if (!d.a_kcontig) return sgemm_kernel<most, false, true, false>;
  if (!d.b_ncontig) return sgemm_kernel<most, true, false, false>;
  return chunks ? sgemm_kernel<most, true, true, true> : sgemm_kernel<TM, true, true, false>;
}

Kernel kernel_for(const GemmDesc &d, int tm, bool chunks) {
  switch (tm) {
    case 8: return kernel_of<8>(d, chunks);
    case 12: return kernel_of<12>(d, chunks);
    case 16: return kernel_of<16>(d, chunks);
    default: return kernel_of<20>(d, chunks);
  }
}

// Rows per thread of one launch.  CTAs of all sizes keep the FFMA pipe about
// equally busy, two to an SM; what differs is the rows past M and the last
// wave, so take the size with the least work per SM: full waves of two CTAs
// per SM, and a last wave that takes a little over half as long where its
// CTAs have an SM each.
int choose_tm(const GemmDesc &d, int z, bool chunks) {
  int best = 16;
  double best_t = 1e30;
  for (int tm : {16, 20, 12, 8}) {
    if (tm > 16 && (chunks || !d.a_kcontig || !d.b_ncontig)) continue;
    const long long ctas = (long long)ceil_div(d.M, 8 * tm) * ceil_div(d.N, BN) * z;
    const long long slots = (long long)kCtasPerSm * num_sms(), rem = ctas % slots;
    const double waves = (double)(ctas / slots) + (rem == 0 ? 0.0 : (rem <= num_sms() ? 0.6 : 1.0));
    const double t = waves * (tm + 2.0);
    if (t < best_t) {
      best_t = t;
      best = tm;
    }
  }
  return best;
}

// How one product runs: its K-chunks, and whether each CTA runs all of them.
struct Plan {
  int splits, kps;
  bool chunks;
};

// A row-invariant product (no split that depends on the rows) still sums K in
// chunks of kInvariantChunk: few rows run them in parallel CTAs with a
// reduction, many rows in one CTA each, with the same additions in the same
// order either way.
bool invariant_chunks(const GemmDesc &d, const GemmWorkspace &ws) {
  return ws.max_splits == 1 && d.node_dim != kNodeK && d.a_kcontig && d.b_ncontig && d.K > kInvariantChunk;
}

// rows up to which the chunks of a row-invariant product run in parallel
// CTAs: fewer than one 128 x 128 tile for every two SMs; from there on the
// tiles alone (choose_tm halves their rows) give every SM work, and the
// partial tiles would cost 13 times the output's bytes
bool few_rows(int M, int N) { return 2LL * ceil_div(M, kPlanTile) * ceil_div(N, BN) <= num_sms(); }

Plan make_plan(const GemmDesc &d, const GemmWorkspace &ws) {
  Plan p{1, 0, false};
  if (invariant_chunks(d, ws)) {
    p.kps = kInvariantChunk;
    p.splits = (int)ceil_div(d.K, p.kps);
    p.chunks = !few_rows(d.M, d.N) || (size_t)p.splits * d.M * d.N > ws.floats;
    return p;
  }
  p.splits = std::min(choose_splits(d.M, d.N, d.K), ws.max_splits);
  if (p.splits > 1 && (size_t)p.splits * d.M * d.N > ws.floats) p.splits = 1;
  p.kps = std::max(kPlanK, (int)(ceil_div(d.K, (long long)p.splits * kPlanK) * kPlanK));
  return p;
}

size_t totals_bytes(int tm) { return (size_t)2 * tm * kThreads * sizeof(float4); }

}  // namespace

size_t gemm_simt_workspace_floats(int M, int N, int K, bool row_invariant) {
  if (row_invariant)
    return K > kInvariantChunk && few_rows(M, N) ? (size_t)ceil_div(K, kInvariantChunk) * M * N : 0;
  const int s = choose_splits(M, N, K);
  return s > 1 ? (size_t)s * M * N : 0;
}

int run_gemm_simt(const GemmDesc &d, DevDims dims, const GemmWorkspace &ws, cudaStream_t s) {
  if (d.M <= 0 || d.N <= 0 || d.K < 0) return GCNN_OK;
  if (d.N % 4 || d.ldc % 4 || reinterpret_cast<uintptr_t>(d.C) % 16)
    return set_error(GCNN_EINVAL, "gemm: N, ldc must be multiples of 4 and C 16-byte aligned");
  if (d.a_kcontig && d.K % 4) return set_error(GCNN_EINVAL, "gemm: K must be a multiple of 4");
  if (!d.b_ncontig && d.K % 4) return set_error(GCNN_EINVAL, "gemm: K must be a multiple of 4");
  if (!operand_ok(d.A, d.a_kcontig) || !operand_ok(d.B, true) || (d.b_ncontig && d.B.nseg != 1))
    return set_error(GCNN_EINVAL, "gemm: bad operand segments (alignment / order)");
  if (!d.a_kcontig && !d.b_ncontig) return set_error(GCNN_EINVAL, "gemm: A along M needs B along N");
  // rows come in fours; a remainder only as the ones row
  if (!d.a_kcontig && d.M % 4 && (d.A.seg[d.A.nseg - 1].ptr || d.A.seg[d.A.nseg - 1].begin != d.M / 4 * 4))
    return set_error(GCNN_EINVAL, "gemm: M must be a multiple of 4 besides the ones row");
  for (int q = 0; q < d.A.nseg; ++q)
    if (d.A.seg[q].mask && (!d.a_kcontig || d.b_ncontig)) return set_error(GCNN_EINVAL, "gemm: no mask on A in this form");
  for (int q = 0; q < d.B.nseg; ++q)
    if (d.B.seg[q].rowscale || (d.B.seg[q].mask && d.a_kcontig)) return set_error(GCNN_EINVAL, "gemm: no mask or scale on B in this form");
  const Plan p = make_plan(d, ws);
  const int tm = choose_tm(d, p.chunks ? 1 : p.splits, p.chunks);
  const Kernel kernel = kernel_for(d, tm, p.chunks);
  if (p.chunks) {
    static std::once_flag once;
    static cudaError_t attr = cudaSuccess;
    std::call_once(once, [&] {
      for (int t : {8, 12, 16})
        if (attr == cudaSuccess)
          attr = cudaFuncSetAttribute(kernel_for(d, t, true), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)totals_bytes(t));
    });
    if (attr != cudaSuccess) return set_error(GCNN_ECUDA, "gemm: %s", cudaGetErrorString(attr));
  }
  const bool reduce = p.splits > 1 && !p.chunks;
  dim3 grid(ceil_div(d.N, BN), ceil_div(d.M, 8 * tm), reduce ? p.splits : 1);
  float *part = reduce ? ws.partial : nullptr;
  GCNN_TRY(launch(kernel, grid, kThreads, p.chunks ? totals_bytes(tm) : 0, s, d, dims, part, p.splits, p.kps));
  if (reduce) GCNN_TRY(run_splitk_reduce(d, dims, part, p.splits, s));
  return GCNN_OK;
}

int run_splitk_reduce(const GemmDesc &d, DevDims dims, const float *partial, int splits, cudaStream_t s) {
  const long long work = (long long)d.M * (d.N / 4);
  GCNN_TRY(launch(splitk_reduce_kernel, ceil_div(work, kReduceThreads), kReduceThreads, 0, s, d, dims, partial, splits));
  return GCNN_OK;
}

GCNN_TIMELINE_ATTACH(gemm_simt)

}  // namespace gcnn
