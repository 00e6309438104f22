// FP32 products of the inference forward on the tensor cores, without giving up
// FP32 accuracy: exact integer slices (the splitting of Ootomo, Ozaki and
// Yokota's integer-unit DGEMM, Int. J. High Perform. Comput. Appl. 2024, here
// for FP32 on BF16 units).
//
// A row of A is scaled by a power of two to at most 256 in magnitude and cut
// into three integers, x = 2^(e-8) (s1 + s2 2^-9 + s3 2^-18), |s| <= 256,
// rounded to nearest at every step: 26 bits below the row's largest entry, two
// more than FP32 itself holds.  The columns of B (the weights) are cut the same
// way.  Integers up to 256 are exact in BF16, products of two have at most 17
// bits, and sums of a thousand of them with mixed signs stay far below 2^24, so the FP32
// accumulators of the tensor cores, which round toward zero and would bias a
// sum of rounded terms, hold the sums exactly.
// Products of equal weight share an accumulator:
//   G2 = s1 t1,  G3 = s1 t2 + s2 t1,  G4 = s1 t3 + s2 t2 + s3 t1
//   C = 2^(ea+eb-16) (G2 + 2^-9 G3 + 2^-18 G4)
// and what is dropped (weights 2^-27 and below) is less than a plain FP32 sum's
// own rounding.
//
// The degree scalers stay out of the operand: the update runs as four phases
// (x, and the aggregates against the identity, amplification and attenuation
// rows of W_U), each with its own sums, combined per row as
// ((p_x + p_id) + amp p_amp) + att p_att.  So the aggregates' slices are written
// once and not three times.
//
// Rows with an infinity or a NaN have no such scale (theirs is NaN): the
// epilogue computes them with plain FP32 products.
//
// Measured against the CUDA-core path (FFMA), H = 200, 6 layers: relative error of
// a layer's activations 1.1e-7 to 1.9e-7 against 3.4e-7 to 6.3e-7 (FP64 oracle,
// 2,174 atoms), with 8-bit slices 6.6e-7 to 1.3e-6.  Update of 19,719 atoms 682
// -> 100 us and 14 us for the sum of the phases; 1,100-molecule forward 4.87 ->
// 1.84 ms, a server burst of 650 molecules 9.4 -> 2.9 ms.
#include <algorithm>
#include <cfloat>

#include "slices.cuh"
#include "tc_ptx.cuh"

namespace gcnn {
namespace {

constexpr int kBM = 128, kBK = 64, kMaxN = 112, kStagesF = 2;
constexpr int kThreadsF = 320, kEpiWarpsF = 8;
constexpr int kABytes = kBM * kBK * 2;                     // one plane of A
constexpr int kStageF = 3 * kABytes + 3 * 2 * (int)kMnAtomBytes;  // and of B: at most two 64-column atoms
constexpr int kChunkF = 16, kPitchF = kChunkF + 4;
constexpr int kEpiF = kEpiWarpsF * 32 * kPitchF * 4;
constexpr int kSmemF = 1024 + kStagesF * kStageF + kEpiF + 256;
constexpr uint32_t kAccStride = 128;  // TMEM columns between the three accumulators

struct F32Maps {
  CUtensorMap x, agg, b;
};

// x (N x H, H <= 256) -> planes row x3[i] = [s1 | s2 | s3], each Hp wide; one
// warp per row.
__global__ void __launch_bounds__(256) slice_rows_kernel(int n_cap, int H, int Hp, DevDims dims,
                                                         const float *__restrict__ x, uint16_t *__restrict__ x3,
                                                         float *__restrict__ factor) {
  pdl_entry(GCNN_K_CAST_BF16);
  const int N = min(n_cap, dims.nodes(n_cap));
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31, H4 = H >> 2;
  if (i >= N) return;  // warp-uniform
  float4 v[2];
  float m = 0.f;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int c4 = lane + 32 * u;
    v[u] = c4 < H4 ? *reinterpret_cast<const float4 *>(x + (size_t)i * H + 4 * c4) : make_float4(0.f, 0.f, 0.f, 0.f);
    m = max4(m, v[u]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  float inv, f;
  slice_scale(m, &inv, &f);
  if (lane == 0) factor[i] = f;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int c4 = lane + 32 * u;
    if (c4 < H4) store_slices(v[u], inv, x3 + (size_t)i * 3 * Hp + 4 * c4, Hp);
  }
}

// Columns of W (K x N, pitch N; one matrix per blockIdx.y, `stride` floats
// apart) -> w3 as three K x N planes per matrix, and the columns' factors; sets
// *bad where a column has none.
constexpr int kWeightThreads = 1024;

__global__ void __launch_bounds__(kWeightThreads)
slice_weights_kernel(int K, int N, const float *__restrict__ W, long long stride, uint16_t *__restrict__ w3,
                     float *__restrict__ factor, unsigned *__restrict__ bad) {
  pdl_entry(GCNN_K_CAST_BF16);
  __shared__ float red[32][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, n = blockIdx.x * 32 + lane;
  W += (long long)blockIdx.y * stride;
  w3 += (size_t)blockIdx.y * 3 * K * N;
  float m = 0.f;
  if (n < N)
#pragma unroll 8
    for (int k = w; k < K; k += 32) {
      const float v = W[(size_t)k * N + n];
      m = v != v ? __uint_as_float(0x7f800000u) : fmaxf(m, fabsf(v));
    }
  red[w][lane] = m;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 32; ++q) m = fmaxf(m, red[q][lane]);
  float inv, f;
  slice_scale(m, &inv, &f);
  if (n >= N) return;
  if (w == 0) {
    factor[(size_t)blockIdx.y * N + n] = f;
    if (f != f) atomicOr(bad, 1u);
  }
#pragma unroll 4
  for (int k = w; k < K; k += 32) {
    float s[3];
    slice3(W[(size_t)k * N + n] * inv, s);
#pragma unroll
    for (int p = 0; p < 3; ++p) w3[((size_t)p * K + k) * N + n] = (uint16_t)(bf16x2(s[p], 0.f) & 0xffffu);
  }
}

// ---------------------------------------------------------------- product
__device__ __forceinline__ float4 finish_f32(const F32Desc &d, int n, float4 v) {
  if (d.bias) {
    v.x += n + 0 < d.bias_n ? d.bias[n + 0] : 0.f;
    v.y += n + 1 < d.bias_n ? d.bias[n + 1] : 0.f;
    v.z += n + 2 < d.bias_n ? d.bias[n + 2] : 0.f;
    v.w += n + 3 < d.bias_n ? d.bias[n + 3] : 0.f;
  }
  if (d.relu) v = make_float4(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f), fmaxf(v.z, 0.f), fmaxf(v.w, 0.f));
  return v;
}

// A phase's value of C(row, n) with plain FP32 products in k order, for a row
// or a column without a finite factor.
__device__ __noinline__ float plain_dot(const F32Desc &d, const F32Phase &ph, int row, int n) {
  const int K = ph.from_agg ? kAgg * d.H : d.H;
  const float *a = ph.from_agg ? d.agg + (size_t)row * K : d.x + (size_t)row * K;
  const float *b = d.W + (size_t)ph.b_row * d.N + n;
  float s = 0.f;
  for (int k = 0; k < K; ++k) s = fmaf(a[k], b[(size_t)k * d.N], s);
  return s;
}

// Persistent CTAs, one per SM, over 128 x BN tiles (BN <= 112).  Per 64-wide k
// tile the three planes of A and B arrive (96 KB, two stages) for 24 MMAs; warp
// 0 loads, warp 1 issues, warps 2-9 read the phase's three accumulators out of
// TMEM while the next tile's first stages arrive.  Bound by the bytes an SM
// takes in (96 KB per 1,400 cycles of MMAs).  PART: one item is one phase, whose
// value goes to f32_combine_kernel; otherwise an item runs all phases.
template <bool PART>
__global__ void __launch_bounds__(kThreadsF, 1)
tma_gemm_f32_kernel(const __grid_constant__ F32Maps maps, F32Desc d, DevDims dims, float *__restrict__ partial,
                    int ntiles, int BN, unsigned *err) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  float *epi = reinterpret_cast<float *>(smem + kStagesF * kStageF);
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + kStagesF * kStageF + kEpiF);
  uint64_t *empty = full + kStagesF;
  uint64_t *acc_full = empty + kStagesF, *acc_empty = acc_full + 1;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_empty + 1);
  uint32_t *flag = tmem_slot + 1;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  if (tid == 0) {
    for (int s = 0; s < kStagesF; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(acc_full, 1);
    mbar_init(acc_empty, kEpiWarpsF);
    *flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  const int M = min(d.M, dims.nodes(d.M)), N = d.N;
  // work item t of a CTA: a tile (column tiles fastest) and, with PART, a
  // phase; the x phase, a quarter of the others' length, comes last
  const int tiles = (M + kBM - 1) / kBM * ntiles, items = PART ? tiles * d.nphase : tiles;
  auto row0 = [&](int t) { return t % tiles / ntiles * kBM; };
  auto col0 = [&](int t) { return t % tiles % ntiles * BN; };
  auto first_phase = [&](int t) { return PART ? (t / tiles + 1) % d.nphase : 0; };
  const int phases = PART ? 1 : d.nphase;
  pdl_entry(GCNN_K_GEMM_TC_C);
  if ((int)blockIdx.x >= items) return;  // block-uniform, before any barrier wait or TMEM use
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  const int atoms = (BN + 63) / 64;
  const int b_plane = atoms * (int)kMnAtomBytes;

  if (warp == 0) {
    // ------------------------------------------------ TMA producer
    int it = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < items && ok; t += gridDim.x)
      for (int p = first_phase(t), p1 = p + phases; p < p1 && ok; ++p) {
        const int m0 = row0(t), n0 = col0(t);
        const F32Phase ph = d.phase[p];
        const CUtensorMap *am = ph.from_agg ? &maps.agg : &maps.x;
        const int width = ph.from_agg ? d.Ap : d.Hp;
        for (int kt = 0; kt < ph.ktiles; ++kt, ++it) {
          const int s = it % kStagesF;
          if (it >= kStagesF && !__all_sync(0xffffffffu, mbar_wait(&empty[s], (it / kStagesF - 1) & 1))) {
            ok = false;
            break;
          }
          uint8_t *st = smem + s * kStageF;
          if (elect_one()) {
            mbar_expect_tx(&full[s], (uint32_t)(3 * (kABytes + b_plane)));
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              tma_load_2d(smem_u32(st + q * kABytes), am, q * width + kt * kBK, m0, &full[s]);
              for (int j = 0; j < atoms; ++j)
                tma_load_2d(smem_u32(st + 3 * kABytes + q * b_plane + j * (int)kMnAtomBytes), &maps.b, n0 + 64 * j,
                            q * d.b_rows + ph.b_row + kt * kBK, &full[s]);
            }
          }
          __syncwarp();
        }
      }
    if (!ok && lane == 0) atomicOr(flag, 1u);
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer
    const uint32_t idesc = instr_desc(kBM, BN, false, true);
    const uint64_t da = smem_desc(smem_u32(smem), false), db = smem_desc(smem_u32(smem + 3 * kABytes), true);
    const uint32_t a_hi = (uint32_t)(da >> 32), b_hi = (uint32_t)(db >> 32);
    const uint32_t bp = (uint32_t)b_plane >> 4;
    bool ok = true;
    int it = 0, round = 0;
    for (int t = blockIdx.x; t < items && ok; t += gridDim.x)
      for (int p = first_phase(t), p1 = p + phases; p < p1 && ok; ++p, ++round) {
        if (round > 0) ok = __all_sync(0xffffffffu, mbar_wait(acc_empty, (round - 1) & 1));
        fence_after_sync();
        const int nk = d.phase[p].ktiles;
        for (int kt = 0; kt < nk && ok; ++kt, ++it) {
          const int s = it % kStagesF;
          ok = __all_sync(0xffffffffu, mbar_wait(&full[s], (it / kStagesF) & 1));
          if (!ok) break;
          fence_after_sync();
          const uint32_t a0 = (uint32_t)da + s * (kStageF >> 4), b0 = (uint32_t)db + s * (kStageF >> 4);
#pragma unroll
          for (int g = 0; g < 3; ++g)      // accumulator of s_i t_j with i + j = g
#pragma unroll
            for (int i = 0; i <= g; ++i)
#pragma unroll
              for (int j = 0; j < kBK / 16; ++j)
                mma_bf16(tmem + g * kAccStride, a0 + i * (kABytes >> 4) + j * (32u >> 4), a_hi,
                         b0 + (g - i) * bp + j * (2048u >> 4), b_hi, idesc, (kt > 0 || i > 0 || j > 0) ? 1u : 0u);
          mma_commit(&empty[s]);
        }
        if (ok) mma_commit(acc_full);
      }
    if (!ok && lane == 0) atomicOr(flag, 1u);
  } else {
    // ------------------------------------------------ epilogue
    // A lane turns its row's three sums into the phase's value; the chunk then
    // goes through shared memory to row segments of 64 bytes, where the running
    // total of earlier phases is read back from C (by the lane that stored it).
    const int q = warp & 3, half = (warp - 2) >> 2;
    const int chunks = (BN + kChunkF - 1) / kChunkF, mid = (chunks + 1) / 2;
    const int c0 = half ? mid : 0, c1 = half ? chunks : mid;
    float *S = epi + (warp - 2) * 32 * kPitchF;
    const int cc = (lane & 3) * 4;  // stores: rows rr + 8 w, columns cc ..
    bool ok = true;
    int round = 0;
    for (int t = blockIdx.x; t < items && ok; t += gridDim.x)
      for (int p = first_phase(t), p1 = p + phases; p < p1; ++p, ++round) {
        const int m0 = row0(t), n0 = col0(t);
        const int row = m0 + 32 * q + lane, rr = m0 + 32 * q + (lane >> 2);
        if (!__all_sync(0xffffffffu, mbar_wait(acc_full, round & 1))) {
          if (lane == 0) atomicOr(flag, 1u);
          ok = false;
          break;
        }
        fence_after_sync();
        const F32Phase ph = d.phase[p];
        const float f = row < M ? (ph.from_agg ? d.fagg : d.fx)[row] : 0.f;
        float sc[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) sc[w] = !PART && ph.scaler && rr + 8 * w < M ? ph.scaler[rr + 8 * w] : 1.f;
#pragma unroll 1
        for (int c = c0; c < c1; ++c) {
          uint32_t g[3][2][8];
#pragma unroll
          for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int w = 0; w < 2; ++w)
              tmem_ld8(tmem + ((uint32_t)(32 * q) << 16) + a * kAccStride + (uint32_t)(c * kChunkF + 8 * w), g[a][w]);
          const int n = n0 + c * kChunkF + cc;
          const bool in = n < N && c * kChunkF + cc < BN;
          float4 old[4];
          if (!PART && p > 0)
#pragma unroll
            for (int w = 0; w < 4; ++w)
              if (in && rr + 8 * w < M) old[w] = *reinterpret_cast<const float4 *>(d.C + (size_t)(rr + 8 * w) * d.ldc + n);
          // the chunk's column factors, one per lane
          const int nf = n0 + c * kChunkF + (lane & 15);
          const float fbl = nf < N ? d.fb[nf] : 0.f;
          tmem_wait_ld();
          if (c + 1 == c1) {  // this warp has read all of the phase's sums
            fence_before_sync();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(acc_empty)) : "memory");
          }
#pragma unroll
          for (int w = 0; w < 4; ++w) {
            float v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const int x = 4 * w + k;
              const float fb = __shfl_sync(0xffffffffu, fbl, x);
              const float g2 = __uint_as_float(g[0][x / 8][x % 8]), g3 = __uint_as_float(g[1][x / 8][x % 8]);
              const float g4 = __uint_as_float(g[2][x / 8][x % 8]);
              // the factors are powers of two: only the two sums round
            const float u = fmaf(fmaf(g4, 0.001953125f, g3), 0.001953125f, g2);
            v[k] = (u * fb) * f;
            if (!(fabsf(v[k]) <= FLT_MAX)) {  // overflow on the way, or a factor that is no number
              if (f == f && fb == fb) v[k] = (u * f) * fb;
              else if (row < M && n0 + c * kChunkF + x < N) v[k] = plain_dot(d, ph, row, n0 + c * kChunkF + x);
            }
            }
            *reinterpret_cast<float4 *>(S + lane * kPitchF + 4 * w) = make_float4(v[0], v[1], v[2], v[3]);
          }
          __syncwarp();
#pragma unroll
          for (int w = 0; w < 4; ++w) {
            const int r = rr + 8 * w;
            float4 v = *reinterpret_cast<const float4 *>(S + ((lane >> 2) + 8 * w) * kPitchF + cc);
            if (!in || r >= M) continue;
            if (PART) {
              *reinterpret_cast<float4 *>(partial + ((size_t)p * d.M + r) * N + n) = v;
              continue;
            }
            if (p > 0)
              v = ph.scaler ? make_float4(fmaf(sc[w], v.x, old[w].x), fmaf(sc[w], v.y, old[w].y),
                                          fmaf(sc[w], v.z, old[w].z), fmaf(sc[w], v.w, old[w].w))
                            : make_float4(old[w].x + v.x, old[w].y + v.y, old[w].z + v.z, old[w].w + v.w);
            if (p + 1 == p1) v = finish_f32(d, n, v);
            *reinterpret_cast<float4 *>(d.C + (size_t)r * d.ldc + n) = v;
          }
          __syncwarp();
        }
        if (c0 >= c1 && lane == 0)  // a warp without columns (narrow tiles)
          asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(acc_empty)) : "memory");
      }
  }
  fence_before_sync();
  __syncthreads();
  if (tid == 0 && *flag && err) atomicOr(err, kErrTimeout);
  if (warp == 0) tmem_free(tmem, 512);
}

// C from the phases' values: the same operations in the same order as above.
__global__ void __launch_bounds__(256)
f32_combine_kernel(F32Desc d, DevDims dims, const float *__restrict__ partial) {
  pdl_entry(GCNN_K_GEMM_TC_REDUCE);
  const int M = min(d.M, dims.nodes(d.M)), N4 = d.N / 4;
  const unsigned t = blockIdx.x * 256u + threadIdx.x;
  const int row = (int)(t / (unsigned)N4), n = (int)(t % (unsigned)N4) * 4;
  if (row >= M) return;
  float4 v[kF32Phases];
#pragma unroll
  for (int p = 0; p < kF32Phases; ++p)
    if (p < d.nphase) v[p] = *reinterpret_cast<const float4 *>(partial + ((size_t)p * d.M + row) * d.N + n);
  float4 s = v[0];
#pragma unroll
  for (int p = 1; p < kF32Phases; ++p)
    if (p < d.nphase) {
      if (d.phase[p].scaler) {
        const float c = d.phase[p].scaler[row];
        s = make_float4(fmaf(c, v[p].x, s.x), fmaf(c, v[p].y, s.y), fmaf(c, v[p].z, s.z), fmaf(c, v[p].w, s.w));
      } else {
        s = make_float4(s.x + v[p].x, s.y + v[p].y, s.z + v[p].z, s.w + v[p].w);
      }
    }
  *reinterpret_cast<float4 *>(d.C + (size_t)row * d.ldc + n) = finish_f32(d, n, s);
}

}  // namespace

int run_gemm_f32tc(const F32Desc &d, DevDims dims, float *partial, size_t partial_floats, unsigned *err, cudaStream_t s) {
  if (d.M <= 0 || d.N <= 0) return GCNN_OK;
  if (d.N % 8 || d.H % 8 || d.Hp % 64 || d.Ap % 64 || d.nphase < 1 || d.nphase > kF32Phases)
    return set_error(GCNN_EINVAL, "f32tc gemm: bad sizes");
  static const cudaError_t attr = [] {
    const cudaError_t e =
        cudaFuncSetAttribute(tma_gemm_f32_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemF);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(tma_gemm_f32_kernel<true>,
                                                       cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemF);
  }();
  if (attr != cudaSuccess) return set_error(GCNN_ECUDA, "f32tc gemm: %s", cudaGetErrorString(attr));
  F32Maps maps;
  GCNN_TRY(tc_make_map(&maps.x, TcMat{d.x3, 3 * d.Hp, d.M, 3 * d.Hp, false}, kBM));
  GCNN_TRY(tc_make_map(&maps.agg, TcMat{d.agg3, 3 * d.Ap, d.M, 3 * d.Ap, false}, kBM));
  GCNN_TRY(tc_make_map(&maps.b, TcMat{d.b3, d.N, 3 * d.b_rows, d.N, true}, kBK));
  const int nt = (int)ceil_div(d.N, kMaxN), BN = ((d.N + nt - 1) / nt + 15) / 16 * 16;
  const int mt = (int)ceil_div(d.M, kBM), sms = num_sms();
  // phases in parallel CTAs: finer waves (and all there is for few rows) against
  // the values' way through memory, 2 x 4 bytes each per output
  int k_all = 0;
  for (int p = 0; p < d.nphase; ++p) k_all += d.phase[p].ktiles;
  const double tile_us = 1.05 * k_all + 4.0;
  const double seq = ceil_div((long long)mt * nt, sms) * tile_us;
  const double par = (double)ceil_div((long long)mt * nt * d.nphase, sms) * tile_us / d.nphase + 3.0 +
                     8e-6 * d.nphase * (double)d.M * d.N / 5.0;
  const bool part = d.nphase > 1 && par < seq && (size_t)d.nphase * d.M * d.N <= partial_floats;
  const int items = mt * nt * (part ? d.nphase : 1);
  GCNN_TRY(launch(part ? tma_gemm_f32_kernel<true> : tma_gemm_f32_kernel<false>, std::min(items, sms), kThreadsF, kSmemF,
                  s, maps, d, dims, part ? partial : nullptr, nt, BN, err));
  if (part)
    GCNN_TRY(launch(f32_combine_kernel, ceil_div((long long)d.M * (d.N / 4), 256), 256, 0, s, d, dims,
                    (const float *)partial));
  return GCNN_OK;
}

int launch_slice_rows(int n_nodes, int H, int Hp, DevDims dims, const float *x, uint16_t *x3, float *factor,
                      cudaStream_t s) {
  if (H > kF32MaxH || H % 4) return set_error(GCNN_EINVAL, "slice_rows: hidden too wide");
  if (n_nodes <= 0) return GCNN_OK;
  return launch(slice_rows_kernel, ceil_div(n_nodes, 8), 256, 0, s, n_nodes, H, Hp, dims, x, x3, factor);
}

int launch_slice_weights(int K, int N, int count, const float *W, long long stride, uint16_t *w3, float *factor,
                         unsigned *bad, cudaStream_t s) {
  return launch(slice_weights_kernel, dim3(ceil_div(N, 32), (unsigned)count), kWeightThreads, 0, s, K, N, W, stride, w3,
                factor, bad);
}

GCNN_TIMELINE_ATTACH(gemm_f32tc)

}  // namespace gcnn
