// Attention of a few query rows against many keys (decode: one new token per sequence; short query chunks against a
// cache): O = softmax(scale * Q K^T) V without a causal mask, for at most 32 query rows per key/value head.
//
// Bound: HBM.  Every key and value is read once and meets only the rows = seq_q * (heads_q / heads_kv) queries that
// share its head, a few FLOPs per byte; what matters is that the cache is streamed once, by all SMs, with enough
// bytes in flight.  (The two-tile kernel gives each query head a 256-row item of its own: one valid row in 256, the
// keys of a group fetched once per query head, and as many CTAs as heads.)  Hence:
//   - the query heads of a group and the query positions are the rows of ONE problem per (batch, key/value head);
//   - its keys are cut into `splits` runs of 64-key blocks, one CTA each, and the CTAs of a problem form a cluster:
//     their partial results are merged through distributed shared memory -- no scratch in global memory, no second
//     launch, a fixed order of additions;
//   - a producer warp streams K and V through a 96 KB TMA ring, two CTAs per SM (192 KB where there are not that many);
//   - four warps take 16 of a block's 64 keys each, with running maxima, sums and outputs of their own, so the main
//     loop has no barrier among them.  Keys are the M dimension of both products (S^T = K Q^T, O^T = V^T P^T) and the
//     8, 16 or 32 query rows the N dimension of mma.sync.m16n8k16: with M = 128 query rows, as tcgen05 wants them,
//     the products would be padding, and the round trip of the scores through tensor memory would be a serial chain.
// Measured (32 query / 8 key-value heads of 128, one query row per sequence, caches rotating through HBM; device time in a
// train, the two-tile kernel -> this): 32 sequences x 2000 keys 218 -> 39.3 us, 7 x 276 17.1 -> 4; 25 x 4217 keys of 12 heads
// of 64 158 -> 49.  A call of the first, one after another: 240 -> 40.4 us, 6.5 TB/s, the rate of a plain copy.  Calls of many
// problems of few keys are faster on the tile kernels: decode_wins (fact_api.cu).
// Masking only in the last block; probabilities are rounded to BF16 for the second product, sums are FP32 and taken
// over the unrounded values, the reference maximum moves (and O is rescaled) only when a score exceeds it by more than
// 8 in log2 units, as in the two-tile kernel.
#pragma once
#include "attention_kernel.cuh"

namespace fact {

constexpr int kDecThreads = 160;     // warps 0-3 compute, warp 4 loads
constexpr int kDecWarps = 4;
constexpr int kDecBlockK = 64;       // keys per ring stage: 16 per computing warp
constexpr int kDecMaxRows = 32;
constexpr uint32_t kDecRingBytes = 96 * 1024;   // two CTAs per SM; twice that where every CTA has an SM to itself
__host__ __device__ constexpr uint32_t dec_stage_bytes(int D) { return 2u * (uint32_t)kDecBlockK * (uint32_t)D * 2u; }
constexpr uint32_t kDecCtrlBytes = 256;               // barriers, abort flag: behind the ring (later: partial results)

struct DecodeParams {
  const __nv_bfloat16* Q;
  __nv_bfloat16* O;
  long long q_sb, q_st, q_sh, o_sb, o_st, o_sh;
  int Tq, Tk, Hkv, group, rows;  // rows = Tq * group; row r is query position r / group, head kvh * group + r % group
  int stages;                    // of the ring
  int splits;                    // CTAs (a cluster) per (batch, key/value head)
  int k_each, v_each;            // mask of the batch coordinate: all ones; 0 where all entries share one K or V
  float scale_log2;
  int* status;
};

template <int HD, int NT>  // NT: groups of 8 query rows
__global__ void __launch_bounds__(kDecThreads, NT <= 2 ? 2 : 1)
    fact_attention_decode_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                                 const DecodeParams p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  constexpr int KS = HD / 16;                               // 16-wide steps over the head dimension
  constexpr uint32_t kv_bytes = dec_stage_bytes(HD) / 2;    // K (or V) of a stage
  constexpr uint32_t chunk_bytes = kDecBlockK * 128u;       // 64 columns of it: 64 swizzled rows of 128 bytes
  constexpr int kPartLd = HD + 4;                           // floats per row of a partial output
  constexpr int kRows = 8 * NT;
  static_assert((kDecWarps + 1) * (kRows * kPartLd + 2 * kRows) * 4 <= (int)kDecRingBytes, "partials fit the ring");
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  const int lane = threadIdx.x & 31;
  const uint32_t smem_base = ptx::smem_u32(smem_raw);
  if (smem_base & 1023u) {  // (every CTA of the grid alike: no cluster is left waiting)
    if (threadIdx.x == 0) atomicExch(p.status, kDeviceTimeoutCode);
    return;
  }
  const int NS = p.stages;
  const uint32_t ring_bytes = (uint32_t)NS * dec_stage_bytes(HD);
  const uint32_t bar_base = smem_base + ring_bytes;
  auto full_bar = [&](int s) { return bar_base + 8u * (uint32_t)s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (uint32_t)(NS + s); };
  volatile int* abort_p = reinterpret_cast<volatile int*>(smem_raw + ring_bytes + 8 * 2 * NS);
  static_assert(8 * 2 * (int)(2 * kDecRingBytes / dec_stage_bytes(HD)) + 4 <= (int)kDecCtrlBytes, "control area");
  if (threadIdx.x < 2 * NS) {
    ptx::mbar_init(bar_base + 8u * threadIdx.x, (int)threadIdx.x < NS ? 1 : kDecWarps);
    if (threadIdx.x == 0) *abort_p = 0;
    ptx::fence_mbar_init();
  }
  if (warp == kDecWarps && lane == 0) {
    ptx::prefetch_tensormap(&tmK);
    ptx::prefetch_tensormap(&tmV);
  }
  __syncthreads();
  ptx::grid_dependency_wait();

  const int rank = (int)(blockIdx.x % (unsigned)p.splits);
  const int pair = (int)(blockIdx.x / (unsigned)p.splits);
  const int b = pair / p.Hkv, kvh = pair - b * p.Hkv;
  const int nb = (p.Tk + kDecBlockK - 1) / kDecBlockK;
  const int blk0 = (int)((long long)rank * nb / p.splits), blk1 = (int)((long long)(rank + 1) * nb / p.splits);
  auto wait_all = [&](uint32_t bar, uint32_t parity) -> bool {
    return __all_sync(0xffffffffu, wait_bar(bar, parity, abort_p, p.status)) != 0;
  };

  // per computing warp: reference maximum and partial row sums of this thread's columns (rows 2 (lane % 4), + 1 of
  // every group of 8), O^T accumulators
  float m[NT][2], l[NT][2], o[NT][KS][4];
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    m[t][0] = m[t][1] = -INFINITY;
    l[t][0] = l[t][1] = 0.f;
#pragma unroll
    for (int k = 0; k < KS; ++k)
#pragma unroll
      for (int i = 0; i < 4; ++i) o[t][k][i] = 0.f;
  }

  if (warp == kDecWarps) {
    // ------------------------------------------------------------ TMA producer
    int s = 0;
    uint32_t phase = 0;
    for (int j = blk0; j < blk1; ++j) {
      if (!wait_all(empty_bar(s), phase ^ 1u)) break;
      if (ptx::elect_one()) {
        const uint32_t dst = smem_base + (uint32_t)s * dec_stage_bytes(HD);
        ptx::mbar_arrive_expect_tx(full_bar(s), dec_stage_bytes(HD));
#pragma unroll
        for (int c = 0; c < HD / 64; ++c)
          ptx::tma_load_4d(dst + (uint32_t)c * chunk_bytes, &tmK, full_bar(s), c * 64, kvh, j * kDecBlockK, b & p.k_each);
#pragma unroll
        for (int c = 0; c < HD / 64; ++c)
          ptx::tma_load_4d(dst + kv_bytes + (uint32_t)c * chunk_bytes, &tmV, full_bar(s), c * 64, kvh, j * kDecBlockK, b & p.v_each);
      }
      __syncwarp();
      if (++s == NS) {
        s = 0;
        phase ^= 1u;
      }
    }
  } else {
    // ------------------------------------------------------------ 16 keys of every block per warp
    // Q as the B operand: this thread's column is query row 8 t + lane / 4, its k values 2 (lane % 4) + {0, 1, 8, 9}
    uint32_t qf[NT][KS][2];
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const int r = 8 * t + (lane >> 2);
      const bool ok = r < p.rows;
      const int tq = ok ? r / p.group : 0, g = ok ? r - tq * p.group : 0;
      const uint32_t* src = reinterpret_cast<const uint32_t*>(p.Q + (long long)b * p.q_sb + (long long)tq * p.q_st +
                                                              (long long)(kvh * p.group + g) * p.q_sh);
#pragma unroll
      for (int k = 0; k < KS; ++k) {
        qf[t][k][0] = ok ? __ldg(src + k * 8 + (lane & 3)) : 0u;
        qf[t][k][1] = ok ? __ldg(src + k * 8 + (lane & 3) + 4) : 0u;
      }
    }
    // ldmatrix addresses of this lane inside a stage.  K (plain): key = lane % 16, 16-byte piece 2 k + lane / 16.
    // V (transposed): key = lane % 8 + 8 (lane / 16), piece 2 k + (lane / 8) % 2.
    const uint32_t key_k = (uint32_t)(16 * warp + (lane & 15)), key_v = (uint32_t)(16 * warp + (lane & 7) + ((lane >> 4) << 3));
    const uint32_t pk = (uint32_t)(lane >> 4), pv = (uint32_t)((lane >> 3) & 1);
    int s = 0;
    uint32_t phase = 0;
    for (int j = blk0; j < blk1; ++j) {
      if (!wait_all(full_bar(s), phase)) break;
      const uint32_t ks0 = smem_base + (uint32_t)s * dec_stage_bytes(HD) + key_k * 128u;
      const uint32_t vs0 = smem_base + (uint32_t)s * dec_stage_bytes(HD) + kv_bytes + key_v * 128u;
      float sc[2][NT][4];  // two chains of sums, even and odd steps
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
          for (int i = 0; i < 4; ++i) sc[e][t][i] = 0.f;
#pragma unroll
      for (int k = 0; k < KS; ++k) {
        uint32_t a[4];
        const uint32_t piece = (uint32_t)(2 * (k & 3)) + pk;
        ptx::ldmatrix_x4(ks0 + (uint32_t)(k >> 2) * chunk_bytes + ((piece ^ (key_k & 7u)) << 4), a);
#pragma unroll
        for (int t = 0; t < NT; ++t) ptx::mma_m16n8k16_bf16(sc[k & 1][t], a, qf[t][k]);
      }
      // scores of keys lane / 4 (i = 0, 1) and lane / 4 + 8 (i = 2, 3), rows 2 (lane % 4) + (i & 1)
      const int left = p.Tk - (j * kDecBlockK + 16 * warp);  // keys of this warp's 16 that exist
      uint32_t pf[NT][2];
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        float x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = (sc[0][t][i] + sc[1][t][i]) * p.scale_log2;
        if (left < 16) {
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if ((lane >> 2) + (i >> 1) * 8 >= left) x[i] = -INFINITY;
        }
        const float mx0 = fmaxf(x[0], x[2]), mx1 = fmaxf(x[1], x[3]);
        if (__any_sync(0xffffffffu, mx0 > m[t][0] + kAttnRescaleThreshold || mx1 > m[t][1] + kAttnRescaleThreshold)) {
          float mn[2] = {mx0, mx1};
#pragma unroll
          for (int i = 0; i < 2; ++i) {  // over the eight lanes that hold the same row
            mn[i] = fmaxf(mn[i], __shfl_xor_sync(0xffffffffu, mn[i], 4));
            mn[i] = fmaxf(mn[i], __shfl_xor_sync(0xffffffffu, mn[i], 8));
            mn[i] = fmaxf(mn[i], __shfl_xor_sync(0xffffffffu, mn[i], 16));
            mn[i] = fmaxf(mn[i], m[t][i]);
            const float alpha = ptx::ex2_approx(m[t][i] - (mn[i] == -INFINITY ? 0.f : mn[i]));
            l[t][i] *= alpha;
            m[t][i] = mn[i];
#pragma unroll
            for (int k = 0; k < KS; ++k) {
              o[t][k][i] *= alpha;
              o[t][k][i + 2] *= alpha;
            }
          }
        }
        const float r0 = m[t][0] == -INFINITY ? 0.f : m[t][0], r1 = m[t][1] == -INFINITY ? 0.f : m[t][1];
        const float e0 = ptx::ex2_approx(x[0] - r0), e1 = ptx::ex2_approx(x[1] - r1);
        const float e2 = ptx::ex2_approx(x[2] - r0), e3 = ptx::ex2_approx(x[3] - r1);
        l[t][0] += e0 + e2;
        l[t][1] += e1 + e3;
        // (key, row) fragments of the accumulator become the (row, key) fragments the second product's B wants
        pf[t][0] = ptx::movmatrix_trans(pack_bf16x2(e0, e1));
        pf[t][1] = ptx::movmatrix_trans(pack_bf16x2(e2, e3));
      }
#pragma unroll
      for (int k = 0; k < KS; ++k) {
        uint32_t a[4];
        const uint32_t piece = (uint32_t)(2 * (k & 3)) + pv;
        ptx::ldmatrix_x4_trans(vs0 + (uint32_t)(k >> 2) * chunk_bytes + ((piece ^ (key_v & 7u)) << 4), a);
#pragma unroll
        for (int t = 0; t < NT; ++t) ptx::mma_m16n8k16_bf16(o[t][k], a, pf[t]);
      }
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(empty_bar(s));
      if (++s == NS) {
        s = 0;
        phase ^= 1u;
      }
    }
  }
  __syncthreads();  // every load has landed and been read: the ring becomes the partial results' place

  float* const part = reinterpret_cast<float*>(smem_raw);       // [warp][row][kPartLd]
  float* const ml = part + kDecWarps * kRows * kPartLd;         // [warp][row][2]
  float* const merged = ml + kDecWarps * kRows * 2;             // [row][kPartLd], then [row][2]
  float* const merged_ml = merged + kRows * kPartLd;
  if (warp < kDecWarps) {
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int row = 8 * t + 2 * (lane & 3) + i;
        float s = l[t][i];
        s += __shfl_xor_sync(0xffffffffu, s, 4);
        s += __shfl_xor_sync(0xffffffffu, s, 8);
        s += __shfl_xor_sync(0xffffffffu, s, 16);
        if (lane < 4) {
          ml[(warp * kRows + row) * 2] = m[t][i];
          ml[(warp * kRows + row) * 2 + 1] = s;
        }
        float* dst = part + (warp * kRows + row) * kPartLd + (lane >> 2);
#pragma unroll
        for (int k = 0; k < KS; ++k) {
          dst[16 * k] = o[t][k][i];
          dst[16 * k + 8] = o[t][k][i + 2];
        }
      }
  }
  __syncthreads();
  // n partial results (their maxima and sums at ml_of(i), outputs at part_of(i)) added up in ascending order, for four
  // columns of one row: O = sum_i 2^(m_i - M) O_i, L = sum_i 2^(m_i - M) l_i
  auto merge = [](int n, auto ml_of, auto part_of, float4& acc, float& mm, float& ll) {
    mm = -INFINITY;
    for (int i = 0; i < n; ++i) mm = fmaxf(mm, ml_of(i).x);
    ll = 0.f;
    acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int i = 0; i < n; ++i) {
      const float2 w = ml_of(i);
      const float f = w.x == -INFINITY ? 0.f : ptx::ex2_approx(w.x - mm);
      const float4 v = part_of(i);
      ll = fmaf(f, w.y, ll);
      acc.x = fmaf(f, v.x, acc.x);
      acc.y = fmaf(f, v.y, acc.y);
      acc.z = fmaf(f, v.z, acc.z);
      acc.w = fmaf(f, v.w, acc.w);
    }
  };
  auto store = [&](int row, int c, const float4& acc, float ll) {
    const float inv = ll > 0.f ? __fdividef(1.f, ll) : 0.f;
    const int tq = row / p.group, g = row - tq * p.group;
    __nv_bfloat16* dst = p.O + (long long)b * p.o_sb + (long long)tq * p.o_st + (long long)(kvh * p.group + g) * p.o_sh + c;
    uint2 w;
    w.x = pack_bf16x2(acc.x * inv, acc.y * inv);
    w.y = pack_bf16x2(acc.z * inv, acc.w * inv);
    *reinterpret_cast<uint2*>(dst) = w;
  };
  const int items = p.rows * (HD / 4);
  for (int i = (int)threadIdx.x; i < items; i += kDecThreads) {
    const int row = i / (HD / 4), c = 4 * (i - row * (HD / 4));
    float4 acc;
    float mm, ll;
    merge(
        kDecWarps, [&](int w) { return *reinterpret_cast<const float2*>(ml + (w * kRows + row) * 2); },
        [&](int w) { return *reinterpret_cast<const float4*>(part + (w * kRows + row) * kPartLd + c); }, acc, mm, ll);
    if (p.splits == 1) {
      store(row, c, acc, ll);
    } else {
      *reinterpret_cast<float4*>(merged + row * kPartLd + c) = acc;
      if (c == 0) *reinterpret_cast<float2*>(merged_ml + row * 2) = make_float2(mm, ll);
    }
  }
  if (p.splits > 1) {
    // the CTAs of the cluster share out the (row, 4 columns) items and add the runs of keys up in order
    ptx::cluster_arrive();
    ptx::cluster_wait();
    const uint32_t merged_s = ptx::smem_u32(merged), merged_ml_s = ptx::smem_u32(merged_ml);
    for (int i = rank * kDecThreads + (int)threadIdx.x; i < items; i += p.splits * kDecThreads) {
      const int row = i / (HD / 4), c = 4 * (i - row * (HD / 4));
      float4 acc;
      float mm, ll;
      merge(
          p.splits, [&](int w) { return ptx::ld_shared_cluster_f2(ptx::mapa(merged_ml_s + (uint32_t)row * 8u, (uint32_t)w)); },
          [&](int w) { return ptx::ld_shared_cluster_f4(ptx::mapa(merged_s + (uint32_t)(row * kPartLd + c) * 4u, (uint32_t)w)); },
          acc, mm, ll);
      store(row, c, acc, ll);
    }
    ptx::grid_launch_dependents();
    ptx::cluster_arrive();  // no CTA leaves while a peer may still read its shared memory
    ptx::cluster_wait();
  } else {
    ptx::grid_launch_dependents();
  }
  if (*abort_p) {  // a wait expired: give copies that may still be in flight time to land
    const unsigned long long t0 = ptx::globaltimer_ns();
    while (ptx::globaltimer_ns() - t0 < 200000ull) {
    }
  }
}

}  // namespace fact
