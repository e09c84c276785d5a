// Tree-mask attention (Section 3.2 / 4.1: every draft-tree row is verified in one forward,
// each conditioned on its own path). Row t attends cache slots [0, nvis[t]) plus the slots
// tbase[t] + b for every bit b of its 128-bit mask. Queries, keys and values are fp32 in
// memory; softmax and accumulation are fp32; the output is written as two bf16 limbs for the
// O-projection GEMM.
//
// One CTA handles one head, a block of up to 32 consecutive rows of ONE episode and one slice
// of that block's key range (split-KV). Keys and values go through shared memory in tiles of
// 32 slots, so a K/V row is read from L2/HBM once per row block instead of once per row; the
// next tile is fetched into registers while the current one is used.
//
// The two contractions run on the tensor cores with fp32-grade operands: every operand (q
// scaled, k, v, the softmax weights p) is split into two bf16 limbs (hi = bf16(x), lo =
// bf16(x - hi): 16 mantissa bits) when it is written to shared memory, and a product is three
// m16n8k16 MMAs (hi hi + hi lo + lo hi) accumulated in fp32. A tile goes through three phases
// separated by CTA barriers: scores (warp = 16 rows x 8 keys, q fragments kept in registers
// for the whole kernel), online softmax (warp = 4 rows, lane = key; running max and sum live
// in that warp's registers), weighted sum (warp = 16 rows x a quarter of the head dimension).
// With several key slices the CTAs of a row block form a thread-block cluster: each leaves
// (max, sum, unnormalised output) in its own shared memory, and after one cluster barrier
// every CTA merges a share of the rows, reading the slices over distributed shared memory in
// ascending order (deterministic; nothing goes through global memory).
#pragma once
#include <cooperative_groups.h>
#include "common.cuh"
#include "gemm_tc.cuh"

namespace attn {

constexpr int RB = 32;            // rows per block
constexpr int KT = 32;            // key slots per tile
constexpr int THREADS = 256;      // 8 warps x 4 rows
constexpr int MAX_SPLITS = 8;         // key slices per row block = cluster size (8: the portable limit)
// (32-row block, head) pairs up to which a launch takes the few-row kernel: up to 64 rows of 32 heads
// its slices are what fills the SMs. Above, 128-row blocks, which one episode has 32 of, catch up: a
// verification of 96 rows here and of 97 rows there takes 4.30 / 4.33 ms against 64 slots, 4.60 / 4.62
// against 290 and 4.97 / 4.93 against 600; a layer's attention at 128 rows 23.3 us here, 22.5 there.
constexpr int FEW_CTAS = 96;
constexpr int MAX_SPLIT_CTAS = 148;   // CTAs of a launch that uses more than one key slice

struct Args {
  const float *q;          // [rows][H * DH], already rotated
  const float *cache;      // [episode][2 (K, V)][max_seq][H * DH]
  size_t ep_stride;
  int max_seq, H;
  RowTable rt;
  float scale;
  bf16 *out;               // two limbs, [rows][H * DH] each
  size_t out_plane;
  int splits;              // few-row launches: key slices per row block; the cluster is (splits, 1, 1)
  unsigned long long wait_ns;   // long launches: limit of every mbarrier wait, and the status word
  int *err;
  int withhold_tile;       // test hook (SPECVLA_OPT_WITHHOLD_KEYS), long launches: key tile never reported (-1: none)
};

__host__ __device__ inline int blocks_of(const EpArgs &ea, int rows) {
  int n = 0;
  for (int i = 0; i < ea.n_ep; i++) n += (ea.nrows[i] + rows - 1) / rows;
  return n;
}
// Shared memory: bf16 limb planes of Q [RB], K [KT], V [KT] (row pitch DH + 8: rows 16-byte
// aligned and ldmatrix conflict-free), of P [RB][KT + 8], and the fp32 scores [RB][KT + 4].
template <int DH> constexpr int smem_bytes() {
  return (2 * (RB + 2 * KT) * (DH + 8) + 2 * RB * (KT + 8)) * (int)sizeof(bf16) + RB * (KT + 4) * (int)sizeof(float);
}

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
// c += a (16 x 16, row) * b (16 x 8, col), bf16 operands, fp32 accumulator
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// four floats -> four hi limbs and four lo limbs, 8 bytes each
__device__ __forceinline__ void split4(const float4 v, uint2 &hi, uint2 &lo) {
  const __nv_bfloat162 h01 = __floats2bfloat162_rn(v.x, v.y), h23 = __floats2bfloat162_rn(v.z, v.w);
  const float2 f01 = __bfloat1622float2(h01), f23 = __bfloat1622float2(h23);
  const __nv_bfloat162 l01 = __floats2bfloat162_rn(v.x - f01.x, v.y - f01.y);
  const __nv_bfloat162 l23 = __floats2bfloat162_rn(v.z - f23.x, v.w - f23.y);
  hi = make_uint2(*reinterpret_cast<const uint32_t *>(&h01), *reinterpret_cast<const uint32_t *>(&h23));
  lo = make_uint2(*reinterpret_cast<const uint32_t *>(&l01), *reinterpret_cast<const uint32_t *>(&l23));
}

// The few-row launches (a verification step, a draft level). SLICED: grid (row blocks x key slices,
// heads), cluster (slices, 1, 1). Launches of 75 to 96 CTAs get one slice: grid (heads, row blocks),
// output straight from the registers. With one slice in the sliced form a verification of 65 / 96 rows
// took 4.71 / 5.10 ms against 600 slots and 4.24 / 4.68 ms against 290, so 4.56 / 4.96 and 4.13 / 4.60 ms.
template <int DH, bool SLICED>
__global__ void __launch_bounds__(THREADS, 1)
tree_attention_kernel(const EpArgs ea, const Args a) {
  constexpr int PER = DH / 32;            // head-dim columns per lane in the slice merge
  constexpr int C4 = DH / 4;              // float4 per row
  constexpr int LD = DH + 8;              // pitch (bf16) of the Q, K, V limb planes
  constexpr int LP = KT + 8;              // pitch (bf16) of the P limb planes
  constexpr int LS = KT + 4;              // pitch (float) of the scores
  constexpr int NLD = KT * C4 / THREADS;  // float4 per thread per tile
  constexpr int KS = DH / 16;             // k steps of the score MMAs
  constexpr int NB = DH / 32;             // 8-column blocks of a warp's quarter of the head dim
  extern __shared__ __align__(16) unsigned char smem_raw[];
  bf16 *sQh = reinterpret_cast<bf16 *>(smem_raw);   // [RB][LD]
  bf16 *sQl = sQh + RB * LD;
  bf16 *sKh = sQl + RB * LD;                        // [KT][LD]
  bf16 *sKl = sKh + KT * LD;
  bf16 *sVh = sKl + KT * LD;
  bf16 *sVl = sVh + KT * LD;
  bf16 *sPh = sVl + KT * LD;                        // [RB][LP]
  bf16 *sPl = sPh + RB * LP;
  float *sS = reinterpret_cast<float *>(sPl + RB * LP);   // [RB][LS]
  __shared__ int s_nvis[RB], s_tbase[RB], s_kmax;
  __shared__ uint32_t s_mask[RB][4];
  __shared__ float s_corr[RB], s_m[RB], s_l[RB];
  // The GEMM that follows is let in only once the tile loop is over (pdl_launch below): its
  // waiting CTAs would otherwise take registers and shared memory and push this grid into waves.
  pdl_wait();

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int mb = warp & 1, wq = warp >> 1;         // 16-row block; key octet (scores) / head-dim quarter (sum)
  const int h = SLICED ? blockIdx.y : blockIdx.x, hd = a.H * DH;
  const int splits = SLICED ? a.splits : 1;
  int bid = SLICED ? (int)blockIdx.x / splits : (int)blockIdx.y;
  const int sp = SLICED ? (int)blockIdx.x - bid * splits : 0;
  int ei = 0;
  for (; ei < ea.n_ep; ei++) {
    const int nb = (ea.nrows[ei] + RB - 1) / RB;
    if (bid < nb) break;
    bid -= nb;
  }
  if (ei >= ea.n_ep) {
    pdl_launch();
    return;
  }
  const int row0 = ea.row0[ei] + bid * RB;
  const int nrows = min(RB, ea.nrows[ei] - bid * RB);
  const float *kbase = a.cache + (size_t)ea.eps[ei] * a.ep_stride + (size_t)h * DH;
  const float *vbase = kbase + (size_t)a.max_seq * hd;

  // the block's query rows (rows past nrows are zero): requested first, used after the metadata
  float4 qv[RB * C4 / THREADS];
#pragma unroll
  for (int k = 0; k < RB * C4 / THREADS; k++) {
    const int i = tid + k * THREADS;
    const int r = i / C4, c = i % C4;
    qv[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < nrows) qv[k] = *reinterpret_cast<const float4 *>(a.q + (size_t)(row0 + r) * hd + h * DH + c * 4);
  }
  if (tid < RB) {
    int nv = 0, tb = 0, km = 0;
    uint32_t m[4] = {0, 0, 0, 0};
    if (tid < nrows) {
      nv = a.rt.nvis[row0 + tid];
      tb = a.rt.tbase[row0 + tid];
      km = nv;
#pragma unroll
      for (int w = 0; w < 4; w++) {
        m[w] = a.rt.mask[(size_t)(row0 + tid) * 4 + w];
        if (m[w]) km = max(km, tb + 32 * w + 32 - __clz(m[w]));
      }
    }
    s_nvis[tid] = nv;
    s_tbase[tid] = tb;
#pragma unroll
    for (int w = 0; w < 4; w++) s_mask[tid][w] = m[w];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) km = max(km, __shfl_xor_sync(0xffffffffu, km, o));
    if (tid == 0) s_kmax = min(km, a.max_seq);
  }
  __syncthreads();
  const int kmax = s_kmax;
  const int tiles = (kmax + KT - 1) / KT;
  const int t0 = sp * tiles / splits, t1 = (sp + 1) * tiles / splits;

  float4 kreg[NLD], vreg[NLD];
  auto fetch = [&](int t) {
#pragma unroll
    for (int k = 0; k < NLD; k++) {
      const int i = tid + k * THREADS;
      const int slot = t * KT + i / C4, c = i % C4;
      if (slot < kmax) {
        kreg[k] = *reinterpret_cast<const float4 *>(kbase + (size_t)slot * hd + c * 4);
        vreg[k] = *reinterpret_cast<const float4 *>(vbase + (size_t)slot * hd + c * 4);
      } else {
        kreg[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        vreg[k] = kreg[k];
      }
    }
  };
  if (t0 < t1) fetch(t0);                  // in flight while the queries are split

  // the query rows, scaled, as limbs
#pragma unroll
  for (int k = 0; k < RB * C4 / THREADS; k++) {
    const int i = tid + k * THREADS;
    const int r = i / C4, c = i % C4;
    float4 v = qv[k];
    v.x *= a.scale; v.y *= a.scale; v.z *= a.scale; v.w *= a.scale;
    uint2 hi, lo;
    split4(v, hi, lo);
    *reinterpret_cast<uint2 *>(sQh + r * LD + c * 4) = hi;
    *reinterpret_cast<uint2 *>(sQl + r * LD + c * 4) = lo;
  }
  __syncthreads();

  // A fragments of this warp's 16 query rows, both limbs, for the whole kernel
  uint32_t qh[KS][4], ql[KS][4];
  {
    const int r = 16 * mb + (lane & 15), c = (lane >> 4) * 8;
#pragma unroll
    for (int ks = 0; ks < KS; ks++) {
      ldsm_x4(smem_addr(sQh + r * LD + 16 * ks + c), qh[ks]);
      ldsm_x4(smem_addr(sQl + r * LD + 16 * ks + c), ql[ks]);
    }
  }
  float m_run = -INFINITY, l_run = 0.f;   // softmax statistics of row 4 warp + lane / 8
  float acc[NB][4];                       // rows 16 mb + lane / 4 (+ 8), columns (DH / 4) wq + 8 nb + 2 (lane % 4) (+ 1)
#pragma unroll
  for (int nb = 0; nb < NB; nb++)
#pragma unroll
    for (int k = 0; k < 4; k++) acc[nb][k] = 0.f;

  for (int t = t0; t < t1; t++) {
    __syncthreads();                       // the previous tile is no longer being read
#pragma unroll
    for (int k = 0; k < NLD; k++) {
      const int i = tid + k * THREADS;
      const int j = i / C4, c = i % C4;
      uint2 hi, lo;
      split4(kreg[k], hi, lo);
      *reinterpret_cast<uint2 *>(sKh + j * LD + c * 4) = hi;
      *reinterpret_cast<uint2 *>(sKl + j * LD + c * 4) = lo;
      split4(vreg[k], hi, lo);
      *reinterpret_cast<uint2 *>(sVh + j * LD + c * 4) = hi;
      *reinterpret_cast<uint2 *>(sVl + j * LD + c * 4) = lo;
    }
    __syncthreads();
    if (t + 1 < t1) fetch(t + 1);          // in flight while this tile is used

    // ---- scores of rows 16 mb .. + 16 against keys 8 wq .. + 8
    {
      // three chains (hi hi, hi lo, lo hi) instead of one of 3 DH / 16 dependent MMAs
      float sc[4] = {0.f, 0.f, 0.f, 0.f}, sc1[4] = {0.f, 0.f, 0.f, 0.f}, sc2[4] = {0.f, 0.f, 0.f, 0.f};
      // B fragments two k steps at a time: lanes 0-7 / 8-15 address the keys' columns
      // 32 kp, 32 kp + 8 (first step), lanes 16-23 / 24-31 the columns 32 kp + 16, + 24 (second)
      const int key = 8 * wq + (lane & 7), c = (lane >> 3) * 8;
#pragma unroll
      for (int kp = 0; kp < KS / 2; kp++) {
        uint32_t bh[4], bl[4];
        ldsm_x4(smem_addr(sKh + key * LD + 32 * kp + c), bh);
        ldsm_x4(smem_addr(sKl + key * LD + 32 * kp + c), bl);
        mma_bf16(sc, qh[2 * kp], bh[0], bh[1]);
        mma_bf16(sc1, qh[2 * kp], bl[0], bl[1]);
        mma_bf16(sc2, ql[2 * kp], bh[0], bh[1]);
        mma_bf16(sc, qh[2 * kp + 1], bh[2], bh[3]);
        mma_bf16(sc1, qh[2 * kp + 1], bl[2], bl[3]);
        mma_bf16(sc2, ql[2 * kp + 1], bh[2], bh[3]);
      }
#pragma unroll
      for (int k = 0; k < 4; k++) sc[k] += sc1[k] + sc2[k];
      float *dst = sS + (16 * mb + (lane >> 2)) * LS + 8 * wq + 2 * (lane & 3);
      *reinterpret_cast<float2 *>(dst) = make_float2(sc[0], sc[1]);
      *reinterpret_cast<float2 *>(dst + 8 * LS) = make_float2(sc[2], sc[3]);
    }
    __syncthreads();
    // ---- online softmax: eight lanes per row (row 4 warp + lane / 8), a lane has the keys
    // lane % 8 + 8 j of the tile
    {
      const int r = warp * 4 + (lane >> 3), tc = lane & 7;
      const int nv = s_nvis[r], tb = s_tbase[r];
      float sv[4];
      bool vis[4];
      float mx = -INFINITY;
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const int slot = t * KT + tc + 8 * j;
        vis[j] = slot < nv;
        const int b = slot - tb;
        if (!vis[j] && b >= 0 && b < 128) vis[j] = (s_mask[r][b >> 5] >> (b & 31)) & 1u;
        sv[j] = sS[r * LS + tc + 8 * j];
        if (vis[j]) mx = fmaxf(mx, sv[j]);
      }
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
      const float mn = fmaxf(m_run, mx);
      const float corr = (mn == -INFINITY) ? 1.f : __expf(m_run - mn);
      m_run = mn;
      float ps = 0.f;
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const float p = vis[j] ? __expf(sv[j] - mn) : 0.f;
        ps += p;
        const bf16 ph = __float2bfloat16(p);
        sPh[r * LP + tc + 8 * j] = ph;
        sPl[r * LP + tc + 8 * j] = __float2bfloat16(p - __bfloat162float(ph));
      }
      ps += __shfl_xor_sync(0xffffffffu, ps, 1);
      ps += __shfl_xor_sync(0xffffffffu, ps, 2);
      ps += __shfl_xor_sync(0xffffffffu, ps, 4);
      l_run = l_run * corr + ps;
      if (tc == 0) s_corr[r] = corr;
    }
    __syncthreads();
    // ---- weighted sum: rows 16 mb .. + 16, head-dim columns (DH / 4) wq .. + DH / 4
    {
      const float c0 = s_corr[16 * mb + (lane >> 2)], c1 = s_corr[16 * mb + (lane >> 2) + 8];
#pragma unroll
      for (int nb = 0; nb < NB; nb++) {
        acc[nb][0] *= c0;
        acc[nb][1] *= c0;
        acc[nb][2] *= c1;
        acc[nb][3] *= c1;
      }
      const int pr = 16 * mb + (lane & 15), pc = (lane >> 4) * 8;
      // V fragments (transposed loads): lanes 0-7 / 8-15 address keys 16 ks .. + 8 / + 8 .. + 16
      // at one 8-column block, lanes 16-31 the same keys at the next block
      const int vk = (lane & 7) + ((lane >> 3) & 1) * 8, vc = (DH / 4) * wq + (lane >> 4) * 8;
#pragma unroll
      for (int ks = 0; ks < KT / 16; ks++) {
        uint32_t ph[4], pl[4];
        ldsm_x4(smem_addr(sPh + pr * LP + 16 * ks + pc), ph);
        ldsm_x4(smem_addr(sPl + pr * LP + 16 * ks + pc), pl);
#pragma unroll
        for (int np = 0; np < NB / 2; np++) {
          uint32_t vh[4], vl[4];
          ldsm_x4_trans(smem_addr(sVh + (16 * ks + vk) * LD + vc + 16 * np), vh);
          ldsm_x4_trans(smem_addr(sVl + (16 * ks + vk) * LD + vc + 16 * np), vl);
          mma_bf16(acc[2 * np], ph, vh[0], vh[1]);
          mma_bf16(acc[2 * np], ph, vl[0], vl[1]);
          mma_bf16(acc[2 * np], pl, vh[0], vh[1]);
          mma_bf16(acc[2 * np + 1], ph, vh[2], vh[3]);
          mma_bf16(acc[2 * np + 1], ph, vl[2], vl[3]);
          mma_bf16(acc[2 * np + 1], pl, vh[2], vh[3]);
        }
      }
    }
  }

  pdl_launch();
  if ((lane & 7) == 0) {
    s_m[warp * 4 + (lane >> 3)] = m_run;
    s_l[warp * 4 + (lane >> 3)] = l_run;
  }
  __syncthreads();
  const int ra = 16 * mb + (lane >> 2), rb = ra + 8;        // this thread's two rows
  const int cbase = (DH / 4) * wq + 2 * (lane & 3);          // + 8 nb: its column pairs
  if (!SLICED) {
    const float ia = 1.f / s_l[ra], ib = 1.f / s_l[rb];
#pragma unroll
    for (int nb = 0; nb < NB; nb++) {
#pragma unroll
      for (int half = 0; half < 2; half++) {
        const int r = half ? rb : ra;
        if (r >= nrows) continue;
        const float inv = half ? ib : ia;
        const float v0 = acc[nb][2 * half] * inv, v1 = acc[nb][2 * half + 1] * inv;
        const size_t idx = (size_t)(row0 + r) * hd + h * DH + cbase + 8 * nb;
        const __nv_bfloat162 hi = __floats2bfloat162_rn(v0, v1);
        const float2 hf = __bfloat1622float2(hi);
        *reinterpret_cast<__nv_bfloat162 *>(a.out + idx) = hi;
        *reinterpret_cast<__nv_bfloat162 *>(a.out + a.out_plane + idx) = __floats2bfloat162_rn(v0 - hf.x, v1 - hf.y);
      }
    }
    return;
  }

  // leave this slice in shared memory (over the query planes, which were
  // only needed for the fragments), then merge rows sp, sp + splits, ... from all slices
  constexpr int LO = DH + 4;
  float *sO = reinterpret_cast<float *>(smem_raw);          // [RB][LO]: output, then max and sum
#pragma unroll
  for (int nb = 0; nb < NB; nb++) {
    *reinterpret_cast<float2 *>(sO + ra * LO + cbase + 8 * nb) = make_float2(acc[nb][0], acc[nb][1]);
    *reinterpret_cast<float2 *>(sO + rb * LO + cbase + 8 * nb) = make_float2(acc[nb][2], acc[nb][3]);
  }
  if (tid < RB) {
    sO[tid * LO + DH] = s_m[tid];
    sO[tid * LO + DH + 1] = s_l[tid];
  }
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  for (int r = sp + splits * warp; r < nrows; r += splits * (THREADS / 32)) {
    // every load of the row's slices is issued before any is used: one latency, not one per slice
    float ms[MAX_SPLITS], ls[MAX_SPLITS], os[MAX_SPLITS][PER];
#pragma unroll
    for (int s2 = 0; s2 < MAX_SPLITS; s2++) {
      if (s2 < splits) {
        const float *src = cluster.map_shared_rank(sO, (unsigned)s2) + r * LO;
        ms[s2] = src[DH];
        ls[s2] = src[DH + 1];
        if (PER == 4) {
          const float4 t4 = *reinterpret_cast<const float4 *>(src + lane * 4);
          os[s2][0] = t4.x; os[s2][1] = t4.y; os[s2][2 % PER] = t4.z; os[s2][3 % PER] = t4.w;
        } else {
          const float2 t2 = *reinterpret_cast<const float2 *>(src + lane * 2);
          os[s2][0] = t2.x; os[s2][1] = t2.y;
        }
      }
    }
    float M = -INFINITY;
#pragma unroll
    for (int s2 = 0; s2 < MAX_SPLITS; s2++)
      if (s2 < splits) M = fmaxf(M, ms[s2]);
    float L = 0.f, o[PER];
#pragma unroll
    for (int k = 0; k < PER; k++) o[k] = 0.f;
#pragma unroll
    for (int s2 = 0; s2 < MAX_SPLITS; s2++)
      if (s2 < splits) {
        const float c = (ms[s2] == -INFINITY) ? 0.f : __expf(ms[s2] - M);
        L += ls[s2] * c;
#pragma unroll
        for (int k = 0; k < PER; k++) o[k] += os[s2][k] * c;
      }
    const float inv = 1.f / L;
#pragma unroll
    for (int k = 0; k < PER; k++) {
      const size_t idx = (size_t)(row0 + r) * hd + h * DH + lane * PER + k;
      const float v = o[k] * inv;
      const bf16 hi = __float2bfloat16(v);
      a.out[idx] = hi;
      a.out[a.out_plane + idx] = __float2bfloat16(v - __bfloat162float(hi));
    }
  }
  // nobody leaves while a peer may still be reading its shared memory (relaxed: nothing is handed over, and
  // a releasing arrival would first wait for the output's stores)
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Launches with enough row blocks to fill the SMs without slicing keys (prefill, batched
// verification): the two products on tcgen05.
//
// mma.sync runs at an eighth of the tcgen05 rate on this chip (23 clocks per m16n8k16 and scheduler
// measured), and with three limb products per contraction it bounded these launches, whatever the
// split of rows and keys over warps. Here a CTA takes 128 rows of one episode and one head:
//   warps 0-3   own a row per thread: scores from TMEM, mask, online softmax, weights back to TMEM as
//               the A operand of the second product (two limbs), rescaling of O when a maximum moved;
//   warps 4-11  load K and V tiles of 64 slots (fp32, the next tile's loads in flight while this one
//               is converted), split them into bf16 limbs and write them as swizzled K-major operands:
//               K as [slot][dim], V transposed; two buffers. A thread transposes 8 slots x 4 dims of V;
//               its four rows of V^T are DH / 4 apart, so that a warp's stores meet no bank twice: row
//               j DH / 4 + i is dim 4 i + j, and so is column j DH / 4 + i of O;
//   warp 12     issues the MMAs: S = Q K^T (hi hi in one accumulator, hi lo + lo hi in another, two
//               buffers), O += P V (three products).
// A row's weight of a slot that it does not see is zero, and zero times a value that is not finite is
// NaN: in a block of 128 causal rows one such V row would reach up to 127 rows before it (32 in the
// few-row kernel, whose tiles 32 rows share). So once the context has cached K and V of a row that is
// not finite (the QKV GEMM, which has the row's sum of squares, says so in a flag), the loaders write
// zeros in place of such values, and the rows that do see them get their NaN on the way out. (Checked in
// every loader, without that flag, it cost 1 us per launch; in the finishing loop of QKV, 0.2 us.)
// The scores of tile t + 1 are computed while the softmax of tile t runs. Arithmetic as in the few-row
// kernel: 16 mantissa bits per operand, fp32 accumulation and softmax.
// Per launch (32 heads of 128; the mma.sync kernel with one CTA per 32 rows before): 16 prefixes of
// 296 rows 474 -> 219 us, one of 290 rows 27.4 -> 18.6 us, 8 trees of 27 rows against 290 slots 72 ->
// 57 us. A tile takes 3500 clocks, bound by the softmax threads (about 2800) and the hand-overs; a
// CTA spends another 5300 on queries and first tile and 3200 on its output.
// Grid (heads, row blocks), the blocks taken last to first: causal rows make the late blocks of an
// episode the long ones, and CTAs are handed out x first, so every head's longest block starts
// before any short one.
constexpr int TC_ROWS = 128, TC_KEYS = 64, TC_LOADERS = 256, TC_THREADS = 128 + TC_LOADERS + 32;
template <int DH> __host__ __device__ constexpr int tc_q_bytes() { return TC_ROWS * DH * 2; }          // one limb
template <int DH> __host__ __device__ constexpr int tc_kv_bytes() { return TC_KEYS * DH * 2; }         // one limb of K or of V
template <int DH> __host__ __device__ constexpr int tc_smem_bytes() { return 2 * tc_q_bytes<DH>() + 8 * tc_kv_bytes<DH>() + 1024; }
constexpr uint32_t TC_S = 0, TC_P = 256, TC_O = 320;       // TMEM columns: S [2][main 64 | cross 64], P hi | lo, O

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void st_shared16(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
// eight floats -> 16 bytes of hi limbs and 16 bytes of lo limbs
__device__ __forceinline__ void store_split8(uint32_t hi_addr, uint32_t lo_addr, const float (&v)[8]) {
  uint2 h0, l0, h1, l1;
  split4(make_float4(v[0], v[1], v[2], v[3]), h0, l0);
  split4(make_float4(v[4], v[5], v[6], v[7]), h1, l1);
  st_shared16(hi_addr, h0.x, h0.y, h1.x, h1.y);
  st_shared16(lo_addr, l0.x, l0.y, l1.x, l1.y);
}

template <int DH>
__global__ void __launch_bounds__(TC_THREADS, 1)
row_attention_kernel(const EpArgs ea, const Args a) {
  using namespace gemm_tc;
  constexpr int QB = tc_q_bytes<DH>(), KVB = tc_kv_bytes<DH>();
  constexpr int C8 = DH / 8;                       // 16-byte chunks (8 dims) per row
  constexpr int C4 = DH / 4;                       // float4 per row
  constexpr int NKC = TC_KEYS * C8 / TC_LOADERS;   // K chunks per loader thread and tile
  static_assert((TC_KEYS / 8) * C4 <= TC_LOADERS, "one 8 x 4 piece of V per loader thread");
  extern __shared__ unsigned char smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  // Q hi | Q lo | per buffer: K hi | K lo | V^T hi | V^T lo
  auto kv_base = [&](int b) { return base + (uint32_t)(2 * QB + b * 4 * KVB); };
  __shared__ __align__(8) unsigned long long s_bar[10];
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail, s_clean, s_non_finite;
  const uint32_t bars = smem_u32(s_bar);
  auto k_full = [&](int b) { return bars + 8u * b; };           // the loaders have written K (V) of buffer b
  auto v_full = [&](int b) { return bars + 8u * (2 + b); };
  auto s_full = [&](int b) { return bars + 8u * (4 + b); };     // scores are in S buffer b, K of buffer b is free
  auto v_free = [&](int b) { return bars + 8u * (6 + b); };     // V of buffer b is free
  const uint32_t p_full = bars + 8u * 8, o_full = bars + 8u * 9;   // weights are in TMEM / O includes their tile

  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  if (tid == 0) {
    for (int b = 0; b < 2; b++) {
      mbar_init(k_full(b), TC_LOADERS / 32);
      mbar_init(v_full(b), TC_LOADERS / 32);
      mbar_init(v_free(b), 1);
      mbar_init(s_full(b), 1);
    }
    mbar_init(p_full, 4);
    mbar_init(o_full, 1);
    s_fail = s_non_finite = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 12) {
    tc_alloc(smem_u32(&s_tmem), 512);
    tc_relinquish();
  }
  pdl_wait();

  const int h = blockIdx.x, hd = a.H * DH;
  int bid = (int)gridDim.y - 1 - (int)blockIdx.y, ei = 0;
  for (; ei + 1 < ea.n_ep; ei++) {
    const int nb = (ea.nrows[ei] + TC_ROWS - 1) / TC_ROWS;
    if (bid < nb) break;
    bid -= nb;
  }
  const int row0 = ea.row0[ei] + bid * TC_ROWS;
  const int nrows = min(TC_ROWS, ea.nrows[ei] - bid * TC_ROWS);
  const float *kbase = a.cache + (size_t)ea.eps[ei] * a.ep_stride + (size_t)h * DH;
  const float *vbase = kbase + (size_t)a.max_seq * hd;

  int flag = 0;
  if (tid == TC_THREADS - 1) flag = a.err[SV_NON_FINITE_V];     // (in flight with the row tables)
  // last slot that any row sees: every warp finds it for itself
  int kmax = 0;
  {
    int vis[TC_ROWS / 32], at[TC_ROWS / 32];
    uint4 m[TC_ROWS / 32];
#pragma unroll
    for (int k = 0; k < TC_ROWS / 32; k++) {               // (all loads first)
      const int r = row0 + min(lane + 32 * k, nrows - 1);
      vis[k] = a.rt.nvis[r];
      at[k] = a.rt.tbase[r];
      m[k] = *reinterpret_cast<const uint4 *>(a.rt.mask + (size_t)r * 4);
    }
#pragma unroll
    for (int k = 0; k < TC_ROWS / 32; k++) {
      const int last = m[k].w ? 128 - __clz(m[k].w) : m[k].z ? 96 - __clz(m[k].z) : m[k].y ? 64 - __clz(m[k].y)
                       : m[k].x ? 32 - __clz(m[k].x) : 0;
      kmax = max(kmax, max(vis[k], last ? at[k] + last : 0));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) kmax = max(kmax, __shfl_xor_sync(0xffffffffu, kmax, o));
  kmax = min(kmax, a.max_seq);
  const int tiles = (kmax + TC_KEYS - 1) / TC_KEYS;
  if (tid == TC_THREADS - 1) s_clean = flag;

  // the loaders' first tile is on its way while the others prepare the queries
  const int lt = tid - 128;
  const int vg = lt / C4, vd = lt % C4;                     // V: this thread's slot group and float4 of dims
  float4 kr[NKC][2], vr[8];
  auto load_k = [&](int t) {
#pragma unroll
    for (int k = 0; k < NKC; k++) {
      const int i = lt + k * TC_LOADERS, slot = t * TC_KEYS + i / C8;
      kr[k][0] = kr[k][1] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (slot < kmax) {
        const float4 *p = reinterpret_cast<const float4 *>(kbase + (size_t)slot * hd + (i % C8) * 8);
        kr[k][0] = p[0];
        kr[k][1] = p[1];
      }
    }
  };
  auto load_v = [&](int t) {
    const float *p = vbase + (size_t)(t * TC_KEYS + vg * 8) * hd + vd * 4;
#pragma unroll
    for (int j = 0; j < 8; j++) {
      vr[j] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (vg < TC_KEYS / 8 && t * TC_KEYS + vg * 8 + j < kmax) vr[j] = *reinterpret_cast<const float4 *>(p + (size_t)j * hd);
    }
  };
  const bool loader = warp >= 4 && warp < 12;
  if (loader && tiles > 0) {
    load_k(0);
    load_v(0);
  }
  // what this thread's row sees (warps 0-3): slots [0, nv) and bits of a 128-bit mask from slot tb on
  int nv = 0, tb = 0;
  unsigned long long mlo = 0, mhi = 0;
  if (warp < 4) {
    if (tid < nrows) {
      const int r = row0 + tid;
      nv = a.rt.nvis[r];
      tb = a.rt.tbase[r];
      const uint4 m = *reinterpret_cast<const uint4 *>(a.rt.mask + (size_t)r * 4);
      mlo = m.x | ((unsigned long long)m.y << 32);
      mhi = m.z | ((unsigned long long)m.w << 32);
    }
  }
  // the query rows, scaled, as limbs (rows past nrows are zero): blocks of 64 dims, 128-byte rows
  if (warp < 12) {
    constexpr int QT = 128 + TC_LOADERS, NQ = (TC_ROWS * C8 + QT - 1) / QT;
    float4 x[NQ][2];
#pragma unroll
    for (int k = 0; k < NQ; k++) {
      const int i = tid + k * QT, r = i / C8;
      x[k][0] = x[k][1] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r < nrows) {
        const float4 *p = reinterpret_cast<const float4 *>(a.q + (size_t)(row0 + r) * hd + h * DH + (i % C8) * 8);
        x[k][0] = p[0];
        x[k][1] = p[1];
      }
    }
#pragma unroll
    for (int k = 0; k < NQ; k++) {
      const int i = tid + k * QT, r = i / C8, c = i % C8;
      if (r >= TC_ROWS) break;
      const uint32_t at = base + (uint32_t)((c >> 3) * (TC_ROWS * 128) + r * 128 + (((c & 7) ^ (r & 7)) << 4));
      const float v[8] = {x[k][0].x * a.scale, x[k][0].y * a.scale, x[k][0].z * a.scale, x[k][0].w * a.scale,
                          x[k][1].x * a.scale, x[k][1].y * a.scale, x[k][1].z * a.scale, x[k][1].w * a.scale};
      store_split8(at, at + QB, v);
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, s_tmem, 0);
  const bool clean = s_clean != 0;
  auto fail = [&](int code) {
    atomicExch(a.err, code);
    s_fail = 1;
  };

  if (loader) {
    // ------------------------------------------------------------------ loaders
    for (int t = 0; t < tiles; t++) {
      const int b = t & 1;
      bool ok = t < 2 || mbar_wait(s_full(b), ((t >> 1) - 1) & 1, a.wait_ns);
      if (!__all_sync(0xffffffffu, ok)) {
        if (lane == 0) fail(SV_ERR_WAIT_EMPTY);
        break;
      }
      const uint32_t kb = kv_base(b);
#pragma unroll
      for (int k = 0; k < NKC; k++) {
        const int i = lt + k * TC_LOADERS, key = i / C8, c = i % C8;
        const uint32_t at = kb + (uint32_t)((c >> 3) * (TC_KEYS * 128) + key * 128 + (((c & 7) ^ (key & 7)) << 4));
        const float v[8] = {kr[k][0].x, kr[k][0].y, kr[k][0].z, kr[k][0].w, kr[k][1].x, kr[k][1].y, kr[k][1].z, kr[k][1].w};
        store_split8(at, at + KVB, v);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0 && t != a.withhold_tile) mbar_arrive(k_full(b));
      if (t + 1 < tiles) load_k(t + 1);
      ok = t < 2 || mbar_wait(v_free(b), ((t >> 1) - 1) & 1, a.wait_ns);
      if (!__all_sync(0xffffffffu, ok)) {
        if (lane == 0) fail(SV_ERR_WAIT_EMPTY);
        break;
      }
      if (clean) {
        bool bad = false;
        auto drop = [&](float &x) {
          if (!limb_finite(x)) {
            x = 0.f;
            bad = true;
          }
        };
#pragma unroll
        for (int j = 0; j < 8; j++) {
          drop(vr[j].x);
          drop(vr[j].y);
          drop(vr[j].z);
          drop(vr[j].w);
        }
        if (bad) s_non_finite = 1;
      }
      if (vg < TC_KEYS / 8) {
        const float v[4][8] = {{vr[0].x, vr[1].x, vr[2].x, vr[3].x, vr[4].x, vr[5].x, vr[6].x, vr[7].x},
                               {vr[0].y, vr[1].y, vr[2].y, vr[3].y, vr[4].y, vr[5].y, vr[6].y, vr[7].y},
                               {vr[0].z, vr[1].z, vr[2].z, vr[3].z, vr[4].z, vr[5].z, vr[6].z, vr[7].z},
                               {vr[0].w, vr[1].w, vr[2].w, vr[3].w, vr[4].w, vr[5].w, vr[6].w, vr[7].w}};
#pragma unroll
        for (int j = 0; j < 4; j++) {
          const int r = j * C4 + vd;
          const uint32_t at = kb + (uint32_t)(2 * KVB + r * 128 + ((vg ^ (r & 7)) << 4));
          store_split8(at, at + KVB, v[j]);
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(v_full(b));
      if (t + 1 < tiles) load_v(t + 1);
    }
    __syncwarp();
    if (clean) asm volatile("bar.arrive 1, %0;" ::"n"(128 + TC_LOADERS) : "memory");   // s_non_finite is final
  } else if (warp == 12) {
    // ------------------------------------------------------------------ MMA issuer
    const bool lead = elect_one();
    constexpr uint32_t idesc_s = instr_desc(TC_KEYS), idesc_o = instr_desc(DH);
    auto scores = [&](int t) {
      const int b = t & 1;
      const bool ok = mbar_wait(k_full(b), (t >> 1) & 1, a.wait_ns);
      if (!__all_sync(0xffffffffu, ok)) return false;
      tc_fence_after();
      const uint64_t qh = smem_desc(base), ql = smem_desc(base + QB);
      const uint64_t kh = smem_desc(kv_base(b)), kl = smem_desc(kv_base(b) + KVB);
      const uint32_t s0 = tmem + TC_S + (uint32_t)(b * 128), s1 = s0 + 64;
      if (lead) {
#pragma unroll
        for (int ks = 0; ks < DH / 16; ks++) {
          const uint64_t qo = (uint64_t)(((ks >> 2) * (TC_ROWS * 128) + (ks & 3) * 32) >> 4);
          const uint64_t ko = (uint64_t)(((ks >> 2) * (TC_KEYS * 128) + (ks & 3) * 32) >> 4);
          tc_mma(s0, qh + qo, kh + ko, idesc_s, ks > 0 ? 1u : 0u);
          tc_mma(s1, qh + qo, kl + ko, idesc_s, ks > 0 ? 1u : 0u);
          tc_mma(s1, ql + qo, kh + ko, idesc_s, 1u);
        }
        tc_commit(s_full(b));
      }
      __syncwarp();
      return true;
    };
    bool ok = tiles == 0 || scores(0);
    for (int t = 0; ok && t < tiles; t++) {
      // whichever comes first: the next tile's keys (its S buffer was read before the weights of tile
      // t - 1 were reported), or this tile's weights
      bool next_done = t + 1 >= tiles;
      uint64_t t0 = 0;
      for (int spin = 0;; spin++) {
        if (!next_done && __all_sync(0xffffffffu, mbar_test(k_full((t + 1) & 1), ((t + 1) >> 1) & 1))) {
          ok = scores(t + 1);
          next_done = true;
        }
        if (!ok || __all_sync(0xffffffffu, mbar_test(p_full, t & 1))) break;
        if ((spin & 1023) == 1023) {
          const uint64_t now = global_ns();
          if (t0 == 0) t0 = now;
          ok = __all_sync(0xffffffffu, now - t0 <= a.wait_ns);
        }
      }
      if (!ok) break;
      ok = mbar_wait(v_full(t & 1), (t >> 1) & 1, a.wait_ns);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const uint32_t vb = kv_base(t & 1) + 2 * KVB;
      const uint64_t vh = smem_desc(vb), vl = smem_desc(vb + KVB);
      const uint32_t ph = tmem + TC_P, pl = ph + 32, o = tmem + TC_O;
      if (lead) {
#pragma unroll
        for (int ks = 0; ks < TC_KEYS / 16; ks++) {
          const uint64_t vo = (uint64_t)((ks * 32) >> 4);
          tc_mma_ta(o, ph + ks * 8, vh + vo, idesc_o, (t > 0 || ks > 0) ? 1u : 0u);
          tc_mma_ta(o, ph + ks * 8, vl + vo, idesc_o, 1u);
          tc_mma_ta(o, pl + ks * 8, vh + vo, idesc_o, 1u);
        }
        tc_commit(v_free(t & 1));
        tc_commit(o_full);
      }
      __syncwarp();
      if (!next_done) ok = scores(t + 1);
    }
    if (!ok && lead) fail(SV_ERR_WAIT_FULL);
    __syncwarp();
  } else if (warp < 4) {
    // ------------------------------------------------------------------ softmax: row tid
    const uint32_t tl = tmem + ((uint32_t)(warp * 32) << 16);
    float m = -INFINITY, l = 0.f;
    bool ok = true;
    for (int t = 0; t < tiles; t++) {
      ok = mbar_wait(s_full(t & 1), (t >> 1) & 1, a.wait_ns);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      float s[TC_KEYS];
#pragma unroll
      for (int c = 0; c < TC_KEYS; c += 32) {
        uint32_t x[32], y[32];
        tmem_ld32(tl + TC_S + (uint32_t)((t & 1) * 128 + c), x);
        tmem_ld32(tl + TC_S + (uint32_t)((t & 1) * 128 + 64 + c), y);
        tc_wait_ld();
#pragma unroll
        for (int j = 0; j < 32; j++) s[c + j] = __uint_as_float(x[j]) + __uint_as_float(y[j]);
      }
      // which of the tile's slots the row sees
      const int p = nv - t * TC_KEYS, off = tb - t * TC_KEYS;
      unsigned long long vis = p >= 64 ? ~0ull : p > 0 ? (1ull << p) - 1ull : 0ull;
      if (off >= 0) {
        if (off < 64) vis |= mlo << off;
      } else if (off > -64) {
        vis |= (mlo >> -off) | (mhi << (64 + off));
      } else if (off > -128) {
        vis |= mhi >> (-off - 64);
      }
      if (!__all_sync(0xffffffffu, vis == ~0ull)) {
        const uint32_t v0 = (uint32_t)vis, v1 = (uint32_t)(vis >> 32);
#pragma unroll
        for (int j = 0; j < 32; j++) {
          if (!((v0 >> j) & 1u)) s[j] = -INFINITY;
          if (!((v1 >> j) & 1u)) s[32 + j] = -INFINITY;
        }
      }
      float mx[4] = {m, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int j = 0; j < TC_KEYS; j++) mx[j & 3] = fmaxf(mx[j & 3], s[j]);
      const float mn = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
      const float z = mn == -INFINITY ? 0.f : mn;            // (a row that has seen nothing yet: weights of zero)
      const float corr = mn == -INFINITY ? 1.f : __expf(m - mn);
      const bool moved = __any_sync(0xffffffffu, mn != m);
      m = mn;
      float ps[4] = {0.f, 0.f, 0.f, 0.f};
      uint32_t hi[32], lo[32];
#pragma unroll
      for (int j = 0; j < TC_KEYS; j += 4) {
        const float4 e = make_float4(__expf(s[j] - z), __expf(s[j + 1] - z), __expf(s[j + 2] - z), __expf(s[j + 3] - z));
        ps[0] += e.x; ps[1] += e.y; ps[2] += e.z; ps[3] += e.w;
        uint2 eh, el;
        split4(e, eh, el);
        hi[j / 2] = eh.x; hi[j / 2 + 1] = eh.y;
        lo[j / 2] = el.x; lo[j / 2 + 1] = el.y;
      }
      l = l * corr + ((ps[0] + ps[1]) + (ps[2] + ps[3]));
      if (t > 0) {
        // the previous tile's product has read the weights and written O
        ok = mbar_wait(o_full, (t - 1) & 1, a.wait_ns);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
        if (moved) {
#pragma unroll 1
          for (int c = 0; c < DH; c += 32) {
            uint32_t o[32];
            tmem_ld32(tl + TC_O + c, o);
            tc_wait_ld();
#pragma unroll
            for (int j = 0; j < 32; j++) o[j] = __float_as_uint(__uint_as_float(o[j]) * corr);
            tc_st32(tl + TC_O + c, o);
          }
        }
      }
      tc_st32(tl + TC_P, hi);
      tc_st32(tl + TC_P + 32, lo);
      tc_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(p_full);
    }
    if (ok && tiles > 0) {
      ok = mbar_wait(o_full, (tiles - 1) & 1, a.wait_ns);
      ok = __all_sync(0xffffffffu, ok);
      tc_fence_after();
    }
    if (!ok && lane == 0) fail(SV_ERR_WAIT_TMEM_FULL);
    // output limbs, through the query planes (every product has been computed): rows of DH + 8 elements
    constexpr int LD = DH + 8;
    bf16 *oh = reinterpret_cast<bf16 *>(smem_raw + (base - smem_u32(smem_raw))) + warp * 32 * LD;
    bf16 *ol = oh + TC_ROWS * LD;
    const float inv = 1.f / l;
    if (ok) {
#pragma unroll 1
      for (int c = 0; c < C4; c += 8) {                    // dims 4 c .. 4 c + 31: eight columns of each quarter
        uint32_t o0[8], o1[8], o2[8], o3[8];
        tc_ld8(tl + TC_O + c, o0);
        tc_ld8(tl + TC_O + C4 + c, o1);
        tc_ld8(tl + TC_O + 2 * C4 + c, o2);
        tc_ld8(tl + TC_O + 3 * C4 + c, o3);
        tc_wait_ld();
#pragma unroll
        for (int j = 0; j < 8; j++) {
          uint2 eh, el;
          split4(make_float4(__uint_as_float(o0[j]) * inv, __uint_as_float(o1[j]) * inv, __uint_as_float(o2[j]) * inv,
                             __uint_as_float(o3[j]) * inv), eh, el);
          *reinterpret_cast<uint2 *>(oh + lane * LD + 4 * (c + j)) = eh;
          *reinterpret_cast<uint2 *>(ol + lane * LD + 4 * (c + j)) = el;
        }
      }
      __syncwarp();
      for (int i = lane; i < 32 * C8; i += 32) {
        const int r = warp * 32 + i / C8, c = (i % C8) * 8;
        if (r >= nrows) break;
        const size_t idx = (size_t)(row0 + r) * hd + h * DH + c;
        *reinterpret_cast<uint4 *>(a.out + idx) = *reinterpret_cast<const uint4 *>(oh + (i / C8) * LD + c);
        *reinterpret_cast<uint4 *>(a.out + a.out_plane + idx) = *reinterpret_cast<const uint4 *>(ol + (i / C8) * LD + c);
      }
    }
    __syncwarp();
    if (clean) {
      asm volatile("bar.sync 1, %0;" ::"n"(128 + TC_LOADERS) : "memory");
      if (ok && s_non_finite) {
        // NaN for the rows of this warp that see a slot whose V is not finite, in the dims where it is not
#pragma unroll 1
        for (int slot = 0; slot < kmax; slot++) {
          const int bit = slot - tb;
          const unsigned long long m64 = bit < 64 ? mlo : mhi;
          const unsigned sees = __ballot_sync(0xffffffffu, slot < nv || (bit >= 0 && bit < 128 && ((m64 >> (bit & 63)) & 1ull)));
#pragma unroll 1
          for (int c = lane; c < DH; c += 32) {
            if (limb_finite(vbase[(size_t)slot * hd + c])) continue;
#pragma unroll 1
            for (unsigned rest = sees; rest; rest &= rest - 1) {
              const size_t idx = (size_t)(row0 + warp * 32 + __ffs(rest) - 1) * hd + h * DH + c;
              a.out[idx] = a.out[a.out_plane + idx] = __float2bfloat16(NAN);
            }
          }
        }
      }
    }
    tc_fence_before();
  }
  pdl_launch();
  __syncthreads();
  tc_fence_after();
  if (s_fail) {
    const uint64_t t0 = global_ns();
    while (global_ns() - t0 < 200000ull) __nanosleep(1000);
  }
  if (warp == 12) tc_dealloc(tmem, 512);
}

}  // namespace attn
