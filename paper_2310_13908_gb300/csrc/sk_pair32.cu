// sk_pair32.cu -- kernels and launchers of the FP32-compensated pair sums
// (device code in sk_pair32.cuh).
#include "sk_pair32.cuh"

namespace sk {
namespace {

using namespace p32;

// One work item (target block tb, source chunk ch) per CTA. In the fused
// kernel (many target blocks) the CTA that completes a block's last chunk
// finishes that block (FP64 near sums, chunk merge): that FP64 work then runs
// beside other CTAs' FP32 pair work instead of in kernels of its own. With
// few blocks a block's finish on one CTA would become the tail, so the plain
// kernel is followed by the finish kernels below.
template <class L, int NP, int TPB, int MINB>
__global__ void __launch_bounds__(TPB, MINB) k_pair32(PairArgs a) {
  extern __shared__ __align__(128) float4 sm[];
  __shared__ PipeSmem<pair_stages<L, NP, TPB>()> ps;
  if (threadIdx.x == 0) ps.initialized = 0;
  const int tb = blockIdx.x / a.n_chunks, ch = blockIdx.x % a.n_chunks;
  pair_item<L, NP, TPB>(a, tb, chunk_tiles(a, ch), sm, ps);
}

template <class L, int NP, int MINB>
__global__ void __launch_bounds__(TPB32, MINB)
    k_pair32_fused(PairArgs a, OverflowArgs oa, FinishArgs fa, int* __restrict__ tb_done,
                   int64_t M) {
  extern __shared__ __align__(128) float4 sm[];
  __shared__ PipeSmem<pair_stages<L, NP>()> ps;
  __shared__ int s_last;
  if (threadIdx.x == 0) ps.initialized = 0;
  const int tb = blockIdx.x / a.n_chunks, ch = blockIdx.x % a.n_chunks;
  pair_item<L, NP>(a, tb, chunk_tiles(a, ch), sm, ps);
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();  // this chunk's partials and near-list entries before the count
    s_last = atomicAdd(&tb_done[tb], 1) == a.n_chunks - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  constexpr int TB = TPB32 * 2 * NP;  // targets per block
  // the source stages are free now: the finish buckets the near lists there
  static_assert(pair_smem_bytes<L, NP>() / 4 >= (size_t)(TPB32 / 32) * near_warp_words(64 * NP),
                "finish scratch");
  finish_block<L, 64 * NP>(oa, fa, M, (int64_t)tb * TB, TB, reinterpret_cast<unsigned*>(sm));
}

// Separate finish for grids too small to fuse it: FIN_PARTS CTAs per target
// group of G targets, each with its share of the targets (and the whole list,
// of which it keeps its own), the near-sum scratch in dynamic shared memory.
// Bound by the FP64 pipe (60% busy) and the latency of its phases; small grids
// by how many SMs get a share. Single layer: 72 us at 24,576 targets (64 chunks, 12
// near pairs per target), 16 us at 1,944, 22 us at 5,766; one CTA per group with a
// thread per target 104, 47 and 61 us; one warp per share instead of four 112 us at
// 24,576 targets.
constexpr int FIN_PARTS = 4, FIN_THREADS = 128;
template <class L, int G>
__global__ void __launch_bounds__(FIN_THREADS) k_finish32(OverflowArgs oa, FinishArgs a,
                                                           int64_t M) {
  extern __shared__ __align__(16) unsigned fsm[];
  constexpr int KP = G / FIN_PARTS;
  const int64_t g = blockIdx.x / FIN_PARTS;
  const int k0 = (int)(blockIdx.x % FIN_PARTS) * KP;
  overflow_targets<L, G>(oa, g, k0, k0 + KP, M);
  int cnt = near_group<L, G, FIN_THREADS>(
      oa, a, g, k0, k0 + KP, fsm, reinterpret_cast<double*>(fsm + near_warp_words(G)), threadIdx.x,
      [&](int64_t t, bool valid, int sub, double n0, double n1, double n2) {
        finish_merge<fin_subs(G)>(a, t, valid && t < M, sub, n0, n1, n2);
      });
  // count near pairs: one atomic per warp
  for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(FULL, cnt, o);
  if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(a.flags + FLAG_NEAR_PAIRS, (unsigned long long)cnt);
  __syncthreads();  // these targets are finished: their partials are dead
  discard_block_partials(a, g * G + k0, KP, threadIdx.x, blockDim.x);
}

}  // namespace

template <class L, int NP>
void launch_pair32_t(const EvalBufs& b, float rt_ratio, double scale,
                     cudaStream_t st, cudaEvent_t pair_end) {
  constexpr int MINB = NP == 2 ? PAIR32_MINB_NP2 : PAIR32_MINB_NP1;
  const unsigned grid = (unsigned)((b.M_pad / (TPB32 * 2 * NP)) * b.n_chunks);
  const size_t smem = pair_smem_bytes<L, NP>();
  PairArgs a{b.srcF,  b.segbox,   b.src_orig, b.meta,     b.tgtF, b.M_pad,
             b.n_chunks, b.part, b.near_cnt, b.near_idx, b.flags, rt_ratio, b.srcLo};
  OverflowArgs oa{b.srcF, b.segbox, b.src_orig, b.meta,  b.tgtF,  b.tgt64,     b.near_cnt,
                  b.src_xyz, b.src_w, b.dens,   b.nrm, scale, b.flags, b.near_ovf};
  FinishArgs fa{b.tgt64, b.tgt_perm, b.M_pad, b.n_chunks, b.part, b.near_cnt, b.near_idx,
                b.near_ovf, b.src_xyz, b.src_w, b.dens, b.nrm, scale, b.u, b.flags};
  oa.group = fa.group = 64 * NP;
  oa.rt_ratio = rt_ratio;
  if (b.fuse_finish) {
    cudaFuncSetAttribute(k_pair32_fused<L, NP, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)smem);
    k_pair32_fused<L, NP, MINB><<<grid, TPB32, smem, st>>>(a, oa, fa, b.tb_done, b.M);
    if (pair_end) cudaEventRecord(pair_end, st);
  } else {
    // One pair per lane, single layer: CTAs of 128 threads. A CTA's warps meet
    // few or many segments inside rho_c delta, and the SM waits for the
    // slowest; smaller CTAs wait less (pair kernel with 256 threads: 1,944 nodes
    // 13% longer, 24,576 nodes and 96,774 sources x 5,766 targets 3%; 64 threads:
    // longer from 24,576 nodes on). The stresslet's larger records leave room for
    // too few of them: 24,576 nodes 3% longer with 128.
    constexpr int TPB = NP == 1 && L::V == V_SL ? 128 : TPB32;
    constexpr size_t smem1 = pair_smem_bytes<L, NP, TPB>();
    const auto k = k_pair32<L, NP, TPB, MINB * (TPB32 / TPB)>;
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem1);
    k<<<grid * (TPB32 / TPB), TPB, smem1, st>>>(a);
    if (pair_end) cudaEventRecord(pair_end, st);
    constexpr int G = 64 * NP;
    const size_t fsmem = (size_t)near_warp_words(G) * sizeof(unsigned) + FIN_THREADS * 3 * sizeof(double);
    k_finish32<L, G><<<(unsigned)(b.M_pad / G * FIN_PARTS), FIN_THREADS, fsmem, st>>>(oa, fa, b.M);
  }
}

void launch_pair32(int layer, const EvalBufs& b, double rho_T, double rho_c, double scale,
                   cudaStream_t st, cudaEvent_t pair_end) {
  const float ratio = near_ratio(rho_T, rho_c);
  if (layer == LAYER_SL) {
    if (b.pair_np == 2)
      launch_pair32_t<SLayer, 2>(b, ratio, scale, st, pair_end);
    else
      launch_pair32_t<SLayer, 1>(b, ratio, scale, st, pair_end);
  } else {
    if (b.pair_np == 2)
      launch_pair32_t<DLayer, 2>(b, ratio, scale, st, pair_end);
    else
      launch_pair32_t<DLayer, 1>(b, ratio, scale, st, pair_end);
  }
}

}  // namespace sk
