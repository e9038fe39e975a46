// sk_pair64.cu -- FP64 pair sums (single and double layer).
//
// Same work decomposition as the FP32 kernels (sorted targets, chunks of
// source tiles staged by bulk async copies, per-segment near/far test), all
// arithmetic in FP64 but the tails of the table's polynomials (terms below 2^-30):
//   rho >= 7   plain Stokeslet / stresslet (s_i = 1 to double precision)
//   rho < 7    s_i / rho^k from a table of local polynomials in rho^2
//              (sk_factors64.h), incl. r = 0
// Two targets per lane; plain FP64 accumulation per chunk; the finish
// kernel adds the chunks of a target in fixed order.
#include <cfloat>

#include "sk_factors64.h"
#include "sk_internal.h"

namespace sk {
namespace {

constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes,
                                          uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity) {
  const long long t0 = clock64();
  while (true) {
    uint32_t ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, "
        "p; }"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
    if (clock64() - t0 > WAIT_CYCLES) return false;
  }
}

template <int LAYER>
__device__ __forceinline__ void far64(const double4_32a& G, const double4_32a& Nn, double dx,
                                      double dy, double dz, double r2, double* u) {
  const double ri = rsqrt_fp64(r2);
  const double ri2 = ri * ri;
  if (LAYER == LAYER_SL) {
    const double gd = fma(G.z, dz, fma(G.y, dy, G.x * dx));
    const double a = gd * ri2;
    u[0] = fma(fma(dx, a, G.x), ri, u[0]);
    u[1] = fma(fma(dy, a, G.y), ri, u[1]);
    u[2] = fma(fma(dz, a, G.z), ri, u[2]);
  } else {
    const double dq = fma(G.z, dz, fma(G.y, dy, G.x * dx));
    const double dn = fma(Nn.z, dz, fma(Nn.y, dy, Nn.x * dx));
    const double c = dq * dn * (ri2 * ri2 * ri);
    u[0] = fma(c, dx, u[0]);
    u[1] = fma(c, dy, u[1]);
    u[2] = fma(c, dz, u[2]);
  }
}

// high words of y = 1 + rho^2 at the end of the smoothed range (rho = RHO_C64)
// and at the end of the table
static_assert(RHO_C64 == 7, "Y_NEAR_HI is the high word of 1 + 49");
constexpr unsigned Y_NEAR_HI = 0x40490000u;
constexpr unsigned Y_TABLE_HI = 0x3ff00000u + (F64_N << (20 - F64_SUB_BITS));

// Factor f of a table (see f64_table_bytes) in interval idx at t = y - middle.
template <int NF, int TAIL>
__device__ __forceinline__ double factor(const double* tab, int f, int idx, double t, float tf) {
  const double* c = tab + f * F64_HEAD * F64_N + idx;
  const float* d = reinterpret_cast<const float*>(tab + NF * F64_HEAD * F64_N) + f * TAIL * F64_N + idx;
  float w = d[(TAIL - 1) * F64_N];
#pragma unroll
  for (int k = TAIL - 2; k >= 0; --k) w = fmaf(w, tf, d[k * F64_N]);
  return fma(fma(fma(c[3 * F64_N] + widen(w * tf), t, c[2 * F64_N]), t, c[F64_N]), t, c[0]);
}

// One pair inside the table's range; v accumulates the sum without its last
// factor 1/delta (invd2 = 1/delta^2).
template <int LAYER>
__device__ __forceinline__ void near64(const double* tab, const double4_32a& G,
                                       const double4_32a& Nn, double dx, double dy, double dz,
                                       double y, double invd2, double* v) {
  const int hi = __double2hiint(y);
  const int idx = (hi - 0x3ff00000) >> (20 - F64_SUB_BITS);
  constexpr int LOW = (1 << (20 - F64_SUB_BITS)) - 1;
  const double t = y - __hiloint2double((hi & ~LOW) | ((LOW + 1) >> 1), 0);
  const float tf = (float)t;
  const double gd = fma(G.z, dz, fma(G.y, dy, G.x * dx)) * invd2;
  if (LAYER == LAYER_SL) {
    const double k1 = factor<2, F64_TAIL_SL>(tab, 0, idx, t, tf);
    const double b = gd * factor<2, F64_TAIL_SL>(tab, 1, idx, t, tf);
    v[0] = fma(dx, b, fma(G.x, k1, v[0]));
    v[1] = fma(dy, b, fma(G.y, k1, v[1]));
    v[2] = fma(dz, b, fma(G.z, k1, v[2]));
  } else {
    const double dn = fma(Nn.z, dz, fma(Nn.y, dy, Nn.x * dx)) * invd2;
    const double c = gd * dn * factor<1, F64_TAIL_DL>(tab, 0, idx, t, tf);
    v[0] = fma(c, dx, v[0]);
    v[1] = fma(c, dy, v[1]);
    v[2] = fma(c, dz, v[2]);
  }
}

// Shared memory: the layer's factor table, then two source buffers.
template <int LAYER>
constexpr size_t pair64_smem_bytes() {
  return f64_table_bytes(LAYER == LAYER_DL) +
         2 * TILE64 * (LAYER == LAYER_DL ? 3 : 2) * sizeof(double4_32a);
}

// Work item: a block of 2 blockDim.x sorted targets against chunk ch of the
// sources. The chunks split the active sources evenly in units of SRC_UNIT
// (not whole tiles: with few tiles per chunk, whole tiles would leave some
// chunks twice as long as others); a CTA stages its chunk in pieces of at most
// TILE64 sources.
constexpr int SRC_UNIT = 8;

template <int LAYER>
__global__ void __launch_bounds__(TPB64, 2)
    k_pair64(const double4_32a* __restrict__ src64, const double4_32a* __restrict__ nrm64,
             const char* __restrict__ table, const float4* __restrict__ segbox,
             const int* __restrict__ meta, const double4_32a* __restrict__ tgt64, int64_t M_pad,
             int n_chunks, double* __restrict__ part, unsigned long long* __restrict__ flags) {
  constexpr int REC = 2;  // double4_32a records per source in src64
  constexpr uint32_t TAB_BYTES = (uint32_t)f64_table_bytes(LAYER == LAYER_DL);
  constexpr uint32_t BUF_D4 = TILE64 * (REC + (LAYER == LAYER_DL ? 1 : 0));
  extern __shared__ __align__(128) char sm_raw[];
  __shared__ __align__(8) uint64_t mbar[3];  // source buffers 0, 1; the table
  const double* tab = reinterpret_cast<const double*>(sm_raw);
  double4_32a* const sm64 = reinterpret_cast<double4_32a*>(sm_raw + TAB_BYTES);

  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int tb = blockIdx.x / n_chunks, ch = blockIdx.x % n_chunks;
  const int units = (meta[META_NS] + SRC_UNIT - 1) / SRC_UNIT;
  const int s0 = (int)((long long)ch * units / n_chunks) * SRC_UNIT;
  const int s1 = (int)((long long)(ch + 1) * units / n_chunks) * SRC_UNIT;
  const int n_it = (s1 - s0 + TILE64 - 1) / TILE64;

  if (tid == 0) {
    for (int b = 0; b < 3; ++b) mbar_init(&mbar[b]);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  int issued[2] = {0, 0}, consumed[2] = {0, 0};
  auto issue = [&](int b, int it) {
    double4_32a* dst = sm64 + (size_t)b * BUF_D4;
    const int j0 = s0 + it * TILE64, n = min(TILE64, s1 - j0);
    const uint32_t bytes = (uint32_t)n * sizeof(double4_32a);
    expect_tx(&mbar[b], LAYER == LAYER_DL ? 3 * bytes : 2 * bytes);
    bulk_copy(dst, src64 + (size_t)j0 * REC, 2 * bytes, &mbar[b]);
    if (LAYER == LAYER_DL) bulk_copy(dst + TILE64 * REC, nrm64 + j0, bytes, &mbar[b]);
    issued[b]++;
  };
  if (tid == 0 && n_it > 0) {
    expect_tx(&mbar[2], TAB_BYTES);
    bulk_copy(sm_raw, table, TAB_BYTES, &mbar[2]);
    for (int b = 0; b < 2; ++b)
      if (b < n_it) issue(b, b);
  }

  const int64_t wbase = (int64_t)tb * (blockDim.x * TPL64) + wid * TGT_WARP64;
  double tx[2], ty[2], tz[2], invd[2], invd2[2];
  float blo[3] = {FLT_MAX, FLT_MAX, FLT_MAX}, bhi[3] = {-FLT_MAX, -FLT_MAX, -FLT_MAX};
  float rc2max = -1.f, amax = 0.f;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const double4_32a x = tgt64[wbase + 32 * h + lane];
    tx[h] = x.x;
    ty[h] = x.y;
    tz[h] = x.z;
    const bool real = x.w > 0.0;
    invd[h] = real ? 1.0 / x.w : 1.0;
    invd2[h] = fmin(invd[h] * invd[h], DBL_MAX);  // finite, so that r = 0 gives y = 1
    if (real) {
      const float fx = (float)x.x, fy = (float)x.y, fz = (float)x.z;
      blo[0] = fminf(blo[0], fx); bhi[0] = fmaxf(bhi[0], fx);
      blo[1] = fminf(blo[1], fy); bhi[1] = fmaxf(bhi[1], fy);
      blo[2] = fminf(blo[2], fz); bhi[2] = fmaxf(bhi[2], fz);
      rc2max = fmaxf(rc2max, (float)((RHO_C64 * x.w) * (RHO_C64 * x.w)));
      amax = fmaxf(amax, fmaxf(fabsf(fx), fmaxf(fabsf(fy), fabsf(fz))));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      blo[c] = fminf(blo[c], __shfl_xor_sync(FULL, blo[c], o));
      bhi[c] = fmaxf(bhi[c], __shfl_xor_sync(FULL, bhi[c], o));
    }
    rc2max = fmaxf(rc2max, __shfl_xor_sync(FULL, rc2max, o));
    amax = fmaxf(amax, __shfl_xor_sync(FULL, amax, o));
  }
  const bool warp_live = rc2max >= 0.f;
  const float pad = 4e-7f * amax;  // covers FP64 -> FP32 rounding of both boxes
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    blo[c] -= pad;
    bhi[c] += pad;
  }
  const float rc2test = rc2max * 1.0001f;
  // Warps with a target whose 1/delta^2 overflows (delta below 7.5e-155) decide pair by
  // pair: there y does not tell r > 0 from far (a smoothed pair's 1/delta^3 would
  // overflow, so only r = 0 takes the table).
  const bool pair_by_pair = __any_sync(FULL, invd2[0] == DBL_MAX || invd2[1] == DBL_MAX);
  const unsigned table_hi = pair_by_pair ? 0u : Y_TABLE_HI;

  double u[2][3] = {{0, 0, 0}, {0, 0, 0}};  // far pairs
  double v[2][3] = {{0, 0, 0}, {0, 0, 0}};  // near pairs, times delta

  bool timed_out = false;
  if (n_it > 0 && __syncthreads_or(!mbar_wait_bounded(&mbar[2], 0))) timed_out = true;
  for (int it = 0; it < n_it && !timed_out; ++it) {
    const int buf = it & 1;
    const bool ok = mbar_wait_bounded(&mbar[buf], (uint32_t)(consumed[buf] & 1));
    consumed[buf]++;
    if (__syncthreads_or(!ok)) {
      timed_out = true;
      break;
    }
    if (warp_live) {
      const int j0 = s0 + it * TILE64, j1 = min(j0 + TILE64, s1);
      const double4_32a* S = sm64 + (size_t)buf * BUF_D4;
      const double4_32a* SN = S + TILE64 * REC;
      bool nb = false;
      const int seg0 = j0 / SEG, n_seg = (j1 - 1) / SEG - seg0 + 1;
      if (lane < n_seg) {
        const float4 lo = segbox[2 * ((size_t)seg0 + lane)];
        const float4 hi = segbox[2 * ((size_t)seg0 + lane) + 1];
        const float dx = fmaxf(0.f, fmaxf(lo.x - bhi[0], blo[0] - hi.x));
        const float dy = fmaxf(0.f, fmaxf(lo.y - bhi[1], blo[1] - hi.y));
        const float dz = fmaxf(0.f, fmaxf(lo.z - bhi[2], blo[2] - hi.z));
        nb = dx * dx + dy * dy + dz * dz < rc2test;
      }
      const unsigned nm = __ballot_sync(FULL, nb);
#pragma unroll 1
      for (int s = 0; s < n_seg; ++s) {
        const int ja = max(0, (seg0 + s) * SEG - j0), jb = min(j1, (seg0 + s + 1) * SEG) - j0;
        if (!((nm >> s) & 1u)) {
#pragma unroll 2
          for (int j = ja; j < jb; ++j) {
            const double4_32a P = S[REC * j], G = S[REC * j + 1];
            const double4_32a Nn = LAYER == LAYER_DL ? SN[j] : make_double4_32a(0, 0, 0, 0);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const double dx = tx[h] - P.x, dy = ty[h] - P.y, dz = tz[h] - P.z;
              far64<LAYER>(G, Nn, dx, dy, dz, fma(dz, dz, fma(dy, dy, dx * dx)), u[h]);
            }
          }
        } else {
#pragma unroll 1
          for (int j = ja; j < jb; ++j) {
            const double4_32a P = S[REC * j], G = S[REC * j + 1];
            const double4_32a Nn = LAYER == LAYER_DL ? SN[j] : make_double4_32a(0, 0, 0, 0);
            double dx[2], dy[2], dz[2], r2[2], y[2];
            unsigned hi[2];  // unsigned: a NaN of either sign lies beyond the table
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              dx[h] = tx[h] - P.x;
              dy[h] = ty[h] - P.y;
              dz[h] = tz[h] - P.z;
              r2[h] = fma(dz[h], dz[h], fma(dy[h], dy[h], dx[h] * dx[h]));
              y[h] = fma(r2[h], invd2[h], 1.0);
              hi[h] = (unsigned)__double2hiint(y[h]);
            }
            // If a lane has a pair inside the smoothed range, every lane inside
            // the table's range (rho < 16) takes the table, so that the warp
            // runs one of the two forms; beyond the smoothed range both give
            // the plain kernel.
            if (__any_sync(FULL, hi[0] < Y_NEAR_HI || hi[1] < Y_NEAR_HI)) {
              if (__all_sync(FULL, hi[0] < table_hi && hi[1] < table_hi)) {
#pragma unroll
                for (int h = 0; h < 2; ++h)
                  near64<LAYER>(tab, G, Nn, dx[h], dy[h], dz[h], y[h], invd2[h], v[h]);
              } else {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                  bool in_table = hi[h] < Y_TABLE_HI;
                  if (pair_by_pair && invd2[h] == DBL_MAX) in_table = r2[h] == 0.0;
                  if (in_table)
                    near64<LAYER>(tab, G, Nn, dx[h], dy[h], dz[h], y[h], invd2[h], v[h]);
                  else
                    far64<LAYER>(G, Nn, dx[h], dy[h], dz[h], r2[h], u[h]);
                }
              }
            } else {
#pragma unroll
              for (int h = 0; h < 2; ++h)
                far64<LAYER>(G, Nn, dx[h], dy[h], dz[h], r2[h], u[h]);
            }
          }
        }
      }
    }
    __syncthreads();
    if (tid == 0 && it + 2 < n_it) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      issue(buf, it + 2);
    }
  }
  if (timed_out) {
    if (tid == 0) {
      atomicExch(flags + FLAG_TIMEOUT, 1ull);
      mbar_wait_bounded(&mbar[2], 0);
      for (int b = 0; b < 2; ++b)
        while (consumed[b] < issued[b]) {
          if (!mbar_wait_bounded(&mbar[b], (uint32_t)(consumed[b] & 1))) break;
          consumed[b]++;
        }
    }
    return;
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    double* o = part + ((size_t)ch * M_pad + wbase + 32 * h + lane) * 3;
#pragma unroll
    for (int c = 0; c < 3; ++c) o[c] = fma(v[h][c], invd[h], u[h][c]);
  }
}

__global__ void k_finish64(const int* __restrict__ perm, int64_t M, int64_t M_pad, int n_chunks,
                           const double* __restrict__ part, double* __restrict__ u_out) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= M) return;
  double u0 = 0, u1 = 0, u2 = 0;
  for (int c = 0; c < n_chunks; ++c) {
    const double* p = part + ((size_t)c * M_pad + t) * 3;
    u0 += p[0];
    u1 += p[1];
    u2 += p[2];
  }
  const int64_t j = perm[t];
  u_out[3 * j] = u0;
  u_out[3 * j + 1] = u1;
  u_out[3 * j + 2] = u2;
}

}  // namespace

void launch_pair64(int layer, const EvalBufs& b, double /*scale*/, cudaStream_t st) {
  // M_pad is a multiple of TGT_CTA64, hence of the smaller CTA's targets too
  const int tpb = b.threads64;
  const unsigned grid = (unsigned)((b.M_pad / ((int64_t)tpb * TPL64)) * b.n_chunks);
  if (layer == LAYER_SL) {
    constexpr size_t smem = pair64_smem_bytes<LAYER_SL>();
    cudaFuncSetAttribute(k_pair64<LAYER_SL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_pair64<LAYER_SL><<<grid, tpb, smem, st>>>(b.src64, b.nrm64, b.factors64, b.segbox, b.meta,
                                                b.tgt64, b.M_pad, b.n_chunks, b.part, b.flags);
  } else {
    constexpr size_t smem = pair64_smem_bytes<LAYER_DL>();
    cudaFuncSetAttribute(k_pair64<LAYER_DL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_pair64<LAYER_DL><<<grid, tpb, smem, st>>>(
        b.src64, b.nrm64, b.factors64 + f64_table_bytes(false), b.segbox, b.meta, b.tgt64, b.M_pad,
        b.n_chunks, b.part, b.flags);
  }
}

void launch_finish64(const EvalBufs& b, cudaStream_t st) {
  k_finish64<<<(unsigned)((b.M + 127) / 128), 128, 0, st>>>(b.tgt_perm, b.M, b.M_pad, b.n_chunks,
                                                            b.part, b.u);
}

}  // namespace sk
