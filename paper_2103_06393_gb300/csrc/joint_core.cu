// The column sums of the joint form (joint.cuh) on the tensor cores:
//   forward  T[c, s]   = sum_j K[j][c] X[j, s]            rows c, summed over the stored columns j
//   adjoint  Psi[j, s] = sum_c conj(K[j][c]) F[c, s]      rows j, summed over all cores' entries c
// One complex GEMM each with P right-hand sides a pass, bound by the read of K (8 bytes an entry) as
// long as the arithmetic keeps up: in FP32 on the CUDA cores it did not (96^3 head coil, 2.7 GB of K,
// 16 right-hand sides: 1.2 / 2.1 ms against 0.4 ms for the bytes).
//
// K stays in FP32 in memory.  A CTA takes 128 rows and walks chunks of 32 summed entries: 8 worker
// warps load the chunk's K (one chunk ahead), scale it by powers of two, split it into fp16 hi + lo
// and write 128-byte swizzled rows (32 (Re, Im) pairs) to one of two buffers, and split the chunk's
// 32 x P right-hand-side entries beside it, scaled per right-hand side; the ninth warp issues the
// hi hi, hi lo and lo hi MMAs (M = 128, N = 2 P, K = 64); the accumulator is added into FP32
// registers with the chunk's scales while the next chunk is converted, so that a tensor-core sum has
// 64 terms.
//
// Scales: K per column j (kscale[j] = 2^(15 - e_j), |K[j]| < 2^e_j, from the build; fp16 hi + lo leave
// an error of max(2^-23 |K|, 2^-40 2^e_j)); the forward's X by 2^(e_j - e), e the component's largest
// e_j; the right-hand sides' entries per chunk.  Each chunk enters the FP32 sums with all scales but
// 2^(e_j - e) taken out, so that these overflow where the product would and not before; an X entry takes
// its own power of two first, so that a small one against a small column keeps its bits.  Scales of K's rows
// taken anew in every chunk of the adjoint cost a fifth of its issue slots (0.61 ms at 96^3, 16 right-hand
// sides).
#include <algorithm>

#include "joint_tc.cuh"

namespace zbc {
namespace {

constexpr int kRows = 128, kSum = 32;
constexpr int kFold = 32;  // chunks of the adjoint per FP32 chain: one over a slice's 300 chunks (96^3) made
                           // more than half of its error
constexpr uint32_t kRowTerm = kRows * 128u;  // one term of K's chunk

__host__ __device__ inline int slices_of(int Cs, int split) { return ((Cs + kSum - 1) / kSum + split - 1) / split; }

template <int P>
constexpr size_t core_smem() {
  return 4 * (size_t)kRowTerm + 4 * (size_t)(2 * P) * 128;
}

template <bool FWD, int P>
__global__ void __launch_bounds__(288, 2)
    joint_core_kernel(const __grid_constant__ JointGeo G, const float2* __restrict__ K, const float* __restrict__ kscale,
                      const float2* __restrict__ R, int64_t ldr, int p, int split, float2* __restrict__ out,
                      int* __restrict__ err, uint32_t polls) {
  constexpr int N = 2 * P, I = P / 8;
  constexpr uint32_t kBTerm = N * 128u, ncols = FWD ? 2 * N : 4 * N;  // two accumulators, the adjoint's sums
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t done[2], ready[2];
  __shared__ uint32_t tmem_base;
  __shared__ float bscale[4][P];            // scales that a chunk's sums still carry, per right-hand side
  unsigned char* sa = smem;                 // [2 buffers][2 terms][128 rows][128 B]
  unsigned char* sb = sa + 4 * kRowTerm;    // [2 buffers][2 terms][N rows][128 B]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0)
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&done[i], 1);
      tc::mbar_init(&ready[i], 8);
    }
  if (warp == 0) tc::tmem_alloc(&tmem_base, ncols);
  __syncthreads();
  const uint32_t tmem = tmem_base;
  Waits waits{err, polls};
  // forward: items are the 128-row tiles of all components, walked by blockIdx.x; adjoint: one item,
  // slice blockIdx.x of `split` chunks of one component (ksplit, first chunk ch0), for rows 128 blockIdx.y
  const int s0 = blockIdx.z * P, Mp = (G.M + kSum - 1) / kSum * kSum;
  int tiles = 0, ksplit = 0, ch0 = blockIdx.x;
  for (int k = 0; k < G.q; ++k) tiles += (G.Cs[k] + kRows - 1) / kRows;
  if (!FWD) {
    for (int n; ch0 >= (n = slices_of(G.Cs[ksplit], split)); ++ksplit) ch0 -= n;
    ch0 *= split;
  }
  const int items = FWD ? (tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 1;
  const int per = FWD ? Mp / kSum : min(split, (G.Cs[ksplit] + kSum - 1) / kSum - ch0);
  if (warp == 8) {
    if (lane == 0) {
      constexpr uint32_t id = tc::instr_desc(128, N, 0);
      int c = 0;
      for (; c < items * per; ++c) {
        const int d = c & 1;
        waits.one(&ready[d], (c >> 1) & 1);
        if (!waits.ok) break;
        tc::fence_after();
        const uint32_t a0 = tc::smem_u32(sa) + d * 2 * kRowTerm, b0 = tc::smem_u32(sb) + d * 2 * kBTerm;
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
          const uint64_t ah = tc::smem_desc_sw128(a0 + ks * 32), al = tc::smem_desc_sw128(a0 + kRowTerm + ks * 32);
          const uint64_t bh = tc::smem_desc_sw128(b0 + ks * 32), bl = tc::smem_desc_sw128(b0 + kBTerm + ks * 32);
          tc::mma<0>(tmem + d * N, al, bh, id, ks > 0);
          tc::mma<0>(tmem + d * N, ah, bl, id, 1);
        }
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
          tc::mma<0>(tmem + d * N, tc::smem_desc_sw128(a0 + ks * 32), tc::smem_desc_sw128(b0 + ks * 32), id, 1);
        tc::commit(&done[d]);
      }
      drain2(done, c);
    }
    __syncwarp();
  } else {
    const int q4 = warp & 3, half = warp >> 2;           // accumulator rows and columns
    const int row0 = warp * 4 + lane / 8, c8 = lane % 8;  // adjoint loader: rows row0 + 32 u, entries entry_of(c8, w)
    bool bad = false;
    float2 x[16], b[I];
    // position of the chunk that fetch() reads next: component, first row of the tile (forward) or first
    // core entry (adjoint)
    int fk = 0, fpos = 0;
    auto locate_tile = [&](int t) {
      fk = 0;
      for (int n; t >= (n = (G.Cs[fk] + kRows - 1) / kRows); ++fk) t -= n;
      fpos = t * kRows;
    };
    auto fetch = [&](int ch) {  // chunk ch of the current item
      if (FWD) {
        const int c = fpos + 32 * q4 + lane, j0 = ch * kSum + 16 * half;
        const float2* g = K + G.koff[fk] + (int64_t)j0 * G.Cs[fk] + c;
        const bool live = c < G.Cs[fk];
#pragma unroll
        for (int u = 0; u < 16; ++u)
          x[u] = live && j0 + u < G.M ? __ldcs(g + (int64_t)u * G.Cs[fk]) : make_float2(0.f, 0.f);
        const int j = ch * kSum + lane;
#pragma unroll
        for (int i = 0; i < I; ++i) {
          const int s = s0 + warp + 8 * i;
          b[i] = j < G.M && s < p ? __ldg(R + j + ldr * s) : make_float2(0.f, 0.f);
        }
      } else {
        const int c = fpos + 2 * c8;  // rows of K are padded to 4 entries: pairs never cross their end
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int j = blockIdx.y * kRows + row0 + 32 * u;
          const float2* g = K + G.koff[fk] + (int64_t)j * G.Cs[fk] + c;
#pragma unroll
          for (int w = 0; w < 2; ++w) {
            const float4 v = j < G.M && c + 16 * w < G.Cs[fk] ? __ldcs((const float4*)(g + 16 * w))
                                                              : make_float4(0.f, 0.f, 0.f, 0.f);
            x[4 * u + 2 * w] = make_float2(v.x, v.y);
            x[4 * u + 2 * w + 1] = make_float2(v.z, v.w);
          }
        }
#pragma unroll
        for (int i = 0; i < I; ++i) {
          const int s = s0 + warp + 8 * i;
          b[i] = fpos + lane < G.Cs[fk] && s < p ? __ldg(R + G.toff[fk] + fpos + lane + ldr * s) : make_float2(0.f, 0.f);
        }
      }
    };
    float kr[4];  // adjoint: scales of the loader's rows
    if (FWD) {
      locate_tile(blockIdx.x);
    } else {
      fk = ksplit;
      fpos = ch0 * kSum;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int j = blockIdx.y * kRows + row0 + 32 * u;
        kr[u] = j < G.M ? __ldg(kscale + (int64_t)fk * 2 * Mp + j) : 1.f;
      }
    }
    fetch(0);
    int c0 = 0;  // the CTA's number of this item's first chunk
    for (int item = 0; item < items; ++item, c0 += per) {
      const int k = fk, row = fpos;
      const float* ks = kscale + (int64_t)k * 2 * Mp;
      // 2^(e - 15) of the component, half of it, and what the accumulators' rounding takes off
      const float kf = __ldg(kscale + (int64_t)G.q * 2 * Mp + k) * (0.5f * lo_first_gain(4));
      float acc[P];
#pragma unroll
      for (int i = 0; i < P; ++i) acc[i] = 0.f;
      auto fold = [&](int c) {
        const int d = c & 1;
        waits.warp(&done[d], (c >> 1) & 1);
        tc::fence_after();
        const uint32_t t0 = tmem + (uint32_t)(d * N + half * P) + ((uint32_t)(32 * q4) << 16);
#pragma unroll
        for (int i = 0; i < I; ++i) {
          uint32_t r[8];
          tmem_ld8(t0 + 8 * i, r);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float cf = bscale[c & 3][half * (P / 2) + 4 * i + u];
#pragma unroll
            for (int e = 0; e < 2; ++e)
              acc[8 * i + 2 * u + e] = fmaf(__uint_as_float(r[2 * u + e]), cf, acc[8 * i + 2 * u + e]);
          }
        }
        tc::fence_before();
      };
      // adjoint: the sums so far wait in tensor memory, after the two accumulators (each thread its own)
      auto put_by = [&](bool first) {
        const uint32_t t0 = tmem + (uint32_t)(2 * N + half * P) + ((uint32_t)(32 * q4) << 16);
#pragma unroll
        for (int i = 0; i < I; ++i) {
          uint32_t r[8];
          if (!first) tmem_ld8(t0 + 8 * i, r);
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            r[u] = __float_as_uint(first ? acc[8 * i + u] : acc[8 * i + u] + __uint_as_float(r[u]));
            acc[8 * i + u] = 0.f;
          }
          tmem_st8(t0 + 8 * i, r);
        }
        tc::tmem_wait_st();
      };
      auto chunk = [&](int ch) {
        const int c = c0 + ch, d = c & 1;
        if (ch >= 2) fold(c - 2);  // also: the MMAs have read this buffer
        const float xs = FWD ? __ldg(ks + Mp + ch * kSum + lane) : 1.f;  // 2^(e_j - e), used after K's split
        unsigned char* ad = sa + (size_t)d * 2 * kRowTerm;
        if (FWD) {
          const int r = 32 * q4 + lane;
          const float4* kp = (const float4*)(ks + ch * kSum + 16 * half);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float4 sc = __ldg(kp + u);
            uint32_t h[4], l[4];
            split2(x[4 * u].x * sc.x, x[4 * u].y * sc.x, h[0], l[0]);
            split2(x[4 * u + 1].x * sc.y, x[4 * u + 1].y * sc.y, h[1], l[1]);
            split2(x[4 * u + 2].x * sc.z, x[4 * u + 2].y * sc.z, h[2], l[2]);
            split2(x[4 * u + 3].x * sc.w, x[4 * u + 3].y * sc.w, h[3], l[3]);
            unsigned char* o = ad + tc::sw128_off(r, 4 * half + u);
            *(uint4*)o = make_uint4(h[0], h[1], h[2], h[3]);
            *(uint4*)(o + kRowTerm) = make_uint4(l[0], l[1], l[2], l[3]);
          }
        } else {
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            uint32_t h[4], l[4];
#pragma unroll
            for (int w = 0; w < 4; ++w) split2(x[4 * u + w].x * kr[u], x[4 * u + w].y * kr[u], h[w], l[w]);
            unsigned char* o = ad + tc::sw128_off(row0 + 32 * u, c8);
            *(uint4*)o = make_uint4(h[0], h[1], h[2], h[3]);
            *(uint4*)(o + kRowTerm) = make_uint4(l[0], l[1], l[2], l[3]);
          }
        }
        // the right-hand sides' rows (two a right-hand side): pair `lane` of the chunk in the rows' order
        const uint32_t kc = FWD ? lane / 4 : lane % 16 / 2, word = FWD ? lane % 4 : lane % 2 + lane / 16 * 2;
#pragma unroll
        for (int i = 0; i < I; ++i) {
          const int n = 2 * (warp + 8 * i);
          // xs |b| < 2^e, so that 2^(kDataShift - e) b is below 2^kDataShift / xs: finite
          const float m = absmax_nan(0.f, b[i].x, b[i].y);
          if (FWD) bad = bad || !(m < INFINITY);
          const int e = exp_of(__uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(FWD ? m * xs : m))), -117);
          if (lane == 0) bscale[c & 3][warp + 8 * i] = pow2f(e - kDataShift + 1) * kf;
          const float sc = pow2f(kDataShift - e);
          uint32_t h, l;
          split2(FWD ? b[i].x * sc * xs : b[i].x * sc, FWD ? b[i].y * sc * xs : b[i].y * sc, h, l);
          const uint32_t hs = __byte_perm(h, 0, 0x1032), ls = __byte_perm(l, 0, 0x1032);
          unsigned char* o0 = sb + (size_t)d * 2 * kBTerm + tc::sw128_off(n, kc) + 4 * word;
          unsigned char* o1 = sb + (size_t)d * 2 * kBTerm + tc::sw128_off(n + 1, kc) + 4 * word;
          // forward: (Re, -Im), (Im, Re) against (Re, Im) K; adjoint: (Re, Im), (Im, -Re)
          *(uint32_t*)o0 = FWD ? h ^ 0x80000000u : h;
          *(uint32_t*)(o0 + kBTerm) = FWD ? l ^ 0x80000000u : l;
          *(uint32_t*)o1 = FWD ? hs : hs ^ 0x80000000u;
          *(uint32_t*)(o1 + kBTerm) = FWD ? ls : ls ^ 0x80000000u;
        }
        if (ch + 1 < per) {
          if (!FWD) fpos += kSum;
          fetch(ch + 1);
        } else if (item + 1 < items) {
          locate_tile((int)blockIdx.x + (item + 1) * (int)gridDim.x);
          fetch(0);
        }
        warp_publish(&ready[d]);
      };
      int ch = 0;
      if (!FWD)
        for (; per - ch > kFold; put_by(ch == kFold))
          for (int end = ch + kFold; ch < end; ++ch) chunk(ch);
      for (; ch < per; ++ch) chunk(ch);
      if (per > 1) fold(c0 + per - 2);
      fold(c0 + per - 1);
      const int r = 32 * q4 + lane;
      if (FWD) {
        if (row + r < G.Cs[k])
#pragma unroll
          for (int i = 0; i < P / 2; ++i) {
            const int s = s0 + half * (P / 2) + i;
            if (s < p) out[(int64_t)s * G.Ct + G.toff[k] + row + r] = make_float2(acc[2 * i], acc[2 * i + 1]);
          }
      } else {
        if (per > kFold) {
          const uint32_t t0 = tmem + (uint32_t)(2 * N + half * P) + ((uint32_t)(32 * q4) << 16);
#pragma unroll
          for (int i = 0; i < I; ++i) {
            uint32_t v[8];
            tmem_ld8(t0 + 8 * i, v);
#pragma unroll
            for (int u = 0; u < 8; ++u) acc[8 * i + u] += __uint_as_float(v[u]);
          }
        }
        const int j = blockIdx.y * kRows + r;
        const float kj = j < G.M ? __ldg(ks + Mp + j) : 0.f;  // 2^(e_j - e)
        if (j < G.M)
#pragma unroll
          for (int i = 0; i < P / 2; ++i) {
            const int s = s0 + half * (P / 2) + i;
            if (s < p) out[((int64_t)blockIdx.x * p + s) * G.M + j] = make_float2(acc[2 * i] * kj, acc[2 * i + 1] * kj);
          }
      }
    }
    if (bad) atomicOr(err, kErrNonFinite);
  }
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, ncols);
}

// e_j of a column's core: one CTA per (column, component); kscale[k][0][j] = e_j as a float for now
__global__ void __launch_bounds__(128) core_exp_kernel(const __grid_constant__ JointGeo G, const float2* __restrict__ K,
                                                       int Mp, float* __restrict__ kscale) {
  const int j = blockIdx.x, k = blockIdx.y;
  __shared__ float red[4];
  float m = 0.f;
  if (j < G.M)
    for (int c = threadIdx.x; c < G.Cs[k]; c += 128) {
      const float2 v = K[G.koff[k] + (int64_t)j * G.Cs[k] + c];
      m = absmax_nan(m, v.x, v.y);
    }
  for (int o = 16; o > 0; o >>= 1) m = max_nan(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 4; ++w) m = max_nan(m, red[w]);
    kscale[(int64_t)k * 2 * Mp + j] = m > 0.f ? (float)exp_of(m, -106) : -1000.f;  // no entries: takes the largest e
  }
}
// the scales from the exponents: kscale[k][0][j] = 2^(15 - e_j), kscale[k][1][j] = 2^(e_j - e), and
// 2^(e - 15) of component k after them
__global__ void __launch_bounds__(256) core_scale_kernel(const __grid_constant__ JointGeo G, int Mp, float* __restrict__ kscale) {
  const int k = blockIdx.x;
  __shared__ int emax;
  if (threadIdx.x == 0) emax = -1000;
  __syncthreads();
  float* row = kscale + (int64_t)k * 2 * Mp;
  for (int j = threadIdx.x; j < Mp; j += 256) atomicMax(&emax, (int)row[j]);
  __syncthreads();
  const int e = emax < -500 ? 0 : emax;
  for (int j = threadIdx.x; j < Mp; j += 256) {
    const int ej = row[j] < -500.f ? e : (int)row[j];
    row[j] = pow2f(15 - ej);
    row[Mp + j] = pow2f(max(-126, ej - e));
  }
  if (threadIdx.x == 0) kscale[(int64_t)G.q * 2 * Mp + k] = pow2f(e - 15);
}

int padded_m(const JointGeo& G) { return ceil_div(G.M, kSum) * kSum; }

template <int P>
int launch_fwd(const JointCache& jc, const float2* X, int64_t ldx, int p, float2* T, int* err, uint32_t polls,
               cudaStream_t st) {
  const JointGeo& G = jc.geo;
  ZBC_TRY((set_smem_limit<joint_core_kernel<true, P>>((int)core_smem<P>())));
  int tiles = 0;
  for (int k = 0; k < G.q; ++k) tiles += ceil_div(G.Cs[k], kRows);
  const int passes = ceil_div(p, P);
  joint_core_kernel<true, P><<<dim3(std::min(tiles, 2 * sm_count()), 1, passes), 288, core_smem<P>(), st>>>(
      G, jc.K, jc.kscale, X, ldx, p, 0, T, err, polls);
  return ZBC_OK;
}
template <int P>
int launch_adj(const JointCache& jc, const float2* F, int p, int split, int splits, float2* part, int* err, uint32_t polls,
               cudaStream_t st) {
  const JointGeo& G = jc.geo;
  ZBC_TRY((set_smem_limit<joint_core_kernel<false, P>>((int)core_smem<P>())));
  joint_core_kernel<false, P><<<dim3(splits, ceil_div(G.M, kRows), ceil_div(p, P)), 288, core_smem<P>(), st>>>(
      G, jc.K, jc.kscale, F, G.Ct, p, split, part, err, polls);
  return ZBC_OK;
}

int rhs_tile(int p) { return p <= 8 ? 8 : p <= 16 ? 16 : 32; }

}  // namespace

size_t joint_core_bytes(const JointGeo& G) { return sizeof(float) * ((size_t)G.q * 2 * padded_m(G) + G.q); }

int joint_core_build(const JointGeo& G, const float2* K, float* kscale, bool* fits, cudaStream_t st) {
  const int Mp = padded_m(G);
  core_exp_kernel<<<dim3(Mp, G.q), 128, 0, st>>>(G, K, Mp, kscale);
  core_scale_kernel<<<G.q, 256, 0, st>>>(G, Mp, kscale);
  count_launch(2);
  ZBC_TRY_CUDA(cudaGetLastError());
  // columns further apart than FP32's exponents reach have no common scale
  std::vector<float> rel((size_t)G.q * 2 * Mp);
  ZBC_TRY_CUDA(cudaMemcpyAsync(rel.data(), kscale, sizeof(float) * rel.size(), cudaMemcpyDeviceToHost, st));
  ZBC_TRY_CUDA(cudaStreamSynchronize(st));
  *fits = true;
  for (int k = 0; k < G.q; ++k)
    for (int j = 0; j < G.M; ++j) *fits = *fits && rel[((size_t)2 * k + 1) * Mp + j] > 1e-35f;
  return ZBC_OK;
}

int joint_core_fwd(const JointCache& jc, const float2* X, int64_t ldx, int p, float2* T, int* err, uint32_t polls,
                   cudaStream_t st) {
  switch (rhs_tile(p)) {
    case 8: ZBC_TRY(launch_fwd<8>(jc, X, ldx, p, T, err, polls, st)); break;
    case 16: ZBC_TRY(launch_fwd<16>(jc, X, ldx, p, T, err, polls, st)); break;
    default: ZBC_TRY(launch_fwd<32>(jc, X, ldx, p, T, err, polls, st)); break;
  }
  count_launch();
  ZBC_TRY_CUDA(cudaGetLastError());
  return ZBC_OK;
}

void joint_core_split(const JointGeo& G, int p, int* split, int* splits) {
  int chunks = 0;
  for (int k = 0; k < G.q; ++k) chunks += ceil_div(G.Cs[k], kSum);
  // one wave of two CTAs an SM, at least 4 chunks each
  const int want = std::max(1, 2 * sm_count() / (ceil_div(G.M, kRows) * ceil_div(p, rhs_tile(p))));
  *split = std::max(4, ceil_div(chunks, want));
  *splits = 0;
  for (int k = 0; k < G.q; ++k) *splits += slices_of(G.Cs[k], *split);
}

int joint_core_adj(const JointCache& jc, const float2* F, int p, float2* part, int* err, uint32_t polls, cudaStream_t st) {
  int split, splits;
  joint_core_split(jc.geo, p, &split, &splits);
  switch (rhs_tile(p)) {
    case 8: ZBC_TRY(launch_adj<8>(jc, F, p, split, splits, part, err, polls, st)); break;
    case 16: ZBC_TRY(launch_adj<16>(jc, F, p, split, splits, part, err, polls, st)); break;
    default: ZBC_TRY(launch_adj<32>(jc, F, p, split, splits, part, err, polls, st)); break;
  }
  count_launch();
  ZBC_TRY_CUDA(cudaGetLastError());
  return ZBC_OK;
}

}  // namespace zbc
