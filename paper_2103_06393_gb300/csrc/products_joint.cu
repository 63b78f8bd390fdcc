// The products through a joint basis of the columns' factors (joint.cuh).
//
// Forward:  T = sum_j K_j X[j, :]        joint_core_fwd_kernel, joint_core.cu   (R1 R2 R3 entries per component)
//           Q[i3] = T x3 B3              joint_mode3_fwd_kernel
//           Y[:, :, i3] = B1 Q[i3] B2^T  joint_planes.cu          (one write of Y)
// Adjoint:  Q[i3] = B1^H Phi[:, :, i3] conj(B2)   joint_planes.cu          (one read of Phi)
//           F = Q x3 B3^H                         joint_mode3_adj_kernel
//           Psi[j, :] = sum conj(K_j) F           joint_core_adj_kernel, joint_core.cu; joint_sum_kernel
// The column sums here are the FP32 ones of a few right-hand sides, which the read of K bounds;
// joint_core.cu has those of more on the tensor cores.
#include <algorithm>

#include "decomp.cuh"
#include "joint.cuh"

namespace zbc {
namespace {

constexpr int kJc = 64;  // columns of X per shared-memory chunk of the forward core sum
constexpr int kJf = 32;  // and per FP32 chain

__device__ __forceinline__ bool finite2(float2 v) { return isfinite(v.x) && isfinite(v.y); }

// T[js][s][toff + c] = sum over columns j of slice js of K[j][c] X[j, s]; two c per thread.
// Grid (c blocks of 256, slices, q * passes of P right-hand sides).
template <int P>
__global__ void __launch_bounds__(128) joint_core_fwd_kernel(const __grid_constant__ JointGeo G, const float2* __restrict__ K,
                                                             const float2* __restrict__ X, int64_t ldx, int p, int JS,
                                                             float2* __restrict__ T, int* __restrict__ err) {
  __shared__ __align__(16) float2 xs[kJc][P];
  const int k = blockIdx.z % G.q, s0 = blockIdx.z / G.q * P;
  const int c = 2 * (blockIdx.x * 128 + threadIdx.x);
  if (2 * blockIdx.x * 128 >= G.Cs[k]) return;
  const bool live = c < G.Cs[k];
  const int per = (G.M + JS - 1) / JS;
  const int j0 = blockIdx.y * per, j1 = min(G.M, j0 + per);
  const int64_t cs = G.Cs[k];
  const float2* Kp = K + G.koff[k] + (live ? c : 0);
  float2 sum[2][P];
#pragma unroll
  for (int s = 0; s < P; ++s) sum[0][s] = sum[1][s] = make_float2(0.f, 0.f);
  bool bad = false;
  for (int jb = j0; jb < j1; jb += kJc) {
    const int nj = min(kJc, j1 - jb);
    __syncthreads();
    for (int e = threadIdx.x; e < kJc * P; e += 128) {
      const int jj = e % kJc, s = e / kJc;
      float2 v = make_float2(0.f, 0.f);
      if (jj < nj && s0 + s < p) v = X[jb + jj + ldx * (s0 + s)];
      bad = bad || !finite2(v);
      xs[jj][s] = v;
    }
    __syncthreads();
    for (int jh = 0; jh < nj; jh += kJf) {
      float2 acc[2][P];  // chains of kJf terms
#pragma unroll
      for (int s = 0; s < P; ++s) acc[0][s] = acc[1][s] = make_float2(0.f, 0.f);
      const int je = min(nj, jh + kJf);
#pragma unroll 4
      for (int jj = jh; jj < je; ++jj) {
        const float4 kv = __ldcs((const float4*)(Kp + (jb + jj) * cs));
#pragma unroll
        for (int s = 0; s < P; ++s) {
          const float2 x = xs[jj][s];
          acc[0][s] = cfma(make_float2(kv.x, kv.y), x, acc[0][s]);
          acc[1][s] = cfma(make_float2(kv.z, kv.w), x, acc[1][s]);
        }
      }
#pragma unroll
      for (int c2 = 0; c2 < 2; ++c2)
#pragma unroll
        for (int s = 0; s < P; ++s) {
          sum[c2][s].x += acc[c2][s].x;
          sum[c2][s].y += acc[c2][s].y;
        }
    }
  }
  if (bad) atomicOr(err, kErrNonFinite);
  if (!live) return;
#pragma unroll
  for (int s = 0; s < P; ++s)
    if (s0 + s < p) {
      float2* o = T + ((int64_t)blockIdx.y * p + s0 + s) * G.Ct + G.toff[k] + c;
      *(float4*)o = make_float4(sum[0][s].x, sum[0][s].y, sum[1][s].x, sum[1][s].y);
    }
}

constexpr int kZ = 16;  // values of i3 (forward) or of the third core index (adjoint) per thread

// Q[s][qoff + i3 RR + xy] = sum_z B3[i3, z] sum_js T[js][s][toff + xy + RR z]
__global__ void __launch_bounds__(128) joint_mode3_fwd_kernel(const __grid_constant__ JointGeo G,
                                                              const float2* __restrict__ basis, const float2* __restrict__ T,
                                                              int p, int JS, float2* __restrict__ Q) {
  __shared__ float2 b3[kJointRmax][kZ];
  const int k = blockIdx.z % G.q, s = blockIdx.z / G.q, R3 = G.R[k][2];
  const int RR = G.R[k][0] * G.R[k][1];
  if ((int)blockIdx.x * 128 >= RR) return;
  const int z0 = blockIdx.y * kZ, xy = blockIdx.x * 128 + threadIdx.x;
  for (int e = threadIdx.x; e < R3 * kZ; e += 128) {
    const int zz = e % kZ, r = e / kZ;
    b3[r][zz] = z0 + zz < G.n3 ? basis[G.boff[k][2] + (int64_t)r * G.n3 + z0 + zz] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  if (xy >= RR) return;
  float2 acc[kZ];
#pragma unroll
  for (int z = 0; z < kZ; ++z) acc[z] = make_float2(0.f, 0.f);
  const float2* Ts = T + (int64_t)s * G.Ct + G.toff[k] + xy;
#pragma unroll 2
  for (int r = 0; r < R3; ++r) {
    float2 t = Ts[(int64_t)r * RR];
    for (int js = 1; js < JS; ++js) {
      const float2 u = Ts[(int64_t)js * p * G.Ct + (int64_t)r * RR];
      t.x += u.x;
      t.y += u.y;
    }
#pragma unroll
    for (int z = 0; z < kZ; ++z) acc[z] = cfma(t, b3[r][z], acc[z]);
  }
  float2* o = Q + (int64_t)s * G.Qt + G.qoff[k] + xy;
#pragma unroll
  for (int z = 0; z < kZ; ++z)
    if (z0 + z < G.n3) o[(int64_t)(z0 + z) * RR] = acc[z];
}

// F[s][toff + xy + RR z] = sum_i3 conj(B3[i3, z]) Q[s][qoff + i3 RR + xy]; entries up to Cs are zero
__global__ void __launch_bounds__(128, 8) joint_mode3_adj_kernel(const __grid_constant__ JointGeo G,
                                                              const float2* __restrict__ basis, const float2* __restrict__ Q,
                                                              float2* __restrict__ F) {
  constexpr int NZ = 8, NC = 32;
  __shared__ float2 b3[NC][NZ];
  const int k = blockIdx.z % G.q, s = blockIdx.z / G.q, R3 = G.R[k][2];
  const int RR = G.R[k][0] * G.R[k][1], z0 = blockIdx.y * NZ;
  if ((int)blockIdx.x * 128 >= RR || z0 >= R3) return;
  const int xy = blockIdx.x * 128 + threadIdx.x;
  const float2* Qs = Q + (int64_t)s * G.Qt + G.qoff[k] + (xy < RR ? xy : 0);
  float2 sum[NZ];
#pragma unroll
  for (int z = 0; z < NZ; ++z) sum[z] = make_float2(0.f, 0.f);
  for (int i0 = 0; i0 < G.n3; i0 += NC) {
    __syncthreads();
    for (int e = threadIdx.x; e < NC * NZ; e += 128) {
      const int i = e % NC, z = e / NC;
      b3[i][z] = z0 + z < R3 && i0 + i < G.n3 ? basis[G.boff[k][2] + (int64_t)(z0 + z) * G.n3 + i0 + i] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    float2 acc[NZ];  // the chunk's sums: a chain of NC terms
#pragma unroll
    for (int z = 0; z < NZ; ++z) acc[z] = make_float2(0.f, 0.f);
    const int ni = min(NC, G.n3 - i0);
#pragma unroll 8
    for (int i = 0; i < ni; ++i) {
      const float2 v = Qs[(int64_t)(i0 + i) * RR];
#pragma unroll
      for (int z = 0; z < NZ; ++z) acc[z] = cfma_conj(b3[i][z], v, acc[z]);
    }
#pragma unroll
    for (int z = 0; z < NZ; ++z) {
      sum[z].x += acc[z].x;
      sum[z].y += acc[z].y;
    }
  }
  float2* o = F + (int64_t)s * G.Ct + G.toff[k];
  if (xy < RR)
#pragma unroll
    for (int z = 0; z < NZ; ++z)
      if (z0 + z < R3) o[xy + (int64_t)RR * (z0 + z)] = sum[z];
  if (blockIdx.x == 0 && blockIdx.y == 0)
    for (int e = RR * R3 + threadIdx.x; e < G.Cs[k]; e += 128) o[e] = make_float2(0.f, 0.f);
}

constexpr int kCj = 64;  // columns per CTA of the adjoint core sum
constexpr int kCc = 32;  // core entries per chunk

// part[split][s][j] = sum over the split's core entries c of conj(K[j][c]) F[s][c].  128 threads:
// 16 groups of 4 columns, P right-hand sides, and KS interleaved slices of the chunk (P = 1 or 2).  Grid (column tiles, splits of all components' entries, passes of P).
template <int P>
__global__ void __launch_bounds__(128) joint_core_adj_kernel(const __grid_constant__ JointGeo G, const float2* __restrict__ K,
                                                             const float2* __restrict__ F, int p, int chunk,
                                                             float2* __restrict__ part) {
  constexpr int KS = 8 / P;
  __shared__ __align__(16) float2 ks[kCc][kCj + 2];
  __shared__ __align__(16) float2 fs[kCc][P];
  __shared__ float2 red[KS][kCj][P];
  int sp = blockIdx.y, k = 0;
  for (; k < G.q; ++k) {
    const int ns = (G.Cs[k] + chunk - 1) / chunk;
    if (sp < ns) break;
    sp -= ns;
  }
  const int c0 = sp * chunk, c1 = min(G.Cs[k], c0 + chunk);
  const int jb = blockIdx.x * kCj, s0 = blockIdx.z * P;
  const int jg = threadIdx.x % 16, sg = threadIdx.x / 16 % P, kq = threadIdx.x / (16 * P);
  const int cl = threadIdx.x % 32, w4 = threadIdx.x / 32;
  const float2* Kp = K + G.koff[k];
  const float2* Fp = F + G.toff[k];
  float2 acc[4], sum[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) acc[a] = sum[a] = make_float2(0.f, 0.f);
  // the running sums go into the totals every 8 chunks: one FP32 sum over a split's several thousand
  // entries made the 96^3 adjoint's error 1.5e-6, against 9.7e-7 of the mode-1 form
  auto fold = [&]() {
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      sum[a].x += acc[a].x;
      sum[a].y += acc[a].y;
      acc[a] = make_float2(0.f, 0.f);
    }
  };
  float2 kr[kCj / 4];
  auto fetch = [&](int c) {
#pragma unroll
    for (int u = 0; u < kCj / 4; ++u) {
      const int j = jb + w4 + 4 * u;
      kr[u] = c + cl < c1 && j < G.M ? __ldcs(Kp + (int64_t)j * G.Cs[k] + c + cl) : make_float2(0.f, 0.f);
    }
  };
  fetch(c0);
  for (int c = c0; c < c1; c += kCc) {
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kCj / 4; ++u) ks[cl][w4 + 4 * u] = kr[u];
    for (int e = threadIdx.x; e < kCc * P; e += 128) {
      const int i = e % kCc, s = e / kCc;
      fs[i][s] = c + i < c1 && s0 + s < p ? Fp[(int64_t)(s0 + s) * G.Ct + c + i] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    if (c + kCc < c1) fetch(c + kCc);
#pragma unroll 4
    for (int i = kq; i < kCc; i += KS) {
      const float4 k0 = *(const float4*)&ks[i][4 * jg], k1 = *(const float4*)&ks[i][4 * jg + 2];
      const float2 f = fs[i][sg];
      acc[0] = cfma_conj(make_float2(k0.x, k0.y), f, acc[0]);
      acc[1] = cfma_conj(make_float2(k0.z, k0.w), f, acc[1]);
      acc[2] = cfma_conj(make_float2(k1.x, k1.y), f, acc[2]);
      acc[3] = cfma_conj(make_float2(k1.z, k1.w), f, acc[3]);
    }
    if ((c - c0) / kCc % 8 == 7) fold();
  }
  fold();
#pragma unroll
  for (int a = 0; a < 4; ++a) red[kq][4 * jg + a][sg] = sum[a];
  __syncthreads();
  if (kq == 0)
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      for (int w = 1; w < KS; ++w) {
        sum[a].x += red[w][4 * jg + a][sg].x;
        sum[a].y += red[w][4 * jg + a][sg].y;
      }
      const int j = jb + 4 * jg + a, s = s0 + sg;
      if (j < G.M && s < p) part[((int64_t)blockIdx.y * p + s) * G.M + j] = sum[a];
    }
}

// out[j, s] = sum over the splits, in order; one warp per 32 columns, the splits over 8 warps
__global__ void __launch_bounds__(256) joint_sum_kernel(const float2* __restrict__ part, int M, int p, int splits,
                                                        float2* __restrict__ out, int64_t ldo) {
  __shared__ float2 red[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, j = blockIdx.x * 32 + lane, s = blockIdx.y;
  float2 a = make_float2(0.f, 0.f);
  if (j < M)
    for (int i = w; i < splits; i += 8) {
      const float2 v = part[((int64_t)i * p + s) * M + j];
      a.x += v.x;
      a.y += v.y;
    }
  red[w][lane] = a;
  __syncthreads();
  if (w == 0 && j < M) {
    for (int i = 1; i < 8; ++i) {
      a.x += red[i][lane].x;
      a.y += red[i][lane].y;
    }
    out[j + ldo * s] = a;
  }
}

// From this many right-hand sides on, the column sums run on the tensor cores (at least 8 a
// pass).  160 x 160 x 128, 4096 columns: whole forward 0.91 ms in FP32 at 4 against 1.11 ms at 8, whole
// adjoint 1.33 / 2.05 ms in FP32 at 2 / 4 against 1.04 ms at 4 and 1.23 ms at 8.
constexpr int kTcFwd = 5, kTcAdj = 3;

int rhs_per_cta(int p) { return p <= 1 ? 1 : p <= 2 ? 2 : 4; }  // FP32 column sums

template <int P>
void launch_core_fwd(const JointGeo& G, const float2* K, const float2* X, int64_t ldx, int p, int JS, float2* T, int* err,
                     int csmax, cudaStream_t st) {
  joint_core_fwd_kernel<P><<<dim3(ceil_div(csmax, 256), JS, G.q * ceil_div(p, P)), 128, 0, st>>>(G, K, X, ldx, p, JS, T, err);
  count_launch();
}
template <int P>
void launch_core_adj(const JointGeo& G, const float2* K, const float2* F, int p, int chunk, int splits, float2* part,
                     cudaStream_t st) {
  joint_core_adj_kernel<P><<<dim3(ceil_div(G.M, kCj), splits, ceil_div(p, P)), 128, 0, st>>>(G, K, F, p, chunk, part);
  count_launch();
}

// work split of ps <= kJointPass right-hand sides
struct FwdPlan {
  int P, JS;              // right-hand sides per CTA, slices of the column sum
  int64_t telems, qelems;
  FwdPlan(const JointGeo& G, int ps) {
    int cblocks = 0;
    for (int k = 0; k < G.q; ++k) cblocks += ceil_div(G.Cs[k], 256);
    P = rhs_per_cta(ps);
    // enough CTAs for 6 per SM, at least 32 columns a slice
    JS = std::max(1, std::min({16, G.M / 32, ceil_div(6 * sm_count(), cblocks * ceil_div(ps, P))}));
    if (ps >= kTcFwd) JS = 1;
    telems = (int64_t)JS * ps * G.Ct;
    qelems = (int64_t)ps * G.Qt;
  }
  size_t bytes() const { return sizeof(float2) * (telems + qelems); }
};
struct AdjPlan {
  int P, chunk, splits;   // core entries per split, number of splits
  int64_t felems, qelems, pelems;
  AdjPlan(const JointGeo& G, int ps) {
    P = rhs_per_cta(ps);
    // about 6 CTAs per SM, at least 256 entries a split
    const int want = std::max(1, 6 * sm_count() / (ceil_div(G.M, kCj) * ceil_div(ps, P)));
    chunk = (int)std::max<int64_t>(256, (G.Ct / want + kCc - 1) / kCc * kCc);
    splits = 0;
    for (int k = 0; k < G.q; ++k) splits += ceil_div(G.Cs[k], chunk);
    if (ps >= kTcAdj) joint_core_split(G, ps, &chunk, &splits);
    felems = (int64_t)ps * G.Ct;
    qelems = (int64_t)ps * G.Qt;
    pelems = (int64_t)splits * ps * G.M;
  }
  size_t bytes() const { return sizeof(float2) * (felems + qelems + pelems); }
};

}  // namespace

void joint_plan_work(JointCache* jc) {
  jc->work[0][0] = jc->work[1][0] = 0;
  for (int ps = 1; ps <= kJointPass; ++ps) {
    jc->work[0][ps] = std::max(jc->work[0][ps - 1], AdjPlan(jc->geo, ps).bytes());
    jc->work[1][ps] = std::max(jc->work[1][ps - 1], FwdPlan(jc->geo, ps).bytes());
  }
}

// tries of the product's bounded waits; a test limit applies to one product
static uint32_t take_wait_limit(Handle& h) {
  const uint32_t polls = std::min(h.test_first_wait, kJointPolls);
  h.test_first_wait = kWaitPolls;
  return polls;
}

int matvec_joint(Handle& h, const float2* X, int64_t ldx, int p, float2* Y, int64_t ldy, cudaStream_t st) {
  const JointCache& jc = *h.joint;
  const JointGeo& G = jc.geo;
  int* err = (int*)h.work_err.ptr;
  const uint32_t polls = take_wait_limit(h);
  ZBC_TRY(h.work_joint_fwd.ensure(joint_work_bytes(h, p, true)));
  int csmax = 0, rrmax = 0;
  for (int k = 0; k < G.q; ++k) {
    csmax = std::max(csmax, G.Cs[k]);
    rrmax = std::max(rrmax, G.R[k][0] * G.R[k][1]);
  }
  for (int s0 = 0; s0 < p; s0 += kJointPass) {
    const int ps = std::min(kJointPass, p - s0);
    const FwdPlan pl(G, ps);
    const int JS = pl.JS;
    float2* T = (float2*)h.work_joint_fwd.ptr;
    float2* Q = T + pl.telems;
    const float2* Xs = X + ldx * s0;
    switch (ps >= kTcFwd ? 0 : pl.P) {
      case 0: ZBC_TRY(joint_core_fwd(jc, Xs, ldx, ps, T, err, polls, st)); break;
      case 1: launch_core_fwd<1>(G, jc.K, Xs, ldx, ps, JS, T, err, csmax, st); break;
      case 2: launch_core_fwd<2>(G, jc.K, Xs, ldx, ps, JS, T, err, csmax, st); break;
      default: launch_core_fwd<4>(G, jc.K, Xs, ldx, ps, JS, T, err, csmax, st); break;
    }
    joint_mode3_fwd_kernel<<<dim3(ceil_div(rrmax, 128), ceil_div(G.n3, kZ), ps * G.q), 128, 0, st>>>(G, jc.basis, T, ps, JS, Q);
    count_launch();
    ZBC_TRY(joint_planes_fwd(jc, Q, ps, Y + ldy * s0, ldy, err, polls, st));
  }
  return ZBC_OK;
}

int rmatvec_joint(Handle& h, const float2* Phi, int64_t ldphi, int p, float2* out, int64_t ldo, cudaStream_t st) {
  const JointCache& jc = *h.joint;
  const JointGeo& G = jc.geo;
  int* err = (int*)h.work_err.ptr;
  const uint32_t polls = take_wait_limit(h);
  ZBC_TRY(h.work_joint_adj.ensure(joint_work_bytes(h, p, false)));
  int r3 = 0, rrmax = 0;
  for (int k = 0; k < G.q; ++k) {
    r3 = std::max(r3, G.R[k][2]);
    rrmax = std::max(rrmax, G.R[k][0] * G.R[k][1]);
  }
  for (int s0 = 0; s0 < p; s0 += kJointPass) {
    const int ps = std::min(kJointPass, p - s0);
    const AdjPlan pl(G, ps);
    const int chunk = pl.chunk, splits = pl.splits;
    float2* Q = (float2*)h.work_joint_adj.ptr;
    float2* F = Q + pl.qelems;
    float2* part = F + pl.felems;
    const float2* Ps = Phi + ldphi * s0;
    ZBC_TRY(joint_planes_adj(jc, Ps, ldphi, ps, Q, err, polls, st));
    joint_mode3_adj_kernel<<<dim3(ceil_div(rrmax, 128), ceil_div(r3, 8), ps * G.q), 128, 0, st>>>(G, jc.basis, Q, F);
    switch (ps >= kTcAdj ? 0 : pl.P) {
      case 0: ZBC_TRY(joint_core_adj(jc, F, ps, part, err, polls, st)); break;
      case 1: launch_core_adj<1>(G, jc.K, F, ps, chunk, splits, part, st); break;
      default: launch_core_adj<2>(G, jc.K, F, ps, chunk, splits, part, st); break;
    }
    joint_sum_kernel<<<dim3(ceil_div(G.M, 32), ps), 256, 0, st>>>(part, G.M, ps, splits, out + ldo * s0, ldo);
    count_launch(2);
    ZBC_TRY_CUDA(cudaGetLastError());
  }
  return ZBC_OK;
}

}  // namespace zbc
