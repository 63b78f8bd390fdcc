// Basis and reduced cores of the joint-subspace products (joint.cuh), built once per handle.
//
// Basis of component k and mode g: pivoted Gram-Schmidt in FP64 on the columns of all weighted
// factors F_t = U_g diag(d) / |U_g diag(d)|_F, d_a the norm of the core's slice a along mode g (for
// an HOSVD tensor d_a is the singular value of that column), so that the residual of F_t outside
// the basis is the relative Frobenius error that the projection makes on tensor t.  Each step takes
// the largest residual column, orthogonalises it once more against the basis and removes it from
// all columns; it ends when every tensor's residual is at most kJointEps.  Rows that are zero in
// every factor (masked voxels) stay exactly zero.
#include <algorithm>
#include <cmath>

#include "decomp.cuh"
#include "joint.cuh"

namespace zbc {

static void free_operands(JointCache* c) {
  if (c->basis) cudaFree(c->basis);
  if (c->K) cudaFree(c->K);
  if (c->bop) cudaFree(c->bop);
  if (c->kscale) cudaFree(c->kscale);
  c->basis = c->K = nullptr;
  c->bop = nullptr;
  c->kscale = nullptr;
  c->bytes = 0;
}

void joint_release(JointCache* c) {
  if (!c) return;
  free_operands(c);
  delete c;
}
int64_t joint_bytes(const JointCache* c) { return c ? c->bytes : 0; }

namespace {

// one weighted factor (tensor t, mode g): r columns of n entries at F, part of problem pr = k + q g
struct FactorJob {
  const float2* G;   // core r1 x r2 x r3
  const float2* U;   // n x r
  double2* F;
  double2* C;        // R x r coefficients B^H U (filled by coef_kernel)
  int64_t col0;      // index of its first column within the problem
  int n, r, r1, r2, r3, g, pr;
};

struct Problem {     // one (k, g)
  double2* F;        // all columns, n each
  double2* Q;        // n x cap basis
  int n, cap;
};

struct PivotState {  // per problem, double buffered by step parity
  unsigned long long col;  // largest column residual^2 (float bits) << 32 | ~column
  unsigned int tensor;     // largest tensor residual^2 (float bits)
};

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// one CTA per factor: F = U diag(d) / norm, and the first pivot (ranks of at most kJointRmax)
__global__ void __launch_bounds__(128) weight_kernel(const FactorJob* jobs, const Problem* prob, PivotState* state,
                                                     double* resid) {
  const FactorJob jb = jobs[blockIdx.x];
  __shared__ double w2[kJointRmax], c2[kJointRmax];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t ne = (int64_t)jb.r1 * jb.r2 * jb.r3;
  const int64_t per = ne / jb.r;  // entries of one slice along mode g
  const int64_t s_in = jb.g == 0 ? 1 : jb.g == 1 ? jb.r1 : (int64_t)jb.r1 * jb.r2;
  for (int a = warp; a < jb.r; a += 4) {
    double s = 0.0, u = 0.0;
    for (int64_t e = lane; e < per; e += 32) {
      const int64_t lo = e % s_in, hi = e / s_in;
      const float2 v = jb.G[lo + s_in * (a + (int64_t)jb.r * hi)];
      s += (double)v.x * v.x + (double)v.y * v.y;
    }
    for (int i = lane; i < jb.n; i += 32) {
      const float2 v = jb.U[i + (int64_t)jb.n * a];
      u += (double)v.x * v.x + (double)v.y * v.y;
    }
    s = warp_sum(s);
    u = warp_sum(u);
    if (lane == 0) {
      w2[a] = s;
      c2[a] = s * u;
    }
  }
  __syncthreads();
  double tot = 0.0;
  for (int a = 0; a < jb.r; ++a) tot += c2[a];
  const double inv = tot > 0.0 ? 1.0 / sqrt(tot) : 0.0;
  for (int64_t e = threadIdx.x; e < (int64_t)jb.n * jb.r; e += blockDim.x) {
    const int a = (int)(e / jb.n);
    const double s = sqrt(w2[a]) * inv;
    const float2 v = jb.U[e];
    jb.F[e] = make_double2(v.x * s, v.y * s);
  }
  if (threadIdx.x == 0) {
    // a non-finite tensor gives a non-finite residual, which never passes the test
    const double res = tot > 0.0 ? 1.0 : (tot == 0.0 ? 0.0 : INFINITY);
    resid[blockIdx.x] = res;
    atomicMax(&state[jb.pr].tensor, __float_as_uint((float)res));
    for (int a = 0; a < jb.r; ++a) {
      const float c = (float)(c2[a] * inv * inv);
      if (c > 0.f)
        atomicMax(&state[jb.pr].col, (unsigned long long)__float_as_uint(c) << 32 | (0xffffffffu - (unsigned)(jb.col0 + a)));
    }
  }
}

// one CTA per problem: the next basis vector from the pivot column, or the end of the problem
__global__ void __launch_bounds__(256) pivot_basis_kernel(const Problem* prob, const PivotState* cur, PivotState* next,
                                                          int* rank, int step, float eps2) {
  const int pr = blockIdx.x;
  const Problem P = prob[pr];
  __shared__ double2 dots[kJointRmax];
  __shared__ double red[8];
  extern __shared__ double2 v[];  // n
  if (threadIdx.x == 0) next[pr] = PivotState{0ull, 0u};
  if (rank[pr] >= 0) return;  // done
  const float worst = __uint_as_float(cur[pr].tensor);
  if (worst <= eps2 || cur[pr].col == 0ull) {
    if (threadIdx.x == 0) rank[pr] = worst <= eps2 ? step : P.cap + 1;
    return;
  }
  if (step >= P.cap || !(worst < 2.f)) {
    if (threadIdx.x == 0) rank[pr] = P.cap + 1;  // no basis within the cap (or a non-finite tensor)
    return;
  }
  const int64_t col = 0xffffffffu - (unsigned)(cur[pr].col & 0xffffffffull);
  const double2* f = P.F + col * P.n;
  for (int i = threadIdx.x; i < P.n; i += blockDim.x) v[i] = f[i];
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int a = warp; a < step; a += 8) {  // dots = Q^H v
    double2 d = make_double2(0.0, 0.0);
    for (int i = lane; i < P.n; i += 32) d = zfma_conj(P.Q[(int64_t)a * P.n + i], v[i], d);
    d.x = warp_sum(d.x);
    d.y = warp_sum(d.y);
    if (lane == 0) dots[a] = d;
  }
  __syncthreads();
  double s = 0.0;
  for (int i = threadIdx.x; i < P.n; i += blockDim.x) {
    double2 x = v[i];
    for (int a = 0; a < step; ++a) {
      const double2 q = P.Q[(int64_t)a * P.n + i], d = dots[a];
      x.x -= q.x * d.x - q.y * d.y;
      x.y -= q.x * d.y + q.y * d.x;
    }
    v[i] = x;
    s += x.x * x.x + x.y * x.y;
  }
  s = warp_sum(s);
  if (lane == 0) red[warp] = s;
  __syncthreads();
  s = 0.0;
  for (int w = 0; w < 8; ++w) s += red[w];
  const double inv = s > 0.0 ? 1.0 / sqrt(s) : 0.0;
  for (int i = threadIdx.x; i < P.n; i += blockDim.x)
    P.Q[(int64_t)step * P.n + i] = make_double2(v[i].x * inv, v[i].y * inv);
}

// one warp per factor: F -= q (q^H F) for the basis vector of this step, the residuals and the next
// pivot.  Factors already inside the basis are left alone (a residual only shrinks).
__global__ void __launch_bounds__(128) project_kernel(const FactorJob* jobs, int nf, const Problem* prob,
                                                      const int* rank, PivotState* next, double* resid, int step,
                                                      double eps2) {
  const int f = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (f >= nf) return;
  const FactorJob jb = jobs[f];
  if (rank[jb.pr] >= 0) return;
  double res = resid[f];
  if (res > eps2) {
    const double2* q = prob[jb.pr].Q + (int64_t)step * jb.n;
    res = 0.0;
    for (int a = 0; a < jb.r; ++a) {
      double2* x = jb.F + (int64_t)a * jb.n;
      double2 d = make_double2(0.0, 0.0);
      for (int i = lane; i < jb.n; i += 32) d = zfma_conj(q[i], x[i], d);
      d.x = warp_sum(d.x);
      d.y = warp_sum(d.y);
      double s = 0.0;
      for (int i = lane; i < jb.n; i += 32) {
        double2 y = x[i];
        const double2 c = q[i];
        y.x -= c.x * d.x - c.y * d.y;
        y.y -= c.x * d.y + c.y * d.x;
        x[i] = y;
        s += y.x * y.x + y.y * y.y;
      }
      s = warp_sum(s);
      res += s;
      if (lane == 0 && s > 0.0)
        atomicMax(&next[jb.pr].col,
                  (unsigned long long)__float_as_uint((float)s) << 32 | (0xffffffffu - (unsigned)(jb.col0 + a)));
    }
    if (lane == 0) resid[f] = res;
  }
  // float rounding up, so that a residual just above the bound stays above it
  if (lane == 0) atomicMax(&next[jb.pr].tensor, __float_as_uint(__double2float_ru(res)));
}

// C = B^H U of one factor, one warp per entry (FP64)
__global__ void __launch_bounds__(256) coef_kernel(const FactorJob* jobs, const Problem* prob, const int* rank) {
  const FactorJob jb = jobs[blockIdx.x];
  const int R = rank[jb.pr], lane = threadIdx.x & 31;
  const double2* Q = prob[jb.pr].Q;
  for (int e = threadIdx.x >> 5; e < R * jb.r; e += 8) {
    const int x = e % R, a = e / R;
    double2 d = make_double2(0.0, 0.0);
    for (int i = lane; i < jb.n; i += 32) {
      const float2 u = jb.U[i + (int64_t)jb.n * a];
      d = zfma_conj(Q[(int64_t)x * jb.n + i], make_double2(u.x, u.y), d);
    }
    d.x = warp_sum(d.x);
    d.y = warp_sum(d.y);
    if (lane == 0) jb.C[e] = d;
  }
}

__global__ void __launch_bounds__(256) round_basis_kernel(const double2* Q, float2* B, int64_t len) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < len; e += (int64_t)gridDim.x * blockDim.x)
    B[e] = make_float2((float)Q[e].x, (float)Q[e].y);
}

// The three mode products of K = G x1 C1 x2 C2 x3 C3 for a batch of tensors, FP64, rounded once.
struct CoreJob {
  const float2* G;
  const double2 *C1, *C2, *C3;  // R_g x r_g
  double2 *T1, *T2;             // R1 x r2 x r3, R1 x R2 x r3
  float2* K;                    // R1 x R2 x R3, then zeros up to Cs
  int r1, r2, r3, R1, R2, R3, Cs;
};
__global__ void __launch_bounds__(256) core1_kernel(const CoreJob* jobs) {
  const CoreJob jb = jobs[blockIdx.y];
  const int ne = jb.R1 * jb.r2 * jb.r3;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < ne; e += gridDim.x * blockDim.x) {
    const int x = e % jb.R1, bc = e / jb.R1;
    double2 s = make_double2(0.0, 0.0);
    for (int a = 0; a < jb.r1; ++a) {
      const float2 g = jb.G[a + (int64_t)jb.r1 * bc];
      s = zfma(jb.C1[x + jb.R1 * a], make_double2(g.x, g.y), s);
    }
    jb.T1[e] = s;
  }
}
__global__ void __launch_bounds__(256) core2_kernel(const CoreJob* jobs) {
  const CoreJob jb = jobs[blockIdx.y];
  const int ne = jb.R1 * jb.R2 * jb.r3;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < ne; e += gridDim.x * blockDim.x) {
    const int x = e % jb.R1, y = e / jb.R1 % jb.R2, c = e / (jb.R1 * jb.R2);
    double2 s = make_double2(0.0, 0.0);
    for (int b = 0; b < jb.r2; ++b) s = zfma(jb.T1[x + jb.R1 * (b + jb.r2 * c)], jb.C2[y + jb.R2 * b], s);
    jb.T2[e] = s;
  }
}
constexpr int kCoreZ = 4;  // values of mode 3 per thread of core3_kernel
__global__ void __launch_bounds__(256) core3_kernel(const CoreJob* jobs) {
  const CoreJob jb = jobs[blockIdx.y];
  const int RR = jb.R1 * jb.R2, nz = (jb.R3 + kCoreZ - 1) / kCoreZ;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < RR * nz; e += gridDim.x * blockDim.x) {
    const int xy = e % RR, z0 = e / RR * kCoreZ;
    double2 s[kCoreZ];
#pragma unroll
    for (int z = 0; z < kCoreZ; ++z) s[z] = make_double2(0.0, 0.0);
    for (int c = 0; c < jb.r3; ++c) {
      const double2 t = jb.T2[xy + (int64_t)RR * c];
#pragma unroll
      for (int z = 0; z < kCoreZ; ++z)
        if (z0 + z < jb.R3) s[z] = zfma(t, jb.C3[z0 + z + jb.R3 * c], s[z]);
    }
#pragma unroll
    for (int z = 0; z < kCoreZ; ++z)
      if (z0 + z < jb.R3) jb.K[xy + (int64_t)RR * (z0 + z)] = make_float2((float)s[z].x, (float)s[z].y);
  }
  if (blockIdx.x == 0)
    for (int e = RR * jb.R3 + threadIdx.x; e < jb.Cs; e += blockDim.x) jb.K[e] = make_float2(0.f, 0.f);
}

int cuda_status(cudaError_t e, const char* what) {
  set_error("joint basis: %s: %s", what, cudaGetErrorString(e));
  return e == cudaErrorMemoryAllocation ? ZBC_ENOMEM : ZBC_ECUDA;
}

}  // namespace

static int build(Handle& h, JointCache* jc, cudaStream_t st) {
  const int q = h.q, T = (int)h.desc.size(), n[3] = {h.n1, h.n2, h.n3}, NP = 3 * q;
  JointGeo& g = jc->geo;
  g.n1 = h.n1;
  g.n2 = h.n2;
  g.n3 = h.n3;
  g.q = q;
  g.M = h.M;
  // A factor of more than kJointRmax columns has no basis of kJointRmax vectors (unless some of its
  // columns carry less than the tolerance), and the kernels below hold its weights in arrays of that size
  for (const TensorDesc& d : h.desc)
    if (std::max({d.r1, d.r2, d.r3}) > kJointRmax) return ZBC_OK;  // unusable
  // factors, grouped by (mode, component) so that a problem's columns are one run
  std::vector<FactorJob> fj;
  std::vector<Problem> prob(NP);
  int64_t fcols = 0, celems = 0, qelems = 0;
  std::vector<int64_t> foff, coff;
  for (int m = 0; m < 3; ++m)
    for (int k = 0; k < q; ++k) {
      const int pr = k + q * m, cap = std::min(kJointRmax, n[m]);
      prob[pr].n = n[m];
      prob[pr].cap = cap;
      int64_t c0 = 0;
      for (int j = 0; j < h.M; ++j) {
        const int t = j * q + k;
        const TensorDesc& d = h.desc[t];
        const int r[3] = {d.r1, d.r2, d.r3};
        const float2* G = h.d_pool + d.off;
        const float2* U = G + (int64_t)d.r1 * d.r2 * d.r3;
        if (m > 0) U += (int64_t)n[0] * d.r1;
        if (m > 1) U += (int64_t)n[1] * d.r2;
        fj.push_back(FactorJob{G, U, nullptr, nullptr, c0, n[m], r[m], d.r1, d.r2, d.r3, m, pr});
        foff.push_back(fcols);
        coff.push_back(celems);
        fcols += (int64_t)n[m] * r[m];
        celems += (int64_t)cap * r[m];
        c0 += r[m];
      }
      if (c0 >= 0xffffffffll) return ZBC_OK;  // unusable: the pivot packs a 32-bit column
      qelems += (int64_t)n[m] * cap;
    }
  const int nf = (int)fj.size();
  DevBuf F, Q, C, jobs, probs, state, rank, resid;
  ZBC_TRY(F.ensure(sizeof(double2) * fcols));
  ZBC_TRY(Q.ensure(sizeof(double2) * qelems));
  ZBC_TRY(C.ensure(sizeof(double2) * celems));
  ZBC_TRY(jobs.ensure(sizeof(FactorJob) * nf));
  ZBC_TRY(probs.ensure(sizeof(Problem) * NP));
  ZBC_TRY(state.ensure(2 * sizeof(PivotState) * NP));
  ZBC_TRY(rank.ensure(sizeof(int) * NP));
  ZBC_TRY(resid.ensure(sizeof(double) * nf));
  std::vector<int64_t> qoff(NP);
  int64_t qo = 0;
  for (int pr = 0; pr < NP; ++pr) {
    qoff[pr] = qo;
    prob[pr].Q = (double2*)Q.ptr + qo;
    qo += (int64_t)prob[pr].n * prob[pr].cap;
    prob[pr].F = (double2*)F.ptr + foff[(size_t)pr * h.M];
  }
  for (int f = 0; f < nf; ++f) {
    fj[f].F = (double2*)F.ptr + foff[f];
    fj[f].C = (double2*)C.ptr + coff[f];
  }
  ZBC_TRY_CUDA(cudaMemcpyAsync(jobs.ptr, fj.data(), sizeof(FactorJob) * nf, cudaMemcpyHostToDevice, st));
  ZBC_TRY_CUDA(cudaMemcpyAsync(probs.ptr, prob.data(), sizeof(Problem) * NP, cudaMemcpyHostToDevice, st));
  ZBC_TRY_CUDA(cudaMemsetAsync(state.ptr, 0, 2 * sizeof(PivotState) * NP, st));
  ZBC_TRY_CUDA(cudaMemsetAsync(rank.ptr, 0xff, sizeof(int) * NP, st));  // -1: running
  const auto* dj = (const FactorJob*)jobs.ptr;
  const auto* dp = (const Problem*)probs.ptr;
  auto* ds = (PivotState*)state.ptr;
  auto* dr = (int*)rank.ptr;
  const double eps2 = kJointEps * kJointEps;
  const int nmax = std::max(n[0], std::max(n[1], n[2]));
  const size_t vsm = sizeof(double2) * nmax;
  if (vsm > 48 * 1024) ZBC_TRY(set_smem_limit<pivot_basis_kernel>(64 * 1024 + 4096));
  weight_kernel<<<nf, 128, 0, st>>>(dj, dp, ds, (double*)resid.ptr);
  count_launch();
  std::vector<int> rk(NP, -1);
  bool running = true;
  for (int step = 0; step <= kJointRmax && running; ++step) {
    PivotState *cur = ds + (step & 1) * NP, *next = ds + (~step & 1) * NP;
    pivot_basis_kernel<<<NP, 256, vsm, st>>>(dp, cur, next, dr, step, (float)eps2);
    project_kernel<<<ceil_div(nf, 4), 128, 0, st>>>(dj, nf, dp, dr, next, (double*)resid.ptr, step, eps2);
    count_launch(2);
    if (step % 8 == 7 || step == kJointRmax) {
      ZBC_TRY_CUDA(cudaMemcpyAsync(rk.data(), dr, sizeof(int) * NP, cudaMemcpyDeviceToHost, st));
      ZBC_TRY_CUDA(cudaStreamSynchronize(st));
      running = false;
      for (int pr = 0; pr < NP; ++pr) {
        running = running || rk[pr] < 0;
        if (rk[pr] > prob[pr].cap) return ZBC_OK;  // no basis within the cap: unusable
      }
    }
  }
  // geometry, and whether the form is worth its memory and work: the columns' sums over R1 R2 R3
  // entries plus one expansion against the decompression of every column, per right-hand side
  double work = 0.0, direct = 0.0, wbytes = 0.0;
  int64_t kelems = 0, belems = 0;
  g.Ct = g.Qt = 0;
  for (int k = 0; k < q; ++k) {
    for (int m = 0; m < 3; ++m) {
      if (rk[k + q * m] < 1) return ZBC_OK;
      g.R[k][m] = rk[k + q * m];
      g.boff[k][m] = belems;
      belems += (int64_t)n[m] * g.R[k][m];
    }
    const int64_t C3 = (int64_t)g.R[k][0] * g.R[k][1] * g.R[k][2];
    g.Cs[k] = (int)((C3 + 3) / 4 * 4);
    g.koff[k] = kelems;
    kelems += (int64_t)h.M * g.Cs[k];
    g.toff[k] = g.Ct;
    g.Ct += g.Cs[k];
    g.qoff[k] = g.Qt;
    g.Qt += (int64_t)g.R[k][0] * g.R[k][1] * n[2];
    work += (double)h.M * C3 + (double)h.nv() * g.R[k][0];
  }
  for (int t = 0; t < T; ++t) {
    direct += (double)h.nv() * h.desc[t].r1;
    wbytes += 8.0 * n[1] * n[2] * ((h.desc[t].r1 + 1) / 2 * 2);
  }
  // K may take twice the bytes of the decompression cache's W where the products are long (the
  // 96^3 head coil: the same 2.7 GB); a handle whose products take microseconds either way keeps it
  // under half of W, less than the operands that tuning would otherwise leave
  jc->large = direct > 1e8;
  if (work > 0.5 * direct || 8.0 * kelems > (jc->large ? 2.0 : 0.5) * wbytes) return ZBC_OK;
  // and it leaves a quarter of its size free (W is built) for the workspaces of the products
  size_t mem_free = 0, mem_total = 0;
  ZBC_TRY_CUDA(cudaMemGetInfo(&mem_free, &mem_total));
  if (sizeof(float2) * (size_t)kelems > mem_free / 5 * 4) return ZBC_ENOMEM;
  cudaError_t e = cudaMalloc(&jc->basis, sizeof(float2) * belems);
  if (e == cudaSuccess) e = cudaMalloc(&jc->K, sizeof(float2) * kelems);
  if (e == cudaSuccess) e = cudaMalloc(&jc->bop, joint_planes_bytes(g));
  if (e == cudaSuccess) e = cudaMalloc(&jc->kscale, joint_core_bytes(g));
  if (e != cudaSuccess) {
    cudaGetLastError();
    return cuda_status(e, "allocation");
  }
  jc->bytes = (int64_t)(sizeof(float2) * (belems + kelems) + joint_planes_bytes(g) + joint_core_bytes(g));
  for (int k = 0; k < q; ++k)
    for (int m = 0; m < 3; ++m) {
      const int64_t len = (int64_t)n[m] * g.R[k][m];
      round_basis_kernel<<<std::min(1024, ceil_div(len, 256)), 256, 0, st>>>((double2*)Q.ptr + qoff[k + q * m],
                                                                             jc->basis + g.boff[k][m], len);
      count_launch();
    }
  ZBC_TRY(joint_planes_build(g, jc->basis, jc->bop, st));
  coef_kernel<<<nf, 256, 0, st>>>(dj, dp, dr);
  count_launch();
  // reduced cores in batches that keep the FP64 intermediates near 1 GB
  int64_t t1max = 0, t2max = 0;
  for (int t = 0; t < T; ++t) {
    const int* R = g.R[t % q];
    t1max = std::max(t1max, (int64_t)R[0] * h.desc[t].r2 * h.desc[t].r3);
    t2max = std::max(t2max, (int64_t)R[0] * R[1] * h.desc[t].r3);
  }
  const int batch = (int)std::max<int64_t>(1, std::min<int64_t>(std::min(T, 32768), ((int64_t)1 << 30) / (16 * (t1max + t2max))));
  DevBuf T1, T2, cjobs;
  ZBC_TRY(T1.ensure(sizeof(double2) * t1max * batch));
  ZBC_TRY(T2.ensure(sizeof(double2) * t2max * batch));
  ZBC_TRY(cjobs.ensure(sizeof(CoreJob) * T));
  std::vector<CoreJob> cj(T);
  for (int t = 0; t < T; ++t) {
    const int j = t / q, k = t % q, b = t % batch;
    const TensorDesc& d = h.desc[t];
    const FactorJob* f[3];
    for (int m = 0; m < 3; ++m) f[m] = &fj[((size_t)(k + q * m)) * h.M + j];
    cj[t] = CoreJob{f[0]->G, f[0]->C, f[1]->C, f[2]->C, (double2*)T1.ptr + t1max * b, (double2*)T2.ptr + t2max * b,
                    jc->K + g.koff[k] + (int64_t)j * g.Cs[k], d.r1, d.r2, d.r3, g.R[k][0], g.R[k][1], g.R[k][2],
                    g.Cs[k]};
  }
  ZBC_TRY_CUDA(cudaMemcpyAsync(cjobs.ptr, cj.data(), sizeof(CoreJob) * T, cudaMemcpyHostToDevice, st));
  int csmax = 0;
  for (int k = 0; k < q; ++k) csmax = std::max(csmax, g.Cs[k]);
  for (int t0 = 0; t0 < T; t0 += batch) {
    const int nt = std::min(batch, T - t0);
    const auto* p = (const CoreJob*)cjobs.ptr + t0;
    core1_kernel<<<dim3(std::min(64, ceil_div(t1max, 256)), nt), 256, 0, st>>>(p);
    core2_kernel<<<dim3(std::min(64, ceil_div(t2max, 256)), nt), 256, 0, st>>>(p);
    core3_kernel<<<dim3(std::min(64, ceil_div(csmax / kCoreZ + 1, 256)), nt), 256, 0, st>>>(p);
    count_launch(3);
  }
  bool fits = false;
  ZBC_TRY(joint_core_build(g, jc->K, jc->kscale, &fits, st));
  e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_status(e, "reduced cores");
  joint_plan_work(jc);
  jc->usable = fits;
  return ZBC_OK;
}

int build_joint(Handle& h, cudaStream_t st) {
  if (h.joint) return ZBC_OK;
  h.joint = new JointCache();  // kept also when unusable, so that the search is not repeated
  const int s = build(h, h.joint, st);
  h.joint->no_room = s == ZBC_ENOMEM;
  if (!h.joint->usable) free_operands(h.joint);
  return s;
}

}  // namespace zbc
