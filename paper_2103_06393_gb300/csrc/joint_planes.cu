// The plane products of the joint form (joint.cuh) on the tensor cores: per right-hand side s,
// component k and plane i3,
//   forward  Y[:, :, i3] = B1 S,  S = Q[i3] B2^T          (one write of Y)
//   adjoint  Q[i3] = V conj(B2),  V = B1^H Phi[:, :, i3]  (one read of Phi)
// The contraction with B1 touches every voxel R1 times and is a tcgen05 GEMM (kind::f16); the one
// with B2 works on R1 rows: a second GEMM before it in the forward, FP32 on the CUDA cores in the
// adjoint.  Operands are split into fp16 hi + lo (x = hi + lo to 2^-22) after scaling by powers of two
// and the three products hi hi, hi lo, lo hi are summed in FP32.  In FP32 on the CUDA cores the same planes took 3.1 / 4.7 ms
// (320 x 320 x 256, 8 right-hand sides, R = 23-25: 57 % of the FP32 rate) against 0.74 ms that
// writing or reading the 5 GB takes.
//
// Operand conventions: a complex row entry is the pair of K elements (Re, Im), so with
//   A[i1] = (Re, Im) B1[i1, :]  and  B rows (Re S, -Im S), (Im S, Re S)
// D's column pair is (Re, Im) Y; the adjoint contracts Phi's own (Re, Im) pairs along i1 with rows
// (Re b, Im b), (-Im b, Re b) of the basis vector b, which gives (Re, Im) of conj(b) Phi.
#include <algorithm>

#include "joint_tc.cuh"

namespace zbc {
namespace {

// ---------------------------------------------------------------------------------------------
// forward
// ---------------------------------------------------------------------------------------------
// A CTA takes a tile of `T2` i2 (at most 112) and up to `nb` blocks of 128 i1, keeps the hi / lo rows of
// B2 and B1 for them in shared memory and walks the planes (s, i3) of its component.  Per plane:
//   workers     Q[i3] (loaded a plane ahead) scaled by its largest entry, split: rows of one MMA operand
//   MMA 1       D1[i2, (Re, Im) x] = B2 Q^T           M = 128, N = 2 R1p, K = 2 R2p
//   workers     D1 -> S's rows for the second MMA (a fixed shift: |S| < 12 max |Q|)
//   MMA 2       D2[i1, (Re, Im) i2] = B1 S            M = 128, N = 2 T2, K = 2 R1p, per i1 block, two
//                                                     accumulators in turn
//   workers     D2 -> Y, 32 consecutive i1 per store
// The ninth warp issues all MMAs.  Where two copies of S fit (ns = 2) the workers make plane t + 1's S
// before they store plane t, so that the MMAs of one plane overlap the stores of the other; else only
// the next plane's Q is split ahead.  S on the CUDA cores (R1 R2 multiply-adds per i2 and plane) took two thirds of the
// issue slots: 0.48 / 1.22 / 1.03 ms for 96^3/16, 160 x 160 x 128/32 and 320 x 320 x 256/8 planes.
// K-major core-matrix layout without swizzle, KB chunks of 16 bytes a row; rows of B1 past n1 are not
// stored: MMA 2 reads what follows, into accumulator rows that nothing reads.
struct FwdShape {
  int R1p, R2p, T2, nt2, nb, gy, ns;
  __host__ __device__ size_t b1_bytes(int n1) const { return (size_t)8 * R1p * min(nb * 128, (n1 + 7) / 8 * 8); }
  __host__ __device__ size_t s_bytes() const { return (size_t)16 * R1p * T2; }
  __host__ __device__ size_t b2_bytes() const { return (size_t)1024 * R2p; }
  __host__ __device__ size_t q_bytes() const { return (size_t)16 * R1p * R2p; }
  __host__ __device__ size_t bytes(int n1) const { return b1_bytes(n1) + ns * s_bytes() + b2_bytes() + q_bytes(); }
};
// 16 worker warps: with one CTA an SM, 8 of them left the schedulers two thirds idle
constexpr int kFwdWorkers = 512, kFwdThreads = kFwdWorkers + 32, kFwdGroups = kFwdWorkers / 128;
constexpr int kQRegs = kJointRmax * kJointRmax / kFwdWorkers;

__global__ void __launch_bounds__(kFwdThreads, 1)
    joint_planes_fwd_kernel(const __grid_constant__ JointGeo G, const __grid_constant__ FwdShape F,
                            const float2* __restrict__ basis, const float2* __restrict__ Q, int p, float2* __restrict__ Y,
                            int64_t ldy, int* __restrict__ err, uint32_t polls) {
  extern __shared__ __align__(128) unsigned char smem_f[];
  __shared__ __align__(8) uint64_t done[2], dfree[2], sready, qready, s1done;
  __shared__ uint32_t tmem_base;
  __shared__ float wmax[2][kFwdWorkers / 32];
  const int k = blockIdx.z, R1 = G.R[k][0], R2 = G.R[k][1], RR = R1 * R2;
  const int R1p = F.R1p, KB = R1p / 4, KB1 = F.R2p / 4, T2 = F.T2;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int i20 = (int)(blockIdx.y % F.nt2) * T2, row0 = (int)(blockIdx.y / F.nt2) * F.nb * 128;
  const int rows = min(F.nb * 128, G.n1 - row0), nblk = (rows + 127) / 128;
  unsigned char* sa = smem_f;                    // B1: [block][term][rows]
  unsigned char* ss = sa + F.b1_bytes(G.n1);     // S: [ns][term][2 T2 rows]
  unsigned char* sb2 = ss + F.ns * F.s_bytes();  // B2: [term][128 rows]
  unsigned char* sq = sb2 + F.b2_bytes();        // Q: [term][2 R1p rows]
  const uint32_t ablk = 128u * KB * 16u, sterm = 2u * T2 * KB * 16u, b2term = 128u * KB1 * 16u, qterm = 2u * R1p * KB1 * 16u;
  const uint32_t alast = (uint32_t)((rows - (nblk - 1) * 128 + 7) / 8) * 8u * KB * 16u;
  constexpr uint32_t ncols = 512;
  const uint32_t d2 = 2 * R1p;                   // D1 in columns 0 .. 2 R1p - 1, two D2 of 2 T2 columns after it
  const int lag = F.ns - 1;
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&done[i], 1);
      tc::mbar_init(&dfree[i], kFwdWorkers / 32);
    }
    tc::mbar_init(&sready, kFwdWorkers / 32);
    tc::mbar_init(&qready, kFwdWorkers / 32);
    tc::mbar_init(&s1done, 1);
  }
  if (warp == 0) tc::tmem_alloc(&tmem_base, ncols);
  auto rows_of = [&](unsigned char* dst, uint32_t lo, int r, int kc, int kb, const float2* b, int n, int i, bool live, int R) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float2 v = live && 4 * kc + u < R ? b[(int64_t)(4 * kc + u) * n + i] : make_float2(0.f, 0.f);
      split2(v.x * pow2f(kBasisShift), v.y * pow2f(kBasisShift), h[u], l[u]);
    }
    unsigned char* d = dst + tc::core_off(r, kc, kb);
    *(uint4*)d = make_uint4(h[0], h[1], h[2], h[3]);
    *(uint4*)(d + lo) = make_uint4(l[0], l[1], l[2], l[3]);
  };
  const int rows8 = (rows + 7) / 8 * 8;
  for (int e = tid; e < rows8 * KB; e += kFwdThreads) {
    const int rr = e % rows8, b = rr / 128;
    rows_of(sa + (size_t)b * 2 * ablk, b == nblk - 1 ? alast : ablk, rr % 128, e / rows8, KB, basis + G.boff[k][0], G.n1,
            row0 + rr, row0 + rr < G.n1, R1);
  }
  for (int e = tid; e < 128 * KB1; e += kFwdThreads) {
    const int r = e % 128;
    rows_of(sb2, b2term, r, e / 128, KB1, basis + G.boff[k][1], G.n2, i20 + r, r < T2 && i20 + r < G.n2, R2);
  }
  for (uint32_t e = tid; e < qterm / 8; e += kFwdThreads) ((uint4*)sq)[e] = make_uint4(0, 0, 0, 0);  // the pad stays zero
  tc::fence_proxy_async();
  __syncthreads();
  const uint32_t tmem = tmem_base;
  const int planes = p * G.n3;
  const int mine = (planes - 1 - (int)blockIdx.x) / (int)gridDim.x + 1;  // grid x <= planes
  Waits waits{err, polls};
  if (warp == kFwdWorkers / 32) {
    if (lane == 0) {
      const uint32_t b1 = tc::smem_u32(sa), s0 = tc::smem_u32(ss), b2 = tc::smem_u32(sb2), q0 = tc::smem_u32(sq);
      const uint32_t sbo = KB * 128u, sbo1 = KB1 * 128u;
      auto chain = [&](uint32_t d, uint32_t a, uint32_t alo, uint32_t b, uint32_t blo, uint32_t st, int steps, uint32_t id) {
        for (int ks = 0; ks < steps; ++ks) {
          const uint64_t ah = tc::smem_desc(a + ks * 256u, 128, st), al = tc::smem_desc(a + alo + ks * 256u, 128, st);
          const uint64_t bh = tc::smem_desc(b + ks * 256u, 128, st), bl = tc::smem_desc(b + blo + ks * 256u, 128, st);
          tc::mma<0>(d, al, bh, id, ks > 0);
          tc::mma<0>(d, ah, bl, id, 1);
          tc::mma<0>(d, ah, bh, id, 1);
        }
      };
      int m1 = 0, n = 0;  // MMAs 1 issued, accumulators of MMA 2 used so far
      auto mma1 = [&](int t) {
        waits.one(&qready, t & 1);
        if (!waits.ok) return;
        tc::fence_after();
        chain(tmem, b2, b2term, q0, qterm, sbo1, KB1 / 2, tc::instr_desc(128, 2 * R1p, 0));
        tc::commit(&s1done);
        ++m1;
      };
      mma1(0);
      for (int t = 0; t < mine && waits.ok; ++t) {
        waits.one(&sready, t & 1);
        if (lag && t + 1 < mine) mma1(t + 1);
        for (int b = 0; b < nblk && waits.ok; ++b, ++n) {
          waits.one(&dfree[n & 1], ((n >> 1) & 1) ^ 1);  // a fresh barrier's preceding phase counts as complete
          if (!waits.ok) break;
          tc::fence_after();
          chain(tmem + d2 + (uint32_t)((n & 1) * 2 * T2), b1 + (uint32_t)b * 2 * ablk, b == nblk - 1 ? alast : ablk,
                s0 + (uint32_t)(t & lag) * 2 * sterm, sterm, sbo, KB / 2, tc::instr_desc(128, 2 * T2, 0));
          tc::commit(&done[n & 1]);
        }
        if (!lag && t + 1 < mine) mma1(t + 1);
      }
      drain1(&s1done, m1);
      drain2(done, n);
    }
    __syncwarp();
  } else {
    const int q4 = warp & 3, grp = warp >> 2;  // accumulator rows; the groups share its columns
    const float gain = mixed_gain(KB1 / 2, KB / 2);
    const float2* Qk = Q + G.qoff[k];
    float2 qr[kQRegs];
    uint32_t qoff[kQRegs];  // of the pair (x, y) in row 2 x; row 2 x + 1 lies 16 bytes further
#pragma unroll
    for (int u = 0; u < kQRegs; ++u) {
      const int x = (tid + kFwdWorkers * u) % R1, y = (tid + kFwdWorkers * u) / R1;
      qoff[u] = tc::core_off(2 * x, y / 4, KB1) + 4 * (y % 4);
    }
    auto fetch_q = [&](int t) {
      const int pl = (int)blockIdx.x + t * (int)gridDim.x;
      const float2* Qp = Qk + (int64_t)(pl / G.n3) * G.Qt + (int64_t)(pl % G.n3) * RR;
#pragma unroll
      for (int u = 0; u < kQRegs; ++u)
        if (tid + kFwdWorkers * u < RR) qr[u] = __ldg(Qp + tid + kFwdWorkers * u);
    };
    auto split_q = [&](int t) {  // returns the plane's exponent; MMA 1 of the plane before has completed
      float m = 0.f;
#pragma unroll
      for (int u = 0; u < kQRegs; ++u)
        if (tid + kFwdWorkers * u < RR) m = absmax_nan(m, qr[u].x, qr[u].y);
      for (int o = 16; o > 0; o >>= 1) m = max_nan(m, __shfl_xor_sync(0xffffffffu, m, o));
      if (lane == 0) wmax[t & 1][warp] = m;
      asm volatile("bar.sync 1, 512;" ::: "memory");
#pragma unroll
      for (int w = 0; w < kFwdWorkers / 32; ++w) m = max_nan(m, wmax[t & 1][w]);
      const int e = exp_of(m, -117);  // 2^(kDataShift - e) stays finite; Y takes 2^-20 and 2^(e - 1) in turn
      const float sc = pow2f(kDataShift - e);
#pragma unroll
      for (int u = 0; u < kQRegs; ++u)
        if (tid + kFwdWorkers * u < RR) {
          uint32_t h, l;
          split2(qr[u].x * sc, qr[u].y * sc, h, l);
          unsigned char* d = sq + qoff[u];  // rows (Re, -Im), (Im, Re)
          *(uint32_t*)d = h ^ 0x80000000u;
          *(uint32_t*)(d + qterm) = l ^ 0x80000000u;
          *(uint32_t*)(d + 16) = __byte_perm(h, 0, 0x1032);
          *(uint32_t*)(d + qterm + 16) = __byte_perm(l, 0, 0x1032);
        }
      warp_publish(&qready);
      return e;
    };
    fetch_q(0);
    int e = split_q(0), elast = 0;
    if (mine > 1) fetch_q(1);
    int n = 0;
    for (int t = 0; t < mine + lag; ++t) {
      const int eout = lag ? elast : e;  // of the plane that is stored in this pass
      if (t < mine) {
        // S's rows 2 i2, 2 i2 + 1 from D1's row i2: D1 = 2^(kDataShift + kBasisShift - e) S, so 2^-9 D1 < 2^15,
        // and D2 = 2^(21 - e) Y
        waits.warp(&s1done, t & 1);
        tc::fence_after();
        const int r = 32 * q4 + lane;
        if (32 * q4 < T2) {
          unsigned char* so = ss + (size_t)(t & lag) * 2 * sterm;
          for (int c = grp; c < R1p / 4; c += kFwdGroups) {
            uint32_t v[8], hr[4], lr[4], hi[4], li[4];
            tmem_ld8(tmem + (uint32_t)(8 * c) + ((uint32_t)(32 * q4) << 16), v);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              split2(__uint_as_float(v[2 * u]) * 0x1p-9f, __uint_as_float(v[2 * u + 1]) * 0x1p-9f, hr[u], lr[u]);
              hi[u] = __byte_perm(hr[u], 0, 0x1032);
              li[u] = __byte_perm(lr[u], 0, 0x1032);
              hr[u] ^= 0x80000000u;
              lr[u] ^= 0x80000000u;
            }
            if (r < T2) {
              unsigned char* d = so + tc::core_off(2 * r, c, KB);
              *(uint4*)d = make_uint4(hr[0], hr[1], hr[2], hr[3]);
              *(uint4*)(d + sterm) = make_uint4(lr[0], lr[1], lr[2], lr[3]);
              *(uint4*)(d + 16) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
              *(uint4*)(d + sterm + 16) = make_uint4(li[0], li[1], li[2], li[3]);
            }
          }
        }
        tc::fence_before();
        warp_publish(&sready);
        elast = e;
        if (t + 1 < mine) {
          e = split_q(t + 1);
          if (t + 2 < mine) fetch_q(t + 2);
        }
      }
      if (t < lag) continue;
      const float us = pow2f(eout - 1) * gain;
      const int pl = (int)blockIdx.x + (t - lag) * (int)gridDim.x, s = pl / G.n3, i3 = pl - s * G.n3;
      float2* Yp = Y + ldy * s + (int64_t)k * ((int64_t)G.n1 * G.n2 * G.n3) +
                   (int64_t)G.n1 * (i20 + (int64_t)G.n2 * i3) + row0;
      const int left = min(T2, G.n2 - i20);
      for (int b = 0; b < nblk; ++b, ++n) {
        const int d = n & 1, i1 = b * 128 + 32 * q4;
        waits.warp(&done[d], (n >> 1) & 1);
        tc::fence_after();
        if (i1 < rows) {
          const uint32_t t0 = tmem + d2 + (uint32_t)(d * 2 * T2) + ((uint32_t)(32 * q4) << 16);
          float2* y0 = Yp + i1 + lane;
          const bool live = i1 + lane < rows && waits.ok;
          for (int c = grp; c < T2 / 8; c += kFwdGroups) {
            float v[16];
            tc::tmem_ld16(t0 + 16 * c, v);
            float2* y = y0 + (int64_t)G.n1 * 8 * c;
#pragma unroll
            for (int w = 0; w < 8; ++w, y += G.n1)
              if (live && 8 * c + w < left) __stcs(y, make_float2(v[2 * w] * 0x1p-20f * us, v[2 * w + 1] * 0x1p-20f * us));
          }
        }
        tc::fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive1(&dfree[d]);
      }
    }
  }
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, ncols);
}

// ---------------------------------------------------------------------------------------------
// adjoint
// ---------------------------------------------------------------------------------------------
// Walks planes (k, s, i3).  Per tile of 128 i2 (the rows of D) Phi streams through registers in
// chunks of 32 i1: 8 lanes hold a row's 32 entries, take the row's exponent, and write its scaled
// hi / lo words (one 128-byte swizzled row per term) to one of two buffers; the basis rows of the
// chunk (N = 2 NC, split once per handle) arrive by bulk copy.  12 MMAs a chunk (K = 64); the
// accumulator is added into FP32 registers with the row's scale while the next chunk's MMAs run, so
// each tensor-core sum has only 64 terms.  Then V (registers -> shared) is contracted with B2 on the
// CUDA cores into Q, which stays in registers over the plane's tiles.
constexpr int kTile2 = 128;   // i2 rows of a tile
constexpr int kChunk1 = 32;   // i1 per chunk
constexpr uint32_t kATerm = kTile2 * 128u;

inline size_t planes_adj_smem(int NC, int kStage2) {
  return 4 * (size_t)kATerm + 2 * 2 * 2 * (size_t)NC * 128 + sizeof(float2) * kStage2 * ((NC + 15) / 16 * 16);
}

// NC = 8 I >= R1, R2 of every component.  VEC: Phi's columns start on 16 bytes, and a lane reads two
// entries at a time (half the loads; the load unit was the busiest one).
// kStage2: i2 per stage of B2, and per FP32 chain of the contraction with it; RAGGED: the last stage ends with
// the tile's rows.
template <int I, bool VEC, int kStage2, bool RAGGED>
__global__ void __launch_bounds__(kThreads, I <= 4 ? 2 : 1)
    joint_planes_adj_kernel(const __grid_constant__ JointGeo G, const unsigned char* __restrict__ bop,
                            const float2* __restrict__ b2t, const float2* __restrict__ Phi, int64_t ldphi, int p,
                            float2* __restrict__ Q, int* __restrict__ err, uint32_t polls) {
  constexpr int NC = 8 * I, N = 2 * NC, RC = (NC + 15) / 16;  // Q: RC x RC entries a thread
  constexpr int R2p = 16 * RC;
  constexpr uint32_t kBTerm = N * 128u;
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t done[2], full[2], ready[2];
  __shared__ uint32_t tmem_base;
  __shared__ int rexp[4][kTile2];
  unsigned char* sa = smem;                       // [2 buffers][2 terms][128 rows][128 B]; V after a tile
  unsigned char* sb = sa + 4 * kATerm;            // [2 buffers][2 terms][N rows][128 B]
  float2* b2s = (float2*)(sb + 4 * kBTerm);       // [kStage2][R2p]
  float2* vs = (float2*)sa;                       // [NC][128]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr uint32_t ncols = N <= 16 ? 32 : N <= 32 ? 64 : N <= 64 ? 128 : 256;
  if (tid == 0)
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&done[i], 1);
      tc::mbar_init(&full[i], 1);
      tc::mbar_init(&ready[i], 8);
    }
  if (warp == 0) tc::tmem_alloc(&tmem_base, ncols);
  __syncthreads();
  const uint32_t tmem = tmem_base;
  const int nch = (G.n1 + kChunk1 - 1) / kChunk1, nt2 = (G.n2 + kTile2 - 1) / kTile2;
  const int planes = G.n3 * p * G.q;  // plane = k + q (i3 + n3 s); a CTA's planes are blockIdx.x + g gridDim.x
  const int mine = (planes - 1 - (int)blockIdx.x) / (int)gridDim.x + 1;  // grid <= planes
  Waits waits{err, polls};
  if (warp == 8) {
    if (lane == 0) {
      // chunk c of this CTA (all tiles of all its planes in order): its B block is copied once the MMAs
      // of chunk c - 2 have read the buffer
      const int per = nch * nt2, total = mine * per;
      int issued = 0;
      auto copy_b = [&](int c) {
        const int k = ((int)blockIdx.x + c / per * (int)gridDim.x) % G.q, ch = c % nch;
        mbar_arrive_expect_tx(&full[c & 1], 2 * kBTerm);
        bulk_g2s(sb + (size_t)(c & 1) * 2 * kBTerm, bop + ((size_t)k * nch + ch) * 2 * kBTerm, 2 * kBTerm, &full[c & 1]);
        ++issued;
      };
      copy_b(0);
      int c = 0;
      for (; c < total; ++c) {
        const int d = c & 1;
        const uint32_t par = (c >> 1) & 1;
        if (c > 0) waits.one(&done[d ^ 1], ((c - 1) >> 1) & 1);
        if (!waits.ok) break;
        if (c + 1 < total) copy_b(c + 1);
        waits.one(&full[d], par);
        waits.one(&ready[d], par);
        if (!waits.ok) break;
        tc::fence_after();
        const uint32_t a0 = tc::smem_u32(sa) + d * 2 * kATerm, b0 = tc::smem_u32(sb) + d * 2 * kBTerm;
        constexpr uint32_t id = tc::instr_desc(128, N, 0);
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
          const uint64_t ah = tc::smem_desc_sw128(a0 + ks * 32), al = tc::smem_desc_sw128(a0 + kATerm + ks * 32);
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
      // after giving up: the copies in flight land before the buffers are left
      for (int i = c; i < issued; ++i) tc::mbar_wait_idle(&full[i & 1], (i >> 1) & 1);
    }
    __syncwarp();
  } else {
    // a limit known at compile time: 320 x 320 x 256, 8 right-hand sides (I = 3) 1.70 against 1.72 ms, but
    // 194 against 188 us at I = 4 (160 x 160 x 128, 4)
    if (I <= 3) waits.polls = kJointPolls;
    const int64_t nv = (int64_t)G.n1 * G.n2 * G.n3;
    const int row0 = warp * 4 + lane / 8, c8 = lane % 8;  // loader: rows row0 + 32 u, i1 = entry_of(c8, w)
    const int q4 = warp & 3, half = warp >> 2;            // accumulator rows and columns
    const int tx = tid % 16, ty = tid / 16;
    bool bad = false;
    // a work item is one tile of one plane: Phi at the loader's first row and i1, and the tile's rows
    const float2* src = nullptr;
    int rows = 0;
    auto locate = [&](int plane, int t2) {
      const int k = plane % G.q, i3 = plane / G.q % G.n3, s = plane / G.q / G.n3;
      rows = min(kTile2, G.n2 - t2 * kTile2);
      src = Phi + ldphi * s + (int64_t)k * nv + (int64_t)G.n1 * ((int64_t)G.n2 * i3 + t2 * kTile2 + row0) + 2 * c8;
    };
    float2 x[4][4];
    auto fetch = [&](int ch) {
      const int left = G.n1 - ch * kChunk1 - 2 * c8;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float2* g = src + (int64_t)G.n1 * (32 * u) + ch * kChunk1;
        const bool live = row0 + 32 * u < rows;
        if (VEC) {
#pragma unroll
          for (int w = 0; w < 2; ++w) {
            const float4 v = live && 16 * w < left ? __ldcs((const float4*)(g + 16 * w)) : make_float4(0.f, 0.f, 0.f, 0.f);
            x[u][2 * w] = make_float2(v.x, v.y);
            x[u][2 * w + 1] = make_float2(v.z, v.w);
          }
        } else {
#pragma unroll
          for (int w = 0; w < 4; ++w) {
            const int o = (w & 1) + 16 * (w >> 1);
            x[u][w] = live && o < left ? __ldcs(g + o) : make_float2(0.f, 0.f);
          }
        }
      }
    };
    float2 qa[RC][RC];
    int c0 = 0;  // the CTA's chunk number of this item's first chunk
    locate(blockIdx.x, 0);
    fetch(0);
    for (int item = 0; item < mine * nt2; ++item, c0 += nch) {
      const int plane = (int)blockIdx.x + item / nt2 * (int)gridDim.x, t2 = item % nt2, k = plane % G.q;
      if (t2 == 0)
#pragma unroll
        for (int a = 0; a < RC; ++a)
#pragma unroll
          for (int b = 0; b < RC; ++b) qa[a][b] = make_float2(0.f, 0.f);
      float acc[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[c] = 0.f;
      auto fold = [&](int c) {  // also: the MMAs have read chunk c's buffer
        const int d = c & 1;
        waits.warp(&done[d], (c >> 1) & 1);
        tc::fence_after();
        if (32 * q4 < rows) {
          const float us = pow2f(rexp[c & 3][32 * q4 + lane] - 2) * (pow2f(2 - kDataShift - kBasisShift) * lo_first_gain(4));
          const uint32_t t0 = tmem + (uint32_t)(d * N + half * NC) + ((uint32_t)(32 * q4) << 16);
#pragma unroll
          for (int i = 0; i < I; ++i) {
            uint32_t r[8];
            tmem_ld8(t0 + 8 * i, r);
#pragma unroll
            for (int u = 0; u < 8; ++u) acc[8 * i + u] = fmaf(__uint_as_float(r[u]), us, acc[8 * i + u]);
          }
        }
        tc::fence_before();
      };
      for (int ch = 0; ch < nch; ++ch) {
        const int c = c0 + ch, d = c & 1;
        if (ch >= 2) fold(c - 2);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (warp * 4 + 32 * u >= rows) continue;  // rows past the grid: their D rows are not used
          float m = 0.f;
#pragma unroll
          for (int w = 0; w < 4; ++w) m = absmax_nan(m, x[u][w].x, x[u][w].y);
          m = max_nan(m, __shfl_xor_sync(0xffffffffu, m, 1));
          m = max_nan(m, __shfl_xor_sync(0xffffffffu, m, 2));
          m = max_nan(m, __shfl_xor_sync(0xffffffffu, m, 4));
          bad = bad || !(m < INFINITY);
          const int e = exp_of(m, -117), r = row0 + 32 * u;  // 2^(kDataShift - e) stays finite
          if (c8 == 0) rexp[c & 3][r] = e;
          const float sc = pow2f(kDataShift - e);
          uint32_t h[4], l[4];
#pragma unroll
          for (int w = 0; w < 4; ++w) split2(x[u][w].x * sc, x[u][w].y * sc, h[w], l[w]);
          unsigned char* o = sa + (size_t)d * 2 * kATerm + tc::sw128_off(r, c8);
          *(uint4*)o = make_uint4(h[0], h[1], h[2], h[3]);
          *(uint4*)(o + kATerm) = make_uint4(l[0], l[1], l[2], l[3]);
        }
        if (ch + 1 < nch) fetch(ch + 1);
        warp_publish(&ready[d]);
      }
      if (nch > 1) fold(c0 + nch - 2);
      fold(c0 + nch - 1);
      // the next item's first chunk is on its way during the contraction with B2
      const int done_rows = rows;
      if (item + 1 < mine * nt2) {
        locate(t2 + 1 < nt2 ? plane : plane + (int)gridDim.x, t2 + 1 < nt2 ? t2 + 1 : 0);
        fetch(0);
      }
      // V: row i2 = 32 q4 + lane, columns (Re, Im) of x = half NC / 2 + c
#pragma unroll
      for (int c = 0; c < NC / 2; ++c)
        vs[(half * (NC / 2) + c) * kTile2 + 32 * q4 + lane] =
            32 * q4 + lane < done_rows ? make_float2(acc[2 * c], acc[2 * c + 1]) : make_float2(0.f, 0.f);
      const float4* bsrc = (const float4*)(b2t + ((int64_t)k * nt2 + t2) * kTile2 * R2p);
      for (int j0 = 0; j0 < done_rows; j0 += kStage2) {
        const int je = RAGGED ? min(kStage2, done_rows - j0) : kStage2;
        if (j0 > 0) worker_barrier();
#pragma unroll
        for (int e = 0; e < kStage2 * R2p / 512; ++e)
          if (!RAGGED || e * (512 / R2p) < je) ((float4*)b2s)[tid + 256 * e] = __ldg(bsrc + j0 * R2p / 2 + tid + 256 * e);
        worker_barrier();
        float2 qs[RC][RC];  // the stage's sums
        auto pair = [&](int j, bool first) {
          float4 v[RC];
#pragma unroll
          for (int a = 0; a < RC; ++a) {
            const int xx = ty + 16 * a;
            v[a] = NC % 16 == 0 || xx < NC ? *(const float4*)&vs[xx * kTile2 + j0 + j] : make_float4(0.f, 0.f, 0.f, 0.f);
          }
#pragma unroll
          for (int b = 0; b < RC; ++b) {
            const float2 e0 = b2s[j * R2p + tx + 16 * b], e1 = b2s[(j + 1) * R2p + tx + 16 * b];
#pragma unroll
            for (int a = 0; a < RC; ++a) {
              qs[a][b] = cfma_conj(e0, make_float2(v[a].x, v[a].y), first ? make_float2(0.f, 0.f) : qs[a][b]);
              qs[a][b] = cfma_conj(e1, make_float2(v[a].z, v[a].w), qs[a][b]);
            }
          }
        };
        // the first pair peeled where it helps: I = 4 188 -> 183 us (160 x 160 x 128, 4 right-hand sides), I = 6
        // 367 -> 362 us (96^3, 16), but I = 3 1.70 -> 1.77 ms (320 x 320 x 256, 8)
        if (I <= 3)
#pragma unroll
          for (int a = 0; a < RC; ++a)
#pragma unroll
            for (int b = 0; b < RC; ++b) qs[a][b] = make_float2(0.f, 0.f);
        else
          pair(0, true);
#pragma unroll 2
        for (int j = I <= 3 ? 0 : 2; j < je; j += 2) pair(j, false);  // rows past the tile's are zero
#pragma unroll
        for (int a = 0; a < RC; ++a)
#pragma unroll
          for (int b = 0; b < RC; ++b) {
            qa[a][b].x += qs[a][b].x;
            qa[a][b].y += qs[a][b].y;
          }
      }
      worker_barrier();  // V is read before the next item overwrites the buffers
      if (t2 == nt2 - 1) {
        const int i3 = plane / G.q % G.n3, s = plane / G.q / G.n3, R1 = G.R[k][0], R2 = G.R[k][1];
        float2* Qp = Q + (int64_t)s * G.Qt + G.qoff[k] + (int64_t)i3 * R1 * R2;
#pragma unroll
        for (int a = 0; a < RC; ++a)
#pragma unroll
          for (int b = 0; b < RC; ++b) {
            const int xx = ty + 16 * a, y = tx + 16 * b;
            if (xx < R1 && y < R2) Qp[xx + R1 * y] = qa[a][b];
          }
      }
    }
    if (bad) atomicOr(err, kErrNonFinite);
  }
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, ncols);
}

// B1's rows of the adjoint: per component and chunk of 32 i1, [term][2 x + e][64 fp16], 128-byte
// swizzled, the 16-byte chunk c holding i1 = entry_of(c, 0 .. 3); one thread per (row pair, 16-byte chunk)
__global__ void __launch_bounds__(256) split_basis_kernel(const __grid_constant__ JointGeo G,
                                                          const float2* __restrict__ basis, int NC, int nch,
                                                          unsigned char* __restrict__ out) {
  const int k = blockIdx.y, e = blockIdx.x * 256 + threadIdx.x;
  const int c8 = e % 8, x = e / 8 % NC, ch = e / (8 * NC);
  if (ch >= nch) return;
  uint32_t h0[4], l0[4], h1[4], l1[4];
  for (int w = 0; w < 4; ++w) {
    const int i1 = ch * kChunk1 + entry_of(c8, w);
    const float2 v = x < G.R[k][0] && i1 < G.n1 ? basis[G.boff[k][0] + (int64_t)x * G.n1 + i1] : make_float2(0.f, 0.f);
    const float re = v.x * pow2f(kBasisShift), im = v.y * pow2f(kBasisShift);
    split2(re, im, h0[w], l0[w]);
    split2(-im, re, h1[w], l1[w]);
  }
  const size_t term = (size_t)2 * NC * 128;
  unsigned char* o = out + ((size_t)k * nch + ch) * 2 * term;
  *(uint4*)(o + tc::sw128_off(2 * x, c8)) = make_uint4(h0[0], h0[1], h0[2], h0[3]);
  *(uint4*)(o + term + tc::sw128_off(2 * x, c8)) = make_uint4(l0[0], l0[1], l0[2], l0[3]);
  *(uint4*)(o + tc::sw128_off(2 * x + 1, c8)) = make_uint4(h1[0], h1[1], h1[2], h1[3]);
  *(uint4*)(o + term + tc::sw128_off(2 * x + 1, c8)) = make_uint4(l1[0], l1[1], l1[2], l1[3]);
}

int max_r(const JointGeo& G, int m) {
  int r = 0;
  for (int k = 0; k < G.q; ++k) r = std::max(r, G.R[k][m]);
  return r;
}
int adj_rows(const JointGeo& G) { return ceil_div(std::max(max_r(G, 0), max_r(G, 1)), 8) * 8; }
size_t bop_bytes(const JointGeo& G) { return (size_t)G.q * ceil_div(G.n1, kChunk1) * 2 * 2 * adj_rows(G) * 128; }
int b2t_rows(const JointGeo& G) { return ceil_div(G.n2, kTile2) * kTile2; }
int b2t_cols(const JointGeo& G) { return ceil_div(adj_rows(G), 16) * 16; }

// B2 by i2: per component [n2 rounded up to tiles][R2p], zeros past n2 and R2
__global__ void __launch_bounds__(256) transpose_basis_kernel(const __grid_constant__ JointGeo G,
                                                              const float2* __restrict__ basis, int rows, int R2p,
                                                              float2* __restrict__ out) {
  const int k = blockIdx.y, e = blockIdx.x * 256 + threadIdx.x, y = e % R2p, i2 = e / R2p;
  if (i2 >= rows) return;
  out[((int64_t)k * rows + i2) * R2p + y] =
      i2 < G.n2 && y < G.R[k][1] ? basis[G.boff[k][1] + (int64_t)y * G.n2 + i2] : make_float2(0.f, 0.f);
}

template <int I, bool VEC, int kStage2, bool RAGGED>
int launch_planes_adj(const JointGeo& G, const unsigned char* bop, const float2* Phi, int64_t ldphi, int p, float2* Q,
                      int* err, uint32_t polls, cudaStream_t st) {
  const float2* b2t = (const float2*)(bop + bop_bytes(G));
  ZBC_TRY((set_smem_limit<joint_planes_adj_kernel<I, VEC, kStage2, RAGGED>>((int)planes_adj_smem(8 * I, kStage2))));
  const size_t sm = planes_adj_smem(8 * I, kStage2);
  const int64_t planes = (int64_t)G.n3 * p * G.q;
  const int grid = (int)std::min<int64_t>(planes, (sm <= 112 * 1024 ? 2 : 1) * sm_count());
  joint_planes_adj_kernel<I, VEC, kStage2, RAGGED><<<grid, kThreads, sm, st>>>(G, bop, b2t, Phi, ldphi, p, Q, err, polls);
  count_launch();
  ZBC_TRY_CUDA(cudaGetLastError());
  return ZBC_OK;
}

template <int I, int kStage2, bool RAGGED>
int planes_adj_vec(const JointGeo& G, const unsigned char* bop, const float2* Phi, int64_t ldphi, int p, float2* Q,
                   int* err, uint32_t polls, cudaStream_t st) {
  // every column of every plane on 16 bytes, and no pair of entries across the end of one
  if (G.n1 % 2 == 0 && (p == 1 || ldphi % 2 == 0) && (uintptr_t)Phi % 16 == 0)
    return launch_planes_adj<I, true, kStage2, RAGGED>(G, bop, Phi, ldphi, p, Q, err, polls, st);
  return launch_planes_adj<I, false, kStage2, RAGGED>(G, bop, Phi, ldphi, p, Q, err, polls, st);
}

template <int I>
int planes_adj(const JointGeo& G, const unsigned char* bop, const float2* Phi, int64_t ldphi, int p, float2* Q, int* err,
               uint32_t polls, cudaStream_t st) {
  // Up to rank 24 stages of 64 i2 where they hold no more padding than stages of 32: 1.68 against 1.70 ms for
  // n2 = 320 (8 right-hand sides), 4.02 against 4.10 ms for 309 (32).  Where stages of 32 would pad by a
  // sixteenth or more, stages of 64 of which the last ends with its rows: 138 against 160 us for 66 (29), 379
  // against 410 us for 74 (13), 78 against 83 us for 135 (11); the loop without a fixed length costs a few per
  // cent, 1.49 against 1.46 ms for 93 (12), and one stage of 31 rows 235 against 229 us.  Above rank 24 a second
  // CTA an SM, or the registers, would not fit.
  if constexpr (I <= 3) {
    const int rows32 = ceil_div(G.n2, 32) * 32;
    if (ceil_div(G.n2, 64) * 64 == rows32)
      return planes_adj_vec<I, 64, false>(G, bop, Phi, ldphi, p, Q, err, polls, st);
    if (G.n2 > 64 && (rows32 - G.n2) * 16 >= G.n2) return planes_adj_vec<I, 64, true>(G, bop, Phi, ldphi, p, Q, err, polls, st);
  }
  return planes_adj_vec<I, 32, false>(G, bop, Phi, ldphi, p, Q, err, polls, st);
}

}  // namespace

int joint_planes_fwd(const JointCache& jc, const float2* Q, int p, float2* Y, int64_t ldy, int* err, uint32_t polls,
                     cudaStream_t st) {
  const JointGeo& G = jc.geo;
  constexpr size_t kLimit = 224 * 1024;
  // balanced tiles of i2 that leave tensor memory for D1 and two D2; where the operands do not fit
  // shared memory together, one copy of S, then fewer i1 blocks, then smaller tiles
  FwdShape F;
  F.R1p = ceil_div(max_r(G, 0), 8) * 8;
  F.R2p = ceil_div(max_r(G, 1), 8) * 8;
  const int nblk = ceil_div(G.n1, 128), t2max = (512 - 2 * F.R1p) / 4 / 16 * 16;
  for (F.nt2 = ceil_div(G.n2, t2max);; ++F.nt2) {
    F.T2 = ceil_div(ceil_div(G.n2, F.nt2), 16) * 16;
    F.nb = nblk;
    F.ns = 2;
    if (F.bytes(G.n1) > kLimit) F.ns = 1;
    while (F.nb > 1 && F.bytes(G.n1) > kLimit) --F.nb;
    if (F.bytes(G.n1) <= kLimit) break;  // 16 i2, one block, one S: at most 213 KB
  }
  F.nt2 = ceil_div(G.n2, F.T2);
  F.gy = ceil_div(nblk, F.nb);
  ZBC_TRY(set_smem_limit<joint_planes_fwd_kernel>((int)kLimit));
  const int walkers = std::min(p * G.n3, std::max(1, sm_count() / (F.gy * F.nt2 * G.q)));
  joint_planes_fwd_kernel<<<dim3(walkers, F.gy * F.nt2, G.q), kFwdThreads, F.bytes(G.n1), st>>>(G, F, jc.basis, Q, p, Y, ldy,
                                                                                            err, polls);
  count_launch();
  ZBC_TRY_CUDA(cudaGetLastError());
  return ZBC_OK;
}

int joint_planes_adj(const JointCache& jc, const float2* Phi, int64_t ldphi, int p, float2* Q, int* err, uint32_t polls,
                     cudaStream_t st) {
  const JointGeo& G = jc.geo;
  switch (adj_rows(G) / 8) {
    case 1: return planes_adj<1>(G, jc.bop, Phi, ldphi, p, Q, err, polls, st);
    case 2: return planes_adj<2>(G, jc.bop, Phi, ldphi, p, Q, err, polls, st);
    case 3: return planes_adj<3>(G, jc.bop, Phi, ldphi, p, Q, err, polls, st);
    case 4: return planes_adj<4>(G, jc.bop, Phi, ldphi, p, Q, err, polls, st);
    case 5: return planes_adj<5>(G, jc.bop, Phi, ldphi, p, Q, err, polls, st);
    case 6: return planes_adj<6>(G, jc.bop, Phi, ldphi, p, Q, err, polls, st);
    case 7: return planes_adj<7>(G, jc.bop, Phi, ldphi, p, Q, err, polls, st);
    default: return planes_adj<8>(G, jc.bop, Phi, ldphi, p, Q, err, polls, st);
  }
}

size_t joint_planes_bytes(const JointGeo& G) {
  return bop_bytes(G) + sizeof(float2) * (size_t)G.q * b2t_rows(G) * b2t_cols(G);
}

int joint_planes_build(const JointGeo& G, const float2* basis, unsigned char* bop, cudaStream_t st) {
  const int NC = adj_rows(G), nch = ceil_div(G.n1, kChunk1);
  split_basis_kernel<<<dim3(ceil_div((int64_t)nch * NC * 8, 256), G.q), 256, 0, st>>>(G, basis, NC, nch, bop);
  const int rows = b2t_rows(G), cols = b2t_cols(G);
  transpose_basis_kernel<<<dim3(ceil_div((int64_t)rows * cols, 256), G.q), 256, 0, st>>>(G, basis, rows, cols,
                                                                                         (float2*)(bop + bop_bytes(G)));
  count_launch(2);
  ZBC_TRY_CUDA(cudaGetLastError());
  return ZBC_OK;
}

}  // namespace zbc
