// Joint-subspace form of the products (joint_build.cu, products_joint.cu).
//
// Every stored column of component k is Z^{kj} = G x1 U1 x2 U2 x3 U3 with factors of its own, but
// the factors of all columns are fields of the same domain and span few directions together (the
// 96^3 head-coil workload: 47-52 directions per axis for 1024 columns of rank 11; the 1 mm grid:
// 23-25 of 320).  With an orthonormal basis B_g (n_g x R_g) of that span per component and mode,
//   Z^{kj} = K^{kj} x1 B1 x2 B2 x3 B3,   K^{kj} = G x1 (B1^H U1) x2 (B2^H U2) x3 (B3^H U3),
// so  Y^k = (sum_j K^{kj} X[j, :]) x1 B1 x2 B2 x3 B3  and the adjoint is its transpose: the sum
// over the columns runs over R1 R2 R3 entries instead of n1 n2 n3 voxels, and the expansion to the
// grid is done once per right-hand side instead of once per column.  This is the same operator to
// the tolerance kJointEps, of the size of the complex64 tensors' rounding.
#pragma once

#include "zbc_internal.cuh"

namespace zbc {

constexpr int kJointQ = 12;      // components of a handle (q <= 12)
constexpr int kJointRmax = 64;   // largest R_g
// largest residual of a tensor's weighted factor outside the basis, relative to its norm.  The
// complex64 rounding of the factors is 6e-8 of their norm; at 1e-7 the products' error against
// 64 bits is that of their FP32 sums.
constexpr double kJointEps = 1e-7;

struct JointGeo {
  int n1, n2, n3, q, M;
  int R[kJointQ][3];
  int Cs[kJointQ];        // R1 R2 R3 rounded up to 4 (row stride of K)
  int64_t koff[kJointQ];  // component k's rows [j][Cs] in K
  int64_t boff[kJointQ][3];  // B_g in the basis array: column r at boff + r n_g
  int64_t toff[kJointQ];  // component k's entries in one right-hand side of T / F
  int64_t qoff[kJointQ];  // component k's planes [i3][R1 R2] in one right-hand side of Q
  int64_t Ct, Qt;         // entries of one right-hand side of T / F and of Q
};

constexpr int kJointPass = 64;  // right-hand sides that the products' workspaces hold at a time

struct JointCache {
  bool usable = false;    // false: the factors share no small basis (the other forms are used)
  bool large = false;     // the products decompress more than 1e8 voxel ranks
  bool untuned_use = false;  // products of untuned classes ran it: captured graphs may hold its operands
  bool no_room = false;   // unusable for want of device memory: zbc_tune tries again
  JointGeo geo;
  float2* basis = nullptr;
  float2* K = nullptr;
  unsigned char* bop = nullptr;  // B1 split for the adjoint's plane product (joint_planes.cu)
  float* kscale = nullptr;       // power-of-two scales of K's columns (joint_core.cu)
  int64_t bytes = 0;
  // workspace bytes of a product (adjoint, forward) of up to p right-hand sides: the largest of every
  // plan up to p.  The plans of few right-hand sides cut the column sum into more slices and may take
  // more than those of more, and a buffer that grows for them would leave a captured graph without its own.
  size_t work[2][kJointPass + 1] = {};
};

// the plane products on the tensor cores (joint_planes.cu): Y from Q, and Q from Phi
size_t joint_planes_bytes(const JointGeo& G);
int joint_planes_build(const JointGeo& G, const float2* basis, unsigned char* bop, cudaStream_t st);
// (polls: tries of each bounded wait, about a microsecond each)
constexpr uint32_t kJointPolls = 1000000;
int joint_planes_fwd(const JointCache& jc, const float2* Q, int p, float2* Y, int64_t ldy, int* err, uint32_t polls,
                     cudaStream_t st);
int joint_planes_adj(const JointCache& jc, const float2* Phi, int64_t ldphi, int p, float2* Q, int* err, uint32_t polls,
                     cudaStream_t st);

// the column sums on the tensor cores (joint_core.cu): T from X, and partial Psi from F in `splits`
// slices of `split` chunks of core entries
size_t joint_core_bytes(const JointGeo& G);
int joint_core_build(const JointGeo& G, const float2* K, float* kscale, bool* fits, cudaStream_t st);
int joint_core_fwd(const JointCache& jc, const float2* X, int64_t ldx, int p, float2* T, int* err, uint32_t polls,
                   cudaStream_t st);
void joint_core_split(const JointGeo& G, int p, int* split, int* splits);
int joint_core_adj(const JointCache& jc, const float2* F, int p, float2* part, int* err, uint32_t polls, cudaStream_t st);

// Builds h.joint (synchronises).  Returns ZBC_OK also when no small basis exists: see usable.
int build_joint(Handle& h, cudaStream_t st);
void joint_plan_work(JointCache* jc);  // fills work from geo
// bytes of h.work_joint_fwd / _adj that a product of p right-hand sides needs (h.joint usable)
inline size_t joint_work_bytes(const Handle& h, int p, bool fwd) {
  return h.joint->work[fwd][p < kJointPass ? p : kJointPass];
}
int matvec_joint(Handle& h, const float2* X, int64_t ldx, int p, float2* Y, int64_t ldy, cudaStream_t st);
int rmatvec_joint(Handle& h, const float2* Phi, int64_t ldphi, int p, float2* out, int64_t ldo, cudaStream_t st);

}  // namespace zbc
